"""What this framework's users have it do, as timed cases.

Every case goes through the public entry points (include/hx.h, hx.py).  Ciphertext words are
integers modulo primes, so every result but a decrypted slot is compared word for word.  A
program keeps its context, its evaluation keys and a product's plan for as long as it serves one
ring; they are made once per ring here, and a state's inputs come from its seed alone.
Results that live in a library handle leave it as they do in a server that answers a request:
by hx_ct_export into a page-locked buffer.  Parameter sets are those of the benchmark
(paper_2207_04620_gb300/workloads.py) and of the tests, or of the same form: a chain of one
60-bit prime and primes of the scale's size, with 60-bit special primes.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2207_04620_gb300 import hx, workloads

_RINGS: dict = {}
_PLANS: dict = {}


def listed():
    return [
        # the smallest call of the method: one rotation of one ciphertext of config 0's ring,
        # on device buffers, where launches and latency are all there is
        dict(name="rotate one, N=2^12", kind="rotate", log_n=12, limbs=3, bits=40, special=1, step=5),
        # forward transforms at the size where only the kernels count (200 polynomials, 8 limbs)
        dict(name="ntt 1600 rows, N=2^14", kind="ntt", log_n=14, limbs=8, polys=200, bits=45, inverse=False),
        # inverse transforms of an odd log N and a ragged batch (19 primes: config 2's chain and specials)
        dict(name="intt 399 rows, N=2^15", kind="ntt", log_n=15, limbs=19, polys=21, bits=40, inverse=True),
        # Mul_ct, RS and Rot of one ciphertext: the ordinary single-ciphertext step of a user's circuit
        dict(name="mul+rotate one, N=2^14", kind="chain", log_n=14, limbs=8, bits=45, special=2, step=3),
        # config 0: one small product with two levels (the depth-2 schedule), an interactive request
        dict(name="matmul 16, N=2^12", kind="matmul", log_n=12, limbs=3, bits=40, special=1, h=16, pairs=1,
             form="one"),
        # an uneven batch of a smaller ring through the batched call, a server's ordinary batch
        dict(name="matmul 32 x5, N=2^13", kind="matmul", log_n=13, limbs=7, bits=45, special=2, h=32, pairs=5,
             form="batch"),
        # config 1, the headline: 16 pairs (32 products) through the executor from host buffers
        dict(name="matmul 64 x16, N=2^14", kind="matmul", log_n=14, limbs=8, bits=45, special=2, h=64, pairs=16,
             form="graph"),
        # config 2: the composite sign of 64 ciphertexts with both collective refreshes
        dict(name="sign x64, N=2^15", kind="sign", log_n=15, limbs=16, bits=40, special=3, alpha=4, count=64, d=4,
             k=8, relu=False),
        # a layer forward and backward (Fig. 5): products, sign, transpose, gradient
        dict(name="dense layer, N=2^14", kind="dense", log_n=14, limbs=16, bits=40, special=3, h=32, n_in=200,
             rows=64, k=2),
        # the client's two directions: encode + encrypt a batch, decrypt + decode it
        dict(name="client x12, N=2^14", kind="client", log_n=14, limbs=8, bits=45, special=2, count=12),
        # a server's mix of small requests over three rings in one call
        dict(name="rotate 24, three rings", kind="rings", log_n=12, limbs=4, bits=45, special=2, count=24),
        # the aggregation server's update: 16 parties, 8 model ciphertexts
        dict(name="aggregate 16x8, N=2^15", kind="aggregate", log_n=15, limbs=16, bits=40, special=3, parties=16,
             count=8),
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.99)))))))


def draw(rng):
    kind = rng.choice(["ntt", "ntt", "rotate", "chain", "matmul", "matmul", "sign", "sign", "client", "rings",
                       "aggregate", "dense"])
    bits = rng.choice([36, 40, 45, 50, 55])
    special = rng.randint(1, 3)
    if kind == "ntt":
        log_n, limbs = rng.randint(11, 16), rng.randint(1, 24)
        polys = _log_int(rng, 1, max(1, (1 << 26 >> log_n) // limbs))
        return dict(kind=kind, log_n=log_n, limbs=limbs, polys=polys, bits=bits, inverse=rng.random() < 0.5)
    if kind == "rotate":
        log_n = rng.randint(11, 14)
        limbs = rng.randint(2, {11: 20, 12: 14, 13: 9, 14: 6}[log_n])
        return dict(kind=kind, log_n=log_n, limbs=limbs, bits=bits, special=max(2, special), step=rng.randint(1, 1000))
    if kind == "chain":
        return dict(kind=kind, log_n=rng.randint(11, 16), limbs=rng.randint(2, 18), bits=bits, special=special,
                    step=rng.randint(1, 1000))
    if kind == "matmul":
        log_n = rng.randint(11, 14)
        h = 1 << rng.randint(2, min(6, (log_n - 1) // 2))
        return dict(kind=kind, log_n=log_n, limbs=rng.randint(3, 9), bits=rng.choice([40, 45, 50]), special=2, h=h,
                    pairs=_log_int(rng, 1, 12), form=rng.choice(["one", "batch", "graph"]))
    if kind == "sign":
        # a composition takes four levels, the last product of ReLU one more
        return dict(kind=kind, log_n=rng.randint(11, 15), limbs=rng.randint(6, 18), bits=40, special=3,
                    alpha=rng.choice([0, 4]), count=_log_int(rng, 1, 48), d=rng.randint(1, 4), k=rng.randint(1, 4),
                    relu=rng.random() < 0.5)
    if kind == "client":
        return dict(kind=kind, log_n=rng.randint(11, 15), limbs=rng.randint(1, 12), bits=rng.choice([36, 40, 45]),
                    special=special, count=_log_int(rng, 1, 24))
    if kind == "rings":
        return dict(kind=kind, log_n=rng.randint(11, 13), limbs=rng.randint(2, 8), bits=bits, special=max(2, special),
                    count=_log_int(rng, 3, 48))
    if kind == "aggregate":
        return dict(kind=kind, log_n=rng.randint(12, 15), limbs=rng.randint(2, 16), bits=40, special=3,
                    parties=_log_int(rng, 1, 24), count=rng.randint(1, 8))
    return dict(kind="dense", log_n=rng.choice([12, 13]), limbs=rng.randint(14, 17), bits=40, special=3, h=16,
                n_in=rng.randint(5, 100), rows=rng.randint(5, 48), k=1)


# ---- rings, keys and plans: made once, kept ------------------------------------------------------

def _ring(case, n_q=None, log_n=None):
    """The context of a case's chain."""
    log_n, n_q = log_n or case["log_n"], n_q or case["limbs"]
    key = (log_n, n_q, case["bits"], case.get("special", 1), case.get("alpha", 0))
    if key not in _RINGS:
        _RINGS[key] = [hx.hx_context_create(log_n, [60] + [case["bits"]] * (n_q - 1), [60] * case.get("special", 1),
                                            case["bits"], alpha=case.get("alpha", 0)), None, set()]
    return _RINGS[key]


def _keys(ring, steps):
    """The ring's key set with Galois keys for these rotation steps."""
    ctx, ks, have = ring
    if ks is None:
        ring[1] = hx.hx_keygen(ctx, 2, 81, sorted(steps))
    elif not steps <= have:
        hx.hx_keyset_add_rotations(ctx, ks, sorted(steps - have))
    have |= steps
    return ring[1]


class _State:
    """A case's inputs and buffers; ciphertext handles go back with it."""

    def __init__(self, case):
        self.case, self.held, self.ex = case, [], None

    def hold(self, handles):
        self.held += handles
        return handles

    def __del__(self):
        if self.ex is not None:
            hx.hx_matmul_exec_destroy(self.ex)
        for c in self.held:
            hx.hx_ct_destroy(c)


def _export(handles, buf):
    """The handles' residues, one after another, into the page-locked buffer; frees the handles."""
    at, lib = buf.data_ptr(), hx.lib()
    left = buf.numel()
    for c in handles:
        words = lib.hx_ct_export(c, ctypes.cast(at, hx.P_u64), left)
        hx.hx_ct_destroy(c)
        if words < 0:
            raise RuntimeError("export failed: %d" % words)
        at, left = at + 8 * words, left - words
    return buf


def _pinned(words):
    return torch.zeros(int(words), dtype=torch.int64).pin_memory()


def _residues(seed, primes, polys, n):
    """Uniform residues [polys][len(primes)][n] on the device."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randint(0, (1 << 63) - 1, (polys, len(primes), n), dtype=torch.int64, device="cuda", generator=g)
    for i, q in enumerate(primes):
        x[:, i] %= q
    return x


def _out_limbs(case):
    """Limbs of a product's or sign's result."""
    if case["kind"] == "matmul":
        return case["limbs"] - 3 if case["limbs"] >= 4 else 1
    depth = min(case["d"], 3) + 1
    left = case["limbs"]
    for it in range(case["k"]):
        if left - 1 < depth + (1 if case["relu"] and it == case["k"] - 1 else 0):
            left = case["limbs"]
        left -= depth
    return left - (1 if case["relu"] else 0)


# ---- prepare and run ----------------------------------------------------------------------------

def prepare(case, seed):
    s = _State(case)
    kind, log_n, limbs = case["kind"], case["log_n"], case["limbs"]
    n = 1 << log_n
    rng = np.random.default_rng(seed)
    if kind == "ntt":
        ring = _ring(case)
        s.ctx = ring[0]
        s.primes = list(range(limbs))
        s.x = _residues(seed, hx.hx_context_primes(s.ctx)[:limbs], case["polys"], n)
        return s
    if kind == "rotate":
        ring = _ring(case)
        s.ctx, s.ks = ring[0], _keys(ring, {case["step"]})
        s.x = _residues(seed, hx.hx_context_primes(s.ctx)[:limbs], 2, n)
        s.out = torch.empty_like(s.x)
        return s
    if kind == "rings":
        s.jobs, words = [], 0
        for i in range(case["count"]):
            j = i % 3
            level = max(1, limbs - i % 4 % limbs)
            ring = _ring(case, log_n=log_n + j)
            ks = _keys(ring, {1, 3, 5})
            z = rng.uniform(-1, 1, (1, n << j >> 1))
            ct = s.hold(hx.hx_encrypt_batch(ring[0], ks, z, [seed + i], level))[0]
            s.jobs.append((ring[0], ks, ct, (1, 3, 5)[i // 3 % 3]))
            words += 2 * level * (n << j)
        s.host = _pinned(words)
        return s
    ring = _ring(case)
    s.ctx = ctx = ring[0]
    if kind == "chain":
        s.ks = _keys(ring, {case["step"]})
        s.a, s.b = s.hold(hx.hx_encrypt_batch(ctx, s.ks, rng.uniform(-1, 1, (2, n // 2)), [seed, seed + 1]))
        s.host = _pinned(2 * (limbs - 1) * n)
    elif kind == "matmul":
        h, pairs = case["h"], case["pairs"]
        beta = n // 2 // (h * h)
        s.ks = _keys(ring, set(hx.hx_matmul_rotation_steps(ctx, h, limbs)))
        z = rng.uniform(-1, 1, (2 * pairs, beta * h * h))
        cts = s.hold(hx.hx_encrypt_batch(ctx, s.ks, z, [seed * 64 + i for i in range(2 * pairs)]))
        s.A, s.B = cts[:pairs], cts[pairs:]
        s.host = _pinned(pairs * 2 * _out_limbs(case) * n)
        if case["form"] == "graph":
            key = (ctx, h, limbs)
            if key not in _PLANS:
                plan = hx.hx_matmul_plan_create(ctx, h, limbs)
                if limbs >= 4:
                    hx.hx_matmul_plan_bind_keys(ctx, plan, s.ks)
                _PLANS[key] = plan
            scale = hx.hx_ct_info(cts[0])[2]
            s.ex = hx.hx_matmul_exec_create(ctx, s.ks, _PLANS[key], pairs, scale)
            s.host_a, s.host_b = _pinned(pairs * 2 * limbs * n), _pinned(pairs * 2 * limbs * n)
            _export(s.A, s.host_a)
            _export(s.B, s.host_b)
            s.held = []
    elif kind == "sign":
        s.ks = _keys(ring, set())
        z = np.stack([workloads.sign_inputs(seed * 64 + i, n // 2) for i in range(case["count"])])
        s.x = s.hold(hx.hx_encrypt_batch(ctx, s.ks, z, [seed * 64 + i for i in range(case["count"])]))
        s.seed = seed
        s.host = _pinned(case["count"] * 2 * _out_limbs(case) * n)
    elif kind == "dense":
        h = case["h"]
        beta = n // 2 // (h * h)
        s.ks = _keys(ring, set(hx.hx_dense_rotation_steps(ctx, h)))
        W, X, G = workloads.dense_inputs(seed, case["rows"], case["n_in"], h)
        Wp, Xp, Gp = workloads.dense_pack(W, X, G, h, beta)
        s.n_out, s.groups, s.seed = len(Wp), len(Xp), seed
        z = np.stack([Wp[i][g] for i in range(s.n_out) for g in range(s.groups)] + Xp + Gp)
        cts = s.hold(hx.hx_encrypt_batch(ctx, s.ks, z, [seed * 64 + i for i in range(len(z))]))
        nw = s.n_out * s.groups
        s.W, s.X, s.G = cts[:nw], cts[nw: nw + s.groups], cts[nw + s.groups:]
        s.host = _pinned(2 * limbs * n * (2 * s.n_out + nw))
    elif kind == "client":
        s.ks = _keys(ring, set())
        s.z = rng.uniform(-1, 1, (case["count"], n // 2))
        s.seeds = [seed * 64 + i for i in range(case["count"])]
        s.host = _pinned(case["count"] * 2 * limbs * n)
    elif kind == "aggregate":
        s.ks = _keys(ring, set())
        parties, count = case["parties"], case["count"]
        z = np.concatenate([rng.normal(0, 0.05, (count, n // 2)), rng.normal(0, 0.01, (count, n // 2))])
        cts = s.hold(hx.hx_encrypt_batch(ctx, s.ks, z, [seed * 64 + i for i in range(2 * count)]))
        s.models, s.grads = cts[:count], []
        for i in range(parties):  # every party's ciphertext of the same gradient, under its own randomness
            s.grads += s.hold(hx.hx_encrypt_batch(ctx, s.ks, z[count:] * (1 + 0.01 * i),
                                                  [(seed + 1) * 4096 + i * 64 + m for m in range(count)]))
        s.host = _pinned(count * 2 * (limbs - 1) * n)
    return s


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "ntt":
        hx.hx_ntt(s.ctx, s.x.data_ptr(), case["polys"], s.primes, inverse=case["inverse"])
        return s.x
    if kind == "rotate":
        hx.hx_rotate_noalloc(s.ctx, s.ks, s.x.data_ptr(), case["limbs"], s.out.data_ptr(), case["step"])
        return s.out
    if kind == "rings":
        return _export(hx.hx_rotate_jobs(s.jobs), s.host)
    ctx, ks = s.ctx, s.ks
    if kind == "chain":
        t = hx.hx_tensor(ctx, s.a, s.b)
        m = hx.hx_relinearize(ctx, ks, t)
        r = hx.hx_rescale(ctx, m)
        out = hx.hx_rotate(ctx, ks, r, case["step"])
        for c in (t, m, r):
            hx.hx_ct_destroy(c)
        return _export([out], s.host)
    if kind == "matmul":
        if case["form"] == "graph":
            hx.hx_matmul_exec_run_host(s.ex, s.host_a.data_ptr(), s.host_b.data_ptr(), s.host.data_ptr())
            return s.host
        if case["form"] == "batch":
            return _export(hx.hx_matmul_batch(ctx, ks, None, s.A, s.B, case["h"]), s.host)
        return _export([hx.hx_matmul(ctx, ks, a, b, case["h"]) for a, b in zip(s.A, s.B)], s.host)
    if kind == "sign":
        return _export(hx.hx_sign_approx_batch(ctx, ks, s.x, case["d"], case["k"], relu=case["relu"],
                                               refresh_seed=s.seed), s.host)
    if kind == "dense":
        E, M, dW = hx.hx_dense_layer(ctx, ks, s.W, s.X, s.G, case["h"], s.n_out, s.groups, 4, case["k"], 4.0,
                                     refresh_seed=s.seed)
        return _export(E + M + dW, s.host)
    if kind == "client":
        cts = hx.hx_encrypt_batch(ctx, ks, s.z, s.seeds)
        slots = [hx.hx_decrypt(ctx, ks, c) for c in cts]
        return {"ciphertexts": _export(cts, s.host), "slots": np.stack(slots)}
    return _export(hx.hx_aggregate(ctx, s.grads, case["parties"], s.models, 0.1 / (4 * case["parties"])), s.host)


# ---- what a pass cannot do without ---------------------------------------------------------------

def _ntt_ops(n, rows):
    """Butterflies of `rows` transforms, a modular product and two additions each."""
    return 3.0 * rows * (n / 2) * math.log2(n)


def _switch(n, limbs, special, alpha, count=1, hoisted=False):
    """(key bytes, operations of `count` key switches): ModUp, inner product, ModDown."""
    digits, ext = -(-limbs // alpha), limbs + special
    up = _ntt_ops(n, limbs + digits * ext - limbs) + 2.0 * n * digits * alpha * ext
    down = _ntt_ops(n, 2 * ext) + 2.0 * n * 2 * special * limbs
    ip = 4.0 * n * digits * ext
    return 16.0 * n * digits * ext, (up / count if hoisted else up) * count + (ip + down) * count


def work(case):
    """Inputs, keys and results once over; the modular operations of the transforms, conversions
    and inner products (a multiplication and an addition are two)."""
    kind, n, limbs = case["kind"], 1 << case["log_n"], case["limbs"]
    special = case.get("special", 1)
    alpha = case.get("alpha", 0) or special
    ct = 16.0 * n * limbs
    if kind == "ntt":
        rows = limbs * case["polys"]
        return {"bytes": 16.0 * n * rows, "flops": _ntt_ops(n, rows)}
    kb, ko = _switch(n, limbs, special, alpha)
    if kind == "rotate":
        return {"bytes": 2 * ct + kb, "flops": ko}
    if kind == "rings":
        per = case["count"] / 3
        return {"bytes": 7 * (per * 2 * ct + 3 * kb), "flops": 7 * per * ko}
    if kind == "chain":
        return {"bytes": 3 * ct + 2 * kb, "flops": 2 * ko + 8.0 * n * limbs}
    if kind == "matmul":
        # Alg. 3: the rotations of U^zeta, U^mu and of Steps 2 and 4, most of them hoisted
        rot = 3 * case["h"] + 5 * math.sqrt(case["h"])
        kb, ko = _switch(n, limbs, special, alpha, int(rot), hoisted=True)
        return {"bytes": 3 * ct * case["pairs"] + rot * kb, "flops": ko * case["pairs"]}
    if kind == "sign":
        # a composition: four products at falling levels
        prods = case["k"] * (min(case["d"], 3) + 1)
        return {"bytes": 2 * ct * case["count"] + kb, "flops": 0.5 * prods * ko * case["count"]}
    if kind == "dense":
        h, beta = case["h"], n // 2 // (case["h"] * case["h"])
        n_out, groups = -(-case["rows"] // h), -(-(-(-case["n_in"] // h)) // beta)
        rot = 8 * h
        kb, ko = _switch(n, limbs, special, alpha, rot, hoisted=True)
        return {"bytes": ct * (3 * n_out * groups + 2 * groups) + rot * kb, "flops": 0.5 * ko * n_out * groups}
    if kind == "client":
        return {"bytes": case["count"] * (ct + 8.0 * n), "flops": case["count"] * (_ntt_ops(n, 4 * limbs))}
    sums = (case["parties"] + 2) * case["count"]
    return {"bytes": sums * ct, "flops": 2.0 * sums * 2 * n * limbs + _ntt_ops(n, 2 * limbs * case["count"])}


def tolerance(case):
    # residues are whole numbers; decrypted slots go through one FP64 transform of the same
    # integers, where another order of its log N sums differs by a few units in the last place
    return {"rel": 1e-14} if case["kind"] == "client" else "exact"


def exact(case, seed):
    """Decrypted slots against the encrypted numbers; the residues have no 64-bit float value."""
    if case["kind"] != "client":
        return None
    z = np.random.default_rng(seed).uniform(-1, 1, (case["count"], (1 << case["log_n"]) // 2))
    return {"ciphertexts": None, "slots": z}
