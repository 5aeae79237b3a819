"""hx_rotate_hoisted: every output in its own handle, written there; bit-exact against the oracle over
groups of several launches, with identity steps between."""
import numpy as np
import pytest

import mempool
from oracle import ckks as C
from paper_2207_04620_gb300 import hx, workloads

from hxpair import PARAMS, Pair

pytestmark = pytest.mark.gpu


PARAMS["hoisted_general"] = dict(log_n=12, q_bits=[60, 45, 45, 45, 45], p_bits=[61, 60], log2_scale=45)


@pytest.fixture(scope="module", params=["alg3", "hoisted_general"])  # the second: outside fold arithmetic
def pair(request):
    from paper_2207_04620_gb300 import build

    build.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pr = Pair(request.param, rot_steps=[1, -3])
    yield pr
    pr.close()


def _input(pr, limbs, comps=2):
    return C.Ciphertext(workloads.residues(limbs, pr.octx.q[:limbs], comps, pr.N).reshape(comps, limbs, pr.N), 2.0 ** 45)


@pytest.mark.parametrize("limbs", [1, 5])
@pytest.mark.parametrize("steps", [[], [0], [1], [-3, 0, 1], [0] + [1, -3] * 17 + [0, 0, -3], [1] * 32 + [-3] * 33])
def test_outputs_in_order(pair, limbs, steps):
    ct = _input(pair, limbs)
    ev = C.Evaluator(pair.octx, pair.oks)
    want = {k: ev.rotate_hoisted(ct, [k])[0] for k in set(steps)}
    a = pair.to_lib(ct)
    got = hx.hx_rotate_hoisted(pair.ctx, pair.ks, a, steps)
    hx.hx_ct_destroy(a)
    assert len(got) == len(steps)
    for i, k in enumerate(steps):  # a destroyed handle leaves the others alone
        assert pair.same(got[i], want[k])
        hx.hx_ct_destroy(got[i])


def test_outputs_are_held_once(pair):
    """256 rotations take their outputs' memory and one group's temporaries, not the outputs twice."""
    import torch

    limbs, n = 5, 256
    row = pair.N * 8
    out = n * 2 * limbs * row
    ext = limbs + 2
    group = 32 * 2 * (ext + limbs) * row   # at most 32 rotations: the extended pairs and the converted rows
    modup = (3 * ext + limbs) * row        # three digits, the coefficients
    a = pair.to_lib(_input(pair, limbs))
    torch.cuda.synchronize()
    mempool.reset_peak()
    before = mempool.used()
    got = hx.hx_rotate_hoisted(pair.ctx, pair.ks, a, [1, -3] * (n // 2))
    torch.cuda.synchronize()
    assert mempool.peak() - before <= out + group + modup + (4 << 20)
    for h in got + [a]:
        hx.hx_ct_destroy(h)


def test_identity_copies_three_components(pair):
    """A step of 0 mod N/2 copies a product before its relinearisation whole, in hx_rotate and here."""
    ct = _input(pair, 4, comps=3)
    a = pair.to_lib(ct)
    for h in [hx.hx_rotate(pair.ctx, pair.ks, a, 0)] + hx.hx_rotate_hoisted(pair.ctx, pair.ks, a, [0, pair.N // 2]):
        assert pair.same(h, ct)
