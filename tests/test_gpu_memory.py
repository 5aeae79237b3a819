"""Grouped rotations on a device without room for their buffers: the calls fall back to one rotation at
a time, as they ran before there were groups, with the same results.  The shortage is a memory pool with
a limit of its own, or for a captured product a tensor that holds the rest of the device."""
import numpy as np
import pytest

import mempool
from paper_2207_04620_gb300 import hx, workloads

pytestmark = pytest.mark.gpu

LOG_N, Q, P, H = 13, [60] + [45] * 6, [60, 60], 32


@pytest.fixture(scope="module")
def ring():
    from paper_2207_04620_gb300 import build

    build.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = hx.hx_context_create(LOG_N, Q, P, 45)
    steps = set(hx.hx_matmul_rotation_steps(ctx, H, len(Q))) | set(hx.hx_transpose_rotation_steps(ctx, H))
    steps |= set(hx.hx_matmul_rotation_steps(ctx, H, 3))
    ks = hx.hx_keygen(ctx, 1, 17, sorted(steps))
    yield ctx, ks, sorted(steps)
    hx.hx_keyset_destroy(ks)
    hx.hx_context_destroy(ctx)


def _batch(ctx, ks, count, limbs, seed):
    beta = (1 << LOG_N) // 2 // (H * H)
    z = np.stack([workloads.pack(workloads.matrices(seed + i, beta, H), H, beta) for i in range(count)])
    return hx.hx_encrypt_batch(ctx, ks, z, [seed + i for i in range(count)], limbs)


def _fits(call, results, mib):
    """call() with `mib` MiB of device memory left, and the same call unlimited needs more and agrees."""
    import torch

    torch.cuda.synchronize()
    mempool.reset_peak()
    before = mempool.used()
    want = results(call())
    torch.cuda.synchronize()
    assert mempool.peak() - before > mib << 20
    with mempool.limited(mib << 20):
        got = results(call())
    assert all(np.array_equal(g, w) for g, w in zip(got, want))


def _export(ctx, handles):
    out = [hx.hx_ct_export(ctx, h) for h in handles]
    for h in handles:
        hx.hx_ct_destroy(h)
    return out


@pytest.mark.parametrize("limbs,mib", [(7, 192), (3, 224)])  # Alg. 3; the depth-2 form
def test_products(ring, limbs, mib):
    ctx, ks, _ = ring
    a, b = _batch(ctx, ks, 5, limbs, 10), _batch(ctx, ks, 5, limbs, 20)
    _fits(lambda: hx.hx_matmul_batch(ctx, ks, None, a, b, H), lambda r: _export(ctx, r), mib)
    for x in a + b:
        hx.hx_ct_destroy(x)


def test_transposes(ring):
    ctx, ks, _ = ring
    x = _batch(ctx, ks, 8, 7, 30)
    _fits(lambda: hx.hx_transpose(ctx, ks, None, x, H), lambda r: _export(ctx, r), 256)
    for c in x:
        hx.hx_ct_destroy(c)


def test_hoisted_rotations(ring):
    ctx, ks, steps = ring
    a = _batch(ctx, ks, 1, 7, 40)[0]
    _fits(lambda: hx.hx_rotate_hoisted(ctx, ks, a, (steps * 32)[:32]), lambda r: _export(ctx, r), 64)
    hx.hx_ct_destroy(a)


@pytest.mark.parametrize("mib", [288, 600])
def test_captured_products(ring, mib):
    import torch

    ctx, ks, _ = ring
    a, b = _batch(ctx, ks, 5, 7, 50), _batch(ctx, ks, 5, 7, 60)
    plan = hx.hx_matmul_plan_create(ctx, H, 7)
    want = _export(ctx, hx.hx_matmul_batch(ctx, ks, plan, a, b, H))
    scale = hx.hx_ct_info(a[0])[2]
    for full in (True, False):
        ex = hx.hx_matmul_exec_create(ctx, ks, plan, 5, scale)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        hold = torch.empty(max(0, torch.cuda.mem_get_info()[0] - (mib << 20)) if full else 0, dtype=torch.uint8, device="cuda")
        before = hx.hx_matmul_exec_launches(ex)
        for _ in range(2):
            got = _export(ctx, hx.hx_matmul_exec_run(ex, a, b))
            assert all(np.array_equal(g, w) for g, w in zip(got, want))
        assert (hx.hx_matmul_exec_launches(ex) > before) == full  # smaller groups, more launches
        del hold
        hx.hx_matmul_exec_destroy(ex)
    hx.hx_matmul_plan_destroy(plan)
    for x in a + b:
        hx.hx_ct_destroy(x)
