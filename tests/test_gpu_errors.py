"""A call that is refused leaves nothing behind that the next call would report."""
import numpy as np
import pytest

from paper_2207_04620_gb300 import hx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2207_04620_gb300 import build

    build.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_a_refused_launch_is_reported_once():
    ctx = hx.hx_context_create(11, [60, 45], [60], 45)
    ks = hx.hx_keygen(ctx, 1, 5, [1])
    a = hx.hx_encrypt(ctx, ks, np.ones(4), 1)
    with pytest.raises(hx.HxError):  # four polynomials an entry: one more than a grid's z extent holds
        hx.hx_encrypt_batch(ctx, ks, np.ones((16384, 1)), np.arange(16384), 1)
    b = hx.hx_add(ctx, a, a)
    assert abs(hx.hx_decrypt(ctx, ks, b, 4) - 2).max() < 1e-6
    for x in (a, b):
        hx.hx_ct_destroy(x)
    hx.hx_keyset_destroy(ks)
    hx.hx_context_destroy(ctx)


@pytest.mark.parametrize("limbs", [5, 3])  # Alg. 3; the depth-2 form
def test_an_executor_without_keys_is_reported_once(limbs):
    """The capture of a product ends in a missing Galois key: the next calls, a product with its keys and
    an executor among them, are as if it had not been tried."""
    h = 4
    ctx = hx.hx_context_create(11, [60, 45, 45, 45, 45], [60, 60], 45)
    steps = hx.hx_matmul_rotation_steps(ctx, h, limbs)
    few, ks = hx.hx_keygen(ctx, 1, 5, steps[:-1]), hx.hx_keygen(ctx, 1, 5, steps)
    a, b = hx.hx_encrypt_batch(ctx, ks, np.ones((2, 8)), [1, 2], limbs)
    plan = hx.hx_matmul_plan_create(ctx, h, limbs)
    scale = hx.hx_ct_info(a)[2]
    for call in (lambda: hx.hx_matmul_exec_create(ctx, few, plan, 1, scale), lambda: hx.hx_matmul(ctx, few, a, b, h)):
        with pytest.raises(hx.HxError) as e:
            call()
        assert e.value.code == -5, e.value
        c = hx.hx_add(ctx, a, b)
        want = hx.hx_matmul(ctx, ks, a, b, h)
        ex = hx.hx_matmul_exec_create(ctx, ks, plan, 1, scale)
        got = hx.hx_matmul_exec_run(ex, [a], [b])[0]
        assert np.array_equal(hx.hx_ct_export(ctx, got), hx.hx_ct_export(ctx, want))
        hx.hx_matmul_exec_destroy(ex)
        for x in (c, want, got):
            hx.hx_ct_destroy(x)
    for x in (a, b):
        hx.hx_ct_destroy(x)
    hx.hx_matmul_plan_destroy(plan)
    for k in (few, ks):
        hx.hx_keyset_destroy(k)
    hx.hx_context_destroy(ctx)
