"""Rescale from a prime of any size onto any other: the remainder goes into the transforms as it is, or
reduced, by the sizes."""
import numpy as np
import pytest

from oracle import ckks as C
from paper_2207_04620_gb300 import hx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2207_04620_gb300 import build

    build.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("bits", [[60, 45, 45, 45], [40, 60, 45], [45, 46], [45, 47], [60, 33, 60], [60, 60], [61, 45]])
@pytest.mark.parametrize("log_n", [11, 15])
def test_remainders_at_the_edges(log_n, bits):
    octx = C.Context(log_n, bits, [60], 40)
    ctx = hx.hx_context_create(log_n, bits, [60], 40)
    try:
        n, top = 1 << log_n, octx.q[-1]
        rng = np.random.default_rng(log_n)
        x = np.stack([np.stack([rng.integers(0, q, n, dtype=np.uint64) for q in octx.q]) for _ in range(2)])
        # the top limb's coefficients: the whole range, then zero, the halves and the largest residue
        c = np.stack([rng.integers(0, top, n, dtype=np.uint64)] * 2)
        c[1, :] = np.resize(np.array([0, 1, top // 2, top // 2 + 1, top - 1], dtype=np.uint64), n)
        for i in range(2):
            x[i, -1] = octx.ntt(c[i][None, :], [top])[0]
        ev = C.Evaluator(octx, None)
        want = ev.rescale(C.Ciphertext(x, 2.0 ** 80))
        h = hx.hx_ct_import(ctx, x, 2.0 ** 80)
        r = hx.hx_rescale(ctx, h)
        assert np.array_equal(hx.hx_ct_export(ctx, r), want.c)
        hx.hx_ct_destroy(r)
        hx.hx_ct_destroy(h)
    finally:
        hx.hx_context_destroy(ctx)
