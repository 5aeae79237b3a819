"""The device encoder at every ring degree, and a batch's encryptions against single ones."""
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


@pytest.mark.parametrize("log_n", [11, 12, 13, 14, 15, 16])
def test_coefficients_and_batches(log_n):
    """Both are the correct rounding of the same exact values: equal."""
    ctx = hx.hx_context_create(log_n, [60, 45], [60], 45)
    try:
        n = 1 << log_n
        z = np.random.default_rng(log_n).uniform(-1, 1, (3, n // 2))
        for scale in (2.0 ** 45, 1099510054913.0):
            want = C.encode_real(n, z, scale)
            assert np.array_equal(hx.hx_encode_batch(ctx, z, scale), want)
            assert np.array_equal(hx.hx_encode_batch(ctx, z[:, :5], scale), C.encode_real(n, z[:, :5], scale))
        ks = hx.hx_keygen(ctx, 2, 5)
        batch = hx.hx_encrypt_batch(ctx, ks, z, [7, 8, 9])
        for ct, row, seed in zip(batch, z, (7, 8, 9)):
            one = hx.hx_encrypt(ctx, ks, row, 0, seed)
            assert np.array_equal(hx.hx_ct_export(ctx, ct), hx.hx_ct_export(ctx, one))
            hx.hx_ct_destroy(one)
            hx.hx_ct_destroy(ct)
        hx.hx_keyset_destroy(ks)
    finally:
        hx.hx_context_destroy(ctx)
