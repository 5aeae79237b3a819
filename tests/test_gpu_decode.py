"""Decryption and decoding on the device at every ring degree, whole and partial slot counts."""
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
def test_slots_of_the_decrypted_coefficients(log_n):
    """hx_decrypt equals the decoding of hx_decrypt_coeffs' integers.  Each of the log N + 1 stages
    rounds within 4 units of 2^-53 of the 2-norm, which grows as the exact transform's, so the 2-norms
    differ by less than (log N + 1) 2^-51 each way; twice that for the two sides."""
    ctx = hx.hx_context_create(log_n, [60, 45], [60], 45)
    try:
        ks = hx.hx_keygen(ctx, 3, 5)
        n = 1 << log_n
        z = np.random.default_rng(log_n).uniform(-1, 1, n // 2)
        ct = hx.hx_encrypt(ctx, ks, z, 0, 9)
        want = C.decode(n, hx.hx_decrypt_coeffs(ctx, ks, ct), 2.0 ** 45).real
        got = hx.hx_decrypt(ctx, ks, ct)
        assert np.linalg.norm(got - want) <= 2 * (log_n + 1) * 2.0 ** -51 * np.linalg.norm(want)
        # encryption noise v e + e0 + e1 s: v ternary, s the sum of three ternary shares, every e of
        # width 3.2; a slot sums its n coefficients, and eight standard deviations cover n / 2 slots
        sigma = 3.2 * np.sqrt(n * (2 / 3 + 3 * 2 / 3) + 1)
        assert np.abs(got - z).max() < 8 * sigma * np.sqrt(n) / 2.0 ** 45
        for count in (1, 3, n // 4 + 1):
            assert np.array_equal(hx.hx_decrypt(ctx, ks, ct, count), got[:count])
        assert np.array_equal(hx.hx_decrypt_parties(ctx, ks, ct, [1, 1, 1]), got)
        hx.hx_ct_destroy(ct)
        hx.hx_keyset_destroy(ks)
    finally:
        hx.hx_context_destroy(ctx)
