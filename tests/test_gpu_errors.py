"""A call that is refused leaves nothing behind that the next call would report."""
import numpy as np
import pytest

from paper_2207_04620_gb300 import hx

pytestmark = pytest.mark.gpu


def test_a_refused_launch_is_reported_once():
    from paper_2207_04620_gb300 import build

    build.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
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
