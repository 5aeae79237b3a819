"""Every split and tile width of the transform on primes just below a power of two, and the untuned ones."""
import numpy as np
import pytest

from oracle import ckks as C
from paper_2207_04620_gb300 import hx, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2207_04620_gb300 import build

    build.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("log_n", [11, 12, 13, 14, 15, 16])
def test_splits_and_widths(log_n):
    import torch

    octx = C.Context(log_n, [60, 45], [60], 40)
    ctx = hx.hx_context_create(log_n, [60, 45], [60], 40)
    try:
        primes = octx.q + octx.p
        x = workloads.residues(3, primes, 2, octx.N)
        want = octx.ntt(x, primes * 2)

        def check(what):
            dev = torch.from_numpy(x.view(np.int64).copy()).cuda()
            hx.hx_ntt(ctx, dev.data_ptr(), 2, [0, 1, 2])
            torch.cuda.synchronize()
            assert np.array_equal(dev.cpu().numpy().view(np.uint64), want), what
            hx.hx_ntt(ctx, dev.data_ptr(), 2, [0, 1, 2], inverse=True)
            torch.cuda.synchronize()
            assert np.array_equal(dev.cpu().numpy().view(np.uint64), x), what

        check("untuned")
        first = hx.hx_ntt_tuning(ctx)[0]
        assert first["split"] == (1 if log_n in (13, 15) else 0)
        cols = log_n // 2 + first["split"]
        assert first["widths"] == [8 if n >= 8 else 16 for n in (cols, log_n - cols)] * 2
        for split in (0, 1) if log_n & 1 else (0,):
            for w in ([4] * 4, [8] * 4, [16] * 4, [32] * 4, [-8] * 4, [-16] * 4):
                hx.hx_ntt_tiles(ctx, w)
                hx.hx_ntt_split(ctx, split)
                check((split, w))
        # the several-ring launch
        hx.hx_ntt_tiles(ctx, [16] * 4)
        assert hx.hx_ntt_tuning(ctx)[0]["split"] == first["split"]
        dev = torch.from_numpy(x.view(np.int64).copy()).cuda()
        hx.hx_ntt_multi([(ctx, dev.data_ptr(), 2, [0, 1, 2])])
        torch.cuda.synchronize()
        assert np.array_equal(dev.cpu().numpy().view(np.uint64), want)
    finally:
        hx.hx_context_destroy(ctx)
