"""Transforms on chains of primes just below powers of two (fold arithmetic): bit-exact against the
oracle at the ends of the prime sizes it takes (33 and 60 bits), with final reductions of one fold and
of two, on inputs that drive its signed, unreduced sums furthest.  Words are integers, so there is no
tolerance."""
import numpy as np
import pytest

from oracle import ckks as C
from paper_2207_04620_gb300 import hx, workloads

pytestmark = pytest.mark.gpu

# 60-bit primes leave the least room above a sum, small ones have the largest d / q
CHAINS = {
    "60": [60] * 8,
    "mixed": [60, 59, 55, 50, 45, 45, 45, 45, 45, 45],
    "40": [60] + [40] * 12,
    "small": [38, 38, 36, 36, 36, 35],
    "33": [33, 33, 34, 34],
    "60_33": [60, 33, 45, 34, 60, 36],
}


def folds(q):
    """How many folds the final reduction of prime q takes; None if fold arithmetic does not hold for it:
    on a unit u >= 2^b with folded values within 17/16 u and products within 25/16 u, sums up to
    127/16 u have to stay inside 63 bits and end within 2^(b-1) of [0, 2^b)."""
    b = q.bit_length()
    one, d = 1 << b, (1 << b) - q
    if not 33 <= b <= 60 or d >= 1 << 26:
        return None

    def folded(v):
        return one + ((v >> b) + 1) * d

    u = max(one, -(-16 * (one + one // 2 + (d << 31)) // 25))
    for _ in range(3):
        u = max(u, -(-16 * folded(u * 127 // 16 + 1) // 17))
    limit = u * 127 // 16 + 1
    if limit >= (1 << 63) - (1 << 32) or 16 * folded(limit) > 17 * u:
        return None
    once = folded(limit)
    if once - one <= one // 2:
        return 1
    return 2 if folded(once) - one <= one // 2 else None


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2207_04620_gb300 import build

    build.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def inputs(seed, primes, n):
    """[8][limbs][n]: random, all q - 1, all 0, q - 1 alternating with 0 (by 1 and by n / 2), one
    q - 1 at each end, near q / 2."""
    q = np.array(primes, dtype=np.uint64)[:, None]
    x = np.zeros((8, len(primes), n), dtype=np.uint64)
    x[0] = workloads.residues(seed, primes, 1, n)
    x[1] = q - np.uint64(1)
    x[3][:, ::2] = (q - np.uint64(1))
    x[4][:, : n // 2] = (q - np.uint64(1))
    x[5][:, 0] = (q - np.uint64(1))[:, 0]
    x[6][:, -1] = (q - np.uint64(1))[:, 0]
    x[7] = q // np.uint64(2) + workloads.residues(seed + 1, [2] * len(primes), 1, n)
    return x


def dev(x, offset=0):
    """x on the device, `offset` words behind an allocation's start."""
    import torch

    buf = torch.zeros(x.size + offset, dtype=torch.int64, device="cuda")
    t = buf[offset:]
    t.copy_(torch.from_numpy(x.view(np.int64).reshape(-1).copy()))
    return buf, t


@pytest.mark.parametrize("log_n", [11, 12, 13, 14, 15, 16])
@pytest.mark.parametrize("chain", sorted(CHAINS))
def test_extreme_inputs_bit_exact(chain, log_n):
    bits = CHAINS[chain]
    octx = C.Context(log_n, bits, [60], 40)
    ctx = hx.hx_context_create(log_n, bits, [60], 40)
    try:
        primes = octx.q + octx.p
        assert all(folds(q) for q in primes)
        if chain in ("33", "60_33") and log_n >= 12:
            assert 2 in [folds(q) for q in primes]
        x = inputs(log_n, primes, octx.N)
        flat = x.reshape(-1, octx.N)
        idx = list(range(len(primes)))
        for inverse, want in ((False, octx.ntt(flat, primes * 8)), (True, octx.intt(flat, primes * 8))):
            for offset in (0, 2):  # 2: rows at 16 mod 32 bytes take the narrower accesses
                buf, t = dev(x, offset)
                hx.hx_ntt(ctx, t.data_ptr(), 8, idx, inverse=inverse)
                got = t.cpu().numpy().view(np.uint64).reshape(-1, octx.N)
                assert np.array_equal(got, want), (inverse, offset)
            buf, t = dev(x)
            hx.hx_ntt_multi([(ctx, t.data_ptr(), 8, idx)], inverse=inverse)
            assert np.array_equal(t.cpu().numpy().view(np.uint64).reshape(-1, octx.N), want), ("multi", inverse)
    finally:
        hx.hx_context_destroy(ctx)


@pytest.mark.parametrize("log_n", [13, 14])
def test_unreduced_inputs(log_n):
    """Forward transforms take values below 4q and inverse ones below 2q, as the Shoup butterflies do."""
    octx = C.Context(log_n, [60, 60, 45], [60], 45)
    ctx = hx.hx_context_create(log_n, [60, 60, 45], [60], 45)
    try:
        primes = octx.q + octx.p
        q = np.array(primes, dtype=np.uint64)[None, :, None]
        x = inputs(5, primes, octx.N)
        for inverse, top in ((False, 3), (True, 1)):
            flat = x.reshape(-1, octx.N)
            want = (octx.intt if inverse else octx.ntt)(flat, primes * 8)
            buf, t = dev(x + np.uint64(top) * q)
            hx.hx_ntt(ctx, t.data_ptr(), 8, [0, 1, 2, 3], inverse=inverse)
            assert np.array_equal(t.cpu().numpy().view(np.uint64).reshape(-1, octx.N), want), inverse
    finally:
        hx.hx_context_destroy(ctx)
