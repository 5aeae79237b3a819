"""Basis conversions on split sums: every source count up to the largest, full sums (60-bit primes),
sources and destinations of 33 to 60 bits in one conversion, chains outside fold arithmetic (Shoup
products), grids split over the destination rows, and overshoots that lie on an integer (where the FP64 sum
decides), bit-exact against the oracle."""
import numpy as np
import pytest

from oracle import ckks as C
from paper_2207_04620_gb300 import hx, workloads

from hxpair import PARAMS, Pair

pytestmark = pytest.mark.gpu

for a, k in ((1, 1), (2, 2), (3, 3), (4, 4), (5, 5), (7, 6)):
    PARAMS["conv%d" % a] = dict(log_n=11, q_bits=[60] * 9, p_bits=[60] * k, log2_scale=45, alpha=a)
MIXED = [60, 33, 34, 60, 36, 33, 35, 60, 34]
PARAMS["conv_mixed3"] = dict(log_n=11, q_bits=MIXED, p_bits=[60, 36, 33], log2_scale=33, alpha=3)
PARAMS["conv_mixed7"] = dict(log_n=11, q_bits=MIXED, p_bits=[60, 33, 60, 36, 60, 34], log2_scale=33, alpha=7)
PARAMS["conv_mixed14"] = dict(log_n=14, q_bits=MIXED, p_bits=[60, 34], log2_scale=33)
PARAMS["conv_general"] = dict(log_n=11, q_bits=[60] * 9, p_bits=[61] * 3, log2_scale=45, alpha=4)
PARAMS["conv40"] = dict(log_n=13, q_bits=[60] + [40] * 8, p_bits=[60] * 3, log2_scale=40, alpha=4)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2207_04620_gb300 import build

    build.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("name", ["conv1", "conv2", "conv3", "conv4", "conv5", "conv7", "conv40", "conv_mixed3", "conv_mixed7",
                                  "conv_mixed14", "conv_general"])
def test_switch_and_joint_division(name):
    pr = Pair(name, rot_steps=[3])
    try:
        ev = C.Evaluator(pr.octx, pr.oks)
        for limbs in (2, 5, 9):
            primes = pr.octx.q[:limbs]
            q = np.array(primes, dtype=np.uint64)[:, None]
            full = np.broadcast_to(q - np.uint64(1), (limbs, pr.N))
            rand = workloads.residues(limbs, primes, 3, pr.N).reshape(3, limbs, pr.N)
            # coefficients at and beside (q_top -+ 1) / 2: P d + h falls on a multiple of P q_top
            rng = np.random.default_rng(limbs)
            co = np.stack([rng.choice(np.array([0, 1, p - 1, p // 2, p // 2 + 1, p // 2 - 1, p // 2 + 2], dtype=np.uint64),
                                      pr.N) for p in primes])
            edge = pr.octx.ntt(co, primes)
            zero = np.zeros((limbs, pr.N), dtype=np.uint64)
            for d in (rand, np.stack([full, full, full]), np.stack([edge, edge[:, ::-1], zero]),
                      np.stack([edge, zero, rand[2]])):
                ct = C.Ciphertext(np.ascontiguousarray(d), 2.0 ** 80)
                a = pr.to_lib(ct)
                assert pr.same(hx.hx_relinearize(pr.ctx, pr.ks, a), ev.relinearize(ct))
                assert pr.same(hx.hx_relin_rescale(pr.ctx, pr.ks, a), ev.relin_rescale(ct))
            two = C.Ciphertext(np.ascontiguousarray(np.stack([full, full])), 2.0 ** 45)
            assert pr.same(hx.hx_rotate(pr.ctx, pr.ks, pr.to_lib(two), 3), ev.rotate(two, 3))
            assert pr.same(hx.hx_rotate_jobs([(pr.ctx, pr.ks, pr.to_lib(two), 3)])[0], ev.rotate(two, 3))
    finally:
        pr.close()
