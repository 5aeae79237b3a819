"""Key inner products over keys split at bit 30: every digit count the kernels are built for and
the general one, up to and past the counts at which their sums make room, with 60-bit primes (the
fullest sums), with primes of 33 to 60 bits, on a chain outside fold arithmetic (a 61-bit special prime:
Montgomery keys, whole-word products, the same groups and schedules), and all words at q - 1, bit-exact against the oracle; batches that fill a block's
entries partly."""
import numpy as np
import pytest

from oracle import ckks as C
from oracle import hercules as Hc
from paper_2207_04620_gb300 import hx, workloads

from hxpair import PARAMS, Pair

pytestmark = pytest.mark.gpu

PARAMS["split60"] = dict(log_n=11, q_bits=[60] * 16, p_bits=[60], log2_scale=45, alpha=1)
PARAMS["split_mixed"] = dict(log_n=11, q_bits=[60, 33, 34, 60] + [36, 33, 60, 35] * 3, p_bits=[60], log2_scale=33, alpha=1)
PARAMS["general"] = dict(log_n=11, q_bits=[60] * 16, p_bits=[61], log2_scale=45, alpha=1)
PARAMS["general_mm"] = dict(log_n=11, q_bits=[60] + [45] * 6, p_bits=[61, 60], log2_scale=45)
PARAMS["split60_mm"] = dict(log_n=11, q_bits=[60] * 9, p_bits=[60], log2_scale=45, alpha=1)
PARAMS["split45_mm"] = dict(log_n=11, q_bits=[60] + [45] * 6, p_bits=[60, 60], log2_scale=45)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2207_04620_gb300 import build

    build.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.fixture(scope="module", params=["split60", "split_mixed", "general"])
def chain(request):
    pr = Pair(request.param, rot_steps=[1, 5, -3])
    yield pr
    pr.close()


@pytest.mark.parametrize("limbs", [1, 2, 3, 4, 5, 6, 7, 8, 14, 15, 16])
def test_rotations_by_digit_count(chain, limbs):
    q = np.array(chain.octx.q[:limbs], dtype=np.uint64)[None, :, None]
    full = np.broadcast_to(q - np.uint64(1), (2, limbs, chain.N)).copy()
    rand = workloads.residues(limbs, chain.octx.q[:limbs], 2, chain.N).reshape(2, limbs, chain.N)
    ev = C.Evaluator(chain.octx, chain.oks)
    jobs = []
    for x in (full, rand):
        ct = C.Ciphertext(x, 2.0 ** 45)
        a = chain.to_lib(ct)
        assert chain.same(hx.hx_rotate(chain.ctx, chain.ks, a, 1), ev.rotate(ct, 1))
        for got, k in zip(hx.hx_rotate_hoisted(chain.ctx, chain.ks, a, [5, -3]), (5, -3)):
            assert chain.same(got, ev.rotate_hoisted(ct, [k])[0])
        jobs.append(((chain.ctx, chain.ks, a, 1), ev.rotate(ct, 1)))
    for got, (_, want) in zip(hx.hx_rotate_jobs([j for j, _ in jobs]), jobs):
        assert chain.same(got, want)


@pytest.mark.parametrize("name,h,limbs", [("split60_mm", 4, 9), ("split60_mm", 4, 5), ("split45_mm", 4, 7), ("general_mm", 4, 7),
                                          ("general_mm", 4, 3)])
@pytest.mark.parametrize("count", [1, 2, 3, 5])
def test_products_bound_and_unbound(name, h, limbs, count):
    p = PARAMS[name]
    beta = (1 << p["log_n"]) // 2 // (h * h)
    pr = Pair(name, rot_steps=Hc.matmul_rotation_steps(h, beta, limbs))
    try:
        A = [pr.encrypt(workloads.pack(workloads.matrices(i, beta, h), h, beta), i, limbs) for i in range(count)]
        B = [pr.encrypt(workloads.pack(workloads.matrices(50 + i, beta, h), h, beta), 50 + i, limbs) for i in range(count)]
        la, lb = [pr.to_lib(x) for x in A], [pr.to_lib(x) for x in B]
        plan = hx.hx_matmul_plan_create(pr.ctx, h, limbs)
        plain = hx.hx_matmul_batch(pr.ctx, pr.ks, plan, la, lb, h)
        if limbs > 3:  # Alg. 3; the depth-2 form has no selections to bind
            hx.hx_matmul_plan_bind_keys(pr.ctx, plan, pr.ks)
        bound = hx.hx_matmul_batch(pr.ctx, pr.ks, plan, la, lb, h)
        masks, ev = Hc.MaskProvider(pr.octx, h, limbs), C.Evaluator(pr.octx, pr.oks)
        for i in sorted({0, count - 1}):
            want = Hc.matmul(ev, A[i], B[i], h, masks)
            assert pr.same(plain[i], want) and pr.same(bound[i], want)
        for i in range(count):
            assert np.array_equal(hx.hx_ct_export(pr.ctx, plain[i]), hx.hx_ct_export(pr.ctx, bound[i]))
        hx.hx_matmul_plan_destroy(plan)
    finally:
        pr.close()


def test_rings_inside_and_outside_fold_arithmetic_in_one_call():
    """hx_rotate_jobs and hx_ntt_multi over rings of both kinds: one arithmetic serves every transform,
    keys and conversions keep their ring's."""
    import torch

    pairs = [Pair("split45_mm", rot_steps=[3]), Pair("general_mm", rot_steps=[3])]
    try:
        jobs, want, rows = [], [], []
        for i, pr in enumerate(pairs):
            limbs = 5 - i
            x = workloads.residues(i, pr.octx.q[:limbs], 2, pr.N).reshape(2, limbs, pr.N)
            ct = C.Ciphertext(x, 2.0 ** 45)
            jobs.append((pr.ctx, pr.ks, pr.to_lib(ct), 3))
            want.append(C.Evaluator(pr.octx, pr.oks).rotate(ct, 3))
            t = torch.from_numpy(x.view(np.int64).copy()).cuda()
            rows.append((t, pr.octx.ntt(x.reshape(-1, pr.N), pr.octx.q[:limbs] * 2)))
        for pr, got, w in zip(pairs, hx.hx_rotate_jobs(jobs), want):
            assert pr.same(got, w)
        hx.hx_ntt_multi([(pr.ctx, t.data_ptr(), 2, list(range(t.shape[1]))) for pr, (t, _) in zip(pairs, rows)])
        for t, w in rows:
            assert np.array_equal(t.cpu().numpy().view(np.uint64).reshape(w.shape), w)
    finally:
        for pr in pairs:
            pr.close()
