"""The selection of a boundary unit at the sizes where its shared memory ends, in both of its forms (one thread block per
unit, or one per task), and where more scores are equal than one warp sorts."""
import numpy as np
import pytest

from paper_2609_03494_b200 import binding as B
from paper_2609_03494_b200 import workload as W
from tests import lockstep as LS

pytestmark = pytest.mark.gpu


# A request of P pages has 16 (P - 1) candidates at its boundary.  Shared memory holds the factors of 1024 / 2G pages at a time
# (G = 8: 64 pages), the scores of 5120 candidates of a whole unit and of 10 240 of a single job.  With overlap_slots = 1 the
# boundary kernel has one thread block, so that it takes whole units; by default two units become six jobs.
@pytest.mark.parametrize("hq,prompt", [(16, 1030), (16, 1046), (4, 5130), (4, 5146), (16, 10250), (16, 10266)])
@pytest.mark.parametrize("slots", [0, 1])
def test_candidate_counts_at_the_edges_of_shared_memory(hq, prompt, slots):
    wl = W.Workload("edge", 5, W.Shape(1, hq, 2, 64), [W.RequestSpec(0, prompt, 30, 0.05)], n_resident=1, initial_pages=0,
                    max_pages_per_req=prompt // 16 + 2, n_pages=prompt // 16 + 1)
    st = LS.run_lockstep(wl, tau=-1.0, overlap_slots=slots)
    assert st.actions.get(B.GP_ACT_COMPRESS_FALLBACK, 0) == 2          # asks to grow, the pool is empty
    assert st.decisions["sel"] > 0 and st.near_ties == {"ws": 0, "sel": 0, "act": 0}


@pytest.mark.parametrize("page,slots", [(16, 0), (16, 1), (64, 0), (64, 1), (256, 0)])
def test_equal_scores_go_by_slot(page, slots):
    """Keys of zero make every score equal: the working sets are ceil(0.99 n), every block keeps its first k_loc slots and the
    last `page` of the other candidates go."""
    import torch
    rng = np.random.default_rng(3)
    P, L, hq, hkv, d, k_loc = 10 if page == 16 else 3, 1, 8, 2, 64, page // 4
    n = P * page - 1
    cfg = B.make_config(L, hq, hkv, d, n_pages=P, max_pages_per_req=P, max_requests=4, k_loc=k_loc, tau=1.0, page_size=page,
                        overlap_slots=slots)
    pool = B.Pool(cfg)
    try:
        zero = np.zeros((L, n, hkv, d), dtype=np.uint16)
        vals = W.f32_to_bf16_bits(rng.standard_normal((L, n, hkv, d)).astype(np.float32))
        assert pool.request_add(-1, 0, zero, vals, n, 0)[0] == B.GP_OK
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda()
        q = W.f32_to_bf16_bits(rng.standard_normal((L, 1, hq, d)).astype(np.float32))
        out = torch.zeros((L, 1, hq, d), dtype=torch.float32, device="cuda")
        act = torch.zeros(1, dtype=torch.int32, device="cuda")
        pool.decode_step(torch.zeros(1, dtype=torch.int32, device="cuda"), dev(q), dev(zero[:, :1]), dev(vals[:, :1]), out, act)
        assert act.tolist() == [B.GP_ACT_COMPRESS]
        n_d, n_e = (P - 1) * page, P * page - 16
        ks, kl, _ = B.gp_debug_boundary(pool.handle, 0, L, hkv)
        # 0.99 n is not a whole number at these sizes, so rounding of the n equal weights cannot move the count
        assert (ks == -(-99 * n_d // 100)).all() and (kl == ks).all()
        quota = min(k_loc, (n_e - page) // -(-n_e // page))
        slots_left = np.arange(n_e)
        rest = slots_left[slots_left % page >= quota]
        want = np.setdiff1d(np.arange(P * page), rest[len(rest) - page:])
        for h in range(hkv):
            assert np.array_equal(B.gp_debug_retained(pool.handle, 0, 0, h, want.size), want)
        assert B.gp_debug_pool(pool.handle)[2][7] == 0
    finally:
        pool.close()
