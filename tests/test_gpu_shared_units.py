"""Boundary units of many candidates, shared out over the thread blocks of a cluster: around the size where that begins, at counts that
leave the last blocks a short part or none, for every group size, head dimension and page size, and where all scores are equal."""
import numpy as np
import pytest

from paper_2609_03494_b200 import binding as B
from paper_2609_03494_b200 import workload as W
from tests import lockstep as LS

pytestmark = pytest.mark.gpu


# A request of P pages of b tokens has P b - 16 candidates; units are shared out above 10 240.  Eight blocks take whole pages each for the softmax
# and whole blocks of Eq. 10, and words of 32 candidates, for the descents.
@pytest.mark.parametrize("hq,hkv,d,page,prompt,rope", [
    (4, 2, 64, 16, 10237, 0.0), (4, 2, 64, 16, 10256, 0.0), (2, 2, 128, 16, 10269, 1e6), (8, 1, 128, 16, 10493, 0.0), (8, 1, 64, 16, 11192, 1e6),
    (8, 2, 128, 64, 10363, 0.0), (8, 2, 64, 128, 11262, 0.0), (8, 2, 64, 256, 10492, 0.0), (8, 1, 64, 256, 12282, 1e6)])
def test_shared_units_against_the_oracle(hq, hkv, d, page, prompt, rope):
    P = prompt // page + 1
    s = W.Shape(1, hq, hkv, d, page_size=page)
    reqs = [W.RequestSpec(i, n, P * page - prompt + 3 + i, 0.05, share_group=-1) for i, n in enumerate((prompt, prompt - 5))]
    wl = W.Workload("shared", 11, s, reqs, n_resident=2, initial_pages=0, max_pages_per_req=P + 1, n_pages=2 * P, k_loc=page // 4)
    st = LS.run_lockstep(wl, tau=-1.0, rope_theta=rope, check_pool_every=16)
    assert st.decisions["sel"] > 0 and st.near_ties == {"ws": 0, "sel": 0, "act": 0}


@pytest.mark.parametrize("page,P", [(16, 643), (16, 675), (64, 163), (256, 43)])
def test_equal_scores_of_shared_units_go_by_slot(page, P):
    """Keys of zero make every score equal: the working sets are ceil(0.99 n), every block keeps its first k_loc slots and the
    last `page` of the other candidates go."""
    import torch
    rng = np.random.default_rng(3)
    L, hq, hkv, d, k_loc = 1, 8, 2, 64, page // 4
    n = P * page - 1
    pool = B.Pool(B.make_config(L, hq, hkv, d, n_pages=P, max_pages_per_req=P, max_requests=4, k_loc=k_loc, tau=1.0, page_size=page))
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


@pytest.mark.parametrize("how", ["early plan", "graph", "four kernels"])
def test_shared_units_whatever_way_the_steps_are_launched(how):
    """Every plan clears the counters the boundary work draws its jobs from: also one that starts beside the compaction, and one that is
    replayed.  The kernel that takes such units on one thread block each gives the same."""
    import torch
    L, hq, hkv, d, steps = 2, 4, 2, 64, 36
    lens = (10300, 10270, 300)
    g = torch.Generator(device="cuda").manual_seed(4)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    prompts = [(rand(L, n, hkv, d), rand(L, n, hkv, d)) for n in lens]
    qs, ks, vs = rand(steps, L, 3, hq, d), rand(steps, L, 3, hkv, d), rand(steps, L, 3, hkv, d)
    pages = sum(n // 16 + 1 for n in lens)

    def run(how):
        pool = B.Pool(B.make_config(L, hq, hkv, d, n_pages=pages + 1, max_pages_per_req=max(lens) // 16 + 3, max_requests=4, tau=-1.0,
                                    overlap_slots=-1 if how == "four kernels" else 0))
        try:
            for (k, v), n in zip(prompts, lens):
                assert pool.request_add(-1, 0, k, v, n, 0)[0] == B.GP_OK
            B.gp_set_early_plan(pool.handle, how == "early plan")
            ids = torch.arange(3, dtype=torch.int32, device="cuda")
            out = torch.zeros((L, 3, hq, d), dtype=torch.float32, device="cuda")
            act = torch.zeros(3, dtype=torch.int32, device="cuda")
            q, k, v = qs[0].clone(), ks[0].clone(), vs[0].clone()
            outs, acts, graph = [], [], None
            if how == "graph":
                side = torch.cuda.Stream()
                side.wait_stream(torch.cuda.current_stream())
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=side):
                    pool.decode_step(ids, q, k, v, out, act)
            torch.cuda.synchronize()
            for t in range(steps):
                if graph is not None:
                    q.copy_(qs[t]); k.copy_(ks[t]); v.copy_(vs[t])
                    graph.replay()
                else:
                    pool.decode_step(ids, qs[t], ks[t], vs[t], out, act)
                outs.append(out.clone()); acts.append(act.clone())
            torch.cuda.synchronize()
            n = B.gp_debug_state(pool.handle, 4)[1]
            kept = [B.gp_debug_retained(pool.handle, r, l, h, int(n[r])) for r in range(3) for l in range(L) for h in range(hkv)]
            assert B.gp_pool_status(pool.handle) == (B.GP_OK, 0)
            return torch.stack(outs).cpu().numpy(), torch.stack(acts).cpu().numpy(), kept
        finally:
            pool.close()

    want, got = run("plain"), run(how)
    assert (want[1][:, :2] != 0).sum() >= 4                            # both long requests at boundaries, growing and compressing
    assert np.array_equal(want[0], got[0]) and np.array_equal(want[1], got[1])
    assert all(np.array_equal(a, b) for a, b in zip(want[2], got[2]))


def _decode(layers, hq, hkv, d, lens, steps, page=16, k_loc=4, tau=-1.0, spare=1, four=False, graph=False, edit=None, spin_limit=0, withhold=0):
    """Decodes `steps` tokens of requests of these lengths in a pool with `spare` free pages, one step captured and replayed with `graph`.  Everything a step decides, and how many units were
    shared out (`four`: the kernels that never do)."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(4)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    pages = [n // page + 1 for n in lens]
    pool = B.Pool(B.make_config(layers, hq, hkv, d, n_pages=sum(pages) + spare, max_pages_per_req=max(pages) + 3, max_requests=len(lens), k_loc=k_loc,
                                tau=tau, page_size=page, overlap_slots=-1 if four else 0))
    try:
        for i, n in enumerate(lens):
            k, v = rand(layers, n, hkv, d), rand(layers, n, hkv, d)
            if edit:
                edit(i, k, v)
            assert pool.request_add(-1, 0, k, v, n, 0)[0] == B.GP_OK
            del k, v
        if spin_limit:
            B.gp_test_withhold(pool.handle, withhold, spin_limit)
        R = len(lens)
        ids = torch.arange(R, dtype=torch.int32, device="cuda")
        out = torch.zeros((layers, R, hq, d), dtype=torch.float32, device="cuda")
        act = torch.zeros(R, dtype=torch.int32, device="cuda")
        ins = [torch.empty((layers, R, heads, d), dtype=torch.bfloat16, device="cuda") for heads in (hq, hkv, hkv)]
        outs, acts, step = [], [], lambda: pool.decode_step(ids, *ins, out, act)
        if graph:
            side, g_step = torch.cuda.Stream(), torch.cuda.CUDAGraph()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.graph(g_step, stream=side):
                step()
            step = g_step.replay
        for _ in range(steps):
            for t in ins:
                t.copy_(rand(*t.shape))
            step()
            outs.append(out.clone()); acts.append(act.clone())
        torch.cuda.synchronize()
        n = B.gp_debug_state(pool.handle, R)[1]
        return dict(out=torch.stack(outs).cpu().numpy(), act=torch.stack(acts).cpu().numpy(), status=B.gp_pool_status(pool.handle),
                    sets=[B.gp_debug_boundary(pool.handle, r, layers, hkv)[:2] for r in range(R)],
                    kept=[B.gp_debug_retained(pool.handle, r, l, h, int(n[r])) for r in range(R) for l in range(layers) for h in range(hkv)],
                    state=[B.gp_debug_request(pool.handle, r, max(pages) + 3) for r in range(R)], shared=int(B.gp_debug_pool(pool.handle)[2][11]))
    finally:
        pool.close()


def _same(a, b):
    assert a["status"] == b["status"] and np.array_equal(a["act"], b["act"])
    assert all(np.array_equal(x, y) for s, t in zip(a["sets"], b["sets"]) for x, y in zip(s, t))
    assert len(a["kept"]) == len(b["kept"]) and all(np.array_equal(x, y) for x, y in zip(a["kept"], b["kept"]))
    assert np.array_equal(a["out"], b["out"], equal_nan=True)


@pytest.mark.parametrize("hq,d", [(8, 64), (64, 64), (16, 128)])
def test_more_shared_units_than_clusters(hq, d):
    """48 units on at most 37 clusters (two blocks on each of 148 SMs): some clusters draw a second one, in the place of the first.  Two units one after the
    other are shared out from 20 480 candidates on.  The second step is a boundary that takes the spare page, the eighteenth one that evicts."""
    got, want = (_decode(6, hq, 8, d, [1302 * 16 - 2], 20, four=four) for four in (False, True))
    assert (got["shared"], want["shared"]) == (2 * 48, 0) and got["status"] == (B.GP_OK, 0)
    assert [t for t in range(20) if got["act"][t, 0]] == [1, 17]
    _same(got, want)


@pytest.mark.parametrize("graph", [False, True])
def test_requests_that_grow_into_shared_units(graph):
    """Admitted with fewer tokens than a unit that is shared out: the third boundary has 10 256 candidates, after 42 steps or as many replays of one."""
    got, want = (_decode(2, 8, 2, 64, [10230, 200], 43, spare=40, four=four, graph=graph and not four) for four in (False, True))
    assert (got["shared"], want["shared"]) == (4, 0) and got["status"] == (B.GP_OK, 0)
    _same(got, want)


def test_shared_units_of_a_request_admitted_by_reference():
    """The donor has gone when the request that took its prompt by reference reaches its boundary."""
    import torch
    L, hq, hkv, d = 2, 8, 2, 64
    g = torch.Generator(device="cuda").manual_seed(5)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    pool = B.Pool(B.make_config(L, hq, hkv, d, n_pages=645, max_pages_per_req=644, max_requests=4, tau=1.0))
    try:
        assert pool.request_add(-1, 0, rand(L, 10260, hkv, d), rand(L, 10260, hkv, d), 10260, 0) == (B.GP_OK, 0)
        assert pool.request_add(0, 641, rand(L, 15, hkv, d), rand(L, 15, hkv, d), 15, 0) == (B.GP_OK, 1)
        pool.release(0)
        out = torch.zeros((L, 1, hq, d), dtype=torch.float32, device="cuda")
        act = torch.zeros(1, dtype=torch.int32, device="cuda")
        pool.decode_step(torch.ones(1, dtype=torch.int32, device="cuda"), rand(L, 1, hq, d), rand(L, 1, hkv, d), rand(L, 1, hkv, d), out, act)
        assert act.tolist() == [B.GP_ACT_COMPRESS]
        counters = B.gp_debug_pool(pool.handle)[2]
        assert counters[11] == L * hkv and counters[7] == 0
    finally:
        pool.close()


def test_a_request_with_more_units_than_clusters_may_take():
    """80 units: more than twice the clusters of a B200, so that pool never launches them."""
    got, want = (_decode(10, 8, 8, 64, [10271], 2, tau=1.0, four=four) for four in (False, True))
    assert (got["shared"], want["shared"]) == (0, 0) and got["status"] == (B.GP_OK, 0) and got["act"][0, 0] == B.GP_ACT_COMPRESS
    _same(got, want)


@pytest.mark.parametrize("what,bit", [(4, 8), (8, 16)])
def test_waits_of_shared_units_that_run_out_are_reported(what, bit):
    """The decisions never told to the waiting blocks (4), the logits never reported complete (8): every block of a cluster gives up by itself, meets
    the others at the cluster's barriers all the same, and the pool steps on."""
    import torch
    L, hq, hkv, d, lens = 1, 8, 2, 64, (642 * 16 - 1, 643 * 16 - 1, 303)
    g = torch.Generator(device="cuda").manual_seed(6)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    pages = [n // 16 + 1 for n in lens]
    pool = B.Pool(B.make_config(L, hq, hkv, d, n_pages=sum(pages), max_pages_per_req=643, max_requests=4, tau=1.0))
    try:
        for n in lens:
            assert pool.request_add(-1, 0, rand(L, n, hkv, d), rand(L, n, hkv, d), n, 0)[0] == B.GP_OK
        ids = torch.arange(3, dtype=torch.int32, device="cuda")
        out = torch.zeros((L, 3, hq, d), dtype=torch.float32, device="cuda")
        act = torch.zeros(3, dtype=torch.int32, device="cuda")
        step = lambda: pool.decode_step(ids, rand(L, 3, hq, d), rand(L, 3, hkv, d), rand(L, 3, hkv, d), out, act)
        B.gp_test_withhold(pool.handle, what, 2000)
        step()
        assert act.tolist() == [B.GP_ACT_COMPRESS] * 3
        status, bits = B.gp_pool_status(pool.handle)
        assert status == B.GP_ERR_CUDA and (bits & bit), bits
        n_free, ref, counters = B.gp_debug_pool(pool.handle, sum(pages))
        assert counters[11] == 2 * L * hkv and n_free == 0 and ref.tolist() == [1] * sum(pages)
        assert [B.gp_debug_request(pool.handle, r, 643)[:2] for r in range(3)] == [(P, (P - 1) * 16) for P in pages]
        B.gp_test_withhold(pool.handle, 0, 0)
        step()
        assert act.tolist() == [B.GP_ACT_NONE] * 3 and bool(torch.isfinite(out).all())
    finally:
        pool.close()


# 8 x 5120 places for scores: 40 960 candidates are the most that a cluster takes; of two units one after the other more than 20 480 each.  With pages
# of b > 16 tokens the larger of the two candidate sets counts: all but the protected window, P b - 16, where `cand` is (P - 1) b.
@pytest.mark.parametrize("hq,d,page,cand,k_loc,shared", [
    (8, 64, 16, 20000, 4, 1), (4, 128, 16, 20000, 0, 1), (1, 64, 16, 40960, 4, 1), (8, 128, 16, 40960, 16, 1), (8, 64, 256, 159 * 256, 64, 1),
    (2, 64, 128, 319 * 128, 0, 1), (8, 64, 16, 40976, 4, 0), (4, 64, 256, 160 * 256, 64, 0)])
def test_shared_units_up_to_the_largest(hq, d, page, cand, k_loc, shared):
    n = cand + page - 1
    got, want = (_decode(1, hq, 1, d, [n], 2, page=page, k_loc=k_loc, tau=1.0, four=four) for four in (False, True))
    assert (got["shared"], want["shared"]) == (shared, 0) and got["status"] == (B.GP_OK, 0) and got["act"][0, 0] == B.GP_ACT_COMPRESS
    _same(got, want)


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
def test_shared_units_with_keys_that_are_no_numbers(value):
    """One key element of one unit.  What the unit's scores then are, and the lists made from them, is what one thread block makes of them."""
    def edit(i, k, v):
        if i == 0:
            k[0, 5000, 1, 7] = value
    got, want = (_decode(1, 8, 2, 64, [642 * 16 - 1, 643 * 16 - 1], 2, tau=1.0, four=four, edit=edit) for four in (False, True))
    assert (got["shared"], want["shared"]) == (4, 0)
    _same(got, want)


@pytest.mark.parametrize("long_at_boundary", [True, False])
def test_shared_units_among_many_requests(long_at_boundary):
    """40 requests at their boundary, two of them long (the 35th and 38th), or only short ones beside long requests that are not at theirs.  One unit
    each: more than the clusters, so that a unit is shared out above 20 480 candidates."""
    lens = [47 + 16 * (i % 18) for i in range(40)]
    lens[34], lens[37] = (1302 * 16 - 1, 1310 * 16 - 1) if long_at_boundary else (1302 * 16 + 3, 1310 * 16 + 4)
    got, want = (_decode(1, 8, 1, 64, lens, 3, tau=1.0, four=four) for four in (False, True))
    assert (got["shared"], want["shared"]) == (2 if long_at_boundary else 0, 0) and got["status"] == (B.GP_OK, 0)
    assert (got["act"][0] == B.GP_ACT_COMPRESS).sum() == (40 if long_at_boundary else 38)
    _same(got, want)
