"""The compaction's two shapes (a ticket is a whole unit, or a part of one whose evicted slots the unit's last part waits for), and
what a request looks like after many of them: rows move into evicted slots, the order of the tokens is kept beside them."""
import numpy as np
import pytest

from paper_2609_03494_b200 import binding as B
from paper_2609_03494_b200 import workload as W
from tests import lockstep as LS

pytestmark = pytest.mark.gpu
SHRINK = dict(policy=B.GP_POLICY_SHRINK, min_capacity=64, tau=-0.03, shrink_below=-0.036)


def _by_part(monkeypatch):
    make = LS.make_pools

    def pools(*a, **kw):
        gpu, ora = make(*a, **kw)
        B.gp_test_withhold(gpu.handle, 32, 0)           # parts of 64 slots
        return gpu, ora
    monkeypatch.setattr(LS, "make_pools", pools)


@pytest.mark.parametrize("config,over", [(1, dict(tau=-0.05)), (3, dict()), (5, dict()), (5, SHRINK), (5, dict(overlap_slots=-1)),
                                         (1, dict(async_boundary=True, tau=-0.05)), (5, dict(async_boundary=True))])
def test_units_in_parts(config, over, monkeypatch):
    _by_part(monkeypatch)
    st = LS.run_lockstep(W.parity_instance(config), **over)
    assert st.decisions["sel"] > 0 and st.counters[8] > 0 and st.near_ties == {"ws": 0, "sel": 0, "act": 0}


@pytest.mark.parametrize("b,over", [(256, dict(tau=-0.05)), (32, dict(tau=-0.03)), (64, dict(policy=B.GP_POLICY_SHRINK, shrink_below=0.0,
                                                                                          min_capacity=128, tau=0.05))])
def test_units_in_parts_with_larger_pages(b, over, monkeypatch):
    _by_part(monkeypatch)
    s = W.Shape(1, 8, 2, 64, page_size=b)
    reqs = [W.RequestSpec(i, p, 4 * b, 0.05, share_group=-1) for i, p in enumerate((b + 44, 40, 2 * b - 1))]
    wl = W.Workload(f"b{b}", 77, s, reqs, n_resident=3, initial_pages=0, max_pages_per_req=5, n_pages=14, k_loc=b // 4)
    st = LS.run_lockstep(wl, summary_every=64, check_pool_every=32, **over)
    assert st.decisions["sel"] > 0


@pytest.mark.parametrize("d", [64, 128])
def test_rows_and_ids_stay_together_through_many_compactions(d):
    """Every retained row is the one its token id had when it was appended, ids ascend, the newest sixteen are there; heads and
    layers each on their own."""
    import torch
    layers, hq, hkv, n0, steps, cap = 2, 4, 2, 75, 165, 6
    rng = np.random.default_rng(23)
    bits = lambda *shape: W.f32_to_bf16_bits(rng.standard_normal(shape).astype(np.float32))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda()
    pool = B.Pool(B.make_config(layers, hq, hkv, d, n_pages=cap, max_pages_per_req=cap, max_requests=4))
    try:
        k, v = bits(layers, n0 + steps, hkv, d), bits(layers, n0 + steps, hkv, d)
        assert pool.request_add(-1, 0, np.ascontiguousarray(k[:, :n0]), np.ascontiguousarray(v[:, :n0]), n0, 0)[0] == B.GP_OK
        ids, act = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        out = torch.zeros((layers, 1, hq, d), dtype=torch.float32, device="cuda")
        compressed = 0
        for t in range(n0, n0 + steps):
            pool.decode_step(ids, dev(bits(layers, 1, hq, d)), dev(k[:, t:t + 1]), dev(v[:, t:t + 1]), out, act)
            if int(act[0]) not in (B.GP_ACT_COMPRESS, B.GP_ACT_COMPRESS_FALLBACK):
                continue
            compressed += 1
            _, n, pos, _ = B.gp_debug_request(pool.handle, 0, cap)
            for l in range(layers):
                for h in range(hkv):
                    tok = B.gp_debug_retained(pool.handle, 0, l, h, n)
                    assert (np.diff(tok) > 0).all() and tok[-1] == t and (tok[-16:] == np.arange(t - 15, t + 1)).all()
                    gk, gv = B.gp_debug_kv(pool.handle, 0, l, h, n, d)
                    assert np.array_equal(gk, k[l, tok, h]) and np.array_equal(gv, v[l, tok, h])
        assert compressed >= 5 and B.gp_pool_status(pool.handle) == (B.GP_OK, 0)
    finally:
        pool.close()


def _decode(lens, steps, forms, layers=2, hq=4, hkv=2, d=64, page=16, tau=10.0, shared=None, **config):
    """`steps` decode steps of requests with prompts of `lens` tokens (the first `shared` pages of each those of request 0) on a pool
    with a page to spare for each, once per form (early planning, compaction switch, overlap_slots; a host wait after every step only
    where there is no early planning): outputs, actions, and every request's state, ids and rows."""
    import torch
    n_req, cap = len(lens), max(lens) // page + 3
    shared = shared or [0] * n_req
    rng = np.random.default_rng(41)
    bits = lambda *shape: W.f32_to_bf16_bits(rng.standard_normal(shape).astype(np.float32))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda()
    prompts = [(m, dev(bits(layers, n - m * page, hkv, d)), dev(bits(layers, n - m * page, hkv, d)), n - m * page) for n, m in zip(lens, shared)]
    ins = [tuple(dev(bits(layers, n_req, h, d)) for h in (hq, hkv, hkv)) for _ in range(steps)]
    ids = torch.arange(n_req, dtype=torch.int32, device="cuda")
    results = []
    for early, switch, overlap in forms:
        pool = B.Pool(B.make_config(layers, hq, hkv, d, n_pages=sum(n // page + 2 for n in lens), max_pages_per_req=cap, page_size=page,
                                    k_loc=page // 4, max_requests=max(4, n_req), overlap_slots=overlap, tau=tau, **config))
        try:
            for m, k, v, n in prompts:
                assert pool.request_add(0 if m else -1, m, k, v, n, 0)[0] == B.GP_OK
            B.gp_set_early_plan(pool.handle, early)
            B.gp_test_withhold(pool.handle, switch, 0)
            outs = torch.zeros((steps, layers, n_req, hq, d), dtype=torch.float32, device="cuda")
            acts = torch.zeros((steps, n_req), dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            for t in range(steps):
                pool.decode_step(ids, *ins[t], outs[t], acts[t])
                if not early:
                    torch.cuda.synchronize()
            torch.cuda.synchronize()
            assert B.gp_pool_status(pool.handle) == (B.GP_OK, 0)
            state = [B.gp_debug_request(pool.handle, r, cap)[:3] for r in range(n_req)]
            kept = [a for r in range(n_req) for l in range(layers) for h in range(hkv)
                    for a in (B.gp_debug_retained(pool.handle, r, l, h, state[r][1]), *B.gp_debug_kv(pool.handle, r, l, h, state[r][1], d))]
            results.append((outs.cpu().numpy(), acts.cpu().numpy(), state, kept))
        finally:
            pool.close()
    return results


def _assert_equal(results):
    (o1, a1, s1, k1) = results[0]
    for o2, a2, s2, k2 in results[1:]:
        assert np.array_equal(a1, a2) and s1 == s2 and np.array_equal(o1, o2)
        assert len(k1) == len(k2) and all(np.array_equal(x, y) for x, y in zip(k1, k2))


def test_parts_beside_an_early_plan():
    """With early planning the plan of a step runs beside the compaction of the step before and writes its own boundary records there.
    Three requests of unequal length compress at every step, other ones from step to step (the records' places in the scratch differ),
    no host wait lies between the steps: parts of 64 slots give what whole units without early planning give, bit for bit."""
    lens = [16 * (4 + (7 * i) % 45) - 1 - i // 3 for i in range(48)]
    results = _decode(lens, 40, [(False, 16, -1), (True, 32, -2), (True, 32, -1), (True, 16, -2), (False, 32, -2)])
    compress = np.isin(results[0][1], (B.GP_ACT_COMPRESS, B.GP_ACT_COMPRESS_FALLBACK))
    assert (compress.sum(axis=1) >= 3).all()
    _assert_equal(results)


def test_parts_of_long_units_beside_an_early_plan():
    """The parts as they are (units of up to three, each of several passes of its thread block), early planning on and off."""
    lens = [16 * m - 1 - i % 2 for i, m in enumerate((257, 300, 513, 520, 770, 40))]
    results = _decode(lens, 20, [(False, 16, -1), (True, 0, -2), (True, 0, -1)], layers=1)
    assert np.isin(results[0][1], (B.GP_ACT_COMPRESS, B.GP_ACT_COMPRESS_FALLBACK)).sum() >= 12
    _assert_equal(results)


@pytest.mark.parametrize("d,page,over", [(128, 16, {}), (64, 16, {}), (64, 32, {}), (128, 16, dict(policy=B.GP_POLICY_SHRINK, min_capacity=64,
                                                                                           shrink_below=0.05))])
def test_copied_units_in_parts(d, page, over):
    """Units that are copied on write are shared out by their tiles: requests that share all, some or few of their pages, that compress in
    the same step or later ones, against whole units."""
    shared = [0, 139, 80, 100, 9, 8, 1, 60, 0, 139]
    lens = [page * m - x for m, x in ((140, 1), (140, 1), (90, 1), (200, 1), (10, 1), (9, 1), (30, 1), (70, 5), (30, 1), (141, 3))]
    results = _decode(lens, page + 6, [(False, 16, -1), (False, 0, -2), (True, 0, -2), (True, 0, -1), (True, 32, -2)], d=d, page=page, shared=shared,
                      **over)
    done = np.isin(results[0][1], (B.GP_ACT_COMPRESS, B.GP_ACT_COMPRESS_FALLBACK, B.GP_ACT_SHRINK))
    assert done.any(axis=0).all() and (done[0].sum() >= 7 if page == 16 else True)
    _assert_equal(results)
