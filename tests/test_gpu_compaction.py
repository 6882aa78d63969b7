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
