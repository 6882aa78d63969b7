"""Admission: prompt rows land where the pool says they are, at the edges of the 16-token tiles and for head counts that do not
divide a block; a refused admission leaves the pool alone; pages return in table order, after a copy-on-write step too."""
import numpy as np
import pytest

from paper_2609_03494_b200 import binding as B
from paper_2609_03494_b200 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hkv,d,layers", [(1, 64, 1), (3, 128, 2), (8, 128, 2), (5, 64, 3)])
def test_prompt_rows_are_in_their_pages(hkv, d, layers):
    rng = np.random.default_rng(5)
    lens = (1, 15, 16, 17, 33, 300)
    pages = sum(n // 16 + 1 for n in lens)
    pool = B.Pool(B.make_config(layers, hkv, hkv, d, n_pages=pages, max_pages_per_req=20, max_requests=8))
    try:
        rows = []
        for n in lens:
            k, v = (W.f32_to_bf16_bits(rng.standard_normal((layers, n, hkv, d)).astype(np.float32)) for _ in range(2))
            st, rid = pool.request_add(-1, 0, k, v, n, 0)
            assert st == B.GP_OK
            rows.append((rid, n, k, v))
        # the pool is full: refused, and nothing of the pool has changed
        assert pool.request_add(-1, 0, rows[0][2], rows[0][3], 1, 0)[0] == B.GP_ERR_NO_PAGES
        assert B.gp_debug_pool(pool.handle)[0] == 0
        for rid, n, k, v in rows:
            assert B.gp_debug_request(pool.handle, rid, 20)[:3] == (n // 16 + 1, n, n)
            for l in range(layers):
                for h in range(hkv):
                    gk, gv = B.gp_debug_kv(pool.handle, rid, l, h, n, d)
                    assert np.array_equal(gk, k[l, :, h]) and np.array_equal(gv, v[l, :, h])
                    assert np.array_equal(B.gp_debug_retained(pool.handle, rid, l, h, n), np.arange(n))
    finally:
        pool.close()


def test_released_pages_come_back_in_table_order():
    # a request of 300 pages (more than a thread block's worth) and sharers of half of it
    rng = np.random.default_rng(6)
    n = 300 * 16 - 1
    k, v = (W.f32_to_bf16_bits(rng.standard_normal((1, n, 1, 64)).astype(np.float32)) for _ in range(2))
    pool = B.Pool(B.make_config(1, 1, 1, 64, n_pages=310, max_pages_per_req=300, max_requests=8))
    try:
        st, a = pool.request_add(-1, 0, k, v, n, 0)
        assert st == B.GP_OK
        sharers = [pool.request_add(a, 150, None, None, 0, 0) for _ in range(3)]
        assert all(s == B.GP_OK for s, _ in sharers)
        n_free, ref, _ = B.gp_debug_pool(pool.handle, 310)
        assert n_free == 310 - 303 and sorted(ref)[-150:] == [4] * 150
        table = B.gp_debug_request(pool.handle, a, 300)[3]
        pool.release(a)                                             # its second half goes, the shared half stays
        assert B.gp_debug_pool(pool.handle)[0] == 310 - 153
        for _, rid in sharers:
            pool.release(rid)
        n_free, ref, counters = B.gp_debug_pool(pool.handle, 310)
        assert n_free == 310 and not ref.any() and counters[7] == 0
        # last in, first out: the shared half was pushed last, in table order, then the last sharer's own page
        st, b = pool.request_add(-1, 0, k[:, :1023], v[:, :1023], 1023, 0)
        got = B.gp_debug_request(pool.handle, b, 300)[3]
        assert st == B.GP_OK and list(got[1:64]) == list(table[149:86:-1])
    finally:
        pool.close()


@pytest.mark.parametrize("sharers", [2, 9, 40])
def test_pages_replaced_in_one_step_return_once_in_the_last_sharers_order(sharers):
    """All sharers of a prompt compress in the same step: each gets its own copies, and the shared pages go back to the free list
    once, when the last of them (the highest request id) has let go, in table order."""
    import torch
    rng = np.random.default_rng(8)
    P, d = 70, 64
    n0 = (P - 1) * 16
    pool = B.Pool(B.make_config(1, 4, 1, d, n_pages=(sharers + 1) * P, max_pages_per_req=P, max_requests=64, tau=10.0))
    bits = lambda *s: W.f32_to_bf16_bits(rng.standard_normal(s).astype(np.float32))
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x).view(np.int16)).cuda()
    try:
        st, a = pool.request_add(-1, 0, bits(1, n0, 1, d), bits(1, n0, 1, d), n0, 0)
        rids = [a] + [pool.request_add(a, P - 1, None, None, 0, 0)[1] for _ in range(sharers - 1)]
        shared = B.gp_debug_request(pool.handle, a, P)[3][:P - 1]
        ids = torch.tensor(rids, dtype=torch.int32, device="cuda")
        out = torch.zeros((1, sharers, 4, d), dtype=torch.float32, device="cuda")
        act = torch.zeros(sharers, dtype=torch.int32, device="cuda")
        for _ in range(16):
            pool.decode_step(ids, dev(bits(1, sharers, 4, d)), dev(bits(1, sharers, 1, d)), dev(bits(1, sharers, 1, d)), out, act)
        assert act.tolist() == [B.GP_ACT_COMPRESS] * sharers
        n_free, ref, counters = B.gp_debug_pool(pool.handle, (sharers + 1) * P)
        tables = [B.gp_debug_request(pool.handle, r, P)[3] for r in rids]
        own = [p for t in tables for p in t]
        assert len(set(own)) == len(own) == sharers * P and not set(own) & set(shared)
        assert n_free == P and counters[7] == 0 and sorted(ref) == [0] * P + [1] * (sharers * P)
        st, b = pool.request_add(-1, 0, bits(1, n0, 1, d), bits(1, n0, 1, d), n0, 0)
        assert st == B.GP_OK and list(B.gp_debug_request(pool.handle, b, P)[3][:P - 1]) == list(shared[::-1])
    finally:
        pool.close()


def test_misaligned_prompt_is_refused_before_any_launch():
    import torch
    pool = B.Pool(B.make_config(1, 2, 2, 64, n_pages=8, max_pages_per_req=4, max_requests=4))
    try:
        rows = torch.zeros(20 * 2 * 64 + 64, dtype=torch.int16, device="cuda")
        good = rows.data_ptr()
        launches = B.gp_launch_count(pool.handle)
        for k, v in ((good + 2, good), (good, good + 8), (good + 14, good + 14)):
            assert B.gp_request_add(pool.handle, -1, 0, k, v, 20, 0, pool.stream()) == (B.GP_ERR_INVALID, -1)
        assert B.gp_launch_count(pool.handle) == launches and B.gp_debug_pool(pool.handle)[0] == 8
        assert B.gp_request_add(pool.handle, -1, 0, good, good, 20, 0, pool.stream()) == (B.GP_OK, 0)
        assert B.gp_request_add(pool.handle, 0, 1, 2, 2, 0, 0, pool.stream()) == (B.GP_OK, 1)       # no tail: the pointers are not looked at
    finally:
        pool.close()


def test_a_prompt_past_the_page_cap_is_refused_without_copying_it():
    """With shared pages the refusal comes from the device (a bad donor is reported first): the prompt is not copied meanwhile, however
    long the caller says it is."""
    import torch
    pool = B.Pool(B.make_config(36, 2, 2, 64, n_pages=8, max_pages_per_req=4, max_requests=4))
    try:
        rows = torch.zeros(36 * 20 * 2 * 64, dtype=torch.int16, device="cuda").data_ptr()
        assert B.gp_request_add(pool.handle, -1, 0, rows, rows, 20, 0, pool.stream()) == (B.GP_OK, 0)
        for donor_pages, n_tail, want in ((1, 49, B.GP_ERR_NO_PAGES), (1, 2 ** 30, B.GP_ERR_NO_PAGES), (1, 2 ** 31 - 1, B.GP_ERR_NO_PAGES),
                                          (2, 2 ** 30, B.GP_ERR_INVALID)):
            launches = B.gp_launch_count(pool.handle)
            assert B.gp_request_add(pool.handle, 0, donor_pages, rows, rows, n_tail, 0, pool.stream()) == (want, -1)
            assert B.gp_launch_count(pool.handle) == launches + 1
        assert B.gp_debug_pool(pool.handle)[0] == 6 and B.gp_debug_request(pool.handle, 0, 4)[:3] == (2, 20, 20)
    finally:
        pool.close()
