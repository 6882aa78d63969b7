"""Numbers at and past the edges of their formats: outputs that overflow, queries near the largest bf16, keys that are
infinite or not numbers."""
import numpy as np
import pytest

from oracle import growpage_oracle as O
from paper_2609_03494_b200 import binding as B
from paper_2609_03494_b200 import workload as W

pytestmark = pytest.mark.gpu


def _bits(rng, *shape):
    return W.f32_to_bf16_bits(rng.standard_normal(shape).astype(np.float32))


def _step(pool, q, k, v):
    """One decode step of request 0: outputs [L][H_q][d], action."""
    import torch
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda()
    L, _, hq, d = q.shape
    out = torch.zeros((L, 1, hq, d), dtype=torch.float32, device="cuda")
    act = torch.zeros(1, dtype=torch.int32, device="cuda")
    pool.decode_step(torch.zeros(1, dtype=torch.int32, device="cuda"), dev(q), dev(k), dev(v), out, act)
    torch.cuda.synchronize()
    return out.cpu().numpy()[:, 0], int(act[0])


# Work items of 32 pages: a request in one piece, in two, in three, in eleven (merged as eight and three) and in seventeen (eight,
# eight and one).  Queries of zero give every token the weight 1, so that the sum over a column of 3e38 is past fp32 in every piece.
@pytest.mark.parametrize("pages", [20, 64, 70, 330, 520])
def test_an_output_that_overflows_is_infinite_however_many_pieces_it_is_merged_from(pages):
    rng = np.random.default_rng(3)
    hq, d, n = 4, 64, pages * 16 - 8
    pool = B.Pool(B.make_config(1, hq, 1, d, n_pages=pages, max_pages_per_req=pages, max_requests=2))
    try:
        k, v = _bits(rng, 1, n + 1, 1, d), _bits(rng, 1, n + 1, 1, d)
        v[..., 9] = W.f32_to_bf16_bits(np.float32([3e38]))[0]
        assert pool.request_add(-1, 0, k[:, :n], v[:, :n], n, 0)[0] == B.GP_OK
        out, act = _step(pool, np.zeros((1, 1, hq, d), np.uint16), k[:, n:], v[:, n:])
        assert act == B.GP_ACT_NONE and np.isposinf(out[..., 9]).all()
        mean = W.bf16_bits_to_f64(v[0, :, 0]).mean(axis=0)
        # sums of n terms of size one, rounded to 24 bits after every sixteen
        assert np.abs(np.delete(out[0] - mean, 9, axis=1)).max() <= n / 16 * 2.0 ** -24 + 1e-6
    finally:
        pool.close()


@pytest.mark.parametrize("hq,d,rope_theta", [(4, 64, 0.0), (16, 128, 0.0), (4, 128, 1e4)])
def test_boundary_after_queries_near_the_largest_bf16(hq, d, rope_theta):
    """The summaries keep most of a one-hot first query while the boundary's own query is large in every element: its size lends
    the calibrated summary one element of more than 2^128.  Keys near the smallest normal bf16 make the logits ordinary."""
    rng = np.random.default_rng(5)
    L, hkv, pages = 1, 2, 5
    n = pages * 16 - 2
    kw = dict(n_pages=pages, max_pages_per_req=pages, max_requests=2, tau=2.0, rope_theta=rope_theta)
    pool, ora = B.Pool(B.make_config(L, hq, hkv, d, **kw)), O.OraclePool(O.OracleConfig(L, hq, hkv, d, **kw))
    f = W.bf16_bits_to_f64
    try:
        keys = W.f32_to_bf16_bits((2e-38 * rng.standard_normal((L, n + 2, hkv, d))).astype(np.float32))
        vals = _bits(rng, L, n + 2, hkv, d)
        assert pool.request_add(-1, 0, keys[:, :n], vals[:, :n], n, 0)[0] == B.GP_OK
        assert ora.request_add(-1, 0, f(keys[:, :n]), f(vals[:, :n]), n, 0)[0] == O.OK
        first = np.zeros((L, 1, hq, d), np.float32)
        first[..., 3] = 1e38
        second = rng.uniform(1e38, 2e38, (L, 1, hq, d)) * rng.choice([-1.0, 1.0], (L, 1, hq, d))
        for t, q in enumerate((first, second.astype(np.float32))):
            q = W.f32_to_bf16_bits(q)
            _, act = _step(pool, q, keys[:, n + t:n + t + 1], vals[:, n + t:n + t + 1])
            rec = ora.decode_step([0], f(q), f(keys[:, n + t:n + t + 1]), f(vals[:, n + t:n + t + 1]))
            assert [act] == rec.actions.tolist()
        assert act == B.GP_ACT_COMPRESS
        ks, kl, delta = B.gp_debug_boundary(pool.handle, 0, L, hkv)
        info = rec.boundary[0]
        assert np.array_equal(ks, info.K_s) and np.array_equal(kl, info.K_l) and (ks > 1).all()
        left = ora.request_state(0)[1]
        for h in range(hkv):
            assert np.array_equal(B.gp_debug_retained(pool.handle, 0, 0, h, left), ora.retained(0, 0, h))
        assert B.gp_debug_pool(pool.handle)[2][7] == 0
    finally:
        pool.close()


# With few units a thread block takes one task of a unit; with overlap_slots = 1 the boundary kernel has one block, which takes
# whole units.
@pytest.mark.parametrize("hq,d", [(2, 64), (8, 64), (16, 128)])
@pytest.mark.parametrize("slots", [0, 1])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_a_key_that_is_no_finite_number_shows_in_its_units_scores(value, slots, hq, d):
    """Against positive query elements a key element of -inf is a token without weight.  With +inf or NaN no score of the unit is a number:
    its working sets are all candidates and, all scores being equal, the evicted slots go by their order.  The other unit is untouched."""
    rng = np.random.default_rng(7)
    L, hkv, pages, k_loc = 1, 2, 6, 4
    n = pages * 16 - 1
    kw = dict(n_pages=pages, max_pages_per_req=pages, max_requests=2, tau=2.0, k_loc=k_loc)
    pool = B.Pool(B.make_config(L, hq, hkv, d, overlap_slots=slots, **kw))
    ora = O.OraclePool(O.OracleConfig(L, hq, hkv, d, **kw))
    f = W.bf16_bits_to_f64
    try:
        keys, vals = _bits(rng, L, n + 1, hkv, d), _bits(rng, L, n + 1, hkv, d)
        q = W.f32_to_bf16_bits(np.abs(rng.standard_normal((L, 1, hq, d))).astype(np.float32) + 0.1)
        bad = keys.copy()
        bad[0, 37, 1, 5] = {True: 0x7fc0, False: 0x7f80 if value > 0 else 0xff80}[bool(np.isnan(value))]
        exact = bad if value == -np.inf else keys                  # what the oracle can follow
        assert pool.request_add(-1, 0, bad[:, :n], vals[:, :n], n, 0)[0] == B.GP_OK
        ora.request_add(-1, 0, f(exact[:, :n]), f(vals[:, :n]), n, 0)
        out, act = _step(pool, q, keys[:, n:], vals[:, n:])
        rec = ora.decode_step([0], f(q), f(keys[:, n:]), f(vals[:, n:]))
        assert act == B.GP_ACT_COMPRESS and rec.actions.tolist() == [act]
        ks, kl, _ = B.gp_debug_boundary(pool.handle, 0, L, hkv)
        G, n_c = hq // hkv, (pages - 1) * 16
        slots_left = np.arange(n_c)
        rest = slots_left[slots_left % 16 >= k_loc]
        by_order = np.setdiff1d(np.arange(n + 1), rest[len(rest) - 16:])
        for h in range(hkv):
            kept = B.gp_debug_retained(pool.handle, 0, 0, h, n_c)
            if h == 1 and value != -np.inf:
                assert np.isnan(out[0, G:]).all() and (ks[0, h], kl[0, h]) == (n_c, n_c)
                assert np.array_equal(kept, by_order)
            else:
                assert np.abs(out[0, h * G:(h + 1) * G] - rec.out[0, 0, h * G:(h + 1) * G]).max() <= 1e-2
                assert (ks[0, h], kl[0, h]) == (rec.boundary[0].K_s[0, h], rec.boundary[0].K_l[0, h])
                assert np.array_equal(kept, ora.retained(0, 0, h))
        assert B.gp_debug_pool(pool.handle)[2][7] == 0
    finally:
        pool.close()
