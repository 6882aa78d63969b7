"""Numbers at and past the edges of their formats: outputs that overflow, queries near the largest bf16."""
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
