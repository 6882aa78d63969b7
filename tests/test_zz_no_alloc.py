"""The allocation-free attention entry point against the pool's own decode step and against the float64 oracle.

Some callers cannot give the library scratch memory or let it allocate (all device memory is committed to
the KV pool, or the host forbids allocator calls from plug-ins); `gp_attention_noalloc` serves them from a
fixed array inside the library.  This test feeds it the same keys and values the pool holds after a decode
step and expects the same attention output, on two consecutive calls (the array keeps the first call's
contents, which must not leak into the second), and compares it with the oracle's dense attention on
requests of ragged lengths, one of them empty.  It is collected last on purpose."""
import numpy as np
import pytest

from oracle import growpage_oracle as O
from paper_2609_03494_b200 import binding as B
from paper_2609_03494_b200 import workload as W

pytestmark = pytest.mark.gpu

ATTN_MAX_ABS = 1e-2      # same bound as the other attention parity tests
ATTN_MEAN_ABS = 1e-3


@pytest.mark.parametrize("hq,hkv,d,prompts", [(8, 2, 64, (37, 130, 300)), (32, 8, 128, (513, 16, 95, 1))])
def test_noalloc_attention_matches_the_pool_on_two_calls(hq, hkv, d, prompts):
    import torch
    rng = np.random.default_rng(7)
    n_req = len(prompts)
    cap = max(prompts) // 16 + 3
    cfg = B.make_config(1, hq, hkv, d, n_pages=n_req * cap, max_pages_per_req=cap, max_requests=8, tau=-1.0)
    pool = B.Pool(cfg)
    bits = lambda *shape: W.f32_to_bf16_bits(rng.standard_normal(shape).astype(np.float32))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda()
    try:
        for n in prompts:
            st, _ = pool.request_add(-1, 0, bits(1, n, hkv, d), bits(1, n, hkv, d), n, 0)
            assert st == B.GP_OK
        ids = torch.arange(n_req, dtype=torch.int32, device="cuda")
        max_len = max(prompts) + 2
        for step in range(2):
            q, k, v = bits(1, n_req, hq, d), bits(1, n_req, hkv, d), bits(1, n_req, hkv, d)
            out = torch.zeros((1, n_req, hq, d), dtype=torch.float32, device="cuda")
            act = torch.zeros(n_req, dtype=torch.int32, device="cuda")
            qd = dev(q)
            pool.decode_step(ids, qd, dev(k), dev(v), out, act)
            # the pool's keys and values after the step (the new token included), as plain dense tensors
            K = np.zeros((n_req, hkv, max_len, d), dtype=np.uint16)
            V = np.zeros((n_req, hkv, max_len, d), dtype=np.uint16)
            lens = np.zeros(n_req, dtype=np.int32)
            for r in range(n_req):
                _, n, _, _ = B.gp_debug_request(pool.handle, r, cap)
                lens[r] = n
                for h in range(hkv):
                    K[r, h, :n], V[r, h, :n] = B.gp_debug_kv(pool.handle, r, 0, h, n, d)
            assert lens.tolist() == [p + step + 1 for p in prompts]
            out2 = torch.full((n_req, hq, d), float("nan"), dtype=torch.float32, device="cuda")
            Kd, Vd, lens_d = dev(K), dev(V), torch.from_numpy(lens).cuda()      # the caller owns every buffer
            B.gp_attention_noalloc(qd.data_ptr(), Kd.data_ptr(), Vd.data_ptr(), lens_d.data_ptr(), n_req, hq, hkv, d,
                                   max_len, out2.data_ptr(), pool.stream())
            torch.cuda.synchronize()
            err = (out2 - out[0]).abs()
            assert float(err.max()) <= ATTN_MAX_ABS and float(err.mean()) <= ATTN_MEAN_ABS, (step, float(err.max()))
    finally:
        pool.close()


@pytest.mark.parametrize("hq,hkv,d,lens", [(8, 2, 64, (37, 0, 300, 1)), (32, 8, 128, (513, 16, 0, 95)), (16, 2, 128, (129,))])
def test_noalloc_attention_matches_the_oracle_and_an_empty_request_gives_zeros(hq, hkv, d, lens):
    import torch
    rng = np.random.default_rng(19)
    n_req, max_len = len(lens), max(lens) + 5
    bits = lambda *shape: W.f32_to_bf16_bits(rng.standard_normal(shape).astype(np.float32))
    q, K, V = bits(n_req, hq, d), bits(n_req, hkv, max_len, d), bits(n_req, hkv, max_len, d)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda()
    qd, Kd, Vd = dev(q), dev(K), dev(V)
    lens_d = torch.tensor(lens, dtype=torch.int32, device="cuda")
    f = W.bf16_bits_to_f64
    for call in range(2):                                    # the second call finds the first one's partials in the array
        out = torch.full((n_req, hq, d), float("nan"), dtype=torch.float32, device="cuda")
        B.gp_attention_noalloc(qd.data_ptr(), Kd.data_ptr(), Vd.data_ptr(), lens_d.data_ptr(), n_req, hq, hkv, d,
                               max_len, out.data_ptr(), 0)
        torch.cuda.synchronize()
        got = out.cpu().numpy().astype(np.float64)
        for r, n in enumerate(lens):
            if n == 0:
                assert np.array_equal(got[r], np.zeros((hq, d))), "an empty request must give a row of zeros"
                continue
            want = O.attention_decode(f(q[r]), f(K[r, :, :n]), f(V[r, :, :n]))
            err = np.abs(got[r] - want)
            assert err.max() <= ATTN_MAX_ABS and err.mean() <= ATTN_MEAN_ABS, (call, r, err.max())


def test_noalloc_rejects_what_does_not_fit():
    import torch
    z = torch.zeros(16, dtype=torch.int32, device="cuda")
    with pytest.raises(B.GpError) as e:
        B.gp_attention_noalloc(z.data_ptr(), z.data_ptr(), z.data_ptr(), z.data_ptr(), 128, 32, 8, 128, 4, z.data_ptr(), 0)
    assert e.value.status == B.GP_ERR_TOO_LARGE and "fixed scratch" in str(e.value)
    with pytest.raises(B.GpError) as e:
        B.gp_attention_noalloc(z.data_ptr(), z.data_ptr(), z.data_ptr(), z.data_ptr(), 1, 8, 2, 96, 4, z.data_ptr(), 0)
    assert e.value.status == B.GP_ERR_INVALID


def _dense(rng, hq, hkv, d, lens, max_len, offset=0):
    """Queries, keys and values on the device, keys and values `offset` elements past a 16-byte boundary; their values as float64."""
    import torch
    f = W.bf16_bits_to_f64
    arrays = [W.f32_to_bf16_bits((2.0 * rng.standard_normal(shape)).astype(np.float32))
              for shape in ((len(lens), hq, d), (len(lens), hkv, max_len, d), (len(lens), hkv, max_len, d))]
    on_gpu = []
    for i, a in enumerate(arrays):
        flat = torch.zeros(a.size + 8, dtype=torch.int16, device="cuda")
        part = flat[offset if i else 0:][:a.size]
        part.copy_(torch.from_numpy(a.view(np.int16).reshape(-1)))
        on_gpu.append(part)
    return on_gpu, [f(a) for a in arrays]


# Lengths at the edges of the 16- and 32-token tiles, of the warps' shares and of the splits (256 tokens of the longest
# request); every size of a group; keys and values on and off a 16-byte boundary.  Products of bf16 numbers are exact
# in fp32, weights keep 24 bits, and a sum of n tokens is rounded at most n / 16 / 4 + 30 times, each within 2^-24 of
# the sum of magnitudes: under 1e-6 of the result at these lengths and widths, where values do not cancel to nothing.
@pytest.mark.parametrize("hq,hkv,d,lens,offset", [
    (8, 2, 64, (1, 15, 16, 17, 31, 32, 33, 0, 127, 128, 129), 0),
    (6, 2, 64, (255, 256, 257, 513), 0),
    (8, 8, 128, (1, 15, 16, 17, 63, 64, 65, 0, 129), 0),
    (16, 2, 128, (1023, 1024, 1025, 3, 2000), 0),
    (5, 1, 128, (300, 7, 0), 0),
    (1, 1, 64, (5000,), 0),
    (8, 2, 128, (77, 300), 1),
    (7, 1, 64, (77, 300), 4),
    (16, 4, 128, (1, 0, 7, 8, 9, 31, 33, 1025), 1),
    (1, 1, 64, (5000,), 3),
    (8, 8, 64, (2500, 1) + (3,) * 118, 1),
])
def test_noalloc_attention_at_tile_and_split_edges(hq, hkv, d, lens, offset):
    import torch
    rng = np.random.default_rng(23)
    max_len = max(lens) + 3
    (q, K, V), (qf, Kf, Vf) = _dense(rng, hq, hkv, d, lens, max_len, offset)
    lens_d = torch.tensor(lens, dtype=torch.int32, device="cuda")
    out = torch.full((len(lens), hq, d), float("nan"), dtype=torch.float32, device="cuda")
    B.gp_attention_noalloc(q.data_ptr(), K.data_ptr(), V.data_ptr(), lens_d.data_ptr(), len(lens), hq, hkv, d, max_len,
                           out.data_ptr(), 0)
    got = out.cpu().numpy().astype(np.float64)
    for r, n in enumerate(lens):
        want = O.attention_decode(qf[r], Kf[r, :, :n], Vf[r, :, :n]) if n else np.zeros((hq, d))
        assert np.linalg.norm(got[r] - want) <= 1e-6 * np.linalg.norm(want), (r, n)


def test_noalloc_attention_with_an_infinite_value_keeps_the_other_columns():
    import torch
    rng = np.random.default_rng(29)
    hq, hkv, d, n = 8, 2, 128, 100
    (q, K, V), (qf, Kf, Vf) = _dense(rng, hq, hkv, d, (n,), n)
    V.view(1, hkv, n, d)[0, 1, 40, 5] = 0x7f80                     # +inf
    lens_d = torch.tensor([n], dtype=torch.int32, device="cuda")
    out = torch.zeros((1, hq, d), dtype=torch.float32, device="cuda")
    B.gp_attention_noalloc(q.data_ptr(), K.data_ptr(), V.data_ptr(), lens_d.data_ptr(), 1, hq, hkv, d, n, out.data_ptr(), 0)
    got = out.cpu().numpy().astype(np.float64)[0]
    want = O.attention_decode(qf[0], Kf[0], Vf[0])
    want[4:, 5] = np.inf
    # weights here are no smaller than about 2^-60, so that inf x weight is inf
    assert np.array_equal(np.isinf(got), np.isinf(want)) and not np.isnan(got).any()
    fin = np.isfinite(want)
    assert np.linalg.norm(got[fin] - want[fin]) <= 1e-6 * np.linalg.norm(want[fin])


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_noalloc_attention_with_a_key_that_is_no_finite_number(value, offset):
    """Against positive query elements a key element of -inf is a token without weight.  With +inf or NaN the weights of the heads that
    read it have no finite sum, and a row without a positive sum of weights is written as zeros.  The other heads are untouched."""
    import torch
    rng = np.random.default_rng(31)
    hq, hkv, d, n, G = 6, 2, 128, 100, 3
    (q, K, V), (qf, Kf, Vf) = _dense(rng, hq, hkv, d, (n,), n, offset)
    q.view(hq, d)[:, 5] = 0x3f80                                   # 1.0
    qf[0][:, 5] = 1.0
    K.view(hkv, n, d)[1, 45, 5] = 0x7fc0 if np.isnan(value) else 0x7f80 if value > 0 else 0xff80 - 0x10000
    if value == -np.inf:
        Kf[0, 1, 45, 5] = value
    lens_d = torch.tensor([n], dtype=torch.int32, device="cuda")
    out = torch.zeros((1, hq, d), dtype=torch.float32, device="cuda")
    B.gp_attention_noalloc(q.data_ptr(), K.data_ptr(), V.data_ptr(), lens_d.data_ptr(), 1, hq, hkv, d, n, out.data_ptr(), 0)
    got = out.cpu().numpy().astype(np.float64)[0]
    want = O.attention_decode(qf[0], Kf[0], Vf[0])
    clean = hq if value == -np.inf else G
    assert np.linalg.norm(got[:clean] - want[:clean]) <= 1e-6 * np.linalg.norm(want[:clean])
    assert not got[clean:].any()
