"""The attention kernel's consumer warps take one 16-token tile at a time at d = 128 and two at d = 64: lengths around the ends of tiles,
of pairs, of a round of the four warps' pairs and of work items, every group size, against the float64 attention.  The weights are
carried as bf16 with their bf16 residual (2^-17 of each), logits and sums in fp32: under 2^-15 of the largest value (4.5 for these
inputs), 1.4e-4."""
import numpy as np
import pytest

from oracle import growpage_oracle as O
from paper_2609_03494_b200 import binding as B
from paper_2609_03494_b200 import workload as W

pytestmark = pytest.mark.gpu
LENS = (1, 14, 15, 16, 17, 30, 31, 32, 33, 47, 48, 62, 63, 64, 65, 95, 126, 127, 128, 129, 159, 254, 255, 256, 257, 300, 510, 511, 512, 513,
        527, 528, 1023, 1024, 1040, 2049)


@pytest.mark.parametrize("rope", [0.0, 1e6])
@pytest.mark.parametrize("hq,hkv,d", [(2, 2, 64), (4, 2, 64), (8, 2, 64), (16, 2, 64), (8, 2, 128), (16, 2, 128)])
def test_lengths_around_tiles_pairs_and_items(hq, hkv, d, rope):
    import torch
    rng = np.random.default_rng(3)
    n_req, cap = len(LENS), max(LENS) // 16 + 3
    bits = lambda *shape: W.f32_to_bf16_bits(rng.standard_normal(shape).astype(np.float32))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda()
    f = W.bf16_bits_to_f64
    pool = B.Pool(B.make_config(1, hq, hkv, d, n_pages=sum(n // 16 + 2 for n in LENS), max_pages_per_req=cap, max_requests=n_req, rope_theta=rope))
    try:
        prompts = [(bits(1, n, hkv, d), bits(1, n, hkv, d)) for n in LENS]
        for n, (k, v) in zip(LENS, prompts):
            assert pool.request_add(-1, 0, k, v, n, 0)[0] == B.GP_OK
        q, k, v = bits(1, n_req, hq, d), bits(1, n_req, hkv, d), bits(1, n_req, hkv, d)
        out = torch.zeros((1, n_req, hq, d), dtype=torch.float32, device="cuda")
        act = torch.zeros(n_req, dtype=torch.int32, device="cuda")
        pool.decode_step(torch.arange(n_req, dtype=torch.int32, device="cuda"), dev(q), dev(k), dev(v), out, act)
        got = out.cpu().numpy().astype(np.float64)[0]
        assert B.gp_pool_status(pool.handle) == (B.GP_OK, 0)
        half = d // 2
        for i, n in enumerate(LENS):
            K, V = np.concatenate([f(prompts[i][0][0]), f(k[0, i:i + 1])]), np.concatenate([f(prompts[i][1][0]), f(v[0, i:i + 1])])
            qq = f(q[0, i])
            if rope:
                ang = n * rope ** (-np.arange(half) / half)
                c, s = np.cos(ang), np.sin(ang)
                qq = np.concatenate([qq[:, :half] * c - qq[:, half:] * s, qq[:, half:] * c + qq[:, :half] * s], axis=1)
            want = O.attention_decode(qq, K.transpose(1, 0, 2), V.transpose(1, 0, 2))
            assert np.abs(got[i] - want).max() <= 1.4e-4, (n, np.abs(got[i] - want).max())
    finally:
        pool.close()


@pytest.mark.parametrize("hq,hkv,lo,hi", [(2, 2, 64, 240), (4, 2, 64, 240), (8, 2, 64, 240), (16, 2, 64, 240), (8, 2, 200, 1800), (16, 2, 200, 1800)])
def test_weights_in_pairs_of_tiles_keep_their_bits(hq, hkv, lo, hi):
    """d = 64, keys of which some are heavy hitters along the queries.  Two bf16 terms of a weight, 2^-17 of each, leave an error of
    1.6e-6 to 1.8e-6 of the outputs' 2-norm with a tile at a time and of 1.7e-6 to 1.9e-6 with two that share a maximum.  Groups of up to
    four carry a third term, 2^-24: what is left is a logit's fp32 sum of 64 products of up to 16 in magnitude, off by some 2^-22 x 16 /
    sqrt(64), and so is its weight: 1e-6 at most.  Groups of eight carry it for every other tile: half of the squared error of 1.9e-6, 1.4e-6."""
    import torch
    rng = np.random.default_rng(29)
    d, n_req = 64, 48
    lens = [int(x) for x in np.linspace(lo, hi, n_req)]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(W.f32_to_bf16_bits(a.astype(np.float32))).view(np.int16)).cuda()
    rounded = lambda a: W.bf16_bits_to_f64(W.f32_to_bf16_bits(a.astype(np.float32)))
    u = rng.standard_normal((hkv, d))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    uq = np.repeat(u, hq // hkv, axis=0)

    def keys(n):
        k = rng.standard_normal((n, hkv, d))
        heavy = rng.random(n) < np.exp(rng.uniform(np.log(0.005), np.log(0.2)))
        k[heavy] = 4.0 * u + 0.1 * k[heavy]
        return rounded(k)
    pool = B.Pool(B.make_config(1, hq, hkv, d, n_pages=sum(n // 16 + 2 for n in lens), max_pages_per_req=hi // 16 + 3, max_requests=n_req))
    try:
        K = [keys(n) for n in lens]
        V = [rounded(rng.standard_normal((n, hkv, d))) for n in lens]
        for n, k, v in zip(lens, K, V):
            assert pool.request_add(-1, 0, dev(k[None, :-1]), dev(v[None, :-1]), n - 1, 0)[0] == B.GP_OK
        q = rounded(2.0 * uq + rng.standard_normal((n_req, hq, d)))
        out = torch.zeros((1, n_req, hq, d), dtype=torch.float32, device="cuda")
        act = torch.zeros(n_req, dtype=torch.int32, device="cuda")
        pool.decode_step(torch.arange(n_req, dtype=torch.int32, device="cuda"), dev(q[None]), dev(np.stack([k[-1] for k in K])[None]),
                         dev(np.stack([v[-1] for v in V])[None]), out, act)
        got = out.cpu().numpy().astype(np.float64)[0]
        want = np.stack([O.attention_decode(q[i], K[i].transpose(1, 0, 2), V[i].transpose(1, 0, 2)) for i in range(n_req)])
        err = np.linalg.norm(got - want) / np.linalg.norm(want)
        assert err < (1e-6 if hq < 8 * hkv else 1.4e-6), err
    finally:
        pool.close()
