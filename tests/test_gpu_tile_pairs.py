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
