"""A layer's launch may start while the layer before it on its stream still runs (its plan has been read by then): only the caller's
tensors are waited for.  Layers back to back on one stream, layers whose tensors are written right before them (one set of
buffers for all layers, so that the kernel before a layer writes what the layer before that one read), and layers that change streams
give what layers with a host wait between them give, bit for bit, through boundaries and compactions; requests of one to several
work items."""
import numpy as np
import pytest

from paper_2609_03494_b200 import binding as B
from paper_2609_03494_b200 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("how", ["back_to_back", "shared_buffers", "two_streams"])
@pytest.mark.parametrize("hq,hkv,d,n_req,rope", [(8, 2, 64, 3, 0.0), (16, 8, 128, 40, 1e6)])
def test_layers_that_overlap_equal_layers_one_by_one(how, hq, hkv, d, n_req, rope):
    import torch
    layers, steps = 5, 18
    lens = [15 + (61 * i) % 1100 for i in range(n_req)]
    cap = max(lens) // 16 + 3
    rng = np.random.default_rng(7)
    bits = lambda *shape: W.f32_to_bf16_bits(rng.standard_normal(shape).astype(np.float32))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda()
    prompts = [(dev(bits(layers, n, hkv, d)), dev(bits(layers, n, hkv, d)), n) for n in lens]
    ins = [tuple(dev(bits(layers, n_req, h, d)) for h in (hq, hkv, hkv)) for _ in range(steps)]
    ids = torch.arange(n_req, dtype=torch.int32, device="cuda")
    results = []
    for way in ("one_by_one", how):
        pool = B.Pool(B.make_config(layers, hq, hkv, d, n_pages=sum(n // 16 + 1 for n in lens) + 3, max_pages_per_req=cap,
                                    max_requests=max(4, n_req), rope_theta=rope))
        try:
            for k, v, n in prompts:
                assert pool.request_add(-1, 0, k, v, n, 0)[0] == B.GP_OK
            outs = torch.zeros((steps, layers, n_req, hq, d), dtype=torch.float32, device="cuda")
            acts = torch.zeros((steps, n_req), dtype=torch.int32, device="cuda")
            bufs = [torch.zeros_like(x[0]) for x in ins[0]] + [torch.zeros_like(outs[0, 0])]
            torch.cuda.synchronize()
            streams = [torch.cuda.current_stream(), torch.cuda.Stream()]
            for t in range(steps):
                q, k, v = ins[t]
                s = pool.stream()
                B.gp_step_begin(pool.handle, ids.data_ptr(), n_req, acts[t].data_ptr(), s)
                for i, l in enumerate((2, 0, 1, 4, 3)):
                    if way == "one_by_one":
                        torch.cuda.synchronize()
                    if way == "shared_buffers":
                        for b, x in zip(bufs, (q, k, v)):
                            b.copy_(x[l])
                        B.gp_attn_layer(pool.handle, l, ids.data_ptr(), n_req, *(b.data_ptr() for b in bufs), s)
                        outs[t, l].copy_(bufs[3])
                        continue
                    if way == "two_streams" and i:
                        streams[i % 2].wait_stream(streams[1 - i % 2])
                        s = streams[i % 2].cuda_stream
                    B.gp_attn_layer(pool.handle, l, ids.data_ptr(), n_req, q[l].data_ptr(), k[l].data_ptr(), v[l].data_ptr(), outs[t, l].data_ptr(), s)
                B.gp_step_end(pool.handle, ids.data_ptr(), n_req, acts[t].data_ptr(), pool.stream())
            torch.cuda.synchronize()
            assert B.gp_pool_status(pool.handle) == (B.GP_OK, 0)
            state = [B.gp_debug_request(pool.handle, r, cap)[:3] for r in range(n_req)]
            kept = [B.gp_debug_retained(pool.handle, r, l, h, state[r][1]) for r in range(0, n_req, 3) for l in (0, layers - 1) for h in range(hkv)]
            results.append((outs.cpu().numpy(), acts.cpu().numpy(), state, kept))
        finally:
            pool.close()
    (o1, a1, s1, k1), (o2, a2, s2, k2) = results
    assert (a1 != B.GP_ACT_NONE).any() and np.array_equal(a1, a2) and s1 == s2
    assert all(np.array_equal(x, y) for x, y in zip(k1, k2)) and np.array_equal(o1, o2)
