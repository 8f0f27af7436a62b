"""mmshift_hidden_stats at the edges of its chunks (512 rows), of the copy
groups (4 rows, 32 ahead) and of a CTA's columns (64 threads of eight, in float32
of four):
compared with float64 in plain torch under the bounds of the statistics tests
(fp32 sums shifted by the chunk's first row, chunks merged pairwise: mean within
5e-5 (|mean| + std), std within 2e-4 std + 1e-6 |mean|)."""
import pytest
import torch

import paper_2607_22586_gb300 as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [(1, 2, 3), (4, 5, 6, 33, 34), (36, 37, 511), (512, 513, 514), (1025, 1600)])
@pytest.mark.parametrize("ncol,dtype", [(64, "bf16"), (520, "bf16"), (3584, "bf16"), (8, "f32"), (264, "f32"),
                                        (2056, "f32")])
def test_statistics_at_edges(lens, ncol, dtype):
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(sum(lens) + ncol)
    L, total = 2, sum(lens)
    mean = torch.randn(ncol, generator=gen, device="cuda")
    mean[::37] = 20.0
    H = (mean + torch.randn((L, total, ncol), generator=gen, device="cuda")).to(dt)
    cu = [0]
    for t in lens:
        cu.append(cu[-1] + t)
    shape = M.make_shape(4, 1, 64, 2, 0 if dtype == "bf16" else 1, cu, [1] * len(lens), n_layers=L,
                         layer_stride_kv=total * 64, layer_stride_q=len(lens) * 2 * 4 * 64)
    nb = M.mmshift_hidden_stats_workspace_size(shape, ncol)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    out = torch.full((L, len(lens), 2, ncol), -1.0, device="cuda")
    M.check(M.mmshift_hidden_stats(shape, ncol, H, 0, out, ws, nb), "hidden_stats")
    torch.cuda.synchronize()
    for l in range(L):
        for b, (lo, hi) in enumerate(zip(cu, cu[1:])):
            x = H[l, lo:hi].double()
            mu = x.mean(0)
            sd = x.std(0, unbiased=True) if hi - lo > 1 else torch.zeros_like(mu)
            assert bool(((out[l, b, 0] - mu).abs() <= 5e-5 * (mu.abs() + sd)).all())
            assert bool(((out[l, b, 1] - sd).abs() <= 2e-4 * sd + 1e-6 * mu.abs()).all())
