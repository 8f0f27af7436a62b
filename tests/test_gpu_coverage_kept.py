"""mmshift_coverage at the edges of its two-softmax form: kept sets with
padding rows anywhere, budgets around the 256-entry copy blocks and the
1024-key splits, decode query counts around 32 per CTA, one query head per KV
head, a KV head with no kept row, float32 and misaligned keys, and a budget so
large that the group-mass form runs. Compared with a float64 softmax in plain
torch: each sum of exponentials is within 2e-6 relative (float32 terms at
most 2^-23 |log2| off, |log2| < 24 where a term matters), so the ratio is
within 5e-6 of the reference plus 1e-9."""
import math

import pytest
import torch

import paper_2607_22586_gb300 as M
from paper_2607_22586_gb300 import _lib as LB

pytestmark = pytest.mark.gpu


def _inputs(lens, budgets, hq, hkv, d, L, n_dec, dt, shift, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    total, w = sum(lens), 2
    buf = torch.randn(L * total * hkv * d + 8, generator=gen, device="cuda").to(dt)
    K = buf[shift:shift + L * total * hkv * d].view(L, total, hkv, d)
    Q = torch.randn((L, len(lens), w, hq, d), generator=gen, device="cuda").to(dt)
    dec = (1.5 * torch.randn((L, len(lens), hq, n_dec, d), generator=gen, device="cuda")).to(dt)
    idx = []
    for t, c in zip(lens, budgets):
        keep = min(c, t)
        pick = torch.rand((L, t, hkv), generator=gen, device="cuda").topk(keep, dim=1).indices
        pick = pick.sort(dim=1).values.to(torch.int32)
        drop = torch.rand((L, keep, hkv), generator=gen, device="cuda") < 0.2
        idx.append(torch.where(drop, -1, pick))
    return K, Q, dec, torch.cat(idx, dim=1).to(torch.int32).contiguous()


def _run(K, Q, dec, idx, lens, budgets, hq, hkv, d, L, n_dec, dt):
    cu = [0]
    for t in lens:
        cu.append(cu[-1] + t)
    shape = M.make_shape(hq, hkv, d, 2, 0 if dt == torch.bfloat16 else 1, cu, budgets, n_layers=L,
                         layer_stride_kv=cu[-1] * hkv * d, layer_stride_q=len(lens) * 2 * hq * d)
    nb = M.mmshift_coverage_workspace_size(shape, n_dec)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    cov = torch.full((L, len(lens), hkv, n_dec), -1.0, device="cuda")
    M.check(M.mmshift_coverage(shape, K, Q, dec, n_dec, 0.0, idx, cov, ws, nb), "coverage")
    return cov, M.mmshift_poll_status(ws)


@pytest.mark.parametrize("lens,budgets,hq,hkv,d,L,n_dec,dtype,shift", [
    ((300, 2, 77), (64, 1, 16), 64, 8, 128, 2, 33, "bf16", 0),
    ((1500, 1025), (255, 257), 28, 4, 128, 1, 32, "bf16", 0),
    ((5000,), (1025,), 8, 2, 64, 1, 100, "bf16", 0),
    ((4097,), (200,), 16, 16, 128, 2, 1, "bf16", 0),
    ((2049,), (512,), 4, 1, 64, 2, 31, "f32", 0),
    ((700,), (100,), 28, 4, 128, 1, 16, "bf16", 1),       # keys at an odd address
    ((600,), (600,), 28, 4, 128, 1, 2, "bf16", 0),        # the group-mass form
])
def test_coverage_of_padded_kept_sets(lens, budgets, hq, hkv, d, L, n_dec, dtype, shift):
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    K, Q, dec, idx = _inputs(lens, budgets, hq, hkv, d, L, n_dec, dt, shift, 3 + sum(lens))
    idx[0, :min(budgets[0], lens[0]), 0] = -1              # a head that kept nothing
    cov, status = _run(K, Q, dec, idx, lens, budgets, hq, hkv, d, L, n_dec, dt)
    assert status == LB.MMSHIFT_OK
    r, scale = hq // hkv, 1.0 / math.sqrt(d)
    for l in range(L):
        lo = off = 0
        for b, (t, c) in enumerate(zip(lens, budgets)):
            keep = min(c, t)
            for h in range(hkv):
                k = K[l, lo:lo + t, h].double()
                q = dec[l, b, h * r:(h + 1) * r].double()
                p = torch.softmax(scale * (q @ k.T), -1)
                i = idx[l, off:off + keep, h].long()
                ref = p[:, :, i[i >= 0]].sum(-1).mean(0)
                err = (cov[l, b, h].double() - ref).abs()
                assert bool((err <= 5e-6 * ref + 1e-9).all()), (l, b, h, float((err / (ref + 1e-9)).max()))
            lo += t
            off += keep
    assert float(cov[0, 0, 0].abs().max()) == 0.0


def test_bad_index_is_left_out_and_reported():
    lens, budgets = (900,), (300,)
    K, Q, dec, idx = _inputs(lens, budgets, 28, 4, 128, 1, 8, torch.bfloat16, 0, 11)
    ref, status = _run(K, Q, dec, idx, lens, budgets, 28, 4, 128, 1, 8, torch.bfloat16)
    assert status == LB.MMSHIFT_OK
    idx[idx == -1] = 900                                   # past the prompt: left out like -1
    got, status = _run(K, Q, dec, idx, lens, budgets, 28, 4, 128, 1, 8, torch.bfloat16)
    assert status == LB.MMSHIFT_ERR_DEVICE
    assert torch.equal(got, ref)
