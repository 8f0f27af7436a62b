"""Steps 2-4 on the CUDA cores (float32 inputs, and keys whose base address a
TMA load cannot take) at the edges of their tiles: 64 proxy rows, 128 keys in
two runs of 64, key splits of 1024 shared by up to eight CTAs, groups spread
over CTAs. Compared with a float64 softmax in plain torch under the parity
contract's mass tolerance (2e-3 relative, 1e-9 absolute)."""
import math

import pytest
import torch

import paper_2607_22586_gb300 as M
from tests import parity as PT

pytestmark = pytest.mark.gpu


def _reference(K, Q, prox, lens, hq, hkv, g):
    r, n = hq // hkv, prox.shape[2]
    total = sum(lens)
    gm = torch.zeros((hkv, max(g, 1), total), dtype=torch.float64, device="cuda")
    an = torch.zeros((hkv, total), dtype=torch.float64, device="cuda")
    scale = 1.0 / math.sqrt(K.shape[-1])
    lo = 0
    for b, t in enumerate(lens):
        for h in range(hkv):
            k = K[lo:lo + t, h].double()
            for i in range(g):
                q = prox[b, h * r:(h + 1) * r, i * (n // g):(i + 1) * (n // g)].double()
                gm[h, i, lo:lo + t] = torch.softmax(scale * (q @ k.T), -1).sum((0, 1))
            a = Q[b, -1, h * r:(h + 1) * r].double()
            an[h, lo:lo + t] = torch.softmax(scale * (a @ k.T), -1).mean(0)
        lo += t
    return gm, an


@pytest.mark.parametrize("lens,hq,hkv,d,n,g,dtype,shift", [
    ((1,), 4, 1, 64, 32, 2, "f32", 0),
    ((63, 64, 65), 4, 2, 64, 16, 2, "f32", 0),          # a run of 64 keys
    ((127, 128, 129), 14, 2, 128, 32, 2, "f32", 0),     # a tile of keys, 112-row groups
    ((1023, 1024, 1025), 4, 1, 64, 64, 4, "f32", 0),    # a key split
    ((2300,), 8, 8, 128, 24, 3, "f32", 1),              # one head per KV head; unaligned base
    ((300, 2), 64, 8, 128, 512, 32, "f32", 0),          # 4,112 proxy rows
    ((700,), 4, 1, 64, 0, 0, "f32", 0),                 # the anchor alone
    ((900, 130), 28, 4, 128, 64, 4, "bf16", 1),         # bf16 keys at an odd address
])
def test_masses_at_tile_edges(lens, hq, hkv, d, n, g, dtype, shift):
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(7 + sum(lens))
    total, w = sum(lens), 4
    buf = torch.randn(total * hkv * d + 8, generator=gen, device="cuda").to(dt)
    K = buf[shift:shift + total * hkv * d].view(total, hkv, d)
    Q = torch.randn((len(lens), w, hq, d), generator=gen, device="cuda").to(dt)
    prox = (4.0 * torch.randn((len(lens), hq, max(n, 1), d), generator=gen, device="cuda")).to(dt)
    cu = [0]
    for t in lens:
        cu.append(cu[-1] + t)
    shape = M.make_shape(hq, hkv, d, w, 1 if dtype == "f32" else 0, cu, [1] * len(lens))
    params = M.default_params(n_proxies=n, n_groups=g)
    nb = M.mmshift_workspace_size(shape, params)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    gm = torch.full((hkv, max(g, 1), total), -1.0, device="cuda")
    an = torch.full((hkv, total), -1.0, device="cuda")
    M.check(M.mmshift_proxy_mass(shape, K, Q, prox if n else None, params, gm if g else None, an,
                                 None, ws, nb), "proxy_mass")
    M.check(M.mmshift_poll_status(ws), "status")
    ref_gm, ref_an = _reference(K, Q, prox, lens, hq, hkv, g)
    if g:
        PT.mass_close(gm.cpu().numpy(), ref_gm.cpu().numpy(), "group masses")
    PT.mass_close(an.cpu().numpy(), ref_an.cpu().numpy(), "anchor")
