"""The tensor-core mass pass has a kernel for each group width of 16 to 256
columns, head size and form of its work lists: few groups with the anchor beside
them (whole teams of CTAs), and 60 blocks of groups over seven key splits, which
152 SMs share by explicit lists. Groups that fill their columns and groups that
leave some as padding. Compared with a float64 softmax in plain torch under the
parity contract's mass tolerance (2e-3 relative, 1e-9 absolute)."""
import math

import pytest
import torch

import paper_2607_22586_gb300 as M
from tests import parity as PT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("r,gs,blocks", [(k, 16, 0) for k in range(1, 17)]
                         + [(1, 16 * k - 3, 60) for k in range(1, 17)])
def test_masses_of_every_group_width(d, r, gs, blocks):
    width = -(-r * gs // 16) * 16
    g, t = (blocks * (256 // width), 7000) if blocks else (3, 700)
    n, w = g * gs, 2
    gen = torch.Generator(device="cuda").manual_seed(width + d)
    K = torch.randn((t, 1, d), generator=gen, device="cuda").bfloat16()
    Q = torch.randn((1, w, r, d), generator=gen, device="cuda").bfloat16()
    prox = (3.0 * torch.randn((1, r, n, d), generator=gen, device="cuda")).bfloat16()
    shape = M.make_shape(r, 1, d, w, 0, [0, t], [1])
    params = M.default_params(n_proxies=n, n_groups=g)
    nb = M.mmshift_workspace_size(shape, params)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    gm = torch.full((1, g, t), -1.0, device="cuda")
    an = torch.full((1, t), -1.0, device="cuda")
    M.check(M.mmshift_proxy_mass(shape, K, Q, prox, params, gm, an, None, ws, nb), "proxy_mass")
    M.check(M.mmshift_poll_status(ws), "status")
    k, scale = K[:, 0].double(), 1.0 / math.sqrt(d)
    ref = torch.empty_like(gm[0], dtype=torch.float64)
    for i in range(g):
        q = prox[0, :, i * gs:(i + 1) * gs].double()
        ref[i] = torch.softmax(scale * (q @ k.T), -1).sum((0, 1))
    PT.mass_close(gm[0].cpu().numpy(), ref.cpu().numpy(), "group masses")
    a = torch.softmax(scale * (Q[0, -1].double() @ k.T), -1).mean(0)
    PT.mass_close(an[0].cpu().numpy(), a.cpu().numpy(), "anchor")
