"""The anchor of a call whose requests all have at most eight key splits of 1024
keys comes from one kernel on a cluster with a CTA per split; a longer request
in the call sends it through two kernels. Both take every sum in the same order,
so the short requests' anchor is the same to the bit, and a float64 softmax is
met under the parity contract's mass tolerance (2e-3 relative, 1e-9 absolute).
The proxies fill whole blocks of 256 rows, so the anchor rows have their own."""
import math

import pytest
import torch

import paper_2607_22586_gb300 as M
from tests import parity as PT

pytestmark = pytest.mark.gpu


def _anchor(K, Q, prox, lens, hq, hkv, w, n, g):
    cu = [0]
    for t in lens:
        cu.append(cu[-1] + t)
    shape = M.make_shape(hq, hkv, K.shape[-1], w, 0, cu, [1] * len(lens))
    params = M.default_params(n_proxies=n, n_groups=g)
    nb = M.mmshift_workspace_size(shape, params)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    gm = torch.full((hkv, g, cu[-1]), -1.0, device="cuda")
    an = torch.full((hkv, cu[-1]), -1.0, device="cuda")
    M.check(M.mmshift_proxy_mass(shape, K, Q, prox, params, gm, an, None, ws, nb), "proxy_mass")
    M.check(M.mmshift_poll_status(ws), "status")
    return an


@pytest.mark.parametrize("lens,hq,hkv,d,n,g", [
    ((1, 1023, 1024), 4, 1, 64, 64, 4),          # one split each
    ((1025, 31, 2048), 28, 4, 128, 256, 4),      # two, seven anchor rows
    ((2049, 3000, 5000), 4, 2, 128, 128, 2),     # clusters of five CTAs
    ((8192, 257), 16, 2, 128, 128, 8),           # eight, eight anchor rows
    ((7169, 8191, 1), 1, 1, 64, 256, 2),         # one anchor row
])
def test_one_kernel_equals_two(lens, hq, hkv, d, n, g):
    gen = torch.Generator(device="cuda").manual_seed(3 + sum(lens))
    longer, w = 8193, 3
    total = sum(lens)
    K = torch.randn((total + longer, hkv, d), generator=gen, device="cuda").bfloat16()
    Q = (3.0 * torch.randn((len(lens) + 1, w, hq, d), generator=gen, device="cuda")).bfloat16()
    prox = torch.randn((len(lens) + 1, hq, n, d), generator=gen, device="cuda").bfloat16()
    one = _anchor(K[:total], Q[:-1], prox[:-1], lens, hq, hkv, w, n, g)
    two = _anchor(K, Q, prox, (*lens, longer), hq, hkv, w, n, g)
    assert torch.equal(one, two[:, :total])
    lo, r = 0, hq // hkv
    for b, t in enumerate(lens):
        for h in range(hkv):
            a, k = Q[b, -1, h * r:(h + 1) * r].double(), K[lo:lo + t, h].double()
            ref = torch.softmax((a @ k.T) / math.sqrt(d), -1).mean(0)
            PT.mass_close(one[h, lo:lo + t].cpu().numpy(), ref.cpu().numpy(), f"request {b} head {h}")
        lo += t
