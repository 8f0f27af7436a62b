"""The mass pass on the CUDA cores (float32) with its groups in ranges of
different lengths: short last ranges, the anchor in a range of its own or with
the last groups, one range for all. Compared with a float64 softmax in plain torch
under the parity contract's mass tolerance (2e-3 relative, 1e-9 absolute). The
ranges follow the number of SMs: those noted at the cases are a GB300's, and are
checked there."""
import pytest
import torch

import paper_2607_22586_gb300 as M
from tests import parity as PT
from tests.group_ranges import ranges
from tests.test_gpu_simt_tiles import _reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,hq,hkv,d,n,g,layout", [
    ((9000,), 8, 2, 64, 40, 5, (3, False, 2)),          # 3 + 2 groups, the anchor with the 2
    ((12000,), 8, 2, 64, 24, 3, (3, False, 1)),         # all groups and the anchor in one range
    ((6000, 300), 16, 2, 128, 72, 9, (3, True, 4)),     # 3 + 3 + 3 and the anchor alone
    ((5000,), 28, 4, 64, 160, 10, (2, True, 6)),        # five ranges of two and the anchor alone
    ((700,), 8, 8, 128, 28, 7, (4, True, 3)),           # 4 + 3 and the anchor, one query head per KV head
    ((1000,), 4, 1, 64, 32, 2, (1, True, 3)),            # one group each and the anchor
])
def test_masses_in_group_ranges(lens, hq, hkv, d, n, g, layout):
    r, nsm = hq // hkv, torch.cuda.get_device_properties(0).multi_processor_count
    rows = lambda k: -(-k // 16) * 16
    keyu = hkv * sum(-(-t // 128) for t in lens)
    gper, own, rs = ranges([(g, rows(r * n // g), rows(r), keyu, nsm)])[0]
    assert nsm != 152 or (gper, own, len(rs)) == layout
    gen = torch.Generator(device="cuda").manual_seed(sum(lens))
    total, w = sum(lens), 4
    K = torch.randn((total, hkv, d), generator=gen, device="cuda")
    Q = torch.randn((len(lens), w, hq, d), generator=gen, device="cuda")
    prox = 4.0 * torch.randn((len(lens), hq, n, d), generator=gen, device="cuda")
    cu = [0]
    for t in lens:
        cu.append(cu[-1] + t)
    shape = M.make_shape(hq, hkv, d, w, 1, cu, [1] * len(lens))
    params = M.default_params(n_proxies=n, n_groups=g)
    nb = M.mmshift_workspace_size(shape, params)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    gm = torch.full((hkv, g, total), -1.0, device="cuda")
    an = torch.full((hkv, total), -1.0, device="cuda")
    M.check(M.mmshift_proxy_mass(shape, K, Q, prox, params, gm, an, None, ws, nb), "proxy_mass")
    M.check(M.mmshift_poll_status(ws), "status")
    ref_gm, ref_an = _reference(K, Q, prox, lens, hq, hkv, g)
    PT.mass_close(gm.cpu().numpy(), ref_gm.cpu().numpy(), "group masses")
    PT.mass_close(an.cpu().numpy(), ref_an.cpu().numpy(), "anchor")
