"""The hidden-space projection on CTA pairs (an even number of 128-proxy tiles)
at its edges: a last tile with few proxies, 128-feature tiles (half a tile of 64
features per CTA), fewer tiles than pairs, and outputs at an address that only
8-byte stores take. Same oracle and bounds as the other hidden-proxy tests."""
import numpy as np
import pytest
import torch

import paper_2607_22586_gb300 as M
from paper_2607_22586_gb300 import synth as S
from tests import parity as PT
from tests.test_gpu_hidden import _check_projection, _gpu_hidden_proxies, _stats

pytestmark = pytest.mark.gpu

BASE = S.WORKLOADS["qwen7b-1layer"].replace(n_q_heads=4, n_kv_heads=1, seq_lens=(300, 77),
                                            n_visual=(250, 50), budgets=(64, 8))


@pytest.mark.parametrize("n_p,hq,d,dm,rope", [(200, 4, 128, 256, 1e6), (256, 6, 64, 128, 0.0),
                                              (129, 2, 64, 64, 1e4), (512, 8, 128, 320, 0.0)])
def test_pair_tiles_match_oracle(n_p, hq, d, dm, rope):
    wl = BASE.replace(n_q_heads=hq, n_kv_heads=1, head_dim=d)
    h = PT.hyper(n_proxies=n_p, n_groups=1, seed=5, layer_id=1, rope_theta=rope, rope_pos_offset=1)
    hid = S.make_hidden_states(wl, 0, dm)
    w, bias = S.make_query_projection(wl, 0, dm, True)
    st = _stats(wl, [hid])
    got = _gpu_hidden_proxies(wl, dm, st, [w], [bias], h)
    for b in range(wl.batch):
        _check_projection(got[0, b], st[0, b], w, bias, h, b, wl.seq_lens[b] + 1, hq, 1)


def test_outputs_at_an_eight_byte_address():
    dm, n_p = 128, 256
    h = PT.hyper(n_proxies=n_p, n_groups=1, seed=6)
    hid = S.make_hidden_states(BASE, 0, dm)
    w, bias = S.make_query_projection(BASE, 0, dm, True)
    st = _stats(BASE, [hid])
    want = _gpu_hidden_proxies(BASE, dm, st, [w], [bias], h)
    shape, params = PT.shape_of(BASE), PT.abi_params(h)
    nb = M.mmshift_hidden_proxies_workspace_size(shape, dm, params)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    buf = torch.zeros(want.size + 4, dtype=torch.bfloat16, device="cuda")
    wq = PT.dev(w[None], S.BF16)
    # the bias two bytes off its alignment as well
    bb = torch.zeros(bias.size + 1, dtype=torch.bfloat16, device="cuda")
    bb[1:] = PT.dev(bias, S.BF16)
    sd = torch.from_numpy(np.ascontiguousarray(st)).cuda()
    M.check(M.mmshift_build_hidden_proxies(shape, dm, sd, wq, 0, bb[1:], None, params, buf[4:], ws, nb),
            "build_hidden_proxies")
    M.check(M.mmshift_poll_status(ws), "status")
    np.testing.assert_array_equal(PT.host(buf[4:]).reshape(want.shape), want)
