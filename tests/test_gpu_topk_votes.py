"""The top-k's votes with more than eight groups (csrc/select.cu): a CTA reads the
coverage words of 4,096 keys and 32 groups at a time along the groups' rows and
turns them in shared memory. Group counts around 32 and 64, lengths around the
4,096 keys and the 32 of a word, requests that start inside a call's words; 512
and 1024 threads. Scores and kept sets equal the oracle's exactly."""
import numpy as np
import pytest
import torch

import paper_2607_22586_gb300 as M
from oracle import mmshift_oracle as O
from paper_2607_22586_gb300 import synth as S
from tests import parity as PT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,hkv,g", [
    ((4096, 31), 1, 9),
    ((4095, 4097, 33), 1, 32),
    ((8193, 2), 2, 33),
    ((1000, 32, 64), 1, 70),
    ((41, 95, 4128) + tuple(range(2, 52)), 3, 10),    # 159 units: 512 threads
])
def test_scores_exact_with_many_groups(lens, hkv, g):
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    total, keep, tau = cu[-1], [max(1, t // 3) for t in lens], 0.95
    gm = S.make_group_masses(hkv, g, total, 112.0, seed=len(lens) + g)
    anchor = S.make_scores(hkv, total, 0, seed=6) * np.float32(0.5)
    shape = M.make_shape(2 * hkv, hkv, 64, 2, 0, cu, keep)
    h = PT.hyper(n_proxies=16 * g, n_groups=g, tau=tau)
    params = PT.abi_params(h)
    nb = M.mmshift_workspace_size(shape, params)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    idx = torch.full((1, M.mmshift_output_rows(shape), hkv), -1, dtype=torch.int32, device="cuda")
    sc = torch.empty((1, hkv, total), device="cuda")
    M.check(M.mmshift_scores_topk(shape, params, torch.from_numpy(gm).cuda(),
                                  torch.from_numpy(anchor).cuda(), sc, idx, ws, nb), "scores_topk")
    M.check(M.mmshift_poll_status(ws), "status")
    sc, idx, olo = PT.host(sc)[0], PT.host(idx)[0], 0
    for b, t in enumerate(lens):
        lo = cu[b]
        for hh in range(hkv):
            v = O.votes(O.cover_sets(gm[hh, :, lo:lo + t].astype(np.float64), tau))
            want = (v.astype(np.float32) + np.float32(h["lam"]) * anchor[hh, lo:lo + t]).astype(np.float32)
            np.testing.assert_array_equal(sc[hh, lo:lo + t], want)
            np.testing.assert_array_equal(idx[olo:olo + keep[b], hh],
                                          O.select_topk(want.astype(np.float64), keep[b]))
        olo += keep[b]
