"""The coverage vote's ranking of its candidates (csrc/select.cu, rank_among):
masses on a coarse grid, so that many candidates have the same key and the lower
index decides, at counts around the quads of keys read at once and the threads
of a CTA (512, or 256 in calls of many units). Votes and kept sets equal the
oracle's exactly."""
import numpy as np
import pytest
import torch

import paper_2607_22586_gb300 as M
from oracle import mmshift_oracle as O
from paper_2607_22586_gb300 import synth as S
from tests import parity as PT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels", [1, 3, 64])
@pytest.mark.parametrize("lens,hkv,g", [
    ((2, 3, 4, 5, 31, 33), 2, 2),
    ((127, 128, 129, 255, 257), 1, 4),
    ((511, 512, 513), 1, 3),
    ((63, 255, 256, 257), 4, 32),     # 512 units: 256 threads each
])
def test_votes_exact_with_equal_masses(lens, hkv, g, levels):
    rng = np.random.default_rng(levels + sum(lens))
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    total, keep = cu[-1], [max(1, t // 3) for t in lens]
    # The parameters hold tau in float32. On a grid of sixths a prefix can weigh
    # 0.9 of the total to within 0.9's rounding (2.4e-8), where the oracle's
    # float64 tau ends one key later; 0.875 and its products are exact in both.
    tau = 0.875
    gm = (0.5 + rng.integers(0, levels, size=(hkv, g, total)) / (2.0 * levels)).astype(np.float32)
    anchor = S.make_scores(hkv, total, 0, seed=5) * np.float32(0.5)
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
