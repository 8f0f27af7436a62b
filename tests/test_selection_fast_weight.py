"""The float32 form of the coverage vote's fixed-point weights (csrc/select.cu,
total_and_max): x + 96 rounds x in [0, 32) to a multiple a of 2^-17, one FMA
rounds (x - a) 2^40 to an integer, and a 2^40 plus that integer is x 2^40
rounded to the nearest integer, halves to even. The steps are restated here
with the kernel's bit-pattern sums and compared with the exact product."""
import numpy as np
import pytest
import torch

import paper_2607_22586_gb300 as M
from oracle import mmshift_oracle as O
from paper_2607_22586_gb300 import synth as S
from tests import parity as PT

F96, F23 = np.float32(96.0), np.float32(12582912.0)


def fast_weights(x: np.ndarray) -> np.ndarray:
    t = (x + F96).astype(np.float32)
    a = (t - F96).astype(np.float32)
    rest = (x - a).astype(np.float32)
    assert np.all(rest.astype(np.float64) == x.astype(np.float64) - a.astype(np.float64))
    # one rounding, as the FMA: the sum fits the wider type except for terms
    # too small to matter
    f = (rest.astype(np.longdouble) * np.longdouble(2.0 ** 40) + np.longdouble(F23)).astype(np.float32)
    hi = t.view(np.uint32).astype(np.int64) - 0x42C00000
    lo = f.view(np.uint32).astype(np.int64) - 0x4B400000
    assert hi.min() >= 0 and hi.max() <= 1 << 22 and np.abs(lo).max() <= 1 << 22
    return (hi << 23) + lo


def _check(x):
    got = fast_weights(x)
    want = np.rint(x.astype(np.float64) * 2.0 ** 40).astype(np.int64)
    bad = np.nonzero(got != want)[0]
    assert bad.size == 0, [(float(x[i]).hex(), int(got[i]), int(want[i])) for i in bad[:5]]


def test_random_values_of_every_exponent():
    rng = np.random.default_rng(0)
    e = rng.integers(127 - 60, 127 + 5, size=400_000)
    bits = (e.astype(np.uint32) << 23) | rng.integers(0, 1 << 23, size=e.size).astype(np.uint32)
    _check(bits.view(np.float32))


def test_edges_and_halves():
    ints = np.arange(0, 1 << 12, dtype=np.float64)
    x = [np.array([0.0, np.nextafter(np.float32(32), np.float32(0)), 2.0 ** -41, 2.0 ** -40, 1e-45])]
    for scale in (2.0 ** -40, 2.0 ** -30, 2.0 ** -18, 2.0 ** -17):
        x += [ints * scale, (ints + 0.5) * scale, (ints + 0.25) * scale]
    x = np.concatenate(x)
    x = x[x < 32.0].astype(np.float32)
    _check(x)


def test_sums_of_a_carry_interval_do_not_wrap():
    # 64 quads of the largest values: the kernel's 32-bit sums less the biases
    x = np.full(256, np.nextafter(np.float32(32), np.float32(0)), dtype=np.float32)
    t = (x + F96).view(np.uint32).astype(np.uint64).sum() % (1 << 32)
    hi = (int(t) - 256 * 0x42C00000) % (1 << 32)
    assert hi < 1 << 31 and hi == 256 * (1 << 22)


@pytest.mark.gpu
def test_votes_exact_with_heavy_keys_and_long_rows():
    """Keys of 32 and more take the integer form, quad by quad, and a row of
    140,000 keys carries its 32-bit sums: votes equal the oracle's."""
    wl = S.WORKLOADS["72b-80l-ragged"].replace(
        name="long", n_layers=1, seq_lens=(140001, 60), n_visual=(0, 0), budgets=(500, 8))
    h = PT.hyper(n_proxies=32, n_groups=2)
    T, hkv, G = wl.total_tokens, wl.n_kv_heads, 2
    gm = S.make_group_masses(hkv, G, T, 112.0, seed=12)
    heavy = np.array([32.0, 31.999998, 100.0, 33.5, 32.000004], dtype=np.float32)
    gm[:, 0, 5:140001:20011] = np.resize(heavy, gm[:, 0, 5:140001:20011].shape)
    anchor = S.make_scores(hkv, T, 0, seed=13) * np.float32(0.5)
    shape, params = PT.shape_of(wl), PT.abi_params(h)
    nb = M.mmshift_workspace_size(shape, params)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    idx = torch.empty((1, M.mmshift_output_rows(shape), hkv), dtype=torch.int32, device="cuda")
    sc = torch.empty((1, hkv, T), device="cuda")
    M.check(M.mmshift_scores_topk(shape, params, torch.from_numpy(gm).cuda(),
                                  torch.from_numpy(anchor).cuda(), sc, idx, ws, nb), "scores_topk")
    got = PT.host(sc)[0]
    for lo, hi in ((0, 140001), (140001, 140061)):
        for hh in range(hkv):
            v = O.votes(O.cover_sets(gm[hh, :, lo:hi].astype(np.float64), h["tau"]))
            want = (v.astype(np.float32) + np.float32(h["lam"]) * anchor[hh, lo:hi]).astype(np.float32)
            np.testing.assert_array_equal(got[hh, lo:hi], want)
