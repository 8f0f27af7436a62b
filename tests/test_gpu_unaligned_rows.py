"""Rows at addresses (or layers at strides) that no 16-byte access takes: the keys
and values of a selection and of the gather alone, the gathered rows, and proxies
written for the caller. The results are those of aligned copies, to the bit."""
import pytest
import torch

import paper_2607_22586_gb300 as M

pytestmark = pytest.mark.gpu


def _at(x, shift):
    """x at an address `shift` elements past a 256-byte boundary."""
    buf = torch.zeros(x.numel() + 64, dtype=x.dtype, device="cuda")
    y = buf[shift:shift + x.numel()].view(x.shape)
    y.copy_(x)
    return y


@pytest.mark.parametrize("dt", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("shifts,pad", [((1, 0, 0, 0), 0), ((0, 3, 0, 0), 0), ((0, 0, 1, 0), 0),
                                        ((0, 0, 0, 5), 0), ((1, 1, 1, 1), 0), ((0, 0, 0, 0), 3)])
def test_gather_of_unaligned_rows(dt, d, shifts, pad):
    L, t, hq, hkv, w, budget = 2, 300, 8, 2, 4, 40
    gen = torch.Generator(device="cuda").manual_seed(d)
    row = t * hkv * d
    K, V = (torch.randn((L, row + pad), generator=gen, device="cuda").to(dt) for _ in range(2))
    Q = torch.randn((L, 1, w, hq, d), generator=gen, device="cuda").to(dt)
    shape = M.make_shape(hq, hkv, d, w, 0 if dt == torch.bfloat16 else 1, [0, t], [budget], n_layers=L,
                         layer_stride_kv=row + pad, layer_stride_q=w * hq * d)
    params = M.default_params(n_proxies=16, n_groups=2)
    nb = max(M.mmshift_workspace_size(shape, p) for p in (params, None))   # the gather's: default parameters
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    idx = torch.empty((L, budget, hkv), dtype=torch.int32, device="cuda")
    ok, ov = (_at(torch.zeros((L, budget, hkv, d), dtype=dt, device="cuda"), s) for s in shifts[2:])
    k, v = _at(K, shifts[0]), _at(V, shifts[1])
    M.check(M.mmshift_select(shape, k, v, Q, None, params, idx, ok, ov, None, ws, nb), "select")
    M.check(M.mmshift_poll_status(ws), "status")
    sel = idx.long()[..., None].expand(-1, -1, -1, d)
    want = [x[:, :row].reshape(L, t, hkv, d).gather(1, sel) for x in (K, V)]
    assert torch.equal(ok, want[0]) and torch.equal(ov, want[1])
    # the gather alone; -1 and other bad indices give zero rows
    idx[0, 0, 0] = -1
    M.check(M.mmshift_gather(shape, k, v, idx, ok, ov, ws, nb), "gather")
    assert M.mmshift_poll_status(ws) != 0
    for got, ref in zip((ok, ov), want):
        ref[0, 0, 0] = 0
        assert torch.equal(got, ref)


@pytest.mark.parametrize("dt", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("shift", [1, 2, 4, 5])
def test_proxies_at_unaligned_addresses(dt, shift):
    hq, hkv, d, w, n, t = 8, 2, 128, 4, 24, 50
    gen = torch.Generator(device="cuda").manual_seed(shift)
    Q = torch.randn((1, w, hq, d), generator=gen, device="cuda").to(dt)
    shape = M.make_shape(hq, hkv, d, w, 0 if dt == torch.bfloat16 else 1, [0, t], [5])
    params = M.default_params(n_proxies=n, n_groups=2, rope_theta=1e6)
    stats = torch.rand((1, 2, hq * d), generator=gen, device="cuda")
    for build, arg in ((M.mmshift_build_proxies, Q), (M.mmshift_build_proxies_from_stats, stats)):
        ref = torch.zeros((1, hq, n, d), dtype=dt, device="cuda")
        got = _at(ref, shift)
        M.check(build(shape, arg, params, ref), "aligned")
        M.check(build(shape, arg, params, got), "unaligned")
        torch.cuda.synchronize()
        assert torch.equal(got, ref) and float(got.abs().max()) > 0


@pytest.mark.parametrize("shift", [1, 4, 8])
@pytest.mark.parametrize("n", [100, 200])         # one tile of proxies, a pair of tiles
def test_projected_proxies_at_unaligned_addresses(shift, n):
    hq, hkv, d, dm = 4, 2, 64, 128
    gen = torch.Generator(device="cuda").manual_seed(n)
    shape = M.make_shape(hq, hkv, d, 2, 0, [0, 30], [5])
    params = M.default_params(n_proxies=n, n_groups=1, rope_theta=1e6)
    stats = torch.rand((1, 1, 2, dm), generator=gen, device="cuda")
    W = (0.1 * torch.randn((1, hq * d, dm), generator=gen, device="cuda")).bfloat16()
    nb = M.mmshift_hidden_proxies_workspace_size(shape, dm, params)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    ref = torch.zeros((1, 1, hq, n, d), dtype=torch.bfloat16, device="cuda")
    got = _at(ref, shift)
    for out in (ref, got):
        M.check(M.mmshift_build_hidden_proxies(shape, dm, stats, W, 0, None, None, params, out, ws, nb),
                "hidden proxies")
        M.check(M.mmshift_poll_status(ws), "status")
    assert torch.equal(got, ref) and float(got.float().abs().max()) > 0
