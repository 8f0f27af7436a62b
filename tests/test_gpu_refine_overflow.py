"""A call that leaves more proxy elements undecided than its refinement list
holds (csrc/proxy.cu) recomputes every element. Window rows that alternate
between two neighbouring bf16 values have means halfway between them, and a
gamma far below the rounding of float32 leaves every element there, rotated ones
too at position 0: all of them overflow a list of elements / 64 + 16,384 entries
(half as many where they take 64 bits). Compared with mmshift_build_proxies, which
has no list; the elements are the mean nudged by the normal's sign, so both of
the mean's neighbours have to appear."""
import pytest
import torch

import paper_2607_22586_gb300 as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,lens,hq,hkv,d,n,g,rope", [
    (1, (40,), 28, 4, 128, 8, 1, 0.0),            # 28,672 elements, a list of 16,832: just above it
    (1, (40,), 28, 4, 128, 8, 1, 1e6),
    (3, (50, 2, 31), 28, 4, 64, 40, 4, 0.0),
    (5, (90, 90, 90), 28, 4, 128, 96, 2, 1e6),
    (4, (200,), 16, 16, 64, 512, 32, 1e6),
    (129, (3,), 33, 33, 64, 2052, 4, 0.0),        # 64-bit entries
    (80, (3,) * 8, 64, 8, 128, 512, 32, 0.0),     # more undecided elements than 2^31
])
def test_overflow_equals_a_full_recomputation(layers, lens, hq, hkv, d, n, g, rope):
    w, dt, b = 8, torch.bfloat16, len(lens)
    gen = torch.Generator(device="cuda").manual_seed(n)
    cu = [0]
    for t in lens:
        cu.append(cu[-1] + t)
    K = torch.randn((layers, cu[-1], hkv, d), generator=gen, device="cuda").to(dt)
    lo = (1.0 + torch.rand((layers, b, 1, hq, d), generator=gen, device="cuda") * 0.9).to(dt)
    step = torch.arange(w, device="cuda").view(1, 1, w, 1, 1) % 2
    Q = (lo.view(torch.int16) + step.to(torch.int16)).contiguous().view(dt)   # lo, the next value, lo, ...
    shape = M.make_shape(hq, hkv, d, w, 0, cu, [1] * b, n_layers=layers,
                         layer_stride_kv=cu[-1] * hkv * d, layer_stride_q=b * w * hq * d)
    params = M.default_params(n_proxies=n, n_groups=g, rope_theta=rope, seed=3, gamma=1e-6,
                              rope_pos_offset=-lens[0])
    nb = M.mmshift_workspace_size(shape, params)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    rows = M.mmshift_output_rows(shape)
    idx = torch.empty((layers, rows, hkv), dtype=torch.int32, device="cuda")
    ok = torch.empty((layers, rows, hkv, d), dtype=dt, device="cuda")
    ov = torch.empty_like(ok)
    listed = torch.zeros((layers, b, hq, n, d), dtype=dt, device="cuda")
    dbg = M.make_debug(proxies=listed)
    M.check(M.mmshift_select(shape, K, K, Q, None, params, idx, ok, ov, dbg, ws, nb), "select")
    M.check(M.mmshift_poll_status(ws), "status")
    full = torch.empty_like(listed)
    M.check(M.mmshift_build_proxies(shape, Q, params, full), "build_proxies")
    torch.cuda.synchronize()
    assert torch.equal(listed.view(torch.int16), full.view(torch.int16))
    for l in range(layers):
        up = listed[l].view(torch.int16) - lo[l].view(torch.int16).view(b, hq, 1, d)
        assert int(up.min()) == 0 and int(up.max()) == 1
        assert 0.4 < float(up.float().mean()) < 0.6
