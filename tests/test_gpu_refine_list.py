"""The list of proxy elements that the sampler leaves undecided (csrc/proxy.cu):
entries pack layer and request, query head, proxy and dimension into 32 bits, or
64 where they need more. A call with the list gives the same bits as one without
(mmshift_build_proxies), which recomputes every element in float64."""
import pytest
import torch

import paper_2607_22586_gb300 as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,lens,hq,hkv,n,g,rope", [
    (1, (40,), 1, 1, 8, 1, 1e6),                  # fields of no bits
    (3, (50, 2, 31), 28, 4, 40, 4, 0.0),          # sizes that are no powers of two
    (5, (90, 40, 7), 28, 4, 96, 2, 1e6),
    (4, (200,), 16, 16, 512, 32, 1e6),            # 24,000 undecided of 4.2 million, rotated
    (129, (3,), 33, 33, 2052, 4, 1e6),            # 33 bits: 64-bit entries
])
def test_listed_elements_equal_a_full_recomputation(layers, lens, hq, hkv, n, g, rope):
    d, w, dt = 128, 9, torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(n)
    cu = [0]
    for t in lens:
        cu.append(cu[-1] + t)
    total, b = cu[-1], len(lens)
    K = torch.randn((layers, total, hkv, d), generator=gen, device="cuda").to(dt)
    Q = (torch.randn((layers, 1, 1, hq, d), generator=gen, device="cuda")
         + torch.randn((layers, b, w, hq, d), generator=gen, device="cuda")).to(dt)
    shape = M.make_shape(hq, hkv, d, w, 0, cu, [1] * b, n_layers=layers,
                         layer_stride_kv=total * hkv * d, layer_stride_q=b * w * hq * d)
    params = M.default_params(n_proxies=n, n_groups=g, rope_theta=rope, seed=3)
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
