"""mmshift_coverage of logits that are not finite: a decode query with a NaN or
+inf logit under any query head of a KV head, or with nothing but -inf logits,
has coverage 0 there, whether such a key is among the kept ones or not; every
other (query, KV head) is as without it. Runs of 16, 32 and 64 keys are the units
in which the passes take their maxima."""
import math

import pytest
import torch

import paper_2607_22586_gb300 as M
from paper_2607_22586_gb300 import _lib as LB

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,shift,keep,n_dec", [
    ("bf16", 128, 0, 200, 3), ("bf16", 64, 0, 100, 33),     # tensor cores
    ("f32", 128, 0, 50, 3), ("bf16", 64, 1, 100, 3),        # CUDA cores
    ("bf16", 128, 0, 1100, 1),                              # the group-mass form
])
@pytest.mark.parametrize("what,val", [
    ("query", math.nan), ("kept key", math.nan), ("other key", math.nan), ("first 64 keys", math.nan),
    ("last 16 keys", math.nan), ("keys 1024-1099", math.nan), ("other key", math.inf),
    ("all keys", -math.inf)])
def test_coverage_of_non_finite_logits(dtype, d, shift, keep, n_dec, what, val):
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    t, hq, hkv = 1100, 8, 2
    r, scale = hq // hkv, 1.0 / math.sqrt(d)
    gen = torch.Generator(device="cuda").manual_seed(5 + d)
    buf = torch.randn(t * hkv * d + 8, generator=gen, device="cuda").to(dt)
    K = buf[shift:shift + t * hkv * d].view(1, t, hkv, d)
    Q = torch.randn((1, 1, 2, hq, d), generator=gen, device="cuda").to(dt)
    dec = torch.randn((1, 1, hq, n_dec, d), generator=gen, device="cuda").to(dt)
    # the value meets a positive element of every query, so an infinite key's
    # logits have its sign
    dec[..., 0] = 1.0
    idx = torch.arange(1, 2 * keep, 2, device="cuda") if 2 * keep < t else torch.arange(t, device="cuda")
    idx = idx.to(torch.int32)[:keep, None].expand(keep, hkv).contiguous()[None]
    bad = torch.zeros((hkv, n_dec), dtype=torch.bool, device="cuda")
    if what == "query":                         # one query of query head 1, so of KV head 0
        dec[0, 0, 1, n_dec - 1, 5] = val
        bad[0, n_dec - 1] = True
    else:
        keys = {"kept key": [1], "other key": [2], "first 64 keys": range(64),
                "last 16 keys": range(1084, 1100), "keys 1024-1099": range(1024, 1100),
                "all keys": range(t)}[what]
        K[0, list(keys), 1, 0] = val
        bad[1] = True
    shape = M.make_shape(hq, hkv, d, 2, 0 if dtype == "bf16" else 1, [0, t], [keep])
    nb = M.mmshift_coverage_workspace_size(shape, n_dec)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    cov = torch.full((1, 1, hkv, n_dec), -1.0, device="cuda")
    M.check(M.mmshift_coverage(shape, K, Q, dec, n_dec, 0.0, idx, cov, ws, nb), "coverage")
    assert M.mmshift_poll_status(ws) == LB.MMSHIFT_OK
    for h in range(hkv):
        # float64 softmax; 5e-6 relative for the two-softmax form (float32 terms), the
        # parity contract's 2e-3 for masses where the group-mass form runs
        p = torch.softmax(scale * (dec[0, 0, h * r:(h + 1) * r].double() @ K[0, :, h].double().T), -1)
        ref = p[:, :, idx[0, :, h].long()].sum(-1).mean(0)
        got = cov[0, 0, h].double()
        assert bool((got[bad[h]] == 0.0).all()), got
        ok = ~bad[h]
        tol = 2e-3 if keep == t else 5e-6
        assert bool(((got - ref).abs()[ok] <= tol * ref[ok] + 1e-9).all()), (got, ref)
