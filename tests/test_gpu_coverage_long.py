"""mmshift_coverage of long prompts. A row's softmax partials (four per 1,024 keys
on the tensor cores, one on the CUDA cores) are merged in runs of 64 first where
they exceed one run: just below and above one run, last runs of one partial, short
requests beside long ones, in the prompt's sums and in the kept rows' as well. The
kept rows of budgets above 16,384 are placed by their chunks' counts: one more
than that, several requests and layers, padding rows anywhere. The query heads of a
KV head are merged side by side, 8 to 128 of them. Reference and bounds as in the tests of the kept rows."""
import math

import pytest
import torch

from paper_2607_22586_gb300 import _lib as LB
from tests.test_gpu_coverage_kept import _inputs, _run

pytestmark = pytest.mark.gpu


def _check(lens, budgets, hq, hkv, d, L, n_dec, dtype):
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    K, Q, dec, idx = _inputs(lens, budgets, hq, hkv, d, L, n_dec, dt, 0, 5 + sum(lens))
    cov, status = _run(K, Q, dec, idx, lens, budgets, hq, hkv, d, L, n_dec, dt)
    assert status == LB.MMSHIFT_OK
    r, scale = hq // hkv, 1.0 / math.sqrt(d)
    for l in range(L):
        lo = off = 0
        for b, (t, c) in enumerate(zip(lens, budgets)):
            keep = min(c, t)
            for h in range(hkv):
                k = K[l, lo:lo + t, h].double()
                p = torch.softmax(scale * (dec[l, b, h * r:(h + 1) * r].double() @ k.T), -1)
                i = idx[l, off:off + keep, h].long()
                ref = p[:, :, i[i >= 0]].sum(-1).mean(0)
                err = (cov[l, b, h].double() - ref).abs()
                assert bool((err <= 5e-6 * ref + 1e-9).all()), (l, b, h, float((err / (ref + 1e-9)).max()))
            lo += t
            off += keep


@pytest.mark.parametrize("lens,budgets,hq,hkv,d,L,n_dec,dtype", [
    ((16384,), (900,), 28, 4, 128, 1, 32, "bf16"),              # one run: merged as it is
    ((16385,), (900,), 28, 4, 128, 2, 33, "bf16"),              # 68 partials
    ((32769, 300, 16384, 1), (2000, 30, 40, 1), 8, 2, 64, 1, 65, "bf16"),
    ((40000,), (17500,), 8, 1, 128, 1, 40, "bf16"),             # kept rows in two runs as well
    ((66000,), (500,), 2, 1, 64, 1, 9, "f32"),                  # CUDA cores: 65 partials
])
def test_coverage_of_long_prompts(lens, budgets, hq, hkv, d, L, n_dec, dtype):
    _check(lens, budgets, hq, hkv, d, L, n_dec, dtype)


@pytest.mark.parametrize("lens,budgets,hq,hkv,d,L,n_dec,dtype", [
    ((40000,), (16384,), 8, 2, 128, 1, 40, "bf16"),             # counted again by each CTA
    ((40000,), (16385,), 8, 2, 128, 1, 40, "bf16"),             # counts, a last chunk of one entry
    ((300, 50000, 1, 700), (77, 17000, 1, 256), 14, 2, 128, 2, 33, "bf16"),
    ((40000, 300), (16640, 257), 4, 1, 64, 1, 70, "f32"),
])
def test_coverage_of_large_budgets(lens, budgets, hq, hkv, d, L, n_dec, dtype):
    _check(lens, budgets, hq, hkv, d, L, n_dec, dtype)


@pytest.mark.parametrize("lens,budgets,hq,hkv,d,L,n_dec,dtype", [
    ((900, 30), (100, 3), 18, 2, 64, 1, 33, "bf16"),            # nine heads: 16 places
    ((700,), (50,), 32, 1, 128, 2, 5, "bf16"),
    ((700,), (50,), 33, 1, 64, 1, 9, "bf16"),                   # eight queries a CTA
    ((500, 1500), (20, 90), 128, 1, 64, 1, 33, "bf16"),
    ((600,), (40,), 136, 1, 64, 1, 4, "bf16"),                  # two rounds
])
def test_coverage_of_many_query_heads(lens, budgets, hq, hkv, d, L, n_dec, dtype):
    _check(lens, budgets, hq, hkv, d, L, n_dec, dtype)
