"""KVSelector calls on a stream of their own: workspaces belong to that stream, so
work pending on the current one neither delays the zeroing of a status word (past
the kernels that report a bad index there) nor gets the workspace while the call
still runs."""
import pytest
import torch

import paper_2607_22586_gb300 as M
from paper_2607_22586_gb300.selector import KVSelector

pytestmark = pytest.mark.gpu

MS = 2_000_000   # clocks of about a millisecond


def _selector(t, hq=28, hkv=4, d=128, w=4):
    return KVSelector(hq, hkv, d, w, torch.bfloat16, [0, t], [t // 8], params=M.default_params(n_proxies=32,
                                                                                              n_groups=2))


@pytest.mark.parametrize("t", [2000, 20000])      # a zeroed workspace, a zeroed status word
@pytest.mark.parametrize("raw", [False, True])    # a torch stream, its handle
def test_coverage_beside_a_busy_current_stream(t, raw):
    gen = torch.Generator(device="cuda").manual_seed(t)
    sel = _selector(t)
    K, V = (torch.randn((1, t, 4, 128), generator=gen, device="cuda").bfloat16() for _ in range(2))
    Q = torch.randn((1, 1, 4, 28, 128), generator=gen, device="cuda").bfloat16()
    dec = torch.randn((1, 1, 28, 16, 128), generator=gen, device="cuda").bfloat16()
    sel(K, V, Q)
    ref = sel.coverage(K, Q, dec)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    bad = sel.out_idx.clone()
    bad[0, 0, 0] = t                               # past the prompt: reported
    torch.cuda.synchronize()
    stream = side.cuda_stream if raw else side
    for _ in range(3):
        torch.cuda._sleep(20 * MS)
        got = sel.coverage(K, Q, dec, stream=stream)
        torch.cuda._sleep(20 * MS)
        with pytest.raises(RuntimeError):
            sel.coverage(K, Q, dec, idx=bad, stream=stream)
        torch.cuda.synchronize()
        assert torch.equal(got, ref)


def test_statistics_keep_their_workspace():
    t = 20000
    gen = torch.Generator(device="cuda").manual_seed(2)
    sel = _selector(t)
    q = torch.randn((1, t, 28, 128), generator=gen, device="cuda").bfloat16()
    ref = sel.prefill_stats(q)
    side = torch.cuda.Stream()
    n = M.mmshift_prefill_stats_workspace_size(sel.shape)
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(5 * MS)
    got = sel.prefill_stats(q, stream=side)
    for _ in range(4000):                          # whoever gets its bytes next writes them
        torch.empty(n, dtype=torch.uint8, device="cuda").fill_(255)
    torch.cuda.synchronize()
    assert torch.equal(got, ref)
