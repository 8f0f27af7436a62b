"""Short calls launch their kernels as programmatic dependents of one another,
longer ones do not. A stack of layers above the limit (1,024 units of 256 proxy
rows x 1,024 keys x KV head x layer) gives what its layers give in calls of their
own below it, to the bit; and short calls on two streams at once, each with its
own buffers, give what they give alone."""
import pytest
import torch

import paper_2607_22586_gb300 as M
from paper_2607_22586_gb300.selector import KVSelector

pytestmark = pytest.mark.gpu


def _inputs(L, B, t, hq, hkv, w, d, dt, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    K = torch.randn((L, B * t, hkv, d), generator=gen, device="cuda").to(dt)
    V = torch.randn((L, B * t, hkv, d), generator=gen, device="cuda").to(dt)
    Q = (2.0 * torch.randn((L, B, w, hq, d), generator=gen, device="cuda")).to(dt)
    return K, V, Q


def _selector(L, B, t, hq, hkv, w, d, dt, budget, **params):
    return KVSelector(hq, hkv, d, w, dt, [t * b for b in range(B + 1)], [budget] * B, n_layers=L,
                      params=M.default_params(**params))


@pytest.mark.parametrize("L,t,hq,hkv,d,dt,n,g,rope", [
    (4, 5000, 28, 4, 128, torch.bfloat16, 512, 32, 1e6),   # 300 units a layer, 1,200 in all
    (12, 9000, 16, 2, 64, torch.bfloat16, 128, 8, 0.0),    # two anchor kernels
    (130, 700, 28, 4, 128, torch.float32, 64, 4, 0.0),     # CUDA cores, votes of few groups
])
def test_layers_below_the_limit_equal_the_stack_above_it(L, t, hq, hkv, d, dt, n, g, rope):
    w, budget = 16, t // 8
    K, V, Q = _inputs(L, 1, t, hq, hkv, w, d, dt, 7 * L)
    units = hkv * -(-t // 1024) * -(-(-(-n // g) * hq // hkv * g + 16) // 256)
    assert units <= 1024 < units * L
    stack = _selector(L, 1, t, hq, hkv, w, d, dt, budget, n_proxies=n, n_groups=g, rope_theta=rope)
    ref = [x.clone() for x in stack(K, V, Q)]
    stack.poll()
    for l in range(L):
        one = _selector(1, 1, t, hq, hkv, w, d, dt, budget, n_proxies=n, n_groups=g, rope_theta=rope,
                        layer_id=l)
        got = one(K[l:l + 1], V[l:l + 1], Q[l:l + 1])
        one.poll()
        for a, b in zip(got, ref):
            assert torch.equal(a[0], b[l]), l


@pytest.mark.parametrize("dt,rope", [(torch.bfloat16, 1e6), (torch.float32, 0.0)])
def test_short_calls_on_two_streams(dt, rope):
    B, t, hq, hkv, w, d = 2, 1500, 28, 4, 8, 128
    calls = []
    for k in range(2):
        K, V, Q = _inputs(1, B, t, hq, hkv, w, d, dt, 40 + k)
        sel = _selector(1, B, t, hq, hkv, w, d, dt, 100 + k, n_proxies=32, n_groups=2, rope_theta=rope,
                        seed=k)
        ref = [x.clone() for x in sel(K, V, Q)]
        sel.poll()
        calls.append((sel, (K, V, Q), ref, torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _ in range(50):
        for sel, _, _, st in calls:
            with torch.cuda.stream(st):
                sel.out_idx.fill_(-7)
                for x in (sel.out_k, sel.out_v):
                    x.zero_()
        for sel, inp, _, st in calls:
            sel(*inp, stream=st)
        for sel, _, ref, st in calls:
            sel.poll(st)
            for a, b in zip((sel.out_idx, sel.out_k, sel.out_v), ref):
                assert torch.equal(a, b)
