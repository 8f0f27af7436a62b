"""Measured cases of the library: calls that a serving program makes after
prefill, through the public entry points, with inputs of the shape and spread
of this repository's synthetic workloads, drawn on the GPU.

A case names its kind:
  select    KVSelector.__call__: the whole selection over all layers of a call
            (optionally with a budget per layer and KV head, or with proxy
            statistics over the whole prompt taken first);
  mass      mmshift_proxy_mass with given proxies: steps 2-4 alone;
  hidden    mmshift_hidden_stats + mmshift_build_hidden_proxies: proxies from
            the prefill hidden states;
  coverage  KVSelector.coverage: the attention-mass coverage of a kept set.
``seq`` and ``budgets`` list the requests' prompt lengths and budgets.
"""
import math

import torch

import paper_2607_22586_gb300 as M
from paper_2607_22586_gb300.selector import KVSelector

_DT = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(name, kind, seq, budgets, hq=28, hkv=4, d=128, layers=1, window=32, dtype="bf16",
          n=512, g=32, mode="vote", head_budgets=False, prompt_stats=False, rope=False, n_dec=0,
          d_model=0):
    return {"name": name, "kind": kind, "seq": seq, "budgets": budgets, "hq": hq, "hkv": hkv,
            "d": d, "layers": layers, "window": window, "dtype": dtype, "n": n, "g": g,
            "mode": mode, "head_budgets": head_budgets, "prompt_stats": prompt_stats,
            "rope": rope, "n_dec": n_dec, "d_model": d_model}


def listed():
    return [
        # the smallest call: one layer of a small float32 model, launches and
        # latency (the tiny workload)
        _case("select_f32_1k", "select", "1024", "128", hq=4, hkv=1, d=64, window=16, dtype="f32"),
        # short ragged requests of a 72B-class model, one layer at a time as a
        # layer-by-layer prefill loop calls it, few proxies: latency
        _case("select_ragged_short", "select", "300,1000,77,2", "64,2000,16,1", hq=64, hkv=8,
              n=32, g=2),
        # one layer of a 7B-class model, ordinary prompt, paper hyper-parameters
        _case("select_layer_4k", "select", "4096", "512"),
        # the 28-layer 8K stack in one call, each layer with its own budget
        # (a pyramid around 1024), wider window
        _case("select_stack_8k_budgets", "select", "8192", "1536", layers=28, window=64,
              head_budgets=True),
        # the 28-layer 32K multi-image stack, paper hyper-parameters: the
        # largest ordinary call
        _case("select_stack_32k", "select", "32768", "2048", layers=28),
        # the same with as many proxies as window queries
        _case("select_stack_32k_few", "select", "32768", "2048", layers=28, n=32, g=2),
        # a slice of the 72B-class ragged batch (GQA 64/8, eight requests)
        _case("select_72b_ragged", "select", "2048,3000,4096,6000,8192,12000,16384,24576",
              "192,320,384,576,832,1216,1664,2432", hq=64, hkv=8, layers=10, n=32, g=2),
        # proxy statistics over all prompt queries, then the selection with them
        _case("select_prompt_stats", "select", "16001", "1600", layers=8, n=64, g=4,
              prompt_stats=True),
        # steps 2-4 alone on proxies a caller made, head_dim 64, ragged
        _case("mass_d64", "mass", "3000,1500", "256,256", hq=8, hkv=2, d=64),
        # steps 2-4 alone in float32, odd length
        _case("mass_f32_4k", "mass", "4001", "512", dtype="f32", n=128, g=8),
        # proxies from the prefill hidden states, projected by W_Q
        _case("hidden_16k", "hidden", "16384", "1024", layers=8, d_model=3584, rope=True),
        # quality metric: coverage of a kept set for 32 decode queries per layer
        _case("coverage_stack_32k", "coverage", "32768", "2048", layers=28, n_dec=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["select"] * 5 + ["mass"] * 2 + ["hidden", "coverage"])
    dtype = "f32" if kind in ("select", "mass") and rng.random() < 0.25 else "bf16"
    hq, hkv, d = rng.choice([(28, 4, 128), (64, 8, 128), (8, 2, 64), (32, 8, 128), (4, 1, 64),
                             (16, 16, 128)])
    total = _log_int(rng, 200, 4096 if dtype == "f32" else 32768)
    batch = rng.choice([1, 1, 1, 2, 3, 5, 8])
    cuts = sorted(rng.sample(range(1, total), batch - 1)) if batch > 1 else []
    lens = [b - a for a, b in zip([0] + cuts, cuts + [total])]
    frac = math.exp(rng.uniform(math.log(0.04), math.log(0.4)))
    budgets = [max(1, int(round(frac * t))) for t in lens]
    n, g = rng.choice([(32, 2), (32, 2), (64, 4), (128, 32), (128, 8), (512, 32), (512, 32)])
    # no more keys, and no more logits, than the 28-layer 32K stacks have
    most = min(28 * 32768 // total, int(28 * 32768 * 28 * 512 // (total * hq * n)))
    if dtype == "f32":
        most = min(most, int(2 * 4001 * 28 * 128 // (total * hq * n)))
        if most < 1:
            n, g, most = 32, 2, 1
    layers = _log_int(rng, 1, max(1, min(28, most)))
    if kind == "hidden":
        hq, hkv, d = rng.choice([(28, 4, 128), (16, 16, 128)])
        layers = min(layers, 8)
    return _case("", kind, ",".join(map(str, lens)), ",".join(map(str, budgets)), hq=hq, hkv=hkv,
                 d=d, layers=max(1, layers), window=rng.choice([8, 16, 32, 33, 64]), dtype=dtype,
                 n=n, g=g, mode="mass" if kind == "select" and rng.random() < 0.2 else "vote",
                 head_budgets=kind == "select" and rng.random() < 0.25,
                 prompt_stats=False, rope=rng.random() < 0.4,
                 n_dec=rng.choice([1, 8, 32, 33]) if kind == "coverage" else 0,
                 d_model=hq * d if kind == "hidden" else 0)


def _ints(text):
    return [int(x) for x in text.split(",")]


def _cu(lens):
    cu = [0]
    for t in lens:
        cu.append(cu[-1] + t)
    return cu


def _keys(case, gen, dt):
    """Keys [L, T, Hkv, d]: 95% visual tokens around per-head cluster centres
    (the cluster of a token shared by the heads), 1% of them scaled by 3, text
    tokens unit normal, four channels scaled by 8 (bf16 models)."""
    lens, hkv, d, L = _ints(case["seq"]), case["hkv"], case["d"], case["layers"]
    dev = "cuda"
    out = torch.empty((L, sum(lens), hkv, d), dtype=dt, device=dev)
    scale = torch.ones(d, device=dev)
    if dt == torch.bfloat16:
        scale[torch.randperm(d, generator=gen, device=dev)[:4]] = 8.0
    cu = _cu(lens)
    for l in range(L):
        for lo, hi in zip(cu, cu[1:]):
            t = hi - lo
            nv = int(0.95 * t)
            k = torch.randn((t, hkv, d), generator=gen, device=dev)
            nc = max(1, min(512, nv // 16))
            centres = torch.randn((nc, hkv, d), generator=gen, device=dev)
            pick = torch.randint(0, nc, (nv,), generator=gen, device=dev)
            k[:nv] = centres[pick] + 0.1 * k[:nv]
            crit = torch.rand((nv, 1, 1), generator=gen, device=dev) < 0.01
            k[:nv] *= torch.where(crit, 3.0, 1.0)
            out[l, lo:hi] = (k * scale).to(dt)
    return out


def _queries(case, K, count, gen, spread):
    """[L, B, count, Hq, d]: half the request's per-head key mean plus noise."""
    lens, hq, hkv = _ints(case["seq"]), case["hq"], case["hkv"]
    L, d = case["layers"], case["d"]
    q = spread * torch.randn((L, len(lens), count, hq, d), generator=gen, device="cuda")
    cu = _cu(lens)
    for l in range(L):
        for b, (lo, hi) in enumerate(zip(cu, cu[1:])):
            q[l, b] += 0.5 * K[l, lo:hi].float().mean(0).repeat_interleave(hq // hkv, 0)
    return q.to(K.dtype)


def _kept(case, gen):
    """A kept set in the output layout [L, R, Hkv]: ascending, the last token in."""
    L, hkv = case["layers"], case["hkv"]
    parts = []
    for t, c in zip(_ints(case["seq"]), _ints(case["budgets"])):
        keep = min(c, t)
        key = torch.rand((L, t, hkv), generator=gen, device="cuda")
        key[:, t - 1] = 2.0
        parts.append(key.topk(keep, dim=1).indices.sort(dim=1).values.to(torch.int32))
    return torch.cat(parts, dim=1).contiguous()


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    lens, budgets = _ints(case["seq"]), _ints(case["budgets"])
    L, hq, hkv, d, w = case["layers"], case["hq"], case["hkv"], case["d"], case["window"]
    dt, total, batch = _DT[case["dtype"]], sum(lens), len(lens)
    params = M.default_params(n_proxies=case["n"], n_groups=case["g"], seed=seed,
                              score_mode=1 if case["mode"] == "mass" else 0,
                              rope_theta=1e6 if case["rope"] else 0.0)
    s = {"case": case, "params": params}
    if case["kind"] == "hidden":
        dm = case["d_model"]
        mean = 0.5 * torch.randn(dm, generator=gen, device="cuda")
        mean[torch.randperm(dm, generator=gen, device="cuda")[:4]] = 20.0
        spread = torch.rand(dm, generator=gen, device="cuda") + 0.5
        s["H"] = torch.empty((L, total, dm), dtype=dt, device="cuda")
        for l in range(L):
            s["H"][l] = (mean + spread * torch.randn((total, dm), generator=gen, device="cuda")).to(dt)
        s["W"] = (torch.randn((L, hq * d, dm), generator=gen, device="cuda") / math.sqrt(dm)).to(dt)
        s["bias"] = (0.5 * torch.randn((L, hq * d), generator=gen, device="cuda")).to(dt)
        s["shape"] = M.make_shape(hq, hkv, d, w, 0, _cu(lens), budgets, n_layers=L,
                                  layer_stride_kv=total * hkv * d,
                                  layer_stride_q=batch * w * hq * d)
        s["sbytes"] = M.mmshift_hidden_stats_workspace_size(s["shape"], dm)
        s["pbytes"] = M.mmshift_hidden_proxies_workspace_size(s["shape"], dm, params)
        s["sws"] = torch.zeros(s["sbytes"], dtype=torch.uint8, device="cuda")
        s["pws"] = torch.zeros(s["pbytes"], dtype=torch.uint8, device="cuda")
        s["stats"] = torch.empty((L, batch, 2, dm), device="cuda")
        s["proxies"] = torch.empty((L, batch, hq, case["n"], d), dtype=dt, device="cuda")
        return s
    s["K"] = _keys(case, gen, dt)
    s["Q"] = _queries(case, s["K"], w, gen, 1.0)
    if case["kind"] == "mass":
        s["proxies"] = (8.0 * torch.randn((L, batch, hq, case["n"], d), generator=gen,
                                          device="cuda")).to(dt)
        s["shape"] = M.make_shape(hq, hkv, d, w, 0 if dt == torch.bfloat16 else 1, _cu(lens),
                                  budgets, n_layers=L, layer_stride_kv=total * hkv * d,
                                  layer_stride_q=batch * w * hq * d)
        s["bytes"] = M.mmshift_workspace_size(s["shape"], params)
        s["ws"] = torch.zeros(s["bytes"], dtype=torch.uint8, device="cuda")
        s["group_mass"] = torch.empty((L, hkv, case["g"], total), device="cuda")
        s["anchor"] = torch.empty((L, hkv, total), device="cuda")
        s["mass"] = torch.empty((L, hkv, total), device="cuda")
        return s
    s["sel"] = KVSelector(hq, hkv, d, w, dt, _cu(lens), budgets, n_layers=L, params=params)
    if case["kind"] == "coverage":
        dec = _queries(case, s["K"], case["n_dec"], gen, 1.5)
        s["dec"] = dec.permute(0, 1, 3, 2, 4).contiguous()
        s["idx"] = _kept(case, gen)
        return s
    s["V"] = torch.randn((L, total, hkv, d), generator=gen, device="cuda", dtype=dt)
    if case["head_budgets"]:
        # from the capacity at the first layer down to a third of it at the last
        f = torch.linspace(1.0, 1.0 / 3.0, L, device="cuda")[:, None, None]
        cap = torch.tensor(budgets, device="cuda")[None, :, None]
        s["hb"] = (f * cap).round().clamp(min=1).to(torch.int32).expand(L, batch, hkv).contiguous()
    if case["prompt_stats"]:
        s["Qfull"] = torch.empty((L, total, hq, d), dtype=dt, device="cuda")
        for l in range(L):
            off = torch.randn((hq, d), generator=gen, device="cuda")
            s["Qfull"][l] = (off + torch.randn((total, hq, d), generator=gen, device="cuda")).to(dt)
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "hidden":
        M.check(M.mmshift_hidden_stats(s["shape"], case["d_model"], s["H"], 0, s["stats"], s["sws"],
                                       s["sbytes"], torch.cuda.current_stream()), "hidden_stats")
        M.check(M.mmshift_build_hidden_proxies(s["shape"], case["d_model"], s["stats"], s["W"], 0,
                                               s["bias"], None, s["params"], s["proxies"], s["pws"],
                                               s["pbytes"], torch.cuda.current_stream()),
                "build_hidden_proxies")
        return {"stats": s["stats"], "proxies": s["proxies"]}
    if case["kind"] == "mass":
        M.check(M.mmshift_proxy_mass(s["shape"], s["K"], s["Q"], s["proxies"], s["params"],
                                     s["group_mass"], s["anchor"], s["mass"], s["ws"], s["bytes"],
                                     torch.cuda.current_stream()), "proxy_mass")
        return {"group_mass": s["group_mass"], "anchor": s["anchor"], "mass": s["mass"]}
    sel = s["sel"]
    if case["kind"] == "coverage":
        return {"coverage": sel.coverage(s["K"], s["Q"], s["dec"], idx=s["idx"])}
    if case["prompt_stats"]:
        stats = sel.prefill_stats(s["Qfull"])
        idx, k, v = sel(s["K"], s["V"], s["Q"], stats=stats)
        return {"stats": stats, "idx": idx, "k": k, "v": v}
    idx, k, v = sel(s["K"], s["V"], s["Q"], head_budgets=s.get("hb"))
    out = {"idx": idx, "k": k, "v": v}
    if case["head_budgets"]:
        out["count"] = sel.out_count
    return out


def work(case):
    """K (or the prompt's queries or hidden states) read once, kept rows read
    and written once, the logits formed once."""
    lens, budgets = _ints(case["seq"]), _ints(case["budgets"])
    L, hq, hkv, d, w = case["layers"], case["hq"], case["hkv"], case["d"], case["window"]
    es = 2 if case["dtype"] == "bf16" else 4
    total, batch = sum(lens), len(lens)
    kept = sum(min(c, t) for c, t in zip(budgets, lens))
    k_bytes = L * total * hkv * d * es
    q_bytes = L * batch * w * hq * d * es
    if case["kind"] == "hidden":
        dm = case["d_model"]
        return {"bytes": L * (total * dm + hq * d * (dm + 1) + batch * hq * case["n"] * d) * es
                + L * batch * 2 * dm * 4,
                "flops": 2.0 * L * batch * case["n"] * dm * hq * d + 3.0 * L * total * dm}
    if case["kind"] == "coverage":
        return {"bytes": k_bytes + L * batch * hq * case["n_dec"] * d * es + L * kept * hkv * 4
                + L * batch * hkv * case["n_dec"] * 4,
                "flops": 2.0 * d * L * total * hq * case["n_dec"]}
    flops = 2.0 * d * L * total * hq * (case["n"] + 1)
    if case["kind"] == "mass":
        return {"bytes": k_bytes + L * batch * hq * (case["n"] + 1) * d * es
                + L * hkv * (case["g"] + 2) * total * 4, "flops": flops}
    out = L * kept * hkv * (4 * d * es + 4)
    if case["prompt_stats"]:
        q_bytes += L * total * hq * d * es + L * batch * 2 * hq * d * 4
    return {"bytes": k_bytes + q_bytes + out, "flops": flops}


def tolerance(case):
    if case["kind"] == "mass":
        # measured against float64: 1.4e-6; single masses carry the rounding of
        # a float32 log2 normaliser near 2^7, 1e-5
        return {"rel": 6e-6, "max": 1e-4}
    if case["kind"] == "coverage":
        # measured against float64: 1.3e-6
        return {"rel": 6e-6, "max": 1e-4}
    if case["kind"] == "hidden":
        # a proxy whose float32 value lies near a bf16 rounding boundary moves
        # by one unit of 2^-8; the statistics are float32 sums
        return {"rel": 5e-4, "max": 1.6e-2}
    # a kept set is a set of whole numbers, and the cache rows are copies
    return "exact"


def exact(case, seed):
    kind, L = case["kind"], case["layers"]
    lens, hkv, d = _ints(case["seq"]), case["hkv"], case["d"]
    cu, r = _cu(lens), case["hq"] // case["hkv"]

    def stats64(x):
        """[L, T, columns] -> [L, B, 2, columns]: mean and unbiased std."""
        out = torch.zeros((L, len(lens), 2, x.shape[-1]), dtype=torch.float64, device="cuda")
        for l in range(L):
            for b, (lo, hi) in enumerate(zip(cu, cu[1:])):
                y = x[l, lo:hi].double()
                out[l, b, 0] = y.mean(0)
                if hi - lo > 1:
                    out[l, b, 1] = y.std(0, unbiased=True)
        return out

    if kind == "hidden":
        s = prepare(case, seed)
        return {"stats": stats64(s["H"]), "proxies": None}
    if kind == "select":
        if not case["prompt_stats"]:
            return None
        s = prepare(case, seed)
        return {"stats": stats64(s["Qfull"].flatten(2)), "idx": None, "k": None, "v": None}
    n = case["n"] if kind == "mass" else case["n_dec"]
    if 2.0 * d * L * sum(lens) * case["hq"] * (n + 1) > 1e12:
        return None
    s = prepare(case, seed)
    scale = 1.0 / math.sqrt(d)
    budgets = _ints(case["budgets"])
    if kind == "coverage":
        cov = torch.empty((L, len(lens), hkv, n), dtype=torch.float64, device="cuda")
        for l in range(L):
            off = 0
            for b, (lo, hi) in enumerate(zip(cu, cu[1:])):
                keep = min(budgets[b], hi - lo)
                for h in range(hkv):
                    k = s["K"][l, lo:hi, h].double()
                    q = s["dec"][l, b, h * r:(h + 1) * r].double()
                    p = torch.softmax(scale * (q @ k.T), dim=-1)
                    t = s["idx"][l, off:off + keep, h].long()
                    cov[l, b, h] = p[:, :, t].sum(-1).mean(0)
                off += keep
        return {"coverage": cov}
    g = case["g"]
    gm = torch.empty((L, hkv, g, cu[-1]), dtype=torch.float64, device="cuda")
    an = torch.empty((L, hkv, cu[-1]), dtype=torch.float64, device="cuda")
    for l in range(L):
        for b, (lo, hi) in enumerate(zip(cu, cu[1:])):
            for h in range(hkv):
                k = s["K"][l, lo:hi, h].double()
                q = s["proxies"][l, b, h * r:(h + 1) * r].double()
                for i in range(g):
                    part = q[:, i * (n // g):(i + 1) * (n // g)]
                    gm[l, h, i, lo:hi] = torch.softmax(scale * (part @ k.T), dim=-1).sum((0, 1))
                a = s["Q"][l, b, -1, h * r:(h + 1) * r].double()
                an[l, h, lo:hi] = torch.softmax(scale * (a @ k.T), dim=-1).mean(0)
    return {"group_mass": gm, "anchor": an, "mass": gm.sum(2)}
