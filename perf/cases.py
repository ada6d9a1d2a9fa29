"""The calls of the HSA hot path whose time is followed, over the sizes users run.

A case is one call, or one short chain of calls, of the library's public entry
points, as a program that serves a video diffusion transformer makes them.
Kinds:

  plan       once per sample and once per iteration: the partition of the
             tokens by their statistic, then one iteration's active set.
  attention  one layer's active attention: bf16 or fp32, head dimension 64 or
             128, the queries read by index or compact, the keys in one cache
             or (token reordering) in a cache prefix and the fresh baseline.
  sync       what moves a layer's rows: gather of the active hidden rows and
             the KV-cache scatter.
  rope       the same scatter with K rotated on its way, and Q's rotation.
  euler      the latent update with the velocity statistic, as in the first,
             full-budget iterations, or without it.
  iteration  a whole iteration of one layer: active set, gather, KV scatter,
             attention, cached Euler.

Token grids are (frames, rows, columns) of patches, tokens row-major.
"""
import math

import torch

import paper_2605_06892_gb300 as hsa

T = 40   # denoising iterations of every case
# Group splits: fraction of the tokens and step budget of each group.
PRESETS = {
    "three": ((0.25, 40), (0.25, 20), (0.5, 10)),
    "four": ((0.25, 40), (0.25, 20), (0.25, 10), (0.25, 5)),
}
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def listed():
    return [
        # A small fp32 layer (4x16x16 tokens, 4 heads x 64), one iteration with a
        # quarter of the tokens active: the smallest use, all launch latency.
        {"name": "iter_tiny_f32", "kind": "iteration", "F": 4, "Hh": 16, "Ww": 16, "H": 4,
         "D": 64, "C": 16, "dtype": "f32", "preset": "four", "iter": 1, "boxes": False},
        # An LTX-like layer (16x16x24 tokens, 32 heads x 64, 128-channel latent)
        # at an iteration with half of the tokens active: the ordinary step of a
        # compressed-latent model.
        {"name": "iter_ltx_half", "kind": "iteration", "F": 16, "Hh": 16, "Ww": 24, "H": 32,
         "D": 64, "C": 128, "dtype": "bf16", "preset": "four", "iter": 2, "boxes": False},
        # Token selection of that layer ...
        {"name": "plan_ltx", "kind": "plan", "N": 6144, "preset": "four", "iter": 1,
         "window": 100, "boxes": False},
        # ... of a 720p-like video (21x45x80 tokens) inside the caching window ...
        {"name": "plan_720p", "kind": "plan", "N": 75600, "preset": "four", "iter": 6,
         "window": 80, "boxes": False},
        # ... and of a long video, as many tokens as the workspace-free partition takes.
        {"name": "plan_long", "kind": "plan", "N": 524288, "preset": "three", "iter": 2,
         "window": 100, "boxes": False},
        # A Wan-1.3B-like layer (21x30x52 tokens, 12 heads x 128), half of the
        # queries, read by index: the ordinary attention call.
        {"name": "attn_wan13b_half", "kind": "attention", "F": 21, "Hh": 30, "Ww": 52, "H": 12,
         "D": 128, "dtype": "bf16", "preset": "three", "iter": 2, "boxes": False,
         "by_index": True, "prefix": False},
        # The same tokens in 24 heads x 64 after token reordering: compact
        # queries, keys in the cache prefix and the fresh baseline rows.
        {"name": "attn_prefix_24x64", "kind": "attention", "F": 21, "Hh": 30, "Ww": 52, "H": 24,
         "D": 64, "dtype": "bf16", "preset": "three", "iter": 2, "boxes": False,
         "by_index": False, "prefix": True},
        # A Wan-14B-like layer (40 heads x 128) of a 720p-like video with a
        # quarter of the tokens active: the largest call.
        {"name": "attn_720p_quarter", "kind": "attention", "F": 21, "Hh": 45, "Ww": 80, "H": 40,
         "D": 128, "dtype": "bf16", "preset": "four", "iter": 1, "boxes": False,
         "by_index": True, "prefix": False},
        # fp32 attention at the LTX-like layer's size, half of the queries: the
        # precise path, for validation runs and models kept in fp32.
        {"name": "attn_ltx_f32", "kind": "attention", "F": 16, "Hh": 16, "Ww": 24, "H": 32,
         "D": 64, "dtype": "f32", "preset": "four", "iter": 2, "boxes": False,
         "by_index": True, "prefix": False},
        # Row movement of a Wan-14B-like layer (hidden 5120) at 480p, the active
        # tokens clustered in boxes of the grid.
        {"name": "sync_wan14b_boxes", "kind": "sync", "F": 21, "Hh": 30, "Ww": 52, "H": 40,
         "D": 128, "dtype": "bf16", "preset": "three", "iter": 2, "boxes": True},
        # K and Q rotated at the Wan-1.3B-like layer.
        {"name": "rope_wan13b_half", "kind": "rope", "F": 21, "Hh": 30, "Ww": 52, "H": 12,
         "D": 128, "dtype": "bf16", "preset": "three", "iter": 2, "boxes": False},
        # A full-budget iteration's latent update with the velocity statistic,
        # 16 channels, a batch of long videos (1048576 tokens).
        {"name": "euler_stat_1m", "kind": "euler", "N": 1048576, "C": 16, "preset": "four",
         "iter": 0, "stat": True, "boxes": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi):
    """A (frames, rows, columns) grid of about lo..hi tokens, odd sides included."""
    n = _log(rng, lo, hi)
    f = rng.randint(1, max(1, min(25, n // 64)))
    side = max(8.0, n / f)
    h = max(4, int(round(math.sqrt(side) * rng.uniform(0.6, 1.0))))
    return {"F": f, "Hh": h, "Ww": max(4, int(round(side / h)))}


def _preset(rng):
    return {"preset": rng.choice(sorted(PRESETS)), "iter": rng.choice([0, 1, 2, 4, 7]),
            "boxes": rng.random() < 0.3}


def draw(rng):
    kind = rng.choice(["plan", "attention", "attention", "sync", "rope", "euler", "iteration"])
    c = {"kind": kind}
    c.update(_preset(rng))
    if kind == "plan":
        c.update(N=_log(rng, 1000, 1000000), window=rng.choice([100, 80]), boxes=False)
    elif kind == "attention":
        c.update(D=rng.choice([64, 128]), by_index=rng.random() < 0.6, prefix=rng.random() < 0.3,
                 dtype="f32" if rng.random() < 0.25 else "bf16")
        if c["dtype"] == "f32":
            c.update(_grid(rng, 512, 8192), H=rng.randint(2, 16))
        else:
            c.update(_grid(rng, 1024, 75600), H=rng.randint(4, 40))
    elif kind in ("sync", "rope"):
        c.update(_grid(rng, 1024, 75600), H=rng.randint(4, 40), D=rng.choice([64, 128]),
                 dtype="f32" if kind == "sync" and rng.random() < 0.2 else "bf16")
    elif kind == "euler":
        c.update(N=_log(rng, 1000, 4000000), C=rng.choice([16, 16, 48, 64, 128]),
                 stat=rng.random() < 0.5, boxes=False)
        c["N"] = min(c["N"], 128 * 2 ** 20 // c["C"])
    else:
        c.update(D=rng.choice([64, 128]), C=rng.choice([16, 48, 128]),
                 dtype=rng.choice(["bf16", "bf16", "f32"]))
        if c["dtype"] == "f32":
            c.update(_grid(rng, 256, 4096), H=rng.randint(2, 8))
        else:
            c.update(_grid(rng, 1024, 12288), H=rng.randint(4, 32))
    # No drawn case costs more than the largest listed one (a quarter of the
    # 720p-like tokens, 40 heads x 128).
    if "H" in c and "D" in c:
        most = 4.0 * 18900 * 75600 * 128 * 40
        while work(c)["flops"] > most:
            c["H"] = max(1, c["H"] // 2)
    return c


# ------------------------------------------------------------------ inputs

def _tokens(case):
    return case["N"] if "N" in case else case["F"] * case["Hh"] * case["Ww"]


def _split(case):
    """(budgets, counts) of the groups, the last one taking the remainder."""
    N, preset = _tokens(case), PRESETS[case["preset"]]
    counts = [int(N * f) for f, _ in preset]
    counts[-1] = N - sum(counts[:-1])
    return tuple(s for _, s in preset), tuple(counts)


def _n_active(case):
    budgets, counts = _split(case)
    margin = (100 - case.get("window", 100)) * T // 200
    i = case["iter"]
    full = i < margin or i > T - margin - 1
    return sum(n for s, n in zip(budgets, counts) if full or i % (T // s) == 0)


def _stat(case, g):
    """Per-token statistic: lognormal, raised inside boxes of the grid where the
    case's high-velocity regions are clustered."""
    N = _tokens(case)
    stat = torch.randn(N, generator=g, device="cuda").exp()
    if case["boxes"]:
        dims = (case["F"], case["Hh"], case["Ww"])
        field = torch.zeros(dims, device="cuda")
        for _ in range(10):
            u = torch.rand(6, generator=g, device="cuda").tolist()
            ext = [max(1, int(d * (0.15 + 0.3 * a))) for d, a in zip(dims, u)]
            org = [int((d - e) * a) for d, e, a in zip(dims, ext, u[3:])]
            field[org[0]:org[0] + ext[0], org[1]:org[1] + ext[1], org[2]:org[2] + ext[2]] = 1e3
        stat += field.reshape(-1)
    return stat


def _groups(case, stat):
    """Group of each token: ranked by the statistic, ties by the lower token
    first, the lowest ranks to the last group."""
    _, counts = _split(case)
    order = torch.sort(stat, stable=True).indices
    group = torch.empty(stat.numel(), dtype=torch.int32, device=stat.device)
    lo = 0
    for k in range(len(counts) - 1, -1, -1):
        group[order[lo:lo + counts[k]]] = k
        lo += counts[k]
    return group


def _active(case, group):
    """(idx, pos) of the case's iteration."""
    budgets, _ = _split(case)
    margin = (100 - case.get("window", 100)) * T // 200
    i = case["iter"]
    full = i < margin or i > T - margin - 1
    on = torch.tensor([full or i % (T // s) == 0 for s in budgets], device=group.device)
    flag = on[group.long()]
    idx = torch.nonzero(flag).reshape(-1).to(torch.int32)
    rank = torch.cumsum(flag.to(torch.int32), 0, dtype=torch.int32) - 1
    return idx, torch.where(flag, rank, torch.full_like(rank, -1))


def _inputs(case, seed):
    """Every input tensor of the case, on the GPU, from the seed alone."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    N, n = _tokens(case), _n_active(case)
    dt = DTYPES[case.get("dtype", "f32")]
    kind = case["kind"]

    def normal(*shape, dtype=dt):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).to(dtype)

    s = {"stat": _stat(case, g)}
    if kind == "plan":
        return s
    s["group"] = _groups(case, s["stat"])
    s["idx"], s["pos"] = _active(case, s["group"])
    if kind in ("sync", "iteration"):
        s["hidden"] = normal(N, case["H"] * case["D"])
    if kind != "euler":
        H, D = case["H"], case["D"]
        if kind == "attention" and case["prefix"]:
            s["base"] = min(N - 1, _split(case)[1][0])
        M = N - s.get("base", 0)
        s["k_cache"], s["v_cache"] = normal(M, H, D), normal(M, H, D)
        if kind == "attention":
            s["q"] = normal(N if case["by_index"] else n, H, D)
            if case["prefix"]:
                s["k_base"], s["v_base"] = normal(N - M, H, D), normal(N - M, H, D)
        else:
            s["k_fresh"], s["v_fresh"] = normal(n, H, D), normal(n, H, D)
            if kind != "sync":
                s["q"] = normal(n, H, D)
    if kind in ("euler", "iteration"):
        C = case["C"]
        s["x"] = normal(N, C, dtype=torch.float32)
        s["velocity"] = normal(N, C, dtype=torch.float32)
        s["fresh"] = normal(n, C, dtype=torch.float32)
        s["sum"] = torch.zeros(N, device="cuda")
    return s


def _step(case):
    """sigma_{i+1} - sigma_i of the linear schedule."""
    return -1.0 / T


def prepare(case, seed):
    s = _inputs(case, seed)
    N, n = _tokens(case), _n_active(case)
    kind = case["kind"]
    s["case"], s["n"] = case, n
    s["budgets"], s["counts"] = _split(case)

    def empty(*shape, dtype):
        return torch.empty(shape, dtype=dtype, device="cuda")

    if kind in ("plan", "iteration"):
        s["out_idx"] = torch.zeros(N, dtype=torch.int32, device="cuda")
        s["out_pos"] = empty(N, dtype=torch.int32)
    if kind == "plan":
        s["out_group"] = empty(N, dtype=torch.int32)
        s["workspace"] = empty(hsa.hsa_partition_workspace_bytes(N), dtype=torch.uint8)
    if kind in ("sync", "iteration"):
        s["rows"] = empty(n, s["hidden"].shape[1], dtype=s["hidden"].dtype)
    if kind in ("attention", "iteration"):
        H, D = case["H"], case["D"]
        s["out"] = empty(n, H, D, dtype=DTYPES[case["dtype"]])
        code = hsa.HSA_BF16 if case["dtype"] == "bf16" else hsa.HSA_F32
        size = hsa.hsa_active_attention_workspace_bytes(n, N, H, D, code)
        s["workspace"] = empty(size, dtype=torch.uint8) if size else None
    if kind == "rope":
        s["table"] = hsa.hsa_rope_table((case["F"], case["Hh"], case["Ww"]), case["D"]).cuda()
    return s


def run(s):
    case, n = s["case"], s["n"]
    kind = case["kind"]
    if kind == "plan":
        hsa.hsa_partition(s["stat"], T, s["budgets"], s["counts"], s["out_group"], s["workspace"])
        hsa.hsa_partition_active(s["out_group"], T, s["budgets"], case["iter"], s["out_idx"],
                                 s["out_pos"], window_pct=case["window"])
        return {"group": s["out_group"], "idx": s["out_idx"][:n], "pos": s["out_pos"]}
    if kind == "attention":
        q_idx = s["idx"] if case["by_index"] else None
        if case["prefix"]:
            hsa.hsa_active_attention_prefix(s["q"], q_idx, n, s["k_cache"], s["v_cache"],
                                            s["k_base"], s["v_base"], s["out"],
                                            workspace=s["workspace"])
        else:
            hsa.hsa_active_attention(s["q"], q_idx, n, s["k_cache"], s["v_cache"], s["out"],
                                     workspace=s["workspace"])
        return {"out": s["out"]}
    if kind == "sync":
        hsa.hsa_gather_active(s["hidden"], s["idx"], n, s["rows"])
        hsa.hsa_kv_sync_scatter(s["k_cache"], s["v_cache"], s["k_fresh"], s["v_fresh"], s["idx"],
                                n)
        return {"rows": s["rows"], "k_cache": s["k_cache"], "v_cache": s["v_cache"]}
    if kind == "rope":
        hsa.hsa_kv_sync_scatter_rope(s["k_cache"], s["v_cache"], s["k_fresh"], s["v_fresh"],
                                     s["idx"], n, s["table"])
        hsa.hsa_rope_rows(s["q"], s["idx"], n, s["table"])
        return {"k_cache": s["k_cache"], "v_cache": s["v_cache"], "q": s["q"]}
    if kind == "euler":
        if case["stat"]:
            hsa.hsa_cached_euler_l1rel(s["x"], s["velocity"], s["fresh"], s["pos"], _step(case),
                                       s["sum"], 0.25)
            return {"x": s["x"], "velocity": s["velocity"], "sum": s["sum"]}
        hsa.hsa_cached_euler(s["x"], s["velocity"], s["fresh"], s["pos"], _step(case))
        return {"x": s["x"], "velocity": s["velocity"]}
    hsa.hsa_partition_active(s["group"], T, s["budgets"], case["iter"], s["out_idx"],
                             s["out_pos"])
    hsa.hsa_gather_active(s["hidden"], s["out_idx"], n, s["rows"])
    hsa.hsa_kv_sync_scatter(s["k_cache"], s["v_cache"], s["k_fresh"], s["v_fresh"], s["out_idx"],
                            n)
    hsa.hsa_active_attention(s["q"], None, n, s["k_cache"], s["v_cache"], s["out"],
                             workspace=s["workspace"])
    hsa.hsa_cached_euler(s["x"], s["velocity"], s["fresh"], s["out_pos"], _step(case))
    return {"idx": s["out_idx"][:n], "pos": s["out_pos"], "rows": s["rows"],
            "k_cache": s["k_cache"], "v_cache": s["v_cache"], "out": s["out"], "x": s["x"],
            "velocity": s["velocity"]}


def work(case):
    N, n = _tokens(case), _n_active(case)
    kind = case["kind"]
    size = 2 if case.get("dtype") == "bf16" else 4
    row = case.get("H", 0) * case.get("D", 0) * size
    nbytes = flops = 0
    if kind == "plan":
        nbytes += 4 * N + 4 * N              # statistic read, groups written
    if kind in ("plan", "iteration"):
        nbytes += 4 * N + 4 * n              # pos and idx written
    if kind == "iteration":
        nbytes += 4 * N                      # groups read
    if kind in ("sync", "iteration"):
        nbytes += 2 * n * row                # hidden rows read and written
    if kind in ("sync", "rope", "iteration"):
        nbytes += 4 * n * row + 4 * n        # K and V rows read and written, idx
    if kind == "rope":
        nbytes += 2 * n * row + n * case["D"] * 4   # Q rows read and written, table rows
        flops += 2 * 3 * n * case["H"] * case["D"]
    if kind in ("attention", "iteration"):
        nbytes += 2 * N * row + 2 * n * row
        flops += 4 * n * N * case["H"] * case["D"]
    if kind in ("euler", "iteration"):
        nbytes += 4 * (3 * N + n) * case["C"] + 4 * N
        flops += 2 * N * case["C"]
        if case.get("stat"):
            nbytes += 4 * n * case["C"] + 8 * n     # old velocities and the running statistic
            flops += 4 * n * case["C"]
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------- the same in 64 bits

def _exact_attention(q, keys, values):
    """softmax(q k^T / sqrt(D)) v per head in fp64, the queries in blocks."""
    n, H, D = q.shape
    out = torch.empty((n, H, D), dtype=torch.float64, device=q.device)
    for h in range(H):
        k, v = keys[:, h].double(), values[:, h].double()
        for lo in range(0, n, 8192):
            p = torch.softmax(q[lo:lo + 8192, h].double() @ k.t() / math.sqrt(D), dim=1)
            out[lo:lo + 8192, h] = p @ v
    return out


def _exact_rope(x, case, idx):
    """Rows of x rotated by their tokens' angles: bands of frame, row and column
    pairs, the fp32 (cos, sin) table as a program holds it."""
    F, Hh, Ww, D = case["F"], case["Hh"], case["Ww"], case["D"]
    pairs, side = D // 2, D // 6
    bands = (pairs - 2 * side, side, side)
    tok = idx.long()
    where = (tok // (Hh * Ww), tok // Ww % Hh, tok % Ww)
    angle = torch.cat([w.double()[:, None] * 10000.0 ** (-torch.arange(
        p, dtype=torch.float64, device=x.device) / p) for w, p in zip(where, bands)], dim=1)
    c, s = (f(angle).float().double()[:, None, :] for f in (torch.cos, torch.sin))
    x0, x1 = x[..., 0::2].double(), x[..., 1::2].double()
    return torch.stack((x0 * c - x1 * s, x0 * s + x1 * c), dim=-1).reshape(x.shape)


def exact(case, seed):
    if work(case)["flops"] > 12e12:
        return None                       # over 20 seconds of fp64
    s = _inputs(case, seed)
    kind = case["kind"]
    out = {}
    if kind == "plan":
        out["group"] = _groups(case, s["stat"])
        out["idx"], out["pos"] = _active(case, out["group"])
        return out
    idx = s["idx"].long()
    if kind == "iteration":
        out["idx"], out["pos"] = s["idx"], s["pos"]
    if kind in ("sync", "iteration"):
        out["rows"] = s["hidden"][idx].double()
    if kind in ("sync", "rope", "iteration"):
        fresh = _exact_rope(s["k_fresh"], case, s["idx"]) if kind == "rope" else s["k_fresh"]
        out["k_cache"], out["v_cache"] = s["k_cache"].double(), s["v_cache"].double()
        out["k_cache"][idx], out["v_cache"][idx] = fresh.double(), s["v_fresh"].double()
    if kind == "rope":
        out["q"] = _exact_rope(s["q"], case, s["idx"])
    if kind == "attention":
        q = s["q"][idx] if case["by_index"] else s["q"]
        pair = [torch.cat((s[a], s[b])) if case["prefix"] else s[a]
                for a, b in (("k_cache", "k_base"), ("v_cache", "v_base"))]
        out["out"] = _exact_attention(q, *pair)
    if kind == "iteration":
        out["out"] = _exact_attention(s["q"], out["k_cache"], out["v_cache"])
    if kind in ("euler", "iteration"):
        old, new = s["velocity"].double(), s["velocity"].double()
        new[idx] = s["fresh"].double()
        step = torch.tensor(_step(case), dtype=torch.float32).double().item()
        out["x"] = s["x"].double() + new * step
        out["velocity"] = new
        if case.get("stat"):
            total = torch.zeros(new.shape[0], dtype=torch.float64, device=new.device)
            total[idx] = 0.25 * (new - old).abs().sum(1)[idx] / new.abs().sum(1)[idx]
            out["sum"] = total
    return out
