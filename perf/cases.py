"""What is timed: calls of the TwinKV pass as a serving or evaluation program makes them.

Every case is one call of a public entry point of paper_2608_27128_gb300.twinkv on a KV
cache of L layers, H KV heads, N positions and head dimension d.  The program holds the
keys, the mask its eviction policy produced, a workspace and the output tensors; it keeps
them from call to call.

A case's fields:
  op      entry point: repair, dedup, redundancy, policy, select, noalloc, host
  L H N d cache shape;  dtype of the keys, "bf16" or "f32"
  keep    share of the positions the policy retains (the budget, for the policy)
  tau     similarity threshold
  all     repair and host: also return b_i(all) and its twin
  pyramid per-layer budgets shrink with depth (the same total)
  keys    "rope" (rotated per position, 15 % near copies), "outlier" (four large
          channels, 10 % near copies) or "plain" (N(0,1), 5 % near copies)
"""
import math

import torch

from paper_2608_27128_gb300 import twinkv as tk

WINDOW, N_SINK, N_RECENT = 32, 4, 64     # the paper's defaults (Sec. 3.2)


def _case(op, L, H, N, d, **kw):
    c = {"op": op, "L": L, "H": H, "N": N, "d": d, "dtype": "bf16", "keep": 0.5,
         "tau": 0.85, "all": False, "pyramid": False, "keys": "rope"}
    c.update(kw)
    return c


def listed():
    return [
        # The smallest call: one head of a short float32 cache, as in a unit test or a
        # notebook.  Launches and latency count.
        _case("repair", 1, 1, 512, 64, dtype="f32", keys="plain", name="repair_one_head_f32"),
        # A serving loop that repairs layer by layer: one layer's heads after a 4k prompt.
        _case("repair", 1, 8, 4096, 128, name="repair_one_layer_4k"),
        # Redundancy statistics (b_i over every key) of a few float32 layers, ragged length.
        _case("redundancy", 2, 8, 5003, 128, dtype="f32", name="redundancy_ragged_f32"),
        # The standalone policy on a ragged d = 64 cache.
        _case("policy", 16, 8, 3001, 64, keep=0.3, tau=0.9, keys="outlier",
              name="policy_llama_ragged"),
        # The standalone policy on a whole Qwen3-4B cache, budgets shrinking with depth.
        _case("policy", 36, 8, 8192, 128, pyramid=True, name="policy_qwen_8k_pyramid"),
        # The repair of a whole Llama-3.2-1B cache (d = 64), default outputs.
        _case("repair", 16, 8, 8192, 64, tau=0.9, keys="outlier", name="repair_llama_8k"),
        # The repair that keeps one of each twin pair, 30 % kept, half a Qwen3-4B cache.
        _case("dedup", 18, 8, 8192, 128, keep=0.3, name="dedup_qwen_half_8k"),
        # The headline workload: a whole Qwen3-4B cache with both audits returned.
        _case("repair", 36, 8, 16384, 128, all=True, name="repair_qwen_16k_all"),
        # One layer of a 128k context, default outputs.
        _case("repair", 1, 8, 131072, 128, keys="plain", name="repair_long_128k"),
        # The swap alone on scores that the program already has (a threshold sweep).
        _case("select", 36, 8, 16384, 128, name="select_qwen_16k"),
        # The same for one layer inside an engine that may not allocate.
        _case("noalloc", 1, 8, 8192, 128, name="select_noalloc_one_layer"),
        # A cache offloaded to page-locked host memory, a quarter of the Qwen3-4B layers.
        _case("host", 9, 8, 8192, 128, name="repair_host_8k"),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["repair", "repair", "repair", "dedup", "redundancy", "policy", "select",
                     "noalloc", "host"])
    d = rng.choice([64, 128])
    dtype = "f32" if rng.random() < 0.25 else "bf16"
    while True:
        L, H, N = rng.randint(1, 36), rng.choice([1, 2, 4, 8]), _spread(rng, 300, 131072)
        if rng.random() < 0.5:
            N = N // 256 * 256 or 256          # half of the lengths are whole tiles
        u = L * H
        if op == "noalloc" and u * N > tk.NOALLOC_MAX_POSITIONS:
            continue
        if op == "host" and u * N * d * 4 > 400e6:
            continue
        if u * N * d <= 36 * 8 * 16384 * 128 and u * N * N * d <= 36 * 8 * 16384 ** 2 * 128:
            break
    return _case(op, L, H, N, d, dtype=dtype, keep=rng.choice([0.3, 0.5, 0.7]),
                 tau=rng.choice([0.85, 0.9]), all=rng.random() < 0.4,
                 pyramid=L > 1 and rng.random() < 0.3,
                 keys=rng.choice(["rope", "outlier", "plain"]))


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _keys(case, g):
    """Keys [L, H, N, d] with near copies planted at random places, one unit at a time."""
    L, H, N, d = case["L"], case["H"], case["N"], case["d"]
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    out = torch.empty((L * H, N, d), dtype=dtype, device="cuda")
    share = {"rope": 0.15, "outlier": 0.10, "plain": 0.05}[case["keys"]]
    n = max(1, int(share * N))
    if case["keys"] == "rope":
        theta = 1.0e6 ** (-2.0 * torch.arange(d // 2, device="cuda", dtype=torch.float64) / d)
        angle = torch.arange(N, device="cuda", dtype=torch.float64)[:, None] * theta
        cos, sin = angle.cos().float(), angle.sin().float()
    for u in range(L * H):
        x = torch.randn((N, d), generator=g, device="cuda")
        if case["keys"] == "outlier":
            x[:, torch.randperm(d, generator=g, device="cuda")[:4]] *= 8.0
        if case["keys"] == "rope":
            a, b = x[:, :d // 2], x[:, d // 2:]
            x = torch.cat([a * cos - b * sin, a * sin + b * cos], dim=1)
        place = torch.randperm(N, generator=g, device="cuda")
        noise = torch.randn((n, d), generator=g, device="cuda")
        x[place[n:2 * n]] = x[place[:n]] + 0.02 * noise
        out[u] = x.to(dtype)
    return out.view(L, H, N, d)


def _budgets(case):
    """Retained positions of each unit (at least the protected ones)."""
    L, H, N = case["L"], case["H"], case["N"]
    mean = math.ceil(case["keep"] * N)
    low = min(N_SINK + N_RECENT, N)
    spread = min(0.5, (N - mean) / mean, (mean - low) / mean) if case["pyramid"] else 0.0
    spread = max(0.0, spread)
    per_layer = [mean * (1.0 + spread * (1.0 - 2.0 * l / max(1, L - 1))) for l in range(L)]
    return [min(N, max(low, int(k))) for k in per_layer for _ in range(H)]


def _mask(case, budgets, g):
    """A retained set of the budget's size per unit: heavy-tailed scores, the sink and the
    recent positions always kept."""
    L, H, N = case["L"], case["H"], case["N"]
    k = torch.tensor(budgets, device="cuda")
    mask = torch.zeros((L * H, N), dtype=torch.uint8, device="cuda")
    place = torch.arange(N, device="cuda")
    for u in range(L * H):
        score = torch.rand(N, generator=g, device="cuda").pow(-1.0 / 1.5)
        score[:N_SINK] = math.inf
        score[max(0, N - N_RECENT):] = math.inf
        order = torch.argsort(score, descending=True, stable=True)
        mask[u].scatter_(0, order, (place < k[u]).to(torch.uint8))
    return mask.view(L, H, N)


def _outputs(case, device, pin=False):
    L, H, N = case["L"], case["H"], case["N"]

    def new(shape, dtype):
        # swap entries past a unit's count stay as the program left them
        return torch.full(shape, -1 if dtype == torch.int32 else 0, dtype=dtype, device=device,
                          pin_memory=pin)

    out = {"mask": new((L, H, N), torch.uint8), "status": new((L * H,), torch.int32)}
    if case["op"] == "policy":
        out["count"] = new((L, H, N), torch.int32)
        return out
    out["swaps"] = new((L * H, N // 2, 2), torch.int32)
    out["nswaps"] = new((L * H,), torch.int32)
    if case["op"] in ("repair", "dedup", "host"):
        out["score_ret"] = new((L, H, N), torch.float64)
        out["twin_ret"] = new((L, H, N), torch.int32)
        if case["all"]:
            out["score_all"] = new((L, H, N), torch.float64)
            out["twin_all"] = new((L, H, N), torch.int32)
    return out


def _scores(case, g):
    """b_i(S0) as an audit leaves it: most keys well below tau, a share near 1."""
    shape = (case["L"], case["H"], case["N"])
    b = 0.35 + 0.08 * torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    twin = torch.rand(shape, generator=g, device="cuda") < 0.2
    near = 1.0 - 4e-4 * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)
    return torch.where(twin, near, b)


def prepare(case, seed):
    g = _generator(seed)
    op, dev = case["op"], torch.device("cuda", torch.cuda.current_device())
    budgets = _budgets(case)
    state = {"case": case}
    if op in ("select", "noalloc"):
        state["scores"] = _scores(case, g)
    else:
        state["keys"] = _keys(case, g)
    if op not in ("redundancy", "policy"):
        state["mask"] = _mask(case, budgets, g)
    state["budget"] = torch.tensor(budgets, dtype=torch.int32, device=dev)
    if op == "host":
        for name in ("keys", "mask", "budget"):
            state[name] = state[name].cpu().pin_memory()
        shape = tk.shape_of(state["keys"])
        state["arena"] = torch.zeros_like(tk.host_arena(shape))
        state["out"] = _outputs(case, "cpu", pin=True)
        return state
    if op == "redundancy":
        size = (case["L"], case["H"], case["N"])
        state["score"] = torch.empty(size, dtype=torch.float64, device=dev)
        state["twin"] = torch.empty(size, dtype=torch.int32, device=dev)
    else:
        state["out"] = _outputs(case, dev)
    if op == "select":
        shape = tk.Shape(case["L"], case["H"], case["N"], 64, tk.BF16)
        state["ws"] = tk.workspace(shape, tk.OP_REPAIR_SELECT, dev)
    elif op != "noalloc":
        number = {"repair": tk.OP_REPAIR, "dedup": tk.OP_REPAIR,
                  "redundancy": tk.OP_REDUNDANCY, "policy": tk.OP_POLICY}[op]
        state["ws"] = tk.workspace(tk.shape_of(state["keys"]), number, dev)
    return state


def run(state):
    case = state["case"]
    op, tau = case["op"], case["tau"]
    if op == "repair":
        return tk.twinkv_repair(state["keys"], state["mask"], state["budget"], tau,
                                want_all=case["all"], out=state["out"], ws=state["ws"])
    if op == "dedup":
        return tk.twinkv_repair_dedup(state["keys"], state["mask"], state["budget"], tau,
                                      want_all=case["all"], out=state["out"], ws=state["ws"])
    if op == "redundancy":
        return tk.twinkv_redundancy(state["keys"], WINDOW, state["score"], state["twin"],
                                    ws=state["ws"])
    if op == "policy":
        return tk.twinkv_policy(state["keys"], state["budget"], tau, out=state["out"],
                                ws=state["ws"])
    if op == "select":
        return tk.twinkv_repair_select(state["scores"], state["mask"], state["budget"], tau,
                                       out=state["out"], ws=state["ws"])
    if op == "noalloc":
        return tk.twinkv_repair_select_noalloc(state["scores"], state["mask"],
                                               state["budget"], tau, out=state["out"])
    return tk.twinkv_repair_host(state["keys"], state["mask"], state["budget"], tau,
                                 want_all=case["all"], out=state["out"], arena=state["arena"])


def work(case):
    """Each input read once, each output written once; the similarity matrix that the
    maxima or the counts run over, entry by entry (2 d operations each): N x N where every
    key counts, N x K where only the K retained ones do."""
    L, H, N, d = case["L"], case["H"], case["N"], case["d"]
    op, u = case["op"], case["L"] * case["H"]
    budgets = _budgets(case)
    key_bytes = u * N * d * (4 if case["dtype"] == "f32" else 2)
    if op == "redundancy":
        return {"bytes": key_bytes + u * N * 12, "flops": 2 * u * N * N * d}
    if op == "policy":
        return {"bytes": key_bytes + u * N * 5, "flops": 2 * u * N * N * d}
    if op in ("select", "noalloc"):
        return {"bytes": u * N * 10, "flops": u * N}
    cols = u * N if case["all"] else sum(budgets)
    out = 1 + 12 * (2 if case["all"] else 1)
    return {"bytes": key_bytes + u * N * (1 + out), "flops": 2 * N * d * cols}


def exact(case, seed):
    """b_i(S0) and b_i(all) in float64.  Positions, counts and masks are whole numbers."""
    op, N, d = case["op"], case["N"], case["d"]
    u = case["L"] * case["H"]
    if op in ("select", "noalloc", "policy") or 2.0 * u * N * N * d > 3e12:
        return None
    state = prepare(case, seed)
    keys = state["keys"].cuda().view(u, N, d)
    mask = state["mask"].cuda().view(u, N).bool() if "mask" in state else None
    best_all = torch.empty((u, N), dtype=torch.float64, device="cuda")
    best_ret = torch.empty_like(best_all)
    place = torch.arange(N, device="cuda")
    rows = max(1, min(N, (1 << 27) // N))
    for i in range(u):
        # the pass is defined on bf16 keys: float32 ones are rounded first
        k = keys[i].to(torch.bfloat16).double()
        norm = (k * k).sum(dim=1)
        for r in range(0, N, rows):
            sim = k[r:r + rows] @ k.T
            sim /= (norm[r:r + rows, None] * norm[None, :]).sqrt_()
            sim.masked_fill_((place[r:r + rows, None] - place[None, :]).abs() <= WINDOW, -1.0)
            best_all[i, r:r + rows] = sim.max(dim=1).values
            if mask is not None:
                sim.masked_fill_(~mask[i][None, :], -1.0)
                best_ret[i, r:r + rows] = sim.max(dim=1).values
    size = (case["L"], case["H"], N)
    if op == "redundancy":
        return best_all.view(size), None
    out = dict.fromkeys(state["out"])
    out["score_ret"] = best_ret.view(size)
    if case["all"]:
        out["score_all"] = best_all.view(size)
    return out
