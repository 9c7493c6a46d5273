"""Performance cases: the work a user of this library has it do, through the
public entry points of paper_2609_32663_gb300.dkv.

A case is a dict of plain values. Its "kind" is the call a program makes:

  step            one decode step of a whole model: dkv_decode_attn on every
                  layer, captured once as a CUDA graph and replayed, as a
                  serving loop does
  layers          the same calls made eagerly, layer by layer, as a program
                  does whose own model code runs between them
  noalloc         dkv_decode_attn_noalloc, layer by layer: the entry point for
                  hosts that own all device memory
  multi           dkv_decode_multi, layer by layer: several queries per
                  sequence over one compressed context
  prune           dkv_map_pattern and dkv_compact into the caller's buffers: the
                  one-time step after prefill
  prune_inplace   dkv_map_pattern_inplace and dkv_compact_inplace, inside the
                  dense cache
  export          dkv_topk_mask: learned probabilities to the binary pattern

Geometries, retention rates and lengths are those of the package's workloads
(inputs.WORKLOADS); `draw` spreads the same kinds over their ranges.
"""
import math

import numpy as np
import torch

from paper_2609_32663_gb300 import dkv, inputs

HEAD = 128       # head_dim of the library
RESERVE = 256    # rows kept free after each slab for generated tokens
DEV = "cuda"


def _case(name, kind, L, H, Hkv, T, B, D, rate, pattern="profile", ragged=0, outliers=0.0, queries=1):
    """ragged: shortest context when the sequences' lengths are uniform in [ragged, T]; 0: every context is T."""
    return {"name": name, "kind": kind, "L": L, "H": H, "Hkv": Hkv, "T": T, "B": B, "D": D, "rate": rate,
            "pattern": pattern, "ragged": ragged, "outliers": outliers, "queries": queries}


def listed():
    return [
        # The smallest call: one layer of a 4K context, called on its own. Launch latency and host work.
        _case("layer-4k", "layers", 1, 32, 8, 4096, 1, 32, 0.35, pattern="bernoulli"),
        # A decode step of the whole model at an ordinary context: 50 MB a layer, short launches back to back.
        _case("step-llama-32k", "step", 32, 32, 8, 32768, 1, 64, 0.35),
        # The headline step: the whole model at 128K, outlier keys as real caches have them.
        _case("step-llama-128k", "step", 32, 32, 8, 131072, 1, 128, 0.346, outliers=0.01),
        # The other head shape in use (group of 7), a small batch.
        _case("step-qwen-64k-b4", "step", 28, 28, 4, 65536, 4, 64, 0.35),
        # Batched serving: sixteen sequences of independent, odd lengths; ragged slabs.
        _case("layers-b16-ragged", "layers", 4, 32, 8, 65536, 16, 64, 0.25, ragged=8192),
        # A host that owns the device pool: the allocation-free entry point.
        _case("noalloc-32k", "noalloc", 4, 32, 8, 32768, 1, 64, 0.35),
        # Shared-context reuse: a few queries at a time (16 columns a KV head) ...
        _case("multi-q4-128k", "multi", 4, 32, 8, 131072, 1, 128, 0.346, outliers=0.01, queries=4),
        # ... a full batch of them (64 columns) ...
        _case("multi-q16-128k", "multi", 4, 32, 8, 131072, 1, 128, 0.346, outliers=0.01, queries=16),
        # ... and the other head shape, 28 columns, a small batch of contexts.
        _case("multi-q4-qwen-64k-b4", "multi", 4, 28, 4, 65536, 4, 64, 0.35, queries=4),
        # After prefill: map the pattern and pack the whole model's cache.
        _case("prune-llama-32k", "prune", 32, 32, 8, 32768, 1, 64, 0.35),
        # The same without a second cache, a short context.
        _case("prune-inplace-16k", "prune_inplace", 32, 32, 8, 16384, 1, 32, 0.35),
        # The export of a model's pattern (32 layers, 32 heads, 128 bins).
        _case("export-llama", "export", 32, 32, 8, 131072, 1, 128, 0.346),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "layers", "layers", "noalloc", "multi", "multi", "multi", "prune",
                       "prune_inplace", "export"])
    H, Hkv = rng.choice([(32, 8), (32, 8), (28, 4), (16, 16), (16, 8), (12, 4), (24, 4), (32, 4), (20, 4)])
    G = H // Hkv
    if kind == "export":
        D = _log_int(rng, 32, 2048)
        L = _log_int(rng, 4, 80)
        return {k: v for k, v in _case("", kind, L, H, Hkv, 131072, 1, D, round(rng.uniform(0.2, 0.5), 3)).items()
                if k != "name"}
    T = _log_int(rng, 2048, 131072)
    B = rng.choice([1, 1, 1, 2, 3, 4, 7, 16])
    rate = round(rng.uniform(0.2, 0.5), 3)
    D = min(rng.choice([32, 64, 128, 253]), T - 1152)
    most = {"step": 32, "layers": 4, "noalloc": 4, "multi": 4, "prune": 32, "prune_inplace": 32}[kind]
    L = _log_int(rng, 1, most)
    # At most about 3 GB of dense rows for the one-time kinds and of packed rows for a decode step.
    per_layer = B * Hkv * T * 512 * (1.0 if kind.startswith("prune") else rate)
    while L > 1 and L * per_layer > 3e9:
        L -= 1
    while B > 1 and L * per_layer > 3e9:
        B -= 1
        per_layer = B * Hkv * T * 512
    ragged = max(1500, T // 8) if B > 1 and rng.random() < 0.6 else 0
    queries = 1
    if kind == "multi":
        queries = min(64 // G, rng.choice([1, 2, 3, 4, 5, 8, 11, 16, 64]))
    c = _case("", kind, L, H, Hkv, T, B, D, rate, pattern=rng.choice(["profile", "profile", "bernoulli"]),
              ragged=ragged, outliers=rng.choice([0.0, 0.01]), queries=queries)
    c.pop("name")
    return c


# ------------------------------------------------------------------ inputs
def _context(case):
    """Context lengths: like the pattern below, a property of the case."""
    if not case["ragged"]:
        return np.full(case["B"], case["T"], np.int32)
    rng = np.random.default_rng([case["T"], case["B"], 11])
    return rng.integers(case["ragged"], case["T"] + 1, size=case["B"]).astype(np.int32)


def _bin_width(case):
    return max(1, -(-(case["T"] - inputs.SINK - inputs.RECENT) // case["D"]))


def _pattern(case):
    """The model's learned pattern: static, so the same for every seed; keys, values and queries are not."""
    wl = inputs.Workload("case", L=case["L"], H=case["H"], Hkv=case["Hkv"], T=case["T"], B=case["B"], D=case["D"],
                         W=_bin_width(case), pattern=case["pattern"], rate=case["rate"],
                         seed=case["T"] + case["D"])
    return inputs.make_pattern(wl)


def _shape(case):
    return dkv.Shape(L=case["L"], H=case["H"], H_kv=case["Hkv"], D=case["D"], bin_width=_bin_width(case))


def _slab_lengths(case, M, ctx):
    """Kept positions of every slab [L][B][Hkv], by the definition of the map."""
    L, H, Hkv, W = case["L"], case["H"], case["Hkv"], _bin_width(case)
    U = M.reshape(L, Hkv, H // Hkv, -1).max(axis=2)
    out = np.zeros((L, len(ctx), Hkv), np.int64)
    for b, Tc in enumerate(int(x) for x in ctx):
        p = np.arange(Tc)
        edge = (p < inputs.SINK) | (p >= Tc - inputs.RECENT)
        d = (Tc - inputs.RECENT - 1 - p[~edge]) // W
        per_bin = np.bincount(d, minlength=U.shape[2])[:U.shape[2]] if d.size else np.zeros(U.shape[2], np.int64)
        out[:, b, :] = edge.sum() + (U * per_bin).sum(axis=2)
    return out


def _layout(case):
    M, ctx = _pattern(case), _context(case)
    ln = _slab_lengths(case, M, ctx)
    off = np.zeros(ln.size + 1, np.int64)
    np.cumsum(ln.reshape(-1) + RESERVE, out=off[1:])
    return M, ctx, ln, off


def _normal(gen, *shape):
    return torch.randn(shape, generator=gen, device=DEV, dtype=torch.bfloat16)


def _rows(gen, n, outliers):
    """n cache rows of keys and of values; a share of the key rows is 8 times as large."""
    K, V = _normal(gen, n, HEAD), _normal(gen, n, HEAD)
    if outliers:
        K *= (1 + 7 * (torch.rand(n, 1, generator=gen, device=DEV) < outliers)).to(torch.bfloat16)
    return K, V


def _decode_tensors(case, seed, rows):
    """Packed caches, the step's queries, keys and values, and how many tokens each sequence has generated."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1000 * seed + 17)
    L, B, H, Hkv, Q = case["L"], case["B"], case["H"], case["Hkv"], case["queries"]
    Kc, Vc = _rows(gen, rows, case["outliers"])
    q = _normal(gen, L, B, Q, H, HEAD) if case["kind"] == "multi" else _normal(gen, L, B, H, HEAD)
    k_new, v_new = _normal(gen, L, B, Hkv, HEAD), _normal(gen, L, B, Hkv, HEAD)
    napp = torch.randint(0, RESERVE - 1, (B,), generator=gen, device=DEV, dtype=torch.int32)
    return Kc, Vc, q, k_new, v_new, napp


def _probabilities(case, seed):
    """Learned retention probabilities [L][H][D]: a near/far mix per head, noise, a logistic."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1000 * seed + 13)
    L, H, D = case["L"], case["H"], case["D"]
    w = torch.rand(L, H, 1, generator=gen, device=DEV)
    x = torch.linspace(0, 1, D, device=DEV)
    z = 6 * (w * (1 - x) + (1 - w) * x - 0.5) + torch.randn(L, H, D, generator=gen, device=DEV)
    return torch.sigmoid(z)


def prepare(case, seed):
    kind, L = case["kind"], case["L"]
    s = {"kind": kind, "L": L, "queries": case["queries"]}
    if kind == "export":
        s["P"] = _probabilities(case, seed)
        s["K"] = dkv.dkv_budget(case["rate"], L, case["H"], case["D"])
        s["M"] = torch.zeros(s["P"].shape, dtype=torch.uint8, device=DEV)
        s["work"] = torch.empty(dkv.dkv_topk_workspace_bytes(), dtype=torch.uint8, device=DEV)
        return s
    shape = _shape(case)
    M, ctx, ln, off = _layout(case)
    if kind.startswith("prune"):
        gen = torch.Generator(device=DEV)
        gen.manual_seed(1000 * seed + 17)
        stride = case["T"] + (RESERVE if kind == "prune_inplace" else 0)
        K, V = _rows(gen, L * case["B"] * case["Hkv"] * stride, case["outliers"])
        s |= {"M": M, "ctx": ctx, "shape": shape, "stride": stride, "K": K, "V": V, "plan": None}
        if kind == "prune":
            s["Kc"], s["Vc"] = (torch.zeros(int(off[-1]), HEAD, dtype=torch.bfloat16, device=DEV) for _ in range(2))
        return s
    Kc, Vc, q, k_new, v_new, napp = _decode_tensors(case, seed, int(off[-1]))
    s |= {"Kc": Kc, "Vc": Vc, "q": q, "k": k_new, "v": v_new, "napp": napp, "shape": shape, "B": case["B"],
          "out": torch.zeros(q.shape, dtype=torch.float32, device=DEV)}
    if kind == "noalloc":
        ioff = np.zeros(ln.size + 1, np.int64)
        np.cumsum(ln.reshape(-1), out=ioff[1:])
        s["len"] = torch.from_numpy(ln.reshape(-1).astype(np.int32)).to(DEV)
        s["off"], s["ioff"] = torch.from_numpy(off).to(DEV), torch.from_numpy(ioff).to(DEV)
        s["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        return s
    s["plan"] = dkv.dkv_map_pattern(M, ctx, shape, reserve_rows=RESERVE)
    if kind == "step":
        _layers(s)  # first calls outside the capture
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _layers(s)
    return s


def _layers(s):
    for l in range(s["L"]):
        dkv.dkv_decode_attn(s["plan"], l, s["q"][l], s["k"][l], s["v"][l], s["napp"], s["Kc"], s["Vc"], s["out"][l])


def run(state):
    s, kind = state, state["kind"]
    if kind == "step":
        s["graph"].replay()
    elif kind == "layers":
        _layers(s)
    elif kind == "noalloc":
        for l in range(s["L"]):
            dkv.dkv_decode_attn_noalloc(s["shape"], s["B"], l, RESERVE, s["len"], s["off"], s["ioff"], s["q"][l],
                                        s["k"][l], s["v"][l], s["napp"], s["Kc"], s["Vc"], s["out"][l],
                                        status=s["status"])
    elif kind == "multi":
        for l in range(s["L"]):
            dkv.dkv_decode_multi(s["plan"], l, s["q"][l], s["queries"], s["napp"], s["Kc"], s["Vc"], s["out"][l])
        return {"out": s["out"]}
    elif kind == "prune":
        s["plan"] = dkv.dkv_map_pattern(s["M"], s["ctx"], s["shape"], reserve_rows=RESERVE)
        dkv.dkv_compact(s["plan"], s["K"], s["V"], s["Kc"], s["Vc"], T_stride=s["stride"])
        return {"Kc": s["Kc"], "Vc": s["Vc"]}
    elif kind == "prune_inplace":
        s["plan"] = dkv.dkv_map_pattern_inplace(s["M"], s["ctx"], s["shape"], s["stride"], reserve_rows=RESERVE)
        dkv.dkv_compact_inplace(s["plan"], s["K"], s["V"])
        return {"Kc": s["K"], "Vc": s["V"]}
    elif kind == "export":
        dkv.dkv_topk_mask(s["P"], s["K"], s["M"], s["work"])
        return s["M"]
    # A decode step's results: the attention outputs, and the caches with this step's rows appended.
    return {"out": s["out"], "Kc": s["Kc"], "Vc": s["Vc"]}


def work(case):
    """K and V rows read once (and written once when they move), queries, new rows and outputs."""
    L, B, H, Hkv, Q = case["L"], case["B"], case["H"], case["Hkv"], case["queries"]
    if case["kind"] == "export":
        return {"bytes": 5 * L * H * case["D"], "flops": 0}
    kept = int(_slab_lengths(case, _pattern(case), _context(case)).sum())
    if case["kind"].startswith("prune"):
        return {"bytes": 2 * kept * 512, "flops": 0}
    rows = kept + L * B * Hkv * (RESERVE // 2)  # half the reserve generated, on average
    new = 0 if case["kind"] == "multi" else L * B * Hkv * 2 * 512
    return {"bytes": rows * 512 + new + L * B * Q * H * (256 + 512), "flops": rows * Q * (H // Hkv) * 4 * HEAD}


def exact(case, seed):
    kind = case["kind"]
    if kind.startswith("prune"):
        return None  # a copy of bytes
    if kind == "export":
        P = _probabilities(case, seed).reshape(-1).cpu().numpy().astype(np.float64)
        keep = int(math.floor(case["rate"] * P.size + 0.5))
        M = np.zeros(P.size, np.uint8)
        M[np.argsort(-P, kind="stable")[:keep]] = 1
        return torch.from_numpy(M.reshape(case["L"], case["H"], case["D"]))
    _, _, ln, off = _layout(case)
    Kc, Vc, q, k_new, v_new, napp = _decode_tensors(case, seed, int(off[-1]))
    L, B, H, Hkv, Q = case["L"], case["B"], case["H"], case["Hkv"], case["queries"]
    G, napp = H // Hkv, napp.tolist()
    out = torch.zeros(q.shape, dtype=torch.float64, device=DEV)
    for l in range(L):
        for b in range(B):
            for g in range(Hkv):
                h = (l * B + b) * Hkv + g
                r0, n = int(off[h]), int(ln[l, b, g]) + napp[b]
                K, V = Kc[r0:r0 + n].double(), Vc[r0:r0 + n].double()
                heads = slice(g * G, (g + 1) * G)
                if kind == "multi":
                    qq = q[l, b, :, heads].double().reshape(Q * G, HEAD)
                else:
                    K = torch.cat([K, k_new[l, b, g].double()[None]])
                    V = torch.cat([V, v_new[l, b, g].double()[None]])
                    qq = q[l, b, heads].double()
                o = torch.softmax(qq @ K.T / math.sqrt(HEAD), dim=-1) @ V
                if kind == "multi":
                    out[l, b, :, heads] = o.reshape(Q, G, HEAD)
                else:
                    out[l, b, heads] = o
    return {"out": out} if kind == "multi" else {"out": out, "Kc": None, "Vc": None}
