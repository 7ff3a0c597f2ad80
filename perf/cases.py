"""The measured cases: what a program that fine-tunes the block scales of an FP4 model
asks of this package, over the range of sizes it asks it for.

Kinds of case (every call goes through Handle, with the buffers a training loop keeps):

  step     one linear of a training step: forward, input gradient and masked scale gradient
  layer    one decoder layer of a training step: projection of its seven latent planes,
           the three contractions of each linear, merge of the seven planes
  planes   projection and merge of every scale plane of a layer (an optimizer step, an export)
  edit     one plane of a served model: hot-swap the base scales in, merge a task, audit the
           change, roll the merge back
  adapter  the low-rank scale adapter of one linear: latent, projection and mask from B and
           A, and the gradients of B and A from a scale gradient
  moe      one expert linear of a mixture-of-experts step: grouped forward, input gradient
           and masked scale gradient over the experts' routed rows
  moe_adapter  the adapters of all experts of one linear

Token counts run from one short example to a 16 x 2048 batch; the shapes are the package's
synthetic workloads' (Llama-3-8B-shaped layers, Qwen3-30B-A3B- and gpt-oss-120B-shaped
experts) and generic ones of the same range.
"""
import math

import torch

import paper_2609_04526_gb300 as pkg
from paper_2609_04526_gb300 import synth

FMT = {"nvfp4": synth.NVFP4, "mxfp4": synth.MXFP4}
BLOCK = {"nvfp4": 16, "mxfp4": 32}

# q, k, v, o, gate, up, down as multiples (out, in) of (hidden, key/value width, intermediate)
LAYER = (("q", "h", "h"), ("k", "kv", "h"), ("v", "kv", "h"), ("o", "h", "h"), ("gate", "f", "h"), ("up", "f", "h"),
         ("down", "h", "f"))


def listed():
    return [
        # the smallest linear of the package's own checks: launches and host calls are what counts
        {"name": "step_tiny", "kind": "step", "fmt": "nvfp4", "M": 64, "N": 256, "K": 512, "act": "gauss"},
        # one short training example (a question with its answer) through an attention projection
        {"name": "step_example", "kind": "step", "fmt": "nvfp4", "M": 187, "N": 4096, "K": 4096, "act": "gauss"},
        # one sequence, its padding removed (a ragged token count), through the down projection
        {"name": "step_down_seq", "kind": "step", "fmt": "nvfp4", "M": 1999, "N": 4096, "K": 14336, "act": "silu"},
        # two sequences through an MXFP4 projection with outlier channels
        {"name": "step_mx", "kind": "step", "fmt": "mxfp4", "M": 4096, "N": 4096, "K": 4096, "act": "outlier"},
        # the largest linear at the full 16 x 2048 batch
        {"name": "step_gate_batch", "kind": "step", "fmt": "nvfp4", "M": 32768, "N": 14336, "K": 4096, "act": "gauss"},
        # a whole layer for one 2048-token sequence: the usual micro-batch of a fine-tuning run
        {"name": "layer_seq", "kind": "layer", "fmt": "nvfp4", "M": 2048, "h": 4096, "kv": 1024, "f": 14336},
        # every scale plane of that layer projected and merged
        {"name": "layer_planes", "kind": "planes", "fmt": "nvfp4", "h": 4096, "kv": 1024, "f": 14336},
        # the plane of one served MXFP4 linear swapped, merged, audited and rolled back
        {"name": "plane_edit", "kind": "edit", "fmt": "mxfp4", "N": 14336, "K": 4096},
        # the adapter of the gate projection at the rank of the 8B runs
        {"name": "adapter_gate", "kind": "adapter", "fmt": "nvfp4", "N": 14336, "K": 4096, "r": 58},
        # 128 small NVFP4 experts, one 2048-token sequence routed top-8
        {"name": "moe_seq", "kind": "moe", "fmt": "nvfp4", "E": 128, "T": 2048, "top": 8, "N": 768, "K": 2048},
        # 128 larger MXFP4 experts, four sequences routed top-4
        {"name": "moe_mx", "kind": "moe", "fmt": "mxfp4", "E": 128, "T": 8192, "top": 4, "N": 2880, "K": 2880},
        # the adapters of the 128 small experts at the rank of the MoE runs
        {"name": "moe_adapter", "kind": "moe_adapter", "fmt": "nvfp4", "E": 128, "N": 768, "K": 2048, "r": 54},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dim(rng, lo, hi, step):
    """A size spread over the logarithm of lo .. hi, a multiple of `step` (the formats' own granularity)."""
    return min(hi, max(lo, step * round(_log(rng, lo, hi) / step)))


def draw(rng):
    fmt = rng.choice(("nvfp4", "nvfp4", "mxfp4"))
    kind = rng.choice(("step", "step", "step", "moe", "moe", "layer", "planes", "edit", "adapter", "moe_adapter"))
    if kind == "step":
        N, K = _dim(rng, 256, 14336, 8), _dim(rng, 512, 14336, 32)
        most = min(32768, 32768 * 14336 * 4096 // (N * K))
        return {"kind": kind, "fmt": fmt, "M": int(_log(rng, 16, most + 0.5)), "N": N, "K": K,
                "act": rng.choice(("gauss", "silu", "outlier"))}
    if kind in ("layer", "planes"):
        h, f = _dim(rng, 1024, 4096, 64), _dim(rng, 2048, 14336, 64)
        c = {"kind": kind, "fmt": fmt, "h": h, "kv": rng.choice((h, h // 4)) // 32 * 32, "f": f}
        if kind == "layer":
            c["M"] = int(_log(rng, 64, 4096.5))
        return c
    if kind == "edit":
        return {"kind": kind, "fmt": fmt, "N": _dim(rng, 512, 14336, 8), "K": _dim(rng, 512, 14336, 32)}
    if kind == "adapter":
        return {"kind": kind, "fmt": fmt, "N": _dim(rng, 512, 14336, 8), "K": _dim(rng, 512, 14336, 32),
                "r": int(_log(rng, 4, 128.5))}
    E = rng.choice((8, 16, 32, 64, 128))
    N, K = _dim(rng, 512, 2880, 32), _dim(rng, 512, 2880, 32)
    if kind == "moe":
        return {"kind": kind, "fmt": fmt, "E": E, "T": int(_log(rng, 64, 16384.5)), "top": rng.choice((2, 4, 8)),
                "N": N, "K": K}
    return {"kind": kind, "fmt": fmt, "E": E, "N": N, "K": K, "r": int(_log(rng, 4, 128.5))}


# ------------------------------------------------------------------ preparation

_handle = None


def _h():
    """The one handle a training process keeps."""
    global _handle
    if _handle is None:
        _handle = pkg.Handle()
    return _handle


def _linears(case):
    return [synth.Linear(n, case[o], case[i], "x_" + ("f" if i == "f" else n)) for n, o, i in LAYER]


def _dense(case, seed, linears, kinds):
    """A dense workload of these linears (inputs come from its seed)."""
    acts = tuple((l.x, l.K, kinds.get(l.x, "gauss")) for l in linears)
    return synth.Workload("case", "case", FMT[case["fmt"]], case.get("M", 1), tuple(linears), acts, seed)


def _mask(shape, seed, device="cuda"):
    """STE mask of a plane: one in a thousand scales at the ceiling."""
    g = torch.Generator(device=device)
    g.manual_seed(seed * 7919 + 13)
    return (torch.rand(shape, generator=g, device=device) >= 1e-3).to(torch.uint8)


def _step_state(wl, lin, seed):
    w = synth.gen_weight(wl, lin, device="cuda")
    X = synth.gen_act(wl, lin.x, device="cuda")
    dY = synth.gen_dy(wl, lin, device="cuda")
    return {"w": pkg.QuantWeight(wl.fmt, lin.N, lin.K, w.codes, w.scales, w.ws2), "X": X, "dY": dY,
            "mask": _mask(w.scales.shape, seed), "Y": torch.empty_like(dY), "dX": torch.empty_like(X),
            "g": torch.empty(w.scales.shape, dtype=torch.float32, device="cuda")}


def _plane_state(wl, lin, w):
    """One plane of the projection and merge: the latent, the training bytes, mask and NaN
    count it is projected to, and the artifact's scale plane it is merged into."""
    z = lambda t: torch.empty(w.scales.shape, dtype=t, device="cuda")  # noqa: E731
    return {"latent": synth.gen_latent(wl, lin, w, device="cuda"), "bytes": z(torch.uint8), "mask": z(torch.uint8),
            "ws2": w.ws2, "nonfinite": torch.zeros(1, dtype=torch.int32, device="cuda"),
            "changed": torch.zeros(1, dtype=torch.int64, device="cuda"), "art": w.scales.clone()}


def _plane_calls(planes):
    proj = [{k: p[k] for k in ("latent", "bytes", "mask", "ws2", "nonfinite")} for p in planes]
    merge = [{"latent": p["latent"], "bytes": p["art"], "ws2": p["ws2"], "changed": p["changed"]} for p in planes]
    return proj, merge


def _experts(case, seed):
    """The workload and weights of one expert linear; a router with log-normal expert
    popularity picks the rows (ragged, some experts may have none)."""
    lin = synth.Linear("w", case["N"], case["K"], "x")
    wl = synth.MoEWorkload("case", "case", FMT[case["fmt"]], case.get("T", 1), min(case.get("top", 1), case["E"]),
                           case["E"], (lin,), (("x", case["K"], "gauss"),), seed)
    ex = synth.gen_experts(wl, lin, device="cuda")
    return wl, lin, ex, pkg.GroupedWeight(ex.fmt, ex.E, ex.N, ex.K, ex.codes, ex.scales, ex.ws2)


def prepare(case, seed):
    kind, h = case["kind"], _h()
    s = {"kind": kind, "h": h, "fmt": FMT[case["fmt"]]}
    empty = lambda shape, t: torch.empty(shape, dtype=t, device="cuda")  # noqa: E731
    if kind == "step":
        lin = synth.Linear("w", case["N"], case["K"], "x")
        s.update(_step_state(_dense(case, seed, [lin], {"x": case["act"]}), lin, seed))
    elif kind in ("layer", "planes"):
        linears = _linears(case)
        wl = _dense(case, seed, linears, {"x_f": "silu"})
        s["planes"], s["steps"] = [], []
        for i, lin in enumerate(linears):
            if kind == "layer":
                t = _step_state(wl, lin, seed + i)
                w = t["w"]
                p = _plane_state(wl, lin, w)
                # the contractions read the projected bytes and mask of this step
                t["w"] = pkg.QuantWeight(w.fmt, w.N, w.K, w.codes, p["bytes"], w.ws2)
                t["mask"] = p["mask"]
                s["steps"].append(t)
            else:
                p = _plane_state(wl, lin, synth.gen_weight(wl, lin, device="cuda"))
            s["planes"].append(p)
        if kind == "layer":  # q, k and v read one activation, gate and up another
            for i, j in ((1, 0), (2, 0), (5, 4)):
                s["steps"][i]["X"] = s["steps"][j]["X"]
        s["project"], s["merge"] = _plane_calls(s["planes"])
    elif kind == "edit":
        lin = synth.Linear("w", case["N"], case["K"], "x")
        wl = _dense(case, seed, [lin], {})
        w = synth.gen_weight(wl, lin, device="cuda")
        s.update(base=w.scales, ws2=w.ws2, latent=synth.gen_latent(wl, lin, w, device="cuda"),
                 art=torch.zeros_like(w.scales), merged=torch.zeros_like(w.scales),
                 delta=empty(w.scales.shape, torch.float32), changed=empty(1, torch.int64),
                 diff=empty(1, torch.int64), undone=empty(1, torch.int64))
    elif kind == "adapter":
        lin = synth.Linear("w", case["N"], case["K"], "x")
        wl = _dense(case, seed, [lin], {})
        w = synth.gen_weight(wl, lin, device="cuda")
        B, A, aor = synth.gen_adapter(wl, lin, w, r=case["r"], device="cuda")
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed + 17)
        s.update(base=w.scales, ws2=w.ws2, B=B, A=A, aor=aor, bytes=torch.empty_like(w.scales),
                 mask=torch.empty_like(w.scales), latent=empty(w.scales.shape, torch.float32),
                 nonfinite=empty(1, torch.int32),
                 g=torch.randn(w.scales.shape, generator=gen, device="cuda") * 1e-2 * _mask(w.scales.shape, seed),
                 dB=empty(B.shape, torch.float32), dA=empty(A.shape, torch.float32))
    elif kind == "moe":
        wl, lin, ex, gw = _experts(case, seed)
        off = synth.offsets_of(synth.gen_routing(wl))
        X = synth.gen_act(wl, "x", M=off[-1], device="cuda")
        dY = synth.gen_dy(wl, lin, M=off[-1], device="cuda")
        s.update(w=gw, off=off, X=X, dY=dY, mask=_mask(ex.scales.shape, seed), Y=torch.empty_like(dY),
                 dX=torch.empty_like(X), g=empty(ex.scales.shape, torch.float32))
    else:
        wl, lin, ex, gw = _experts(case, seed)
        B, A, aor = synth.gen_expert_adapters(wl, lin, ex, r=case["r"], device="cuda")
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed + 17)
        s.update(w=gw, B=B, A=A, aor=aor, bytes=torch.empty_like(ex.scales), mask=torch.empty_like(ex.scales),
                 latent=empty(ex.scales.shape, torch.float32), nonfinite=empty(1, torch.int32),
                 g=torch.randn(ex.scales.shape, generator=gen, device="cuda") * 1e-2 * _mask(ex.scales.shape, seed),
                 dB=empty(B.shape, torch.float32), dA=empty(A.shape, torch.float32))
    return s


# ------------------------------------------------------------------ one pass

def _contractions(h, t):
    h.sq_fwd(t["w"], t["X"], t["Y"])
    h.sq_bwd_dx(t["w"], t["dY"], t["dX"])
    h.sq_scale_grad(t["w"], t["X"], t["dY"], mask=t["mask"], g=t["g"])
    return [t["Y"], t["dX"], t["g"]]


def run(s):
    kind, h, fmt = s["kind"], s["h"], s["fmt"]
    if kind == "step":
        return _contractions(h, s)
    if kind in ("layer", "planes"):
        h.sq_project_planes(fmt, s["project"])
        out = [_contractions(h, t) for t in s["steps"]]
        h.sq_merge_planes(fmt, s["merge"])
        # the changed-byte counters are not returned: a second merge of the same latents changes nothing
        return [out, [[p["bytes"], p["mask"], p["nonfinite"], p["art"]] for p in s["planes"]]]
    if kind == "edit":
        h.sq_swap_scales(s["base"], s["art"])
        h.sq_merge(fmt, s["latent"], s["ws2"], s["art"], ongrid_delta=s["delta"], changed=s["changed"])
        h.sq_count_diff(s["art"], s["base"], s["diff"])
        h.sq_swap_scales(s["art"], s["merged"])
        h.sq_rollback(fmt, s["delta"], s["ws2"], s["art"], s["undone"])
        return [s["merged"], s["delta"], s["changed"], s["diff"], s["art"], s["undone"]]
    if kind == "adapter":
        h.sq_project_lowrank(fmt, s["base"], s["B"], s["A"], s["ws2"], s["aor"], bytes_out=s["bytes"],
                             mask_out=s["mask"], nonfinite=s["nonfinite"], latent_out=s["latent"])
        h.sq_lowrank_grad(s["g"], s["B"], s["A"], s["aor"], dB=s["dB"], dA=s["dA"])
        return [s["bytes"], s["mask"], s["nonfinite"], s["latent"], s["dB"], s["dA"]]
    if kind == "moe":
        h.sq_grouped_fwd(s["w"], s["off"], s["X"], s["Y"])
        h.sq_grouped_bwd_dx(s["w"], s["off"], s["dY"], s["dX"])
        h.sq_grouped_scale_grad(s["w"], s["off"], s["X"], s["dY"], mask=s["mask"], g=s["g"])
        return [s["Y"], s["dX"], s["g"]]
    h.sq_grouped_project_lowrank(s["w"], s["B"], s["A"], s["aor"], bytes_out=s["bytes"], mask_out=s["mask"],
                                 nonfinite=s["nonfinite"], latent_out=s["latent"])
    h.sq_grouped_lowrank_grad(s["g"], s["B"], s["A"], s["aor"], dB=s["dB"], dA=s["dA"])
    return [s["bytes"], s["mask"], s["nonfinite"], s["latent"], s["dB"], s["dA"]]


# ------------------------------------------------------------------ necessary work and tolerance

def _step_work(M, N, K, G, weights=1):
    """Forward, input gradient and scale gradient of `weights` weights over M rows in all:
    X and dY, the codes, the scale bytes and mask read once, Y, dX and g written once."""
    nbytes = 2 * 2 * M * (N + K) + weights * (N * K // 2 + N * G * (1 + 1 + 4))
    return nbytes, 6 * M * N * K


def work(case):
    kind, B = case["kind"], BLOCK[case["fmt"]]
    if kind in ("layer", "planes"):
        nbytes = flops = 0
        for lin in _linears(case):
            N, K, G = lin.N, lin.K, lin.K // B
            # latent, projected byte, mask byte, old and new artifact byte
            nbytes += N * G * 8
            if kind == "layer":
                b, f = _step_work(case["M"], N, K, G)
                nbytes, flops = nbytes + b - 2 * N * G, flops + f  # the projection's bytes stay on the chip at best
        if kind == "layer":
            nbytes -= 2 * case["M"] * 3 * case["h"]  # q, k, v share an input, gate and up another
        return {"bytes": nbytes, "flops": flops}
    N, K = case["N"], case["K"]
    G = K // B
    if kind == "step":
        b, f = _step_work(case["M"], N, K, G)
        return {"bytes": b, "flops": f}
    if kind == "edit":  # base and latent read, merged plane, delta and rolled-back plane written
        return {"bytes": N * G * (1 + 4 + 1 + 4 + 1), "flops": 0}
    if kind == "moe":
        b, f = _step_work(case["T"] * min(case["top"], case["E"]), N, K, G, case["E"])
        return {"bytes": b, "flops": f}
    E, r = case.get("E", 1), case["r"]
    # base byte, B and A read, byte, mask and latent written; g read, dB and dA written; three products of rank r
    return {"bytes": E * (N * G * (1 + 1 + 1 + 4 + 4) + r * (N + G) * (2 + 4)), "flops": E * 6 * N * G * r}


def tolerance(case):
    kind = case["kind"]
    if kind in ("step", "layer", "moe"):
        return {"rel": 7e-3, "max": 0.05}  # Y and dX are rounded to bf16: 1.7e-3 off a 64-bit result
    if kind in ("adapter", "moe_adapter"):
        return {"rel": 1e-5, "max": 1e-3}  # fp32 sums; the bytes and mask stay as they are
    return "exact"


# ------------------------------------------------------------------ the same results in 64 bits

_E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


def _codes64(codes):
    """Packed nibbles [.., K/2] (even element low) -> fp64 E2M1 values [.., K]."""
    table = torch.tensor(_E2M1 + tuple(-v for v in _E2M1), dtype=torch.float64, device=codes.device)
    pair = torch.stack((codes & 15, codes >> 4), dim=-1).flatten(-2)
    return table[pair.long()]


def _scales64(fmt, scales, ws2):
    if fmt == synth.NVFP4:
        return scales.view(torch.float8_e4m3fn).double() * ws2
    return torch.exp2(scales.double() - 127)


def _step64(fmt, codes, scales, ws2, mask, X, dY):
    B = 16 if fmt == synth.NVFP4 else 32
    c = _codes64(codes)
    W = c * _scales64(fmt, scales, ws2).repeat_interleave(B, dim=1)
    X, dY = X.double(), dY.double()
    Y, dX = X @ W.T, dY @ W
    g = ((dY.T @ X) * c).unflatten(1, (-1, B)).sum(2) * mask
    return [Y, dX, g]


def exact(case, seed):
    if work(case)["flops"] > 6e12 or case["kind"] == "planes":
        return None  # too long in 64 bits; or bytes alone
    s = prepare(case, seed)
    kind, fmt = s["kind"], s["fmt"]
    if kind == "step":
        w = s["w"]
        return _step64(fmt, w.codes, w.scales, w.ws2, s["mask"], s["X"], s["dY"])
    if kind == "layer":
        # the projected bytes come from a torch cast of the clamped latents (E4M3) or their
        # rounded logarithm (E8M0), the mask from the clamp
        out = []
        for t, p in zip(s["steps"], s["planes"]):
            L, w = p["latent"], t["w"]
            if fmt == synth.NVFP4:
                cap = torch.tensor(448.0, device="cuda") * torch.tensor(w.ws2, dtype=torch.float32, device="cuda")
                q = (L.clamp(-cap, cap) / torch.tensor(w.ws2, dtype=torch.float32, device="cuda"))
                byte = q.clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)
                mask = (L.abs() <= cap).double()
            else:
                m, e = torch.frexp(L.double())  # L = m 2^e, m in [0.5, 1)
                e = e - 1 + (m > math.sqrt(0.5)).to(e.dtype)
                ok = (L > 0) & (e >= -127) & (e <= 127)
                byte = torch.where(L > 0, (e + 127).clamp(0, 254), torch.zeros_like(e)).to(torch.uint8)
                mask = ok.double()
            out.append(_step64(fmt, w.codes, byte, w.ws2, mask, t["X"], t["dY"]))
        return [out, [[None] * 4 for _ in s["planes"]]]
    if kind == "edit":
        return None  # bytes, counts and a difference of two scales that is exact by definition
    if kind == "moe":
        w, off = s["w"], s["off"]
        Y, dX, g = s["Y"].double(), s["dX"].double(), s["g"].double()
        for e in range(w.E):
            a, b = off[e], off[e + 1]
            Y[a:b], dX[a:b], g[e] = _step64(fmt, w.codes[e], w.scales[e], w.ws2[e], s["mask"][e], s["X"][a:b],
                                            s["dY"][a:b])
        return [Y, dX, g]
    if kind == "adapter":
        eff = _scales64(fmt, s["base"], s["ws2"])
    else:
        eff = torch.stack([_scales64(fmt, s["w"].scales[e], s["w"].ws2[e]) for e in range(s["w"].E)])
    B, A, g = s["B"].double(), s["A"].double(), s["g"].double()
    return [None, None, None, eff + s["aor"] * (B @ A), s["aor"] * (g @ A.mT), s["aor"] * (B.mT @ g)]
