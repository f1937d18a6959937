"""The work that users of this library have it do, as cases that can be timed.

A case is one call of a public entry point on the tensors that a training (or
export) program holds at that moment: one weight matrix, the seven linear
weights of a decoder layer, or the linear weights of several layers.  Shapes
and distributions are those of ``paper_2608_13966_gb300.workloads``.

Keys of a case:
  call      "single" (one tensor), "batch" (several tensors, outputs allocated
            by the call) or "model" (the C entry point over buffers the
            program keeps: one flat buffer per output, as for a whole model)
  kind      "int" (asymmetric codes), "sym" (symmetric codes), "nvfp4", "lut"
  shapes    "rowsxcols,..." of the tensors, repeated ``layers`` times
  bits, group, clip   integer bits, group size, factor grid ("8": 1.00..0.65,
            "16": 1.00..0.25, "paper": 0.30..1.00)
  g, r      gradient ("bf16", "f32", "none") and reconstruction dtype
  codes     "none", "u8" or "packed"
  saliency  "ema", "ema_squared" or "uniform"
  adamw     the call also takes the AdamW step
  amax      NVFP4: the program supplies each tensor's absmax
  dist      distribution of w ("t4", "t3_outliers", "normal")
"""
import math

import numpy as np
import torch

from paper_2608_13966_gb300 import api, quasar, workloads as wl

BETA2 = 0.999
CLIPS = {"8": wl.CLIP_8, "16": wl.CLIP_16, "paper": wl.CLIP_PAPER}
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32, "none": None}
DEV = "cuda"


def _layer(layout):
    return ",".join(f"{rows}x{cols}" for _, rows, cols in layout)


LLAMA = _layer(wl.LLAMA31_8B_LAYER)
QWEN = _layer(wl.QWEN3_8B_LAYER)
BASE = {"call": "batch", "kind": "int", "shapes": LLAMA, "layers": 1, "bits": 3, "group": 128,
        "clip": "8", "g": "bf16", "r": "bf16", "codes": "none", "saliency": "ema", "adamw": False,
        "amax": False, "dist": "t4"}


def listed():
    def case(name, **kw):
        return dict(BASE, name=name, **kw)

    return [
        # the smallest call: one small fp32 matrix (a unit test, a probe of one
        # projection); latency and the launch count
        case("matrix_int4_f32", call="single", shapes="256x1024", bits=4, g="f32", r="f32",
             codes="u8", dist="normal"),
        # a layer wrapped at each step by a program that reconstructs layer by
        # layer, with the codes kept for statistics
        case("llama_layer_int3", codes="u8"),
        # small groups, a wide grid of 16 factors, outliers
        case("qwen_layer_int2_k16", shapes=QWEN, bits=2, group=64, clip="16", codes="u8",
             dist="t3_outliers"),
        # the paper's own ascending grid of 15 factors
        case("llama_layer_int3_paper_grid", clip="paper"),
        # a training step's whole pass: many tensors in one call, buffers kept
        # by the program (the largest case: 8 layers, 1.7e9 weights)
        case("llama_model_int3", call="model", layers=8),
        # the optimizer step fused with the reconstruction
        case("llama_layer_int3_adamw", adamw=True),
        # NVFP4 with the tensor absmax taken by the call, codes kept
        case("llama_layer_nvfp4", kind="nvfp4", bits=4, group=16, codes="u8"),
        # the optimizer step, then NVFP4 of the updated weights
        case("llama_layer_nvfp4_adamw", kind="nvfp4", bits=4, group=16, adamw=True),
        # the lookup-table format with its deployment codes
        case("llama_layer_lut", kind="lut", bits=3, group=512, codes="packed"),
        # symmetric codes
        case("llama_layer_int4_sym", kind="sym", bits=4),
        # odd row counts, small groups, fp32 gradients and reconstruction
        case("ragged_int4_g32_f32", shapes="1023x1056,517x2880,2049x736", bits=4, group=32,
             g="f32", r="f32"),
        # export of an attention block: no gradient, packed codes, absmax known
        case("export_nvfp4_packed", kind="nvfp4", bits=4, group=16, g="none", codes="packed",
             shapes="4096x4096,1024x4096,1024x4096,4096x4096", amax=True),
    ]


def draw(rng):
    c = dict(BASE)
    c["kind"] = rng.choice(["int"] * 8 + ["nvfp4"] * 5 + ["lut"] * 4 + ["sym"] * 3)
    c["adamw"] = c["kind"] in ("int", "nvfp4") and rng.random() < 0.25
    c["bits"] = {"int": rng.choice([2, 3, 3, 4, 4, 8]), "sym": rng.choice([3, 4, 4, 8]),
                 "nvfp4": 4, "lut": 3}[c["kind"]]
    c["group"] = {"nvfp4": 16, "lut": 512}.get(c["kind"], rng.choice([32, 64, 128, 128, 128, 256]))
    c["clip"] = rng.choice(["8", "8", "8", "16", "paper"])
    c["g"] = "f32" if rng.random() < 0.25 else "bf16"
    if not c["adamw"] and rng.random() < 0.15:
        c["g"] = "none"
    c["r"] = rng.choice(["bf16", "bf16", "f32"])
    c["codes"] = rng.choice(["none", "none", "u8", "packed"])
    c["saliency"] = rng.choice(["ema"] * 6 + ["ema_squared", "uniform"])
    c["dist"] = rng.choice(["t4", "t4", "t3_outliers", "normal"])
    c["amax"] = c["kind"] == "nvfp4" and not c["adamw"] and rng.random() < 0.3
    unit_r, unit_c = (8, 64) if c["kind"] == "lut" else (1, c["group"])
    n_t = rng.choice([1, 1, 2, 3, 7])
    total = 2.0 ** rng.uniform(15, 27.6)
    shapes = []
    for _ in range(n_t):
        n = total / n_t * 2.0 ** rng.uniform(-0.5, 0.5)
        cols = min(n, 2.0 ** rng.uniform(8, 13.8))
        cols = unit_c * max(1, round(cols / unit_c))
        rows = unit_r * max(1, min(round(n / cols / unit_r), 28672 // unit_r))
        shapes.append(f"{rows}x{cols}")
    c["shapes"] = ",".join(shapes)
    if n_t == 1 and c["kind"] in ("int", "nvfp4") and not c["adamw"] and c["saliency"] == "ema" \
            and c["codes"] != "packed":
        c["call"] = "single"
    return c


def _shapes(case):
    one = [tuple(int(x) for x in s.split("x")) for s in case["shapes"].split(",")]
    return one * case["layers"]


def _hyper(case):
    return dict(wl.ADAMW_NVFP4 if case["kind"] == "nvfp4" else wl.ADAMW_LLAMA_INT3)


def _inputs(case, seed):
    """(w, g, v, m) of each tensor, drawn as the workloads draw theirs."""
    g_dtype = DTYPES[case["g"]]
    for j, (rows, cols) in enumerate(_shapes(case)):
        spec = wl.TensorSpec(f"t{j}", rows, cols, j // 7, j)
        like = wl.Workload("case", "int", case["bits"], case["group"], CLIPS[case["clip"]], BETA2,
                           g_dtype or torch.float32, torch.float32, False, (spec,), case["dist"],
                           "warm_g2" if case["dist"] == "normal" else "lognormal",
                           adamw=_hyper(case) if case["adamw"] else {})
        d = wl.make_tensor(like, spec, device=DEV, seed=seed)
        yield d["w"], d["g"] if g_dtype else None, d["v"], d.get("m")


def prepare(case, seed):
    items = []
    for w, g, v, m in _inputs(case, seed):
        if case["adamw"]:
            items.append((w, g, m, v))
        elif case["amax"]:
            items.append((w, g, v, w.abs().max().reshape(1)))
        else:
            items.append((w, g, v))
    state = {"case": case, "items": items}
    if case["call"] == "model":
        n = sum(it[0].numel() for it in items)
        flat = {"r": torch.empty(n, dtype=DTYPES[case["r"]], device=DEV),
                "a": torch.empty(n // case["group"], dtype=torch.float32, device=DEV),
                "b": torch.empty(n // case["group"], dtype=torch.float32, device=DEV),
                "cand_idx": torch.empty(n // case["group"], dtype=torch.uint8, device=DEV),
                "v": torch.cat([it[2].reshape(-1) for it in items])}
        descs, at = [], 0
        for i, (w, g, v) in enumerate(items):
            k, p, q = w.numel(), at // case["group"], (at + w.numel()) // case["group"]
            items[i] = (w, g, flat["v"][at:at + k])
            descs.append({"w": w, "g": g, "v": flat["v"][at:at + k], "r": flat["r"][at:at + k],
                          "a": flat["a"][p:q], "b": flat["b"][p:q],
                          "cand_idx": flat["cand_idx"][p:q], "rows": w.shape[0],
                          "cols": w.shape[1]})
            at += k
        state["flat"], state["descs"] = flat, quasar.int_tensor_array(descs)
    return state


def run(state):
    c, items = state["case"], state["items"]
    clip, r_dtype = CLIPS[c["clip"]], DTYPES[c["r"]]
    if c["call"] == "model":
        st = quasar.quasar_recon_int_batch(state["descs"], BETA2, c["bits"], c["group"], clip,
                                           g_dtype=quasar.F32 if c["g"] == "f32" else quasar.BF16,
                                           r_dtype=quasar.F32 if c["r"] == "f32" else quasar.BF16)
        if st != quasar.QuasarStatus.OK:
            raise quasar.QuasarError(st)
        return state["flat"]
    keep = dict(codes=c["codes"] != "none", r_dtype=r_dtype, beta2=BETA2)
    if c["call"] == "single":
        w, g, v = items[0][:3]
        if c["kind"] == "nvfp4":
            out = [api.recon_nvfp4(w, g, v, clip=clip, tensor_amax=items[0][3] if c["amax"] else None,
                                   **keep)]
        else:
            out = [api.recon_int(w, g, v, bits=c["bits"], group_size=c["group"], clip=clip, **keep)]
    else:
        keep.update(saliency=c["saliency"], packed_codes=c["codes"] == "packed")
        h = _hyper(c)
        if c["kind"] == "nvfp4":
            out = (api.adamw_recon_nvfp4_batch(items, clip=clip, **h, **keep) if c["adamw"]
                   else api.recon_nvfp4_batch(items, clip=clip, **keep))
        elif c["kind"] == "lut":
            out = api.recon_lut_batch(items, clip=clip, **keep)
        elif c["adamw"]:
            out = api.adamw_recon_int_batch(items, bits=c["bits"], group_size=c["group"], clip=clip,
                                            **h, **keep)
        else:
            out = api.recon_int_batch(items, bits=c["bits"], group_size=c["group"], clip=clip,
                                      symmetric=c["kind"] == "sym", **keep)
    for res, it in zip(out, items):
        if c["adamw"]:
            res.update(w=it[0], m=it[2], v=it[3])
        elif c["g"] != "none":
            res["v"] = it[2]
    return out


def work(case):
    n = sum(rows * cols for rows, cols in _shapes(case))
    k = len(CLIPS[case["clip"]])
    per = 8.0 + {"bf16": 2, "f32": 4, "none": 0}[case["g"]]              # w, v, g in
    per += {"bf16": 2, "f32": 4}[case["r"]] + (4 if case["g"] != "none" else 0)  # r, v' out
    per += 12 if case["adamw"] else 0                                    # m in; w', m' out
    code_bits = 4 if case["kind"] == "nvfp4" else case["bits"]
    per += {"none": 0.0, "u8": 1.0, "packed": code_bits / 8}[case["codes"]]
    group = {"int": 9, "sym": 9, "nvfp4": 2, "lut": 9}[case["kind"]]     # fit and index of a group
    # per weight and factor: the code, its moments and error (int: 5 fused or
    # plain operations beside the rounding; NVFP4 also sums its error directly;
    # the table only sums h and h w of each index)
    flops = {"int": 10, "sym": 8, "nvfp4": 12, "lut": 5}[case["kind"]] * k + 25
    return {"bytes": n * per + n // case["group"] * group, "flops": float(n * flops)}


def tolerance(case):
    # Measured against exact() rounded to the output's type, on the listed cases
    # and fourteen drawn ones.  Where both keep the same factor and codes, fp32
    # outputs agree to 1e-7 and bf16 ones to a rare rounding flip (1e-4); what is
    # larger comes from the few groups whose two best factors are within
    # rounding of each other, or whose weight lies on a code boundary, and where
    # a correct computation may keep the other one: such a group moves by up to
    # a code step, 1.9 times the rms of a heavy-tailed tensor.  Largest seen:
    # int 8.4e-4, lut 9.7e-4, nvfp4 4.6e-4, sym 2.0e-4 of r's norm; 1.5e-5 of
    # the whole values (a single group of a small tensor is more than that).
    rel = {"int": 4e-3, "lut": 4e-3, "nvfp4": 2e-3, "sym": 1e-3}[case["kind"]]
    groups = min(rows * cols // case["group"] for rows, cols in _shapes(case))
    return {"rel": rel, "max": 0.99, "differ": min(0.01, max(6e-5, 1.0 / groups))}


# ------------------------------------------------------------------ exact

def _f32(x):
    return float(np.float32(x))


def _best(best, new, better):
    return [torch.where(better.reshape(-1, *([1] * (x.dim() - 1))), x, y) for x, y in zip(new, best)]


def _exact_int(w, h, case):
    """Groups in rows: w, h [groups, G] fp64 -> r, a, b, codes, index."""
    qmax = 2 ** case["bits"] - 1
    h = torch.where(h.sum(1, keepdim=True) == 0, torch.ones_like(h), h)
    hs = h.sum(1)
    wb = (h * w).sum(1) / hs
    ww = (h * (w - wb[:, None]) ** 2).sum(1)
    mn, mx = w.min(1).values, w.max(1).values
    c, rho = (mn + mx) / 2, (mx - mn) / 2
    best, err = None, None
    for k, f in enumerate(CLIPS[case["clip"]]):
        f = _f32(f)
        z, s = c - f * rho, 2 * f * rho / qmax
        q = torch.round((w - z[:, None]) / s[:, None]).clamp_(0, qmax)
        qb = (h * q).sum(1) / hs
        dq = q - qb[:, None]
        hdq = h * dq
        dd, nn = (hdq * dq).sum(1), (hdq * (w - wb[:, None])).sum(1)
        a = torch.where(dd > 0, nn / dd, s)
        e = torch.where(dd > 0, ww - nn * a, ww)
        new = [a, wb - a * qb, q.to(torch.uint8), torch.full_like(c, k).to(torch.uint8)]
        best, err = (new, e) if best is None else (_best(best, new, e < err), torch.minimum(e, err))
    a, b, q, k = best
    flat = rho == 0
    a, b = torch.where(flat, torch.zeros_like(a), a), torch.where(flat, mn, b)
    q[flat] = 0
    k[flat] = 0
    r = torch.where(flat[:, None], w, a[:, None] * q + b[:, None])
    return r, a, b, q, k


def _exact_sym(w, h, case):
    top = 2 ** (case["bits"] - 1) - 1
    h = torch.where(h.sum(1, keepdim=True) == 0, torch.ones_like(h), h)
    amax = w.abs().max(1).values
    best, err = None, None
    for k, f in enumerate(CLIPS[case["clip"]]):
        s = _f32(f) * amax / top
        q = torch.round(w / s[:, None]).clamp_(-top, top)
        q = torch.where(amax[:, None] > 0, q, torch.zeros_like(q))
        qq = (h * q * q).sum(1)
        a = torch.where(qq > 0, (h * q * w).sum(1) / qq, s)
        e = (h * (a[:, None] * q - w) ** 2).sum(1)
        new = [a, q.to(torch.int8), torch.full_like(amax, k).to(torch.uint8)]
        best, err = (new, e) if best is None else (_best(best, new, e < err), torch.minimum(e, err))
    a, q, k = best
    return a[:, None] * q, a, -a * top, (q.to(torch.int16) + top).to(torch.uint8), k


def _e4m3(x):
    """The nearest E4M3 value of x (ties to even, at most 448) and its bits."""
    b = x.clamp(-448, 448).to(torch.float8_e4m3fn)
    v = b.double()
    bits = torch.where(v == 0, torch.zeros_like(b.view(torch.uint8)), b.view(torch.uint8))
    return v, bits


def _exact_nvfp4(w, h, case, amax):
    grid = torch.tensor([0, 0.5, 1, 1.5, 2, 3, 4, 6], dtype=torch.float64, device=w.device)
    s_t = float(np.float32(amax) / np.float32(2688.0)) if amax > 0 else 1.0
    h = torch.where(h.sum(1, keepdim=True) == 0, torch.ones_like(h), h)
    mag = w.abs()
    top = mag.max(1).values
    best, err = None, None
    for k, f in enumerate(CLIPS[case["clip"]]):
        sigma = _f32(f) * top / 6
        y = mag / torch.where(sigma > 0, sigma, torch.ones_like(sigma))[:, None]
        # ties go to the even code: up from codes 1, 3, 5, down from 0, 2, 4, 6
        i = ((y > 0.25).to(torch.int8) + (y >= 0.75) + (y > 1.25) + (y >= 1.75) + (y > 2.5)
             + (y >= 3.5) + (y > 5.0)).to(torch.int8)
        q = grid[i.long()]
        qq = (h * q * q).sum(1)
        x = torch.where(qq > 0, (h * q * mag).sum(1) / qq, sigma)
        sc, bits = _e4m3(x / s_t)
        a = s_t * sc
        e = (h * (a[:, None] * q - mag) ** 2).sum(1)
        new = [a, i, bits, torch.full_like(top, k).to(torch.uint8)]
        best, err = (new, e) if best is None else (_best(best, new, e < err), torch.minimum(e, err))
    a, i, bits, k = best
    zero = top == 0
    i[zero], bits[zero], k[zero] = 0, 0, 0
    r = torch.where(zero[:, None], torch.zeros_like(w), a[:, None] * grid[i.long()] * w.sign())
    return r, bits, s_t, (i + 8 * ((w < 0) & (i > 0))).to(torch.uint8), k


def _exact_lut(w, h, case):
    h = torch.where(h.sum(1, keepdim=True) == 0, torch.ones_like(h), h)
    mn, mx = w.min(1).values, w.max(1).values
    c, rho = (mn + mx) / 2, (mx - mn) / 2
    best, err = None, None
    for k, f in enumerate(CLIPS[case["clip"]]):
        z, s = c - _f32(f) * rho, 2 * _f32(f) * rho / 7
        q = torch.round((w - z[:, None]) / s[:, None]).clamp_(0, 7)
        q = torch.where(rho[:, None] > 0, q, torch.zeros_like(q))
        sums = []
        for j in range(8):
            hj = torch.where(q == j, h, torch.zeros_like(h))
            t = hj.sum(1)
            sums.append(torch.where(t > 0, (hj * w).sum(1) / t, z + j * s))
        v, bits = _e4m3(torch.stack(sums, 1))
        r = v.gather(1, q.long())
        e = (h * (r - w) ** 2).sum(1)
        new = [r, bits, q.to(torch.uint8), torch.full_like(c, k).to(torch.uint8)]
        best, err = (new, e) if best is None else (_best(best, new, e < err), torch.minimum(e, err))
    r, bits, q, k = best
    flat = rho == 0
    v, cb = _e4m3(c)
    r[flat], bits[flat], q[flat], k[flat] = v[flat, None], cb[flat, None], 0, 0
    return r, bits, q, k


def _exact_adamw(w, g, m, v, hp):
    lr, b1, b2, eps, wd = (_f32(x) for x in (hp["lr"], hp["beta1"], BETA2, hp["eps"],
                                             hp["weight_decay"]))
    m = b1 * m + (1 - b1) * g
    v = b2 * v + (1 - b2) * g * g
    den = v.sqrt() / math.sqrt(1 - b2 ** hp["step"]) + eps
    return w * (1 - lr * wd) - lr / (1 - b1 ** hp["step"]) * m / den, m, v


def exact(case, seed):
    results = []
    for w, g, v, m in _inputs(case, seed):
        rows, cols = w.shape
        w, v = w.double(), v.double()
        if case["adamw"]:
            w, m, v = _exact_adamw(w, g.double(), m.double(), v, _hyper(case))
        elif g is not None:
            v = _f32(BETA2) * v + (1 - _f32(BETA2)) * g.double() ** 2
        h = {"ema": lambda: v, "ema_squared": lambda: v * v,
             "uniform": lambda: torch.ones_like(v)}[case["saliency"]]()
        if case["kind"] == "lut":
            def blocks(x):
                return x.reshape(rows // 8, 8, cols // 64, 64).transpose(1, 2).reshape(-1, 512)

            def back(x):
                return x.reshape(rows // 8, cols // 64, 8, 64).transpose(1, 2).reshape(rows, cols)

            r, book, q, k = _exact_lut(blocks(w), blocks(h), case)
            res = {"r": back(r), "book": book, "cand_idx": k}
            q = back(q)
        elif case["kind"] == "nvfp4":
            amax = float(w.abs().max().float())
            r, bits, s_t, q, k = _exact_nvfp4(w.reshape(-1, 16), h.reshape(-1, 16), case, amax)
            res = {"r": r.reshape(rows, cols), "block_scale": bits, "cand_idx": k,
                   "tensor_scale": torch.tensor([s_t], dtype=torch.float64)}
        else:
            fit = _exact_sym if case["kind"] == "sym" else _exact_int
            r, a, b, q, k = fit(w.reshape(-1, case["group"]), h.reshape(-1, case["group"]), case)
            res = {"r": r.reshape(rows, cols), "a": a, "b": b, "cand_idx": k}
        if case["codes"] != "none":
            res["codes"] = None if case["codes"] == "packed" else q.reshape(rows, cols)
        if case["adamw"]:
            res.update(w=w, m=m, v=v)
        elif g is not None:
            res["v"] = v
        results.append(res)
    if case["call"] == "model":
        return {k: torch.cat([x[k].reshape(-1) for x in results]) for k in results[0]}
    return results
