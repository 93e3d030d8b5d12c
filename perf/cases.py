"""The work a user of this framework has it do, as timed cases.

One call of a serving or generation loop each, through the package's public
functions: decode attention over a compressed cache (from one short request
to the long-context batches), several requests in one launch, the many-query
attention of image generation and editing, the prefill's observation scores
and compression, re-compression under a shrinking budget, and one whole
request batch (prefill and graphed decode steps). Shapes are those of the
repository's workloads (28 query / 4 KV heads of 128 channels) and their
neighbours; inputs are seeded Gaussian K / V with a few outlier key channels,
as everywhere else in the repository.

Segments are written as text, one per cache type in context order:
  "full N"            every token kept in bf16 (a view of the prompt's rows)
  "quant/B N"         every token at B bits
  "evict N K"         the K best of N tokens in bf16
  "evict_quant/B N K" the K best of N tokens at B bits
``spread`` in [0, 1) makes the batch's kept counts differ (budgets are per
sequence): sequence b of an evicted type keeps K (1 - spread b / batch).
"""
import math

import torch

import paper_2609_32831_gb300 as uc
from paper_2609_32831_gb300.engine import CacheType, RequestCache

HQ, HKV, D, GROUP = 28, 4, 128, 32
DEV = "cuda"


# ------------------------------------------------------------------- cases

def listed():
    return [
        # one short request: 256 prompt tokens, an image evicted to 20 % at
        # int4, a few generated tokens; latency is all that counts
        {"name": "decode_1k_b1", "op": "attend", "batch": 1, "tokens": 1, "stats": False, "spread": 0.0,
         "segs": "full 256; evict_quant/4 768 153; evict 21 21"},
        # multi-image understanding, batch 8: prompt in bf16, four images
        # evicted to 30 % at int4, 512 generated tokens at int2
        {"name": "decode_8k_b8", "op": "attend", "batch": 8, "tokens": 1, "stats": True, "spread": 0.1,
         "segs": "full 512; evict_quant/4 7168 2150; quant/2 512"},
        # long-context serving, batch 16: both calibrated types at int2 and
        # the generated tokens so far
        {"name": "decode_32k_b16", "op": "attend", "batch": 16, "tokens": 1, "stats": False, "spread": 0.0,
         "segs": "quant/2 3276; quant/2 29492; evict 130 130"},
        # very long context, few sequences: the context is split over all SMs
        {"name": "decode_128k_b2", "op": "attend", "batch": 2, "tokens": 1, "stats": False, "spread": 0.0,
         "segs": "quant/2 13107; quant/2 117965; evict 77 77"},
        # four query tokens at once (a drafted continuation being checked)
        {"name": "decode_draft4_16k_b4", "op": "attend", "batch": 4, "tokens": 4, "stats": True, "spread": 0.2,
         "segs": "full 1000; quant/4 12288; evict 3072 921"},
        # requests of very different lengths served in one launch
        {"name": "batch_8_requests", "op": "batch", "longest": 32768, "calls": 8, "tokens": 1},
        # text-to-image: 4096 latent queries over the prompt, the int4 latent
        # cache and the current latents
        {"name": "denoise_4k_b4", "op": "attend", "batch": 4, "tokens": 4096, "stats": True, "spread": 0.0,
         "segs": "full 256; quant/4 4096; full 4096"},
        # editing one small image: ragged sizes throughout
        {"name": "edit_1k_b1", "op": "attend", "batch": 1, "tokens": 1000, "stats": True, "spread": 0.0,
         "segs": "full 77; quant/4 1023; evict 700 140; full 1000"},
        # prefill: observation-window scores of one long-context layer
        {"name": "scores_32k_b16", "op": "scores", "batch": 16, "n": 32768, "window": 32},
        # prefill: the image tokens of that layer to int2
        {"name": "quantize_32k_b16", "op": "compress", "batch": 16, "n": 29492, "begin": 3276, "kind": "quant",
         "bits": 2, "keep": 29492, "recent": 0, "then": "", "then_bits": 16, "then_keep": 0},
        # an image type evicted to 20 %, then, in the next chunk of the
        # schedule, its budget halves and what it holds is evicted and quantized
        {"name": "evict_shrink_32k_b4", "op": "compress", "batch": 4, "n": 29492, "begin": 3276, "kind": "evict",
         "bits": 16, "keep": 5898, "recent": 32, "then": "evict_quant", "then_bits": 4, "then_keep": 2949},
        # a whole request batch: prefill (scores, masses, budgets, compression
        # of every layer) and the decode steps that follow, as a CUDA graph
        {"name": "generate_8k_b8", "op": "generate", "batch": 8, "n": 8192, "layers": 4, "steps": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_segs(rng, ctx):
    n0 = max(1, ctx // rng.choice([8, 10, 20]))
    n1 = max(2, ctx - n0)
    keep = max(1, int(n1 * rng.choice([0.1, 0.2, 0.3, 0.5])))
    first = rng.choice(["full %d" % n0, "quant/4 %d" % n0, "quant/2 %d" % n0])
    second = rng.choice(["quant/2 %d" % n1, "quant/4 %d" % n1, "evict %d %d" % (n1, keep),
                         "evict_quant/4 %d %d" % (n1, keep), "evict_quant/2 %d %d" % (n1, keep)])
    g = rng.randint(1, 250)
    return "; ".join([first, second] + rng.choice([[], ["evict %d %d" % (g, g)]]))


def draw(rng):
    op = rng.choice(["decode", "decode", "decode", "draft", "dense", "dense", "batch", "scores", "compress",
                     "compress", "generate"])
    if op in ("decode", "draft"):
        tokens = 1 if op == "decode" else rng.randint(2, 8)
        ctx = _log(rng, 300, 130000)
        batch = _log(rng, 1, max(1, min(16, 32768 * 16 // ctx)))
        if op == "draft":
            batch = max(1, min(batch, 65536 // ctx))
        return {"op": "attend", "batch": batch, "tokens": tokens, "stats": rng.random() < 0.5,
                "spread": rng.choice([0.0, 0.1, 0.3]), "segs": _draw_segs(rng, ctx)}
    if op == "dense":
        tokens = _log(rng, 200, 4096)
        batch = rng.randint(1, 4)
        n_text, n_cache = rng.randint(20, 256), _log(rng, 200, 4096)
        cache = rng.choice(["quant/4 %d" % n_cache, "quant/2 %d" % n_cache, "evict %d %d" % (n_cache, n_cache // 5)])
        return {"op": "attend", "batch": batch, "tokens": tokens, "stats": True, "spread": 0.0,
                "segs": "full %d; %s; full %d" % (n_text, cache, tokens)}
    if op == "batch":
        return {"op": "batch", "longest": _log(rng, 2000, 32768), "calls": rng.randint(2, 8),
                "tokens": rng.choice([1, 1, 1, 2])}
    if op == "scores":
        n = _log(rng, 500, 131072)
        return {"op": "scores", "batch": max(1, min(rng.randint(1, 16), 32768 * 16 // n)), "n": n,
                "window": rng.choice([8, 16, 32, 32])}
    if op == "compress":
        n = _log(rng, 500, 118000)
        kind, bits = rng.choice([("quant", 2), ("quant", 4), ("evict", 16), ("evict_quant", 4), ("evict_quant", 2)])
        keep = n if kind == "quant" else max(2, int(n * rng.choice([0.1, 0.2, 0.3])))
        then = rng.choice(["", "", "evict_quant"])
        return {"op": "compress", "batch": max(1, min(rng.randint(1, 16), 29492 * 16 // n)), "n": n,
                "begin": rng.randint(0, 300), "kind": kind, "bits": bits, "keep": keep,
                "recent": rng.choice([0, 0, 1]) and min(32, keep) if kind != "quant" else 0,
                "then": then, "then_bits": rng.choice([2, 4]) if then else 16, "then_keep": max(1, keep // 2) if then else 0}
    n = _log(rng, 1000, 16384)
    return {"op": "generate", "batch": max(1, min(rng.randint(1, 8), 65536 // n)), "n": n,
            "layers": rng.randint(2, 4), "steps": rng.randint(2, 16)}


# ------------------------------------------------------------------ inputs

def _gen(seed, k=0):
    return torch.Generator(device=DEV).manual_seed(1000003 * k + int(seed))


def _kv(seed, batch, n, k=0):
    """bf16 K, V [batch, HKV, n, D]: Gaussian, four key channels ten times larger."""
    g = _gen(seed, k)
    kk = torch.randn((batch, HKV, n, D), generator=g, device=DEV)
    ch = torch.randperm(D, generator=g, device=DEV)[:4]
    kk[..., ch] *= 10.0
    kk = kk.to(torch.bfloat16)
    return kk, torch.randn((batch, HKV, n, D), generator=g, device=DEV).to(torch.bfloat16)


def _q(seed, batch, tokens, k=0):
    return torch.randn((batch, HQ, tokens, D), generator=_gen(seed, 500 + k), device=DEV).to(torch.bfloat16)


def _scores(seed, batch, n, k=0):
    """Positive eviction scores with the long tail of attention masses."""
    return torch.empty((batch, HKV, n), device=DEV).exponential_(1.0, generator=_gen(seed, 900 + k))


def _parse(segs):
    out = []
    for s in segs.split(";"):
        kind, *nums = s.split()
        kind, _, bits = kind.partition("/")
        n = int(nums[0])
        out.append((kind, int(bits or 16), n, int(nums[1]) if len(nums) > 1 else n))
    return out


def _keeps(batch, kind, keep, spread):
    return [max(1, int(keep * (1.0 - spread * b / batch))) if kind.startswith("evict") else keep
            for b in range(batch)]


def _build(kk, vv, sc, segs, spread, ws):
    """The compressed segments of one layer, as a prefill leaves them."""
    out, begin, batch = [], 0, kk.shape[0]
    for kind, bits, n, keep in segs:
        if kind == "full":
            out.append(uc.Segment.view(kk, vv, begin, n))
        else:
            keeps = _keeps(batch, kind, keep, spread)
            seg = uc.Segment(kind, bits, batch, HKV, n, max(keeps), DEV)
            seg.set_keep(keeps)
            uc.compress_segment(kk, vv, seg, begin=begin, scores=sc if kind.startswith("evict") else None, ws=ws)
            out.append(seg)
        begin += n
    return out


def _batch_calls(case):
    """(context, segments text) of each request: halving lengths, an int4 prompt and the rest at int2."""
    out = []
    for i in range(case["calls"]):
        n = max(64, case["longest"] >> i)
        out.append((n, "quant/4 %d; quant/2 %d" % (n // 10, n - n // 10)))
    return out


def _attend_inputs(case, seed):
    segs = _parse(case["segs"])
    n = sum(s[2] for s in segs)
    kk, vv = _kv(seed, case["batch"], n)
    return segs, kk, vv, _scores(seed, case["batch"], n), _q(seed, case["batch"], case["tokens"])


def _compress_inputs(case, seed):
    n = case["begin"] + case["n"]
    kk, vv = _kv(seed, case["batch"], n)
    return kk, vv, _scores(seed, case["batch"], n)


def _generate_inputs(case, seed):
    L, B, S = case["layers"], case["batch"], case["steps"]
    kv = [_kv(seed, B, case["n"], l) for l in range(L)]
    g = _gen(seed, 77)
    rnd = lambda *shape: torch.randn(shape, generator=g, device=DEV).to(torch.bfloat16)  # noqa: E731
    return ([k for k, _ in kv], [v for _, v in kv], rnd(L, B, HQ, 32, D), rnd(S, L, B, HQ, 1, D),
            rnd(S, L, B, HKV, D), rnd(S, L, B, HKV, D))


def prepare(case, seed):
    op = case["op"]
    ws = uc.Workspace(DEV)
    if op == "attend":
        segs, kk, vv, sc, q = _attend_inputs(case, seed)
        return {"op": op, "q": q, "segs": _build(kk, vv, sc, segs, case["spread"], ws), "ws": ws,
                "out": torch.empty_like(q), "stats": case["stats"]}
    if op == "batch":
        calls = []
        for i, (n, text) in enumerate(_batch_calls(case)):
            kk, vv = _kv(seed, 1, n, i)
            q = _q(seed, 1, case["tokens"], i)
            calls.append((q, _build(kk, vv, None, _parse(text), 0.0, ws), torch.empty_like(q)))
        return {"op": op, "calls": calls, "ws": ws}
    if op == "scores":
        kk, _ = _kv(seed, case["batch"], case["n"])
        out = torch.empty((case["batch"], HKV, case["n"]), device=DEV)
        return {"op": op, "k": kk, "q": _q(seed, case["batch"], case["window"]), "out": out, "ws": ws}
    if op == "compress":
        kk, vv, sc = _compress_inputs(case, seed)
        seg = uc.Segment(case["kind"], case["bits"], case["batch"], HKV, case["n"], case["keep"], DEV)
        seg.set_keep([case["keep"]] * case["batch"])
        st = {"op": op, "k": kk, "v": vv, "scores": sc if case["kind"] != "quant" or case["then"] else None,
              "seg": seg, "case": case, "ws": ws, "then": None}
        if case["then"]:
            st["then"] = uc.Segment(case["then"], case["then_bits"], case["batch"], HKV, case["n"],
                                    case["then_keep"], DEV)
            st["then"].set_keep([case["then_keep"]] * case["batch"])
        return st
    k, v, qwin, q, kn, vn = _generate_inputs(case, seed)
    n_text = case["n"] // 10
    rc = RequestCache([CacheType("text", n_text), CacheType("image", case["n"] - n_text)], case["layers"],
                      case["batch"], DEV, rho=0.25, gen_capacity=64)
    # the policies an offline calibration chose; the decode step is captured
    # once for the layout and replayed for every request batch of its shape
    rc.policy = {"text": uc.POLICY_QUANT, "image": uc.POLICY_QUANT}
    rc.prefill(k, v, qwin)
    rc.capture_decode()
    return {"op": "generate", "rc": rc, "k": k, "v": v, "qwin": qwin, "q": q, "kn": kn, "vn": vn}


# --------------------------------------------------------------- one pass

def _arrays(seg):
    out = {name: seg.tensor(name) for name in ("n_kept", "kept_idx", "k", "v", "k_codes", "k_params", "v_codes",
                                               "v_params")}
    return {name: t for name, t in out.items() if t is not None}


def run(state):
    op = state["op"]
    if op == "attend":
        out, lse, mass = uc.attend(state["q"], state["segs"], out=state["out"], want_lse=state["stats"],
                                   want_mass=state["stats"], ws=state["ws"])
        return {"out": out, "lse": lse, "mass": mass} if state["stats"] else {"out": out}
    if op == "batch":
        return [list(r) for r in uc.attend_batch(state["calls"], ws=state["ws"])]
    if op == "scores":
        return uc.score_accumulate(state["q"], state["k"], out=state["out"], ws=state["ws"])
    if op == "compress":
        c, seg = state["case"], state["seg"]
        uc.compress_segment(state["k"], state["v"], seg, begin=c["begin"], scores=state["scores"],
                            n_recent=c["recent"], ws=state["ws"])
        if state["then"] is None:
            return _arrays(seg)
        uc.recompress_segment(seg, state["then"], scores=state["scores"], scores_begin=c["begin"],
                              n_recent=c["recent"], ws=state["ws"])
        return [_arrays(seg), _arrays(state["then"])]
    rc = state["rc"]
    rc.prefill(state["k"], state["v"], state["qwin"])
    for s in range(state["q"].shape[0]):
        out = rc.decode_step_graph(state["q"][s], state["kn"][s], state["vn"][s])
    return {"out": out, "mass": rc.mass_buf}


# -------------------------------------------------------------------- work

def _stored(kind, bits, n):
    """Bytes of n stored tokens of one KV head (K and V)."""
    if bits == 16:
        return 4.0 * D * n
    full = n // GROUP * GROUP
    return full * (2.0 * D * bits / 8 + 4.0 * D / GROUP + 16.0) + 4.0 * D * (n - full)


def _attend_work(batch, tokens, segs, spread, stats):
    b, f = 2.0 * batch * HQ * tokens * D * 2, 0.0
    for kind, bits, _, keep in segs:
        for n in _keeps(batch, kind, keep, spread):
            b += HKV * _stored(kind, bits, n)
            f += 4.0 * HQ * tokens * n * D
    if stats:
        b += 4.0 * batch * HQ * tokens * (1 + len(segs))
    return b, f


def work(case):
    op = case["op"]
    if op == "attend":
        b, f = _attend_work(case["batch"], case["tokens"], _parse(case["segs"]), case["spread"], case["stats"])
    elif op == "batch":
        b = f = 0.0
        for _, text in _batch_calls(case):
            x, y = _attend_work(1, case["tokens"], _parse(text), 0.0, True)
            b, f = b + x, f + y
    elif op == "scores":
        rows = case["batch"] * HQ * case["window"]
        b = case["batch"] * HKV * case["n"] * (2.0 * D + 4.0) + rows * D * 2.0
        f = 2.0 * rows * case["n"] * D
    elif op == "compress":
        # read: every score and the kept tokens' rows; written: the packed
        # tokens and their indices
        bh, n, keep = case["batch"] * HKV, case["n"], case["keep"]
        b = bh * (keep * 4.0 * D + _stored(case["kind"], case["bits"], keep) + 4.0 * keep)
        b += bh * 4.0 * n if case["kind"] != "quant" else 0.0
        if case["then"]:
            t = case["then_keep"]
            b += bh * (4.0 * keep + _stored(case["kind"], case["bits"], t) + _stored("", case["then_bits"], t) + 4.0 * t)
        f = 0.0
    else:
        L, B, n, S = case["layers"], case["batch"], case["n"], case["steps"]
        segs = [("quant", 2, n // 10, n // 10), ("quant", 2, n - n // 10, n - n // 10)]
        one, flops = _attend_work(B, 1, segs, 0.0, False)
        packed = sum(B * HKV * _stored("quant", 2, s[2]) for s in segs)
        b = L * (B * HKV * n * 4.0 * D + packed + S * one + B * HKV * 4.0 * D * S * (S + 1) / 2)
        f = L * (2.0 * B * HQ * 32 * n * D + S * flops)
    return {"bytes": b, "flops": f}


def tolerance(case):
    # measured against exact(): outputs 1.7e-3 (their own bf16 rounding), lse and
    # masses below 2e-6, scores 4e-7; about four times that, scores ten times
    # (fp32 sums over the window in another order)
    return {"attend": {"rel": 6e-3}, "batch": {"rel": 6e-3}, "scores": {"rel": 4e-6}, "compress": "exact",
            "generate": {"rel": 6e-3}}[case["op"]]


# ------------------------------------------------------------ 64-bit values

def _group_quant(x, bits, dim):
    """x [.., G, ..] float64 holding bf16 values, groups along ``dim``: the
    values that the packed codes stand for, code * s + z."""
    x32 = x.float()
    mn, mx = x32.amin(dim, keepdim=True), x32.amax(dim, keepdim=True)
    qmax = float(2 ** bits - 1)
    s, z = ((mx - mn) / qmax).half().float(), mn.half().float()
    code = torch.round((x32 - z) / torch.where(s == 0, torch.ones_like(s), s)).clamp(0, qmax)
    code = torch.where(s == 0, torch.zeros_like(code), code)
    return code.double() * s.double() + z.double()


def _values(kk, vv, sc, kind, bits, keep):
    """What one sequence's segment stores, in float64: kk, vv [HKV, n, D] bf16, sc [HKV, n]."""
    if kind.startswith("evict"):
        idx = torch.sort(sc, dim=1, descending=True, stable=True).indices[:, :keep].sort(dim=1).values
        kk = torch.gather(kk, 1, idx[..., None].expand(-1, -1, D))
        vv = torch.gather(vv, 1, idx[..., None].expand(-1, -1, D))
    k, v = kk.double(), vv.double()
    if bits != 16:
        n = k.shape[1] // GROUP * GROUP
        kq = _group_quant(k[:, :n].reshape(HKV, -1, GROUP, D), bits, 2).reshape(HKV, n, D)
        vq = _group_quant(v[:, :n].reshape(HKV, n, D // GROUP, GROUP), bits, 3).reshape(HKV, n, D)
        k, v = torch.cat([kq, k[:, n:]], 1), torch.cat([vq, v[:, n:]], 1)
    return k, v


def _attention(q, parts):
    """q [HQ, T, D] bf16; parts: (k, v) [HKV, n, D] float64 per segment -> O, lse, mass."""
    T = q.shape[1]
    out = torch.empty((HQ, T, D), dtype=torch.float64, device=q.device)
    lse = torch.empty((HQ, T), dtype=torch.float64, device=q.device)
    mass = torch.empty((HQ, T, len(parts)), dtype=torch.float64, device=q.device)
    k, v = torch.cat([p[0] for p in parts], 1), torch.cat([p[1] for p in parts], 1)
    step = max(1, int(2e8 // max(1, T * k.shape[1])))
    for j in range(HKV):
        h0 = j * (HQ // HKV)
        for h in range(h0, h0 + HQ // HKV, step):
            e = min(h + step, h0 + HQ // HKV)
            x = q[h:e].double().reshape(-1, D) @ k[j].T / math.sqrt(D)
            lz = torch.logsumexp(x, 1)
            p = torch.exp(x - lz[:, None])
            out[h:e] = (p @ v[j]).reshape(e - h, T, D)
            lse[h:e] = lz.reshape(e - h, T)
            at = 0
            for s, part in enumerate(parts):
                n = part[0].shape[1]
                mass[h:e, :, s] = p[:, at:at + n].sum(1).reshape(e - h, T)
                at += n
    return out, lse, mass


def _attend_exact(q, kk, vv, sc, segs, spread):
    outs = []
    for b in range(q.shape[0]):
        parts, begin = [], 0
        for kind, bits, n, keep in segs:
            kb = _keeps(q.shape[0], kind, keep, spread)[b]
            parts.append(_values(kk[b, :, begin:begin + n], vv[b, :, begin:begin + n],
                                 None if sc is None else sc[b, :, begin:begin + n], kind, bits, kb))
            begin += n
        outs.append(_attention(q[b], parts))
    return [torch.stack(x) for x in zip(*outs)]


def exact(case, seed):
    op = case["op"]
    if op == "attend":
        segs, kk, vv, sc, q = _attend_inputs(case, seed)
        out, lse, mass = _attend_exact(q, kk, vv, sc, segs, case["spread"])
        return {"out": out, "lse": lse, "mass": mass} if case["stats"] else {"out": out}
    if op == "batch":
        res = []
        for i, (n, text) in enumerate(_batch_calls(case)):
            kk, vv = _kv(seed, 1, n, i)
            res.append(_attend_exact(_q(seed, 1, case["tokens"], i), kk, vv, None, _parse(text), 0.0))
        return res
    if op == "scores":
        kk, _ = _kv(seed, case["batch"], case["n"])
        q = _q(seed, case["batch"], case["window"])
        g = HQ // HKV
        out = torch.empty((case["batch"], HKV, case["n"]), dtype=torch.float64, device=DEV)
        for b in range(case["batch"]):
            for j in range(HKV):
                x = q[b, j * g:(j + 1) * g].double().reshape(-1, D) @ kk[b, j].double().T / math.sqrt(D)
                out[b, j] = torch.softmax(x, 1).sum(0)
        return out
    if op == "compress":
        return None  # codes, 16-bit parameters, indices and copied rows: the same bytes always
    k, v, qwin, q, kn, vn = _generate_inputs(case, seed)
    L, B, n, S = case["layers"], case["batch"], case["n"], case["steps"]
    n_text = n // 10
    g = HQ // HKV
    out = torch.empty((L, B, HQ, 1, D), dtype=torch.float64, device=DEV)
    mass = torch.zeros(((L + 3) // 4, B, 2), dtype=torch.float64, device=DEV)
    for l in range(L):
        size = min(4, L - l // 4 * 4)
        for b in range(B):
            for j in range(HKV):
                x = qwin[l, b, j * g:(j + 1) * g].double().reshape(-1, D) @ k[l][b, j].double().T / math.sqrt(D)
                p = torch.softmax(x, 1)
                for s, (lo, hi) in enumerate([(0, n_text), (n_text, n)]):
                    mass[l // 4, b, s] += p[:, lo:hi].sum() / (HQ * 32 * size)
            parts = [_values(k[l][b, :, lo:hi], v[l][b, :, lo:hi], None, "quant", 2, hi - lo)
                     for lo, hi in [(0, n_text), (n_text, n)]]
            parts.append((kn[:, l, b].transpose(0, 1).double(), vn[:, l, b].transpose(0, 1).double()))
            out[l, b] = _attention(q[S - 1, l, b], parts)[0]
    return {"out": out, "mass": mass}
