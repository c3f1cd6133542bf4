"""What a serving program has this library do, as cases that can be timed and compared.

Four kinds of call, each through the package's public Python entry points, with the library-owned workspace and
outputs allocated by the call, as a decode loop uses them:

  step    commit_step: LM head, softmax statistics and threshold commit of one forward's window
  decode  commit_step, then commit_sweep on the window it resolved (one whole iteration of the decode loop)
  verify  verify_step: speculative-decoding verification of n_req x (n_draft + 1) rows
  tp      one rank of a vocabulary-parallel head: lmhead_partials on its shard, its partials placed beside the other
          ranks' (what an all-gather leaves), merge_commit

Head formats: "f32", "bf16", "e4m3" (codes with a scale per row), "w8a8" (the same head with the hidden rows quantised
to E4M3 by the call) and "nvfp4" (E2M1 codes, an E4M3 scale per 16 elements, a scale per row).

Inputs: hidden states N(0, 1) and head rows N(0, 1/d), so logits are about N(0, 1), with 40% of the rows moved along one
head row so that its logit rises by 2 to 10 (18 for verification, whose targets are confident): confidences from 1e-4 to
0.99, as a partly denoised window has them.
"""

import math

import torch

import paper_2609_33887_gb300 as bdc

EPS = (0.8, 0.7, 0.6, 0.5, 0.45, 0.4, 0.3, 0.2, 0.1, 0.05, 0.02)  # typical acceptance: the settings one verification scores
E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


def _window(name, kind, head, n_seq, n_slots, block_len, masked, d, V, T, idle=0, mask_id=-1):
    """A window of n_seq sequences x n_slots slots x block_len positions; `masked` of the active slots' positions are
    still masked, the last `idle` slots of each sequence are placeholders."""
    c = {"kind": kind, "head": head, "n_seq": n_seq, "n_slots": n_slots, "block_len": block_len, "masked": masked,
         "d": d, "V": V, "T": T, "idle": idle, "mask_id": mask_id}
    return dict(c, name=name) if name else c


def _verify(name, head, n_req, n_draft, d, V):
    c = {"kind": "verify", "head": head, "n_req": n_req, "n_draft": n_draft, "d": d, "V": V}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a window and head small enough to check by hand, in exact float32: the latency of one call
        _window("f32_1x1x32_d256", "step", "f32", 1, 1, 32, 32, 256, 4096, 1),
        # a small model served in float32 to check a 16-bit deployment against
        _window("f32_2x2x32_d1024", "step", "f32", 2, 2, 32, 77, 1024, 50304, 4),
        # one request alone: the whole iteration whose latency a user of one stream sees
        _window("decode_1x2x32_bf16", "decode", "bf16", 1, 2, 32, 38, 2048, 151936, 4, mask_id=151666),
        # a few requests, ragged sizes, placeholder slots, a vocabulary that no tile divides
        _window("decode_5x3x20_bf16", "decode", "bf16", 5, 3, 20, 131, 1544, 102401, 8, idle=1, mask_id=102400),
        # the usual small serving batch
        _window("step_8x2x32_bf16", "step", "bf16", 8, 2, 32, 294, 2048, 151936, 4),
        # the same batch with the head in each of the stored precisions that save memory
        _window("step_8x2x32_e4m3", "step", "e4m3", 8, 2, 32, 294, 2048, 151936, 4),
        _window("step_8x2x32_w8a8", "step", "w8a8", 8, 2, 32, 294, 2048, 151936, 4),
        _window("step_8x2x32_nvfp4", "step", "nvfp4", 8, 2, 32, 294, 2048, 151936, 4),
        # a full serving batch of a mid-size model, sixteen operating points scored at once
        _window("step_64x4x64_bf16", "step", "bf16", 64, 4, 64, 8192, 4096, 151936, 16),
        # the largest window: 131072 positions, a large model's 8-bit head
        _window("step_256x8x64_e4m3", "step", "e4m3", 256, 8, 64, 52429, 5120, 157184, 16),
        # speculative decoding: 64 requests x (4 drafts + 1) against an 8-bit target head
        _verify("verify_64x5_e4m3", "e4m3", 64, 4, 3584, 152064),
        # the same against a bf16 head
        _verify("verify_64x5_bf16", "bf16", 64, 4, 4096, 128256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.choice(["bf16", "bf16", "bf16", "e4m3", "e4m3", "w8a8", "nvfp4", "nvfp4", "f32", "verify", "verify", "tp"])
    V = _log(rng, 32000, 157184)
    if pick == "verify":
        return _verify(None, rng.choice(["bf16", "e4m3", "nvfp4"]), _log(rng, 1, 128), rng.randint(1, 8),
                       256 * rng.randint(3, 16), V)
    L, slots = rng.randint(4, 64), rng.randint(1, 8)
    idle = rng.randint(0, slots - 1) if rng.random() < 0.4 else 0
    T = rng.randint(1, 32)
    frac = rng.uniform(0.1, 1.0)
    if pick == "f32":
        n_seq, slots, idle = _log(rng, 1, 4), min(slots, 2), 0
        d, V = _log(rng, 64, 1024), _log(rng, 1000, 50304)
    elif pick == "nvfp4":
        n_seq, d = _log(rng, 1, 32), 32 * rng.randint(16, 128)
    elif pick in ("e4m3", "w8a8"):
        n_seq, d = _log(rng, 1, 256), 16 * rng.randint(32, 320)
    else:
        n_seq, d = _log(rng, 1, 64), 8 * _log(rng, 64, 640)
    head = "bf16" if pick == "tp" else pick
    while True:
        masked = max(1, int(frac * n_seq * (slots - idle) * L))
        if n_seq == 1 or 2.0 * masked * d * V <= 2e13:
            break
        n_seq //= 2
    kind = "tp" if pick == "tp" else rng.choice(["step", "step", "decode"])
    return _window(None, kind, head, n_seq, slots, L, masked, d, V, T, idle, rng.choice([-1, V - 1, V // 3]))


# ----------------------------------------------------------------------------------------------------------- inputs --
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _round_up(x, a):
    return (x + a - 1) // a * a


def _nvfp4(w):
    """[V, d] float32 -> (codes [V, round_up(d / 2, 16)], block scales [V, round_up(d / 16, 16)], row scale [V])."""
    V, d = w.shape
    nb = (d + 15) // 16
    codes = torch.zeros(V, _round_up((d + 1) // 2, 16), dtype=torch.uint8, device=w.device)
    bscale = torch.zeros(V, _round_up(nb, 16), dtype=torch.uint8, device=w.device)
    rscale = torch.empty(V, dtype=torch.float32, device=w.device)
    mids = torch.tensor([0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0], device=w.device)
    for r0 in range(0, V, 16384):
        x = torch.nn.functional.pad(w[r0:r0 + 16384], (0, nb * 16 - d)).view(-1, nb, 16)
        amax = x.abs().amax(dim=2)
        rs = (amax.amax(dim=1) / (6.0 * 448.0)).clamp_min(1e-30)
        bs = (amax / (6.0 * rs[:, None])).to(torch.float8_e4m3fn)
        q = x / (bs.float() * rs[:, None]).clamp_min(1e-38)[:, :, None]
        code = torch.bucketize(q.abs(), mids) | ((q < 0).long() << 3)
        code = code.view(-1, nb * 16).to(torch.uint8)
        codes[r0:r0 + 16384, : nb * 8] = code[:, 0::2] | (code[:, 1::2] << 4)
        bscale[r0:r0 + 16384, :nb] = bs.view(torch.uint8)
        rscale[r0:r0 + 16384] = rs
    return codes, bscale, rscale


def _head(head, V, d, g):
    """(weight as the entry points take it, row scale or None)."""
    if head == "nvfp4":
        codes, bscale, rscale = _nvfp4(torch.randn(V, d, generator=g, device="cuda") / math.sqrt(d))
        return bdc.Nvfp4Head(codes, bscale, d), rscale
    dtype = {"f32": torch.float32, "bf16": torch.bfloat16}.get(head, torch.float8_e4m3fn)
    w = torch.empty(V, d, dtype=dtype, device="cuda")
    scale = torch.empty(V, device="cuda") if dtype == torch.float8_e4m3fn else None
    for r0 in range(0, V, 32768):
        x = torch.randn(min(32768, V - r0), d, generator=g, device="cuda") / math.sqrt(d)
        if scale is not None:
            s = x.abs().amax(dim=1) / 448.0
            scale[r0:r0 + 32768] = s
            x = x / s[:, None]
        w[r0:r0 + 32768] = x.to(dtype)
    return w, scale


def _rows(w, scale, rows):
    """The head's rows `rows` in float64, as the stored format says."""
    if isinstance(w, bdc.Nvfp4Head):
        c = w.codes[rows]
        nib = torch.stack([c & 15, c >> 4], dim=2).view(len(rows), -1)[:, : w.dim].long()
        val = torch.tensor(E2M1, device="cuda", dtype=torch.float64)[nib & 7] * (1 - 2 * (nib >> 3)).double()
        bs = w.block_scale[rows].view(torch.float8_e4m3fn).double().repeat_interleave(16, dim=1)[:, : w.dim]
        return val * bs * scale[rows, None].double()
    if w.dtype == torch.float8_e4m3fn:
        return w.view(torch.uint8)[rows].view(torch.float8_e4m3fn).double() * scale[rows, None].double()
    return w[rows].double()


def _hidden(n, d, w, scale, V, g, dtype, lo, hi, share, draft_of=None):
    h = torch.empty(n, d, dtype=dtype, device="cuda")
    tok = torch.randint(0, V, (n,), generator=g, device="cuda")
    b = lo + (hi - lo) * torch.rand(n, generator=g, device="cuda")
    b = torch.where(torch.rand(n, generator=g, device="cuda") < share, b, torch.zeros_like(b))
    for r0 in range(0, n, 8192):
        t = tok[r0:r0 + 8192]
        wr = _rows(w, scale, t).float()
        x = torch.randn(len(t), d, generator=g, device="cuda") + b[r0:r0 + 8192, None] * wr / (wr * wr).sum(1, keepdim=True)
        h[r0:r0 + 8192] = x.to(dtype)
    return h, tok


def _inputs(case, seed):
    g = _gen(seed)
    d, V, head = case["d"], case["V"], case["head"]
    w, scale = _head(head, V, d, g)
    s = {"case": case, "w": w, "scale": scale}
    dtype = torch.float32 if head == "f32" else torch.bfloat16
    if case["kind"] == "verify":
        q, D = case["n_req"], case["n_draft"]
        s["hidden"], tok = _hidden(q * (D + 1), d, w, scale, V, g, dtype, 8.0, 18.0, 1.1)
        # a draft agrees with the row's boosted entry nine times in ten
        other = torch.randint(0, V, (q, D), generator=g, device="cuda")
        agree = torch.rand(q, D, generator=g, device="cuda") < 0.9
        s["draft"] = torch.where(agree, tok.view(q, D + 1)[:, :D], other).to(torch.int32).reshape(-1).contiguous()
        return s
    B, slots, L, idle = case["n_seq"], case["n_slots"], case["block_len"], case["idle"]
    P, act = B * slots * L, slots - idle
    s["hidden"], _ = _hidden(P, d, w, scale, V, g, dtype, 2.0, 10.0, 0.4)
    mask = torch.ones(B, slots, L, dtype=torch.uint8, device="cuda")
    live = torch.zeros(B * act * L, dtype=torch.uint8, device="cuda")
    live[torch.randperm(B * act * L, generator=g, device="cuda")[: case["masked"]]] = 1
    mask[:, :act] = live.view(B, act, L)
    flags = torch.zeros(B, slots, dtype=torch.uint8, device="cuda")
    flags[:, :act] = bdc.BD_BLOCK_ACTIVE
    flags[:, 0] |= bdc.BD_BLOCK_FALLBACK_ELIGIBLE
    s["mask"], s["flags"] = mask.view(-1).contiguous(), flags.view(-1).contiguous()
    s["tau"] = [0.5 + 0.48 * k / max(1, case["T"] - 1) for k in range(case["T"])]
    if case["kind"] == "decode":
        tokens = torch.randint(0, V, (P,), generator=g, device="cuda", dtype=torch.int32)
        s["window"] = torch.where(s["mask"] != 0, torch.full_like(tokens, case["mask_id"]), tokens)
    if case["kind"] == "tp":
        # this rank holds rows [lo, hi) of the head; the other three ranks' partials, as their calls left them
        edges = [V * r // 4 for r in range(5)]
        s["lo"], s["hi"] = edges[1], edges[2]
        pos = torch.nonzero(_is_live(s)).view(-1)
        s["pm"] = torch.full((4, P), -math.inf, device="cuda")
        s["ps"] = torch.zeros(4, P, device="cuda")
        s["pa"] = torch.full((4, P), -1, dtype=torch.int32, device="cuda")
        for r in (0, 2, 3):
            x = s["hidden"][pos].float() @ w[edges[r]:edges[r + 1]].float().t()
            if edges[r] <= case["mask_id"] < edges[r + 1]:
                x[:, case["mask_id"] - edges[r]] = -math.inf
            m, a = x.max(dim=1)
            s["pm"][r, pos], s["pa"][r, pos] = m, (a + edges[r]).to(torch.int32)
            s["ps"][r, pos] = (x - m[:, None]).exp().sum(1)
    return s


def _is_live(s):
    return (s["mask"] != 0) & (s["flags"].repeat_interleave(s["case"]["block_len"]) & 1 != 0)


def prepare(case, seed):
    return _inputs(case, seed)


# -------------------------------------------------------------------------------------------------------------- run --
def run(s):
    c = s["case"]
    if c["kind"] == "verify":
        return bdc.verify_step(s["hidden"], s["w"], s["draft"], c["n_req"], c["n_draft"], EPS, weight_scale=s["scale"])
    shape = (c["n_seq"], c["n_slots"], c["block_len"])
    if c["kind"] == "tp":
        lo, hi = s["lo"], s["hi"]
        m, e, a = bdc.lmhead_partials(s["hidden"], s["w"][lo:hi], lo, s["mask"], s["flags"], *shape,
                                      mask_token_id=c["mask_id"])
        s["pm"][1], s["ps"][1], s["pa"][1] = m, e, a
        return (m, e, a) + bdc.merge_commit(s["pm"], s["ps"], s["pa"], s["mask"], s["flags"], *shape, s["tau"], counts=True)
    out = bdc.commit_step(s["hidden"], s["w"], s["mask"], s["flags"], *shape, s["tau"], weight_scale=s["scale"],
                          mask_token_id=c["mask_id"], counts=True, fp8_activations=c["head"] == "w8a8")
    if c["kind"] == "step":
        return out
    # the scheduler keeps the window it served from beside the one the sweep moves on
    window, mask, flags = s["window"].clone(), s["mask"].clone(), s["flags"].clone()
    swept = bdc.commit_sweep(window, mask, flags, *shape, out[0], out[2], c["T"] // 2, mask_token_id=c["mask_id"],
                             options=bdc.BD_SWEEP_ELIGIBLE_OLDEST)
    return out + (window, mask, flags) + swept


# ------------------------------------------------------------------------------------------------------ work, error --
def work(case):
    """The head and the rows that need a prediction read once, the masks read and the outputs written once."""
    d, V = case["d"], case["V"]
    per = {"f32": d * 4, "bf16": d * 2, "e4m3": d + 4, "w8a8": d + 4, "nvfp4": d / 2 + d / 16 + 4}[case["head"]]
    el = 4 if case["head"] == "f32" else 2
    if case["kind"] == "verify":
        rows = case["n_req"] * (case["n_draft"] + 1)
        return {"bytes": V * per + rows * d * el + 20 * rows + case["n_req"] * 48, "flops": 2.0 * rows * d * V}
    P = case["n_seq"] * case["n_slots"] * case["block_len"]
    V = V * 2 // 4 - V // 4 if case["kind"] == "tp" else V
    extra = {"step": 0, "decode": 22, "tp": 12 * 4}[case["kind"]]
    return {"bytes": V * per + case["masked"] * d * el + (13 + extra) * P, "flops": 2.0 * case["masked"] * d * V}


def tolerance(case):
    # float32 sums of up to 5120 products and of V exponentials: 2e-6 from float64 with FMA sums, up to 3.4e-5 with the
    # tensor cores' float32 accumulation. Whole values: a top-two gap or a threshold closer than that rounding moves a
    # token or a bit of one row.
    rel = 8e-6 if case["head"] == "f32" else 1.2e-4
    return {"rel": rel, "max": 10 * rel, "differ": 0.005}


# ------------------------------------------------------------------------------------------------------------ exact --
def _act(s):
    """The hidden rows as the step multiplies them, in float64: W8A8 quantises each row to E4M3 with its own scale."""
    h = s["hidden"]
    if s["case"]["head"] != "w8a8":
        return h.double()
    amax = h.float().abs().amax(dim=1, keepdim=True)
    top = torch.full_like(amax, 448.0)  # tensor by tensor: one correctly rounded division each
    code = (h.float() * (top / amax)).clamp(-448, 448).to(torch.float8_e4m3fn)
    return code.double() * (amax / top).double()


def _stats(h, s, lo, hi, mask_id, draft=None):
    """Per row of h over head rows [lo, hi): max, sum of exp(l - max), argmax, mean of (l - max), the draft's logit."""
    m = torch.full((len(h),), -math.inf, dtype=torch.float64, device="cuda")
    e, a, t, x = torch.zeros_like(m), torch.zeros_like(m).long(), torch.zeros_like(m), torch.zeros_like(m)
    for r0 in range(0, len(h), 1024):
        l = torch.empty(len(h[r0:r0 + 1024]), hi - lo, dtype=torch.float64, device="cuda")
        for v0 in range(lo, hi, 16384):
            rows = torch.arange(v0, min(hi, v0 + 16384), device="cuda")
            l[:, v0 - lo:v0 - lo + len(rows)] = h[r0:r0 + 1024] @ _rows(s["w"], s["scale"], rows).t()
        if lo <= mask_id < hi:
            l[:, mask_id - lo] = -math.inf
        sl = slice(r0, r0 + 1024)
        m[sl], a[sl] = l.max(dim=1)
        if draft is not None:
            x[sl] = l.gather(1, draft[sl].clamp_min(0)[:, None])[:, 0]
        l -= m[sl, None]
        p = l.exp()
        e[sl] = p.sum(1)
        if draft is not None:
            t[sl] = (p * l).sum(1) / e[sl]
    return m, e, a + lo, t, x


def _commit(s, tok, conf):
    """The threshold commit with the top-1 fallback: (tokens, conf, commit bits, counts)."""
    c = s["case"]
    blocks, L = c["n_seq"] * c["n_slots"], c["block_len"]
    live, cf = _is_live(s).view(blocks, L), conf.view(blocks, L)
    best = torch.where(live, cf, torch.full_like(cf, -1.0)).argmax(dim=1)
    first = torch.zeros_like(live).scatter_(1, best[:, None], True) & live
    fall = ((s["flags"] & 2) != 0) & live.any(dim=1)
    bits, counts = torch.zeros(blocks, L, dtype=torch.int64, device="cuda"), []
    for k, tau in enumerate(torch.tensor(s["tau"], dtype=torch.float32).tolist()):
        b = live & (cf >= tau)
        b = torch.where((~b.any(dim=1) & fall)[:, None], first, b)
        bits |= b.long() << k
        counts.append(b.view(c["n_seq"], -1).sum(1))
    bits = torch.where(bits >= 2 ** 31, bits - 2 ** 32, bits)
    return tok.to(torch.int32), conf, bits.view(-1).to(torch.int32), torch.stack(counts, 1).to(torch.int32)


def exact(case, seed):
    if work(case)["flops"] > 3e12:
        return None  # minutes of float64
    s = _inputs(case, seed)
    h = _act(s)
    if case["kind"] == "verify":
        q, D = case["n_req"], case["n_draft"]
        draft = torch.full((q, D + 1), -1, dtype=torch.int64, device="cuda")
        draft[:, :D] = s["draft"].view(q, D)
        draft = draft.view(-1)
        m, e, a, t, x = _stats(h, s, 0, case["V"], -1, draft)
        p = torch.where(draft >= 0, (x - m).exp() / e, torch.zeros_like(m))
        H = e.log() - t
        bits = torch.zeros_like(draft)
        for k, eps in enumerate(torch.tensor(EPS, dtype=torch.float32).double().tolist()):
            bits |= ((p > torch.minimum(torch.full_like(H, eps), math.sqrt(eps) * (-H).exp())) & (draft >= 0)).long() << k
        bits |= ((draft == a) & (draft >= 0)).long() << 31
        ok = torch.stack([(bits >> k) & 1 for k in list(range(len(EPS))) + [31]], 1).view(q, D + 1, -1)[:, :D]
        bits = torch.where(bits >= 2 ** 31, bits - 2 ** 32, bits)
        return {"tokens": a.to(torch.int32), "p_draft": p, "entropy": H, "accept": bits.to(torch.int32),
                "accepted": ok.cumprod(dim=1).sum(1).to(torch.int32)}
    live = _is_live(s)
    pos = torch.nonzero(live).view(-1)
    lo, hi = (s["lo"], s["hi"]) if case["kind"] == "tp" else (0, case["V"])
    m = torch.full((len(live),), -math.inf, dtype=torch.float64, device="cuda")
    e, a = torch.zeros_like(m), torch.full_like(m, -1).long()
    m[pos], e[pos], a[pos], _, _ = _stats(h[pos], s, lo, hi, case["mask_id"])
    if case["kind"] == "tp":
        pm, ps, pa = s["pm"].double(), s["ps"].double(), s["pa"].long()
        pm[1], ps[1], pa[1] = m, e, a
        top, r = pm.max(dim=0)
        total = (ps * (pm - top).exp()).nan_to_num(0.0).sum(0)
        tok = torch.where(live, pa.gather(0, r[None])[0], torch.full_like(a, -1))
        conf = torch.where(live, 1.0 / total, torch.zeros_like(total))
        return (m, e, a.to(torch.int32)) + _commit(s, tok, conf)
    conf = torch.where(live, 1.0 / e, torch.zeros_like(e))
    out = _commit(s, a, conf)
    return out if case["kind"] == "step" else out + (None,) * 6
