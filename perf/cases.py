"""The work that a program using libispa has it do, as cases that can be timed and compared.

A case is one call, or one short run of calls that belong together, through the public entry
points (``paper_2607_00712_gb300.abi``), with device buffers the program keeps between steps.

* ``listed()``  the named cases, each a point of a range that ``draw`` covers;
* ``prepare``   what the program holds before the call, made on the GPU from the seed alone;
* ``run``       one pass; it leaves its state so that the next pass computes the same;
* ``exact``     the same outputs in 64 bits, by plain torch;
* ``work``      the bytes and operations one pass cannot do without.

Inputs follow the recipe of the package's ``synth`` module (q, k, v ~ N(0, 1), one N(0, 0.5^2)
offset per frame and head on the keys, everything in bf16), drawn by torch's generator on the
device.
"""
import math

import torch

from paper_2607_00712_gb300 import abi
from paper_2607_00712_gb300.device import LS, Ring, Window

DEV = "cuda"
BF16, F32, F64, U8 = torch.bfloat16, torch.float32, torch.float64, torch.uint8
E4M3_MAX = 448.0
LAMBDA = 1e-3          # ridge weight of the closed-form solve (the paper's default)
MAX_ATTN_FLOPS = 3.2e12


def listed():
    m13 = dict(heads=12, head_dim=128, frame_tokens=1560)
    m14 = dict(heads=40, head_dim=128, frame_tokens=1560)
    return [
        # The smallest call: an F-layer of the tiny configuration (two heads of 64, 64 tokens per
        # frame), where launches and latency are all there is.
        dict(name="full_tiny", kind="attn", mode="full", fmt="bf16", heads=2, head_dim=64, frame_tokens=64,
             chunk_frames=2, past_frames=4, capacity=6, pinned=0, win_sink=0, win_recent=0, causal=False, lse=True),
        # The F-layer of a 1.3B-shaped chunk step: half of the layers, every denoising step.
        dict(name="full_1.3b", kind="attn", mode="full", fmt="bf16", **m13, chunk_frames=3, past_frames=18,
             capacity=18, pinned=0, win_sink=0, win_recent=0, causal=False, lse=False),
        # An L-layer of a stream that is generated frame by frame: a wrapped ring with a pinned sink
        # frame, a window of the sink and the six newest frames, one frame of queries.
        dict(name="local_frame", kind="attn", mode="local", fmt="bf16", **m13, chunk_frames=1, past_frames=17,
             capacity=10, pinned=1, win_sink=1, win_recent=6, causal=False, lse=False),
        # The warmup step of a 1.3B-shaped layer: both outputs and their discrepancy in one pass.
        dict(name="dual_1.3b", kind="attn", mode="dual", fmt="bf16", **m13, chunk_frames=3, past_frames=18,
             capacity=18, pinned=0, win_sink=0, win_recent=6, causal=False, lse=False),
        # The F-layer of a 14B-shaped chunk step: the largest call of the path.
        dict(name="full_14b", kind="attn", mode="full", fmt="bf16", **m14, chunk_frames=3, past_frames=18,
             capacity=18, pinned=0, win_sink=0, win_recent=0, causal=False, lse=False),
        # The 8-bit F-layer with all it takes: the chunk's q, k and v quantised, the attention over
        # the 8-bit ring, and the finished chunk appended to that ring.
        dict(name="kv8_1.3b", kind="attn", mode="full", fmt="kv8", **m13, chunk_frames=3, past_frames=18,
             capacity=21, pinned=0, win_sink=0, win_recent=0, causal=False, lse=False),
        # The finished chunk appended to the rings of all 30 layers (half F-layers, half L-layers)
        # in one launch, once per chunk.
        dict(name="append_1.3b", kind="append", layers=30, **m13, chunk_frames=3, cap_full=6, cap_local=4),
        # The least-squares sums of one layer over the four denoising steps of a warmup chunk.
        dict(name="ls_1.3b", kind="ls", dim=1536, tokens=4680, steps=4, exact_delta=False),
        # The same sums at the 14B width, one step.
        dict(name="ls_14b", kind="ls", dim=5120, tokens=4680, steps=1, exact_delta=False),
        # The closed-form solve of one layer, once per layer at the transition, at both widths.
        dict(name="solve_1.3b", kind="solve", dim=1536, d_out=1536, tokens=37440),
        dict(name="solve_14b", kind="solve", dim=5120, d_out=5120, tokens=37440),
        # The 8-bit output projection after the attention: activations quantised, then the GEMM.
        dict(name="w8a8_1.3b", kind="w8a8", tokens=4680, dim=1536, d_out=1536),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["attn"] * 6 + ["append", "ls", "ls", "solve", "w8a8", "w8a8"])
    if kind == "attn":
        mode = rng.choice(["full", "full", "local", "dual"])
        fmt = rng.choice(["bf16", "bf16", "bf16", "kv8", "qk8"])
        head_dim = 128 if fmt != "bf16" else rng.choice([64, 128, 128, 128])
        while True:
            heads, chunk = rng.choice([2, 4, 8, 12, 16, 24, 40]), rng.randint(1, 3)
            tokens = _log(rng, 60, 1600)
            if fmt == "kv8":
                tokens = (tokens + 3) // 4 * 4     # the d-major value ring wants multiples of 4
            pinned = rng.choice([0, 1])
            capacity = rng.randint(max(4, chunk + pinned), 24)
            # an 8-bit case also appends its chunk, so its ring has the room; the others may have wrapped
            past = rng.randint(1, max(1, capacity - chunk)) if fmt != "bf16" else rng.randint(1, capacity + 8)
            recent = rng.randint(1, min(6, capacity - pinned))
            case = dict(kind="attn", mode=mode, fmt=fmt, heads=heads, head_dim=head_dim, frame_tokens=tokens,
                        chunk_frames=chunk, past_frames=past, capacity=capacity, pinned=pinned, win_sink=pinned,
                        win_recent=recent, causal=fmt == "bf16" and rng.random() < 0.25, lse=rng.random() < 0.3)
            if work(case)["flops"] <= MAX_ATTN_FLOPS:
                return case
    if kind == "append":
        return dict(kind="append", layers=rng.randint(1, 30), heads=rng.choice([2, 4, 8, 12, 16]),
                    head_dim=rng.choice([64, 128]), frame_tokens=_log(rng, 60, 1600), chunk_frames=rng.randint(1, 3),
                    cap_full=rng.randint(4, 6), cap_local=4)
    if kind == "ls":
        return dict(kind="ls", dim=128 * _log(rng, 2, 40), tokens=_log(rng, 60, 4800), steps=rng.randint(1, 4),
                    exact_delta=rng.random() < 0.3)
    if kind == "solve":
        dim = 128 * _log(rng, 2, 24)
        return dict(kind="solve", dim=dim, d_out=rng.choice([dim, dim, dim + 96, dim // 2 + 8]),
                    tokens=dim * rng.randint(3, 8))
    return dict(kind="w8a8", tokens=_log(rng, 40, 9400), dim=128 * _log(rng, 4, 40), d_out=128 * _log(rng, 4, 40))


# ---------------------------------------------------------------- key sets of an attention case
def _resident(c):
    """Past frames still in the ring, in order."""
    n, cap, pin = c["past_frames"], c["capacity"], c["pinned"]
    return [f for f in range(n) if f < pin or n - f <= cap - pin]


def _local(c):
    n = c["past_frames"]
    return [f for f in _resident(c) if f < c["win_sink"] or f >= n - c["win_recent"]]


def _seen(c):
    """Past frames whose keys the pass visits."""
    return _local(c) if c["mode"] == "local" else _resident(c)


def _chunk_pairs(c):
    """Visible (query, key) pairs inside the chunk."""
    n, P = c["chunk_frames"], c["frame_tokens"]
    return P * P * (n * (n + 1) // 2 if c["causal"] else n * n)


# ---------------------------------------------------------------- work
def work(case):
    k = case["kind"]
    if k == "attn":
        H, d, P = case["heads"], case["head_dim"], case["frame_tokens"]
        nq, past = case["chunk_frames"] * P, len(_seen(case)) * P
        flops = 4.0 * d * H * (nq * past + _chunk_pairs(case))
        row = H * d
        out = nq * row * 2 * (2 if case["mode"] == "dual" else 1)
        if case["fmt"] == "bf16":
            return {"bytes": 3 * nq * row * 2 + past * row * 4 + out, "flops": flops}
        key = 2 if case["fmt"] == "kv8" else 3     # bytes of one ring key and value
        # bf16 chunk in, the ring's past read, the codes of q, k (and v), the output, the appended chunk
        return {"bytes": 3 * nq * row * 2 + past * row * key + nq * row * key + out + nq * row * key, "flops": flops}
    if k == "append":
        n = case["layers"] * case["chunk_frames"] * case["frame_tokens"] * case["heads"] * case["head_dim"]
        return {"bytes": 2 * 2 * 2 * n, "flops": 0}
    if k == "ls":
        D, T, s = case["dim"], case["tokens"], case["steps"]
        return {"bytes": s * 2 * T * D * 2 + 4 * (2 * D * D + D), "flops": s * 2.0 * T * (2.0 * D * D + D)}
    if k == "solve":
        D, n = case["dim"], case["d_out"]
        # factorisation, X W and S W, two triangular solves; G, X and S read, W read, dW written
        return {"bytes": 4 * (2 * D * D + D) + 8 * D * n, "flops": D ** 3 / 3 + 4.0 * D * D * n + 2.0 * D * D * n}
    T, D, n = case["tokens"], case["dim"], case["d_out"]
    return {"bytes": T * D * 2 + T * D + 4 * T + n * D + 4 * n + T * n * 2, "flops": 2.0 * T * D * n}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=F32)


def _keys(g, frames, P, H, d):
    k = _normal(g, frames, P, H, d)
    k += 0.5 * _normal(g, frames, 1, H, d)
    return k.to(BF16).reshape(frames * P, H, d)


def _attn_inputs(c, seed):
    """The chunk's q, k, v and the past frames' k, v in order, bf16 [tokens][H][d]."""
    g = _gen(seed)
    P, H, d, n = c["frame_tokens"], c["heads"], c["head_dim"], c["chunk_frames"]
    q = _normal(g, n * P, H, d).to(BF16)
    k = _keys(g, n, P, H, d)
    v = _normal(g, n * P, H, d).to(BF16)
    k_past = _keys(g, c["past_frames"], P, H, d)
    v_past = _normal(g, c["past_frames"] * P, H, d).to(BF16)
    return q, k, v, k_past, v_past


def _head_scale(x):
    """One fp32 e4m3 scale per head, from the first frames' largest magnitude."""
    return (x.float().abs().amax(dim=(0, 2)) / E4M3_MAX).contiguous()


def _calibration(c, past):
    return _head_scale(past[:c["frame_tokens"]])


def _activations(g, T, D):
    """A_loc and A_full of T tokens: A_full = A_loc + 0.5 N(0, 1)."""
    a = _normal(g, T, D).to(BF16)
    return a, (a.float() + 0.5 * _normal(g, T, D)).to(BF16)


def _solve_inputs(c, seed):
    """A least-squares state of the warmup (the blocks the solve reads) and the projection weight.

    The features of attention outputs differ in size; a log-normal factor per feature stands for it."""
    g = _gen(seed)
    D, T = c["dim"], c["tokens"]
    spread = torch.exp(0.5 * _normal(g, D))
    gram = torch.zeros(2 * D, 2 * D, dtype=F32, device=DEV)
    for t0 in range(0, T, 4096):
        n = min(4096, T - t0)
        a = _normal(g, n, D) * spread
        delta = 0.5 * _normal(g, n, D) * spread + 0.2 * a
        ad = torch.cat([a, delta], 1)
        gram[:D].addmm_(a.t(), ad)
        gram[D:, D:].addmm_(delta.t(), delta)
    W = _normal(g, D, c["d_out"]) / math.sqrt(D)
    return gram, W.contiguous()


def _w8a8_inputs(c, seed):
    g = _gen(seed)
    x = _normal(g, c["tokens"], c["dim"]).to(BF16)
    W = _normal(g, c["dim"], c["d_out"]) / math.sqrt(c["dim"])
    # the weight codes a program keeps: one scale per output channel, codes [d_out][dim]
    amax = W.abs().amax(dim=0)
    scale = (amax / E4M3_MAX).contiguous()
    codes = (W * (E4M3_MAX / amax)).t().clamp(-E4M3_MAX, E4M3_MAX).contiguous().to(torch.float8_e4m3fn)
    return x, codes, scale


# ---------------------------------------------------------------- states
def _prepare_attn(c, seed):
    q, k, v, k_past, v_past = _attn_inputs(c, seed)
    P, H, d, n = c["frame_tokens"], c["heads"], c["head_dim"], c["chunk_frames"]
    fmt, nq, D = c["fmt"], n * P, H * d
    ring = Ring(H, d, P, c["capacity"], c["pinned"], DEV, k_e4m3=fmt == "qk8", kv_e4m3=fmt == "kv8")
    s = dict(case=c, ring=ring, q=q, k=k, v=v, win=Window(c["win_sink"], c["win_recent"]))
    if fmt != "bf16":
        s["k_scale"], s["v_scale"] = _calibration(c, k_past), _calibration(c, v_past)
    step = min(3, c["capacity"] - c["pinned"])
    for f in range(0, c["past_frames"], step):
        m = min(step, c["past_frames"] - f)
        _append(s, k_past[f * P:(f + m) * P], v_past[f * P:(f + m) * P], m)
    s["out"] = torch.empty(nq, D, dtype=BF16, device=DEV)
    s["lse"] = torch.empty(H, nq, dtype=F32, device=DEV) if c["lse"] else None
    if c["mode"] == "dual":
        s["loc"] = torch.empty(nq, D, dtype=BF16, device=DEV)
        s["lse_loc"] = torch.empty(H, nq, dtype=F32, device=DEV) if c["lse"] else None
        s["disc"] = torch.empty(nq, dtype=F32, device=DEV)
        s["disc_sum"] = torch.zeros(1, dtype=F32, device=DEV)
        s["ws_bytes"] = abi.ispa_attn_dual_workspace_size(H, nq)
        s["ws"] = torch.empty(s["ws_bytes"], dtype=U8, device=DEV)
    if fmt != "bf16":
        s["q8"] = torch.empty(nq, H, d, dtype=U8, device=DEV)
        s["q_scale"] = torch.empty(H, (nq + 127) // 128, dtype=F32, device=DEV)
        s["k8"] = torch.empty(nq, H, d, dtype=U8, device=DEV)
        if fmt == "kv8":
            s["vt_ld"] = (nq + 15) // 16 * 16
            s["vt8"] = torch.zeros(H, d, s["vt_ld"], dtype=U8, device=DEV)
    torch.cuda.synchronize()
    return s


def _append(s, k, v, n, stream=None):
    ring, fmt = s["ring"].c, s["case"]["fmt"]
    if fmt == "bf16":
        abi.ispa_kv_append(ring, k, v, n, stream)
    elif fmt == "qk8":
        abi.ispa_kv_append_qk8(ring, k, v, n, s["k_scale"], stream)
    else:
        abi.ispa_kv_append_kv8(ring, k, v, n, s["k_scale"], s["v_scale"], stream)


def prepare(case, seed):
    k = case["kind"]
    if k == "attn":
        return _prepare_attn(case, seed)
    if k == "append":
        g = _gen(seed)
        P, H, d, n, L = (case[x] for x in ("frame_tokens", "heads", "head_dim", "chunk_frames", "layers"))
        rings = [Ring(H, d, P, case["cap_full"] if i % 2 == 0 else case["cap_local"], 1, DEV) for i in range(L)]
        arr = (abi.KVRing * L)(*[r.c for r in rings])
        ks = [_normal(g, n * P, H, d).to(BF16) for _ in range(L)]
        vs = [_normal(g, n * P, H, d).to(BF16) for _ in range(L)]
        for i in range(L):
            arr[i].frames_written = 5      # the stream is past its first frames: the slots wrap
        return dict(case=case, rings=rings, arr=arr, k=ks, v=vs)
    if k == "ls":
        g = _gen(seed)
        D, T = case["dim"], case["tokens"]
        pairs = [_activations(g, T, D) for _ in range(case["steps"])]
        n = abi.ispa_ls_accumulate_workspace_size(D, T)
        return dict(case=case, pairs=pairs, ls=LS(D, DEV), ws=torch.empty(n, dtype=U8, device=DEV), ws_bytes=n)
    if k == "solve":
        gram, W = _solve_inputs(case, seed)
        D, d_out = case["dim"], case["d_out"]
        n = abi.ispa_ls_solve_workspace_size(D, d_out)
        return dict(case=case, gram=gram, state=abi.LSState(D, 0, case["tokens"], gram.data_ptr()), W=W,
                    dW=torch.empty(D, d_out, dtype=F32, device=DEV), ws=torch.empty(n, dtype=U8, device=DEV),
                    ws_bytes=n)
    x, codes, scale = _w8a8_inputs(case, seed)
    T, D, n = case["tokens"], case["dim"], case["d_out"]
    return dict(case=case, x=x, w8=codes.view(U8), w_scale=scale, x8=torch.empty(T, D, dtype=U8, device=DEV),
                x_scale=torch.empty(T, dtype=F32, device=DEV), out=torch.empty(T, n, dtype=BF16, device=DEV))


# ---------------------------------------------------------------- one pass
def _run_bf16(s, st):
    c, ring, nq = s["case"], s["ring"].c, s["q"].shape[0]
    flags = abi.ISPA_ATTN_FRAME_CAUSAL if c["causal"] else 0
    if c["mode"] == "full":
        abi.ispa_attn_full_ex(ring, s["q"], s["k"], s["v"], nq, 0.0, flags, s["out"], s["lse"], st)
        return dict(out=s["out"], lse=s["lse"])
    if c["mode"] == "local":
        abi.ispa_attn_local_ex(ring, s["win"], s["q"], s["k"], s["v"], nq, 0.0, flags, s["out"], s["lse"], st)
        return dict(out=s["out"], lse=s["lse"])
    s["disc_sum"].zero_()
    abi.ispa_attn_dual_ex(ring, s["win"], s["q"], s["k"], s["v"], nq, 0.0, flags, s["out"], s["loc"], s["disc"],
                          s["disc_sum"], s["lse"], s["lse_loc"], s["ws"], s["ws_bytes"], st)
    return dict(out=s["out"], loc=s["loc"], disc=s["disc"], disc_sum=s["disc_sum"], lse=s["lse"],
                lse_loc=s["lse_loc"])


def _run_8bit(s, st):
    c, ring, q = s["case"], s["ring"].c, s["q"]
    nq, H, d = q.shape
    kv8 = c["fmt"] == "kv8"
    ring.frames_written = c["past_frames"]     # the step is run again on the same chunk
    abi.ispa_quantize_q_e4m3(q, nq, H, d, s["q8"], s["q_scale"], st)
    abi.ispa_quantize_k_e4m3(s["k"], nq, H, d, s["k_scale"], s["k8"], st)
    head = (ring, s["k_scale"])
    tail = (s["q8"], s["q_scale"], s["k8"], s["k_scale"], s["v"])
    if kv8:
        abi.ispa_quantize_vt_e4m3(s["v"], nq, H, d, s["v_scale"], s["vt8"], s["vt_ld"], st)
        head = (ring, s["k_scale"], s["v_scale"])
        tail = (s["q8"], s["q_scale"], s["k8"], s["k_scale"], s["vt8"], s["vt_ld"])
    out = dict(out=s["out"], lse=s["lse"], q8=s["q8"], q_scale=s["q_scale"], k8=s["k8"])
    if c["mode"] == "full":
        call = abi.ispa_attn_full_kv8 if kv8 else abi.ispa_attn_full_qk8
        call(*head, *tail, nq, 0.0, s["out"], s["lse"], st)
    elif c["mode"] == "local":
        call = abi.ispa_attn_local_kv8 if kv8 else abi.ispa_attn_local_qk8
        call(*head, s["win"], *tail, nq, 0.0, s["out"], s["lse"], st)
    else:
        s["disc_sum"].zero_()
        call = abi.ispa_attn_dual_kv8 if kv8 else abi.ispa_attn_dual_qk8
        call(*head, s["win"], *tail, nq, 0.0, s["out"], s["loc"], s["disc"], s["disc_sum"], s["lse"], s["lse_loc"],
             s["ws"], s["ws_bytes"], st)
        out.update(loc=s["loc"], disc=s["disc"], disc_sum=s["disc_sum"], lse_loc=s["lse_loc"])
    _append(s, s["k"], s["v"], c["chunk_frames"], st)
    out.update(ring_k=s["ring"].k, ring_v=s["ring"].v)
    if kv8:
        out["vt8"] = s["vt8"]
    return out


def run(state):
    s, c = state, state["case"]
    st = torch.cuda.current_stream()
    if c["kind"] == "attn":
        return _run_bf16(s, st) if c["fmt"] == "bf16" else _run_8bit(s, st)
    if c["kind"] == "append":
        for r in s["arr"]:
            r.frames_written = 5
        abi.ispa_kv_append_layers(s["arr"], s["k"], s["v"], c["chunk_frames"], st)
        return dict(k=[r.k for r in s["rings"]], v=[r.v for r in s["rings"]])
    if c["kind"] == "ls":
        abi.ispa_ls_state_reset(s["ls"].c, st)
        flags = abi.ISPA_LS_EXACT_DELTA if c["exact_delta"] else 0
        for a_loc, a_full in s["pairs"]:
            abi.ispa_ls_accumulate_ex(s["ls"].c, a_loc, a_full, c["tokens"], flags, s["ws"], s["ws_bytes"], st)
        return dict(gram=s["ls"].gram)
    if c["kind"] == "solve":
        eps = abi.ispa_ls_solve(s["state"], s["W"], c["d_out"], LAMBDA, s["dW"], s["ws"], s["ws_bytes"], st)
        return dict(dW=s["dW"], eps=eps)
    T, D, n = c["tokens"], c["dim"], c["d_out"]
    abi.ispa_quantize_rows_e4m3(s["x"], T, D, s["x8"], s["x_scale"], st)
    abi.ispa_linear_w8a8(s["x8"], s["x_scale"], s["w8"], s["w_scale"], T, D, n, s["out"], st)
    return dict(x8=s["x8"], x_scale=s["x_scale"], out=s["out"])


# ---------------------------------------------------------------- 64 bits
def _e4m3(x, inv):
    """Codes of x * inv (fp32), as the fp64 values they stand for."""
    return (x.float() * inv).clamp(-E4M3_MAX, E4M3_MAX).to(torch.float8_e4m3fn).to(F64)


def _dequant_heads(x, scale):
    """[n][H][d] after coding with one scale per head."""
    inv = (1.0 / scale)[None, :, None]
    return _e4m3(x, inv) * scale.to(F64)[None, :, None]


def _dequant_q(q):
    """[n][H][d] after coding with one scale per head and 128 tokens."""
    out = torch.empty(q.shape, dtype=F64, device=DEV)
    for t in range(0, q.shape[0], 128):
        b = q[t:t + 128]
        scale = _head_scale(b)
        out[t:t + 128] = _dequant_heads(b, torch.where(scale == 0, torch.ones_like(scale), scale))
    return out


def _attend(q, k, v, c, past):
    """Softmax attention of one head in 64 bits; the last keys are the chunk's.  Output, LSE."""
    nq, P = q.shape[0], c["frame_tokens"]
    out = torch.empty_like(q)
    lse = torch.empty(nq, dtype=F64, device=DEV)
    for r in range(0, nq, 2048):
        s = (q[r:r + 2048] @ k.t()) / math.sqrt(q.shape[1])
        if c["causal"]:
            frame = torch.arange(r, min(nq, r + 2048), device=DEV) // P
            key = torch.arange(k.shape[0] - past, device=DEV) // P
            s[:, past:].masked_fill_(key[None, :] > frame[:, None], -math.inf)
        m = s.amax(dim=1, keepdim=True)
        s.sub_(m).exp_()
        z = s.sum(dim=1, keepdim=True)
        out[r:r + 2048] = (s @ v) / z
        lse[r:r + 2048] = (m + z.log())[:, 0]
    return out, lse


def _exact_attn(c, seed):
    q, k, v, k_past, v_past = _attn_inputs(c, seed)
    P, H, d, nq = c["frame_tokens"], c["heads"], c["head_dim"], q.shape[0]
    if c["fmt"] != "bf16":
        ks, vs = _calibration(c, k_past), _calibration(c, v_past)
        q, k, k_past = _dequant_q(q), _dequant_heads(k, ks), _dequant_heads(k_past, ks)
        if c["fmt"] == "kv8":
            v, v_past = _dequant_heads(v, vs), _dequant_heads(v_past, vs)

    def attend(frames):
        o = torch.empty(nq, H, d, dtype=F64, device=DEV)
        lse = torch.empty(H, nq, dtype=F64, device=DEV)
        rows = torch.cat([torch.arange(f * P, (f + 1) * P, device=DEV) for f in frames]) if frames else \
            torch.empty(0, dtype=torch.int64, device=DEV)
        for h in range(H):
            kh = torch.cat([k_past[rows, h].to(F64), k[:, h].to(F64)])
            vh = torch.cat([v_past[rows, h].to(F64), v[:, h].to(F64)])
            o[:, h], lse[h] = _attend(q[:, h].to(F64), kh, vh, c, rows.numel())
        return o.reshape(nq, H * d), lse

    full, lse = attend(_seen(c))
    out = dict(out=full, lse=lse if c["lse"] else None)
    if c["mode"] == "dual":
        loc, lse_loc = attend(_local(c))
        disc = (full - loc).square().sum(dim=1)
        out.update(loc=loc, disc=disc.sqrt(), disc_sum=disc.sum().reshape(1), lse_loc=lse_loc if c["lse"] else None)
    if c["fmt"] != "bf16":
        out.update(q8=None, q_scale=None, k8=None, ring_k=None, ring_v=None)
        if c["fmt"] == "kv8":
            out["vt8"] = None
    return out


def _maintained(D):
    """The parts of the [2D][2D] state that hold sums (1) and the rest, which stays zero (0)."""
    nb = D // 128
    up = torch.ones(nb, nb, dtype=F64, device=DEV).triu()
    if D % 256 == 0:
        i = torch.arange(0, nb, 2, device=DEV)
        up[i + 1, i] = 1.0
    up = up.repeat_interleave(128, 0).repeat_interleave(128, 1)
    return torch.cat([torch.cat([up, torch.ones_like(up)], 1), torch.cat([torch.zeros_like(up), up], 1)], 0)


def _exact_ls(c, seed):
    g = _gen(seed)
    D, T = c["dim"], c["tokens"]
    gram = torch.zeros(2 * D, 2 * D, dtype=F64, device=DEV)
    for _ in range(c["steps"]):
        a, f = _activations(g, T, D)
        ad = torch.cat([a.to(F64), f.to(F64) - a.to(F64)], 1)
        gram.addmm_(ad.t(), ad)
    return dict(gram=(gram * _maintained(D)).reshape(-1))


def _exact_solve(c, seed):
    gram, W = _solve_inputs(c, seed)
    D = c["dim"]

    def sym(m):
        return m.triu() + m.triu(1).t()

    G, X, S = sym(gram[:D, :D].to(F64)), gram[:D, D:].to(F64), sym(gram[D:, D:].to(F64))
    W = W.to(F64)
    rhs = X @ W
    L = torch.linalg.cholesky(G + LAMBDA * torch.eye(D, dtype=F64, device=DEV))
    dW = torch.cholesky_solve(rhs, L)
    eps = (dW * (G @ dW)).sum() - 2 * (dW * rhs).sum() + (W * (S @ W)).sum()
    return dict(dW=dW, eps=float(eps))


def exact(case, seed):
    k = case["kind"]
    if k == "attn":
        return _exact_attn(case, seed)
    if k == "append":
        return None      # copies: the bytes themselves
    if k == "ls":
        return _exact_ls(case, seed)
    if k == "solve":
        return _exact_solve(case, seed)
    x, codes, w_scale = _w8a8_inputs(case, seed)
    amax = x.float().abs().amax(dim=1)
    a = _e4m3(x, (E4M3_MAX / amax)[:, None]) * (amax / E4M3_MAX).to(F64)[:, None]
    y = a @ (codes.to(F64) * w_scale.to(F64)[:, None]).t()
    return dict(x8=None, x_scale=None, out=y)
