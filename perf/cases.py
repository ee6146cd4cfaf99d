"""The calls a user of this framework makes, as cases to time: whole replayed steps, loss evaluation, and the groups of
C-ABI calls that replay or audit one part of a step (linears, attention, LM head and loss, reductions, update and hash).

Sizes are the repository's own configurations (the 1B-shaped decoder, the paper's block, the kernel-level workloads, the
smoke step) and odd or ragged sizes in between.  Every result is defined to the bit, so every case is compared exactly."""
import math

import numpy as np
import torch

import paper_2609_17380_b200 as det
from paper_2609_17380_b200 import step as dstep

F32, I32, I16, I8 = torch.float32, torch.int32, torch.int16, torch.int8


def listed():
    return [
        # the smoke step: one narrow layer, two micro-batches; what is run to check an installation or bisect a mismatch,
        # and the smallest calls the driver makes
        dict(name="step_miniature", kind="step", block="plain", layers=1, d=256, kv=2, ffn=512, vocab=512, seq=128, mb=1,
             accum=1, shard=2, rep=1, arith=1),
        # one micro-batch step of the 1B-shaped decoder at full width (sequence 2048, micro-batch 4, vocabulary 50304),
        # eight of its 24 layers so that several states fit the card
        dict(name="step_1b_8_layers", kind="step", block="plain", layers=8, d=2048, kv=16, ffn=8192, vocab=50304, seq=2048,
             mb=4, accum=1, shard=1, rep=1, arith=1),
        # the paper's block (grouped queries, QK-norm, RoPE, embedding norm, sliding windows with every fifth layer full,
        # int8 P.V, fixed-point query gradient, z-loss) at its sequence length and vocabulary, one sequence
        dict(name="step_paper_5_layers", kind="step", block="paper", layers=5, d=2048, kv=4, ffn=5632, vocab=128256, seq=4096,
             mb=1, accum=1, shard=1, rep=1, arith=1),
        # a medium model in arithmetic version 2 (LM head and its gradients on the int8 tensor cores), four micro-batches
        dict(name="step_v2_medium", kind="step", block="plain", layers=4, d=1024, kv=8, ffn=2816, vocab=32768, seq=1024, mb=1,
             accum=2, shard=2, rep=1, arith=2),
        # evaluation: the loss of one short ragged batch under a medium model, forward only
        dict(name="eval_medium", kind="eval", block="plain", layers=6, d=1024, kv=8, ffn=2816, vocab=16384, seq=832, mb=2,
             accum=1, shard=1, rep=1, arith=1),
        # a single quantised linear, forward and backward, 256 tokens 512 -> 512: latency
        dict(name="linear_single", kind="linear", m=256, shapes="512x512", hb=128),
        # the 1B-shaped linear set (QKV, output, gate/up, down) at 16384 tokens, forward and backward
        dict(name="linear_set_16k", kind="linear", m=16384, shapes="6144x2048,2048x2048,16384x2048,2048x8192", hb=128),
        # causal attention forward and backward, two ragged sequences, eight heads
        dict(name="attention_ragged", kind="attention", mode="plain", b=2, h=8, kv=8, s=1088, window=0),
        # attention of a local layer of the paper's block: grouped heads, window 512, both integer devices
        dict(name="attention_window", kind="attention", mode="integer", b=1, h=16, kv=4, s=4096, window=512),
        # LM head and cross-entropy, forward and backward, for a short stretch of tokens over the full vocabulary
        dict(name="head_loss_short", kind="head", m=384, vocab=50304, d=2048, z=1e-4, arith=1),
        # the order-fixed reductions: RMSNorm forward and backward on 16384 x 2048 f32, cross-entropy of 4096 x 50304
        # logits, global gradient norm over 1.2e9 values
        dict(name="reductions", kind="reductions", dtype="f32", rows=16384, d=2048, xrows=4096, vocab=50304, n=1200000000),
        # the end of a step: eight gradient pushes in mesh order (2,2,2), clip, AdamW and the state hashes of a small model
        # with many tensors
        dict(name="update_and_hash", kind="update", layers=12, d=1024, ffn=2816, vocab=16384, accum=2, shard=2, rep=2),
    ]


def _log(rng, lo, hi, unit):
    """A multiple of unit, spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / unit)) * unit))


def _draw(rng):
    kind = rng.choice(["step", "step", "eval", "linear", "linear", "attention", "attention", "head", "reductions", "update"])
    if kind in ("step", "eval"):
        paper = kind == "step" and rng.random() < 0.35
        d = 128 * rng.choice([2, 4, 6, 8, 12, 16])
        heads = d // 128
        seq, mb = 64 * rng.randrange(2, 33), rng.choice([1, 2, 4])
        if seq % 128 and mb % 2:                 # tokens of a micro-batch come in multiples of 128
            seq += 64
        return dict(kind=kind, block="paper" if paper else "plain", layers=rng.randrange(1, 7), d=d,
                    kv=(heads // 2 if heads % 4 else heads // 4) if paper else heads, ffn=_log(rng, 256, 8192, 128),
                    vocab=_log(rng, 512, 50304, 128), seq=seq, mb=mb, accum=rng.choice([1, 2]) if kind == "step" else 1,
                    shard=rng.choice([1, 2]) if kind == "step" else 1, rep=1, arith=2 if not paper and rng.random() < 0.25 else 1)
    if kind == "linear":
        pairs = ["%dx%d" % (_log(rng, 256, 16384, 128), _log(rng, 256, 8192, 128)) for _ in range(rng.choice([1, 1, 4]))]
        return dict(kind=kind, m=_log(rng, 128, 16384, 128), shapes=",".join(pairs), hb=rng.choice([128, 128, 128, 0]))
    if kind == "attention":
        mode = rng.choice(["plain", "plain", "integer", "v2"])
        h = rng.choice([2, 4, 8, 12, 16])
        s = 64 * int(round(math.exp(rng.uniform(math.log(2), math.log(64)))))
        if mode == "v2":
            return dict(kind=kind, mode=mode, b=rng.choice([1, 2, 4]), h=h, kv=h, s=max(128, s // 128 * 128), window=0)
        return dict(kind=kind, mode=mode, b=rng.choice([1, 2, 3, 4]), h=h, kv=h // rng.choice([1, 1, 2]), s=s,
                    window=rng.choice([0, 0, 0, 128, 256, 512]))
    if kind == "head":
        return dict(kind=kind, m=_log(rng, 128, 8192, 128), vocab=_log(rng, 512, 50304, 128), d=128 * rng.randrange(2, 17),
                    z=rng.choice([0.0, 1e-4]), arith=rng.choice([1, 1, 2]))
    if kind == "reductions":
        return dict(kind=kind, dtype=rng.choice(["f32", "bf16"]), rows=_log(rng, 64, 16384, 1), d=8 * _log(rng, 16, 512, 1),
                    xrows=_log(rng, 64, 8192, 1), vocab=_log(rng, 512, 50304, 4), n=_log(rng, 1000, 1200000000, 1))
    return dict(kind=kind, layers=rng.randrange(1, 13), d=128 * rng.randrange(1, 13), ffn=_log(rng, 256, 4096, 128),
                vocab=_log(rng, 512, 32768, 128), accum=rng.choice([1, 2, 3]), shard=rng.choice([1, 2]), rep=rng.choice([1, 2, 3]))


def _seconds(case):
    w = work(case)
    return max(w["bytes"] / 6e12, w["flops"] / 60e12)


def draw(rng):
    most = max(_seconds(c) for c in listed())
    while True:
        case = _draw(rng)
        if _seconds(case) <= most:
            return case


# ---- inputs ---------------------------------------------------------------------------------------------------------
def _config(case):
    kw = dict(n_layers=case["layers"], d_model=case["d"], n_heads=case["d"] // 128, ffn=case["ffn"], vocab=case["vocab"],
              seq=case["seq"], micro_batch=case["mb"], mesh=(case["accum"], case["shard"], case["rep"]), lr=1e-5,
              arith=case["arith"])
    if case["block"] == "paper":
        ang = np.arange(case["seq"], dtype=np.float64)[:, None] * (5.0e5 ** (-2.0 * np.arange(64, dtype=np.float64) / 128))[None, :]
        kw.update(n_kv_heads=case["kv"], qk_norm=True, embed_norm=True, window=512, full_every=5, z_weight=1e-4, pv_int8=True,
                  dq_fixed=True, rope_tables=(np.cos(ang).astype(np.float32), np.sin(ang).astype(np.float32)))
    return dstep.ModelConfig(**kw)


def _bf16(g, n, std=1.0):
    return (torch.randn(n, generator=g, device="cuda") * std).to(torch.bfloat16).view(I16)


def _f32(g, n, std=1.0):
    return torch.randn(n, generator=g, device="cuda").mul_(std)


def _empty(n, dtype=F32):
    return torch.empty(n, dtype=dtype, device="cuda")


def _ws(nbytes):
    return torch.empty(int(nbytes) + 256, dtype=torch.uint8, device="cuda")


def _roots(hashes):
    return np.frombuffer(bytes.fromhex("".join(hashes.values())), np.uint8)


def _prepare_step(case, seed, g):
    r = dstep.Replay(_config(case))
    r.init_params_on_device(seed)
    n_mb = case["accum"] * case["shard"] * case["rep"]
    tok = torch.randint(0, case["vocab"], (n_mb, case["mb"], case["seq"] + 1), generator=g, device="cuda", dtype=I32)
    r.calibrate(tok[0])
    return dict(r=r, tok=tok)


def _run_step(s):
    """One optimizer step; the caller counts the steps."""
    r = s["r"]
    res = r.step(s["tok"])
    r.cfg.step += 1
    return dict(params=r.pbf, steps=r.sx, m=r.m, v=r.v, grad=r.gout, losses=res["losses"], norm=res["grad_norm"],
                status=res["status"], roots=_roots(res["hashes"]))


def _run_eval(s):
    r = s["r"]
    r.forward(s["tok"][0])
    return dict(loss=r.loss_mean, rows=r.loss_row, lse=r.lse_x, logits=r.logits)


def _prepare_linear(case, seed, g):
    m, jobs = case["m"], []
    for shape in case["shapes"].split(","):
        n, k = (int(v) for v in shape.split("x"))
        j = dict(m=m, n=n, k=k, hb=case["hb"], X=_bf16(g, m * k), W=_bf16(g, n * k, 0.02), dY=_bf16(g, m * n, 0.01), s_w=_empty(n),
                 s_x=_empty(1), s_u=_empty(1), qW=_empty(n * k, I8), qWt=_empty(n * k, I8), qX=_empty(m * k, I8), Y=_empty(m * n, I16),
                 dX=_empty(m * k, I16), dW=_empty(n * k), ds=_empty(1))
        j["ws"] = _ws(max(det.det_linear_bwd_ws_bytes(m, n, k), det.det_lsq_act_scale_init_ws_bytes(m * k),
                          det.det_lsq_weight_scale_ws_bytes(n, k), det.det_lsq_quantize_weight_ws_bytes(n, k)))
        det.det_lsq_weight_scale(j["W"], n, k, 0, j["s_w"], j["ws"])
        det.det_lsq_act_scale_init(j["X"], m * k, j["s_x"], j["ws"])
        det.det_lsq_quantize_weight(j["W"], j["s_w"], n, k, case["hb"], j["qW"], j["qWt"], j["s_u"], j["ws"])
        jobs.append(j)
    return dict(jobs=jobs, status=torch.zeros(1, dtype=I32, device="cuda"))


def _run_linear(s):
    for j in s["jobs"]:
        det.det_linear_fwd(j["X"], j["qW"], j["s_x"], j["s_w"], j["m"], j["n"], j["k"], j["Y"], j["qX"], s["status"])
    for j in s["jobs"]:
        det.det_linear_bwd(j["dY"], j["X"], j["qX"], j["W"], j["qWt"], j["s_x"], j["s_w"], j["s_u"], j["m"], j["n"], j["k"], j["hb"],
                           j["dX"], j["dW"], j["ds"], j["ws"], s["status"])
    return [dict(Y=j["Y"], qX=j["qX"], dX=j["dX"], dW=j["dW"], ds=j["ds"]) for j in s["jobs"]] + [s["status"]]


def _prepare_attention(case, seed, g):
    b, h, kv, s = case["b"], case["h"], case["kv"], case["s"]
    ld = (h + 2 * kv) * 128
    st = dict(case, ld=ld, qkv=_bf16(g, b * s * ld), dout=_bf16(g, b * s * h * 128, 0.1), out=_empty(b * s * h * 128, I16),
              lse=_empty(b * h * s), dqkv=_empty(b * s * ld, I16), status=torch.zeros(1, dtype=I32, device="cuda"))
    st["ws"] = _ws(det.det_attn_fwd_v2_ws_bytes(b, h, s) if case["mode"] == "v2" else
                   det.det_attn_bwd_fixq_ws_bytes(b, h, s, kv) if case["mode"] == "integer" else det.det_attn_bwd_ws_bytes(b, h, s, kv))
    return st


def _run_attention(s):
    b, h, kv, n, ld, win = s["b"], s["h"], s["kv"], s["s"], s["ld"], s["window"]
    q = s["qkv"].data_ptr()
    k, v, dm = q + 2 * 128 * h, q + 2 * 128 * (h + kv), 128 * h
    if s["mode"] == "v2":                        # the version-2 attention has a forward pass only
        det.det_attn_fwd_v2(q, k, v, ld, b, h, n, s["out"], dm, s["lse"], s["ws"], s["status"])
        return dict(out=s["out"], lse=s["lse"], status=s["status"])
    dq = s["dqkv"].data_ptr()
    dk, dv = dq + 2 * 128 * h, dq + 2 * 128 * (h + kv)
    if s["mode"] == "integer":
        det.det_attn_fwd_int8pv(q, k, v, ld, b, h, n, s["out"], dm, s["lse"], s["status"], Hkv=kv, window=win)
        det.det_attn_bwd_fixq(s["dout"], q, k, v, s["out"], s["lse"], ld, dm, b, h, n, dq, dk, dv, ld, s["ws"], Hkv=kv, window=win)
    else:
        det.det_attn_fwd(q, k, v, ld, b, h, n, s["out"], dm, s["lse"], Hkv=kv, window=win)
        det.det_attn_bwd(s["dout"], q, k, v, s["out"], s["lse"], ld, dm, b, h, n, dq, dk, dv, ld, s["ws"], Hkv=kv, window=win)
    return dict(out=s["out"], lse=s["lse"], grads=s["dqkv"], status=s["status"])


def _prepare_head(case, seed, g):
    m, v, d = case["m"], case["vocab"], case["d"]
    st = dict(case, H=_bf16(g, m * d), W=_bf16(g, v * d, 0.02), target=torch.randint(0, v, (m,), generator=g, device="cuda", dtype=I32),
              logits=_empty(m * v), loss_row=_empty(m), lse=_empty(m), loss=_empty(1), z_mean=_empty(1), dH=_empty(m * d, I16),
              dW=_empty(v * d), status=torch.zeros(1, dtype=I32, device="cuda"))
    st["ws"] = _ws(max(det.det_xent_ws_bytes(m, v), det.det_lmhead_fwd_v2_ws_bytes(m, v, d), det.det_lmhead_bwd_v2_ws_bytes(m, v, d)))
    return st


def _run_head(s):
    m, v, d = s["m"], s["vocab"], s["d"]
    if s["arith"] == 2:
        det.det_lmhead_fwd_v2(s["H"], s["W"], m, v, d, s["logits"], s["ws"], s["status"])
    else:
        det.det_lmhead_fwd(s["H"], s["W"], m, v, d, s["logits"])
    det.det_xent_fwd(s["logits"], s["target"], m, v, s["z"], s["loss_row"], s["lse"], s["loss"], s["z_mean"], s["ws"], s["status"])
    det.det_xent_bwd(s["logits"], s["target"], s["lse"], m, v, s["z"], 1.0 / m)      # in place: the logits become their gradient
    if s["arith"] == 2:
        det.det_lmhead_bwd_v2(s["logits"], s["H"], s["W"], m, v, d, s["dH"], s["dW"], s["ws"], s["status"])
    else:
        det.det_lmhead_bwd(s["logits"], s["H"], s["W"], m, v, d, s["dH"], s["dW"], 1)
    return dict(loss=s["loss"], z=s["z_mean"], rows=s["loss_row"], lse=s["lse"], dlogits=s["logits"], dH=s["dH"], dW=s["dW"],
                status=s["status"])


def _prepare_reductions(case, seed, g):
    rows, d, xr, v, n = case["rows"], case["d"], case["xrows"], case["vocab"], case["n"]
    bf = case["dtype"] == "bf16"
    vec = (lambda k: _bf16(g, k)) if bf else (lambda k: _f32(g, k))
    gain = 1 + 0.02 * torch.randn(d, generator=g, device="cuda")
    st = dict(case, io=det.DET_BF16 if bf else det.DET_F32, x=vec(rows * d), dy=vec(rows * d),
              gain=gain.to(torch.bfloat16).view(I16) if bf else gain, y=_empty(rows * d, I16 if bf else F32),
              dx=_empty(rows * d, I16 if bf else F32), rstd=_empty(rows), dgain=_empty(d), logits=_f32(g, xr * v, 2.0),
              target=torch.randint(0, v, (xr,), generator=g, device="cuda", dtype=I32), loss_row=_empty(xr), lse=_empty(xr),
              loss=_empty(1), z_mean=_empty(1), grad=_f32(g, n, 1e-3), norm=_empty(1), coef=_empty(1),
              status=torch.zeros(1, dtype=I32, device="cuda"))
    st["ws"] = _ws(max(det.det_rmsnorm_bwd_ws_bytes(rows, d), det.det_xent_ws_bytes(xr, v), det.det_grad_norm_ws_bytes([st["grad"]])))
    return st


def _run_reductions(s):
    rows, d, xr, v = s["rows"], s["d"], s["xrows"], s["vocab"]
    det.det_rmsnorm_fwd(s["io"], s["x"], s["gain"], rows, d, 1e-6, s["y"], s["rstd"])
    det.det_rmsnorm_bwd(s["io"], s["dy"], s["x"], s["gain"], s["rstd"], rows, d, s["dx"], s["dgain"], s["ws"])
    det.det_xent_fwd(s["logits"], s["target"], xr, v, 1e-4, s["loss_row"], s["lse"], s["loss"], s["z_mean"], s["ws"], s["status"])
    det.det_grad_norm([s["grad"]], 1.0, s["norm"], s["coef"], s["ws"], s["status"])
    return dict(y=s["y"], rstd=s["rstd"], dx=s["dx"], dgain=s["dgain"], loss=s["loss"], z=s["z_mean"], rows=s["loss_row"],
                lse=s["lse"], norm=s["norm"], coef=s["coef"], status=s["status"])


def _prepare_update(case, seed, g):
    r = dstep.Replay(dstep.ModelConfig(n_layers=case["layers"], d_model=case["d"], n_heads=case["d"] // 128, ffn=case["ffn"],
                                       vocab=case["vocab"], seq=128, micro_batch=1,
                                       mesh=(case["accum"], case["shard"], case["rep"]), lr=1e-5))
    r.init_params_on_device(seed)
    r.sx.fill_(0.05)
    r.gmb.normal_(0, 1e-3, generator=g)
    return dict(r=r)


def _run_update(s):
    """The end of a step as the driver makes it; every micro-batch leaves its gradient in the same buffer."""
    r = s["r"]
    cfg = r.cfg
    st = det.det_accum()
    det.det_grad_accum_init(st, cfg.mesh[0], cfg.mesh[1], cfg.mesh[2], r.n_grad, r.abufs)
    for _ in range(cfg.n_microbatches):
        det.det_grad_accum_push(st, r.gmb)
    det.det_grad_accum_result(st, r.gout)
    r.optimizer()
    hashes = r.hashes()
    cfg.step += 1
    return dict(params=r.pbf, steps=r.sx, m=r.m, v=r.v, grad=r.gout, norm=r.norm, coef=r.coef, roots=_roots(hashes))


PREPARE = dict(step=_prepare_step, eval=_prepare_step, linear=_prepare_linear, attention=_prepare_attention, head=_prepare_head,
               reductions=_prepare_reductions, update=_prepare_update)
RUN = dict(step=_run_step, eval=_run_eval, linear=_run_linear, attention=_run_attention, head=_run_head,
           reductions=_run_reductions, update=_run_update)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return dict(PREPARE[case["kind"]](case, seed, g), kind=case["kind"])


def run(state):
    return RUN[state["kind"]](state)


# ---- what a pass cannot do without ------------------------------------------------------------------------------------
def _pairs(s, window):
    """(query, key) pairs of one head of one causal sequence."""
    w = window if 0 < window < s else s
    return w * (w + 1) // 2 + (s - w) * w


def _n_params(layers, d, kv, ffn, vocab):
    lin = layers * ((d + 256 * kv) * d + d * d + 3 * ffn * d)
    return lin, lin + 2 * vocab * d + (2 * layers + 1) * d


def work(case):
    kind = case["kind"]
    if kind in ("step", "eval"):
        t, heads, d = case["seq"] * case["mb"], case["d"] // 128, case["d"]
        lin, total = _n_params(case["layers"], d, case["kv"], case["ffn"], case["vocab"])
        mbs = case["accum"] * case["shard"] * case["rep"]
        windows = [512 if case["block"] == "paper" and l != case["layers"] - 1 and (l + 1) % 5 else 0 for l in range(case["layers"])]
        pairs = case["mb"] * heads * sum(_pairs(case["seq"], w) for w in windows)
        if kind == "eval":
            return dict(bytes=2 * total + 4 * t + 4 * t * case["vocab"],
                        flops=2 * t * (lin + case["vocab"] * d) + 4 * 128 * pairs)
        return dict(bytes=28 * total + 4 * t * mbs, flops=mbs * (6 * t * (lin + case["vocab"] * d) + 14 * 128 * pairs))
    if kind == "linear":
        m, b, f = case["m"], 0, 0
        for shape in case["shapes"].split(","):
            n, k = (int(v) for v in shape.split("x"))
            b += 2 * m * k + m * k + 2 * m * n + 2 * m * n + 2 * m * k + 2 * n * k + 2 * n * k + 4 * n * k
            f += 6 * m * n * k
        return dict(bytes=b, flops=f)
    if kind == "attention":
        b, h, kv, s = case["b"], case["h"], case["kv"], case["s"]
        io, pairs = 2 * b * s * 128 * (h + 2 * kv), b * h * _pairs(s, case["window"])
        if case["mode"] == "v2":
            return dict(bytes=io + 2 * b * s * 128 * h, flops=4 * 128 * pairs)
        return dict(bytes=2 * io + 4 * b * s * 128 * h, flops=14 * 128 * pairs)
    if kind == "head":
        m, v, d = case["m"], case["vocab"], case["d"]
        return dict(bytes=4 * m * v + 4 * m * d + 6 * v * d, flops=6 * m * v * d)
    if kind == "reductions":
        e, rd, x = 2 if case["dtype"] == "bf16" else 4, case["rows"] * case["d"], case["xrows"] * case["vocab"]
        return dict(bytes=4 * e * rd + 4 * x + 4 * case["n"], flops=12 * rd + 4 * x + 2 * case["n"])
    _, total = _n_params(case["layers"], case["d"], case["d"] // 128, case["ffn"], case["vocab"])
    pushes = case["accum"] * case["shard"] * case["rep"]
    return dict(bytes=(4 * pushes + 4 + 20) * total, flops=(2 * pushes + 20) * total)


def tolerance(case):
    """Every operation has one defined order and rounding, so any correct implementation returns the same bits."""
    return "exact"
