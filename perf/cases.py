"""Performance cases of the translation library: what a program that uses it
calls, from one sentence to a full batch, and the layers below it.

Whole calls: `translate` (mnmt_translate, greedy and beam, int8 and 4-bit
models) and `first_step` (encode + the first decode step: the time to the first
token).  Single layers, each through its own entry point: the int8 linear, the
tensor-core linear over fp16 codes, the 4-bit linear, the greedy vocabulary
head, incremental attention, LayerNorm, and a quantisation-aware training step
of one linear (forward and the two fake-quant backward passes).

Every result of the library is defined to the last bit (integer accumulation,
fixed-point sums, stated roundings), so outputs compare exactly; only the fp64
gradient sums of the fake-quant backward pass depend on the order of addition.
"""
import math

import numpy as np
import torch

from paper_2306_04235_gb300 import mnmt, synth

SMALL, WIDE = "small-12x2-d256-v32k-e128", "wide-6x6-d512-v32k"
MB10, MB20 = "mobilenmt-10mb", "mobilenmt-20mb"
TINY = "tiny-2x1-d128-v8k"
MODES = {"q8": mnmt.EPI_Q8, "relu_q8": mnmt.EPI_RELU_Q8, "resid": mnmt.EPI_RESID, "f32": mnmt.EPI_F32}
GAMMA = 0.75  # residual gain of the `resid` epilogue: repeated passes stay bounded


def listed():
    return [
        # an interactive request: one sentence, greedy, the deep-encoder small model
        dict(name="translate_one", kind="translate", model=SMALL, wq=8, batch=1, beam=1, S=46, T=64),
        # the paper's 20MB shape at its own length (30 -> 30), with 4-bit min-max rows
        dict(name="translate_one_4bit", kind="translate", model=MB20, wq=synth.WQ_INT4_MINMAX, batch=1, beam=1, S=30, T=30),
        # an ordinary server batch: 32 sentences, beam 4
        dict(name="translate_batch", kind="translate", model=SMALL, wq=8, batch=32, beam=4, S=80, T=128),
        # the largest: 128 sentences, beam 4, the wide model
        dict(name="translate_large", kind="translate", model=WIDE, wq=8, batch=128, beam=4, S=128, T=160),
        # time to the first token of a batch: the encoder direction
        dict(name="first_step", kind="first_step", model=WIDE, wq=8, batch=64, beam=4, S=100),
        # a layer on int8 operands, a ragged few hundred tokens (QKV of the wide model)
        dict(name="linear_int8", kind="linear", M=1000, N=1536, K=512, mode="q8"),
        # the encoder's largest contraction (FFN2 of the wide model, residual epilogue)
        dict(name="linear_tc_ffn2", kind="linear_tc", M=16384, N=512, K=2048, mode="resid"),
        # the greedy head of a batch over the full vocabulary
        dict(name="vocab_argmax", kind="argmax", M=512, N=32000, K=512),
        # the smallest: a few rows through one 4-bit layer
        dict(name="linear_4bit", kind="linear_w4", M=8, N=2048, K=512, mode="relu_q8", minmax=True),
        # incremental attention of a beam batch late in a translation
        dict(name="attention_decode", kind="attention", R=512, H=8, dh=64, T=160),
        # LayerNorm over an encoder batch
        dict(name="layernorm", kind="layernorm", M=16384, d=512),
        # quantisation-aware training of one FFN layer: forward, activation and weight gradients
        dict(name="qat_step", kind="qat", M=4096, N=2048, K=512, wbits=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult(x, m, lo):
    return max(lo, x // m * m)


def draw(rng):
    kind = rng.choice(["translate", "translate", "first_step", "linear", "linear_tc", "linear_w4", "argmax", "attention",
                       "layernorm", "qat"])
    if kind == "translate":
        model = rng.choice([SMALL, SMALL, WIDE, MB10, MB20, TINY])
        beam = rng.choice([1, 1, 4, 2, 5])
        wq = rng.choice([8, 8, 8, synth.WQ_INT4, synth.WQ_INT4_MINMAX])
        batch = _log(rng, 1, 24 if wq == synth.WQ_INT4_MINMAX else 128)
        batch = max(1, min(batch, 512 // beam))
        return dict(kind=kind, model=model, wq=wq, batch=batch, beam=beam, S=rng.randint(5, 128), T=_log(rng, 8, 96))
    if kind == "first_step":
        return dict(kind=kind, model=rng.choice([SMALL, WIDE, MB10, MB20]), wq=8, batch=_log(rng, 1, 128),
                    beam=rng.choice([1, 4]), S=rng.randint(5, 128))
    mode = rng.choice(list(MODES))
    if kind == "linear":
        M = _log(rng, 1, 16384)
        return dict(kind=kind, M=M, N=_log(rng, 96, 4096), K=_mult(_log(rng, 64, 2048), 64, 64), mode=mode)
    if kind == "linear_tc":
        return dict(kind=kind, M=_log(rng, 17, 16384), N=_log(rng, 96, 4096), K=_mult(_log(rng, 64, 2048), 8, 64), mode=mode)
    if kind == "linear_w4":
        return dict(kind=kind, M=_log(rng, 1, 64), N=_log(rng, 96, 4096), K=_mult(_log(rng, 64, 2048), 32, 64), mode=mode,
                    minmax=rng.random() < 0.5)
    if kind == "argmax":
        return dict(kind=kind, M=_log(rng, 1, 1024), N=rng.randint(8000, 33000), K=rng.choice([128, 256, 384, 512, 1024]))
    if kind == "attention":
        return dict(kind=kind, R=_log(rng, 1, 512), H=rng.choice([4, 6, 8]), dh=rng.choice([32, 64, 64, 128]),
                    T=_log(rng, 4, 512))
    if kind == "layernorm":
        return dict(kind=kind, M=_log(rng, 1, 16384), d=rng.choice([128, 256, 384, 512, 768, 1024, rng.randint(65, 1100)]))
    return dict(kind=kind, M=_log(rng, 1, 8192), N=_log(rng, 96, 3072), K=_mult(_log(rng, 64, 1024), 64, 64),
                wbits=rng.choice([4, 8]))


# --------------------------------------------------------------------------- inputs
_models = {}  # (model, format) -> (config, blob, handle): a program loads its model once


def _model(name, wq):
    if (name, wq) not in _models:
        cfg = synth.MODELS[name]
        blob = synth.build_blob(cfg, 1, wq=wq)
        stream = torch.cuda.Stream()
        _models[name, wq] = (cfg, stream, mnmt.mnmt_load_weights(blob, stream))
    return _models[name, wq]


class _Session:
    """A session and its sources; freed with the state."""

    def __init__(self, case, seed):
        cfg, self.stream, model = _model(case["model"], case["wq"])
        B, S, self.beam = case["batch"], case["S"], case["beam"]
        self.T = case.get("T", 16)
        self.B, self.S, self.R, self.d = B, S, B * self.beam, cfg.d_model
        rng = np.random.default_rng(seed)
        # lengths from a fifth of the longest up to it; ids as a shuffled corpus would give them
        self.lens = rng.integers(max(1, S // 5), S + 1, B).astype(np.int32)
        self.lens[0] = S
        self.ids = rng.integers(3, cfg.vocab, (B, S)).astype(np.int32)
        self.ids[np.arange(S)[None, :] >= self.lens[:, None]] = cfg.pad_id
        self.handle = mnmt.mnmt_session_create(model, B, S, self.beam, self.T)

    def __del__(self):
        if getattr(self, "handle", None):
            mnmt.mnmt_session_free(self.handle)
            self.handle = None


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _codes(g, *shape):
    """int8 codes of a quantised Gaussian tensor (clipped at about four deviations)."""
    return torch.randn(shape, generator=g, device="cuda").mul_(127 / 4).round_().clamp_(-127, 127).to(torch.int8)


def _unit(g, *shape):
    return torch.rand(shape, generator=g, device="cuda")


def prepare(case, seed):
    k = case["kind"]
    if k in ("translate", "first_step"):
        return {"kind": k, "s": _Session(case, seed)}
    g = _gen(seed)
    st = {"kind": k, "case": case}
    if k in ("linear", "linear_tc", "argmax", "linear_w4"):
        M, N, K = case["M"], case["N"], case["K"]
        st["A"], st["W"] = _codes(g, M, K), None
        st["s_x"] = 4 / 127
        st["s_w"] = _unit(g, N) * 2e-4 + 5e-4
        st["b"] = (_unit(g, N) - 0.5) * 0.04
        st["inv"] = 1.0 / (_unit(g, N) * 0.01 + 0.01)
        if k == "linear_w4":
            st["W"] = torch.randint(0, 256, (N, K // 2), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8)
            st["s_w"] = _unit(g, N) * 2e-3 + 5e-3
            st["m"] = (-7.5 * st["s_w"]).contiguous() if case["minmax"] else None
        else:
            st["W"] = _codes(g, N, K)
        if k == "linear_tc":
            for n in ("A", "W"):
                h = torch.empty(st[n].shape, dtype=torch.float16, device="cuda")
                mnmt.mnmt_codes_to_f16(st[n], h, h.numel())
                st[n + "16"] = h
            st["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        if k == "argmax":
            st["ids"] = torch.zeros(M, dtype=torch.int32, device="cuda")
        elif case["mode"] in ("resid", "f32"):
            st["f"] = torch.randn((M, N), generator=g, device="cuda")
            st["q"] = None
        else:
            st["q"] = torch.zeros((M, N), dtype=torch.int8, device="cuda")
            st["f"] = None
    elif k == "attention":
        R, H, dh, T = case["R"], case["H"], case["dh"], case["T"]
        st["q"] = _codes(g, R, H, dh)
        st["k"], st["v"] = _codes(g, R, H, T, dh), _codes(g, R, H, T, dh)
        st["n"] = torch.randint(max(1, T // 2), T + 1, (R,), generator=g, device="cuda", dtype=torch.int32)
        st["sigma"], st["rho"] = float(np.float32((2 / 127) ** 2 / math.sqrt(dh))), 1.25
        st["ctx"] = torch.zeros((R, H, dh), dtype=torch.int8, device="cuda")
    elif k == "layernorm":
        M, d = case["M"], case["d"]
        st["r"] = torch.randn((M, d), generator=g, device="cuda") * (_unit(g, M, 1) * 4 + 0.5) + _unit(g, M, 1) - 0.5
        st["g"], st["b"] = torch.randn(d, generator=g, device="cuda") * 0.02 + 1, torch.randn(d, generator=g, device="cuda") * 0.02
        st["f"] = torch.empty((M, d), device="cuda")
        st["q"] = torch.empty((M, d), dtype=torch.int8, device="cuda")
    else:  # qat
        M, N, K = case["M"], case["N"], case["K"]
        st["X"], st["W"] = torch.randn((M, K), generator=g, device="cuda"), torch.randn((N, K), generator=g, device="cuda") * 0.05
        st["gX"], st["gW"] = torch.randn((M, K), generator=g, device="cuda"), torch.randn((N, K), generator=g, device="cuda")
        qmax = 2 ** (case["wbits"] - 1) - 1
        st["s_w"] = (st["W"].abs().amax(1) * 0.9 / qmax).contiguous()  # learned scales clip a little
        st["s_x"], st["s_wt"] = 3.0 / 127, float(np.float32(0.15 / qmax))
        st["b"] = torch.randn(N, generator=g, device="cuda") * 0.02
        st["ws"] = torch.empty((M * K + 15) // 16 * 16 + N * K, dtype=torch.uint8, device="cuda")
        st["y"] = torch.empty((M, N), device="cuda")
        st["dX"], st["dW"] = torch.empty((M, K), device="cuda"), torch.empty((N, K), device="cuda")
        st["ds"] = torch.zeros(2, dtype=torch.float64, device="cuda")
    return st


# --------------------------------------------------------------------------- one pass
def run(st):
    k = st["kind"]
    if k == "translate":
        s = st["s"]
        ids, lens = np.empty((s.B, s.T), np.int32), np.empty(s.B, np.int32)
        scores = np.empty(s.B, np.float32)
        mnmt.mnmt_translate(s.handle, s.ids, s.lens, s.B, s.S, s.T, 0, ids, lens, scores)
        # beside the tokens: the last step's quantised decoder output, the input of the vocabulary projection
        return {"ids": ids, "lens": lens, "scores": scores,
                "dec_out": mnmt.mnmt_debug_tap(s.handle, mnmt.TAP_DEC_OUT, 0, np.int8, (s.R, s.d))}
    if k == "first_step":
        s = st["s"]
        mnmt.mnmt_encode(s.handle, s.ids, s.lens, s.B, s.S)
        tok, par, sc, _ = mnmt.mnmt_decode_step(s.handle, s.R)
        return {"tokens": tok, "parents": par, "scores": sc,
                "dec_out": mnmt.mnmt_debug_tap(s.handle, mnmt.TAP_DEC_OUT, 0, np.int8, (s.R, s.d))}
    c = st["case"]
    if k == "linear":
        mnmt.mnmt_linear(st["A"], st["W"], st["s_w"], st["b"], st["s_x"], st["inv"], GAMMA, c["M"], c["N"], c["K"],
                         MODES[c["mode"]], st["q"], st["f"])
        return st["q"] if st["f"] is None else st["f"]
    if k == "linear_tc":
        mnmt.mnmt_linear_tc(st["A16"], st["W16"], st["s_w"], st["b"], st["s_x"], st["inv"], GAMMA, c["M"], c["N"], c["K"],
                            MODES[c["mode"]], st["q"], st["f"], None, st["status"])
        return [st["q"] if st["f"] is None else st["f"], st["status"]]
    if k == "linear_w4":
        mnmt.mnmt_linear_w4(st["A"], st["W"], st["s_w"], st["m"], st["b"], st["s_x"], st["inv"], GAMMA, c["M"], c["N"],
                            c["K"], MODES[c["mode"]], st["q"], st["f"])
        return st["q"] if st["f"] is None else st["f"]
    if k == "argmax":
        mnmt.mnmt_linear_argmax_ids_noalloc(st["A"], st["W"], st["s_w"], st["b"], st["s_x"], c["M"], c["N"], c["K"], st["ids"])
        return st["ids"]
    if k == "attention":
        mnmt.mnmt_attention_decode(st["q"], st["k"], st["v"], st["n"], c["R"], c["H"], c["dh"], c["T"], st["sigma"],
                                   st["rho"], st["ctx"])
        return st["ctx"]
    if k == "layernorm":
        mnmt.mnmt_layernorm(st["r"], st["g"], st["b"], c["M"], c["d"], 127 / 4, st["f"], st["q"])
        return {"f": st["f"], "q": st["q"]}
    # one training step of a linear: forward; the activation's and the weight's straight-through and scale gradients
    M, N, K = c["M"], c["N"], c["K"]
    mnmt.mnmt_fake_quant_linear(st["X"], st["W"], st["s_x"], st["s_w"], st["b"], M, N, K, c["wbits"], st["ws"], st["y"])
    ds = st["ds"]
    mnmt.mnmt_fake_quant_backward(st["X"], st["gX"], M * K, st["s_x"], st["dX"], ds[0:1])
    mnmt.mnmt_fake_quant_backward(st["W"], st["gW"], N * K, st["s_wt"], st["dW"], ds[1:2], bits=c["wbits"])
    return {"y": st["y"], "dX": st["dX"], "dW": st["dW"], "ds": ds}


# --------------------------------------------------------------------------- what a pass cannot do without
def _encode_work(cfg, wbytes, B, S):
    d, F, L, D = cfg.d_model, cfg.d_ffn, cfg.n_enc, cfg.n_dec
    per_layer = 4 * d * d + 2 * d * F
    lin = L * per_layer + D * 2 * d * d + (d * cfg.d_embed if cfg.d_embed != d else 0)
    flops = 2 * B * S * lin + L * 4 * B * S * S * d
    byts = lin * wbytes + B * S * (cfg.d_embed + D * 2 * d)
    return byts, flops


def _step_work(cfg, wbytes, R, B, S, t):
    d, F, D = cfg.d_model, cfg.d_ffn, cfg.n_dec
    lin = D * (6 * d * d + 2 * d * F) + (d * cfg.d_embed if cfg.d_embed != d else 0)
    byts = lin * wbytes + cfg.vocab * (d + 8) + D * 2 * d * (B * S + R * t)
    return byts, 2 * R * (lin + cfg.vocab * d) + D * 4 * R * (S + t) * d


def work(case):
    k = case["kind"]
    if k in ("translate", "first_step"):
        cfg = synth.MODELS[case["model"]]
        wb = 1.0 if case["wq"] == 8 else 0.5
        B, S, R = case["batch"], case["S"], case["batch"] * case["beam"]
        T = case["T"] if k == "translate" else 1
        eb, ef = _encode_work(cfg, wb, B, S)
        sb, sf = _step_work(cfg, wb, R, B, S, (T + 1) / 2)
        return {"bytes": eb + T * sb, "flops": ef + T * sf}
    if k in ("linear", "linear_tc", "linear_w4", "argmax"):
        M, N, K = case["M"], case["N"], case["K"]
        e = {"linear_tc": 2, "linear_w4": 0.5}.get(k, 1)
        out = 4 * M if k == "argmax" else M * N * {"q8": 1, "relu_q8": 1, "resid": 8, "f32": 4}[case["mode"]]
        return {"bytes": M * K * (2 if k == "linear_tc" else 1) + N * K * e + 8 * N + out, "flops": 2 * M * N * K}
    if k == "attention":
        R, H, dh, T = case["R"], case["H"], case["dh"], case["T"]
        n = (max(1, T // 2) + T) / 2
        return {"bytes": R * H * dh * (2 * n + 2) + 4 * R, "flops": 4 * R * H * dh * n}
    if k == "layernorm":
        return {"bytes": case["M"] * case["d"] * 9 + 8 * case["d"], "flops": 8 * case["M"] * case["d"]}
    M, N, K = case["M"], case["N"], case["K"]
    return {"bytes": 4 * (M * K + N * K + M * N) + 12 * (M * K + N * K), "flops": 2 * M * N * K}


def tolerance(case):
    # the scale gradients are fp64 sums in no fixed order: 4e-16 seen between two
    # orders at the listed size; the terms have both signs, so a draw whose sum
    # nearly cancels may show a few hundred times that.  All else is exact.
    return {"rel": 1e-13, "max": 1e-13, "differ": 0.0} if case["kind"] == "qat" else "exact"


# --------------------------------------------------------------------------- the same in 64 bits
def _f64(x):
    return x.to(torch.float64)


def _affine(st, acc):
    return acc * (float(np.float32(st["s_x"])) * _f64(st["s_w"])) + _f64(st["b"])


def _fq64(x, s, bits):
    """codes of the symmetric quantiser (its own fp32 rounding points) and the unrounded code"""
    qmax = 2 ** (bits - 1) - 1
    inv = torch.ones((), device=x.device) / s
    t = x * inv
    return torch.round(t).clamp(-qmax, qmax).to(torch.float64), t.to(torch.float64), qmax


def exact(case, seed):
    """The floating outputs in 64 bits; None for codes, ids and whole translations (they have no other value)."""
    k = case["kind"]
    if k in ("translate", "first_step", "attention", "argmax") or case.get("mode") in ("q8", "relu_q8"):
        return None
    st = prepare(case, seed)
    if k in ("linear", "linear_tc", "linear_w4"):
        A = _f64(st["A"])
        if k == "linear_w4":
            w = st["W"].view(case["N"], case["K"] // 32, 16).to(torch.int16)
            u = torch.cat([w & 15, w >> 4], 2).reshape(case["N"], case["K"]).to(torch.float64)
            s_x = float(np.float32(st["s_x"]))
            if case["minmax"]:
                y = (A @ u.T) * (s_x * _f64(st["s_w"])) + A.sum(1, keepdim=True) * (s_x * _f64(st["m"])) + _f64(st["b"])
            else:
                y = _affine(st, A @ (u - 8).T)
        else:
            y = _affine(st, A @ _f64(st["W"]).T)
        y = y + GAMMA * _f64(st["f"]) if case["mode"] == "resid" else y
        return [y, None] if k == "linear_tc" else y
    if k == "layernorm":
        r = _f64(st["r"])
        c = r - r.mean(1, keepdim=True)
        y = c / torch.sqrt((c * c).mean(1, keepdim=True) + 1e-5) * _f64(st["g"]) + _f64(st["b"])
        return {"f": y, "q": None}
    X, W = st["X"], st["W"]
    s_x = torch.tensor(st["s_x"], dtype=torch.float32, device="cuda")
    s_wt = torch.tensor(st["s_wt"], dtype=torch.float32, device="cuda")
    qx, tx, mx = _fq64(X, s_x, 8)
    qw, _, _ = _fq64(W, st["s_w"][:, None], case["wbits"])
    y = (qx @ qw.T) * (_f64(s_x) * _f64(st["s_w"])) + _f64(st["b"])
    out, ds = [], []
    for x, gr, s, bits in ((X, st["gX"], s_x, 8), (W, st["gW"], s_wt, case["wbits"])):
        q, t, m = _fq64(x, s, bits)
        inside = t.abs() <= m
        out.append(_f64(gr) * inside)
        ds.append((_f64(gr) * torch.where(inside, q - t, q)).sum())
    return {"y": y, "dX": out[0], "dW": out[1], "ds": torch.stack(ds)}
