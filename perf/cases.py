"""What users of this library have it do, as cases that can be timed and checked.

A case is a dict of plain values.  ``prepare`` makes what a program holds
before the call (inputs, weights, optimiser state), ``run`` makes one pass
through the public entry points and returns its outputs whole, ``exact`` gives
the same values from plain torch in 64 bits.

Kinds of case:
  steps   training steps of one layer on operand images, captured once as a CUDA
          graph and replayed with new update constants (small layers are run so)
  layer   one training step of a DQTBitLinear module: forward, dX and the
          weight update in its backward (each grid, activation type, optimiser
          and code storage that the module takes)
  codes   the same step through the calls on int8 codes
  mlp     the training step of an MLP's three projections on operand images:
          gate and up stacked, both weight gradients in one grouped launch
  update  AdamW + stochastic rounding of a gradient in memory (a data-parallel
          rank's shard)
  ops     what the decoder runs between its projections: RMSNorm, the rotary
          embedding and the SwiGLU gate, forward and backward
  loss    token cross-entropy over the vocabulary, forward and gradient
  logits  the decoder evaluated on one sequence (no gradient)
  train   one training step of the decoder, replayed from a CUDA graph
"""
import math

import torch
import torch.nn.functional as F

from paper_2412_04787_gb300 import dqt
from paper_2412_04787_gb300.bitlinear import DQTBitLinear
from paper_2412_04787_gb300.decoder import DecoderConfig, DQTDecoder

LR, BETAS, EPS, STEP = 1e-3, (0.9, 0.999), 1e-8, 100
THETA, NORM_EPS = 10000.0, 1e-6


def _layer(name, T, K, N, bits=1.58, act="int8", optimizer="adamw", packed=False):
    return {"name": name, "kind": "layer", "T": T, "K": K, "N": N, "bits": bits, "act": act,
            "optimizer": optimizer, "packed": packed}


def listed():
    return [
        # a small layer: a few microseconds of work, so latency and launches
        {"name": "steps_small", "kind": "steps", "T": 256, "K": 512, "N": 512, "bits": 1.58,
         "steps": 8},
        # q, k, v or o of the 12-layer, 768-wide decoder at 16 x 1024 tokens
        {"name": "steps_768", "kind": "steps", "T": 16384, "K": 768, "N": 768, "bits": 1.58,
         "steps": 2},
        # the down projection of a 2048-wide decoder with 8-bit codes
        _layer("layer_down_8bit", 8192, 5632, 2048, bits=8.0),
        # the FP8 environment on sizes that no tile divides
        _layer("layer_fp8_ragged", 3001, 1040, 2744, bits=4.0, act="fp8"),
        # the memory-efficient set-up: Adafactor and 2-bit codes, a gate projection
        _layer("layer_adafactor_packed", 8192, 2048, 5632, optimizer="adafactor", packed=True),
        # a program on the C interface that holds int8 codes only
        {"name": "codes_gate", "kind": "codes", "T": 8192, "K": 2048, "N": 5632, "bits": 1.58},
        # the MLP of the benchmark: 4 x 2048 tokens, 2048 -> 5632 -> 2048
        {"name": "mlp_step", "kind": "mlp", "T": 8192, "H": 2048, "I": 5632, "bits": 1.58},
        # a shard of 2^26 weights updated after a reduce-scatter
        {"name": "update_8bit", "kind": "update", "n": 1 << 26, "bits": 8.0},
        # one block's norms, rotations and gate in a 2048-wide decoder, 8 x 2048 tokens
        {"name": "ops_2048", "kind": "ops", "B": 8, "S": 2048, "D": 2048, "H": 32, "I": 5632},
        # the head's loss over a 32000-word vocabulary
        {"name": "loss_32000", "kind": "loss", "M": 8192, "V": 32000},
        # evaluating a prompt
        {"name": "logits_prompt", "kind": "logits", "layers": 2, "D": 768, "H": 12, "I": 2048,
         "V": 32000, "B": 1, "S": 333, "bits": 1.58},
        # a training step of the decoder
        {"name": "train_step", "kind": "train", "layers": 2, "D": 768, "H": 12, "I": 2048,
         "V": 32000, "B": 4, "S": 1024, "bits": 1.58},
    ]


def _log(rng, lo, hi, step=1):
    """An integer in [lo, hi], spread over its logarithm, a multiple of `step`."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step
    return max(lo, min(hi, v))


def draw(rng):
    kind = rng.choice(["steps", "steps", "layer", "layer", "layer", "codes", "mlp", "update", "ops",
                       "loss", "logits", "train"])
    bits = rng.choice([1.58, 1.58, 4.0, 8.0])
    if kind == "layer":
        T, K, N = _log(rng, 64, 16384), _log(rng, 256, 5632, 16), _log(rng, 256, 5632, 8)
        act = rng.choice(["int8", "int8", "fp8"])
        optimizer = rng.choice(["adamw", "adamw", "adafactor"])
        packed = bits == 1.58 and rng.random() < 0.4
        if act == "fp8" and bits == 8.0:
            K = max(256, K // 128 * 128)  # the split E4M3 image's rows
        T = min(T, 200_000_000_000 // (K * N))  # no more work than the MLP's step
        c = _layer("", T, K, N, bits, act, optimizer, packed)
        del c["name"]
        return c
    if kind == "steps":
        return {"kind": kind, "T": _log(rng, 128, 16384), "K": _log(rng, 256, 1536, 8),
                "N": _log(rng, 256, 1536, 8), "bits": bits, "steps": rng.choice([2, 4])}
    if kind == "codes":
        return {"kind": kind, "T": _log(rng, 64, 8192), "K": _log(rng, 256, 5632, 16),
                "N": _log(rng, 256, 5632, 8), "bits": bits}
    if kind == "mlp":
        return {"kind": kind, "T": _log(rng, 256, 8192), "H": _log(rng, 512, 2048, 8),
                "I": _log(rng, 1024, 5632, 256), "bits": bits}
    if kind == "update":
        return {"kind": kind, "n": _log(rng, 1 << 16, 1 << 26), "bits": bits}
    if kind == "ops":
        hd, H = rng.choice([32, 64, 128]), rng.randint(4, 16)
        return {"kind": kind, "B": rng.randint(1, 8), "S": _log(rng, 64, 2048), "D": hd * H, "H": H,
                "I": _log(rng, 256, 5632, 8)}
    if kind == "loss":
        return {"kind": kind, "M": _log(rng, 64, 8192), "V": _log(rng, 1000, 32000, 8)}
    H = rng.randint(4, 12)
    return {"kind": kind, "layers": rng.randint(1, 2), "D": 64 * H, "H": H,
            "I": _log(rng, 512, 2048, 8), "V": _log(rng, 1000, 32000, 8),
            "B": 1 if kind == "logits" else rng.randint(1, 4),
            "S": _log(rng, 16 if kind == "logits" else 128, 1024),
            "bits": rng.choice([1.58, 8.0])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(g, shape, std, dtype=torch.float32):
    return (torch.randn(shape, generator=g, device="cuda") * std).to(dtype)


def _moments(g, shape):
    # moments of a run under way, of the size that gradients of 1e-2 leave
    return _normal(g, shape, 1e-4), _normal(g, shape, 1e-4).square_()


def _weight(g, N, K, bits):
    return dqt.dqt_absmean_init(_normal(g, (N, K), 0.02), bits)


def _tensors(case, seed):
    """The input tensors of a case, in one fixed order of draws."""
    g, kind = _gen(seed), case["kind"]
    bf = torch.bfloat16
    if kind in ("steps", "layer", "codes"):
        T, K, N = case["T"], case["K"], case["N"]
        t = {"x": _normal(g, (T, K), 1.0, bf), "dy": _normal(g, (T, N), 1e-2, bf)}
        if case.get("optimizer") != "adafactor":
            t["m"], t["v"] = _moments(g, (N, K))
        if kind != "layer":
            t["W"], t["s_w"] = _weight(g, N, K, case["bits"])
        return t
    if kind == "mlp":
        T, H, I = case["T"], case["H"], case["I"]
        t = {"x": _normal(g, (T, H), 1.0, bf), "h": _normal(g, (T, I), 1.0, bf),
             "dgu": _normal(g, (T, 2 * I), 1e-2, bf), "dd": _normal(g, (T, H), 1e-2, bf)}
        t["m_gu"], t["v_gu"] = _moments(g, (2 * I, H))
        t["m_d"], t["v_d"] = _moments(g, (H, I))
        Wg, t["s_g"] = _weight(g, I, H, case["bits"])
        Wu, t["s_u"] = _weight(g, I, H, case["bits"])
        t["W_gu"] = torch.cat((Wg, Wu))
        t["W_d"], t["s_d"] = _weight(g, H, I, case["bits"])
        return t
    if kind == "update":
        n = case["n"]
        t = {"grad": _normal(g, (n,), 1e-3)}
        t["m"], t["v"] = _moments(g, (n,))
        t["W"], t["s_w"] = dqt.dqt_absmean_init(_normal(g, (n,), 0.02), case["bits"])
        return t
    if kind == "ops":
        B, S, D, I = case["B"], case["S"], case["D"], case["I"]
        R = B * S
        t = {"x": _normal(g, (R, D), 1.0, bf),
             "w": (1.0 + 0.1 * _normal(g, (D,), 1.0)).to(bf), "dy": _normal(g, (R, D), 1e-2, bf),
             "q": _normal(g, (B, S, case["H"], D // case["H"]), 1.0, bf),
             "g": _normal(g, (R, I), 1.0, bf), "u": _normal(g, (R, I), 1.0, bf),
             "dh": _normal(g, (R, I), 1e-2, bf)}
        hd = D // case["H"]
        inv = 1.0 / THETA ** (torch.arange(0, hd, 2, device="cuda", dtype=torch.float32) / hd)
        ang = torch.outer(torch.arange(S, device="cuda", dtype=torch.float32), inv)
        t["cs"] = torch.stack((torch.cos(ang), torch.sin(ang)), dim=-1).contiguous()
        return t
    if kind == "loss":
        M, V = case["M"], case["V"]
        return {"logits": _normal(g, (M, V), 2.0, bf),
                "targets": torch.randint(0, V, (M,), generator=g, device="cuda"),
                "scale": torch.full((1,), 1.0 / M, device="cuda")}
    ids = torch.randint(0, case["V"], (case["B"], case["S"] + 1), generator=g, device="cuda")
    return {"ids": ids[:, :-1].contiguous(), "targets": ids[:, 1:].contiguous()}


def _module(case, seed, t):
    layer = DQTBitLinear(case["K"], case["N"], bits=case["bits"], lr=LR, betas=BETAS, eps=EPS,
                         seed=seed, tensor_id=3, init_seed=seed, act=case["act"],
                         optimizer=case["optimizer"], packed=case["packed"])
    if case["optimizer"] == "adamw":
        layer.m.copy_(t["m"])
        layer.v.copy_(t["v"])
        layer.step = STEP - 1
    return layer


def _decoder(case, seed):
    return DQTDecoder(DecoderConfig(layers=case["layers"], hidden=case["D"], heads=case["H"],
                                    ffn=case["I"], vocab=case["V"], bits=case["bits"], lr=LR,
                                    seed=seed, rope_theta=THETA, norm_eps=NORM_EPS))


class _Steps:
    """Captured training steps of one layer: two weight images that each step
    swaps, update constants in a device block fed from two host blocks."""

    def __init__(self, case, seed, t):
        self.case, self.t, self.count, self.step = case, t, case["steps"], STEP - 1
        T, K, N = case["T"], case["K"], case["N"]
        self.grid, self.sr = dqt.grid(case["bits"]), dqt.sr_stream(seed=seed, tensor_id=3)
        row = (dqt.lib().dqt_update_consts_size() + 63) // 64 * 64
        self.host = [torch.zeros((self.count, row), dtype=torch.uint8).pin_memory() for _ in range(2)]
        self.dev = torch.zeros((self.count, row), dtype=torch.uint8, device="cuda")
        self.copied, self.turn = [None, None], 0
        self.images = [dqt.dqt_codes_to_bf16(t["W"]), torch.empty_like(t["W"], dtype=torch.bfloat16)]
        bf, dev = torch.bfloat16, "cuda"
        self.s_x = torch.empty(T, device=dev)
        self.q, self.xdq = (torch.empty((T, K), dtype=bf, device=dev) for _ in range(2))
        self.y, self.dx = torch.empty((T, N), dtype=bf, device=dev), torch.empty((T, K), dtype=bf, device=dev)
        sizes = (dqt.dqt_fwd_img_workspace_size(T, K, N), dqt.dqt_bwd_dx_img_workspace_size(T, N, K),
                 dqt.dqt_bwd_dw_img_workspace_size(T, N, K))
        self.ws = [torch.empty(n, dtype=torch.uint8, device=dev) if n else False for n in sizes]
        self.pass_on_current_stream(forward_only=True)  # the library's first use, outside the capture
        torch.cuda.synchronize()
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(self.graph):
            self.pass_on_current_stream()

    def pass_on_current_stream(self, forward_only=False):
        t, s_w = self.t, self.t["s_w"]
        for i in range(self.count):
            img, img_next = self.images[i % 2], self.images[(i + 1) % 2]
            dqt.dqt_act_quant_images(t["x"], None, self.s_x, self.q, self.xdq, want=())
            dqt.dqt_bitlinear_fwd_img(self.q, self.s_x, img, s_w, self.grid, Y=self.y, ws=self.ws[0])
            if forward_only:
                return
            dqt.dqt_bitlinear_bwd_dx_img(t["dy"], img, s_w, dX=self.dx, ws=self.ws[1])
            dqt.dqt_bitlinear_bwd_dw_update_dev(t["dy"], self.xdq, t["W"], t["m"], t["v"], self.dev[i],
                                                ws=self.ws[2], W_img_next=img_next)

    def replay(self):
        slot = self.turn % 2
        self.turn += 1
        if self.copied[slot] is not None:
            self.copied[slot].synchronize()  # the copy that last read this host block is done
        for i in range(self.count):
            self.step += 1
            hp = dqt.adamw(lr=LR, beta1=BETAS[0], beta2=BETAS[1], eps=EPS, step=self.step)
            dqt.dqt_update_consts(hp, self.sr, self.grid, self.t["s_w"], out=self.host[slot][i])
        self.dev.copy_(self.host[slot], non_blocking=True)
        self.copied[slot] = torch.cuda.Event()
        self.copied[slot].record()
        self.graph.replay()


class _Train:
    """A decoder whose training step (gradients of the dense parameters, updates
    of the BitLinear codes) is captured once and replayed."""

    def __init__(self, case, seed, t):
        self.model, self.t, self.turn = _decoder(case, seed), t, 0
        self.model.enable_graph_updates()
        layers = self.model.bitlinear_layers()
        # warm up without the updates, so that the captured step is the first
        for b in layers:
            b.update_in_backward = False
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            for _ in range(2):
                self.forward_backward()
                self.model.zero_grad(set_to_none=True)
        torch.cuda.current_stream().wait_stream(side)
        for b in layers:
            b.update_in_backward = True
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(self.graph):
            self.loss = self.forward_backward()

    def forward_backward(self):
        loss = self.model(self.t["ids"], self.t["targets"])
        loss.backward()
        return loss.detach()

    def replay(self):
        self.model.prepare_step(self.turn % 2)
        self.model.upload_update_consts(self.turn % 2)
        self.turn += 1
        self.graph.replay()


def prepare(case, seed):
    t, kind = _tensors(case, seed), case["kind"]
    s = {"case": case, "seed": seed, "t": t}
    if kind == "steps":
        s["steps"] = _Steps(case, seed, t)
    elif kind == "layer":
        s["layer"] = _module(case, seed, t)
    elif kind == "codes":
        T, K, N = case["T"], case["K"], case["N"]
        sizes = (dqt.dqt_fwd_workspace_size(T, K, N), dqt.dqt_bwd_dx_workspace_size(T, N, K),
                 dqt.dqt_bwd_dw_workspace_size(T, N, K))
        s["ws"] = torch.empty(max(sizes), dtype=torch.uint8, device="cuda")
        s["step"] = STEP - 1
    elif kind == "mlp":
        s["img_gu"] = [dqt.dqt_codes_to_bf16(t["W_gu"]), torch.empty_like(t["W_gu"], dtype=torch.bfloat16)]
        s["img_d"] = [dqt.dqt_codes_to_bf16(t["W_d"]), torch.empty_like(t["W_d"], dtype=torch.bfloat16)]
        s["step"] = STEP - 1
    elif kind == "update":
        s["step"] = STEP - 1
    elif kind == "logits":
        s["model"] = _decoder(case, seed)
    elif kind == "train":
        s["train"] = _Train(case, seed, t)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _hp(s):
    s["step"] += 1
    return dqt.adamw(lr=LR, beta1=BETAS[0], beta2=BETAS[1], eps=EPS, step=s["step"])


def run(s):
    case, t = s["case"], s["t"]
    kind = case["kind"]
    if kind == "steps":
        p = s["steps"]
        p.replay()
        return {"y": p.y, "dx": p.dx, "codes": t["W"], "m": t["m"], "v": t["v"]}
    if kind == "layer":
        layer = s["layer"]
        x = t["x"].detach().requires_grad_()  # a new activation, as a network hands it on
        y = layer(x)
        (dx,) = torch.autograd.grad(y, (x,), t["dy"])
        state = (layer.m, layer.v) if case["optimizer"] == "adamw" else (layer.R, layer.C)
        return {"y": y.detach(), "dx": dx, "codes": layer.codes, "state": state}
    if kind == "codes":
        g, s_w, ws = dqt.grid(case["bits"]), t["s_w"], s["ws"]
        xq, s_x = dqt.dqt_act_quant(t["x"])
        y = dqt.dqt_bitlinear_fwd(xq, s_x, t["W"], s_w, g, ws=ws)
        dx = dqt.dqt_bitlinear_bwd_dx(t["dy"], t["W"], s_w, ws=ws)
        dqt.dqt_bitlinear_bwd_dw_update(t["dy"], xq, s_x, t["W"], s_w, t["m"], t["v"], _hp(s),
                                        dqt.sr_stream(seed=s["seed"], tensor_id=3), g, ws=ws)
        return {"xq": xq, "s_x": s_x, "y": y, "dx": dx, "codes": t["W"], "m": t["m"], "v": t["v"]}
    if kind == "mlp":
        g, I, hp, seed = dqt.grid(case["bits"]), case["I"], _hp(s), s["seed"]
        img_gu, img_d = s["img_gu"], s["img_d"]
        _, sx, xi, xd = dqt.dqt_act_quant_images(t["x"], want=("Xq_img", "Xdq"))
        gu = dqt.dqt_bitlinear_fwd_img_pair(xi, sx, img_gu[0], I, t["s_g"], t["s_u"], g)
        _, sh, hi, hd = dqt.dqt_act_quant_images(t["h"], want=("Xq_img", "Xdq"))
        y = dqt.dqt_bitlinear_fwd_img(hi, sh, img_d[0], t["s_d"], g)
        dh = dqt.dqt_bitlinear_bwd_dx_img(t["dd"], img_d[0], t["s_d"])
        dxg = dqt.dqt_bitlinear_bwd_dx_img(t["dgu"][:, :I], img_gu[0][:I], t["s_g"])
        dxu = dqt.dqt_bitlinear_bwd_dx_img(t["dgu"][:, I:], img_gu[0][I:], t["s_u"])
        sr = [dqt.sr_stream(seed=seed, tensor_id=j) for j in range(3)]
        dqt.dqt_bitlinear_bwd_dw_update_group(
            [{"dY": t["dgu"], "Xdq": xd, "W": t["W_gu"], "m": t["m_gu"], "v": t["v_gu"], "N0": I,
              "s_w0": t["s_g"], "s_w1": t["s_u"], "sr0": sr[0], "sr1": sr[1],
              "W_img_next": img_gu[1]},
             {"dY": t["dd"], "Xdq": hd, "W": t["W_d"], "m": t["m_d"], "v": t["v_d"],
              "s_w0": t["s_d"], "sr0": sr[2], "W_img_next": img_d[1]}], hp, g)
        img_gu.reverse()  # the next step reads the images that this update wrote
        img_d.reverse()
        return {"gu": gu, "y": y, "dh": dh, "dxg": dxg, "dxu": dxu, "codes": (t["W_gu"], t["W_d"]),
                "m": (t["m_gu"], t["m_d"]), "v": (t["v_gu"], t["v_d"])}
    if kind == "update":
        dqt.dqt_sr_update(t["grad"], t["W"], t["s_w"], t["m"], t["v"], _hp(s),
                          dqt.sr_stream(seed=s["seed"], tensor_id=3), case["bits"])
        return {"codes": t["W"], "m": t["m"], "v": t["v"]}
    if kind == "ops":
        y, rstd = dqt.dqt_rmsnorm_bf16(t["x"], t["w"], NORM_EPS)
        r = dqt.dqt_rope_bf16(t["q"], t["cs"])
        h = dqt.dqt_swiglu_bf16(t["g"], t["u"])
        dg, du = dqt.dqt_swiglu_bwd_bf16(t["g"], t["u"], t["dh"])
        dq = dqt.dqt_rope_bf16(r, t["cs"], inverse=True)
        dx, dw = dqt.dqt_rmsnorm_bwd_bf16(t["x"], t["w"], rstd, t["dy"])
        return {"y": y, "r": r, "h": h, "dg": dg, "du": du, "dq": dq, "dx": dx, "dw": dw}
    if kind == "loss":
        lse, rows = dqt.dqt_cross_entropy_fwd_bf16(t["logits"], t["targets"])
        d = dqt.dqt_cross_entropy_bwd_bf16(t["logits"], t["targets"], lse, t["scale"])
        return {"lse": lse, "rows": rows, "dlogits": d}
    if kind == "logits":
        with torch.no_grad():
            return s["model"](t["ids"])
    p = s["train"]
    p.replay()
    return {"loss": p.loss, "grads": [w.grad for w in p.model.dense_parameters()],
            "layers": [(b.codes, b.m, b.v) for b in p.model.bitlinear_layers()]}


# ---------------------------------------------------------------------------
# 64 bits
# ---------------------------------------------------------------------------
def _quant64(x, act):
    """Activation codes, their scales, and the dequantised activation as the
    weight gradient reads it (bf16), in 64 bits.  The scale and the product
    that decide a code are single precision by the method's definition."""
    top = 448.0 if act == "fp8" else 127.0
    s = (top / x.float().abs().amax(-1, keepdim=True).clamp_min(1e-5).double()).float()
    p = x.float() * s
    if act == "fp8":
        q = p.clamp(-448.0, 448.0).to(torch.float8_e4m3fn).float()
    else:
        q = p.round().clamp_(-128.0, 127.0)
    return q.double(), s.double(), (q / s).to(torch.bfloat16).double()


def _step64(x, dy, W, s_w, act):
    """(y, dx, gradient) of one BitLinear in 64 bits."""
    q, s, xd = _quant64(x, act)
    c, d = W.double(), dy.double()
    return (q @ c.t()) / (s * s_w), (d @ c) / s_w, d.t() @ xd


def _adam64(grad, m, v):
    return (BETAS[0] * m.double() + (1 - BETAS[0]) * grad,
            BETAS[1] * v.double() + (1 - BETAS[1]) * grad.square())


class _Model64:
    """The decoder in 64 bits on a model's weights: activation codes as above,
    straight through in the backward."""

    def __init__(self, model, case):
        self.case = case
        self.p = [p.detach().double().requires_grad_() for p in model.dense_parameters()]
        self.named = dict(zip((n for n, _ in model.named_parameters() if not n.endswith("_anchor")),
                              self.p))
        self.blocks = [{n: b.int8_codes().double() / b.s_w for n, b in
                        (("q", k.q), ("k", k.k), ("v", k.v), ("o", k.o), ("gate", k.gate),
                         ("up", k.up), ("down", k.down))} for k in model.blocks]

    def lin(self, x, w, store):
        q, s, xd = _quant64(x.detach(), "int8")
        y = (x + (q / s - x).detach()) @ w.t()
        if y.requires_grad:
            y.register_hook(lambda d: store.append(
                d.reshape(-1, d.shape[-1]).t() @ xd.reshape(-1, xd.shape[-1])))
        return y

    def norm(self, x, w):
        return x / (x.square().mean(-1, keepdim=True) + NORM_EPS).sqrt() * w

    def __call__(self, ids):
        c, n = self.case, self.named
        B, S = ids.shape
        hd = c["D"] // c["H"]
        inv = 1.0 / THETA ** (torch.arange(0, hd, 2, device="cuda", dtype=torch.float64) / hd)
        rot = torch.polar(torch.ones((), dtype=torch.float64, device="cuda"),
                          torch.outer(torch.arange(S, device="cuda", dtype=torch.float64), inv))

        def rope(x):
            z = torch.view_as_complex(x.reshape(B, S, c["H"], hd // 2, 2).contiguous())
            return torch.view_as_real(z * rot[:, None]).reshape(B, S, c["H"], hd).transpose(1, 2)

        x = n["embed"][ids]
        self.grads = []
        hide = torch.ones((S, S), dtype=torch.bool, device="cuda").triu(1)
        for i, w in enumerate(self.blocks):
            st = {k: [] for k in w}
            self.grads.append(st)
            a = self.norm(x, n["blocks.%d.attn_norm.weight" % i])
            q, k = rope(self.lin(a, w["q"], st["q"])), rope(self.lin(a, w["k"], st["k"]))
            v = self.lin(a, w["v"], st["v"]).view(B, S, c["H"], hd).transpose(1, 2)
            p = (q @ k.transpose(-1, -2) / math.sqrt(hd)).masked_fill(hide, -math.inf).softmax(-1)
            x = x + self.lin((p @ v).transpose(1, 2).reshape(B, S, c["D"]), w["o"], st["o"])
            a = self.norm(x, n["blocks.%d.mlp_norm.weight" % i])
            x = x + self.lin(F.silu(self.lin(a, w["gate"], st["gate"]))
                             * self.lin(a, w["up"], st["up"]), w["down"], st["down"])
        return self.norm(x, n["norm.weight"]) @ n["head"].t()


def exact(case, seed):
    """What ``run`` returns on a new state, in 64 bits; None for codes that a
    random draw decides."""
    kind, t = case["kind"], _tensors(case, seed)
    if kind == "steps":  # the gradient is every step's; y and dx follow from the drawn codes
        g = t["dy"].double().t() @ _quant64(t["x"], "int8")[2]
        m, v = t["m"], t["v"]
        for _ in range(case["steps"]):
            m, v = _adam64(g, m, v)
        return {"y": None, "dx": None, "codes": None, "m": m, "v": v}
    if kind == "layer":
        layer = _module(case, seed, t)
        y, dx, g = _step64(t["x"], t["dy"], layer.int8_codes(), layer.s_w, case["act"])
        if case["optimizer"] == "adamw":
            state = _adam64(g, t["m"], t["v"])
        else:  # the first step: the statistics are the means themselves
            g2 = g.square() + 1e-30
            state = (g2.mean(1), g2.mean(0))
        return {"y": y, "dx": dx, "codes": None, "state": state}
    if kind == "codes":
        q, s, _ = _quant64(t["x"], "int8")
        y, dx, g = _step64(t["x"], t["dy"], t["W"], t["s_w"], "int8")
        m, v = _adam64(g, t["m"], t["v"])
        return {"xq": q.to(torch.int8), "s_x": s[:, 0], "y": y, "dx": dx, "codes": None, "m": m, "v": v}
    if kind == "mlp":
        I, W = case["I"], t["W_gu"]
        g, dxg, gg = _step64(t["x"], t["dgu"][:, :I], W[:I], t["s_g"], "int8")
        u, dxu, gu = _step64(t["x"], t["dgu"][:, I:], W[I:], t["s_u"], "int8")
        y, dh, gd = _step64(t["h"], t["dd"], t["W_d"], t["s_d"], "int8")
        a, b = _adam64(torch.cat((gg, gu)), t["m_gu"], t["v_gu"]), _adam64(gd, t["m_d"], t["v_d"])
        return {"gu": torch.cat((g, u), 1), "y": y, "dh": dh, "dxg": dxg, "dxu": dxu,
                "codes": (None, None), "m": (a[0], b[0]), "v": (a[1], b[1])}
    if kind == "update":
        m, v = _adam64(t["grad"].double(), t["m"], t["v"])
        return {"codes": None, "m": m, "v": v}
    if kind == "ops":
        x, w = t["x"].double().requires_grad_(), t["w"].double().requires_grad_()
        y = x / (x.square().mean(-1, keepdim=True) + NORM_EPS).sqrt() * w
        dx, dw = torch.autograd.grad(y, (x, w), t["dy"].double())
        g, u = t["g"].double().requires_grad_(), t["u"].double().requires_grad_()
        h = F.silu(g) * u
        dg, du = torch.autograd.grad(h, (g, u), t["dh"].double())
        q, rot = t["q"].double(), torch.view_as_complex(t["cs"].double())[:, None]
        z = torch.view_as_complex(q.view(*q.shape[:-1], -1, 2)) * rot
        r = torch.view_as_real(z).flatten(-2)
        dq = torch.view_as_real(z * rot.conj()).flatten(-2)
        return {"y": y.detach(), "r": r, "h": h.detach(), "dg": dg, "du": du, "dq": dq, "dx": dx,
                "dw": dw}
    if kind == "loss":
        x = t["logits"].double()
        lse = x.logsumexp(-1)
        rows = torch.arange(case["M"], device="cuda")
        d = (x - lse[:, None]).exp_()
        d[rows, t["targets"]] -= 1.0
        return {"lse": lse, "rows": lse - x[rows, t["targets"]], "dlogits": d.mul_(t["scale"].double())}
    m = _Model64(_decoder(case, seed), case)
    if kind == "logits":
        with torch.no_grad():
            return m(t["ids"])
    loss = F.cross_entropy(m(t["ids"]).flatten(0, 1), t["targets"].flatten())
    grads = torch.autograd.grad(loss, m.p)
    layers = []
    for st in m.grads:
        for k in ("q", "k", "v", "o", "gate", "up", "down"):
            g = st[k][0]
            layers.append((None,) + _adam64(g, torch.zeros_like(g), torch.zeros_like(g)))
    return {"loss": loss.detach(), "grads": list(grads), "layers": layers}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "steps":
        T, K, N, n = case["T"], case["K"], case["N"], case["steps"]
        return {"bytes": n * (4 * T * (K + N) + (2 + 2 + 16) * N * K), "flops": 6.0 * n * T * K * N}
    if kind in ("layer", "codes"):
        T, K, N = case["T"], case["K"], case["N"]
        code = 0.25 if case.get("packed") else 1.0
        state = 8 * (N + K) if case.get("optimizer") == "adafactor" else 16 * N * K
        b = 4 * T * (K + N) + 2 * code * N * K + state
        if kind == "codes":
            b += T * (K + 4)  # the activation codes are an output here
        return {"bytes": b, "flops": 6.0 * T * K * N}
    if kind == "mlp":
        T, H, I = case["T"], case["H"], case["I"]
        # in: x, h, dgu, dd; out: gu, y, dh, dxg, dxu; codes and moments both ways, images once
        return {"bytes": 2 * T * (H + I + 2 * I + H) + 2 * T * (2 * I + H + I + 2 * H) + 3 * H * I * (18 + 4),
                "flops": 18.0 * T * H * I}
    if kind == "update":
        return {"bytes": 22 * case["n"], "flops": 0}
    if kind == "ops":
        R, D, I = case["B"] * case["S"], case["D"], case["I"]
        # x, dy, q in, y, r, dq, dx out; g, u, dh in, h, dg, du out
        return {"bytes": 2 * R * (3 * D + 4 * D + 6 * I), "flops": 0}
    if kind == "loss":
        return {"bytes": 4 * case["M"] * case["V"], "flops": 0}
    D, I, V, L, S = case["D"], case["I"], case["V"], case["layers"], case["S"]
    T, P = case["B"] * S, L * (4 * D * D + 3 * D * I)
    attn = 2.0 * T * S * D * L  # causal: half of the two products
    if kind == "logits":
        return {"bytes": 2 * T * D + P + 2 * V * D + 2 * T * V, "flops": 2.0 * T * (P + V * D) + attn}
    return {"bytes": 18 * P + 10 * V * D + 4 * T * V, "flops": 6.0 * T * (P + V * D) + 3.5 * attn}


def tolerance(case):
    kind = case["kind"]
    # y is exact integer arithmetic with one rounding to bf16 (int8 codes);
    # dx and the FP8 y are fp32 sums rounded once to bf16, so another order of
    # sums moves a few values by one bf16 step; codes: the share of draws that
    # a gradient's last bits decide
    if kind in ("steps", "layer", "codes", "mlp"):
        return {"rel": 2e-3, "max": 0.05, "differ": 1e-4}
    if kind == "update":
        return {"rel": 1e-6, "max": 1e-5, "differ": 1e-6}
    if kind == "ops":
        return {"rel": 2e-3, "max": 0.05}
    if kind == "loss":
        return {"rel": 2e-3, "max": 0.05}
    # a whole model: one layer's rounding moves activation codes in all that follow
    if kind == "logits":
        return {"rel": 2e-2, "max": 0.3}
    return {"rel": 3e-2, "max": 0.9, "differ": 5e-3}
