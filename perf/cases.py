"""What this library is asked to do in earnest, as cases that can be timed.

A case is a plain dict.  Its "kind" says which public calls one pass makes:

  linear   quantize_act, then mp_gemm: one quantized linear layer
  conv     quantize_act, then mp_conv2d: one quantized convolution
  mlp      quantize_act, mp_gemm writing the next layer's codes from its
           epilogue, then that layer's mp_gemm: an MLP block
  phase2   FakeQuantMLP.forward: master weights and activations quantized on
           the fly, then the integer products, layer by layer

Weights are packed once in prepare() (phase2 packs them in every pass); output
buffers are kept by the program, as a serving loop keeps them.  With "graph"
the pass is captured once and replayed, as decode loops do.
"""
import math

import numpy as np
import torch

from paper_2311_14114_gb300 import soniq as sq
from paper_2311_14114_gb300.phase2 import FakeQuantMLP

OUT = {"f16": torch.float16, "bf16": torch.bfloat16}


def _linear(name, M, K, N, lo, hi, frac, scale="tensor", out="f16", outliers=0, gain=1.0, signed=False, sub_k=0,
            graph=False):
    c = dict(kind="linear", M=M, K=K, N=N, lo=lo, hi=hi, frac=frac, scale=scale, out=out, outliers=outliers,
             gain=gain, signed=signed, sub_k=sub_k, graph=graph)
    return dict(name=name, **c) if name else c


def _conv(name, batch, H, W, C, C_out, R, stride, pad, lo, hi, frac):
    c = dict(kind="conv", batch=batch, H=H, W=W, C=C, C_out=C_out, R=R, stride=stride, pad=pad, lo=lo, hi=hi,
             frac=frac)
    return dict(name=name, **c) if name else c


def _mlp(name, M, K, N, K_out, lo, hi, frac, outliers, gain):
    c = dict(kind="mlp", M=M, K=K, N=N, K_out=K_out, lo=lo, hi=hi, frac=frac, outliers=outliers, gain=gain)
    return dict(name=name, **c) if name else c


def _phase2(name, M, K, N, K_out, lo, hi, frac):
    c = dict(kind="phase2", M=M, K=K, N=N, K_out=K_out, lo=lo, hi=hi, frac=frac)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one small layer of a small network: latency and launches
        _linear("linear_64x512x512", 64, 512, 512, 2, 8, 0.25, outliers=4, gain=10.0),
        # one token through an LLM's up-projection, the decode loop replayed as a graph
        _linear("decode_m1", 1, 4096, 11008, 3, 6, 0.15, graph=True),
        # a few sequences decoded together, one scale per token, plain calls
        _linear("decode_m4_row", 4, 4096, 11008, 3, 6, 0.15, scale="row"),
        # a batch of sequences decoded together
        _linear("decode_m16", 16, 4096, 11008, 3, 6, 0.15, graph=True),
        # a short prompt (an odd number of tokens), one scale per token, bf16 outputs
        _linear("prompt_m137_row_bf16", 137, 4096, 11008, 3, 6, 0.15, scale="row", out="bf16"),
        # signed activations with scale runs along K (group-wise scales) at ragged sizes
        _linear("runs_1001x3000x1111", 1001, 3000, 1111, 4, 8, 0.25, scale="row", signed=True, sub_k=128),
        # a transformer MLP block whose up-projection writes the down-projection's codes
        _mlp("mlp_16384x768x3072", 16384, 768, 3072, 768, 2, 8, 0.20, 8, 20.0),
        # a residual block's 3x3 convolution on a batch of images
        _conv("conv_64x14x14x256", 64, 14, 14, 256, 256, 3, 1, 1, 4, 8, 0.30),
        # the same of an early layer on one image: latency
        _conv("conv_1x56x56x64", 1, 56, 56, 64, 64, 3, 1, 1, 4, 8, 0.30),
        # a long prompt through a square layer: the benchmark's headline workload
        _linear("sweep_lo4_hi8_f25", 8192, 4096, 4096, 4, 8, 0.25),
        # the same with 2-bit codes in most channels
        _linear("sweep_lo2_hi8_f10", 8192, 4096, 4096, 2, 8, 0.10),
        # one fine-tuning forward of an LLM's MLP block: fp32 master weights quantized on the fly
        _phase2("phase2_2048x4096x11008", 2048, 4096, 11008, 4096, 3, 6, 0.15),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _bits(rng):
    return rng.choice([1, 2, 3, 4]), rng.choice([4, 6, 8])


def draw(rng):
    kind = rng.choices(["linear", "runs", "conv", "mlp", "phase2"], [6, 1, 2, 1, 1])[0]
    lo, hi = _bits(rng)
    if kind == "linear":
        while True:
            M, K, N = _log_int(rng, 1, 16384), _log_int(rng, 256, 8192), _log_int(rng, 64, 11008)
            if M * K * N <= 8192 * 4096 * 4096:
                break
        if rng.random() < 0.5:
            K = -(-K // 64) * 64        # most layers have round widths, some do not
            N = -(-N // 64) * 64
        return _linear(None, M, K, N, lo, hi, rng.choice([0.0, 0.1, 0.15, 0.25, 0.5, 1.0]),
                       scale=rng.choice(["tensor", "tensor", "row", "calibrated"]), out=rng.choice(["f16", "bf16"]),
                       outliers=rng.choice([0, 4]), gain=10.0, graph=M <= 32 and rng.random() < 0.5)
    if kind == "runs":
        return _linear(None, _log_int(rng, 64, 2048), _log_int(rng, 512, 4096), _log_int(rng, 256, 2048), lo, hi,
                       rng.choice([0.1, 0.25, 0.5]), scale=rng.choice(["tensor", "row"]), signed=rng.random() < 0.5,
                       sub_k=rng.choice([128, 256]))
    if kind == "conv":
        while True:
            batch, H, C, C_out = _log_int(rng, 1, 64), rng.randint(7, 56), _log_int(rng, 32, 512), _log_int(rng, 32, 512)
            W, R, stride = max(7, H + rng.choice([0, 0, 1, -3])), rng.choice([1, 3, 3, 5]), rng.choice([1, 1, 2])
            if (H // stride) * (W // stride) * batch * C * C_out * R * R <= 3 * 10 ** 10 and batch * H * W * C <= 5 * 10 ** 7:
                break
        return _conv(None, batch, H, W, C, C_out, R, stride, R // 2, lo, hi, rng.choice([0.1, 0.3, 0.5]))
    if kind == "mlp":
        K = _log_int(rng, 256, 1024)
        return _mlp(None, _log_int(rng, 256, 16384), K, 4 * K, K, lo, hi, rng.choice([0.1, 0.2, 0.5]), 8, 20.0)
    K = _log_int(rng, 512, 4096)
    return _phase2(None, _log_int(rng, 64, 2048), K, min(11008, int(2.7 * K)), K, lo, hi, rng.choice([0.1, 0.15, 0.25]))


# ---- inputs -----------------------------------------------------------------

def _assignment(rng, K, frac, outliers):
    """Outlier channels and a random choice of others take the high precision;
    the permutation lists the low channels, then the high ones, each ascending."""
    n_hi = int(np.floor(frac * K + 0.5))
    order = rng.permutation(K)
    high = np.zeros(K, dtype=bool)
    high[order[:n_hi]] = True
    out = order[: min(outliers, n_hi)]
    return np.concatenate([np.flatnonzero(~high), np.flatnonzero(high)]).astype(np.int32), [K - n_hi, n_hi], out


def _inputs(case, seed):
    """Everything random about a case: activations, and per layer weights and permutation."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32)

    if case["kind"] == "conv":
        C, taps = case["C"], case["R"] ** 2
        perm, count, _ = _assignment(rng, C, case["frac"], 0)
        X = normal(case["batch"], case["H"], case["W"], C).relu_().half()
        return X, [dict(W=normal(case["C_out"], taps, C) * math.sqrt(2.0 / (taps * C)), perm=perm, count=count)]
    widths = [case["K"], case["N"]] + ([case["K_out"]] if case["kind"] != "linear" else [])
    layers, out = [], None
    for i, (K, N) in enumerate(zip(widths[:-1], widths[1:])):
        perm, count, o = _assignment(rng, K, case["frac"], case.get("outliers", 0) if i == 0 else 0)
        layers.append(dict(W=normal(N, K) * 0.02, perm=perm, count=count))
        out = o if i == 0 else out
    A = normal(case["M"], case["K"])
    if len(out):
        A[:, torch.as_tensor(out, device="cuda")] *= case["gain"]
    return A.half(), layers


def _mlp_scales(case):
    """The down-projection's calibrated input scales: a few standard deviations of the up-projection's outputs."""
    return [0.08 * math.sqrt(case["K"])] * 2


def _calibrated(A, perm, count):
    """Calibrated scales of a layer's input, a little under what the data reach (the largest values clip)."""
    p = torch.as_tensor(perm.astype(np.int64), device=A.device)
    return torch.stack([A[:, p[a:b]].abs().max().float() * 0.9 if b > a else torch.ones((), device=A.device)
                        for a, b in ((0, count[0]), (count[0], count[0] + count[1]))])


def prepare(case, seed):
    x, layers = _inputs(case, seed)
    kind = case["kind"]
    bits = [case["lo"], case["hi"]]
    if kind == "phase2":
        return dict(kind=kind, X=x, model=FakeQuantMLP([dict(l, bits=bits) for l in layers], case["M"]))
    first = layers[0]
    if kind == "conv":
        lay = sq.Layout(first["perm"], first["count"], bits, pad_unit=32)
        Wp, s_w = sq.pack_weights(lay, first["W"])
        cd = sq.conv_desc(case["batch"], case["H"], case["W"], case["C_out"], case["R"], case["R"],
                          (case["stride"],) * 2, (case["pad"],) * 2)
        rows = x.reshape(-1, case["C"])
        P, Q = sq.conv_out_hw(cd)
        return dict(kind=kind, lay=lay, cd=cd, A=rows, Wp=Wp, s_w=s_w, s_a=torch.empty(2, device="cuda"),
                    Ap=torch.empty(rows.shape[0], lay.row_bytes(), dtype=torch.uint8, device="cuda"),
                    Y=torch.empty(case["batch"], P, Q, case["C_out"], dtype=torch.float16, device="cuda"))
    M = case["M"]
    act = (sq.ACT_SIGNED,) * 2 if case.get("signed") else (sq.ACT_UNSIGNED,) * 2
    lay = sq.Layout(first["perm"], first["count"], bits, act_kind=act, sub_k=case.get("sub_k", 0))
    Ap = torch.empty(M, lay.row_bytes(), dtype=torch.uint8, device="cuda")
    if kind == "mlp":
        second = layers[1]
        lay2 = sq.Layout(second["perm"], second["count"], bits)
        order = torch.as_tensor(sq.next_layer_row_order(lay2), device="cuda")
        W1 = torch.where((order >= 0)[:, None], first["W"][order.clamp(min=0)], 0.0)
        Wp, s_w = sq.pack_weights(lay, W1.contiguous())
        Wp2, s_w2 = sq.pack_weights(lay2, second["W"])
        s2 = torch.tensor(_mlp_scales(case), dtype=torch.float32, device="cuda")
        return dict(kind=kind, lay=lay, lay2=lay2, A=x, Wp=Wp, s_w=s_w, Wp2=Wp2, s_w2=s_w2, s2=s2, Ap=Ap,
                    s_a=torch.empty(2, device="cuda"), nxt=sq.NextLayer(lay2, s2, M=M),
                    Y=torch.empty(M, case["K_out"], dtype=torch.float16, device="cuda"))
    Wp, s_w = sq.pack_weights(lay, first["W"])
    scale = case["scale"]
    s_a = (_calibrated(x, first["perm"], first["count"]) if scale == "calibrated"
           else torch.empty(lay.scale_shape(M if scale == "row" else None), dtype=torch.float32, device="cuda"))
    state = dict(kind=kind, lay=lay, A=x, Wp=Wp, s_w=s_w, s_a=s_a, Ap=Ap, scale=scale,
                 Y=torch.empty(M, case["N"], dtype=OUT[case["out"]], device="cuda"))
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _linear_pass(state)
        torch.cuda.current_stream().wait_stream(side)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            _linear_pass(state)
        state["graph"] = graph
    return state


# ---- one pass ---------------------------------------------------------------

def _linear_pass(s):
    sq.quantize_act(s["lay"], s["A"], s["scale"], s_a=s["s_a"], Ap=s["Ap"])
    sq.mp_gemm(s["lay"], s["Ap"], s["s_a"], s["Wp"], s["s_w"], s["scale"], Y=s["Y"])


def run(s):
    kind = s["kind"]
    if kind == "phase2":
        m = s["model"]
        m.forward(s["X"])
        return dict(y=m.Y, Ap=m.Ap, s_a=m.s_a, Wp=m.Wp, s_w=m.s_w)
    if kind == "linear":
        if "graph" in s:
            s["graph"].replay()
        else:
            _linear_pass(s)
        return dict(y=s["Y"], Ap=s["Ap"], s_a=s["s_a"])
    sq.quantize_act(s["lay"], s["A"], s_a=s["s_a"], Ap=s["Ap"])
    if kind == "conv":
        sq.mp_conv2d(s["lay"], s["cd"], s["Ap"], s["s_a"], s["Wp"], s["s_w"], Y=s["Y"])
        return dict(y=s["Y"], Ap=s["Ap"], s_a=s["s_a"])
    nxt = s["nxt"]
    sq.mp_gemm(s["lay"], s["Ap"], s["s_a"], s["Wp"], s["s_w"], next=nxt, write_y=False)
    sq.mp_gemm(s["lay2"], nxt.Ap, s["s2"], s["Wp2"], s["s_w2"], "calibrated", Y=s["Y"])
    return dict(y=s["Y"], Ap=s["Ap"], s_a=s["s_a"], next_Ap=nxt.Ap)


# ---- the least one pass has to do -------------------------------------------

def _code_bytes(case, K):
    n_hi = int(np.floor(case["frac"] * K + 0.5))
    return ((K - n_hi) * case["lo"] + n_hi * case["hi"]) / 8.0


def work(case):
    if case["kind"] == "conv":
        P = (case["H"] + 2 * case["pad"] - case["R"]) // case["stride"] + 1
        Q = (case["W"] + 2 * case["pad"] - case["R"]) // case["stride"] + 1
        pixels, out, taps = case["batch"] * case["H"] * case["W"], case["batch"] * P * Q, case["R"] ** 2
        code = _code_bytes(case, case["C"])
        return dict(bytes=pixels * (2 * case["C"] + code) + case["C_out"] * (taps * code + 8) + 2 * out * case["C_out"],
                    flops=2.0 * out * case["C_out"] * taps * case["C"])
    M, K, N = case["M"], case["K"], case["N"]
    code = _code_bytes(case, K)
    if case["kind"] == "linear":
        runs = -(-K // case["sub_k"]) if case["sub_k"] else 2
        rows = M if case["scale"] == "row" else 1
        return dict(bytes=M * (2 * K + code) + N * (code + 4 * runs) + 4 * runs * rows + 2 * M * N, flops=2.0 * M * N * K)
    K2 = case["K_out"]
    code2 = _code_bytes(case, N)
    flops = 2.0 * M * N * (K + K2)
    if case["kind"] == "mlp":
        return dict(bytes=M * (2 * K + code + code2) + N * (code + 8) + K2 * (code2 + 8) + 2 * M * K2, flops=flops)
    return dict(bytes=M * (2 * K + code + code2 + 2 * N + 2 * K2) + 4 * N * K + 4 * K2 * N + N * (code + 8) + K2 * (code2 + 8),
                flops=flops)


# ---- the same in 64 bits ----------------------------------------------------
# The codes are defined in 32 bits (a / s rounded, times 2^n - 1 rounded, then
# to the nearest integer, ties to even); everything after them is exact.

def _ranges(count, sub_k):
    """Per group the runs of packed positions that share a scale."""
    for g, (a, b) in enumerate(((0, count[0]), (count[0], count[0] + count[1]))):
        step = sub_k or max(b - a, 1)
        yield g, [(p, min(p + step, b)) for p in range(a, b, step)]


def _scaled(v, s):
    return torch.where(s > 0, v / torch.where(s > 0, s, 1.0), torch.zeros_like(v))


def _act_codes(v, s, n, signed):
    q = _scaled(v, s)
    if signed:
        return torch.clamp(torch.round(q * 2.0 ** (n - 1)), -(2.0 ** (n - 1)), 2.0 ** (n - 1) - 1), 2.0 ** (n - 1)
    return torch.clamp(torch.round(q * (2.0 ** n - 1)), 0, 2.0 ** n - 1), 2.0 ** n - 1


def _weight_codes(v, s, n):
    return torch.clamp(torch.round(_scaled(v, s) * 2.0 ** (n - 1)), -(2.0 ** (n - 1)), 2.0 ** (n - 1) - 1)


def _exact_layer(A, layer, bits, signed=False, sub_k=0, scale="tensor", given=None):
    """Outputs in 64 bits, activation scales, weight scales of one linear layer (A: the fp16 input)."""
    perm = torch.as_tensor(layer["perm"].astype(np.int64), device=A.device)
    Ag, Wg = A.float()[:, perm], layer["W"][:, perm]
    M, N = A.shape[0], Wg.shape[0]
    runs = [r for _, r in _ranges(layer["count"], sub_k)]
    nb = max(len(r) for r in runs) if sub_k else 1
    rows = M if scale == "row" else 1
    s_a, s_w = torch.zeros(rows, 2, nb, device=A.device), torch.zeros(N, 2, nb, device=A.device)
    y = torch.zeros(M, N, dtype=torch.float64, device=A.device)
    for g in (0, 1):
        for i, (a, b) in enumerate(runs[g]):
            va, vw, n = Ag[:, a:b], Wg[:, a:b], bits[g]
            s_w[:, g, i] = vw.abs().amax(1)
            s_a[:, g, i] = given[g] if given is not None else va.abs().amax(1) if scale == "row" else va.abs().max()
            u, L = _act_codes(va, s_a[:, g, i, None], n, signed)
            j = _weight_codes(vw, s_w[:, g, i, None], n)
            alpha = s_a[:, g, i, None].double() * s_w[None, :, g, i].double() / (L * 2.0 ** (n - 1))
            y += alpha * (u.double() @ j.double().T)
    shape = (2,) if not sub_k else (2, nb)
    return y, s_a.reshape(((M,) if scale == "row" else ()) + shape), s_w.reshape((N,) + shape)


def exact(case, seed):
    x, layers = _inputs(case, seed)
    bits = [case["lo"], case["hi"]]
    kind = case["kind"]
    if kind == "conv":
        layer, R = layers[0], case["R"]
        perm = torch.as_tensor(layer["perm"].astype(np.int64), device=x.device)
        X, W = x.float()[..., perm], layer["W"][..., perm]
        y, s_a = 0.0, torch.zeros(2, device=x.device)
        for g, runs in _ranges(layer["count"], 0):
            for a, b in runs:
                v, w, n = X[..., a:b], W[..., a:b], bits[g]
                s_a[g] = v.abs().max()
                s_w = w.abs().amax((1, 2))
                u, L = _act_codes(v, s_a[g], n, False)
                j = _weight_codes(w, s_w[:, None, None], n).double()
                u = torch.nn.functional.pad(u.double(), (0, 0, case["pad"], case["pad"], case["pad"], case["pad"]))
                st = case["stride"]
                P, Q = (u.shape[1] - R) // st + 1, (u.shape[2] - R) // st + 1
                acc = 0.0
                for t in range(R * R):
                    r, c = divmod(t, R)
                    acc = acc + u[:, r:r + (P - 1) * st + 1:st, c:c + (Q - 1) * st + 1:st] @ j[:, t].T
                y = y + acc * (s_a[g].double() * s_w.double() / (L * 2.0 ** (n - 1)))
        return dict(y=y, Ap=None, s_a=s_a)
    if kind == "linear":
        given = None
        if case["scale"] == "calibrated":
            given = _calibrated(x, layers[0]["perm"], layers[0]["count"])
        y, s_a, _ = _exact_layer(x, layers[0], bits, case["signed"], case["sub_k"], case["scale"], given)
        return dict(y=y, Ap=None, s_a=s_a if given is None else given)
    if kind == "mlp":
        y1, s_a, _ = _exact_layer(x, layers[0], bits)
        s2 = torch.tensor(_mlp_scales(case), dtype=torch.float32, device=x.device)
        y2, _, _ = _exact_layer(y1.half(), layers[1], bits, given=s2)
        return dict(y=y2, Ap=None, s_a=s_a, next_Ap=None)
    y1, s_a1, s_w1 = _exact_layer(x, layers[0], bits)
    y2, s_a2, s_w2 = _exact_layer(y1.half(), layers[1], bits)
    return dict(y=[y1, y2], Ap=None, s_a=[s_a1, s_a2], Wp=None, s_w=[s_w1, s_w2])
