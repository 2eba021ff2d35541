"""The workloads this library is timed on, through its public entry points.

A case is a dict of plain values.  `kind` names the call:

  qlinear   one dptq_qlinear call: rotate, quantize, integer GEMM, scales (Sections 2, 4.2)
  shared    dptq_qlinear_quantize once, then dptq_qlinear_gemm for each layer that reads the
            same activations (q, k, v of one attention block)
  stack     the four projection groups (q|k|v, o, gate|up, down) of consecutive decoder
            layers, replayed as one CUDA graph: the body of a decode or prefill step
  rotquant  dptq_rotate_quant_act: codes and scales in the public format
  kv4       dptq_kv4_quantize over a layer's K cache, groups of 128
  policy    dptq_sensitivity_policy over the layers' residual states

Projection sizes, block Hadamard sizes, bit masks and outlier patterns are those of
paper_2606_12487_gb300/inputs.py (LLaMA-2-7B decode, LLaMA-3-8B and LLaMA-2-13B prefill,
LLaMA-2-70B, the single 256 -> 512 layer).  Inputs are drawn on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_2606_12487_gb300 import dptq

DEV = "cuda"
W_STD = 0.02
POLICY_EPS, POLICY_TAU_JR, POLICY_TAU_SNR = 1e-6, 0.1, 20.0


def listed():
    return [
        # The smallest layer, 16 tokens: launch latency.
        dict(name="single_m16_a4", kind="qlinear", M=16, N=512, K=256, B=256, bits=4, acts="fixed", rh=False),
        # LLaMA-2-7B down for one sequence: one token, blocks of 256, a long K.
        dict(name="decode_down_m1_a4", kind="qlinear", M=1, N=4096, K=11008, B=256, bits=4, acts="channels", rh=False),
        # LLaMA-2-7B q|k|v of a sensitive (8-bit) layer, 8 sequences.
        dict(name="decode_qkv_m8_a8", kind="qlinear", M=8, N=12288, K=4096, B=4096, bits=8, acts="channels", rh=False),
        # Two LLaMA-2-7B layers (8-bit, then 4-bit) of a decode step at 32 sequences.
        dict(name="decode_stack_m32", kind="stack", M=32, d=4096, kv=4096, f=11008, B=4096, Bd=256, mask="84",
             acts="channels"),
        # LLaMA-2-70B down at 64 sequences: the longest K.
        dict(name="batch_70b_down_m64_a4", kind="qlinear", M=64, N=8192, K=28672, B=4096, bits=4, acts="first",
             rh=False),
        # LLaMA-3-8B q, k, v of a short prompt of odd length, one quantization for all
        # three, randomized Hadamard.
        dict(name="prompt_qkv_shared_m333_a4", kind="shared", M=333, Ns="4096,1024,1024", K=4096, B=2048, bits=4,
             acts="tokens", rh=True),
        # LLaMA-3-8B prefill of 2048 tokens: gate|up (wide N) and down (long K).
        dict(name="prefill_gateup_m2048_a4", kind="qlinear", M=2048, N=28672, K=4096, B=2048, bits=4, acts="tokens",
             rh=False),
        dict(name="prefill_down_m2048_a4", kind="qlinear", M=2048, N=4096, K=14336, B=2048, bits=4, acts="tokens",
             rh=False),
        # LLaMA-2-70B down, four sequences of 2048 tokens, 8-bit layer: the largest.
        dict(name="prefill_70b_down_m8192_a8", kind="qlinear", M=8192, N=8192, K=28672, B=4096, bits=8, acts="first",
             rh=False),
        # LLaMA-2-13B down activations for another GEMM: 13 blocks of 1024 and a tail of 512.
        dict(name="rotquant_m1024_a8", kind="rotquant", M=1024, K=13824, B=1024, bits=8, acts="student", rh=False),
        # LLaMA-2-7B K cache of 8192 tokens (32 heads of 128).
        dict(name="kv4_8192x4096", kind="kv4", rows=8192, cols=4096),
        # Calibration statistics of 32 layers over 512 tokens of width 4096.
        dict(name="policy_32x512x4096", kind="policy", L=32, T=512, d=4096, bits=4),
    ]


# (K, N, B) of the projections of the workloads above, and plain sizes.
_PROJ = [(256, 512, 256), (4096, 12288, 4096), (4096, 4096, 4096), (4096, 22016, 4096), (11008, 4096, 256),
         (4096, 4096, 2048), (4096, 1024, 2048), (4096, 28672, 2048), (14336, 4096, 2048), (5120, 5120, 1024),
         (5120, 27648, 1024), (13824, 5120, 1024), (8192, 10240, 4096), (8192, 8192, 4096), (8192, 57344, 4096),
         (28672, 8192, 4096), (11008, 4096, 4096), (1536, 2064, 512), (3072, 3072, 1024), (2080, 1008, 128)]
_ACTS = {4096: "channels", 2048: "tokens", 1024: "student", 256: "channels"}
_MAX_FLOPS = 2.0 * 8192 * 8192 * 28672


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["qlinear"] * 8 + ["shared", "stack", "rotquant", "rotquant", "kv4", "policy"])
    bits = rng.choice([4, 4, 8])
    if kind == "stack":
        # Small decoder geometries, so that a drawn case stays cheap.
        d = rng.choice([2048, 4096, 4096])
        f = rng.choice([5632, 11008]) if d == 2048 else rng.choice([11008, 14336])
        return dict(kind=kind, M=_log_int(rng, 1, 256), d=d, kv=rng.choice([d, d // 4]), f=f,
                    B=rng.choice([d, d // 2]), Bd=rng.choice([256, 512]), mask=rng.choice(["4", "84", "44"]),
                    acts="channels")
    if kind == "shared":
        K = rng.choice([4096, 5120, 8192])
        n = rng.choice([1024, K])
        return dict(kind=kind, M=_log_int(rng, 1, 4096), Ns="%d,%d,%d" % (K, n, n), K=K, B=rng.choice([1024, 512]),
                    bits=bits, acts=rng.choice(["tokens", "student"]), rh=rng.random() < 0.5)
    if kind == "rotquant":
        K, _, B = rng.choice(_PROJ)
        return dict(kind=kind, M=_log_int(rng, 1, 8192), K=K, B=B, bits=bits, acts=_ACTS.get(B, "channels"),
                    rh=rng.random() < 0.3)
    if kind == "kv4":
        return dict(kind=kind, rows=_log_int(rng, 1, 65536), cols=128 * rng.choice([1, 8, 32, 40, 64]))
    if kind == "policy":
        return dict(kind=kind, L=rng.choice([8, 32, 40]), T=_log_int(rng, 16, 1024), d=rng.choice([1024, 4096, 5120, 8192]),
                    bits=bits)
    K, N, B = rng.choice(_PROJ)
    cap = min(8192, max(64, int(_MAX_FLOPS / (2.0 * N * K))))
    return dict(kind=kind, M=_log_int(rng, 1, cap), N=N, K=K, B=B, bits=bits, acts=_ACTS.get(B, "channels"),
                rh=rng.random() < 0.2)


# ------------------------------------------------------------------------------ inputs
def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + 7919 * stream + 1)
    return g


def _host_rng(seed, stream):
    return np.random.default_rng([int(seed), stream])


def _half(x):
    return x.clamp_(-65504.0, 65504.0).to(torch.float16)


def _acts(M, K, kind, seed, stream):
    """fp16 activations [M, K] with massive-activation outliers in fixed channels, in a few
    tokens, in the first token of a sequence, or with heavy tails."""
    g, r = _gen(seed, stream), _host_rng(seed, stream)
    x = torch.randn((M, K), generator=g, device=DEV)
    ch = lambda n: torch.from_numpy(np.sort(r.choice(K, n, replace=False))).to(DEV)  # noqa: E731
    if kind == "fixed":
        x[:, ch(2)] *= 50.0
    elif kind == "channels":
        x[:, ch(4)] *= 100.0
    elif kind == "tokens":
        rows = torch.from_numpy(np.sort(r.choice(M, max(1, M // 100), replace=False))).to(DEV)
        c = ch(3)
        x[rows[:, None], c[None, :]] *= 300.0
    elif kind == "first":
        c = ch(2)
        rows = torch.arange(0, M, 2048, device=DEV)
        x[rows[:, None], c[None, :]] *= 1000.0
    elif kind == "student":   # Student's t with 3 degrees of freedom
        q = torch.zeros_like(x)
        for _ in range(3):
            q += torch.randn((M, K), generator=g, device=DEV).square_()
        x *= (q / 3.0).rsqrt_()
    return _half(x)


def _weights(N, K, seed, stream):
    return _half(torch.randn((N, K), generator=_gen(seed, stream), device=DEV).mul_(W_STD))


def _signs(K, seed):
    return _host_rng(seed, 999).choice(np.array([-1, 1], dtype=np.int8), K)


def _pack(W, B, signs):
    return dptq.dptq_pack_weights(W, B) if signs is None else dptq.dptq_pack_weights_rh(W, B, signs)


def _stack_groups(case):
    """(K, N, B, bits) of each projection group of the stack, in order."""
    d, kv, f = case["d"], case["kv"], case["f"]
    out = []
    for m in case["mask"]:
        b = int(m)
        out += [(d, d + 2 * kv, case["B"], b), (d, d, case["B"], b), (d, 2 * f, case["B"], b), (f, d, case["Bd"], b)]
    return out


def _out(M, N):
    return torch.empty((M, N), dtype=torch.float16, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "kv4":
        R, C = case["rows"], case["cols"]
        kv = torch.randn((R, C), generator=_gen(seed, 0), device=DEV)
        kv[:, torch.from_numpy(_host_rng(seed, 0).choice(C, max(1, C // 64), replace=False)).to(DEV)] *= 10.0
        return dict(case=case, kv=_half(kv), codes=torch.empty((R, C // 2), dtype=torch.uint8, device=DEV),
                    scales=torch.empty((R, C // 128), dtype=torch.float32, device=DEV))
    if kind == "policy":
        L, T, d = case["L"], case["T"], case["d"]
        x, dx = _policy_inputs(case, seed)
        return dict(case=case, x=x, dx=dx, jr=torch.empty((L,), dtype=torch.float64, device=DEV),
                    snr=torch.empty((L,), dtype=torch.float64, device=DEV),
                    bits=torch.empty((L,), dtype=torch.uint8, device=DEV))
    if kind == "rotquant":
        M, K, bits = case["M"], case["K"], case["bits"]
        st = dict(case=case, x=_acts(M, K, case["acts"], seed, 0),
                  codes=torch.empty((M, K // 2), dtype=torch.uint8, device=DEV) if bits == 4
                  else torch.empty((M, K), dtype=torch.int8, device=DEV),
                  scales=torch.empty((M,), dtype=torch.float32, device=DEV))
        if case["rh"]:
            st["signs"] = torch.from_numpy(_signs(K, seed)).to(DEV)
        return st
    if kind == "qlinear":
        signs = _signs(case["K"], seed) if case["rh"] else None
        layer = _pack(_weights(case["N"], case["K"], seed, 1), case["B"], signs)
        return dict(case=case, layer=layer, x=_acts(case["M"], case["K"], case["acts"], seed, 0),
                    out=_out(case["M"], case["N"]))
    if kind == "shared":
        signs = _signs(case["K"], seed) if case["rh"] else None
        Ns = [int(n) for n in case["Ns"].split(",")]
        layers = [_pack(_weights(n, case["K"], seed, 1 + i), case["B"], signs) for i, n in enumerate(Ns)]
        return dict(case=case, layers=layers, x=_acts(case["M"], case["K"], case["acts"], seed, 0),
                    outs=[_out(case["M"], n) for n in Ns])
    # stack: the graph of one step, as a serving loop keeps it
    M, groups = case["M"], _stack_groups(case)
    dptq.dptq_reserve(M, max(K for K, _, _, _ in groups), 0)
    layers = [dptq.dptq_pack_weights(_weights(N, K, seed, 100 + i), B) for i, (K, N, B, _) in enumerate(groups)]
    xs = [_acts(M, K, case["acts"], seed, i) for i, (K, _, _, _) in enumerate(groups)]
    outs = [_out(M, N) for _, N, _, _ in groups]

    def step():
        for layer, x, (_, _, _, bits), out in zip(layers, xs, groups, outs):
            dptq.dptq_qlinear(layer, x, bits, out)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    return dict(case=case, layers=layers, xs=xs, outs=outs, graph=graph)


def _policy_inputs(case, seed):
    """Residual states and updates; the first two layers and the last one carry large
    updates in four channels."""
    L, T, d = case["L"], case["T"], case["d"]
    g, r = _gen(seed, 0), _host_rng(seed, 0)
    x = torch.randn((L, T, d), generator=g, device=DEV)
    dx = torch.randn((L, T, d), generator=g, device=DEV).mul_(0.05)
    ch = torch.from_numpy(np.sort(r.choice(d, 4, replace=False))).to(DEV)
    for l in (0, 1, L - 1):
        dx[l][:, ch] += 40.0 * torch.randn((T, 4), generator=g, device=DEV)
    return x, dx


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "qlinear":
        dptq.dptq_qlinear(state["layer"], state["x"], case["bits"], state["out"])
        return state["out"]
    if kind == "stack":
        state["graph"].replay()
        return state["outs"]
    if kind == "shared":
        dptq.dptq_qlinear_quantize(state["layers"][0], state["x"], case["bits"])
        for layer, out in zip(state["layers"], state["outs"]):
            dptq.dptq_qlinear_gemm(layer, case["M"], case["bits"], out)
        return state["outs"]
    if kind == "rotquant":
        if "signs" in state:
            dptq.dptq_rotate_quant_act_rh(state["x"], case["B"], case["bits"], state["signs"], state["codes"],
                                          state["scales"])
        else:
            dptq.dptq_rotate_quant_act(state["x"], case["B"], case["bits"], state["codes"], state["scales"])
        return [state["codes"], state["scales"]]
    if kind == "kv4":
        dptq.dptq_kv4_quantize(state["kv"], 128, state["codes"], state["scales"])
        return [state["codes"], state["scales"]]
    dptq.dptq_sensitivity_policy(state["x"], state["dx"], case["bits"], POLICY_EPS, POLICY_TAU_JR, POLICY_TAU_SNR,
                                 state["jr"], state["snr"], state["bits"])
    return [state["jr"], state["snr"], state["bits"]]


# ------------------------------------------------------------------------------ work
def _linear_work(M, K, N, x_bytes=True):
    return N * K // 2 + 4 * N + 2 * M * N + (2 * M * K if x_bytes else 0), 2.0 * M * N * K


def work(case):
    kind = case["kind"]
    if kind == "qlinear":
        b, f = _linear_work(case["M"], case["K"], case["N"])
        return {"bytes": b, "flops": f}
    if kind == "shared":
        parts = [_linear_work(case["M"], case["K"], int(n), i == 0) for i, n in enumerate(case["Ns"].split(","))]
    elif kind == "stack":
        parts = [_linear_work(case["M"], K, N) for K, N, _, _ in _stack_groups(case)]
    else:
        parts = None
    if parts is not None:
        return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}
    if kind == "rotquant":
        M, K = case["M"], case["K"]
        return {"bytes": 2 * M * K + M * K * case["bits"] // 8 + 4 * M, "flops": M * K * math.log2(case["B"])}
    if kind == "kv4":
        n = case["rows"] * case["cols"]
        return {"bytes": 2 * n + n // 2 + 4 * n // 128, "flops": 3.0 * n}
    n = case["L"] * case["T"] * case["d"]
    return {"bytes": 8 * n, "flops": 12.0 * n}


def tolerance(case):
    kind = case["kind"]
    if kind in ("qlinear", "shared", "stack"):
        # The accumulators are whole numbers; fp32 scales and one rounding to fp16 remain:
        # 2.1e-4 off 64 bits as a 2-norm, at most one fp16 ulp (2^-10) in a value.  A code at
        # a rounding tie (1e-5 of them at most) may move by one: less than 0.02 of a row.
        return {"rel": 1e-3, "max": 0.02}
    if kind == "rotquant":
        # Codes but for ties, scales to a rounding of 32 bits.
        return {"rel": 3e-7, "max": 5e-7, "differ": 2e-5}
    if kind == "kv4":
        # The quantizer is defined step by step in fp32: nothing is left open.
        return {"rel": 1e-7, "max": 2e-7, "differ": 0.0}
    # Norms and errors in 32 bits per element and token, means in 64.
    return {"rel": 1e-5, "max": 3e-5, "differ": 0.0}


# ------------------------------------------------------------------------------ 64-bit results
def _paley(p):
    """Paley's first construction of order p (p - 1 prime, 3 mod 4): H = I + S."""
    q = p - 1
    chi = np.full(q, -1)
    chi[[(i * i) % q for i in range(1, q)]] = 1
    chi[0] = 0
    H = np.eye(p)
    H[0, 1:] += 1
    H[1:, 0] -= 1
    i = np.arange(q)
    H[1:, 1:] += chi[(i[None, :] - i[:, None]) % q]
    return torch.from_numpy(H).to(DEV)


def _is_prime(n):
    return n > 1 and all(n % d for d in range(2, int(n ** 0.5) + 1))


def _fwht(x):
    """Rows of x [.., n] times the Sylvester Hadamard matrix of order n."""
    n, h = x.shape[-1], 1
    shape = x.shape
    while h < n:
        v = x.reshape(-1, n // (2 * h), 2, h)
        x = torch.cat([v[:, :, :1] + v[:, :, 1:], v[:, :, :1] - v[:, :, 1:]], dim=2).reshape(shape)
        h *= 2
    return x


def _rotate64(x, B, signs):
    """x R in 64 bits: whole blocks of B, then a tail of 2^k or p 2^k elements."""
    x = x.double()
    if signs is not None:
        x = x * torch.from_numpy(signs).to(DEV)
    M, K = x.shape
    r = K % B
    parts = []
    if K - r:
        parts.append((_fwht(x[:, :K - r].reshape(-1, B)) / math.sqrt(B)).reshape(M, K - r))
    if r:
        t, odd, tz = x[:, K - r:], r, 0
        while odd % 2 == 0:
            odd, tz = odd // 2, tz + 1
        p = 1 if odd == 1 else next(odd << m for m in range(2, tz + 1) if _is_prime((odd << m) - 1))
        z = _fwht(t.reshape(M, p, r // p)) if r // p > 1 else t.reshape(M, p, r // p)
        if p > 1:
            z = torch.einsum("mab,ac->mcb", z, _paley(p))
        parts.append((z / math.sqrt(r)).reshape(M, r))
    return torch.cat(parts, dim=1)


def _quant64(y, bits):
    """Codes and scales per row: the quantizer reads y and keeps s = max|y| / qmax in 32
    bits, which is its definition."""
    y = y.float()
    qmax = float(2 ** (bits - 1) - 1)
    s = y.abs().amax(dim=1, keepdim=True) / qmax
    c = torch.where(s > 0, torch.clamp(torch.round(y / torch.where(s > 0, s, torch.ones_like(s))), -qmax - 1, qmax),
                    torch.zeros_like(y))
    return c, s.squeeze(1)


def _rows(fn, x, step):
    return [fn(x[i:i + step]) for i in range(0, x.shape[0], step)]


def _quantized64(x, B, signs, bits):
    """Codes [rows, K] as float64 and scales as float64, a few thousand rows at a time."""
    step = max(1, (1 << 26) // x.shape[1])
    got = _rows(lambda v: _quant64(_rotate64(v, B, signs), bits), x, step)
    return torch.cat([c.to(torch.float32) for c, _ in got]), torch.cat([s for _, s in got]).double()


def _linear64(x, W, B, signs, bits):
    a, sa = _quantized64(x, B, signs, bits)
    w, sw = _quantized64(W, B, signs, 4)
    del W
    out = torch.empty((x.shape[0], w.shape[0]), dtype=torch.float64, device=DEV)
    a = a.double()
    step = max(1, (1 << 27) // w.shape[1])
    for i in range(0, w.shape[0], step):
        out[:, i:i + step] = (a @ w[i:i + step].double().t()) * sa[:, None] * sw[None, i:i + step]
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "kv4":
        kv = prepare(case, seed)["kv"]
        am = kv.double().reshape(kv.shape[0], -1, 128).abs().amax(dim=2)
        return [None, am / 7.0]
    if kind == "policy":
        x, dx = _policy_inputs(case, seed)
        jrs, snrs = [], []
        for l in range(case["L"]):
            u = x[l] + dx[l]
            c, s = _quant64(u, case["bits"])
            err = (c.double() * s.double()[:, None] - dx[l].double()) - x[l].double()
            nx, nd = x[l].double().square().sum(1), dx[l].double().square().sum(1)
            jrs.append((nd.sqrt() / (nx.sqrt() + POLICY_EPS)).mean())
            snrs.append((10.0 * torch.log10(nx / (err.square().sum(1) + POLICY_EPS))).mean())
        return [torch.stack(jrs), torch.stack(snrs), None]
    if kind == "stack":
        return [_linear64(_acts(case["M"], K, case["acts"], seed, i), _weights(N, K, seed, 100 + i), B, None, bits)
                for i, (K, N, B, bits) in enumerate(_stack_groups(case))]
    signs = _signs(case["K"], seed) if case["rh"] else None
    x = _acts(case["M"], case["K"], case["acts"], seed, 0)
    if kind == "rotquant":
        y = _rows(lambda v: _rotate64(v, case["B"], signs).abs().amax(dim=1), x, max(1, (1 << 26) // case["K"]))
        return [None, torch.cat(y) / float(2 ** (case["bits"] - 1) - 1)]
    if kind == "shared":
        return [_linear64(x, _weights(int(n), case["K"], seed, 1 + i), case["B"], signs, case["bits"])
                for i, n in enumerate(case["Ns"].split(","))]
    return _linear64(x, _weights(case["N"], case["K"], seed, 1), case["B"], signs, case["bits"])
