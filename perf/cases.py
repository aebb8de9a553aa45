"""The work that a user of this library has it do, as cases that can be timed and compared.

Every case is one use of the public binding (paper_2501_19090_gb300.pifa) on synthetic operands of
the recipe in paper_2501_19090_gb300/inputs.py: activations N(0, 1), W_p ~ N(0, 1/r), C of the
spread that compressed layers show (standard deviation 0.18), random index sets; all drawn on the
GPU from the case's seed. Row pitches are rounded up to 8 elements, as the library asks.

kinds:
  eager        one forward call, launched from Python: a program without CUDA graphs
  decode       a decode step over `layers` layers of one shape, captured once into a CUDA graph and
               replayed per token batch, as a serving loop does
  mlp          gate and up (grouped, one call) and down over `layers` blocks; T <= 64 replayed from a
               CUDA graph, larger T launched directly
  prefill      one forward call over a long token batch
  backward     the gradients of one layer (fine-tuning): dX, dW_p, dC
  accumulate   the M method's calibration of one layer: cleared accumulators, `batches` batches
  compress     Algorithm 1 on the GPU, float64
  reconstruct  the M method's two solves, float64
"""
import math

import torch

from paper_2501_19090_gb300 import pifa as P

DEV = "cuda"


def _layer(name, kind, m, n, r, T, **more):
    return dict({"name": name, "kind": kind, "m": m, "n": n, "r": r, "T": T}, **more)


def listed():
    return [
        # the smallest layer of the configurations, one call from Python: latency and host work
        _layer("eager_tiny_T16", "eager", 256, 256, 128, 16, c="bf16"),
        # decode of a 7B model's attention projections, a batch of 8 sequences
        _layer("decode_attn7b_T8", "decode", 4096, 4096, 2048, 8, c="bf16", layers=4),
        # batched decode at a rank that is no multiple of a tile, C stored as fp16
        _layer("decode_r2458_fp16_T50", "decode", 4096, 4096, 2458, 50, c="fp16", layers=3),
        # decode of a 70B model's gate / up projections: the benchmark's headline workload
        _layer("decode_gateup70b_T16", "decode", 28672, 8192, 4096, 16, c="bf16", layers=2),
        # a 7B MLP block for one sequence: gate and up grouped, then down
        _layer("mlp7b_T1", "mlp", 11008, 4096, 2048, 1, c="bf16", layers=2),
        # a 7B attention projection over a long prompt
        _layer("prefill_attn7b_T2048", "prefill", 4096, 4096, 2048, 2048, c="bf16"),
        # a short, ragged prompt through a 7B down projection
        _layer("prefill_down7b_T300", "prefill", 4096, 11008, 2048, 300, c="bf16"),
        # a 70B attention projection over a long prompt
        _layer("prefill_qo70b_T4096", "prefill", 8192, 8192, 4096, 4096, c="bf16"),
        # a fine-tuning step's gradients of a 7B attention projection
        _layer("backward_attn7b_T2048", "backward", 4096, 4096, 2048, 2048),
        # the M method's calibration of a 7B attention layer, two batches of 2048 samples
        _layer("accumulate_attn7b_T2048", "accumulate", 4096, 4096, 0, 2048, lam=0.25, batches=2),
        # Algorithm 1 on a 7B attention layer
        _layer("compress_attn7b", "compress", 4096, 4096, 2048, 0),
        # the M method's solves for a layer half that size
        _layer("reconstruct_2048", "reconstruct", 2048, 2048, 1024, 0, alpha=1e-3),
    ]


# ---- draws ---------------------------------------------------------------------------------------
_SHAPES = [(4096, 4096), (11008, 4096), (4096, 11008), (8192, 8192), (28672, 8192)]
_FRACTIONS = (0.25, 0.4, 0.5, 0.6, 0.75)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, hi=8192):
    """A layer of the model shapes at one of the swept rank fractions, or any layer at any rank."""
    if rng.random() < 0.5:
        m, n = rng.choice([s for s in _SHAPES if max(s) <= 4 * hi])
        return m, n, int(rng.choice(_FRACTIONS) * min(m, n) + 0.5)
    m, n = _log(rng, 256, hi), _log(rng, 256, hi)
    return m, n, max(8, int(rng.uniform(0.2, 0.8) * min(m, n)))


def draw(rng):
    kind = rng.choice(["eager", "decode", "decode", "decode", "mlp", "prefill", "prefill", "prefill", "backward",
                       "backward", "accumulate", "compress", "reconstruct"])
    c = rng.choice(["bf16", "bf16", "fp16"])
    if kind == "eager":
        m, n, r = _shape(rng, 4096)
        return {"kind": kind, "m": m, "n": n, "r": r, "T": _log(rng, 1, 64), "c": c}
    if kind == "decode":
        m, n, r = _shape(rng)
        return {"kind": kind, "m": m, "n": n, "r": r, "T": _log(rng, 1, 64), "c": c, "layers": rng.choice([1, 2, 3, 4])}
    if kind == "mlp":  # the grouped call asks for (m - r) % 128 == 0 and r % 8 == 0
        n = 128 * _log(rng, 4, 40)
        r = 128 * max(1, int(rng.uniform(0.25, 0.75) * n / 128))
        m = r + 128 * _log(rng, 8, 90)
        return {"kind": kind, "m": m, "n": n, "r": r, "T": _log(rng, 1, 2048), "c": c, "layers": rng.choice([1, 2])}
    if kind in ("prefill", "backward"):
        m, n, r = _shape(rng)
        most = 4096 * 4096 * (8192 + 4096) // (1 if kind == "prefill" else 3)
        T = _log(rng, 65, 4096)
        T = max(65, min(T, most // (r * (n + m - r))))
        case = {"kind": kind, "m": m, "n": n, "r": r, "T": T}
        return dict(case, c=c) if kind == "prefill" else case
    if kind == "accumulate":
        return {"kind": kind, "m": _log(rng, 256, 4096), "n": _log(rng, 256, 4096), "r": 0, "T": _log(rng, 64, 2048),
                "lam": rng.choice([0.0, 0.25, 0.5, 1.0]), "batches": rng.choice([1, 2])}
    if kind == "compress":
        m, n = _log(rng, 256, 4096), _log(rng, 256, 4096)
        return {"kind": kind, "m": m, "n": n, "r": max(8, int(rng.uniform(0.25, 0.5) * min(m, n))), "T": 0}
    m, n = _log(rng, 256, 2048), _log(rng, 256, 2048)
    return {"kind": kind, "m": m, "n": n, "r": max(8, int(rng.uniform(0.25, 0.5) * min(m, n))), "T": 0,
            "alpha": rng.choice([0.0, 1e-3])}


# ---- inputs --------------------------------------------------------------------------------------
def _pad8(v):
    return (v + 7) // 8 * 8


def _padded(rows, cols, dtype, gen=None, scale=1.0):
    """A rows x cols tensor of pitch round_up(cols, 8): N(0, scale^2) values, or zeros without `gen`."""
    t = torch.zeros((rows, _pad8(cols)), dtype=dtype, device=DEV)[:, :cols]
    if gen is not None:
        t.copy_(torch.randn((rows, cols), device=DEV, generator=gen).mul_(scale))
    return t


def _index_sets(gen, m, r, groups=1):
    piv, nonp = [], []
    for g in range(groups):
        p = torch.randperm(m, device=DEV, generator=gen)
        piv.append(p[:r].sort().values + g * m)
        nonp.append(p[r:].sort().values + g * m)
    return torch.cat(piv).to(torch.int32), torch.cat(nonp).to(torch.int32)


def _cdt(case):
    return torch.float16 if case.get("c") == "fp16" else torch.bfloat16


def _one_layer(gen, m, n, r, cdt, groups=1):
    piv, nonp = _index_sets(gen, m, r, groups)
    return {"Wp": _padded(groups * r, n, torch.bfloat16, gen, r ** -0.5),
            "C": _padded(groups * (m - r), r, cdt, gen, 0.18), "piv": piv, "nonp": nonp, "groups": groups, "m": m}


def _with_io(gen, layer, X, workspace_bytes):
    T = X.shape[0]
    layer["X"] = X
    layer["Y"] = _padded(T, layer["groups"] * layer["m"], torch.bfloat16)
    layer["ws"] = torch.empty(workspace_bytes + 256, dtype=torch.uint8, device=DEV)
    return layer


def _forward(a, stream=None):
    if a["groups"] > 1:
        return P.pifa_forward_grouped(a["groups"], a["X"], a["Wp"], a["C"], a["piv"], a["nonp"], Y=a["Y"],
                                      workspace_tensor=a["ws"], stream=stream)
    return P.pifa_forward(a["X"], a["Wp"], a["C"], a["piv"], a["nonp"], Y=a["Y"], workspace_tensor=a["ws"], stream=stream)


def _captured(calls):
    """The calls captured into a CUDA graph, after one eager pass."""
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    for a in calls:
        _forward(a, stream)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for a in calls:
            _forward(a, stream)
    torch.cuda.synchronize()
    return graph


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    kind, m, n, r, T = (case[k] for k in ("kind", "m", "n", "r", "T"))
    bf16 = torch.bfloat16
    state = {"case": case}
    if kind in ("eager", "decode", "prefill", "mlp"):
        cdt = _cdt(case)
        code = P.PIFA_DTYPE_FP16 if case.get("c") == "fp16" else P.PIFA_DTYPE_BF16
        calls = []
        for _ in range(case.get("layers", 1)):
            if kind == "mlp":
                calls.append(_with_io(gen, _one_layer(gen, m, n, r, cdt, 2), _padded(T, n, bf16, gen),
                                      P.pifa_workspace_size_grouped(2, T, m, n, r, code)))
                calls.append(_with_io(gen, _one_layer(gen, n, m, r, cdt), _padded(T, m, bf16, gen),
                                      P.pifa_workspace_size(T, n, m, r, c_dtype=code)))
            else:
                calls.append(_with_io(gen, _one_layer(gen, m, n, r, cdt), _padded(T, n, bf16, gen),
                                      P.pifa_workspace_size(T, m, n, r, c_dtype=code)))
        state["calls"] = calls
        if kind == "decode" or (kind == "mlp" and T <= 64):
            state["graph"] = _captured(calls)
    elif kind == "backward":
        state.update(_one_layer(gen, m, n, r, bf16))
        state["X"], state["dY"] = _padded(T, n, bf16, gen), _padded(T, m, bf16, gen)
        state["ws"] = torch.empty(P.pifa_backward_workspace_size(T, m, n, r) + 256, dtype=torch.uint8, device=DEV)
    elif kind == "accumulate":
        state["Xu"] = [_padded(T, n, bf16, gen) for _ in range(case["batches"])]
        state["Xo"] = []
        for Xu in state["Xu"]:  # the dense flow's input: close to the compressed one's
            Xo = _padded(T, n, bf16)
            Xo.copy_(Xu.float() + 0.1 * torch.randn((T, n), device=DEV, generator=gen))
            state["Xo"].append(Xo)
        state["W"] = _padded(m, n, bf16, gen, n ** -0.5)
        state["XXt"], state["YtXt"] = _padded(n, n, torch.float32), _padded(m, n, torch.float32)
        state["ws"] = torch.empty(P.pifa_m_accumulate_workspace_size(T, m, n) + 256, dtype=torch.uint8, device=DEV)
    elif kind == "compress":
        state["U"] = torch.randn((m, r), device=DEV, generator=gen).mul_(r ** -0.5).double()
        state["V"] = torch.randn((n, r), device=DEV, generator=gen).mul_(r ** -0.5).double()
    elif kind == "reconstruct":  # accumulators of 2 n samples, as the calibration leaves them
        Xu = torch.randn((2 * n, n), device=DEV, generator=gen).to(bf16).float()
        Xo = (Xu + 0.1 * torch.randn((2 * n, n), device=DEV, generator=gen)).to(bf16).float()
        W = (torch.randn((m, n), device=DEV, generator=gen) * n ** -0.5).to(bf16)
        state["XXt"], state["YtXt"], state["W"] = (_padded(n, n, torch.float32), _padded(m, n, torch.float32),
                                                   _padded(m, n, bf16))
        state["XXt"].copy_(Xu.t() @ Xu)
        state["YtXt"].copy_(((0.25 * Xo + 0.75 * Xu) @ W.float().t()).t() @ Xu)
        state["W"].copy_(W)
        state["V"] = torch.randn((n, r), device=DEV, generator=gen).mul_(n ** -0.5).double()
    else:
        raise ValueError(kind)
    return state


# ---- one pass ------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("eager", "decode", "prefill", "mlp"):
        if "graph" in state:
            state["graph"].replay()
        else:
            for a in state["calls"]:
                _forward(a)
        return [a["Y"] for a in state["calls"]]
    if kind == "backward":
        dX, dWp, dC = P.pifa_backward(state["X"], state["Wp"], state["C"], state["piv"], state["nonp"], state["dY"],
                                      workspace_tensor=state["ws"])
        return {"dX": dX, "dWp": dWp, "dC": dC}
    if kind == "accumulate":
        state["XXt"].zero_()
        state["YtXt"].zero_()
        for Xo, Xu in zip(state["Xo"], state["Xu"]):
            P.pifa_m_accumulate(Xo, Xu, state["W"], case["lam"], state["XXt"], state["YtXt"],
                                workspace_tensor=state["ws"])
        return {"XXt": state["XXt"], "YtXt": state["YtXt"]}
    if kind == "compress":
        piv, nonp, Wp, C, _ = P.pifa_compress_device(state["U"], state["V"])
        return {"piv": piv, "nonp": nonp, "Wp": Wp, "C": C}
    U_r, V_r = P.pifa_m_reconstruct(state["XXt"], state["YtXt"], state["V"], W=state["W"], alpha=case["alpha"])
    return {"U_r": U_r, "V_r": V_r}


# ---- what a pass cannot do without ---------------------------------------------------------------
def _forward_work(T, m, n, r, groups=1):
    """Weights, indices, X and Y once; the multiply-adds of Algorithm 2 (the indices are int32)."""
    g = groups
    return (2 * g * r * (n + m - r) + 2 * T * (n + g * m) + 4 * g * m, 2 * T * g * r * (n + m - r))


def work(case):
    kind, m, n, r, T = (case[k] for k in ("kind", "m", "n", "r", "T"))
    if kind in ("eager", "decode", "prefill"):
        b, f = _forward_work(T, m, n, r)
        k = case.get("layers", 1)
        return {"bytes": k * b, "flops": k * f}
    if kind == "mlp":
        (b0, f0), (b1, f1) = _forward_work(T, m, n, r, 2), _forward_work(T, n, m, r)
        return {"bytes": case["layers"] * (b0 + b1), "flops": case["layers"] * (f0 + f1)}
    if kind == "backward":  # X, dY, W_p, C and the indices in, dX (bf16), dW_p and dC (fp32) out
        return {"bytes": 2 * T * (2 * n + m) + 6 * r * n + 6 * r * (m - r) + 4 * m,
                "flops": 2 * T * r * (2 * n + 2 * (m - r))}
    if kind == "accumulate":  # X_o and X_u per batch, W once, the accumulators written once
        k = case["batches"]
        return {"bytes": k * 4 * T * n + 2 * m * n + 4 * (n * n // 2 + m * n),
                "flops": k * (T * n * (n + 1) + 4 * T * m * n)}
    if kind == "compress":  # Gram, Cholesky, Z = U L, greedy steps, R^-1, C, W_p; U, V in, W_p, C, indices out
        greedy = 6 * (m * r * r / 2 - r ** 3 / 6)
        return {"bytes": 8 * (m * r + n * r + r * n + (m - r) * r) + 4 * m,
                "flops": r * r * n + m * r * r + greedy + 2 * r ** 3 / 3 + (m - r) * r * r + 2 * r * r * n}
    # reconstruct: the two normal matrices, their Cholesky solves and the products of Eqs. 4 and 8
    return {"bytes": 4 * (n * n // 2 + m * n) + 2 * m * n + 16 * n * r + 8 * m * r,
            "flops": 2 * n * n * r + n * r * r + 2 * m * n * r + r ** 3 / 3 + 2 * m * r * r + m * r * r + r ** 3 / 3
            + 2 * m * n * r + 2 * r * r * n + n ** 3 / 3 + 2 * n * n * r}


def tolerance(case):
    """About four times what the outputs differ by from the 64-bit values rounded to their type
    (forward and dX: rel 3.6e-4, one bf16 step at most; the fp32 accumulators 1.8e-5, the float64
    paths 1.4e-13 and 4.2e-14)."""
    kind = case["kind"]
    if kind in ("eager", "decode", "prefill", "mlp", "backward"):
        return {"rel": 1.5e-3, "max": 3e-2}
    if kind == "accumulate":
        return {"rel": 8e-5, "max": 2e-4}
    if kind == "compress":
        return {"rel": 2e-12, "max": 1e-10}
    return {"rel": 1e-12, "max": 1e-11}


# ---- the same in 64 bits ---------------------------------------------------------------------------
def _exact_forward(a):
    X, m = a["X"].double(), a["m"]
    G = a["groups"]
    Y = torch.empty((X.shape[0], G * m), dtype=torch.float64, device=DEV)
    r, q = a["Wp"].shape[0] // G, a["C"].shape[0] // G
    for g in range(G):
        Yp = X @ a["Wp"][g * r:(g + 1) * r].double().t()
        Y[:, a["piv"][g * r:(g + 1) * r].long()] = Yp
        Y[:, a["nonp"][g * q:(g + 1) * q].long()] = Yp @ a["C"][g * q:(g + 1) * q].double().t()
    return Y


def _exact_compress(U, V):
    """Greedy selection with every residual norm recomputed, then W_p = W'[I] and C = W'[I^c] W_p^+."""
    m, r = U.shape
    Z = U @ torch.linalg.qr(V, mode="r").R.t()  # the row inner products of U V^T
    R, chosen = Z.clone(), torch.zeros(m, dtype=torch.bool, device=DEV)
    for _ in range(r):
        norms = R.square().sum(1)
        p = norms.masked_fill(chosen, -1.0).argmax().view(1)
        chosen[p] = True
        q = R.index_select(0, p)[0]
        q = q / q.norm()
        R -= torch.outer(R @ q, q)
    piv, nonp = chosen.nonzero().view(-1), (~chosen).nonzero().view(-1)
    C = torch.linalg.solve(Z[piv].t(), Z[nonp].t()).t()
    return {"piv": piv.to(torch.int32), "nonp": nonp.to(torch.int32), "Wp": U[piv] @ V.t(), "C": C.contiguous()}


def exact(case, seed):
    state = prepare(case, seed)
    kind = case["kind"]
    if kind in ("eager", "decode", "prefill", "mlp"):
        return [_exact_forward(a) for a in state["calls"]]
    if kind == "backward":
        X, dY, Wp, C = (state[k].double() for k in ("X", "dY", "Wp", "C"))
        dYnp = dY[:, state["nonp"].long()]
        dYp = dY[:, state["piv"].long()] + dYnp @ C
        return {"dX": dYp @ Wp, "dWp": dYp.t() @ X, "dC": dYnp.t() @ (X @ Wp.t())}
    if kind == "accumulate":
        XXt = YtXt = 0.0
        lam, W = case["lam"], state["W"].double()
        for Xo, Xu in zip(state["Xo"], state["Xu"]):
            Xo, Xu = Xo.double(), Xu.double()
            XXt = XXt + Xu.t() @ Xu
            YtXt = YtXt + ((lam * Xo + (1.0 - lam) * Xu) @ W.t()).t() @ Xu
        b = torch.arange(case["n"], device=DEV) // 128  # the 128 x 128 blocks on and above the diagonal
        return {"XXt": XXt.masked_fill(b[:, None] > b[None, :], 0.0), "YtXt": YtXt}
    if kind == "compress":
        return _exact_compress(state["U"], state["V"])
    A = state["XXt"].double().triu()
    A = A + A.triu(1).t()
    B, V, alpha = state["YtXt"].double(), state["V"], case["alpha"]
    U_r = torch.linalg.solve(V.t() @ A @ V, (B @ V).t()).t()
    if alpha:
        B = B + alpha * state["W"].double()
        A = A + alpha * torch.eye(A.shape[0], dtype=torch.float64, device=DEV)
    V_r = torch.linalg.solve(A, torch.linalg.solve(U_r.t() @ U_r, U_r.t() @ B).t())
    return {"U_r": U_r.contiguous(), "V_r": V_r.contiguous()}
