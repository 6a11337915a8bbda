"""Workloads that time this library through its public entry points.

Each case is one whole job as a user's program runs it: a context made from an
initial tensor (or chain state), its steps, and the results read back; or one
call of the stand-alone FP64-grade GEMM.  The sizes are those of the benchmark
configurations in ``workloads`` and sizes between them.

Kinds of job:

* ``model`` -- HOTRG of a classical lattice model: ln Z per site and the spectrum
  of the first environment that is cut;
* ``sweep`` -- many instances with their own couplings and cuts in one context;
* ``chain`` -- HOTRG of an XXZ quantum chain along imaginary time, the same results;
* ``itebd`` -- ground-state iteration of a batch of XXZ chains;
* ``gemm``  -- the exact-slice GEMM on device matrices.

The modes whose contractions accumulate in FP32 (TF32, BF16X3, BF16X6) return
single precision, the precision of the sums behind the results; the others
return FP64.  Tensors and isometries are left out: they are fixed only up to an
orthogonal change of basis of the kept states.  So are the spectra of later
steps, which near the transition magnify rounding by the flow along the
temperature direction.
"""
import math

import numpy as np
import torch

import paper_2602_05900_gb300 as hotrg

BETA_C_ISING = 0.5 * math.log(1.0 + math.sqrt(2.0))
BETA_C_POTTS3 = math.log(1.0 + math.sqrt(3.0))
FP64_GRADE = ("fp64", "bf16xs")
# Cuts of the XXZ chains that keep whole multiplets of the spin symmetry (where a
# cut splits one, the kept states and so ln Z depend on the eigenvectors chosen
# inside it), or are large enough for that to be below the modes' accuracy.
CHAIN_CUTS = (6, 7, 8, 10, 13, 15, 18, 19, 22, 28, 30, 31, 32)


def listed():
    return [
        # plain FP64 reference job at the smallest cut: launches and latency
        {"name": "ising_d8_fp64", "kind": "model", "q": 2, "field": 0.0, "cut": 8, "steps": 20, "mode": "fp64"},
        # the headline job: one Ising instance to its thermodynamic limit
        {"name": "ising_d32_tf32", "kind": "model", "q": 2, "field": 0.0, "cut": 32, "steps": 30, "mode": "tf32"},
        # FP64-grade job on the tensor cores at a ragged cut
        {"name": "ising_d21_bf16xs", "kind": "model", "q": 2, "field": 0.0, "cut": 21, "steps": 18, "mode": "bf16xs"},
        # split products in a field at the large cut of the accuracy target
        {"name": "ising_field_d48_bf16x3", "kind": "model", "q": 2, "field": 0.01, "cut": 48, "steps": 12,
         "mode": "bf16x3"},
        # the largest bond dimension: three-state Potts, gigabytes of intermediates
        {"name": "potts3_d64_bf16x3", "kind": "model", "q": 3, "field": 0.0, "cut": 64, "steps": 9,
         "mode": "bf16x3"},
        # the batched coupling sweep: uneven cuts side by side
        {"name": "sweep24_tf32", "kind": "sweep", "count": 24, "cuts": "16,24,32,40", "steps": 12, "mode": "tf32"},
        # a quantum chain at finite temperature, small and ordinary cut
        {"name": "chain_d13_bf16xs", "kind": "chain", "tau": 0.03125, "time": 7, "space": 16, "cut": 13,
         "mode": "bf16xs"},
        {"name": "chain_d32_bf16xs", "kind": "chain", "tau": 0.03125, "time": 7, "space": 16, "cut": 32,
         "mode": "bf16xs"},
        # ground-state iteration: one chain at the paper's largest bond dimension,
        # and a batch at a middle one
        {"name": "itebd_1x_d30", "kind": "itebd", "chains": 1, "cut": 30, "updates": 30},
        {"name": "itebd_64x_d16", "kind": "itebd", "chains": 64, "cut": 16, "updates": 30},
        # an environment times a block of vectors (D = 48), the eigensolver's product
        {"name": "gemm_2304x64", "kind": "gemm", "m": 2304, "n": 64, "k": 2304, "pad": 0, "slices": 8},
        # a large general product of ragged sizes in padded rows
        {"name": "gemm_ragged_3k", "kind": "gemm", "m": 3001, "n": 2777, "k": 3203, "pad": 5, "slices": 8},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("model", "model", "model", "sweep", "chain", "chain", "itebd", "itebd", "gemm", "gemm"))
    if kind == "model":
        mode = rng.choice(("fp64", "tf32", "tf32", "bf16x3", "bf16x6", "bf16xs"))
        cut = _log_int(rng, 4, 20 if mode == "fp64" else 40)
        # the Potts cuts split doublets, which costs up to 1e-6: split products only
        potts = mode in ("bf16x3", "bf16x6") and cut >= 16
        return {"kind": kind, "q": rng.choice((2, 3)) if potts else 2, "field": rng.choice((0.0, 0.0, 0.01)), "cut": cut,
                "steps": rng.randint(8, 14 if mode in FP64_GRADE or cut > 32 else 24), "mode": mode}
    if kind == "sweep":
        cuts = sorted({_log_int(rng, 6, 32) for _ in range(rng.randint(1, 4))})
        return {"kind": kind, "count": _log_int(rng, 4, 24), "cuts": ",".join(map(str, cuts)),
                "steps": rng.randint(8, 12), "mode": "tf32"}
    if kind == "chain":
        return {"kind": kind, "tau": rng.choice((0.03125, 0.0625, 0.125)), "time": rng.randint(4, 7),
                "space": rng.randint(6, 16), "cut": rng.choice(CHAIN_CUTS), "mode": rng.choice(("bf16xs", "bf16xs", "fp64"))}
    if kind == "itebd":
        cut = _log_int(rng, 4, 48)
        return {"kind": kind, "chains": _log_int(rng, 1, 64), "cut": cut,
                "updates": rng.randint(10, 30 if cut <= 32 else 16)}
    return {"kind": kind, "m": _log_int(rng, 64, 3000), "n": _log_int(rng, 16, 3000), "k": _log_int(rng, 64, 3200),
            "pad": rng.choice((0, 0, 1, 7)), "slices": rng.choice((6, 7, 8, 8))}


# ---------------------------------------------------------------- inputs

def _rng(case, seed):
    return np.random.default_rng([20260205, int(seed) & 0x7FFFFFFF])


def _model_inputs(case, seed):
    """Inverse temperature within two per cent of the transition."""
    beta_c = BETA_C_ISING if case["q"] == 2 else BETA_C_POTTS3
    return beta_c * float(_rng(case, seed).uniform(0.98, 1.01))


def _sweep_inputs(case, seed):
    """Couplings over both phases, the cuts dealt out in turn."""
    cuts = [int(v) for v in case["cuts"].split(",")]
    betas = _rng(case, seed).uniform(0.35, 0.55, size=case["count"])
    return [float(b) for b in betas], [cuts[i % len(cuts)] for i in range(case["count"])]


def _chain_inputs(case, seed):
    """An antiferromagnetic chain of the XXZ family off its isotropic point."""
    return 1.0, float(_rng(case, seed).uniform(0.5, 0.9))


def _itebd_inputs(case, seed):
    """Couplings and a random normalised two-site cell for every chain."""
    rng, D, n = _rng(case, seed), case["cut"], case["chains"]
    couplings = np.stack([rng.uniform(0.5, 1.5, n), rng.uniform(0.5, 1.5, n), np.full(n, 0.05)], axis=1)
    P = rng.standard_normal((n, D, 2, D))
    Q = rng.standard_normal((n, D, 2, D))
    lam = -np.sort(-rng.uniform(0.1, 1.0, size=(n, D)), axis=1)
    return couplings, P, Q, lam / np.linalg.norm(lam, axis=1, keepdims=True)


def _gemm_inputs(case, seed):
    """Two matrices with rows of uneven size, in rows `pad` elements longer."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) & 0x7FFFFFFF)

    def matrix(rows, cols):
        a = torch.randn(rows, cols + case["pad"], dtype=torch.float64, device=dev, generator=g)
        a *= torch.exp(2.0 * torch.randn(rows, 1, dtype=torch.float64, device=dev, generator=g))
        return a[:, :cols]

    return matrix(case["m"], case["k"]), matrix(case["n"], case["k"])


def prepare(case, seed):
    kind, state = case["kind"], {"case": dict(case)}
    if kind == "gemm":
        state["a"], state["b"] = _gemm_inputs(case, seed)
        state["c"] = torch.empty(case["m"], case["n"], dtype=torch.float64, device="cuda")
        return state
    state["stream"] = torch.cuda.Stream()
    if kind == "model":
        beta = _model_inputs(case, seed)
        state["T0"] = hotrg.ising_tensor(beta, case["field"]) if case["q"] == 2 else hotrg.potts_tensor(case["q"], beta)
    elif kind == "sweep":
        betas, state["cuts"] = _sweep_inputs(case, seed)
        state["T0s"] = [hotrg.ising_tensor(b) for b in betas]
    elif kind == "chain":
        jxy, jz = _chain_inputs(case, seed)
        state["T0"] = hotrg.xxz_tensor(jxy, jz, case["tau"])
    else:
        state["couplings"], P, Q, lam = _itebd_inputs(case, seed)
        state["init"] = [(P[i], Q[i], lam[i]) for i in range(case["chains"])]
    return state


# ---------------------------------------------------------------- one pass

def _first_cut(case):
    """Index of the first step that discards states."""
    return next(i for i, (D, _, K) in enumerate(_dims(case)) if K < D * D)


def _results(case, h):
    ln_z, spectrum = np.float64(h.ln_z_per_site()), h.spectrum(_first_cut(case))
    if case["mode"] in FP64_GRADE:
        return {"ln_z": ln_z, "spectrum": spectrum}
    return {"ln_z": np.float32(ln_z), "spectrum": spectrum.astype(np.float32)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gemm":
        stream = torch.cuda.current_stream()
        return {"c": hotrg.dgemm_emu(state["a"], state["b"], state["c"], case["slices"], stream)}
    if kind == "model":
        with hotrg.Hotrg(state["T0"], case["cut"], case["mode"], state["stream"]) as h:
            h.run(case["steps"])
            return _results(case, h)
    if kind == "sweep":
        with hotrg.HotrgBatch(state["T0s"], state["cuts"], case["mode"], state["stream"]) as h:
            h.run(case["steps"])
            return {"ln_z": h.ln_z_per_site().astype(np.float32)}
    if kind == "chain":
        with hotrg.Hotrg(state["T0"], case["cut"], case["mode"], state["stream"]) as h:
            h.run_quantum(case["time"], case["space"])
            return _results(case, h)
    with hotrg.Itebd(state["couplings"], case["cut"], state["init"], state["stream"]) as h:
        h.step(case["updates"])
        return {"energy": h.energy(), "lam": h.lam(case["chains"] - 1)}


# ---------------------------------------------------------------- work of one pass

def _dims(case):
    """(fused, contracted, kept) bond dimensions of every step."""
    cut = case["cut"]
    out = []
    if case["kind"] == "chain":
        d = 4
        for _ in range(case["time"]):
            k = min(d * d, cut)
            out.append((d, 4, k))
            d = k
        out += [(1, d, 1)] * case["space"]
        return out
    dx = dy = case["q"]
    for i in range(case["steps"]):
        if i % 2 == 0:
            k = min(dy * dy, cut)
            out.append((dy, dx, k))
            dy = k
        else:
            k = min(dx * dx, cut)
            out.append((dx, dy, k))
            dx = k
    return out


def _step_flops(D, E, K):
    """Contractions of one step, and the leading pairs of both environments
    taken as two products of each with the K + 1 vectors."""
    f = 8 * D**3 * E**3 + 4 * D**4 * E**2 + 2 * K * D**3 * E**2 + 2 * K * D**3 * E**3 + 2 * K * K * D**2 * E**2
    return f + (8 * D**4 * (K + 1) if D * D > K else 0)


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8 * (m * k + n * k + m * n), "flops": 2 * m * n * k}
    if kind == "itebd":
        d, n = case["cut"], 2 * case["cut"]
        # four products of the bond matrices and one reduction to its eigenvectors
        one = 2 * (n * n * d + n**3 + n * n * d) + 9 * n**3
        return {"bytes": 8 * case["chains"] * (8 * d * d + n * n) * case["updates"],
                "flops": case["chains"] * one * case["updates"]}
    if kind == "sweep":
        cuts = [int(v) for v in case["cuts"].split(",")]
        each = [work({"kind": "model", "q": 2, "cut": cuts[i % len(cuts)], "steps": case["steps"]})
                for i in range(case["count"])]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    dims = _dims(case)
    return {"bytes": sum(8 * (D * D * E * E + K * K * E * E) for D, E, K in dims),
            "flops": sum(_step_flops(D, E, K) for D, E, K in dims)}


# ---------------------------------------------------------------- 64-bit values

def _exact_seconds(case):
    """Rough cost of the plain 64-bit calculation below."""
    if case["kind"] in ("gemm", "itebd"):
        return 1.0
    if case["kind"] == "sweep":
        cuts = [int(v) for v in case["cuts"].split(",")]
        return sum(_exact_seconds({"kind": "model", "q": 2, "cut": cuts[i % len(cuts)], "steps": case["steps"]})
                   for i in range(case["count"]))
    return sum(_step_flops(D, E, K) / 0.8e12 + (2 * (D / 40.0) ** 6 * 0.25 + 0.01 if D > 1 else 0.002)
               for D, E, K in _dims(case))


def _y_step(T, cut):
    """One step along y of T[x, x', y, y'] (left, right, down, up): the step's
    tensor over its largest entry, the log of that entry, and the spectrum."""
    D = T.shape[0]
    n = D * D
    K = min(n, cut)
    td = torch.tensordot

    def gram(low, up):
        A = td(T, T, dims=(low, low))
        B = td(T, T, dims=(up, up))
        G = td(A, B, dims=([1, 3], [1, 3])).permute(0, 2, 1, 3).reshape(n, n)
        return 0.5 * (G + G.T)

    lam, V = [], []
    for low, up in (([1, 2], [1, 3]), ([0, 2], [0, 3])):
        w, v = torch.linalg.eigh(gram(low, up))
        lam.append(w.flip(0))
        V.append(v.flip(1))
    side = 0 if K == n or lam[0][K:].sum() <= lam[1][K:].sum() else 1
    U = (torch.eye(n, dtype=T.dtype, device=T.device) if K == n else V[side][:, :K]).reshape(D, D, K)
    P = td(U, T, dims=([0], [0]))                       # x2, a, x1', y, k
    Q = td(P, T, dims=([0, 4], [0, 2]))                 # a, x1', y, x2', y'
    out = td(Q, U, dims=([1, 3], [0, 1])).permute(0, 3, 1, 2).contiguous()
    c = out.abs().max()
    keep = K if K == n else K + 1
    return out / c, float(torch.log(c)), lam[side][:keep] / lam[side][0]


def _step(T, cut, direction):
    if direction == "y":
        return _y_step(T, cut)
    T, lc, spec = _y_step(T.permute(2, 3, 0, 1).contiguous(), cut)
    return T.permute(2, 3, 0, 1).contiguous(), lc, spec


def _classical_tensor(q, beta, field):
    if q == 2:
        s = np.array([1.0, -1.0])
        B, w = np.exp(beta * np.outer(s, s)), np.exp(beta * field * s)
    else:
        B, w = np.exp(beta * np.eye(q)), np.ones(q)
    v, X = np.linalg.eigh(B)
    W = (X * np.sqrt(v)) @ X.T
    return np.einsum("s,sa,sb,sc,sd->abcd", w, W, W, W, W)


def _bond_operators(jxy, jz, tau):
    """h and exp(-tau h) of a bond in the basis uu, ud, du, dd."""
    h = np.zeros((4, 4))
    h[0, 0] = h[3, 3] = 0.25 * jz
    h[1, 1] = h[2, 2] = -0.25 * jz
    h[1, 2] = h[2, 1] = 0.5 * jxy
    w, X = np.linalg.eigh(h)
    return h, (X * np.exp(-tau * w)) @ X.T


def _chain_tensor(jxy, jz, tau):
    """Two sites over one period: T[x, x', (e0 o0), (e2 o2)]; the bond between
    cells is cut by a singular value decomposition of its gate."""
    g = _bond_operators(jxy, jz, tau)[1].reshape(2, 2, 2, 2)        # a' b' a b
    # gate between the right site of one cell and the left site of the next
    u, s, vt = np.linalg.svd(g.transpose(0, 2, 1, 3).reshape(4, 4))
    A = (u * np.sqrt(s)).reshape(2, 2, 4)                            # o2 o1 x'
    B = (np.sqrt(s)[:, None] * vt).reshape(4, 2, 2)                  # x e2 e1
    T = np.einsum("pqef,xcp,dqy->xyefcd", g, B, A)                   # p = e1, q = o1
    return T.reshape(4, 4, 4, 4)


def _exact_hotrg(T0, case, directions):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    T = torch.from_numpy(np.ascontiguousarray(T0)).to(dev)
    c = T.abs().max()
    T, ln, n, spec = T / c, float(torch.log(c)), 0, None
    for d in directions:
        if d == "trace":
            T = torch.einsum("abcc->ab", T)[:, :, None, None]
            c = T.abs().max()
            T, lc = T / c, float(torch.log(c))
        else:
            n += 1
            T, lc, s = _step(T, case["cut"], d)
            if spec is None and len(s) > case["cut"]:
                spec = s.cpu().numpy()
        ln += lc / 2.0**n
    ln += math.log(float(torch.einsum("aacc->", T))) / 2.0**n
    return np.float64(ln), spec


def _exact_itebd(case, seed):
    couplings, P, Q, lam = _itebd_inputs(case, seed)
    n, D = case["chains"], case["cut"]
    ops = [_bond_operators(*c) for c in couplings]
    h = np.stack([o[0] for o in ops]).reshape(n, 2, 2, 2, 2)
    g = np.stack([o[1] for o in ops]).reshape(n, 2, 2, 2, 2)
    other = np.full((n, D), 1.0 / math.sqrt(D))

    def pair(P, Q):
        return np.einsum("ziaj,zjbm->ziabm", P, Q, optimize=True)

    def energy(P, Q, lam):
        th = lam[:, :, None, None, None] * pair(P, Q)
        ht = np.einsum("zABab,ziabm->ziABm", h, th, optimize=True)
        return (th * ht).sum((1, 2, 3, 4)) / (th * th).sum((1, 2, 3, 4))

    for _ in range(case["updates"]):
        phi = np.einsum("zABab,ziabm->ziABm", g, pair(P, Q), optimize=True)
        theta = lam[:, :, None, None, None] * phi
        _, s, yt = np.linalg.svd(theta.reshape(n, 2 * D, 2 * D))
        s, yt = s[:, :D], yt[:, :D]
        norm = np.linalg.norm(s, axis=1)[:, None]
        Pn = (phi.reshape(n, 2 * D, 2 * D) @ yt.transpose(0, 2, 1) / norm[:, :, None]).reshape(n, D, 2, D)
        P, Q, lam, other = yt.reshape(n, D, 2, D), Pn, s / norm, lam
    return {"energy": 0.5 * (energy(P, Q, lam) + energy(Q, P, other)), "lam": lam[-1]}


def exact(case, seed):
    kind = case["kind"]
    if _exact_seconds(case) > 15.0:
        return None
    if kind == "gemm":
        a, b = _gemm_inputs(case, seed)
        return {"c": a @ b.T}
    if kind == "itebd":
        return _exact_itebd(case, seed)
    if kind == "sweep":
        betas, cuts = _sweep_inputs(case, seed)
        directions = ["xy"[i % 2] for i in range(case["steps"])]
        ln = [_exact_hotrg(_classical_tensor(2, b, 0.0), {"cut": c}, directions) for b, c in zip(betas, cuts)]
        return {"ln_z": np.array([v for v, _ in ln])}
    if kind == "model":
        T0 = _classical_tensor(case["q"], _model_inputs(case, seed), case["field"])
        ln, spec = _exact_hotrg(T0, case, ["xy"[i % 2] for i in range(case["steps"])])
    else:
        jxy, jz = _chain_inputs(case, seed)
        T0 = _chain_tensor(jxy, jz, case["tau"])
        ln, spec = _exact_hotrg(T0, case, ["y"] * case["time"] + ["trace"] + ["x"] * case["space"])
    return {"ln_z": ln, "spectrum": spec}
