"""Performance cases of the quaternion pseudoinverse library: calls that its
users make through the public binding (paper_2605_01464_gb300.qpinv.Context),
from the smallest product to the 2048 x 2048 solve.

Kinds (case["kind"]):
  gemm     Context.qgemm: C = A B in one precision ("tc": BF16 splits of
           `split` terms, "emu": `split` exact slices, "fp64": CUDA cores)
  solve    Context.solve: X = A^dagger of a matrix with a prescribed spectrum
           (or a Gaussian one), one method, one precision
  batched  Context.solve_batched: many small uneven blocks in one call
  cur      Context.cur_complete: colour image completion (Sec. 5.1)
  filter   Context.toeplitz_filter: filter design on Lorenz signals (Sec. 5.2)
  krylov   Context.global_krylov: Gl-QGMRES / Gl-QFOM (Sec. 3.5)

Quaternion matrices are (4, rows, cols) float64 planes (s, x, y, z) on the
GPU.  Inputs come from the seed alone; a program keeps one context per set of
options, so the contexts live as long as the process.
"""
import functools
import math

import numpy as np
import torch

from paper_2605_01464_gb300 import inputs, qpinv

DEV = "cuda"
_contexts = {}


def _context(**options):
    key = tuple(sorted(options.items()))
    if key not in _contexts:
        _contexts[key] = qpinv.Context(0, **options)
    return _contexts[key]


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # one small product in the binding's default precision: latency of a call
        {"name": "gemm_tc_64x48x80", "kind": "gemm", "precision": "tc", "split": 3, "m": 64, "k": 48, "n": 80},
        # a ragged product of the size of the solver's polynomial blocks
        {"name": "gemm_tc_2176x2056x2100", "kind": "gemm", "precision": "tc", "split": 2, "m": 2176, "k": 2056,
         "n": 2100},
        # an FP64-accurate product on the tensor cores
        {"name": "gemm_emu_2048", "kind": "gemm", "precision": "emu", "split": 8, "m": 2048, "k": 2048, "n": 2048},
        # an FP64 product of the paper's 1000 x 500 example
        {"name": "gemm_fp64_1000x500", "kind": "gemm", "precision": "fp64", "split": 1, "m": 1000, "k": 500,
         "n": 1000},
        # the small dense Gaussian workload: a handful of iterations of tiny products
        {"name": "solve_64x48", "kind": "solve", "method": "qhpi19", "precision": "mixed", "m": 64, "n": 48,
         "rank": 48, "smin": 0.0},
        # the paper's rectangular example, order-10 iteration
        {"name": "solve_1000x500_qsai", "kind": "solve", "method": "qsai", "precision": "mixed", "m": 1000, "n": 500,
         "rank": 500, "smin": 0.0},
        # the headline workload: square, sigma log-spaced 1 .. 1e-6, mixed precision
        {"name": "solve_2048_kappa1e6", "kind": "solve", "method": "qhpi19", "precision": "mixed", "m": 2048,
         "n": 2048, "rank": 2048, "smin": 1e-6},
        # rank-deficient input: every product FP64-accurate
        {"name": "solve_rankdef_2048x1024", "kind": "solve", "method": "qhpi19", "precision": "emu", "m": 2048,
         "n": 1024, "rank": 512, "smin": 3e-2},
        # blocks of 16 .. 256 rows and columns, solved in one call
        {"name": "batched_512", "kind": "batched", "count": 512, "lo": 16, "hi": 256, "method": "qhpi19"},
        # image completion: 512 x 768 colour image, 70 % of the pixels missing, rank 60
        {"name": "cur_512x768", "kind": "cur", "m": 512, "n": 768, "rank": 60, "iters": 10, "method": "qhpi19"},
        # filter design at 0.05 and finer sampling: an 801 x 801 data matrix
        {"name": "filter_801", "kind": "filter", "dt": 0.025, "method": "qsai"},
        # preconditioned GMRES on the 14 x 17 reservoir grid, three right-hand sides
        {"name": "krylov_238", "kind": "krylov", "nx": 14, "ny": 17, "cols": 3, "solver": "gmres", "precond": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "gemm", "solve", "solve", "solve", "batched", "cur", "filter", "krylov"])
    if kind == "gemm":
        precision = rng.choice(["tc", "emu", "emu", "fp64"])
        hi = 1000 if precision == "fp64" else 2200
        m, k, n = (_log(rng, 40, hi) for _ in range(3))
        split = {"tc": rng.randint(1, 3), "emu": rng.choice([4, 6, 8, 8]), "fp64": 1}[precision]
        return {"kind": kind, "precision": precision, "split": split, "m": m, "k": k, "n": n}
    if kind == "solve":
        form = rng.choice(["gauss", "square", "rankdef"])
        if form == "gauss":  # full rank, either orientation
            m, n = _log(rng, 48, 1024), _log(rng, 48, 1024)
            return {"kind": kind, "method": rng.choice(["qhpi19", "qsai", "qrapid", "ns"]), "precision": "mixed",
                    "m": m, "n": n, "rank": min(m, n), "smin": 0.0}
        if form == "square":
            n = _log(rng, 100, 2048)
            return {"kind": kind, "method": rng.choice(["qhpi19", "qsai"]), "precision": "mixed", "m": n, "n": n,
                    "rank": n, "smin": 10.0 ** -rng.uniform(2, 6)}
        m, n = _log(rng, 100, 2048), _log(rng, 100, 1024)
        return {"kind": kind, "method": rng.choice(["qhpi19", "qsai", "ns"]), "precision": "emu", "m": m, "n": n,
                "rank": max(1, min(m, n) // 2), "smin": 3e-2}
    if kind == "batched":
        return {"kind": kind, "count": _log(rng, 40, 512), "lo": 16, "hi": rng.choice([96, 160, 256]),
                "method": rng.choice(["qhpi19", "qsai"])}
    if kind == "cur":
        m, n = _log(rng, 128, 512), _log(rng, 128, 768)
        return {"kind": kind, "m": m, "n": n, "rank": rng.randint(16, 60), "iters": rng.randint(2, 8),
                "method": "qhpi19"}
    if kind == "filter":
        return {"kind": kind, "dt": rng.choice([0.04, 0.05, 0.08, 0.1]), "method": rng.choice(["qsai", "qhpi19", "ns"])}
    return {"kind": "krylov", "nx": rng.randint(8, 14), "ny": rng.randint(8, 17), "cols": rng.randint(1, 12),
            "solver": rng.choice(["gmres", "fom"]), "precond": rng.choice([0, 2])}


# ------------------------------------------------- quaternion planes in torch

def _gen(seed, stream=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _normal(seed, stream, *shape):
    return torch.randn(*shape, generator=_gen(seed, stream), device=DEV, dtype=torch.float64)


def _hamilton(p, q, op):
    """The Hamilton product of plane stacks p and q, real products by `op`."""
    s = op(p[0], q[0]) - op(p[1], q[1]) - op(p[2], q[2]) - op(p[3], q[3])
    x = op(p[0], q[1]) + op(p[1], q[0]) + op(p[2], q[3]) - op(p[3], q[2])
    y = op(p[0], q[2]) - op(p[1], q[3]) + op(p[2], q[0]) + op(p[3], q[1])
    z = op(p[0], q[3]) + op(p[1], q[2]) - op(p[2], q[1]) + op(p[3], q[0])
    return torch.stack([s, x, y, z])


def _mul(P, Q):
    return _hamilton(P, Q, torch.matmul)


def _scale(p, q):
    return _hamilton(p, q, torch.mul)


def _conj(q):
    return torch.stack([q[0], -q[1], -q[2], -q[3]])


def _chi(Q):
    """Complex representation [[s + x i, y + z i], [-y + z i, s - x i]] by blocks, (2m, 2n)."""
    a, b = torch.complex(Q[0], Q[1]), torch.complex(Q[2], Q[3])
    return torch.cat([torch.cat([a, b], 1), torch.cat([-b.conj(), a.conj()], 1)], 0)


def _unchi(C):
    m, n = C.shape[0] // 2, C.shape[1] // 2
    a, b = C[:m, :n], C[:m, n:]
    return torch.stack([a.real, a.imag, b.real, b.imag]).contiguous()


def _pinv_full_rank(A):
    """A^dagger of a full-rank A in 64 bits: the normal equations, then Newton-Schulz steps."""
    C = _chi(A)
    H = C.mH
    wide = C.shape[0] < C.shape[1]
    X = (torch.linalg.solve(C @ H, C)).mH if wide else torch.linalg.solve(H @ C, H)
    I = torch.eye(min(C.shape), dtype=C.dtype, device=C.device)
    for _ in range(2):
        X = X + X @ (I - C @ X) if wide else X + (I - X @ C) @ X
    return _unchi(X)


@functools.lru_cache(maxsize=8)
def _dct(n):
    """Orthonormal DCT-II matrix, rows = frequencies."""
    k = torch.arange(n, device=DEV)
    C = torch.cos(math.pi / (2 * n) * ((2 * k[None, :] + 1) * k[:, None] % (4 * n)).double()) * math.sqrt(2.0 / n)
    C[0] *= math.sqrt(0.5)
    return C


def _unit(seed, stream, n):
    q = _normal(seed, stream, 4, n)
    return q / q.square().sum(0, keepdim=True).sqrt()


def _spectrum(case):
    r, smin = case["rank"], case["smin"]
    return torch.logspace(0.0, math.log10(smin), r, device=DEV, dtype=torch.float64)


def _with_spectrum(case, seed):
    """A and A^dagger (m x n, n x m) with singular values _spectrum(case):
    A = L Q_m diag(sigma p) Q_n^T R with random unit quaternion diagonals L, R,
    p and randomly chosen columns of the DCT matrices Q_m, Q_n."""
    m, n, r = case["m"], case["n"], case["rank"]
    sig = _spectrum(case)
    L, R, p = _unit(seed, 1, m), _unit(seed, 2, n), _unit(seed, 3, r)
    Qm = _dct(m)[torch.randperm(m, generator=_gen(seed, 4), device=DEV)[:r]].T
    Qn = _dct(n)[torch.randperm(n, generator=_gen(seed, 5), device=DEV)[:r]].T
    mid = torch.stack([(Qm * (sig * p[c])) @ Qn.T for c in range(4)])
    A = _scale(_scale(L[:, :, None], mid), R[:, None, :])

    def pinv():
        inv = torch.stack([(Qn * (c / sig)) @ Qm.T for c in _conj(p)])
        return _scale(_scale(_conj(R)[:, :, None], inv), _conj(L)[:, None, :])

    return A.contiguous(), pinv


# ------------------------------------------------------------ inputs by kind

def _matrix(case, seed):
    if case["smin"] > 0:
        return _with_spectrum(case, seed)
    A = _normal(seed, 6, 4, case["m"], case["n"])  # Gaussian: full rank
    return A, lambda: _pinv_full_rank(A)


def _shapes(case):
    """The blocks' shapes: the same for every seed, as a program's blocks are."""
    g = np.random.RandomState(case["count"])
    return [(int(a), int(b)) for a, b in g.randint(case["lo"], case["hi"] + 1, size=(case["count"], 2))]


@functools.lru_cache(maxsize=4)
def _trajectory(dt):
    return inputs.lorenz_trajectory(dt, 40.0 + round(1.0 / dt) * dt)


def _signals(case, seed):
    """Lorenz signals of the filtering example: s(t) and x(t) = s(t - 1) + noise."""
    dt = case["dt"]
    d, count = int(round(1.0 / dt)), int(round(40.0 / dt)) + 1
    tr = torch.from_numpy(_trajectory(dt)).to(DEV).T
    x = torch.zeros(4, count, device=DEV, dtype=torch.float64)
    s = torch.zeros_like(x)
    s[1:] = tr[:, d:d + count]
    x[1:] = tr[:, :count] + 0.5 * _normal(seed, 7, 3, count)
    return x, s, (count - 1) // 2


@functools.lru_cache(maxsize=4)
def _image(m, n):
    return torch.from_numpy(inputs.synthetic_rgb_image(m, n)).to(DEV)


def _completion(case, seed):
    m, n = case["m"], case["n"]
    M = _image(m, n).clone()
    M[1:] = (M[1:] + 0.01 * _normal(seed, 8, 3, m, n)).clamp_(0.0, 1.0)
    mask = (torch.rand(m, n, generator=_gen(seed, 9), device=DEV) < 0.3).to(torch.uint8)
    g = np.random.RandomState(int(seed) % (1 << 31))
    I = np.stack([np.sort(g.permutation(m)[:case["rank"]]) for _ in range(case["iters"])]).astype(np.int32)
    J = np.stack([np.sort(g.permutation(n)[:case["rank"]]) for _ in range(case["iters"])]).astype(np.int32)
    return M, mask, I, J


def _system(case, seed):
    """The preconditioning example's system A_s + A_x i + A_y j + A_z k on a
    reservoir grid, with a storage term that keeps it well posed."""
    As = torch.from_numpy(inputs.reservoir_matrix(case["nx"], case["ny"], int(seed), log_sd=1.0, storage=0.1)).to(DEV)
    A = torch.stack([As, -As, 2.0 * As, 1.5 * As])
    B = torch.rand(4, As.shape[0], case["cols"], generator=_gen(seed, 10), device=DEV, dtype=torch.float64)
    return A.contiguous(), B


# ------------------------------------------------------------------ interface

def prepare(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        return {"case": case, "ctx": _context(), "A": _normal(seed, 11, 4, case["m"], case["k"]),
                "B": _normal(seed, 12, 4, case["k"], case["n"])}
    if kind == "solve":
        A, _ = _matrix(case, seed)
        return {"case": case, "ctx": _context(precision=case["precision"]), "A": A}
    if kind == "batched":
        shapes = _shapes(case)
        total = 4 * sum(m * n for m, n in shapes)
        a, x = _normal(seed, 13, total), torch.zeros(total, device=DEV, dtype=torch.float64)
        As, Xs, at = [], [], 0
        for m, n in shapes:
            As.append(a[at:at + 4 * m * n].view(4, m, n))
            Xs.append(x[at:at + 4 * m * n].view(4, n, m))
            at += 4 * m * n
        return {"case": case, "ctx": _context(), "As": As, "Xs": Xs, "X": x}
    if kind == "cur":
        M, mask, I, J = _completion(case, seed)
        return {"case": case, "ctx": _context(), "M": M, "mask": mask, "I": I, "J": J}
    if kind == "filter":
        x, s, p = _signals(case, seed)
        return {"case": case, "ctx": _context(), "x": x, "s": s, "p": p}
    A, B = _system(case, seed)
    return {"case": case, "ctx": _context(), "A": A, "B": B}


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "gemm":
        return ctx.qgemm(state["A"], state["B"], precision=case["precision"], split_level=case["split"])
    if kind == "solve":
        X, _ = ctx.solve(state["A"], case["method"], tol=1e-12, max_iter=200)
        return X
    if kind == "batched":
        ctx.solve_batched(state["As"], case["method"], tol=1e-12, max_iter=200, Xs=state["Xs"])
        return state["X"]
    if kind == "cur":
        C, _ = ctx.cur_complete(state["M"], state["mask"], state["I"], state["J"], case["method"], tol=1e-12,
                                max_iter=200, sigma=0.5)
        return C
    if kind == "filter":
        h, s_hat, _, _ = ctx.toeplitz_filter(state["x"], state["s"], state["p"], method=case["method"], tol=1e-12,
                                             max_iter=2000)
        return {"h": h, "s_hat": s_hat}
    X, _ = ctx.global_krylov(state["A"], state["B"], case["solver"], precond_iters=case["precond"], tol=1e-11,
                             max_iter=3000)
    return X


#: method: (order, products per iteration)
_METHOD = {"ns": (2, 2), "qsai": (10, 6), "qhpi19": (19, 7), "qrapid": (89, 18)}


def _solve_flops(m, n, smin, method):
    """The residual goes from 1 - alpha sigma_r^2 (safe alpha, about
    smin^2 / n) to 1e-16 in log_order steps; four products for E1 .. E4."""
    order, products = _METHOD[method]
    s = min(m, n)
    steps = math.ceil(math.log(37.0 * max(4.0, s) / (smin * smin), order))
    return 32.0 * (steps * ((products - 2) * s ** 3 + 2 * m * n * s) + 2 * m * n * (m + n))


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        m, k, n = case["m"], case["k"], case["n"]
        return {"bytes": 32.0 * (m * k + k * n + m * n), "flops": 32.0 * m * k * n}
    if kind == "solve":
        m, n = case["m"], case["n"]
        smin = case["smin"] or max(abs(m - n), 1) / (4.0 * max(m, n))
        return {"bytes": 64.0 * m * n, "flops": _solve_flops(m, n, smin, case["method"])}
    if kind == "batched":
        shapes = _shapes(case)
        return {"bytes": sum(64.0 * m * n for m, n in shapes),
                "flops": sum(_solve_flops(m, n, max(abs(m - n), 1) / (4.0 * max(m, n)), case["method"])
                             for m, n in shapes)}
    if kind == "cur":
        m, n, r, it = case["m"], case["n"], case["rank"], case["iters"]
        each = _solve_flops(m, r, 1e-1, case["method"]) + _solve_flops(r, n, 1e-1, case["method"])
        return {"bytes": 65.0 * m * n, "flops": it * (each + 32.0 * (2 * m * n * r + r * r * (m + n)))}
    if kind == "filter":
        n = int(round(40.0 / case["dt"])) // 2 + 1
        return {"bytes": 64.0 * 4 * n, "flops": _solve_flops(n, n, 1e-3, case["method"])}
    n, c = case["nx"] * case["ny"], case["cols"]
    steps = n // 2
    return {"bytes": 32.0 * (n * n + 2 * n * c), "flops": 32.0 * n * n * c * steps + 16.0 * n * c * steps * steps}


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        return _mul(_normal(seed, 11, 4, case["m"], case["k"]), _normal(seed, 12, 4, case["k"], case["n"]))
    if kind == "solve":
        return _matrix(case, seed)[1]()
    if kind == "batched":
        shapes = _shapes(case)
        a = _normal(seed, 13, 4 * sum(m * n for m, n in shapes))
        out, at = [], 0
        for m, n in shapes:
            out.append(_pinv_full_rank(a[at:at + 4 * m * n].view(4, m, n)).reshape(-1))
            at += 4 * m * n
        return torch.cat(out)
    if kind == "cur":
        M, mask, I, J = _completion(case, seed)
        obs = mask.bool()[None]
        g = torch.exp(-2.0 * torch.arange(-1, 2, device=DEV, dtype=torch.float64) ** 2)
        g = g / g.sum()
        C = torch.where(obs, M, torch.zeros_like(M))
        for i, j in zip(I, J):
            i, j = torch.from_numpy(i).long().to(DEV), torch.from_numpy(j).long().to(DEV)
            CJ, RI = C[:, :, j].contiguous(), C[:, i, :].contiguous()
            U = _mul(_mul(_pinv_full_rank(CJ), C), _pinv_full_rank(RI))
            X = _mul(_mul(CJ, U), RI)
            m, n = X.shape[1:]
            P = torch.nn.functional.pad(X[None], (1, 1, 1, 1), mode="replicate")[0]
            X = sum(g[a] * g[b] * P[:, a:a + m, b:b + n] for a in range(3) for b in range(3))
            C = torch.where(obs, M, X)
        return C
    if kind == "filter":
        x, s, p = _signals(case, seed)
        at = p + torch.arange(p + 1, device=DEV)[:, None] - torch.arange(p + 1, device=DEV)[None, :]
        X, S = x[:, at], s[:, p:2 * p + 1, None]
        h = torch.linalg.solve(_chi(X), _chi(S))
        return {"h": _unchi(h), "s_hat": S.contiguous()}
    A, B = _system(case, seed)
    return _unchi(torch.linalg.solve(_chi(A), _chi(B)))
