"""The workloads this library's speed is measured on, through its public entry points.

listed()              the fixed cases
draw(rng)             one more case of the same ranges
prepare(case, seed)   inputs on the device and what a program keeps between calls
run(state)            one pass; returns every output
work(case)            the bytes and flops one pass cannot do without
exact(case, seed)     the same outputs by plain torch in 64 bits

Kinds of case:
  solve     the SLSQP iteration on a dense matrix: new values into A and B, H12
            factorization in place, Q^T B, back-substitution
  stacked   the same on the stacked SLSQP matrix [L^T; C], structure-aware
  resident  a factorization that is kept (with its compact-WY store): Q^T B and
            back-substitution for new right-hand sides
  batch     many independent problems in one call (factor, Q^T b, solve)
  plan      the same problems replayed from a plan, as an SLSQP loop does
  mixed     a large least-squares problem by a low-precision factorization and
            refinement to FP64 accuracy
  requests  a burst of host-side requests through the request loop
"""
import math

import numpy as np
import torch

from paper_2506_09463_gb300 import abi, api

DEV = "cuda"
F64 = torch.float64
PREC = {"fp64": abi.SLQR_FP64, "fp32": abi.SLQR_FP32, "tf32": abi.SLQR_TF32,
        "bf16x3": abi.SLQR_BF16X3}


def listed():
    return [
        # one small subproblem on its own: latency of the panels and launches
        {"name": "solve_256x128", "kind": "solve", "m": 256, "n": 128, "nrhs": 1},
        # a mid-size subproblem, nearly square, sizes that are no multiple of a tile
        {"name": "solve_1203x1001", "kind": "solve", "m": 1203, "n": 1001, "nrhs": 1},
        # tall problem with a block of right-hand sides
        {"name": "solve_16384x2048_64rhs", "kind": "solve", "m": 16384, "n": 2048, "nrhs": 64},
        # the largest: the dense square matrices of the paper's measurements
        {"name": "solve_8192x8192", "kind": "solve", "m": 8192, "n": 8192, "nrhs": 1},
        # the SLSQP matrix [L^T; C] with many constraint rows
        {"name": "stacked_4000+1000", "kind": "stacked", "n": 4000, "m_eq": 1000, "nrhs": 1},
        # an SLSQP iteration that reuses the factorization it has
        {"name": "resident_4096x2048", "kind": "resident", "m": 4096, "n": 2048, "nrhs": 1},
        # many concurrent SLSQP runs: uneven problems in one launch, FP64
        {"name": "batch_fp64_2000", "kind": "batch", "prec": "fp64", "count": 2000, "m_lo": 16,
         "m_hi": 512, "shapes": 7},
        # the same, FP32 factorization refined to FP64 accuracy
        {"name": "batch_fp32_2000", "kind": "batch", "prec": "fp32", "count": 2000, "m_lo": 16,
         "m_hi": 512, "shapes": 7},
        # an SLSQP loop over few small problems: the plan's launch latency
        {"name": "plan_fp64_256_small", "kind": "plan", "prec": "fp64", "count": 256, "m_lo": 16,
         "m_hi": 64, "shapes": 9},
        # one large well-conditioned problem in mixed precision (FP32 pipe)
        {"name": "mixed_fp32_8192x4096", "kind": "mixed", "prec": "fp32", "m": 8192, "n": 4096,
         "kappa": 1e2},
        # ragged sizes, tensor-core updates on split BF16
        {"name": "mixed_bf16x3_3001x700", "kind": "mixed", "prec": "bf16x3", "m": 3001, "n": 700,
         "kappa": 1e2},
        # requests of several SLSQP runs arriving together, [L^T; C] of mixed sizes
        {"name": "requests_stacked_24", "kind": "requests", "count": 24, "n_lo": 50, "n_hi": 2000,
         "shapes": 8},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "stacked", "resident", "batch", "plan", "mixed",
                       "mixed", "requests"])
    if kind in ("solve", "resident"):
        while True:
            m = _log(rng, 64, 16384)
            n = _log(rng, 32, min(m, 8192))
            if rng.random() < 0.4:             # sizes as programs pad them
                m, n = max(64, m // 64 * 64), max(32, n // 32 * 32)
            # a quarter of the largest listed case is enough for an extra one, and so few
            # columns of so many rows are no least-squares problem of an SLSQP step
            if 64 * n >= m and 2.0 * m * n * n < 2.0e11:
                break
        return {"kind": kind, "m": m, "n": n, "nrhs": rng.choice([1, 1, 1, 3, 17, 64])}
    if kind == "stacked":
        n = _log(rng, 50, 4000)
        return {"kind": kind, "n": n, "m_eq": rng.randint(n // 16 + 1, n // 2),
                "nrhs": rng.choice([1, 1, 1, 5])}
    if kind in ("batch", "plan"):
        lo = rng.choice([8, 16, 40])
        hi = _log(rng, 64, 512)
        return {"kind": kind, "prec": rng.choice(["fp64", "fp64", "fp32"]),
                "count": _log(rng, 16, 2000), "m_lo": lo, "m_hi": hi,
                "shapes": rng.randint(10, 10 ** 6)}
    if kind == "mixed":
        prec = rng.choice(["fp32", "tf32", "bf16x3"])
        m = _log(rng, 512, 8192)
        n = _log(rng, max(128, m // 16), m // 2)
        return {"kind": kind, "prec": prec, "m": m, "n": n,
                "kappa": float(_log(rng, 10, {"fp32": 10 ** 5, "tf32": 100, "bf16x3": 1000}[prec]))}
    return {"kind": kind, "count": rng.randint(4, 32), "n_lo": 50, "n_hi": _log(rng, 200, 2000),
            "shapes": rng.randint(10, 10 ** 6)}


# -- inputs ---------------------------------------------------------------------

_context = None


def _ctx():
    """The one context a program keeps for its direct calls."""
    global _context
    if _context is None:
        _context = api.Context(0)
    return _context


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn_cm(m, n, g):
    """m x n iid N(0,1), column-major."""
    return torch.randn(n, m, generator=g, dtype=F64, device=DEV).t()


def _stack(n, m_eq, g):
    """[L^T; C]: L lower triangular, diagonal U[0.5, 2], below it N(0, 0.1); C N(0,1)."""
    A = _randn_cm(n + m_eq, n, g)
    top = torch.triu(A[:n] * 0.1, 1)
    top.diagonal().copy_(torch.rand(n, generator=g, dtype=F64, device=DEV) * 1.5 + 0.5)
    A[:n] = top
    return A


def _conditioned(m, n, kappa, g):
    """U diag(sigma) V^T with sigma_i = kappa^(-i/(n-1)), U and V random orthogonal."""
    U = torch.linalg.qr(torch.randn(m, n, generator=g, dtype=F64, device=DEV))[0]
    V = torch.linalg.qr(torch.randn(n, n, generator=g, dtype=F64, device=DEV))[0]
    s = kappa ** (-torch.arange(n, dtype=F64, device=DEV) / max(1, n - 1))
    return (V @ (U * s).t()).t()


def _dense_inputs(case, seed):
    g = _gen(seed)
    if case["kind"] == "stacked":
        n = case["n"]
        m = n + case["m_eq"]
        A = _stack(n, case["m_eq"], g)
    else:
        m, n = case["m"], case["n"]
        A = _randn_cm(m, n, g)
    return A, _randn_cm(m, case["nrhs"], g)


def _batch_shapes(case):
    """m ~ U{m_lo..m_hi}, n ~ U{ceil(m/4)..m}."""
    rng = np.random.default_rng(case["shapes"])
    ms = [int(v) for v in rng.integers(case["m_lo"], case["m_hi"] + 1, size=case["count"])]
    ns = [int(rng.integers(-(-m // 4), m + 1)) for m in ms]
    return ms, ns


def _batch_inputs(case, seed):
    ms, ns = _batch_shapes(case)
    g = _gen(seed)
    A = torch.randn(sum(m * n for m, n in zip(ms, ns)), generator=g, dtype=F64, device=DEV)
    b = torch.randn(sum(ms), generator=g, dtype=F64, device=DEV)
    if case["prec"] == "fp32":
        # refinement is for problems of moderate condition: square Gaussian ones get
        # a heavier diagonal
        o = 0
        for m, n in zip(ms, ns):
            A[o:o + m * n].view(n, m).diagonal().add_(2.0 * math.sqrt(m))
            o += m * n
    return ms, ns, A, b


def _mixed_inputs(case, seed):
    g = _gen(seed)
    A = _conditioned(case["m"], case["n"], case["kappa"], g)
    return A, torch.randn(case["m"], generator=g, dtype=F64, device=DEV)


def _request_shapes(case):
    """n ~ log-U[n_lo, n_hi], m_eq ~ U{0..n/2}."""
    rng = np.random.default_rng(case["shapes"])
    n = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), size=case["count"]))
    return [(int(k), int(rng.integers(0, int(k) // 2 + 1))) for k in n]


def _request_inputs(case, seed):
    rng = np.random.default_rng(seed)
    out = []
    for n, m_eq in _request_shapes(case):
        A = np.zeros((n, n + m_eq)).T
        A[:n] = np.triu(rng.standard_normal((n, n)) * 0.1, 1)
        A[np.arange(n), np.arange(n)] = rng.uniform(0.5, 2.0, n)
        A[n:] = rng.standard_normal((m_eq, n))
        out.append((A, rng.standard_normal(n + m_eq)))
    return out


# -- what a program holds, and one pass --------------------------------------------


class _Plan:
    """A batch plan, destroyed with the state that holds it."""

    def __init__(self, *args):
        st, self.handle = abi.slqr_batch_plan_create(*args)
        abi.check(args[0], st, "slqr_batch_plan_create")

    def __del__(self):
        torch.cuda.synchronize()
        abi.slqr_batch_plan_destroy(self.handle)


def _offsets(sizes):
    return [0] + [int(v) for v in np.cumsum(sizes)[:-1]]


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": dict(case)}
    if kind in ("solve", "stacked", "resident"):
        A0, B0 = _dense_inputs(case, seed)
        m, n = A0.shape
        ctx = _ctx()
        s.update(ctx=ctx, A0=A0, B0=B0, A=torch.empty_like(A0), B=torch.empty_like(B0),
                 up=torch.empty(n, dtype=F64, device=DEV), wy=ctx.wy_buffer(m, n))
        if kind == "resident":
            s["A"].copy_(A0)
            ctx.factor(s["A"], s["up"], s["wy"])
    elif kind in ("batch", "plan"):
        ms, ns, A0, b0 = _batch_inputs(case, seed)
        A, b = torch.empty_like(A0), torch.empty_like(b0)
        up = torch.zeros(sum(ns), dtype=F64, device=DEV)
        status = torch.zeros(len(ms), dtype=torch.int32, device=DEV)
        ao, bo, uo = (_offsets(v) for v in ([m * n for m, n in zip(ms, ns)], ms, ns))
        Ap = [A.data_ptr() + 8 * o for o in ao]
        bp = [b.data_ptr() + 8 * o for o in bo]
        upp = [up.data_ptr() + 8 * o for o in uo]
        s.update(ctx=_ctx(), A0=A0, b0=b0, A=A, b=b, up=up, status=status, ms=ms, ns=ns, Ap=Ap,
                 bp=bp, upp=upp, prec=PREC[case["prec"]])
        # rows n.. of b are the residual part of Q^T b in FP64 and unspecified in FP32
        s["keep"] = torch.cat([torch.arange(o, o + (m if s["prec"] == 0 else n), device=DEV)
                               for o, m, n in zip(bo, ms, ns)])
        if kind == "plan":
            s["plan"] = _Plan(s["ctx"].ctx, ms, ns, None, Ap, ms, upp, bp, s["prec"],
                              status.data_ptr(), None)
    elif kind == "mixed":
        A, b = _mixed_inputs(case, seed)
        s.update(ctx=_ctx(), A=A, b=b, x=torch.empty(case["n"], dtype=F64, device=DEV),
                 prec=PREC[case["prec"]])
    else:
        s.update(ctx=_ctx(), server=api.Server(_ctx()), problems=_request_inputs(case, seed))
    return s


def run(s):
    kind = s["kind"]
    if kind in ("solve", "stacked", "resident"):
        ctx, A, B, up, wy = s["ctx"], s["A"], s["B"], s["up"], s["wy"]
        B.copy_(s["B0"])
        if kind == "stacked":
            A.copy_(s["A0"])
            ctx.factor_stacked(A, up, wy)
            ctx.apply_qt_stacked(A, up, B, wy=wy)
        else:
            if kind == "solve":
                A.copy_(s["A0"])
                ctx.factor(A, up, wy)
            ctx.apply_qt(A, up, B, wy=wy)
        ctx.solve_r(A, B)
        return {"B": B} if kind == "resident" else {"A": A, "up": up, "B": B}
    if kind in ("batch", "plan"):
        s["A"].copy_(s["A0"])
        s["b"].copy_(s["b0"])
        stream = torch.cuda.current_stream().cuda_stream
        if kind == "plan":
            abi.check(s["ctx"].ctx, abi.slqr_batch_plan_launch(s["plan"].handle, stream), "plan")
        else:
            st = abi.slqr_batch_factor(s["ctx"].ctx, s["ms"], s["ns"], s["Ap"], s["ms"], s["upp"],
                                       s["bp"], s["prec"], s["status"].data_ptr(), None, stream)
            abi.check(s["ctx"].ctx, st, "slqr_batch_factor")
        if s["prec"] == abi.SLQR_FP64:
            return {"A": s["A"], "b": s["b"], "status": s["status"], "up": s["up"]}
        return {"b": s["b"][s["keep"]], "status": s["status"]}
    if kind == "mixed":
        A, x = s["A"], s["x"]
        st, info = abi.slqr_lstsq_mixed_ex(s["ctx"].ctx, A.shape[0], A.shape[1], A.data_ptr(),
                                           A.stride(1), s["b"].data_ptr(), x.data_ptr(), s["prec"],
                                           torch.cuda.current_stream().cuda_stream,
                                           fp64_fallback=1)
        abi.check(s["ctx"].ctx, st, "slqr_lstsq_mixed_ex")
        return {"x": x, "status": st}
    server = s["server"]
    tickets = [server.submit(abi.SLQR_REQ_FACTOR_SOLVE, A, b, structure=abi.SLQR_STACKED)
               for A, b in s["problems"]]
    done = [server.wait(t) for t in tickets]
    return {"x": [x for _, x in done], "status": [r.status for r, _ in done]}


# -- the least work of a pass, and its values in 64 bits ------------------------------


def _flops(m, n, nrhs):
    """Householder factorization, Q^T of nrhs right-hand sides, back-substitution."""
    return 2.0 * m * n * n - 2.0 * n ** 3 / 3.0 + nrhs * (4.0 * m * n - 2.0 * n * n + 1.0 * n * n)


def _stacked_flops(n, m_eq, nrhs):
    return 2.0 * (m_eq + 1) * n * n + nrhs * (4.0 * (m_eq + 1) * n + 1.0 * n * n)


def work(case):
    kind = case["kind"]
    if kind == "solve":
        m, n, k = case["m"], case["n"], case["nrhs"]
        return {"bytes": 16.0 * m * n + 16.0 * m * k, "flops": _flops(m, n, k)}
    if kind == "stacked":
        n, e, k = case["n"], case["m_eq"], case["nrhs"]
        return {"bytes": 16.0 * (n * (n + 1) / 2 + e * n) + 16.0 * (n + e) * k,
                "flops": _stacked_flops(n, e, k)}
    if kind == "resident":
        m, n, k = case["m"], case["n"], case["nrhs"]
        return {"bytes": 8.0 * m * n + 16.0 * m * k, "flops": k * (4.0 * m * n - 1.0 * n * n)}
    if kind in ("batch", "plan"):
        ms, ns = _batch_shapes(case)
        out = 16.0 if case["prec"] == "fp64" else 8.0
        return {"bytes": sum(out * m * n + 16.0 * m for m, n in zip(ms, ns)),
                "flops": sum(_flops(m, n, 1) for m, n in zip(ms, ns))}
    if kind == "mixed":
        m, n = case["m"], case["n"]
        return {"bytes": 8.0 * m * n + 8.0 * (m + n), "flops": _flops(m, n, 1)}
    shapes = _request_shapes(case)
    return {"bytes": sum(8.0 * (n + e) * n + 8.0 * (2 * n + e) for n, e in shapes),
            "flops": sum(_stacked_flops(n, e, 1) for n, e in shapes)}


def _h12(A, B):
    """The H12 factorization of A (R, reflector tails and pivot entries), Q^T B with its
    first n rows replaced by R^-1 of them.  LAPACK's reflectors are the same ones scaled
    to a leading 1: up = -tau R_kk."""
    n = A.shape[1]
    F, tau = torch.geqrf(A)
    up = -tau * F.diagonal()[:n]
    QB = torch.ormqr(F, tau, B, left=True, transpose=True)
    QB[:n] = torch.linalg.solve_triangular(F[:n].triu(), QB[:n], upper=True)
    return torch.triu(F) + torch.tril(F, -1) * up, up, QB


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "stacked", "resident"):
        A, up, B = _h12(*_dense_inputs(case, seed))
        return {"B": B} if kind == "resident" else {"A": A, "up": up, "B": B}
    if kind in ("batch", "plan"):
        ms, ns, A, b = _batch_inputs(case, seed)
        A, b = A.cpu(), b.cpu()
        oA, ob, oup, ao, bo = [], [], [], 0, 0
        for m, n in zip(ms, ns):
            F, up, x = _h12(A[ao:ao + m * n].view(n, m).t(), b[bo:bo + m, None])
            oA.append(F.t().reshape(-1))
            oup.append(up)
            ob.append(x[:m if case["prec"] == "fp64" else n, 0])
            ao += m * n
            bo += m
        if case["prec"] == "fp64":
            return {"A": torch.cat(oA), "b": torch.cat(ob), "status": None, "up": torch.cat(oup)}
        return {"b": torch.cat(ob), "status": None}
    if kind == "mixed":
        A, b = _mixed_inputs(case, seed)
        return {"x": _h12(A, b[:, None])[2][:case["n"], 0], "status": None}
    out = []
    for A, b in _request_inputs(case, seed):
        A, b = torch.from_numpy(A).to(DEV), torch.from_numpy(b).to(DEV)
        out.append(_h12(A, b[:, None])[2][:A.shape[1], 0])
    return {"x": out, "status": None}
