"""The workloads that the speed of this library is measured on.

Each case is one pass through the public binding (`paper_2609_15217_gb300.tinylu`)
as a finite-element code that integrates its material law on the GPU calls it:

  gesv     tl_gesv_batched: one fresh linear system per integration point
           (optionally keeping the factors for a later solve)
  factor   tl_getrf_batched, then tl_getrs_batched with nrhs right-hand sides
  ragged   tl_lupp_solve_batched: the systems of several laws, every one with
           its own n, in binary64 or in mixed precision
  norton   tl_newton_integrate(_tangent): the fused Newton loop of the Norton law
  tanh     tl_newton_integrate with the dense law, n unknowns per point

Systems are those of the library's sweep (half U[-1, 1] entries, half with a
prescribed condition number of 1e2..1e8, b = A x with x in U[-1, 1]); the points
are those of its Newton workloads.  The handle is untuned, as tl_create gives it.
"""
import math

import numpy as np
import torch

from paper_2609_15217_gb300 import inputs, layout as lay, tinylu as tl

DEVICE = "cuda"
RTOL, MAX_ITER = 1e-10, 20
# the Norton steel of the library's Newton workload: E, nu, A, m, dt
NORTON = (200000.0, 0.3, 1e-12, 4.0, 1.0)
# sizes and weights of the ragged workload, and every size alike
MIXES = {
    "laws": ((6, 7, 12, 13, 19, 25, 32), (0.2, 0.25, 0.15, 0.15, 0.1, 0.1, 0.05)),
    "all": (tuple(range(1, 33)), (1.0 / 32,) * 32),
}
# Norton points of this workload take 3 to 8 linear solves, 6.2 in the mean;
# the dense law takes 3 to 4
NORTON_SOLVES, TANH_SOLVES = 6.2, 3.1


def listed():
    return [
        # the integration points of one small element group: launch latency
        {"name": "gesv_n6_b64", "op": "gesv", "n": 6, "batch": 64, "interleaved": False, "factors": False},
        # 512 hexahedra with 8 points each, one state vector of 8
        {"name": "gesv_n8_b4096", "op": "gesv", "n": 8, "batch": 4096, "interleaved": False, "factors": False},
        # a whole mesh, a small viscoplastic law (7 unknowns), a batch that fills no tile
        {"name": "gesv_n7_b1000003", "op": "gesv", "n": 7, "batch": 1000003, "interleaved": True, "factors": False},
        # a whole mesh, a crystal law of middle size
        {"name": "gesv_n19_b150001", "op": "gesv", "n": 19, "batch": 150001, "interleaved": True, "factors": False},
        # the largest systems, one after another in memory as LAPACK-style callers keep them
        {"name": "gesv_n32_b60000", "op": "gesv", "n": 32, "batch": 60000, "interleaved": False, "factors": False},
        # solve and keep the factors (the tangent operator is solved with them later)
        {"name": "gesv_lu_n13_b50000", "op": "gesv", "n": 13, "batch": 50000, "interleaved": True, "factors": True},
        # factor once, solve for the six strain directions
        {"name": "factor_n12_b90001_r6", "op": "factor", "n": 12, "batch": 90001, "interleaved": True, "nrhs": 6},
        # factor, then one solve, large systems, one after another in memory
        {"name": "factor_n27_b20011_r1", "op": "factor", "n": 27, "batch": 20011, "interleaved": False, "nrhs": 1},
        # a structure of seven materials in one call
        {"name": "ragged_laws_b262144", "op": "ragged", "mix": "laws", "batch": 262144, "mixed": False},
        # every size, binary32 factors with binary64 refinement
        {"name": "ragged_mixed_all_b100003", "op": "ragged", "mix": "all", "batch": 100003, "mixed": True},
        # one time step of a viscoplastic structure, tangent included
        {"name": "norton_tangent_b400000", "op": "norton", "batch": 400000, "tangent": True},
        # the same with a dense law of 20 unknowns
        {"name": "tanh_n20_b65537", "op": "tanh", "n": 20, "batch": 65537},
    ]


# No drawn case costs more floating-point work, or more memory, than these.
MOST_FLOPS, MOST_BYTES = 1.3e9, 6e8


def draw(rng):
    """One more case: sizes 1..32, batches of 1 to a million (by their logarithm), both layouts, every option."""
    op = rng.choice(["gesv", "gesv", "gesv", "factor", "factor", "ragged", "norton", "tanh"])
    c = {"op": op, "batch": 1}
    if op in ("gesv", "factor", "tanh"):
        c["n"] = rng.randint(1, 32)
    if op in ("gesv", "factor"):
        c["interleaved"] = rng.random() < 0.5
    if op == "gesv":
        c["factors"] = rng.random() < 0.3
    elif op == "factor":
        c["nrhs"] = rng.choice([1, 1, 2, 3, 6, 6, 12, 32])
    elif op == "ragged":
        c["mix"], c["mixed"] = rng.choice(sorted(MIXES)), rng.random() < 0.5
    elif op == "norton":
        c["tangent"] = rng.random() < 0.5
    one = work(c)
    most = min(1e6, MOST_FLOPS / max(one["flops"], 1.0), MOST_BYTES / one["bytes"])
    c["batch"] = max(1, int(math.exp(rng.uniform(0.0, math.log(most)))))
    return c


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def factor_flops(n):
    return 2 * ((n - 1) * n * (2 * n - 1) // 6) + n * (n - 1) // 2 + n


def solve_flops(n):
    return 2 * n * (n - 1) + n


def work(case):
    """Each input read once, each output written once; multiplies and adds of the elimination and the solves."""
    batch, op = case["batch"], case["op"]
    if op == "gesv":
        n = case["n"]
        size, flops = 8 * n * n + 20 * n + 4, factor_flops(n) + solve_flops(n)
        if case["factors"]:
            size += 8 * n * n
    elif op == "factor":
        n, r = case["n"], case["nrhs"]
        size, flops = 16 * n * n + 16 * n * r + 4 * n + 4, factor_flops(n) + r * solve_flops(n)
    elif op == "ragged":
        sizes, weights = MIXES[case["mix"]]
        size = sum(w * (8 * n * n + 20 * n + 8 + 24) for n, w in zip(sizes, weights))
        flops = sum(w * (factor_flops(n) + solve_flops(n)) for n, w in zip(sizes, weights))
    elif op == "norton":
        size, evaluation = 12 * 8 + 13 * 8 + 8, 244
        flops = NORTON_SOLVES * (factor_flops(7) + solve_flops(7) + evaluation) + evaluation
        if case["tangent"]:
            size += 36 * 8
            flops += factor_flops(7) + 6 * solve_flops(7) + 6 * 15
    else:
        n = case["n"]
        size, evaluation = 8 * n * n + 24 * n + 8, 2 * n * n + 20 * n
        flops = TANH_SOLVES * (factor_flops(n) + solve_flops(n) + evaluation) + evaluation
    return {"bytes": int(size * batch), "flops": int(flops * batch)}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

_handle = None


def handle():
    """The program's handle: made once, kept for as long as the program runs."""
    global _handle
    if _handle is None:
        _handle = tl.tl_create()
    return _handle


def systems(n, batch, seed):
    """A (batch, n, n) and b (batch, n) of the sweep."""
    A, b, _ = inputs.sweep_systems_torch(n, batch, seed, DEVICE)
    return A, b


def right_hand_sides(case, seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed + 1)
    shape = (case["batch"], case["nrhs"], case["n"])
    return torch.empty(shape, dtype=torch.float64, device=DEVICE).uniform_(-1.0, 1.0, generator=g)


def ragged_sizes(case, seed):
    """The sizes of the batch: their weights' shares, in random order."""
    sizes, weights = MIXES[case["mix"]]
    ends = np.rint(np.cumsum(weights) * case["batch"]).astype(np.int64)
    n = np.repeat(np.array(sizes, dtype=np.int64), np.diff(ends, prepend=0))
    return np.random.default_rng(seed).permutation(n)


def ragged_systems(case, seed):
    """Sizes and offsets of the systems, one after another in memory, and the systems of each size."""
    n = torch.from_numpy(ragged_sizes(case, seed)).to(DEVICE)
    a_off = torch.cumsum(n * n, 0) - n * n
    b_off = torch.cumsum(n, 0) - n
    parts = []
    for k in sorted(set(MIXES[case["mix"]][0])):
        at = torch.nonzero(n == k).reshape(-1)
        if at.numel():
            parts.append((k, at, *systems(k, at.numel(), seed * 64 + k)))
    return n, a_off, b_off, parts


def norton_inputs(case, seed):
    sig0, deps = inputs.norton_points_torch(case["batch"], seed, DEVICE)
    return torch.cat([sig0.t(), deps.t()], dim=0).contiguous()


def doubles(*shape):
    return torch.zeros(shape, dtype=torch.float64, device=DEVICE)


def ints(*shape):
    return torch.zeros(shape, dtype=torch.int32, device=DEVICE)


def prepare(case, seed):
    op, batch = case["op"], case["batch"]
    s = {"op": op, "h": handle(), "batch": batch, "case": case}
    if op in ("gesv", "factor"):
        n, L = case["n"], int(case["interleaved"])
        ld = lay.pad_ld(batch)
        rows = ld if L else batch
        A, b = systems(n, batch, seed)
        s.update(n=n, layout=L, ld=ld, A=lay.matrices_to_layout(A, L, ld), ipiv=ints(n * rows), info=ints(batch))
        if op == "gesv":
            s.update(b=lay.vectors_to_layout(b, L, ld), x=doubles(n * rows),
                     LU=doubles(n * n * rows) if case["factors"] else None)
        else:
            B = lay.multi_rhs_to_layout(right_hand_sides(case, seed), L, ld)
            s.update(B=B, LU=torch.zeros_like(s["A"]), X=torch.zeros_like(B), nrhs=case["nrhs"])
    elif op == "ragged":
        n, a_off, b_off, parts = ragged_systems(case, seed)
        A, b = doubles(int((n * n).sum())), doubles(int(n.sum()))
        for k, at, Ak, bk in parts:
            step = torch.arange(k * k, device=DEVICE)
            A[a_off[at][:, None] + step] = Ak.transpose(1, 2).reshape(-1, k * k)
            b[b_off[at][:, None] + step[:k]] = bk
        s.update(n=n.to(torch.int32), a_off=a_off, b_off=b_off, A=A, b=b, x=torch.zeros_like(b),
                 ipiv=ints(b.numel()), info=ints(batch), steps=ints(batch) if case["mixed"] else None,
                 prec=tl.TL_PREC_FP32_IR if case["mixed"] else tl.TL_PREC_FP64)
    elif op == "norton":
        s.update(fields=norton_inputs(case, seed), law=tl.make_law(tl.TL_LAW_NORTON, 7, NORTON), x=doubles(7, batch),
                 sig=doubles(6, batch), D=doubles(36, batch) if case["tangent"] else None, iters=ints(batch),
                 status=ints(batch))
    else:
        n = case["n"]
        s.update(fields=inputs.tanh_points_torch(n, batch, seed, DEVICE), law=tl.make_law(tl.TL_LAW_TANH, n),
                 x=doubles(n, batch), iters=ints(batch), status=ints(batch))
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(s):
    op, h, batch = s["op"], s["h"], s["batch"]
    if op == "gesv":
        tl.check("tl_gesv_batched", tl.tl_gesv_batched(h, s["n"], s["A"], s["LU"], s["b"], s["x"], s["ipiv"], s["info"],
                                                       s["layout"], s["ld"], batch), h)
        return {"x": s["x"], "LU": s["LU"], "ipiv": s["ipiv"], "info": s["info"]}
    if op == "factor":
        # both calls work in place: the program copies what it still needs
        s["LU"].copy_(s["A"])
        s["X"].copy_(s["B"])
        tl.check("tl_getrf_batched", tl.tl_getrf_batched(h, s["n"], s["LU"], s["layout"], s["ld"], s["ipiv"], s["info"],
                                                         batch), h)
        tl.check("tl_getrs_batched", tl.tl_getrs_batched(h, s["n"], s["nrhs"], s["LU"], s["ipiv"], s["layout"], s["ld"],
                                                         s["X"], batch), h)
        return {"x": s["X"], "LU": s["LU"], "ipiv": s["ipiv"], "info": s["info"]}
    if op == "ragged":
        tl.check("tl_lupp_solve_batched",
                 tl.tl_lupp_solve_batched(h, batch, s["n"], s["a_off"], s["A"], s["b_off"], s["b"], s["x"], s["b_off"],
                                          s["ipiv"], s["info"], s["prec"], s["steps"]), h)
        return {"x": s["x"], "ipiv": s["ipiv"], "info": s["info"], "steps": s["steps"]}
    if op == "norton" and s["D"] is not None:
        tl.check("tl_newton_integrate_tangent",
                 tl.tl_newton_integrate_tangent(h, s["law"], batch, s["fields"], s["x"], s["sig"], s["D"], s["iters"],
                                                s["status"], RTOL, MAX_ITER), h)
    else:
        tl.check("tl_newton_integrate",
                 tl.tl_newton_integrate(h, s["law"], batch, s["fields"], s["x"], s.get("sig"), s["iters"], s["status"],
                                        RTOL, MAX_ITER), h)
    return {"x": s["x"], "sig": s.get("sig"), "D": s.get("D"), "iters": s["iters"], "status": s["status"]}


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def residual(A, x, b):
    """b - A x with error-free products (Dekker's split) and compensated sums, rounded once."""
    def split(v):
        c = 134217729.0 * v
        hi = c - (c - v)
        return hi, v - hi
    total, rest = b.clone(), torch.zeros_like(b)
    for j in range(A.shape[2]):
        a, y = A[:, :, j], -x[:, j:j + 1].expand_as(b)
        p = a * y
        (ah, al), (yh, yl) = split(a), split(y)
        e = ((ah * yh - p) + ah * yl + al * yh) + al * yl
        t = total + p
        z = t - total
        rest += ((total - (t - z)) + (p - z)) + e
        total = t
    return total + rest


def solve(A, b):
    """A x = b by torch, refined with residuals in twice the precision."""
    LU, piv = torch.linalg.lu_factor(A)
    x = torch.linalg.lu_solve(LU, piv, b[:, :, None])[:, :, 0]
    for _ in range(2):
        x = x + torch.linalg.lu_solve(LU, piv, residual(A, x, b)[:, :, None])[:, :, 0]
    return LU, piv.to(torch.int32), x


def newton(evaluate, x, solves):
    """The Newton loop of every point at once: state, iteration counts and the Jacobian where each stopped."""
    F, J = evaluate(x, slice(None))
    r0 = F.norm(dim=1)
    live = torch.nonzero(r0 > 0.0).reshape(-1)
    iters = torch.zeros(x.shape[0], dtype=torch.int32, device=x.device)
    for _ in range(solves):
        Fl, Jl = evaluate(x[live], live)
        live, Fl, Jl = (v[Fl.norm(dim=1) > RTOL * r0[live]] for v in (live, Fl, Jl))
        if not live.numel():
            break
        x[live] += torch.linalg.solve(Jl, -Fl[:, :, None])[:, :, 0]
        iters[live] += 1
    return x, iters


def norton_exact(case, fields):
    E, nu, coef, m, dt = NORTON
    lam, mu = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    sig0, deps = fields[:6].t(), fields[6:].t()
    one = torch.tensor([1.0, 1, 1, 0, 0, 0], dtype=torch.float64, device=fields.device)
    eye = torch.eye(6, dtype=torch.float64, device=fields.device)
    K = eye - one[:, None] * one / 3
    C = lam * one[:, None] * one + 2 * mu * eye

    def evaluate(x, at):
        sig = sig0[at] + x[:, :6] @ C
        dev = sig @ K
        seq = torch.sqrt(1.5 * (dev * dev).sum(1))
        inv = torch.where(seq > 0, 1 / seq, torch.zeros_like(seq))
        nrm = 1.5 * dev * inv[:, None]
        dp = x[:, 6]
        F = torch.cat([x[:, :6] - deps[at] + dp[:, None] * nrm, (dp - dt * coef * seq ** m)[:, None]], 1)
        J = torch.zeros((x.shape[0], 7, 7), dtype=torch.float64, device=x.device)
        c = (dp * 2 * mu * inv)[:, None, None]
        J[:, :6, :6] = eye + c * (1.5 * K - nrm[:, :, None] * nrm[:, None, :])
        J[:, :6, 6] = nrm
        J[:, 6, :6] = (-dt * coef * m * seq ** (m - 1) * 2 * mu)[:, None] * nrm
        J[:, 6, 6] = 1.0
        return F, J

    x, iters = newton(evaluate, torch.cat([deps, torch.zeros_like(deps[:, :1])], 1), MAX_ITER)
    D = None
    if case["tangent"]:
        rhs = torch.zeros((x.shape[0], 7, 6), dtype=torch.float64, device=x.device)
        rhs[:, :6] = eye
        X = torch.linalg.solve(evaluate(x, slice(None))[1], rhs)[:, :6]
        D = (C @ X).permute(2, 1, 0).reshape(36, -1).contiguous()
    sig = (sig0 + x[:, :6] @ C).t().contiguous()
    return {"x": x.t().contiguous(), "sig": sig, "D": D, "iters": iters, "status": torch.zeros_like(iters)}


def tanh_exact(case, fields):
    n = case["n"]
    A = fields[:n * n].t().reshape(-1, n, n).transpose(1, 2)
    c, b = fields[n * n:n * n + n].t(), fields[n * n + n:].t()

    def evaluate(x, at):
        t = torch.tanh(x)
        F = (A[at] @ x[:, :, None])[:, :, 0] + c[at] * t - b[at]
        return F, A[at] + torch.diag_embed(c[at] * (1 - t * t))

    x, iters = newton(evaluate, torch.zeros_like(c), MAX_ITER)
    return {"x": x.t().contiguous(), "sig": None, "D": None, "iters": iters, "status": torch.zeros_like(iters)}


def exact(case, seed):
    op, batch = case["op"], case["batch"]
    if op in ("gesv", "factor"):
        n, L = case["n"], int(case["interleaved"])
        ld = lay.pad_ld(batch)
        A, b = systems(n, batch, seed)
        if op == "gesv":
            LU, piv, x = solve(A, b)
            x = lay.vectors_to_layout(x, L, ld)
        else:
            B = right_hand_sides(case, seed)
            each = [solve(A, B[:, r]) for r in range(case["nrhs"])]
            LU, piv, _ = each[0]
            x = lay.multi_rhs_to_layout(torch.stack([v[2] for v in each], dim=1), L, ld)
        keeps = op == "factor" or case["factors"]
        return {"x": x, "LU": lay.matrices_to_layout(LU, L, ld) if keeps else None,
                "ipiv": lay.vectors_to_layout(piv, L, ld), "info": ints(batch)}
    if op == "ragged":
        n, _, b_off, parts = ragged_systems(case, seed)
        x, ipiv = doubles(int(n.sum())), ints(int(n.sum()))
        for k, at, A, b in parts:
            _, piv, xk = solve(A, b)
            place = b_off[at][:, None] + torch.arange(k, device=DEVICE)
            x[place], ipiv[place] = xk, piv
        # the pivots and refinement counts of the binary32 factors have no 64-bit value
        return {"x": x, "ipiv": None if case["mixed"] else ipiv, "info": ints(batch), "steps": None}
    if op == "norton":
        return norton_exact(case, norton_inputs(case, seed))
    return tanh_exact(case, inputs.tanh_points_torch(case["n"], batch, seed, DEVICE))


def tolerance(case):
    """About four times what is measured between the path and `exact`.

    The solutions carry eps times the condition number of the worst systems
    (1e8 by construction, and the tail of the random half): 2e-11 to 4e-10 measured.
    Newton states agree to 3e-16, but a point whose residual lies on the
    stopping threshold may take one iteration more, which moves it by up to 1e-10.
    Whole numbers (pivots, info, counts) are the same but for such ties.
    """
    if case["op"] in ("norton", "tanh"):
        return {"rel": 1e-12, "max": 1e-8, "differ": 1e-4}
    return {"rel": 2e-9, "max": 1e-5, "differ": 1e-4}
