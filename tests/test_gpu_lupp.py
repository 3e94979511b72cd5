"""GPU parity of the batched LUpp kernels against the CPU oracle, through
the C ABI (tl_gesv_batched / tl_getrf_batched / tl_getrs_batched).

Bar (paper Sec. 2.2 arithmetic, identical on both sides):
  * pivots, info and the LU factors: bit-identical to the oracle;
  * x: normwise backward error ||Ax - b|| / (||A|| ||x|| eps) <= 10 n and
    forward error against the oracle's x <= 1e-12 * kappa(A) (the GPU back
    substitution multiplies by RN(1/u_ii) where the oracle divides).
Sizes span several thread blocks and end on a ragged tail.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2609_15217_gb300 import inputs  # noqa: E402
from paper_2609_15217_gb300 import layout as L  # noqa: E402

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps
DEV = "cuda"


@pytest.fixture(scope="module")
def tl():
    from paper_2609_15217_gb300 import tinylu
    return tinylu


@pytest.fixture(scope="module")
def h(tl):
    hh = tl.tl_create()
    yield hh
    tl.tl_destroy(hh)


def gpu_gesv(tl, h, A, b, layout, want_lu=True, ld=None):
    batch, n, _ = A.shape
    ld = ld or L.pad_ld(batch)
    dA = L.matrices_to_layout(torch.from_numpy(A).to(DEV), layout, ld)
    db = L.vectors_to_layout(torch.from_numpy(b).to(DEV), layout, ld)
    dx = torch.full_like(db, -7.0)
    dLU = torch.full_like(dA, -7.0) if want_lu else None
    dpiv = torch.full((db.numel(),), -7, dtype=torch.int32, device=DEV)
    dinfo = torch.full((batch,), -7, dtype=torch.int32, device=DEV)
    st = tl.tl_gesv_batched(h, n, dA, dLU, db, dx, dpiv, dinfo, layout, ld, batch)
    tl.check("tl_gesv_batched", st, h)
    torch.cuda.synchronize()
    x = L.vectors_from_layout(dx, batch, n, layout, ld).cpu().numpy()
    piv = L.vectors_from_layout(dpiv, batch, n, layout, ld).cpu().numpy()
    info = dinfo.cpu().numpy()
    LU = L.matrices_from_layout(dLU, batch, n, layout, ld).cpu().numpy() if want_lu else None
    return x, piv, info, LU


def backward_error(A, x, b):
    r = np.einsum("sij,sj->si", A.astype(np.longdouble), x.astype(np.longdouble)) - b.astype(np.longdouble)
    r = np.abs(r).max(axis=1).astype(np.float64)
    return r / (np.abs(A).sum(axis=2).max(axis=1) * np.abs(x).max(axis=1) * EPS)


def check_solution(A, b, x_gpu, x_orc):
    n = A.shape[-1]
    be = backward_error(A, x_gpu, b)
    assert (be <= 10 * n).all(), f"backward error {be.max():.3g} > {10 * n}"
    kappa = np.linalg.cond(A)
    fe = np.abs(x_gpu - x_orc).max(axis=1) / np.maximum(np.abs(x_orc).max(axis=1), 1e-300)
    assert (fe <= 1e-12 * kappa).all(), f"forward error / kappa {np.max(fe / kappa):.3g}"


ALL_N = list(range(1, 33))


@pytest.mark.parametrize("layout", [0, 1], ids=["per_system", "interleaved"])
@pytest.mark.parametrize("n", ALL_N)
def test_gesv_parity(tl, h, n, layout):
    batch = 3 * 128 + 37
    A, b, _, _ = inputs.sweep_systems(n, batch, inputs.config_seed(2, n))
    x_o, piv_o, info_o, gap, LU_o = oracle.gesv(A, b, want_lu=True)
    x_g, piv_g, info_g, LU_g = gpu_gesv(tl, h, A, b, layout)
    assert np.array_equal(info_g, info_o)
    assert np.array_equal(piv_g, piv_o), f"pivot mismatches: {(piv_g != piv_o).any(axis=1).sum()}"
    assert np.array_equal(LU_g.view(np.int64), LU_o.view(np.int64)), "LU factors differ from the oracle (bitwise)"
    check_solution(A, b, x_g, x_o)
    # without the factors output (the fused kernel that keeps L unpermuted)
    x_g2, piv_g2, info_g2, _ = gpu_gesv(tl, h, A, b, layout, want_lu=False)
    assert np.array_equal(piv_g2, piv_o) and np.array_equal(info_g2, info_o)
    assert np.array_equal(x_g2, x_g)


@pytest.mark.parametrize("layout", [0, 1], ids=["per_system", "interleaved"])
@pytest.mark.parametrize("n", [1, 2, 5, 8, 9, 10, 12, 13, 16, 17, 24, 25, 31, 32])
def test_getrf_getrs_parity(tl, h, n, layout):
    batch = 2 * 128 + 5
    A, b = inputs.uniform_systems(n, batch, 4000 + n)
    LU_o, piv_o, info_o, _ = oracle.getrf(A)
    ld = L.pad_ld(batch)
    dA = L.matrices_to_layout(torch.from_numpy(A).to(DEV), layout, ld)
    dpiv = torch.zeros(n * (ld if layout else batch), dtype=torch.int32, device=DEV)
    dinfo = torch.zeros(batch, dtype=torch.int32, device=DEV)
    tl.check("getrf", tl.tl_getrf_batched(h, n, dA, layout, ld, dpiv, dinfo, batch), h)
    torch.cuda.synchronize()
    LU_g = L.matrices_from_layout(dA, batch, n, layout, ld).cpu().numpy()
    piv_g = L.vectors_from_layout(dpiv, batch, n, layout, ld).cpu().numpy()
    assert np.array_equal(dinfo.cpu().numpy(), info_o)
    assert np.array_equal(piv_g, piv_o)
    assert np.array_equal(LU_g.view(np.int64), LU_o.view(np.int64))
    for nrhs in (1, 3):
        B = inputs.rng(4100 + n).uniform(-1, 1, size=(batch, nrhs, n))
        dB = L.multi_rhs_to_layout(torch.from_numpy(B).to(DEV), layout, ld)
        tl.check("getrs", tl.tl_getrs_batched(h, n, nrhs, dA, dpiv, layout, ld, dB, batch), h)
        torch.cuda.synchronize()
        X_g = L.multi_rhs_from_layout(dB, batch, nrhs, n, layout, ld).cpu().numpy()
        for r in range(nrhs):
            x_o = oracle.getrs(LU_o, piv_o, B[:, r, :])
            check_solution(A, B[:, r, :], X_g[:, r, :], x_o)


@pytest.mark.parametrize("n", [3, 8, 11, 16, 20, 32])
def test_edge_cases(tl, h, n):
    """Zero pivots, all-zero and non-finite systems, exact ties, a pivot
    below DBL_MIN, and the stress magnitude range of Sec. 4.2."""
    batch = 70
    A, b = inputs.uniform_systems(n, batch, 4200 + n)
    A[0, :, min(2, n - 1)] = 0.0                 # zero pivot at step 2 (or n-1)
    A[1] = 0.0                                   # every pivot zero
    A[2, n // 2, n // 3] = np.nan                # non-finite
    A[3, 0, 0] = np.inf
    A[4, :, 0] = 1.0                             # exact tie in column 0
    A[4, :, 0] *= np.where(np.arange(n) % 2, -1.0, 1.0)
    A[5] *= 2.0 ** -1060                         # subnormal pivots (quotient branch)
    A[6] = np.ldexp(A[6], -31)                   # stress range, U[-4.7e-10, 4.7e-10]
    A[7] = np.eye(n)[::-1] * 3.0                 # anti-diagonal permutation
    A[8, :, :] = A[8, :, :] * 0 + np.triu(np.ones((n, n)))  # upper triangular ones
    for layout in (0, 1):
        x_o, piv_o, info_o, _, LU_o = oracle.gesv(A, b, want_lu=True)
        x_g, piv_g, info_g, LU_g = gpu_gesv(tl, h, A, b, layout)
        assert np.array_equal(info_g, info_o)
        assert np.array_equal(piv_g, piv_o)
        ok = info_o == 0
        bad = info_o < 0
        assert np.array_equal(LU_g[~bad].view(np.int64), LU_o[~bad].view(np.int64))
        assert np.array_equal(LU_g[bad], A[bad], equal_nan=True)  # nothing factored
        assert np.isnan(x_g[~ok]).all()
        normal = ok & (np.arange(batch) != 5)
        check_solution(A[normal], b[normal], x_g[normal], x_o[normal])
        # pivots below DBL_MIN: both sides divide in the substitution, so the
        # solution is bit-identical too
        assert np.array_equal(x_g[5], x_o[5], equal_nan=True)


def test_x_aliases_b_and_tiny_batches(tl, h):
    n = 8
    for batch in (1, 2, 31, 33):
        A, b = inputs.uniform_systems(n, batch, 4300 + batch)
        x_o, piv_o, info_o, _ = oracle.gesv(A, b)
        for layout in (0, 1):
            ld = L.pad_ld(batch)
            dA = L.matrices_to_layout(torch.from_numpy(A).to(DEV), layout, ld)
            db = L.vectors_to_layout(torch.from_numpy(b).to(DEV), layout, ld)
            dpiv = torch.zeros(db.numel(), dtype=torch.int32, device=DEV)
            dinfo = torch.zeros(batch, dtype=torch.int32, device=DEV)
            tl.check("gesv", tl.tl_gesv_batched(h, n, dA, None, db, db, dpiv, dinfo, layout, ld, batch), h)
            torch.cuda.synchronize()
            x_g = L.vectors_from_layout(db, batch, n, layout, ld).cpu().numpy()
            check_solution(A, b, x_g, x_o)


def test_argument_errors(tl, h):
    d = torch.zeros(64, dtype=torch.float64, device=DEV)
    i = torch.zeros(64, dtype=torch.int32, device=DEV)
    assert tl.tl_gesv_batched(h, 0, d, None, d, d, i, i, 0, 0, 1) == tl.TL_ERR_INVALID_ARG
    assert tl.tl_last_bad_arg(h) == 2
    assert tl.tl_gesv_batched(h, 33, d, None, d, d, i, i, 0, 0, 1) == tl.TL_ERR_INVALID_ARG
    assert tl.tl_gesv_batched(h, 4, d, None, d, d, i, i, 1, 3, 4) == tl.TL_ERR_INVALID_ARG
    assert tl.tl_last_bad_arg(h) == 10          # ld_batch < batch
    assert tl.tl_gesv_batched(h, 4, None, None, d, d, i, i, 0, 0, 1) == tl.TL_ERR_INVALID_ARG
    assert tl.tl_last_bad_arg(h) == 3
    assert tl.tl_gesv_batched(h, 4, d, None, d, d, i, i, 7, 0, 1) == tl.TL_ERR_INVALID_ARG
    assert tl.tl_last_bad_arg(h) == 9
    assert tl.tl_gesv_batched(h, 4, d, None, d, d, i, i, 0, 0, -1) == tl.TL_ERR_INVALID_ARG
    assert tl.tl_gesv_batched(h, 4, d, None, d, d, i, i, 0, 0, 0) == tl.TL_OK  # empty batch
    assert tl.tl_getrs_batched(h, 4, 0, d, i, 0, 0, d, 1) == tl.TL_ERR_INVALID_ARG
    assert tl.tl_last_bad_arg(h) == 3
    assert tl.tl_getrf_batched(h, 4, d.data_ptr() + 4, 0, 0, i, i, 1) == tl.TL_ERR_INVALID_ARG
    assert tl.tl_last_bad_arg(h) == 3           # misaligned


@pytest.mark.parametrize("layout", [0, 1], ids=["per_system", "interleaved"])
@pytest.mark.parametrize("n", list(range(1, 10)))
def test_one_thread_kernels(tl, h, n, layout):
    """The one-thread register kernels at a batch that ends inside a warp and
    inside a block, with systems that take the exact general path (zero,
    subnormal, huge and non-finite entries) next to ordinary ones."""
    batch = 2 * 128 + 45
    A, b, _, _ = inputs.sweep_systems(n, batch, 6200 + n)
    A[3, :, n // 2] = 0.0
    A[35, n - 1, 0] = np.nan
    A[36] *= 2.0 ** -1060
    A[130, 0, 0] = 1e308
    A[batch - 1, 0, n - 1] = np.inf
    x_o, piv_o, info_o, _, LU_o = oracle.gesv(A, b, want_lu=True)
    assert tl.tl_dispatch_set(h, n, layout, 1, 0) == tl.TL_OK
    try:
        x_g, piv_g, info_g, LU_g = gpu_gesv(tl, h, A, b, layout)
        x_2, piv_2, info_2, _ = gpu_gesv(tl, h, A, b, layout, want_lu=False)
    finally:
        tl.tl_dispatch_set(h, n, layout, 0, 0)
    ok = info_o >= 0
    assert np.array_equal(info_g, info_o) and np.array_equal(info_2, info_o)
    assert np.array_equal(piv_g, piv_o) and np.array_equal(piv_2, piv_o)
    assert np.array_equal(LU_g[ok].view(np.int64), LU_o[ok].view(np.int64))
    assert np.array_equal(x_2, x_g, equal_nan=True) and np.isnan(x_g[info_o != 0]).all()


# (n, side): the batch rules change the default kernel at warps per SM, so the
# lines are given as systems per SM (plus a remainder) and follow the device.
@pytest.mark.parametrize("n,per_sm,more", [(5, 0, 1), (6, 48, 0), (8, 48, 0), (8, 48, 1), (9, 16, 0), (10, 4, 0),
                                           (13, 4, 1), (16, 16, 0), (16, 16, 1), (20, 16, 0), (20, 16, 1), (26, 32, 1),
                                           (32, 54, 0), (32, 54, 1)])
def test_small_batch_rule(tl, h, n, per_sm, more):
    """Both sides of the lines where the default kernel changes with the
    batch, with zero, subnormal, huge and non-finite systems among ordinary
    ones: every output of every call equal bit for bit to one fixed variant's."""
    batch = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
    g = torch.Generator(device=DEV)
    g.manual_seed(17 * n + batch)
    A0 = torch.empty((batch, n, n), dtype=torch.float64, device=DEV).uniform_(-1, 1, generator=g)
    b0 = torch.empty((batch, n), dtype=torch.float64, device=DEV).uniform_(-1, 1, generator=g)
    if batch > 40:
        A0[3, :, n // 2] = 0.0
        A0[5] = 0.0
        A0[7, n - 1, 0] = float("nan")
        A0[8] *= 2.0 ** -1060
        A0[19, 0, 0] = 1e308
        A0[21] *= 2.0 ** 1020
        A0[batch - 2, n // 2] *= 2.0 ** -1040
        A0[batch - 1, 0, n - 1] = float("inf")
    for layout in (0, 1):
        ld = L.pad_ld(batch)
        A = L.matrices_to_layout(A0, layout, ld)
        b = L.vectors_to_layout(b0, layout, ld)
        out = []
        for variant in (0, tl.variant_id(8, shared=True)):
            assert tl.tl_dispatch_set(h, n, layout, variant, 0) == tl.TL_OK
            res = []
            for call in ("gesv", "gesv_lu", "getrf"):
                F = torch.full_like(A, -7.0) if call != "getrf" else A.clone()
                x = torch.full_like(b, -7.0)
                piv = torch.full((b.numel(),), -7, dtype=torch.int32, device=DEV)
                info = torch.full((batch,), -7, dtype=torch.int32, device=DEV)
                if call == "getrf":
                    st = tl.tl_getrf_batched(h, n, F, layout, ld, piv, info, batch)
                else:
                    LU = F if call == "gesv_lu" else None
                    st = tl.tl_gesv_batched(h, n, A, LU, b, x, piv, info, layout, ld, batch)
                tl.check(call, st, h)
                res += [(call, name, t.cpu().numpy().reshape(-1)) for name, t in
                        (("F", F), ("x", x), ("piv", piv), ("info", info))]
            out.append(res)
        tl.tl_dispatch_set(h, n, layout, 0, 0)
        if batch > 40:
            info = out[0][3][2]
            assert info[3] == n // 2 + 1 and info[5] == 1 and info[7] == -1 and info[batch - 1] == -1
        for (call, name, u), (_, _, v) in zip(*out):
            # bit for bit; a NaN of x or of a factor that overflowed may carry another payload
            same = u == v if u.dtype == np.int32 else (u.view(np.int64) == v.view(np.int64)) | (np.isnan(u) & np.isnan(v))
            assert same.all(), (n, batch, layout, call, name, np.flatnonzero(~same)[:5])


@pytest.mark.parametrize("layout", [0, 1], ids=["per_system", "interleaved"])
@pytest.mark.parametrize("n,nrhs,batch", [(5, 1, 61), (6, 2, 64), (7, 1, 333), (8, 2, 1), (9, 1, 45), (4, 6, 2432),
                                          (8, 16, 700), (9, 17, 97), (10, 6, 1), (12, 3, 609), (13, 7, 333),
                                          (16, 32, 61), (20, 3, 700), (24, 5, 612), (27, 12, 41), (32, 6, 2433),
                                          (32, 32, 9), (17, 1, 4865), (24, 2, 4870), (25, 1, 4866), (32, 2, 4867)])
def test_getrs_kernels_agree(tl, h, n, nrhs, batch, layout):
    """The default solves with given factors (one row per lane in small
    batches; in shared memory one thread per right-hand side or 8 lanes per
    system) at partial blocks and warps: equal bit for bit to the register
    kernel of large batches, with a pivot below DBL_MIN (every row of that
    system takes quotients) and a zero pivot among the factors."""
    A, _, _, _ = inputs.sweep_systems(n, batch, 7300 + n)
    A[0, n // 2] *= 2.0 ** -1040
    if batch > 40:
        A[40, :, 1] = 0.0
    ld = L.pad_ld(batch)
    F = L.matrices_to_layout(torch.from_numpy(A).to(DEV), layout, ld)
    piv = torch.zeros(n * (ld if layout else batch), dtype=torch.int32, device=DEV)
    info = torch.zeros(batch, dtype=torch.int32, device=DEV)
    tl.check("getrf", tl.tl_getrf_batched(h, n, F, layout, ld, piv, info, batch), h)
    B = inputs.rng(7400 + n).uniform(-1, 1, size=(batch, nrhs, n))
    B[0, :, n // 2] *= 2.0 ** -1040  # so that x is finite
    B = L.multi_rhs_to_layout(torch.from_numpy(B).to(DEV), layout, ld)
    register_lanes = 1 if n <= 9 else 2 if n <= 12 else 4 if n <= 16 else 8 if n <= 24 else 16
    out = []
    for variant in (0, register_lanes):
        assert tl.tl_dispatch_set(h, n, layout, variant, 0) == tl.TL_OK
        X = B.clone()
        tl.check("getrs", tl.tl_getrs_batched(h, n, nrhs, F, piv, layout, ld, X, batch), h)
        out.append(L.multi_rhs_from_layout(X, batch, nrhs, n, layout, ld).cpu().numpy())
    tl.tl_dispatch_set(h, n, layout, 0, 0)
    finite = np.isfinite(out[0])
    assert np.array_equal(out[0], out[1], equal_nan=True)
    assert np.array_equal(out[0][finite].view(np.int64), out[1][finite].view(np.int64))
    assert finite[0].all()
    if batch > 40:
        assert not np.isfinite(out[0][40]).all(axis=-1).any()
