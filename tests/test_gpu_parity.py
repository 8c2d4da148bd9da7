"""GPU parity of the FP64 tile QR against the CPU oracle (same list, same
seeded inputs), through the C ABI.

Tolerances: the factor R within max|dR| / ||A||_F <= 1e-11; the Householder
vectors (|v| <= 1 by construction) and T factors within 1e-10 absolute; Q
within 1e-12. Integer outputs (lists) are compared bit-exactly elsewhere.
"""
import itertools

import numpy as np
import pytest

from oracle.elim_list import BINARY, FIBONACCI, FLAT, GREEDY, hqr_elim_list
from oracle.householder import householder_qr
from oracle.lstsq import lstsq, lstsq_unblocked
from oracle.tile_qr import apply_q as o_apply_q
from oracle.tile_qr import explicit_q, tile_qr
from paper_1110_1553_gb300 import inputs

torch = pytest.importorskip("torch")
hqr = pytest.importorskip("paper_1110_1553_gb300.hqr")

pytestmark = pytest.mark.gpu
TREES = (FLAT, BINARY, GREEDY, FIBONACCI)
R_TOL = 1e-11
VT_TOL = 1e-10


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1110_1553_gb300 import _build
    _build.build()
    hqr.load()
    hqr.set_timeout_ms(20000)


def pad(A, nb):
    M, N = A.shape
    Mp, Np = -(-M // nb) * nb, -(-N // nb) * nb
    P = np.zeros((Mp, Np))
    P[:M, :N] = A
    return P


def run_both(A, nb, ib, recs):
    Fo = tile_qr(pad(A, nb), nb, ib, recs)
    Fg = hqr.geqrf(torch.from_numpy(np.ascontiguousarray(A)).cuda(), nb, ib, recs)
    return Fo, Fg


def compare_factors(Fo, Fg, A):
    nrm = np.linalg.norm(A)
    tiles = Fg.tiles().cpu().numpy()
    N = Fg.N
    Rg = Fg.R().cpu().numpy()
    Ro = np.triu(Fo.A[:N, :N])
    assert np.max(np.abs(Rg - Ro)) <= R_TOL * nrm
    # every stored V / R entry of every tile
    d = np.abs(tiles - Fo.A)
    assert np.max(d) <= max(VT_TOL, R_TOL * nrm), np.unravel_index(np.argmax(d), d.shape)
    T = Fg.T().cpu().numpy()
    for (r, k), To in Fo.Tg.items():
        assert np.max(np.abs(T[k, r, 0].T - To)) <= VT_TOL, ("Tg", r, k)
    for (i, k), To in Fo.Tk.items():
        assert np.max(np.abs(T[k, i, 1].T - To)) <= VT_TOL, ("Tk", i, k)


@pytest.mark.parametrize("nb,ib", [(16, 4), (64, 16), (256, 32)])
@pytest.mark.parametrize("shape,a,p", [((1, 1), 1, 1), ((2, 1), 2, 1), ((2, 1), 1, 1), ((2, 2), 2, 1),
                                       ((2, 2), 1, 1), ((3, 2), 1, 2)])
def test_each_kernel(nb, ib, shape, a, p):
    # (1,1): GEQRT; (2,1) a=2: +TSQRT; a=1: +TTQRT; (2,2): +UNMQR and TSMQR / TTMQR
    m, n = shape
    A = inputs.gaussian(m * nb, n * nb, seed=100 + nb + 7 * m + n + a)
    recs = hqr_elim_list(m, n, a, p, FLAT, FLAT)
    Fo, Fg = run_both(A, nb, ib, recs)
    compare_factors(Fo, Fg, A)


@pytest.mark.parametrize("low,high", list(itertools.product(TREES, TREES)))
def test_all_tree_pairs(low, high):
    nb, ib, m, n = 16, 4, 9, 4
    A = inputs.gaussian(m * nb, n * nb, seed=3)
    for a, p in ((1, 1), (2, 3), (4, 2), (m, 1)):
        recs = hqr_elim_list(m, n, a, p, low, high)
        Fo, Fg = run_both(A, nb, ib, recs)
        compare_factors(Fo, Fg, A)


def test_square_flat_ts_c1_shape():
    # 512 x 512, nb = 64, ib = 16, flat TS domains a = 8, p = 1: R, T and Q I
    nb, ib = 64, 16
    A = inputs.gaussian(512, 512, seed=1)
    recs = hqr_elim_list(8, 8, 8, 1, FLAT, FLAT)
    Fo, Fg = run_both(A, nb, ib, recs)
    compare_factors(Fo, Fg, A)
    I = torch.eye(512, dtype=torch.float64, device="cuda").t().contiguous().t()
    Qg = Fg.apply_q(I.clone(), trans=False).cpu().numpy()
    Qo = explicit_q(Fo)
    assert np.max(np.abs(Qg - Qo)) <= 1e-12
    assert np.linalg.norm(Qg.T @ Qg - np.eye(512)) <= 1e-12
    Rg = Fg.R().cpu().numpy()
    assert np.linalg.norm(A - Qg @ Rg) / np.linalg.norm(A) <= 1e-13


def test_apply_q_both_ways():
    nb, ib, m, n = 32, 8, 6, 3
    A = inputs.gaussian(m * nb, n * nb, seed=5)
    recs = hqr_elim_list(m, n, 2, 2, GREEDY, FIBONACCI)
    Fo, Fg = run_both(A, nb, ib, recs)
    B = inputs.gaussian(m * nb, 37, seed=6)  # ragged number of columns
    for trans in (True, False):
        Bg = torch.from_numpy(B.copy()).cuda()
        out = Fg.apply_q(Bg, trans=trans).cpu().numpy()
        ref = o_apply_q(Fo, B, trans=trans)
        assert np.max(np.abs(out - ref)) <= 1e-12 * np.linalg.norm(B)
    # Q^T A = [R; 0]
    QtA = Fg.apply_q(torch.from_numpy(A.copy()).cuda(), trans=True).cpu().numpy()
    R = Fg.R().cpu().numpy()
    assert np.max(np.abs(QtA[:n * nb] - R)) <= 1e-12 * np.linalg.norm(A)
    assert np.max(np.abs(QtA[n * nb:])) <= 1e-12 * np.linalg.norm(A)


def test_gels_matches_oracle():
    nb, ib, m, n = 32, 8, 8, 3
    A = inputs.gaussian(m * nb, n * nb, seed=7)
    b = inputs.gaussian(m * nb, 2, seed=8)
    recs = hqr_elim_list(m, n, 2, 2, GREEDY, FIBONACCI)
    x = hqr.gels_qr(torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda(), nb, ib, recs).cpu().numpy()
    for c in range(2):
        xo, _ = lstsq(A, b[:, c], nb, ib, recs)
        kappa = np.linalg.cond(A)
        assert np.linalg.norm(x[:, c] - xo) / np.linalg.norm(xo) <= 1e-15 * kappa * kappa * 10 + 1e-13


@pytest.mark.parametrize("M,N,nb,ib", [(100, 37, 16, 4), (65, 65, 32, 8), (300, 20, 64, 16), (17, 3, 8, 2)])
def test_ragged_shapes(M, N, nb, ib):
    A = inputs.gaussian(M, N, seed=M + N)
    m, n = -(-M // nb), -(-N // nb)
    recs = hqr_elim_list(m, n, 2, 2, GREEDY, BINARY)
    Fo, Fg = run_both(A, nb, ib, recs)
    compare_factors(Fo, Fg, pad(A, nb))
    Ru = householder_qr(A)[0]
    Rg = Fg.R().cpu().numpy()
    s = np.sign(np.diag(Rg)) * np.sign(np.diag(Ru))
    assert np.max(np.abs(Rg * s[:, None] - Ru)) <= 1e-12 * np.linalg.norm(A)


def test_triangular_input_is_exact():
    nb, ib, m = 16, 4, 5
    A = np.triu(inputs.gaussian(m * nb, m * nb, seed=9))
    for low, high, a, p in ((FLAT, FLAT, 1, 1), (GREEDY, FIBONACCI, 2, 2), (BINARY, GREEDY, 5, 1)):
        Fg = hqr.geqrf(torch.from_numpy(A).cuda(), nb, ib, hqr_elim_list(m, m, a, p, low, high))
        assert np.array_equal(Fg.R().cpu().numpy(), A)


def test_zero_matrix_and_single_tile():
    Z = np.zeros((40, 24))
    Fg = hqr.geqrf(torch.from_numpy(Z).cuda(), 8, 4)
    assert not Fg.R().cpu().numpy().any()
    A = inputs.gaussian(8, 8, seed=10)
    Fg = hqr.geqrf(torch.from_numpy(A).cuda(), 8, 2)
    Ro = np.triu(tile_qr(A, 8, 2, hqr_elim_list(1, 1, 1, 1, FLAT, FLAT)).A)
    assert np.max(np.abs(Fg.R().cpu().numpy() - Ro)) <= 1e-13


def test_refactor_is_bitwise_deterministic():
    nb, ib, m, n = 32, 8, 12, 4
    A = torch.from_numpy(inputs.gaussian(m * nb, n * nb, seed=11)).cuda()
    Fg = hqr.geqrf(A, nb, ib, hqr_elim_list(m, n, 2, 3, GREEDY, FIBONACCI))
    t1 = Fg.tiles()
    for _ in range(3):
        Fg.refactor(A)
        assert torch.equal(Fg.tiles(), t1)


def test_invalid_list_rejected():
    recs = hqr_elim_list(4, 2, 1, 1, FLAT, FLAT)
    bad = recs[:-1]
    A = torch.from_numpy(inputs.gaussian(32, 16, seed=12)).cuda()
    with pytest.raises(hqr.HQRError) as e:
        hqr.geqrf(A, 8, 4, bad)
    assert e.value.status == -8


def test_device_wait_times_out_instead_of_hanging():
    # a task given an input that never arrives: the persistent kernel must
    # give up after the time limit, report HQR_ERR_TIMEOUT and leave the
    # context usable
    nb, ib, m, n = 16, 4, 4, 2
    A = torch.from_numpy(inputs.gaussian(m * nb, n * nb, seed=13)).cuda()
    recs = hqr_elim_list(m, n, 1, 1, FLAT, FLAT)
    Fg = hqr.geqrf(A, nb, ib, recs)
    good = Fg.tiles().clone()
    hqr.set_timeout_ms(300)
    try:
        Fg.debug_block_task(Fg.ntasks // 2, 1)
        with pytest.raises(hqr.HQRError) as e:
            Fg.refactor(A)
        assert e.value.status == hqr.ERR_TIMEOUT
        Fg.debug_block_task(Fg.ntasks // 2, 0)
    finally:
        hqr.set_timeout_ms(20000)
    Fg.refactor(A)
    assert torch.equal(Fg.tiles(), good)


# ---------------------------------------------------------------- FP32 --
# FP32 storage and arithmetic against the FP64 oracle run on the same
# (float-rounded) input: R within 5e-6 ||A||_F, Q^T B within 5e-6 ||B||.

@pytest.mark.parametrize("nb,ib", [(16, 4), (64, 16), (256, 32)])
@pytest.mark.parametrize("shape,a,p", [((1, 1), 1, 1), ((2, 1), 2, 1), ((2, 1), 1, 1), ((2, 2), 2, 1),
                                       ((2, 2), 1, 1), ((3, 2), 1, 2)])
def test_each_kernel_fp32(nb, ib, shape, a, p):
    m, n = shape
    A = inputs.gaussian(m * nb, n * nb, seed=300 + nb + 7 * m + n + a).astype(np.float32)
    recs = hqr_elim_list(m, n, a, p, FLAT, FLAT)
    Fo = tile_qr(A.astype(np.float64), nb, ib, recs)
    Fg = hqr.geqrf(torch.from_numpy(np.ascontiguousarray(A)).cuda(), nb, ib, recs)
    Rg = Fg.R().cpu().numpy().astype(np.float64)
    nrm = np.linalg.norm(A.astype(np.float64))
    assert np.max(np.abs(Rg - Fo.R())) <= 5e-6 * nrm
    tiles = Fg.tiles().cpu().numpy().astype(np.float64)
    assert np.max(np.abs(tiles - Fo.A)) <= 5e-5 * max(1.0, nrm)


@pytest.mark.parametrize("low,high", [(FLAT, FLAT), (GREEDY, FIBONACCI), (BINARY, GREEDY), (FIBONACCI, BINARY)])
def test_tree_pairs_fp32_and_apply_q(low, high):
    nb, ib, m, n = 32, 8, 9, 4
    A = inputs.gaussian(m * nb, n * nb, seed=41).astype(np.float32)
    recs = hqr_elim_list(m, n, 2, 3, low, high)
    Fo = tile_qr(A.astype(np.float64), nb, ib, recs)
    Fg = hqr.geqrf(torch.from_numpy(A).cuda(), nb, ib, recs)
    nrm = np.linalg.norm(A.astype(np.float64))
    assert np.max(np.abs(Fg.R().cpu().numpy() - Fo.R())) <= 5e-6 * nrm
    B = inputs.gaussian(m * nb, 5, seed=42).astype(np.float32)
    for trans in (True, False):
        out = Fg.apply_q(torch.from_numpy(B.copy()).cuda(), trans=trans).cpu().numpy()
        ref = o_apply_q(Fo, B.astype(np.float64), trans=trans)
        assert np.max(np.abs(out - ref)) <= 5e-6 * np.linalg.norm(B.astype(np.float64))


# ------------------------------------------------------- split panels --
# CUDA-core panels of tiles with nb >= 64 run as one task per ib block plus
# the updates of the panel's own trailing columns. Same tolerances as whole
# panels; R also against a whole-panel run (split turned off).

@pytest.mark.parametrize("low,high,a,p,ib", [(FLAT, FLAT, 4, 1, 16), (GREEDY, FIBONACCI, 2, 2, 16),
                                             (BINARY, GREEDY, 1, 3, 16), (GREEDY, GREEDY, 2, 1, 8)])
def test_split_panels_fp64(low, high, a, p, ib):
    """ib = 8: blocks narrower than the 16-column update slabs (a block's trailing work starts
    inside its own slab)."""
    nb, m, n = 64, 7, 4
    A = inputs.gaussian(m * nb, n * nb - 3, seed=61 + a)  # ragged last tile column
    recs = hqr_elim_list(m, n, a, p, low, high)
    Fo, Fs = run_both(A, nb, ib, recs)
    compare_factors(Fo, Fs, pad(A, nb))
    B = inputs.gaussian(A.shape[0], 3, seed=62)
    for trans in (True, False):
        out = Fs.apply_q(torch.from_numpy(B.copy()).cuda(), trans=trans).cpu().numpy()
        ref = o_apply_q(Fo, B, trans=trans)
        assert np.max(np.abs(out - ref)) <= 1e-12 * np.linalg.norm(B)
    hqr.set_panel_split(0)
    try:
        Fw = hqr.geqrf(torch.from_numpy(np.ascontiguousarray(A)).cuda(), nb, ib, recs)
    finally:
        hqr.set_panel_split(64)
    assert np.max(np.abs(Fs.R().cpu().numpy() - Fw.R().cpu().numpy())) <= 1e-13 * np.linalg.norm(A)


@pytest.mark.parametrize("nb,ib", [(128, 16), (128, 32), (256, 32)])
def test_split_panels_fp32(nb, ib):
    """FP32 panels are split where a block spans whole update slabs (here slabs of 16)."""
    m, n = 6, 3
    A = inputs.gaussian(m * nb, n * nb, seed=63 + ib).astype(np.float32)
    recs = hqr_elim_list(m, n, 2, 2, GREEDY, FIBONACCI)
    Fo = tile_qr(A.astype(np.float64), nb, ib, recs)
    hqr.set_slab_widths(16, 0, 0)
    try:
        Fg = hqr.geqrf(torch.from_numpy(A).cuda(), nb, ib, recs)
    finally:
        hqr.set_slab_widths(0, 0, 0)
    nrm = np.linalg.norm(A.astype(np.float64))
    assert np.max(np.abs(Fg.R().cpu().numpy().astype(np.float64) - Fo.R())) <= 5e-6 * nrm
    tiles = Fg.tiles().cpu().numpy().astype(np.float64)
    assert np.max(np.abs(tiles - Fo.A)) <= 5e-5 * max(1.0, nrm)


def test_split_panels_least_squares_plan():
    """A least-squares plan whose panels are split: x equals the FP64 oracle's."""
    nb, ib = 64, 16
    A = inputs.gaussian(700, 190, seed=64)
    b = inputs.rng(64, 1).standard_normal(700)
    x = torch.zeros(190, dtype=torch.float64, device="cuda")
    plan = hqr.LSPlan([(torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda(), x)], refine_iters=0,
                      configs=[hqr.tile_config(nb, ib, 2, 2, "greedy", "fibonacci")])
    plan.run()
    assert plan.status() == 0
    xo = lstsq_unblocked(A, b)
    assert np.linalg.norm(x.cpu().numpy() - xo) / np.linalg.norm(xo) <= 1e-12


@pytest.mark.parametrize("shape,a,nb,ib", [((1, 1), 1, 64, 16), ((2, 1), 2, 64, 16), ((2, 1), 1, 64, 16), ((2, 1), 2, 24, 6),
                                           ((2, 1), 1, 256, 32), ((2, 1), 2, 16, 16), ((2, 2), 2, 8, 2)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_panel_scaled_columns(shape, a, nb, ib, dtype):
    """GEQRT, TSQRT and TTQRT blocks on columns whose sums of squares lie inside
    and far outside the range whose columns are used unscaled: QR commutes
    with a column scaling by powers of two, so R must be the unscaled R with
    scaled columns, each column within R_TOL (FP32: 5e-6) of its own norm; zero
    columns stay zero."""
    if dtype == "f32" and ib % 4:
        pytest.skip("FP32 inner blocks are multiples of 4")
    m, n = shape
    A = inputs.gaussian(m * nb, n * nb, seed=170 + nb + a)
    recs = hqr_elim_list(m, n, a, 1, FLAT, FLAT)
    exps = [0, -400, 400, 0, -60, 60, -480] if dtype == "f64" else [0, -60, 60, 0, -30, 30, -90]
    scale = np.ldexp(1.0, np.resize(exps, n * nb))
    scale[[1, 6]] = 0.0
    A = A.astype(np.float32).astype(np.float64) if dtype == "f32" else A
    base = tile_qr(A * (scale != 0), nb, ib, recs).R()
    As = torch.from_numpy(A * scale).cuda()
    R = hqr.geqrf(As if dtype == "f64" else As.float(), nb, ib, recs).R().double().cpu().numpy()
    assert np.all(R[:, scale == 0] == 0)
    keep = scale != 0
    err = np.abs(R[:, keep] / scale[keep] - base[:, keep]) / np.linalg.norm(A, axis=0)[keep]
    assert np.max(err) <= (R_TOL if dtype == "f64" else 5e-6)


@pytest.mark.parametrize("shape,a,nb,ib", [((1, 1), 1, 64, 16), ((2, 1), 2, 64, 16), ((2, 1), 1, 64, 16), ((2, 1), 2, 128, 32),
                                           ((3, 2), 2, 16, 8)])
@pytest.mark.parametrize("dtype,exps", [("f32", (13, 116)), ("f32", (10, 119)), ("f32", (6, 121)), ("f32", (-23, -116)),
                                        ("f32", (-20, -120)), ("f32", (120, -120, 0)), ("f64", (60, 965)), ("f64", (60, 980)),
                                        ("f64", (-60, -1000)), ("f64", (1000, -1000, 0))])
def test_panel_columns_of_far_sizes(shape, a, nb, ib, dtype, exps):
    """GEQRT, TSQRT and TTQRT blocks whose columns are of ordinary size next to
    columns near the type's largest or smallest numbers: R must be the unscaled
    R with scaled columns (a column scaling by powers of two commutes with QR),
    each column within R_TOL (FP32: 5e-6) of its own norm."""
    m, n = shape
    A = inputs.gaussian(m * nb, n * nb, seed=270 + nb + a)
    recs = hqr_elim_list(m, n, a, 1, FLAT, FLAT)
    scale = np.ldexp(1.0, np.resize(exps, n * nb))
    A = A.astype(np.float32).astype(np.float64) if dtype == "f32" else A
    base = tile_qr(A, nb, ib, recs).R()
    As = torch.from_numpy(A * scale).cuda()
    R = hqr.geqrf(As if dtype == "f64" else As.float(), nb, ib, recs).R().double().cpu().numpy()
    err = np.abs(R / scale - base) / np.linalg.norm(A, axis=0)
    assert np.max(err) <= (R_TOL if dtype == "f64" else 5e-6)


@pytest.mark.parametrize("shape,a", [((1, 1), 1), ((2, 1), 2), ((2, 1), 1)])
@pytest.mark.parametrize("prec,nb,ib", [("f64", 32, 8), ("f64", 64, 16), ("f32", 32, 8), ("f32", 128, 16), ("tensor", 128, 128)])
@pytest.mark.parametrize("dense", [False, True])
def test_nan_reaches_r(shape, a, prec, nb, ib, dense):
    """One NaN below the diagonal, in column c of the last tile, among zeros or
    in a full tile (where the reflectors before c spread it over the column,
    so that nothing else is left there): R(c, c) is NaN, and the columns before
    c are what they are without it."""
    m, n = shape
    A = inputs.gaussian(m * nb, nb, seed=290 + nb)
    row = m * nb - 2 if m == 1 or a == 2 else nb
    if not dense:
        A[(m - 1) * nb + 1:] = 0
        A[(m - 1) * nb] = 0 if m > 1 else A[0]
    recs = hqr_elim_list(m, 1, a, 1, FLAT, FLAT)
    dt = torch.float64 if prec == "f64" else torch.float32
    for c in (0, 1, ib - 1, nb // 2, nb - 3):
        B = torch.from_numpy(A.copy()).to(dt)
        R0 = hqr.geqrf(B.cuda(), nb, ib, recs, tensor=prec == "tensor").R().cpu()
        B[row, c] = float("nan")
        R = hqr.geqrf(B.cuda(), nb, ib, recs, tensor=prec == "tensor").R().cpu()
        assert torch.isnan(R[c, c]), c
        assert torch.equal(R[:, :c], R0[:, :c]), c


@pytest.mark.parametrize("dtype,nb,ib,w", [("f64", 64, 32, 16), ("f64", 88, 8, 16), ("f64", 96, 16, 8), ("f64", 96, 16, 16),
                                           ("f64", 104, 8, 4), ("f64", 40, 4, 4), ("f32", 128, 16, 16), ("f32", 128, 16, 12),
                                           ("f32", 128, 32, 16), ("f32", 64, 8, 64), ("f32", 136, 8, 8)])
def test_updates_on_both_sides_of_the_resident_limit(dtype, nb, ib, w):
    """Update tasks with the reflector tile staged whole (small tiles, narrow
    slabs) and block by block (the others), and right-hand sides of 1 and 19
    columns, which may take the other way than the tiles: R, Q^T B and Q B
    against the oracle, with TS and TT kernels and a ragged last tile."""
    m, n = 4, 2
    A = inputs.gaussian(m * nb - 5, n * nb - 3, seed=180 + nb + w)
    recs = hqr_elim_list(m, n, 2, 1, GREEDY, GREEDY)
    rt, bt = (R_TOL, 1e-12) if dtype == "f64" else (5e-6, 5e-6)
    if dtype == "f32":
        A = A.astype(np.float32).astype(np.float64)
    Fo = tile_qr(pad(A, nb), nb, ib, recs)
    Ad = torch.from_numpy(A).cuda()
    hqr.set_slab_widths(w, 0, 0)
    try:
        F = hqr.geqrf(Ad if dtype == "f64" else Ad.float(), nb, ib, recs)
    finally:
        hqr.set_slab_widths(0, 0, 0)
    N = A.shape[1]
    assert np.max(np.abs(F.R().double().cpu().numpy() - np.triu(Fo.A[:N, :N]))) <= rt * np.linalg.norm(A)
    for k in (1, 19):
        B = pad(inputs.gaussian(A.shape[0], k, seed=181 + k).astype(np.float32).astype(np.float64), 1)
        for trans in (True, False):
            Bd = torch.from_numpy(B.copy()).cuda()
            out = F.apply_q(Bd if dtype == "f64" else Bd.float(), trans=trans).double().cpu().numpy()
            ref = o_apply_q(Fo, np.vstack([B, np.zeros((m * nb - B.shape[0], k))]), trans=trans)[:B.shape[0]]
            assert np.max(np.abs(out - ref)) <= bt * np.linalg.norm(B)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_apply_q_block_widths(dtype):
    """Right-hand sides of sizes that take blocks of 4, 8 and 16 columns, in turn
    on one factorization (the block layout changes between calls)."""
    nb, ib, m, n = 16, 8, 40, 2
    A = inputs.gaussian(m * nb, n * nb, seed=190).astype(np.float32).astype(np.float64)
    recs = hqr_elim_list(m, n, 4, 2, GREEDY, BINARY)
    Fo = tile_qr(A, nb, ib, recs)
    Ad = torch.from_numpy(A).cuda()
    F = hqr.geqrf(Ad if dtype == "f64" else Ad.float(), nb, ib, recs)
    for k in (3, 110, 450, 102, 103, 5, 401, 62, 63, 150, 151, 400):
        B = inputs.gaussian(m * nb, k, seed=191 + k).astype(np.float32).astype(np.float64)
        for trans in (True, False):
            Bd = torch.from_numpy(B.copy()).cuda()
            out = F.apply_q(Bd if dtype == "f64" else Bd.float(), trans=trans).double().cpu().numpy()
            err = np.max(np.abs(out - o_apply_q(Fo, B, trans=trans)))
            assert err <= (1e-12 if dtype == "f64" else 5e-6) * np.linalg.norm(B), (k, trans)


@pytest.mark.parametrize("prec,nb,ib", [("f64", 64, 16), ("f64", 256, 32), ("f32", 64, 16), ("tensor", 128, 128)])
def test_reflector_scalars(prec, nb, ib):
    """beta, tau and v of reflectors of (alpha, x) over the range whose columns are
    used unscaled, against 60 digits: A = [diag(alpha); diag(x)] killed by one TSQRT
    has nb independent ones. In units u of rounding (2^-53, FP32 2^-24): n2 =
    alpha^2 + x^2 carries 2 (x^2 and the sum), so h = sqrt(n2) 1 of them, 0.5 of the
    rounded n2 y0 and 1 of its own, 2.5, with the series and Newton steps below
    0.1: beta within 3. |alpha| / h <= 1 adds the 2.5 of 1 / h (FP32: 3, formed from
    h) and a rounding to tau in [1, 2]: 4 (5). x / (alpha - beta): 2.5 of h, one
    each of the sum, the reciprocal and the product: 6."""
    from decimal import Decimal, getcontext
    getcontext().prec = 60
    u = Decimal(2) ** (-53 if prec == "f64" else -24)
    rng = np.random.default_rng(nb)
    xr, ar = {"f64": (60, 120), "f32": (19, 39), "tensor": (48, 49)}[prec]  # |x| and |alpha| up to (x: and from 1 over) 2^this
    dt = np.float64 if prec == "f64" else np.float32
    for trial in range(6):
        x = (rng.choice([-1, 1], nb) * 2.0 ** rng.uniform(-xr, xr, nb)).astype(dt)
        al = (rng.choice([-1, 1], nb) * 2.0 ** rng.uniform(-ar, ar, nb)).astype(dt)
        near = rng.random(nb) < 0.5  # half of them of one size
        al[near] = (x[near] * rng.uniform(0.01, 100, near.sum()) * rng.choice([-1, 1], near.sum())).astype(dt)
        al[:2] = 0.0, -0.0
        A = torch.from_numpy(np.vstack([np.diag(al), np.diag(x)])).cuda()
        F = hqr.geqrf(A, nb, ib, hqr_elim_list(2, 1, 2, 1, FLAT, FLAT), tensor=prec == "tensor")
        R, V, T = F.R().cpu().numpy(), F.tiles().cpu().numpy()[nb:2 * nb], F.T().cpu().numpy()[0, 1, 1]
        for j in range(nb):
            a, b = Decimal(float(al[j])), Decimal(float(x[j]))
            h = (a * a + b * b).sqrt()
            beta = -h if a >= 0 else h
            for got, ref, tol in ((R[j, j], beta, 3), (T[j, j % ib], 1 + abs(a) / h, 4 if prec == "f64" else 5),
                                  (V[j, j], b / (a - beta), 6)):
                assert abs(Decimal(float(got)) - ref) <= tol * u * abs(ref), (trial, j, got, ref)


def test_captured_refactor_between_block_widths():
    """A factorization captured in a CUDA graph gives the same bits when replayed
    after right-hand sides of another block width than those before the capture.
    FP64 tiles of 256 with blocks of 16 and slabs of 8 columns: right-hand-side
    blocks of 4 columns leave an update 58,368 bytes of shared memory and stage
    8 columns of V at once, blocks of 16 columns 91,008 and 16 (72,448 used), so
    the descriptor of one width must not reach the launch of another."""
    nb, ib, m, n = 256, 16, 12, 2
    A = [torch.from_numpy(inputs.gaussian(m * nb, n * nb, seed=230 + q)).cuda().t().contiguous().t() for q in range(2)]
    F = hqr.geqrf(A[0], nb, ib, hqr_elim_list(m, n, 4, 1, GREEDY, GREEDY))
    ref = F.tiles().clone()
    F.apply_q(torch.ones(m * nb, 3, dtype=torch.float64, device="cuda"), trans=True)  # blocks of 4
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        F.refactor_async(A[0], s)
    F.refactor(A[1])
    F.apply_q(torch.ones(m * nb, 2000, dtype=torch.float64, device="cuda"), trans=True)  # blocks of 16
    g.replay()
    torch.cuda.synchronize()
    assert F.status() == 0
    assert torch.equal(F.tiles(), ref)
