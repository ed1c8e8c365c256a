"""GPU parity of gemv / ger / symv / trmv / trsv against the CPU oracle, through the C ABI."""
import itertools

import numpy as np
import pytest
import torch

from oracle import blas_oracle as orc
from paper_2411_07211_b200 import synth
from tests.gpu_util import TOL, Guarded, assert_close, assert_same_gaps, pick, place

pytestmark = pytest.mark.gpu

DTYPES = [np.float32, np.float64]
ORDERS = [orc.ROW_MAJOR, orc.COL_MAJOR]
UPLOS = [orc.UPPER, orc.LOWER]
TRANSES = [orc.NO_TRANS, orc.TRANS]
DIAGS = [orc.NON_UNIT, orc.UNIT]


@pytest.fixture(scope="module")
def b2():
    from paper_2411_07211_b200 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(b2):
    c = b2.Context()
    c.reset()
    return c


def matbuf(seed, major, minor, lda, dtype):
    """major x lda buffer, pad columns NaN."""
    buf = synth.vector_np(seed, 7, major * lda, dtype).reshape(major, lda)
    buf[:, minor:] = np.nan
    return buf.ravel()


GEMV_SHAPES = [(1, 1), (3, 5), (17, 33), (64, 64), (100, 700), (700, 100), (257, 1031), (1500, 40), (40, 3000),
               (2049, 513), (130, 2100), (4100, 24),
               # narrow shapes of the paper's skinny study (Section 6.2.2): N = 40, N <= 88 / 44, M a power of 2 or 3
               (2187, 40), (2187, 44), (4096, 88), (88, 4096), (44, 2187), (6561, 8)]


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("order", ORDERS)
@pytest.mark.parametrize("trans", TRANSES)
@pytest.mark.parametrize("m,n", GEMV_SHAPES)
def test_gemv(b2, ctx, dtype, order, trans, m, n):
    minor, major = (n, m) if order == orc.ROW_MAJOR else (m, n)
    lenx, leny = (n, m) if trans == orc.NO_TRANS else (m, n)
    cases = [(0, 0, 1, 1, 0.5), (0, 0, 1, 1, 0.0), (1, 0, 2, 2, 0.5), (4, 1, -1, 3, 0.0), (3, 0, 1, -2, 0.5),
             (0, 0, -2, 3, 0.5)]  # unpadded with strided vectors: the narrow-matrix kernels see every increment
    for pad, offset, incx, incy, beta in cases:
        lda = minor + pad
        a = matbuf(m * 31 + n, major, minor, lda, dtype)
        x = synth.vector_np(1, m + n, lenx, dtype)
        y = synth.vector_np(2, m + n, leny, dtype) if beta != 0 else np.full(leny, np.nan, dtype=dtype)
        hx, hy = place(x, incx), place(y, incy)
        ga, gx, gy = Guarded(a, offset), Guarded(hx), Guarded(hy)
        b2.gemv(ctx, order, trans, m, n, 1.25, ga.t, lda, gx.t, incx, beta, gy.t, incy)
        oy = hy.copy()
        absterms = orc.gemv(order, trans, m, n, dtype(1.25), a, lda, hx, incx, dtype(beta), oy, incy)
        ry = gy.host()
        assert_close(pick(ry, leny, incy), pick(oy, leny, incy), absterms, dtype, f"gemv pad={pad} off={offset}")
        assert_same_gaps(ry, hy, leny, incy)
        assert np.array_equal(ga.host(), a, equal_nan=True) and np.array_equal(gx.host(), hx, equal_nan=True)
        ga.check_guards(), gx.check_guards(), gy.check_guards()
    # alpha == 0: y <- beta*y, A and x may hold anything
    lda = minor
    y = synth.vector_np(2, 5, leny, dtype)
    gy = Guarded(y)
    junk = Guarded(np.full(major * lda, np.nan, dtype=dtype))
    jx = Guarded(np.full(lenx, np.nan, dtype=dtype))
    b2.gemv(ctx, order, trans, m, n, 0.0, junk.t, lda, jx.t, 1, 0.5, gy.t, 1)
    assert np.array_equal(gy.host(), dtype(0.5) * y)
    b2.gemv(ctx, order, trans, m, n, 0.0, junk.t, lda, jx.t, 1, 0.0, gy.t, 1)
    assert np.array_equal(gy.host(), np.zeros(leny, dtype=dtype))


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("order", ORDERS)
@pytest.mark.parametrize("m,n", GEMV_SHAPES)
def test_ger(b2, ctx, dtype, order, m, n):
    minor, major = (n, m) if order == orc.ROW_MAJOR else (m, n)
    for pad, offset, incx, incy in [(0, 0, 1, 1), (1, 0, 2, 2), (4, 1, -1, 3), (2, 0, 1, -2), (0, 0, -1, 2)]:
        lda = minor + pad
        a = matbuf(m * 17 + n, major, minor, lda, dtype)
        x = synth.vector_np(3, m + n, m, dtype)
        y = synth.vector_np(4, m + n, n, dtype)
        hx, hy = place(x, incx), place(y, incy)
        ga, gx, gy = Guarded(a, offset), Guarded(hx), Guarded(hy)
        b2.ger(ctx, order, m, n, 1.25, gx.t, incx, gy.t, incy, ga.t, lda)
        oa = a.copy()
        absterms = orc.ger(order, m, n, dtype(1.25), hx, incx, hy, incy, oa, lda)
        ra = ga.host()
        view = (lambda b: b.reshape(major, lda)[:, :minor]) if True else None
        got, want = view(ra), view(oa)
        if order == orc.COL_MAJOR:
            got, want = got.T, want.T
        assert_close(got, want, absterms, dtype, f"ger pad={pad} off={offset}")
        assert_same_gaps(ra, a)
        ga.check_guards()
        assert np.array_equal(gx.host(), hx, equal_nan=True) and np.array_equal(gy.host(), hy, equal_nan=True)
    ga = Guarded(a)
    b2.ger(ctx, order, m, n, 0.0, gx.t, incx, gy.t, incy, ga.t, lda)
    assert np.array_equal(ga.host(), a, equal_nan=True)


def tri_buf(seed, n, lda, dtype, order, uplo, diag):
    """Conditioned triangular matrix; everything the routine must not use is NaN."""
    buf = synth.matrix_np(seed, 30 + n, n, n, lda, dtype, tri_n=n)
    p, q = np.indices((n, lda))
    r, c = (p, q) if order == orc.ROW_MAJOR else (q, p)
    inside = (r <= c) if uplo == orc.UPPER else (r >= c)
    bad = ~inside | (q >= n)
    if diag == orc.UNIT:
        bad |= (r == c)
    buf[bad] = np.nan
    return buf.ravel()


TRI_SIZES = [1, 2, 5, 31, 64, 65, 127, 128, 129, 200, 513, 1100]
TRI_CASES = [(0, 0, 1), (1, 0, 2), (4, 1, -1), (0, 0, 2)]  # pad, offset, inc


@pytest.fixture(params=[0, 2], ids=["general-kernel", "ring-kernel"])
def symv_kernel(request, b2):
    """symv picks its kernel by the size of the triangle; both are run on every test size."""
    old = b2.get_tuning(b2.KNOB_TRI_TILE)
    b2.set_tuning(b2.KNOB_TRI_TILE, request.param)
    yield request.param
    b2.set_tuning(b2.KNOB_TRI_TILE, old)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("order", ORDERS)
@pytest.mark.parametrize("uplo", UPLOS)
@pytest.mark.parametrize("n", TRI_SIZES)
def test_symv(b2, ctx, dtype, order, uplo, n, symv_kernel):
    for (pad, offset, inc), beta in zip(TRI_CASES, [0.5, 0.0, 0.5, 0.0]):
        lda = n + pad
        a = tri_buf(9, n, lda, dtype, order, uplo, orc.NON_UNIT)
        x = synth.vector_np(5, n, n, dtype)
        y = synth.vector_np(6, n, n, dtype) if beta != 0 else np.full(n, np.nan, dtype=dtype)
        hx, hy = place(x, inc), place(y, -inc)
        ga, gx, gy = Guarded(a, offset), Guarded(hx), Guarded(hy)
        b2.symv(ctx, order, uplo, n, 1.25, ga.t, lda, gx.t, inc, beta, gy.t, -inc)
        oy = hy.copy()
        absterms = orc.symv(order, uplo, n, dtype(1.25), a, lda, hx, inc, dtype(beta), oy, -inc)
        ry = gy.host()
        assert_close(pick(ry, n, -inc), pick(oy, n, -inc), absterms, dtype, f"symv pad={pad}")
        assert_same_gaps(ry, hy, n, -inc)
        ga.check_guards(), gy.check_guards()


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("order", ORDERS)
@pytest.mark.parametrize("uplo", UPLOS)
@pytest.mark.parametrize("trans", TRANSES)
@pytest.mark.parametrize("diag", DIAGS)
@pytest.mark.parametrize("n", TRI_SIZES)
def test_trmv_trsv(b2, ctx, dtype, order, uplo, trans, diag, n):
    for pad, offset, inc in TRI_CASES:
        lda = n + pad
        a = tri_buf(12, n, lda, dtype, order, uplo, diag)
        x = synth.vector_np(7, n, n, dtype)
        hx = place(x, inc)
        ga, gx = Guarded(a, offset), Guarded(hx)
        b2.trmv(ctx, order, uplo, trans, diag, n, ga.t, lda, gx.t, inc)
        ox = hx.copy()
        absterms = orc.trmv(order, uplo, trans, diag, n, a, lda, ox, inc)
        rx = gx.host()
        assert_close(pick(rx, n, inc), pick(ox, n, inc), absterms, dtype, f"trmv pad={pad}")
        assert_same_gaps(rx, hx, n, inc)
        ga.check_guards(), gx.check_guards()
        # trsv: residual of the GPU solution, then forward error against the oracle's solution
        gx = Guarded(hx)
        b2.trsv(ctx, order, uplo, trans, diag, n, ga.t, lda, gx.t, inc)
        assert ctx.device_status() == 0
        rx = gx.host()
        assert_same_gaps(rx, hx, n, inc)
        gx.check_guards()
        resid, scale = orc.trsv_residual(order, uplo, trans, diag, n, a, lda, hx, inc, rx, inc)
        tol = TOL[np.dtype(dtype)]
        assert np.all(resid <= tol * scale), f"trsv residual pad={pad}: worst {np.max(resid / scale):.3e}"
        ox = hx.copy()
        absterms = orc.trsv(order, uplo, trans, diag, n, a, lda, ox, inc)
        assert_close(pick(rx, n, inc), pick(ox, n, inc), 8 * absterms, dtype, "trsv forward")  # |a_ii| >= 1
        assert np.array_equal(ga.host(), a, equal_nan=True)


def test_trsv_bounded_wait_reports_timeout(b2):
    """Host-injected failure: one block of the solve order never publishes (a test hook in the
    library), so its dependants' waits run out.  They must return a status, not hang."""
    ctx = b2.Context(wait_limit=2000)
    ctx.reset()
    n = 128 * 6
    a = Guarded(tri_buf(3, n, n, np.float32, orc.ROW_MAJOR, orc.LOWER, orc.NON_UNIT))
    x = Guarded(synth.vector_np(1, 1, n, np.float32))
    b2.set_tuning(b2.KNOB_TRSV_DEBUG_SKIP, 2)
    try:
        b2.trsv(ctx, orc.ROW_MAJOR, orc.LOWER, orc.NO_TRANS, orc.NON_UNIT, n, a.t, n, x.t, 1)
        torch.cuda.synchronize()
        assert ctx.device_status() == b2.STATUS_TIMEOUT
    finally:
        b2.set_tuning(b2.KNOB_TRSV_DEBUG_SKIP, -1)
    # a timed-out call leaves the control block dirty: without a reset the next call must say so
    # (and leave x as it was) instead of returning an unsolved vector with status 0
    ctx.status.zero_()
    x = Guarded(synth.vector_np(1, 1, n, np.float32))
    b2.trsv(ctx, orc.ROW_MAJOR, orc.LOWER, orc.NO_TRANS, orc.NON_UNIT, n, a.t, n, x.t, 1)
    torch.cuda.synchronize()
    assert ctx.device_status() == b2.STATUS_TIMEOUT
    assert np.array_equal(x.host(), synth.vector_np(1, 1, n, np.float32))
    ctx.reset()
    x = Guarded(synth.vector_np(1, 1, n, np.float32))
    b2.trsv(ctx, orc.ROW_MAJOR, orc.LOWER, orc.NO_TRANS, orc.NON_UNIT, n, a.t, n, x.t, 1)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    resid, scale = orc.trsv_residual(orc.ROW_MAJOR, orc.LOWER, orc.NO_TRANS, orc.NON_UNIT, n, a.host(), n,
                                     synth.vector_np(1, 1, n, np.float32), 1, x.host(), 1)
    assert np.all(resid <= 2e-6 * scale)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("front,cluster,pm_from", [(0, 0, 16), (2, 0, 0), (2, 0, 5), (2, 2, 0), (2, 2, 3)])
def test_trsv_every_kernel_choice(b2, ctx, dtype, front, cluster, pm_from):
    """Behind the cluster kernel trsv has three more code paths (block-row kernel; sub-block kernel block by block;
    sub-block kernel in clusters), and the sub-block kernel premultiplies the last tile of a block row from
    a given row on.  Workspaces too small for the cluster kernel reach them; here each is forced for every
    view, on sizes with a ragged last block and more block rows than one cluster holds, with the
    premultiplied tile starting at the first row and inside the matrix."""
    old = (b2.get_tuning(b2.KNOB_TRSV_FRONT), b2.get_tuning(b2.KNOB_TRSV_CLUSTER), b2.get_tuning(b2.KNOB_TRSV_PM_FROM))
    b2.set_tuning(b2.KNOB_TRSV_FRONT, front)
    b2.set_tuning(b2.KNOB_TRSV_CLUSTER, cluster)
    b2.set_tuning(b2.KNOB_TRSV_PM_FROM, pm_from)
    try:
        tol = TOL[np.dtype(dtype)]
        for n in (130, 1100, 2052):
            for uplo, trans, diag in itertools.product(UPLOS, TRANSES, DIAGS):
                a = tri_buf(21, n, n, dtype, orc.ROW_MAJOR, uplo, diag)
                hx = synth.vector_np(9, n, n, dtype)
                ga, gx = Guarded(a), Guarded(hx)
                b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, diag, n, ga.t, n, gx.t, 1)
                assert ctx.device_status() == 0
                rx = gx.host()
                gx.check_guards()
                resid, scale = orc.trsv_residual(orc.ROW_MAJOR, uplo, trans, diag, n, a, n, hx, 1, rx, 1)
                assert np.all(resid <= tol * scale), f"n={n} {uplo} {trans} {diag}: worst {np.max(resid / scale):.3e}"
    finally:
        b2.set_tuning(b2.KNOB_TRSV_FRONT, old[0])
        b2.set_tuning(b2.KNOB_TRSV_CLUSTER, old[1])
        b2.set_tuning(b2.KNOB_TRSV_PM_FROM, old[2])


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("m,n", [(1, 5), (3, 1), (7, 3), (257, 31), (1025, 1), (2, 4099), (4100, 3), (1024, 5)])
def test_ger_unpadded_odd_widths(b2, ctx, dtype, m, n):
    """Matrices that are one contiguous run with rows off 16-byte boundaries: elements before the first and after the
    last pack, packs that hold several rows, one row per element, rows longer than a chunk."""
    for off, incx, incy in ((0, 1, 1), (1, 2, -1), (3, -1, 3)):
        a, x, y = synth.matrix_np(3, m, m, n, n, dtype).ravel(), synth.vector_np(5, m, m, dtype), synth.vector_np(6, n, n, dtype)
        ga, gx, gy = Guarded(a, off), Guarded(place(x, incx)), Guarded(place(y, incy))
        b2.ger(ctx, orc.ROW_MAJOR, m, n, 0.75, gx.t, incx, gy.t, incy, ga.t, n)
        oa = a.copy()
        absterms = orc.ger(orc.ROW_MAJOR, m, n, dtype(0.75), place(x, incx), incx, place(y, incy), incy, oa, n)
        assert_close(ga.host(), oa, np.asarray(absterms).ravel(), dtype, f"ger off={off}")
        ga.check_guards()


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("n", [5, 16, 31, 33, 36, 63, 66, 127, 131, 252, 255, 509, 515, 1030])
def test_ger_padded_rows(b2, ctx, dtype, n):
    """Rows on 16-byte boundaries that end inside a pack or behind one, in every row segment length of the kernel (8, 16, 32
    and 128 packs): the last tile cut by both edges, by one, by none; the padding keeps its NaN."""
    lda = (n + 4) // 4 * 4
    for m in (1, 129, 300):
        a = synth.matrix_np(3, m, m, n, lda, dtype)
        a[:, n:] = np.nan
        x, y = synth.vector_np(5, m, m, dtype), synth.vector_np(6, n, n, dtype)
        ga, gx, gy = Guarded(a.ravel()), Guarded(x), Guarded(place(y, -2))
        b2.ger(ctx, orc.ROW_MAJOR, m, n, 0.75, gx.t, 1, gy.t, -2, ga.t, lda)
        oa = a.ravel().copy()
        absterms = orc.ger(orc.ROW_MAJOR, m, n, dtype(0.75), x, 1, place(y, -2), -2, oa, lda)
        got = ga.host().reshape(m, lda)
        assert_close(got[:, :n], oa.reshape(m, lda)[:, :n], absterms, dtype, f"ger m={m}")
        assert np.isnan(got[:, n:]).all()
        ga.check_guards()


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("mode", [0, 2, 3])
def test_cluster_gather_kernel(b2, ctx, dtype, mode):
    """The one-launch kernel at its edges: one output more and less than a cluster owns, one element more and less
    than a chunk of the row part (256 / 128 columns) and a batch of the column part (128 rows), every residue of the
    rows' starts; mode 3 sends every output of trmv through the workspace first, mode 0 keeps these sizes on the tile
    kernels."""
    old = b2.get_tuning(b2.KNOB_GATHER)
    b2.set_tuning(b2.KNOB_GATHER, mode)
    try:
        for n, pad, off in ((1, 0, 0), (31, 0, 0), (32, 1, 0), (33, 0, 1), (127, 2, 0), (129, 0, 0), (255, 0, 0), (257, 3, 1), (512, 0, 0), (1030, 1, 0)):
            lda, inc = n + pad, -2 if pad else 1
            x, y = synth.vector_np(7, n, n, dtype), synth.vector_np(8, n, n, dtype)
            for uplo, trans in itertools.product(UPLOS, TRANSES):
                diag = orc.UNIT if n % 2 else orc.NON_UNIT
                a = tri_buf(12, n, lda, dtype, orc.ROW_MAJOR, uplo, diag)
                ga, gx = Guarded(a, off), Guarded(place(x, inc))
                b2.trmv(ctx, orc.ROW_MAJOR, uplo, trans, diag, n, ga.t, lda, gx.t, inc)
                ox = place(x, inc)
                absterms = orc.trmv(orc.ROW_MAJOR, uplo, trans, diag, n, a, lda, ox, inc)
                assert_close(pick(gx.host(), n, inc), pick(ox, n, inc), absterms, dtype, f"trmv {n} {pad} {uplo} {trans}")
                gx.check_guards()
            if mode == 3:
                continue
            for uplo in UPLOS:
                a = tri_buf(9, n, lda, dtype, orc.ROW_MAJOR, uplo, orc.NON_UNIT)
                ga, gx, gy = Guarded(a, off), Guarded(place(x, inc)), Guarded(place(y, 1))
                b2.symv(ctx, orc.ROW_MAJOR, uplo, n, 1.25, ga.t, lda, gx.t, inc, 0.5, gy.t, 1)
                oy = y.copy()
                absterms = orc.symv(orc.ROW_MAJOR, uplo, n, dtype(1.25), a, lda, place(x, inc), inc, dtype(0.5), oy, 1)
                assert_close(gy.host(), oy, absterms, dtype, f"symv {n} {pad} {uplo}")
                gy.check_guards()
            for m, trans in itertools.product((n + 1, 200), TRANSES):
                a = synth.matrix_np(3, m, m, n, lda, dtype).ravel()
                lx, ly = (n, m) if trans == orc.NO_TRANS else (m, n)
                vx, vy = synth.vector_np(5, lx, lx, dtype), np.full(ly, np.nan, dtype=dtype)
                ga, gx, gy = Guarded(a, off), Guarded(place(vx, inc)), Guarded(vy)
                b2.gemv(ctx, orc.ROW_MAJOR, trans, m, n, 1.25, ga.t, lda, gx.t, inc, 0.0, gy.t, 1)
                oy = vy.copy()
                absterms = orc.gemv(orc.ROW_MAJOR, trans, m, n, dtype(1.25), a, lda, place(vx, inc), inc, dtype(0.0), oy, 1)
                assert_close(gy.host(), oy, absterms, dtype, f"gemv {m} {n} {pad} {trans}")
                gy.check_guards()
    finally:
        b2.set_tuning(b2.KNOB_GATHER, old)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("n,pad", [(63, 1), (130, 2), (513, 3), (516, 0), (641, 7), (1090, 2), (1151, 1), (1153, 0)])
@pytest.mark.parametrize("rows", [512, 0])
def test_cut_longest_column_tile(b2, ctx, dtype, n, pad, rows):
    """The tile kernels' column sums where the last column tile of an upper triangle (64 or 128 columns, the longest
    of them) is cut by the matrix edge: on a pack boundary, inside a pack, with one column and with all but one, in
    blocks of 512 rows that lie above the diagonal whole, in part and not at all, and of as many as the size asks for
    (one step of 64); rows on and off 16-byte boundaries."""
    old = b2.get_tuning(b2.KNOB_GATHER), b2.get_tuning(b2.KNOB_TRI_TILE), b2.get_tuning(b2.KNOB_TRI_ROWS)
    b2.set_tuning(b2.KNOB_GATHER, 0)
    b2.set_tuning(b2.KNOB_TRI_TILE, 0)
    b2.set_tuning(b2.KNOB_TRI_ROWS, rows)
    try:
        for lda, diag, inc in ((n + pad, orc.NON_UNIT, 1), ((n + 7) // 4 * 4, orc.UNIT, 2)):
            x, y = synth.vector_np(7, n, n, dtype), synth.vector_np(8, n, n, dtype)
            a = tri_buf(12, n, lda, dtype, orc.ROW_MAJOR, orc.UPPER, diag)
            ga, gx = Guarded(a), Guarded(place(x, inc))
            b2.trmv(ctx, orc.ROW_MAJOR, orc.UPPER, orc.TRANS, diag, n, ga.t, lda, gx.t, inc)
            ox = place(x, inc)
            absterms = orc.trmv(orc.ROW_MAJOR, orc.UPPER, orc.TRANS, diag, n, a, lda, ox, inc)
            assert_close(pick(gx.host(), n, inc), pick(ox, n, inc), absterms, dtype, f"trmv lda={lda}")
            gx.check_guards()
            for uplo, off in itertools.product(UPLOS, (0, 1)):  # (off 16-byte boundaries a lower triangle's first tile is cut too)
                a = tri_buf(9, n, lda, dtype, orc.ROW_MAJOR, uplo, orc.NON_UNIT)
                ga, gx, gy = Guarded(a, off), Guarded(place(x, inc)), Guarded(y)
                b2.symv(ctx, orc.ROW_MAJOR, uplo, n, 1.25, ga.t, lda, gx.t, inc, 0.5, gy.t, 1)
                oy = y.copy()
                absterms = orc.symv(orc.ROW_MAJOR, uplo, n, dtype(1.25), a, lda, place(x, inc), inc, dtype(0.5), oy, 1)
                assert_close(gy.host(), oy, absterms, dtype, f"symv lda={lda} {uplo} off={off}")
                gy.check_guards()
    finally:
        b2.set_tuning(b2.KNOB_GATHER, old[0])
        b2.set_tuning(b2.KNOB_TRI_TILE, old[1])
        b2.set_tuning(b2.KNOB_TRI_ROWS, old[2])


# Geometries of the cluster trsv kernel: type, value of the knob that cuts float into block rows of 64, unknowns of a block row.
TRSV_ROWS = [(np.float32, 0, 128), (np.float32, 1 << 30, 64), (np.float64, -1, 64)]


def trsv_near(dtype, nb, aligned):
    """Rows behind the front whose tiles the solving cluster multiplies itself (off 16-byte boundaries: of 15 block rows at most)."""
    return (6 if nb == 128 else 8) if aligned else (3 if nb == 128 else 4)


@pytest.fixture
def trsv_rows(b2, rows):
    """The knob that cuts float into block rows of 64 at the value of the test's parameter `rows`."""
    old = b2.get_tuning(b2.KNOB_TRSV_SHORT_ROWS)
    b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, rows)
    yield
    b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, old)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("streams", [-1, 1, 0])
def test_trsv_cluster_kernel(b2, ctx, dtype, streams):
    """The cluster kernel at its edges: one unknown more and less than a block row, than the rows the solving
    cluster multiplies itself, than one turn of the cluster; more strips than streaming blocks; with all
    streaming clusters, with one, and with none (the solving cluster then does their work)."""
    nb, near, cs = (128, 4, 16) if dtype == np.float32 else (64, 6, 16)
    sizes = [1, nb, nb + 1, (near + 1) * nb, (near + 1) * nb + 1, cs * nb - 1, cs * nb + 3]
    if streams != 0:
        sizes += [(cs + near + 2) * nb + 5] if streams == 1 else [(2 * cs + 7) * nb + 5, 70 * nb]
    old = b2.get_tuning(b2.KNOB_TRSV_STREAMS)
    b2.set_tuning(b2.KNOB_TRSV_STREAMS, streams)
    try:
        for n, pad in itertools.product(sizes, (0, 1)):
            for uplo, trans in itertools.product(UPLOS, TRANSES):
                diag = orc.UNIT if n % 2 else orc.NON_UNIT
                a = tri_buf(22, n, n + pad, dtype, orc.ROW_MAJOR, uplo, diag)
                hx = place(synth.vector_np(9, n, n, dtype), -2 if pad else 1)
                ga, gx = Guarded(a), Guarded(hx)
                b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, diag, n, ga.t, n + pad, gx.t, -2 if pad else 1)
                assert ctx.device_status() == 0
                rx = gx.host()
                gx.check_guards()
                inc = -2 if pad else 1
                resid, scale = orc.trsv_residual(orc.ROW_MAJOR, uplo, trans, diag, n, a, n + pad, hx, inc, rx, inc)
                assert np.all(resid <= TOL[np.dtype(dtype)] * scale), (n, pad, uplo, trans, np.max(resid / scale))
    finally:
        b2.set_tuning(b2.KNOB_TRSV_STREAMS, old)


@pytest.mark.parametrize("dtype,rows,nb", TRSV_ROWS)
@pytest.mark.parametrize("streams", [-1, 1, 0])
def test_trsv_cluster_kernel_in_rows(b2, ctx, dtype, rows, nb, streams, trsv_rows):
    """The cluster kernel at its edges, in rows of 128 and of 64: one unknown more and less than a block row, than the rows the solving
    cluster multiplies itself, than one turn of the cluster; more strips than streaming blocks; with all
    streaming clusters, with one, and with none (the solving cluster then does their work)."""
    cs, old = 16, b2.get_tuning(b2.KNOB_TRSV_STREAMS)
    b2.set_tuning(b2.KNOB_TRSV_STREAMS, streams)
    try:
        for aligned in (True, False):
            near = trsv_near(dtype, nb, aligned)
            sizes = [1, nb, nb + 1, (near + 1) * nb, (near + 1) * nb + 1, cs * nb - 1, cs * nb + 3]
            if streams != 0:
                sizes += [(cs + near + 2) * nb + 5]
            for n, uplo, trans in itertools.product(sizes, UPLOS, TRANSES):
                lda, inc = ((n + 3) // 4 * 4, 1) if aligned else (n | 1, -2)
                diag = orc.UNIT if n % 2 else orc.NON_UNIT
                a = tri_buf(22, n, lda, dtype, orc.ROW_MAJOR, uplo, diag)
                hx = place(synth.vector_np(9, n, n, dtype), inc)
                ga, gx = Guarded(a), Guarded(hx)
                b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, diag, n, ga.t, lda, gx.t, inc)
                assert ctx.device_status() == 0
                rx = gx.host()
                gx.check_guards()
                resid, scale = orc.trsv_residual(orc.ROW_MAJOR, uplo, trans, diag, n, a, lda, hx, inc, rx, inc)
                assert np.all(resid <= TOL[np.dtype(dtype)] * scale), (n, aligned, uplo, trans, np.max(resid / scale))
    finally:
        b2.set_tuning(b2.KNOB_TRSV_STREAMS, old)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("streams", [-1, 1])
def test_trsv_cluster_last_tiles(b2, ctx, dtype, streams):
    """Solves whose strips end with the first and with the second tile of a pair (the streaming blocks take tiles in
    pairs), whole and ragged, on and off 16-byte boundaries (one near row fewer in float); with one strip for each streaming
    block and, on one cluster of them, with several."""
    nb, near = (128, 4) if dtype == np.float32 else (64, 6)
    old = b2.get_tuning(b2.KNOB_TRSV_STREAMS)
    b2.set_tuning(b2.KNOB_TRSV_STREAMS, streams)
    try:
        for n, pad in [((near + 2) * nb - 4, 0), ((near + 3) * nb, 0), ((near + 4) * nb + 4, 4), (near * nb + 1, 0), ((near + 3) * nb - 1, 2),
                       ((near + 9) * nb, 0), ((near + 10) * nb + 4, 0)]:
            for uplo, trans in itertools.product(UPLOS, TRANSES):
                a = tri_buf(23, n, n + pad, dtype, orc.COL_MAJOR, uplo, orc.NON_UNIT)
                hx = synth.vector_np(9, n, n, dtype)
                ga, gx = Guarded(a), Guarded(hx)
                b2.trsv(ctx, orc.COL_MAJOR, uplo, trans, orc.NON_UNIT, n, ga.t, n + pad, gx.t, 1)
                assert ctx.device_status() == 0
                resid, scale = orc.trsv_residual(orc.COL_MAJOR, uplo, trans, orc.NON_UNIT, n, a, n + pad, hx, 1, gx.host(), 1)
                gx.check_guards()
                assert np.all(resid <= TOL[np.dtype(dtype)] * scale), (n, pad, uplo, trans, np.max(resid / scale))
    finally:
        b2.set_tuning(b2.KNOB_TRSV_STREAMS, old)


@pytest.mark.parametrize("dtype,rows,nb", TRSV_ROWS)
@pytest.mark.parametrize("streams", [-1, 1])
def test_trsv_cluster_last_tiles_in_rows(b2, ctx, dtype, rows, nb, streams, trsv_rows):
    """Solves whose strips end with the first and with the second tile of a pair (the streaming blocks take tiles in
    pairs), whole and ragged, on and off 16-byte boundaries (fewer near rows there); with one strip for each streaming
    block and, on one cluster of them, with several."""
    old = b2.get_tuning(b2.KNOB_TRSV_STREAMS)
    b2.set_tuning(b2.KNOB_TRSV_STREAMS, streams)
    try:
        for aligned in (True, False):
            near = trsv_near(dtype, nb, aligned)
            for n, uplo, trans in itertools.product([(near + 2) * nb - 4, (near + 3) * nb, (near + 4) * nb + 4, near * nb + 1, (near + 3) * nb - 1, (near + 9) * nb,
                                                     (near + 10) * nb + 4], UPLOS, TRANSES):
                lda = (n + 3) // 4 * 4 if aligned else n | 1
                a = tri_buf(23, n, lda, dtype, orc.COL_MAJOR, uplo, orc.NON_UNIT)
                hx = synth.vector_np(9, n, n, dtype)
                ga, gx = Guarded(a), Guarded(hx)
                b2.trsv(ctx, orc.COL_MAJOR, uplo, trans, orc.NON_UNIT, n, ga.t, lda, gx.t, 1)
                assert ctx.device_status() == 0
                resid, scale = orc.trsv_residual(orc.COL_MAJOR, uplo, trans, orc.NON_UNIT, n, a, lda, hx, 1, gx.host(), 1)
                gx.check_guards()
                assert np.all(resid <= TOL[np.dtype(dtype)] * scale), (n, aligned, uplo, trans, np.max(resid / scale))
    finally:
        b2.set_tuning(b2.KNOB_TRSV_STREAMS, old)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("n", [1, 3, 4, 31, 33, 129, 240, 241, 255, 256, 257, 416, 417, 511, 512])
def test_trmv_one_launch_rows(b2, ctx, dtype, n):
    """Row sums of small triangles in place and in one launch: one row more and less than a warp, a cluster of 8 and one of 16 has, and
    the sizes at which the tile kernel takes over; on and off 16-byte boundaries, strided, both triangles and diagonals."""
    old = b2.get_tuning(b2.KNOB_GATHER)
    try:
        for knob, pad, inc, diag in [(1, 0, 1, orc.NON_UNIT), (1, 1, -2, orc.UNIT), (2, -n % 16, 3, orc.UNIT), (2, 3, 1, orc.NON_UNIT)]:
            b2.set_tuning(b2.KNOB_GATHER, knob)
            for uplo in UPLOS:
                a = tri_buf(28, n, n + pad, dtype, orc.ROW_MAJOR, uplo, diag)
                hx = place(synth.vector_np(9, n, n, dtype), inc)
                ga, gx = Guarded(a), Guarded(hx)
                b2.trmv(ctx, orc.ROW_MAJOR, uplo, orc.NO_TRANS, diag, n, ga.t, n + pad, gx.t, inc)
                ox = hx.copy()
                absterms = orc.trmv(orc.ROW_MAJOR, uplo, orc.NO_TRANS, diag, n, a, n + pad, ox, inc)
                rx = gx.host()
                assert_close(pick(rx, n, inc), pick(ox, n, inc), absterms, dtype, f"trmv {n} {uplo} {pad}")
                assert_same_gaps(rx, hx, n, inc)
                gx.check_guards()
    finally:
        b2.set_tuning(b2.KNOB_GATHER, old)


@pytest.mark.parametrize("dtype,rows,room", [(np.float32, 0, True), (np.float32, 1 << 30, True), (np.float32, 1 << 30, False), (np.float64, -1, False)])
def test_trsv_cluster_block_rows(b2, dtype, rows, room):
    """Float in block rows of 128 where it would take 64 and the other way round; block rows of 64 with a workspace that holds the
    inverses beyond one turn of the cluster and no premultiplied tiles.  One unknown more and less than a block row, than the
    rows the solving cluster multiplies itself, than a turn; several strips for a streaming block."""
    nb = 128 if rows == 0 else 64
    sizes = [(21 * nb - 7) // 4 * 4, 22 * nb + 1] if not room else [nb - 1, nb + 4, 7 * nb, 9 * nb + 1, 17 * nb + 4, 45 * nb - 3]
    ws = None
    if not room:  # control block, x and far sums, flags, inverses
        s = np.dtype(dtype).itemsize
        ws = 4096 + 2 * 23 * nb * 2 * s + 512 + 7 * nb * nb * s
    c = b2.Context() if ws is None else b2.Context(workspace_bytes=ws)
    c.reset()
    old = b2.get_tuning(b2.KNOB_TRSV_SHORT_ROWS)
    b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, rows)
    try:
        for n, order, trans, uplo in itertools.product(sizes, ORDERS, TRANSES, UPLOS):
            a = tri_buf(27, n, n, dtype, order, uplo, orc.NON_UNIT)
            hx = synth.vector_np(9, n, n, dtype)
            ga, gx = Guarded(a), Guarded(hx)
            b2.trsv(c, order, uplo, trans, orc.NON_UNIT, n, ga.t, n, gx.t, 1)
            assert c.device_status() == 0
            resid, scale = orc.trsv_residual(order, uplo, trans, orc.NON_UNIT, n, a, n, hx, 1, gx.host(), 1)
            gx.check_guards()
            assert np.all(resid <= TOL[np.dtype(dtype)] * scale), (n, order, uplo, trans, np.max(resid / scale))
    finally:
        b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, old)


@pytest.mark.parametrize("dtype", DTYPES)
def test_trsv_premultiplied_tile_overflows(b2, ctx, dtype):
    """Tiles beside the diagonal whose products with the block's inverse are beyond the type, in the cluster's first turn and
    after it, times unknowns that are zero: the solution is the right-hand side over the diagonal and exact."""
    small, big = (-60, 90) if dtype == np.float32 else (-600, 500)
    n = 18 * 64 + 8
    m = np.diag(np.full(n, 2.0 ** small, dtype=dtype))
    b = synth.vector_np(3, 1, n, dtype)
    for k in (1, 17):  # tile (k, k - 1), and zeros for the unknowns it meets
        m[k * 64:(k + 1) * 64, (k - 1) * 64:k * 64] = 2.0 ** big
        b[(k - 1) * 64:k * 64] = 0
    want = b / dtype(2.0 ** small)
    for flip, order, trans in itertools.product((False, True), ORDERS, TRANSES):  # op(A) lower, upper
        op = m[::-1, ::-1] if flip else m
        stored = op if (order == orc.ROW_MAJOR) == (trans == orc.NO_TRANS) else op.T
        uplo = orc.UPPER if flip != (trans == orc.TRANS) else orc.LOWER
        da = torch.from_numpy(np.ascontiguousarray(stored).ravel()).cuda()
        x = torch.from_numpy(b[::-1].copy() if flip else b.copy()).cuda()
        # (blocks of 64 from the other end: whole when the order is turned round)
        if flip:
            da, x, length = da.view(n, n)[8:, 8:].reshape(-1).contiguous(), x[8:].contiguous(), n - 8
        else:
            length = n
        b2.trsv(ctx, order, uplo, trans, orc.NON_UNIT, length, da, length, x, 1)
        assert ctx.device_status() == 0
        expect = want[::-1][8:] if flip else want
        assert np.array_equal(x.cpu().numpy(), expect), (flip, order, trans)


@pytest.mark.parametrize("dtype,rows,nb", TRSV_ROWS)
@pytest.mark.parametrize("block,length", [(0, 0), (1, 0), (4, 0), (18, 30)])
def test_trsv_infinite_right_hand_side(b2, ctx, dtype, rows, nb, block, length):
    """An infinite element of the right-hand side in every place of a block row: that unknown is infinite, the block rows before it are
    what they are without it, bit for bit, and what follows it is not finite.  In the first rows, in one with sums of rows further
    back and in the ragged last one."""
    n, length = 18 * nb + 30, length or nb
    x = torch.from_numpy(synth.vector_np(9, n, n, dtype)).cuda()
    old = b2.get_tuning(b2.KNOB_TRSV_SHORT_ROWS)
    b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, rows)
    try:
        for uplo, trans in itertools.product(UPLOS, TRANSES):
            upper = (uplo == orc.UPPER) == (trans == orc.NO_TRANS)  # of op(A): solved from the last row on
            a = tri_buf(24, n, n, dtype, orc.ROW_MAJOR, uplo, orc.NON_UNIT)
            da, signs = torch.from_numpy(a).cuda(), np.sign(a.reshape(n, n).diagonal())

            def solve(v):
                b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, da, n, v, 1)
                assert ctx.device_status() == 0
                return v.cpu().numpy()
            whole = solve(x.clone())
            before = slice(min(n, (block + 1) * nb), n) if upper else slice(0, block * nb)
            for q in range(length):
                i = block * nb + (length - 1 - q if upper else q)
                v = x.clone()
                v[i] = np.inf if q % 2 else -np.inf
                want, got = float(v[i]) * signs[i], solve(v)
                assert got[i] == want, (q, uplo, trans, got[i])
                assert np.array_equal(got[before], whole[before]), (q, uplo, trans)
                assert not np.any(np.isfinite(got[:i] if upper else got[i + 1:])), (q, uplo, trans)
    finally:
        b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, old)


def _solve_turned(b2, ctx, m, b, want):
    """op(A) = m in blocks of 64 and one of 8, lower triangular, and turned round, in both orders and stored either way; the last block does
    not count when it is turned, so that the blocks of 64 are whole from the other end."""
    n = len(b)
    for flip, order, trans in itertools.product((False, True), ORDERS, TRANSES):
        op, rhs, expect = (v[::-1][8:] if flip else v for v in (m[:, ::-1] if flip else m, b, want))
        if flip:
            op = op[:, 8:]
        stored = op if (order == orc.ROW_MAJOR) == (trans == orc.NO_TRANS) else op.T
        uplo = orc.UPPER if flip != (trans == orc.TRANS) else orc.LOWER
        length = len(rhs)
        da = torch.from_numpy(np.ascontiguousarray(stored).ravel()).cuda()
        x = torch.from_numpy(rhs.copy()).cuda()
        b2.trsv(ctx, order, uplo, trans, orc.NON_UNIT, length, da, length, x, 1)
        assert ctx.device_status() == 0
        assert np.array_equal(x.cpu().numpy(), expect), (flip, order, trans)


@pytest.mark.parametrize("dtype", DTYPES)
def test_trsv_premultiplied_tile_overflows_in_row_4(b2, ctx, dtype):
    """The same in a row of the cluster's first turn whose tile is premultiplied (those of rows 1 and 2 are not)."""
    small, big = (-60, 90) if dtype == np.float32 else (-600, 500)
    n = 18 * 64 + 8
    m, b = np.diag(np.full(n, 2.0 ** small, dtype=dtype)), synth.vector_np(3, 1, n, dtype)
    m[256:320, 192:256], b[192:256] = 2.0 ** big, 0
    _solve_turned(b2, ctx, m, b, b / dtype(2.0 ** small))


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("rest", [0.0, 2.0])
def test_trsv_premultiplied_tile_underflows(b2, ctx, dtype, rest):
    """Tiles beside the diagonal whose products with the block's inverse are below the type, times large unknowns, in the cluster's
    first turn and after it; in double also products that vanish beside others that do not.  Powers of two: exact."""
    diag, tile, size = (84, -66, 100) if dtype == np.float32 else (600, -500, 600)
    n = 18 * 64 + 8
    m, b = np.eye(n, dtype=dtype), np.ones(n, dtype=dtype)
    want = b.copy()
    for k in (1, 4, 17):
        here, before = slice(k * 64, (k + 1) * 64), slice((k - 1) * 64, k * 64)
        m[here, here] *= dtype(2.0 ** diag)
        m[here, before] = np.diag(np.full(64, 2.0 ** tile))
        b[before] = want[before] = 2.0 ** size
        b[here], want[here] = 0, -2.0 ** (tile + size - diag)
        if rest:  # the first column beside them: a product of ordinary size with an unknown that is small
            m[here, before][:, 0] = 2.0 ** diag * rest
            b[(k - 1) * 64] = want[(k - 1) * 64] = 2.0 ** (tile + size - diag)
            want[here] *= 3
            want[k * 64] = -2.0 ** (tile + size - diag) * rest
    _solve_turned(b2, ctx, m, b, want)


@pytest.mark.parametrize("dtype,rows,nb", TRSV_ROWS[1:])
@pytest.mark.parametrize("block,length", [(0, 64), (1, 64), (4, 64), (7, 30)])
def test_trsv_infinite_element_and_its_block_row(b2, ctx, dtype, rows, nb, block, length):
    """In rows of 64 the unknowns of the same block row that precede an infinite element of the right-hand side do not depend on it
    either."""
    n = 7 * nb + 30
    old = b2.get_tuning(b2.KNOB_TRSV_SHORT_ROWS)
    b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, rows)
    try:
        for uplo, trans, q in itertools.product(UPLOS, TRANSES, (1, 18, length - 1)):
            upper = (uplo == orc.UPPER) == (trans == orc.NO_TRANS)  # of op(A): solved from the last row on
            a, hx = tri_buf(24, n, n, dtype, orc.ROW_MAJOR, uplo, orc.NON_UNIT), synth.vector_np(9, n, n, dtype)
            i = block * nb + (length - 1 - q if upper else q)
            hx[i] = np.inf
            ga, gx = Guarded(a), Guarded(hx)
            b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, ga.t, n, gx.t, 1)
            assert ctx.device_status() == 0
            got = gx.host()
            gx.check_guards()
            assert got[i] == np.inf * np.sign(a.reshape(n, n)[i, i]), (q, uplo, trans, got[i])
            resid, scale = orc.trsv_residual(orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, a, n, hx, 1, got, 1)
            before = slice(i + 1, n) if upper else slice(0, i)
            assert np.all(resid[before] <= TOL[np.dtype(dtype)] * scale[before]), (q, uplo, trans)
    finally:
        b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, old)


@pytest.mark.parametrize("dtype", DTYPES)
def test_trsv_product_beyond_the_type(b2, ctx, dtype):
    """Right-hand sides and tiles whose products with the block's inverse are beyond the type, while the right-hand side less the tile's
    product with the unknowns before is not.  Powers of two: exact."""
    diag, size, rest = (-100, 33, 12) if dtype == np.float32 else (-750, 300, 250)
    n = 18 * 64 + 8
    m, b = np.eye(n, dtype=dtype), np.ones(n, dtype=dtype)
    want = b.copy()
    for k in (1, 4, 17):
        here, before = slice(k * 64, (k + 1) * 64), slice((k - 1) * 64, k * 64)
        m[here, here] *= dtype(2.0 ** diag)
        m[here, before] = np.eye(64)
        b[before] = want[before] = 2.0 ** size
        b[here], want[here] = 2.0 ** size + 2.0 ** rest, 2.0 ** (rest - diag)
    _solve_turned(b2, ctx, m, b, want)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("at", [0, 70, 300])
def test_trsv_solution_overflows(b2, ctx, dtype, at):
    """A solution beyond the type from one unknown on, with a matrix and a right-hand side that make all later ones infinite of the same
    sign by substitution: so they are in its block row and the next, and nowhere finite."""
    n = 18 * 64 + 30
    big = np.finfo(dtype).maxexp - 4
    for pad in (0, 1):
        m = np.full((n, n), -1.0 / n, dtype=dtype)
        m[np.diag_indices(n)] = 1
        b = np.ones(n, dtype=dtype)
        m[at, at], b[at] = 2.0 ** -big, 2.0 ** 40
        for uplo, trans in ((orc.LOWER, orc.NO_TRANS), (orc.UPPER, orc.TRANS)):
            buf = np.zeros((n, n + pad), dtype=dtype)
            buf[:, :n] = m if trans == orc.NO_TRANS else m.T
            ga, gx = Guarded(buf), Guarded(b)
            b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, ga.t, n + pad, gx.t, 1)
            assert ctx.device_status() == 0
            got = gx.host()
            assert np.all(np.isfinite(got[:at])) and not np.any(np.isfinite(got[at:])), (pad, uplo, trans)
            assert np.all(got[at:(at // 64 + 2) * 64] == np.inf), (pad, uplo, trans, np.flatnonzero(got[at:] != np.inf)[:4])


def test_trsv_small_workspace_takes_longer_rows(b2):
    """Float with the smallest workspace, where the inverses of block rows of 64 do not fit and rows of 128 need none: these, bit for bit."""
    small = b2.Context(workspace_bytes=b2.lib().b2_workspace_min_bytes())
    small.reset()
    old = b2.get_tuning(b2.KNOB_TRSV_SHORT_ROWS)
    for n, pad in [(1412, 0), (1601, 2), (2048, 0), (2047, 0)]:
        for uplo, trans in itertools.product(UPLOS, TRANSES):
            ga = Guarded(tri_buf(29, n, n + pad, np.float32, orc.ROW_MAJOR, uplo, orc.NON_UNIT))
            hx, got = synth.vector_np(9, n, n, np.float32), []
            for rows in (old, 0):
                b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, rows)
                try:
                    gx = Guarded(hx)
                    b2.trsv(small, orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, ga.t, n + pad, gx.t, 1)
                finally:
                    b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, old)
                assert small.device_status() == 0
                gx.check_guards()
                got.append(gx.host())
            assert np.array_equal(*got), (n, pad, uplo, trans)


@pytest.mark.parametrize("n,room,unit", [(6000, 320 << 10, 4), (2304, 230 << 10, 4), (6500, 0, 2)])
def test_ring_units(b2, ctx, n, room, unit):
    """trmv's float row sums with a strided x and symv on the ring kernel, bit for bit as with units of so many tiles: with a workspace that
    holds the partials of units of four only, and on rows off 32-byte boundaries."""
    c = b2.Context(workspace_bytes=4096 + room) if room else ctx
    c.reset()
    old = b2.get_tuning(b2.KNOB_TRI_TILE_UNIT)
    for uplo in UPLOS:
        ga = Guarded(tri_buf(26, n, n, np.float32, orc.ROW_MAJOR, uplo, orc.NON_UNIT))
        x, y, got = place(synth.vector_np(7, n, n, np.float32), 2), synth.vector_np(8, n, n, np.float32), []
        for where, asked in ((c, 0), (ctx, unit)):
            b2.set_tuning(b2.KNOB_TRI_TILE_UNIT, asked)
            try:
                gx, gy = Guarded(x), Guarded(y)
                if n == 2304:
                    b2.symv(where, orc.ROW_MAJOR, uplo, n, 1.25, ga.t, n, gx.t, 2, 0.5, gy.t, 1)
                else:
                    b2.trmv(where, orc.ROW_MAJOR, uplo, orc.NO_TRANS, orc.NON_UNIT, n, ga.t, n, gx.t, 2)
            finally:
                b2.set_tuning(b2.KNOB_TRI_TILE_UNIT, old)
            gx.check_guards(), gy.check_guards()
            got += [gx.host(), gy.host()]
        assert np.array_equal(got[0], got[2], equal_nan=True) and np.array_equal(got[1], got[3]), uplo


@pytest.mark.parametrize("dtype,rows,nb", TRSV_ROWS[1:])
def test_trsv_premultiplied_last_rows(b2, ctx, dtype, rows, nb):
    """Off 16-byte boundaries only the last block rows' tiles are premultiplied: one more block row than beyond the first turn and those,
    and several; ragged, from either end."""
    old = b2.get_tuning(b2.KNOB_TRSV_SHORT_ROWS)
    b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, rows)
    try:
        for n, uplo, trans in [(73 * nb - 1, orc.LOWER, orc.NO_TRANS), (76 * nb + 5, orc.LOWER, orc.TRANS)]:
            a = tri_buf(30, n, n | 1, dtype, orc.ROW_MAJOR, uplo, orc.NON_UNIT)
            hx = synth.vector_np(9, n, n, dtype)
            ga, gx = Guarded(a), Guarded(hx)
            b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, ga.t, n | 1, gx.t, 1)
            assert ctx.device_status() == 0
            resid, scale = orc.trsv_residual(orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, a, n | 1, hx, 1, gx.host(), 1)
            gx.check_guards()
            assert np.all(resid <= TOL[np.dtype(dtype)] * scale), (n, uplo, trans, np.max(resid / scale))
    finally:
        b2.set_tuning(b2.KNOB_TRSV_SHORT_ROWS, old)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("extra", [0, 400 << 10])
def test_small_workspace_off_boundaries(b2, dtype, extra):
    """symv and trmv's column sums with the smallest workspace and with a little more, off 16-byte boundaries, at sizes where
    the tile kernels' partials would need more, up to the largest that the gather kernel takes; the next one is refused."""
    small = b2.Context(workspace_bytes=b2.lib().b2_workspace_min_bytes() + extra)
    small.reset()
    for n in (2401, 3001, 4001, 4601) if dtype == np.float32 else (2043, 2501, 3101):
        x, y = synth.vector_np(7, n, n, dtype), synth.vector_np(8, n, n, dtype)
        for uplo in UPLOS:
            a = tri_buf(26, n, n, dtype, orc.ROW_MAJOR, uplo, orc.NON_UNIT)
            ga, gx, gy = Guarded(a), Guarded(x), Guarded(y)
            b2.symv(small, orc.ROW_MAJOR, uplo, n, 1.25, ga.t, n, gx.t, 1, 0.5, gy.t, 1)
            oy = y.copy()
            absterms = orc.symv(orc.ROW_MAJOR, uplo, n, dtype(1.25), a, n, x, 1, dtype(0.5), oy, 1)
            assert_close(gy.host(), oy, absterms, dtype, f"symv {n} {uplo}")
            b2.trmv(small, orc.ROW_MAJOR, uplo, orc.TRANS, orc.NON_UNIT, n, ga.t, n, gx.t, 1)
            ox = x.copy()
            absterms = orc.trmv(orc.ROW_MAJOR, uplo, orc.TRANS, orc.NON_UNIT, n, a, n, ox, 1)
            assert_close(gx.host(), ox, absterms, dtype, f"trmv {n} {uplo}")
            gx.check_guards(), gy.check_guards()
    n = 4701 if dtype == np.float32 else 3201
    a, v = torch.zeros(n * n, dtype=torch.from_numpy(y).dtype, device="cuda"), torch.from_numpy(np.resize(y, n)).cuda()
    with pytest.raises(b2.B2Error) as e:
        b2.symv(small, orc.ROW_MAJOR, orc.UPPER, n, 1.25, a, n, v, 1, 0.5, v.clone(), 1)
    assert e.value.status == b2.STATUS_WORKSPACE_TOO_SMALL


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("n", [8, 77, 300])
@pytest.mark.parametrize("power", [0, 90, -90])
def test_trsv_divides_by_the_diagonal(b2, ctx, dtype, n, power):
    """Multiples of the diagonal below ones in every eighth row, right-hand side one there and else zero: the solution is the
    negated factors and exact, for each unknown is one quotient of whole numbers.  The product with a rounded reciprocal is
    not that quotient for many of the divisors (49 in double, 41 in float).  Scaled also by powers of two, in double beyond the
    range in which such a product is corrected."""
    scale = 2.0 ** (power if dtype == np.float32 else 4 * power)
    a = np.zeros((n, n), dtype=dtype)
    want = np.zeros(n, dtype=dtype)
    for i in range(n):
        one = i % 8 == 0
        a[i, i] = 1 if one else (2 * i + 27) * scale
        want[i] = 1 if one else -(i % 5)
        if not one:
            a[i, i - i % 8] = -want[i] * a[i, i]
    hx = np.where(np.arange(n) % 8 == 0, 1, 0).astype(dtype)
    for lda in (n + n % 2 * 3, n | 1):  # on and off 16-byte boundaries
        for uplo, trans, view in ((orc.LOWER, orc.NO_TRANS, a), (orc.UPPER, orc.TRANS, a.T)):
            buf = np.full((n, lda), np.nan, dtype=dtype)
            buf[:, :n] = view
            gm, gx = Guarded(buf), Guarded(hx)
            b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, gm.t, lda, gx.t, 1)
            assert ctx.device_status() == 0
            assert np.array_equal(gx.host(), want), (lda, uplo, trans)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_trsv_keeps_what_precedes_a_bad_element(b2, ctx, dtype, bad):
    """An infinite or NaN element of the matrix in a diagonal block: the unknowns that the solve reaches before it do not depend
    on it.  The element lies beside the diagonal, on it, and in the lower left part of a block of every level of the
    inversion; in a whole block, in one that the streaming blocks invert and in the ragged last one."""
    nb = 128 if dtype == np.float32 else 64
    n = 18 * nb + 44
    places = [(1, 0), (3, 1), (7, 0), (7, 6), (7, 7), (12, 3), (15, 2), (23, 16), (30, 9), (39, 37), (45, 45), (63, 1), (61, 35)]
    if nb == 128:
        places += [(76, 65), (99, 10), (100, 63), (127, 64), (127, 127)]
    for block, length, where in ((1, nb, places), (17, nb, places[3::4]), (18, 44, [(43, 40), (20, 3), (43, 43)])):
        for (row, col), uplo, trans in itertools.product(where, UPLOS, TRANSES):
            upper = (uplo == orc.UPPER) == (trans == orc.NO_TRANS)  # of op(A): solved from the last row on
            i, j = (block * nb + (length - 1 - q if upper else q) for q in (row, col))
            a = tri_buf(24, n, n, dtype, orc.ROW_MAJOR, uplo, orc.NON_UNIT)
            a.reshape(n, n)[(i, j) if trans == orc.NO_TRANS else (j, i)] = bad
            hx = synth.vector_np(9, n, n, dtype)
            ga, gx = Guarded(a), Guarded(hx)
            b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, ga.t, n, gx.t, 1)
            assert ctx.device_status() == 0
            resid, scale = orc.trsv_residual(orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, a, n, hx, 1, gx.host(), 1)
            before = slice(i + 1, n) if upper else slice(0, i)
            assert np.all(resid[before] <= TOL[np.dtype(dtype)] * scale[before]), (block, row, col, uplo, trans)


@pytest.mark.parametrize("dtype,rows,nb", TRSV_ROWS[1:2])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_trsv_keeps_what_precedes_a_bad_element_in_rows(b2, ctx, dtype, rows, nb, bad, trsv_rows):
    """An infinite or NaN element of the matrix in a diagonal block: the unknowns that the solve reaches before it do not depend
    on it.  The element lies beside the diagonal, on it, and in the lower left part of a block of every level of the
    inversion; in a whole block, in one that the streaming blocks invert and in the ragged last one."""
    n = 18 * nb + 44
    places = [(1, 0), (3, 1), (7, 0), (7, 6), (7, 7), (12, 3), (15, 2), (23, 16), (30, 9), (39, 37), (45, 45), (63, 1), (61, 35)]
    if nb == 128:
        places += [(76, 65), (99, 10), (100, 63), (127, 64), (127, 127)]
    for block, length, where in ((1, nb, places), (17, nb, places[3::4]), (18, 44, [(43, 40), (20, 3), (43, 43)])):
        for (row, col), uplo, trans in itertools.product(where, UPLOS, TRANSES):
            upper = (uplo == orc.UPPER) == (trans == orc.NO_TRANS)  # of op(A): solved from the last row on
            i, j = (block * nb + (length - 1 - q if upper else q) for q in (row, col))
            a = tri_buf(24, n, n, dtype, orc.ROW_MAJOR, uplo, orc.NON_UNIT)
            a.reshape(n, n)[(i, j) if trans == orc.NO_TRANS else (j, i)] = bad
            hx = synth.vector_np(9, n, n, dtype)
            ga, gx = Guarded(a), Guarded(hx)
            b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, ga.t, n, gx.t, 1)
            assert ctx.device_status() == 0
            resid, scale = orc.trsv_residual(orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, a, n, hx, 1, gx.host(), 1)
            before = slice(i + 1, n) if upper else slice(0, i)
            assert np.all(resid[before] <= TOL[np.dtype(dtype)] * scale[before]), (block, row, col, uplo, trans)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("streams", [-1, 1])
def test_trsv_first_cluster_overtaken(b2, ctx, dtype, streams):
    """The first cluster, whose blocks have staged their diagonal blocks by then, draws a ticket other than the first and
    streams: with fewer block rows than blocks in a cluster, with more, ragged, on and off 16-byte boundaries."""
    nb, near = (128, 4) if dtype == np.float32 else (64, 6)
    old = b2.get_tuning(b2.KNOB_TRSV_STREAMS)
    b2.set_tuning(b2.KNOB_TRSV_STREAMS, streams)
    b2.set_tuning(b2.KNOB_TRSV_DEBUG_LATE, 1 << 16)  # (polls; the other clusters draw their tickets within a hundred)
    try:
        for n, pad in [((near + 3) * nb, 0), ((near + 4) * nb + 1, 0), (18 * nb + 4, 0), (21 * nb + 3, 2)]:
            for uplo, trans in itertools.product(UPLOS, TRANSES):
                a = tri_buf(25, n, n + pad, dtype, orc.ROW_MAJOR, uplo, orc.NON_UNIT)
                hx = synth.vector_np(9, n, n, dtype)
                ga, gx = Guarded(a), Guarded(hx)
                b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, ga.t, n + pad, gx.t, 1)
                assert ctx.device_status() == 0
                gx.check_guards()
                resid, scale = orc.trsv_residual(orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, a, n + pad, hx, 1, gx.host(), 1)
                assert np.all(resid <= TOL[np.dtype(dtype)] * scale), (n, pad, uplo, trans, np.max(resid / scale))
    finally:
        b2.set_tuning(b2.KNOB_TRSV_STREAMS, old)
        b2.set_tuning(b2.KNOB_TRSV_DEBUG_LATE, 0)


@pytest.mark.parametrize("dtype,rows,nb", TRSV_ROWS[:2])
@pytest.mark.parametrize("streams", [-1, 1])
def test_trsv_first_cluster_overtaken_in_rows(b2, ctx, dtype, rows, nb, streams, trsv_rows):
    """The first cluster, whose blocks have staged their diagonal blocks by then, draws a ticket other than the first and
    streams: with fewer block rows than blocks in a cluster, with more, ragged, on and off 16-byte boundaries."""
    old = b2.get_tuning(b2.KNOB_TRSV_STREAMS)
    b2.set_tuning(b2.KNOB_TRSV_STREAMS, streams)
    b2.set_tuning(b2.KNOB_TRSV_DEBUG_LATE, 1 << 16)  # (polls; the other clusters draw their tickets within a hundred)
    try:
        for aligned in (True, False):
            near = trsv_near(dtype, nb, aligned)
            for n, uplo, trans in itertools.product([(near + 3) * nb, (near + 4) * nb + 1, 18 * nb + 4, 21 * nb + 3], UPLOS, TRANSES):
                lda = (n + 3) // 4 * 4 if aligned else n | 1
                a = tri_buf(25, n, lda, dtype, orc.ROW_MAJOR, uplo, orc.NON_UNIT)
                hx = synth.vector_np(9, n, n, dtype)
                ga, gx = Guarded(a), Guarded(hx)
                b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, ga.t, lda, gx.t, 1)
                assert ctx.device_status() == 0
                gx.check_guards()
                resid, scale = orc.trsv_residual(orc.ROW_MAJOR, uplo, trans, orc.NON_UNIT, n, a, lda, hx, 1, gx.host(), 1)
                assert np.all(resid <= TOL[np.dtype(dtype)] * scale), (n, aligned, uplo, trans, np.max(resid / scale))
    finally:
        b2.set_tuning(b2.KNOB_TRSV_STREAMS, old)
        b2.set_tuning(b2.KNOB_TRSV_DEBUG_LATE, 0)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("n,pad", [(1985, 0), (3440, 0), (3441, 0), (4130, 2), (5801, 0)])
def test_rows_per_block_by_size(b2, ctx, dtype, n, pad):
    """symv and trmv's column sums on the tile kernel in blocks of 64, 128 and more rows, off 16-byte boundaries up to
    the longest of 256, the last one cut."""
    old = b2.get_tuning(b2.KNOB_GATHER), b2.get_tuning(b2.KNOB_TRI_TILE)
    b2.set_tuning(b2.KNOB_GATHER, 0)
    b2.set_tuning(b2.KNOB_TRI_TILE, 0)
    try:
        lda, x, y = n + pad, synth.vector_np(7, n, n, dtype), synth.vector_np(8, n, n, dtype)
        for uplo in UPLOS:
            a = tri_buf(12, n, lda, dtype, orc.ROW_MAJOR, uplo, orc.NON_UNIT)
            ga, gx = Guarded(a), Guarded(x)
            b2.trmv(ctx, orc.ROW_MAJOR, uplo, orc.TRANS, orc.NON_UNIT, n, ga.t, lda, gx.t, 1)
            ox = x.copy()
            absterms = orc.trmv(orc.ROW_MAJOR, uplo, orc.TRANS, orc.NON_UNIT, n, a, lda, ox, 1)
            assert_close(gx.host(), ox, absterms, dtype, f"trmv {uplo}")
            gx, gy = Guarded(x), Guarded(y)
            b2.symv(ctx, orc.ROW_MAJOR, uplo, n, 1.25, ga.t, lda, gx.t, 1, 0.5, gy.t, 1)
            oy = y.copy()
            absterms = orc.symv(orc.ROW_MAJOR, uplo, n, dtype(1.25), a, lda, x, 1, dtype(0.5), oy, 1)
            assert_close(gy.host(), oy, absterms, dtype, f"symv {uplo}")
            gx.check_guards(), gy.check_guards()
    finally:
        b2.set_tuning(b2.KNOB_GATHER, old[0])
        b2.set_tuning(b2.KNOB_TRI_TILE, old[1])


@pytest.mark.parametrize("order", ORDERS)
@pytest.mark.parametrize("trans", TRANSES)
@pytest.mark.parametrize("m,n", [(1999, 2001), (2001, 2001), (1023, 4099), (1025, 3911), (31009, 129), (8009, 511), (7999, 513)])
def test_gemv_double_unaligned_steps(b2, ctx, order, trans, m, n):
    """gemv in double off 16-byte boundaries around the size from which a step of the tile kernel has four rows instead of two
    per thread, and where a block has a whole row and where it has not."""
    minor, major = (n, m) if order == orc.ROW_MAJOR else (m, n)
    lda = minor + 1 - minor % 2  # odd
    lenx, leny = (n, m) if trans == orc.NO_TRANS else (m, n)
    a = matbuf(m + n, major, minor, lda, np.float64)
    x, y = synth.vector_np(1, m + n, lenx, np.float64), synth.vector_np(2, m + n, leny, np.float64)
    ga, gx, gy = Guarded(a), Guarded(x), Guarded(y)
    old = b2.get_tuning(b2.KNOB_GATHER)
    b2.set_tuning(b2.KNOB_GATHER, 0)
    try:
        b2.gemv(ctx, order, trans, m, n, 1.25, ga.t, lda, gx.t, 1, 0.5, gy.t, 1)
    finally:
        b2.set_tuning(b2.KNOB_GATHER, old)
    oy = y.copy()
    absterms = orc.gemv(order, trans, m, n, 1.25, a, lda, x, 1, 0.5, oy, 1)
    assert_close(gy.host(), oy, absterms, np.float64, f"gemv {m} {n} {order} {trans}")
    gy.check_guards()


@pytest.mark.parametrize("dtype", DTYPES)
def test_small_integer_level2_is_bit_exact(b2, ctx, dtype):
    rng = np.random.default_rng(2)
    m, n = 300, 1100
    a = rng.integers(-2, 3, size=(m, n)).astype(dtype)
    x = rng.integers(-2, 3, size=n).astype(dtype)
    xm = rng.integers(-2, 3, size=m).astype(dtype)
    ga, gx, gxm = Guarded(a.ravel()), Guarded(x), Guarded(xm)
    gy = Guarded(np.zeros(m, dtype=dtype))
    b2.gemv(ctx, orc.ROW_MAJOR, orc.NO_TRANS, m, n, 2.0, ga.t, n, gx.t, 1, 0.0, gy.t, 1)
    assert np.array_equal(gy.host(), 2 * (a.astype(np.int64) @ x.astype(np.int64)).astype(dtype))
    gy = Guarded(np.zeros(n, dtype=dtype))
    b2.gemv(ctx, orc.ROW_MAJOR, orc.TRANS, m, n, 2.0, ga.t, n, gxm.t, 1, 0.0, gy.t, 1)
    assert np.array_equal(gy.host(), 2 * (a.astype(np.int64).T @ xm.astype(np.int64)).astype(dtype))
    k = 700
    t = rng.integers(-2, 3, size=(k, k)).astype(dtype)
    v = rng.integers(-2, 3, size=k).astype(dtype)
    gt = Guarded(t.ravel())
    for uplo, tri in [(orc.UPPER, np.triu(t)), (orc.LOWER, np.tril(t))]:
        for trans, diag in itertools.product(TRANSES, DIAGS):
            tt = tri.astype(np.int64)
            if diag == orc.UNIT:
                np.fill_diagonal(tt, 1)
            gv = Guarded(v)
            b2.trmv(ctx, orc.ROW_MAJOR, uplo, trans, diag, k, gt.t, k, gv.t, 1)
            assert np.array_equal(gv.host(), ((tt.T if trans == orc.TRANS else tt) @ v.astype(np.int64)).astype(dtype))
        symm = (tri + tri.T - np.diag(np.diag(t))).astype(np.int64)
        gv, gy = Guarded(v), Guarded(v.copy())
        b2.symv(ctx, orc.ROW_MAJOR, uplo, k, 1.0, gt.t, k, gv.t, 1, -1.0, gy.t, 1)
        assert np.array_equal(gy.host(), (symm @ v.astype(np.int64) - v.astype(np.int64)).astype(dtype))


@pytest.mark.parametrize("dtype", DTYPES)
def test_level2_determinism(b2, ctx, dtype):
    n = 900
    a = Guarded(synth.vector_np(1, 1, n * n, dtype))
    x = synth.vector_np(1, 2, n, dtype)
    outs = []
    for _ in range(3):
        gx, gy = Guarded(x), Guarded(np.zeros(n, dtype=dtype))
        b2.gemv(ctx, orc.ROW_MAJOR, orc.TRANS, n, n, 1.0, a.t, n, gx.t, 1, 0.0, gy.t, 1)
        b2.symv(ctx, orc.ROW_MAJOR, orc.UPPER, n, 1.0, a.t, n, gx.t, 1, 1.0, gy.t, 1)
        b2.trmv(ctx, orc.ROW_MAJOR, orc.LOWER, orc.TRANS, orc.NON_UNIT, n, a.t, n, gy.t, 1)
        outs.append(gy.host().copy())
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("kernel", [0, 2, 3])
def test_trsv_replayed_from_a_graph(b2, dtype, kernel):
    """A captured solve is replayed with other data in the same buffers: every replay gives the bits of a plain call.
    (Its values in the workspace carry the tag of the captured call every time.)"""
    old = b2.get_tuning(b2.KNOB_TRSV_FRONT)
    b2.set_tuning(b2.KNOB_TRSV_FRONT, kernel)
    try:
        for n in (131, 2435):
            ctx = b2.Context()
            ctx.reset()
            mats = [torch.from_numpy(tri_buf(s, n, n + 1, dtype, orc.ROW_MAJOR, orc.LOWER, orc.NON_UNIT)).cuda() for s in (21, 22, 23)]
            rhs = [torch.from_numpy(synth.vector_np(s, n, n, dtype)).cuda() for s in (5, 6, 7)]
            call = lambda c, a, x: b2.trsv(c, orc.ROW_MAJOR, orc.LOWER, orc.NO_TRANS, orc.NON_UNIT, n, a, n + 1, x, 1)
            want = []
            for a, b in zip(mats, rhs):
                want.append(b.clone())
                call(ctx, a, want[-1])
            a, x = mats[0].clone(), rhs[0].clone()
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                call(ctx, a, x)
                b2.scal(ctx, n, 1.0, x, 1)
            for k in (0, 1, 2, 2, 0):
                a.copy_(mats[k])
                x.copy_(rhs[k])
                graph.replay()
                torch.cuda.synchronize()
                assert ctx.device_status() == 0 and torch.equal(x, want[k]), (n, k)
            del graph
    finally:
        b2.set_tuning(b2.KNOB_TRSV_FRONT, old)


@pytest.mark.parametrize("dtype", DTYPES)
def test_workspace_query_keeps_the_kernels(b2, ctx, dtype):
    """With exactly b2_workspace_query bytes trsv and symv run on the kernels they run on with the default workspace:
    equal bits, which the kernels behind them do not give (their sums run in another order)."""
    s = np.dtype(dtype).itemsize

    def solve(c, n):
        gx = Guarded(synth.vector_np(9, n, n, dtype))
        b2.trsv(c, orc.ROW_MAJOR, orc.LOWER, orc.NO_TRANS, orc.NON_UNIT, n, tri.t, n, gx.t, 1)
        assert c.device_status() == 0
        return gx.host()

    def product(c, n):
        gx, gy = Guarded(synth.vector_np(9, n, n, dtype)), Guarded(np.zeros(n, dtype=dtype))
        b2.symv(c, orc.ROW_MAJOR, orc.UPPER, n, 1.25, sym.t, n, gx.t, 1, 0.0, gy.t, 1)
        return gy.host()

    for n in (300, 2100, 2432):
        tri = Guarded(tri_buf(21, n, n, dtype, orc.ROW_MAJOR, orc.LOWER, orc.NON_UNIT))
        sym = Guarded(tri_buf(9, n, n, dtype, orc.ROW_MAJOR, orc.UPPER, orc.NON_UNIT))
        small = b2.Context(workspace_bytes=b2.lib().b2_workspace_query(n, n, s))
        small.reset()
        for routine, knob, other in ((solve, b2.KNOB_TRSV_FRONT, 2), (product, b2.KNOB_TRI_TILE, 0)):
            want = routine(ctx, n)
            assert np.array_equal(routine(small, n), want), (n, routine.__name__)
            old = b2.get_tuning(knob)
            b2.set_tuning(knob, other)
            try:
                assert not np.array_equal(routine(ctx, n), want), (n, routine.__name__)
            finally:
                b2.set_tuning(knob, old)


@pytest.mark.parametrize("dtype", DTYPES)
def test_workspace_query_is_enough(b2, dtype):
    """A workspace of exactly b2_workspace_query(m, n, s) bytes serves every level-2 routine on an
    m x n problem (the recommended default is only a default): a matrix of a few very long rows,
    where the column splits of the row-dot kind must all be merged, and a triangular one."""
    s = np.dtype(dtype).itemsize
    tol = TOL[np.dtype(dtype)]
    m, n = 6, 300000
    small = b2.Context(workspace_bytes=b2.lib().b2_workspace_query(m, n, s))
    small.reset()
    a = synth.vector_np(41, 1, m * n, dtype)
    ga = Guarded(a)
    for trans in TRANSES:
        lenx, leny = (n, m) if trans == orc.NO_TRANS else (m, n)
        x, y = synth.vector_np(41, 2, lenx, dtype), synth.vector_np(41, 3, leny, dtype)
        gx, gy = Guarded(x), Guarded(y)
        b2.gemv(small, orc.ROW_MAJOR, trans, m, n, 1.25, ga.t, n, gx.t, 1, 0.5, gy.t, 1)
        oy = y.copy()
        absterms = orc.gemv(orc.ROW_MAJOR, trans, m, n, dtype(1.25), a, n, x, 1, dtype(0.5), oy, 1)
        assert_close(gy.host(), oy, absterms, dtype, f"gemv trans={trans} on the queried workspace")
        gy.check_guards()
    k = 2100
    tri = Guarded(synth.matrix_np(41, 4, k, k, k, dtype, tri_n=k).ravel())
    small = b2.Context(workspace_bytes=b2.lib().b2_workspace_query(k, k, s))
    small.reset()
    v = synth.vector_np(41, 5, k, dtype)
    gv, gy = Guarded(v), Guarded(v.copy())
    b2.symv(small, orc.ROW_MAJOR, orc.LOWER, k, 1.25, tri.t, k, gv.t, 1, 0.5, gy.t, 1)
    oy = v.copy()
    absterms = orc.symv(orc.ROW_MAJOR, orc.LOWER, k, dtype(1.25), tri.host(), k, v, 1, dtype(0.5), oy, 1)
    assert_close(gy.host(), oy, absterms, dtype, "symv on the queried workspace")
    for trans in TRANSES:
        gx = Guarded(v)
        b2.trmv(small, orc.ROW_MAJOR, orc.UPPER, trans, orc.NON_UNIT, k, tri.t, k, gx.t, 1)
        ox = v.copy()
        absterms = orc.trmv(orc.ROW_MAJOR, orc.UPPER, trans, orc.NON_UNIT, k, tri.host(), k, ox, 1)
        assert_close(gx.host(), ox, absterms, dtype, "trmv on the queried workspace")
        gx = Guarded(v)
        b2.trsv(small, orc.ROW_MAJOR, orc.UPPER, trans, orc.NON_UNIT, k, tri.t, k, gx.t, 1)
        assert small.device_status() == 0
        resid, scale = orc.trsv_residual(orc.ROW_MAJOR, orc.UPPER, trans, orc.NON_UNIT, k, tri.host(), k, v, 1,
                                         gx.host(), 1)
        assert np.all(resid <= tol * scale), "trsv on the queried workspace"


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("c", [2.0, 8.0])
def test_trsv_moderately_conditioned(b2, ctx, dtype, c):
    """Matrices that are NOT diagonally dominant: unit diagonal, off-diagonal uniform[-1, 1] * c / sqrt(n)
    (at c = 8 the solution grows to about 3e4 from a right-hand side in [-1, 1]).  The kernels apply
    explicit inverses of the 128 x 128 / 64 x 64 diagonal blocks, whose error grows with the blocks'
    condition number; the row-wise residual of the device solution must still meet the bound."""
    n = 1100
    tol = TOL[np.dtype(dtype)]
    u = synth.vector_np(5, n, n * n, np.float64).reshape(n, n)
    a = (u * c / np.sqrt(n)).astype(dtype)
    np.fill_diagonal(a, 1.0)
    b = synth.vector_np(5, 1, n, dtype)
    ga = Guarded(a.ravel())
    for uplo, trans, diag in ((orc.LOWER, orc.NO_TRANS, orc.UNIT), (orc.UPPER, orc.TRANS, orc.NON_UNIT),
                              (orc.UPPER, orc.NO_TRANS, orc.UNIT), (orc.LOWER, orc.TRANS, orc.NON_UNIT)):
        gx = Guarded(b)
        b2.trsv(ctx, orc.ROW_MAJOR, uplo, trans, diag, n, ga.t, n, gx.t, 1)
        assert ctx.device_status() == 0
        resid, scale = orc.trsv_residual(orc.ROW_MAJOR, uplo, trans, diag, n, a.ravel(), n, b, 1, gx.host(), 1)
        assert np.all(resid <= tol * scale), f"c={c} {uplo} {trans} {diag}: worst {np.max(resid / scale) / tol:.3f} of the bound"


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("unit", [1, 2, 4])
def test_symv_trmv_every_unit_length(b2, ctx, dtype, unit):
    """The tile kernel of symv / trmv cuts block rows (columns) into units of 1, 2 or 4 tiles,
    chosen by the matrix size; here each length is forced on sizes small enough for the full oracle
    and large enough to have rows of several units, a ragged edge, units of a single tile next to
    full ones, and several units per block (more units than SMs)."""
    old = b2.get_tuning(b2.KNOB_TRI_TILE_UNIT), b2.get_tuning(b2.KNOB_TRI_TILE)
    b2.set_tuning(b2.KNOB_TRI_TILE_UNIT, unit)
    b2.set_tuning(b2.KNOB_TRI_TILE, 2)  # every trmv through the tile kernel too
    try:
        for n in (700, 2443, 1280, 2560):  # (the last two: every tile full)
            a = synth.matrix_np(17, 3, n, n, n, dtype, tri_n=n).ravel()
            x, y = synth.vector_np(17, 4, n, dtype), synth.vector_np(17, 5, n, dtype)
            ga = Guarded(a)
            for uplo in UPLOS:
                gx, gy = Guarded(x), Guarded(y)
                b2.symv(ctx, orc.ROW_MAJOR, uplo, n, 1.25, ga.t, n, gx.t, 1, 0.5, gy.t, 1)
                oy = y.copy()
                absterms = orc.symv(orc.ROW_MAJOR, uplo, n, dtype(1.25), a, n, x, 1, dtype(0.5), oy, 1)
                assert_close(gy.host(), oy, absterms, dtype, f"symv n={n} uplo={uplo} unit={unit}")
                for trans, diag in itertools.product(TRANSES, DIAGS):
                    gx = Guarded(x)
                    b2.trmv(ctx, orc.ROW_MAJOR, uplo, trans, diag, n, ga.t, n, gx.t, 1)
                    ox = x.copy()
                    absterms = orc.trmv(orc.ROW_MAJOR, uplo, trans, diag, n, a, n, ox, 1)
                    assert_close(gx.host(), ox, absterms, dtype, f"trmv n={n} {uplo} {trans} {diag} unit={unit}")
    finally:
        b2.set_tuning(b2.KNOB_TRI_TILE_UNIT, old[0])
        b2.set_tuning(b2.KNOB_TRI_TILE, old[1])


@pytest.mark.parametrize("dtype", DTYPES)
def test_tile_kernel_tma_delivery(b2, ctx, dtype):
    """The ring kernel with its tiles delivered by one tiled TMA copy each (tensor map over the
    matrix, zero fill outside it, a shared-memory barrier per ring slot with bounded waits): symv
    and every trmv on sizes with ragged edges, with only full tiles, and with more units than SMs;
    the device status must stay clean (a barrier wait that ran out would set it)."""
    old = b2.get_tuning(b2.KNOB_TRI_TILE), b2.get_tuning(b2.KNOB_TRI_BULK)
    b2.set_tuning(b2.KNOB_TRI_TILE, 2)
    b2.set_tuning(b2.KNOB_TRI_BULK, 1)
    try:
        for n, pad in ((130, 0), (700, 4), (1280, 0), (2443, 0), (2560, 8)):
            lda = n + pad
            a = synth.matrix_np(19, 3, n, lda, lda, dtype, tri_n=n).ravel()
            x, y = synth.vector_np(19, 4, n, dtype), synth.vector_np(19, 5, n, dtype)
            ga = Guarded(a)
            for uplo in UPLOS:
                gx, gy = Guarded(x), Guarded(y)
                b2.symv(ctx, orc.ROW_MAJOR, uplo, n, 1.25, ga.t, lda, gx.t, 1, 0.5, gy.t, 1)
                oy = y.copy()
                absterms = orc.symv(orc.ROW_MAJOR, uplo, n, dtype(1.25), a, lda, x, 1, dtype(0.5), oy, 1)
                assert_close(gy.host(), oy, absterms, dtype, f"symv n={n} uplo={uplo}")
                for trans, diag in itertools.product(TRANSES, DIAGS):
                    gx = Guarded(x)
                    b2.trmv(ctx, orc.ROW_MAJOR, uplo, trans, diag, n, ga.t, lda, gx.t, 1)
                    ox = x.copy()
                    absterms = orc.trmv(orc.ROW_MAJOR, uplo, trans, diag, n, a, lda, ox, 1)
                    assert_close(gx.host(), ox, absterms, dtype, f"trmv n={n} {uplo} {trans} {diag}")
            assert ctx.device_status() == 0
            ga.check_guards()
    finally:
        b2.set_tuning(b2.KNOB_TRI_TILE, old[0])
        b2.set_tuning(b2.KNOB_TRI_BULK, old[1])


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("order", ORDERS)
def test_trmv_tile_kernel_forced(b2, ctx, dtype, order):
    """trmv through the shared-memory-ring tile kernel for every option combination (by default
    only the cases where it is the faster one take it): padded leading dimension, strided and
    reversed x, guard bands, the unreferenced triangle and a unit diagonal NaN-poisoned."""
    old = b2.get_tuning(b2.KNOB_TRI_TILE)
    b2.set_tuning(b2.KNOB_TRI_TILE, 2)
    try:
        for n, (pad, inc) in itertools.product((129, 700), ((0, 1), (4, 2), (8, -1))):
            lda = n + pad
            for uplo, trans, diag in itertools.product(UPLOS, TRANSES, DIAGS):
                a = tri_buf(12, n, lda, dtype, order, uplo, diag)
                x = synth.vector_np(7, n, n, dtype)
                hx = place(x, inc)
                ga, gx = Guarded(a), Guarded(hx)
                b2.trmv(ctx, order, uplo, trans, diag, n, ga.t, lda, gx.t, inc)
                ox = hx.copy()
                absterms = orc.trmv(order, uplo, trans, diag, n, a, lda, ox, inc)
                rx = gx.host()
                assert_close(pick(rx, n, inc), pick(ox, n, inc), absterms, dtype, f"trmv n={n} pad={pad} inc={inc}")
                assert_same_gaps(rx, hx, n, inc)
                ga.check_guards(), gx.check_guards()
    finally:
        b2.set_tuning(b2.KNOB_TRI_TILE, old)
