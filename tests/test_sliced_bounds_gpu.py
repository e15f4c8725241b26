"""Error bounds of the sliced FP64 products: an output of K terms within
(K + 2) 2^-53 of sum |h x| (the bound of a K-term multiply-add chain, and the
epilogue), on operands that sit just above the kernels' checks and on panels whose
entries fall over many orders of magnitude."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from synthetic.structures import BlockPattern

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _handle(pat, vals):
    from paper_2609_04397_gb300 import VBCSR
    return VBCSR.from_pattern(pat, vals, torch.float64, "cuda:0")


def _kernels(fn):
    """Names of the library's kernels that fn launches (never empty)."""
    from torch.profiler import ProfilerActivity, profile
    for _ in range(5):   # a trace can come back before its buffers fill
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            fn()
            torch.cuda.synchronize()
        names = [e.name for e in prof.events() if "vbcsr" in e.name]
        if names:
            return names
    raise AssertionError("no trace of the launches")


def _uniform(rows, K, b=16):
    """rows block rows of b x b blocks, all over the same K / b block columns."""
    n = K // b
    return BlockPattern(np.full(rows, b), np.full(n, b), np.arange(rows + 1) * n, np.tile(np.arange(n), rows))


def _block_values(h, rows, b=16):
    """The same stored row h everywhere."""
    blocks = np.broadcast_to(h.reshape(-1, 1, b), (len(h) // b, b, b))
    return np.tile(blocks.reshape(-1), rows)


def _sums(h, x):
    terms = [Fraction(a) * Fraction(b) for a, b in zip(h.tolist(), x.tolist())]
    return sum(terms), sum(abs(t) for t in terms)


def _products(K):
    """(h, x) of K terms: large entries of one side meet entries of the other that the
    fixed point rounds by half a unit, and the sum rests on a few products."""
    half = 0.99 * 2.0 ** -55   # 0.495 of the last place at a scale of 1.97
    h, x = np.full(K, half), np.full(K, 1.97)
    h[0], x[0] = 1.97, 4.6 * 2.0 ** -6
    yield "one product", h, x
    for n in (9, 33, 35, 60):   # n products of leading digits 126 x 1
        h, x = np.full(K, half), np.full(K, 1.97)
        h[:n], x[:n] = 1.97, 0.504 * 2.0 ** -6
        yield f"{n} products", h, x


@pytest.mark.parametrize("K", [64, 320, 768])
@pytest.mark.parametrize("k", [5, 16])
def test_products_just_above_the_check(K, k):
    rows = -(-(1 << 24) // (16 * K * (8 if k < 8 else k)))
    pat = _uniform(rows, K)
    for name, h, x in _products(K):
        H = _handle(pat, _block_values(h, rows))
        sign = np.where(np.arange(k) % 2, -1.0, 1.0)
        X = torch.from_numpy(x[:, None] * sign).cuda()
        exact, mag = _sums(h, x)
        got = H.spmm(X).cpu().numpy()
        bound = float((K + 2) * U * mag)
        for s in (1, -1):
            err = max(abs(Fraction(v) - s * exact) for v in np.unique(got[:, sign == s]).tolist())
            assert err <= bound, (name, float(err / mag) / U)
    assert any("slice_product" in n for n in _kernels(lambda: H.spmm(X)))


@pytest.mark.parametrize("k", [6, 16, 18, 40])
def test_sampled_products_just_above_the_check(k):
    """Every common column of the two rows has a small leading digit and six of -128."""
    n = -(-(1 << 22) // (k * 1024)) + 1
    pat = _uniform(max(n // 4, 1), 1024)
    for d in (1, 2, 3, 4, 6, 8, 11):
        e = float((d << 56) - 128 * sum(1 << (8 * i) for i in range(1, 7))) * 2.0 ** -62
        A = np.full((pat.n_rows, k), e)
        B = np.full((pat.n_cols, k), e)
        A[:, 0], A[:, 1], B[:, 0], B[:, 1] = 1.97, 0.0, 0.0, 1.97
        exact, mag = _sums(A[0], B[0])
        H = _handle(pat, np.zeros(pat.nnz))
        got = H.sddmm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()).cpu().numpy()
        err = max(abs(Fraction(v) - exact) for v in np.unique(got).tolist())
        assert err <= (k + 2) * Fraction(U) * mag, (d, float(err / mag) / U)
    assert any("slice_sddmm" in s for s in _kernels(lambda: H.sddmm(torch.from_numpy(A).cuda(),
                                                                    torch.from_numpy(B).cuda())))


@pytest.mark.parametrize("K", [128, 320, 752])
@pytest.mark.parametrize("fall", [3.0, 7.0, 14.0])
def test_falling_panels(K, fall, monkeypatch):
    """Columns of X that fall by e^-fall within a row of H, in random order: inside the bound,
    and no further off than the multiply-adds of the same call (a handle with device checks)."""
    rng = np.random.default_rng(int(K + fall))
    rows = -(-(1 << 24) // (16 * K * 16))
    pat = _uniform(rows, K)
    vals = rng.standard_normal(pat.nnz)
    H = _handle(pat, vals)
    monkeypatch.setenv("VBCSR_DEBUG_CHECKS", "1")
    plain = _handle(pat, vals)
    X = rng.standard_normal((K, 16)) * np.exp(-fall * rng.random((K, 16)))
    dense = vals.reshape(rows, K // 16, 16, 16).transpose(0, 2, 1, 3).reshape(rows * 16, K)[:2048].astype(np.longdouble)
    exact = dense @ X.astype(np.longdouble)
    mag = (np.abs(dense) @ np.abs(X).astype(np.longdouble)).astype(np.float64)
    Xd = torch.from_numpy(X).cuda()
    e, ec = (np.abs((P.spmm(Xd)[:2048].cpu().numpy() - exact).astype(np.float64)) / mag / U for P in (H, plain))
    assert e.max() <= K + 2
    assert np.sqrt(np.mean(e ** 2)) <= np.sqrt(np.mean(ec ** 2))
    assert any("slice_product" in n for n in _kernels(lambda: H.spmm(Xd)))
    assert not any("slice" in n for n in _kernels(lambda: plain.spmm(Xd)))


def _spiked(b, cols, k, complex_values, seed):
    """A dense operator of b-row items with one huge entry in every seventh row, met by a panel
    whose row there is zero in the odd columns: one unresolved output a column pair."""
    rng = np.random.default_rng(seed)
    wb = -(-cols // b)
    rows = max(-(-(1 << 24) // (b * wb * b * (16 if k > 8 else 8))), 4)
    pat = BlockPattern(np.full(rows, b), np.full(wb, b), np.arange(rows + 1) * wb, np.tile(np.arange(wb), rows))
    K = wb * b
    D = rng.standard_normal((rows * b, K))
    X = rng.standard_normal((K, k))
    if complex_values:
        D = D + 1j * rng.standard_normal(D.shape)
        X = X + 1j * rng.standard_normal(X.shape)
    D[::7, K - 2] *= 1e9
    X[K - 2, 1::4] = 0.0
    vals = D.reshape(rows, b, wb, b).transpose(0, 2, 1, 3).reshape(-1)
    return pat, np.ascontiguousarray(vals), D, X


@pytest.mark.parametrize("b", [3, 8, 9, 13, 16])
@pytest.mark.parametrize("k", [5, 8, 16, 21])
@pytest.mark.parametrize("kind", [np.float64, np.complex128])
def test_single_unresolved_outputs(b, k, kind):
    """Forward and adjoint, with the fused epilogue, alpha a power of two and not."""
    from paper_2609_04397_gb300 import VBCSR
    cplx = kind is np.complex128
    pat, vals, D, X = _spiked(b, 160, k, cplx, b + k)
    H = VBCSR.from_pattern(pat, vals, torch.complex128 if cplx else torch.float64, "cuda:0")
    rng = np.random.default_rng(1)
    K = D.shape[1]
    some = np.unique(np.concatenate([np.arange(0, min(200, len(D))), np.arange(0, len(D), max(len(D) // 200, 1))]))
    wide = np.clongdouble if cplx else np.longdouble
    for alpha in (2.0, -0.3):
        Y0, Z, R = (rng.standard_normal((len(D), k)).astype(kind) for _ in range(3))
        Y, dot = torch.from_numpy(Y0.copy()).cuda(), torch.zeros(1, dtype=torch.float64, device="cuda:0")
        H.spmm_ex(torch.from_numpy(X).cuda(), alpha, -1.0, Y, gamma=0.5, Z=torch.from_numpy(Z).cuda(),
                  R=torch.from_numpy(R).cuda(), dot_out=dot)
        got = Y.cpu().numpy()
        ref = alpha * (D[some].astype(wide) @ X.astype(wide)) - Y0[some] + 0.5 * Z[some]
        mag = abs(alpha) * (np.abs(D[some]) @ np.abs(X)) + np.abs(Y0[some]) + np.abs(Z[some])
        # a complex term is two real ones of each component
        bound = ((4 if cplx else 1) * K + 8) * U * mag
        assert (np.abs((got[some] - ref).astype(kind)) <= bound).all()
        terms = np.sum(np.abs(R * got))
        assert abs(dot.item() - np.sum((np.conj(R) * got).real)) <= 1e-12 * terms
    G = rng.standard_normal((len(D), k)).astype(kind)
    G[:, 1] = 0.0
    G[0, 1] = 1.0
    got = H.spmm_adjoint(torch.from_numpy(G).cuda()).cpu().numpy()
    ref = np.conj(D.T).astype(kind) @ G
    mag = np.abs(D.T) @ np.abs(G)
    # both sides are chains of len(D) terms at most (blocked on the host)
    assert (np.abs(got - ref) <= 2 * (4 if cplx else 1) * len(D) * U * mag).all()
    assert any("slice_product" in n for n in _kernels(lambda: H.spmm(torch.from_numpy(X).cuda())))


@pytest.mark.parametrize("k", [5, 16, 40])
@pytest.mark.parametrize("b", [9, 13])
def test_heavy_tailed_panels(b, k):
    """Panels whose largest entries are far above the rest (Student's t with 2 degrees of
    freedom): second attempts at most passes, single outputs, items left to multiply-adds."""
    rng = np.random.default_rng(b * k)
    wb = 340 // b
    rows = -(-(1 << 24) // (b * wb * b * (16 if k > 8 else 8)))
    pat = BlockPattern(np.full(rows, b), np.full(40 * wb, b), np.arange(rows + 1) * wb,
                       np.sort(np.argsort(rng.random((rows, 40 * wb)), axis=1)[:, :wb], axis=1).reshape(-1))
    vals = rng.standard_normal(pat.nnz)
    X = rng.standard_t(2, (pat.n_cols, k))
    Y0 = rng.standard_normal((pat.n_rows, k))
    H = _handle(pat, vals)
    Y = torch.from_numpy(Y0.copy()).cuda()
    H.spmm(torch.from_numpy(X).cuda(), -2.0, 0.5, Y)
    got = Y.cpu().numpy()
    K = wb * b
    cols = pat.block_col_idx.reshape(rows, wb)
    for r in range(0, rows, max(rows // 40, 1)):
        D = vals.reshape(rows, wb, b, b)[r].transpose(1, 0, 2).reshape(b, K).astype(np.longdouble)
        x = X.reshape(-1, b, k)[cols[r]].reshape(K, k).astype(np.longdouble)
        ref = -2.0 * (D @ x) + 0.5 * Y0[r * b:(r + 1) * b]
        mag = 2.0 * (np.abs(D) @ np.abs(x)) + 0.5 * np.abs(Y0[r * b:(r + 1) * b])
        assert (np.abs(got[r * b:(r + 1) * b] - ref) <= (K + 4) * U * mag).all()
    assert any("slice_product" in n for n in _kernels(lambda: H.spmm(torch.from_numpy(X).cuda())))


def _time(fn, n=10):
    fn()
    best = 1e9
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(n):
            fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / n)
    return best


@pytest.mark.parametrize("k", [8, 16])
def test_panels_of_mostly_tiny_entries_are_not_tried(k):
    """Columns of 1 and -1 and one entry 2^9 or 2^13 times as large: neither is resolved, both
    run multiply-adds without a digit product before them."""
    rng = np.random.default_rng(k)
    n, wb, b = 6000, 24, 13
    cols = np.sort((np.arange(n)[:, None] + 7 * np.arange(wb)) % n, axis=1)
    pat = BlockPattern(np.full(n, b), np.full(n, b), np.arange(n + 1) * wb, cols.reshape(-1))
    H = _handle(pat, rng.standard_normal(pat.nnz))
    X = torch.randn(pat.n_cols, k, dtype=torch.float64, device="cuda:0").sign()
    Y = torch.empty(pat.n_rows, k, dtype=torch.float64, device="cuda:0")
    times = []
    for peak in (2.0 ** 9, 2.0 ** 13):
        X[77] = peak
        times.append(_time(lambda: H.spmm(X, 1.0, 0.0, Y)))
        assert any("slice_product" in s for s in _kernels(lambda: H.spmm(X, 1.0, 0.0, Y)))
    assert times[0] <= 1.05 * times[1], times


@pytest.mark.parametrize("k", [5, 8, 13])
@pytest.mark.parametrize("kpoint", [[0.13, -0.27, 0.41], [0.0, 0.0, 0.0]])
def test_real_panels_of_complex_operators_are_sliced(k, kpoint):
    """Zero imaginary parts are no reason for multiply-adds (a panel of unit columns takes
    them and gives their time), nor are the outputs that they make exact zeros where the
    operator is real as well."""
    import oracle
    import synthetic as syn
    from paper_2609_04397_gb300 import VBCSR
    w = syn.zincblende_crystal(8)
    H = VBCSR.from_images(w.bsize, w.edge_i, w.edge_j, w.edge_R, w.edge_values, device="cuda:0")
    H.set_kpoint(kpoint)
    rb, cb, rp, ci = H.pattern
    pat = BlockPattern(rb, cb, rp, ci)
    rng = np.random.default_rng(k)
    full = rng.standard_normal((pat.n_rows, k)) + 1j * rng.standard_normal((pat.n_rows, k))
    vals = H.get_values().cpu().numpy()
    assert any(kpoint) or (vals.imag == 0).all()
    times = {}
    unit = np.eye(pat.n_rows, k, dtype=complex)
    for name, P in (("real", full.real.astype(complex)), ("nearly real", full.real + 1e-9j * full.imag), ("unit", unit)):
        Xd = torch.from_numpy(P).cuda()
        Y = torch.empty_like(Xd)
        for fn, ref in ((H.spmm, oracle.spmm_complex), (H.spmm_adjoint, oracle.spmm_adjoint_complex)):
            got = fn(Xd, 1.0, 0.0, Y).cpu().numpy()
            mag = (oracle.spmm if fn == H.spmm else oracle.spmm_adjoint)(pat, np.abs(vals), np.abs(P))
            # two chains of at most 2 x 380 terms
            assert (np.abs(got - ref(pat, vals, P)) <= 4 * 760 * U * mag).all(), name
            if not any(kpoint) and name == "real":
                assert (got.imag == 0).all()
        times[name] = _time(lambda: H.spmm(Xd, 1.0, 0.0, Y))
    assert times["real"] <= 0.85 * times["unit"], times


@pytest.mark.parametrize("k", [17, 33, 40, 560])
def test_one_bad_column_leaves_the_other_passes_sliced(k):
    """A column with a NaN, an Inf or one entry only sends its own 16 columns to multiply-adds:
    the bits of the others are those of a panel without it (from column 496 on a panel's
    columns are taken together)."""
    rng = np.random.default_rng(k)
    n, wb, b = 400, 24, 13
    cols = np.sort((np.arange(n)[:, None] + 7 * np.arange(wb)) % n, axis=1)
    pat = BlockPattern(np.full(n, b), np.full(n, b), np.arange(n + 1) * wb, cols.reshape(-1))
    vals = rng.standard_normal(pat.nnz)
    H = _handle(pat, vals)
    X = rng.standard_normal((pat.n_cols, k))
    clean = H.spmm(torch.from_numpy(X).cuda()).cpu().numpy()
    import oracle
    for bad in sorted({0, 16, k - 1, min(k - 1, 500)}):
        for kind in ("nan", "inf", "unit"):
            Z = X.copy()
            if kind == "unit":
                Z[:, bad] = 0.0
                Z[7, bad] = 1.0
            else:
                Z[7, bad] = float(kind)
            got = H.spmm(torch.from_numpy(Z).cuda()).cpu().numpy()
            lo = 16 * (bad // 16)
            hi = lo + 16
            if bad >= 496:
                lo, hi = 496, k
            same = np.r_[0:lo, min(hi, k):k]
            assert np.array_equal(got[:, same], clean[:, same]), (bad, kind)
            own = slice(lo, min(hi, k, lo + 16))
            with np.errstate(invalid="ignore"):
                ref = oracle.spmm(pat, vals, np.ascontiguousarray(Z[:, own]))
            mag = oracle.spmm(pat, np.abs(vals), np.abs(np.ascontiguousarray(Z[:, own])))
            assert np.array_equal(np.isnan(got[:, own]), np.isnan(ref))
            fin = np.isfinite(ref)
            # two chains of 312 terms
            assert (np.abs(got[:, own][fin] - ref[fin]) <= 640 * U * mag[fin]).all(), (bad, kind)
    assert any("slice_product" in s for s in _kernels(lambda: H.spmm(torch.from_numpy(X).cuda())))


def test_panel_that_does_not_fit_leaves_narrower_ones_sliced():
    """With the device almost full a wide product and a wide sampled one run multiply-adds;
    narrower ones keep their buffers, and the wide ones are sliced again when there is room."""
    import synthetic as syn
    w = syn.amorphous(700, side=60.0 * (700 / 20000) ** (1 / 3))
    H = _handle(w.pattern, w.values)
    k, wide = 16, 8192
    X, A = (torch.randn(w.pattern.n_rows, wide, dtype=torch.float64, device="cuda:0") for _ in range(2))
    Xk, Ak, Xs, As = X[:, :k].contiguous(), A[:, :k].contiguous(), X[:, :700].contiguous(), A[:, :700].contiguous()
    Y, D = torch.empty_like(X), torch.empty(w.pattern.nnz, dtype=torch.float64, device="cuda:0")
    first = H.spmm(Xk)
    H.sddmm(Ak, Xk)
    Yp = torch.cat([H.spmm(X[:, c:c + 4].contiguous()) for c in range(0, 64, 4)], 1)   # multiply-adds
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    leave = 24 << 20
    full = []
    for part in (1 << 32, 1 << 28, 1 << 24):
        while torch.cuda.mem_get_info()[0] > leave + part:
            full.append(torch.empty(part, dtype=torch.uint8, device="cuda:0"))
    H.spmm(X, 1.0, 0.0, Y)
    H.sddmm(As, Xs, 1.0, 0.0, D)
    again = torch.empty_like(first)
    H.spmm(Xk, 1.0, 0.0, again)
    torch.cuda.synchronize()
    full.clear()
    torch.cuda.empty_cache()
    bound = 1600 * U * H_abs_product(w, X[:, :64])   # two chains of at most 768 terms
    assert ((Y[:, :64] - Yp).abs() <= bound).all()
    assert torch.equal(again, first)
    names = _kernels(lambda: (H.spmm(Xk), H.sddmm(Ak, Xk)))
    assert any("slice_product" in s for s in names) and any("slice_sddmm" in s for s in names)
    for _ in range(70):
        H.spmm(X, 1.0, 0.0, Y)
        H.sddmm(As, Xs, 1.0, 0.0, D)
    names = _kernels(lambda: (H.spmm(X, 1.0, 0.0, Y), H.sddmm(As, Xs, 1.0, 0.0, D)))
    assert any("slice_product" in s for s in names) and any("slice_sddmm" in s for s in names)


def H_abs_product(w, X):
    """sum |h x| of every output"""
    return _handle(w.pattern, np.abs(w.values)).spmm(X.abs().contiguous())


def _amorphous():
    import synthetic as syn
    w = syn.amorphous(700, side=60.0 * (700 / 20000) ** (1 / 3))
    return w, _handle(w.pattern, w.values)


def test_autotune_times_the_multiply_adds():
    """At a width that runs sliced the tuner still chooses the multiply-adds' tiles by their
    own times: narrower products use them."""
    w, H = _amorphous()
    X = torch.randn(w.pattern.n_cols, 16, dtype=torch.float64, device="cuda:0")
    names = _kernels(lambda: H.autotune(16))
    assert any("fma" in s for s in names) and not any("slice" in s for s in names)
    assert any("slice_product" in s for s in _kernels(lambda: H.spmm(X)))


def test_captured_values_before_any_product():
    """A captured change of the values on a handle without digit tiles does not keep its products
    off the tensor cores: every call rebuilds the tiles, a recurrence and a graph once."""
    import oracle
    import synthetic as syn
    w, H = _amorphous()
    pat, k = w.pattern, 16
    X = np.random.default_rng(1).standard_normal((pat.n_cols, k))
    Xd = torch.from_numpy(X).cuda()
    v = [syn.random_values(pat, s) / 40 for s in range(4)]
    buf = torch.from_numpy(v[0]).cuda()
    H.set_values(buf)
    setv = torch.cuda.CUDAGraph()
    with torch.cuda.graph(setv):
        H.set_values(buf)

    def same(i, y):
        ref, mag = oracle.spmm(pat, v[i], X), oracle.spmm(pat, np.abs(v[i]), np.abs(X))
        assert (np.abs(y.cpu().numpy() - ref) <= 1600 * U * mag).all()   # two chains of at most 768 terms

    assert any("slice_product" in s for s in _kernels(lambda: H.spmm(Xd)))
    same(0, H.spmm(Xd))
    buf.copy_(torch.from_numpy(v[1]))
    setv.replay()
    same(1, H.spmm(Xd))
    Y = torch.empty(2, pat.n_rows, k, dtype=torch.float64, device="cuda:0")
    prod = torch.cuda.CUDAGraph()
    with torch.cuda.graph(prod):
        H.spmm(Xd, 1.0, 0.0, Y[0])
        H.spmm(Xd, 1.0, 0.0, Y[1])
    for i in (2, 3):
        buf.copy_(torch.from_numpy(v[i]))
        setv.replay()
        prod.replay()
        same(i, Y[0])
        same(i, Y[1])
    assert sum("slice_values" in s for s in _kernels(prod.replay)) == 1
    R = torch.randn(pat.n_rows, k, dtype=torch.float64, device="cuda:0")
    names = _kernels(lambda: H.chebyshev(R, 6))
    assert sum("slice_product" in s for s in names) == 5 and sum("slice_values" in s for s in names) == 1


def _device_bytes(H):
    import ctypes
    from paper_2609_04397_gb300 import _lib
    info = _lib.Info()
    assert _lib.lib().vbcsr_get_info(H.handle, ctypes.byref(info)) == 0
    return info.device_bytes


def test_digit_buffers_leave_memory_and_are_given_back():
    """No digit buffers while they would leave less than a quarter of the device's memory;
    set_sliced(False) frees those that no graph holds, and products run multiply-adds."""
    w, H = _amorphous()
    k = 16
    X = torch.randn(w.pattern.n_cols, k, dtype=torch.float64, device="cuda:0")
    Y = torch.empty(w.pattern.n_rows, k, dtype=torch.float64, device="cuda:0")
    bare = _device_bytes(H)
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    full = [torch.empty(1 << 32, dtype=torch.uint8, device="cuda:0") for _ in range((free - total // 5) >> 32)]
    assert not any("slice" in s for s in _kernels(lambda: H.spmm(X, 1.0, 0.0, Y)))
    assert _device_bytes(H) == bare
    full.clear()
    torch.cuda.empty_cache()
    for _ in range(70):
        H.spmm(X, 1.0, 0.0, Y)
    assert any("slice_product" in s for s in _kernels(lambda: H.spmm(X, 1.0, 0.0, Y)))
    first = Y.clone()
    D = H.sddmm(X[:, :6].contiguous(), X[:, :6].contiguous())
    assert _device_bytes(H) > bare + 7 * w.pattern.nnz
    H.set_sliced(False)
    assert _device_bytes(H) == bare
    names = _kernels(lambda: (H.spmm(X, 1.0, 0.0, Y), H.sddmm(X[:, :6].contiguous(), X[:, :6].contiguous())))
    assert names and not any("slice" in s for s in names)
    assert ((Y - first).abs() <= 1600 * U * H_abs_product(w, X)).all()   # two chains of at most 768 terms
    H.set_sliced(True)
    assert torch.equal(H.spmm(X), first) and torch.equal(H.sddmm(X[:, :6].contiguous(), X[:, :6].contiguous()), D)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        H.spmm(X, 1.0, 0.0, Y)
    H.set_sliced(False)
    Y.zero_()
    graph.replay()
    assert torch.equal(Y, first)
    H.set_values(torch.from_numpy(2.0 * w.values).cuda())
    graph.replay()
    assert torch.equal(Y, 2.0 * first)


@pytest.mark.parametrize("small,sliced", [(1, True), (8, False)])
def test_batches_are_sliced_for_their_share_of_large_structures(small, sliced):
    """One structure above the size line beside small ones: sliced when it holds two fifths of the
    batch's entries, else multiply-adds throughout, as one launch without passes over X."""
    import oracle
    import synthetic as syn
    from paper_2609_04397_gb300 import VBCSR
    pats = [syn.random_pattern(n, n, (4, 9, 13), 0.15, n, empty_rows=0, unsorted=True)
            for n in [330] + [220 + s for s in range(small)]]
    pats = [BlockPattern(p.row_bsize, p.row_bsize, p.block_row_ptr, p.block_col_idx) for p in pats]
    nnz = np.array([p.nnz for p in pats])
    assert nnz[0] * 16 >= 1 << 24 > nnz[1] * 16 and (nnz[0] / nnz.sum() >= 0.5 if sliced else nnz[0] / nnz.sum() <= 0.35)
    offs = np.cumsum([0] + [len(p.row_bsize) for p in pats])
    ptr = np.concatenate([[0]] + [p.block_row_ptr[1:] + s for p, s in zip(pats, np.cumsum([0] + [p.nblk for p in pats]))])
    col = np.concatenate([p.block_col_idx for p in pats])
    rb = np.concatenate([p.row_bsize for p in pats])
    vals = [syn.random_values(p, i) for i, p in enumerate(pats)]
    H = VBCSR.from_batched(offs, offs, rb, rb, ptr, col, np.concatenate(vals), torch.float64, "cuda:0")
    X = np.random.default_rng(0).standard_normal((int(rb.sum()), 16))
    Xd = torch.from_numpy(X).cuda()
    names = _kernels(lambda: H.spmm(Xd))
    assert any("slice" in s for s in names) == sliced
    got, r, c = H.spmm(Xd).cpu().numpy(), 0, 0
    for p, v in zip(pats, vals):
        x = np.ascontiguousarray(X[c:c + p.n_cols])
        mag = oracle.spmm(p, np.abs(v), np.abs(x))
        # two chains of a row's terms
        assert (np.abs(got[r:r + p.n_rows] - oracle.spmm(p, v, x)) <= 2 * p.n_cols * U * mag).all()
        r, c = r + p.n_rows, c + p.n_cols
    # in a recurrence the lines are lower
    assert any("slice_product" in s for s in _kernels(lambda: H.chebyshev(Xd, 4)))


def test_what_is_not_sliced_runs_multiply_adds():
    """The column floors, the size line and small work items, each seen in a trace that shows the
    multiply-add kernel that ran instead."""
    import synthetic as syn

    def sliced(fn, plain):
        names = _kernels(fn)
        yes = any("slice" in s for s in names)
        assert yes or any(plain in s for s in names), names
        return yes

    w, H = _amorphous()
    lo, hi = H.gershgorin()
    H.shift_scale((lo + hi) / 2, 0.51 * (hi - lo))
    X = torch.randn(w.pattern.n_cols, 16, dtype=torch.float64, device="cuda:0")
    for k in (1, 2, 3, 4, 5, 8, 16):
        Xk = X[:, :k].contiguous()
        kc = max(8, 1 << (k - 1).bit_length())
        single = k >= 5 and w.pattern.nnz * kc >= 1 << 24
        repeated = k >= 3 and w.pattern.nnz * k >= 1 << 22
        assert sliced(lambda: H.spmm(Xk), "fma") == single
        assert sliced(lambda: H.spmm_adjoint(Xk), "fma") == single
        assert sliced(lambda: H.chebyshev(Xk, 4), "fma") == repeated
        assert sliced(lambda: H.sddmm(Xk, Xk), "sddmm") == (k >= 6 and w.pattern.nnz * k >= 1 << 22)
    n = 14_000   # 2 x 2 blocks, 40 a row: 160 entries a work item
    cols = np.sort((np.arange(n)[:, None] + 3 * np.arange(40)) % n, axis=1)
    pat = BlockPattern(np.full(n, 2), np.full(n, 2), np.arange(n + 1) * 40, cols.reshape(-1))
    H = _handle(pat, syn.random_values(pat, 1))
    X = torch.randn(pat.n_cols, 8, dtype=torch.float64, device="cuda:0")
    assert not sliced(lambda: H.spmm(X), "fma")
    assert not sliced(lambda: H.spmm_adjoint(X), "fma")
    assert not sliced(lambda: H.sddmm(X, X), "sddmm")
