"""The sliced form of native FP64 products (csrc/sliced.cuh): FP64 operands as
base-256 digits on the FP16 tensor cores, with FP64 multiply-adds wherever the
fixed point does not resolve an output.

Every element is held to 1e-13 of sum |h x|: the oracle's own chain of up to
768 multiply-adds stays within 768 2^-53 = 8.5e-14 of it, and an output that
passes the sliced kernel's check within about 1e-14."""
import numpy as np
import pytest
import torch

import oracle
import synthetic as syn
from synthetic.structures import BlockPattern

pytestmark = pytest.mark.gpu
TOL = 1e-13


def _handle(pat, vals):
    from paper_2609_04397_gb300 import VBCSR
    return VBCSR.from_pattern(pat, vals, torch.float64, "cuda:0")


def _kernels(fn):
    from torch.profiler import ProfilerActivity, profile
    for _ in range(2):   # the first trace of a process can come back before its buffers fill
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            fn()
            torch.cuda.synchronize()
        names = [e.name for e in prof.events() if "vbcsr" in e.name]
        if names:
            return names
    return []


def _check(H, pat, vals, X, transpose=False, alpha=1.0, beta=0.0, Y0=None, tol=TOL):
    fn, ref_fn = (H.spmm_adjoint, oracle.spmm_adjoint) if transpose else (H.spmm, oracle.spmm)
    Xd = torch.from_numpy(X).cuda()
    if Y0 is None:
        got = fn(Xd, alpha).cpu().numpy()
        Y0 = np.zeros_like(got)
    else:
        got = fn(Xd, alpha, beta, torch.from_numpy(Y0.copy()).cuda()).cpu().numpy()
    ref = ref_fn(pat, vals, X, alpha, beta, Y0)
    scale = ref_fn(pat, np.abs(vals), np.abs(X), abs(alpha), 0.0) + abs(beta) * np.abs(Y0)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    fin = np.isfinite(ref)
    assert np.array_equal(got[~fin & ~np.isnan(ref)], ref[~fin & ~np.isnan(ref)])
    bad = np.abs(got[fin] - ref[fin]) > tol * scale[fin]
    assert not bad.any(), (bad.sum(), np.max(np.abs(got[fin] - ref[fin]) / np.maximum(scale[fin], 1e-300)))
    return got


def _pattern(sizes, n=64, density=0.5, seed=1):
    return syn.random_pattern(n, n - 3, sizes, density, seed, empty_rows=2, unsorted=True)


# row heights 1 .. 16 and taller (chunked), rows of a multiple of 16 columns, ragged ones, some
# wider than the 768 columns a sliced row may have, widths around the 8- and 16-column tiles
@pytest.mark.parametrize("sizes,n,density", [((4, 9, 13), 64, 0.5), ((16,), 48, 0.6), ((1, 2, 3), 300, 0.6),
                                             ((17, 20, 33), 40, 0.4), ((13, 15), 80, 0.6)])
@pytest.mark.parametrize("k", [2, 8, 9, 16, 17, 40])
def test_sliced_products_against_oracle(sizes, n, density, k):
    pat = _pattern(sizes, n, density, seed=k)
    vals = syn.random_values(pat, k)
    H = _handle(pat, vals)
    rng = np.random.default_rng(k)
    wide = max(k, -(-(1 << 24) // pat.nnz) + 1)        # columns from which this operator is sliced
    for cols in sorted({k, wide}):
        X = rng.standard_normal((pat.n_cols, cols))
        Y0 = rng.standard_normal((pat.n_rows, cols))
        _check(H, pat, vals, X, alpha=2.0, beta=-1.0, Y0=Y0)
        Xa = rng.standard_normal((pat.n_rows, cols))
        _check(H, pat, vals, Xa, transpose=True)
    assert any("slice_product" in n for n in _kernels(lambda: H.spmm(torch.from_numpy(X).cuda())))
    H.check()


def test_exact_level_sums_at_the_widest_row():
    """768 equal products whose digits are all 127 or all -128 but the leading one:
    the largest level sums there are. The exact sum is 768 h x."""
    b = 16
    pat = BlockPattern(np.full(120, b), np.full(48, b), np.arange(121) * 48, np.tile(np.arange(48), 120))
    assert pat.n_cols == 768
    for digits in (0x7D7F7F7F7F7F7F, 0x7D808080808080 - 0x01010101010100, 0x3E7F7F7F7F7F7F):
        h = float(digits) * 2.0 ** -54
        H = _handle(pat, np.full(pat.nnz, h))
        for x in (h, -h, 0.75 * h):
            X = torch.full((768, 16), x, dtype=torch.float64, device="cuda:0")
            from fractions import Fraction
            exact = float(768 * Fraction(h) * Fraction(x))
            got = H.spmm(X)
            assert (got - exact).abs().max().item() <= 4e-16 * abs(exact)


@pytest.mark.parametrize("k", [7, 8, 16, 19])
def test_items_of_nine_rows(k):
    """The ninth row's digits are the N side of its own products: the largest digit sums of
    765 columns, and ninth rows that are zero, far smaller than the others or unresolved."""
    b = 9
    nr = 310
    pat = BlockPattern(np.full(nr, b), np.full(85, b), np.arange(nr + 1) * 85, np.tile(np.arange(85), nr))
    h = float(0x7D808080808080 - 0x01010101010100) * 2.0 ** -54
    H = _handle(pat, np.full(pat.nnz, h))
    X = torch.full((765, k), -h, dtype=torch.float64, device="cuda:0")
    from fractions import Fraction
    exact = float(-765 * Fraction(h) * Fraction(h))
    got = H.spmm(X)
    assert (got - exact).abs().max().item() <= 4e-16 * abs(exact)
    assert any("slice_product" in n for n in _kernels(lambda: H.spmm(X)))
    rng = np.random.default_rng(k)
    vals = rng.standard_normal(pat.nnz).reshape(nr, 85, b, b)   # blocks of a block row are b x b
    vals[0, :, 8] = 0.0
    vals[1, :, 8] *= 1e-200
    vals[2, :, 8, :] = 0.0
    vals[2, 3, 8, 4] = 1.0
    vals[3, :, 8] *= np.exp(-np.arange(85) / 3.0)[:, None]
    vals = vals.reshape(-1)
    X = rng.standard_normal((765, k))
    X[:40, k // 2] = 0.0
    H = _handle(pat, vals)
    Y0 = rng.standard_normal((nr * b, k))
    _check(H, pat, vals, X, alpha=0.3, beta=2.0, Y0=Y0)
    _check(H, pat, vals, rng.standard_normal((nr * b, k)), transpose=True)


def test_unresolved_outputs_take_multiply_adds():
    """Graded rows and columns, zero rows and columns, panels supported on a few
    rows, tiny and huge magnitudes, Inf and NaN: every output as accurate as the
    multiply-add chain's, and NaN and Inf only where they belong."""
    pat = _pattern((4, 9, 13), 260, 0.25, 5)
    rng = np.random.default_rng(0)
    assert 32 * pat.nnz >= 1 << 24   # sliced
    vals = syn.random_values(pat, 5)
    k = 24
    X = rng.standard_normal((pat.n_cols, k))
    cases = {}
    cases["graded columns"] = X * np.exp(-np.arange(pat.n_cols) / 5.0)[:, None]
    cases["one-hot"] = np.eye(pat.n_cols)[:, :k]
    local = np.zeros_like(X)
    local[100:180] = X[100:180]
    cases["local"] = local
    z = X.copy()
    z[:, 3] = 0.0
    z[:, 5] *= 1e-200
    z[:, 7] *= 1e200
    z[:, 9] = 5e-324
    cases["scales"] = z
    bad = X.copy()
    bad[17, 2], bad[200, 4], bad[3, 6] = np.nan, np.inf, -np.inf
    cases["not finite"] = bad
    spike = X.copy()
    spike[50] *= 1e9
    cases["spike"] = spike
    graded = vals * 10.0 ** rng.uniform(-12, 3, len(vals))
    rows = np.repeat(np.arange(pat.nblk), pat.block_sizes())
    zero = np.where(np.isin(pat.block_rows()[rows], (4, 5, 6)), 0.0, vals)
    for v in (vals, graded, zero):
        H = _handle(pat, v)
        for X in cases.values():
            with np.errstate(invalid="ignore", over="ignore"):
                _check(H, pat, v, np.ascontiguousarray(X))
    Xt = np.random.default_rng(1).standard_normal((pat.n_rows, k)) * np.exp(-np.arange(pat.n_rows) / 7.0)[:, None]
    _check(H, pat, zero, Xt, transpose=True)


def test_structures_of_a_batch_keep_their_own_scales():
    """A batched operator's structures are independent: one structure's huge panel leaves
    the bits of the others alone."""
    from paper_2609_04397_gb300 import VBCSR
    w = syn.batched_uneven(6, 600, 900, seed=3)
    offs = w.struct_brow_offsets
    rows = w.pattern.block_rows()
    local = w.pattern.block_col_idx - offs[np.searchsorted(offs, rows, side="right") - 1]
    H = VBCSR.from_batched(offs, offs, w.pattern.row_bsize, w.pattern.col_bsize, w.pattern.block_row_ptr, local,
                           w.values, torch.float64, "cuda:0")
    X = np.random.default_rng(2).standard_normal((w.pattern.n_cols, 16))
    Y = _check(H, w.pattern, w.values, X)
    cut = int(w.pattern.row_bsize[:offs[1]].sum())
    X2 = X.copy()
    X2[:cut] *= 1e7
    Y2 = _check(H, w.pattern, w.values, X2)
    assert np.array_equal(Y[cut:], Y2[cut:])


def test_tiles_follow_the_values():
    """Eager and captured changes of the values reach eager and captured products."""
    w = syn.amorphous(700, side=60.0 * (700 / 20000) ** (1 / 3))
    pat, k = w.pattern, 16
    rng = np.random.default_rng(1)
    X = rng.standard_normal((pat.n_cols, k))
    Xd = torch.from_numpy(X).cuda()
    v = [syn.random_values(pat, s) for s in range(5)]
    H = _handle(pat, v[0])
    Y = torch.empty(pat.n_rows, k, dtype=torch.float64, device="cuda:0")
    buf = torch.from_numpy(v[0]).cuda()

    def same(i, y=None):
        y = H.spmm(Xd) if y is None else y
        ref = oracle.spmm(pat, v[i], X)
        scale = oracle.spmm(pat, np.abs(v[i]), np.abs(X))
        assert (np.abs(y.cpu().numpy() - ref) <= TOL * scale).all()

    # a product captured before its tiles exist runs multiply-adds
    first = torch.cuda.CUDAGraph()
    with torch.cuda.graph(first):
        H.spmm(Xd, 1.0, 0.0, Y)
    first.replay()
    same(0, Y)
    same(0)
    H.set_values(torch.from_numpy(v[1]).cuda())
    same(1)
    first.replay()
    same(1, Y)
    H.set_values(torch.from_numpy(v[2]).cuda())          # stale tiles at capture
    prod = torch.cuda.CUDAGraph()
    with torch.cuda.graph(prod):
        H.spmm(Xd, 1.0, 0.0, Y)
    same(2)
    prod.replay()
    same(2, Y)
    H.set_values(torch.from_numpy(v[3]).cuda())
    prod.replay()
    same(3, Y)
    setv = torch.cuda.CUDAGraph()
    with torch.cuda.graph(setv):
        H.set_values(buf)
    same(3)
    buf.copy_(torch.from_numpy(v[4]))
    setv.replay()
    prod.replay()
    same(4, Y)
    same(4)
    # values changed by a capture before the adjoint's tiles exist
    G = rng.standard_normal((pat.n_rows, k))
    _check(H, pat, v[4], G, transpose=True)
    buf.copy_(torch.from_numpy(v[1]))
    setv.replay()
    _check(H, pat, v[1], G, transpose=True)


def test_captured_products_outlive_larger_ones():
    """A graph's buffers stay when a wider product, or a wider sampled one, needs larger ones."""
    w = syn.amorphous(700, side=60.0 * (700 / 20000) ** (1 / 3))
    pat = w.pattern
    H = _handle(pat, w.values)
    rng = np.random.default_rng(3)
    X, Xw = (rng.standard_normal((pat.n_cols, k)) for k in (16, 90))
    Xd, Xwd = torch.from_numpy(X).cuda(), torch.from_numpy(Xw).cuda()
    A, Aw = torch.randn_like(Xd[:pat.n_rows]), torch.randn_like(Xwd[:pat.n_rows])
    Y, D = H.spmm(Xd), H.sddmm(A, Xd)
    Yg, Dg = torch.empty_like(Y), torch.empty_like(D)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        H.spmm(Xd, 1.0, 0.0, Yg)
        H.sddmm(A, Xd, 1.0, 0.0, Dg)
    _check(H, pat, w.values, Xw)
    H.sddmm(Aw, Xwd)
    graph.replay()
    assert torch.equal(Yg, Y) and torch.equal(Dg, D)


@pytest.mark.parametrize("k", [6, 7, 16, 17, 40, 200])
def test_sliced_sddmm_against_oracle(k):
    """The pattern-sampled product, contracting over the panel columns: row heights 1 to 33,
    rows wider than the 512-column window, ragged tiles, leading dimensions above k, graded
    rows, rows whose large columns do not meet, zero rows, Inf and NaN."""
    pat = syn.random_pattern(230, 225, (1, 4, 9, 13, 33), 0.35, k, empty_rows=2, unsorted=True)
    assert pat.nnz * k >= 1 << 22
    H = _handle(pat, syn.random_values(pat, k))
    rng = np.random.default_rng(k)
    A0, B0 = rng.standard_normal((pat.n_rows, k + 1)), rng.standard_normal((pat.n_cols, k + 2))
    D0 = rng.standard_normal(pat.nnz)
    grade = 10.0 ** -np.arange(k + 2)
    for A, B in ((A0, B0), (A0 * 10.0 ** rng.uniform(-30, 30, (pat.n_rows, 1)), B0),
                 (A0 * np.clip(grade[:k + 1], 1e-30, None), B0 * np.clip(grade[k - 1::-1].tolist() + [1.0, 1.0], 1e-30, None))):
        A, B = A.copy(), B.copy()
        A[5] = 0.0
        B[7] = 0.0
        for alpha, beta in ((1.0, 0.0), (1.5, -0.5)):
            Ad, Bd = torch.from_numpy(A).cuda()[:, :k], torch.from_numpy(B).cuda()[:, :k]
            Dd = torch.from_numpy(D0.copy()).cuda()
            H.sddmm(Ad, Bd, alpha, beta, Dd)
            got = Dd.cpu().numpy()
            ref = oracle.sddmm(pat, A[:, :k], B[:, :k], alpha, beta, D0)
            scale = oracle.sddmm(pat, np.abs(A[:, :k]), np.abs(B[:, :k]), abs(alpha), 0.0) + abs(beta) * np.abs(D0)
            assert (np.abs(got - ref) <= TOL * scale).all(), np.max(np.abs(got - ref) / np.maximum(scale, 1e-300))
    A, B = A0.copy(), B0.copy()
    A[3, 0], A[40, 1], B[9, 1], B[5] = np.nan, np.inf, -np.inf, 0.0
    with np.errstate(invalid="ignore"):
        ref = oracle.sddmm(pat, A[:, :k], B[:, :k], 1.0, 0.0, None)
    got = H.sddmm(torch.from_numpy(A).cuda()[:, :k], torch.from_numpy(B).cuda()[:, :k]).cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
    assert any("slice_sddmm" in n for n in _kernels(lambda: H.sddmm(torch.from_numpy(A0).cuda()[:, :k],
                                                                    torch.from_numpy(B0).cuda()[:, :k])))


def test_fewest_columns():
    """Five columns, forward and adjoint, over every row height of a random pattern, with
    outputs that are not resolved; four are sliced in a recurrence only, two never."""
    pat = syn.random_pattern(430, 425, (1, 2, 4, 9, 13, 16, 33), 0.13, 3, empty_rows=2, unsorted=True)
    assert 8 * pat.nnz >= 1 << 24
    vals = syn.random_values(pat, 3)
    H = _handle(pat, vals)
    rng = np.random.default_rng(3)
    X = rng.standard_normal((pat.n_cols, 5))
    _check(H, pat, vals, X, alpha=-0.3, beta=2.0, Y0=rng.standard_normal((pat.n_rows, 5)))
    _check(H, pat, vals, rng.standard_normal((pat.n_rows, 5)), transpose=True)
    assert any("slice_product" in n for n in _kernels(lambda: H.spmm(torch.from_numpy(X).cuda())))
    assert not any("slice" in n for n in _kernels(lambda: H.spmm(torch.from_numpy(X[:, :4].copy()).cuda())))
    X[:, 1] *= np.exp(-np.arange(pat.n_cols) / 50.0)
    X[9, 0] = np.inf
    with np.errstate(invalid="ignore"):
        _check(H, pat, vals, X)
    w = syn.amorphous(700, side=60.0 * (700 / 20000) ** (1 / 3))
    H = _handle(w.pattern, w.values)
    lo, hi = H.gershgorin()
    H.shift_scale((lo + hi) / 2, 0.51 * (hi - lo))
    for k in (2, 3, 4):
        R = torch.randn(w.pattern.n_rows, k, dtype=torch.float64, device="cuda:0")
        sliced = any("slice_product" in n for n in _kernels(lambda: H.chebyshev(R, 5)))
        assert sliced == (k * w.pattern.nnz >= 1 << 22 and k > 2)
        mu, _ = H.chebyshev(R, 5)
        t = [R, H.spmm(R)]
        for _ in range(3):
            t.append(2.0 * H.spmm(t[-1]) - t[-2])
        ref = torch.stack([(R * x).sum() for x in t]) / R.numel()
        assert (mu - ref).abs().max().item() <= 1e-13 * ref[0].abs().item()


def test_small_items_are_not_sliced():
    """2 x 2 blocks, 40 a row: 160 entries a work item, too few for the digit products."""
    n = 14_000
    cols = np.sort((np.arange(n)[:, None] + 3 * np.arange(40)) % n, axis=1)
    pat = BlockPattern(np.full(n, 2), np.full(n, 2), np.arange(n + 1) * 40, cols.reshape(-1))
    assert 8 * pat.nnz >= 1 << 24
    vals = syn.random_values(pat, 1)
    H = _handle(pat, vals)
    X = np.random.default_rng(1).standard_normal((pat.n_cols, 8))
    _check(H, pat, vals, X)
    Xd = torch.from_numpy(X).cuda()
    assert not any("slice" in k for k in _kernels(lambda: (H.spmm(Xd), H.spmm_adjoint(Xd), H.sddmm(Xd, Xd))))


@pytest.mark.parametrize("k", [1, 3, 8, 13])
def test_sliced_complex_products(k):
    """A complex operator as two real virtual columns a value, forward and
    conjugate-transpose, at two k-points (the tiles follow the values), with the
    fused epilogue, and on a panel that is not resolved."""
    from paper_2609_04397_gb300 import VBCSR
    w = syn.zincblende_crystal(4)
    H = VBCSR.from_images(w.bsize, w.edge_i, w.edge_j, w.edge_R, w.edge_values, device="cuda:0")
    rb, cb, rp, ci = H.pattern
    pat = BlockPattern(rb, cb, rp, ci)
    rng = np.random.default_rng(k)

    def crandn(n):
        return rng.standard_normal((n, k)) + 1j * rng.standard_normal((n, k))

    X, Y0, Z, R = (crandn(pat.n_rows) for _ in range(4))
    local = X * np.exp(-np.arange(pat.n_rows) / 9.0)[:, None]
    for kp in ([0.13, -0.27, 0.41], [0.3, 0.2, -0.1]):
        H.set_kpoint(kp)
        vals = H.get_values().cpu().numpy()
        for P in (X, local):
            mag = oracle.spmm(pat, np.abs(vals), np.abs(P))
            Yd, dot = torch.from_numpy(Y0.copy()).cuda(), torch.zeros(1, dtype=torch.float64, device="cuda:0")
            H.spmm_ex(torch.from_numpy(P).cuda(), 2.0, -1.0, Yd, gamma=0.5, Z=torch.from_numpy(Z).cuda(),
                      R=torch.from_numpy(R).cuda(), dot_out=dot)
            ref = oracle.spmm_complex(pat, vals, P, 2.0, -1.0, Y0) + 0.5 * Z
            got = Yd.cpu().numpy()
            # four real products a complex one
            assert (np.abs(got - ref) <= 2 * TOL * (2 * mag + np.abs(Y0) + np.abs(Z))).all()
            assert abs(dot.item() - np.sum((np.conj(R) * got).real)) <= 1e-12 * np.sum(np.abs(R * got))
            ref = oracle.spmm_adjoint_complex(pat, vals, P, 1.0, 0.0, Y0)
            got = H.spmm_adjoint(torch.from_numpy(P).cuda()).cpu().numpy()
            assert (np.abs(got - ref) <= 2 * TOL * oracle.spmm_adjoint(pat, np.abs(vals), np.abs(P))).all()
    if k > 1:   # from this width the operator has enough work
        assert any("slice_product" in n for n in _kernels(lambda: H.spmm(torch.from_numpy(X).cuda())))


def test_shift_scale_divides_correctly_rounded():
    """(H - c I) / d by reciprocal and exact remainder equals the division bit for bit:
    random and hard quotients, zeros, infinities, NaN, values and divisors at the ends
    of the exponent range, a divisor with every significand bit set."""
    pat = syn.random_pattern(40, 40, (4, 9, 13), 0.4, 1)
    pat = BlockPattern(pat.row_bsize, pat.row_bsize, pat.block_row_ptr, pat.block_col_idx)
    rng = np.random.default_rng(0)
    n = pat.nnz
    vals = rng.standard_normal(n) * 2.0 ** rng.integers(-40, 40, n)
    vals[::7] = rng.integers(1, 1 << 53, len(vals[::7])).astype(np.float64)
    vals[:9] = [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e308, 2.2e-308, 1.0]
    for d in (3.0, 1.0 / 3.0, -7.7, np.pi, 1e-3, float.fromhex("0x1.fffffffffffffp+3"), float.fromhex("0x1.fffffffffffffp+0"),
              float.fromhex("0x1.0000000000001p+0"), 1e-300, 1e300, 4.0):
        H = _handle(pat, vals)
        H.shift_scale(0.0, d)
        with np.errstate(all="ignore"):
            ref = vals / d
        got = H.get_values().cpu().numpy()
        assert np.array_equal(got, ref, equal_nan=True), (d, (got != ref).sum())
