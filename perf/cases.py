"""The work whose speed is measured: what a user of the library has it do.

Every case is one call (or one short sequence) of the public Python API on an
atom-centred operator, with the structures of the repository's own workloads
(zinc-blende nanoparticles, disordered and uniformly random periodic systems,
batches of small structures, scalar graphs, periodic crystals). The patterns
are deterministic in the case; stored values and panels come from the seed.

A case is a dict of plain values:
  kind       spmm | matmul | chebyshev | kpm_grad | kspace
  structure  zincblende | disordered | uniform | batched | scalar | variable | crystal
  n          atoms asked for (batched: structures; crystal: cells along a side)
  k          panel columns
  precision  the library's name of the block-product arithmetic
and what one kind alone needs (dtype, transpose, epilogue, moments, every).
"""
import functools
import math

import numpy as np
import torch

from paper_2609_04397_gb300 import VBCSR, chebyshev_moments, vbcsr_matmul

DEV = "cuda"


def listed():
    return [
        # A small molecule-sized cell: one product of a few microseconds, where launches and latency count.
        {"name": "spmm_tiny_f64_k8", "kind": "spmm", "structure": "uniform", "n": 200, "k": 8, "dtype": "f64",
         "precision": "native", "transpose": False, "epilogue": False},
        # Matrix-vector product of a nanoparticle, the step of Lanczos and conjugate-gradient iterations.
        {"name": "spmv_zb50k_f64", "kind": "spmm", "structure": "zincblende", "n": 50000, "k": 1, "dtype": "f64",
         "precision": "native", "transpose": False, "epilogue": False},
        # The same operator on a wide panel, as in subspace iteration and filtering.
        {"name": "spmm_zb50k_f64_k32", "kind": "spmm", "structure": "zincblende", "n": 50000, "k": 32, "dtype": "f64",
         "precision": "native", "transpose": False, "epilogue": False},
        # Many block sizes (9 to 20) and an odd panel width, with the fused epilogue of a recurrence step.
        {"name": "spmm_variable_f64_k13_ex", "kind": "spmm", "structure": "variable", "n": 3000, "k": 13,
         "dtype": "f64", "precision": "native", "transpose": False, "epilogue": True},
        # A mixed-precision product wider than one 16-column tile.
        {"name": "spmm_zb50k_tf32x3_k24", "kind": "spmm", "structure": "zincblende", "n": 50000, "k": 24,
         "dtype": "f64", "precision": "tf32x3", "transpose": False, "epilogue": False},
        # Scalar operator (every block 1 x 1): the tight-binding graph with one orbital per site.
        {"name": "spmm_scalar_f64_k4", "kind": "spmm", "structure": "scalar", "n": 400000, "k": 4, "dtype": "f64",
         "precision": "native", "transpose": False, "epilogue": False},
        # 256 independent structures of uneven size in one operator, FP32: the batch of a learned Hamiltonian.
        {"name": "spmm_batched256_f32_k8", "kind": "spmm", "structure": "batched", "n": 256, "k": 8, "dtype": "f32",
         "precision": "native", "transpose": False, "epilogue": False},
        # One training step through a product: new values set, forward, adjoint and pattern-sampled gradient.
        {"name": "matmul_grad_dis20k_f64_k16", "kind": "matmul", "structure": "disordered", "n": 20000, "k": 16,
         "precision": "native"},
        # The FP64 recurrence of the kernel polynomial method, with checkpoints.
        {"name": "chebyshev_zb100k_f64_k16", "kind": "chebyshev", "structure": "zincblende", "n": 100000, "k": 16,
         "precision": "native", "moments": 8, "every": 4},
        # The same recurrence at scale with tensor-core block products.
        {"name": "chebyshev_zb200k_bf16x2_k16", "kind": "chebyshev", "structure": "zincblende", "n": 200000, "k": 16,
         "precision": "bf16x2", "moments": 11, "every": 8},
        # Differentiable moments of a predicted operator: recurrence, reverse recurrence, value gradient.
        {"name": "kpm_grad_dis20k_f64_k8", "kind": "kpm_grad", "structure": "disordered", "n": 20000, "k": 8,
         "precision": "native", "moments": 30, "every": 10},
        # A periodic crystal sampled at a k-point and multiplied (complex).
        {"name": "kspace_crystal12_c128_k8", "kind": "kspace", "structure": "crystal", "n": 12, "k": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges (sizes log-uniform, odd widths among them)."""
    kind = rng.choice(["spmm"] * 5 + ["matmul", "chebyshev", "chebyshev", "kpm_grad", "kspace"])
    if kind == "spmm":
        s = rng.choice(["uniform", "zincblende", "zincblende", "disordered", "variable", "batched", "scalar"])
        n = {"uniform": lambda: _log(rng, 150, 6000), "zincblende": lambda: _log(rng, 500, 60000),
             "disordered": lambda: _log(rng, 400, 30000), "variable": lambda: _log(rng, 300, 8000),
             "batched": lambda: _log(rng, 4, 256), "scalar": lambda: _log(rng, 3000, 400000)}[s]()
        dtype = "f32" if s == "batched" else rng.choice(["f64", "f64", "f64", "f32"])
        prec = "native" if dtype == "f32" else rng.choice(["native"] * 4 + ["f32", "tf32x3", "bf16x2", "df32"])
        k = rng.choice([1, 2, 3, 4, 5, 7, 8, 12, 13, 16, 21, 24, 31, 32])
        return {"kind": kind, "structure": s, "n": n, "k": k, "dtype": dtype, "precision": prec,
                "transpose": rng.random() < 0.3, "epilogue": dtype == "f64" and rng.random() < 0.3}
    if kind == "matmul":
        s = rng.choice(["disordered", "zincblende", "uniform"])
        n = _log(rng, 500, 20000) if s != "uniform" else _log(rng, 200, 6000)
        return {"kind": kind, "structure": s, "n": n, "k": rng.choice([1, 4, 8, 11, 16, 32]), "precision": "native"}
    if kind == "chebyshev":
        prec = rng.choice(["native", "native", "bf16x2", "tf32x3"])
        return {"kind": kind, "structure": "zincblende", "n": _log(rng, 1000, 100000),
                "k": rng.choice([4, 8, 9, 16]), "precision": prec, "moments": rng.randint(4, 9), "every": 4}
    if kind == "kpm_grad":
        return {"kind": kind, "structure": rng.choice(["disordered", "zincblende"]), "n": _log(rng, 500, 12000),
                "k": rng.choice([3, 4, 8, 16]), "precision": "native", "moments": rng.randint(8, 30), "every": 10}
    return {"kind": kind, "structure": "crystal", "n": rng.randint(3, 12), "k": rng.choice([1, 4, 7, 8])}


# ----------------------------------------------------------------------------
# patterns (deterministic in the case)


class Pattern:
    """Block sizes, row pointer, sorted columns and a scale per block (numpy)."""

    def __init__(self, bsize, i, j, scale, offsets=None):
        n = len(bsize)
        self.bsize = np.ascontiguousarray(bsize, np.int32)
        self.i, self.j = i.astype(np.int64), j.astype(np.int32)
        self.ptr = np.zeros(n + 1, np.int64)
        np.cumsum(np.bincount(i, minlength=n), out=self.ptr[1:])
        self.off = np.zeros(n + 1, np.int64)
        np.cumsum(self.bsize, out=self.off[1:])
        size = self.bsize[self.i].astype(np.int64) * self.bsize[self.j]
        self.voff = np.zeros(len(i) + 1, np.int64)
        np.cumsum(size, out=self.voff[1:])
        self.rows, self.nnz, self.nblk = int(self.off[-1]), int(self.voff[-1]), len(i)
        # entries N(0, 1) / sqrt(entries of the row) unless the structure gives its own decay
        if scale is None:
            per = np.bincount(i, weights=self.bsize[self.j].astype(np.float64), minlength=n)
            scale = (per[self.i] * per[self.j]) ** -0.25
        self.scale = scale
        self.offsets = offsets          # batched: first atom of every structure


def _spread(v):
    v = v.astype(np.uint64) & np.uint64(0x1FFFFF)
    for s, m in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F), (4, 0x10C30C30C30C30C3),
                 (2, 0x1249249249249249)):
        v = (v | (v << np.uint64(s))) & np.uint64(m)
    return v


def _morton(pos):
    q = np.floor(pos - pos.min(axis=0)).astype(np.int64)
    return np.argsort(_spread(q[:, 0]) | (_spread(q[:, 1]) << np.uint64(1)) | (_spread(q[:, 2]) << np.uint64(2)),
                      kind="stable")


def _zincblende(n):
    """Spherical cluster, cation b = 13 and anion b = 9, blocks to the third shell; entries exp(-r / 2 A)."""
    a = 5.87
    radius = 4.0 * (3.0 * n / (32.0 * math.pi)) ** (1.0 / 3.0)          # in units of a / 4
    m = int(math.ceil(radius / 4.0)) + 1
    r = 4 * np.arange(-m, m + 1)
    cells = np.stack(np.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 1, 3)
    cat = (cells + np.array([[0, 0, 0], [0, 2, 2], [2, 0, 2], [2, 2, 0]])).reshape(-1, 3)
    pos = np.concatenate([cat, cat + 1])
    bs = np.concatenate([np.full(len(cat), 13), np.full(len(cat), 9)])
    keep = (pos * pos).sum(1) <= radius * radius
    pos, bs = pos[keep], bs[keep]
    order = _morton(pos * (a / 4.0))
    pos, bs = pos[order], bs[order]
    side = int(pos.max() - pos.min()) + 9
    q = torch.from_numpy(pos - pos.min(axis=0) + 4).to(DEV)
    grid = torch.full((side, side, side), -1, dtype=torch.int64, device=DEV)
    grid[q[:, 0], q[:, 1], q[:, 2]] = torch.arange(len(pos), device=DEV)
    ii, jj, dd = [], [], []
    for x in range(-3, 4):
        for y in range(-3, 4):
            for z in range(-3, 4):
                d2 = x * x + y * y + z * z
                if d2 in (0, 3, 8, 11):
                    nb = grid[q[:, 0] + x, q[:, 1] + y, q[:, 2] + z]
                    at = torch.nonzero(nb >= 0).squeeze(1)
                    ii.append(at)
                    jj.append(nb[at])
                    dd.append(torch.full((len(at),), math.sqrt(d2) * a / 4.0, dtype=torch.float64, device=DEV))
    ii, jj, dd = torch.cat(ii), torch.cat(jj), torch.cat(dd)
    o = torch.argsort(ii * len(pos) + jj)
    return Pattern(bs, ii[o].cpu().numpy(), jj[o].cpu().numpy(), torch.exp(-dd[o] / 2.0).cpu().numpy())


def _pairs(pos, side, cutoff):
    """(i, j) of every pair closer than the cutoff in a periodic cube, and (i, i), sorted."""
    n = len(pos)
    p = torch.from_numpy(pos).to(DEV)
    nc = int(side / cutoff)
    if nc < 4:
        d = p[:, None, :] - p[None, :, :]
        d -= side * torch.round(d / side)
        near = (d * d).sum(-1) < cutoff * cutoff
        ij = torch.nonzero(near)
        return ij[:, 0].cpu().numpy(), ij[:, 1].cpu().numpy()
    c = torch.clamp((p * (nc / side)).long(), 0, nc - 1)
    cell = (c[:, 0] * nc + c[:, 1]) * nc + c[:, 2]
    order = torch.argsort(cell)
    count = torch.bincount(cell, minlength=nc ** 3)
    start = torch.cumsum(count, 0) - count
    ii, jj = [], []
    for x in (-1, 0, 1):
        for y in (-1, 0, 1):
            for z in (-1, 0, 1):
                o = (((c[:, 0] + x) % nc) * nc + (c[:, 1] + y) % nc) * nc + (c[:, 2] + z) % nc
                cnt = count[o]
                i = torch.repeat_interleave(torch.arange(n, device=DEV), cnt)
                at = torch.arange(len(i), device=DEV) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
                j = order[start[o][i] + at]
                d = p[i] - p[j]
                d -= side * torch.round(d / side)
                near = (d * d).sum(1) < cutoff * cutoff
                ii.append(i[near])
                jj.append(j[near])
    ii, jj = torch.cat(ii), torch.cat(jj)
    o = torch.argsort(ii * n + jj)
    return ii[o].cpu().numpy(), jj[o].cpu().numpy()


def _uniform_pos(rng, n, density):
    side = (n / density) ** (1.0 / 3.0)
    pos = rng.uniform(0.0, side, size=(n, 3))
    return pos[_morton(pos)], side


def _species(rng, n, sizes, parts):
    counts = [int(round(f * n)) for f in parts]
    counts[-1] = n - sum(counts[:-1])
    return rng.permutation(np.repeat(sizes, counts))


@functools.lru_cache(maxsize=4)
def _pattern(structure, n):
    rng = np.random.default_rng(n)
    if structure == "zincblende":
        return _zincblende(n)
    if structure == "disordered":
        # n atoms on a displaced lattice at 0.0926 per cubic Angstrom, b in {4, 9, 13} at 40/40/20 %, 4.5 A cutoff
        side = (n / 0.0926) ** (1.0 / 3.0)
        m = int(math.ceil(n ** (1.0 / 3.0) - 1e-9))
        g = (np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5) * (side / m)
        pos = g[np.sort(rng.permutation(len(g))[:n])]
        pos = np.mod(pos + rng.uniform(-0.25, 0.25, size=pos.shape), side)
        pos = pos[_morton(pos)]
        i, j = _pairs(pos, side, 4.5)
        return Pattern(_species(rng, n, [4, 9, 13], [0.4, 0.4, 0.2]), i, j, None)
    if structure == "batched":
        # n periodic structures of 50 to 2000 atoms (log-uniform), b in {4, 9, 13} in equal parts, 5 A cutoff
        sizes = np.rint(np.exp(rng.uniform(math.log(50), math.log(2000), size=n))).astype(int)
        off = np.concatenate([[0], np.cumsum(sizes)])
        ii, jj, bs = [], [], []
        for s, m in enumerate(sizes):
            pos, side = _uniform_pos(rng, int(m), 0.0488)
            i, j = _pairs(pos, side, 5.0)
            ii.append(i + off[s])
            jj.append(j + off[s])
            bs.append(_species(rng, int(m), [4, 9, 13], [1 / 3, 1 / 3, 1 / 3]))
        return Pattern(np.concatenate(bs), np.concatenate(ii), np.concatenate(jj), None, off.astype(np.int64))
    # uniformly random positions at 0.0488 per cubic Angstrom, 5 A cutoff
    pos, side = _uniform_pos(rng, n, 0.0488)
    i, j = _pairs(pos, side, 5.0)
    if structure == "scalar":
        b = np.ones(n, np.int32)
    elif structure == "variable":
        b = rng.integers(9, 21, size=n)
    else:
        b = _species(rng, n, [4, 9], [0.5, 0.5])
    return Pattern(b, i, j, None)


@functools.lru_cache(maxsize=2)
def _crystal(n):
    """Images of a periodic zinc-blende crystal of n^3 cells (n >= 2: one image per pair): (bsize, i, j, R, scale)."""
    r = 4 * np.arange(n)
    cells = np.stack(np.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 1, 3)
    cat = (cells + np.array([[0, 0, 0], [0, 2, 2], [2, 0, 2], [2, 2, 0]])).reshape(-1, 3)
    pos = np.concatenate([cat, cat + 1])
    bs = np.concatenate([np.full(len(cat), 13, np.int32), np.full(len(cat), 9, np.int32)])
    L = 4 * n
    grid = np.full((L, L, L), -1, np.int64)
    grid[tuple(pos.T)] = np.arange(len(pos))
    ii, jj, RR, dd = [], [], [], []
    for x in range(-3, 4):
        for y in range(-3, 4):
            for z in range(-3, 4):
                d2 = x * x + y * y + z * z
                if d2 in (0, 3, 8, 11):
                    q = pos + np.array([x, y, z])
                    nb = grid[tuple((q % L).T)]
                    at = np.nonzero(nb >= 0)[0]
                    ii.append(at)
                    jj.append(nb[at])
                    RR.append((q // L)[at])
                    dd.append(np.full(len(at), math.sqrt(d2) * 5.87 / 4.0))
    ii, jj, RR, dd = np.concatenate(ii), np.concatenate(jj), np.concatenate(RR), np.concatenate(dd)
    o = np.lexsort((jj, ii))
    return bs, ii[o], jj[o], RR[o].astype(np.int32), np.exp(-dd[o] / 2.0)


# ----------------------------------------------------------------------------
# values and panels (from the seed)


def _hash(x, key):
    """SplitMix64 finaliser of a counter (int64 arithmetic wraps)."""
    def shr(v, s):
        return (v >> s) & ((1 << (64 - s)) - 1)
    x = x * -7046029254386353131 + key
    x = (x ^ shr(x, 30)) * -4658895280553007687
    x = (x ^ shr(x, 27)) * -7723592293110705685
    return shr(x ^ shr(x, 31), 11)                              # 53 bits


def _normal(index, seed):
    u = (_hash(index, 2 * seed + 1).double() + 0.5) * 2.0 ** -53
    v = _hash(index, 2 * seed + 1000003).double() * 2.0 ** -53
    return torch.sqrt(-2.0 * torch.log(u)) * torch.cos(2.0 * math.pi * v)


def _values(p, seed, chunk=1 << 25):
    """Packed FP64 values of a symmetric operator: N(0, 1) by the (row, column) pair, times the block's scale."""
    out = torch.empty(p.nnz, dtype=torch.float64, device=DEV)
    bi, bj = torch.from_numpy(p.bsize[p.i]).to(DEV), torch.from_numpy(p.bsize[p.j]).to(DEV)
    ri, cj = torch.from_numpy(p.off[p.i]).to(DEV), torch.from_numpy(p.off[p.j]).to(DEV)
    sc, vo = torch.from_numpy(p.scale).to(DEV), torch.from_numpy(p.voff).to(DEV)
    u0 = 0
    while u0 < p.nblk:
        u1 = min(p.nblk, max(u0 + 1, int(np.searchsorted(p.voff, p.voff[u0] + chunk, side="right")) - 1))
        e0, e1 = int(p.voff[u0]), int(p.voff[u1])
        u = torch.repeat_interleave(torch.arange(u0, u1, device=DEV), vo[u0 + 1:u1 + 1] - vo[u0:u1], output_size=e1 - e0)
        q = torch.arange(e0, e1, device=DEV) - vo[u]
        w = bj[u].long()
        r, c = ri[u] + q // w, cj[u] + q % w
        lo, hi = torch.minimum(r, c), torch.maximum(r, c)
        out[e0:e1] = _normal(lo * p.rows + hi, seed) * sc[u]
        u0 = u1
    return out


def _panel(rows, k, seed, stream, dtype=torch.float64):
    g = torch.Generator(device=DEV).manual_seed(1000 * seed + stream)
    return torch.randn(rows, k, dtype=torch.float64, device=DEV, generator=g).to(dtype)


def _signs(rows, k, seed):
    g = torch.Generator(device=DEV).manual_seed(1000 * seed + 7)
    return torch.randint(0, 2, (rows, k), device=DEV, generator=g).double() * 2.0 - 1.0


def _row_sum(p, v):
    """The largest absolute row sum: a bound of the spectrum."""
    s = torch.zeros(p.rows, dtype=torch.float64, device=DEV)
    for u, bi, bj in _classes(p):
        s.index_add_(0, _rows(p.off[p.i[u]], bi).reshape(-1), _blocks(p, v, u, bi, bj).abs().sum(2).reshape(-1))
    return float(s.max())


def _operator(p, v, dtype):
    if p.offsets is None:
        return VBCSR.from_arrays(p.bsize, p.bsize, p.ptr, p.j, v, dtype, DEV)
    local = (p.j - p.offsets[np.searchsorted(p.offsets, p.i, side="right") - 1]).astype(np.int32)
    return VBCSR.from_batched(p.offsets, p.offsets, p.bsize, p.bsize, p.ptr, local, v, dtype, DEV)


def _inputs(c, seed):
    """Values and panels of a case, as both prepare and exact start from."""
    k = c["k"]
    if c["kind"] == "kspace":
        bs, i, j, R, scale = _crystal(c["n"])
        n = int((bs[i].astype(np.int64) * bs[j]).sum())
        g = torch.Generator(device=DEV).manual_seed(1000 * seed + 1)
        per = torch.from_numpy(np.repeat(scale, bs[i].astype(np.int64) * bs[j])).to(DEV)
        v = torch.randn(n, dtype=torch.float64, device=DEV, generator=g) * per
        rows = int(bs.sum())
        X = torch.complex(_panel(rows, k, seed, 2), _panel(rows, k, seed, 3))
        q = np.random.default_rng(seed).uniform(0.0, 1.0, 3)
        return (bs, i, j, R), v, {"X": X, "q": q}
    p = _pattern(c["structure"], c["n"])
    v = _values(p, seed)
    if c["kind"] == "spmm":
        dt = torch.float32 if c["dtype"] == "f32" else torch.float64
        t = {"X": _panel(p.rows, k, seed, 2, dt)}
        if c["epilogue"]:
            t |= {"Z": _panel(p.rows, k, seed, 3, dt), "R": _panel(p.rows, k, seed, 4, dt)}
        return p, v.to(dt), t
    if c["kind"] == "matmul":
        return p, v, {"X": _panel(p.rows, k, seed, 2), "dY": _panel(p.rows, k, seed, 3)}
    d = 1.01 * _row_sum(p, v)
    if c["kind"] == "chebyshev":
        return p, v / d, {"X": _signs(p.rows, k, seed)}
    return p, v, {"X": _signs(p.rows, k, seed), "d": d, "c": 0.01 * d}


def prepare(case, seed):
    p, v, t = _inputs(case, seed)
    s = dict(t, case=case)
    if case["kind"] == "kspace":
        bs, i, j, R = p
        s["H"] = VBCSR.from_images(bs, i, j, R, v.cpu().numpy(), device=DEV)
        return s
    s["H"] = _operator(p, v, v.dtype)
    if case["kind"] in ("matmul", "kpm_grad"):
        s["v"] = v.requires_grad_(True)
    if case["kind"] == "matmul":
        s["X"].requires_grad_(True)
    if case["kind"] == "spmm" and case["epilogue"]:
        s["Y"] = torch.empty_like(s["Z"])
        s["dot"] = torch.empty(1, dtype=torch.float64, device=DEV)
    return s


def run(s):
    c, H = s["case"], s["H"]
    if c["kind"] == "kspace":
        H.set_kpoint(s["q"])
        return H.spmm(s["X"])
    if c["kind"] == "spmm":
        if c["epilogue"]:
            Y = H.spmm_ex(s["X"], 2.0, 0.0, s["Y"], transpose=c["transpose"], gamma=-1.0, Z=s["Z"], R=s["R"],
                          dot_out=s["dot"], precision=c["precision"])
            return {"Y": Y, "dot": s["dot"]}
        fn = H.spmm_adjoint if c["transpose"] else H.spmm
        return fn(s["X"], precision=c["precision"])
    if c["kind"] == "matmul":
        Y = vbcsr_matmul(H, s["v"], s["X"], c["precision"])
        dv, dX = torch.autograd.grad(Y, (s["v"], s["X"]), s["dY"])
        return {"Y": Y.detach(), "dvalues": dv, "dX": dX}
    if c["kind"] == "chebyshev":
        mu, ck = H.chebyshev(s["X"], c["moments"], ckpt_every=c["every"], precision=c["precision"])
        return {"moments": mu, "checkpoints": ck}
    mu = chebyshev_moments(H, s["v"], s["X"], c["moments"], c["every"], c["precision"], c=s["c"], d=s["d"])
    dv, = torch.autograd.grad((mu * mu).sum(), (s["v"],))
    return {"moments": mu.detach(), "dvalues": dv}


def work(case):
    """Bytes: stored values and one column index per block once, panels read and written once (per product of a
    recurrence); flops: 2 per stored entry and column of every product (8 for complex)."""
    k, kind = case["k"], case["kind"]
    if kind == "kspace":
        bs, i, j, _, _ = _crystal(case["n"])
        nnz, rows = int((bs[i].astype(np.int64) * bs[j]).sum()), int(bs.sum())
        return {"bytes": 8 * nnz + 16 * len(i) + 2 * 16 * rows * k, "flops": 4 * nnz + 8 * nnz * k}
    p = _pattern(case["structure"], case["n"])
    e = 4 if case.get("dtype") == "f32" else 8
    # a mixed mode reads the values in its own format (4 bytes)
    ev = 4 if case["precision"] in ("f32", "tf32", "tf32x3", "bf16x2") else e
    one = ev * p.nnz + 4 * p.nblk
    panel = e * p.rows * k
    if kind == "spmm":
        return {"bytes": one + (4 if case["epilogue"] else 2) * panel, "flops": 2 * p.nnz * k}
    if kind == "matmul":
        # values in, X in, Y out; dY in, dX out, the gradient of the values out
        return {"bytes": 8 * p.nnz + 2 * panel + 8 * p.nnz + 2 * panel, "flops": 6 * p.nnz * k}
    m = case["moments"]
    if kind == "chebyshev":
        ck = 2 * -(-(m - 1) // case["every"])
        return {"bytes": (m - 1) * (one + 4 * panel) + ck * panel, "flops": 2 * p.nnz * k * (m - 1)}
    # recurrence, reverse recurrence and the sampled gradient over all steps
    return {"bytes": 2 * (m - 1) * (one + 4 * panel) + 8 * p.nnz, "flops": 2 * p.nnz * k * 3 * (m - 1)}


# ----------------------------------------------------------------------------
# the same results in plain 64-bit torch


def _classes(p, most=1 << 25):
    """(block indices, b_i, b_j) of equal-shaped blocks, in pieces."""
    bi, bj = p.bsize[p.i].astype(np.int64), p.bsize[p.j].astype(np.int64)
    key = bi * 100000 + bj
    order = np.argsort(key, kind="stable")
    kk = key[order]
    cut = np.concatenate([[0], np.nonzero(np.diff(kk))[0] + 1, [len(kk)]])
    for a, b in zip(cut[:-1], cut[1:]):
        x, y = int(bi[order[a]]), int(bj[order[a]])
        step = max(1, most // (x * y))
        for s in range(a, b, step):
            yield order[s:min(b, s + step)], x, y


def _rows(first, b):
    return torch.from_numpy(first).to(DEV)[:, None] + torch.arange(b, device=DEV)


def _blocks(p, v, u, bi, bj):
    at = torch.from_numpy(p.voff[u]).to(DEV)[:, None] + torch.arange(bi * bj, device=DEV)
    return v[at.reshape(-1)].reshape(len(u), bi, bj)


def _apply(p, v, X, transpose=False):
    """H X or H^T X, block by block in the width of X."""
    Y = torch.zeros(p.rows, X.shape[1], dtype=X.dtype, device=DEV)
    for u, bi, bj in _classes(p, max(1 << 16, (1 << 27) // X.shape[1])):
        B = _blocks(p, v, u, bi, bj)
        ri, cj = _rows(p.off[p.i[u]], bi), _rows(p.off[p.j[u]], bj)
        if transpose:
            ri, cj, B = cj, ri, B.transpose(1, 2)
        Y.index_add_(0, ri.reshape(-1), torch.bmm(B, X[cj]).reshape(-1, X.shape[1]))
    return Y


def _sample(p, A, B):
    """A[rows_i] B[cols_j]^T on the stored blocks, packed."""
    D = torch.empty(p.nnz, dtype=torch.float64, device=DEV)
    for u, bi, bj in _classes(p, max(1 << 16, (1 << 26) // max(1, A.shape[1] // 4))):
        at = torch.from_numpy(p.voff[u]).to(DEV)[:, None] + torch.arange(bi * bj, device=DEV)
        blk = torch.bmm(A[_rows(p.off[p.i[u]], bi)], B[_rows(p.off[p.j[u]], bj)].transpose(1, 2))
        D[at.reshape(-1)] = blk.reshape(-1)
    return D


def exact(case, seed):
    p, v, t = _inputs(case, seed)
    X, kind = t["X"], case["kind"]
    if kind == "kspace":
        bs, i, j, R = p
        q = Pattern(bs, i, j, np.ones(len(i)))
        # n >= 3: every pair has one image, so the edges are the blocks
        ph = torch.from_numpy(np.exp(-2j * np.pi * (R.astype(np.float64) @ t["q"]))).to(DEV)
        size = torch.from_numpy(np.diff(q.voff)).to(DEV)
        return _apply(q, v * torch.repeat_interleave(ph, size), X)
    v, X = v.double(), X.double()
    if kind == "spmm":
        Y = _apply(p, v, X, case["transpose"])
        if not case["epilogue"]:
            return Y
        Y = 2.0 * Y - t["Z"].double()
        return {"Y": Y, "dot": (t["R"].double() * Y).sum().reshape(1)}
    if kind == "matmul":
        return {"Y": _apply(p, v, X), "dvalues": _sample(p, t["dY"], X), "dX": _apply(p, v, t["dY"], True)}
    m, every = case["moments"], case["every"]
    h = v
    if kind == "kpm_grad":
        h = v / t["d"]
    shift = t["c"] / t["d"] if kind == "kpm_grad" else 0.0

    def ham(x, transpose=False):
        y = _apply(p, h, x, transpose)
        return y - shift * x if shift else y

    scale = 1.0 / X.numel()
    T = [X, ham(X)]
    for _ in range(2, m):
        T.append(2.0 * ham(T[-1]) - T[-2])
    mu = torch.stack([(X * x).sum() * scale for x in T[:m]])
    if kind == "chebyshev":
        ck = torch.stack([torch.stack([T[a], T[a + 1]]) for a in range(0, m - 1, every)])
        return {"moments": mu, "checkpoints": ck}
    g = 2.0 * mu * scale
    D = torch.zeros(p.nnz, dtype=torch.float64, device=DEV)
    lam, nxt = g[m - 1] * X, torch.zeros_like(X)
    for n in range(m - 2, -1, -1):
        D += _sample(p, (2.0 if n else 1.0) * lam, T[n])
        if n:
            lam, nxt = g[n] * X + 2.0 * ham(lam, True) - nxt, lam
    return {"moments": mu, "dvalues": D / t["d"]}
