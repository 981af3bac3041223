"""The work a user of this framework has it do, as cases that can be timed and compared.

Every matrix is one of the covariance matrices the framework is made for: uniform random points in
the unit square or cube, a KD cluster tree, Chebyshev interpolation bases, coupling blocks from the
kernel at the interpolation points and dense near-field blocks from the kernel at the points. The
arrays are formed here, in plain torch FP64 from their definitions (`covariance`), and handed to the
framework's entry points, so that `exact` can multiply the same arrays without the framework.

Kinds:
  product   y = A x with a stored matrix: FP64 vectors on the FP64 form, FP32 vectors on the scaled
            16-bit forms (whose arithmetic is FP32)
  kernel    the same with the coupling blocks evaluated from the kernel in each product and the
            dense blocks generated on the device (how the largest 3D problems fit)
  batch     many independent matrices of uneven size in one call
  compress  compression of the far field to a threshold, its result made into a matrix, one product
  build     construction of the tree, block structure and bases on the device from the points
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1902_01829_gb300 as h2

DEV = "cuda:0"


# ------------------------------------------------------------------------------- the cases
def listed():
    return [
        # one vector through an oracle-sized matrix: the smallest call, latency and launches
        dict(name="fp64_small", kind="product", dim=2, n=4096, m=32, p=4, eta=0.9, kernel="exp", ell=0.1,
             storage="fp64", bases_fp32=False, nv=1),
        # the headline product (2D, 64-point leaves, rank 16, one FP64 vector), the matrix far larger than L2
        dict(name="fp64_one", kind="product", dim=2, n=131072, m=64, p=4, eta=0.9, kernel="exp", ell=0.1,
             storage="fp64", bases_fp32=False, nv=1),
        # a block of vectors (block solver, sampling) with ragged leaves
        dict(name="fp64_block", kind="product", dim=2, n=50001, m=64, p=4, eta=0.9, kernel="exp", ell=0.1,
             storage="fp64", bases_fp32=False, nv=16),
        # 3D, rank 64: most of the bytes are coupling blocks
        dict(name="fp64_3d", kind="product", dim=3, n=16384, m=64, p=4, eta=0.9, kernel="exp", ell=0.2,
             storage="fp64", bases_fp32=False, nv=1),
        # the precision form at its recommended accuracy, one vector (an iterative solver's inner product)
        dict(name="int16_one", kind="product", dim=2, n=131072, m=64, p=4, eta=0.9, kernel="exp", ell=0.1,
             storage="int16", bases_fp32=True, nv=1),
        # the same form with many vectors (vectors/s)
        dict(name="int16_block", kind="product", dim=2, n=65536, m=64, p=4, eta=0.9, kernel="exp", ell=0.1,
             storage="int16", bases_fp32=True, nv=64),
        # fp16 codes and 16-bit bases, a block of vectors, 64-point leaves
        dict(name="fp16_block", kind="product", dim=2, n=65536, m=64, p=4, eta=0.9, kernel="exp", ell=0.1,
             storage="fp16", bases_fp32=False, nv=32),
        # bf16 in 3D at rank 64, a block of vectors
        dict(name="bf16_3d", kind="product", dim=3, n=16384, m=64, p=4, eta=0.9, kernel="exp", ell=0.2,
             storage="bf16", bases_fp32=False, nv=16),
        # 3D problems too large to store: coupling from the kernel, dense blocks generated
        dict(name="kernel_3d", kind="kernel", dim=3, n=65536, m=64, p=4, eta=0.9, kernel="exp", ell=0.2,
             storage="int16", bases_fp32=True, nv=8),
        # independent matrices of uneven size and uneven vector counts, 32-point leaves, fp16
        dict(name="batch", kind="batch", count=32, n_lo=1024, n_hi=16384, m=32, p=4, eta=0.9, kernel="exp", ell=0.1,
             storage="fp16", bases_fp32=False),
        # the paper's 3D compression problem (threshold 1e-3)
        dict(name="compress_3d", kind="compress", dim=3, n=8192, m=64, p=4, eta=0.9, kernel="exp", ell=0.2, eps=1e-3),
        # construction from the points: tree, block structure, bases
        dict(name="build", kind="build", dim=2, n=200000, m=64, p=4, eta=0.9, kernel="exp", ell=0.1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product"] * 5 + ["kernel", "batch", "compress", "build"])
    dim = rng.choice([2, 2, 3])
    ell = 0.1 if dim == 2 else 0.2
    if kind == "product":
        storage, bases = rng.choice([("fp64", False), ("fp64", False), ("int16", True), ("fp16", False), ("bf16", False),
                                     ("fp16", True)])
        nv = rng.choice([1, 1, 2, 3, 4, 6, 8, 13, 16] + ([] if storage == "fp64" else [32, 64]))
        p = rng.choice([4, 4, 4, 3])
        hi = (16384 if p == 4 else 32768) if dim == 3 else (131072 if nv <= 4 else 50001 if storage == "fp64" else 65536)
        n = _log_int(rng, 1000, hi)
        if rng.random() < 0.25:
            n = 1 << max(10, min(n.bit_length() - 1, 17))  # full, equal leaves
        return dict(kind=kind, dim=dim, n=n, m=rng.choice([64, 64, 32]) if dim == 2 else 64, p=p, eta=0.9, kernel="exp",
                    ell=ell, storage=storage, bases_fp32=bases, nv=nv)
    if kind == "kernel":
        storage, bases = rng.choice([("int16", True), ("fp16", False)])
        return dict(kind=kind, dim=dim, n=_log_int(rng, 4000, 65536), m=64, p=rng.choice([4, 4, 3]), eta=rng.choice([0.9, 0.7]),
                    kernel=rng.choice(["exp", "matern32"]), ell=ell, storage=storage, bases_fp32=bases,
                    nv=rng.choice([1, 2, 4, 8]))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 32), n_lo=1024, n_hi=_log_int(rng, 2048, 16384), m=rng.choice([32, 32, 64]),
                    p=4, eta=0.9, kernel="exp", ell=0.1, storage=rng.choice(["fp16", "bf16", "int16"]), bases_fp32=False)
    if kind == "compress":
        return dict(kind=kind, dim=dim, n=_log_int(rng, 2000, 8192), m=64, p=8 if dim == 2 else 4, eta=0.9, kernel="exp",
                    ell=ell, eps=1e-7 if dim == 2 else 1e-3)
    return dict(kind=kind, dim=dim, n=_log_int(rng, 8192, 200000), m=rng.choice([32, 64]), p=4, eta=0.9, kernel="exp", ell=ell)


# ------------------------------------------------------------------------------- the matrices
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _kernel(kind, ell, r):
    if kind == "exp":
        return torch.exp(-r / ell)
    s = math.sqrt(3.0) * r / ell
    return (1.0 + s) * torch.exp(-s)


def _dist(X, Y):
    """Distances of points X (b, r, dim) and Y (b, c, dim): (b, r, c)."""
    r2 = torch.zeros(X.shape[0], X.shape[1], Y.shape[1], dtype=torch.float64, device=X.device)
    for d in range(X.shape[2]):
        r2 += (X[:, :, None, d] - Y[:, None, :, d]) ** 2
    return torch.sqrt(r2)


def _lagrange(xi, t):
    """Tensor Lagrange polynomials of the nodes xi (b, dim, p) at the points t (b, r, dim): (b, r, p^dim),
    dimension 0 slowest."""
    b, dim, p = xi.shape
    out = torch.ones(b, t.shape[1], 1, dtype=torch.float64, device=t.device)
    for d in range(dim):
        cols = []
        for a in range(p):
            v = torch.ones_like(t[:, :, d])
            for c in range(p):
                if c != a:
                    v = v * (t[:, :, d] - xi[:, d, c, None]) / (xi[:, d, a, None] - xi[:, d, c, None])
            cols.append(v)
        out = (out[:, :, :, None] * torch.stack(cols, 2)[:, :, None, :]).reshape(b, t.shape[1], -1)
    return out


def _grid(xi):
    """Interpolation points of the nodes xi (b, dim, p): (b, p^dim, dim), dimension 0 slowest."""
    b, dim, p = xi.shape
    idx = torch.arange(p ** dim, device=xi.device)
    return torch.stack([xi[:, d, (idx // p ** (dim - 1 - d)) % p] for d in range(dim)], 2)


class _Cov:
    """The structure of a covariance H^2 matrix (heap-ordered complete tree, block-sparse rows)."""


def structure(points, m, p, eta):
    """KD tree, tight boxes, Chebyshev nodes and the dual traversal of `points` (n, dim)."""
    n, dim = points.shape
    q = 0
    while (m << q) < n:
        q += 1
    A = _Cov()
    A.n, A.dim, A.m, A.p, A.k, A.q = n, dim, m, p, p ** dim, q
    perm = torch.arange(n, device=points.device)
    bounds = np.array([0, n], dtype=np.int64)
    for _ in range(q):  # a node's points by (coordinate along its longest side, index); the first ceil(s / 2) go left
        node = torch.repeat_interleave(torch.arange(bounds.size - 1, device=perm.device),
                                       torch.from_numpy(np.diff(bounds)).to(perm.device))
        P = points[perm]
        mn, mx = _segment(P, node, bounds.size - 1)
        side = torch.argmax(mx - mn, 1)[node]
        x = P.gather(1, side[:, None])[:, 0]
        o = torch.argsort(perm, stable=True)
        o = o[torch.argsort(x[o], stable=True)]
        perm = perm[o[torch.argsort(node[o], stable=True)]]
        mid = bounds[:-1] + (np.diff(bounds) + 1) // 2
        bounds = np.sort(np.concatenate([bounds, mid]))
    A.perm, A.leaf_offset = perm, bounds
    A.points = points[perm]
    leaves = 1 << q
    A.leaf = torch.repeat_interleave(torch.arange(leaves, device=perm.device),
                                     torch.from_numpy(np.diff(bounds)).to(perm.device))
    mn, mx = _segment(A.points, A.leaf, leaves)
    lo, hi = [mn], [mx]
    while lo[0].shape[0] > 1:
        lo.insert(0, torch.minimum(lo[0][0::2], lo[0][1::2]))
        hi.insert(0, torch.maximum(hi[0][0::2], hi[0][1::2]))
    bmin, bmax = torch.cat(lo), torch.cat(hi)
    c = 0.5 * (bmin + bmax)
    thin = (bmax - bmin) < 1e-10
    a, b = torch.where(thin, c - 0.5e-10, bmin), torch.where(thin, c + 0.5e-10, bmax)
    v = torch.arange(p, dtype=torch.float64, device=c.device)
    A.cheb = 0.5 * (a + b)[:, :, None] + 0.5 * (b - a)[:, :, None] * torch.cos((2.0 * v + 1.0) * math.pi / (2.0 * p))
    diam = torch.sqrt(((bmax - bmin) ** 2).sum(1))
    I = torch.zeros(1, dtype=torch.int64, device=c.device)
    J, S = I.clone(), []
    for level in range(q + 1):
        gap = torch.clamp(torch.maximum(bmin[J] - bmax[I], bmin[I] - bmax[J]), min=0.0)
        dist = torch.sqrt((gap ** 2).sum(1))
        far = (dist > 0) & (torch.maximum(diam[I], diam[J]) <= eta * dist) if eta > 0 else torch.zeros_like(I, dtype=torch.bool)
        S.append(torch.stack([I[far], J[far]]))
        I, J = I[~far], J[~far]
        if level < q:
            I, J = (torch.cat([2 * I + u for u in (1, 2) for _ in (1, 2)]), torch.cat([2 * J + w for _ in (1, 2) for w in (1, 2)]))
    nodes = 2 * leaves - 1
    A.leaves, A.nodes = leaves, nodes

    def bsr(i, j, rows):
        o = torch.argsort(i * nodes + j)
        return i[o], j[o], torch.cat([torch.zeros(1, dtype=torch.int64, device=i.device),
                                      torch.cumsum(torch.bincount(i, minlength=rows), 0)])

    S = torch.cat(S, 1)
    A.Si, A.Sj, A.Sptr = bsr(S[0], S[1], nodes)
    A.Di, A.Dj, A.Dptr = bsr(I - (leaves - 1), J - (leaves - 1), leaves)
    return A


def _segment(P, seg, count):
    ix = seg[:, None].expand_as(P)
    z = torch.empty(count, P.shape[1], dtype=P.dtype, device=P.device)
    return (z.scatter_reduce(0, ix, P, "amin", include_self=False), z.scatter_reduce(0, ix, P, "amax", include_self=False))


def covariance(case, points, values="UESD"):
    """The matrix of `case` over `points`: its structure and, as asked, the values of its blocks.
    U and D are held padded to the largest leaf (zero rows and columns)."""
    A = structure(points, case["m"], case["p"], case["eta"])
    A.kernel, A.ell = case["kernel"], case["ell"]
    size = torch.from_numpy(np.diff(A.leaf_offset)).to(points.device)
    A.mm = int(size.max())
    slot = torch.arange(A.mm, device=points.device)
    A.mask = slot[None, :] < size[:, None]
    A.at = torch.clamp(torch.from_numpy(A.leaf_offset[:-1]).to(points.device)[:, None] + slot[None, :], max=A.n - 1)
    A.leafpts = A.points[A.at]
    first = A.leaves - 1
    if "U" in values:
        A.U = _lagrange(A.cheb[first:], A.leafpts) * A.mask[:, :, None]
    if "E" in values:
        c = torch.arange(1, A.nodes, device=points.device)
        A.E = _lagrange(A.cheb[(c - 1) // 2], _grid(A.cheb[c]))
    if "S" in values:
        A.S = coupling(A, slice(None))
    if "D" in values:
        A.D = dense(A, slice(None))
    return A


def coupling(A, b):
    return _kernel(A.kernel, A.ell, _dist(_grid(A.cheb[A.Si[b]]), _grid(A.cheb[A.Sj[b]])))


def dense(A, b):
    i, j = A.Di[b], A.Dj[b]
    return _kernel(A.kernel, A.ell, _dist(A.leafpts[i], A.leafpts[j])) * (A.mask[i][:, :, None] & A.mask[j][:, None, :])


def arrays(A, values="UESD"):
    """The matrix's description in host memory, as the entry points take it (blocks column-major)."""
    def host(t, dt=None):
        t = t.cpu().numpy()
        return t if dt is None else t.astype(dt)

    d = dict(n=A.n, depth=A.q, rank=A.k, leaf_offset=A.leaf_offset, S_rowptr=host(A.Sptr, np.int32),
             S_colidx=host(A.Sj, np.int32), D_rowptr=host(A.Dptr, np.int32), D_colidx=host(A.Dj, np.int32))
    if "U" in values:
        Ut = A.U.transpose(1, 2)
        d["U"] = host(Ut[A.mask[:, None, :].expand_as(Ut)])
    if "E" in values:
        d["E"] = host(A.E.transpose(1, 2).reshape(-1))
    d["S_val"] = host(A.S.transpose(1, 2).reshape(-1)) if "S" in values else None
    d["D_val"] = None
    if "D" in values:
        Dt = A.D.transpose(1, 2)
        if bool(A.mask.all()):
            d["D_val"] = host(Dt.reshape(-1))
        else:
            d["D_val"] = host(Dt[A.mask[A.Dj][:, :, None] & A.mask[A.Di][:, None, :]])
    return d


def multiply(A, x, far_only=False):
    """y = A x in FP64 (x (n, nv) in cluster order): upsweep, coupling, downsweep, dense blocks."""
    nv, step = x.shape[1], 8192
    first = A.leaves - 1
    xl = x[A.at] * A.mask[:, :, None]
    xh = torch.zeros(A.nodes, A.k, nv, dtype=torch.float64, device=x.device)
    yh = torch.zeros_like(xh)
    xh[first:] = torch.bmm(A.U.transpose(1, 2), xl)
    for level in range(A.q - 1, -1, -1):
        lo, hi = 2 ** (level + 1) - 1, 2 ** (level + 2) - 1
        xh[2 ** level - 1:lo] = torch.bmm(A.E[lo - 1:hi - 1].transpose(1, 2), xh[lo:hi]).reshape(-1, 2, A.k, nv).sum(1)
    for b in range(0, A.Si.numel(), step):
        s = slice(b, b + step)
        yh.index_add_(0, A.Si[s], torch.bmm(A.S[s] if hasattr(A, "S") else coupling(A, s), xh[A.Sj[s]]))
    for level in range(1, A.q + 1):
        lo, hi = 2 ** level - 1, 2 ** (level + 1) - 1
        c = torch.arange(lo, hi, device=x.device)
        yh[lo:hi] += torch.bmm(A.E[lo - 1:hi - 1], yh[(c - 1) // 2])
    yl = torch.bmm(A.U, yh[first:])
    if not far_only:
        for b in range(0, A.Di.numel(), step):
            s = slice(b, b + step)
            yl.index_add_(0, A.Di[s], torch.bmm(A.D[s] if hasattr(A, "D") else dense(A, s), xl[A.Dj[s]]))
    return yl[A.mask]


def _points(case, g):
    if case["kind"] == "build":
        # the block lists' lengths depend on the points: one cloud per case, in another order (and
        # another unit of length, a power of two) for every seed
        P = torch.rand(case["n"], case["dim"], dtype=torch.float64, device=DEV, generator=_generator(case["n"]))
        P = P[torch.randperm(case["n"], device=DEV, generator=g)]
        return P * 2.0 ** int(torch.randint(-3, 4, (1,), device=DEV, generator=g))
    return torch.rand(case["n"], case["dim"], dtype=torch.float64, device=DEV, generator=g)


def _vectors(n, nv, g, dtype):
    return torch.randn(nv, n, dtype=torch.float64, device=DEV, generator=g).to(dtype).t()


def _members(case, seed):
    """The batch's matrices: (case of the member, points) each, sizes log-uniform, 1, 4 or 16 vectors."""
    rs = np.random.RandomState(seed % (1 << 32))
    out = []
    for i in range(case["count"]):
        # the sizes come from the case, so that every seed's batch is the same amount of work
        t = (i + 0.5) / case["count"]
        n = int(round(math.exp(math.log(case["n_lo"]) * (1 - t) + math.log(case["n_hi"]) * t))) + (i % 3)
        out.append(dict(case, dim=2, n=n, nv=(1, 4, 16)[i % 3]))
    rs.shuffle(out)
    return out


# ------------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    g, kind = _generator(seed), case["kind"]
    if kind == "build":
        return dict(kind=kind, case=case, points=_points(case, g).cpu().numpy())
    if kind == "batch":
        mats, sizes = [], []
        for c in _members(case, seed):
            d = arrays(covariance(c, _points(c, g)))
            mats.append(h2.H2Matrix(**d, storage=case["storage"], bases_fp32=case["bases_fp32"]))
            sizes.append((c["n"], c["nv"]))
        total = sum(n * nv for n, nv in sizes)
        # the members' vectors lie one after another in one FP32 buffer of the program's; the batched
        # call takes FP64 vectors, so they are widened before it and its results narrowed after it
        x = torch.randn(total, dtype=torch.float64, device=DEV, generator=g).float()
        x64, y64, y = torch.empty(total, dtype=torch.float64, device=DEV), torch.empty(total, dtype=torch.float64, device=DEV), torch.empty_like(x)
        xs, ys, at = [], [], 0
        for n, nv in sizes:
            xs.append(x64[at:at + n * nv].view(nv, n).t())
            ys.append(y64[at:at + n * nv].view(nv, n).t())
            at += n * nv
        B = h2.H2Batch(mats)
        return dict(kind=kind, B=B, args=B.prepare(xs, ys), x=x, x64=x64, y64=y64, y=y, keep=(xs, ys))
    pts = _points(case, g)
    if kind == "compress":
        d = arrays(covariance(case, pts, "UES"), "UES")
        C = h2.Compressor(**{k: v for k, v in d.items() if k != "D_val"})
        d["D_rowptr"] = np.zeros_like(d["D_rowptr"])  # the far field alone
        d["D_colidx"], d["D_val"] = np.empty(0, np.int32), np.empty(0)
        x = _vectors(case["n"], 1, g, torch.float64)
        return dict(kind=kind, C=C, d=d, eps=case["eps"], x=x)
    if kind == "kernel":
        A = covariance(case, pts, "UE")
        d = arrays(A, "UE")
        M = h2.H2Matrix(**d, storage=case["storage"], bases_fp32=case["bases_fp32"], points=A.points.cpu().numpy(),
                        coupling_kernel=dict(kernel=case["kernel"], ell=case["ell"], cheb=A.cheb.cpu().numpy()))
    else:
        M = h2.H2Matrix(**arrays(covariance(case, pts)), storage=case["storage"], bases_fp32=case["bases_fp32"])
    x = _vectors(case["n"], case["nv"], g, torch.float64 if case["storage"] == "fp64" else torch.float32)
    y = torch.empty(case["nv"], case["n"], dtype=x.dtype, device=DEV).t()
    return dict(kind=kind, M=M, x=x, y=y)


BUILT = ("perm", "leaf_offset", "points", "cheb", "S_rowptr", "S_colidx", "D_rowptr", "D_colidx", "U", "E")


def run(s):
    kind = s["kind"]
    if kind == "product" or kind == "kernel":
        if s["x"].dtype == torch.float64:
            return s["M"].matvec(s["x"], s["y"])
        return s["M"].matvec_f32(s["x"], s["y"])
    if kind == "batch":
        s["x64"].copy_(s["x"])
        s["B"].matvec_prepared(s["args"])
        s["y"].copy_(s["y64"])
        return s["y"]
    if kind == "compress":
        C, d = s["C"], s["d"]
        C.run(s["eps"])
        rank, rows, cols = C.result()
        M = h2.H2Matrix(**{**d, "rank": rank, "U": C.read("U"), "E": C.read("E"), "S_val": C.read("S")})
        return {"y": M.matvec(s["x"]), "sigma": C.read("sigma_U"), "ranks": np.array(rows + cols, dtype=np.int64)}
    c = s["case"]
    B = h2.Built(s["points"], m=c["m"], p=c["p"], eta=c["eta"], kernel=c["kernel"], ell=c["ell"], values=("U", "E"))
    out = {w: B.read(w) for w in BUILT}
    B.close()
    return out


# ------------------------------------------------------------------------------- what the work is
@functools.lru_cache(maxsize=None)
def _counts(dim, n, m, p, eta):
    A = structure(torch.rand(n, dim, dtype=torch.float64, device=DEV, generator=_generator(7)), m, p, eta)
    size = torch.from_numpy(np.diff(A.leaf_offset)).to(DEV)
    return int(A.Si.numel()), int((size[A.Di] * size[A.Dj]).sum()), int(A.Di.numel()), A.nodes


def _product_work(c, nv, vec):
    """Bytes and flops of one product: every stored entry and every vector entry once."""
    k = c["p"] ** c["dim"]
    nS, nDval, nD, nodes = _counts(c["dim"], c["n"], c["m"], c["p"], c["eta"])
    bases, coup = 2 * c["n"] * k + 2 * (nodes - 1) * k * k, nS * k * k
    if c["storage"] == "fp64":
        b = 8 * (bases + coup + nDval)
    else:
        kc = c["kind"] == "kernel"
        b = (4 if c["bases_fp32"] else 2) * bases + 2 * nDval + 4 * nD + (0 if kc else 2 * coup + 4 * nS)
        b += 4 * nS + 16 * nodes * k if kc else 0  # the column list and the interpolation points
    return b + 2 * vec * c["n"] * nv, 2 * nv * (bases + coup + nDval)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_product_work(c, c["nv"], 4) for c in _members(case, 0)]
        return {"bytes": sum(a for a, _ in w), "flops": sum(f for _, f in w)}
    k, n, dim = case["p"] ** case["dim"], case["n"], case["dim"]
    if kind in ("product", "kernel"):
        b, f = _product_work(case, case["nv"], 8 if case["storage"] == "fp64" else 4)
        return {"bytes": b, "flops": f}
    nS, nDval, nD, nodes = _counts(dim, n, case["m"], case["p"], case["eta"])
    if kind == "compress":  # the low-rank part in; the two projections and the R trees' reductions
        b = 8 * (nS * k * k + n * k + nodes * k * k)
        return {"bytes": b, "flops": nS * (2 * k * k * (k + 1) + 2 * k * k * (k - 1))}
    b = 8 * n * dim * 2 + 8 * n + 4 * (nS + nD) + 8 * (n * k + nodes * k * k)
    return {"bytes": b, "flops": (n + nodes * k) * (k + 3 * case["p"] ** 2 * dim)}


def exact(case, seed):
    g, kind = _generator(seed), case["kind"]
    if kind == "build":
        A = covariance(case, _points(case, g), "UE")
        d = arrays(A, "UE")
        return {"points": A.points.reshape(-1), "cheb": A.cheb.reshape(-1), "U": d["U"], "E": d["E"],
                **{w: None for w in ("perm", "leaf_offset", "S_rowptr", "S_colidx", "D_rowptr", "D_colidx")}}
    if kind == "batch":
        made = [(c, covariance(c, _points(c, g))) for c in _members(case, seed)]
        x = torch.randn(sum(c["n"] * c["nv"] for c, _ in made), dtype=torch.float64, device=DEV, generator=g).float().double()
        out, at = [], 0
        for c, A in made:
            size = c["n"] * c["nv"]
            out.append(multiply(A, x[at:at + size].view(c["nv"], c["n"]).t()).t().reshape(-1))
            at += size
        return torch.cat(out)
    A = covariance(case, _points(case, g), "UE" if kind == "kernel" else "UES" if kind == "compress" else "UESD")
    if kind == "compress":  # the compressed far field's product is the far field's to the threshold
        return {"y": multiply(A, _vectors(case["n"], 1, g, torch.float64), far_only=True), "sigma": None, "ranks": None}
    return multiply(A, _vectors(case["n"], case["nv"], g, torch.float64 if case["storage"] == "fp64" else torch.float32).double())
