"""Performance cases: the calls a user of the library makes, over the sizes, types and options it is used with.

Every case is a dict of plain values.  `op` names the call:

  trsv       sptrsv_lower, then sptrsv_upper, on ILU(0) factors (default plan)
  apply      IluSolver.apply: the ILU(0) preconditioner inside a Krylov loop (pencils > 0: partitioned sweeps)
  ras        RasSolver.apply: restricted additive Schwarz on box subdomains
  sgs        SgsSmoother.smooth: one symmetric Gauss-Seidel sweep (the multigrid smoother)
  spmv       spmv: the FP64 matrix product of the outer solver
  ilu        ilu_factor: ILU(k) of a new matrix
  ilut       ilut_factor: ILUT(10, 1e-3) of a new matrix, the solver made from it and its first application
  setup      IluSolver(...) and partition(...), then its first application and product: what a new matrix
             costs besides its factorization
  ras_setup  RasSolver(...) with every subdomain one part, and its first application
  solve      IluSolver.solve: FGMRES(30) to 1e-8
  net        Net.backward: loss and gradients of the correction network on one minibatch of crops

Matrices are the ones of paper_1606_00541_gb300.synth, built here on the GPU because a preparation has to be
quick: 5- and 7-point Poisson, the 7-point log-normal finite-volume matrix (ln k ~ N(0, 2^2)) and the jittered
27-point stencil, on nx x ny x nz grids with x fastest.
"""
import math

import torch

from paper_1606_00541_gb300 import hec, learn

DEV = "cuda"
VALUE_BYTES = {"f64": 8, "f32": 4, "bf16": 2}


# --- cases ---------------------------------------------------------------------------------------

def _case(name, op, stencil, dims, vdt="f64", nrhs=1, **more):
    nx, ny, nz = dims
    return dict(name=name, op=op, stencil=stencil, nx=nx, ny=ny, nz=nz, vdt=vdt, nrhs=nrhs, **more)


def listed():
    cube = lambda m: (m, m, m)  # noqa: E731
    return [
        # the smallest calls: one lower and one upper solve on a 64 x 64 grid (a coarse grid, a unit test, one
        # block of a larger program), where launches and the latency of a level are all there is
        _case("trsv_poisson5_64", "trsv", "poisson5", (64, 64, 1)),
        # the preconditioner of a Krylov loop on a million-row model problem, used as the constructor leaves it
        _case("apply_poisson7_100", "apply", "poisson7", cube(100), pencils=0),
        # the same call tuned by its user: FP32 factor values and one thread block for each of 256 x-pencils,
        # the configuration of the time-to-solution benchmark
        _case("apply_fv7_128_parts", "apply", "fv7", cube(128), vdt="f32", pencils=16),
        # many right-hand sides at once: restricted additive Schwarz on 64 boxes, 16 right-hand sides
        _case("ras_fv7_128_16rhs", "ras", "fv7", cube(128), vdt="f32", nrhs=16, bx=4, by=4, bz=4),
        # the triangular solve as a smoother, on rows of 27 entries
        _case("sgs_stencil27_100", "sgs", "stencil27", cube(100)),
        # the matrix product of the outer solver on the largest grid in use (8 million rows)
        _case("spmv_fv7_200", "spmv", "fv7", cube(200)),
        # a new matrix in every time step of a simulation: its ILU(0) factorization ...
        _case("ilu0_fv7_128", "ilu", "fv7", cube(128), k=0),
        # ... or, for harder problems with longer rows, its ILUT factorization and the solver made from that
        _case("ilut_stencil27_100", "ilut", "stencil27", cube(100)),
        # ... and the analysis, packing, plans and partition that follow a factorization
        _case("setup_fv7_128", "setup", "fv7", cube(128), vdt="f32", pencils=16),
        # the same for the Schwarz form with one part per subdomain (576 boxes)
        _case("ras_setup_fv7_128", "ras_setup", "fv7", cube(128), vdt="f32", bx=4, by=12, bz=12),
        # the whole solve, time to 1e-8: the number the library is judged by
        _case("solve_fv7_128", "solve", "fv7", cube(128), vdt="f32", pencils=16),
        # training of the learned correction: one minibatch of eight 32^3 crops, forward and backward
        _case("net_backward_8x32", "net", "crops", (32, 32, 256), vdt="bf16", zs=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, lo, hi):
    """A grid near a cube whose extents are drawn one by one (odd and unequal ones among them)."""
    m = _log(rng, lo, hi)
    return tuple(max(4, min(hi, int(m * rng.uniform(0.75, 1.25)))) for _ in range(3))


def draw(rng):
    op = rng.choice(["trsv", "apply", "apply", "apply", "ras", "ras", "sgs", "spmv", "spmv", "ilu", "ilu", "ilut", "setup",
                     "ras_setup", "solve", "net"])
    vdt = rng.choice(["f64", "f32", "bf16"])
    if op == "trsv":
        return _draw(op, "poisson5", (_log(rng, 64, 1024), _log(rng, 64, 1024), 1), vdt, rng.choice([1, 1, 2, 3, 8]))
    if op == "apply":
        nrhs = rng.choice([1, 1, 1, 2, 4, 5, 8, 16])
        dims = _dims(rng, 16, 128 if nrhs == 1 else 100)
        return _draw(op, rng.choice(["poisson7", "fv7"]), dims, vdt, nrhs,
                     pencils=rng.choice([0, _pencils(dims)]) if nrhs == 1 else 0)
    if op == "ras":
        dims = _dims(rng, 24, 128)
        return _draw(op, "fv7", dims, vdt, rng.choice([1, 3, 4, 8, 12, 16]), bx=rng.randint(1, 4), by=rng.randint(2, 4),
                     bz=rng.randint(2, 4))
    if op == "sgs":
        return _draw(op, rng.choice(["stencil27", "fv7"]), _dims(rng, 16, 100), vdt, rng.choice([1, 1, 2, 4]))
    if op == "spmv":
        nrhs = rng.choice([1, 1, 2, 4, 7, 16])
        stencil = rng.choice(["fv7", "stencil27", "poisson7"])
        return _draw(op, stencil, _dims(rng, 24, 200 if nrhs == 1 and stencil != "stencil27" else 100), "f64", nrhs)
    if op == "ilu":
        stencil = rng.choice(["fv7", "fv7", "poisson7", "stencil27"])
        return _draw(op, stencil, _dims(rng, 16, 128 if stencil != "stencil27" else 48), "f64", 1,
                     k=rng.choice([0, 0, 1]) if stencil != "stencil27" else 0)
    if op == "ilut":
        return _draw(op, rng.choice(["stencil27", "fv7"]), _dims(rng, 12, 100), "f64", 1)
    if op in ("setup", "solve"):
        dims = _dims(rng, 24, 128)
        return _draw(op, "fv7", dims, vdt, 1, pencils=rng.choice([0, _pencils(dims)]))
    if op == "ras_setup":
        dims = _dims(rng, 24, 128)
        return _draw(op, "fv7", dims, vdt, 1, bx=max(1, dims[0] // 32), by=max(1, dims[1] // 11), bz=max(1, dims[2] // 11))
    m, batch = rng.choice([16, 20, 24, 32]), rng.randint(1, 8)
    return _draw(op, "crops", (m, m, m * batch), "bf16", 1, zs=m)


def _draw(*a, **k):
    c = _case(None, *a, **k)
    del c["name"]
    return c


def _pencils(dims):
    """Pencils along y and along z: 8 cells thick, as in the listed case, and at most 16 of them."""
    return max(1, min(16, min(dims[1], dims[2]) // 8))


# --- matrices ------------------------------------------------------------------------------------

STENCILS = {
    "poisson5": [(0, -1, 0), (0, 0, -1), (0, 0, 0), (0, 0, 1), (0, 1, 0)],
    "poisson7": [(-1, 0, 0), (0, -1, 0), (0, 0, -1), (0, 0, 0), (0, 0, 1), (0, 1, 0), (1, 0, 0)],
    "stencil27": [(z, y, x) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)],
}
STENCILS["fv7"] = STENCILS["poisson7"]


def _matrix(case, gen):
    """(rowptr int32, col int32, val float64) on the GPU."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = nx * ny * nz
    g = torch.arange(n, device=DEV)
    x, y, z = g % nx, (g // nx) % ny, g // (nx * ny)
    offs = STENCILS[case["stencil"]]
    cols, vals, mask = [], [], []
    perm = torch.exp(2.0 * torch.randn(n, device=DEV, dtype=torch.float64, generator=gen)) if case["stencil"] == "fv7" else None
    diag = torch.zeros(n, device=DEV, dtype=torch.float64)
    edge = {}
    for dz, dy, dx in offs:
        d = dz * nx * ny + dy * nx + dx
        ok = (x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) & (z + dz >= 0) & (z + dz < nz)
        c = g + d
        cols.append(c)
        mask.append(ok)
        if d == 0:
            vals.append(None)
            continue
        cc = c.clamp(0, n - 1)
        if case["stencil"] == "fv7":  # harmonic face average, Dirichlet faces at the boundary
            t = torch.where(ok, 2.0 * perm * perm[cc] / (perm + perm[cc]), 0.0)
            diag += t + torch.where(ok, 0.0, 2.0 * perm)
            vals.append(-t)
        elif case["stencil"] == "stencil27":  # one draw for each undirected edge, kept on its smaller end
            key, at = ((dz, dy, dx), g) if d > 0 else ((-dz, -dy, -dx), cc)
            if key not in edge:
                edge[key] = 2.0 * torch.rand(n, device=DEV, dtype=torch.float64, generator=gen) - 1.0
            v = torch.where(ok, -(1.0 + 0.3 * edge[key][at]), 0.0)
            diag += 1.05 * v.abs()
            vals.append(v)
        else:
            vals.append(torch.full((n,), -1.0, device=DEV, dtype=torch.float64))
    if case["stencil"].startswith("poisson"):
        diag += len(offs) - 1
    vals = torch.stack([diag if v is None else v for v in vals], dim=1)
    cols, mask = torch.stack(cols, dim=1), torch.stack(mask, dim=1)
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    rowptr[1:] = mask.sum(1).cumsum(0).to(torch.int32)
    return rowptr, cols[mask].to(torch.int32), vals[mask]


def _boxes(case, bx, by, bz):
    """The box of each cell: near-equal extents along each axis."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    g = torch.arange(nx * ny * nz, device=DEV)
    x, y, z = g % nx, (g // nx) % ny, g // (nx * ny)
    part = (x * bx) // nx + bx * ((y * by) // ny + by * ((z * bz) // nz))
    return part.to(torch.int32), bx * by * bz


def _inputs(case, seed):
    """(A, right-hand side or start vectors), the same for prepare() and exact()."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    A = _matrix(case, gen)
    n, k = A[0].numel() - 1, case["nrhs"]
    shape = (n,) if k == 1 else (n, k)
    rand = lambda: 2.0 * torch.rand(shape, device=DEV, dtype=torch.float64, generator=gen) - 1.0  # noqa: E731
    return A, rand(), rand()


def _net_inputs(case, seed):
    """Residual and log-permeability fields of a minibatch, the targets, and the initial weights."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    n = case["nx"] * case["ny"] * case["nz"]
    x = torch.zeros(n, learn.C, dtype=torch.bfloat16, device=DEV)
    x[:, :2] = torch.randn(n, 2, device=DEV, generator=gen).to(torch.bfloat16)
    return x, torch.randn(n, device=DEV, generator=gen), learn.init_params(seed % 1000)


# --- the calls -----------------------------------------------------------------------------------

def _ilu0(A):
    Lh, Uh = hec.ilu_factor(*A, k=0)
    return Lh.tensors(), Uh.tensors()


def _partition(s, case):
    if case["pencils"]:
        part, count = _boxes(case, 1, case["pencils"], case["pencils"])
        s.partition(part, count, threads=512)


def prepare(case, seed):
    op = case["op"]
    if op == "net":
        x, target, params = _net_inputs(case, seed)
        return dict(op=op, net=hec.Net(params), x=x, target=target, dims=(case["nx"], case["ny"], case["nz"]), zs=case["zs"])
    A, b, c = _inputs(case, seed)
    st = dict(op=op, case=case, A=A, b=b, c=c)
    vdt, k = case["vdt"], case["nrhs"]
    if op in ("trsv", "apply", "solve"):
        L, U = _ilu0(A)
        st["s"] = hec.IluSolver(L, U, A=A if op == "solve" else None, vdt=vdt, max_nrhs=k)
        if op != "trsv":
            _partition(st["s"], case)
        if op == "solve":  # c is the solution, b = A c
            st["b"] = hec.spmv(st["s"].A, c)
    elif op in ("ras", "ras_setup"):
        st["part"], st["nsub"] = _boxes(case, case["bx"], case["by"], case["bz"])
        if op == "ras":
            st["s"] = hec.RasSolver(A, st["part"], st["nsub"], vdt=vdt, max_nrhs=k)
    elif op == "sgs":
        st["s"] = hec.SgsSmoother(A, vdt=vdt, max_nrhs=k)
    elif op == "spmv":
        st["s"] = hec.hec_from_csr(*A)
    elif op == "setup":
        st["L"], st["U"] = _ilu0(A)
        st["part"], st["nparts"] = _boxes(case, 1, case["pencils"], case["pencils"]) if case["pencils"] else (None, 0)
    return st


def run(st):
    op = st["op"]
    if op == "net":
        loss = st["net"].backward(st["x"], st["target"], st["dims"], zs=st["zs"])
        return loss, st["net"].params(grads=True)[1]
    A, b, case = st["A"], st["b"], st["case"]
    if op == "trsv":
        y = hec.sptrsv_lower(st["s"].pL, b)
        return y, hec.sptrsv_upper(st["s"].pU, y)
    if op in ("apply", "ras"):
        return st["s"].apply(b)
    if op == "sgs":
        return st["s"].smooth(st["c"], b)
    if op == "spmv":
        return hec.spmv(st["s"], b)
    if op == "ilu":
        L, U = hec.ilu_factor(*A, k=case["k"])
        return L.tensors() + U.tensors()
    if op == "ilut":
        L, U = hec.ilut_factor(*A, p=10, tol=1e-3)
        return hec.IluSolver(L.tensors(), U.tensors(), vdt=case["vdt"]).apply(b)
    if op == "setup":
        s = hec.IluSolver(st["L"], st["U"], A=A, vdt=case["vdt"])
        if st["part"] is not None:
            s.partition(st["part"], st["nparts"], threads=512)
        z = s.apply(b)
        return z, hec.spmv(s.A, z)
    if op == "ras_setup":
        s = hec.RasSolver(A, st["part"], st["nsub"], vdt=case["vdt"])
        sub = torch.arange(st["nsub"], dtype=torch.int32, device=DEV)
        s.partition(torch.repeat_interleave(sub, s.ext_ptr.diff()), st["nsub"], threads=256)
        return s.ext_ptr, s.ext2glob, s.owned, s.apply(b)
    return st["s"].solve(b, max_iters=5000)[0]


# --- the work ------------------------------------------------------------------------------------

def _entries(case):
    """Stored entries of the matrix."""
    dims = (case["nz"], case["ny"], case["nx"])
    return sum(math.prod(d - abs(o) for d, o in zip(dims, off)) for off in STENCILS[case["stencil"]])


def _sweeps(n, nnz, k, sv):
    """Both factors of an ILU(0) with values and column indices, their row pointers, and the vectors in and out."""
    tri = (nnz + n) // 2
    return dict(bytes=2 * tri * (sv + 4) + 8 * (n + 1) + 16 * n * k, flops=4 * tri * k)


def work(case):
    op, k = case["op"], case["nrhs"]
    n = case["nx"] * case["ny"] * case["nz"]
    if op == "net":  # input channels, targets and gradients; forward and two products backward
        return dict(bytes=n * (32 + 4) + 4 * hec.net_param_count(), flops=3 * 2 * 27 * (2 * 16 + 2 * 16 * 16 + 16) * n)
    nnz, sv = _entries(case), VALUE_BYTES[case["vdt"]]
    if op == "spmv":
        return dict(bytes=12 * nnz + 4 * n + 16 * n * k, flops=2 * nnz * k)
    if op in ("trsv", "apply"):
        w = _sweeps(n, nnz, k, sv)
        return dict(w, bytes=w["bytes"] + (16 * n * k if op == "trsv" else 0))
    if op == "sgs":  # both triangles with FP64 residual products; x and b in, x out
        w = _sweeps(n, nnz, k, sv)
        return dict(bytes=w["bytes"] + 12 * (nnz - n) + 8 * n * k, flops=w["flops"] + 2 * (nnz - n) * k)
    if op == "ilu":  # A in, L and U out (about twice the entries for one level of fill); ~3 updates an entry
        out = (1 + case["k"]) * nnz + n
        return dict(bytes=12 * (nnz + out) + 12 * n, flops=6 * out)
    if op == "ilut":  # at most 10 entries in each part of a row besides the diagonal
        out = 2 * n * (min(10, (nnz // n - 1) // 2 + 4) + 1)
        return dict(bytes=12 * (nnz + 2 * out) + 28 * n, flops=22 * out)
    if op == "setup":  # the factors and A in, their packed forms and maps out, one application, one product
        w = _sweeps(n, nnz, 1, sv)
        return dict(bytes=12 * (2 * nnz + n) + w["bytes"] + 12 * nnz + 16 * n + 16 * n, flops=w["flops"] + 2 * nnz)
    if op == "solve":  # about as many iterations as the longest extent; a basis of 15 vectors on average
        w, its = _sweeps(n, nnz, 1, sv), max(case["nx"], case["ny"], case["nz"])
        return dict(bytes=its * (w["bytes"] + 12 * nnz + 20 * n + 17 * 8 * n), flops=its * (w["flops"] + 2 * nnz + 62 * n))
    # Schwarz: the extended rows, with about 6.4 entries in a row
    ne = n + 2 * ((case["bx"] - 1) * case["ny"] * case["nz"] + (case["by"] - 1) * case["nx"] * case["nz"] +
                  (case["bz"] - 1) * case["nx"] * case["ny"])
    nnz_e = int(6.4 * ne)
    w = _sweeps(ne, nnz_e, k, sv)
    w["bytes"] += 16 * (n - ne) * k + 5 * ne
    if op == "ras_setup":  # A in, the extended system and its factors out, then as above
        w = dict(bytes=w["bytes"] + 12 * nnz + 24 * nnz_e + 20 * ne, flops=w["flops"] + 6 * nnz_e)
    return w


# --- the same results in 64 bits -----------------------------------------------------------------

def _rows(rowptr):
    """The row of each entry."""
    count = rowptr.long().diff()
    return torch.repeat_interleave(torch.arange(count.numel(), device=DEV), count)


def _ell(n, row, col, val):
    """Entries (sorted by row) as padded [n, w] columns and values."""
    count = torch.bincount(row, minlength=n)
    start = count.cumsum(0) - count
    w = max(1, int(count.max()))
    c = torch.zeros(n, w, dtype=torch.long, device=DEV)
    v = torch.zeros(n, w, dtype=torch.float64, device=DEV)
    slot = torch.arange(row.numel(), device=DEV) - start[row]
    c[row, slot], v[row, slot] = col, val
    return c, v


def _product(c, v, x):
    if x.dim() == 1:
        return (v * x[c]).sum(1)
    return torch.stack([(v * x[:, q].contiguous()[c]).sum(1) for q in range(x.shape[1])], dim=1)


def _rounded(val, vdt):
    return val if vdt == "f64" else val.to(torch.float32 if vdt == "f32" else torch.bfloat16).double()


def _solve(n, row, col, val, b):
    """T x = b for a triangular T: x = D^-1 (b - N x) repeated; N is nilpotent, so it ends at the substitution."""
    off = row != col
    c, v = _ell(n, row[off], col[off], val[off])
    d = torch.empty(n, dtype=torch.float64, device=DEV)
    d[row[~off]] = val[~off]
    d = d if b.dim() == 1 else d[:, None]
    x = b / d
    for _ in range(20000):
        y = (b - _product(c, v, x)) / d
        if bool((y - x).abs().max() <= 1e-16 * y.abs().max()):
            return y
        x = y
    return x


def _factors(A, k=0):
    """ILU(k) values for k = 0 or 1, as (row, col, value) sorted by row and column: the equations
    l_ij u_jj = a_ij - sum l_iq u_qj and u_ij = a_ij - sum l_iq u_qj repeated to their fixed point."""
    n = A[0].numel() - 1
    row, col, val = _rows(A[0]), A[1].long(), A[2]
    key = row * n + col

    def updates(row, col, key):
        """(entry (i, j), entry (i, q), entry (q, j)) for q < i, q < j; the first is a key, or an index if it is there."""
        end = torch.searchsorted(key, (torch.arange(n, device=DEV) + 1) * n)
        first = torch.searchsorted(key, torch.arange(n, device=DEV) * (n + 1) + 1)  # right of the diagonal
        low = (col < row).nonzero().flatten()
        out = []
        for s in range(int((end - first).max())):
            e2 = first[col[low]] + s
            ok = e2 < end[col[low]]
            e1, e2 = low[ok], e2[ok]
            out.append((row[e1] * n + col[e2], e1, e2))
        return out

    if k:
        fill = torch.unique(torch.cat([key] + [t[0] for t in updates(row, col, key)]))
        full = torch.zeros(fill.numel(), dtype=torch.float64, device=DEV)
        full[torch.searchsorted(fill, key)] = val
        key, val, row, col = fill, full, fill // n, fill % n
    found = []
    for t, e1, e2 in updates(row, col, key):
        at = torch.searchsorted(key, t).clamp(max=key.numel() - 1)
        hit = key[at] == t
        found.append((at[hit], e1[hit], e2[hit]))
    at, e1, e2 = (torch.cat([f[i] for f in found]) for i in range(3))
    order = torch.argsort(at * key.numel() + e1) if key.numel() < 2 ** 31 else torch.argsort(at, stable=True)
    at, e1, e2 = at[order], e1[order], e2[order]
    target, count = torch.unique_consecutive(at, return_counts=True)
    slot = torch.arange(at.numel(), device=DEV) - torch.repeat_interleave(count.cumsum(0) - count, count)
    mine = torch.repeat_interleave(torch.arange(target.numel(), device=DEV), count)
    w = int(count.max())
    none = key.numel()  # an entry of value zero behind the others
    i1 = torch.full((target.numel(), w), none, device=DEV)
    i2 = torch.full((target.numel(), w), none, device=DEV)
    i1[mine, slot], i2[mine, slot] = e1, e2
    diag = torch.searchsorted(key, col * (n + 1))
    low = col < row
    f = torch.cat([val, val.new_zeros(1)])
    for _ in range(20000):
        new = val.clone()
        new[target] -= (f[i1] * f[i2]).sum(1)
        new = torch.where(low, new / f[diag], new)
        if bool((new - f[:-1]).abs().max() <= 1e-16 * new.abs().max()):
            break
        f = torch.cat([new, val.new_zeros(1)])
    return n, row, col, new


def _split(n, row, col, f):
    """(row, col, value) of the unit lower and of the upper factor."""
    low, up = col < row, col >= row
    i = torch.arange(n, device=DEV)
    key = torch.cat([row[low] * n + col[low], i * (n + 1)])
    val = torch.cat([f[low], torch.ones(n, dtype=torch.float64, device=DEV)])
    order = torch.argsort(key)
    return (key[order] // n, key[order] % n, val[order]), (row[up], col[up], f[up])


def _extended(case, A):
    """The Schwarz system: (ext_ptr, ext2glob, owned, block-diagonal matrix)."""
    n = A[0].numel() - 1
    part, nsub = _boxes(case, case["bx"], case["by"], case["bz"])
    part, row, col = part.long(), _rows(A[0]), A[1].long()
    key = torch.unique(torch.cat([part[row] * n + col, part * n + torch.arange(n, device=DEV)]))
    sub, glob = key // n, key % n
    count = A[0].long().diff()[glob]
    e = torch.repeat_interleave(torch.arange(key.numel(), device=DEV), count)
    src = A[0].long()[glob][e] + torch.arange(e.numel(), device=DEV) - (count.cumsum(0) - count)[e]
    want = sub[e] * n + col[src]
    at = torch.searchsorted(key, want).clamp(max=key.numel() - 1)
    hit = key[at] == want
    rowptr = torch.zeros(key.numel() + 1, dtype=torch.int32, device=DEV)
    rowptr[1:] = torch.bincount(e[hit], minlength=key.numel()).cumsum(0).to(torch.int32)
    ext_ptr = torch.searchsorted(sub, torch.arange(nsub + 1, device=DEV))
    return ext_ptr, glob, part[glob] == sub, (rowptr, at[hit].to(torch.int32), A[2][src[hit]])


def _apply(A, b, vdt):
    n, row, col, f = _factors(A)
    L, U = _split(n, row, col, f)
    y = _solve(n, L[0], L[1], _rounded(L[2], vdt), b)
    return y, _solve(n, U[0], U[1], _rounded(U[2], vdt), y)


def _exact_net(case, seed):
    x, target, params = _net_inputs(case, seed)
    nx, ny, zs = case["nx"], case["ny"], case["zs"]
    p = torch.tensor(params, device=DEV, dtype=torch.float64).reshape(4, learn.LAYER).requires_grad_()
    a = x.double().reshape(-1, zs, ny, nx, learn.C)
    for layer in range(4):
        wgt = p[layer, :27 * learn.C * learn.C].reshape(27, learn.C, learn.C)
        pad = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1, 1, 1))
        a = p[layer, 27 * learn.C * learn.C:] + sum(
            pad[:, dz:dz + zs, dy:dy + ny, dx:dx + nx] @ wgt[(dz * 3 + dy) * 3 + dx]
            for dz in range(3) for dy in range(3) for dx in range(3))
        a = torch.relu(a) if layer < 3 else a
    loss = ((a[..., 0].reshape(-1) - target.double()) ** 2).mean()
    loss.backward()
    return loss.item(), p.grad.reshape(-1)


def exact(case, seed):
    op, vdt = case["op"], case["vdt"]
    if op == "net":
        return _exact_net(case, seed)
    if op == "ilut":  # a serial dual-threshold factorization: far too slow in plain torch
        return None
    A, b, c = _inputs(case, seed)
    n = A[0].numel() - 1
    row, col = _rows(A[0]), A[1].long()
    if op == "spmv":
        return _product(*_ell(n, row, col, A[2]), b)
    if op == "solve":  # b was made from c
        return c
    if op == "sgs":
        val = _rounded(A[2], vdt)
        lo, up = col < row, col > row
        x = _solve(n, row[~up], col[~up], val[~up], b - _product(*_ell(n, row[up], col[up], A[2][up]), c))
        return _solve(n, row[~lo], col[~lo], val[~lo], b - _product(*_ell(n, row[lo], col[lo], A[2][lo]), x))
    if op == "ilu":
        L, U = _split(*_factors(A, case["k"]))
        return None, None, L[2], None, None, U[2]
    if op in ("ras", "ras_setup"):
        _, glob, owned, E = _extended(case, A)
        z = torch.empty_like(b)
        z[glob[owned]] = _apply(E, b[glob], vdt)[1][owned]
        return z if op == "ras" else (None, None, None, z)
    y, x = _apply(A, b, vdt)
    if op == "setup":
        return x, _product(*_ell(n, row, col, A[2]), x)
    return (y, x) if op == "trsv" else x
