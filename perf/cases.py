"""The calls a user of the GenEO library makes, with their sizes.

A program that uses the library does one of three things: it builds a
preconditioner and solves with it (``setup_solve``: geneo_setup +
geneo_pcg_solve + geneo_destroy, the benchmark's step), it solves with a
handle that stays resident (``solve``: one to eight right-hand sides in one
geneo_pcg_solve, the serving trace's request), or it applies M^{-1} inside an
iteration of its own (``apply``: geneo_apply).  The problem families are the
ones of the tests, the benchmark and the serving trace:

* ``darcy2d``: 2D Darcy, channels and inclusions at contrast 1e4 (at 1e6 the
  FP64 rounding of x keeps some of the larger grids above a residual of 1e-8),
  boxes of 16^2 elements, overlap 1, at most 10 eigenvectors;
* ``darcy3d``: 3D Darcy, kappa = exp(Gaussian field) with four slabs at 1e6,
  boxes of about 16^3 elements, overlap 2, at most 20 eigenvectors;
* ``laminate``: 3D elasticity of a fibre/resin laminate, boxes of about 12^3
  elements, overlap 2, at most 30 eigenvectors;
* ``uneven``: 3D Darcy on an irregular k-d partition (sides 6-20 elements),
  overlap 1-3 per box, one inclusion of contrast 1e2-1e6 per box.

Right-hand sides are loads: a constant source (or body force) and a few
smooth ones of random place, width and sign.  Everything solves to a true
residual of 1e-8.  Precisions: FP64 is the library's default, FP32 (mixed
precision) is what the benchmark and the serving trace use.
"""
import math

import numpy as np
import torch

import gen
from paper_1906_10944_gb300 import geneo as G

TOL = 1e-8
FAMILY = {
    # family: (box side, overlap, nev_max, dofs per node)
    "darcy2d": (16, 1, 10, 1),
    "darcy3d": (16, 2, 20, 1),
    "laminate": (12, 2, 30, 3),
    "uneven": (13, None, 20, 1),
}


def _case(name, kind, family, nel, prec, nrhs=1):
    nx, ny, nz = (tuple(nel) + (0,))[:3]
    c = {"kind": kind, "family": family, "nx": nx, "ny": ny, "nz": nz, "prec": prec, "nrhs": nrhs}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a handle of the smallest 2D configuration solving one load: latency and launches
        _case("solve_2d_64", "solve", "darcy2d", (64, 64), "fp64"),
        # the same configuration from its matrices to the solution (default options)
        _case("setup_2d_64", "setup_solve", "darcy2d", (64, 64), "fp64"),
        # serving: the smallest 3D request, one right-hand side on a resident handle
        _case("serve_32_r1", "solve", "darcy3d", (32, 32, 32), "fp32"),
        # serving: an ordinary size with the most right-hand sides a request brings
        _case("serve_64_r8", "solve", "darcy3d", (64, 64, 64), "fp32", 8),
        # serving: a large ragged grid, an odd number of right-hand sides
        _case("serve_99_r3", "solve", "darcy3d", (99, 96, 90), "fp32", 3),
        # serving: elasticity, one right-hand side
        _case("serve_el32_r1", "solve", "laminate", (32, 32, 32), "fp32"),
        # admission of a new elasticity problem and its first solve, ragged boxes
        _case("setup_el38", "setup_solve", "laminate", (38, 31, 24), "fp32"),
        # uneven boxes, widths and overlaps in one batch, some of them factored again in FP64
        _case("setup_uneven_44", "setup_solve", "uneven", (44, 40, 36), "fp32"),
        # FP64 throughout (the default precision) on a 3D problem
        _case("setup_48_fp64", "setup_solve", "darcy3d", (48, 48, 48), "fp64"),
        # M^{-1} r in FP64 for a caller's own Krylov iteration
        _case("apply_64_fp64", "apply", "darcy3d", (64, 64, 64), "fp64"),
        # an ordinary size from its matrices to the solution, mixed precision
        _case("setup_64", "setup_solve", "darcy3d", (64, 64, 64), "fp32"),
        # the benchmark's step: 2.1 million dofs, 512 subdomains
        _case("setup_128", "setup_solve", "darcy3d", (128, 128, 128), "fp32"),
    ]


def draw(rng):
    """One more case: kind, family and precision by how often programs use
    them, grids of any (ragged) size over the family's range."""
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi, most):
        """A grid whose mean side lies in [lo, hi] (over the logarithm), its
        sides within a sixth of it, at most ``most`` each."""
        m = side(lo, hi)
        return tuple(max(lo, min(most, m + rng.randint(-(m // 6), m // 6))) for _ in range(3))

    kind = rng.choice(["solve", "solve", "solve", "setup_solve", "setup_solve", "apply"])
    if kind == "apply":
        return _case(None, kind, "darcy3d", box(24, 72, 72), "fp64", rng.choice([1, 1, 2, 3]))
    nrhs = 1 if kind == "setup_solve" else rng.choice([1, 1, 2, 3, 4, 5, 6, 8])
    family = rng.choice(["darcy3d", "darcy3d", "darcy3d", "laminate", "laminate", "uneven", "darcy2d"])
    if family == "darcy2d":
        return _case(None, kind, family, (side(40, 320), side(40, 320)), rng.choice(["fp64", "fp32"]), nrhs)
    if family == "laminate":
        hi = 52 if kind == "solve" else 38
        return _case(None, kind, family, box(20, hi, hi), "fp32", nrhs)
    if family == "uneven":
        return _case(None, kind, family, box(24, 40, 44), "fp32", nrhs)
    prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
    hi = 120 if prec == "fp32" else (64 if kind == "solve" else 48)
    return _case(None, kind, family, box(24, hi, hi), prec, nrhs)


# ----------------------------------------------------------------------------
# Inputs, made on the device from the seed
# ----------------------------------------------------------------------------
def _nel(case):
    return tuple(v for v in (case["nx"], case["ny"], case["nz"]) if v)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _splits(n, p):
    return [(n * i) // p for i in range(p + 1)]


def _boxes(case, seed):
    """Element boxes (lo, hi) of the subdomains, grown by their overlap."""
    nel = _nel(case)
    side, overlap, _, _ = FAMILY[case["family"]]
    if case["family"] == "uneven":
        n = max(4, round(float(np.prod(nel)) / side ** 3))
        cores = gen.kd_partition(nel, n, 6, 20, seed)
        rng = np.random.default_rng(seed)
        over = [int(v) for v in rng.integers(1, 4, len(cores))]
    else:
        cores, _ = gen.box_partition(nel, tuple(max(1, round(v / side)) for v in nel), 0)
        over = [overlap] * len(cores)
    grown = [(tuple(max(0, a - o) for a in lo), tuple(min(m, b + o) for b, m in zip(hi, nel)))
             for (lo, hi), o in zip(cores, over)]
    return cores, grown


def _coefficient(case, seed, cores):
    """kappa per element, x fastest (Darcy families)."""
    nel = _nel(case)
    if case["family"] == "darcy2d":
        return torch.from_numpy(gen.kappa_channels_2d(nel, seed=seed, contrast=1e4)).cuda().reshape(-1)
    if case["family"] == "uneven":
        rng = np.random.default_rng(seed + 1)
        kap = np.ones(nel[::-1])
        for lo, hi in cores:
            a = [int(rng.integers(lo[d], max(lo[d] + 1, hi[d] - 1))) for d in range(3)]
            b = [min(hi[d], a[d] + int(rng.integers(1, max(2, (hi[d] - lo[d]) // 2)))) for d in range(3)]
            kap[a[2]:b[2], a[1]:b[1], a[0]:b[0]] = 10.0 ** rng.uniform(2.0, 6.0)
        return torch.from_numpy(kap).cuda().reshape(-1)
    # stationary Gaussian field, covariance 4 exp(-r / 0.1), by circulant embedding
    m = [2 * v for v in nel[::-1]]
    axes = [torch.minimum(torch.arange(v, device="cuda"), v - torch.arange(v, device="cuda")).double() / nel[0]
            for v in m]
    r = torch.sqrt(axes[0][:, None, None] ** 2 + axes[1][None, :, None] ** 2 + axes[2][None, None, :] ** 2)
    lam = torch.fft.fftn(4.0 * torch.exp(-r / 0.1)).real.clamp_min(0.0)
    g = _gen(seed)
    xi = torch.complex(torch.randn(m, generator=g, device="cuda", dtype=torch.float64),
                       torch.randn(m, generator=g, device="cuda", dtype=torch.float64))
    field = torch.fft.fftn(torch.sqrt(lam / lam.numel()) * xi).real
    k = torch.exp(field[tuple(slice(0, v) for v in nel[::-1])])
    for z0 in (24, 56, 88, 120):
        z = (z0 * nel[2]) // 128
        k[z:z + 2] *= 1e6
    return k.reshape(-1)


def _element_matrices(case, seed, cores):
    """Unconstrained element matrices [n_elem, k, k] and a mesh width."""
    nel = _nel(case)
    if case["family"] != "laminate":
        h = 1.0 / nel[0]
        ref = torch.from_numpy(gen.q1_reference_stiffness(len(nel), h)).cuda()
        return _coefficient(case, seed, cores)[:, None, None] * ref, h
    h = 1.0 / nel[2]
    fib = gen.orthotropic_stiffness(135.0, 10.0, 10.0, 0.3, 0.3, 0.4, 5.0, 5.0, 10.0 / 2.8)
    turn = [1, 0, 2, 4, 3, 5]
    table = torch.from_numpy(np.stack([
        gen.q1_elasticity_element(c, h)
        for c in (gen.isotropic_stiffness(3.0, 0.35), fib, fib[np.ix_(turn, turn)])])).cuda()
    # layers of two elements: fibre at 0 or 90 degrees (drawn), resin of drawn modulus
    rng = np.random.default_rng(seed)
    layer = np.arange(nel[2]) // 2
    nl = int(layer[-1]) + 1
    orient, scale = rng.integers(1, 3, nl), 2.0 ** rng.uniform(-1.0, 1.0, nl)
    kind = np.where(layer % 2 == 1, 0, orient[layer])
    fac = np.where(kind == 0, scale[layer], 1.0)
    per_z = table[torch.from_numpy(kind).cuda()] * torch.from_numpy(fac).cuda()[:, None, None]
    return per_z.repeat_interleave(nel[0] * nel[1], dim=0), h


def _grid(dims):
    """Coordinates (x fastest) of the points of a dims-sized grid."""
    total = int(np.prod(dims))
    i, out = torch.arange(total, device="cuda"), []
    for d in dims:
        out.append(i % d)
        i = i // d
    return out


def _matrix(nel, ndn, elem_mats, dirichlet_nodes):
    """CSR of the assembled matrix (Dirichlet rows and columns eliminated, the
    full element pattern kept) and the element -> dof table."""
    dim = len(nel)
    nn = [v + 1 for v in nel]
    node = _grid(nn)
    strides = [1, nn[0], nn[0] * nn[1]][:dim]
    lo = [(c > 0).long() for c in node]                                  # neighbours below
    cnt = [1 + l + (c < v - 1).long() for l, c, v in zip(lo, node, nn)]  # neighbours per direction
    deg = cnt[0] * cnt[1] * (cnt[2] if dim == 3 else 1)
    n_nodes = int(np.prod(nn))
    per_row = (deg * ndn).repeat_interleave(ndn)
    row_ptr = torch.zeros(n_nodes * ndn + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(per_row, 0, out=row_ptr[1:])
    first = row_ptr[:-1].reshape(n_nodes, ndn)[:, 0]                     # first entry of a node's rows
    nnz = int(row_ptr[-1])
    col = torch.zeros(nnz, dtype=torch.int32, device="cuda")
    val = torch.zeros(nnz, dtype=torch.float64, device="cuda")
    ids = torch.arange(n_nodes, device="cuda")

    def entry(at, off, c, cc):
        """Position of (node at, comp c) -> (node at + off, comp cc)."""
        slot = torch.zeros_like(at)
        for d in reversed(range(dim)):
            slot = slot * cnt[d][at] + (off[d] + lo[d][at])
        return first[at] + c * ndn * deg[at] + ndn * slot + cc

    offs = [(x, y, z) for z in ((-1, 0, 1) if dim == 3 else (0,)) for y in (-1, 0, 1) for x in (-1, 0, 1)]
    for off in offs:
        ok = torch.ones(n_nodes, dtype=torch.bool, device="cuda")
        for d in range(dim):
            ok &= (node[d] + off[d] >= 0) & (node[d] + off[d] < nn[d])
        at = ids[ok]
        to = at + sum(off[d] * strides[d] for d in range(dim))
        for c in range(ndn):
            for cc in range(ndn):
                col[entry(at, off, c, cc)] = (to * ndn + cc).int()
    lower = sum(c * s for c, s in zip(_grid(nel), strides))
    bits = [[(a >> d) & 1 for d in range(dim)] for a in range(2 ** dim)]
    nodes = torch.stack([lower + sum(b * s for b, s in zip(bb, strides)) for bb in bits], dim=1)
    for a in range(2 ** dim):
        for b in range(2 ** dim):
            off = [bits[b][d] - bits[a][d] for d in range(dim)]
            for c in range(ndn):
                for cc in range(ndn):  # one entry per element: no two of them meet
                    e = entry(nodes[:, a], off, c, cc)
                    val[e] = val[e] + elem_mats[:, a * ndn + c, b * ndn + cc]
    elem_dofs = (nodes[:, :, None] * ndn + torch.arange(ndn, device="cuda")).reshape(nodes.shape[0], -1).int()
    dirichlet = dirichlet_nodes.repeat_interleave(ndn)
    rows = torch.repeat_interleave(torch.arange(n_nodes * ndn, device="cuda"), per_row)
    hit = dirichlet[rows] | dirichlet[col.long()]
    val[hit] = 0.0
    val[hit & (rows == col)] = 1.0
    return row_ptr, col, val, elem_dofs, dirichlet


def _lists(nel, ndn, grown, dirichlet):
    """Elements and free dofs of every subdomain, each list ascending."""
    dim = len(nel)
    nn = [v + 1 for v in nel]
    es, ns = [1, nel[0], nel[0] * nel[1]][:dim], [1, nn[0], nn[0] * nn[1]][:dim]

    def ids(lo, hi, strides):
        out = np.zeros(1, dtype=np.int64)
        for d in reversed(range(dim)):
            out = (out[:, None] + np.arange(lo[d], hi[d]) * strides[d]).reshape(-1)
        return out

    free = ~dirichlet.cpu().numpy()
    se, sd = [], []
    for lo, hi in grown:
        se.append(ids(lo, hi, es))
        dofs = (ids(lo, [v + 1 for v in hi], ns)[:, None] * ndn + np.arange(ndn)).reshape(-1)
        sd.append(dofs[free[dofs]])
    ptr = [torch.from_numpy(np.concatenate([[0], np.cumsum([v.size for v in x])])).cuda() for x in (se, sd)]
    return (ptr[0], torch.from_numpy(np.concatenate(se).astype(np.int32)).cuda(),
            ptr[1], torch.from_numpy(np.concatenate(sd).astype(np.int32)).cuda())


def _loads(case, seed, h, dirichlet):
    """nrhs load vectors (stride n): a constant plus four smooth sources each."""
    nel = _nel(case)
    dim, ndn = len(nel), FAMILY[case["family"]][3]
    node = [c.double() / max(nel) for c in _grid([v + 1 for v in nel])]
    rng = np.random.default_rng(seed + 7)
    out = torch.zeros(case["nrhs"], node[0].numel(), ndn, dtype=torch.float64, device="cuda")
    for k in range(case["nrhs"]):
        if ndn == 1:
            out[k] = 1.0
        else:
            out[k, :, 2] = -1.0
        for _ in range(4):
            at = [rng.uniform(0.1, 0.9) * v / max(nel) for v in nel]
            r2 = sum((c - a) ** 2 for c, a in zip(node, at))
            bump = torch.exp(-r2 / (2.0 * rng.uniform(0.08, 0.3) ** 2))
            for c in range(ndn):
                out[k, :, c] += float(rng.uniform(-3.0, 3.0)) * bump
    out = out.reshape(case["nrhs"], -1) * h ** dim
    out[:, dirichlet] = 0.0
    return out.contiguous()


def _inputs(case, seed):
    nel = _nel(case)
    dim, ndn = len(nel), FAMILY[case["family"]][3]
    cores, grown = _boxes(case, seed)
    mats, h = _element_matrices(case, seed, cores)
    node = _grid([v + 1 for v in nel])
    if case["family"] == "laminate":
        on = node[0] == 0                                   # clamped at x = 0
    else:
        on = torch.zeros_like(node[0], dtype=torch.bool)    # u = 0 on the whole boundary
        for c, v in zip(node, nel):
            on |= (c == 0) | (c == v)
    row_ptr, col, val, elem_dofs, dirichlet = _matrix(nel, ndn, mats, on)
    sep, se, sdp, sd = _lists(nel, ndn, grown, dirichlet)
    arrays = {"row_ptr": row_ptr, "col": col, "val": val, "dirichlet": dirichlet.to(torch.uint8),
              "elem_dofs": elem_dofs.contiguous(), "elem_mats": mats.contiguous(),
              "sub_elem_ptr": sep, "sub_elem": se, "sub_dof_ptr": sdp, "sub_dof": sd}
    return arrays, len(grown), ndn, _loads(case, seed, h, dirichlet)


class _State:
    """A program's problem, options, vectors and (resident kinds) handle."""

    def __init__(self, case, seed):
        self.kind, self.nrhs = case["kind"], case["nrhs"]
        self.arrays, n_sub, ndn, self.b = _inputs(case, seed)
        self.x = torch.zeros_like(self.b)
        n = self.b.shape[1]
        self.problem = G.make_problem(self.arrays, n, n_sub, self.arrays["elem_dofs"].shape[1], ndn,
                                      G.GENEO_MEM_DEVICE)
        self.options = G.geneo_default_options(
            nev_max=FAMILY[case["family"]][2], tau=0.3,
            precision=G.GENEO_PREC_FP32 if case["prec"] == "fp32" else G.GENEO_PREC_FP64)
        self.h = None
        if self.kind != "setup_solve":
            self.h = G.geneo_setup(self.problem, self.options)
            self.arrays = self.problem = None  # the handle has its own copies

    def __del__(self):
        if self.h:
            G.geneo_destroy(self.h)
            self.h = None


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    if state.kind == "apply":
        G.geneo_apply(state.h, state.b, state.x, state.nrhs)
        return state.x
    if state.kind == "solve":
        G.geneo_pcg_solve(state.h, state.b, state.x, state.nrhs, TOL, 2000)
        return state.x
    h = G.geneo_setup(state.problem, state.options)
    try:
        G.geneo_pcg_solve(h, state.b, state.x, state.nrhs, TOL, 2000)
        return {"x": state.x, "dim_coarse": G.geneo_query(h)["dim_coarse"]}
    finally:
        G.geneo_destroy(h)


def work(case):
    """What one pass cannot do without: every input once, every output once;
    for a solve A and one copy of the subdomain factors once per iteration
    (50 iterations, what these problems take), for a setup the band Cholesky
    factorisations of the A_j and K_j."""
    nel = _nel(case)
    side, overlap, nev, ndn = FAMILY[case["family"]]
    dim, esz = len(nel), (4.0 if case["prec"] == "fp32" else 8.0)
    n = ndn * float(np.prod([v + 1 for v in nel]))
    nnz = n * ndn * 3 ** dim
    k = ndn * 2 ** dim
    elems = float(np.prod(nel))
    # the grown boxes: their sides clipped to the grid
    parts = [max(1, round(v / side)) for v in nel]
    subs = float(np.prod(parts))
    grown = [min(v, v / p + 2 * (overlap or 2)) for v, p in zip(nel, parts)]
    rows = ndn * float(np.prod([g + 1 for g in grown]))
    width = ndn * (float(np.prod([g + 1 for g in grown[:-1]])) + sum(1 for _ in grown))
    factor = subs * rows * width
    vec = 16.0 * n * case["nrhs"]
    one = 12.0 * nnz + esz * factor
    if case["kind"] == "apply":
        return {"bytes": esz * factor + vec, "flops": 4.0 * factor * case["nrhs"]}
    its = 50.0
    solve = {"bytes": its * one + vec, "flops": its * case["nrhs"] * (2.0 * nnz + 4.0 * factor)}
    if case["kind"] == "solve":
        return solve
    inputs = 12.0 * nnz + elems * (8.0 * k * k + 4.0 * k) + 4.0 * subs * (rows / ndn + rows)
    return {"bytes": inputs + solve["bytes"], "flops": 2.0 * factor * width + solve["flops"]}


def exact(case, seed):
    """The solution of A x = b in 64 bits: a dense Cholesky for small systems,
    Jacobi-preconditioned CG restarted on its true residual otherwise.  The
    preconditioner itself (apply) depends on the eigenvectors a solver
    returns, so its result has no such value."""
    if case["kind"] == "apply":
        return None
    arrays, _, _, b = _inputs(case, seed)
    n = b.shape[1]
    a = torch.sparse_csr_tensor(arrays["row_ptr"], arrays["col"].long(), arrays["val"], size=(n, n))
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), arrays["row_ptr"].diff())
    diag = torch.zeros(n, dtype=torch.float64, device="cuda")
    on = rows == arrays["col"]
    diag[rows[on]] = arrays["val"][on]
    s = diag.rsqrt()
    scaled = torch.sparse_csr_tensor(arrays["row_ptr"], arrays["col"].long(),
                                     arrays["val"] * s[rows] * s[arrays["col"].long()], size=(n, n))
    del rows, on
    x = torch.zeros(n, b.shape[0], dtype=torch.float64, device="cuda")
    rhs = b.t().contiguous()
    if n <= 12000:
        low = torch.linalg.cholesky(scaled.to_dense())
        for _ in range(4):
            r = (rhs - a @ x) * s[:, None]
            x += s[:, None] * torch.cholesky_solve(r, low)
    else:
        left = 24000 if n < 400000 else 7000
        for _ in range(6):
            r = (rhs - a @ x) * s[:, None]
            y, p, rr = torch.zeros_like(r), r.clone(), (r * r).sum(0)
            start, step = rr.clone(), 0
            while left > 0:
                q = scaled @ p
                alpha = rr / (p * q).sum(0).clamp_min(1e-300)
                y += alpha * p
                r -= alpha * q
                new = (r * r).sum(0)
                p = r + (new / rr.clamp_min(1e-300)) * p
                rr = new
                step, left = step + 1, left - 1
                if step % 50 == 0 and bool((rr <= 1e-22 * start).all()):
                    break
            x += s[:, None] * y
            if left <= 0:
                return None  # would take too long
    x = x.t().contiguous()
    return x if case["kind"] == "solve" else {"x": x, "dim_coarse": None}
