"""The work that users of the DDLR library have it do, as measurable cases.

Every case goes through the public classes ``DDLR`` and ``Server``.  A case is
a dict of plain values:

kind       what one pass does with the prepared state:
             solve  ``DDLR.pcg`` on new right-hand sides (the handle is kept)
             build  ``DDLR.refactor`` with new matrix values, then ``DDLR.pcg``
             new    a new handle from host arrays, ``DDLR.pcg`` on a host
                    vector, the handle closed
             apply  ``DDLR.apply``, the preconditioner inside a caller's own
                    Krylov loop
             gmres  ``DDLR.gmres`` on an indefinite matrix
             serve  requests of several models through one ``Server``
matrix     lap   unscaled 5/7-point Laplacian, Dirichlet boundary
           jump  7-point finite volumes, cell coefficient 10^u per 8^3 block
           shift the Laplacian minus sigma I
nx, ny, nz / px, py, pz   grid and boxes per axis (nz = pz = 1: two dimensions);
           cuts "equal" (at floor(i N / P)) or "random" (drawn from the case)
k, variant, factor, order, precision, nrhs   as the library's options
           (order: multicolour or natural for the interior blocks and C_a;
           precision: f64, f32 or bf16 for a mixed handle with that U_k)
"""
import math

import numpy as np
import torch

import paper_1505_04341_gb300 as pkg

TOL = 1e-8


# ------------------------------------------------------------------- the cases
def _case(name, kind, shape, boxes, **kw):
    c = dict(name=name, kind=kind, matrix="lap", nx=shape[0], ny=shape[1], nz=shape[2], px=boxes[0], py=boxes[1],
             pz=boxes[2], cuts="equal", k=16, variant=1, factor=0, order="multicolour", precision="f64", nrhs=1)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest problem of the benchmark's configurations: a 2-D grid
        # with exact local factors, where latency and launches are everything
        _case("solve_2d_64_exact", "solve", (64, 64, 1), (2, 2, 1), k=8, factor=1, order="natural"),
        # one right-hand side on the smallest model of the serving stream
        _case("solve_32", "solve", (32, 32, 32), (2, 2, 2)),
        # a user who sets no options: natural elimination orders, deep factors
        _case("solve_64_defaults", "solve", (64, 64, 64), (4, 4, 4), order="natural"),
        # new matrix values on the middle grid (a time step or a Newton step),
        # preconditioner rebuilt, DDLR-2
        _case("build_64_ddlr2", "build", (64, 64, 64), (4, 4, 4), k=32, variant=2),
        # the benchmark's headline: device setup and solve of the 128^3 grid
        _case("build_128", "build", (128, 128, 128), (8, 8, 8), k=32),
        # the same grid in mixed precision, the handle kept between solves
        _case("solve_128_bf16", "solve", (128, 128, 128), (8, 8, 8), k=32, precision="bf16"),
        # a caller's own Krylov loop on the largest grid: one M^-1 x
        _case("apply_128", "apply", (128, 128, 128), (8, 8, 8), k=32),
        # the same call on a small ragged grid, the lowest latency there is
        _case("apply_33x17x21", "apply", (33, 17, 21), (3, 2, 2), k=8),
        # many right-hand sides at once on jump coefficients with uneven
        # boxes, FP32 preconditioner inside FP64 flexible CG
        _case("batch_jump_96", "solve", (96, 96, 96), (5, 5, 5), matrix="jump", cuts="random", k=24,
              precision="f32", nrhs=32, contrast=1.0),
        # an indefinite problem: GMRES(40) with a preconditioner that is not SPD
        _case("gmres_32", "gmres", (32, 32, 32), (2, 2, 2), matrix="shift", sigma=0.035, k=32),
        # the first solve with a matrix that the library has not seen, from
        # host arrays to a host solution (host analysis, copies, setup, PCG)
        _case("new_96", "new", (96, 96, 96), (6, 6, 6)),
        # a burst of requests over three resident models, batched by the server
        _case("serve_24", "serve", (64, 64, 64), (4, 4, 4), requests=24, edge0=32, edge1=48),
    ]


def draw(rng):
    """One more case of the same families: grid edges from 16 to 128 (drawn on
    a logarithmic scale, unequal and odd ones among them), boxes of about 10
    to 20 nodes per edge, every order, precision, variant and width in use;
    two-dimensional grids up to 64 by 64."""
    kind = rng.choice(["solve", "solve", "solve", "build", "build", "apply", "apply", "batch", "gmres", "new", "serve"])
    top = {"solve": 128, "build": 112, "apply": 128, "batch": 80, "gmres": 40, "new": 80, "serve": 64}[kind]
    order = "natural" if kind in ("solve", "build", "new") and rng.random() < 0.25 else "multicolour"
    if order == "natural":
        top = 64
    edge = math.exp(rng.uniform(math.log(20), math.log(top)))
    shape = [max(16, min(top, int(round(edge * rng.uniform(0.8, 1.2))))) for _ in range(3)]
    width = rng.uniform(10, 20)
    boxes = [max(2, int(round(e / width))) for e in shape]
    kw = dict(k=rng.choice([4, 8, 12, 16, 20, 24, 32]), order=order, variant=rng.choice([1, 1, 2]))
    if kind == "apply":
        kw["variant"] = 1
        kw["nrhs"] = rng.choice([1, 1, 1, 5, 8])
    elif kind == "batch":
        kind = "solve"
        kw["nrhs"] = rng.choice([2, 5, 8, 16, 31])
        kw["precision"] = rng.choice(["f64", "f32", "bf16"])
        if rng.random() < 0.5:
            kw.update(matrix="jump", contrast=1.0)
    elif kind == "solve":
        kw["precision"] = rng.choice(["f64", "f64", "f32", "bf16"])
        if rng.random() < 0.25:
            e = rng.randint(16, 64)
            shape, boxes = [e, max(16, e - rng.randint(0, 12)), 1], [2, rng.choice([2, 3]), 1]
            kw.update(factor=1, order="natural", k=rng.choice([4, 8]), precision="f64", variant=1)
    elif kind == "gmres":
        # 1.3 times the smallest eigenvalue: below the second one on these grids
        sigma = 1.3 * sum(2 - 2 * math.cos(math.pi / (e + 1)) for e in shape)
        kw.update(matrix="shift", sigma=sigma, variant=1, k=rng.choice([16, 32]))
    elif kind == "serve":
        kw.update(variant=1, k=16, requests=rng.randint(4, 24), edge0=rng.choice([16, 24, 32]),
                  edge1=rng.choice([40, 48]))
        shape, boxes = [shape[0]] * 3, [boxes[0]] * 3
    c = _case("", kind, shape, boxes, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------ the inputs
def _shape(c):
    return (c["nx"], c["ny"], c["nz"])


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _cuts(c, N, P, axis):
    """The P + 1 cut positions of an axis of N nodes."""
    if c["cuts"] == "equal" or P == 1:
        return [i * N // P for i in range(P + 1)]
    rng = np.random.RandomState(1000 * axis + N + P)
    while True:                                        # every width within 8 to 32 nodes
        cut = np.concatenate([[0], np.sort(rng.choice(np.arange(1, N), P - 1, replace=False)), [N]])
        if 8 <= np.diff(cut).min() and np.diff(cut).max() <= 32:
            return cut.tolist()


def _part(c):
    """Box of every node as an (nz, ny, nx) tensor, and the number of boxes."""
    idx = []
    for axis, (N, P) in enumerate(zip(_shape(c), (c["px"], c["py"], c["pz"]))):
        cut = torch.tensor(_cuts(c, N, P, axis)[1:-1], dtype=torch.int64)
        idx.append(torch.bucketize(torch.arange(N), cut, right=True))
    x, y, z = idx
    part = x[None, None, :] + c["px"] * (y[None, :, None] + c["py"] * z[:, None, None])
    return part.to(torch.int32).cuda(), c["px"] * c["py"] * c["pz"]


def _operator(c, seed):
    """The matrix on the grid: its diagonal (nz, ny, nx) and the weights of the
    couplings to the next node along x, y and z (zero past the last node)."""
    shape = (c["nz"], c["ny"], c["nx"])
    one = torch.ones(shape, dtype=torch.float64, device="cuda")
    if c["matrix"] == "jump":
        blocks = [(e + 7) // 8 for e in shape]
        u = (2 * torch.rand(blocks, generator=_gen(seed), dtype=torch.float64, device="cuda") - 1) * c["contrast"]
        kap = 10.0 ** u
        for a in range(3):
            kap = kap.repeat_interleave(8, dim=a).narrow(a, 0, shape[a])
        kap = kap.contiguous()
    else:
        kap = one
        if c["kind"] == "build":
            # other values on the same pattern: the operator of another step size
            kap = one * (0.5 + torch.rand((), generator=_gen(seed), dtype=torch.float64, device="cuda"))
    diag = torch.zeros_like(one)
    off = []
    for a in (2, 1, 0):
        if shape[a] == 1:
            off.append(torch.zeros_like(one))
            continue
        lo, hi = kap.narrow(a, 0, shape[a] - 1), kap.narrow(a, 1, shape[a] - 1)
        t = 2 * lo * hi / (lo + hi)
        w = torch.zeros_like(one)
        w.narrow(a, 0, shape[a] - 1).copy_(t)
        off.append(w)
        diag.narrow(a, 0, shape[a] - 1).add_(t)
        diag.narrow(a, 1, shape[a] - 1).add_(t)
        edge = 2.0 if c["matrix"] == "jump" else 1.0   # the boundary face: half a cell away, or a whole node
        diag.select(a, 0).add_(edge * kap.select(a, 0))
        diag.select(a, shape[a] - 1).add_(edge * kap.select(a, shape[a] - 1))
    if c["matrix"] == "shift":
        diag -= c["sigma"]
    return diag, off


def _shifted(w, a, shape):
    """w moved one node up along axis a: the coupling to the previous node."""
    out = torch.zeros_like(w)
    if shape[a] > 1:
        out.narrow(a, 1, shape[a] - 1).copy_(w.narrow(a, 0, shape[a] - 1))
    return out


def _csr(c, diag, off):
    """Host CSR (n, rowptr, colind, val) with ascending columns, and the values
    as a device tensor in the same order."""
    shape = (c["nz"], c["ny"], c["nx"])
    n = diag.numel()
    g = torch.arange(n, device="cuda")
    steps = (1, shape[2], shape[1] * shape[2])
    up = [w.reshape(-1) for w in off]
    dn = [_shifted(w, a, shape).reshape(-1) for w, a in zip(off, (2, 1, 0))]
    cols = torch.stack([g - steps[2], g - steps[1], g - steps[0], g, g + steps[0], g + steps[1], g + steps[2]], 1)
    vals = torch.stack([-dn[2], -dn[1], -dn[0], diag.reshape(-1), -up[0], -up[1], -up[2]], 1)
    there = vals != 0
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = there.sum(1).cumsum(0)
    val = vals[there]
    return (n, rowptr.to(torch.int32).cpu().numpy(), cols[there].to(torch.int32).cpu().numpy(),
            val.cpu().numpy()), val


def _rhs(c, seed):
    """Right-hand sides uniform in [-1, 1), column-major (n, nrhs) or a vector."""
    n = c["nx"] * c["ny"] * c["nz"]
    b = 2 * torch.rand((c["nrhs"], n), generator=_gen(seed + 7919), dtype=torch.float64, device="cuda") - 1
    return b[0].contiguous() if c["nrhs"] == 1 else b.T


def _options(c):
    order = 1 if c["order"] == "multicolour" else 0
    return dict(variant=c["variant"], rank_k=c["k"], factor=c["factor"], c_order=order, b_order=order,
                precision=0 if c["precision"] == "f64" else 1, uk_bf16=1 if c["precision"] == "bf16" else 0,
                scale_diag=1 if c["matrix"] == "jump" else 0, max_nrhs=c["nrhs"],
                indefinite=1 if c["matrix"] == "shift" else 0)


def _lowrank(c, s, seed):
    """Low-rank data as a program restores them from its checkpoint: k nearly
    orthonormal columns, Ritz values that fall from near 1, the next one."""
    k = c["k"]
    U = torch.randn((s, k), generator=_gen(seed + 104729), dtype=torch.float64, device="cuda") / math.sqrt(s)
    lam = 0.97 - 0.4 * torch.arange(k + 1, dtype=torch.float64) / k
    return U, lam[:k], float(lam[k])


def _edge_case(c, edge):
    boxes = max(2, edge // 16)
    return dict(c, kind="solve", nx=edge, ny=edge, nz=edge, px=boxes, py=boxes, pz=boxes)


def _requests(c):
    """(model, edge) of every request: an even mix in a shuffled order."""
    edges = [c["edge0"], c["edge1"], c["nx"]]
    pick = [i % 3 for i in range(c["requests"])]
    np.random.RandomState(c["requests"]).shuffle(pick)
    return [(i, edges[i]) for i in pick]


def prepare(case, seed):
    c = case
    if c["kind"] == "serve":
        srv = pkg.Server(max_concurrent=8, max_batch=16, tol=TOL)
        models = []
        for edge in (c["edge0"], c["edge1"], c["nx"]):
            ce = _edge_case(c, edge)
            A, _ = _csr(ce, *_operator(ce, seed))
            part, p = _part(ce)
            models.append(srv.add_model(A, part.reshape(-1).cpu().numpy(), p, **_options(ce)))
        reqs = [(models[i], edge, _rhs(_edge_case(c, edge), seed + 31 * j).cpu().numpy())
                for j, (i, edge) in enumerate(_requests(c))]
        return dict(kind="serve", server=srv, requests=reqs)
    diag, off = _operator(c, seed)
    A, val = _csr(c, diag, off)
    part, p = _part(c)
    part = part.reshape(-1).cpu().numpy()
    b = _rhs(c, seed)
    if c["kind"] == "new":
        return dict(kind="new", A=A, part=part, p=p, b=b.cpu().numpy(), options=_options(c))
    h = pkg.DDLR(A, part, p, **_options(c))
    if c["kind"] == "apply":
        U, lam, theta = _lowrank(c, h.info()["s"], seed)
        h.set_lowrank(U.cpu().numpy(), lam.numpy(), theta)
    x = torch.zeros_like(b) if c["nrhs"] == 1 else torch.zeros_like(b.T).T
    return dict(kind=c["kind"], handle=h, b=b, x=x, val=val)


# ------------------------------------------------------------------- one pass
def run(state):
    kind = state["kind"]
    if kind == "serve":
        srv = state["server"]
        ids = [srv.submit(m, b) for m, _, b in state["requests"]]
        got = [srv.wait(i, len(b)) for i, (_, _, b) in zip(ids, state["requests"])]
        return dict(x=[g[0] for g in got], its=np.array([g[1]["its"] for g in got]))
    if kind == "new":
        h = pkg.DDLR(state["A"], state["part"], state["p"], **state["options"])
        x, info = h.pcg(state["b"], tol=TOL)
        h.close()
        return dict(x=x, its=info[0]["its"])
    h, b, x = state["handle"], state["b"], state["x"]
    if kind == "apply":
        return h.apply(b, x)
    if kind == "gmres":
        x, info = h.gmres(b, x, tol=TOL, maxit=2000)
        return dict(x=x, its=info["its"])
    if kind == "build":
        h.refactor(state["val"])
    x, info = h.pcg(b, x, tol=TOL, maxit=2000)
    return dict(x=x, its=np.array([i["its"] for i in info]))


# ------------------------------------------------------------------- its floor
def _iterations(c):
    """About how many iterations such a solve takes (measured on the listed
    cases: they grow with the longest edge)."""
    edge = max(c["nx"], c["ny"], c["nz"])
    if c["kind"] == "gmres":
        return 6 * edge
    if c["factor"] == 1:
        return 0.5 * edge
    if c["matrix"] == "jump":
        return 3 * edge
    return (1.4 if c["order"] == "natural" else 1.75) * edge


def _sizes(c):
    """n, nonzeros of A, interface nodes and factor entries of the grid."""
    n = c["nx"] * c["ny"] * c["nz"]
    inner, nnz = 1, n
    for e, p in zip(_shape(c), (c["px"], c["py"], c["pz"])):
        inner *= e - 2 * (p - 1)
        nnz += 2 * n * (e - 1) // e
    return n, nnz, n - inner, (nnz + n) // 2


def _apply_work(c):
    """One M^-1 x for nrhs vectors: the factors once per solve with A0 (DDLR-1
    solves twice), U_k once for U_k^T y and once for the sum, vectors in and
    out."""
    n, nnz, s, nf = _sizes(c)
    v = 8 if c["precision"] == "f64" else 4
    u = {"f64": 8, "f32": 4, "bf16": 2}[c["precision"]]
    rows, solves = (s, 2) if c["variant"] == 1 else (n, 1)
    b = solves * nf * (v + 4) + 2 * rows * c["k"] * u + c["nrhs"] * 16 * n
    f = c["nrhs"] * (solves * 4 * nf + 4 * rows * c["k"])
    return b, f


def _solve_work(c):
    n, nnz, s, _ = _sizes(c)
    its, r = _iterations(c), c["nrhs"]
    b, f = _apply_work(c)
    b += 12 * nnz + r * 9 * 8 * n                        # A once, x, r, p, q, z of one iteration
    f += r * (2 * nnz + 12 * n)
    return its * b, its * f


def work(case):
    c = case
    n, nnz, s, nf = _sizes(c)
    if c["kind"] == "apply":
        b, f = _apply_work(c)
    elif c["kind"] == "serve":
        got = [_solve_work(_edge_case(c, e)) for _, e in _requests(c)]
        b, f = sum(g[0] for g in got), sum(g[1] for g in got)
    else:
        b, f = _solve_work(c)
        if c["kind"] in ("build", "new"):
            # 5k Lanczos steps: E, the solves with A0, E^T, and the earlier
            # vectors once for the reorthogonalisation; then the Ritz vectors
            m = 5 * c["k"]
            b += 12 * nnz + m * (c["variant"] * (12 * nf + 16 * n) + 4 * m * s) + 8 * s * (m + c["k"])
            f += m * (c["variant"] * 4 * nf + 2 * m * s) + 2 * s * m * c["k"]
    return dict(bytes=float(b), flops=float(f))


# ------------------------------------------- the same outputs in plain 64 bits
def _sine(N):
    i = torch.arange(1, N + 1, dtype=torch.float64, device="cuda")
    S = math.sqrt(2.0 / (N + 1)) * torch.sin(math.pi * i[:, None] * i[None, :] / (N + 1))
    return S, 2 - 2 * torch.cos(math.pi * i / (N + 1))


def _solve_by_sines(c, b, scale):
    """A^-1 b for the (shifted) Laplacian times scale, diagonalised by the
    discrete sine transform of each axis."""
    shape = (c["nz"], c["ny"], c["nx"])
    v = b.reshape((-1,) + shape)
    lam = torch.zeros(shape, dtype=torch.float64, device="cuda")
    S = []
    for a in range(3):
        M, e = (_sine(shape[a]) if shape[a] > 1
                else (torch.ones((1, 1), dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")))
        S.append(M)
        lam = lam + e.reshape([-1 if d == a else 1 for d in range(3)])
    lam = scale * lam - (c["sigma"] if c["matrix"] == "shift" else 0.0)

    def transform(t):
        t = torch.matmul(t, S[2])
        t = torch.matmul(S[1], t)
        return torch.tensordot(t, S[0], dims=([1], [0])).permute(0, 3, 1, 2)
    return transform(transform(v) / lam).reshape(b.shape[0], -1)


def _grid_product(diag, off, v):
    """A v on the grid; v: (r,) + shape."""
    out = diag * v
    for w, a in zip(off, (2, 1, 0)):
        N = diag.shape[a]
        if N == 1:
            continue
        wc = w.narrow(a, 0, N - 1)
        out.narrow(a + 1, 0, N - 1).sub_(wc * v.narrow(a + 1, 1, N - 1))
        out.narrow(a + 1, 1, N - 1).sub_(wc * v.narrow(a + 1, 0, N - 1))
    return out


def _solve_by_cg(diag, off, b):
    """A^-1 b by Jacobi preconditioned conjugate gradients to rounding."""
    b = b.reshape((-1,) + tuple(diag.shape))
    dot = lambda u, w: (u * w).flatten(1).sum(1).reshape(-1, 1, 1, 1)  # noqa: E731
    x, r = torch.zeros_like(b), b.clone()
    z = r / diag
    p, rz, bb = z.clone(), dot(r, z), dot(b, b)
    for it in range(4000):
        q = _grid_product(diag, off, p)
        a = rz / dot(p, q)
        x += a * p
        r -= a * q
        if it % 20 == 19 and float((dot(r, r) / bb).max()) < 1e-28:
            break
        z = r / diag
        new = dot(r, z)
        p = z + (new / rz) * p
        rz = new
    return x.flatten(1)


def _apply_exact(c, seed):
    """M^-1 x of DDLR-1 with IC(0) blocks in two-colour order and the given
    low-rank data, on the grid.  Every box is at least three nodes wide, so
    that no two interior nodes share an interface node, and the interface nodes
    are connected."""
    shape = (c["nz"], c["ny"], c["nx"])
    diag, off = _operator(c, seed)
    part, _ = _part(c)
    cut = torch.zeros(shape, dtype=torch.bool, device="cuda")
    for a in range(3):
        N = shape[a]
        d = part.narrow(a, 0, N - 1) != part.narrow(a, 1, N - 1)
        cut.narrow(a, 0, N - 1).logical_or_(d)
        cut.narrow(a, 1, N - 1).logical_or_(d)
    # colour classes: the node of lowest index of each component is in class 0
    z, y, x = torch.meshgrid(*[torch.arange(e, device="cuda") for e in shape], indexing="ij")
    parity = ((x + y + z) % 2).reshape(-1)
    comp = torch.where(cut, torch.full_like(part, int(part.max()) + 1), part).reshape(-1).long()
    order = torch.arange(parity.numel(), device="cuda")
    first = torch.full((int(comp.max()) + 1,), parity.numel() - 1, device="cuda").scatter_reduce(0, comp, order, "amin")
    colour = (parity ^ parity[first][comp]).reshape(shape).bool()
    same, cross, cdiag = [], [], torch.where(cut, diag + 1.0, diag)
    for w, a in zip(off, (2, 1, 0)):
        N = shape[a]
        s_, x_ = torch.zeros_like(w), torch.zeros_like(w)
        lo, hi = cut.narrow(a, 0, N - 1), cut.narrow(a, 1, N - 1)
        wc = w.narrow(a, 0, N - 1)
        s_.narrow(a, 0, N - 1).copy_(torch.where(lo == hi, wc, 0.0))
        x_.narrow(a, 0, N - 1).copy_(torch.where(lo != hi, wc, 0.0))
        sq = torch.where(lo != hi, wc * wc, 0.0)        # the diagonal of Ehat Ehat^T
        cdiag.narrow(a, 0, N - 1).add_(torch.where(~lo, sq, 0.0))
        cdiag.narrow(a, 1, N - 1).add_(torch.where(~hi, sq, 0.0))
        same.append(s_)
        cross.append(x_)
    zero = torch.zeros_like(diag)
    l0 = torch.sqrt(cdiag)                              # first colour
    sq = _grid_product(zero, [-w * w for w in same], torch.where(colour, 0.0, 1.0 / cdiag)[None])[0]
    l1 = torch.sqrt(cdiag - sq)                         # second colour
    li = torch.where(colour, l1, l0)

    def a0(v):
        f = torch.where(colour, 0.0, v / li)
        f = torch.where(colour, (v + _grid_product(zero, [-w for w in same], f / li)) / li, f)
        g = torch.where(colour, f / li, 0.0)
        return torch.where(colour, g, (f + _grid_product(zero, [-w for w in same], g) / li) / li)

    def e_cross(v):                                     # the coupling between interior and interface
        return _grid_product(zero, cross, v)

    b = _rhs(c, seed)
    b = b[None] if c["nrhs"] == 1 else b.T
    v = b.reshape((-1,) + shape)
    U, lam, theta = _lowrank(c, int(cut.sum()), seed)
    lam = lam.cuda()
    coef = 1 / (1 - lam) - 1 / (1 - theta)
    zv = a0(v)
    yv = (e_cross(torch.where(cut, 0.0, zv)) - zv)[:, cut]
    wv = yv / (1 - theta) + ((yv @ U) * coef) @ U.T
    wg = torch.zeros_like(v)
    wg[:, cut] = wv
    out = a0(v + torch.where(cut, -wg, e_cross(wg))).flatten(1)
    return out[0] if c["nrhs"] == 1 else out.T


def exact(case, seed):
    """The solution of the linear system (the outputs carry the stopping
    tolerance of the iteration beside it), M^-1 x for the apply cases; the
    iteration counts have no such value."""
    c = case
    if c["kind"] == "apply":
        return _apply_exact(c, seed)
    if c["kind"] == "serve":
        xs = []
        for j, (_, edge) in enumerate(_requests(c)):
            ce = _edge_case(c, edge)
            xs.append(_solve_by_sines(ce, _rhs(ce, seed + 31 * j)[None], 1.0)[0].cpu().numpy())
        return dict(x=xs, its=None)
    b = _rhs(c, seed)
    b = b[None] if c["nrhs"] == 1 else b.T
    diag, off = _operator(c, seed)
    if c["matrix"] == "jump":
        x = _solve_by_cg(diag, off, b)
    else:
        scale = float(off[0].reshape(-1)[0])
        x = _solve_by_sines(c, b, scale)
    x = x[0] if c["nrhs"] == 1 else x.T
    return dict(x=x.cpu().numpy() if c["kind"] == "new" else x, its=None)
