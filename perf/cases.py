"""The work that a user of the library has it do, as measurable cases.

A case is one call (or one short, fixed sequence of calls) of the public binding on a mesh, a
medium and vectors made from a seed:

  operator      y = A x on device buffers (Solver.apply_operator_device)
  precondition  z = P^{-1} r on device buffers, all shots stacked (apply_preconditioner_device)
  step          upload the carried state of every shot, advance some slabs, read the state back
  gradient      one iteration of a waveform inversion: binding.misfit and its backward pass

Meshes are the constructions of the repository's workloads: a layered rectangle of jittered
triangles with a free surface and, where ``slivers`` is set, a hundredth of the cells flattened
to slivers; a periodic square; a periodic cube of jittered Kuhn tetrahedra.  Slab sizes are those
of the configurations: ten times the explicit limit in 2D, 1.28 cells in 3D.  Solves run to
1e-10, where the states of two runs agree to more digits than at the default 1e-8.
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_1802_04516_gb300 import binding

F64 = torch.float64
REL_TOL = 1e-10


# ----------------------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------------------
def _case(call, dim, p, pg, cells, precision, pre, shots=1, slabs=1, krylov=0, scheme="stdg", slivers=False):
    """cells: cells along the short side in 2D (twice as many along the long one), along each
    side in 3D; krylov: Krylov iterations a slab typically takes (for ``work`` alone)."""
    return dict(call=call, dim=dim, p=p, pg=pg, cells=cells, precision=precision, pre=pre, shots=shots, slabs=slabs,
                krylov=krylov, scheme=scheme, slivers=slivers)


def listed():
    return [
        # the smallest call: the Crank-Nicolson operator on the periodic plane-wave square (p = 1), where launches count
        dict(_case("operator", 2, 1, 0, 14, "fp64", 1, scheme="cn"), name="operator-2d-cn-p1"),
        # the benchmark mesh and orders: the operator of the FP32 inner solve on 200,704 triangles
        dict(_case("operator", 2, 3, 3, 224, "mixed", 1, slivers=True), name="operator-2d-p3-f32"),
        # the orders of the sliver study, FP64, a ragged size
        dict(_case("operator", 2, 4, 2, 67, "fp64", 1, slivers=True), name="operator-2d-p4-f64"),
        # the 3D configuration's operator, FP32
        dict(_case("operator", 3, 2, 2, 24, "mixed", 1), name="operator-3d-p2-f32"),
        # the highest order in 3D, an odd number of cells
        dict(_case("operator", 3, 3, 3, 11, "mixed", 1), name="operator-3d-p3-f32"),
        # the stencil preconditioner for the 64 stacked shots of the multi-shot workload
        dict(_case("precondition", 2, 2, 2, 56, "mixed", 2, shots=64, slivers=True), name="precondition-64-shots"),
        # the plane-wave problem: ten Crank-Nicolson slabs by conjugate gradients
        dict(_case("step", 2, 1, 0, 14, "fp64", 1, slabs=10, krylov=58, scheme="cn"), name="step-2d-cn-p1"),
        # the headline: one slab of the 200,704-triangle sliver mesh, mixed precision, stencil preconditioner
        dict(_case("step", 2, 3, 3, 224, "mixed", 2, krylov=141, slivers=True), name="step-2d-p3-mixed"),
        # the binding's defaults (FP64, block Jacobi) on a mid-sized mesh
        dict(_case("step", 2, 2, 2, 45, "fp64", 1, krylov=171), name="step-2d-p2-f64"),
        # the 3D configuration on a small cube
        dict(_case("step", 3, 2, 2, 12, "mixed", 2, krylov=242), name="step-3d-p2-mixed"),
        # a batch of shots in one stacked solve
        dict(_case("step", 2, 2, 2, 32, "mixed", 2, shots=32, krylov=176, slivers=True), name="step-32-shots"),
        # one inversion iteration: new medium, eight shots forward and adjoint
        dict(_case("gradient", 2, 2, 2, 31, "mixed", 2, shots=8, slabs=6, krylov=36), name="gradient-8-shots"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["operator", "operator", "precondition", "step", "step", "gradient"])
    dim = 2 if call == "gradient" else rng.choice([2, 2, 3])
    precision = rng.choice(["fp64", "mixed"])
    if call == "gradient":
        return _case(call, 2, 2, 2, _log(rng, 9, 31), precision, rng.choice([1, 2]), shots=rng.randint(1, 8),
                     slabs=rng.randint(2, 4), krylov=100)
    if call == "operator":
        p = rng.randint(1, 4 if dim == 2 else 3)
        scheme = rng.choice(["stdg", "stdg", "cn"])
        pg = 0 if scheme == "cn" else rng.randint(1, p)
        top = (224 if p < 4 else 120) if dim == 2 else {1: 32, 2: 24, 3: 14}[p]
        if precision == "fp64":
            top = top // 2
        return _case(call, dim, p, pg, _log(rng, 6, top), precision, 1, scheme=scheme, slivers=dim == 2 and rng.random() < 0.5)
    p = rng.randint(1, 3 if dim == 2 else 2)
    pg = p
    pre = rng.choice([1, 2])
    shots = rng.choice([1, 1, rng.randint(2, 40)])
    if call == "precondition":
        top = {1: 120, 2: 100, 3: 75}[p] if dim == 2 else {1: 16, 2: 12}[p]
        if shots > 1:
            top = top // 2
        return _case(call, dim, p, pg, _log(rng, 6, top), precision, pre, shots=shots, slivers=dim == 2 and rng.random() < 0.5)
    scheme = rng.choice(["stdg", "stdg", "cn"]) if shots == 1 else "stdg"
    pg = 0 if scheme == "cn" else p
    top = {1: 100, 2: 70, 3: 50}[p] if dim == 2 else {1: 12, 2: 9}[p]
    if shots > 1 or precision == "fp64":
        top = top // 2
    return _case(call, dim, p, pg, _log(rng, 6, top), precision, pre, shots=shots if dim == 2 else 1,
                 slabs=rng.randint(1, 3), krylov=100, scheme=scheme)


# ----------------------------------------------------------------------------------------
# inputs: meshes, media, states
# ----------------------------------------------------------------------------------------
def _volumes(X):
    return np.linalg.det(X[:, 1:] - X[:, :1])


def _corners(xyz, elem, period):
    X = xyz[elem]
    if period is not None:
        X = X - period * np.round((X - X[:, :1]) / period)
    return X


def _jitter(xyz, elem, period, off):
    """Moves the vertices by ``off``, halved around elements that would turn over."""
    for _ in range(60):
        bad = _volumes(_corners(xyz + off, elem, period)) <= 0
        if not bad.any():
            break
        off[np.unique(elem[bad])] *= 0.5
    return xyz + off


def _triangles(n, periodic, rng):
    """2n x n cells (n x n where periodic) of two triangles each."""
    nx, ny, size = (n, n, np.array([1.0, 1.0])) if periodic else (2 * n, n, np.array([2.0, 1.0]))
    sx, sy = (nx, ny) if periodic else (nx + 1, ny + 1)
    j, i = (a.ravel() for a in np.meshgrid(np.arange(sy), np.arange(sx), indexing="ij"))
    xyz = np.stack([i * size[0] / nx, j * size[1] / ny], axis=1)
    jc, ic = (a.ravel() for a in np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij"))
    at = lambda a, b: (b % sy) * sx + a % sx  # noqa: E731
    v00, v10, v01, v11 = at(ic, jc), at(ic + 1, jc), at(ic, jc + 1), at(ic + 1, jc + 1)
    elem = np.stack([np.stack([v00, v10, v11], 1), np.stack([v00, v11, v01], 1)], axis=1).reshape(-1, 3)
    if periodic:
        return xyz, elem.astype(np.int32), size
    off = rng.uniform(-0.3, 0.3, xyz.shape) * size / (nx, ny)
    off[(i == 0) | (i == nx), 0] = 0.0
    off[(j == 0) | (j == ny), 1] = 0.0
    return _jitter(xyz, elem, None, off), elem.astype(np.int32), None


def _slivers(xyz, elem, n, rng):
    """Flattens about a hundredth of the triangles: in cells seven apart, an inner vertex moves to
    1/70 of a cell from the opposite edge (moves that would turn a triangle over are undone)."""
    cells = np.arange(elem.shape[0] // 2).reshape(n, 2 * n)[3:n - 3:7, 3:2 * n - 3:7].ravel()
    tri = 2 * cells + rng.integers(0, 2, cells.size)
    P = xyz[elem[tri]]
    edge = np.linalg.norm(np.roll(P, -1, axis=1) - np.roll(P, -2, axis=1), axis=2)
    k, rows = np.argmax(edge, axis=1), np.arange(tri.size)
    a, b, c = P[rows, k], P[rows, (k + 1) % 3], P[rows, (k + 2) % 3]
    t = (c - b) / np.linalg.norm(c - b, axis=1, keepdims=True)
    foot = b + np.sum((a - b) * t, axis=1, keepdims=True) * t
    new, vert = xyz.copy(), elem[tri, k]
    new[vert] = foot + (a - foot) / np.linalg.norm(a - foot, axis=1, keepdims=True) / (70.0 * n)
    undo = np.intersect1d(vert, elem[_volumes(new[elem]) <= 0])
    new[undo] = xyz[undo]
    return new


def _tetrahedra(n, rng):
    k, j, i = (a.ravel() for a in np.meshgrid(*[np.arange(n)] * 3, indexing="ij"))
    xyz = np.stack([i, j, k], axis=1) / n
    tets = []
    for perm in itertools.permutations(range(3)):
        at, path = np.zeros(3, dtype=int), [np.zeros(3, dtype=int)]
        for axis in perm:
            at = at + np.eye(3, dtype=int)[axis]
            path.append(at)
        ids = [((k + q[2]) % n * n + (j + q[1]) % n) * n + (i + q[0]) % n for q in path]
        if np.linalg.det(np.eye(3)[list(perm)]) < 0:
            ids[2], ids[3] = ids[3], ids[2]
        tets.append(np.stack(ids, axis=1))
    elem = np.stack(tets, axis=1).reshape(-1, 4)
    return _jitter(xyz, elem, np.ones(3), rng.uniform(-0.2, 0.2, xyz.shape) / n), elem.astype(np.int32), np.ones(3)


def _smooth(rng, x, n_out, modes=6):
    """n_out smooth random fields of unit size at the points x (..., dim), and their gradients."""
    f, g = np.zeros(x.shape[:-1] + (n_out,)), np.zeros(x.shape[:-1] + (n_out, x.shape[-1]))
    for _ in range(modes):
        k = 2 * np.pi * rng.integers(-2, 3, x.shape[-1])
        amp, ph = rng.normal(size=n_out) / math.sqrt(modes), rng.uniform(0, 2 * np.pi, n_out)
        arg = (x @ k)[..., None] + ph
        f += amp * np.sin(arg)
        g += (amp * np.cos(arg))[..., None] * k
    return f, g


def _problem(case, seed):
    """Mesh, medium and slab size of a case."""
    dim, p, n = case["dim"], case["p"], case["cells"]
    rng = np.random.default_rng([n, dim])   # a user has one mesh and many media, states and shots on it
    if dim == 3:
        xyz, elem, period = _tetrahedra(n, rng)
    else:
        xyz, elem, period = _triangles(n, case["scheme"] == "cn" and p == 1, rng)
        if case["slivers"] and period is None and n >= 14:
            xyz = _slivers(xyz, elem, n, rng)
    X = _corners(xyz, elem, period)
    centre = X.mean(axis=1)
    rng = np.random.default_rng([seed, 1])
    if dim == 2 and period is None:   # three layers, faster with depth
        layer = np.clip((centre[:, 1] * 3).astype(int), 0, 2)
        vp, vs, rho = (np.array(a)[layer] for a in ([4.0, 3.0, 2.0], [2.3, 1.7, 1.2], [2.0, 1.5, 1.0]))
    else:
        vp, vs, rho = (np.full(len(elem), a) for a in (math.sqrt(3.0), 1.0, 1.0))
    f, _ = _smooth(rng, centre, 3)
    rho = rho * (1 + 0.05 * np.tanh(f[:, 0]))
    mu = rho * vs ** 2 * (1 + 0.05 * np.tanh(f[:, 1]))
    lam = (rho * vp ** 2 - 2 * rho * vs ** 2) * (1 + 0.05 * np.tanh(f[:, 2]))
    dt = 1.28 / n if dim == 3 else 10.0 / (n * dim * (2 * p + 1) * float(vp.max()))
    return dict(xyz=xyz, elem=elem, period=period, X=X, lam=lam, mu=mu, rho=rho, dt=dt)


def _solver(case, pr):
    stream = torch.cuda.Stream()
    s = binding.Solver(case["dim"], case["p"], case["pg"], scheme=case["scheme"], precision=case["precision"], rel_tol=REL_TOL,
                       gmres_restart=20 if case["pre"] == 2 else 30, stream=stream.cuda_stream, preconditioner=case["pre"])
    s.perf_stream = stream   # the solver's work is issued on it: it lives as long as the solver
    s.set_mesh(pr["xyz"], pr["elem"], pr["period"])
    s.set_material(pr["lam"], pr["mu"], pr["rho"])
    return s


def _vector(case, seed, n):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dtype = torch.float32 if case["precision"] == "mixed" else F64
    return torch.randn(n, generator=g, device="cuda", dtype=F64).to(dtype)


def _states(case, pr, seed):
    """Per shot a smooth carried state: velocity at the element nodes; stress as constant and linear
    Taylor coefficients about each dual cell's centre."""
    geo = _faces(pr["elem"], pr["X"])
    dim, nodes = case["dim"], _lattice(case["dim"], case["p"])
    x = pr["X"][:, :1] + nodes @ (pr["X"][:, 1:] - pr["X"][:, :1])
    out = []
    for shot in range(case["shots"]):
        rng = np.random.default_rng([seed, 2, shot])
        v, _ = _smooth(rng, x, dim)
        s, g = _smooth(rng, geo["xc"], dim * (dim + 1) // 2)
        sig = np.zeros(s.shape + (len(nodes),))
        sig[..., 0], sig[..., 1:dim + 1] = s, g * geo["h"][:, None, None]
        out.append((np.ascontiguousarray(1e-2 * v.transpose(0, 2, 1)), 1e-2 * sig))
    return out


def prepare(case, seed):
    pr = _problem(case, seed)
    s = _solver(case, pr)
    st = dict(case=case, solver=s, dt=pr["dt"])
    if case["call"] == "operator":
        st["x"] = _vector(case, seed, s.nvel)
        st["y"] = torch.empty_like(st["x"])
    elif case["call"] == "precondition":
        s.set_shots(case["shots"])
        st["x"] = _vector(case, seed, s.nvel * case["shots"])
        st["y"] = torch.empty_like(st["x"])
        torch.cuda.synchronize()
        s.apply_preconditioner_device(st["dt"], st["x"].data_ptr(), st["y"].data_ptr(), fp32=case["precision"] == "mixed")
    elif case["call"] == "step":
        if case["shots"] > 1:
            s.set_shots(case["shots"])
        st["states"] = _states(case, pr, seed)
        pinned = lambda a: torch.empty(a.shape, dtype=F64, pin_memory=True).numpy()  # noqa: E731
        st["out"] = [tuple(pinned(a) for a in vs) for vs in st["states"]]
    else:
        rng = np.random.default_rng([seed, 3])
        n = case["shots"]
        st["sources"] = dict(xs=torch.tensor(np.stack([0.2 + 1.6 * (np.arange(n) + rng.uniform(0.2, 0.8, n)) / n, np.full(n, 0.85)], 1)),
                             force=torch.tensor(rng.normal(size=(n, 2))), f0=10.0, t_delay=0.0, n_shots=n)
        s.set_receivers(np.stack([0.02 + 1.96 * np.arange(100) / 99, np.full(100, 0.95)], 1))
        st["data"] = rng.normal(size=(n, case["slabs"], 100, 2)) * 1e-2
        st["model"] = [torch.tensor(pr[k], requires_grad=True) for k in ("lam", "mu", "rho")]
        for k in ("xs", "force"):
            st["sources"][k].requires_grad_(True)
    torch.cuda.synchronize()
    return st


def run(state):
    s, case, dt = state["solver"], state["case"], state["dt"]
    if case["call"] == "operator":
        s.apply_operator_device(dt, state["x"].data_ptr(), state["y"].data_ptr(), fp32=case["precision"] == "mixed")
        return state["y"]
    if case["call"] == "precondition":
        s.apply_preconditioner_device(dt, state["x"].data_ptr(), state["y"].data_ptr(), fp32=case["precision"] == "mixed")
        return state["y"]
    if case["call"] == "step":
        for k, (v, sig) in enumerate(state["states"]):
            s.set_state(v, sig, shot=k)
        s.time = 0.0
        s.step(dt, case["slabs"])
        return [s.get_state(shot=k, out=o) for k, o in enumerate(state["out"])]
    src = state["sources"]
    loss = binding.misfit(s, *state["model"], dt, case["slabs"], state["data"], sources=src)
    grads = torch.autograd.grad(loss, [*state["model"], src["xs"], src["force"]])
    return [loss.detach(), *grads]


# ----------------------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------------------
def _sizes(case):
    dim, p, n = case["dim"], case["p"], case["cells"]
    periodic = dim == 3 or (case["scheme"] == "cn" and p == 1)
    ne = 6 * n ** 3 if dim == 3 else (2 if periodic else 4) * n * n
    nf = (2 * ne if dim == 3 else 3 * ne // 2) + (0 if periodic else 3 * n)
    return ne, nf, math.comb(p + dim, dim), case["pg"] + 1


def work(case):
    """Bytes and operations: each block of the operator (D~, Lame parameters, face ids) and of the
    preconditioner once per application, each vector in and out once; a slab applies the operator and
    the preconditioner ``krylov`` times and streams the vector it orthogonalises."""
    dim, shots = case["dim"], case["shots"]
    ne, nf, N, G = _sizes(case)
    w = 4 if case["precision"] == "mixed" else 8
    nv, n = ne * dim * G * N, dim * N
    op_b = nf * (2 * dim * N * N * w + 2 * w + 8) + ne * w
    op_f = shots * (nf * 8 * dim * dim * G * N * N + nv * 2 * (G + N))
    v_b = 2 * nv * shots * w
    if case["pre"] == 1:
        pc_b, pc_f = ne * (n * n + n * G * G) * w, shots * ne * 2 * n * G * (2 * n + G)
    else:
        half = 2 if w == 4 and shots == 1 else w
        pc_b, pc_f = ne * ((n * G) ** 2 * half + (n * n + n * G * G) * w) + op_b, shots * ne * 2 * ((n * G) ** 2 + n * G * (2 * n + G)) + op_f
    if case["call"] == "operator":
        return dict(bytes=op_b + v_b, flops=op_f)
    if case["call"] == "precondition":
        return dict(bytes=pc_b + v_b, flops=pc_f)
    solves = case["slabs"] * (3 if case["call"] == "gradient" else 1)   # forward, recomputed and adjoint slabs
    state = 2 * 8 * shots * (ne * n + nf * dim * (dim + 1) // 2 * N)
    return dict(bytes=solves * (case["krylov"] * (op_b + pc_b + 2 * v_b) + state), flops=solves * case["krylov"] * (op_f + pc_f))


# ----------------------------------------------------------------------------------------
# the same results in 64 bits, from the equations alone
# ----------------------------------------------------------------------------------------
def _lattice(dim, p):
    """Equispaced nodes of the reference simplex, z outer, then y, x fastest."""
    ax = range(p + 1)
    pts = [q[::-1] for q in itertools.product(*[ax] * dim) if sum(q) <= p]
    return np.array(pts, dtype=float) / p


def _exponents(dim, p):
    """Graded lexicographic: degree ascending, then the x exponent descending, then y."""
    e = [q for q in itertools.product(range(p + 1), repeat=dim) if sum(q) <= p]
    return sorted(e, key=lambda q: (sum(q),) + tuple(-a for a in q))


def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1), 0.5 * w


def _rule(dim, n):
    """Collapsed Gauss rule on the reference simplex."""
    x, w = _gauss(n)
    if dim == 1:
        return x[:, None], w
    pts, wts = [], []
    for idx in itertools.product(range(n), repeat=dim):
        q, left, wt = [], 1.0, 1.0
        for d, i in enumerate(idx):
            q.append(left * x[i])
            wt *= w[i] * left if d else w[i]
            left *= 1 - x[i]
        pts.append(q)
        wts.append(wt)
    return np.array(pts), np.array(wts)


def _mono(y, exps):
    """Monomials at the points y (..., dim) -> (..., N)."""
    return torch.stack([functools.reduce(lambda a, b: a * b, [y[..., r] ** e for r, e in enumerate(q)]) for q in exps], dim=-1)


def _faces(elem, X):
    """Faces by ascending sorted vertex tuple; per (face, side) element and local index; dual-cell centre
    (in the frame of the smaller element), scale and the translation of the other side into that frame."""
    ne, nv = elem.shape
    dim = nv - 1
    opp = [[k for k in range(nv) if k != f] for f in range(nv)]
    tup = np.sort(np.stack([elem[:, o] for o in opp], axis=1).reshape(-1, dim), axis=1).astype(np.int64)
    big = int(elem.max()) + 1
    key = functools.reduce(lambda a, c: a * big + tup[:, c], range(1, dim), tup[:, 0])
    _, first, face = np.unique(key, return_index=True, return_inverse=True)
    face, nf, at = face.ravel(), len(first), np.arange(ne * nv)
    last = np.zeros(nf, dtype=np.int64)
    np.maximum.at(last, face, at)
    pair = np.stack([first, np.where(last != first, last, -1)], axis=1)      # element * nv + local face
    el, lf = pair // nv, pair % nv
    opp = np.array(opp)
    corners = []
    for side in (0, 1):
        e = np.where(el[:, side] >= 0, el[:, side], el[:, 0])
        f = np.where(el[:, side] >= 0, lf[:, side], lf[:, 0])
        order = np.argsort(np.take_along_axis(elem[e], opp[f], axis=1), axis=1)   # the same vertex order on both sides
        V = np.take_along_axis(X[e], np.take_along_axis(opp[f], order, axis=1)[..., None], axis=1)
        corners.append((V, X[e].mean(axis=1), np.abs(_volumes(X[e])), X[e][np.arange(nf), f]))
    inside = el[:, 1] >= 0
    shift = (corners[0][0] - corners[1][0]).mean(axis=1)
    w = np.stack([corners[0][2], np.where(inside, corners[1][2], 0.0)], axis=1)
    w /= w.sum(axis=1, keepdims=True)
    cen = [(c[0].sum(axis=1) + c[1]) / (dim + 1) for c in corners]
    xc = w[:, :1] * cen[0] + w[:, 1:] * (cen[1] + shift)
    far = np.linalg.norm(np.concatenate([corners[0][0], corners[0][1][:, None], (corners[1][1] + shift)[:, None]], 1) - xc[:, None], axis=2)
    return dict(el=el, corners=corners, shift=shift, inside=inside, w=w, xc=xc, h=far.max(axis=1))


class _Exact:
    """The scheme's matrices by quadrature, on whatever device torch has, in 64 bits."""

    def __init__(self, case, pr):
        self.case, self.dt = case, pr["dt"]
        dim, p, G = case["dim"], case["p"], case["pg"] + 1
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=self.dev)  # noqa: E731
        geo, exps = _faces(pr["elem"], pr["X"]), _exponents(dim, p)
        self.N = N = len(exps)
        self.ne, self.nf = len(pr["elem"]), len(geo["xc"])
        coef = np.linalg.inv(_mono(torch.tensor(_lattice(dim, p)), exps).numpy())     # phi_k = sum_a coef[a, k] mono_a
        qp, qw = _rule(dim, p + 3)
        fp, fw = _rule(dim - 1, p + 3)
        ph = _mono(torch.tensor(qp), exps).numpy() @ coef
        self.M = t(ph.T @ (qw[:, None] * ph))
        # time: nodes, W, T = g(1) g(1)^T - K, S = W T^-1 W
        x, wt = _gauss(G)
        vander = np.linalg.inv(np.vander(x, G, increasing=True))
        at = lambda s, d=0: np.array([[math.perm(k, d) * s_ ** (k - d) if k >= d else 0.0 for k in range(G)] for s_ in np.atleast_1d(s)]) @ vander  # noqa: E731
        g0, g1 = at(0.0)[0], at(1.0)[0]
        self.T = np.outer(g1, g1) - (wt[:, None] * at(x, 1)).T @ np.eye(G)
        Ti = np.linalg.inv(self.T)
        self.S, self.g0, self.g1, self.kappa, self.u = wt[:, None] * Ti * wt, g0, g1, g1 @ Ti @ g0, (g1 @ Ti) * wt
        self.coef_rhs = self.dt * (np.ones(1) if case["scheme"] == "cn" else wt * (Ti @ g0))
        self.c = (0.25 if case["scheme"] == "cn" else 1.0) * self.dt ** 2
        el = geo["el"]
        self.el = [t(el[:, 0]), t(np.where(el[:, 1] >= 0, el[:, 1], 0))]
        lam, mu, rho = pr["lam"], pr["mu"], pr["rho"]
        mean = lambda a: t(geo["w"][:, 0] * a[el[:, 0]] + geo["w"][:, 1] * a[el[:, 1]])  # noqa: E731
        self.lam, self.mu = mean(lam), mean(mu)
        vol = np.abs(_volumes(pr["X"]))
        self.rhoJ = t(rho * vol)
        X = t(pr["X"])
        Jinv = torch.linalg.inv((X[:, 1:] - X[:, :1]).transpose(1, 2))
        # orthonormal dual basis from monomials of whitened coordinates y = B (x - x_j)
        self.D = torch.zeros(self.nf, 2, dim, N, N, dtype=F64, device=self.dev)
        self.E = torch.zeros(self.nf, N, N, dtype=F64, device=self.dev)               # Taylor -> orthonormal
        qp, qw, fp, fw, coef = t(qp), t(qw), t(fp), t(fw), t(coef)
        inside, xc, h = t(geo["inside"]), t(geo["xc"]), t(geo["h"])
        sides = [tuple(t(a) for a in c) for c in geo["corners"]]
        shift = t(geo["shift"])
        lat = t(2.0 * _lattice(dim, p) - 0.5)
        inv_lat = torch.linalg.inv(_mono(lat, exps))
        for f0 in range(0, self.nf, 8192):
            f = slice(f0, min(f0 + 8192, self.nf))
            pts, wts = [], []
            for s, (V, b, vol_e, _) in enumerate(sides):
                V, b = V[f], b[f]
                x = V[:, :1] + qp @ torch.cat([V[:, 1:], b[:, None]], 1).sub(V[:, :1])
                w = qw * (vol_e[f] / (dim + 1))[:, None]
                pts.append(x)
                wts.append(w if s == 0 else w * inside[f, None])
            d = [pts[0] - xc[f, None], pts[1] + shift[f, None] - xc[f, None]]
            cov = sum(torch.einsum("fq,fqa,fqb->fab", w, y, y) for w, y in zip(wts, d)) / sum(w.sum(1) for w in wts)[:, None, None]
            L = torch.linalg.cholesky(cov)
            white = lambda y: torch.linalg.solve_triangular(L, y.transpose(1, 2), upper=False).transpose(1, 2)  # noqa: E731,B023
            psi = [_mono(white(y), exps) for y in d]
            C = torch.linalg.cholesky(sum(torch.einsum("fq,fqm,fqn->fmn", w, q, q) for w, q in zip(wts, psi)))
            orth = lambda q: torch.linalg.solve_triangular(C, q.transpose(1, 2), upper=False).transpose(1, 2)  # noqa: E731,B023
            for s, (V, _, _, apex) in enumerate(sides):
                e = self.el[s][f]
                ji, x0 = Jinv[e], X[e, 0]
                ref = lambda x: (x - x0[:, None]) @ ji.transpose(1, 2)  # noqa: E731,B023
                xi, grad = ref(pts[s]), []
                for r in range(dim):
                    low = [tuple(a - (i == r) for i, a in enumerate(q)) for q in exps]
                    fac = torch.tensor([q[r] for q in exps], dtype=F64, device=self.dev)
                    grad.append((_mono(xi, [tuple(max(a, 0) for a in q) for q in low]) * fac) @ coef)
                gphi = torch.einsum("rfqk,frl->flqk", torch.stack(grad), ji)
                self.D[f, s] = -torch.einsum("fq,flqk,fqm->flkm", wts[s], gphi, orth(psi[s]))
                # the face: normal out of this element, from the edge vectors
                E = V[f][:, 1:] - V[f][:, :1]
                nrm = torch.stack([E[:, 0, 1], -E[:, 0, 0]], 1) if dim == 2 else torch.linalg.cross(E[:, 0], E[:, 1])
                nrm = nrm * torch.sign(((V[f][:, 0] - apex[f]) * nrm).sum(1, keepdim=True)) * inside[f, None]
                x = V[f][:, :1] + fp @ E
                y = x - xc[f, None] + (shift[f, None] if s else 0.0)
                phi = _mono(ref(x), exps) @ coef
                self.D[f, s] += torch.einsum("q,fl,fqk,fqm->flkm", fw, nrm, phi, orth(_mono(white(y), exps)))
            self.D[f, 1] *= inside[f, None, None, None]
            taylor = _mono((lat @ L.transpose(1, 2)) / h[f, None, None], exps)
            self.E[f] = C.transpose(1, 2) @ (inv_lat @ taylor)
        self.pairs = [(0, 0), (1, 1), (0, 1)] if dim == 2 else [(0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2)]

    def grad(self, v):
        """D~^T v: (.., elem, k, time, n) -> (.., face, k, l, time, m)."""
        return sum(torch.einsum("flnm,...fkbn->...fklbm", self.D[:, s], v[..., self.el[s], :, :, :]) for s in (0, 1))

    def stress(self, g):
        """E : g as a full tensor."""
        tr = torch.einsum("...fkkbm->...fbm", g)[..., :, None, None, :, :]
        eye = torch.eye(self.case["dim"], dtype=F64, device=self.dev)[:, :, None, None]
        by = lambda a: a[:, None, None, None, None]  # noqa: E731
        return by(self.lam) * tr * eye + by(self.mu) * (g + g.transpose(-4, -3))

    def div(self, h):
        """D~ h: (.., face, k, l, time, m) -> (.., elem, k, time, n)."""
        out = torch.zeros(h.shape[:-5] + (self.ne, self.case["dim"], h.shape[-2], self.N), dtype=F64, device=self.dev)
        for s in (0, 1):
            out.index_add_(out.dim() - 4, self.el[s], torch.einsum("flnm,...fklbm->...fkbn", self.D[:, s], h))
        return out

    def mass(self, v, T):
        return self.rhoJ[:, None, None, None] * torch.einsum("ab,...ekbn,nm->...ekam", torch.as_tensor(T, device=self.dev), v, self.M)

    def face(self, v):
        S = torch.as_tensor(self.S, device=self.dev)
        return self.c * self.div(torch.einsum("ab,...fklbm->...fklam", S, self.stress(self.grad(v))))

    def apply(self, v):
        return self.mass(v, self.T) + self.face(v)

    def coupling(self, s, s2):
        """K of the faces from side s2 to side s, as (face, dim N, dim N)."""
        P = torch.einsum("flnm,fkqm->flknq", self.D[:, s], self.D[:, s2])            # P[l][k] = D_l D_k^T
        K = self.lam[:, None, None, None, None] * P + self.mu[:, None, None, None, None] * P.transpose(1, 2)
        d = range(self.case["dim"])
        tr = self.mu[:, None, None] * sum(P[:, k, k] for k in d)
        for k in d:
            K[:, k, k] += tr
        return K.permute(0, 1, 3, 2, 4).reshape(self.nf, K.shape[1] * self.N, -1)

    def blocks(self):
        """Diagonal blocks of A, (elem, n G, n G) in the order (k, n, time)."""
        n, G = self.case["dim"] * self.N, len(self.T)
        K = torch.zeros(self.ne, n, n, dtype=F64, device=self.dev)
        for s in (0, 1):
            K.index_add_(0, self.el[s], self.coupling(s, s))
        M = torch.block_diag(*[self.M] * self.case["dim"])
        S, T = torch.as_tensor(self.S, device=self.dev), torch.as_tensor(self.T, device=self.dev)
        return self.rhoJ[:, None, None] * torch.kron(M, T) + self.c * torch.einsum("eij,ab->eiajb", K, S).reshape(self.ne, n * G, n * G)

    def flat(self, v):
        """(.., elem, k, time, n) <-> (elem, (k, n, time), shots)."""
        return v.transpose(-1, -2).reshape(v.shape[0], self.ne, -1).permute(1, 2, 0)

    def unflat(self, z):
        return z.permute(2, 0, 1).reshape(z.shape[2], self.ne, self.case["dim"], self.N, len(self.T)).transpose(-1, -2)

    def precondition(self, r):
        A, r = self.blocks(), self.flat(r)
        y = torch.linalg.solve(A, r)
        if self.case["pre"] == 1:
            return self.unflat(y)
        S, G = torch.as_tensor(self.S, device=self.dev), len(self.T)
        rhs, schur, K = r.clone(), A.clone(), self.c * self.coupling(0, 1)
        for f0 in range(0, self.nf, 4096):
            f = slice(f0, min(f0 + 4096, self.nf))
            N01 = torch.einsum("fij,ab->fiajb", K[f], S).reshape(len(K[f]), -1, K.shape[2] * G)
            N10 = torch.einsum("fji,ab->fiajb", K[f], S).reshape(len(K[f]), -1, K.shape[1] * G)
            l, q = self.el[0][f], self.el[1][f]
            schur.index_add_(0, l, N01 @ torch.linalg.solve(A[q], N10), alpha=-1)
            schur.index_add_(0, q, N10 @ torch.linalg.solve(A[l], N01), alpha=-1)
            rhs.index_add_(0, l, N01 @ y[q], alpha=-1)
            rhs.index_add_(0, q, N10 @ y[l], alpha=-1)
        return self.unflat(torch.linalg.solve(schur, rhs))

    def solve(self, b, tol=2e-14, most=400):
        """GMRES with exact diagonal blocks, restarted once or twice, to the rounding of 64 bits."""
        inv = torch.linalg.inv(self.blocks())
        pre = lambda r: self.unflat(inv @ self.flat(r))  # noqa: E731
        x, size = torch.zeros_like(b), torch.linalg.vector_norm(b)
        for _ in range(4):
            r = b - self.apply(x)
            beta = torch.linalg.vector_norm(r)
            if beta <= tol * size:
                break
            V, H = torch.empty((most + 1, b.numel()), dtype=F64, device=self.dev), np.zeros((most + 1, most))
            V[0], j = (r / beta).reshape(-1), 0
            while j < most:
                w = self.apply(pre(V[j].view_as(b))).reshape(-1)
                for _ in (0, 1):
                    h = V[:j + 1] @ w
                    w -= h @ V[:j + 1]
                    H[:j + 1, j] += h.cpu().numpy()
                H[j + 1, j] = float(torch.linalg.vector_norm(w))
                V[j + 1] = w / H[j + 1, j]
                j += 1
                if j % 10 == 0 or j == most:
                    e = np.zeros(j + 1)
                    e[0] = float(beta)
                    y = np.linalg.lstsq(H[:j + 1, :j], e, rcond=None)[0]
                    if np.linalg.norm(H[:j + 1, :j] @ y - e) <= 0.5 * tol * float(size):
                        break
            x += pre((torch.as_tensor(y, device=self.dev) @ V[:j]).view_as(b))
        return x

    def step(self, v, sig, slabs):
        """v (shot, elem, k, n), sig (shot, face, component, Taylor mode): the state after the slabs."""
        dim, cn = self.case["dim"], self.case["scheme"] == "cn"
        full = [[next(c for c, ab in enumerate(self.pairs) if sorted(ab) == sorted((k, l))) for l in range(dim)] for k in range(dim)]
        s = torch.einsum("fmn,zfcn->zfcm", self.E, sig)
        u = torch.as_tensor(self.u, device=self.dev)
        for _ in range(slabs):
            h = s[:, :, full][..., None, :]                                           # (shot, face, k, l, 1, m)
            flux = self.div(h) * torch.as_tensor(self.coef_rhs, device=self.dev)[:, None]
            if cn:
                b = self.mass(v[..., None, :], np.ones((1, 1))) - self.face(v[..., None, :]) + flux
            else:
                b = self.mass(v[..., None, :], np.asarray(self.g0)[:, None]) + flux
            x = self.solve(b)
            t = self.stress(self.grad(0.5 * (x + v[..., None, :]) if cn else x))
            s = self.kappa * s - self.dt * torch.stack([torch.einsum("b,zfbm->zfm", u, t[:, :, a, b]) for a, b in self.pairs], dim=2)
            v = torch.einsum("b,zekbn->zekn", torch.as_tensor(self.g1, device=self.dev), x)
        return v, torch.linalg.solve(self.E[None], s.transpose(2, 3)).transpose(2, 3)


def exact(case, seed):
    """None where 64-bit solves would take too long: the benchmark mesh's slab and the gradients."""
    ne, _, N, G = _sizes(case)
    if case["call"] == "gradient" or (case["call"] == "step" and case["shots"] * case["slabs"] * ne * N * G * case["dim"] > 8e6):
        return None
    pr = _problem(case, seed)
    ex = _Exact(case, pr)
    if case["call"] in ("operator", "precondition"):
        x = _vector(case, seed, case["shots"] * ne * case["dim"] * G * N).double().view(case["shots"], ne, case["dim"], G, N)
        return (ex.apply(x) if case["call"] == "operator" else ex.precondition(x)).reshape(-1)
    states = _states(case, pr, seed)
    v, sig = ex.step(*(torch.as_tensor(np.stack([st[i] for st in states]), device=ex.dev) for i in (0, 1)), case["slabs"])
    return [(a.cpu().numpy(), b.cpu().numpy()) for a, b in zip(v, sig)]
