"""The operator from assembled couplings (csrc/coupling*.cu) over every order it is instantiated for,
against the assembled oracle; the off-diagonal form inside the stencil preconditioner for shot counts
around the four that a thread carries; and the face kernels when the couplings do not fit the device.
Bars: 1e-12 in FP64 and 2e-5 in FP32 for the operator (as the other operator tests), 1e-9 / 1e-3 for
the preconditioner (FP64; FP32 with 16-bit or TF32 blocks)."""
import numpy as np
import pytest

import synth
from helpers import extended_patch_rows, need_gpu, oracle_sim, rel_l2, rel_l2_ext

pytestmark = pytest.mark.gpu

SHAPES = [(2, p, pg) for p in (1, 2, 3, 4) for pg in range(5)] + [(3, p, pg) for p in (1, 2, 3) for pg in (0, 1, 3)] + \
    [(3, 2, 2), (3, 1, 4)]


def _workload(dim, p, pg, n=2):
    if dim == 2:
        xyz, ev, per = synth.tri_grid(n + 1, n, 1.0, 1.0, periodic=False, jitter=0.2, seed=3)
    else:
        xyz, ev, per = synth.tet_kuhn(1 if p == 3 else 2, 1.0, periodic=False, jitter=0.1, seed=3)
    ne = ev.shape[0]
    rng = np.random.default_rng(5)
    return synth.Workload("coupling", dim, xyz, ev, per, rng.uniform(1, 2, ne), rng.uniform(.5, 1, ne),
                          rng.uniform(.8, 1.2, ne), p=p, p_gamma=pg, scheme="stdg", dt=0.05, n_steps=1, h=1.0 / n)


def _solver(w, **kw):
    from paper_1802_04516_gb300.binding import Solver
    s = Solver(w.dim, w.p, w.p_gamma, scheme=w.scheme, **kw)
    s.set_mesh(w.xyz, w.elem_vert, w.period)
    s.set_material(w.lam, w.mu, w.rho)
    return s


@pytest.mark.parametrize("dim,p,pg", SHAPES)
def test_operator_of_every_order(dim, p, pg):
    torch = need_gpu()
    w = _workload(dim, p, pg)
    A = oracle_sim(w).A
    s = _solver(w, precision="mixed", preconditioner=0)
    x = np.random.default_rng(6).normal(size=A.shape[0])
    ref = A @ x
    y = s.apply_operator(w.dt, x)
    if p == 4:   # the FP64 oracle's own rounding is above the bar there: every row in extended precision
        elems = list(range(w.n_elem))
        assert rel_l2_ext(y.reshape(w.n_elem, -1), extended_patch_rows(w, elems, x)) < 1e-12
    else:
        assert rel_l2(y, ref) < 1e-12
    xd = torch.tensor(x, dtype=torch.float32, device="cuda")
    yd = torch.zeros_like(xd)
    torch.cuda.synchronize()
    s.apply_operator_device(w.dt, xd.data_ptr(), yd.data_ptr(), fp32=True)
    assert rel_l2(yd.double().cpu().numpy(), ref) < 2e-5


@pytest.mark.parametrize("dim,p,pg,shots", [(2, 1, 1, 3), (2, 2, 2, 4), (2, 2, 2, 29), (2, 3, 2, 5), (2, 3, 3, 2), (3, 1, 1, 6),
                                            (3, 2, 1, 1)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_off_diagonal_form_for_stacked_shots(dim, p, pg, shots, precision):
    torch = need_gpu()
    from oracle.precond import pre2
    w = _workload(dim, p, pg)
    sim = oracle_sim(w)
    P = pre2(sim.A, w.n_elem, sim.mesh.elem_nbr)
    s = _solver(w, precision=precision, preconditioner=2)
    s.set_shots(shots)
    r = np.random.default_rng(7).normal(size=(shots, sim.A.shape[0]))
    dtype = torch.float64 if precision == "fp64" else torch.float32
    rd = torch.tensor(r, dtype=dtype, device="cuda")
    zd = torch.zeros_like(rd)
    torch.cuda.synchronize()
    s.apply_preconditioner_device(w.dt, rd.data_ptr(), zd.data_ptr(), fp32=precision == "mixed")
    z = zd.double().cpu().numpy()
    for k in range(shots):
        assert rel_l2(z[k], P @ r[k]) < (1e-9 if precision == "fp64" else 1e-3)


@pytest.mark.parametrize("p,pre", [(3, 1), (2, 2)])
def test_face_kernels_when_the_couplings_do_not_fit(p, pre):
    torch = need_gpu()
    w = _workload(2, p, p, n=120)
    n = w.n_elem * 2 * (p + 1) * (p + 1) * (p + 2) // 2
    x = np.random.default_rng(8).normal(size=n)

    def run():
        s = _solver(w, preconditioner=pre)
        s.set_shots(1)
        try:
            couplings = 8 * (s.n_face + s.n_elem) * (w.dim * s.Nphi) ** 2
            return s.apply_operator(w.dt, x), s.apply_preconditioner(w.dt, x), s.query(10), couplings
        finally:
            s.close()

    y, z, held, couplings = run()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    # all but the couplings fits: half their size is left for the granularity of the allocator
    fill = torch.empty(free - (held - couplings // 2), dtype=torch.uint8, device="cuda")
    try:
        y2, z2, held2, _ = run()
    finally:
        del fill
        torch.cuda.empty_cache()
    assert held2 < held
    assert rel_l2(y2, y) < 1e-12 and rel_l2(z2, z) < 1e-10


@pytest.mark.parametrize("shots", [25, 32, 57, 64, 90])
@pytest.mark.parametrize("pre", [1, 2])
def test_ring_of_slots_of_one_element_a_warp(shots, pre):
    # 32 lanes on one element: its slot buffers are refilled by lanes other than their readers, across one to three
    # chunks of shots. The off-diagonal form (stencil preconditioner) against the oracle; the form with the element's own
    # block through one mixed slab, every shot against the same shot alone (rel_tol 1e-11, bar 1e-8 as for mixed states).
    torch = need_gpu()
    from oracle.precond import pre2
    w = _workload(2, 2, 2, n=3)
    s = _solver(w, precision="mixed", preconditioner=pre, rel_tol=1e-11, max_iters=20000)
    s.set_shots(shots)
    rng = np.random.default_rng(shots)
    if pre == 2:
        sim = oracle_sim(w)
        P = pre2(sim.A, w.n_elem, sim.mesh.elem_nbr)
        r = rng.normal(size=(shots, sim.A.shape[0]))
        rd = torch.tensor(r, dtype=torch.float32, device="cuda")
        zd = torch.zeros_like(rd)
        torch.cuda.synchronize()
        s.apply_preconditioner_device(w.dt, rd.data_ptr(), zd.data_ptr(), fp32=True)
        z = zd.double().cpu().numpy()
        for k in range(shots):
            assert rel_l2(z[k], P @ r[k]) < 2e-3    # TF32 blocks
    alone = _solver(w, precision="mixed", preconditioner=pre, rel_tol=1e-11, max_iters=20000)
    alone.set_shots(1)
    v0, sig0 = alone.get_state()
    states = [(rng.normal(size=v0.shape), rng.normal(size=sig0.shape)) for _ in range(shots)]
    for k, (v, sig) in enumerate(states):
        s.set_state(v, sig, shot=k)
    s.step(w.dt, 1)
    for k in sorted({0, 7, 24, shots // 2, shots - 1}):
        alone.set_state(*states[k])
        alone.step(w.dt, 1)
        assert rel_l2(s.get_state(k)[0], alone.get_state()[0]) < 1e-8


def test_recorded_operator_outlives_the_couplings():
    # a caller's graph of the operator and of the residual, replayed after the couplings were given back (an allocation
    # of the context that cannot succeed takes them first) and their room was overwritten
    torch = need_gpu()
    from paper_1802_04516_gb300 import binding
    w = _workload(2, 2, 2, n=16)
    stream = torch.cuda.Stream()
    s = _solver(w, preconditioner=0, stream=stream.cuda_stream)
    lib = binding.load()
    g = torch.Generator(device="cuda").manual_seed(3)
    x, b = (torch.randn(s.nvel, dtype=torch.float64, device="cuda", generator=g) for _ in range(2))
    y, r, out = torch.zeros_like(x), torch.zeros_like(x), torch.zeros(2, dtype=torch.float64, device="cuda")

    def calls():
        s.apply_operator_device(w.dt, x.data_ptr(), y.data_ptr())
        assert lib.stdg_residual_noalloc(s.h, w.dt, x.data_ptr(), b.data_ptr(), r.data_ptr(), out.data_ptr()) == 0

    torch.cuda.synchronize()
    calls()
    torch.cuda.synchronize()
    want = y.clone(), r.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        calls()
    held = s.query(10)
    with pytest.raises(binding.StdgError):
        s.set_shots(1 << 24)
    assert s.query(10) < held
    junk = torch.full((1 << 27,), float("nan"), dtype=torch.float64, device="cuda")
    y.fill_(float("nan"))
    r.fill_(float("nan"))
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert rel_l2(y.cpu().numpy(), want[0].cpu().numpy()) < 1e-12 and rel_l2(r.cpu().numpy(), want[1].cpu().numpy()) < 1e-12
    del junk


@pytest.mark.parametrize("room,share,held", [(4, None, False), (12, None, True), (4, 0.5, True), (12, 0.0, False)])
def test_couplings_take_no_more_than_their_share_of_the_free_memory(room, share, held):
    # a mesh whose couplings are 1/room of the memory that is free when they are laid out (the rest stays for others):
    # by default they may take 1/6 of it
    torch = need_gpu()
    w = _workload(2, 3, 3, n=120)
    x = np.random.default_rng(8).normal(size=w.n_elem * 80)

    def run(share):
        from paper_1802_04516_gb300.binding import Solver
        s = Solver(2, 3, 3, preconditioner=0)
        try:
            if share is not None:
                s.set_coupling_share(share)
            s.set_mesh(w.xyz, w.elem_vert, w.period)
            s.set_material(w.lam, w.mu, w.rho)
            return s.apply_operator(w.dt, x), s.query(10), s.coupling_bytes
        finally:
            s.close()

    y0, base, none = run(0.0)
    assert none == 0
    y1, full, couplings = run(1.0)
    assert couplings == full - base > 0
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    fill = torch.empty(free - base - room * couplings, dtype=torch.uint8, device="cuda")
    try:
        y, _, c = run(share)
    finally:
        del fill
        torch.cuda.empty_cache()
    assert (c > 0) == held
    assert rel_l2(y, y0) < 1e-12 and rel_l2(y1, y0) < 1e-12


def test_couplings_given_back_at_once():
    need_gpu()
    from paper_1802_04516_gb300.binding import STDG_EINVAL, StdgError
    w = _workload(2, 2, 2, n=4)
    s = _solver(w, precision="mixed", preconditioner=2)
    x = np.random.default_rng(8).normal(size=s.nvel)
    y = s.apply_operator(w.dt, x)
    held, c = s.query(10), s.coupling_bytes
    assert c > 0
    for bad in (-0.1, 1.5, float("nan")):
        with pytest.raises(StdgError) as ei:
            s.set_coupling_share(bad)
        assert ei.value.code == STDG_EINVAL
    s.set_coupling_share(0.0)
    assert s.coupling_bytes == 0 and s.query(10) == held - c
    assert rel_l2(s.apply_operator(w.dt, x), y) < 1e-12
    s.set_material(w.lam, w.mu, w.rho)
    assert s.coupling_bytes == 0
    s.set_coupling_share(1.0)
    s.set_material(w.lam, w.mu, w.rho)
    assert s.coupling_bytes == c


@pytest.mark.parametrize("dim,p", [(2, 1), (2, 3), (3, 1)])
def test_fp32_results_that_overflow_are_infinite(dim, p):
    # one large value: every row is one product (plus the mass term), scaled by dt^2 / 4 at the end; results far above
    # the largest FP32 number are infinite, those whose product before the scaling is far below it are finite
    torch = need_gpu()
    w = _workload(dim, p, 0)
    w.lam[:], w.mu[:], w.scheme = w.lam * 1e12, w.mu * 1e12, "cn"
    s = _solver(w, precision="mixed", preconditioner=0)
    x = np.zeros(s.nvel)
    x[s.nvel // 2] = 1e30
    ref = s.apply_operator(w.dt, x)
    xd = torch.tensor(x, dtype=torch.float32, device="cuda")
    yd = torch.zeros_like(xd)
    torch.cuda.synchronize()
    s.apply_operator_device(w.dt, xd.data_ptr(), yd.data_ptr(), fp32=True)
    y = yd.double().cpu().numpy()
    big, small = np.abs(ref) > 1e39, np.abs(ref) < 1e38 * w.dt ** 2 / 4
    assert big.any() and np.array_equal(y[big], np.sign(ref[big]) * np.inf)
    assert np.isfinite(y[small]).all()


@pytest.mark.parametrize("shots", [19, 20, 21, 33, 64])
def test_stacked_shots_from_the_face_blocks(shots):
    # without the couplings, batches around the 20 shots from which a lane takes a shot, and around its 32 lanes
    need_gpu()
    w = _workload(2, 2, 2, n=3)
    rng = np.random.default_rng(shots)
    out = []
    for share in (0.0, 1.0):
        s = _solver(w, precision="mixed", preconditioner=1, rel_tol=1e-11, max_iters=20000)
        s.set_coupling_share(share)
        s.set_material(w.lam, w.mu, w.rho)
        assert (s.coupling_bytes > 0) == (share > 0)
        s.set_shots(shots)
        v0, sig0 = s.get_state(0)
        if not out:
            states = [(rng.normal(size=v0.shape), rng.normal(size=sig0.shape)) for _ in range(shots)]
        for k, st in enumerate(states):
            s.set_state(*st, shot=k)
        s.step(w.dt, 1)
        out.append(np.array([s.get_state(k)[0] for k in range(shots)]))
    for k in range(shots):
        assert rel_l2(out[0][k], out[1][k]) < 1e-8
    sim = oracle_sim(w)
    sim.set_state(*states[-1])
    sim.step(1)
    assert rel_l2(out[0][-1], sim.v_tr) < 1e-8


@pytest.mark.parametrize("dim,p,pg", [(2, 1, 0), (2, 2, 2), (2, 4, 2), (3, 1, 1), (3, 3, 3)])
@pytest.mark.parametrize("shift", [0.0, 1e-3])
def test_constant_and_nearly_constant_vectors_lose_nothing_to_cancellation(dim, p, pg, shift):
    # the face term of a constant is zero: the operator leaves the mass term, a few roundings of each value (20 eps in
    # FP64, 5 in FP32 in norm). A small rough part on top of the constant comes out as the operator on that part alone.
    torch = need_gpu()
    from paper_1802_04516_gb300 import binding
    w = synth.scaled("c2", ny=10, p=p, steps=1) if dim == 2 else _workload(dim, p, pg)
    w.p_gamma, w.scheme = pg, "cn" if pg == 0 else "stdg"
    s = _solver(w, precision="mixed", preconditioner=0)
    assert s.coupling_bytes > 0
    NP, NG = s.query(2), s.query(4)
    M, T = np.zeros((NP, NP)), np.zeros((NG, NG))
    d = lambda a: a.ctypes.data_as(binding._D)  # noqa: E731
    binding.load().stdg_reference_tables(dim, p, pg, d(M), None, d(T), None, None, None)
    X = np.asarray(w.xyz)[w.elem_vert]
    det = np.linalg.det(X[:, 1:] - X[:, :1])
    rng = np.random.default_rng(4)
    x = np.broadcast_to(rng.uniform(1.1, 1.9, (1, dim, 1, 1)), (w.n_elem, dim, NG, NP)).astype(np.float32).astype(np.float64)
    rough = (shift * rng.uniform(-1, 1, x.shape)).astype(np.float32).astype(np.float64)
    full = (x + rough).astype(np.float32).astype(np.float64)   # stays within the binade 1..2
    rough = full - x

    def run(v, fp32):
        if not fp32:
            return s.apply_operator(w.dt, v.ravel()).reshape(v.shape)
        vd = torch.tensor(v.ravel(), dtype=torch.float32, device="cuda")
        yd = torch.zeros_like(vd)
        torch.cuda.synchronize()
        s.apply_operator_device(w.dt, vd.data_ptr(), yd.data_ptr(), fp32=True)
        return yd.double().cpu().numpy().reshape(v.shape)

    mass = np.einsum("e,ab,nm,ekbm->ekan", np.asarray(w.rho) * det, T, M, x)
    exact = mass + (run(rough, False) if shift else 0.0)
    for fp32, eps in ((False, 2.0 ** -53), (True, 2.0 ** -24)):
        bar = (5 if fp32 else 20) * eps
        assert rel_l2(run(full, fp32), exact) < bar
