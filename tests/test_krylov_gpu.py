"""Krylov kernels at the sizes where their reductions and vector accesses can go wrong: fewer values
than one block, shots whose segments start off a 16-byte boundary, restart lengths around the 16
columns that one pass of the multi-dot kernel takes, and shots that converge at different steps.
Every shot against its own oracle run, at the stated state bars (1e-10 FP64, 1e-8 mixed)."""
import numpy as np
import pytest

import synth
from helpers import need_gpu, oracle_sim, rel_l2

pytestmark = pytest.mark.gpu

CASES = [  # cells, p, p_gamma, scheme, shots, restart, preconditioner, precision
    (2, 1, 0, "cn", 1, 30, 1, "fp64"),
    (3, 1, 0, "cn", 3, 30, 1, "mixed"),
    (3, 2, 0, "cn", 2, 30, 0, "fp64"),
    (4, 2, 0, "cn", 1, 30, 1, "mixed"),
    (3, 3, 0, "cn", 1, 30, 1, "fp64"),
    (2, 4, 0, "cn", 1, 30, 1, "mixed"),
    (2, 1, 1, "stdg", 1, 2, 1, "fp64"),
    (3, 2, 1, "stdg", 3, 15, 1, "fp64"),
    (3, 2, 1, "stdg", 3, 16, 1, "mixed"),
    (3, 2, 2, "stdg", 2, 17, 2, "mixed"),
    (4, 3, 2, "stdg", 1, 64, 0, "fp64"),
]


@pytest.mark.parametrize("cells,p,pg,scheme,shots,restart,pre,precision", CASES)
def test_small_and_unaligned_solves(cells, p, pg, scheme, shots, restart, pre, precision):
    need_gpu()
    from paper_1802_04516_gb300.binding import Solver
    xyz, ev, per = synth.tri_grid(cells + 1, cells, 1.0, 1.0, periodic=False, jitter=0.2, seed=4)
    rng = np.random.default_rng(8)
    n = ev.shape[0]
    w = synth.Workload("krylov", 2, xyz, ev, per, rng.uniform(1, 2, n), rng.uniform(.5, 1, n), rng.uniform(.8, 1.2, n),
                       p=p, p_gamma=pg, scheme=scheme, dt=0.05, n_steps=2, h=1.0 / cells)
    s = Solver(2, p, pg, scheme=scheme, precision=precision, rel_tol=1e-13 if precision == "fp64" else 1e-12, max_iters=20000,
               gmres_restart=restart, preconditioner=pre)
    s.set_mesh(xyz, ev, per)
    s.set_material(w.lam, w.mu, w.rho)
    s.set_shots(shots)
    sims = [oracle_sim(w) for _ in range(shots)]
    for k, sim in enumerate(sims):
        v, sig = rng.normal(size=sim.v_tr.shape) * 10.0 ** -k, rng.normal(size=sim.sig_tr.shape) * 10.0 ** -k
        if k == 2:
            v, sig = 0 * v, 0 * sig      # a shot with nothing to solve
        sim.set_state(v, sig)
        s.set_state(v, sig, shot=k)
        sim.step(2)
    s.step(w.dt, 2)
    tol = 1e-10 if precision == "fp64" else 1e-8
    for k, sim in enumerate(sims):
        v, _ = s.get_state(k)
        assert rel_l2(v, sim.v_tr) < tol


@pytest.mark.parametrize("p,precision", [(1, "fp64"), (2, "mixed"), (3, "fp64"), (1, "mixed")])
def test_crank_nicolson_3d(p, precision):
    need_gpu()
    from paper_1802_04516_gb300.binding import Solver
    xyz, ev, per = synth.tet_kuhn(1 if p == 3 else 2, 1.0, periodic=False, jitter=0.1, seed=4)
    rng = np.random.default_rng(9)
    n = ev.shape[0]
    w = synth.Workload("cg3", 3, xyz, ev, per, rng.uniform(1, 2, n), rng.uniform(.5, 1, n), rng.uniform(.8, 1.2, n),
                       p=p, p_gamma=0, scheme="cn", dt=0.05, n_steps=3, h=0.5)
    s = Solver(3, p, 0, scheme="cn", precision=precision, rel_tol=1e-13 if precision == "fp64" else 1e-12, max_iters=20000)
    s.set_mesh(xyz, ev, per)
    s.set_material(w.lam, w.mu, w.rho)
    sim = oracle_sim(w)
    v, sig = rng.normal(size=sim.v_tr.shape), rng.normal(size=sim.sig_tr.shape)
    sim.set_state(v, sig)
    s.set_state(v, sig)
    s.step(w.dt, 3)
    sim.step(3)
    assert rel_l2(s.get_state()[0], sim.v_tr) < (1e-10 if precision == "fp64" else 1e-8)


@pytest.mark.parametrize("nx,ny,p,precision", [  # one cluster holds 1,360 triangles at p = 1 and 672 at p = 2
    (20, 34, 1, "fp64"), (21, 33, 1, "fp64"), (21, 33, 1, "mixed"), (40, 31, 1, "fp64"),
    (16, 21, 2, "mixed"), (17, 21, 2, "mixed"), (17, 21, 2, "fp64")])
def test_crank_nicolson_around_the_cluster_limit(nx, ny, p, precision):
    need_gpu()
    from paper_1802_04516_gb300.binding import Solver
    xyz, ev, per = synth.tri_grid(nx, ny, 1.0, 1.0, periodic=False, jitter=0.2, seed=6)
    rng = np.random.default_rng(12)
    n = ev.shape[0]
    w = synth.Workload("krylov", 2, xyz, ev, per, rng.uniform(1, 2, n), rng.uniform(.5, 1, n), rng.uniform(.8, 1.2, n),
                       p=p, p_gamma=0, scheme="cn", dt=0.02, n_steps=2, h=1.0 / nx)
    sim = oracle_sim(w)
    v, sig = rng.normal(size=sim.v_tr.shape), rng.normal(size=sim.sig_tr.shape)
    sim.set_state(v, sig)
    sim.step(2)
    s = Solver(2, p, 0, scheme="cn", precision=precision, rel_tol=1e-13 if precision == "fp64" else 1e-12, max_iters=20000,
               preconditioner=1)
    s.set_mesh(xyz, ev, per)
    s.set_material(w.lam, w.mu, w.rho)
    s.set_state(v, sig)
    s.step(w.dt, 2)
    out, _ = s.get_state()
    assert rel_l2(out, sim.v_tr) < (1e-10 if precision == "fp64" else 1e-8)
