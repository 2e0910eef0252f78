"""Block-Jacobi apply with one thread per (element, row): meshes on which the rule for the elements per block takes
one, some and the most elements, with ragged last blocks, against the oracle. Bars: 1e-9 in FP64, 2e-5 in FP32 (as the
other preconditioner and FP32 operator tests)."""
import numpy as np
import pytest

import synth
from helpers import need_gpu, oracle_sim, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n,shots", [(1, 20, 1), (1, 39, 5), (2, 14, 1), (2, 19, 3), (2, 25, 1), (3, 14, 1), (3, 16, 2)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_elements_per_block(p, n, shots, precision):
    torch = need_gpu()
    from oracle.precond import pre1
    from paper_1802_04516_gb300.binding import Solver
    xyz, ev, per = synth.tri_grid(n + 1, n, 1.0, 1.0, periodic=False, jitter=0.2, seed=3)
    ne = ev.shape[0]
    rng = np.random.default_rng(5)
    w = synth.Workload("rows", 2, xyz, ev, per, rng.uniform(1, 2, ne), rng.uniform(.5, 1, ne), rng.uniform(.8, 1.2, ne),
                       p=p, p_gamma=p, scheme="stdg", dt=0.02, n_steps=1, h=1.0 / n)
    sim = oracle_sim(w)
    P = pre1(sim.A, w.n_elem)
    s = Solver(2, p, p, precision=precision, preconditioner=1)
    s.set_mesh(w.xyz, w.elem_vert, w.period)
    s.set_material(w.lam, w.mu, w.rho)
    s.set_shots(shots)
    r = np.random.default_rng(7).normal(size=(shots, sim.A.shape[0]))
    rd = torch.tensor(r, dtype=torch.float64 if precision == "fp64" else torch.float32, device="cuda")
    zd = torch.zeros_like(rd)
    torch.cuda.synchronize()
    s.apply_preconditioner_device(w.dt, rd.data_ptr(), zd.data_ptr(), fp32=precision == "mixed")
    z = zd.double().cpu().numpy()
    for k in range(shots):
        assert rel_l2(z[k], P @ r[k]) < (1e-9 if precision == "fp64" else 2e-5)
