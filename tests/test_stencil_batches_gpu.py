"""The FP32 stencil preconditioner of stacked shots on both sides of the 25 shots from which its element-local step
runs on the tensor cores (kind::tf32): below, the FP32 blocks at their own accuracy (1e-4, as the 32-bit blocks of
one shot); from there on the TF32 blocks (2e-3), full and partial groups of shots, with the iteration counts and the
convergence of FP32 blocks, on an image that only contexts with that many shots hold; and the launch settings that the
autotuner searches for each of these kernels."""
import dataclasses

import numpy as np
import pytest

import synth
from helpers import gpu_solver, need_gpu, oracle_sim, rel_l2

pytestmark = pytest.mark.gpu


def _applied(s, w, r):
    import torch
    rd = torch.tensor(r, dtype=torch.float32, device="cuda")
    zd = torch.zeros_like(rd)
    torch.cuda.synchronize()
    s.apply_preconditioner_device(w.dt, rd.data_ptr(), zd.data_ptr(), fp32=True)
    return zd.double().cpu().numpy()


def test_local_step_around_the_tensor_core_limit():
    # one context through growing and shrinking batches at one slab size, then another
    need_gpu()
    from oracle.precond import pre2
    w = synth.scaled("c4", ny=8, steps=1, n_shots=1)
    s = gpu_solver(w, precision="mixed", with_sources=False, with_receivers=False, preconditioner=2)
    for dt in (w.dt, 0.5 * w.dt):
        wd = dataclasses.replace(w, dt=dt)
        sim = oracle_sim(wd)
        P = pre2(sim.A, w.n_elem, sim.mesh.elem_nbr)
        for shots in (2, 24, 25, 29, 24, 40, 8):
            s.set_shots(shots)
            r = np.random.default_rng(shots).normal(size=(shots, sim.A.shape[0]))
            z = _applied(s, wd, r)
            worst = max(rel_l2(z[k], P @ r[k]) for k in range(shots))
            assert worst < (1e-4 if shots < 25 else 2e-3), (shots, worst)


def test_only_large_batches_hold_the_tensor_core_image():
    need_gpu()
    w = synth.scaled("c4", ny=8, steps=1, n_shots=1)
    s = gpu_solver(w, precision="mixed", with_sources=False, with_receivers=False, preconditioner=2)
    held = {}
    for shots in (23, 24, 25, 26, 24):
        s.set_shots(shots)
        held.setdefault(shots, []).append(s.query(10))
    assert held[24][0] == held[24][1]
    image = held[25][0] - held[24][0] - (held[26][0] - held[25][0])
    assert image >= 4 * 36 * 36 * w.n_elem
    assert abs((held[24][0] - held[23][0]) - (held[26][0] - held[25][0])) < image / 2   # no image between 23 and 24


@pytest.mark.parametrize("shots", [29, 40])
def test_tensor_core_blocks_keep_iteration_counts(shots):
    # as many iterations as the slowest shot alone (FP32 arithmetic), with the margin of the per-shot test
    need_gpu()
    w = synth.scaled("c4", ny=10, steps=3, n_shots=shots)
    kw = dict(precision="mixed", rel_tol=1e-10, max_iters=20000, preconditioner=2)
    st = gpu_solver(w, **kw).step(w.dt, 3)
    assert st["status"] == 0
    singles = []
    for k in range(shots):
        wk = dataclasses.replace(w, shots_xs=w.shots_xs[k:k + 1], shots_dir=w.shots_dir[k:k + 1])
        singles.append(gpu_solver(wk, **kw).step(w.dt, 3)["iters_max"])
    assert st["iters_max"] <= 1.15 * max(singles) + 5


def test_tensor_core_blocks_converge_on_the_inversion_medium():
    # 30 slabs of the 60,024-triangle heterogeneous medium with 29 shots: bounded inner iterations in every slab (blocks
    # of fewer bits once stagnated there after 16 slabs)
    need_gpu()
    w = synth.c5_adjoint(steps=30, true_model=True, n_shots=29)
    w = dataclasses.replace(w, shots_xs=np.stack([np.linspace(0.1, 1.9, 29), np.full(29, 0.85)], axis=1))
    s = gpu_solver(w, precision="mixed", rel_tol=1e-8, max_iters=1500, preconditioner=2, gmres_restart=10, inner_tol=1e-2)
    worst = 0
    for _ in range(w.n_steps):
        st = s.step(w.dt, 1)
        assert st["status"] == 0
        worst = max(worst, st["iters_max"])
    assert worst < 400, worst


@pytest.mark.parametrize("p,precision,pre,shots,face,local", [
    (2, "mixed", 2, 1, 24, 3), (2, "mixed", 2, 9, 3, 1), (2, "mixed", 2, 29, 3, 2), (2, "fp64", 2, 1, 0, 1), (1, "mixed", 1, 1, 1, 0)])
def test_autotuner_searches_what_the_kernels_read(p, precision, pre, shots, face, local):
    # candidates: the face kernel's settings (the generic kernel of p = p_gamma = 1 has none) and the local step's; what
    # is not searched keeps its default
    need_gpu()
    w = synth.scaled("c4", ny=8, p=p, steps=1, n_shots=shots)
    s = gpu_solver(w, precision=precision, preconditioner=pre)
    t = s.autotune(w.dt)
    assert t["candidates"] == face + local
    assert (t["face_ms"] > 0) == (face > 0) and (t["pre2_ms"] > 0) == (local > 0)
    if face <= 3:
        assert t["face_register_cap"] == 1 and t["face_blocks_per_sm"] == 16
    if face <= 1:
        assert t["face_warps_per_block"] == 4
    if local != 3:
        assert t["pre2_warps_per_block"] == 4
    if local != 2:
        assert t["mma_ctas_per_sm"] == 2
