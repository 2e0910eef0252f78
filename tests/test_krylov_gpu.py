"""Krylov kernels at the sizes where their reductions and vector accesses can go wrong: fewer values
than one block, shots whose segments start off a 16-byte boundary, restart lengths around the 16
columns that one pass of the multi-dot kernel takes, and shots that converge at different steps.
Every shot against its own oracle run, at the stated state bars (1e-10 FP64, 1e-8 mixed)."""
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

import synth
from helpers import ROOT, need_gpu, oracle_sim, rel_l2

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


# runtime of a device that cannot schedule a cluster of 16 blocks: the occupancy query answers none, a launch fails
NO_CLUSTERS = r"""
#include <dlfcn.h>
#include <cuda_runtime_api.h>
extern "C" cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
    *n = 0;
    return cudaSuccess;
}
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* f, void** args) {
    for (unsigned i = 0; i < cfg->numAttrs; ++i)
        if (cfg->attrs[i].id == cudaLaunchAttributeClusterDimension && cfg->attrs[i].val.clusterDim.x > 8)
            return cudaErrorInvalidClusterSize;
    using F = cudaError_t (*)(const cudaLaunchConfig_t*, const void*, void**);
    return ((F)dlsym(RTLD_NEXT, "cudaLaunchKernelExC"))(cfg, f, args);
}
"""

SMALL_CN = """
import sys
import numpy as np
sys.path.insert(0, {root!r})
import synth
from paper_1802_04516_gb300.binding import Solver
xyz, ev, per = synth.tri_grid(8, 7, 1.0, 1.0, periodic=False, jitter=0.2, seed=6)
out = []
for precision, use_graph in (("fp64", True), ("mixed", True), ("fp64", False)):
    s = Solver(2, 2, 0, scheme="cn", precision=precision, rel_tol=1e-13 if precision == "fp64" else 1e-12, max_iters=20000,
               preconditioner=1, use_graph=use_graph)
    s.set_mesh(xyz, ev, per)
    s.set_material(*synth.homogeneous(ev.shape[0], 2.0, 1.0, 1.0))
    v, sig = s.get_state()
    rng = np.random.default_rng(12)
    s.set_state(rng.normal(size=v.shape), rng.normal(size=sig.shape))
    s.step(0.02, 2)
    out.append(s.get_state()[0])
np.save(sys.argv[1], np.array(out))
"""


def test_small_crank_nicolson_without_clusters_of_sixteen(tmp_path):
    need_gpu()
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    src, lib = tmp_path / "fake.cpp", tmp_path / "fake.so"
    src.write_text(NO_CLUSTERS)
    subprocess.run([gxx, "-shared", "-fPIC", "-I", "/usr/local/cuda/include", "-o", str(lib), str(src), "-ldl"], check=True)
    got = []
    for fake in (False, True):
        env = dict(os.environ, LD_PRELOAD=str(lib)) if fake else dict(os.environ)
        path = tmp_path / ("%d.npy" % fake)
        r = subprocess.run([sys.executable, "-c", SMALL_CN.format(root=ROOT), str(path)], env=env, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        got.append(np.load(path))
    for k, tol in enumerate((1e-10, 1e-8, 1e-10)):
        assert rel_l2(got[1][k], got[0][k]) < tol
    assert not np.array_equal(got[1][0], got[0][0])   # the runtime was the fake one: another order of the sums
