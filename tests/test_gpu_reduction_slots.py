"""GPU: solves whose first or last sums follow another sum's read at once, on
several blocks with next to no work between them, repeated: the diagonal and
unpreconditioned solve, DIC on a mesh without faces (one level), systems that
start converged and diagonal systems in a batch.  Every repetition has to give
the same report and solution, and those of the oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_cases import assemble_oracle, case, dev, mesh_of

pytestmark = pytest.mark.gpu
REPEATS = 50


@pytest.mark.parametrize("precond", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
def test_diagonal_solves_repeat(precond, precision):
    from paper_2512_22215_gb300 import SolverControls
    c = case((9, 9, 8), jitter=0.2, permute=True, seed=171, lognormal=True)
    m = c.mesh
    M = mesh_of(c)
    uo, do = assemble_oracle(c)
    ctl = SolverControls(precond=precond, precision=precision, tolerance=0.0 if precision == 0 else 1e-9,
                         max_iter=4 if precision == 0 else 20000, block_threads=32)
    d, u, b = dev(do), dev(uo), dev(c.b)
    x0, p0 = M.solve(d, u, b, None, ctl)
    assert p0["status"] == 0
    if precision == 0:
        xo, po = oracle.pcg(m.lower, m.upper_addr, do, uo, c.b, precond=precond, tol=0.0, max_iter=4)
        assert np.linalg.norm(x0.cpu().numpy() - xo) <= 1e-10 * np.linalg.norm(xo)
        assert p0["initial_residual"] == pytest.approx(po["initial_residual"], rel=1e-12)
    for _ in range(REPEATS):
        x, p = M.solve(d, u, b, None, ctl)
        assert p == p0 and torch.equal(x, x0)


@pytest.mark.parametrize("precision", [0, 1, 3])
def test_dic_without_faces(precision):
    from paper_2512_22215_gb300 import LduMesh, SolverControls
    n = 2000
    rng = np.random.default_rng(172)
    diag, b = rng.uniform(1.0, 2.0, n), rng.standard_normal(n)
    M = LduMesh(np.zeros(0, np.int32), np.zeros(0, np.int32), n)
    assert M.n_levels == 1
    ctl = SolverControls(precond=2, precision=precision, tolerance=1e-12, block_threads=32)
    d, u, bb = dev(diag), dev(np.zeros(0)), dev(b)
    for _ in range(REPEATS):
        x, p = M.solve(d, u, bb, None, ctl)
        assert p["status"] == 0 and p["converged"] == 1 and p["n_iter"] <= 4
        assert np.abs(x.cpu().numpy() - b / diag).max() <= 1e-12 * np.abs(b).sum() + 1e-15   # |r|_1 < tol |b|_1, diag >= 1


@pytest.mark.parametrize("precision", [0, 1, 3])
@pytest.mark.parametrize("precond", [1, 2])
def test_batch_of_converged_and_short_systems(precision, precond):
    from paper_2512_22215_gb300 import BatchSolve, SolverControls
    cs = [case(n, jitter=0.2, permute=True, seed=173 + k, lognormal=True) for k, n in enumerate([(9, 9, 8), (12, 7, 5), (20, 20, 3)])]
    sys_ = [assemble_oracle(c) for c in cs]
    meshes = [mesh_of(c) for c in cs]
    sol = [oracle.pcg(c.mesh.lower, c.mesh.upper_addr, d, u, c.b, precond=2, tol=1e-15, max_iter=2000)[0]
           for c, (u, d) in zip(cs, sys_)]
    ctl = SolverControls(precond=precond, precision=precision, tolerance=1e-9, block_threads=64)
    x = [dev(s) for s in sol]            # the first two start converged, the last from zero
    batch = BatchSolve(meshes, [dev(d) for _, d in sys_], [dev(u) for u, _ in sys_], [dev(c.b) for c in cs], x, ctl,
                       autotune=False)
    first = None
    for _ in range(REPEATS):
        for k, s in enumerate(sol):
            x[k].copy_(dev(s)) if k < 2 else x[k].zero_()
        batch.run()
        reports = batch.results()
        assert all(p["status"] == 0 and p["converged"] == 1 for p in reports)
        assert [p["n_iter"] for p in reports[:2]] == [0, 0] and reports[2]["n_iter"] > 0
        out = [t.clone() for t in x]
        first = first or (reports, out)
        assert reports == first[0] and all(torch.equal(s, t) for s, t in zip(out, first[1]))
        for p, (u, d), c, t in zip(reports, sys_, cs, out):
            r = c.b - oracle.amul(c.mesh.lower, c.mesh.upper_addr, d, u, t.cpu().numpy())
            assert p["true_rel_residual_l2"] == pytest.approx(np.linalg.norm(r) / np.linalg.norm(c.b), rel=1e-6, abs=1e-15)
