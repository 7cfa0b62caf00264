"""GPU: meshes of many DIC levels (natural order): threads without a row for
more levels than the sweeps look ahead, more levels than the chunk table holds
(512), on the grid, on the first block alone and in a batch, against the
oracle; and the default block size against the largest one, whose sweeps
have no loads ahead."""
import numpy as np
import pytest
import torch

import oracle
from gpu_cases import assemble_oracle, case, dev, mesh_of

pytestmark = pytest.mark.gpu

# levels: 1107, past the table; 78 and 68 with levels that grow and shrink by a row or a few
MESHES = [(1100, 8, 1), (40, 40, 1), (40, 20, 10), (24, 24, 24)]


@pytest.mark.parametrize("tail", [None, "0", "64"], ids=["tail", "grid", "short-tail"])
@pytest.mark.parametrize("n", MESHES)
def test_matched_iterations(n, tail, monkeypatch):
    from paper_2512_22215_gb300 import SolverControls
    if tail is not None:
        monkeypatch.setenv("SPUMA_TAIL_ROWS", tail)
    c = case(n, jitter=0.2 if min(n) > 1 else 0.0, seed=131, lognormal=True)
    m = c.mesh
    M = mesh_of(c)
    assert M.n_levels == sum(n) - 2
    uo, do = assemble_oracle(c)
    xo, _ = oracle.pcg(m.lower, m.upper_addr, do, uo, c.b, precond=2, tol=0.0, max_iter=8)
    for threads in (0, 64, 256, 512, 1024):
        x, p = M.solve(dev(do), dev(uo), dev(c.b), None,
                       SolverControls(precond=2, tolerance=0.0, max_iter=8, block_threads=threads))
        assert p["status"] == 0 and p["n_iter"] == 8
        assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-10 * np.linalg.norm(xo)
        x, p = M.solve(dev(do), dev(uo), dev(c.b), None,
                       SolverControls(precond=2, precision=1, tolerance=1e-9, block_threads=threads))
        r = c.b - oracle.amul(m.lower, m.upper_addr, do, uo, x.cpu().numpy())
        assert p["status"] == 0 and p["converged"] == 1 and np.abs(r).sum() < 2e-9 * np.abs(c.b).sum()


@pytest.mark.parametrize("precision", [0, 1])
def test_batch(precision):
    from paper_2512_22215_gb300 import BatchSolve, SolverControls
    cs = [case(n, jitter=0.2 if min(n) > 1 else 0.0, seed=132, lognormal=True) for n in MESHES]
    sys_ = [assemble_oracle(c) for c in cs]
    x = [torch.zeros(c.mesh.n_cells, dtype=torch.float64, device="cuda") for c in cs]
    batch = BatchSolve([mesh_of(c) for c in cs], [dev(d) for _, d in sys_], [dev(u) for u, _ in sys_],
                       [dev(c.b) for c in cs], x, SolverControls(precond=2, precision=precision, tolerance=1e-9),
                       autotune=False)
    batch.run()
    for c, (u, d), t, p in zip(cs, sys_, x, batch.results()):
        r = c.b - oracle.amul(c.mesh.lower, c.mesh.upper_addr, d, u, t.cpu().numpy())
        assert p["status"] == 0 and p["converged"] == 1 and np.abs(r).sum() < 2e-9 * np.abs(c.b).sum()


@pytest.mark.parametrize("precision", [0, 1])
def test_default_keeps_up(precision):
    """599 levels of at most 300 rows: the default may cost no more than 1.2 times blocks of 1024 threads (3.9 times,
    when threads looked through all the levels left)."""
    from paper_2512_22215_gb300 import SolverControls
    c = case((300, 300, 1), seed=133, lognormal=True)
    M = mesh_of(c)
    uo, do = assemble_oracle(c)
    d, u, b = dev(do), dev(uo), dev(c.b)

    def ms(threads):
        ctl = SolverControls(precond=2, precision=precision, tolerance=0.0, max_iter=20, block_threads=threads)
        best = 1e9
        for _ in range(5):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            M.solve(d, u, b, None, ctl)
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1))
        return best
    assert ms(0) < 1.2 * ms(1024)
