"""GPU: the solver kernels that a solve is routed to by its size and shape, each
at the ends of its range, against the oracle's PCG at the same iteration count:
one block (small systems), a cluster of blocks, the grid with loads ahead (up
to 512 threads) and without (1024), FP64 and mixed; PBiCG on rows wider than
its entry groups; and GAMG by the sizes of its levels."""
import numpy as np
import pytest
import torch

import hexmesh
import oracle
from gpu_cases import assemble_oracle, case, dev, mesh_of

pytestmark = pytest.mark.gpu

# (mesh, permuted, iterations): 1 face; 31 and 33 rows (a piece's edge); 1024 and 1025 rows (one block's and
# beyond); 38400 and 38440 rows (the cluster's 16 x 2400 slots and beyond); 256 and 259 levels (the level tables' 256
# and beyond).  DIC factors a chain exactly: one iteration.  20 iterations are few enough for sums taken in another
# order to stay within 1e-10.
SHAPES = [((2, 1, 1), False, 1), ((31, 1, 1), False, 1), ((11, 3, 1), True, 8), ((16, 16, 4), False, 20),
          ((41, 25, 1), True, 20), ((17, 16, 16), False, 20), ((29, 23, 20), True, 20), ((40, 40, 24), True, 20),
          ((31, 31, 40), True, 20), ((199, 58, 1), False, 20), ((200, 60, 1), False, 20), ((150, 60, 2), False, 20)]


@pytest.mark.parametrize("n,permute,its", SHAPES)
def test_dic_pcg_matched_iterations(n, permute, its):
    from paper_2512_22215_gb300 import SolverControls
    c = case(n, jitter=0.2, permute=permute, seed=91, lognormal=True)
    m = c.mesh
    M = mesh_of(c, centres=permute)
    uo, do = assemble_oracle(c)
    x0 = np.random.default_rng(92).standard_normal(m.n_cells)
    xo, po = oracle.pcg(m.lower, m.upper_addr, do, uo, c.b, x0=x0, precond=2, tol=0.0, max_iter=its)
    assert po["n_iter"] == its
    for threads in (0, 512, 1024):
        x, p = M.solve(dev(do), dev(uo), dev(c.b), dev(x0),
                       SolverControls(precond=2, tolerance=0.0, max_iter=its, block_threads=threads))
        assert p["n_iter"] == its and p["status"] == 0 and p["n_levels"] == M.n_levels
        assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-10 * np.linalg.norm(xo)
        assert p["initial_residual"] == pytest.approx(po["initial_residual"], rel=1e-12)
        assert p["final_residual"] == pytest.approx(po["final_residual"], rel=1e-6, abs=1e-13)


@pytest.mark.parametrize("n,permute", [((2, 1, 1), False), ((33, 5, 3), True), ((26, 25, 24), True), ((150, 60, 2), False)])
@pytest.mark.parametrize("threads", [0, 64, 512, 1024])
def test_mixed_dic_residual(n, permute, threads):
    from paper_2512_22215_gb300 import MIXED, SolverControls
    c = case(n, jitter=0.2, permute=permute, seed=93, lognormal=True)
    m = c.mesh
    M = mesh_of(c, centres=permute)
    uo, do = assemble_oracle(c)
    x, p = M.solve(dev(do), dev(uo), dev(c.b), None,
                   SolverControls(precond=2, precision=MIXED, tolerance=1e-11, block_threads=threads))
    assert p["converged"] == 1 and p["status"] == 0
    r = c.b - oracle.amul(m.lower, m.upper_addr, do, uo, x.cpu().numpy())
    assert np.abs(r).sum() / np.abs(c.b).sum() < 1e-11
    # no more iterations than the oracle's form with the Amul, by the 15 % that FP32 trajectories differ
    _, po = oracle.mixed_reliable(m.lower, m.upper_addr, do, uo, c.b, precond=2, tol=1e-11, delta=1e-2)
    assert p["n_iter"] <= po["n_iter"] + max(3, (3 * po["n_iter"]) // 20)


def test_small_solver_reports_device_errors():
    from paper_2512_22215_gb300 import SolverControls, SpumaError, lib
    for n in (9, 20):      # one block, a cluster
        c = case(n, jitter=0.2, permute=True, seed=94, lognormal=True)
        M = mesh_of(c)
        uo, do = assemble_oracle(c)
        b = c.b.copy()
        b[-1] = np.inf
        for args, status in (((-do, -uo, c.b), 6), ((do, uo, b), 7), ((np.where(np.arange(len(do)) == 3, np.nan, do), uo, c.b), 7)):
            with pytest.raises(SpumaError) as e:
                M.solve(*(dev(t) for t in args), None, SolverControls(precond=2))
            assert e.value.status == status
        x, p = M.solve(dev(do), dev(uo), dev(c.b), None, SolverControls(precond=2, tolerance=1e-10))
        assert p["converged"] == 1 and p["status"] == 0
        # the prepared matrix it leaves behind is the one spuma_matrix_prepare makes
        w = M.precondition(dev(c.b), 2)
        rD = M.read_rD()
        M.prepare(dev(do), dev(uo), 2)
        assert torch.equal(w, M.precondition(dev(c.b), 2)) and torch.equal(rD, M.read_rD())
    # a time limit of zero is the grid solver's (n = 20: several blocks, whose wait runs out)
    lib().spuma_set_barrier_timeout_ns(0)
    try:
        _, p = M.solve(dev(do), dev(uo), dev(c.b), None, SolverControls(precond=2), check_status=False)
    finally:
        lib().spuma_set_barrier_timeout_ns(2_000_000_000)
    assert p["status"] == 8 and p["converged"] == 0


@pytest.mark.parametrize("threads", [256, 1024])
def test_pbicg_wide_rows(threads):
    """Rows of more than six entries on a side (the DILU sweeps' groups), and the row-extent Amul."""
    from paper_2512_22215_gb300 import LduMesh, SolverControls
    c = hexmesh.pressure_case((10, 9, 8), jitter=0.2, permute=True, seed=95, lognormal_gamma=True)
    m, rng = c.mesh, np.random.default_rng(96)
    n = m.n_cells
    pairs = set(zip(m.lower.tolist(), m.upper_addr.tolist()))
    for hub in (0, n // 2, n - 1):
        pairs |= {(min(hub, int(o)), max(hub, int(o))) for o in rng.choice(n, 16, replace=False) if o != hub}
    keys = np.array(sorted(pairs), dtype=np.int32)
    lo, ua = np.ascontiguousarray(keys[:, 0]), np.ascontiguousarray(keys[:, 1])
    lower, upper = -1.0 - rng.random(len(lo)), -1.0 - rng.random(len(lo))
    d = np.zeros(n)
    np.add.at(d, ua, np.abs(lower))
    np.add.at(d, lo, np.abs(upper))
    d /= 0.7
    M = LduMesh(lo, ua, n, asymmetric=True)
    x, p = M.pbicg_solve(dev(d), dev(lower), dev(upper), dev(c.b), None,
                         SolverControls(precond=3, tolerance=1e-10, block_threads=threads))
    assert p["converged"] == 1 and p["status"] == 0
    xo, _ = oracle.pbicg(lo, ua, d, lower, upper, c.b, precond=3, tol=0.0, max_iter=p["n_iter"])
    assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-9 * np.linalg.norm(xo)


# levels of the sizes where the rows per team change: 240 and 112 cells on the first block (two rows, one); 12560 on the
# grid (one) and 17770 (two: 128 rows per block, 124 teams)
@pytest.mark.parametrize("n", [(8, 8, 8), (30, 30, 30), (34, 34, 33)])
@pytest.mark.parametrize("smoother,name", [(0, "richardson"), (1, "gs2")])
def test_gamg_level_sizes(n, smoother, name):
    from oracle import gamg
    from paper_2512_22215_gb300 import GamgSolver, SolverControls
    c = case(n, jitter=0.2, permute=True, seed=108, lognormal=True)
    m = c.mesh
    uo, do = assemble_oracle(c)
    w = np.linalg.norm(m.sf, axis=1)
    S = GamgSolver(mesh_of(c, centres=True), dev(w), smoother=smoother)
    x, p = S.solve(dev(do), dev(uo), dev(c.b), None, SolverControls(tolerance=0.0, max_iter=3))
    assert p["n_iter"] == 3 and p["status"] == 0
    xo, _, _ = gamg.gamg(m.lower, m.upper_addr, do, uo, c.b, w, tol=0.0, max_iter=3, smoother=name)
    assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-8 * np.linalg.norm(xo)
