"""GPU: rows around the kernels' groups of six entries (6, 7, 12, 13, 18, 19 and
more on a side): the Amul on the caller's arrays bit for bit, and the solves at
matched iterations, whose sweeps load six entries ahead of the barrier and the
rest of a row in groups."""
import numpy as np
import pytest

import oracle
from gpu_cases import bits, dev

pytestmark = pytest.mark.gpu
WIDTHS = (5, 6, 7, 11, 12, 13, 17, 18, 19, 25)


def mesh_with_rows(n=600, seed=141):
    """A chain with, for every width w, a cell that has w upper neighbours and another that has w lower ones."""
    rng = np.random.default_rng(seed)
    pairs = {(i, i + 1) for i in range(n - 1)}
    for k, w in enumerate(WIDTHS):
        low, high = 3 + 7 * k, n - 4 - 7 * k
        pairs = {p for p in pairs if p[0] != low and p[1] != high}
        pairs |= {(low, int(v)) for v in rng.choice(np.arange(low + 1, low + 200), w, replace=False)}
        pairs |= {(int(v), high) for v in rng.choice(np.arange(high - 200, high), w, replace=False) if int(v) != low}
    keys = np.array(sorted(pairs), dtype=np.int32)
    lo, up = np.ascontiguousarray(keys[:, 0]), np.ascontiguousarray(keys[:, 1])
    upper = -rng.uniform(0.5, 1.5, len(lo))
    diag = np.full(n, 0.05)
    np.add.at(diag, lo, -upper)
    np.add.at(diag, up, -upper)
    return n, lo, up, upper, diag, rng


def test_caller_order_amul_bitwise():
    from paper_2512_22215_gb300 import LduMesh
    n, lo, up, upper, diag, rng = mesh_with_rows()
    M, x = LduMesh(lo, up, n), rng.standard_normal(n)
    for dt in (np.float64, np.float32):
        a = [t.astype(dt) for t in (diag, upper, x)]
        y = M.amul(*(dev(t) for t in a)).cpu().numpy()
        assert np.array_equal(bits(y), bits(oracle.amul(lo, up, *a)))


@pytest.mark.parametrize("threads", [0, 64, 256, 512, 1024])
def test_solves_at_matched_iterations(threads):
    from paper_2512_22215_gb300 import LduMesh, SolverControls
    n, lo, up, upper, diag, rng = mesh_with_rows()
    M, b = LduMesh(lo, up, n), rng.standard_normal(n)
    x, p = M.solve(dev(diag), dev(upper), dev(b), None,
                   SolverControls(precond=2, tolerance=0.0, max_iter=12, block_threads=threads))
    xo, _ = oracle.pcg(lo, up, diag, upper, b, precond=2, tol=0.0, max_iter=12)
    assert p["status"] == 0 and p["n_iter"] == 12
    assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-10 * np.linalg.norm(xo)
    x, p = M.solve(dev(diag), dev(upper), dev(b), None,
                   SolverControls(precond=2, precision=1, tolerance=1e-10, block_threads=threads))
    r = b - oracle.amul(lo, up, diag, upper, x.cpu().numpy())
    assert p["status"] == 0 and p["converged"] == 1 and np.abs(r).sum() <= 1e-10 * 2 * np.abs(b).sum()


@pytest.mark.parametrize("threads", [0, 64, 1024])
def test_preconditioner_bitwise(threads):
    """Row order is the sequential sweeps' (through the preconditioner call, 0) and does not depend on the block size."""
    from paper_2512_22215_gb300 import LduMesh, SolverControls
    n, lo, up, upper, diag, rng = mesh_with_rows()
    M, b = LduMesh(lo, up, n), rng.standard_normal(n)
    rD, _ = oracle.dic_factor(lo, up, diag, upper)
    if threads == 0:
        M.prepare(dev(diag), dev(upper), 2)
        assert np.array_equal(bits(M.read_rD().cpu().numpy()), bits(rD))
        assert np.array_equal(bits(M.precondition(dev(b), 2).cpu().numpy()), bits(oracle.dic_precondition(lo, up, upper, rD, b)))
        return
    # one iteration from 0: x = alpha w
    x, _ = M.solve(dev(diag), dev(upper), dev(b), None,
                   SolverControls(precond=2, tolerance=0.0, max_iter=1, block_threads=threads))
    w = oracle.dic_precondition(lo, up, upper, rD, b)
    alpha = x.cpu().numpy()[0] / w[0]
    assert np.abs(x.cpu().numpy() - alpha * w).max() <= 1e-13 * np.abs(alpha * w).max()
