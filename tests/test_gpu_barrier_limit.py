"""GPU: a time limit that a grid barrier's wait cannot keep ends the solve with
its status whatever the system's size, small systems (one block, a cluster of
blocks) included; a limit of a second does not."""
import pytest

from gpu_cases import assemble_oracle, case, dev, mesh_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limit,status", [(0, 8), (1, 8), (1_000_000_000, 0)])
@pytest.mark.parametrize("n", [(8, 8, 8), (12, 12, 12), (20, 20, 20)])
def test_small_systems_keep_the_limit(n, limit, status):
    from paper_2512_22215_gb300 import SolverControls, lib
    c = case(n, jitter=0.2, permute=True, seed=161, lognormal=True)
    M = mesh_of(c)
    uo, do = assemble_oracle(c)
    lib().spuma_set_barrier_timeout_ns(limit)
    try:
        _, p = M.solve(dev(do), dev(uo), dev(c.b), None, SolverControls(precond=2), check_status=False)
    finally:
        lib().spuma_set_barrier_timeout_ns(2_000_000_000)
    assert p["status"] == status and p["converged"] == (status == 0)
