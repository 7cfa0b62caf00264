"""GPU: the face kernels' division and square root (shared reciprocals from a
float-float start, built-in operations outside their exponent range) against
the oracle bit for bit, on geometry scaled across that range's ends, with zero
area components (a box without jitter), faces beyond the 0.05 |d| limit, cells
with several Dirichlet faces, and diffusivities that are zero, negative, tiny
or huge."""
import dataclasses

import numpy as np
import pytest

import hexmesh
import oracle
from gpu_cases import bits, dev, mesh_of

pytestmark = pytest.mark.gpu


def _scaled(c, s):
    m = c.mesh
    m = dataclasses.replace(m, sf=m.sf * s * s, bface_sf=m.bface_sf * s * s, c=m.c * s, cf=m.cf * s,
                            bface_cf=m.bface_cf * s, v=m.v * s * s * s)
    return dataclasses.replace(c, mesh=m)


@pytest.mark.parametrize("jitter", [0.0, 0.2], ids=["box", "jittered"])
@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e-25, 1e25, 1e-46, 1e46, 1e-60, 1e60])
def test_assembly_and_operators_bitwise(scale, jitter):
    c = hexmesh.pressure_case((9, 7, 6), jitter=jitter, permute=True, seed=71, lognormal_gamma=True,
                              dirichlet=("xmax", "ymin", "zmin"))
    c = _scaled(c, scale)
    m = c.mesh
    rng = np.random.default_rng(72)
    # faces beyond the limit: the area vector turned across d (and against it)
    turn = rng.permutation(m.n_faces)[:40]
    d = m.c[m.upper_addr[turn]] - m.c[m.lower[turn]]
    t = np.cross(d, rng.standard_normal(d.shape))
    mag = np.linalg.norm(m.sf[turn], axis=1)[:, None]
    t *= mag / np.linalg.norm(t, axis=1)[:, None]
    m.sf[turn] = t + np.linspace(-0.08, 0.08, 40)[:, None] * mag * d / np.linalg.norm(d, axis=1)[:, None]
    c.gamma[:6] = [0.0, -0.0, -1.5, 1e-200, 1e95, 5e-324]
    M = mesh_of(c, centres=True)
    g = dict(sf=dev(m.sf), c=dev(m.c), bc=dev(m.bface_cell), bs=dev(m.bface_sf), bf=dev(m.bface_cf))
    up, dg = M.assemble_laplacian(g["sf"], g["c"], dev(c.gamma), g["bc"], g["bs"], g["bf"], dev(c.bgamma), dev(c.btype))
    uo, do = oracle.assemble_laplacian(m, c.gamma, c.bgamma, c.btype)
    assert np.array_equal(bits(up.cpu().numpy()), bits(uo))
    assert np.array_equal(bits(dg.cpu().numpy()), bits(do))
    w = M.fv_weights(g["sf"], dev(m.cf), g["c"])
    wo = oracle.fv_weights(m)
    assert np.array_equal(bits(w.cpu().numpy()), bits(wo))
    p = rng.standard_normal(m.n_cells)
    p[::5] = 0.0
    gr = M.fv_grad(g["sf"], w, dev(m.v), dev(p), g["bc"], g["bs"], dev(c.btype))
    go = oracle.fv_grad(m, wo, c.btype, p)
    assert np.array_equal(bits(gr.cpu().numpy()), bits(go))
    phi, bphi = rng.standard_normal(m.n_faces), rng.standard_normal(m.n_bfaces)
    corr, b = M.pressure_rhs(g["sf"], g["c"], w, dev(c.gamma), gr, dev(phi), g["bc"], dev(bphi))
    corro, bo = oracle.pressure_rhs(m, wo, c.gamma, go, phi, bphi)
    assert np.array_equal(bits(corr.cpu().numpy()), bits(corro))
    assert np.array_equal(bits(b.cpu().numpy()), bits(bo))


@pytest.mark.parametrize("n", [(1, 1, 1), (2, 1, 1), (33, 5, 3)], ids=["one-cell", "two-cells", "33x5x3"])
def test_caller_order_amul_bitwise(n):
    """The grouped row loop of the Amul on the caller's arrays at its ends: no faces, one face, partial groups."""
    c = hexmesh.pressure_case(n, jitter=0.2, permute=True, seed=73, lognormal_gamma=True)
    m = c.mesh
    uo, do = oracle.assemble_laplacian(m, c.gamma, c.bgamma, c.btype)
    M = mesh_of(c)
    x = np.random.default_rng(74).standard_normal(m.n_cells)
    for dt in (np.float64, np.float32):
        y = M.amul(dev(do.astype(dt)), dev(uo.astype(dt)), dev(x.astype(dt))).cpu().numpy()
        assert np.array_equal(bits(y), bits(oracle.amul(m.lower, m.upper_addr, do.astype(dt), uo.astype(dt), x.astype(dt))))
