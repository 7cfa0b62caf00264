"""GPU: the assembly's per-cell boundary lists: any number of Dirichlet faces
on one cell, among the boundary's others and zero-gradient faces, added in
face order (bit for bit the oracle's diagonal), at a cost in proportion to
their number."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from gpu_cases import bits, case, dev, mesh_of

pytestmark = pytest.mark.gpu


def with_hub(m_faces, n=(9, 8, 7)):
    """The box with m_faces more Dirichlet faces on one inner cell, scattered over the face numbering."""
    c = case(n, jitter=0.2, permute=True, seed=151, lognormal=True)
    m, rng = c.mesh, np.random.default_rng(152)
    B = m.n_bfaces + m_faces
    at = np.ones(B, bool)
    at[rng.choice(B, m_faces, replace=False)] = False      # where the box's own faces go

    def merge(own, extra):
        out = np.empty((B,) + own.shape[1:], own.dtype)
        out[at], out[~at] = own, extra
        return out
    hub = int(m.lower[m.n_faces // 2])
    mesh = dataclasses.replace(
        m, bface_cell=merge(m.bface_cell, hub), bface_sf=merge(m.bface_sf, rng.uniform(0.1, 1.0, (m_faces, 3))),
        bface_cf=merge(m.bface_cf, m.c[hub] + rng.uniform(0.1, 1.0, (m_faces, 3))),
        bface_patch=merge(m.bface_patch, 0))
    return mesh, c.gamma, merge(c.bgamma, rng.uniform(0.5, 2.0, m_faces)), merge(c.btype, 1)


@pytest.mark.parametrize("wide", [False, True], ids=["fixed-width", "row-lists"])
@pytest.mark.parametrize("m_faces", [1, 2, 3, 5, 8, 16, 17, 33, 300])
def test_diagonal_bitwise(m_faces, wide):
    from paper_2512_22215_gb300 import LduMesh
    m, gamma, bgamma, btype = with_hub(m_faces)
    if wide:    # one more row of many faces: no fixed-width layout
        o, n = 3, m.n_cells
        have = set(zip(m.lower.tolist(), m.upper_addr.tolist()))
        new = [p for p in ((o, k) for k in range(o + 1, n, 7)) if p not in have]
        lo = np.concatenate([m.lower, [p[0] for p in new]]).astype(np.int32)
        up = np.concatenate([m.upper_addr, [p[1] for p in new]]).astype(np.int32)
        order = np.lexsort((up, lo))
        sf = np.concatenate([m.sf, np.ones((len(new), 3))])[order]
        gamma = np.concatenate([gamma, np.ones(len(new))])[order]
        m = dataclasses.replace(m, n_faces=len(lo), lower=lo[order], upper_addr=up[order], sf=sf)
    M = LduMesh(m.lower, m.upper_addr, m.n_cells)
    up, dg = M.assemble_laplacian(dev(m.sf), dev(m.c), dev(gamma), dev(m.bface_cell), dev(m.bface_sf), dev(m.bface_cf),
                                  dev(bgamma), dev(btype))
    uo, do = oracle.assemble_laplacian(m, gamma, bgamma, btype)
    assert np.array_equal(bits(up.cpu().numpy()), bits(uo))
    assert np.array_equal(bits(dg.cpu().numpy()), bits(do))


def test_cost_in_proportion():
    def us(m_faces):
        m, gamma, bgamma, btype = with_hub(m_faces, n=(20, 20, 20))
        M = mesh_of(dataclasses.make_dataclass("C", ["mesh"])(m))
        args = [dev(t) for t in (m.sf, m.c, gamma, m.bface_cell, m.bface_sf, m.bface_cf, bgamma, btype)]
        best = 1e9
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            M.assemble_laplacian(*args)
            b.record()
            torch.cuda.synchronize()
            best = min(best, 1e3 * a.elapsed_time(b))
        return best
    # 16 times the faces: the sort's log factor and the cell's loads past the first-level cache leave at most 2 x 16;
    # a search over the list for every face takes 16 x 16
    assert us(2048) < 32 * us(128)
