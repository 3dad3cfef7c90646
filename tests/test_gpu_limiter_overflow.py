"""GPU: the binary32 limiter where the sums of the antidiffusive fluxes pass the
binary32 range (P = +infinity): a cell without room, Q = 0, must let nothing
in.  A step profile of height M in a solid-body flow, the time step and the
layer mass chosen so that P overflows and q, F q and the tendencies do not:
where a cell and its neighbours are at M (or 0) it has no room above (below).
(Where Q overflows too, their ratio is not a number and counts as 1.)"""
import numpy as np
import pytest

from grist_inputs import states as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 2, 4])
@pytest.mark.parametrize("ring", [True, False])
@pytest.mark.parametrize("M", [1.0, 2e37])
def test_overflowing_sums_let_nothing_through(mesh_cache, L, ring, M):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import run_tracer
    assert torch.cuda.is_available()
    m = mesh_cache(3)
    mesh = G.Mesh(m)
    mesh.set_tracer_tuning(cell_edges=ring)
    dt, dpi = 1e9, 25000.0
    # Courant number 0.2 over the mesh spacing; a layer-mass flux of at most 5
    spacing = float(np.mean(m["edge_dc"]))
    un = S.normal_wind_from_psi(m, S.solid_body_psi(m, 1.0))
    F = un / np.abs(un).max() * (0.2 * dpi * spacing / dt)
    assert np.abs(F).max() <= 8.0
    q = np.where(m["cell_xyz"][:, 0] > 0, M, 0.0)
    q = np.repeat(q[None, :, None], L, 2)
    got = run_tracer(mesh, m, q, np.full((m["n_cells"], L), dpi), np.repeat(F[:, None], L, 1), dt, prec="mix")
    assert mesh.last_status() == 0
    # a dozen binary32 roundings of numbers up to M
    tol = 12 * 2.0 ** -23
    near = np.where(m["cells_on_cell"] >= 0, m["cells_on_cell"], np.arange(m["n_cells"])[:, None])
    ring = np.concatenate([q[0, :, 0][near], q[0, :, :1]], axis=1)
    full, empty = (ring == M).all(1), (ring == 0).all(1)
    assert full.sum() > 200 and empty.sum() > 200
    assert got[0, full].max() <= M * (1 + tol) and got[0, empty].min() >= -M * tol
    assert got.std() > 0.3 * M
    mesh.close()
