"""GPU: the hydrostatic equation of state seen through the pressure gradient.
From rest, the wind of one short step is the pressure gradient times the time
step, so that a relative error of alpha or phi shows in u at its own size."""
import numpy as np
import pytest

import oracle as O
from grist_inputs import states as S

pytestmark = pytest.mark.gpu


def _case(m, L, pi_top):
    """Columns over the table's two octaves and beyond both ends, the bins'
    edges and their neighbours among them."""
    rng = np.random.default_rng(23)
    nC = m["n_cells"]
    st = S.dycore_jet_case(m, L)
    mass = 2.0 ** rng.uniform(14.5, 17.5, nC)
    edge = np.ldexp(1.0 + np.arange(128) / 128.0, 15)
    special = np.concatenate([edge, np.nextafter(edge, 0), 2 * edge, [2.0 ** 17, np.nextafter(2.0 ** 17, 0)]])
    mass[rng.permutation(nC)[:special.size]] = special
    st["b_int"], st["pi_top"] = S.sigma_uniform(L), pi_top
    st["ps"] = pi_top + mass
    st["dpi_theta"] = mass[:, None] * np.diff(st["b_int"])[None, :] * rng.uniform(250.0, 400.0, (nC, L))
    st["u"] = np.zeros((m["n_edges"], L))
    return st


@pytest.mark.parametrize("pi_top", [0.0, 225.0, 20000.0])
@pytest.mark.parametrize("L", [2, 33, 60])
def test_wind_from_rest(mesh_cache, pi_top, L):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import oracle_params, run_dycore
    assert torch.cuda.is_available()
    m = mesh_cache(3)
    st = _case(m, L, pi_top)
    M = O.Mesh(m)
    ref = O.dycore_step_hydro(M, oracle_params(st, L), st, 1.0)
    # alpha larger by 1e-12 (Rd and cp together: the same kappa) is well outside the bound
    P = oracle_params(st, L)
    off = O.Params(L, st["b_int"], st["pi_top"], st["phi_s"], rd=287.04 * (1 + 1e-12), cp=1004.64 * (1 + 1e-12),
                   beta=0.55)
    assert O.max_rel_diff(O.dycore_step_hydro(M, off, st, 1.0)["u"], ref["u"]) > 5e-13
    mesh = G.Mesh(m)
    got = run_dycore(mesh, st, L, 1.0, nh=False)
    # phi reaches 4e5 in up to 60 additions, and the oracle's layers carry the
    # cancellation in p_(k+1/2) - p_(k-1/2), up to 130 units of 2^-53: with both
    # cells of an edge 4e5 (60 + 130) 2^-53 2 = 1.7e-8 against the largest
    # difference of phi, 1.7e5: 1e-13, and as much again for the later stages
    assert O.max_rel_diff(got["u"], ref["u"]) <= 2e-13
    mesh.close()
