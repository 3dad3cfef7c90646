"""GPU: the hydrostatic diagnostics take the equation of state from a table of
reference columns over two octaves of the column mass and from pow() outside
it; both, the table's ends and the bins' edges against the oracle."""
import numpy as np
import pytest

import oracle as O
from grist_inputs import states as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pi_top", [0.0, 225.0, 20000.0])
@pytest.mark.parametrize("L", [2, 33])
def test_columns_inside_and_outside_the_table(mesh_cache, pi_top, L):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import oracle_params, run_dycore
    assert torch.cuda.is_available()
    m = mesh_cache(3)
    rng = np.random.default_rng(17)
    nC = m["n_cells"]
    st = S.dycore_jet_case(m, L)
    # column masses from a quarter of the table's lower end to twice its upper
    # end, bin edges (multiples of 2^-7 of a power of two) and their
    # neighbours among them
    mass = 2.0 ** rng.uniform(13.0, 18.0, nC)
    edge = np.ldexp(1.0 + np.arange(128) / 128.0, 15)
    special = np.concatenate([edge, np.nextafter(edge, 0), 2 * edge, [2.0 ** 17, np.nextafter(2.0 ** 17, 0)]])
    mass[:special.size] = special
    theta = rng.uniform(250.0, 400.0, (nC, L))
    st["b_int"], st["pi_top"] = S.sigma_uniform(L), pi_top
    st["ps"] = pi_top + mass
    st["dpi_theta"] = mass[:, None] * np.diff(st["b_int"])[None, :] * theta
    st["u"] = st["u"][:, :L]
    mesh = G.Mesh(m)
    ref = O.dycore_step_hydro(O.Mesh(m), oracle_params(st, L), st, 1.0)
    got = run_dycore(mesh, st, L, 1.0, nh=False)
    # one FP64 step: the parity bound of the other FP64 tests
    for k in ("u", "ps", "dpi_theta"):
        assert O.max_rel_diff(got[k], ref[k]) <= 1e-12, k
    mesh.close()
