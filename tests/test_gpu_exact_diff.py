"""GPU: the mixed and FP64 momentum equations against the oracle where the
integer subtraction leaves its fast case: cells whose p, phi and K differ by
more than a factor of two, equal values, zero winds, and level counts of every
vector width of the edge PV pass."""
import numpy as np
import pytest

import oracle as O
from grist_inputs import states as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mix", "mix_dbl_mass", "mix_df"])
@pytest.mark.parametrize("L,ld", [(4, 4), (6, 6), (6, 7), (7, 8)])
@pytest.mark.parametrize("case", ["jet", "calm", "ridges"])
def test_momentum_against_the_oracle(mesh_cache, prec, L, ld, case):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import oracle_params, run_dycore
    assert torch.cuda.is_available()
    m = mesh_cache(3)
    rng = np.random.default_rng(5)
    st = S.dycore_jet_case(m, L)
    if case == "calm":        # zeros and single cells of wind: K from 0, exact zeros of u
        st["u"] = np.where(rng.uniform(size=st["u"].shape) < 0.2, st["u"], 0.0)
    if case == "ridges":      # surface geopotential and pressure that jump between cells
        st["phi_s"] = 10.0 ** rng.uniform(0.0, 4.5, m["n_cells"])
        st["ps"] = st["ps"] * rng.uniform(0.4, 1.0, m["n_cells"])
        dpi = np.diff(st["b_int"])[None, :] * (st["ps"][:, None] - st["pi_top"])
        st["dpi_theta"] = dpi * st["theta"]
    mesh = G.Mesh(m)
    # a short step: one stage's tendencies, not their growth
    ref = O.dycore_step_hydro(O.Mesh(m), oracle_params(st, L), st, 0.5)
    got = run_dycore(mesh, st, L, 0.5, nh=False, prec=prec, ld=ld)
    # the parity bounds of the other one-step tests: 1e-12, binary32 u 2e-5
    assert O.max_rel_diff(got["u"], ref["u"]) <= (1e-12 if prec == "fp64" else 2e-5)
    mesh.close()
