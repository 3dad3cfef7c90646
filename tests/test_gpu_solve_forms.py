"""GPU: the column solve has a one-warp and a block form, picked by the numbers
of columns and levels, and the FP64 policy short forms of its series: both
forms on either side of every line of the rule, against the oracle."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level,L", [(3, 2), (3, 3), (3, 31), (3, 70), (3, 71), (3, 128), (5, 33), (5, 71), (6, 71)])
@pytest.mark.parametrize("pad", [0, 3])
def test_fp64_step_against_the_oracle(mesh_cache, level, L, pad):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import oracle_params, run_dycore, spun_up_nh
    assert torch.cuda.is_available()
    if pad and level > 3:
        pytest.skip("padding is independent of the mesh size")
    m = mesh_cache(level)
    mesh = G.Mesh(m)
    dt = 60.0
    st = spun_up_nh(m, L, steps=1, dt=dt)
    ref = O.dycore_step_nh(O.Mesh(m), oracle_params(st, L), st, dt)
    got = run_dycore(mesh, st, L, dt, nh=True, ld=L + pad, ld_int=L + 1 + pad)
    # the parity bounds of the other FP64 tests; w on the scale of its terms
    for k in ("u", "ps", "dpi_theta", "phi"):
        assert O.max_rel_diff(got[k], ref[k]) <= 1e-12, k
    assert float(np.max(np.abs(got["w"] - ref["w"]))) <= 1e-12 * 0.55 * dt * 9.80616
    mesh.close()
