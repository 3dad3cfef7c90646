"""GPU: the FP64 limiter compares, bounds and signs in integer arithmetic.
Against the oracle for values at the ends of the format's range, and a
NaN must stay where it was: outside the reach of one step the result is the
one without it."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def _case(m, L, scale, sign, rng):
    q = rng.uniform(0.0, 1.0, (1, m["n_cells"], L))
    q[rng.uniform(size=q.shape) < 0.3] = 0.0          # plateaus: no allowed change, no antidiffusion
    q[rng.uniform(size=q.shape) < 0.1] = -0.0
    if sign:
        q *= np.where(rng.uniform(size=q.shape) < 0.5, -1.0, 1.0)
    F = rng.standard_normal((m["n_edges"], L)) * 2e4
    F[rng.uniform(size=F.shape) < 0.05] = 0.0
    F[rng.uniform(size=F.shape) < 0.05] = -0.0
    return q * scale, 3000.0 + rng.uniform(0, 200, (m["n_cells"], L)), F


@pytest.mark.parametrize("L", [3, 8])
@pytest.mark.parametrize("scale", [1.0, 1e-300, 1e150])
@pytest.mark.parametrize("sign", [False, True])
@pytest.mark.parametrize("ring", [True, False])
def test_values_against_oracle(mesh_cache, L, scale, sign, ring):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import run_tracer
    assert torch.cuda.is_available()
    m = mesh_cache(3)
    mesh = G.Mesh(m)
    mesh.set_tracer_tuning(cell_edges=ring)
    q, dpi, F = _case(m, L, scale, sign, np.random.default_rng(31))
    ref = O.tracer_step(O.Mesh(m), q, dpi, F, 300.0)
    got = run_tracer(mesh, m, q, dpi, F, 300.0)
    assert O.max_rel_diff(got, ref) <= 1e-12
    mesh.close()


@pytest.mark.parametrize("bad", [float("nan"), -float("nan")])
def test_nan_reaches_no_further_than_the_stencils(mesh_cache, bad):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import run_tracer
    m = mesh_cache(3)
    mesh = G.Mesh(m)
    q, dpi, F = _case(m, 4, 1.0, True, np.random.default_rng(32))
    clean = run_tracer(mesh, m, q, dpi, F, 300.0)
    assert mesh.last_status() == 0
    p = q.copy()
    p[0, 40, 1] = bad
    got = run_tracer(mesh, m, p, dpi, F, 300.0)
    assert mesh.last_status() & G.GRIST_FLAG_NONFINITE
    # three stages of two rings each and the limiter's two
    reach = {40}
    for _ in range(8):
        reach |= {int(c) for i in reach for c in m["cells_on_cell"][i] if c >= 0}
    far = np.array(sorted(set(range(m["n_cells"])) - reach))
    assert far.size > 0
    assert np.array_equal(got[0, far], clean[0, far])
    # the other levels are untouched, and next to the NaN nothing but NaN and numbers
    assert np.array_equal(got[0][:, [0, 2, 3]], clean[0][:, [0, 2, 3]])
    assert np.isnan(got[0, 40, 1])
    mesh.close()
