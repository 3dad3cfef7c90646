"""GPU: device memory that the first dycore step of a handle takes, against the
arrays it needs, and the step's bits where the edge PV lies in the theta flux's
array."""
import numpy as np
import pytest

from grist_inputs import states as S

pytestmark = pytest.mark.gpu


def _state(mesh, st, prec, torch):
    fu = torch.float64 if prec == "fp64" else torch.float32
    keys = ["u", "ps", "dpi_theta"] + (["w", "phi"] if "w" in st else [])
    return {k: torch.from_numpy(mesh.to_internal(st[k], "edge" if k == "u" else "cell")).to(
        "cuda", fu if k == "u" else torch.float64) for k in keys}


@pytest.mark.parametrize("prec,level,L,nh", [("fp64", 6, 30, True), ("fp64", 6, 30, False), ("mix", 7, 16, True),
                                             ("mix", 7, 16, False)])
def test_scratch_holds_the_arrays_of_a_step(mesh_cache, prec, level, L, nh):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import dycore_params
    assert torch.cuda.is_available()

    def first_step(m):
        mesh = G.Mesh(m)
        st = S.dycore_jet_case(m, L, nonhydrostatic=nh, bubble=nh)
        s, P = _state(mesh, st, prec, torch), dycore_params(mesh, st, L)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        (mesh.dycore_step_nh if nh else mesh.dycore_step_hydro)(s, P, 20.0, prec=prec)
        torch.cuda.synchronize()
        taken = free - torch.cuda.mem_get_info()[0]
        n = (mesh.nC, mesh.nE, mesh.nV)
        mesh.close()
        return taken, n
    first_step(mesh_cache(3))        # code and stacks of the kernels
    taken, (nC, nE, nV) = first_step(mesh_cache(level))
    s4 = 8 if prec == "fp64" else 4
    # edges: two winds, the mass flux, the theta flux; two scalars
    need = 4 * nE * L * s4 + 2 * nE * 8
    # cells: two dpi theta, theta, p, alpha, layer phi, dp/dpi, K; interfaces: M; scalars
    need += nC * L * (7 * 8 + s4) + nC * (L + 1) * 8 + 5 * nC * 8
    if nh:   # t^n pressure, dphi and 1/th of t^n (FP64: their product); two w, two phi, w**, phi**, the forcing
        need += nC * L * 8 * (2 if prec == "fp64" else 3) + 7 * nC * (L + 1) * 8
    need += nV * L * s4 + nV * 8     # vertex PV
    need += 256 * L * 16             # table of reference columns
    # 2 MB pages, rounding of each array
    assert taken <= need + (6 << 20)


@pytest.mark.parametrize("nh", [True, False])
def test_large_mixed_step_in_either_schedule(mesh_cache, nh):
    """Level 7 is above the line: one chain (profiling), the default schedule
    and the early placement give the same bits."""
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import dycore_params
    m = mesh_cache(7)
    mesh = G.Mesh(m)
    L = 6
    st = S.dycore_jet_case(m, L, nonhydrostatic=nh, bubble=nh)
    P = dycore_params(mesh, st, L)

    def run():
        s = _state(mesh, st, "mix", torch)
        for _ in range(3):
            (mesh.dycore_step_nh if nh else mesh.dycore_step_hydro)(s, P, 20.0, prec="mix")
        torch.cuda.synchronize()
        return s
    mesh.profile(True)
    ref = run()
    mesh.profile(False)
    for place in (0, 1, 2):
        mesh.set_dycore_tuning(wind_placement=place)
        got = run()
        for k in ref:
            assert torch.equal(got[k], ref[k]), (place, k)
    assert mesh.last_status() == 0
    mesh.close()
