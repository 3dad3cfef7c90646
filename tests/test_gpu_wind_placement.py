"""GPU: the non-hydrostatic step runs the wind's diagnostics on a side stream,
from the start of the stage or beside the column solve (large meshes).  Either
gives the bits of one chain (profiling on), in every policy and with both forms
of the solve: on the default stream, on a created one whose buffers are reused
behind the step, recorded in a graph, and beside a tracer step of the handle."""
import numpy as np
import pytest

from grist_inputs import states as S

pytestmark = pytest.mark.gpu
KEYS = ["u", "ps", "dpi_theta", "w", "phi"]


@pytest.mark.parametrize("prec", ["fp64", "mix", "mix_dbl_mass", "mix_df"])
@pytest.mark.parametrize("place,solve", [(1, 1), (1, 2), (2, 1), (2, 2)])
def test_either_placement_gives_the_bits_of_one_chain(mesh_cache, prec, place, solve):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import dycore_params
    assert torch.cuda.is_available()
    m = mesh_cache(5)
    mesh = G.Mesh(m)
    mesh.set_dycore_tuning(column_solve=solve, wind_placement=place)
    L, dt, steps = 20, 60.0, 4
    st = S.dycore_jet_case(m, L, nonhydrostatic=True, bubble=True)
    P = dycore_params(mesh, st, L)
    fu = torch.float64 if prec == "fp64" else torch.float32
    host = {k: torch.from_numpy(mesh.to_internal(st[k], "edge" if k == "u" else "cell")) for k in KEYS}
    q0 = torch.from_numpy(mesh.to_internal(S.tracer_mixture(m, 2, L, np.random.default_rng(1)), "cell", 1)).to("cuda", fu)

    def state():
        return {k: host[k].to("cuda", fu if k == "u" else torch.float64) for k in KEYS}

    def step(s):
        mesh.dycore_step_nh(s, P, dt, prec=prec)

    mesh.profile(True)
    ref = state()
    for _ in range(steps):
        step(ref)
    torch.cuda.synchronize()
    mesh.profile(False)

    def same(s):
        torch.cuda.synchronize()
        for k in KEYS:
            assert torch.equal(s[k], ref[k]), k
    for _ in range(3):                      # an order that is wrong need not show every time
        a = state()
        for _ in range(steps):
            step(a)
        same(a)
    stream, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        b = state()
        for _ in range(steps):
            for k in ("u", "w"):
                old, b[k] = b[k], b[k].clone()
                del old
            step(b)
            for k in ("u", "w"):
                old, b[k] = b[k], b[k].clone()
                del old                     # the next allocation overwrites it behind the step
                torch.full_like(b[k], float("nan"))
    same(b)
    with torch.cuda.stream(stream):
        c = state()
        step(c)
        for k in KEYS:
            c[k].copy_(host[k])
    g = G.capture(lambda: step(c), stream)
    for _ in range(steps):
        g.launch()
    same(c)
    mb = {"q": q0, "dpi": torch.full((mesh.nC, L), 1e3, dtype=torch.float64, device="cuda"),
          "mass_flux": torch.zeros((mesh.nE, L), dtype=torch.float64, device="cuda"), "n_levels": L}
    e = state()
    torch.cuda.synchronize()
    for _ in range(steps):
        with torch.cuda.stream(stream):
            step(e)
        with torch.cuda.stream(other):
            mesh.tracer_step([mb], dt, prec=prec)
    same(e)
    assert mesh.last_status() == 0
    g.close()
    mesh.close()


def test_only_the_placements_there_are(mesh_cache):
    import paper_2404_08849_gb300 as G
    mesh = G.Mesh(mesh_cache(2))
    for bad in (-1, 3):
        with pytest.raises(G.GristError):
            mesh.set_dycore_tuning(wind_placement=bad)
    assert mesh.dycore_tuning() == {"column_solve": 0, "wind_placement": 0}
    mesh.close()
