"""GPU: a dycore step runs parts of its stages on side streams of the handle.
With the kernels timed one by one (profiling) they run in one chain, so the two
must give the same bits: on the default stream, on a created one whose buffers
are freed and reused behind the step, recorded in a graph, and beside a tracer
step of the same handle on another stream."""
import numpy as np
import pytest

from grist_inputs import states as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mix"])
@pytest.mark.parametrize("nh", [False, True])
def test_side_streams_give_the_bits_of_one_chain(mesh_cache, prec, nh):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import dycore_params
    assert torch.cuda.is_available()
    m = mesh_cache(4)
    mesh = G.Mesh(m)
    L, dt, steps = 12, 60.0, 4
    st = S.dycore_jet_case(m, L, nonhydrostatic=nh, bubble=nh)
    P = dycore_params(mesh, st, L)
    fu = torch.float64 if prec == "fp64" else torch.float32
    keys = ["u", "ps", "dpi_theta"] + (["w", "phi"] if nh else [])
    host = {k: torch.from_numpy(mesh.to_internal(st[k], "edge" if k == "u" else "cell")) for k in keys}
    q0 = torch.from_numpy(mesh.to_internal(S.tracer_mixture(m, 2, L, np.random.default_rng(1)), "cell", 1)).to("cuda", fu)

    def state():
        return {k: host[k].to("cuda", fu if k == "u" else torch.float64) for k in keys}

    def step(s):
        (mesh.dycore_step_nh if nh else mesh.dycore_step_hydro)(s, P, dt, prec=prec)

    mesh.profile(True)
    ref = state()
    for _ in range(steps):
        step(ref)
    torch.cuda.synchronize()
    mesh.profile(False)

    def same(s):
        torch.cuda.synchronize()
        for k in keys:
            assert torch.equal(s[k], ref[k]), k
    a = state()
    for _ in range(steps):
        step(a)
    same(a)
    stream, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        b = state()
        for _ in range(steps):
            u = b["u"]
            b["u"] = u.clone()            # the old buffer goes back to the allocator ...
            del u
            step(b)
            b["u"], old = b["u"].clone(), b["u"]
            del old                       # ... and the next allocations overwrite them behind the step
            torch.full_like(b["u"], float("nan"))
    same(b)
    with torch.cuda.stream(stream):
        c = state()
        step(c)
        for k in keys:
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
    g.close()
    mesh.close()
