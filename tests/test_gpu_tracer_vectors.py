"""GPU: a tracer work item is a vector of 4 or 2 levels where the member's rows
and pointers allow one, else single levels; every width against the
one-level form, for level counts and row lengths around the widths,
misaligned buffers, a group with fewer tracers than a thread takes, and
members of different widths in one batch."""
import numpy as np
import pytest

from grist_inputs import states as S

pytestmark = pytest.mark.gpu


def _member(torch, mesh, m, rng, T, L, ld, shift, dt_q, vertical):
    """One member; shift moves every buffer off its allocation by that many
    elements."""
    def place(a, kind, axis, dtype, n):
        b = mesh.to_internal(a, kind, axis)
        pad = np.full(b.shape[:-1] + (n,), np.nan)
        pad[..., :b.shape[-1]] = b
        flat = torch.full((pad.size + shift,), float("nan"), dtype=dtype, device="cuda")
        flat[shift:] = torch.from_numpy(pad.ravel()).to("cuda", dtype)
        return flat[shift:].view(pad.shape)
    F = rng.standard_normal((m["n_edges"], L)) * 2e4
    out = {"q": place(S.tracer_mixture(m, T, L, rng), "cell", 1, dt_q, ld),
           "dpi": place(3000.0 + rng.uniform(0, 200, (m["n_cells"], L)), "cell", 0, torch.float64, ld),
           "mass_flux": place(F, "edge", 0, torch.float64, ld), "n_levels": L}
    if vertical:
        M = rng.uniform(-0.5, 0.5, (m["n_cells"], L + 1))
        M[:, 0] = M[:, L] = 0.0
        out["vmass_flux"] = place(M, "cell", 0, torch.float64, ld + 1)
    return out


@pytest.mark.parametrize("prec", ["mix", "fp64"])
@pytest.mark.parametrize("limiter,beta,ring", [(True, 1.0, True), (False, 1.0, True), (True, 1.0, False),
                                                (True, 0.5, True)])
@pytest.mark.parametrize("shapes", [[(1, 4, 4, 0)], [(5, 6, 6, 0)], [(4, 8, 10, 0)], [(3, 7, 8, 0)], [(2, 12, 12, 1)],
                                    [(2, 12, 12, 2)], [(1, 60, 60, 0), (4, 30, 30, 0), (6, 9, 9, 0), (3, 16, 17, 0)]])
def test_every_width_equals_single_levels(mesh_cache, prec, limiter, beta, ring, shapes):
    import torch
    import paper_2404_08849_gb300 as G
    assert torch.cuda.is_available()
    m = mesh_cache(3)
    mesh = G.Mesh(m)
    dt_q = torch.float64 if prec == "fp64" else torch.float32
    got = []
    for lpt in (1, 2):
        rng = np.random.default_rng(8)
        mb = [_member(torch, mesh, m, rng, T, L, ld, shift, dt_q, L == 60) for T, L, ld, shift in shapes]
        mesh.set_tracer_tuning(block=128, tracers_per_thread=4, levels_per_thread=lpt, cell_edges=ring)
        mesh.tracer_step(mb, 100.0, prec=prec, limiter=limiter, beta=beta)
        torch.cuda.synchronize()
        got.append([x["q"][..., :x["n_levels"]].double() for x in mb])
        for x in mb:   # the rows' padding is never written
            assert bool(torch.isnan(x["q"][..., x["n_levels"]:]).all())
    assert mesh.last_status() == 0
    # the same operations on the same operands; a compiler may contract a
    # product and a sum differently: a few roundings of the type
    tol = 1e-13 if prec == "fp64" else 1e-6
    for a, b in zip(*got):
        assert float((a - b).abs().max()) <= tol * float(a.abs().max())
    mesh.close()


@pytest.mark.parametrize("prec", ["mix", "fp64"])
@pytest.mark.parametrize("L,ld", [(2, 2), (31, 31), (32, 32), (33, 33), (60, 60), (60, 61), (64, 64), (65, 66), (96, 96),
                                  (97, 97), (128, 128), (127, 128)])
@pytest.mark.parametrize("cmax,courant", [(0.0, 6.0), (0.5, 6.0), (float("inf"), 0.4)])
def test_vertical_layouts_against_the_oracle(mesh_cache, prec, L, ld, cmax, courant):
    """Lanes hold 1 to 4 consecutive levels, as vectors or one by one; more
    tracers than one group of loads.  Column fluxes, and so the bounds, of the
    other vertical tests (no layer loses more than about half its mass)."""
    import oracle as O
    import torch
    import paper_2404_08849_gb300 as G
    from test_gpu_vertical import _column_flux, _member as vertical_member
    m = mesh_cache(3)
    mesh = G.Mesh(m)
    rng = np.random.default_rng(L)
    T, dt = 5, 400.0
    dpi = rng.uniform(600, 1200, (m["n_cells"], L))
    M = _column_flux(rng, m["n_cells"], L, dt, 600.0, courant)
    M[::3] = 0.0
    q = rng.uniform(0.1, 1.0, (T, m["n_cells"], L))
    mb = vertical_member(mesh, q, dpi, np.zeros((m["n_edges"], L)), M, prec, ld, ld + 1)
    mesh.tracer_step([mb], dt, prec=prec, vertical_courant_max=cmax)
    torch.cuda.synchronize()
    ref = O.tracer_vertical_step(q, dpi, M, dt, cmax)
    got = mesh.from_internal(mb["q"].double().cpu().numpy()[..., :L], "cell", 1)
    assert O.max_rel_diff(got, ref) <= (1e-12 if prec == "fp64" else 2e-5)
    assert mesh.last_status() == 0
    mesh.close()
