"""GPU: the dycore's kernels take vectors of 4 or 2 levels where rows are whole,
aligned vectors, else single levels.  A padded row or a shifted buffer changes
the widths and nothing else: every field must come out bit for bit the same."""
import numpy as np
import pytest

from grist_inputs import states as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mix", "mix_dbl_mass", "mix_df"])
@pytest.mark.parametrize("nh", [False, True])
@pytest.mark.parametrize("L", [4, 6, 7, 60])
def test_same_bits_at_every_width(mesh_cache, prec, nh, L):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import spun_up_nh, to_dev
    assert torch.cuda.is_available()
    m = mesh_cache(3)
    mesh = G.Mesh(m)
    st = spun_up_nh(m, L, steps=1) if nh else S.dycore_jet_case(m, L)
    phis = to_dev(mesh, st["phi_s"], "cell", 0, torch.float64)
    fu = torch.float64 if prec == "fp64" else torch.float32

    def run(pad, shift):
        def place(a, kind, n, dtype=torch.float64):
            b = mesh.to_internal(a, kind, 0)
            rows = np.full((b.shape[0], n), np.nan)
            rows[:, :b.shape[1]] = b
            flat = torch.full((rows.size + shift,), float("nan"), dtype=dtype, device="cuda")
            flat[shift:] = torch.from_numpy(rows.ravel()).to("cuda", dtype)
            return flat[shift:].view(rows.shape)
        s = {"u": place(st["u"], "edge", L + pad, fu), "ps": to_dev(mesh, st["ps"], "cell", 0, torch.float64),
             "dpi_theta": place(st["dpi_theta"], "cell", L + pad)}
        if nh:
            s.update(w=place(st["w"], "cell", L + 1 + pad), phi=place(st["phi"], "cell", L + 1 + pad),
                     p_nh=place(np.zeros((m["n_cells"], L)), "cell", L + pad), p_nh_valid=False)
        P = G.DycoreParams(L, st["b_int"], st["pi_top"], phis, ld=L + pad, ld_int=L + 1 + pad)
        for _ in range(2):
            (mesh.dycore_step_nh if nh else mesh.dycore_step_hydro)(s, P, 60.0, prec=prec)
        torch.cuda.synchronize()
        out = {"u": s["u"][:, :L], "ps": s["ps"], "dpi_theta": s["dpi_theta"][:, :L]}
        if nh:
            out.update(w=s["w"][:, :L + 1], phi=s["phi"][:, :L + 1], p_nh=s["p_nh"][:, :L])
        return {k: v.clone() for k, v in out.items()}
    ref = run(0, 0)
    assert all(bool(torch.isfinite(v).all()) for v in ref.values())
    for pad, shift in ((1, 0), (2, 0), (4, 0), (0, 1), (0, 2)):
        got = run(pad, shift)
        for k in ref:
            assert torch.equal(ref[k], got[k]), (k, pad, shift)
    assert mesh.last_status() == 0
    mesh.close()


@pytest.mark.parametrize("prec", ["fp64", "mix"])
@pytest.mark.parametrize("L,pad", [(1, 0), (4, 0), (6, 0), (7, 1), (8, 1), (60, 0)])
def test_vorticity_at_every_width(mesh_cache, prec, L, pad):
    """Against numpy: 3 products and 2 sums of FP64, so a few ulp of the terms."""
    import torch
    import paper_2404_08849_gb300 as G
    m = mesh_cache(3)
    mesh = G.Mesh(m)
    rng = np.random.default_rng(L)
    u = rng.standard_normal((m["n_edges"], L)) * 10.0
    u = u if prec == "fp64" else u.astype(np.float32)
    rows = np.full((m["n_edges"], L + pad), np.nan, u.dtype)
    rows[:, :L] = mesh.to_internal(u, "edge", 0)
    vor = mesh.vorticity(torch.from_numpy(rows).cuda(), L)
    torch.cuda.synchronize()
    got = mesh.from_internal(vor.cpu().numpy()[:, :L], "vertex", 0)
    ev = m["edges_on_vertex"]
    w = m["edge_sign_on_vertex"] * m["edge_dc"][ev] / m["vertex_area"][:, None]
    terms = w[:, :, None] * u[ev].astype(np.float64)
    assert np.all(np.abs(got - terms.sum(1)) <= 8 * np.finfo(float).eps * np.abs(terms).sum(1))
    mesh.close()
