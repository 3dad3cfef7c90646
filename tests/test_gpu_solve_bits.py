"""GPU: the one-warp and the block form of the column solve do the same
arithmetic: every field and the pressure come out bit for bit the same, whatever
the precision, the number of levels, the rows' padding and the columns left over
of 32; and the one-warp form alone, which only large meshes take by themselves,
against the oracle."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu
WARP, BLOCK = 1, 2


@pytest.mark.parametrize("prec", ["fp64", "mix", "mix_dbl_mass", "mix_df"])
@pytest.mark.parametrize("L", [2, 3, 4, 7, 31, 60, 71, 128])
@pytest.mark.parametrize("pad", [0, 3])
def test_both_forms_give_the_same_bits(mesh_cache, prec, L, pad):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import dycore_params, spun_up_nh, to_dev
    assert torch.cuda.is_available()
    m = mesh_cache(3)
    mesh = G.Mesh(m)
    dt = 60.0
    st = spun_up_nh(m, L, steps=1, dt=dt)
    P = dycore_params(mesh, st, L, ld=L + pad, ld_int=L + 1 + pad)
    fu = torch.float64 if prec == "fp64" else torch.float32

    def run(form):
        mesh.set_dycore_tuning(column_solve=form)
        assert mesh.dycore_tuning()["column_solve"] == form
        s = {"u": to_dev(mesh, st["u"], "edge", 0, fu, L + pad), "ps": to_dev(mesh, st["ps"], "cell", 0, torch.float64),
             "dpi_theta": to_dev(mesh, st["dpi_theta"], "cell", 0, torch.float64, L + pad),
             "w": to_dev(mesh, st["w"], "cell", 0, torch.float64, L + 1 + pad),
             "phi": to_dev(mesh, st["phi"], "cell", 0, torch.float64, L + 1 + pad),
             "p_nh": torch.zeros((mesh.nC, L + pad), dtype=torch.float64, device="cuda"), "p_nh_valid": False}
        for _ in range(3):
            mesh.dycore_step_nh(s, P, dt, prec=prec)
        torch.cuda.synchronize()
        assert mesh.last_status() == 0
        cut = {"u": L, "dpi_theta": L, "w": L + 1, "phi": L + 1, "p_nh": L}
        return {k: s[k][:, :n].clone() for k, n in cut.items()} | {"ps": s["ps"].clone()}
    a, b = run(WARP), run(BLOCK)
    for k in a:
        assert torch.equal(a[k], b[k]), k
    mesh.close()


@pytest.mark.parametrize("rows", [{"eos"}, {"nh_adv", "wind"}])
def test_both_forms_of_the_emulating_variant(mesh_cache, rows):
    import torch
    import paper_2404_08849_gb300 as G
    from gpu_cases import spun_up_nh, to_dev
    m = mesh_cache(3)
    mesh = G.Mesh(m)
    L, dt = 12, 60.0
    st = spun_up_nh(m, L, steps=1, dt=dt)
    phis = to_dev(mesh, st["phi_s"], "cell", 0, torch.float64)
    P = G.DycoreParams(L, st["b_int"], st["pi_top"], phis, emulate_fp32_rows=sum(G.GRIST_ROWS[r] for r in rows))
    out = []
    for form in (WARP, BLOCK):
        mesh.set_dycore_tuning(column_solve=form)
        s = {k: to_dev(mesh, st[k], "edge" if k == "u" else "cell", 0, torch.float64)
             for k in ("u", "ps", "dpi_theta", "w", "phi")}
        for _ in range(2):
            mesh.dycore_step_nh(s, P, dt)
        out.append(s)
    torch.cuda.synchronize()
    for k in out[0]:
        assert torch.equal(out[0][k], out[1][k]), k
    mesh.close()


@pytest.mark.parametrize("L", [2, 5, 30, 60, 128])
@pytest.mark.parametrize("pad", [0, 3])
def test_one_warp_form_against_the_oracle(mesh_cache, L, pad):
    import paper_2404_08849_gb300 as G
    from gpu_cases import oracle_params, run_dycore, spun_up_nh
    m = mesh_cache(3)
    mesh = G.Mesh(m)
    mesh.set_dycore_tuning(column_solve=WARP)
    dt = 60.0
    st = spun_up_nh(m, L, steps=1, dt=dt)
    ref = O.dycore_step_nh(O.Mesh(m), oracle_params(st, L), st, dt)
    got = run_dycore(mesh, st, L, dt, nh=True, ld=L + pad, ld_int=L + 1 + pad)
    # the parity bounds of the other FP64 tests; w on the scale of its terms
    for k in ("u", "ps", "dpi_theta", "phi"):
        assert O.max_rel_diff(got[k], ref[k]) <= 1e-12, k
    assert float(np.max(np.abs(got["w"] - ref["w"]))) <= 1e-12 * 0.55 * dt * 9.80616
    mesh.close()


def test_only_the_forms_there_are(mesh_cache):
    import paper_2404_08849_gb300 as G
    mesh = G.Mesh(mesh_cache(2))
    assert mesh.dycore_tuning()["column_solve"] == 0
    for bad in (-1, 3):
        with pytest.raises(G.GristError):
            mesh.set_dycore_tuning(column_solve=bad)
    assert mesh.dycore_tuning()["column_solve"] == 0
    mesh.close()
