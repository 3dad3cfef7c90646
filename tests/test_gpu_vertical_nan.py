"""GPU: a NaN in one level of the vertical transport reaches no level that does
not read it.  Without motion a level's upper interface takes the level itself and
its lower one the level below, so that only the level and the one above it may
become NaN; column lengths that fill the warp's 32 lanes among them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mix"])
@pytest.mark.parametrize("L", [5, 31, 32, 33, 64, 70, 96, 128])
def test_nan_stays_where_it_is_read(mesh_cache, prec, L):
    import torch
    import paper_2404_08849_gb300 as G
    assert torch.cuda.is_available()
    mesh = G.Mesh(mesh_cache(2))
    fq = torch.float64 if prec == "fp64" else torch.float32
    rng = np.random.default_rng(L)
    q0 = torch.from_numpy(rng.uniform(0.5, 1.5, (2, mesh.nC, L))).to("cuda", fq)
    dpi = torch.from_numpy(rng.uniform(900.0, 1100.0, (mesh.nC, L))).cuda()

    def step(q):
        mesh.tracer_step([{"q": q, "dpi": dpi, "mass_flux": torch.zeros((mesh.nE, L), dtype=torch.float64, device="cuda"),
                           "vmass_flux": torch.zeros((mesh.nC, L + 1), dtype=torch.float64, device="cuda"),
                           "n_levels": L}], 60.0, prec=prec)
        torch.cuda.synchronize()
        return q
    clean = step(q0.clone())
    assert mesh.last_status() == 0
    K = (L + 31) // 32
    # the first level of the last lane, the last level, and some in between
    for n in sorted({0, L // 2, min(31 * K, L - 1), L - 1}):
        q = q0.clone()
        q[:, :, n] = float("nan")
        step(q)
        assert mesh.last_status() & G.GRIST_FLAG_NONFINITE
        keep = [k for k in range(L) if k not in (n, n - 1)]
        assert torch.equal(q[:, :, keep], clean[:, :, keep]), n
        assert bool(torch.isnan(q[:, :, n]).all())
    mesh.close()
