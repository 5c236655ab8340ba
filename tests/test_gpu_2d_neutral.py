"""Level-0 fields of a 2D gap without net charge, its electrode charged.

With co-located pairs every transverse mode is exactly zero: E_x must be the
mean's field on every row, to the last bit the same along y, and E_y zero.
"""
import numpy as np
import pytest

from paper_2603_24010_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nx,Ny", [(2, 8), (33, 32), (9, 1024), (4, 4096), (2049, 8)])
def test_neutral_level0_fields(Nx, Ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import gap2d
    from paper_2603_24010_gb300 import native
    cfg = W.scaled(W.gap_2d(0, Nx=Nx, Ny=Ny, n_pairs=3000, steps=10, beam_per_step=0), sigma0=1e-6)
    xi, eta, ue, we, ui, wi = (np.asarray(v, np.float32).astype(np.float64) for v in W.load_pairs_2d(cfg))
    xi = np.minimum(xi, np.nextafter(np.float32(Nx), np.float32(0)))
    eta = np.where(eta >= Ny, 0.0, eta)
    g = native.Gap2D(cfg, max_steps=1)
    o = gap2d.Oracle2D(cfg)
    for s, u, w in ((0, ue, we), (1, ui, wi)):
        g.set_particles(s, xi, eta, u, w)
        o.set_particles(s, xi, eta, u, w)
    g.step(native.WEAK, 0)
    assert o.step(1, 0) == 0
    f = g.fields()
    g.close()
    E = cfg["sigma0"] / cfg["eps0"]
    assert not np.any(f["G"]) and not np.any(f["Ey"])
    assert np.all(f["Ex"] == f["Ex"][:, :1]) and np.all(f["phi"] == f["phi"][:, :1])
    # FP32 rounding of the FP64 field (2^-24) and the rounding of a few FP64 operations
    np.testing.assert_allclose(f["Ex"], np.full((Nx, Ny), E), rtol=6.1e-8)
    np.testing.assert_allclose(f["Ex"], o.Ex, rtol=1.3e-7)
    np.testing.assert_allclose(f["phi"], o.phi, rtol=0, atol=1e-12 * E * cfg["d"])
