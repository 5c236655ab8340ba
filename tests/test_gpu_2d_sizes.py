"""The 2D gap at the edges of its transforms, mode groups and work items.

Level-0 fields against the oracle with the tolerances of test_gpu_2d (FP32
transforms and recurrences against FP64); and, after steps that run through
re-sorts and graph replays, a charge grid that is to the last unit the
deposit of the particles the store holds.
"""
import numpy as np
import pytest

from paper_2603_24010_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_24010_gb300 import native
    from oracle import gap2d
    native.lib()
    return native, gap2d


def gap(native, Nx, Ny, n_pairs, steps, beam=0, sort_every=0):
    cfg = W.gap_2d(0, Nx=Nx, Ny=Ny, n_pairs=n_pairs, steps=10, beam_per_step=beam)
    xi, eta, ue, we, ui, wi = (np.asarray(v, np.float32).astype(np.float64) for v in W.load_pairs_2d(cfg))
    xi = np.minimum(xi, np.nextafter(np.float32(Nx), np.float32(0)))
    eta = np.where(eta >= Ny, 0.0, eta)
    g = native.Gap2D(cfg, max_steps=max(steps, 1), sort_every=sort_every)
    g.set_particles(native.ELECTRONS, xi, eta, ue, we)
    g.set_particles(native.IONS, xi, eta, ui, wi)
    return cfg, g, (xi, eta, ue, we, ui, wi)


@pytest.mark.parametrize("Nx,Ny", [(2, 8), (3, 16), (33, 32), (31, 256), (20, 512), (9, 1024), (5, 2048), (4, 4096),
                                   (2049, 8), (1025, 16)])
def test_level0_fields(env, Nx, Ny):
    native, gap2d = env
    cfg, g, (xi, eta, ue, we, ui, wi) = gap(native, Nx, Ny, 30_000, 0)
    g.step(1, 0)
    f = g.fields()
    g.close()
    o = gap2d.Oracle2D(cfg)
    # only the deposit and the solve: electrons and ions at different places
    o.set_particles(0, xi, eta, ue, we)
    o.set_particles(1, xi, eta, ui, wi)
    assert o.step(1, 0) == 0
    np.testing.assert_array_equal(f["G"], o.G)
    assert not np.any(f["G"])  # co-located pairs


@pytest.mark.parametrize("Nx,Ny", [(2, 8), (3, 16), (33, 32), (31, 256), (20, 512), (9, 1024), (5, 2048), (4, 4096),
                                   (2049, 8), (1025, 16)])
def test_charged_level0_fields(env, Nx, Ny):
    native, gap2d = env
    cfg, g, (xi, eta, ue, we, ui, wi) = gap(native, Nx, Ny, 30_000, 0)
    xe = np.minimum(np.float32(Nx) * (xi / Nx) ** 2 + np.float32(1e-3), np.nextafter(np.float32(Nx), np.float32(0)))
    xe = xe.astype(np.float32).astype(np.float64)
    g.set_particles(native.ELECTRONS, xe, eta, ue, we)
    g.step(1, 0)
    f = g.fields()
    g.close()
    o = gap2d.Oracle2D(cfg)
    o.set_particles(0, xe, eta, ue, we)
    o.set_particles(1, xi, eta, ui, wi)
    assert o.step(1, 0) == 0
    np.testing.assert_array_equal(f["G"], o.G)
    assert np.any(f["G"])
    np.testing.assert_allclose(f["phi"], o.phi, rtol=0, atol=2e-5 * np.abs(o.phi).max())
    ex_s = np.abs(o.Ex).max()
    np.testing.assert_allclose(f["Ex"], o.Ex, rtol=0, atol=2e-4 * ex_s)
    np.testing.assert_allclose(f["Ey"], o.Ey, rtol=0, atol=2e-4 * ex_s)


@pytest.mark.parametrize("Nx,Ny,n_pairs,beam,sort_every", [(40, 8, 700, 3, 0), (64, 64, 5, 0, 3), (100, 128, 40_001, 33, 4),
                                                           (33, 64, 90_000, 700, 0)])
def test_grid_is_the_deposit_of_the_particles(env, Nx, Ny, n_pairs, beam, sort_every):
    native, gap2d = env
    steps = 37  # whole graphs, a re-sort and single steps
    _, g, _ = gap(native, Nx, Ny, n_pairs, steps, beam, sort_every)
    for n in (20, 17):
        g.step(0, n)
        G = np.zeros((Nx + 1, Ny), dtype=np.int64)
        live = g.history()["n_live"][-1]
        for s, sign in ((0, -1), (1, 1), (2, -1)):
            x, y, _, _, ids = g.particles(s)
            assert x.size == live[s]
            if x.size:
                gap2d.deposit2d(Nx, Ny, x, y, sign, G)
            if s == 1:
                assert np.unique(ids).size == ids.size
        np.testing.assert_array_equal(g.fields()["G"], G)
    g.close()
