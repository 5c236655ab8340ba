"""When the 2D gap's particle store is re-sorted.

The re-sort pads every tile's segment to whole 16-byte vectors, so it needs
more slots than the particles themselves.  It belongs to the step that follows
it: a call that ends where a re-sort is due returns its steps, whatever the
padded store would need.
"""
import numpy as np
import pytest

from paper_2603_24010_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_24010_gb300 import native
    native.lib()
    return native


def full_store(native):
    """Four ions in each of 64 tiles and a beam that fills the ions' 576 slots in
    16 steps.  One ion of every other tile moves on by a tile meanwhile, so that
    the sorted store would need 128 slots more."""
    cfg = W.gap_2d(0, Nx=256, Ny=256, n_pairs=256, steps=40, beam_per_step=20)
    g = native.Gap2D(cfg, max_steps=40, capacity=(4096, 576, 4096))
    t = np.repeat(np.arange(64), 4)
    xi, eta, z = 32.0 * (t // 8) + 16.5, 32.0 * (t % 8) + 16.5, np.zeros(256)
    w = np.where((np.arange(256) % 4 == 0) & (t % 2 == 0), 2.0, 0.0)
    g.set_particles(native.ELECTRONS, xi, eta, z, z)
    g.set_particles(native.IONS, xi, eta, z, w)
    return g


def test_a_call_that_ends_at_a_resort_keeps_its_particles(native):
    g = full_store(native)
    g.step(native.WEAK, 16)
    assert g.level == 16
    assert g.history()["n_live"][-1, 1] == 576
    assert g.particles(native.IONS)[0].size == 576
    with pytest.raises(native.CpError) as e:  # the next step's re-sort does not fit
        g.step(native.WEAK, 1)
    assert e.value.status == native.ERR_CAPACITY
    g.close()


@pytest.mark.parametrize("sort_every", [5, 16, 17, 40, 1000])
def test_any_period_gives_the_same_steps(native, sort_every):
    """Graphs, single steps and re-sorts in every mixture against one step a call."""
    cfg = W.gap_2d(3, Nx=64, Ny=64, n_pairs=20_000, steps=80, beam_per_step=32)
    p = W.load_pairs_2d(cfg)

    def run(calls, every):
        g = native.Gap2D(cfg, max_steps=80, sort_every=every)
        g.set_particles(native.ELECTRONS, *p[:4])
        g.set_particles(native.IONS, p[0], p[1], p[4], p[5])
        for n in calls:
            g.step(native.WEAK, n)
        h, G = g.history(), g.fields()["G"]
        g.close()
        return h, G

    want, G0 = run([1] * 80, 16)
    for calls in ([80], [7, 33, 40], [20, 60]):
        h, G = run(calls, sort_every)
        for k in ("absorbed", "emitted", "injected", "n_live", "conv_count", "V_gap"):
            np.testing.assert_array_equal(h[k], want[k], err_msg=k)
        np.testing.assert_array_equal(G, G0)


def test_a_long_period_makes_no_long_graph(native):
    """The device memory of a call's graph does not grow with the period."""
    import torch
    steps = 20_000
    cfg = W.gap_2d(0, Nx=32, Ny=32, n_pairs=100, steps=steps, beam_per_step=0)
    p = W.load_pairs_2d(cfg)
    g = native.Gap2D(cfg, max_steps=steps, sort_every=steps)
    g.set_particles(native.ELECTRONS, *p[:4])
    g.set_particles(native.IONS, p[0], p[1], p[4], p[5])
    g.step(native.WEAK, 0)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    g.step(native.WEAK, steps)
    # a graph of 16 steps takes 2 MB, one of 20000 takes 200
    assert free - torch.cuda.mem_get_info()[0] < 32 << 20
    assert g.level == steps
    g.close()
