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
