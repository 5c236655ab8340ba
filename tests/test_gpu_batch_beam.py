"""An ensemble whose beam counts overflow 32 bits when added up over it."""
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


@pytest.mark.parametrize("E,beam", [(2, 2**31 - 1), (600, 2**31 - 512)])
def test_a_beam_beyond_the_store_is_reported(native, E, beam):
    cfgs = [W.scaled(W.gap_1d_fp64(seed=k), n_cells=16, n_pairs=8, beam_per_step=beam if k == 0 else 1,
                     precision=W.FP32) for k in range(E)]
    b = native.Batch(cfgs, max_steps=1, capacity=(64, 1024, 64))
    for i, cfg in enumerate(cfgs):
        xi, ue, ui = W.load_pairs(cfg)
        b.set_particles(i, native.ELECTRONS, xi, ue)
        b.set_particles(i, native.IONS, xi, ui)
    assert b.step(native.WEAK, 1) == native.ERR_CAPACITY
    st = b.status()
    assert st[0] == native.ERR_CAPACITY and not np.any(st[1:])
    np.testing.assert_array_equal(b.history(1)["injected"], [0, 1])  # the others go on
    b.close()
