"""Steps launched one by one right behind a removal of absorbed particles.

The removal swaps the store's buffers.  The step behind it must take its
particles from the new ones, in calls of every length against the removal's
period, with particles removed and with none (the slot counts are then the
same before and after it, and only the buffers differ).
"""
import numpy as np
import pytest

from paper_2603_24010_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("absorbed", "emitted", "injected", "n_live", "conv_count", "ion_energy_eV", "V_gap")


@pytest.fixture(scope="module")
def native():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_24010_gb300 import native
    native.lib()
    return native


def config(pairs, precision, absorbing):
    over = dict(beam_per_step=37, see_scale=10.0, d=4e-5, weight=5e8 / pairs) if absorbing else dict(beam_per_step=0)
    return W.scaled(W.gap_1d_fp64(seed=2), n_cells=200, n_pairs=pairs,
                    precision=W.FP32 if precision == "fp32" else W.FP64, **over)


def result(native, cfg, every, calls, timing=False):
    g = native.Gap(cfg, max_steps=sum(calls), compact_every=every)
    xi, ue, ui = W.load_pairs(cfg)
    if cfg["beam_per_step"] == 0:  # resting, away from the electrodes: none is absorbed
        xi, ue, ui = 80.0 + 0.2 * xi, 0.0 * ue, 0.0 * ui
    g.set_particles(native.ELECTRONS, xi, ue)
    g.set_particles(native.IONS, xi, ui, np.arange(xi.size, dtype=np.uint32) + 5)
    if timing:
        native.lib().cp_enable_timing(g.ctx, 1)
    for n in calls:
        g.step(native.WEAK, n)
    stores = []
    for s in (native.ELECTRONS, native.IONS, native.SECONDARIES):
        x, u, ids = g.particles(s)
        o = np.lexsort((u, x)) if ids is None else np.argsort(ids)
        stores += [x[o], u[o]] + ([ids[o]] if s == native.IONS else [])
    out = g.history(), g.grid()["G"], stores
    g.close()
    return out


@pytest.mark.parametrize("absorbing", [False, True])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("pairs", [500, 400_000])
def test_steps_behind_a_removal(native, pairs, precision, absorbing):
    cfg = config(pairs, precision, absorbing)
    h0, G0, s0 = result(native, cfg, 1000, [60])
    assert (h0["absorbed"].sum() > 0) == absorbing
    # every = 3: calls of 2 and 4 cross removals between steps launched one by
    # one; of 7, whole graphs with such steps behind them
    for calls, timing in (([2] * 30, False), ([4] * 15, False), ([7] * 8 + [4], False), ([1, 59], False), ([60], True)):
        h, G, s = result(native, cfg, 3, calls, timing)
        for k in KEYS:
            np.testing.assert_array_equal(h[k], h0[k], err_msg="%s %s" % (k, calls[:2]))
        np.testing.assert_array_equal(G, G0)
        for a, b in zip(s, s0):
            np.testing.assert_array_equal(a, b)
