"""The removal of absorbed particles at the edges of its blocks.

A block takes 16 chunks of 128 slots from 16 regions of a store and leaves the
live ones interleaved; a removal after every step, on stores from one slot to
several blocks, must give the integers of a run that removes nothing, and keep
every ion's id with its position and velocity.
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


def config(pairs, precision, seed):
    return W.scaled(W.gap_1d_fp64(seed=seed), n_cells=200, n_pairs=pairs, beam_per_step=37, see_scale=10.0, d=4e-5,
                    weight=5e8 / pairs, precision=W.FP32 if precision == "fp32" else W.FP64)


def fill(native, g, cfg, *at):
    xi, ue, ui = W.load_pairs(cfg)
    g.set_particles(*at, native.ELECTRONS, xi, ue)
    g.set_particles(*at, native.IONS, xi, ui, np.arange(xi.size, dtype=np.uint32) + 5)


def result(native, cfg, every, steps):
    g = native.Gap(cfg, max_steps=steps, compact_every=every)
    fill(native, g, cfg)
    g.step(native.WEAK, steps)
    x, u, i = g.particles(native.IONS)
    o = np.argsort(i)
    out = g.history(), g.grid()["G"], (x[o], u[o], i[o])
    g.close()
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("pairs", [1, 127, 128, 129, 2047, 2049, 30_011])
def test_removal_changes_nothing(native, pairs, precision):
    cfg = config(pairs, precision, 3 + pairs % 7)
    steps = 60
    h0, G0, p0 = result(native, cfg, 1000, steps)
    assert h0["absorbed"].sum() > 0
    for every in (1, 7):
        h, G, p = result(native, cfg, every, steps)
        for k in KEYS:
            np.testing.assert_array_equal(h[k], h0[k], err_msg="%s %d" % (k, every))
        np.testing.assert_array_equal(G, G0)
        for a, b in zip(p, p0):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_ensemble_removal(native, precision):
    cfgs = [config(p, precision, 11 + k) for k, p in enumerate((3, 128, 2049, 9000, 40_001, 1))]
    b = native.Batch(cfgs, max_steps=60, compact_every=3)
    for i, cfg in enumerate(cfgs):
        fill(native, b, cfg, i)
    assert b.step(native.WEAK, 60) == 0
    for i, cfg in enumerate(cfgs):
        h0, G0, p0 = result(native, cfg, 1000, 60)
        h = b.history(i)
        for k in KEYS:
            np.testing.assert_array_equal(h[k], h0[k], err_msg="%s %d" % (k, i))
        np.testing.assert_array_equal(b.grid(i)["G"], G0)
        x, u, ids = b.particles(i, native.IONS)
        o = np.argsort(ids)
        for a, c in zip((x[o], u[o], ids[o]), p0):
            np.testing.assert_array_equal(a, c)
    b.close()
