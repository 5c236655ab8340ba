"""The ensemble push at the edges of its split.

A CTA lists eight (instance, species) segments of its share at a time, so
hundreds of tiny gaps make it list again; a gap of 1.2e7 particles adds more
tiles to a CTA's node sums than 32 bits hold; a beam larger than a block is
dealt in pieces.  Every instance must give the integers it gives alone.
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


def put(native, g, cfg, *at):
    xi, ue, ui = W.load_pairs(cfg)
    g.set_particles(*at, native.ELECTRONS, xi, ue)
    g.set_particles(*at, native.IONS, xi, ui)


def same(a, b):
    for k in ("absorbed", "emitted", "injected", "n_live", "conv_count", "ion_energy_eV", "max_cfl", "V_gap"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


def check(native, cfgs, picks, shapes, calls, capacity=(0, 0, 0)):
    steps = sum(calls) * len(shapes)
    b = native.Batch(cfgs, max_steps=steps, capacity=capacity)
    for i, cfg in enumerate(cfgs):
        put(native, b, cfg, i)
    assert b.step(native.WEAK, 0) == 0
    for threads, per_sm in shapes:
        assert b.set_launch(threads, per_sm) == native.OK
        for n in calls:
            assert b.step(native.WEAK, n) == 0
    for i in picks:
        g = native.Gap(cfgs[i], max_steps=steps)
        put(native, g, cfgs[i])
        g.step(native.WEAK, steps)
        same(b.history(i), g.history())
        np.testing.assert_array_equal(b.grid(i)["G"], g.grid()["G"])
        g.close()
    b.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_many_tiny_gaps(native, precision):
    cfgs = []
    for i in range(620):
        c = W.scaled(W.gap_1d_fp64(seed=i), n_cells=8 + i % 60, n_pairs=1 + (i * 7) % 90, see_scale=6.0,
                     beam_per_step=(0, 3, 40)[i % 3], d=2e-5, weight=1e4,
                     precision=W.FP32 if precision == "fp32" else W.FP64)
        cfgs.append(c)
    cfgs[300] = W.scaled(cfgs[300], n_cells=700, n_pairs=90_000, beam_per_step=1500)
    shapes = [(512, 1), (256, 1), (1024, 1)]
    check(native, cfgs, [0, 1, 2, 77, 299, 300, 301, 450, 618, 619], shapes, [1, 64, 5],
          capacity=(100_000, 500_000, 400_000))


def test_more_tiles_than_a_node_sum_holds(native):
    big = W.scaled(W.gap_1d_fp32_large(3), n_cells=300, n_pairs=6_000_000, beam_per_step=2600, weight=1e6)
    small = W.scaled(big, n_cells=97, n_pairs=3001, beam_per_step=0)
    check(native, [small, big, small], [0, 1], [(512, 1), (1024, 1)], [3],
          capacity=(6_000_100, 6_100_000, 100_000))
