"""The single-gap push at the edges of its tiles and rounds.

The charge grid the push leaves must be, to the last unit, the fixed-point
deposit of the particles it leaves (every copy, vector edge, fold and flush
in between), and the particle counts must match the diagnostics' ledger.
"""
import numpy as np
import pytest

from paper_2603_24010_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_24010_gb300 import native
    native.lib()
    return native


def deposit(N, x, sign, G):
    i = np.floor(x).astype(np.int64)
    w = np.floor((x - i) * 65536.0).astype(np.int64)
    for k, v in ((i, 65536 - w), (i + 1, w)):  # sums below 2^53: exact in the weights' doubles
        G += sign * np.bincount(k, weights=v, minlength=N + 1).astype(np.int64)


def check(g, N):
    h = g.history()
    G = np.zeros(N + 1, dtype=np.int64)
    ids = None
    for s, sign in ((0, -1), (1, 1), (2, -1)):
        x, u, i = g.particles(s)
        assert x.size == h["n_live"][-1][s]
        assert np.all((x > 0) & (x < N)) and np.all(np.isfinite(u))
        deposit(N, x, sign, G)
        if s == 1:
            ids = i
    G[[0, N]] *= 2
    np.testing.assert_array_equal(g.grid()["G"], G)
    assert np.unique(ids).size == ids.size
    return h


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("N,n_pairs,beam", [(2, 1, 0), (64, 5, 3), (257, 1023, 1), (300, 2049, 305),
                                            (4096, 312_321, 7), (1531, 700_001, 0)])
def test_grid_is_the_deposit_of_the_particles(nat, precision, N, n_pairs, beam):
    cfg = W.scaled(W.gap_1d_fp64(seed=N), n_cells=N, n_pairs=n_pairs, beam_per_step=beam, precision=precision)
    cfg["weight"] = cfg["n0"] * cfg["d"] * cfg["area"] / n_pairs
    g = nat.Gap(cfg, max_steps=40, compact_every=7)
    g.load_species(n_pairs, 40.0, 3)
    for _ in range(3):
        g.step(0, 5)
        check(g, N)
    g.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("beam,law,scale", [(400, 1, 40.0), (90_000, 0, 10.0), (180_000, 1, 30.0)])
def test_many_impacts_and_large_beams(nat, precision, beam, law, scale):
    """Beams of more than one round of draws per CTA, whose impacts arrive
    together (several rounds of records and several electrons per impact)."""
    cfg = W.scaled(W.gap_1d_fp64(seed=5), d=1e-4, n_cells=48, n_pairs=2000, beam_per_step=beam, precision=precision,
                   see_scale=scale, see_count_law=law, weight=10.0)
    g = nat.Gap(cfg, max_steps=70, compact_every=50)
    g.load_species(2000, 1.0, 3)
    g.step(1, 60)
    h = check(g, 48)
    assert h["absorbed"][:, 0, 1].max() >= beam // 2
    assert h["emitted"].sum() > h["absorbed"][:, :, 1].sum()  # more than one electron an impact
    assert np.all(h["injected"][1:] == beam)
    g.close()
