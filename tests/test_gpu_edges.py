"""Edge cases of the walker cycle on the GPU against the oracle, through the C ABI: the largest supported
size (64 electrons in 64 spatial orbitals: both words of every determinant full, 2016 electron pairs),
a single electron (no pairs, so every attempt is a single), two electrons in two orbitals (a four-
determinant space), and an empty walker list. Walker lists identical after every iteration, every
integer counter identical, the shift bit-identical."""
from __future__ import annotations

import numpy as np
import pytest

from oracle.oracle import Oracle
from parity import compare_rows, same_lists
from paper_1305_6981_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def make_pair(system, tau, thr, **kw):
    from paper_1305_6981_gb300 import Fciqmc
    caps = {k: kw.pop(k) for k in ("main_capacity", "spawn_capacity") if k in kw}
    g = Fciqmc(system, tau, thr, **kw, **caps)
    q = Oracle(system, tau=tau, initiator_threshold=thr, **kw)
    return g, q


def lockstep(g, q, n_iter):
    rows_q = []
    for k in range(n_iter):
        g.step(1)
        rows_q += q.iterate(1)
        assert same_lists(g.walkers(), q.walkers()), f"walker lists differ after iteration {k + 1}"
    compare_rows(g.history(n_iter), rows_q)
    return rows_q


def test_largest_supported_size_64e64o():
    """8 irreps, slowly decaying Cholesky vectors and a near-degenerate window at the Fermi level, so
    that the reference spawns onto hundreds of determinants per iteration."""
    s = synth.make_system(64, 64, seed=11, n_chol=64, symmetry=True, chol_decay_len=8.0,
                          energies=synth.frontier_energies(64, lo=28, hi=35), name="64e64o")
    g, q = make_pair(s, 0.002, 3, initial_population=3000, initial_shift=0.0, seed=4, main_capacity=1 << 16)
    info = g.info()
    assert info["words"] == 2 and info["reference_excitations"] > 0
    ref = info["reference"]
    assert int(ref[0]) == (1 << 64) - 1 and int(ref[1]) == 0  # 32 doubly occupied orbitals fill word 0
    rows = lockstep(g, q, 6)
    assert rows[-1]["nd_out"] > 100 and sum(r["spawn_events"] for r in rows) > 100
    g.close()


def test_one_electron_only_singles():
    s = synth.small_system(6, 1, seed=2)
    g, q = make_pair(s, 0.01, -1, ms2=1, initial_population=200, initial_shift=0.1, seed=8, main_capacity=1 << 10)
    assert g.info()["n_double_ref"] == 0 and g.info()["p_double"] == 0.0
    rows = lockstep(g, q, 200)
    d, _, _ = g.walkers()
    assert len(d) >= 3  # the electron has left the reference orbital
    assert sum(r["spawn_events"] for r in rows) > 0
    g.close()


def test_two_electrons_in_two_orbitals():
    s = synth.small_system(2, 2, seed=3)
    g, q = make_pair(s, 0.01, -1, initial_population=100, initial_shift=0.1, seed=6, main_capacity=1 << 10)
    lockstep(g, q, 200)
    d, _, _ = g.walkers()
    assert 1 < len(d) <= 4
    g.close()


def test_empty_walker_list():
    s = synth.tiny_8e8o()
    g, q = make_pair(s, 0.01, -1, initial_population=50, seed=2, main_capacity=1 << 10)
    none_d = np.zeros((0, 1), dtype=np.uint64)
    none_p = np.zeros(0, dtype=np.int32)
    g.set_walkers(none_d, none_p, iteration=7, shift=0.3, vary=0)
    q.set_walkers(none_d, none_p, iteration=7, shift=0.3)
    rows = lockstep(g, q, 3)
    assert all(r["nw_out"] == 0 and r["attempts"] == 0 for r in rows)
    assert len(g.walkers()[1]) == 0
    g.close()


@pytest.mark.parametrize("steps,want", [(5, 16), (16, 16), (21, 16), (40, 7)])
def test_history_ring_in_one_or_two_pieces(steps, want):
    """The newest rows, oldest first, before and after the ring of 16 rows has wrapped."""
    from paper_1305_6981_gb300 import Fciqmc
    runs = [Fciqmc(synth.tiny_8e8o(), 0.01, -1, initial_population=50, seed=3, main_capacity=1 << 12, history_capacity=c)
            for c in (16, 64)]
    for g in runs:
        g.step(steps)
    short, full = (g.history(want) for g in runs)
    assert [r["iteration"] for r in short] == list(range(max(0, steps - want), steps)) and len(short) == min(steps, want, 16)
    ints = [k for k in short[0] if k != "num_in"]  # (the numerator is summed in slot order)
    assert [[r[k] for k in ints] for r in short] == [[r[k] for k in ints] for r in full]
    for g in runs:
        g.close()


def test_target_does_not_size_the_run():
    """A run made for a target of one walker (the shift varies from the start) and loaded with a list of 1e6 advances as
    fast as one made for 1e6 (20 times slower when the grid for heavily populated determinants followed the target)."""
    from paper_1305_6981_gb300 import Fciqmc
    s = synth.large_24e60o()
    dets, pops = synth.walker_snapshot(s, 1_000_000, seed=2)

    def best(target):
        g = Fciqmc(s, 0.001, 3, target_walkers=target, seed=1, main_capacity=1 << 20, spawn_capacity=1 << 18)
        g.set_walkers(dets, 8 * pops, iteration=5, shift=0.0, vary=0)
        g.step(3)
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.step(5)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        assert g.history(1)[0]["heavy_attempts"] > 100_000
        g.close()
        return min(times)

    assert best(1) < 2 * best(1_000_000)


@pytest.mark.parametrize("walkers,tau", [(40, 0.0005), (300, 0.0001)])
def test_every_determinant_of_a_short_list_heavily_populated(walkers, tau):
    """20,000 determinants in a capacity of 32,768, all above the threshold of heavily populated determinants (32 walkers
    for a list as short as this, from its second iteration on): as the oracle, and no capacity is exceeded."""
    s = synth.make_system(20, 10, seed=4, n_chol=8)
    g, q = make_pair(s, tau, 3, seed=6, main_capacity=1 << 15, spawn_capacity=1 << 18)
    dets, _ = synth.walker_snapshot(s, 200_000, seed=3)
    dets = dets[:20_000]
    assert len(dets) == 20_000
    pops = np.where(np.random.default_rng(1).random(20_000) < 0.5, -walkers, walkers).astype(np.int32)
    for x in (g, q):
        x.set_walkers(dets, pops, iteration=3, shift=0.0)
    rows_q = q.iterate(3)
    g.step(3)
    rows_g = g.history(3)
    compare_rows(rows_g, rows_q)
    assert rows_g[1]["heavy_attempts"] > 0.9 * rows_g[1]["attempts"]
    assert same_lists(g.walkers(), q.walkers())
    g.close()
