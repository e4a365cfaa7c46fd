"""Imported lists at the edges of the spawning and annihilation kernels.

One list per system with amplitudes around every boundary of the spawning
kernel: windows of 32 attempts, powers of two (C / n_att by the exponent) and
other counts (by division), slices of 512 attempts and the smaller slices of
short lists, zero and fractional amplitudes; orbitals 0 and 63 in use; one
bucket (many warps per bucket, crowded buckets) and many buckets (one warp per
bucket).  Everything is an exact sum or a keyed draw, so the GPU's list and
statistics must equal the oracle's bit for bit.
"""
import numpy as np
import pytest

import oracle
import workloads
from tests.test_gpu_parity import _fq, assert_states_equal, assert_stats_equal

pytestmark = pytest.mark.gpu

EDGES = [0.25, 0.75, 1.0, 1.5, 2.0, 2.5, 3.0, 4.0, 5.5, 7.0, 8.0, 15.5, 16.0, 31.0, 32.0, 32.5, 33.0, 63.5, 64.0, 64.5, 65.0,
         127.0, 128.0, 511.5, 512.0, 512.5, 513.0, 1024.0, 1500.25, 3000.0]


def _words(rng, norb, n_el, n):
    out = []
    for _ in range(n):
        w = 0
        for p in rng.choice(norb, n_el, replace=False):
            w |= 1 << int(p)
        out.append(w)
    return np.array(out, np.uint64)


def _list(sysd, norb, n, seed):
    """n distinct determinants (a third with orbitals 0 and norb - 1 occupied), amplitudes through EDGES, the
    reference among them."""
    rng = np.random.default_rng(seed)
    s = oracle.system_from_workload(sysd)
    ra, rb = s.ref
    a, b = _words(rng, norb, sysd["n_alpha"], n), _words(rng, norb, sysd["n_beta"], n)
    a[0], b[0] = ra, rb
    key = sorted({(int(x), int(y)) for x, y in zip(a, b)}, key=lambda k: (k != (ra, rb), rng.random()))
    a = np.array([k[0] for k in key], np.uint64)
    b = np.array([k[1] for k in key], np.uint64)
    c = np.ones(a.size)
    c[1::2] = rng.choice([0.5, 1.0, 1.25, 2.0, 3.0], c[1::2].size)
    k = min(len(EDGES), a.size)
    c[:k] = np.array(EDGES[::-1])[:k]
    return s, a, b, c * rng.choice([-1.0, 1.0], c.size)


def _abinitio(norb, na, nb, seed):
    h, eri = workloads.synthetic_abinitio(norb, 8, seed)
    return dict(kind="abinitio", norb=norb, n_alpha=na, n_beta=nb, h1=h, eri=eri, ecore=0.0)


CASES = {
    "orb64": (lambda: _abinitio(64, 3, 2, 3), 64, dict(tau=2e-4, p_single=0.3, initiator_threshold=3.0)),
    "orb33_one_beta": (lambda: _abinitio(33, 4, 1, 4), 33, dict(tau=2e-4, c_min=0.3, initiator_threshold=1.0)),
    "orb20_heatbath": (lambda: _abinitio(20, 4, 3, 5), 20, dict(tau=5e-4, generator=1, initiator_threshold=3.0)),
    "orb20_adaptive": (lambda: _abinitio(20, 4, 3, 6), 20, dict(tau=5e-4, adaptive_shift=1, initiator_threshold=3.0)),
    # no initiator but the reference: the spawns of heavily populated determinants are weighed too
    "orb20_adaptive_heavy": (lambda: _abinitio(20, 4, 3, 7), 20, dict(tau=5e-4, adaptive_shift=1, initiator_threshold=1e6)),
    "hubbard_8x8": (lambda: dict(workloads.hubbard_2d(8, 8, 4.0)), 64, dict(tau=2e-3)),
}


@pytest.mark.parametrize("max_dets", [16, 20000, 8000000])
@pytest.mark.parametrize("name", sorted(CASES))
def test_imported_list_at_the_edges_bit_exact(name, max_dets):
    fq = _fq()
    make, norb, prm = CASES[name]
    sysd = make()
    prm = dict(dict(target_walkers=1e9, seed=77, shift_damping=0.5, shift_interval=5), **prm)
    s, a, b, c = _list(sysd, norb, 700, 11)
    g = fq.fciqmc_create(sysd, dict(prm, max_dets=max_dets))
    o = oracle.Run(s, **prm)
    fq.fciqmc_import_state(g, a, b, c, 0, 0.1)
    o.import_state(a, b, c, 0, 0.1)
    fq.fciqmc_step(g, 3)
    o.step(3)
    assert_states_equal(fq.fciqmc_export_state(g), o.export())
    assert_stats_equal(fq.fciqmc_iter_stats_get(g), o.stats(), first=0)


@pytest.mark.parametrize("max_dets", [16, 4000])
def test_crowded_buckets_bit_exact(max_dets):
    """Hundreds of walkers on every determinant of a small space, alone and in
    a batch: every bucket holds more spawns than a warp annihilates, some more
    than fit shared memory, and the two kinds are annihilated side by side."""
    fq = _fq()
    sysd = workloads.hubbard_1d(8, 1.0, 4.0)
    s = oracle.system_from_workload(sysd)
    a, b = np.array(s.determinants(), np.uint64).T
    rng = np.random.default_rng(5)
    c = rng.normal(0.0, 1.0, a.size) * np.where(rng.random(a.size) < 0.3, 400.0, 20.0)
    prm = dict(tau=0.01, target_walkers=1e9, seed=3, shift_damping=0.5, shift_interval=5, initiator_threshold=3.0)
    o = oracle.Run(s, **prm)
    o.import_state(a, b, c, 0, -2.0)
    o.step(4)
    gs = [fq.fciqmc_create(sysd, dict(prm, max_dets=max_dets)) for _ in range(4)]
    for g in gs:
        fq.fciqmc_import_state(g, a, b, c, 0, -2.0)
    fq.fciqmc_step(gs[0], 4)
    fq.fciqmc_step_batch(gs[1:], 4)
    for g in gs:
        assert_states_equal(fq.fciqmc_export_state(g), o.export())
        assert_stats_equal(fq.fciqmc_iter_stats_get(g), o.stats())


@pytest.mark.parametrize("count", [2, 33, 70])
def test_batch_deals_slices_and_crowded_buckets_of_all_runs(count):
    """Runs with different numbers of heavy slices and crowded buckets (some
    with none), fewer and more than a warp's 32 lanes: each equals its run alone."""
    fq = _fq()
    sysd = workloads.hubbard_1d(6, 1.0, 4.0)
    s = oracle.system_from_workload(sysd)
    a, b = np.array(s.determinants(), np.uint64).T
    prm = dict(tau=0.01, target_walkers=1e9, shift_damping=0.5, shift_interval=5, initiator_threshold=3.0)
    rng = np.random.default_rng(9)
    runs = []
    for i in range(count):
        c = rng.normal(0.0, 1.0, a.size) * [1.0, 40.0, 600.0][i % 3]
        runs.append((dict(prm, seed=100 + i, max_dets=[16, 4000][i % 2]), c))
    gs = []
    for p, c in runs + runs:
        g = fq.fciqmc_create(sysd, p)
        fq.fciqmc_import_state(g, a, b, c, 0, -2.0)
        gs.append(g)
    fq.fciqmc_step_batch(gs[:count], 3)
    for g, h in zip(gs[:count], gs[count:]):
        fq.fciqmc_step(h, 3)
        assert_states_equal(fq.fciqmc_export_state(g), fq.fciqmc_export_state(h))
        x, y = fq.fciqmc_iter_stats_get(g), fq.fciqmc_iter_stats_get(h)
        for name in x:
            np.testing.assert_array_equal(x[name], y[name], err_msg=name)


@pytest.mark.parametrize("max_dets", [[16, 8000000], [8000000, 16, 4000000]])
def test_batch_with_claimed_buckets(max_dets):
    """Batches with so many buckets that both kernels claim the last of them
    through the first run's counters, in a short or a long run: each run equals
    the same run alone, twice over (the counters are cleared in between)."""
    fq = _fq()
    sysd = _abinitio(20, 4, 3, 8)
    _, a, b, c = _list(sysd, 20, 700, 12)
    prm = dict(tau=5e-4, target_walkers=1e9, shift_damping=0.5, shift_interval=5, initiator_threshold=3.0)
    gs = []
    for i, m in enumerate(max_dets + max_dets):
        g = fq.fciqmc_create(sysd, dict(prm, seed=200 + i % len(max_dets), max_dets=m))
        fq.fciqmc_import_state(g, a, b, c, 0, 0.1)
        gs.append(g)
    k = len(max_dets)
    for _ in range(2):
        fq.fciqmc_step_batch(gs[:k], 2)
        for g, h in zip(gs[:k], gs[k:]):
            fq.fciqmc_step(h, 2)
            assert_states_equal(fq.fciqmc_export_state(g), fq.fciqmc_export_state(h))
            x, y = fq.fciqmc_iter_stats_get(g), fq.fciqmc_iter_stats_get(h)
            for name in x:
                np.testing.assert_array_equal(x[name], y[name], err_msg=name)


def test_more_than_64_electrons_bit_exact():
    """Beyond the table of electron pairs: H_ii of an imported list and of new
    determinants by the sums that need no table."""
    fq = _fq()
    sysd = _abinitio(64, 34, 33, 10)
    prm = dict(target_walkers=1e9, seed=79, shift_damping=0.5, shift_interval=5, tau=2e-5, initiator_threshold=3.0)
    s, a, b, c = _list(sysd, 64, 300, 14)
    g = fq.fciqmc_create(sysd, prm)
    o = oracle.Run(s, **prm)
    fq.fciqmc_import_state(g, a, b, c, 0, 0.1)
    o.import_state(a, b, c, 0, 0.1)
    fq.fciqmc_step(g, 3)
    o.step(3)
    assert o.export()["alpha"].size > 310  # new determinants among them
    assert_states_equal(fq.fciqmc_export_state(g), o.export())
    assert_stats_equal(fq.fciqmc_iter_stats_get(g), o.stats(), first=0)
