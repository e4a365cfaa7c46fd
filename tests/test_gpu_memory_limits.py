"""Runs at the limit of their device memory: what does not fit is refused or
left out, nothing stays allocated for it, and the run goes on as it was."""
import numpy as np
import pytest

import oracle
import workloads
from tests.test_gpu_parity import DAMP, _fq, assert_states_equal, assert_stats_equal

pytestmark = pytest.mark.gpu


def _determinants(norb, na, nb, n, seed):
    """n distinct determinants, the reference (lowest orbitals) among them: an import adds it where it is absent."""
    rng = np.random.default_rng(seed)
    key = {((1 << na) - 1, (1 << nb) - 1)}
    while len(key) < n:
        for _ in range(n - len(key)):
            a = sum(1 << int(p) for p in rng.choice(norb, na, replace=False))
            b = sum(1 << int(p) for p in rng.choice(norb, nb, replace=False))
            key.add((a, b))
    k = np.array(sorted(key), np.uint64)
    return k[:, 0].copy(), k[:, 1].copy()


@pytest.mark.parametrize("use_torch", [True, False])
def test_import_that_does_not_fit_leaves_the_run_and_its_memory_alone(use_torch):
    fq = _fq()
    sysd = workloads.small_abinitio(12, 4, 4, seed=9)
    prm = dict(DAMP, tau=0.002, target_walkers=500, initiator_threshold=3.0, seed=21, max_dets=100)
    bytes0 = fq.fciqmc_layout(fq.fciqmc_create(sysd, prm, use_torch=use_torch))["device_bytes"]
    a, b = _determinants(12, 4, 4, 20000, 1)
    # room for the scratch of the import (24 bytes each) but not for 2^8 buckets of 192 slots
    g = fq.fciqmc_create(sysd, dict(prm, max_device_bytes=bytes0 + (2 << 20)), use_torch=use_torch)
    fq.fciqmc_step(g, 10)
    before = fq.fciqmc_layout(g)
    for _ in range(2):
        with pytest.raises(fq.FciqmcError) as e:
            fq.fciqmc_import_state(g, a, b, np.ones(a.size), 0, 0.0)
        assert e.value.code == fq.FCIQMC_ERR_OUT_OF_MEMORY
        assert fq.fciqmc_layout(g) == before
    fq.fciqmc_step(g, 10)
    o = oracle.Run(oracle.system_from_workload(sysd), **{k: v for k, v in prm.items() if k != "max_dets"})
    o.step(20)
    assert_states_equal(fq.fciqmc_export_state(g), o.export())
    assert_stats_equal(fq.fciqmc_iter_stats_get(g), o.stats())


class _Refusing:
    """PyTorch's allocator, answering NULL to requests of the sizes in `refuse` after the first `skip` of them."""
    refuse = ()
    skip = 0

    @classmethod
    def install(cls, fq, monkeypatch):
        base = fq._TorchAllocator

        class Refusing(base):
            def _alloc(self, nbytes, ctx):
                cls.skip -= nbytes in cls.refuse
                return None if nbytes in cls.refuse and cls.skip < 0 else super()._alloc(nbytes, ctx)

        monkeypatch.setattr(fq, "_TorchAllocator", Refusing)
        monkeypatch.setattr(cls, "refuse", ())
        monkeypatch.setattr(cls, "skip", 0)
        return cls


def test_a_step_after_a_call_that_failed_half_way_uses_the_buffers_of_now(monkeypatch):
    """An import that has replaced the buckets and then finds no memory for
    the selection of D fails; the run stands at the imported list."""
    fq = _fq()
    alloc = _Refusing.install(fq, monkeypatch)
    sysd = workloads.small_abinitio(12, 4, 4, seed=9)
    prm = dict(DAMP, tau=0.002, target_walkers=1e5, initiator_threshold=3.0, seed=22)
    g = fq.fciqmc_create(sysd, dict(prm, max_dets=100, semistoch_size=50, semistoch_start=5))
    fq.fciqmc_step(g, 2)
    a, b = _determinants(12, 4, 4, 3000, 2)
    c = np.random.default_rng(3).normal(0.0, 2.0, a.size)
    shift = (5, 0.1, 1, 0, 0, sum(int(x) for x in np.floor(np.abs(c) * 2.0 ** 32)))
    alloc.refuse = (65536 * 4,)  # the histogram of the selection
    with pytest.raises(fq.FciqmcError) as e:
        fq.fciqmc_import_state(g, a, b, c, *shift)
    assert e.value.code == fq.FCIQMC_ERR_OUT_OF_MEMORY
    alloc.refuse = ()
    o = oracle.Run(oracle.system_from_workload(sysd), **prm)
    o.import_state(a, b, c, *shift)
    for step in (lambda: fq.fciqmc_step(g, 2), lambda: fq.fciqmc_step_batch([g], 2),
                 lambda: (fq.fciqmc_step_async(g, 2), fq.fciqmc_sync(g))):
        step()
        o.step(2)
        assert_states_equal(fq.fciqmc_export_state(g), o.export())


EARLY = {"alone": dict(), "plain": dict(), "adaptive": dict(adaptive_shift=1), "pair": dict(replicas=2)}


@pytest.mark.parametrize("kind", sorted(EARLY))
def test_early_split_that_does_not_fit_is_left_out(monkeypatch, kind):
    """Buckets that hold more walkers and spawns than a warp annihilates (in a
    run alone also those that are half full) are split to save time.  Where the
    memory for that is missing (any limit from the run's own bytes to several
    splits; an allocator that refuses a run or one replica of a pair), the run
    finishes on what it has."""
    fq = _fq()
    alloc = _Refusing.install(fq, monkeypatch)
    sysd = dict(workloads.hubbard_1d(8, 1.0, 4.0), n_beta=3, ref=(0x55, 0x2a))
    s = oracle.system_from_workload(sysd)
    a, b = (x.copy() for x in np.array(s.determinants(), np.uint64).T)
    c = 4.5 * np.random.default_rng(4).choice([-1.0, 1.0], a.size)  # 122 walkers and 45 spawns to a bucket, evenly
    prm = dict(DAMP, tau=0.01, target_walkers=1e9, initiator_threshold=3.0, seed=31, max_dets=4000, **EARLY[kind])
    o = oracle.Run(s, **{k: v for k, v in prm.items() if k not in ("max_dets", "replicas")})
    o.import_state(a, b, c, 0, 4.0)
    o.step(20)

    def run(limit, refuse=(), skip=0):
        g = fq.fciqmc_create(sysd, dict(prm, max_device_bytes=limit))
        both = [g] if kind != "pair" else [g, fq.fciqmc_replica(g, 1)]
        for r in both:
            fq.fciqmc_import_state(r, a, b, c, 0, 4.0)
        first = fq.fciqmc_layout(g)
        alloc.refuse, alloc.skip = refuse, skip
        for _ in range(5):
            if kind == "alone":
                fq.fciqmc_step(g, 4)
            else:
                fq.fciqmc_step_batch(both, 4)
        alloc.refuse = ()
        assert_states_equal(fq.fciqmc_export_state(g), o.export())
        last = [fq.fciqmc_layout(r) for r in both]
        assert all(x == last[0] for x in last)
        assert last[0]["cap_spawn"] == first["cap_spawn"]  # no growth that the run could not do without
        return first, last[0]

    first, last = run(0)
    assert first["buckets"] == 32 and last["buckets"] > 32
    keys = 2 * first["buckets"] * first["cap_main"] * 16  # bytes of a key array of the split layout, two of them to a run
    for skip in (0, 2) if kind == "pair" else (0,):
        assert run(0, (keys,), skip) == (first, first)
    for more in np.linspace(16 << 10, 6 << 20, 13).astype(int):
        limit = first["device_bytes"] + int(more)
        assert run(limit)[1]["device_bytes"] <= limit


@pytest.mark.parametrize("refused", ["partner_split", "first_lists", "second_lists"])
def test_pair_goes_on_whole_after_a_growth_that_failed_half_way(monkeypatch, refused):
    """The first replica's first iteration needs more buckets, and the second
    follows.  The allocator refuses them to the second replica, or the lists of the join to one of the two: the call
    fails, and the next one, with memory, gives what the oracle's pair gives,
    cross estimators included."""
    from tests.test_gpu_replicas import check_pair
    fq = _fq()
    alloc = _Refusing.install(fq, monkeypatch)
    sysd = dict(workloads.hubbard_1d(8, 1.0, 4.0), n_beta=3, ref=(0x55, 0x2a))
    s = oracle.system_from_workload(sysd)
    a, b = (x.copy() for x in np.array(s.determinants(), np.uint64).T)
    c = 9.0 * np.random.default_rng(5).choice([-1.0, 1.0], a.size)  # 97 spawns to each of 32 buckets
    prm = dict(DAMP, tau=0.01, target_walkers=1e9, initiator_threshold=3.0, seed=33)
    g = fq.fciqmc_create(sysd, dict(prm, max_dets=4000, replicas=2))
    pair = oracle.Pair(s, **prm)
    for r in (0, 1):
        fq.fciqmc_import_state(fq.fciqmc_replica(g, r), a, b, c / (1 + 4 * r), 0, 4.0)
        pair.r[r].import_state(a, b, c / (1 + 4 * r), 0, 4.0)
    lay = fq.fciqmc_layout(g)
    assert (lay["buckets"], lay["cap_spawn"]) == (32, 96)
    keys, lists = 64 * lay["cap_main"] * 16, 64 * (lay["cap_main"] + lay["cap_spawn"]) * 48
    alloc.refuse = (keys,) if refused == "partner_split" else (lists,)
    alloc.skip = {"partner_split": 2, "first_lists": 0, "second_lists": 1}[refused]
    with pytest.raises(fq.FciqmcError) as e:
        fq.fciqmc_step(g, 24)
    assert e.value.code == fq.FCIQMC_ERR_OUT_OF_MEMORY
    alloc.refuse = ()
    fq.fciqmc_step(g, 24 - fq.fciqmc_export_shift(g)["iteration"])
    pair.step(24)
    check_pair(fq, g, pair)


@pytest.mark.parametrize("dets", [145, 145 << 6, 155 << 10, 160 << 11, 161 << 11])
def test_a_list_of_a_stated_length_gets_few_slots_per_determinant(dets):
    """At most 160 determinants to a bucket of 192 slots, in a power of two of buckets: below 2.4 slots each."""
    fq = _fq()
    lay = fq.fciqmc_layout(fq.fciqmc_create(workloads.small_abinitio(12, 4, 4, seed=9), dict(tau=0.002, max_dets=dets)))
    assert dets / 160 <= lay["buckets"] < dets / 80 + 1


def test_create_without_room_for_spread_buckets_takes_fewer(monkeypatch):
    fq = _fq()
    alloc = _Refusing.install(fq, monkeypatch)
    sysd = workloads.small_abinitio(12, 4, 4, seed=9)
    prm = dict(tau=0.002, target_walkers=1e4)
    lay = fq.fciqmc_layout(fq.fciqmc_create(sysd, prm))
    alloc.refuse = (lay["buckets"] * lay["cap_main"] * 16,)
    few = fq.fciqmc_layout(fq.fciqmc_create(sysd, prm))
    assert few["buckets"] < lay["buckets"] and few["device_bytes"] < lay["device_bytes"]


REQUESTS = {
    "lattice": (workloads.hubbard_2d(4, 4, 4.0), dict(tau=0.005, target_walkers=1e4)),
    "adaptive": (workloads.small_abinitio(12, 4, 4, seed=9), dict(tau=0.002, target_walkers=3e4, adaptive_shift=1)),
    "heatbath": (workloads.config_abinitio_24()[0], dict(tau=2e-4, target_walkers=1e4, generator=1)),
    "stated_length": (workloads.config_abinitio_24()[0], dict(tau=2e-4, max_dets=150000)),
}


@pytest.mark.parametrize("kind", sorted(REQUESTS))
def test_server_counts_at_least_what_create_takes(kind):
    """A second request of the same kind is not admitted into a budget that it
    would exceed as soon as it is created, and is into one with room."""
    fq = _fq()
    sysd, prm = REQUESTS[kind]
    prm = dict(DAMP, seed=41, max_device_bytes=8 << 30, **prm)
    size = fq.fciqmc_layout(fq.fciqmc_create(sysd, prm, use_torch=False))["device_bytes"]
    for budget, second in ((2 * size - 1, "queued"), (8 * size, "running")):
        srv = fq.fciqmc_server_create(budget, max_active=8)
        ids = [fq.fciqmc_server_submit(srv, sysd, prm, target_sigma=1e-12, max_iters=50) for _ in range(2)]
        fq.fciqmc_server_tick(srv, 1)
        got = [fq.fciqmc_server_poll(srv, i)["state_name"] for i in ids]
        assert got == ["running", second], budget
        fq.fciqmc_server_destroy(srv)


@pytest.mark.parametrize("batch", [False, True])
def test_slices_that_only_save_time_are_left_out_without_room(batch):
    """4900 determinants of 100 walkers on a short list, one slice each, for a
    queue of 4096 that cannot grow: the warps draw them where they find them."""
    fq = _fq()
    sysd = workloads.hubbard_1d(8, 1.0, 4.0)
    s = oracle.system_from_workload(sysd)
    a, b = (x.copy() for x in np.array(s.determinants(), np.uint64).T)
    c = 100.0 * np.random.default_rng(6).choice([-1.0, 1.0], a.size)
    c[:20] *= 40.0  # some with several slices
    prm = dict(DAMP, tau=1e-5, target_walkers=1e5, initiator_threshold=3.0, seed=35)
    sizes = dict(prm, max_dets=8000)
    free = fq.fciqmc_layout(fq.fciqmc_create(sysd, sizes))
    g = fq.fciqmc_create(sysd, dict(sizes, max_device_bytes=free["device_bytes"] + (200 << 10)))
    assert fq.fciqmc_layout(g) == free
    o = oracle.Run(s, **prm)
    fq.fciqmc_import_state(g, a, b, c, 0, 4.0)
    o.import_state(a, b, c, 0, 4.0)
    for _ in range(2):
        if batch:
            fq.fciqmc_step_batch([g], 2)
        else:
            fq.fciqmc_step(g, 2)
        o.step(2)
    assert_states_equal(fq.fciqmc_export_state(g), o.export())
    assert_stats_equal(fq.fciqmc_iter_stats_get(g), o.stats())
    assert fq.fciqmc_layout(g) == free


def test_asynchronous_blocks_split_crowded_buckets_too():
    """A list that a run alone would split (122 walkers to a bucket of 192) is split at the end of an asynchronous block."""
    fq = _fq()
    sysd = dict(workloads.hubbard_1d(8, 1.0, 4.0), n_beta=3, ref=(0x55, 0x2a))
    s = oracle.system_from_workload(sysd)
    a, b = (x.copy() for x in np.array(s.determinants(), np.uint64).T)
    c = 4.5 * np.random.default_rng(4).choice([-1.0, 1.0], a.size)
    prm = dict(DAMP, tau=0.01, target_walkers=1e9, initiator_threshold=3.0, seed=31)
    g = fq.fciqmc_create(sysd, dict(prm, max_dets=4000))
    o = oracle.Run(s, **prm)
    fq.fciqmc_import_state(g, a, b, c, 0, 4.0)
    o.import_state(a, b, c, 0, 4.0)
    assert fq.fciqmc_layout(g)["buckets"] == 32
    for _ in range(3):
        fq.fciqmc_step_async(g, 4)
        fq.fciqmc_sync(g)
        o.step(4)
        assert fq.fciqmc_layout(g)["buckets"] == 64
    assert_states_equal(fq.fciqmc_export_state(g), o.export())
    assert_stats_equal(fq.fciqmc_iter_stats_get(g), o.stats())


@pytest.mark.parametrize("skip,which", [(0, "keys"), (2, "keys"), (1, "lists")])
def test_create_a_pair_with_one_layout_for_both(monkeypatch, skip, which):
    """The spread layout's keys refused to the first or to the second replica, or its lists to the second: both get
    the tight one."""
    fq = _fq()
    alloc = _Refusing.install(fq, monkeypatch)
    sysd = workloads.small_abinitio(12, 4, 4, seed=9)
    prm = dict(DAMP, tau=0.002, target_walkers=1e4, initiator_threshold=3.0, seed=36, replicas=2)
    lay = fq.fciqmc_layout(fq.fciqmc_create(sysd, prm))
    keys = lay["buckets"] * lay["cap_main"] * 16
    alloc.refuse = (keys if which == "keys" else lay["buckets"] * (lay["cap_main"] + lay["cap_spawn"]) * 48,)
    alloc.skip = skip
    g = fq.fciqmc_create(sysd, prm)
    alloc.refuse = ()
    a, b = (fq.fciqmc_layout(fq.fciqmc_replica(g, r)) for r in (0, 1))
    assert a == b and a["buckets"] < lay["buckets"]
    fq.fciqmc_step(g, 10)
