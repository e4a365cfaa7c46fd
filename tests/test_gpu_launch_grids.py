"""Launch configurations whose launches differ: lists with enough buckets for
every grid, with the last buckets claimed and not, and the autotuner's choice
among launches that are not the same."""
import pytest

import oracle
import workloads
from tests.test_gpu_parity import DAMP, _fq, assert_states_equal, assert_stats_equal
from tests.test_gpu_spawn_edges import _abinitio, _list

pytestmark = pytest.mark.gpu


@pytest.fixture
def fq():
    lib = _fq()
    saved = lib.fciqmc_get_launch_config()
    yield lib
    lib.fciqmc_set_launch_config(saved["spawn"], saved["heavy"], saved["annihilate"])


# 2^16 buckets: 13, 27, 7 and 3 rounds of the spawning warps, 18, 6, 2 and 18 of the annihilation's (from 8 on claimed)
CONFIGS = [(1, 1, 0), (2, 4, 9), (8, 16, 24), (16, 2, 3)]


@pytest.mark.parametrize("cfg", CONFIGS)
@pytest.mark.parametrize("adaptive", [0, 1])
def test_long_list_under_every_grid_bit_exact(fq, cfg, adaptive):
    fq.fciqmc_set_launch_config(*cfg)
    sysd = _abinitio(20, 4, 3, 9)
    prm = dict(DAMP, tau=5e-4, target_walkers=1e9, seed=78, initiator_threshold=3.0, adaptive_shift=adaptive)
    s, a, b, c = _list(sysd, 20, 700, 13)
    g = fq.fciqmc_create(sysd, dict(prm, max_dets=8000000))
    assert fq.fciqmc_layout(g)["buckets"] == 1 << 16
    o = oracle.Run(s, **prm)
    fq.fciqmc_import_state(g, a, b, c, 0, 0.1)
    o.import_state(a, b, c, 0, 0.1)
    fq.fciqmc_step(g, 4)
    o.step(4)
    assert_states_equal(fq.fciqmc_export_state(g), o.export())
    assert_stats_equal(fq.fciqmc_iter_stats_get(g), o.stats(), first=0)


@pytest.mark.parametrize("max_dets,adaptive,spawn,annihilate", [
    (16, 0, {1}, {0}), (8000000, 0, {1, 2, 8, 16}, {0, 9, 24}), (8000000, 1, {1, 2, 4, 8, 16}, {0, 9, 24})])
def test_autotune_does_not_choose_between_equal_launches(fq, max_dets, adaptive, spawn, annihilate):
    """One bucket: every grid is the same.  Many: 4 blocks per SM are the
    spawning's resident wave (3 with the adaptive shift), 3 the annihilation's."""
    prm = dict(DAMP, tau=0.002, target_walkers=100, seed=5, max_dets=max_dets, adaptive_shift=adaptive)
    g = fq.fciqmc_create(workloads.small_abinitio(8, 3, 3, seed=5), prm)
    for _ in range(4):
        got = fq.fciqmc_autotune([g], 2)
        assert got["spawn_blocks_per_sm"] in spawn and got["annihilate_blocks_per_sm"] in annihilate, got
