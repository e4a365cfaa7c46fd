"""Runs at the limit of their device memory: what does not fit is refused or
left out, nothing stays allocated for it, and the run goes on as it was."""
import numpy as np
import pytest

import oracle
import workloads
from tests.test_gpu_parity import DAMP, _fq, assert_states_equal, assert_stats_equal

pytestmark = pytest.mark.gpu


def _determinants(norb, na, nb, n, seed):
    rng = np.random.default_rng(seed)
    key = set()
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
