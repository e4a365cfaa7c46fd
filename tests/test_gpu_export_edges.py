"""Export and import at the edges of the sort and of the H_ii kernels.

The export sorts by the ranks of the occupation words with 8-bit digits in
tiles of 4096 keys: list lengths around a tile, rank widths below, at and above
64 bits, words with no choice at all, orbital 63 in use.  The import computes
H_ii by eight lanes per determinant, or by one where there is a determinant
for every thread of the GPU.  Order, amplitudes and flags are compared with
numpy's sort of the input, H_ii with the oracle's exact sums, bit for bit.
"""
import numpy as np
import pytest

import oracle
import workloads
from tests.test_gpu_parity import _fq, bits

pytestmark = pytest.mark.gpu


def _words(rng, norb, k, n):
    order = np.argsort(rng.random((n, norb)), axis=1)[:, :k]
    w = np.zeros(n, np.uint64)
    for j in range(k):
        w |= np.uint64(1) << order[:, j].astype(np.uint64)
    return w


def _unique(a, b):
    key = np.unique(np.stack([a, b], 1), axis=0)
    return key[:, 0].copy(), key[:, 1].copy()


@pytest.mark.parametrize("norb,na,nb,n", [
    (8, 4, 4, 4095), (50, 10, 10, 4096), (64, 16, 16, 4097), (64, 16, 16, 20001), (64, 2, 0, 2016), (33, 1, 0, 33),
    (64, 64, 0, 1), (40, 20, 3, 9000), (20, 6, 6, 700), (24, 6, 6, 160001), (64, 3, 20, 170003),
])
def test_imported_list_comes_back_sorted_with_exact_diagonals(norb, na, nb, n):
    fq = _fq()
    rng = np.random.default_rng(norb + n)
    h, eri = workloads.synthetic_abinitio(norb, 6, norb)
    sysd = dict(kind="abinitio", norb=norb, n_alpha=na, n_beta=nb, h1=h, eri=eri, ecore=0.0)
    s = oracle.system_from_workload(sysd)
    a, b = _unique(_words(rng, norb, na, n), _words(rng, norb, nb, n))
    ra, rb = (np.uint64(x) for x in s.ref)
    if not ((a == ra) & (b == rb)).any():
        a, b = np.append(a, ra), np.append(b, rb)
    p = rng.permutation(a.size)
    a, b = a[p], b[p]
    c = rng.normal(0.0, 3.0, a.size)
    g = fq.fciqmc_create(sysd, dict(tau=1e-4, seed=1))
    fq.fciqmc_import_state(g, a, b, c, 0, 0.0)
    got = fq.fciqmc_export_state(g)
    o = np.lexsort((b, a))
    np.testing.assert_array_equal(got["alpha"], a[o])
    np.testing.assert_array_equal(got["beta"], b[o])
    np.testing.assert_array_equal(bits(got["c"]), bits(c[o]))
    np.testing.assert_array_equal(got["flags"], ((a[o] == ra) & (b[o] == rb)).astype(np.int32))
    for k in np.unique(np.concatenate([[0, a.size - 1], rng.integers(0, a.size, 300)])):
        want = s.hdiag_rel(int(got["alpha"][k]), int(got["beta"][k]))
        assert bits(np.array([got["hdiag"][k]]))[0] == bits(np.array([want]))[0], k


@pytest.mark.parametrize("norb,na,nb,n", [(64, 32, 32, 5000), (64, 31, 30, 4097), (63, 31, 32, 5003)])
def test_ranks_of_more_than_120_bits(norb, na, nb, n):
    """Half-filled words of 63 and 64 orbitals: 120 and 122 bits of rank; with 122 the low word is used whole."""
    test_imported_list_comes_back_sorted_with_exact_diagonals(norb, na, nb, n)
