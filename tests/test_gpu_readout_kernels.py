"""Readout kernels at the edges of their splits, against the FP64 oracle on the same amplitudes.

Marginals: states smaller than one load per lane, selections of low bits only, high bits only and both,
every bin count from the norm to all qubits, one and several loads per warp.  Pauli sums: few-term X
masks inside one tile, spread over several, and wider than any tile, with odd and even numbers of Y,
next to groups that go through the other kernels.  Tolerances as in test_gpu_parity.py: 1e-12 / 1e-6
for probabilities, 1e-9 n / 1e-4 n for expectations."""
import numpy as np
import pytest

import oracle
from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PTOL = {qs.QS_C64: 1e-6, qs.QS_C128: 1e-12}


def state(n, dtype, seed):
    rng = np.random.default_rng(seed)
    v = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    v = (v / np.linalg.norm(v)).astype(np.complex64 if dtype == qs.QS_C64 else np.complex128)
    return v, v.astype(np.complex128)


@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
@pytest.mark.parametrize("n", [1, 2, 4, 5, 6, 7, 9, 12, 16, 19])
def test_marginals_over_sizes_and_selections(n, dtype):
    v, ref = state(n, dtype, n)
    sm = W.SplitMix64(n)
    sets = [[], [0], [n - 1], list(range(min(n, 5))), list(range(n - 1, max(-1, n - 6), -1)), list(range(min(n, 14)))]
    sets += [sm.distinct(n, k) for k in (1, 3, 6, 10, 13) if k <= n]
    with qs.State(n, dtype) as s:
        qs.qs_copy_from_host(s.h, v)
        ptr, _ = qs.qs_get_buffer(s.h, n)
        for q in sets:
            want = oracle.probs(ref, n, q)
            assert np.max(np.abs(s.probs(q) - want)) <= PTOL[dtype], q
            assert np.max(np.abs(qs.qs_probs_noalloc(ptr, n, dtype, q) - want)) <= PTOL[dtype], q


@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
def test_marginals_of_all_qubits(dtype):
    n = 17
    v, ref = state(n, dtype, 3)
    with qs.State(n, dtype) as s:
        qs.qs_copy_from_host(s.h, v)
        order = W.SplitMix64(2).distinct(n, n)
        assert np.max(np.abs(s.probs(order) - oracle.probs(ref, n, order))) <= PTOL[dtype]


@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
@pytest.mark.parametrize("n", [1, 2, 3, 8, 12, 13, 15, 18])
def test_few_term_x_masks(n, dtype):
    v, ref = state(n, dtype, 50 + n)
    sm = W.SplitMix64(n)
    full = (1 << n) - 1
    terms = [(1.0, full, 0), (0.5, full, full), (-0.7, full, 1), (0.3, 0, full)]
    for i in range(n - 1):
        pair = 3 << i
        terms += [(0.4 + 0.1 * i, pair, 0), (0.3, pair, pair), (0.2, 0, pair), (-0.6, pair, 1 << i)]
    for i in range(90):  # scattered masks, many Z bits, some masks more than once
        terms.append((2.0 * sm.uniform() - 1.0, sm.next_u64() & sm.next_u64() & full, sm.next_u64() & full))
    for i in range(20):  # one mask with more terms than a tile takes
        terms.append((0.05 * i, 1 << (n - 1), sm.next_u64() & full))
    tol = (1e-9 if dtype == qs.QS_C128 else 1e-4) * n
    with qs.State(n, dtype) as s:
        qs.qs_copy_from_host(s.h, v)
        for part in (terms, terms[:1], terms[4:12], [t for t in terms if t[1]]):
            want = oracle.expect_pauli(ref, n, part)
            got = s.expect(part)
            assert abs(got.real - want.real) <= tol and abs(got.imag - want.imag) <= tol
