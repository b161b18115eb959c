"""Pauli sums of few X masks on both sides of every rule that chooses a shared-tile pass, a Walsh-Hadamard pass or a
plain pass: one mask of 1 to 9 terms, two to five masks of four and of eight terms, few-term masks beside
them, masks wider than a tile, no term at all.  Against the FP64 oracle on the same amplitudes; tolerance as
in test_gpu_readout_kernels.py: 1e-9 n (complex128), 1e-4 n (complex64)."""
import numpy as np
import pytest

import oracle
from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
@pytest.mark.parametrize("n", [3, 12, 15, 16, 17, 18, 20])
def test_routes(n, dtype):
    rng = np.random.default_rng(n)
    v = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    v = (v / np.linalg.norm(v)).astype(np.complex64 if dtype == qs.QS_C64 else np.complex128)
    ref = v.astype(np.complex128)
    sm = W.SplitMix64(n)
    full = (1 << n) - 1

    def mask(xm, terms):
        return [(2.0 * sm.uniform() - 1.0, xm, sm.next_u64() & full) for _ in range(terms)]

    sums = [[]] + [mask(3 << (n - 2), k) for k in (1, 3, 4, 5, 8, 9)] + [mask(full, 2)]
    for masks in (2, 3, 4, 5):
        for terms in (2, 3, 4, 8):
            sums.append([t for m in range(masks) for t in mask((1 + m) << (m % 2) & full, terms)])
    sums.append(sums[-1] + mask(1 << (n - 1), 1) + mask(full, 1) + mask(0, 6))
    sums.append([t for _ in range(70) for t in mask(sm.next_u64() & full, 1)])
    tol = (1e-9 if dtype == qs.QS_C128 else 1e-4) * n
    with qs.State(n, dtype) as s:
        qs.qs_copy_from_host(s.h, v)
        for terms in sums:
            want = oracle.expect_pauli(ref, n, terms) if terms else 0.0
            assert abs(s.expect(terms) - want) <= tol, len(terms)
