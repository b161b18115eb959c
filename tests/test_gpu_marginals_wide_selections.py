"""Marginals that leave at most three of the bits above a warp's unselected, beside those that leave more, for every
state size around the two kernels' line, with and without selected low bits, and amplitudes that FP32
squares hold, do not hold, or are 0.  Against exactly rounded sums; tolerance as for the other marginals:
1e-13 relative (complex64 bins are float-float sums of eight amplitudes, and of lanes)."""
import math

import numpy as np
import pytest

from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
@pytest.mark.parametrize("n", [1, 3, 5, 6, 7, 8, 9, 10, 12, 14, 15])
def test_few_unselected_bits(n, dtype):
    rng = np.random.default_rng(n)
    sm = W.SplitMix64(n)
    v = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    v[rng.random(1 << n) < 0.2] = 0
    v[: 1 << (n - 1)] *= np.exp2(-90 * rng.random(1 << (n - 1)))  # half of the state is small
    v = v.astype(np.complex64 if dtype == qs.QS_C64 else np.complex128)
    w = v.astype(np.complex128)
    p = w.real ** 2 + w.imag ** 2
    x = np.arange(1 << n)
    with qs.State(n, dtype) as s:
        qs.qs_copy_from_host(s.h, v)
        ptr, _ = qs.qs_get_buffer(s.h, n)
        for left in range(0, min(n, 5) + 1):
            for low in range(0, 8, 1 if n < 10 else 3):
                q = list(range(low, n))
                q = [q[i] for i in sm.distinct(len(q), max(0, len(q) - left))] if q else []
                if len(q) > 14:
                    continue
                m = np.zeros(1 << n, dtype=int)
                for j, b in enumerate(q):
                    m |= ((x >> b) & 1) << j
                rows = p[np.argsort(m, kind="stable")].reshape(1 << len(q), -1)
                want = np.array([math.fsum(r) for r in rows])
                for got in (s.probs(q), qs.qs_probs_noalloc(ptr, n, dtype, q)):
                    assert np.all(np.abs(got - want) <= 1e-13 * want), q


@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
@pytest.mark.parametrize("n,nq", [(17, 12), (18, 12), (19, 13), (20, 14), (20, 15), (22, 16)])
def test_several_settings_per_step(n, nq, dtype):
    """More settings of the upper bits than resident warps: a step covers two, four or eight of them."""
    rng = np.random.default_rng(n * nq)
    v = (rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)).astype(np.complex64 if dtype == qs.QS_C64 else np.complex128)
    v[rng.integers(0, 1 << n, 1000)] = 1e-30
    w = v.astype(np.complex128)
    p = w.real ** 2 + w.imag ** 2
    x = np.arange(1 << n)
    with qs.State(n, dtype) as s:
        qs.qs_copy_from_host(s.h, v)
        for q in (list(range(n - nq, n)), list(range(n - nq + 1, n)) + [0], list(range(n - 1, n - nq, -1)) + [3]):
            m = np.zeros(1 << n, dtype=int)
            for j, b in enumerate(q):
                m |= ((x >> b) & 1) << j
            want = p[np.argsort(m, kind="stable")].reshape(1 << nq, -1).sum(axis=1)  # (pairwise sums)
            assert np.all(np.abs(s.probs(q) - want) <= 1e-13 * want), q
