"""Complex64 marginals of up to five qubits and the allocation-free entry hold FP64 accuracy for amplitudes whose FP32
squares underflow, as marginals of six qubits and more do (test_gpu_marginals_precision.py).  Tolerance per
bin as there: 1e-13 relative, against exactly rounded sums."""
import math

import numpy as np
import pytest

from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["gauss", "wide", "tiny", "zeros"])
@pytest.mark.parametrize("nq", [0, 1, 3, 5, 7])
@pytest.mark.parametrize("n", [5, 8, 14, 19])
def test_bins_hold_64_bits(n, nq, kind):
    if nq > n:
        pytest.skip("more selected qubits than qubits")
    rng = np.random.default_rng(100 * n + nq)
    v = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    if kind == "wide":
        v *= np.exp2(-90 * rng.random(1 << n))
    elif kind == "tiny":
        v *= 2.0 ** -80
    elif kind == "zeros":
        v *= rng.random(1 << n) < 0.3
    v = v.astype(np.complex64)
    w = v.astype(np.complex128)
    for q in (W.SplitMix64(n).distinct(n, nq), list(range(nq)), list(range(n - nq, n))):
        x = np.arange(1 << n)
        m = sum(((x >> b) & 1) << j for j, b in enumerate(q)) if q else np.zeros(1 << n, dtype=int)
        p = (w.real ** 2 + w.imag ** 2)[np.argsort(m, kind="stable")].reshape(1 << nq, -1)
        want = np.array([math.fsum(row) for row in p])
        with qs.State(n, qs.QS_C64) as s:
            qs.qs_copy_from_host(s.h, v)
            ptr, _ = qs.qs_get_buffer(s.h, n)
            for got in (s.probs(q), qs.qs_probs_noalloc(ptr, n, qs.QS_C64, q)):
                assert np.all(np.abs(got - want) <= 1e-13 * want), q
