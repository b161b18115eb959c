"""Complex64 marginals over six qubits and more hold FP64 accuracy: amplitudes over many orders of magnitude
(also far below where an FP32 square is exact), zeros, and NaN.  Tolerance per bin: eight amplitudes per
float-float sum, each addition within a few 2^-48 of the sum, so 1e-13 relative."""
import numpy as np
import pytest

from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["gauss", "wide", "tiny", "zeros", "nan"])
@pytest.mark.parametrize("n,nq", [(9, 6), (16, 6), (18, 10)])
def test_bins_hold_64_bits(n, nq, kind):
    rng = np.random.default_rng(n + nq)
    v = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    if kind == "wide":
        v *= np.exp2(-90 * rng.random(1 << n))
    elif kind == "tiny":
        v *= 2.0 ** -80
    elif kind == "zeros":
        v *= rng.random(1 << n) < 0.3
    v = v.astype(np.complex64)
    if kind == "nan":
        v[5] = np.nan
    q = W.SplitMix64(n).distinct(n, nq)
    w = v.astype(np.complex128)
    x = np.arange(1 << n)
    m = sum(((x >> b) & 1) << j for j, b in enumerate(q))
    want = np.bincount(m, weights=w.real ** 2 + w.imag ** 2, minlength=1 << nq)
    with qs.State(n, qs.QS_C64) as s:
        qs.qs_copy_from_host(s.h, v)
        got = s.probs(q)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    ok = ~np.isnan(want)
    assert np.all(np.abs(got - want)[ok] <= 1e-13 * want[ok])
