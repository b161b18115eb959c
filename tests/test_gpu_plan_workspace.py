"""Plans that live within one call share a device workspace owned by the state: calls of growing and
shrinking plan sizes, with remaps and layout changes between them, against the FP64 oracle
(1e-12 for complex128, 1e-5 for complex64)."""
import numpy as np
import pytest

import oracle
from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,tol", [(qs.QS_C64, 1e-5), (qs.QS_C128, 1e-12)])
def test_repeated_calls_of_changing_plan_size(dtype, tol):
    n = 14
    want = oracle.basis_state(n, 3)
    with qs.State(n, dtype) as s:
        s.set_basis(3)
        for i, gates in enumerate((W.random_circuit(n, 5, 1), W.layered(n, 6, 2), W.qft(n), W.random_circuit(n, 60, 4),
                                   W.random_circuit(n, 1, 5), W.qaoa_complete(n, 2, 6))):
            s.apply(gates, qs.options(dtype=dtype))
            want = oracle.apply_circuit(n, gates, want)
            if i % 2:
                qs.qs_remap(s.h, [0, 2], [n - 1, 7])  # a layout the next readout has to undo
        got = s.amplitudes().astype(np.complex128)
    assert np.max(np.abs(got - want)) <= tol
