"""Deep circuits on few qubits, whose thousands of rotations share one register stage, against the FP64 oracle, on the
in-place engine and (with a 4x4 matrix in the stage) on the general one.  Tolerance: that of the other
circuit tests, 1e-5 / 1e-12, which hold some hundred gates, times ten."""
import numpy as np
import pytest

import oracle
from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W
from paper_2406_14084_gb300.workloads import Gate

pytestmark = pytest.mark.gpu

FORMS = [(qs.QS_C64, 0, 1e-4), (qs.QS_C128, 0, 1e-11), (qs.QS_C128, qs.QS_ARITH_DF, 1e-11)]


@pytest.mark.parametrize("dtype,arith,tol", FORMS)
@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("n", [4, 5, 7])
def test_many_rotations_in_one_stage(n, real, general, dtype, arith, tol):
    rng = W.SplitMix64(n)
    gates = [Gate("T", (0,))] + [Gate("RY", (rng.below(min(n, 5)),), (), (rng.angle(),)) for _ in range(2000)] if real \
        else W.layered(n, 400, n)
    if general:
        gates.insert(len(gates) // 2, Gate("UNITARY", (0, 1), (), (), W.random_unitary(2, 8)))
    want = oracle.apply_circuit(n, gates)
    with qs.State(n, dtype) as s:
        s.apply(gates, qs.options(dtype=dtype, arith=arith, fuse_width=0 if real else 2))
        got = s.amplitudes().astype(np.complex128)
    assert np.max(np.abs(got - want)) <= tol
