"""Slabs with fewer register groups than threads, where whole warps have none, beside full ones, alone and in passes
with a 4x4 matrix (general kernel), against the FP64 oracle: one group, less than a warp of them, one warp,
half of the threads, all.  Tolerance as for every circuit test: 1e-12 (complex128), 1e-5 (complex64)."""
import numpy as np
import pytest

import oracle
from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W
from paper_2406_14084_gb300.workloads import Gate

pytestmark = pytest.mark.gpu

FORMS = [(qs.QS_C64, 0, 1e-5), (qs.QS_C128, 0, 1e-12), (qs.QS_C128, qs.QS_ARITH_DF, 1e-12)]


@pytest.mark.parametrize("dtype,arith,tol", FORMS)
@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("narrow", [0, 1])
@pytest.mark.parametrize("n,slab", [(4, 0), (5, 0), (9, 0), (11, 0), (13, 4), (13, 5), (13, 9), (14, 11), (14, 12)])
def test_warps_without_groups(n, slab, narrow, general, dtype, arith, tol):
    gates = W.layered(n, 3, n + slab) + [Gate("CX", (0,), (n - 1,))]
    if general:
        gates += [Gate("UNITARY", (0, n - 2), (), (), W.random_unitary(2, 8))] + W.layered(n, 2, 5)
    want = oracle.apply_circuit(n, gates, oracle.basis_state(n, 5))
    with qs.State(n, dtype) as s:
        s.set_basis(5)
        s.apply(gates, qs.options(dtype=dtype, arith=arith, slab_bits=slab,
                                  stage_bits=(5 if dtype == qs.QS_C64 else 4) - narrow))
        got = s.amplitudes().astype(np.complex128)
    assert np.max(np.abs(got - want)) <= tol
