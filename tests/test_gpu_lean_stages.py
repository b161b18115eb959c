"""Register stages on the in-place engine against the FP64 oracle, at the sizes and forms where its
records can go wrong: states smaller than one slab and slabs with fewer groups than threads, both stage
widths, rotations on either side of the row exchange (|cos| < |sin|), reflections, X and CX with
controls in registers, in the slab and outside it (controls on flipped bits), tables with conditions
inside and outside the slab, and passes long enough for each program size.  Tolerance as for every
circuit test: max |delta amplitude| 1e-12 (complex128), 1e-5 (complex64)."""
import math

import numpy as np
import pytest

import oracle
from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W
from paper_2406_14084_gb300.workloads import Gate

pytestmark = pytest.mark.gpu

FORMS = [(qs.QS_C64, 0, 1e-5), (qs.QS_C128, 0, 1e-12), (qs.QS_C128, qs.QS_ARITH_DF, 1e-12)]


def check(n, gates, dtype, tol, x0=1, **kw):
    want = oracle.apply_circuit(n, gates, oracle.basis_state(n, x0 % (1 << n)))
    with qs.State(n, dtype) as s:
        s.set_basis(x0 % (1 << n))
        s.apply(gates, qs.options(dtype=dtype, **kw))
        got = s.amplitudes().astype(np.complex128)
    assert np.max(np.abs(got - want)) <= tol


def mixed(n, count, seed):
    rng = W.SplitMix64(seed)
    out = []
    for _ in range(count):
        k = rng.below(10)
        q = rng.distinct(n, 2)
        if k < 2:
            out.append(Gate("RY", (q[0],), (), (rng.angle(),)))
        elif k == 2:
            out.append(Gate("RY", (q[0],), (), (math.pi - 0.01 * rng.uniform(),)))  # |cos| << |sin|
        elif k == 3:
            out.append(Gate("H", (q[0],)))
        elif k == 4:
            out.append(Gate("X", (q[0],)))
        elif k < 7:
            out.append(Gate("CX", (q[0],), (q[1],)))
        elif k == 7:
            out.append(Gate("U3", (q[0],), (), (rng.angle(), rng.angle(), rng.angle())))
        elif k == 8:
            out.append(Gate("CP", tuple(q), (), (rng.angle(),)))
        else:
            out.append(Gate("RZZ", tuple(q), (), (rng.angle(),)))
    return out


@pytest.mark.parametrize("dtype,arith,tol", FORMS)
@pytest.mark.parametrize("n", [4, 5, 6, 9, 12, 13, 14, 17])
def test_mixed_records_over_sizes(n, dtype, arith, tol):
    check(n, mixed(n, 120, 40 + n), dtype, tol, x0=5, arith=arith)


@pytest.mark.parametrize("dtype,arith,tol", FORMS)
@pytest.mark.parametrize("slab,narrow", [(6, 0), (8, 1), (10, 0), (0, 1)])
def test_slab_and_stage_widths(slab, narrow, dtype, arith, tol):
    width = (5 if dtype == qs.QS_C64 else 4) - narrow
    check(15, mixed(15, 160, 7 + slab), dtype, tol, slab_bits=slab, stage_bits=width, arith=arith)


@pytest.mark.parametrize("dtype,arith,tol", FORMS)
@pytest.mark.parametrize("merge", [1, 6, 10])
def test_conditional_tables(merge, dtype, arith, tol):
    n = 15
    check(n, W.qft(n) + W.qaoa_complete(n, 1, 3), dtype, tol, merge_bits=merge, slab_bits=9, arith=arith)


@pytest.mark.parametrize("depth", [2, 30, 150])
def test_program_sizes(depth):
    """One pass of a 13-qubit state: words in 8 KB and 32 KB of parameters, then in device memory."""
    check(13, W.layered(13, depth, 11), qs.QS_C64, 1e-5)


@pytest.mark.parametrize("dtype,arith,tol", FORMS)
@pytest.mark.parametrize("n,slab", [(8, 0), (14, 0), (15, 7), (17, 11)])
def test_separable_tables(n, slab, dtype, arith, tol):
    """Many conditional phases at one place: condition groups inside the slab, outside it and in both."""
    check(n, W.qaoa_complete(n, 2, 3 + n) + W.qft(n), dtype, tol, slab_bits=slab, arith=arith)


@pytest.mark.parametrize("dtype,arith,tol", FORMS)
@pytest.mark.parametrize("k", [7, 8, 10, 11])
def test_wide_diagonals(k, dtype, arith, tol):
    """Diagonals of up to eleven qubits, controls included (ten: the widest that stages take), between rotations, with bits inside and outside the slab."""
    n = 14
    rng = W.SplitMix64(300 + k)
    tables = []
    for i in range(2):
        q = tuple(rng.distinct(n, k))
        tables.append(Gate("DIAG", q[:7], q[7:], (), W.random_diag(7, 70 + i)))
    check(n, mixed(n, 30, k) + tables[:1] + mixed(n, 30, 90 + k) + tables[1:] + mixed(n, 20, 50 + k), dtype, tol, slab_bits=9,
          arith=arith)
