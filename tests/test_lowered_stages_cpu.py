"""Records of the in-place stage engine against the sub-ops that they stand for, executed on the host
(lowered_stages.cpp) with the records' numbers rounded as the device holds them: conditional phases on
every pair of qubits, so that separable records appear, with X gates and wide rotations that hold register
bits flipped, and diagonals and matrices that are not unitary.

Tolerance, relative to the largest amplitude of a group: a record rounds its numbers once, at most a few
hundred records per stage, errors adding at random: 1e-5 (FP32), 1e-12 (double-float, 48 bits), 1e-13
(FP64)."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W
from paper_2406_14084_gb300.workloads import Gate

HERE = os.path.dirname(os.path.abspath(__file__))
FORMS = {"c64": (dict(dtype=qs.QS_C64), 1e-5), "c128": (dict(dtype=qs.QS_C128), 1e-13),
         "df": (dict(dtype=qs.QS_C128, arith=qs.QS_ARITH_DF), 1e-12)}


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    qs.lib()
    so, lib = qs.library_path(), str(tmp_path_factory.mktemp("lowered") / "lowered_stages.so")
    pkg = os.path.dirname(os.path.abspath(qs.__file__))
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(pkg, "..", "include"), "-I",
                    os.path.join(pkg, "csrc"), os.path.join(HERE, "lowered_stages.cpp"), so, "-o", lib,
                    "-Wl,-rpath," + os.path.dirname(so)], check=True)
    dll = ctypes.CDLL(lib)
    dll.lowered_difference.restype = ctypes.c_double
    return dll


def call(fn, numbers, gates, n, **kw):
    arr, keep = qs.marshal_gates(gates)
    opts, out = qs.options(**kw), (ctypes.c_int64 * numbers)()
    rc = fn(arr, ctypes.c_size_t(len(gates)), n, ctypes.byref(opts), out)
    del keep
    assert rc >= 0
    return rc, tuple(out)


@pytest.fixture(scope="module")
def compare(host):
    def run(gates, n, **kw):
        """Largest difference and (stages, lowered stages, separable records, records)."""
        return call(host.lowered_difference, 4, gates, n, **kw)

    return run


def pairs(n, seed, diagonals):
    """Controlled phases on every pair between X gates, rotations and the given one-qubit diagonals."""
    rng = W.SplitMix64(seed)
    out = [Gate("H", (q,)) for q in range(n)] + [Gate("X", (q,)) for q in range(n) if rng.below(2)]
    for a in range(n):
        out += [Gate("CP", (a, b), (), (rng.angle(),)) for b in range(a + 1, n)]
        if rng.below(3) == 0:
            out.append(Gate("X", (a,)))
        if rng.below(4) == 0:
            out.append(Gate("RY", (rng.below(n),), (), (math.pi - 0.01 * rng.uniform(),)))
        if diagonals and rng.below(3) == 0:
            out.append(Gate("DIAG", (rng.below(n),), (), (), np.array(diagonals[rng.below(len(diagonals))], dtype=complex)))
    return out


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("fuse", [0, 2])
@pytest.mark.parametrize("diagonals", [None, ((1, 0),), ((0, 1), (1, 0)), ((1, 1e-3), (0.5, 1)), ((0, 0),)],
                         ids=["unitary", "zero", "zeros", "moduli", "null"])
def test_separable_records_with_any_diagonal(compare, diagonals, fuse, form):
    opts, tol = FORMS[form]
    separable = 0
    for seed in range(24):
        n = (10, 13, 16)[seed % 3]
        worst, count = compare(pairs(n, seed, diagonals), n, fuse_width=fuse, slab_bits=(0, 9)[seed % 2], **opts)
        assert worst <= tol, (seed, worst)
        separable += count[2]
    assert separable or form == "c128"  # FP64 tables take more conditions and mostly stay cheaper


@pytest.mark.parametrize("form", ["c128", "df"])
@pytest.mark.parametrize("n", [15, 16, 18, 20, 22])
def test_separable_records_from_fused_tables(compare, n, form):
    """Two QAOA rounds on the complete graph: separable records out of diagonals of up to ten qubits, each the
    product of some 45 phases.  An entry is off by sqrt(45) roundings of 2^-53 (7e-16); ratios of entries keep
    that, 20 diagonals a stage add at random, the worst of a few hundred amplitudes is at three to four
    sigma: 1.2e-14, and 2^-48 twice more in double-float."""
    tol = 1.2e-14 if form == "c128" else 2e-14
    for seed in range(2):
        worst, count = compare(W.qaoa_complete(n, 2, seed), n, **FORMS[form][0])
        assert count[2] > 0
        assert worst <= tol, (seed, worst)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("n", [4, 5, 6])
@pytest.mark.parametrize("real", [False, True])
def test_long_stages(compare, real, n, form):
    """Thousands of rotations in one stage: their common factor, below 2^-126, has to stay within FP32."""
    opts, tol = FORMS[form]
    rng = W.SplitMix64(n)
    gates = [Gate("T", (0,))] + [Gate("RY", (rng.below(n),), (), (rng.angle(),)) for _ in range(3000)] if real \
        else W.layered(n, 500, n)
    worst, _ = compare(gates, n, fuse_width=0 if real else 2, **opts)
    assert worst <= tol * 10  # ten times the records of the other tests


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("merge", [1, 2, 4, 6, 8])
def test_merge_bits_limits_what_is_put_together(host, merge, form):
    """Tables and separable groups read at most merge_bits conditions, unless one diagonal alone reads more."""
    for gates, n in ((W.qft(16), 16), (pairs(13, 3, None), 13), (W.qaoa_complete(14, 2, 1), 14)):
        for fuse in (0, 2):
            _, most = call(host.lowered_widths, 5, gates, n, merge_bits=merge, fuse_width=fuse, slab_bits=9, **FORMS[form][0])
            assert max(most[0], most[1]) <= max(merge, most[2])


@pytest.mark.parametrize("form", FORMS)
def test_kept_matrices_stay_on_the_general_engine(host, form):
    """factor = 1 keeps full 2x2 matrices and euler = 1 complex ones: no stage with one is lowered."""
    opts = FORMS[form][0]
    _, on = call(host.lowered_widths, 5, W.layered(12, 4, 3), 12, fuse_width=1, **opts)
    assert on[3] == on[4] > 0
    _, off = call(host.lowered_widths, 5, W.layered(12, 4, 3), 12, fuse_width=1, factor=1, **opts)
    assert off[3] == 0 < off[4]
    _, off = call(host.lowered_widths, 5, W.layered(12, 4, 3), 12, fuse_width=1, euler=1, **opts)
    assert off[3] < off[4]


def test_batch_circuits_lower_throughout(compare):
    """The circuits of test_gpu_batch_lean_sizes.py have register stages only, and all of them are lowered."""
    import test_gpu_batch_lean_sizes as B

    for slab, width in B.CASES:
        for n, gates in B.circuits_of(width):
            opts = dict(dtype=qs.QS_C64, slab_bits=slab, stage_bits=width)
            _, count = compare(gates, n, **opts)
            assert 0 < count[0] == count[1], (n, slab, width)
            plan = qs.qs_fuse(gates, n, qs.options(**opts))
            info = qs.qs_plan_info_get(plan)
            qs.qs_plan_destroy(plan)
            assert info["smem_ops"] == 0, (n, slab, width)


@pytest.mark.parametrize("form", ["c128", "df"])
@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("off", [1e-15, 5e-14, 8e-13])
def test_nearly_unitary_matrices(compare, off, real, form):
    """A 2x2 matrix whose last entry is off the unitary one is applied as it is given, however little that is."""
    opts, tol = FORMS[form]
    rng = W.SplitMix64(7)
    gates = []
    for i in range(40):
        a, b, c = rng.angle(), 0.0 if real else rng.angle(), 0.0 if real else rng.angle()
        u = np.array([[math.cos(a), -np.exp(1j * c) * math.sin(a)],
                      [np.exp(1j * b) * math.sin(a), np.exp(1j * (b + c)) * math.cos(a)]])
        u[1, 1] *= 1 + off
        gates.append(Gate("UNITARY", (rng.below(6),), (), (), u))
    worst, _ = compare(gates, 6, fuse_width=0, **opts)
    assert worst <= (1e-13 if form == "c128" else tol * 0.1)
