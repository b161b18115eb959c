"""Batches on the in-place stage engine (two CTAs per SM) and beside them batches that hold one pass for
the general engine, against the FP64 oracle: states smaller than a warp, a slab and the CTA, slabs of few
amplitudes, runs of several slabs, both stage widths, one and two CTAs per SM.  Tolerance on <H> as for
every batch: 1e-4 n."""
import numpy as np
import pytest

import oracle
from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 4, 5, 6, 7, 8, 9, 12, 13, 14, 17]


def run(circuits, **kw):
    n = np.array([c[0] for c in circuits])
    want = [oracle.expect_pauli(oracle.apply_circuit(k, g), k, W.zz_chain_hamiltonian(k)).real for k, g in circuits]
    b = qs.qs_batch_create(circuits, qs.options(dtype=qs.QS_C64, **kw))
    try:
        got = qs.qs_apply_batch(b, W.zz_chain_hamiltonian(int(n.max())), len(circuits))
    finally:
        qs.qs_batch_destroy(b)
    assert np.all(np.abs(got - want) <= 1e-4 * n), np.max(np.abs(got - want))


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("width", [5, 4])
@pytest.mark.parametrize("slab", [0, 6, 9])
def test_sizes_and_widths(slab, width, general):
    circuits = [(n, W.vqe_circuit(n, 3, 60 + n)) for n in SIZES]
    if general:
        circuits.insert(4, (7, [W.Gate("UNITARY", (0, 5), (), (), W.random_unitary(2, 8))] + W.vqe_circuit(7, 2, 3)))
    run(circuits, slab_bits=slab, stage_bits=width)


def test_two_ctas_per_sm():
    run([(n, W.vqe_circuit(n, 2, 90 + n)) for n in [17, 18, 16] * 6])
