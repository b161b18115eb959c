"""Batches that run on the in-place stage engine throughout (test_lowered_stages_cpu.py checks that their passes all
lower), from states of one register group up: slabs of 4 to 13 bits, states smaller than a warp, than the CTA
and larger than a slab, both stage widths, circuits without gates beside them.  Against the FP64 oracle;
tolerance on <H> as for every batch: 1e-4 n."""
import numpy as np
import pytest

import oracle
from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W

SIZES = [4, 5, 6, 7, 8, 9, 10, 12, 13, 14, 15, 17]


def circuits_of(width):
    return [(n, W.vqe_circuit(n, 3, 160 + n)) for n in SIZES if n >= width]


CASES = [(slab, width) for width in (4, 5) for slab in (0, 5, 6, 7, 8, 9, 11) if slab == 0 or slab >= width]


@pytest.mark.gpu
@pytest.mark.parametrize("slab,width", CASES)
@pytest.mark.parametrize("empty", [False, True])
def test_slab_bits_and_widths(slab, width, empty):
    circuits = circuits_of(width)
    if empty:
        circuits = [(3, [])] + circuits + [(9, [])]
    n = np.array([c[0] for c in circuits])
    want = [oracle.expect_pauli(oracle.apply_circuit(k, g), k, W.zz_chain_hamiltonian(k)).real for k, g in circuits]
    b = qs.qs_batch_create(circuits, qs.options(dtype=qs.QS_C64, slab_bits=slab, stage_bits=width))
    try:
        for _ in range(2):
            got = qs.qs_apply_batch(b, W.zz_chain_hamiltonian(int(n.max())), len(circuits))
            assert np.all(np.abs(got - want) <= 1e-4 * n), np.max(np.abs(got - want))
    finally:
        qs.qs_batch_destroy(b)
