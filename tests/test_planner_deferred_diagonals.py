"""Plans whose passes leave trailing diagonals to the pass that needs them, replayed on the FP64 oracle:
diagonals of one and several qubits at the end of a pass, before the last pass, and as the whole rest of a
circuit, over slab sizes.  Tolerance as for every plan replay: max |delta amplitude| 1e-12."""
import pytest

from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W
from paper_2406_14084_gb300.workloads import Gate

from test_planner_cpu import check_plan


@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
@pytest.mark.parametrize("slab", [4, 5, 7])
@pytest.mark.parametrize("tail", ["none", "phases", "pairs"])
def test_deferred_diagonals(tail, slab, dtype):
    n = 9
    rest = {"none": [], "phases": [Gate("T", (q,)) for q in range(n)],
            "pairs": [Gate("CP", (q, (q + 4) % n), (), (0.3 + q,)) for q in range(n)]}[tail]
    for gates in (W.qft(n), W.layered(n, 5, 17), W.qaoa_complete(n, 2, 5)):
        check_plan(list(gates) + rest, n, qs.options(slab_bits=slab, seg_bits=1, dtype=dtype))
