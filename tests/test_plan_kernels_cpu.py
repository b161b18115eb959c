"""Which kernel a plan's passes run on, as qs_plan_info and the bench's record state it: stages only, a 4x4 matrix in one
pass, remaps, gates without blocking."""
import pytest

import bench
from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W
from paper_2406_14084_gb300.workloads import Gate


@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
@pytest.mark.parametrize("case", ["stages", "matrix", "remaps", "unblocked"])
def test_kernels_of_a_plan(case, dtype):
    n = 16
    gates = W.layered(n, 6, 3)
    if case == "matrix":
        gates = gates + [Gate("UNITARY", (0, n - 1), (), (), W.random_unitary(2, 8))]
    opts = qs.options(dtype=dtype, slab_mode=qs.QS_SLAB_REMAP if case == "remaps" else qs.QS_SLAB_GATHER,
                      blocking=int(case != "unblocked"))
    plan = qs.qs_fuse(gates, n, opts)
    info = qs.qs_plan_info_get(plan)
    qs.qs_plan_destroy(plan)
    label = bench.pass_kernels(info)
    if case == "stages":
        assert info["lean_passes"] == info["passes"] > 0 and label == "lean_pass_kernel"
    elif case == "matrix":
        assert 0 < info["lean_passes"] < info["passes"] and label == "lean_pass_kernel + slab_pass_kernel"
    elif case == "remaps":
        assert info["remaps"] > 0 and "slab_pass_kernel" in label
    else:
        assert info["passes"] == 0 and label == "unblocked_kernel"
