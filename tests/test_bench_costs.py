"""Roofline costs that bench.py charges the kernels of its solves (no GPU)."""
import math

import bench


def test_fp64_solves_are_charged_the_modal_operators():
    """The bench's material runs the modal operators in both precisions: FP64
    entries have their operations (45 products and 117 sums per node and load of
    the elastic block, not 576 products), operands of 8 bytes and the FP64 peak."""
    for cls in bench.MODAL_COST:
        flops, nbytes, bound, dtype, dof = bench.class_cost(cls, 0)
        assert (bound, dtype) == ("alu", "f64")
        ref = bench.MODAL_COST["full32" if cls == "full64" else cls]
        assert flops == ref[0] and dof == ref[4]
        assert math.isclose(nbytes, 2 * ref[1], rel_tol=1e-15)
        assert bench.class_cost(cls, 1) == bench.MODAL_COST[cls]
    assert bench.class_cost("elastic0", 0)[0] == 2 * 45 + 117
