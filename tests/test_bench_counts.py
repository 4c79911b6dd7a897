"""What bench.py reports of the column-sum pass's own operations: the ordered form's count, 48N of
the general form's 54N that the library's kernel timing gives, so that no utilisation is
reported from additions that were not issued."""
import types

import bench


def test_issued_operations_are_the_ordered_forms():
    bn = types.SimpleNamespace(alg_flops_pass=1.0, candk_pass=1.0)
    r = bench.roofline_mixed(bn, {"sums": (1, 1000.0, 54e12)}, None)
    assert abs(r["achieved_issued"] - 48.0) < 1e-9
    assert abs(r["frac_issued"] - 48e12 / (152 * 128 * 2 * 2070e6)) < 1e-3
    assert abs(bench.ISSUED_SUMS_GRAD * 103 - 91) < 1e-9
