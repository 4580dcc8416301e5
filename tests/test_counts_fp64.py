"""The count of FP64 instructions of the present two-center passes, on cases counted by hand."""
import numpy as np

from paper_1701_06588_gb300 import counts

CO, ERFC, ERF, OV = (counts.OP_COULOMB, 0.0), (counts.OP_ERFC, 0.3), (counts.OP_ERF, 0.3), (counts.OP_OVERLAP, 0.0)


def _count(la, lb, ka, kb, ops, **kw):
    sh = dict(l=np.array([la, lb]), nprim=np.array([ka, kb]))
    return counts.workload_fp64_instructions(sh, np.array([0]), np.array([1]), ops, **kw)


def test_hand_counted_pairs():
    # (s|s): R^2 6; per operator F_0 1 and its far part 1, p F 1, X 1, element 1
    assert _count(0, 0, 1, 1, [CO]) == 1 + 6 + 5
    assert _count(0, 0, 3, 2, [CO, ERFC]) == 2 * 6 + 1 + 6 + 2 * 5
    assert _count(0, 0, 3, 2, [CO], n_far=[4]) == 6 + 6 + 5
    # (p|s): C, S 4, one step of p_{L,M}; F 2, products 2, X 1 + element 1 for m = 0, X 1 + elements 2 for |m| = 1
    assert _count(1, 0, 2, 2, [OV]) == 4 + 1 + 6 + (4 + 3) + (2 + 2 + 2 + 3)
    # (p|p): orders 2; C, S 8, steps 9; F 5, products 4, elements (0,0): 2 + 1, (0,1), (1,0): 1 + 2, (1,1): 2 + 1 + 6
    assert _count(1, 1, 1, 1, [ERF]) == 2 + 2 + 6 + 17 + (5 + 4 + 3 + 3 + 3 + 9)


def test_shared_sums_and_double_float_classes():
    assert _count(2, 2, 4, 4, [ERF, ERFC]) < _count(2, 2, 4, 4, [ERF, (counts.OP_ERFC, 0.2)])
    assert _count(2, 2, 4, 4, [CO], mixed=True) < _count(2, 2, 4, 4, [CO])
    assert _count(1, 4, 4, 4, [CO], mixed=True) == _count(1, 4, 4, 4, [CO])
    assert _count(4, 4, 4, 4, [CO], mixed=True) == _count(4, 4, 4, 4, [CO])
