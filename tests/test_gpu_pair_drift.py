"""The columns of Z keep their length over the many rotations that restore T's
triangular blocks, most of them by almost nothing.

A column takes part in about n / 2 swaps here, whose errors in its squared
length are independent and at most a few u = 2^-53 (standard deviation 1.2 u for
a rotation): sqrt(500) 1.2 u = 27 u a column at n = 1000, and 0.85 u for the mean
over the columns.  4 u is five standard deviations; errors with a mean of 0.1 u
and more each add up to well above that.
"""
import numpy as np
import pytest

import schur_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_mean_length_of_columns():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1905_04975_gb300 as g
    n = 1000
    S, T, _, _, sel = si.gen_problem(n, 3, select_frac=0.5, reflectors=1)
    d = [g.to_device(x) for x in (S, T, np.eye(n), np.eye(n))]
    r = g.reorder_gen(*d, sel, window=64, chain=32)
    assert r.status == 0
    for X in d[2:]:
        drift = float((X * X).sum(0).sub(1.0).mean())
        assert abs(drift) <= 4 * 2.0 ** -53, drift
