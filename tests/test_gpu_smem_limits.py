"""A problem keeps running when another one with smaller buffers, and the same kernels, is created after it: the kernels'
shared-memory limits are raised and never lowered."""
import numpy as np
import pytest

import synthetic
from oracle import kolmogorov as okol
from tests.gpu_util import dev
from tests.rb_util import gpu_problem as rb_problem
from tests.test_gpu_couette import gpu_problem as couette_problem
from tests.test_gpu_kolmogorov import gpu_problem as kol_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _same_before_and_after(large, make_small, x):
    a, b = (torch.zeros_like(x) for _ in range(2))
    large.eval_F(x, a)
    small = make_small()
    large.eval_F(x, b)
    assert torch.equal(a, b)
    small.close()
    large.close()


def test_rayleigh_benard():
    """x transforms of 2 rows per CTA: 147 KB, then 74 KB."""
    p = rb_problem(1536, 8)
    p.set_option(8, 2)
    x = synthetic.random_coeffs((3, 768, 8), seed=1)
    x[:, 0] = x[:, 0].real
    _same_before_and_after(p, lambda: rb_problem(768, 8), dev(x))


def test_couette():
    """y transforms: 222 KB, then 50 KB."""
    p = couette_problem(16, 576, 8)
    _same_before_and_after(p, lambda: couette_problem(16, 128, 8), dev(synthetic.random_coeffs((3, 576, 8, 8), seed=2)))


def test_kolmogorov():
    """98 KB, then 74 KB."""
    x = okol.Kolmogorov(1024, 100.0).project(synthetic.kolmogorov_ic(1024, 3)).ravel()
    _same_before_and_after(kol_problem([1024]), lambda: kol_problem([768]), dev(np.ascontiguousarray(x)))
