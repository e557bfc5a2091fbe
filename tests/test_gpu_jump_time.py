"""The jump time where the root search's estimate of its own error is wrong.

Two cavities, a photon in the first: the output a_1 + a_2 passes through zero and revives, so the loss rate
p(s) falls and rises again.  At this threshold the first trial of the search (the root of the cubic through norm
and rate at both ends) lies where p has the value of the interval's end to 1e-15: the secant of the two
rates is zero, a Newton step of 2 % of the interval seems exact, and is off by 2e-4."""
import numpy as np
import pytest
import scipy.linalg
import scipy.optimize

from paper_1801_04382_gb300 import Problem, cascaded_chain
from paper_1801_04382_gb300.problem import generator_dense

pytestmark = pytest.mark.gpu

DT, R = 1.56, 0.5163244116006138


# FP64: the norm's rounding, 2^-52 K ~ 1e-14, over the rate 0.3 at the jump; FP32: 2^-23 K ~ 7e-6 likewise
@pytest.mark.parametrize("precision,items,tol", [("fp64", 0, 1e-12), ("fp64", 1, 1e-12), ("fp64", 4, 1e-12), ("fp32", 0, 2e-4)])
def test_equal_rates_do_not_end_the_search(precision, items, tol):
    net = cascaded_chain(2, 1, delta=10.0)
    net.psi0 = np.zeros(36, dtype=np.complex128)
    net.psi0[6] = 1.0                                     # |g 1, g 0>
    eps = np.full((2, 2), 0.3)
    U = np.full((1, 1, 13), 1e-3)
    U[0, 0, 0] = R
    args = (net, 2 * DT, 2, 1, eps, np.ones_like(eps), np.full(2, 10.0), U)
    G = generator_dense(*args, eps[:, 0])
    norm2 = lambda s: float(np.linalg.norm(scipy.linalg.expm(-1j * G * s) @ net.psi0) ** 2)
    root = scipy.optimize.brentq(lambda s: norm2(s) - R, 0.0, DT, xtol=1e-15)
    with Problem(*args, precision=precision, items_per_thread=items) as p:
        p.forward()
        rec = p.records()[0]
    assert rec[0][0] == 1 and abs(rec[0][1] - root) <= tol, (rec[0][1], root)
