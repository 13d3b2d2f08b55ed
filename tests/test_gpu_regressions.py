"""GPU: inputs at the edges of what the entry points take, each of which once gave a wrong result, an error
or a needless cost; against the oracle."""
import numpy as np
import pytest

from oracle import ks_oracle as ko
from paper_2106_03872_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ks():
    from paper_2106_03872_gb300 import ks as mod
    mod.load()
    assert torch.cuda.is_available()
    return mod


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("bf16x3", 1e-4)])
def test_teter_step_of_negative_length(ks, meas, prec, tol):
    """A coupling D far below zero makes every step length 1 / (T + span V + D) negative (T <= 20 Ha, the
    cutoff): the states move all the same.  Bounds: those of the plain parity tests."""
    cell = dict(inputs.small_cell(10.0, 24, 1, 3, 71), proj_D=-60.0)
    ref = ko.Cell(cell)
    c = inputs.random_coeffs(71, 3, ref.nG)
    g = ks.Grid(cell, prec=prec)
    g.set_states(c)
    g.block_iteration(1, precond="teter")
    meas("states after a step of negative length", rel(g.get_states(), ko.block_iteration_teter(ref, c, 1)[1]), tol)
    g.close()
