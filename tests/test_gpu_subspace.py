"""GPU: the mixed path's Hermitian eigensolver at the edges of its size ranges (one CTA, one CTA for
the tridiagonalisation only, a cluster of CTAs), through ks_rayleigh_ritz against the oracle."""
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


@pytest.mark.parametrize("n", [1, 2, 16, 17, 33, 127, 128, 129, 161, 255, 256])
def test_rayleigh_ritz_sizes(ks, meas, n):
    """Random block: Ritz values within the FP32 subspace bound (2.5e-5 Ha at 12 states, growing as
    the 2-norm of the entries' rounding, sqrt(n / 12)), orthonormal Ritz states that diagonalise H."""
    cell = inputs.small_cell(10.0, 24, 3, n, 500 + n, depth=-3.0)
    ref = ko.Cell(cell)
    q, _ = ko.cholqr(inputs.random_coeffs(500 + n, n, ref.nG))
    tol = 2.5e-5 * max(1.0, np.sqrt(n / 12.0))
    g = ks.Grid(cell, prec="bf16x3")
    g.set_states(q)
    eps = g.rayleigh_ritz()
    e_ref = ko.rayleigh_ritz(q, ko.apply_h(ref, q))[0]
    meas("n=%d Ritz values" % n, np.max(np.abs(eps - e_ref)), tol)
    x = g.get_states()
    meas("n=%d orthonormality" % n, np.max(np.abs(ko.gram(x) - np.eye(n))), 1e-4)
    h = ko.gram(x, ko.apply_h(ref, x))
    meas("n=%d off-diagonal of the rotated H" % n, np.max(np.abs(h - np.diag(np.diag(h)))), 10 * tol)
    g.close()


@pytest.mark.parametrize("m2max,nshell", [(10, 147), (13, 203), (14, 251)])
def test_degenerate_shells_above_128(ks, meas, m2max, nshell):
    """Free electrons in complete shells, mixed by a random unitary: exactly degenerate levels through
    the cluster tridiagonalisation and the inverse iteration inside clusters."""
    cell = inputs.small_cell(8.0, 24, 0, nshell, 19)
    ref = ko.Cell(cell)
    picks = np.flatnonzero(np.sum(ref.m ** 2, axis=1) <= m2max)
    assert len(picks) == nshell
    c = np.zeros((nshell, ref.nG), complex)
    c[np.arange(nshell), picks] = 1.0
    rng = np.random.default_rng(4)
    Q, _ = np.linalg.qr(rng.normal(size=(nshell, nshell)) + 1j * rng.normal(size=(nshell, nshell)))
    g = ks.Grid(cell, prec="bf16x3")
    g.set_states(Q @ c)
    eps = g.rayleigh_ritz()
    meas("shells of %d states" % nshell, np.max(np.abs(eps - np.sort(0.5 * ref.g2[picks]))), 1e-4)
    x = g.get_states()
    meas("orthonormality, %d states" % nshell, np.max(np.abs(ko.gram(x) - np.eye(nshell))), 1e-4)
    g.close()


@pytest.mark.parametrize("n", [1, 16, 17, 32, 33, 64, 65, 128, 129, 256])
def test_cholqr_sizes(ks, meas, n):
    """CholQR at the edges of the factor's forms (blocked to 16 states; one CTA of three sizes, then a
    cluster): orthonormal to the overlap's precision, the span kept, and a dependent last state
    reported with the states unchanged."""
    cell = inputs.small_cell(10.0, 24, 2, n, 900 + n)
    ref = ko.Cell(cell)
    c = inputs.random_coeffs(900 + n, n, ref.nG)
    g = ks.Grid(cell, prec="bf16x3")
    g.set_states(c)
    g.orthonormalize()
    q = g.get_states()
    meas("n=%d orthonormality" % n, np.max(np.abs(ko.gram(q) - np.eye(n))), 1e-4)   # split-bf16 overlaps
    q_ref, _ = ko.cholqr(c)
    meas("n=%d factor" % n, np.linalg.norm(q - q_ref) / np.linalg.norm(q_ref), 1e-4)
    if n > 1:
        c[n - 1] = 0.5 * c[0]
        g.set_states(c)
        before = g.get_states()
        with pytest.raises(Exception, match="not positive definite"):
            g.orthonormalize()
        assert np.array_equal(g.get_states(), before)
    g.close()
