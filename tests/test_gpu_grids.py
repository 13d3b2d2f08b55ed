"""GPU: the fused path on the grids of 54, 72 and 108 points (6 x 9, 12 x 6 and 6 x 18 team plans, whose
elements straddle the bitmap words) against the oracle."""
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


# (N, L, atoms, states): full and ragged bands, one state, more atoms than fit one plane
@pytest.mark.parametrize("N,L,natoms,ns", [(54, 20.0, 9, 5), (54, 16.875, 4, 1), (72, 22.5, 14, 9), (72, 28.0, 3, 2),
                                           (108, 33.75, 20, 3)])
def test_fused_grid(ks, meas, N, L, natoms, ns):
    """H psi (2e-5, as on the other fused grids), the density (1e-5) and one ETRS step with Hartree and
    exchange (5e-5: nine H applications and two densities of FP32 rounding)."""
    cell = inputs.small_cell(L, N, natoms, ns, 700 + N + ns, depth=-3.0)
    ref = ko.Cell(cell)
    q, _ = ko.cholqr(inputs.random_coeffs(700 + N, ns, ref.nG))
    g = ks.Grid(cell, prec="bf16x3")
    psi = torch.from_numpy(q).to("cuda", torch.complex64)
    h = torch.empty_like(psi)
    g.apply_h(psi.data_ptr(), h.data_ptr(), ns)
    torch.cuda.synchronize()
    meas("N=%d H psi" % N, rel(h.cpu().numpy().astype(np.complex128), ko.apply_h(ref, q)), 2e-5)
    g.set_states(q)
    n = torch.empty((N, N, N), dtype=torch.float32, device="cuda")
    g.density(n.data_ptr())
    meas("N=%d density" % N, rel(n.cpu().numpy().astype(float), ko.density(ref, q)), 1e-5)
    norms, energies = g.td_step(0.05, 1, "etrs", True)
    q2, n_ref, e_ref = ko.td_step(ref, q, 0.05, "etrs", True)
    meas("N=%d ETRS state" % N, rel(g.get_states(), q2), 5e-5)
    meas("N=%d ETRS norm and energy" % N, max(abs(norms[0] / n_ref - 1), abs(energies[0] / e_ref - 1)), 1e-4)
    g.close()


@pytest.mark.parametrize("N,L,natoms,ns", [(24, 10.0, 3, 1), (36, 12.0, 3, 9), (54, 20.0, 5, 3), (72, 28.0, 4, 2),
                                           (96, 30.0, 4, 2)])
def test_fp64_planes(ks, meas, N, L, natoms, ns):
    """FP64 H psi and density through whole (y, z) planes: 1e-12, as on every FP64 path."""
    cell = inputs.small_cell(L, N, natoms, ns, 800 + N, depth=-3.0)
    ref = ko.Cell(cell)
    c = inputs.random_coeffs(800 + N, ns, ref.nG)
    g = ks.Grid(cell, prec="fp64")
    psi = torch.from_numpy(c).to("cuda")
    h = torch.full_like(psi, float("nan"))
    g.apply_h(psi.data_ptr(), h.data_ptr(), ns)
    torch.cuda.synchronize()
    meas("N=%d FP64 H psi" % N, rel(h.cpu().numpy(), ko.apply_h(ref, c)), 1e-12)
    g.set_states(c)
    n = torch.empty((N, N, N), dtype=torch.float64, device="cuda")
    g.density(n.data_ptr())
    meas("N=%d FP64 density" % N, rel(n.cpu().numpy(), ko.density(ref, c)), 1e-12)
    g.close()


@pytest.mark.parametrize("ns", [1, 80, 81, 128])
def test_realtime_32_plane_forms(ks, meas, ns):
    """One ETRS step on 32^3 either side of the line between the plane kernel's two forms (bounds of
    test_fused_grid)."""
    test_fused_grid(ks, meas, 32, 10.0, 3, ns)
