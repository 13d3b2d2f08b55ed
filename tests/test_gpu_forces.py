"""GPU: forces through planes on the grids with team transforms, the plain FP32 path with atoms, and their
edges, against the oracle."""
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


def smooth_block(ref, seed, ns):
    """Orthonormal states whose spectra fall off at graded rates."""
    t = 0.7 + 3.0 * np.arange(ns)[:, None] / ns
    return ko.cholqr(inputs.random_coeffs(seed, ns, ref.nG) * np.exp(-0.25 * ref.g2[None, :] / t))[0]


# Bound of the mixed forces, 1e-5 of the largest: gradient densities of FP32 transforms (a few 2^-24 of their
# largest value), which a force's sums cancel by a factor of ten and more.
# (N, L, atoms, projectors, states): one state; chunks of states (16 at most) full and ragged; covered points
# whose bitmap words the plan's radix divides (32, 96) and straddles (54, 72, 108); one projector per atom
@pytest.mark.parametrize("N,L,natoms,nproj,ns", [(32, 10.0, 3, 4, 1), (32, 13.0, 5, 4, 19), (48, 15.0, 4, 1, 16),
                                                 (54, 16.875, 6, 4, 17), (54, 22.5, 3, 1, 1), (64, 20.0, 4, 4, 35),
                                                 (72, 22.5, 7, 4, 5), (72, 30.0, 3, 1, 18), (96, 30.0, 9, 4, 3),
                                                 (108, 33.75, 12, 4, 2), (108, 33.75, 3, 1, 17), (128, 40.0, 6, 4, 2)])
def test_forces_through_planes(ks, meas, N, L, natoms, nproj, ns):
    cell = inputs.small_cell(L, N, natoms, ns, 81 + N, depth=-3.0, nproj=nproj)
    cell["pos"][0] = [0.05, L - 0.05, 0.5 * L]                       # spheres and boxes across the faces
    occ = 2.0 - 1.7 * np.arange(ns) / ns
    ref = ko.Cell(dict(cell, occ=occ))
    q = smooth_block(ref, 82, ns)
    g = ks.Grid(cell, prec="bf16x3", occ=occ)
    g.set_states(q)
    F_ref = ko.forces(ref, q)
    meas("N=%d, %d states" % (N, ns), np.max(np.abs(g.forces() - F_ref)), 1e-5 * np.max(np.abs(F_ref)))
    assert np.array_equal(g.forces(), g.forces())
    g.close()


def test_forces_of_two_chunks_of_grids(ks, meas):
    """130 states of 128^3: more than the 2 GB of state grids hold at once (128).  Four states on either side of
    the line are occupied."""
    ns, pick = 130, [0, 127, 128, 129]
    cell = inputs.small_cell(40.0, 128, 4, ns, 83, depth=-3.0)
    occ = np.zeros(ns)
    occ[pick] = [2.0, 1.0, 0.5, 1.5]
    ref = ko.Cell(dict(cell, nstates=4, occ=occ[pick]))
    q = smooth_block(ref, 84, 4)
    c = np.zeros((ns, ref.nG), complex)
    c[pick] = q
    g = ks.Grid(cell, prec="bf16x3", occ=occ)
    g.set_states(c)
    F_ref = ko.forces(ref, q)
    meas("two chunks", np.max(np.abs(g.forces() - F_ref)), 1e-5 * np.max(np.abs(F_ref)))
    g.close()


def test_forces_where_the_atoms_first_cover_no_point(ks, meas):
    """Projector spheres between the grid points, then moved onto them: the forces change from full grids to
    planes in the life of a handle."""
    N, L = 32, 10.0
    h = L / N
    cell = dict(inputs.small_cell(L, N, 2, 3, 85, depth=-3.0), proj_rc=0.4 * h, proj_sigma=0.2 * h)
    cell["pos"] = (np.array([[5, 9, 20], [17, 2, 11]]) + 0.5) * h
    ref = ko.Cell(cell)
    q = smooth_block(ref, 86, 3)
    g = ks.Grid(cell, prec="bf16x3")
    g.set_states(q)
    F_ref = ko.forces(ref, q)
    meas("no covered point", np.max(np.abs(g.forces() - F_ref)), 1e-5 * np.max(np.abs(F_ref)))
    moved = cell["pos"] + 0.4 * h
    g.set_positions(moved)
    F_ref = ko.forces(ko.Cell(dict(cell, pos=moved)), q)
    meas("covered points", np.max(np.abs(g.forces() - F_ref)), 1e-5 * np.max(np.abs(F_ref)))
    g.close()


@pytest.mark.parametrize("N,L,nproj", [(12, 4.5, 4), (16, 5.0, 4), (16, 6.0, 1)])
def test_plain_fp32_path_with_atoms(ks, meas, N, L, nproj):
    """Grids without plane kernels, with projectors: H psi (2e-5), density (1e-5), forces (1e-5) and one ETRS
    step (5e-5), the bounds of the fused grids."""
    cell = inputs.small_cell(L, N, 2, 5, 87, depth=-3.0, nproj=nproj)
    ref = ko.Cell(cell)
    q = smooth_block(ref, 88, 5)
    g = ks.Grid(cell, prec="bf16x3")
    psi = torch.from_numpy(q).to("cuda", torch.complex64)
    h = torch.full_like(psi, float("nan"))
    g.apply_h(psi.data_ptr(), h.data_ptr(), 5)
    torch.cuda.synchronize()
    meas("N=%d H psi" % N, rel(h.cpu().numpy().astype(complex), ko.apply_h(ref, q)), 2e-5)
    g.set_states(q)
    n = torch.empty((N, N, N), dtype=torch.float32, device="cuda")
    g.density(n.data_ptr())
    meas("N=%d density" % N, rel(n.cpu().numpy().astype(float), ko.density(ref, q)), 1e-5)
    F_ref = ko.forces(ref, q)
    meas("N=%d forces" % N, np.max(np.abs(g.forces() - F_ref)), 1e-5 * np.max(np.abs(F_ref)))
    g.td_step(0.05, 1, "etrs", True)
    meas("N=%d ETRS state" % N, rel(g.get_states(), ko.td_step(ref, q, 0.05, "etrs", True)[0]), 5e-5)
    g.close()
