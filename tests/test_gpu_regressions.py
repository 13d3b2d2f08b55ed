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


@pytest.mark.parametrize("N,L", [(54, 16.875), (96, 30.0)])
def test_first_call_under_capture(ks, meas, N, L):
    """H psi and the density captured into a graph by the first calls of their size class (130 states: no
    other test's): nothing is timed on the capturing stream.  Bounds of the fused grids' parity tests."""
    ns = 130
    cell = inputs.small_cell(L, N, 2, ns, 72, depth=-3.0)
    g = ks.Grid(cell, prec="bf16x3")
    c = inputs.random_coeffs(72, 2, g.nG)
    ref = ko.Cell(cell)
    psi = torch.from_numpy(c).to("cuda", torch.complex64).repeat(ns // 2, 1)
    h, n = torch.zeros_like(psi), torch.zeros((N, N, N), dtype=torch.float32, device="cuda")
    g.set_states(np.tile(c, (ns // 2, 1)))
    torch.cuda.synchronize()
    graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=s):
        g.apply_h(psi.data_ptr(), h.data_ptr(), ns, stream=s)
        g.density(n.data_ptr(), stream=s)
    for _ in range(2):
        h.zero_()
        graph.replay()
        torch.cuda.synchronize()
    got = h.cpu().numpy().astype(np.complex128)
    expect = ko.apply_h(ref, c)
    for k in (0, 1, ns - 2, ns - 1):
        meas("N=%d captured H psi" % N, rel(got[k], expect[k % 2]), 2e-5)
    meas("N=%d captured density" % N, rel(n.cpu().numpy().astype(float), ns // 2 * ko.density(ref, c)), 1e-5)
    g.close()


@pytest.mark.parametrize("width", [4e7, 1e11, np.inf])
def test_forces_of_a_flat_local_potential(ks, meas, width):
    """Widths whose box of grid points overflowed an integer: V_loc is constant, so the local sums cancel to
    the rounding of V times the gradient density (FP64 1e-12; FP32 gradients of a few 6e-8: 1e-6)."""
    cell = dict(inputs.small_cell(10.0, 24, 2, 3, 73, depth=-0.1), vloc_width=width)
    ref = ko.Cell(cell)
    q, _ = ko.cholqr(inputs.random_coeffs(73, 3, ref.nG))
    F_ref = ko.forces(ref, q)
    scale = np.max(np.abs(F_ref)) + np.max(np.abs(ref.vloc))
    for prec, tol in (("fp64", 1e-12), ("bf16x3", 1e-6)):
        g = ks.Grid(cell, prec=prec)
        g.set_states(q)
        meas("width %g, %s" % (width, prec), np.max(np.abs(g.forces() - F_ref)), tol * scale)
        g.close()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("bf16x3", 1e-4)])
@pytest.mark.parametrize("N,L,face", [(48, 15.0, 0.1), (64, 20.0, 19.9), (72, 30.0, 0.0)])
def test_local_force_boxes(ks, meas, prec, tol, N, L, face):
    """The local force over boxes that are the whole grid (48 points) or a part of it that wraps around the
    cell's faces, with occupations of every size.  Bounds of the force parity tests."""
    cell = inputs.small_cell(L, N, 2, 3, 74, depth=-3.0)
    cell["pos"][0] = [face, L - 0.3, 0.5 * L]
    occ = np.array([2.0, 1.25, 0.5])
    ref = ko.Cell(dict(cell, occ=occ))
    q, _ = ko.cholqr(inputs.random_coeffs(74, 3, ref.nG))
    q = ko.block_iteration(ref, q, 2)[1]
    F_ref = ko.forces(ref, q)
    g = ks.Grid(cell, prec=prec, occ=occ)
    g.set_states(q)
    meas("N=%d forces" % N, np.max(np.abs(g.forces() - F_ref)), tol * np.max(np.abs(F_ref)))
    g.close()


@pytest.mark.parametrize("N,L,ns", [(32, 13.3, 1), (36, 11.25, 2), (36, 11.25, 3), (48, 20.0, 1), (48, 20.0, 2), (54, 16.875, 1),
                                    (54, 22.5, 4), (64, 20.0, 1), (64, 26.6, 3), (72, 30.0, 1), (72, 22.5, 3),
                                    (72, 30.0, 3), (72, 30.0, 4), (96, 30.0, 1), (108, 33.75, 2), (128, 40.0, 1)])
def test_fp64_routes(ks, meas, N, L, ns):
    """FP64 H psi and density either side of the line between whole planes and line passes, and on the grids
    that have line passes only: 1e-12, as on every FP64 path."""
    cell = inputs.small_cell(L, N, 3, ns, 75, depth=-3.0)
    ref = ko.Cell(cell)
    c = inputs.random_coeffs(75, ns, ref.nG)
    g = ks.Grid(cell, prec="fp64")
    psi = torch.from_numpy(c).to("cuda")
    h = torch.full_like(psi, float("nan"))
    g.apply_h(psi.data_ptr(), h.data_ptr(), ns)
    torch.cuda.synchronize()
    meas("N=%d, %d states: H psi" % (N, ns), rel(h.cpu().numpy(), ko.apply_h(ref, c)), 1e-12)
    g.set_states(c)
    n = torch.empty((N, N, N), dtype=torch.float64, device="cuda")
    g.density(n.data_ptr())
    meas("N=%d, %d states: density" % (N, ns), rel(n.cpu().numpy(), ko.density(ref, c)), 1e-12)
    g.close()


@pytest.mark.parametrize("N,h,natoms,ns", [(54, 0.3125, 1, 1), (54, 0.3125, 33, 5), (72, 0.375, 40, 3), (108, 10.0 / 24, 17, 2)])
def test_projections_of_fp32_accuracy(ks, meas, N, h, natoms, ns):
    """H psi of smooth states (large projections beside the kinetic part) on the grids of 54, 72 and 108 points
    at the accuracy of sums over the grid: a coefficient's last two roundings, 2^-24 / sqrt(3) rms each, are
    4.9e-8, the transforms and projections come to less: 6.5e-8.  (Split-BF16 projections: 7e-8 to 1.4e-7.)"""
    cell = inputs.small_cell(N * h, N, natoms, ns, 76, depth=-3.0)
    ref = ko.Cell(cell)
    t = 0.5 + np.arange(ns)[:, None]
    c = (inputs.random_coeffs(76, ns, ref.nG) * np.exp(-0.25 * ref.g2[None, :] / t)).astype(np.complex64)
    g = ks.Grid(cell, prec="bf16x3")
    psi = torch.from_numpy(c).to("cuda")
    out = torch.empty_like(psi)
    g.apply_h(psi.data_ptr(), out.data_ptr(), ns)
    torch.cuda.synchronize()
    meas("N=%d, %d atoms" % (N, natoms), rel(out.cpu().numpy().astype(complex), ko.apply_h(ref, c.astype(complex))), 6.5e-8)
    g.close()


@pytest.mark.parametrize("natoms,nproj,ns", [(1, 1, 1), (16, 4, 2), (5, 4, 3), (17, 4, 9), (73, 1, 99), (73, 1, 100)])
def test_projection_groups(ks, meas, natoms, nproj, ns):
    """Projections summed on the grid, either side of the lines between two and eight states a CTA (four and one
    warps per atom and state), full and ragged groups, states of different sizes; bound of the fused grids'
    H psi."""
    cell = inputs.small_cell(16.875, 54, natoms, ns, 77, depth=-3.0, nproj=nproj)
    ref = ko.Cell(cell)
    c = inputs.random_coeffs(77, ns, ref.nG) * np.logspace(-3, 3, ns)[:, None]
    g = ks.Grid(cell, prec="bf16x3")
    buf = torch.zeros((ns + 1, ref.nG), dtype=torch.complex64, device="cuda")
    buf[1:] = torch.from_numpy(c).to("cuda", torch.complex64)
    out = torch.full_like(buf, float("nan"))
    g.apply_h(buf[1:].data_ptr(), out[1:].data_ptr(), ns)
    torch.cuda.synchronize()
    got, expect = out[1:].cpu().numpy().astype(complex), ko.apply_h(ref, c)
    meas("%d x %d" % (natoms * nproj, ns), max(rel(got[k], expect[k]) for k in range(ns)), 2e-5)
    g.close()


@pytest.mark.parametrize("N,L,grids", [(64, 20.0, 1), (54, 16.875, 1), (36, 11.25, 2)])
def test_force_buffers(ks, N, L, grids):
    """The first force call allocates the states' full grids once, and the gradients' beside them only on grids
    without team transforms: that many grids of the block, plus less than half a one for the rest."""
    ns = 24
    cell = inputs.small_cell(L, N, 2, ns, 78)
    g = ks.Grid(cell, prec="bf16x3")
    g.set_states(inputs.random_coeffs(78, ns, g.nG))
    before = g.device_bytes()
    g.forces()
    grown, block = g.device_bytes() - before, 8 * ns * N ** 3
    assert grids * block <= grown <= (grids + 0.5) * block
    g.close()
