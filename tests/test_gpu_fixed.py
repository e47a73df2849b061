"""The fixed-point arithmetic of the FP64 kernels (dirac_fixed.cuh): the limits
of its shared exponents, against the oracle and against exact scaling."""
import numpy as np
import pytest

from oracle import hamiltonian as ham, lanczos as lz
from paper_1407_7370_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def prop_of(g, m, order, boundary, V=None, A=(0.0, 0.0), mode="auto"):
    import torch
    from paper_1407_7370_gb300 import Propagator
    p = Propagator(g.nx, g.ny, g.dx, g.dy, order=order, boundary=boundary, m_max=m)
    p.set_fields(None if V is None else torch.from_numpy(V).cuda(), A=A)
    p.set_step_mode(mode)
    return p


@pytest.mark.parametrize("nx,ny,dy,order", [(35, 11, 0.1, 2), (64, 64, 0.13, 4), (97, 50, 0.1, 4), (130, 33, 0.1, 2)])
def test_t_entries_keep_fp64_accuracy(nx, ny, dy, order):
    """beta_m has no later norm to correct it: it is the square root of s2 = Y -
    P^2/X, whose relative error is the sums' rounding times kappa = Y / s2 (the
    rows of y^ cancel by several digits against their largest terms)."""
    import torch
    g = wl.Grid(nx, ny, 0.1, dy)
    for psi0 in (wl.random_spinor(g, 3), wl.positive_energy_packet(g, p0=(10.0, -4.0), sigma_x=0.4)):
        for m in (2, 5):
            op = ham.Operator(nx, ny, 0.1, dy, A=(3.0, -1.5), order=order)
            _, inf = lz.krylov_step(op, psi0.copy(), 1e-4, m)
            p = prop_of(g, m, order, "periodic", A=(3.0, -1.5))
            info = p.step(torch.from_numpy(psi0.copy()).cuda(), 1e-4, m, info=True)
            tol = 64 * U * max(1.0, info.kappa_max)
            scale = np.max(np.abs(inf.beta)) + np.max(np.abs(inf.alpha))
            assert np.max(np.abs(info.beta * 1e-4 / inf.beta - 1.0)) <= tol
            assert np.max(np.abs(info.alpha * 1e-4 - inf.alpha)) <= 64 * U * scale


@pytest.mark.parametrize("mode", ["one_launch", "passes"])
@pytest.mark.parametrize("order,boundary,hasv", [(2, "periodic", True), (4, "dirichlet", False)])
def test_power_of_two_scaling_is_exact(mode, order, boundary, hasv):
    """Every scale is a power of two, so a state times 2^k gives 2^k times the result, bit for bit."""
    import torch
    g = wl.Grid(75, 41, 0.1, 0.1)
    psi0 = wl.random_spinor(g, 5)
    V = wl.random_potential(g, 2, scale=30.0) if hasv else None
    outs = []
    for k in (0, 300, -300):
        psi = torch.from_numpy(psi0 * 2.0 ** k).cuda()
        p = prop_of(g, 8, order, boundary, V, A=(2.0, 1.0), mode=mode)
        p.steps(psi, 2, 1e-4, 8)
        p.sync()
        outs.append(psi.cpu().numpy() * 2.0 ** -k)
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])


@pytest.mark.parametrize("order", [2, 4])
def test_small_numbers_far_from_large_ones_keep_their_digits(order):
    """A region 1e30 times smaller than the rest of the state has its own
    exponents: its relative error is that of a state of its own size."""
    import torch
    g = wl.Grid(160, 48, 0.1, 0.1)
    psi0 = wl.random_spinor(g, 8)
    psi0[:, :80] *= 1e-30
    m, steps = 6, 2
    op = ham.Operator(g.nx, g.ny, g.dx, g.dy, order=order, boundary=ham.DIRICHLET)
    ref, _ = lz.propagate(op, psi0.copy(), 1e-4, m, steps)
    psi = torch.from_numpy(psi0.copy()).cuda()
    p = prop_of(g, m, order, "dirichlet")
    p.steps(psi, steps, 1e-4, m)
    p.sync()
    out = psi.cpu().numpy()
    far = slice(0, 30)   # out of reach of 2 x 6 products of half width 2, and in tiles of small numbers only
    assert lz.rel_l2(out[:, far], ref[:, far]) <= 3e-14 * steps
    assert lz.rel_l2(out, ref) <= 1e-14 * steps


def test_zero_regions_and_zero_state_stay_zero():
    import torch
    g = wl.Grid(128, 64, 0.1, 0.1)
    psi0 = np.zeros((64, 128, 2), dtype=np.complex128)
    psi0[30:33, 100:103] = 1.0 + 0.5j
    psi = torch.from_numpy(psi0).cuda()
    p = prop_of(g, 5, 2, "periodic")
    p.step(psi, 1e-4, 5)
    p.sync()
    out = psi.cpu().numpy()
    reach = np.zeros((64, 128), dtype=bool)
    reach[30 - 4:33 + 4, 100 - 4:103 + 4] = True
    assert not np.any(out[~reach]) and np.all(np.isfinite(out))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_state_is_reported(bad):
    import torch
    from paper_1407_7370_gb300._native import DiracError
    g = wl.Grid(70, 40, 0.1, 0.1)
    psi0 = wl.random_spinor(g, 1)
    psi0[11, 69, 1] = bad
    psi = torch.from_numpy(psi0).cuda()
    p = prop_of(g, 5, 2, "periodic")
    p.step(psi, 1e-4, 5)
    with pytest.raises(DiracError):
        p.sync()
