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


def hnorm(g, order, A, V):
    """Bound of ||H|| of the discretised operator (m c^2 included)."""
    c, mc2 = 137.036, 137.036 ** 2
    f = 1.0 if order == 2 else 1.372
    p = [f / h + abs(a) for h, a in zip((g.dx, g.dy), A)]
    return np.sqrt(mc2 ** 2 + c * c * (p[0] ** 2 + p[1] ** 2)) + (0.0 if V is None else np.max(np.abs(V)))


# short tiles (rows of 4) below two 32 x 16 tiles per SM, tall tiles above
@pytest.mark.parametrize("nx,ny,order,boundary,hasv,A", [
    (1, 1, 2, "periodic", False, (0.0, 0.0)), (33, 5, 4, "periodic", True, (3.0, -2.0)),
    (31, 18, 2, "dirichlet", True, (0.0, 4.0)), (64, 16, 4, "dirichlet", False, (1.0, 0.0)),
    (513, 420, 2, "periodic", True, (2.0, 1.0)), (705, 333, 4, "dirichlet", False, (0.0, -1.0))])
def test_hamiltonian_product_matches_oracle(nx, ny, order, boundary, hasv, A):
    import torch
    g = wl.Grid(nx, ny, 0.1, 0.13)
    psi = wl.random_spinor(g, nx + ny)
    V = wl.random_potential(g, 4, scale=200.0) if hasv else None
    p = prop_of(g, 1, order, boundary, V, A=A)
    out = p.apply(torch.from_numpy(psi).cuda()).cpu().numpy()
    op = ham.Operator(nx, ny, 0.1, 0.13, order=order, V=V, A=A,
                      boundary=ham.DIRICHLET if boundary == "dirichlet" else ham.PERIODIC)
    # a row has seven terms, each rounded a few times on either side
    assert ham.norm(out - ham.apply(op, psi)) <= 16 * U * hnorm(g, order, A, V) * ham.norm(psi)


@pytest.mark.parametrize("order", [2, 4])
def test_hamiltonian_product_keeps_nan_inf_and_tiny_numbers_local(order):
    """Tiles that fixed point cannot hold take the floating-point form."""
    import torch
    g = wl.Grid(96, 70, 0.1, 0.1)
    psi = wl.random_spinor(g, 3)
    p = prop_of(g, 1, order, "periodic")
    clean = p.apply(torch.from_numpy(psi).cuda()).cpu().numpy()
    psi[20, 40, 0] = np.nan
    psi[60, 5, 1] = np.inf
    out = p.apply(torch.from_numpy(psi).cuda()).cpu().numpy()
    w = order // 2
    near = np.zeros((70, 96), dtype=bool)
    for y, x in ((20, 40), (60, 5)):
        for k in range(-w, w + 1):
            near[(y + k) % 70, x] = near[y, (x + k) % 96] = True
    assert np.all(np.isfinite(out[~near])) and not np.any(np.all(np.isfinite(out[near]), axis=-1))
    assert np.max(np.abs(out[~near] - clean[~near])) <= 16 * U * hnorm(g, order, (0, 0), None) * np.max(np.abs(clean)) / 1e3
    tiny = wl.random_spinor(g, 3) * 1e-280
    out = p.apply(torch.from_numpy(tiny).cuda()).cpu().numpy()
    assert np.max(np.abs(out * 1e280 - clean)) <= 64 * U * hnorm(g, order, (0, 0), None) * 6


@pytest.mark.parametrize("nx,ny", [(33, 20), (256, 192), (251, 173)])
def test_gram_schmidt_reproduces_the_whole_of_t(nx, ny):
    """All Ritz values of 30 iterations (no convergence asked for): every T entry
    counts.  Chunks of 32 sites and eight warps per site on the small grid, full
    chunks and one thread per site on the others."""
    import torch
    g = wl.Grid(nx, ny, 0.1, 0.1)
    V = wl.smoothed_coulomb(g, 20.0, 0.5)
    start = wl.random_spinor(g, 12)
    start[:, : nx // 2] *= 1e-3
    op = ham.Operator(nx, ny, 0.1, 0.1, V=V, shift=137.036 ** 2)
    ref = lz.lanczos_eigs(op, start, n_want=30, max_iter=30, tol=1e9, window=(-1e9, 1e9), check_every=30)
    p = prop_of(g, 1, 2, "periodic")
    p.set_fields(torch.from_numpy(V).cuda(), shift=137.036 ** 2)
    res = p.eigs(torch.from_numpy(start).cuda(), n_want=30, max_iter=30, tol=1e9, window=(-1e9, 1e9), check_every=30,
                 vectors=True)
    assert res.values.size == ref.values.size == 30
    assert np.max(np.abs(res.values - ref.values)) <= 1e-11 * hnorm(g, 2, (0, 0), V)
    v = res.vectors.cpu().numpy().reshape(30, -1)
    assert np.max(np.abs(v.conj() @ v.T - np.eye(30))) <= 1e-12


@pytest.mark.parametrize("scale", [1e-140, 1e140])
def test_eigen_mode_start_vector_scale(scale):
    import torch
    g = wl.Grid(40, 33, 0.1, 0.1)
    start = torch.from_numpy(wl.random_spinor(g, 2)).cuda()
    p = prop_of(g, 1, 2, "dirichlet")
    kw = dict(n_want=10, max_iter=20, tol=1e9, window=(-1e9, 1e9), check_every=20)
    a, b = p.eigs(start, **kw), p.eigs(start * scale, **kw)
    assert np.max(np.abs(a.values - b.values)) <= 1e-11 * hnorm(g, 2, (0, 0), None)


@pytest.mark.parametrize("mode", ["one_launch", "passes"])
@pytest.mark.parametrize("m", [16, 17])
def test_gradient_in_both_launch_forms(mode, m):
    """The backward sweep's Krylov spaces without recombination (one launch) and
    from a copy of the state (per pass); m up to 16 and above take different
    contraction widths.  Tolerances of the gradient's parity with the oracle (the
    Krylov error is below 1e-18)."""
    import torch
    from oracle import adjoint as adj
    C = 137.036
    g = wl.Grid(6, 5, 0.4, 0.4)
    V = wl.soft_core(g, 2.0) + 0.3 * wl.random_potential(g, 3, scale=1.0)
    op = ham.Operator(6, 5, 0.4, 0.4, V=V, shift=C * C)
    psi0 = wl.positive_energy_packet(g, p0=(2.0, 1.0), sigma_x=0.8)
    A = np.random.default_rng(3).uniform(-1.0, 1.0, (4, 2))
    p = prop_of(g, m, 2, "periodic", mode=mode)
    p.set_fields(torch.from_numpy(V).cuda(), shift=C * C)
    res = p.adjoint_gradient(torch.from_numpy(psi0).cuda(), 4, 2e-5, m, A, observable="px", checkpoint_every=3)
    ref = adj.gradient(op, psi0, 2e-5, A, "px", None)
    dV = res.dV.cpu().numpy().reshape(-1)
    assert np.max(np.abs(dV - ref.dV)) <= 1e-9 * np.max(np.abs(ref.dV))
    assert np.max(np.abs(res.dA - ref.dA)) <= 1e-9 * np.max(np.abs(ref.dA))
