"""States, potentials and call sequences at the ends of what the fixed-point FP64
kernels take: wide ranges of values inside a tile or a vector, norms that change
between calls, adaptive steps, and fields that are refused."""
import numpy as np
import pytest

from oracle import hamiltonian as ham, lanczos as lz
from paper_1407_7370_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
C = 137.036
MC2 = C * C


def make(g, m, order=2, boundary="periodic", V=None, A=(0.0, 0.0), shift=0.0, mode="auto", precision="fp64"):
    import torch
    from paper_1407_7370_gb300 import Propagator
    p = Propagator(g.nx, g.ny, g.dx, g.dy, order=order, boundary=boundary, m_max=m, precision=precision)
    p.set_fields(None if V is None else torch.from_numpy(V).cuda(), A=A, shift=shift)
    p.set_step_mode(mode)
    return p


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def bnd(boundary):
    return ham.DIRICHLET if boundary == "dirichlet" else ham.PERIODIC


def hnorm(g, order, A=(0.0, 0.0)):
    """Bound of ||H|| without V."""
    f = 1.0 if order == 2 else 1.372
    p = [f / h + abs(a) for h, a in zip((g.dx, g.dy), A)]
    return np.sqrt(MC2 ** 2 + C * C * (p[0] ** 2 + p[1] ** 2))


# --- adaptive steps ---------------------------------------------------------

@pytest.mark.parametrize("mode", ["one_launch", "passes"])
@pytest.mark.parametrize("tol", [1e-3, 1e-6, 1e-9])
def test_adaptive_step_leaves_one_diagonal_for_both_rows(mode, tol):
    """A step that the tolerance ends early leaves the coefficients of pass 1 of
    the next step, not parts of those of the pass it called off: the diagonals of
    the upper and the lower row (doubles 3 and 4 of the exported scalars) differ by
    2 m c^2."""
    g = wl.Grid(75, 41, 0.1, 0.1)
    psi0 = wl.positive_energy_packet(g, p0=(10.0, -4.0), sigma_x=0.5)
    p = make(g, 20, mode=mode)
    psi = dev(psi0)
    ref = psi0.copy()
    op = ham.Operator(g.nx, g.ny, g.dx, g.dy)
    for s in range(3):
        info = p.step(psi, 1e-4, 20, tol=tol, info=True)
        ref, oi = lz.krylov_step(op, ref, 1e-4, 20, tol=tol)
        assert info.k_used == oi.k_used < 20
        au0, ad0 = np.frombuffer(p.export_state()[:40], dtype=np.float64)[3:5]
        assert abs(au0 - ad0 - 2 * MC2) <= 4 * U * 2 * MC2
    assert lz.rel_l2(psi.cpu().numpy(), ref) <= 1e-14 * 3


# --- potentials with a wide range -------------------------------------------

@pytest.mark.parametrize("wall", [1e8, 1e12, 1e30])
@pytest.mark.parametrize("nx,ny,order,boundary", [(75, 41, 2, "periodic"), (97, 50, 4, "dirichlet"),
                                                  (513, 420, 4, "periodic"), (705, 333, 2, "dirichlet")])
def test_hamiltonian_product_beside_a_wall(nx, ny, order, boundary, wall):
    """Sites where V = 0 keep the accuracy that they have without the wall, in the
    tiles that hold a part of it too; sites of the wall that of the wall's size."""
    g = wl.Grid(nx, ny, 0.1, 0.13)
    psi = wl.random_spinor(g, nx)
    V = np.zeros((ny, nx))
    V[:, nx - 21:] = wall
    V[ny // 2, 10] = -wall
    op = ham.Operator(nx, ny, 0.1, 0.13, order=order, V=V, A=(3.0, -2.0), boundary=bnd(boundary))
    ref = ham.apply(op, psi)
    out = make(g, 1, order, boundary, V, A=(3.0, -2.0)).apply(dev(psi)).cpu().numpy()
    free = V == 0.0
    assert ham.norm((out - ref)[free]) <= 16 * U * hnorm(g, order, (3.0, -2.0)) * ham.norm(psi)
    assert ham.norm((out - ref)[~free]) <= 16 * U * wall * ham.norm(psi)


@pytest.mark.parametrize("nx,ny,order", [(75, 41, 2), (513, 420, 4)])
def test_hamiltonian_product_with_potential_over_many_decades(nx, ny, order):
    g = wl.Grid(nx, ny, 0.1, 0.13)
    rng = np.random.default_rng(5)
    psi = wl.random_spinor(g, 3)
    V = 10.0 ** rng.uniform(-6.0, 14.0, size=(ny, nx)) * rng.choice([-1.0, 1.0], size=(ny, nx))
    op = ham.Operator(nx, ny, 0.1, 0.13, order=order, V=V)
    out = make(g, 1, order, V=V).apply(dev(psi)).cpu().numpy()
    err = np.max(np.abs(out - ham.apply(op, psi)), axis=-1)
    assert np.max(err / (hnorm(g, order) + np.abs(V))) <= 16 * U * np.max(np.abs(psi))


@pytest.mark.parametrize("order", [2, 4])
def test_eigen_mode_does_not_see_a_wall_out_of_reach(order):
    """Ten products of half width 1 (2) reach 10 (20) sites; the wall is further
    away but in the same tiles."""
    g = wl.Grid(97, 83, 0.1, 0.1)
    start = np.zeros((83, 97, 2), complex)
    start[36:46, 40:50] = wl.random_spinor(wl.Grid(10, 10, 0.1, 0.1), 4)
    V = np.zeros((83, 97))
    V[:, :18] = V[:, 72:] = 1e14
    kw = dict(n_want=10, max_iter=10, tol=1e9, window=(-1e9, 1e9), check_every=10)
    free = make(g, 1, order, shift=MC2).eigs(dev(start), **kw)
    wall = make(g, 1, order, V=V, shift=MC2).eigs(dev(start), **kw)
    assert free.values.size == wall.values.size == 10
    assert np.max(np.abs(free.values - wall.values)) <= 1e-11 * hnorm(g, order)


# --- norms at the ends of the range, and norms that change ------------------

def run_steps(p, psi0, k, n=2, m=8):
    psi = dev(psi0 * 2.0 ** k)
    info = p.steps(psi, n, 1e-4, m, info=True)
    return psi.cpu().numpy() * 2.0 ** -k, info


@pytest.mark.parametrize("mode", ["one_launch", "passes"])
@pytest.mark.parametrize("order", [2, 4])
def test_norm_may_change_between_calls(mode, order):
    """The scalars that a context carries from step to step are those of the state
    before; the next state may have any norm whose square is a normal number."""
    g = wl.Grid(75, 41, 0.1, 0.1)
    psi0 = wl.random_spinor(g, 5)
    V = wl.random_potential(g, 2, scale=30.0)
    ref, ri = run_steps(make(g, 8, order, V=V, mode=mode), psi0, 0)
    p = make(g, 8, order, V=V, mode=mode)
    for k in (0, 260, -260, 480, -480, 0, -300):
        out, info = run_steps(p, psi0, k)
        assert lz.rel_l2(out, ref) <= 1e-14 * 2, k
        assert info.k_used == 8 and not info.breakdown
        assert np.allclose(info.alpha, ri.alpha, rtol=1e-12, atol=1e-12 * hnorm(g, order))
        assert np.allclose(info.beta, ri.beta, rtol=1e-9, atol=0)


@pytest.mark.parametrize("mode", ["one_launch", "passes"])
def test_state_whose_squared_norm_is_subnormal(mode):
    """2^-517 |psi0| ~ 2^-512: the sum of squares keeps 2^-1074 of about 2^-1024, so
    norms are good to 2^-50 and what they scale likewise."""
    g = wl.Grid(33, 20, 0.1, 0.1)
    psi0 = wl.random_spinor(g, 5)
    psi0 *= 2.0 ** 5 / ham.norm(psi0)
    ref, _ = run_steps(make(g, 8, mode=mode), psi0, 0)
    out, info = run_steps(make(g, 8, mode=mode), psi0, -517)
    assert info.k_used == 8 and not info.breakdown
    assert lz.rel_l2(out, ref) <= 16 * 2.0 ** -50


@pytest.mark.parametrize("k", [260, -260])
def test_step_of_another_norm_after_a_gradient(k):
    """The gradient's multiply-add passes leave no scale of y^."""
    g = wl.Grid(12, 10, 0.4, 0.4)
    V = wl.soft_core(g, 2.0)
    psi0 = wl.positive_energy_packet(g, p0=(2.0, 1.0), sigma_x=0.8)
    ref, _ = run_steps(make(g, 8, V=V, shift=MC2), psi0, 0)
    p = make(g, 8, V=V, shift=MC2)
    p.adjoint_gradient(dev(psi0), 2, 2e-5, 8, np.zeros((2, 2)), observable="px", checkpoint_every=2)
    out, _ = run_steps(p, psi0, k)
    assert lz.rel_l2(out, ref) <= 1e-14 * 2


@pytest.mark.parametrize("mode", ["one_launch", "passes"])
def test_all_zero_state_stays_zero(mode):
    import torch
    g = wl.Grid(70, 40, 0.1, 0.1)
    p = make(g, 6, mode=mode)
    psi = torch.zeros((40, 70, 2), dtype=torch.complex128, device="cuda")
    info = p.steps(psi, 2, 1e-4, 6, info=True)
    assert not np.any(psi.cpu().numpy()) and info.k_used == 1 and info.norm == 0.0
    psi0 = wl.random_spinor(g, 1)
    ref, _ = lz.propagate(ham.Operator(70, 40, 0.1, 0.1), psi0.copy(), 1e-4, 6, 2)
    out, _ = run_steps(p, psi0, 0, m=6)
    assert lz.rel_l2(out, ref) <= 1e-14 * 2


# --- fields that are refused ------------------------------------------------

@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_refused_potential_leaves_the_fields_as_they_were(precision, bad):
    from paper_1407_7370_gb300._native import DiracError
    g = wl.Grid(70, 40, 0.1, 0.1)
    psi0 = wl.positive_energy_packet(g, p0=(3.0, 1.0), sigma_x=0.5)
    V = wl.random_potential(g, 2, scale=30.0)
    outs = []
    for refuse in (False, True):
        p = make(g, 8, V=V, shift=MC2, precision=precision)
        psi = dev(psi0)
        p.step(psi, 1e-4, 8)
        if refuse:
            W = V * 1e6
            W[3, 5] = bad
            with pytest.raises(DiracError):
                p.set_fields(dev(W), shift=MC2)
        p.step(psi, 1e-4, 8)
        p.sync()
        outs.append(psi.cpu().numpy())
    assert np.array_equal(outs[0], outs[1])


# --- accuracy of the products and sums --------------------------------------

def product_longdouble(psi, g, order, A):
    """(H - m c^2) psi with periodic boundaries in extended precision."""
    f = psi.astype(np.clongdouble)
    c = np.longdouble(C)
    r = lambda o, ax: np.roll(f, -o, axis=ax)

    def d(ax, h):
        if order == 2:
            return (r(1, ax) - r(-1, ax)) * (c / (2 * np.longdouble(h)))
        return (8 * (r(1, ax) - r(-1, ax)) - (r(2, ax) - r(-2, ax))) * (c / (12 * np.longdouble(h)))
    px, py = -1j * d(1, g.dx) + c * np.longdouble(A[0]) * f, -1j * d(0, g.dy) + c * np.longdouble(A[1]) * f
    mc2 = c * c
    up = px[..., 1] - 1j * py[..., 1]
    lo = -2 * mc2 * f[..., 1] + px[..., 0] + 1j * py[..., 0]
    return np.stack((up, lo), axis=-1)


@pytest.mark.parametrize("nx,ny", [(96, 64), (544, 400)])
@pytest.mark.parametrize("order", [2, 4])
def test_product_is_as_accurate_as_in_fp64(nx, ny, order):
    """On a state without a wide range the root mean square error of H psi against
    extended precision is no larger than that of the oracle's FP64 arithmetic."""
    g = wl.Grid(nx, ny, 0.1, 0.13)
    A = (7.0, -5.0)
    psi = wl.random_spinor(g, 9)
    exact = product_longdouble(psi, g, order, A)
    op = ham.Operator(nx, ny, 0.1, 0.13, order=order, A=A, shift=MC2)
    out = make(g, 1, order, A=A, shift=MC2).apply(dev(psi)).cpu().numpy()
    rms = lambda a: float(np.sqrt(np.mean(np.abs(a - exact) ** 2)))
    assert rms(out) <= rms(ham.apply(op, psi))


@pytest.mark.parametrize("mode", ["one_launch", "passes"])
def test_small_component_of_a_slow_packet(mode):
    """The lower components (2^-20 of the upper ones, and fed by them) keep their own
    accuracy through the recombination: one short step against the Taylor series."""
    g = wl.Grid(75, 41, 0.1, 0.1)
    psi0 = wl.random_spinor(g, 5)
    psi0[..., 1] *= 2.0 ** -20
    dt = 1e-9
    op = ham.Operator(g.nx, g.ny, g.dx, g.dy)
    ref, term = psi0.copy(), psi0.copy()
    for k in range(1, 8):   # (dt ||H||)^8 / 8! < 1e-38
        term = ham.apply(op, term) * (-1j * dt / k)
        ref = ref + term
    psi = dev(psi0)
    p = make(g, 7, mode=mode)
    p.step(psi, dt, 7)
    p.sync()
    out = psi.cpu().numpy()
    assert lz.rel_l2(out[..., 0], ref[..., 0]) <= 1e-14
    assert lz.rel_l2(out[..., 1], ref[..., 1]) <= 1e-14


def ritz_gram(p, start, k):
    """|Y^H Y - 1| of all Ritz vectors Y of k iterations, and their values."""
    import torch
    res = p.eigs(dev(start), n_want=k, max_iter=k, tol=1e9, window=(-1e9, 1e9), check_every=k, vectors=True)
    assert res.values.size == k
    v = res.vectors.reshape(k, -1)
    return (v.conj() @ v.T - torch.eye(k, device=v.device)).abs().cpu().numpy(), res.values


def test_gram_schmidt_of_a_peak_on_a_flat_floor():
    """The floor (2^-29 of the peak, a million sites) carries 2^-37 of the squared
    norm: products of small numbers count.  Three vectors: nine inner products, each
    good to a few 2^-53 of the norms, and T's eigenvectors, whose values are far
    apart, as good."""
    g = wl.Grid(1024, 1024, 0.1, 0.1)
    start = wl.random_spinor(g, 12) * 2.0 ** -29
    start[500, 500] = (1.0, 0.5j)
    gram, _ = ritz_gram(make(g, 1, shift=MC2), start, 3)
    assert np.max(gram) <= 256 * U


@pytest.mark.parametrize("nx,ny,k", [(61, 47, 250), (251, 173, 140)])
def test_values_of_many_iterations(nx, ny, k):
    """T of k iterations, with every coefficient of the update counting: the small ones
    are applied in FP32, 128 vectors at a time (by eight warps a site on the small
    grid)."""
    g = wl.Grid(nx, ny, 0.1, 0.1)
    V = wl.smoothed_coulomb(g, 20.0, 0.5)
    start = wl.random_spinor(g, 12)
    kw = dict(n_want=k, max_iter=k, tol=1e9, window=(-1e9, 1e9), check_every=k)
    res = make(g, 1, V=V, shift=MC2).eigs(dev(start), **kw)
    ref = lz.lanczos_eigs(ham.Operator(nx, ny, 0.1, 0.1, V=V, shift=MC2), start, **kw)
    assert res.values.size == ref.values.size == k
    assert np.max(np.abs(res.values - ref.values)) <= 1e-11 * (hnorm(g, 2) + np.max(np.abs(V)))


# --- the autotuner's cache --------------------------------------------------

def test_autotune_cache_of_other_kernels_is_not_taken(tmp_path, monkeypatch):
    """A line without the kernels' tag (tile heights that meant others) is not
    taken; a batch of the same sites in other shapes has a line of its own."""
    from paper_1407_7370_gb300 import BatchPropagator
    f = tmp_path / "tune.txt"
    monkeypatch.setenv("DIRAC_AUTOTUNE_CACHE", str(f))

    def tune(grids):
        bp = BatchPropagator(grids, m_max=4)
        psis = []
        for k, (nx, ny, dx, dy) in enumerate(grids):
            bp.set_fields(k)
            psis.append(dev(wl.random_spinor(wl.Grid(nx, ny, dx, dy), k)))
        return bp.autotune(psis, 1e-4, 4, steps=1)
    grids = [(64, 48, 0.1, 0.1), (96, 32, 0.1, 0.1)]
    assert not tune(grids)["from_cache"] and tune(grids)["from_cache"]
    key, rest = f.read_text().split(" ", 1)
    old = [s for s in key.split(",") if s.split("=")[0] in ("prec", "order", "bnd", "nprob", "sites", "m", "sm", "gpu")]
    f.write_text(",".join(old) + " " + rest)
    assert not tune(grids)["from_cache"]
    assert not tune([(3072, 1, 0.1, 0.1), (1, 3072, 0.1, 0.1)])["from_cache"]
