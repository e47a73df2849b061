"""Call sequences, states and potentials at the ends of what the fixed-point FP64
kernels take."""
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
