"""Where the fixed-point Taylor launches of FP64 orbitals could fall short of FP64: the digits of the diagonal
coefficient."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1804_01404_gb300 import tdks, workloads as W  # noqa: E402


def box(n, h, periodic, norb, atoms=(), proj=None):
    return W.System(n=n, h=h, periodic=periodic, atoms=list(atoms), proj=proj or W.Projectors(r_cut=1.5),
                    kpts=np.zeros((1, 3)), kw=np.ones(1), norb=norb, dt=0.02, field=W.Field("none"))


def test_diagonal_beyond_its_digits():
    """A wave vector whose kinetic term and the potential add to a coefficient of 4 or more, which the digits do not
    hold: the FP64 kernel's result, bit for bit.  Spacing 12, dt = 1: bound 4.06, diagonal 3.12, potential 0.95."""
    n, h = (8, 8, 8), (12.0,) * 3
    proj = W.Projectors(E_s=1e-3, E_p=1e-3, r_cut=13.0, width=8.0)
    top = 0.0
    for Z in (-1.0, None):
        s = box(n, h, True, 2, [W.Atom((48.0,) * 3, Z if top == 0.0 else -0.95 / top, sigma=12.0)], proj)
        ctx = tdks.Context(s, precision="f64", hartree=False, xc=False)
        top = float(ctx.grid_array(0).max()) if Z else top
    assert 0.9 < float(ctx.grid_array(0).max()) < 1.0
    r2 = sum(((np.arange(8) * 12.0 - 48.0) ** 2).reshape((-1,) + (1,) * a) for a in range(3))
    u0 = 1.01 * np.stack([1 - 0.93 * np.exp(-r2 / 200), 1 - 0.9 * np.exp(-r2 / 180)])[None].astype(complex)
    got = []
    for scheme in (None, 0):
        if scheme is not None:
            ctx.cell_variant(scheme)
        u = torch.from_numpy(u0).cuda()
        ctx.update_potential(u)
        ctx.taylor_step(u, 1.0, [1.4353] * 3)
        got.append(u.cpu().numpy())
    assert np.array_equal(got[0], got[1])
