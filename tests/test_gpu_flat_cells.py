"""Grids of four planes that fill an SM's shared memory: an orbital copy of 205 to 210 KB and nothing behind it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import tdks_oracle as O  # noqa: E402
from paper_1804_01404_gb300 import tdks, workloads as W  # noqa: E402


@pytest.mark.parametrize("n,periodic,precision", [((81, 81, 4), False, "f32"), ((80, 80, 4), True, "f32"), ((57, 57, 4), True, "f64")],
                         ids=str)
def test_four_full_planes(n, periodic, precision):
    s = W.tiny(periodic=periodic, n=n, norb=2, natom=0, nk=2 if periodic else 1)
    psi0 = W.initial_orbitals(s, 0)
    ctx = tdks.Context(s, precision=precision)
    u = torch.from_numpy(psi0).to("cuda", ctx.cdtype)
    ctx.update_potential(u)
    V = (ctx.grid_array(0) + ctx.grid_array(1)).cpu().numpy()
    A = [0.05, -0.1, 0.2] if periodic else None
    ctx.taylor_step(u, s.dt, A)
    o = ctx.observables(u, A or [0.0] * 3)
    ref = O.propagate_all(s, [], V, psi0, A or np.zeros(3), s.dt)
    tol = 2e-5 if precision == "f32" else 1e-12          # (as in test_gpu_cell_edges.py)
    assert np.linalg.norm(u.cpu().numpy() - ref) < tol * np.linalg.norm(ref)
    if periodic:
        assert np.abs(o["J"] - O.current(s, [], ref, A)).max() < 10 * tol
