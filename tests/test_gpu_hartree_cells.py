"""Potential of a batch of periodic cells with correlation (xc = 2), every cell against the oracle: whole planes of
several cells per CTA, the last CTA of a batch with fewer.  The library hands out the arrays of the first cell, so
the cells take turns in being first."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import tdks_oracle as O  # noqa: E402
from paper_1804_01404_gb300 import tdks, workloads as W  # noqa: E402


@pytest.mark.parametrize("n,ncell", [((22, 13, 10), 2), ((6, 7, 9), 3), ((15, 14, 12), 4), ((16, 16, 16), 3)], ids=str)
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_every_cell(n, ncell, precision):
    s = W.System(n=n, h=(0.5, 0.45, 0.55), periodic=True, atoms=[], proj=W.Projectors(r_cut=1.5), kpts=np.zeros((1, 3)),
                 kw=np.ones(1), norb=2, dt=0.02, field=W.Field("none"))
    ctx = tdks.Context(s, precision=precision, xc=2, ncell=ncell)
    u = torch.from_numpy(np.stack([W.initial_orbitals(s, i) * (1 + 0.2 * i) for i in range(ncell)])).to("cuda", ctx.cdtype)
    for i in range(ncell):
        v = torch.roll(u, -i, 0).contiguous()
        ctx.update_potential(v)
        rho, got = ctx.grid_array(2).cpu().numpy(), ctx.grid_array(1).cpu().numpy()
        want = 2 * (u[i].abs().double() ** 2).sum((0, 1)).cpu().numpy()
        assert np.abs(rho - want).max() < (1e-6 if precision == "f32" else 1e-14) * want.max()
        ref = O.hxc(s, rho, True, 2)
        assert np.abs(got - ref).max() < 1e-13 * np.abs(ref).max()
    ctx.close()
