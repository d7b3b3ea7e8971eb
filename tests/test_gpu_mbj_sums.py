"""Rounding of the FP32 sums over orbitals behind the TB-mBJ potential where a thread adds many of them: 64 k-points
of 32 orbitals on a grid few chunks cover.  The sums over segments of planes against the general kernel (which
orbitals that are not 16-byte aligned take, a k-point's orbitals first, then the k-points), both against FP64: no
further off."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1804_01404_gb300 import tdks, workloads as W  # noqa: E402


def test_long_sums():
    n, h, norb = (24, 24, 23), (0.45, 0.45, 0.45), 32
    kp, kw = W.mp_shifted(4, n[0] * h[0])
    s = W.System(n=n, h=h, periodic=True, atoms=[], proj=W.Projectors(r_cut=1.5), kpts=kp, kw=kw, norb=norb, dt=0.02,
                 field=W.Field("none"))
    g = torch.Generator("cuda").manual_seed(11)
    u = torch.randn((len(kp), norb, n[2], n[1], n[0]), generator=g, dtype=torch.complex64, device="cuda")
    k2 = sum(torch.fft.fftfreq(m, device="cuda").reshape((-1,) + (1,) * a) ** 2 for a, m in enumerate(n))
    u = torch.fft.ifftn(torch.fft.fftn(u, dim=(-3, -2, -1)) * torch.exp(-60 * k2), dim=(-3, -2, -1))
    u = u / (u.abs() ** 2).sum((-3, -2, -1), keepdim=True).sqrt() / np.sqrt(s.dV)
    buf = torch.zeros(u.numel() + 1, dtype=torch.complex64, device="cuda")
    v = {}
    for off in (0, 1):
        ctx = tdks.Context(s, precision="f32", hartree=False, xc=3, mbj_c=1.1)
        w = buf[off:off + u.numel()].view(u.shape)
        w.copy_(u)
        ctx.update_potential(w)
        v[off] = ctx.grid_array(1)
        ctx.close()
    ctx = tdks.Context(s, precision="f64", hartree=False, xc=3, mbj_c=1.1)
    ctx.update_potential(u.to(torch.complex128))
    ref = ctx.grid_array(1)
    err = [float((v[i] - ref).norm() / ref.norm()) for i in (0, 1)]
    assert err[0] <= err[1], err
