"""Where the fixed-point Taylor launches of FP64 orbitals could fall short of FP64: the digits of the diagonal
coefficient, the density of points far below an orbital's largest value, orbitals that decay into a vacuum, and the
current."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1804_01404_gb300 import tdks, workloads as W  # noqa: E402


def box(n, h, periodic, norb, atoms=(), proj=None):
    return W.System(n=n, h=h, periodic=periodic, atoms=list(atoms), proj=proj or W.Projectors(r_cut=1.5),
                    kpts=np.zeros((1, 3)), kw=np.ones(1), norb=norb, dt=0.02, field=W.Field("none"))


@pytest.mark.parametrize("n,periodic", [((19, 10, 12), False), ((16, 16, 16), True), ((9, 13, 20), False)], ids=str)
def test_density_of_small_values(n, periodic):
    """Every point of the density to FP64 accuracy: 2^-53 from the orbitals' rounding in each of the squares, as
    much from the digits of the product, and an addition per orbital, below 2e-15 for eight of them."""
    s = box(n, (0.45, 0.5, 0.4), periodic, 8)
    ctx = tdks.Context(s, precision="f64")
    u0 = W.initial_orbitals(s, 4)
    u0[0, :, 3, 4:6, :] *= 1e-9                          # values of 1e-9 of an orbital's largest beside ordinary ones
    u = torch.from_numpy(u0).cuda()
    ctx.update_potential(u)
    ctx.step(u, 0.0, 1e-7)
    rho, v = ctx.grid_array(2).cpu().numpy(), u.cpu().numpy()
    ref = 2 * (v.real ** 2 + v.imag ** 2).sum((0, 1))
    assert ref.min() < 1e-9 * ref.max()
    assert np.abs(rho / ref - 1).max() < 2e-15


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


def test_orbitals_in_a_vacuum():
    """Localised orbitals in a wide box: the tail keeps FP64 accuracy (the same bits as the FP64 kernel's) and so
    does the exchange potential, the cube root of the density (relative 1e-14: a third of the density's few units
    and the rounding of the cube root)."""
    s = box((20, 22, 18), (0.5,) * 3, False, 3)
    x = [(np.arange(m) - 0.5 * (m - 1)) * 0.5 for m in s.n]
    r2 = lambda c: (x[2][:, None, None] - c[2]) ** 2 + (x[1][:, None] - c[1]) ** 2 + (x[0] - c[0]) ** 2
    u0 = np.stack([np.exp(-r2(c) / (2 * 0.6 ** 2)) * (1 + 0.1j) for c in ((0, 0, 0), (1, 0.5, -1), (-1, 1, 0))])[None]
    u0 /= np.sqrt((np.abs(u0) ** 2).sum((-3, -2, -1), keepdims=True) * s.dV)
    res = []
    for scheme in (None, 0):
        ctx = tdks.Context(s, precision="f64", hartree=False)
        if scheme is not None:
            ctx.cell_variant(scheme)
        u = torch.from_numpy(u0).cuda()
        ctx.update_potential(u)
        ctx.taylor_step(u, 0.02)
        w = torch.from_numpy(u0).cuda()
        ctx.step(w, 0.0, 0.02)
        res.append((u.cpu().numpy(), w.cpu().numpy(), ctx.grid_array(1).cpu().numpy()))
    assert np.array_equal(res[0][0], res[1][0])
    w, v = res[0][1:]
    rho = 2 * (w.real ** 2 + w.imag ** 2).sum((0, 1))
    assert rho.min() < 1e-25 * rho.max()
    assert np.abs(v / (-np.cbrt(3 / np.pi * rho)) - 1).max() < 1e-14
    assert np.abs(v - res[1][2]).max() < 1e-14 * np.abs(v).max()


@pytest.mark.parametrize("n,natom", [((9, 10, 11), 0), ((12, 13, 14), 3)], ids=str)
def test_current_no_further_off_than_fp64(n, natom):
    """J of a step against sums in extended precision over the orbital it returns, the mean over 48 single orbitals:
    no larger an error than the FP64 kernel's."""
    ld = np.longdouble
    d1 = [ld(4) / 5, -ld(1) / 5, ld(4) / 105, -ld(1) / 280]
    h = (0.5, 0.45, 0.4)
    L = np.array(n) * h
    atoms = [W.Atom(tuple(np.array(f) * L), 4.0) for f in ((0.21, 0.33, 0.4), (0.7, 0.64, 0.18), (0.45, 0.9, 0.77))[:natom]]
    proj = W.Projectors()
    tabs = []                                            # grid points, displacements and s, p projectors of an atom
    for at in atoms:
        d = [np.arange(n[a]) * h[a] - at.R[a] for a in range(3)]
        d = [x - l * np.round(x / l) for x, l in zip(d, L)]
        r2 = d[2][:, None, None] ** 2 + d[1][:, None] ** 2 + d[0] ** 2
        iz, iy, ix = np.nonzero(r2 < proj.r_cut ** 2)
        dd = np.stack([d[0][ix], d[1][iy], d[2][iz]])
        r2 = r2[iz, iy, ix]
        g = np.exp(-r2 / (2 * proj.width ** 2)) * (1 - r2 / proj.r_cut ** 2) ** 2
        b = np.stack([g, *(dd * g)])
        tabs.append(((iz, iy, ix), dd.astype(ld), (b / np.sqrt((b ** 2).sum(1, keepdims=True) * np.prod(h))).astype(ld)))
    err = {None: [], 0: []}
    for at_start in (False, True):
        s = box(n, h, True, 1, atoms, proj)
        ctxs = {}
        for scheme in err:
            ctxs[scheme] = tdks.Context(s, precision="f64", obs_at_start=at_start)
            if scheme is not None:
                ctxs[scheme].cell_variant(scheme)
        for seed in range(24):
            u0 = W.initial_orbitals(s, seed)
            for scheme, ctx in ctxs.items():
                u = torch.from_numpy(u0).cuda()
                ctx.update_potential(u)
                ctx.step(u, 0.0, 0.02)
                v = (u0 if at_start else u.cpu().numpy())[0, 0].astype(np.clongdouble)
                norm = (v.real ** 2 + v.imag ** 2).sum()
                J = ctx.read_step_observables()["J"]
                for a in range(3):
                    D = sum(d1[m - 1] / ld(h[a]) * (np.roll(v, -m, 2 - a) - np.roll(v, m, 2 - a)) for m in range(1, 5))
                    ref = (v.conj() * D).imag.sum()
                    for at, (idx, dd, b) in enumerate(tabs):
                        f = v[idx]
                        for p in range(4):
                            E = proj.E_s if p == 0 else proj.E_p
                            ref += 2 * ld(E) * ((dd[a] * b[p] * f).sum().conj() * (b[p] * f).sum()).imag * ld(s.dV)
                    ref *= -2 * ld(s.dV) / ld(s.dV * s.npts)
                    err[scheme].append(float(abs(J[a] - ref) / (norm / s.npts)))
    assert np.mean(err[None]) <= np.mean(err[0]), (np.mean(err[None]), np.mean(err[0]))


def test_potential_beyond_its_digits():
    """A well of |dt V| > 1: every orbital through the FP64 kernel, bit for bit; in a batch only the cell that has it
    (and the next step, with the well gone by a smaller dt, in fixed point again)."""
    n, h = (12, 10, 9), (0.5,) * 3
    s = box(n, h, True, 3, [W.Atom((2.0, 2.5, 2.0), 60.0)], W.Projectors(r_cut=1.5))
    u0 = torch.from_numpy(W.initial_orbitals(s, 1)).cuda()
    ctx = tdks.Context(s, precision="f64", hartree=False, xc=False)
    assert float(ctx.grid_array(0).abs().max()) * 0.02 > 1.0
    got = {}
    for path in (tdks.PATH_FIXED, tdks.PATH_KERNELS):
        ctx.taylor_path(path)
        for dt in (0.02, 0.002, -0.02):
            u = u0.clone()
            ctx.update_potential(u)
            ctx.taylor_step(u, dt, [0.1, 0.2, -0.1])
            got[path, dt] = u
    for dt in (0.02, -0.02):
        assert torch.equal(got[tdks.PATH_FIXED, dt], got[tdks.PATH_KERNELS, dt])
    a, b = got[tdks.PATH_FIXED, 0.002], got[tdks.PATH_KERNELS, 0.002]
    assert not torch.equal(a, b) and float((a - b).norm() / b.norm()) < 2e-15


def test_one_cell_of_a_batch_beyond():
    """Cells of a batch whose densities differ: the Hartree potential of one exceeds the digits, the others' do not."""
    s = box((10, 9, 8), (0.5, 0.55, 0.6), True, 2)
    ctx = tdks.Context(s, precision="f64", ncell=3)
    u0 = torch.from_numpy(np.stack([W.initial_orbitals(s, i) for i in range(3)])).cuda()
    u0[1] *= 60.0                                        # 3600 times the electrons
    ctx.update_potential(u0)
    out = []
    for path in (tdks.PATH_FIXED, tdks.PATH_KERNELS):
        ctx.taylor_path(path)
        u = u0.clone()
        ctx.taylor_step(u, 0.02)
        out.append(u)
    assert torch.equal(out[0][1], out[1][1])
    for i in (0, 2):
        assert not torch.equal(out[0][i], out[1][i]) and float((out[0][i] - out[1][i]).norm() / out[1][i].norm()) < 2e-15
