"""Which kernels run a context's Taylor launches (tdks_taylor_path): what is in use, how a scheme that was set is
left again, and the slab launches forced on every kind of grid that test_gpu_slab.py lists (there the trial run at
set-up decides whether they run), to the tolerances derived there."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1804_01404_gb300 import tdks  # noqa: E402
from test_gpu_slab import SYSTEMS, orbitals, rel, system  # noqa: E402

KERNELS, SLAB, FIXED = tdks.PATH_KERNELS, tdks.PATH_SLAB, tdks.PATH_FIXED
MORE = [((16, 16, 16), (0.5,) * 3, True, 9, 2, 2), ((20, 20, 20), (0.5,) * 3, True, 5, 8, 1)]   # built-in geometries


@pytest.mark.parametrize("spec", SYSTEMS + MORE, ids=lambda s: "x".join(map(str, s[0])) + ("p" if s[2] else "i"))
@pytest.mark.parametrize("at_start,off", [(False, 0), (True, 0), (False, 1), (True, 1)])
def test_forced_slabs(spec, at_start, off):
    s = system(*spec)
    u0 = orbitals(s)
    out = {}
    for path in (SLAB, None):
        try:
            ctx = tdks.Context(s, precision="f64" if path is None else "f32", obs_at_start=at_start)
        except tdks.TdksError:                            # too large for FP64 cells: the FP32 cell kernels
            ctx = tdks.Context(s, precision="f32", obs_at_start=at_start)
            path = KERNELS
        if path is not None:
            assert ctx.taylor_path(path) == path
        buf = torch.empty(u0.numel() + 1, dtype=ctx.cdtype, device="cuda")
        u = buf[off:off + u0.numel()].view(u0.shape)      # 8 bytes off: pairs of points are not 16-byte aligned
        u.copy_(u0)
        ctx.update_potential(u)
        t = u.clone()
        ctx.taylor_step(t, 0.02, [0.1, -0.2, 0.05] if s.periodic else None)
        J = []
        for i in range(2):
            ctx.step(u, 0.02 * i, 0.02)
            J.append(ctx.read_step_observables()["J"])
        ctx.check()
        assert ctx.taylor_path() == (path or ctx.taylor_path())
        out[path == SLAB] = (t, u, ctx.grid_array(2), np.array(J))
    for i in range(3):
        assert rel(out[True][i], out[False][i].to(out[False][i].dtype)) < 1e-6, i
    if s.periodic:
        assert np.abs(out[True][3] - out[False][3]).max() < 1e-6 * 2 * s.norb / (s.dV * s.npts)


def test_paths_of_contexts():
    s = system((12, 14, 10), (0.5, 0.45, 0.5), True, 4, 2, 1)
    u0 = orbitals(s).to(torch.complex128)
    ctx = tdks.Context(s, precision="f64")
    assert ctx.taylor_path() == FIXED
    got = []
    for change in (lambda: None, lambda: ctx.cell_variant(ctx.cell_variant()[0]), lambda: ctx.taylor_path(tdks.PATH_AUTO)):
        change()
        u = u0.clone()
        ctx.update_potential(u)
        ctx.taylor_step(u, 0.02, [0.1, -0.2, 0.05])
        got.append((ctx.taylor_path(), u))
    assert [p for p, _ in got] == [FIXED, KERNELS, FIXED]       # a scheme that is set runs, and can be left again
    assert torch.equal(got[0][1], got[2][1]) and not torch.equal(got[0][1], got[1][1])
    with pytest.raises(tdks.TdksError, match="EUNSUPPORTED"):
        ctx.taylor_path(SLAB)
    for bad in (-2, 4):
        with pytest.raises(tdks.TdksError, match="EINVAL"):
            ctx.taylor_path(bad)
    ctx.close()
    for periodic in (True, False):                        # cell and tile contexts of FP32 orbitals
        s = system((14, 15, 16) if periodic else (32, 32, 32), (0.4,) * 3, periodic, 6, 2, 1)
        ctx = tdks.Context(s, precision="f32")
        auto = ctx.taylor_path()
        assert auto in (KERNELS, SLAB)
        assert ctx.taylor_path(SLAB) == SLAB
        (ctx.cell_variant if periodic else ctx.tile_variant)(0)
        assert ctx.taylor_path() == KERNELS
        assert ctx.taylor_path(tdks.PATH_AUTO) == auto
        with pytest.raises(tdks.TdksError, match="EUNSUPPORTED"):
            ctx.taylor_path(FIXED)
        ctx.close()


def test_smallest_fp64_grids():
    """Grids that fill less than a CTA keep the FP64 kernel, and can be put on the fixed-point path."""
    for n, periodic, want in (((4, 4, 4), True, KERNELS), ((4, 4, 8), True, FIXED), ((5, 5, 5), False, KERNELS),
                              ((6, 6, 6), False, FIXED)):
        s = system(n, (0.6,) * 3, periodic, 3, 0, 1)
        ctx = tdks.Context(s, precision="f64")
        assert ctx.taylor_path() == want
        u0 = orbitals(s).to(torch.complex128)
        out = []
        for path in (KERNELS, FIXED, tdks.PATH_AUTO):
            ctx.taylor_path(path)
            u = u0.clone()
            ctx.update_potential(u)
            ctx.taylor_step(u, 0.02)
            out.append(u)
        assert rel(out[1], out[0]) < 2e-15                   # (as in test_gpu_fixed.py)
        assert torch.equal(out[2], out[want == FIXED])
        ctx.close()


def test_graph_of_predicted_steps_follows_the_path():
    s = system((14, 15, 16), (0.5, 0.45, 0.4), True, 7, 2, 3)
    u0 = orbitals(s)
    res = []
    for paths in ((KERNELS,) * 8, (SLAB,) * 8, (KERNELS, SLAB) * 4):
        ctx = tdks.Context(s, precision="f32")
        u = u0.clone()
        ctx.update_potential(u)
        ctx.set_predictor(tdks.PRED_EXTRAP, 1e-2)
        for i, p in enumerate(paths):
            ctx.taylor_path(p)
            ctx.step(u, 0.02 * i, 0.02)
        assert ctx.read_step_observables()["fallbacks"] == 0
        ctx.check()
        res.append(u)
    assert rel(res[1], res[0].to(torch.complex128)) < 1e-6 and rel(res[2], res[0].to(torch.complex128)) < 1e-6
