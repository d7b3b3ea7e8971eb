"""Contexts on a device that has room for them and little more: what only serves a faster path (the trial runs at
tdks_init, the tables of that path) must not make the set-up fail."""
import gc

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1804_01404_gb300 import tdks, workloads as W  # noqa: E402

MiB = 1 << 20


def room():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("n,periodic,norb", [((40, 40, 40), False, 400), ((32, 28, 28), True, 1216)], ids=["tiled", "cell"])
def test_set_up_with_little_room(n, periodic, norb):
    s = W.System(n=n, h=(0.4, 0.4, 0.4), periodic=periodic, atoms=[W.Atom((4.0, 4.0, 4.0) if periodic else (0.3, 0.2, 0.1), 4.0)],
                 proj=W.Projectors(r_cut=1.5), kpts=np.zeros((1, 3)), kw=np.ones(1), norb=norb, dt=0.02, field=W.Field("none"))
    tdks.Context(s, precision="f32").close()              # (the kernels' code is loaded now)
    gc.collect()
    before = room()
    ctx = tdks.Context(s, precision="f32")
    need = before - room()
    ctx.close()
    one = norb * s.npts * 8                               # one set of orbitals: what a trial run would like to have
    assert one > 160 * MiB
    fill, left = [], room() - need - 64 * MiB
    while left > 0:
        fill.append(torch.empty(min(left, 1 << 34), dtype=torch.uint8, device="cuda"))
        left -= fill[-1].numel()
    try:
        ctx = tdks.Context(s, precision="f32")
        ctx.close()
    finally:
        del fill
        torch.cuda.empty_cache()


def test_training_after_the_device_filled_up():
    """The predictor's set-up takes what training one sample at a time needs; a device that is full afterwards only
    costs the larger groups."""
    s = W.tiny(periodic=True, n=(12, 12, 12), norb=2, natom=1)
    ctx = tdks.Context(s, precision="f32")
    g = torch.Generator("cuda").manual_seed(1)
    v = torch.randn((40, 12, 12, 12), generator=g, dtype=torch.float64, device="cuda")
    ctx.nn_init(0)
    p = ctx.nn_params()
    want = ctx.nn_train(v, epochs=1, batch=8, lr=1e-3, seed=0), ctx.nn_params()
    ctx.close()
    ctx = tdks.Context(s, precision="f32")
    ctx.nn_init(0)
    ctx.nn_params(p)
    fill = []
    for size in (1 << 34, 1 << 30, 1 << 26, 1 << 22, 2 * MiB):
        while True:
            try:
                fill.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
            except torch.OutOfMemoryError:
                break
    try:
        loss, grad = ctx.nn_gradient(v[1:5], v[5])
        got = ctx.nn_train(v, epochs=1, batch=8, lr=1e-3, seed=0), ctx.nn_params()
    finally:
        del fill
        torch.cuda.empty_cache()
    assert np.isfinite(loss) and np.isfinite(grad).all()
    # the same samples in groups of other sizes: FP32 sums in another order, then Adam's normalised step of 1e-3
    assert np.allclose(got[0], want[0], rtol=1e-5)
    assert np.linalg.norm(got[1] - want[1]) < 1e-4 * np.linalg.norm(want[1])
