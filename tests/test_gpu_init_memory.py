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
