"""Host-side check of the fused 3D step's decomposition (no GPU): every cell
has exactly one owner, and every cell a block loads lies within two ghost
layers.  The ownership rules are restated from classic3d.cuh (constants read
from it) for grid sizes that put the edges in every position."""
import os
import re

import pytest

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                      "paper_1111_6583_gb300", "csrc", "classic3d.cuh")


def _const(name):
    with open(HEADER) as f:
        return int(re.search(r"constexpr int %s = (\d+);" % name, f.read()).group(1))


XOWN, LINES, ZSEG = _const("kXOwn3d"), _const("kXSweepLines"), _const("kZSeg3d")


def _layout(nx, ny, nz, prec):
    nxc, nyb = -(-nx // XOWN), -(-ny // (LINES - 4))
    slots, best, nzs = 152 if prec == 0 else 304, 0, 1
    s = -(-nz // ZSEG)
    while s <= nz:
        cost = -(-(nxc * nyb * s) // slots) * (-(-nz // s) + 4)
        if best == 0 or cost < best:
            best, nzs = cost, s
        s += 1 if s < 16 else s // 4
    return nxc, nyb, nzs


@pytest.mark.parametrize("n3", [(4, 4, 4), (28, 12, 64), (29, 13, 65), (56, 24, 5), (57, 25, 130)])
@pytest.mark.parametrize("prec", [0, 1])
def test_every_cell_has_one_owner(n3, prec):
    nx, ny, nz = n3
    nxc, nyb, nzs = _layout(nx, ny, nz, prec)
    seen = set()
    for t in range(nxc * nyb * nzs):
        bx, by, bz = t % nxc, (t // nxc) % nyb, t // (nxc * nyb)
        z0, z1 = bz * nz // nzs, (bz + 1) * nz // nzs
        assert 1 <= z1 - z0 <= ZSEG
        x0, y0 = bx * XOWN, by * (LINES - 4)
        planes = list(range(z0 - 2, z1 + 2))
        assert planes[0] >= -2 and planes[-1] <= nz + 1
        for w in range(LINES):
            assert -2 <= min(y0 - 2 + w, ny + 1) <= ny + 1
            for lane in range(32):
                i, j = x0 - 2 + lane, y0 - 2 + w
                assert -2 <= min(i, nx + 1)
                if 2 <= lane <= 29 and i < nx and 2 <= w <= LINES - 3 and j < ny:
                    # the owner's stencil of raw cells lies in the block
                    assert lane - 2 >= 0 and lane + 2 <= 31 and w - 2 >= 0 and w + 2 <= LINES - 1
                    for k in range(z0, z1):
                        assert (i, j, k) not in seen
                        seen.add((i, j, k))
    assert len(seen) == nx * ny * nz
