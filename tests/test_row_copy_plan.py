"""Host replay of the row kernel's copies (lbm_kernels_row.cuh, producer warp).

Every bulk copy of every item starts on a 16-byte boundary in global and shared
memory, lies inside the population buffer (rounded up to its 256-byte region) and
inside its own slot; the copied blocks put the pulled populations where the
density warps read them; no two copies of a slot overlap.
"""
import numpy as np
import pytest

from oracle import lattice as L

XI = [tuple(int(c) for c in v) for v in L.D3Q19]
GROUPS = [0, 7, 11, 15, 19]


def wrap(g, n):
    return g + n if g < 0 else (g - n if g >= n else g)


@pytest.mark.parametrize("nx,ny,nz,es,by,zc", [
    (16, 9, 5, 4, 4, 2), (13, 9, 5, 4, 4, 2), (3, 7, 4, 4, 5, 1), (3, 3, 5, 4, 2, 5), (4, 3, 5, 4, 3, 2),
    (7, 11, 3, 4, 10, 3), (9, 5, 6, 4, 4, 4), (16, 6, 5, 2, 6, 2), (24, 10, 4, 2, 3, 3), (157, 20, 3, 4, 8, 3),
])
def test_row_copies(nx, ny, nz, es, by, zc, R=1):
    ve, N = 16 // es, nx * ny * nz
    aligned = nx % ve == 0
    slot = -(-((by + 2 * R) * nx + 4 * ve) // 4) * 4
    slot = -(-slot // ve) * ve
    delta = 0 if aligned else ve + (-ny * nx) % ve
    cols, chunks = -(-ny // by), -(-nz // zc)
    region = -(-19 * N * es // 256) * 256
    for item in range(cols * chunks):
        y0, z0 = (item % cols) * by, (item // cols) * zc
        h, rows = min(by, ny - y0), min(by, ny - y0) + 2 * R
        for q in range(min(zc, nz - z0) + 2 * R):
            z = wrap(z0 - R + q, nz)
            for g in range(4):
                for i in range(GROUPS[g], GROUPS[g + 1]):
                    cx, cy, cz = XI[i]
                    held = np.full(slot, -1, dtype=np.int64)
                    first = wrap(y0 - R - cy, ny)
                    e_first = i * N + first * nx
                    zo = wrap(z - cz, nz) * ny * nx
                    for seg in range(4):
                        y, r0 = first, 0
                        n = min(rows, ny - y)
                        for _ in range(seg):
                            r0, y = r0 + n, 0
                            n = min(rows - r0, ny)
                        if n <= 0:
                            continue
                        e = i * N + y * nx + zo
                        pos, count = r0 * nx + (0 if aligned or seg == 0 else delta), n * nx
                        if not aligned:
                            a = e % ve
                            pos += (e_first + zo) % ve - a
                            e, count = e - a, -(-(a + count) // ve) * ve
                        assert e * es % 16 == 0 and pos * es % 16 == 0 and count * es % 16 == 0
                        assert 0 <= e and (e + count) * es <= region
                        assert 0 <= pos and pos + count <= slot
                        assert np.all(held[pos:pos + count] == -1)
                        held[pos:pos + count] = np.arange(e, e + count)
                    shift = 0 if aligned else (e_first + zo) % ve
                    for j in range(rows * nx):
                        r, x = divmod(j, nx)
                        src = wrap(x - cx, nx)
                        at = r * nx + src + shift + (0 if first + r < ny else delta)
                        want = i * N + zo + ((y0 - R - cy + r) % ny) * nx + src
                        assert held[at] == want, (item, q, i, j)
