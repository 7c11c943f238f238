"""CPU model of the 16-byte chunk copies of the staged step kernels (the 3-D strip kernel and
the 2-D staged kernel): every copy is aligned and inside its array and stage, no byte of a stage
is written twice, and every staged value that a thread reads is the periodic source node of its
pull.  Tiles, storage types, edges and thin boxes as the kernels run them."""
import pytest

C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0),
      (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
      (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]


class Stage:
    """Bytes of one stage: byte offset of each staged element -> its source."""

    def __init__(self, nbytes):
        self.nbytes, self.at = nbytes, {}

    def copy(self, dst, src_elem, esz, n, source):
        """n elements of esz bytes from element src_elem of a row; source(j): what element j is."""
        assert dst % 16 == 0 and (src_elem * esz) % 16 == 0 and (n * esz) % 16 == 0
        assert 0 <= dst and dst + n * esz <= self.nbytes
        for j in range(n):
            assert dst + j * esz not in self.at
            self.at[dst + j * esz] = source(src_elem + j)


@pytest.mark.parametrize("ssize", [2, 4])
@pytest.mark.parametrize("bx,by", [(64, 4), (64, 2), (32, 8)])
@pytest.mark.parametrize("strips,ny", [(2, 3), (3, 9), (2, 16)])
def test_strip_chunks(ssize, bx, by, strips, ny):
    nx, es, et, nr = strips * bx, 16 // ssize, 4, by + 2
    ws, wt = bx + 2 * es, bx + 2 * et
    gm_off = 19 * by * ws * ssize
    j_off = gm_off + 6 * nr * ws * ssize
    g0_off = j_off + 3 * by * bx * 4
    total = g0_off + 2 * nr * wt * 4
    for x0 in range(0, nx, bx):
        for y0 in range(0, ny, by):
            st = Stage(total)

            def row(name, r, dz, x, esz, dst, n):
                assert 0 <= x and x + n <= nx
                st.copy(dst, x, esz, n, lambda j: (name, j, (y0 + r) % ny, dz))

            for i, (cx, cy, cz) in enumerate(C3):  # the rows and their chunks beside the strip
                for r in range(by):
                    base = (i * by + r) * ws
                    row(("f", i), r - cy, 1 - cz, x0, ssize, (base + es) * ssize, bx)
            for u in range(10):
                i = u + 1 if u < 2 else u + 5
                cx, cy, cz = C3[i]
                assert cx != 0
                for r in range(by):
                    base = (i * by + r) * ws
                    x = (x0 - es + nx) % nx if cx == 1 else (x0 + bx) % nx
                    row(("f", i), r - cy, 1 - cz, x, ssize,
                        (base + (0 if cx == 1 else es + bx)) * ssize, es)
            for m in range(1, 7):
                cx, cy, cz = C3[m]
                for r in range(nr):
                    row(("g", m), r - 1 - cy, 2 - cz, x0, ssize,
                        gm_off + (((m - 1) * nr + r) * ws + es) * ssize, bx)
            for u in range(10):
                m = u + 1 if u < 2 else 3 + (u - 2) // 2
                left = u == 0 if u < 2 else u % 2 == 0
                cx, cy, cz = C3[m]
                for r in range(nr):
                    x = (x0 - es + nx) % nx if left else (x0 + bx) % nx
                    row(("g", m), r - 1 - cy, 2 - cz, x, ssize,
                        gm_off + (((m - 1) * nr + r) * ws + (0 if left else es + bx)) * ssize, es)
            for c in range(3):
                for r in range(by):
                    row(("J", c), r, 1, x0, 4, j_off + (c * by + r) * bx * 4, bx)
            for h in range(2):
                for r in range(nr):
                    base = (h * nr + r) * wt
                    row(("g0", h), r - 1, 2, x0, 4, g0_off + (base + et) * 4, bx)
                    row(("g0", h), r - 1, 2, (x0 - et + nx) % nx, 4, g0_off + base * 4, et)
                    row(("g0", h), r - 1, 2, (x0 + bx) % nx, 4, g0_off + (base + et + bx) * 4, et)
            # what the threads read: own nodes, and phase A over the halo ring as well
            for y in range(by):
                for x in range(bx):
                    for i, (cx, cy, cz) in enumerate(C3):
                        got = st.at[((i * by + y) * ws + x - cx + es) * ssize]
                        assert got == (("f", i), (x0 + x - cx) % nx, (y0 + y - cy) % ny, 1 - cz)
                    for c in range(3):
                        assert st.at[j_off + ((c * by + y) * bx + x) * 4] == (
                            ("J", c), x0 + x, (y0 + y) % ny, 1)
            for r in range(nr):
                for x in range(-1, bx + 1):
                    for m in range(1, 7):
                        cx, cy, cz = C3[m]
                        got = st.at[gm_off + (((m - 1) * nr + r) * ws + x - cx + es) * ssize]
                        assert got == (("g", m), (x0 + x - cx) % nx, (y0 + r - 1 - cy) % ny, 2 - cz)
                    for h in range(2):
                        assert st.at[g0_off + ((h * nr + r) * wt + x + et) * 4] == (
                            ("g0", h), (x0 + x) % nx, (y0 + r - 1) % ny, 2)


@pytest.mark.parametrize("esz", [4, 8])
@pytest.mark.parametrize("bx,nx", [(128, 128), (128, 100), (128, 132), (128, 384), (32, 36),
                                   (64, 4), (96, 96), (128, 130), (192, 192), (256, 260)])
def test_row_chunks(esz, bx, nx):
    e = 16 // esz
    if nx % e:
        pytest.skip("the staged kernel takes whole chunks")
    cc, seg = bx // e, bx + 8
    ny = 3
    for x0 in range(0, nx, bx):
        wact, frow = min(bx, nx - x0), x0 == 0 and nx <= bx
        for r in range(ny):
            for full in (True, False):
                st = Stage((18 * seg + 2 * bx) * esz)

                def put(name, elem, x, cy, n):
                    assert 0 <= x and x + n <= nx
                    st.copy(elem * esz, x, esz, n, lambda j: (name, j, (r - cy) % ny))

                for tid in range(bx):  # one chunk per thread and pass
                    c = tid % cc * e
                    for it in range((20 + e - 1) // e):
                        p = tid // cc + it * e
                        if p >= (20 if full else 9) or c >= wact:
                            continue
                        if p < 18:
                            put(p, p * seg + 4 + c, x0 + c, C2[p % 9][1], e)
                        else:
                            put(p, 18 * seg + (p - 18) * bx + c, x0 + c, 0, e)
                for q in range(0 if frow else (18 if full else 12)):
                    g, left = q < 12, q < 6 if q < 12 else q < 15
                    u = (q if left else q - 6) if g else (q - 12 if left else q - 15)
                    i = (((0x854210 if left else 0x764320) if g else (0x851 if left else 0x763))
                         >> (4 * u)) & 15
                    x = (nx if x0 == 0 else x0) - e if left else (0 if x0 + wact >= nx else x0 + wact)
                    p = i if g else 9 + i
                    put(p, p * seg + (4 - e if left else 4 + wact), x, C2[i][1], e)

                def pos(col, d):  # staged position of local column col + d
                    j = col + d
                    return (j % nx if frow else j) + 4

                for col in range(-1, wact + 1):  # halo columns: g alone
                    for p in range(18 if full else 9):
                        cx, cy = C2[p % 9]
                        if p >= 9 and not 0 <= col < wact:
                            continue
                        got = st.at[(p * seg + pos(col, -cx)) * esz]
                        assert got == (p, (x0 + col - cx) % nx, (r - cy) % ny)
