"""Index arithmetic of the two-step kernel on the CPU: its tasks cover every
node once, and its 16-byte loads, stores and ghost columns stay inside a row's
padded planes and the u* rows.

Layout (FP32, as the library creates it): xoff = 32 columns, a plane's row is
pitch0 = round_up(32 + nx + 4, 32) elements, u* pitch = round_up(nx + 4, 16)
doubles. Lane l of strip s holds columns c .. c + 3, c = 4 (30 s + l - 1); lanes
1 to 30 write those below nx; a lane loads if c <= nx (nx + 1 with periodic x)."""
import math
import random


def rup(a, b):
    return (a + b - 1) // b * b


def chunks_of(nx, ny, yper, warps=4 * 2 * 152):
    """(nlong, hlong, hend, nchunk) of the library's rule."""
    strips = (nx + 119) // 120
    rounds = lambda h: ((ny + h - 1) // h) * strips / warps  # noqa: E731
    hend = 0
    if rounds(16) > 3.0:
        hl, hend = (24 if rounds(16) > 16.0 else 16), 6
    else:
        best, hl = 0.0, 0
        for h in (4, 6, 8, 12, 16, max(4, (ny * strips + warps - 1) // warps)):
            t = math.ceil(rounds(h)) * (h + 1.0)
            if rounds(h) <= 1.0 and h > 40:
                t *= 1.35
            if not yper:
                t = max(t, h + 12.0)
            if best == 0.0 or t < best:
                best, hl = t, h
    tail = min(ny, int((2.0 if hl == 16 else 1.5) * warps / strips * hend)) if hend else 0
    nlong = (ny - tail) // hl if hend else (ny + hl - 1) // hl
    nchunk = nlong + ((ny - nlong * hl + hend - 1) // hend if hend else 0)
    return nlong, hl, hend, nchunk


def rows_of(chunk, ny, nlong, hl, hend):
    over = max(chunk - nlong, 0)
    ya = (chunk - over) * hl + over * hend
    return ya, min(ny, ya + (hl if chunk < nlong else hend))


def test_tasks_cover_every_row_once():
    r = random.Random(1)
    sizes = [(8192, 8192), (4096, 2048), (2048, 2048), (1025, 1025), (8, 140000), (45000, 24), (1 << 20, 16)]
    sizes += [(r.randint(8, 9000), r.randint(8, 9000)) for _ in range(300)]
    for nx, ny in sizes:
        for yper in (False, True):
            nlong, hl, hend, n = chunks_of(nx, ny, yper)
            at = 0
            for c in range(n):
                ya, yb = rows_of(c, ny, nlong, hl, hend)
                assert ya == at and yb > ya, (nx, ny, c)
                at = yb
            assert at == ny, (nx, ny)
            # the order in which the tasks are taken: the bottom and top rows' chunks first, each once
            order = [0 if i == 0 else n - 1 if i == 1 else i - 1 for i in range(n)]
            assert sorted(order) == list(range(n))


def check_columns(nx, xper):
    pitch0, upitch = rup(32 + nx + 4, 32), rup(nx + 4, 16)
    written = 0
    for s in range((nx + 119) // 120):
        for lane in range(32):
            c = 4 * (30 * s + lane - 1)
            if c <= (nx + 1 if xper else nx):
                assert (32 + c) % 4 == 0 and 0 <= 32 + c and 32 + c + 4 <= pitch0
            if 1 <= lane <= 30 and c < nx:
                written += min(4, nx - c)
                assert c % 2 == 0 and c >= 0 and c + 4 <= upitch
        # the first step is valid one column beyond what the strip writes, and those columns are loaded two beyond
        lo, hi = 120 * s, min(120 * (s + 1), nx)
        assert 4 * (30 * s - 1) <= lo - 2 and hi + 1 < 4 * (30 * s + 31)
    assert written == nx
    assert 32 - 2 >= 0 and 32 + nx + 1 < pitch0  # the ghost columns -2, -1, nx, nx + 1


def test_columns_in_bounds_for_every_width():
    for nx in list(range(8, 400)) + [1000, 2896, 4095, 4096, 4097, 8192, 12345]:
        check_columns(nx, False)
        check_columns(nx, True)
