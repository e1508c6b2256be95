"""The register strips' schedule, replayed on the CPU: the windows of 32 column pairs that a group's
warps hold (stretches of several samples with two halo lanes on each side, or rows closed on
themselves), the rings between the phases (two rows of the c_y = +1 group by the parity of the
iteration, one row of the c_y = 0 group), the split of the rows into ranges (equal ones, and equal parts of
one group of samples), launches of fewer steps, and the columns that are stored.  Lanes outside the halo's
reach hold NaN, so a stored value that depends on one is found.  Every destination column is written
exactly once and one launch equals its number of plain collide-and-stream steps.  The CUDA source is
mirrored, not imported."""
import numpy as np
import pytest

from tests.test_strip3_schedule import plain_steps
from tests.test_strip_schedule import CX, CY, collide

HALO = 2
UP, FLAT, DOWN = (2, 5, 6), (0, 1, 3), (4, 7, 8)


def stretches(units, samples):
    """(warp, first lane, sample, first pair, pairs) of rows of `units` pairs laid end to end."""
    out, w, free = [], 0, 32
    for c in range(samples):
        done = 0
        while done < units:
            if free < 2 * HALO + 1:
                w, free = w + 1, 32
            count = min(free - 2 * HALO, units - done)
            out.append((w, 32 - free, c, done, count))
            free -= count + 2 * HALO
            done += count
    return out, w + 1


def lanes_of(nx, samples):
    """Per warp: task, columns xa and xb, useful, left and right lane of each lane."""
    units = (nx + 1) // 2
    lane = np.arange(32)
    if nx % 2 == 0 and units <= 32:
        samples = min(samples, 32 // units)
        task = np.where(lane // units < samples, lane // units, -1)
        px = np.where(task >= 0, lane - task * units, 0)
        left = np.where(task >= 0, task * units + (px - 1) % units, (lane - 1) % 32)
        right = np.where(task >= 0, task * units + (px + 1) % units, (lane + 1) % 32)
        warps = [(task, px, task >= 0, left, right)]
    else:
        parts, n = stretches(units, samples)
        warps = []
        for w in range(n):
            task, px, useful = np.full(32, -1), np.zeros(32, int), np.zeros(32, bool)
            for ww, l0, c, first, count in parts:
                at = lane - l0
                here = (ww == w) & (at >= 0) & (at < count + 2 * HALO)
                task[here], px[here] = c, (first + at - HALO)[here]
                useful |= here & (at >= HALO) & (at < count + HALO)
            warps.append((task, px, useful, (lane - 1) % 32, (lane + 1) % 32))
    return samples, [(t, (2 * p) % nx, ((2 * p) % nx + 1) % nx, u, le, ri) for t, p, u, le, ri in warps]


def collide_pair(g, omega):
    return collide(g.reshape(9, -1), omega).reshape(g.shape)


def from_left(v, left):
    return np.stack([v[1][left], v[0]])


def from_right(v, right):
    return np.stack([v[1], v[0][right]])


def shift(v, i, left, right):
    return v if CX[i] == 0 else (from_left(v, left) if CX[i] > 0 else from_right(v, right))


def piece(src, dst, writes, warp, ya, yb, n, omega):
    """Rows ya .. yb - 1 of a group's samples (src, dst: one array [9, ny, nx] each) on one warp."""
    task, xa, xb, useful, left, right = warp
    ny, nx = src[0].shape[1:]
    total = yb - ya + 2 * (n - 1)
    ring_p = np.full((n, 2, 9, 2, 32), np.nan)
    ring_z = np.full((n, 9, 2, 32), np.nan)
    for it in range(total):
        y = (ya - (n - 1) + it) % ny
        g = np.full((9, 2, 32), np.nan)
        for c, f in enumerate(src):
            on = task == c
            g[:, 0, on], g[:, 1, on] = f[:, y, xa[on]], f[:, y, xb[on]]
        g = collide_pair(g, omega)
        done = True
        for k in range(1, n):
            h = np.empty_like(g)
            for i in FLAT:
                h[i] = shift(ring_z[k, i], i, left, right)
            for i in UP:
                h[i] = shift(ring_p[k, it & 1, i], i, left, right)
            for i in DOWN:
                h[i] = shift(g[i], i, left, right)
            for i in FLAT:
                ring_z[k, i] = g[i]
            for i in UP:
                ring_p[k, it & 1, i] = g[i]
            if it < 2 * k:
                done = False
                break
            g = collide_pair(h, omega)
        if not done:
            continue
        row = ya + it - 2 * (n - 1)
        assert ya <= row < yb
        for i in range(9):
            v = shift(g[i], i, left, right)
            for lane in np.flatnonzero(useful):
                for half in (0, 1):
                    col = xa[lane] + half
                    if col < nx:  # past an odd width: the row's padding
                        to = (task[lane], i, (row + CY[i]) % ny, col)
                        dst[to[0]][to[1:]] = v[half, lane]
                        writes[to] = writes.get(to, 0) + 1


def ranges(nsup, ny, groups, part):
    """(group of samples, first row, last row) of each piece."""
    rows = nsup * ny
    parts = -(-ny // part) if part else 0
    per = part if part else -(-rows // groups)
    for q in range(nsup * parts if part else groups):
        r = q // parts * ny + q % parts * per if part else q * per
        end = min(rows, r + per, (q // parts + 1) * ny if part else rows)
        while r < end:
            m = r // ny
            yb = min(ny, end - m * ny)
            yield m, r - m * ny, yb
            r = m * ny + yb


@pytest.mark.parametrize("nx,ny,samples,side,groups,part", [
    (2, 3, 5, 6, 2, 0), (10, 4, 7, 6, 3, 0), (64, 5, 2, 6, 2, 0),            # closed rows
    (3, 5, 4, 3, 2, 0), (31, 6, 5, 2, 4, 0), (57, 2, 1, 1, 1, 0),            # odd widths
    (66, 5, 4, 3, 5, 0), (112, 7, 3, 2, 2, 3), (97, 9, 2, 1, 2, 4), (256, 3, 3, 3, 1, 1)])
@pytest.mark.parametrize("n", [1, 2, 3, 4])
def test_one_launch_equals_plain_steps(nx, ny, samples, side, groups, part, n):
    rng = np.random.default_rng(nx * 100 + n)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    src = [w * (1 + 0.05 * rng.standard_normal((9, ny, nx))) for _ in range(samples)]
    dst = [np.full((9, ny, nx), np.nan) for _ in range(samples)]
    side, warps = lanes_of(nx, min(side, samples))
    writes = {}
    for m, ya, yb in ranges(-(-samples // side), ny, groups, part):
        at = slice(m * side, min((m + 1) * side, samples))
        mine = {}
        for warp in warps:
            task = np.where(warp[0] < at.stop - at.start, warp[0], -1)
            piece(src[at], dst[at], mine, (task, *warp[1:3], warp[3] & (task >= 0), *warp[4:]), ya, yb, n, 1.3)
        for (c, *rest), count in mine.items():
            key = (c + at.start, *rest)
            writes[key] = writes.get(key, 0) + count
    assert len(writes) == samples * 9 * ny * nx and set(writes.values()) == {1}
    for f, out in zip(src, dst):
        # the same operations in the same order up to the reductions over nine populations: a few ulp per step
        assert np.abs(out - plain_steps(f, 1.3, n)).max() < 1e-14
