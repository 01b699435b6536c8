"""Index arithmetic of the kernels that take several steps per launch, replayed
on the host: the tile kernel's shared-memory slots (every slot read was written
by the step before, every access inside the block's allocation, every core cell
left once), for ragged sizes and the smallest lattices."""
import pytest

C = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]


def tile_replay(nx, ny, W, H, T, stefan):
    left = {}
    rows = ny if stefan else H + 2 * T
    pitch = W + 2 * T
    for tx in range(-(-nx // W)):
        for ty in range(-(-ny // H)):
            x0, y0 = tx * W, ty * H
            x1, y1 = min(x0 + W, nx), min(y0 + H, ny)
            gx, gy = x0 - T, 0 if stefan else y0 - T
            stamp = {}  # slot -> the step that wrote it

            def slot(x, y, i):
                assert 0 <= y - gy < rows and 0 <= x - gx < pitch, (nx, ny, W, H, T, x, y)
                return ((y - gy) * pitch + (x - gx)) * 9 + i

            for t in range(1, T + 1):
                h = T - t
                xa, xb = max(0, x0 - h), min(nx, x1 + h)
                ya, yb = (0, ny) if stefan else (max(0, y0 - h), min(ny, y1 + h))
                wr, hr = xb - xa, yb - ya
                inv = ((1 << 20) + wr - 1) // wr
                touched = set()
                for c in range(wr * hr):
                    ry = (c * inv) >> 20
                    assert c * inv < 1 << 32 and ry == c // wr
                    x, y = xa + c - ry * wr, ya + ry
                    for i, (cx, cy) in enumerate(C):
                        sx, sy = x - cx, y - cy
                        if stefan:
                            sy %= ny
                        inside = 0 <= sx < nx and 0 <= sy < ny
                        if t > 1:
                            if t % 2 == 0:
                                r = slot(x, y, OPP[i])
                            else:
                                r = slot(sx, sy, i) if inside else slot(x, y, OPP[i])
                            assert stamp.get(r) == t - 1, (nx, ny, W, H, T, t, x, y, i)
                        if t == T:
                            continue
                        px, py = x + cx, y + cy
                        if stefan:
                            py %= ny
                        if t % 2 == 0:
                            w = slot(x, y, i)
                        elif 0 <= px < nx and 0 <= py < ny:
                            w = slot(px, py, OPP[i])
                        else:
                            w = slot(x, y, i)
                        assert w not in touched  # no two cells write one slot in a step
                        touched.add(w)
                    if t == T:
                        assert x0 <= x < x1 and y0 <= y < y1 and (x, y) not in left
                        left[x, y] = 1
                for w in touched:
                    stamp[w] = t
    assert len(left) == nx * ny


@pytest.mark.parametrize("nx,ny,W,H,T,stefan", [
    (2, 2, 32, 2, 2, False), (2, 12, 32, 3, 9, False), (33, 7, 32, 4, 3, False), (70, 21, 32, 5, 4, False),
    (64, 32, 32, 2, 9, False), (130, 9, 64, 9, 5, False), (65, 40, 32, 16, 16, False), (97, 13, 32, 6, 2, False),
    (100, 4, 8, 4, 7, True), (17, 2, 8, 2, 16, True), (40, 8, 16, 8, 4, True), (9, 5, 8, 5, 3, True)])
def test_tile_slots(nx, ny, W, H, T, stefan):
    tile_replay(nx, ny, W, H, T, stefan)
