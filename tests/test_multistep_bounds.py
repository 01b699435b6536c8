"""Index arithmetic of the kernels that take several steps per launch, replayed
on the host: the tile kernel's shared-memory slots (every slot read was written
by the step before, every access inside the block's allocation, every core cell
left once) and the band kernel's ring of rows (the three rows a step-2 row needs
are still in the ring, neighbours inside the block, every cell left once), for
ragged sizes, the smallest lattices and both marching directions."""
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


def band_replay(nx, ny, strips, bands, threads, up):
    left = set()
    pairs = (nx + 1) // 2
    for s in range(strips):
        xs, xe = 2 * (s * pairs // strips), min(nx, 2 * ((s + 1) * pairs // strips))
        x_first, x_end = max(0, xs - 2), min(nx, xe + 2)
        assert (x_end - x_first + 1) // 2 <= threads
        for b in range(bands):
            ya, yb = b * ny // bands, (b + 1) * ny // bands
            r0, r1 = max(0, ya - 1), min(ny, yb + 1)
            rows = r1 - r0
            last = rows if (yb == ny if up else ya == 0) else rows - 1
            ring = {}
            for k in range(last + 1):
                y = r0 + k if up else r1 - 1 - k
                if k < rows:
                    assert 0 <= y < ny
                    ring[k & 3] = y
                    # global loads of the row: within the tiles' rows, a pair in one tile
                    for x in range(x_first, x_end, 2):
                        assert x // 128 == (x + 1) // 128
                        for j in (0, 1):
                            for cx, cy in C:
                                sx, sy = x + j - cx, y - cy
                                wall = (cx > 0 and x + j == 0) or (cx < 0 and x + j >= nx - 1)
                                wall |= (cy > 0 and y == 0) or (cy < 0 and y == ny - 1)
                                if not wall:
                                    assert 0 <= sx < -(-nx // 128) * 128 and 0 <= sy < ny
                r = y - 1 if up else y + 1
                if not ya <= r < yb:
                    continue
                assert ring[(k - 1) & 3] == r
                for x in range(xs, xe):
                    for cx, cy in C:
                        sx, sy = x - cx, r - cy
                        if not (0 <= sx < nx and 0 <= sy < ny):
                            continue  # a wall: the cell's own slots
                        assert x_first <= sx < x_end
                        newer = (cy < 0) == up
                        want = (k - 1) if cy == 0 else (k if newer else k - 2)
                        assert ring[want & 3] == sy
                    assert (x, r) not in left
                    left.add((x, r))
    assert len(left) == nx * ny


@pytest.mark.parametrize("up", [True, False])
@pytest.mark.parametrize("nx,ny,strips,bands,threads", [
    (2, 2, 1, 1, 32), (2, 9, 1, 2, 32), (300, 37, 2, 9, 96), (257, 12, 3, 3, 64), (63, 31, 1, 7, 32),
    (129, 8, 2, 1, 64), (250, 5, 4, 1, 64), (125, 6, 2, 2, 64)])
def test_band_ring(nx, ny, strips, bands, threads, up):
    band_replay(nx, ny, strips, bands, threads, up)


# ---- two cells per thread (PairPlace): the sweeps' offsets, element by element
TW, RS = 128, 18 * 128


def place(x, y, plane, ny, paired):
    ofs = 2 * ((plane % 9) * TW + x % TW) + plane // 9 if paired else plane * TW + x % TW
    return ((x // TW) * ny + y) * RS + ofs


@pytest.mark.parametrize("paired", [False, True])
@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 3), (5, 4), (64, 3), (126, 3), (127, 4), (128, 3), (129, 4),
                                   (130, 3), (255, 3), (256, 4), (257, 3), (300, 3)])
def test_pair_offsets(nx, ny, paired):
    """Every load and store of a pair, as PairPlace computes it, is the element
    that pull streaming and the push sweep's rule name; a cell's loads and stores
    are the same elements; no element is stored by two cells; a missing second
    cell loads padding of its own column and stores nothing."""
    cs = 2 if paired else 1
    stored = {}
    for x in range(0, nx, 2):
        lx, tile = x % TW, ny * RS
        dL = cs * (TW - 1) - tile if lx == 0 and x > 0 else -cs
        dR = tile - cs * (TW - 2) if lx == TW - 2 and x + 2 < nx else 2 * cs
        left, right0, right1, has1 = x == 0, x == nx - 1, x + 1 >= nx - 1, x + 1 < nx
        for y in range(ny):
            p = place(x, y, 0, ny, paired)
            bottom, top = y == 0, y == ny - 1
            loads, stores = [set(), set()], [set(), set()]
            for i, (cx, cy) in enumerate(C):
                slot = 2 * i * TW if paired else i * TW
                oslot = 2 * OPP[i] * TW if paired else OPP[i] * TW

                def walls(j):
                    wcx, wcy = C[j]
                    w = (wcy > 0 and bottom) or (wcy < 0 and top)
                    return ((wcx > 0 and left) or (wcx < 0 and right0) or w,
                            not has1 or (wcx < 0 and right1) or w)

                # pull
                w0, w1 = walls(i)
                src = slot - cy * RS
                o0 = oslot if w0 else src + (dL if cx > 0 else cs if cx < 0 else 0)
                o1 = oslot + cs if w1 else src + (0 if cx > 0 else dR if cx < 0 else cs)
                if not (bottom or top):  # the side path's selects
                    if cx == 0:
                        s0, s1 = src, src + cs
                    elif cx > 0:
                        s0, s1 = oslot if left else src + dL, src if has1 else oslot + cs
                    else:
                        s0, s1 = oslot if right0 else src + cs, oslot + cs if right1 else src + dR
                    assert s0 == o0 and (s1 == o1 or (not has1 and cx == 0))
                    o1 = s1
                for c, o in ((0, o0), (1, o1)):
                    if c and not has1:
                        # padding of the same column (cx = 0: of the row the direction comes from)
                        assert any(p + o == place(x + 1, yy, q, ny, paired)
                                   for yy in (y, y - cy) for q in (i, OPP[i]))
                        continue
                    sx, sy = x + c - cx, y - cy
                    inside = 0 <= sx < nx and 0 <= sy < ny
                    want = place(sx, sy, i, ny, paired) if inside else place(x + c, y, OPP[i], ny, paired)
                    assert p + o == want, (nx, ny, x + c, y, i)
                    loads[c].add(want)
                # push
                w0, w1 = walls(OPP[i])
                out = oslot + cy * RS
                t0 = slot if w0 else out + (cs if cx > 0 else dL if cx < 0 else 0)
                t1 = slot + cs if w1 else out + (dR if cx > 0 else 0 if cx < 0 else cs)
                if not (bottom or top) and cx != 0:
                    t0 = (slot if right0 else out + cs) if cx > 0 else (slot if left else out + dL)
                    t1 = slot + cs if cx > 0 and right1 else out + (dR if cx > 0 else 0)
                for c, o in ((0, t0), (1, t1)):
                    if c and not has1:
                        continue
                    tx, ty = x + c + cx, y + cy
                    inside = 0 <= tx < nx and 0 <= ty < ny
                    want = place(tx, ty, OPP[i], ny, paired) if inside else place(x + c, y, i, ny, paired)
                    assert p + o == want, (nx, ny, x + c, y, i)
                    stores[c].add(want)
                    assert want not in stored
                    stored[want] = 1
            assert loads[0] == stores[0] and loads[1] == stores[1]


@pytest.mark.parametrize("paired", [False, True])
@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 3), (5, 4), (64, 3), (65, 3), (126, 3), (127, 4), (128, 3), (129, 4),
                                   (130, 3), (191, 3), (255, 3), (256, 4), (257, 3), (300, 3)])
def test_pair_offsets_by_path(nx, ny, paired):
    """The pull and the push of a pair as the kernels take them: one path with the wall
    rules for every lane of a warp that touches a side wall and for the bottom and top
    rows, fixed offsets for the others.  A missing second cell loads its own row's padding
    and stores nothing."""
    cs = 2 if paired else 1
    tile = ny * RS
    slot = [(2 * i if paired else i) * TW for i in range(9)]
    pairs = range(0, -(-nx // TW) * TW, 2)  # all lanes of the tiles' warps
    touches = {x: x == 0 or x + 1 >= nx - 1 for x in pairs}
    for x in range(0, nx, 2):
        warp = range(x // 64 * 64, x // 64 * 64 + 64, 2)
        side = any(touches[w] for w in warp)
        lx = x % TW
        dL = cs * (TW - 1) - tile if lx == 0 and x > 0 else -cs
        dR = tile - cs * (TW - 2) if lx == TW - 2 and x + 2 < nx else 2 * cs
        left, right0, right1, has1 = x == 0, x == nx - 1, x + 1 >= nx - 1, x + 1 < nx
        for y in range(ny):
            bottom, top = y == 0, y == ny - 1
            p = place(x, y, 0, ny, paired)

            def wall0(i):
                cx, cy = C[i]
                return (cx > 0 and left) or (cx < 0 and right0) or (cy > 0 and bottom) or (cy < 0 and top)

            def wall1(i):
                cx, cy = C[i]
                return not has1 or (cx < 0 and right1) or (cy > 0 and bottom) or (cy < 0 and top)

            for i, (cx, cy) in enumerate(C):
                o = OPP[i]
                into, own = slot[i] - cy * RS, slot[o]
                out, mine = slot[o] + cy * RS, slot[i]
                if side or bottom or top:
                    pull = (own if wall0(i) else into + (dL if cx > 0 else cs if cx < 0 else 0),
                            own + cs if wall1(i) else into + (0 if cx > 0 else dR if cx < 0 else cs))
                    push = (mine if wall0(o) else out + (cs if cx > 0 else dL if cx < 0 else 0),
                            mine + cs if wall1(o) else out + (dR if cx > 0 else 0 if cx < 0 else cs))
                elif cx == 0:
                    pull, push = (into, into + cs), (out, out + cs)
                else:
                    pull = (into + (dL if cx > 0 else cs), into + (0 if cx > 0 else dR))
                    push = (out + (cs if cx > 0 else dL), out + (dR if cx > 0 else 0))
                for c in (0, 1):
                    if c and not has1:
                        assert p + pull[1] == place(x + 1, y, o, ny, paired)
                        continue
                    for at, sx, sy, there, here in ((pull[c], x + c - cx, y - cy, i, o), (push[c], x + c + cx, y + cy, o, i)):
                        inside = 0 <= sx < nx and 0 <= sy < ny
                        want = place(sx, sy, there, ny, paired) if inside else place(x + c, y, here, ny, paired)
                        assert p + at == want, (nx, ny, x + c, y, i)
