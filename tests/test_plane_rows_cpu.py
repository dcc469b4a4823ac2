"""Host model of the shifted-plane sweeps' row table and frames (no GPU).

A stored frame has nx columns and, per block, the rows of its band and one halo
row (the next band's first row, or row 0 after the last band).  The row table
gives each row of a block's band the block and row that store it and, for the
first row of a band, the halo row of the band before; a node's column is
shifted modulo nx.  The next step reads the corners of node (x, y) at columns x and
x + 1 (0 for x + 1 = nx) of rows y and y + 1 of its own block.

This replays that arithmetic (fill_dest, shifted and the reads of plane_sweep.cuh,
which plane_var.cuh and ml_plane.cuh share) for every shift of many planes and checks
that every position of every frame is written exactly once, that each corner read
holds the node it should, that bands beyond a block's rows are never addressed, and
that the bytes a block posts on its mbarrier before a plane arrives (nx vectors for each
stored row whose source row belongs to another block) are what the others send.
"""

import pytest


def band_of(y, rows):
    magic = ((1 << 32) + rows - 1) // rows
    return (y * magic) >> 32


def replay(nx, ny, nb, sx, sy):
    rows = -(-ny // nb)
    lastrows = ny - (nb - 1) * rows
    frame, received = {}, [0] * nb
    for rank in range(nb):
        y0 = rank * rows
        for yl in range(min(rows, ny - y0)):
            ys = y0 + yl - sy
            ys += ny if ys < 0 else 0
            ob = band_of(ys, rows) if nb > 1 else 0
            lr = ys - ob * rows
            targets = [(ob, lr)]
            if lr == 0:
                hb = nb - 1 if ob == 0 else ob - 1
                targets.append((hb, lastrows if hb == nb - 1 else rows))
            for block, row in targets:
                assert 0 <= row <= rows
                received[block] += nx if block != rank else 0
                for x in range(nx):
                    xs = x - sx
                    key = (block, row, xs + nx if xs < 0 else xs)
                    assert key not in frame, key
                    frame[key] = (x, y0 + yl)
    for rank in range(nb):
        y0 = rank * rows
        myrows = min(rows, ny - y0)
        for yl in range(myrows):
            for x in range(nx):
                x1 = 0 if x + 1 == nx else x + 1
                for row, col, dx, dy in ((yl, x, 0, 0), (yl, x1, 1, 0), (yl + 1, x, 0, 1),
                                         (yl + 1, x1, 1, 1)):
                    want = ((x + dx + sx) % nx, (y0 + yl + dy + sy) % ny)
                    assert frame[(rank, row, col)] == want, (nx, ny, nb, sx, sy)
        posted = 0
        for j in range(myrows + 1):
            ys = y0 + j if j < myrows else (0 if rank == nb - 1 else y0 + rows)
            src = ys + sy
            src -= ny if src >= ny else 0
            posted += nx if band_of(src, rows) != rank else 0
        assert posted == received[rank], (nx, ny, nb, sx, sy, rank)
    assert len(frame) == (ny + nb) * nx


@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 3), (3, 5), (8, 13), (12, 16), (5, 31)])
def test_every_position_once_corners_and_counts(nx, ny):
    for nb in range(1, 17):
        if nb > ny or (nb - 1) * -(-ny // nb) >= ny:
            continue
        for sx in range(nx):
            for sy in range(ny):
                replay(nx, ny, nb, sx, sy)
