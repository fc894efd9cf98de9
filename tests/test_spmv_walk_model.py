"""CPU model of the lane-walk SpMV kernel's row assembly, on the oracle's own plan.

A warp takes a unit of c tiles.  Per tile every lane walks its steps (rows that begin and end
in the lane are written; its first row end and its open run are kept), the open runs are
joined by a segmented scan whose steps stop with the longest run, and the run open after the
tile is carried into the next tile of the unit.  The unit's first row and the row open at its
end go to an accumulator found through the tile slots (the first tile boundary in that row);
each distinct row of the unit boundaries is written once, at its first boundary.

Every row has to be written exactly once and equal the oracle's product, for every unit."""
import numpy as np
import pytest

import inputs
import oracle

MSB = 0x80000000


def _scan(a, head):
    """The kernel's shuffle scan, with its distances and its early end."""
    start, last = [], 0
    for l in range(32):
        last = l if head[l] else last
        start.append(last)
    run = sum(1 << l for l in range(1, 32) if not head[l])
    o = 1
    while o < 32 and run:
        a = [a[l] + a[l - o] if o <= l - start[l] else a[l] for l in range(32)]
        run &= run >> o
        o <<= 1
    return a


def _model(a, x, sigma, c):
    t = oracle.build_tile(a.row_ptr, sigma)
    T, n = t["tile_num"], a.n_rows
    tx, ty = t["tile_x"].astype(np.int64), t["tile_y"].astype(np.int64)
    rows = ty & ~MSB
    slot = np.searchsorted(rows, rows, side="left")
    desc = t["lane_desc"].astype(np.int64)
    steps = int(a.row_ptr[-1]) + n
    prod = a.val * x[a.col]
    y, writes, acc = np.zeros(n), np.zeros(n, np.int64), np.zeros(T + 1)
    for u0 in range(0, T, c):
        u1, carry = min(u0 + c, T), 0.0
        y_unit = int(rows[u0])
        for ti in range(u0, u1):
            x0, y_ws, n_t = tx[ti], int(rows[ti]), int(rows[ti + 1] - rows[ti])
            if ty[ti] & MSB:
                carry += float(prod[x0:tx[ti + 1]].sum())
                assert n_t == 0
                continue
            sy = np.full(n_t, np.nan)
            A, head, hsum, y0s = [], [], [], []
            for lane in range(32):
                j = ti * 32 + lane
                d = int(desc[j]) if j < t["lane_num"] else 0
                ln = min(sigma, steps - j * sigma) if j < t["lane_num"] else 0
                dm, xo, y0 = (d >> 18) & ((1 << ln) - 1), d & 511, (d >> 9) & 511
                s, h, nd = 0.0, 0.0, 0
                for k in range(ln):
                    if (dm >> k) & 1:
                        if nd == 0:
                            h = s
                        else:
                            sy[y0 + nd] = s
                        s, nd = 0.0, nd + 1
                    else:
                        s += prod[x0 + xo + k - nd]
                A.append(s)
                head.append(dm != 0)
                hsum.append(h)
                y0s.append(y0)
            if not head[0]:
                A[0] += carry
            A = _scan(A, head)
            for lane in range(32):
                if head[lane]:
                    sy[y0s[lane]] = hsum[lane] + (carry if lane == 0 else A[lane - 1])
            carry = A[31]
            for r in range(n_t):
                if y_ws + r == y_unit:
                    acc[slot[u0]] += sy[r]
                else:
                    y[y_ws + r] = sy[r]
                    writes[y_ws + r] += 1
        if rows[u1] < n:
            acc[slot[u1]] += carry
    bounds = [min(k * c, T) for k in range(-(-T // c) + 1)]
    for k, i in enumerate(bounds):
        r = int(rows[i])
        if r < n and (k == 0 or rows[bounds[k - 1]] != r):
            y[r] = acc[slot[i]]
            writes[r] += 1
    return y, writes


CASES = {
    "rmat9_hubs": lambda: inputs.add_hubs(inputs.rmat_uniform(9, 8, 3, 3), 2, 600, 1500, 5),
    "ragged": lambda: inputs.row_lengths_csr([0, 1, 900, 0, 0, 3, 448, 447, 449, 0, 13, 14, 15] * 3, 1200, 2),
    "one_row": lambda: inputs.row_lengths_csr([5000], 6000, 3),
    "empty30": lambda: inputs.empty_rows(inputs.rmat_uniform(8, 16, 4, 4), 0.3, 4),
}


@pytest.mark.parametrize("c", [1, 2, 4, 8])
@pytest.mark.parametrize("sigma", [14, 5])
@pytest.mark.parametrize("case", sorted(CASES))
def test_units_write_every_row_once(case, sigma, c):
    a = CASES[case]()
    x = np.random.default_rng(1).random(a.n_cols)
    y, writes = _model(a, x, sigma, c)
    assert (writes == 1).all(), np.flatnonzero(writes != 1)[:10]
    ref, d = oracle.spmv(a.row_ptr, a.col, a.val, x)
    assert oracle.relative_errors(y, ref, d).max() <= 1e-12


@pytest.mark.parametrize("sigma", [14, 5])
@pytest.mark.parametrize("case", sorted(CASES))
def test_tile_shares_add_up_to_the_rows(case, sigma):
    """The one-launch PageRank stores, per tile, its share of its first row (if the row ends in
    it) and of the row open at its end; the first tile that starts in a row adds them up."""
    a = CASES[case]()
    x = np.random.default_rng(1).random(a.n_cols)
    t = oracle.build_tile(a.row_ptr, sigma)
    T, n = t["tile_num"], a.n_rows
    tx, rows = t["tile_x"].astype(np.int64), t["tile_y"].astype(np.int64) & ~MSB
    prod = a.val * x[a.col]
    y, writes = np.zeros(n), np.zeros(n, np.int64)
    head, tail = np.full(T, np.nan), np.full(T, np.nan)
    for i in range(T):
        for r in range(rows[i], rows[i + 1]):
            s = float(prod[max(tx[i], a.row_ptr[r]):a.row_ptr[r + 1]].sum())
            if r == rows[i]:
                head[i] = s
            else:
                y[r] = s
                writes[r] += 1
        last = rows[i + 1]
        tail[i] = float(prod[max(tx[i], a.row_ptr[last]) if last < n else tx[i + 1]:tx[i + 1]].sum())
    for i in range(T):
        if np.searchsorted(rows, rows[i], side="left") == i:
            span = int(np.searchsorted(rows, rows[i], side="right")) - i
            y[rows[i]] = head[i + span - 1] + sum(tail[i + q - 1] for q in range(span) if i + q > 0)
            writes[rows[i]] += 1
    assert (writes == 1).all()
    ref, d = oracle.spmv(a.row_ptr, a.col, a.val, x)
    assert oracle.relative_errors(y, ref, d).max() <= 1e-12
