"""The records that the K^T kernel reads (pat_adjoint_records; host only): they hold every ray segment
of the work list exactly once, start at even radius indexes inside their data rows, and what they add
to a segment (a point before it or after it, for pairs) has no tap in the tile."""
import math

import numpy as np
import pytest

import paper_1707_02245_gb300 as P
import synthetic as S

WTILE, AROWS, STEP, EXACT = 32, 4, 16, 1 << 24


def _tables(n, det_xy, quad_m, extent):
    (xmin, xmax, ymin, ymax) = extent
    hx, hy = (xmax - xmin) / n, (ymax - ymin) / n
    det = np.stack([(det_xy[:, 0] - xmin) / hx - 0.5, (det_xy[:, 1] - ymin) / hy - 0.5], 1).astype(np.float32)
    phi = 2 * math.pi * (np.arange(quad_m) + 0.5) / quad_m
    return det, np.stack([np.cos(phi) / hx, np.sin(phi) / hy], 1).astype(np.float32)


def _check(n, det_xy, n_t, r0, dr, quad_m, slots, extent=(-1.0, 1.0, -1.0, 1.0)):
    det_xy = np.asarray(det_xy, dtype=np.float64)
    ref = P.pat_adjoint_worklist(n, det_xy, n_t, r0, dr, quad_m, slots, extent)["rays"]
    got = P.pat_adjoint_records(n, det_xy, n_t, r0, dr, quad_m, slots, extent)
    rec, items = got["records"], got["items"]
    det, cs = _tables(n, det_xy, quad_m, extent)
    tp = n_t + n_t % 2
    tiles_x = (n + WTILE - 1) // WTILE

    # items: consecutive records, whole groups of the first kind
    assert np.array_equal(items[:, 1], np.concatenate([[0], np.cumsum(items[:-1, 2])])) and items[:, 2].sum() == rec.size
    assert np.all(items[:, 3] % AROWS == 0) and np.all((0 <= items[:, 3]) & (items[:, 3] <= items[:, 2]))
    tile = np.repeat(items[:, 0], items[:, 2])
    second = np.arange(rec.size) - np.repeat(items[:, 1], items[:, 2]) >= np.repeat(items[:, 3], items[:, 2])
    for t, first, count, split in items:
        for a, b in ((first, first + split), (first + split, first + count)):
            assert np.all(np.diff(rec["n"][a:b]) <= 0), "longest first"
        pad = np.flatnonzero(rec["n"][first:first + count] == 0)
        assert pad.size < AROWS or count == pad.size
        assert np.all(pad < split) and np.all(np.diff(pad) == 1) and (not pad.size or pad[-1] == split - 1)
        assert not rec[first + pad].tobytes().strip(b"\0")

    full = rec["n"] > 0
    r, t_, sec = rec[full], tile[full], second[full]
    k = r["k"].astype(np.int64)
    d = r["yraw"].astype(np.int64) // n_t
    assert np.array_equal(r["yraw"] - d * n_t, k) and np.array_equal(r["ypad"], d * tp + k)
    assert np.all(k % 2 == 0) and np.all(k >= 0) and np.all(k + r["n"] <= n_t)
    assert np.all((k + r["n"] <= EXACT) | ((r["n"] <= STEP) & (k % STEP == 0)))
    # axes: detector and angle from the floats, the faster one first
    dirs = {}
    for m, (c, s) in enumerate(cs):
        dirs.setdefault((c.tobytes(), s.tobytes()), []).append(m)
    x = np.where(sec, r["cs"], r["cm"]).astype(np.float32)
    y = np.where(sec, r["cm"], r["cs"]).astype(np.float32)
    assert np.array_equal(np.where(sec, r["ds"], r["dm"]), det[d, 0]) and np.array_equal(np.where(sec, r["dm"], r["ds"]), det[d, 1])
    assert np.all(np.where(sec, np.abs(y) > np.abs(x), np.abs(x) >= np.abs(y)))
    m = []
    for c, s in zip(x, y):
        q = dirs[(c.tobytes(), s.tobytes())]
        assert len(q) == 1
        m.append(q[0])
    m = np.array(m, dtype=np.int64)

    # the list's segments, per (tile, detector, angle): each once and whole
    seg = {}
    tnum, i = 0, 0
    for row, nxt in zip(ref, np.vstack([ref[1:], ref[-1:]])):
        if row[0] < 0:
            tnum += 1
            continue
        seg[(tnum, int(row[0]), int(row[1]))] = (int(row[2]), int(row[2]) + int(nxt[3]) - int(row[3]))
    have = {}
    for tt, dd, mm, kk, nn in zip(t_, d, m, k, r["n"]):
        have.setdefault((int(tt), int(dd), int(mm)), []).append((int(kk), int(kk) + int(nn)))
    assert have.keys() == seg.keys()
    dr_f, rh_f = np.float32(dr), np.float32(r0 + 0.5 * dr)

    def in_tile(tt, dd, mm, kk):
        rk = np.float32(np.float64(np.float32(kk)) * np.float64(dr_f) + np.float64(rh_f))
        fx = np.float32(np.float64(rk) * np.float64(cs[mm, 0]) + np.float64(det[dd, 0]))
        fy = np.float32(np.float64(rk) * np.float64(cs[mm, 1]) + np.float64(det[dd, 1]))
        li, lj = math.floor(fx) - (tt % tiles_x) * WTILE + 1, math.floor(fy) - (tt // tiles_x) * WTILE + 1
        return 0 <= li <= WTILE and 0 <= lj <= WTILE

    for key, (a, b) in seg.items():
        pieces = sorted(have[key])
        assert pieces[0][0] == a - a % (STEP if b > EXACT else 2) and pieces[-1][1] == b
        assert all(p[1] == q[0] for p, q in zip(pieces, pieces[1:]))
        assert len(pieces) == 1 or b > EXACT
        assert not any(in_tile(*key, kk) for kk in range(pieces[0][0], a))
        if (b - pieces[0][0]) % 2 and b < n_t:
            assert not in_tile(*key, b)
    return r


def _circle(n_det, radius):
    a = 2 * math.pi * (np.arange(n_det) + 0.5) / n_det
    return np.stack([radius * np.cos(a), radius * np.sin(a)], 1)


@pytest.mark.parametrize("n,n_det,radius,n_t,m,slots", [(64, 12, 1.2, 127, 96, 304), (33, 5, 0.4, 64, 100, 304), (72, 7, 1.2, 95, 64, 3),
                                                        (2, 1, 1.2, 1, 16, 304), (40, 3, 9.0, 31, 72, 16)])
def test_records_hold_every_segment_once(n, n_det, radius, n_t, m, slots):
    det = _circle(n_det, radius)
    r0, dr = S.radial_sampling(det, n_t)
    _check(n, det, n_t, r0, dr, m, slots)


def test_records_non_square_extent():
    det = np.array([[2.0, 0.0], [0.0, 2.5], [-1.5, -1.0], [0.3, 1.2]])
    _check(40, det, 91, 0.1, 0.05, 112, 24, extent=(-1.5, 1.0, -0.5, 1.5))


def test_records_of_an_image_that_no_circle_meets():
    det = np.array([[50.0, 0.0]])
    got = P.pat_adjoint_records(16, det, 4, 0.0, 0.1, 16, 8)
    assert got["items"].tolist() == [[0, 0, 0, 0]] and got["records"].size == 0


def test_records_past_the_exact_radius_indexes():
    """A detector 2000 image sides away with 2^24 + 4001 radii: the image lies on both sides of index
    2^24, where FP32 holds every second integer only."""
    n_t = EXACT + 4001
    phi = 2 * math.pi * 0.5 / 16
    dist = 2000.0
    det = np.array([[-dist * math.cos(phi), -dist * math.sin(phi)]])
    dr = dist / (EXACT - 3000)
    r = _check(32, det, n_t, 0.0, dr, 16, 304)
    assert np.any(r["k"] + r["n"] > EXACT)


def test_records_reject_bad_input():
    with pytest.raises(P.PatError):
        P.pat_adjoint_records(16, np.array([[1.5, 0.0]]), 8, 0.0, 0.4, 16, slots=0)
    with pytest.raises(P.PatError):
        P.pat_adjoint_records(1, np.zeros((1, 2)), 10, 0.0, 0.1, 16, slots=8)
