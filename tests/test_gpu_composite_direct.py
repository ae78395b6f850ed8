"""Pixels that the searches over pooled pieces leave to the direct sweeps give the bits of those schedules."""
import numpy as np
import pytest

from gpu_run import compact_from_numpy

pytestmark = pytest.mark.gpu


def _compact(pixels, e):
    """PE e's (counts, offsets, fb, rgba) of pixels[p][e] = [(f, b, R, G, B, A), ...]."""
    rows = [np.asarray(p[e], np.float64).reshape(-1, 6) for p in pixels]
    cnt = np.array([len(r) for r in rows], np.uint32)
    off = np.concatenate([[0], np.cumsum(cnt)]).astype(np.uint64)
    rec = np.concatenate(rows).astype(np.float32)
    return cnt, off, rec[:, :2], rec[:, 2:]


def _run(lists, prec, n_s, schedule):
    import paper_2206_14503_gb300 as vdi

    pes = [compact_from_numpy(*l, 2 if prec else 1) for l in lists]
    npix = len(lists[0][0])
    reg = vdi.Regular(npix, n_s, prec)
    ws = vdi.Workspace(vdi.vdi_composite_workspace(len(pes), npix, 1, n_s))
    vdi.check(vdi.vdi_composite([p.struct() for p in pes], npix, 1, reg.struct(), vdi.make_params(schedule=schedule),
                                ws.ptr, ws.nbytes), f"schedule {schedule}")
    out = [reg.counts, reg.gamma, reg.rgba] + ([] if prec else [reg.fb])
    return [a.cpu().numpy().view(np.int32) for a in out] + [np.int32(ws.status())]


def _sorted(rng, n):
    t = np.sort(rng.integers(0, 1 << 20, 2 * n)).reshape(n, 2) / float(1 << 20)
    a = rng.random((n, 1))
    return np.concatenate([t, a * rng.random((n, 3)), a], axis=1)


def _same(lists, prec, n_s, direct, schedules):
    ref = _run(lists, prec, n_s, direct)
    assert ref[0].max() > 0
    for s in schedules:
        for x, y in zip(ref, _run(lists, prec, n_s, s)):
            assert np.array_equal(x, y), s


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("steps", [1, 5, 60, 470])
def test_lists_out_of_depth_order(steps, prec):
    # every other record of PE 0 steps back to the front: the sweep of 470 of them cuts more than 2047 pieces.  (What
    # such lists give depends on the sweep: the lane schedule leaves them to schedule 1's, the pooled one to 2's.)
    import paper_2206_14503_gb300 as vdi

    rng = np.random.default_rng(steps)
    k, pixels = 8, []
    for p in range(70):
        lists = [_sorted(rng, 4) for _ in range(k)]
        if p % 7 == 3:
            back = _sorted(rng, steps)
            back[0::2, :2] = 0.95, 0.96
            back[1::2, :2] = 0.0, 0.0001
            lists = [back] + [np.concatenate([[0.1 * e, 2.0 + e], r[0, 2:]])[None] for e, r in enumerate(lists[1:], 1)]
        pixels.append(lists)
    lists = [_compact(pixels, e) for e in range(k)]
    _same(lists, prec, 4, 1, (vdi.VDI_SCHED_LANE,))
    _same(lists, prec, 4, 2, (vdi.VDI_SCHED_STAGED,))


ODD = {"opacity above 1": (5, 1.5), "opacity NaN": (5, np.nan), "colour NaN": (3, np.nan), "colour infinite": (2, np.inf),
       "colour large": (2, 3e30), "colour -0": (3, -0.0), "front -0": (0, -0.0), "opacity negative": (5, -0.5),
       "back far": (1, 1e20)}


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("k", [8, 11])
@pytest.mark.parametrize("kind", sorted(ODD) + ["short behind opaque"])
def test_values_outside_the_packed_search(kind, k, prec):
    # one odd record, a piece by itself, and plain ones behind it, whose supersegments are as the direct sweep gives them
    import paper_2206_14503_gb300 as vdi

    rng = np.random.default_rng(len(kind) + k)
    pixels = []
    for p in range(40):
        lists = [_sorted(rng, 5) for _ in range(k)]
        for r in lists:
            r[:, :2] += 2.0  # behind the odd record, whose depths are 0 to 1
        if p % 3 == 1:
            rec = np.array([[0.0, 1.0, 0.25, 0.5, 0.125, 0.5]])
            if kind == "short behind opaque":
                # 1e-36 of the opaque record's length
                rec = np.array([[-1.0, 0.0, 0.25, 0.5, 0.125, 1.0], [0.0, 1e-36, 0.5, 0.0, 0.125, 0.5]])
            else:
                at, v = ODD[kind]
                rec[0, at] = v
            if kind == "back far":  # the last of its list
                rec[0, 0] = 10.0
            e = p % k
            lists[e] = np.concatenate([lists[e], rec] if kind == "back far" else [rec, lists[e]])
        pixels.append(lists)
    with np.errstate(invalid="ignore", over="ignore", divide="ignore"):
        lists = [_compact(pixels, e) for e in range(k)]
        _same(lists, prec, 3, 2, (vdi.VDI_SCHED_STAGED,) + ((1, vdi.VDI_SCHED_LANE) if k <= 8 else ()))


@pytest.mark.parametrize("n", [3, 26, 33, 93])
@pytest.mark.parametrize("full", [0.1, 0.9])
def test_records_without_length(n, full):
    # the pooled builds (one warp up to 288 records a pixel, four above) move the others forward over the empty ones
    import paper_2206_14503_gb300 as vdi

    rng = np.random.default_rng(n)
    k, pixels = 11, []
    for p in range(45):
        lists = [_sorted(rng, n) for _ in range(k)]
        for r in lists:
            r[rng.random(n) > full, 1] = 0.0
        pixels.append(lists)
    _same([_compact(pixels, e) for e in range(k)], 0, 5, 2, (vdi.VDI_SCHED_STAGED,))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("total", [287, 288, 289, 1023, 1024, 1025])
def test_stage_limits_of_many_lists(total, prec):
    # K = 64 (every lane of the count's two loads), the longest pixel at the limits of one warp's stage and of four's
    import paper_2206_14503_gb300 as vdi

    rng = np.random.default_rng(total)
    k = 64
    pixels = [[_sorted(rng, (total + k - 1 - e) // k if p in (3, 40) else (p + e) % 3) for e in range(k)] for p in range(44)]
    _same([_compact(pixels, e) for e in range(k)], prec, 7, 2, (vdi.VDI_SCHED_STAGED,))
