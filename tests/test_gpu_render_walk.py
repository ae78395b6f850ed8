"""The walk of another view's rays through the generating view's columns: columns whose lists a ray's piece misses,
touches and holds, lists of 1 to 33 records around the bisection's sizes, views from 0.5 to 177 degrees (the closest
approach to the generating eye before, inside and behind the volume), against the FP64 oracle's renderer."""
import numpy as np
import pytest

import oracle

from test_gpu_render import Cam, device_regular, gpu_render, rotated

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 8, 17, 33])
def test_columns_missed_touched_and_held(n):
    W, H = 45, 37
    gen = Cam((0.0, 0.0, -3.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), 40.0, W, H)
    rng = np.random.default_rng(n)
    counts, recs = np.zeros(W * H, np.int32), np.zeros((W * H, n, 6))
    for p in range(W * H):
        kind = (p * 7 + p // W) % 5  # none | touching records | records with gaps | one in front | all at the back
        counts[p] = (0, n, n, 1, n)[kind]
        c = counts[p]
        t = np.linspace(0.0, 1.0, 2 * c + 1)
        f, b = (t[:-1:2], t[2::2]) if kind == 1 else (t[:-1:2], t[1::2])
        lo, length = ((2.4, 1.2), (2.4, 1.2), (2.4, 1.2), (2.4, 0.3), (3.4, 0.2))[kind]
        a = rng.uniform(0.2, 0.8) / max(c, 1)  # a list's opacity does not grow with n: extinctions up to about 10
        recs[p, :c, 0], recs[p, :c, 1], recs[p, :c, 5] = lo + length * f, lo + length * b, a
        recs[p, :c, 2:5] = a * rng.random((c, 3))
    recs = recs.astype(np.float32).astype(np.float64)
    reg = device_regular(counts, recs, 0)
    seen = 0
    for theta in (0.5, 5.0, 20.0, 50.0, 90.0, 177.0):
        view = rotated(gen, theta, 41, 31)
        want = oracle.render_view(counts, recs, gen, view)
        # a face at s of about 3 is met within 2^-23: a sliver of that length times an extinction of 16 at most changes
        # hands at each of under 45 + 37 crossings on both sides of the closest approach, and as many roundings
        assert np.abs(gpu_render(reg, gen, view) - want).max() <= 2 * 82 * 2.0 ** -23 * 17, theta
        seen += int((want[:, 3] > 0.05).sum())
    assert seen > 500
