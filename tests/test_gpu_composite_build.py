"""The pooled schedule's builds and packed search against the direct sweep, bit for bit, where they change hands: the
longest pixel of a 32-pixel batch at the single warps' limit (288 records) and at the stage's (1024), batches that end
early, records without length, opaque records, fronts at depth 0, one slot and more slots than pieces."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

K = 11


def _sets(lengths, seed):
    """Per PE (counts, offsets, fb, rgba): a pixel's records dealt out to the PEs in turn."""
    rng = np.random.default_rng(seed)
    out = []
    for e in range(K):
        cnt = np.array([(n + K - 1 - e) // K for n in lengths], dtype=np.int32)
        off = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int64)
        fbs, cols = [], []
        for c in cnt:
            t = np.sort(rng.integers(0, 1 << 20, 2 * c)).astype(np.float32) / np.float32(1 << 20)
            if c and e == 0:
                t[0] = 0.0
            fbs.append(t.reshape(c, 2))  # equal neighbours give records with b = f
            a = rng.random((c, 1), dtype=np.float32)
            a[rng.random((c, 1)) < 0.02] = 1.0
            a[rng.random((c, 1)) < 0.02] = 0.0
            cols.append(np.concatenate([a * rng.random((c, 3), dtype=np.float32), a], axis=1))
        out.append((cnt, off, np.concatenate(fbs), np.concatenate(cols).astype(np.float32)))
    return out


@pytest.mark.parametrize("longest", [1, 287, 288, 289, 1023, 1024, 1025])
@pytest.mark.parametrize("n_s", [1, 20])
def test_pooled_equals_direct(longest, n_s):
    import torch

    import paper_2206_14503_gb300 as vdi

    # three batches: the long pixel among short and empty ones, short ones only, six pixels
    lengths = [longest if p == 5 else (p * 7) % 40 for p in range(32)] + [p % 30 for p in range(32)] + [0, 1, 2, 30, 3, 0]
    npix = len(lengths)
    pes = [vdi.Compact.from_tensors(*(torch.from_numpy(a).cuda() for a in (c, o, r, f)))
           for c, o, f, r in _sets(lengths, 7 * longest + n_s)]
    structs = [p.struct() for p in pes]
    got = {}
    for sched in (vdi.VDI_SCHED_STAGED, 2):
        reg = vdi.Regular(npix, n_s)
        ws = vdi.Workspace(vdi.vdi_composite_workspace(K, npix, 1, n_s))
        vdi.check(vdi.vdi_composite(structs, npix, 1, reg.struct(), vdi.make_params(schedule=sched), ws.ptr, ws.nbytes),
                  "composite")
        vdi.check(ws.status(), "status")
        got[sched] = reg
    a, b = got[vdi.VDI_SCHED_STAGED], got[2]
    assert int(b.counts.sum()) > 0
    for name in ("counts", "gamma", "fb", "rgba"):
        x, y = getattr(a, name), getattr(b, name)
        assert torch.equal(x.view(torch.int32), y.view(torch.int32)), name
