"""The batched call's pool, sized from the outputs' N_S, with lists of other lengths: a long pixel among short ones takes
a run of its own and leaves the others their room; what does not fit is swept directly; the bits are the direct sweep's."""
import numpy as np
import pytest

from gpu_run import compact_from_numpy

pytestmark = pytest.mark.gpu

LIST_AT = 512  # the list in the workspace: [entries, ...] 8 words, then entries of 8 words, the first word's top bit: direct


def _lists(lengths, k, seed):
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(k):
        cnt = np.asarray(lengths, np.uint32)
        off = np.concatenate([[0], np.cumsum(cnt)]).astype(np.uint64)
        fb = np.concatenate([np.sort(rng.random(2 * n)).reshape(n, 2) for n in lengths]).astype(np.float32)
        a = rng.random((len(fb), 1))
        out.append((cnt, off, fb, np.concatenate([a * rng.random((len(fb), 3)), a], axis=1).astype(np.float32)))
    return out


# (K, N_S, records per list of the short pixels, of one pixel in 32, whether every pixel's pieces fit the pool)
@pytest.mark.parametrize("k,n_s,short,long,fits", [(16, 8, 4, 60, True), (16, 8, 24, 24, False), (64, 4, 1, 16, True),
                                                   (12, 2, 4, 30, False), (9, 6, 6, 6, True)])
@pytest.mark.parametrize("prec", [0, 1])
def test_lists_longer_than_the_output(k, n_s, short, long, fits, prec):
    import torch

    import paper_2206_14503_gb300 as vdi

    w, h = 64, 33
    lengths = [long if p % 32 == 11 else short for p in range(w * h - 9)] + [0] * 9
    pes = [compact_from_numpy(*l, 2 if prec else 1) for l in _lists(lengths, k, k + long)]
    structs = [p.struct() for p in pes]
    direct, reg = vdi.Regular(w * h, n_s, prec), vdi.Regular(w * h, n_s, prec)
    ws = vdi.Workspace(vdi.vdi_composite_workspace(k, w, h, n_s))
    vdi.check(vdi.vdi_composite(structs, w, h, direct.struct(), vdi.make_params(schedule=2), ws.ptr, ws.nbytes), "direct")
    vdi.check(ws.status(), "direct status")
    host = vdi.vdi_batch_table_pack(vdi.Requests([(structs, w, h, reg.struct(), 0)]))
    dev = torch.frombuffer(bytearray(host), dtype=torch.uint8).cuda()
    wb = vdi.Workspace(vdi.vdi_composite_batched_workspace(host))
    vdi.check(vdi.vdi_composite_batched(dev.data_ptr(), host, vdi.make_params(), wb.ptr, wb.nbytes), "batched")
    vdi.check(wb.status(), "batched status")
    for name in ("counts", "gamma", "rgba") + (() if prec else ("fb",)):
        assert torch.equal(getattr(reg, name).view(torch.int32), getattr(direct, name).view(torch.int32)), name
    words = wb.buf[LIST_AT:].view(torch.int32)
    n = int(words[0])
    swept = int((words[8:8 + 8 * n].view(n, 8)[:, 0] < 0).sum())
    assert n == w * h - 9
    assert (swept == 0) == fits
