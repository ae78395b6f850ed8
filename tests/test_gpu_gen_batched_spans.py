"""Batched generation's recorded spans: emission over them writes the records of emission over every sample."""
import numpy as np
import pytest

import synth

from gpu_run import to_dev

pytestmark = pytest.mark.gpu


# searched and fixed gamma, both precisions, images that end inside a tile; the second request's spans start after
# the first one's
@pytest.mark.parametrize("prec", [0, 1])
def test_batched_spans_change_no_record(prec):
    import torch

    import paper_2206_14503_gb300 as vdi

    lut_d = to_dev(synth.transfer_function(synth.SEED_TF))
    keep, items, outs = [], [], {True: [], False: []}
    for r, (dims, grid, (W, H), n_s, gamma) in enumerate([((48, 40, 56), (2, 1, 2), (72, 61), 5, -1.0),
                                                          ((40, 64, 33), (1, 3, 1), (37, 90), 9, 0.02)]):
        br = vdi.Bricks(to_dev(synth.volume(dims, 12, 3, 900 + r, np.uint16)), dims, vdi.vdi_split_boxes(dims, grid))
        keep.append(br)
        for spans in (True, False):
            outs[spans].append([vdi.Compact(W * H, W * H * n_s, prec) for _ in br.boxes])
        items.append((br, vdi.make_camera(synth.orbit(dims, 1, W, H, 70 + r)[0]), n_s, gamma))
    for spans in (True, False):
        R = vdi.GenRequests([(br.bricks, lut_d.data_ptr(), cam, n_s, gamma, [o.struct() for o in os_])
                             for (br, cam, n_s, gamma), os_ in zip(items, outs[spans])])
        host = vdi.vdi_gen_batch_table_pack(R, vdi.make_params())
        dev = torch.frombuffer(bytearray(host), dtype=torch.uint8).cuda()
        full = vdi.vdi_generate_batched_workspace(host)
        ws = vdi.Workspace(full)
        size = full if spans else full - 512  # (sizes are rounded to 256: the cache still fits, the spans do not)
        vdi.check(vdi.vdi_generate_batched(dev.data_ptr(), host, ws.ptr, size), "batched")
        vdi.check(ws.status(), "status")
    for a, b in zip(outs[True], outs[False]):
        for x, y in zip(a, b):
            assert torch.equal(x.counts, y.counts) and torch.equal(x.offsets, y.offsets)
            assert int(x.offsets[-1]) > 0
            assert torch.equal(x.gamma, y.gamma) and torch.equal(x.rgba, y.rgba)
            assert prec == 1 or torch.equal(x.fb, y.fb)
