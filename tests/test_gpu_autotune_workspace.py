"""GPU: the plans that autotuning makes share the slice workspace of the batch's own plans,
whichever contraction form those (or the candidates) would take on their own. An odd number
of column blocks, 3 slices: packed in pairs the last block's partner has a place, too."""
import numpy as np
import pytest

import bsmm_gen as G
import paper_1504_05046_gb300 as P
from test_gpu_wide import _is_wide

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own,candidate", [(0, dict(cluster=2, stages=0, fp64_tile=0, store_warps=0)),
                                           (2, dict(cluster=2, stages=0, fp64_tile=0, store_warps=2)),
                                           (2, dict(cluster=1, stages=0, fp64_tile=0, store_warps=0))])
def test_replans_share_the_workspace(own, candidate):
    import torch
    r, c, q = (np.full(n, 128, np.int32) for n in (32, 32, 32))
    c[-1] = 96  # 127 column blocks
    am, bm = np.ones((32, 32), np.uint8), np.ones((32, 32), np.uint8)
    plan = P.bsmm_plan(r, c, q, am, bm, mode=P.BSMM_SPLIT_BF16, nslices=3, cluster=own, ksplit=1)
    assert _is_wide(plan) == (own == 2)
    offs = [G.layout_arena(np.ones((32, 32), np.uint8), a, b) for a, b in ((r, q), (q, c), (r, c))]
    gen = torch.Generator(device="cuda").manual_seed(2)
    A, B = (torch.rand(t, generator=gen, device="cuda", dtype=torch.float64) for _, t in offs[:2])
    C = torch.zeros(offs[2][1], dtype=torch.float64, device="cuda")
    ao, bo, co = (torch.from_numpy(o).cuda() for o, _ in offs)
    P.bsmm_execute(plan, 1.0, A, ao, B, bo, 0.0, C, co)
    P.bsmm_status_device(plan)
    want = C.clone()
    C.zero_()
    batch = P.bsmm_batch_create([plan])
    P.bsmm_batch_set_args(batch, [1.0], [A], [ao], [B], [bo], [0.0], [C], [co])
    P.bsmm_batch_execute(batch)  # the kernels' code is on the device
    P.bsmm_batch_status_device(batch)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    P.bsmm_batch_autotune(batch, [candidate], reps=1)
    torch.cuda.synchronize()
    grown = before - torch.cuda.mem_get_info()[0]
    C.zero_()
    P.bsmm_batch_execute(batch)
    P.bsmm_batch_status_device(batch)
    assert bool((C == want).all())
    workspace = 2 * 3 * 2 * 4096 * 4064  # A's and B's slices, about
    assert grown < workspace // 4, (grown, workspace)
