"""GPU: a batch's contraction is the 32-column form, whatever form its plans run on their own.
Plans whose own executes pack column blocks in pairs (3 and 4 slices) are packed block by
block there: the same bits, and no slower than plans without pairs."""
import numpy as np
import pytest

import bsmm_gen as G
import paper_1504_05046_gb300 as P
from test_gpu_wide import _is_wide

pytestmark = pytest.mark.gpu


def _tiles(n, b):
    return np.asarray([b] * (n // b) + ([n % b] if n % b else []), np.int32)


def _batch(s, cluster, sizes):
    import torch
    plans, args = [], []
    for n in sizes:
        t, q = _tiles(n, 128), _tiles(n, 256)
        am, bm = np.ones((len(t), len(q)), np.uint8), np.ones((len(q), len(t)), np.uint8)
        plan = P.bsmm_plan(t, t, q, am, bm, mode=P.BSMM_SPLIT_BF16, nslices=s, cluster=cluster)
        assert _is_wide(plan) == (cluster > 1)
        gen = torch.Generator(device="cuda").manual_seed(n)
        offs = [G.layout_arena(m, a, b) for m, a, b in ((am, t, q), (bm, q, t), (np.ones((len(t), len(t)), np.uint8), t, t))]
        A, B = (torch.rand(tot, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1 for _, tot in offs[:2])
        C = torch.zeros(offs[2][1], dtype=torch.float64, device="cuda")
        ao, bo, co = (torch.from_numpy(o).cuda() for o, _ in offs)
        plans.append(plan)
        args.append((A, ao, B, bo, C, co))
    batch = P.bsmm_batch_create(plans)
    k = len(plans)
    P.bsmm_batch_set_args(batch, [1.0] * k, *[[a[i] for a in args] for i in range(4)], [0.0] * k,
                          [a[4] for a in args], [a[5] for a in args])
    return batch, plans, args


def _us(batch, passes=10):
    import torch
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(passes):
        P.bsmm_batch_execute(batch)
    b.record()
    torch.cuda.synchronize()
    return 1000 * a.elapsed_time(b) / passes


def test_pairs_cost_a_batch_nothing():
    """3 slices, where the copies of a chunk cost most: 1600 us against 1312 when the batch took
    the pairs slice by slice; the bound leaves half of that difference to noise."""
    sizes = (2048, 2048, 2560, 3072)
    pairs, plans, args = _batch(3, 2, sizes)
    single, _, sargs = _batch(3, 0, sizes)
    ratio = []
    for _ in range(9):
        ratio.append(_us(pairs) / _us(single))
    P.bsmm_batch_status_device(pairs)
    P.bsmm_batch_status_device(single)
    for a, b in zip(args, sargs):
        assert bool((a[4] == b[4]).all())
    assert np.median(ratio) <= 1.1, ratio
    # a plan's own execute between two of the batch packs the same workspace in pairs
    A, ao, B, bo, C, co = args[0]
    want = C.clone()
    C.zero_()
    P.bsmm_execute(plans[0], 1.0, A, ao, B, bo, 0.0, C, co)
    P.bsmm_status_device(plans[0])
    assert bool((C == want).all())
    C.zero_()
    P.bsmm_batch_execute(pairs)
    P.bsmm_batch_status_device(pairs)
    assert bool((C == want).all())
