"""Back-to-back calls on one handle that switch between the streaming and the
tensor-core kernels (and their batch tiles) on one stream, with no
synchronisation in between: the per-handle counters that each launch re-arms
in its last CTA, and programmatic dependent launch across kernels, must leave
every result equal to what the same call gives alone."""
import numpy as np
import pytest

import oracle
from acceptance import check_topk
from gpu_cases import to_device_bits, workload

pytestmark = pytest.mark.gpu

CALLS = [(1, 50), (4, 50), (1, 300), (40, 50), (1, 50), (9, 128), (2, 1), (64, 64), (3, 300), (1, 7)]


@pytest.mark.parametrize("storage", ["bf16", "e4m3"])
def test_mixed_paths_back_to_back(vie, storage):
    import torch
    V, d = 30011, 512
    W, h = workload(V, d, 64, seed=83)
    hd = torch.from_numpy(h).cuda()
    with vie.Head(to_device_bits(W), storage=storage) as head:
        # each call alone first
        alone = []
        for b, k in CALLS:
            i, v = head.topk(hd[:b], k)
            torch.cuda.synchronize()
            alone.append((i.cpu().numpy(), v.cpu().numpy()))
        paths = {head.plan(b, k).path for b, k in CALLS}
        assert paths == {0, 1}
        # then all of them back to back, twice over, sparse tensors included
        outs = []
        for rep in range(2):
            for b, k in CALLS:
                if rep:
                    outs.append(head.topk_sparse(hd[:b], k))
                else:
                    outs.append(head.topk(hd[:b], k))
        torch.cuda.synchronize()
        assert head.device_status() == vie.VIE_OK
    for n, out in enumerate(outs):
        ai, av = alone[n % len(CALLS)]
        np.testing.assert_array_equal(out[0].cpu().numpy(), ai)
        np.testing.assert_array_equal(out[1].cpu().numpy().view(np.uint32), av.view(np.uint32))
    if storage == "e4m3":
        q, sc = oracle.quantize_e4m3(W)
        z = oracle.logits_e4m3(q, sc, h)
    else:
        z = oracle.logits(W, h)
    for (b, k), (ai, av) in zip(CALLS, alone):
        for r in range(b):
            assert not check_topk(ai[r], av[r], z[r], k), (b, k, r)


@pytest.mark.parametrize("storage,batch,k", [("bf16", 1, 50), ("bf16", 1, 300), ("bf16", 4, 50), ("bf16", 5, 300),
                                             ("bf16", 300, 2), ("e4m3", 1, 50), ("e4m3", 12, 50)])
def test_queries_written_just_before_each_call(vie, storage, batch, k):
    """Launches overlap the kernels before them on the stream: each step's
    queries are written into the same buffer right before its call and the
    next step's right behind it, with nothing waiting in between."""
    import torch
    V, d, steps = 30011, 512, 12
    W, h = workload(V, d, steps * batch, seed=61)
    src = torch.from_numpy(h).cuda().view(steps, batch, d)
    with vie.Head(to_device_bits(W), storage=storage) as head:
        alone = [tuple(t.clone() for t in head.topk(src[s].contiguous(), k)) for s in range(steps)]
        torch.cuda.synchronize()
        buf = torch.empty((batch, d), device="cuda")
        outs = []
        for s in range(steps):
            buf.copy_(src[s])
            outs.append(head.topk(buf, k))
        torch.cuda.synchronize()
        assert head.device_status() == vie.VIE_OK
    for (ai, av), (i, v) in zip(alone, outs):
        np.testing.assert_array_equal(i.cpu().numpy(), ai.cpu().numpy())
        np.testing.assert_array_equal(v.cpu().numpy().view(np.uint32), av.cpu().numpy().view(np.uint32))
