"""GPU parity of the batched (tensor-core) path and of its merge in the last
CTA: path selection, the largest k of the path, two query groups, and inputs
whose winners crowd into a few per-CTA lists, which the warp merge cannot
settle from the lists' heads and hands to the full merge."""
import numpy as np
import pytest

import oracle
from acceptance import check_topk
from gpu_cases import assert_parity, run_head, to_device_bits, workload
from paper_2608_27460_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["bf16", "e4m3"])
@pytest.mark.parametrize("V,d", [(8000, 16384), (8192, 8192), (20011, 48)])
def test_handle_memory_is_what_its_props_say(vie, storage, V, d):
    """Weights and scratch of a handle, the query matrix with it: for 512 queries
    only where a call can take that many at once (bf16, V >= 8192, d >= 64)."""
    import torch
    W = torch.zeros((V, d), dtype=torch.int16, device="cuda")
    vie.Head(W, storage=storage).close()  # the kernels' own memory is there now
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    with vie.Head(W, storage=storage) as head:
        used = before - torch.cuda.mem_get_info()[0]
        p = head.props
        rows = 1024 if storage == "bf16" and V >= 8192 and d >= 64 else 128
        assert p.scratch_bytes >= rows * p.d_pad * 2
        assert p.scratch_bytes <= rows * p.d_pad * 2 + p.ctas * (8 * 1056 + 256) * 8 + (64 << 10)
        assert used <= p.weight_bytes + p.scratch_bytes + (10 << 20)  # whole 2 MB pages


def test_plan_selects_paths(vie):
    W, _ = workload(20011, 640, 1, seed=3)
    with vie.Head(to_device_bits(W)) as head:
        p = head.plan(1, 50)
        assert (p.path, p.groups, p.launches) == (0, 1, 1)
        p = head.plan(2, 50)  # query prep, then the projection
        assert (p.path, p.groups, p.launches) == (1, 1, 2)
        p = head.plan(40, 50)  # one 64-query group: one pass over W
        assert (p.path, p.groups, p.launches) == (1, 1, 2)
        p = head.plan(40, 65)  # k above the 64-query tile's lists: 32 + 8
        assert (p.path, p.groups, p.launches) == (1, 2, 4)
        p = head.plan(100, 50)  # 64 + 36
        assert (p.path, p.groups, p.launches) == (1, 2, 4)
        p = head.plan(4, 129)  # above the tensor-core path's k
        assert p.path == 0


@pytest.mark.parametrize("V,d,batch,k", [
    (20011, 512, 3, 128),    # largest k of the tensor-core path
    (20011, 512, 3, 129),    # smallest k above it (streaming path)
    (30011, 256, 40, 50),    # 64-query tile, four queries per selector warp
    (30011, 256, 64, 64),    # full 64-query tile at its largest k
    (30011, 256, 40, 65),    # two 32-query groups, two queries per selector warp
    (20011, 1152, 100, 50),  # 64 + 36 queries
    (30011, 256, 32, 1),     # greedy, full group of 32
    (30011, 1000, 64, 1),    # no shared bound: greedy on 64 slots, rows of odd sectors
    (30011, 1000, 20, 3),
    (50021, 1024, 17, 77),
    (100, 64, 4, 50),        # one tile: most CTAs draw nothing and write empty lists
    (64, 128, 2, 64),        # k = V on one CTA
    (200, 256, 40, 64),      # 64-query tile over two tiles
    (129, 128, 8, 128),      # largest k, a one-row last tile
    (2000, 256, 4, 128),     # every row is a candidate: logits of both signs crowd the ranking's bins
    (600, 128, 4, 100),      # the same, few enough to rank by all pairs
])
def test_tensor_core_parity(vie, V, d, batch, k):
    W, h = workload(V, d, batch, seed=V + batch + k)
    assert_parity(vie, W, h, k, reps=2)


# fewer CTAs than 2 k (64 rows each): every CTA publishes four maxima per query
@pytest.mark.parametrize("storage", ["bf16", "e4m3"])
@pytest.mark.parametrize("V,k", [(1000, 20), (1000, 50), (1100, 64), (2500, 20), (2500, 50), (2500, 64),
                                 (5000, 50), (6000, 50), (8127, 64)])
@pytest.mark.parametrize("d", [64, 1024, 3072])
def test_bound_words_of_small_vocabularies(vie, storage, V, d, k):
    """The words of the CTAs' shared bound and the query matrix lie next to
    each other: groups of 8 to 64 queries, repeated without waiting, give the
    oracle's top-k and every launch the same bits."""
    import torch
    W, h = workload(V, d, 100, seed=V + d + k)
    z = oracle.logits(W, h) if storage == "bf16" else oracle.logits_e4m3(*oracle.quantize_e4m3(W), h)
    hd = torch.from_numpy(h).cuda()
    with vie.Head(to_device_bits(W), storage=storage) as head:
        for b in (8, 32, 33, 64, 100):
            outs = [head.topk(hd[:b], k) for _ in range(4)]
            torch.cuda.synchronize()
            assert head.device_status() == vie.VIE_OK
            idx, val = (t.cpu().numpy() for t in outs[0])
            for i, v in outs[1:]:
                np.testing.assert_array_equal(i.cpu().numpy(), idx)
                np.testing.assert_array_equal(v.cpu().numpy().view(np.uint32), val.view(np.uint32))
            for q in range(b):
                assert not check_topk(idx[q], val[q], z[q], k), (b, q)


def _crowded(V, d, batch, rows, seed):
    """Rows `rows` scaled by 64 (exact in bf16): the winners of every query
    sit in one or two 128-row tiles, so in one or two per-CTA lists."""
    W, h = workload(V, d, batch, seed=seed)
    f = synth.bf16_bits_to_f32(W)
    f[rows] *= 64.0
    return synth.f32_to_bf16_bits(f), h


@pytest.mark.parametrize("batch,k", [(1, 50), (4, 50), (4, 128), (20, 50), (40, 50)])
@pytest.mark.parametrize("where", ["head", "tail"])
def test_crowded_winners_take_the_full_merge(vie, batch, k, where):
    V, d = 40009, 256
    rows = np.arange(0, 200) if where == "head" else np.arange(V - 200, V)
    W, h = _crowded(V, d, batch, rows, seed=11 + batch + k)
    idx, _, _ = assert_parity(vie, W, h, k)
    assert np.isin(idx[:, :20], rows).all()  # the scaled rows do win


def test_all_rows_equal_full_groups(vie):
    """Every logit equal, in 32- and 64-query tiles: every query leaves the
    fast merge for the full merge, which ranks by index."""
    V, d = 30011, 64
    row = synth.f32_to_bf16_bits(np.full(d, 0.25, np.float32))
    W = np.tile(row, (V, 1))
    for b, k in ((20, 1), (20, 128), (48, 64)):
        h = np.ones((b, d), np.float32)
        idx, val = run_head(vie, W, h, k)
        np.testing.assert_array_equal(idx, np.tile(np.arange(k, dtype=np.int32), (b, 1)))
        assert np.all(val == np.float32(0.25 * d))


@pytest.mark.parametrize("V,d,batch,k", [
    (8192, 64, 256, 1),        # the smallest batch and vocabulary of the filtered GEMM, one K-block
    (20011, 200, 257, 8),      # a group of one query, a ragged last K-block, every 64th row
    (20011, 512, 300, 9),      # every 32nd row
    (30000, 256, 513, 64),     # two blocks, the second of one query
    (20011, 128, 260, 65),     # every 8th row
    (8193, 320, 256, 128),     # the largest k, a one-row last tile
])
def test_many_queries(vie, V, d, batch, k):
    """Batches of 256 queries or more: a sample of the rows bounds each query's
    k-th logit, the logits above it are gathered and ranked."""
    W, h = workload(V, d, batch, seed=V + batch + k)
    assert_parity(vie, W, h, k, reps=2)


@pytest.mark.parametrize("k", [1, 50])
def test_many_queries_whose_candidates_overflow(vie, k):
    """Rows the sample takes (every 64th, hence every 16th) are zero, so every
    positive logit is a candidate: ~10000 of them, more than are kept, and the
    query is recomputed; and a zero query, whose logits all tie."""
    V, d, batch = 20011, 128, 256
    W, h = workload(V, d, batch, seed=5)
    W[::16] = 0
    h[3] = 0.0
    idx, _, _ = assert_parity(vie, W, h, k)
    np.testing.assert_array_equal(idx[3], np.arange(k))


def _rare_low_rows(V, d, n, low, seed):
    """Every 8th row (all that a sample of any stride takes) has -1 in column 0
    and the others +1; the queries in `low` are mostly that column, so seven
    eighths of the rows reach their sampled bound."""
    W, h = workload(V, d, n, seed=seed)
    f = synth.bf16_bits_to_f32(W)
    f[:, 0] = 1.0
    f[::8, 0] = -1.0
    h[:, 0] = 0.0
    h[low] *= 0.01
    h[low, 0] = 5.0
    return synth.f32_to_bf16_bits(f), h


@pytest.mark.parametrize("V,d,batch,low,k", [
    (8192, 64, 256, [7], 1),               # 256 slices of 32 rows
    (20011, 100, 257, [0, 255, 256], 50),  # 40 slices; rows that are no multiple of 16 bytes of h
    (30000, 72, 513, [512], 8),            # alone in the second block of launches
    (20011, 264, 300, list(range(0, 300, 2)), 128),  # 16 slices of more rows than one round
])
def test_many_queries_some_recomputed(vie, V, d, batch, low, k):
    """Queries whose candidates overflow are recomputed by all CTAs of the
    final launch, among queries that are not; the sparse rows of both."""
    import torch
    W, h = _rare_low_rows(V, d, batch, low, seed=V + k)
    z = oracle.logits(W, h)
    with vie.Head(to_device_bits(W)) as head:
        hd = torch.from_numpy(h).cuda()
        for _ in range(2):  # the counters are re-armed
            i, v, sp = head.topk_sparse(hd, k)
            want = head.sparse_logits(i, v)
            torch.cuda.synchronize()
            assert head.device_status() == vie.VIE_OK
            np.testing.assert_array_equal(sp.cpu().numpy().view(np.uint32), want.cpu().numpy().view(np.uint32))
            idx, val = i.cpu().numpy(), v.cpu().numpy()
            for q in range(batch):
                assert not check_topk(idx[q], val[q], z[q], k), q


def test_a_recomputed_query_is_no_cliff(vie):
    """One query of 512 whose candidates overflow: its rows are shared by the
    CTAs of the launch (its own CTA alone took over 100 times the call)."""
    import torch
    V, d, batch, k = 100003, 512, 512, 2
    W, h = _rare_low_rows(V, d, batch, [7], seed=9)
    plain = h.copy()
    plain[7] = plain[8]
    with vie.Head(to_device_bits(W)) as head:
        t = []
        for x in (plain, h):
            xd = torch.from_numpy(x).cuda()
            out = head.topk(xd, k)
            ms = []
            for _ in range(5):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                head.topk(xd, k, out_idx=out[0], out_logits=out[1])
                b.record()
                b.synchronize()
                ms.append(a.elapsed_time(b))
            t.append(min(ms))
    assert t[1] < 10 * t[0], t


def test_many_queries_sparse_and_captured(vie):
    """The sparse rows of a filtered-GEMM call equal the scatter of its own
    top-k, and replaying the captured call gives the eager bits."""
    import torch
    V, d, batch, k = 8300, 128, 260, 50
    W, h = workload(V, d, batch, seed=77)
    hd = torch.from_numpy(h).cuda()
    with vie.Head(to_device_bits(W)) as head:
        assert head.plan(batch, k).launches == 5
        ei, ev, es = head.topk_sparse(hd, k)
        want = head.sparse_logits(ei, ev)
        oi, ov, osp = torch.empty_like(ei), torch.empty_like(ev), torch.empty_like(es)
        cap = torch.cuda.Stream()
        cap.wait_stream(torch.cuda.current_stream())
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(cap), torch.cuda.graph(g, stream=cap):
            head.topk_sparse(hd, k, out_idx=oi, out_logits=ov, out_sparse=osp, stream=cap)
        torch.cuda.current_stream().wait_stream(cap)
        for _ in range(2):
            osp.zero_()
            g.replay()
        torch.cuda.synchronize()
        assert head.device_status() == vie.VIE_OK
    for a, b in ((es, want), (oi, ei), (ov, ev), (osp, es)):
        np.testing.assert_array_equal(a.cpu().numpy().view(np.uint32), b.cpu().numpy().view(np.uint32))
