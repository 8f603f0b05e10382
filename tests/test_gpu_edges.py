"""GPU checks of the edges of the product path: parts of short prefixes, rows that only pad a block, NaN
and infinite keys, crowded boundary bins, the status word of a packed batch."""
import os
import re

import numpy as np
import pytest
import torch

from paper_2607_24593_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pv():
    from paper_2607_24593_b200 import binding
    return binding


def _sorted(out):
    return torch.sort(out.reshape(-1, out.shape[-1]), dim=1).values.cpu().numpy()


def _operands(x):
    kw = {} if x.qscale is None else dict(q_scale=x.qscale.cuda(), k_scale=x.kscale.cuda())
    return x.q.cuda(), x.w.cuda(), x.k.cuda(), kw


@pytest.mark.parametrize("dtype,g,mode,W,L,row0,c,k", [
    ("fp8", 4, 1, 0, 880, 832, 24, 24),
    ("bf16", 4, 1, 0, 880, 832, 24, 24),
    ("fp8", 4, 0, 0, 900, 644, 256, 16),
    ("fp8", 4, 0, 1004, 1500, 1024, 1024, 64),
    ("bf16", 4, 1, 0, 1003, 960, 16, 16),
    ("fp8", 2, 0, 0, 1100, 1000, 16, 8),
    ("fp8", 1, 0, 0, 300, 290, 2, 1),
    ("bf16", 16, 1, 8, 1201, 1104, 40, 9),
])
def test_chunk_of_a_short_prefix_and_a_small_budget(pv, dtype, g, mode, W, L, row0, c, k):
    """Small budgets allow many parts of a prefix of few key tiles: every part has to have a tile (one that has
    none is never scanned, and its list would be whatever the workspace held).  The workspace starts full of
    words that read as positions with large scores."""
    x = inputs.make_prefill(L, dtype=dtype, seed=L + k)
    q, w, kk, kw = _operands(x)
    ws = torch.full((pv.pivot_workspace_bytes(L, (L + g - 1) // g, c, k),), 0x44, dtype=torch.uint8, device="cuda")
    whole = torch.full((L, k), -7, dtype=torch.int32, device="cuda")
    part = torch.full((L, k), -7, dtype=torch.int32, device="cuda")
    pv.pivot_index_prefill(q, w, kk, L, 64, 128, g, c, k, mode, whole, W=W, **kw)
    pv.pivot_index_prefill(q, w, kk, L, 64, 128, g, c, k, mode, part, W=W, rows=(row0, L), workspace=ws, **kw)
    torch.cuda.synchronize()
    assert pv.pivot_device_status() == 0
    assert np.array_equal(_sorted(whole[row0:]), _sorted(part[row0:]))
    assert (part[:row0] == -7).all()


def _nan_rows(q, rows):
    """e4m3 queries with NaN codes in the given rows."""
    q = q.clone()
    q.view(torch.uint8)[rows] = 0x7f
    return q


def test_chunk_does_not_read_queries_outside_its_rows(pv):
    """A chunk's rows are all it indexes: the other rows of the query tensor may hold anything (they arrive
    later, or were overwritten).  33 groups: the last block of scan rows is padded where the prefix is scanned in parts."""
    L, g, c, k, row0 = 8192, 4, 256, 128, 8192 - 132
    x = inputs.make_prefill(L, dtype="fp8", seed=3)
    q, w, kk, kw = _operands(x)
    a = torch.full((L, k), -7, dtype=torch.int32, device="cuda")
    b = torch.full((L, k), -7, dtype=torch.int32, device="cuda")
    pv.pivot_index_prefill(q, w, kk, L, 64, 128, g, c, k, pv.REFINE, a, rows=(row0, L), **kw)
    pv.pivot_index_prefill(_nan_rows(q, slice(0, row0)), w, kk, L, 64, 128, g, c, k, pv.REFINE, b, rows=(row0, L), **kw)
    torch.cuda.synchronize()
    assert np.array_equal(_sorted(a), _sorted(b))


def test_packed_request_is_not_touched_by_its_first_row_in_its_last_block(pv):
    """Packed requests are padded to whole blocks of scan rows: what a padding row holds must not reach the live
    rows of its block, so NaN queries in the first group change that group's selections only, as in separate calls."""
    lens, g, c, k = [1004, 2003], 4, 256, 128
    cu = [0, 1004, 3007]
    x = inputs.make_prefill(cu[-1], dtype="fp8", seed=4)
    q, w, kk, kw = _operands(x)
    q = _nan_rows(q, slice(1004, 1008))
    packed = torch.full((cu[-1], k), -7, dtype=torch.int32, device="cuda")
    one = torch.full((cu[-1], k), -7, dtype=torch.int32, device="cuda")
    pv.pivot_index_prefill_varlen(q, w, kk, cu, 64, 128, g, c, k, pv.REFINE, packed, **kw)
    for a, b in zip(cu[:-1], cu[1:]):
        pv.pivot_index_prefill(q[a:b], w[a:b], kk[a:b], b - a, 64, 128, g, c, k, pv.REFINE, one[a:b],
                               q_scale=kw["q_scale"][a:b], k_scale=kw["k_scale"][a:b])
    torch.cuda.synchronize()
    assert lens == [b - a for a, b in zip(cu[:-1], cu[1:])]
    assert np.array_equal(_sorted(packed), _sorted(one))


NAN_AT, ZERO_AT = [5, 70, 130, 201], 250


def _all_but_nan(n):
    return np.array([p for p in range(n) if p not in NAN_AT])


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("B,n", [(2, 257), (3, 5000), (80, 700)])
def test_nan_key_scales_rank_behind_every_number_in_decode(pv, mode, B, n):
    """A NaN score counts in the scan's histogram as what the select takes it for: -0."""
    g = 2
    c = k = n - len(NAN_AT)
    x = inputs.make_decode(B, g, n, n, dtype="fp8", seed=9)
    x.kscale[:, NAN_AT] = float("nan")
    q, w, kk, kw = _operands(x)
    out = torch.full((B, g, k), -7, dtype=torch.int32, device="cuda")
    pv.pivot_index_decode(q, w, kk, x.pos0.cuda(), B, kk.shape[1], 64, 128, g, c, k, mode, out, **kw)
    torch.cuda.synchronize()
    assert pv.pivot_device_status() == 0
    assert (_sorted(out) == _all_but_nan(n)).all()


def _keys_without_a_score(x, nan_at, zero_at):
    """NaN entries in the keys at nan_at (any leading dimensions, positions second to last), a key of zeros at zero_at."""
    k = x.k.clone()
    if k.dtype == torch.bfloat16:
        k[..., nan_at, 17] = float("nan")
        k[..., zero_at, :] = 0.0
    else:
        k.view(torch.uint8)[..., nan_at, 17] = 0x7f
        k.view(torch.uint8)[..., zero_at, :] = 0
    x.k = k
    return x


@pytest.mark.parametrize("dtype,impl", [("bf16", 0), ("fp8", 0), ("fp8", 2)])
@pytest.mark.parametrize("mode", [0, 1])
def test_nan_keys_rank_behind_every_number_in_prefill(pv, dtype, impl, mode):
    """A NaN in a key makes its products, and so its score, NaN in every form of the head sum.  A NaN ranks as -0:
    behind a later key whose score is exactly 0, which behind keys of equal score it would not."""
    L, g, c = 401, 4, 257                        # the group at 256 sees exactly c keys, all of them candidates
    k = c - len(NAN_AT)
    x = _keys_without_a_score(inputs.make_prefill(L, dtype=dtype, seed=6), NAN_AT, ZERO_AT)
    q, w, kk, kw = _operands(x)
    out = torch.full((L, k), -7, dtype=torch.int32, device="cuda")
    pv.pivot_index_prefill(q, w, kk, L, 64, 128, g, c, k, mode, out, impl=impl, **kw)
    dense = torch.full((L, k), -7, dtype=torch.int32, device="cuda")
    pv.dense_index(q, w, kk, L, 64, 128, k, dense, impl=impl, **kw)
    torch.cuda.synchronize()
    assert pv.pivot_device_status() == 0
    assert (_sorted(out[256:260]) == _all_but_nan(c)).all()
    assert (_sorted(dense[256:257]) == _all_but_nan(c)).all()


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
@pytest.mark.parametrize("mode", [0, 1])
def test_nan_keys_rank_behind_every_number_in_decode(pv, dtype, mode):
    B, g, c = 3, 2, 257
    k = c - len(NAN_AT)
    x = _keys_without_a_score(inputs.make_decode(B, g, c, c, dtype=dtype, seed=7), NAN_AT, ZERO_AT)
    q, w, kk, kw = _operands(x)
    out = torch.full((B, g, k), -7, dtype=torch.int32, device="cuda")
    pv.pivot_index_decode(q, w, kk, x.pos0.cuda(), B, kk.shape[1], 64, 128, g, c, k, mode, out, **kw)
    torch.cuda.synchronize()
    assert pv.pivot_device_status() == 0
    assert (_sorted(out) == _all_but_nan(c)).all()


def test_status_of_an_earlier_set_of_requests_survives(pv):
    """A packed batch beyond one set of launches (more than 64 requests) is prepared in several: a condition that
    the first set recorded is still there at the end of the call, and the next call starts clean.  The condition
    is planted into a captured call between its two sets."""
    cudart = pytest.importorskip("cuda.bindings.runtime")
    lens, g, c, k = [64] * 70, 4, 32, 16
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(int)
    x = inputs.make_prefill(int(cu[-1]), dtype="bf16", seed=12)
    q, w, kk, kw = _operands(x)
    out = torch.full((int(cu[-1]), k), -7, dtype=torch.int32, device="cuda")
    ws = torch.empty(pv.pivot_workspace_bytes(int(cu[-1]) + 4 * 70, int(cu[-1]) // g, c, k), dtype=torch.uint8, device="cuda")
    call = lambda: pv.pivot_index_prefill_varlen(q, w, kk, cu, 64, 128, g, c, k, pv.REFINE, out, workspace=ws, **kw)
    pv.lib.pivot_launch_count_reset()
    call()                                       # (function attributes are set before the capture)
    per_set = pv.lib.pivot_launch_count_reset() // 2
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    raw = cudart.cudaGraph_t(graph.raw_cuda_graph())

    def ok(r):
        assert r[0] == cudart.cudaError_t.cudaSuccess, r[0]
        return r[1:] if len(r) > 2 else (r[1] if len(r) == 2 else None)

    n = ok(cudart.cudaGraphGetNodes(raw, 0))[1]
    nodes = ok(cudart.cudaGraphGetNodes(raw, n))[0]
    assert n == 2 * per_set == len(nodes)
    edges = ok(cudart.cudaGraphGetEdges_v2(raw, 0))[-1]
    src, dst = ok(cudart.cudaGraphGetEdges_v2(raw, edges))[:2]
    after = {int(a): int(b) for a, b in zip(src, dst)}
    order = [next(int(v) for v in nodes if int(v) not in after.values())]
    while order[-1] in after:
        order.append(after[order[-1]])
    assert len(order) == n                       # a chain
    by_id = {int(v): v for v in nodes}
    end_first, begin_second = by_id[order[per_set - 1]], by_id[order[per_set]]
    p = cudart.cudaMemsetParams()
    p.dst, p.value, p.elementSize, p.width, p.height, p.pitch = ws.data_ptr(), pv.DEV_CAND_OVERFLOW, 4, 1, 1, 4
    node = ok(cudart.cudaGraphAddMemsetNode(raw, [end_first], 1, p))
    ok(cudart.cudaGraphAddDependencies(raw, [node], [begin_second], 1))
    graph.instantiate()
    graph.replay()
    torch.cuda.synchronize()
    assert pv.pivot_device_status() == pv.DEV_CAND_OVERFLOW
    call()
    assert pv.pivot_device_status() == 0


def test_packed_batch_where_only_the_longest_request_fits(pv, monkeypatch):
    """The binding's own workspace shares a batch's launches where there is memory for that; where there is not,
    the call runs with room for its longest request, as it always could."""
    lens, g, c, k = [400, 1600, 900, 1200], 4, 256, 128
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(int)
    x = inputs.make_prefill(int(cu[-1]), dtype="fp8", seed=13)
    q, w, kk, kw = _operands(x)
    run = lambda: pv.pivot_index_prefill_varlen(q, w, kk, cu, 64, 128, g, c, k, pv.REFINE,
                                                torch.full((int(cu[-1]), k), -7, dtype=torch.int32, device="cuda"), **kw)
    want = _sorted(run())
    longest = pv.pivot_workspace_bytes(max(lens), (max(lens) + g - 1) // g, c, k)
    empty = torch.empty

    refused = []

    def small_gpu(*a, **kw_):
        if kw_.get("dtype") == torch.uint8 and a and isinstance(a[0], int) and a[0] > longest:
            refused.append(a[0])
            raise torch.cuda.OutOfMemoryError("no room")
        return empty(*a, **kw_)

    keep = pv._workspaces.get(torch.cuda.current_device())
    pv.pivot_set_workspace(None)
    monkeypatch.setattr(torch, "empty", small_gpu)
    try:
        got = [_sorted(run()) for _ in range(4)]
        assert pv._workspaces[torch.cuda.current_device()].numel() <= longest
        assert len(refused) <= 2                 # not on every call
    finally:
        monkeypatch.undo()
        pv.pivot_set_workspace(keep)
    assert all(np.array_equal(v, want) for v in got)
    assert np.array_equal(_sorted(run()), want)


def test_workspace_that_a_batch_outgrows_stays_valid(pv):
    """A graph captured with the registered workspace goes on using it after a packed batch made the binding
    register a larger one: the memory is not handed to anyone else, and the graph's results stay right."""
    dev = torch.cuda.current_device()
    pv.pivot_set_workspace(None)
    g, c, k, n = 2, 128, 64, 600
    xd = inputs.make_decode(2, g, n, n, dtype="fp8", seed=14)
    q, w, kk, kw = _operands(xd)
    pos0, out = xd.pos0.cuda(), torch.full((2, g, k), -7, dtype=torch.int32, device="cuda")
    xp = inputs.make_prefill(6000, dtype="fp8", seed=15)
    pq, pw, pk, pkw = _operands(xp)
    pv.ensure_workspace(2000, 500, 512, 256)                       # room for any one request
    first = pv._workspaces[dev]
    step = lambda: pv.pivot_index_decode(q, w, kk, pos0, 2, kk.shape[1], 64, 128, g, c, k, pv.REFINE, out, **kw)
    step()
    want = _sorted(out)
    assert pv._workspaces[dev] is first
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    at, size = first.data_ptr(), first.numel()
    del first
    pv.pivot_index_prefill_varlen(pq, pw, pk, [0, 2000, 4000, 6000], 64, 128, 4, 512, 256, pv.REFINE,
                                  torch.full((6000, 256), -7, dtype=torch.int32, device="cuda"), **pkw)
    assert pv._workspaces[dev].numel() > size
    others = [torch.zeros(size, dtype=torch.uint8, device="cuda") for _ in range(3)]
    assert all(o.data_ptr() + size <= at or o.data_ptr() >= at + size for o in others)
    out.fill_(-7)
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(_sorted(out), want)
    assert not any(o.any() for o in others)
    pv.pivot_set_workspace(None)
    assert not pv._outgrown


def test_current_stream_with_and_without_the_raw_handle(pv, monkeypatch):
    """The stream of a call without a `stream` argument, also on a torch release that lacks the raw accessor."""
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert pv._stream(None) == side.cuda_stream
        monkeypatch.setattr(pv, "_raw_stream", None)
        assert pv._stream(None) == side.cuda_stream
    assert pv._stream(None) == torch.cuda.current_stream().cuda_stream


@pytest.mark.parametrize("dtype,mode,c,k,row0", [("fp8", 0, 1280, 1280, 11264), ("bf16", 1, 1280, 700, 11904), ("fp8", 1, 2000, 1000, 12000)])
def test_chunk_whose_parts_fill_their_segments(pv, dtype, mode, c, k, row0):
    """Budgets whose candidate segments are thinned out on the way (more than 1024, a few refresh intervals of
    keys): however the prefix is cut, the rows of a chunk are the whole call's."""
    L, g = 12288, 4
    x = inputs.make_prefill(L, dtype=dtype, seed=16)
    q, w, kk, kw = _operands(x)
    whole = torch.full((L, k), -7, dtype=torch.int32, device="cuda")
    part = torch.full((L, k), -7, dtype=torch.int32, device="cuda")
    pv.pivot_index_prefill(q, w, kk, L, 64, 128, g, c, k, mode, whole, **kw)
    pv.pivot_index_prefill(q, w, kk, L, 64, 128, g, c, k, mode, part, rows=(row0, L), **kw)
    torch.cuda.synchronize()
    assert pv.pivot_device_status() == 0
    assert np.array_equal(_sorted(whole[row0:]), _sorted(part[row0:]))


@pytest.mark.parametrize("B", [2, 40, 80])
@pytest.mark.parametrize("n_tied", [4096, 4097, 9000, 11988, 11989, 12400])
def test_decode_crowded_boundary_bin(pv, B, n_tied):
    """The boundary bin holds n_tied equal scores (one key repeated) and c cuts it: on either side of the lists
    that the select ranks in shared memory (4096 boundary entries; 12288 survivors, 300 of them above the bin), for every cluster size
    (batches of up to 37, up to 74 and more).  The lowest positions of the tie win."""
    g, c, k, n = 1, 1024, 512, 14000
    x = inputs.make_decode(1, g, n, n, dtype="fp8", seed=21)
    kk = x.k.clone()
    raw = kk.view(torch.uint8)
    scale = x.kscale.clone()
    gen = torch.Generator().manual_seed(n_tied)
    tied = torch.randperm(n, generator=gen)[:n_tied].sort().values
    free = torch.ones(n, dtype=torch.bool)
    free[tied] = False
    above = torch.nonzero(free).view(-1)[:300]
    raw[0, tied] = raw[0, 7].clone()
    scale[0, :] = scale[0, :] * 1e-3
    scale[0, tied] = 1.0
    raw[0, above] = raw[0, 7].clone()
    scale[0, above] = 4.0
    rep = lambda t: t.cuda().view(torch.uint8).expand(B, *t.shape[1:]).contiguous().view(t.dtype) if t.element_size() == 1 \
        else t.cuda().expand(B, *t.shape[1:]).contiguous()
    pos0 = torch.full((B,), n - 1, dtype=torch.int32, device="cuda")
    out = torch.full((B, g, k), -7, dtype=torch.int32, device="cuda")
    cand = torch.full((B, c), -7, dtype=torch.int32, device="cuda")
    pv.pivot_index_decode(rep(x.q), rep(x.w), rep(kk), pos0, B, kk.shape[1], 64, 128, g, c, k, pv.REFINE, out, dbg_cand=cand,
                          q_scale=rep(x.qscale), k_scale=rep(scale))
    torch.cuda.synchronize()
    assert pv.pivot_device_status() == 0
    want = np.sort(np.concatenate([above.numpy(), tied.numpy()[: c - len(above)]]))
    assert (_sorted(cand) == want).all()
    want = np.sort(np.concatenate([above.numpy(), tied.numpy()[: k - len(above)]]))
    assert (_sorted(out) == want).all()


@pytest.mark.parametrize("impl", [0, 2])
@pytest.mark.parametrize("L,K,slope", [
    (513, 1, 2.0 ** -10), (1409, 1024, 2.0 ** -10), (1537, 100, 2.0 ** -10), (2100, 777, -2.0 ** -16),
    (12000, 512, 2.0 ** -12), (12000, 1024, 2.0 ** -8), (16500, 1300, 2.0 ** -13), (9999, 64, -2.0 ** -18),
    (20000, 700, -2.0 ** -16), (20001, 900, 2.0 ** -10), (24000, 64, 2.0 ** -13),
])
def test_scores_that_rise_or_fall_along_the_prefix(pv, L, K, slope, impl):
    """One key under scales that rise (every key beats all before it: no threshold drops anything, segments of 8192
    entries fill up and are thinned, by the threshold or, where the scores outgrow the histogram, to the K best) or fall
    with its position (nothing is appended after the first K).  Row t selects its last or its first K keys; on
    either side of the first thresholds (5/4 K keys, four tiles), of a block's last refresh, and of the mean prefix up to
    which each row has a finisher warp of its own (6144 keys: dense requests of 12288)."""
    x = inputs.make_prefill(L, dtype="fp8", seed=3)
    raw = x.k.clone().view(torch.uint8)
    raw[:] = raw[5].clone()
    scale = 1.0 + slope * torch.arange(L, dtype=torch.float32)
    q, w, _, kw = _operands(x)
    kw["k_scale"] = scale.cuda()
    out = torch.full((L, K), -7, dtype=torch.int32, device="cuda")
    pv.dense_index(q, w, raw.view(x.k.dtype).cuda(), L, 64, 128, K, out, impl=impl, **kw)
    torch.cuda.synchronize()
    assert pv.pivot_device_status() == 0
    t = torch.arange(L, device="cuda", dtype=torch.int32).view(-1, 1)
    j = torch.arange(K, device="cuda", dtype=torch.int32).view(1, -1)
    want = torch.where(t - K + 1 + j >= 0, t - K + 1 + j, -1) if slope > 0 else torch.where(j <= t, j, -1).sort(dim=1).values
    assert torch.equal(out.sort(dim=1).values, want)


@pytest.mark.parametrize("scored", [False, True])
@pytest.mark.parametrize("mode", ["dense", 0, 1])
def test_rows_select_the_same_whatever_the_finishers(pv, mode, scored):
    """Requests on either side of the mean prefix up to which each row has a finisher warp of its own: the rows that both
    have select the same keys, with the same scores."""
    sizes, g, c, k = (9001, 24000), 4, 1024, 500
    header = open(os.path.join(os.path.dirname(pv.__file__), "csrc", "kernels.h")).read()
    bound = int(re.search(r"kShortBlockKeys = (\d+);", header).group(1))
    L = sizes[-1]
    x = inputs.make_prefill(L, dtype="fp8", seed=27)
    q, w, kk, kw = _operands(x)
    outs = []
    for n in sizes:
        rows = list(range(n)) if mode == "dense" else list(range(c)) + list(range(c, n, g))
        mean = sum(t + 1 for t in rows) / len(rows)
        assert mean < bound * 3 / 4 if n == sizes[0] else mean > bound * 4 / 3
        out = torch.full((n, k), -7, dtype=torch.int32, device="cuda")
        sc = torch.full((n, k), float("nan"), device="cuda") if scored else None
        part = dict(q_scale=kw["q_scale"][:n], k_scale=kw["k_scale"][:n], dbg_scores=sc)
        if mode == "dense":
            pv.dense_index(q[:n], w[:n], kk[:n], n, 64, 128, k, out, **part)
        else:
            pv.pivot_index_prefill(q[:n], w[:n], kk[:n], n, 64, 128, g, c, k, mode, out, **part)
        torch.cuda.synchronize()
        assert pv.pivot_device_status() == 0
        # (the last group of the shorter request has one member: its proxy is another)
        ids, at = out[:sizes[0] - 1].sort(dim=1)
        outs.append((ids, sc[:sizes[0] - 1].gather(1, at) if scored else None))
    assert torch.equal(outs[0][0], outs[1][0])
    assert not scored or torch.equal(outs[0][1], outs[1][1])


@pytest.mark.parametrize("dtype,impl", [("bf16", 0), ("fp8", 2)])
@pytest.mark.parametrize("g,L", [(4, 4001), (6, 4003), (2, 3001), (9, 4000)])
def test_members_missing_from_a_group_lend_nothing(pv, dtype, impl, g, L):
    """fp32 head sums take no queries for members that a group (or its last chunk) does not have: what the groups before
    it left in their place -- here NaN -- reaches no other member's selection."""
    c, k = 512, 256
    x = inputs.make_prefill(L, dtype=dtype, seed=31)
    q, w, kk, kw = _operands(x)
    first = torch.arange(L, device="cuda") % g == 0
    bad = q.clone()
    if dtype == "bf16":
        bad[~first] = float("nan")
    else:
        bad.view(torch.uint8)[~first] = 0x7f
    outs = []
    for queries in (q, bad):
        out = torch.full((L, k), -7, dtype=torch.int32, device="cuda")
        pv.pivot_index_prefill(queries, w, kk, L, 64, 128, g, c, k, pv.REFINE, out, impl=impl, pool=pv.POOL_FIRST, **kw)
        torch.cuda.synchronize()
        assert pv.pivot_device_status() == 0
        outs.append(_sorted(out[first]))
    assert np.array_equal(*outs)


@pytest.mark.parametrize("dtype,impl", [("fp8", 0), ("fp8", 2), ("bf16", 0)])
@pytest.mark.parametrize("K,form", [(1, ""), (255, ""), (257, ""), (700, "rising"), (300, "tied"), (1300, "")])
def test_rows_that_return_scores_select_the_same(pv, dtype, impl, K, form):
    """Rows with their scores against the same rows without, and every score against the one that the row's key has when all
    keys are wanted.  Rows hold 1 .. 2300 entries: on either side of the sweep's chunks of 256; rising scores append
    every key, tied ones leave a boundary too crowded to rank."""
    L = 2300
    x = inputs.make_prefill(L, dtype=dtype, seed=41)
    q, w, kk, kw = _operands(x)
    if form == "rising":
        b = kk.view(torch.uint8) if dtype == "fp8" else kk
        b[:] = b[5].clone()
        if dtype == "fp8":
            kw["k_scale"] = (1.0 + 2.0 ** -10 * torch.arange(L, dtype=torch.float32)).cuda()
        else:                                   # (bf16 keys have no scale: 16 magnitudes, rising)
            kk = (kk.float() * 2.0 ** (torch.arange(L, device="cuda") * 16 // L - 8).view(-1, 1)).to(kk.dtype)
    if form == "tied":
        w = torch.zeros_like(w)

    def index(k, scored):
        out = torch.full((L, k), -7, dtype=torch.int32, device="cuda")
        sc = torch.full((L, k), float("nan"), device="cuda") if scored else None
        pv.dense_index(q, w, kk, L, 64, 128, k, out, dbg_scores=sc, impl=impl, **kw)
        torch.cuda.synchronize()
        assert pv.pivot_device_status() == 0
        return out, sc

    every, score = index(L, True)
    table = torch.full((L, L + 1), float("-inf"), device="cuda")         # column 0: the -1 of short rows
    table.scatter_(1, every.long() + 1, score)
    table[:, 0] = float("-inf")
    plain, _ = index(K, False)
    out, sc = index(K, True)
    assert np.array_equal(_sorted(plain), _sorted(out))
    assert torch.equal(sc, table.gather(1, out.long() + 1))
