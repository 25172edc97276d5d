"""Single kernels at the edges of their tiles, against the oracle on the same seeded inputs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

import paper_2509_05165_b200 as kvc
from paper_2509_05165_b200 import binding, workloads as W
from paper_2509_05165_b200.binding import alloc_outputs

import parity as Pz


def _setup(cfg, **desc_kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    return dev, W.make_workload(cfg, dev), kvc.desc_from_config(cfg, **desc_kw)


@pytest.mark.parametrize("N", [1, 63, 129, 1030])
@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("bf16", 128), ("f32", 64), ("f32", 128)])
def test_value_norms_at_tile_edges(dtype, d, N):
    """One row, a CTA's rows less and more than full, and several CTAs, for every row width."""
    import oracle
    cfg = W.WorkloadConfig("norm_edges", 2, 4, 2, d, N, 1, batch=2, dtype=dtype, elem_std=1.0, n_sinks=min(4, N), hh_frac=0.0)
    dev, wl, desc = _setup(cfg)
    out = alloc_outputs(desc, 1, wl.k[0].dtype, dev)
    kvc.kvc_score_weighted(desc, wl.q, wl.k, wl.v, out.scores, out.workspace)
    torch.cuda.synchronize()
    S = out.scores.cpu().numpy()
    for l in range(cfg.n_layers):
        for b in range(cfg.batch):
            ref = oracle.score_layer_vnorm(Pz.to_f32_numpy(wl.q[l][b]), Pz.to_f32_numpy(wl.k[l][b]), Pz.to_f32_numpy(wl.v[l][b]),
                                           1.0 / np.sqrt(d), desc.q_pos0, desc.agg_task, desc.agg_group, bool(desc.augment_head_mean))
            Pz.assert_scores_close(S[l, b], ref)


@pytest.mark.parametrize("Hq,Hkv,w,agg_group", [
    (4, 2, 8, 1), (6, 2, 16, 0),        # whole heads inside a 32-column chunk, the last of them not there
    (8, 2, 9, 1), (8, 2, 31, 0),        # columns taken 8 and 16 at a time, the last ones overlapping
    (14, 2, 33, 1), (4, 2, 127, 0),     # ... and 32 at a time; row tiles of three heads and of one
    (2, 1, 129, 1), (4, 2, 256, 0),     # row tiles of 128 rows and one row; of exactly 128
    (10, 5, 128, 1), (18, 9, 128, 1),   # parts of more KV heads than four, and than eight
])
def test_max_over_windows_of_any_length(Hq, Hkv, w, agg_group):
    """Pass 2 on tiles no mask touches: every way a tile's columns are split into query heads."""
    cfg = W.WorkloadConfig("windows", 2, Hq, Hkv, 128, 700, w, dtype="bf16", elem_std=1.0, hh_frac=0.01)
    dev, wl, desc = _setup(cfg, agg_group=agg_group, q_pos0=700)
    out = alloc_outputs(desc, 1, wl.k[0].dtype, dev)
    kvc.kvc_score(desc, wl.q, wl.k, out.scores, out.workspace)
    torch.cuda.synchronize()
    Pz.assert_scores_close(out.scores.cpu().numpy(), Pz.oracle_scores(wl, desc))


@pytest.mark.parametrize("dtype,Hq,Hkv,w,N,agg_task,explicit", [
    ("f32", 2, 2, 1, 129, 0, False),       # one row per unit; one token more than a tile
    ("f32", 6, 2, 43, 1027, 1, False),     # 129 rows: a second row tile of one row; three tokens into the second chunk
    ("f32", 8, 2, 600, 4100, 0, False),    # a unit's logits fill most of the buffer: one unit per group
    ("f32", 8, 1, 600, 4100, 0, False),    # ... and do not fit it: the two sweeps
    ("bf16", 5, 2, 40, 333, 0, True),      # uneven groups, converted operands
])
def test_scoring_on_the_cuda_cores(dtype, Hq, Hkv, w, N, agg_task, explicit):
    import ctypes
    heads = Hq if explicit else Hkv       # (the generator draws equal groups)
    cfg = W.WorkloadConfig("generic", 1, Hq, heads, 64, N, w, dtype=dtype, elem_std=1.0, hh_frac=0.0)
    dev, wl, desc = _setup(cfg, agg_task=agg_task)
    if explicit:
        wl = W.Workload(cfg, wl.q, [t[:, :Hkv].contiguous() for t in wl.k], [t[:, :Hkv].contiguous() for t in wl.v])
        desc = kvc.kvc_desc_init(1, 1, Hq, Hkv, 64, N, w, kvc.BF16)
        members = (ctypes.c_int32 * Hq)(0, 1, 0, 0, 0)
        desc.q_to_kv = ctypes.cast(members, ctypes.POINTER(ctypes.c_int32))
    out = alloc_outputs(desc, 1, wl.k[0].dtype, dev)
    kvc.kvc_score(desc, wl.q, wl.k, out.scores, out.workspace)
    torch.cuda.synchronize()
    assert not kvc.kvc_score_uses_tensor_cores(desc)
    Pz.assert_scores_close(out.scores.cpu().numpy(), Pz.oracle_scores(wl, desc))


@pytest.mark.parametrize("L,Hkv,N,kind", [
    (32, 8, 1500, "uniform"), (32, 8, 1500, "ties"),      # 256 rows: the most that one CTA selects from, 8 samples each
    (43, 6, 400, "uniform"),                              # 258 rows: the histogram passes
    (17, 2, 61, "uniform"), (33, 1, 63, "ties"),          # 2074 and 2079 entries: one round before the last step
    (32, 1, 64, "uniform"),                               # 2048 entries: the last step alone
])
def test_selection_at_the_limits_of_its_kernel(L, Hkv, N, kind):
    import oracle
    cfg = W.WorkloadConfig("select_limits", L, Hkv, Hkv, 64, N, 1, dtype="f32", elem_std=1.0)
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    desc = kvc.desc_from_config(cfg)
    g = np.random.default_rng(N)
    S = g.random((L, 1, Hkv, N), dtype=np.float32) if kind == "uniform" else \
        (np.round(g.random((L, 1, Hkv, N)) * 3) / 4).astype(np.float32)
    scores = torch.from_numpy(S).to(dev)
    ws = torch.empty(kvc.kvc_workspace_size(desc, 0), dtype=torch.uint8, device=dev)
    idx = torch.empty((L, 1, Hkv, N), dtype=torch.int32, device=dev)
    n_keep = torch.empty((1, L, Hkv), dtype=torch.int32, device=dev)
    off = torch.empty((1, L * Hkv + 1), dtype=torch.int64, device=dev)
    for B in (1, L * Hkv * N // 5, L * Hkv * N - 1):
        kvc.kvc_select_unstructured(desc, scores, B, idx, n_keep, off, ws)
        torch.cuda.synchronize()
        n_ref, off_ref = oracle.select_unstructured(S[:, 0].astype(np.float64), B)
        assert np.array_equal(n_ref, n_keep.cpu().numpy()[0]) and np.array_equal(off_ref, off.cpu().numpy()[0])


@pytest.mark.parametrize("N", [8, 1024, 1025, 2048, 2049, 6144, 6145, 12288, 12289, 16384, 16385, 24576, 24577])
def test_ranking_at_the_switches_of_the_cta_size(N):
    """Eq. 17 on random and heavily tied scores of two segments: CTAs of every size up to 8192 elements, full and barely started;
    longer segments are cut into chunks of about that for the sake of idle SMs (in two, three and four here) and merged."""
    cfg = W.WorkloadConfig("rank_switch", 1, 2, 2, 64, N, 1, dtype="f32", elem_std=1.0)
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    desc = kvc.desc_from_config(cfg)
    g = np.random.default_rng(N)
    S = np.stack([g.random(N, dtype=np.float32), (np.round(g.random(N) * 5) / 8).astype(np.float32)])[None, None]
    idx = torch.empty((1, 1, 2, N), dtype=torch.int32, device=dev)
    comp = torch.empty((1, 1, N), dtype=torch.float32, device=dev)
    ws = torch.empty(kvc.kvc_workspace_size(desc, 0), dtype=torch.uint8, device=dev)
    kvc.kvc_compose(desc, torch.from_numpy(S).to(dev), idx, comp, ws)
    torch.cuda.synchronize()
    Pz.assert_rank_exact(S, idx.cpu().numpy())
    Pz.assert_compose_exact(S, idx.cpu().numpy(), comp.cpu().numpy(), desc.agg_head)


def _rank_many_segments(N):
    """Eq. 17 on 80 segments (so many that none is cut for the sake of idle SMs) of five kinds of scores in turn."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    L, Hkv = 10, 8
    desc = kvc.kvc_desc_init(L, 1, Hkv, Hkv, 64, N, 1, kvc.F32)
    g = np.random.default_rng(N)
    x = g.random((5, N), dtype=np.float32)
    kinds = np.stack([x[0], np.round(x[1] * 5) / 8, (1 + x[2] * 1e-4) / N, np.full(N, 0.25), np.exp(-80 * x[4])]).astype(np.float32)
    S = kinds[np.arange(L * Hkv) % 5].reshape(L, 1, Hkv, N)
    idx = torch.empty((L, 1, Hkv, N), dtype=torch.int32, device=dev)
    comp = torch.empty((L, 1, N), dtype=torch.float32, device=dev)
    ws = torch.empty(kvc.kvc_workspace_size(desc, 0), dtype=torch.uint8, device=dev)
    kvc.kvc_compose(desc, torch.from_numpy(S).to(dev), idx, comp, ws)
    torch.cuda.synchronize()
    got = idx.cpu().numpy().reshape(L * Hkv, N)
    Pz.assert_rank_exact(kinds, got[:5])
    assert np.array_equal(got, got[:5][np.arange(L * Hkv) % 5])
    Pz.assert_compose_exact(S, idx.cpu().numpy(), comp.cpu().numpy(), desc.agg_head)


@pytest.mark.parametrize("N", [8193, 12288, 12289, 16384, 16385, 24576, 24577, 32767, 32768])
def test_ranking_at_the_switches_of_the_larger_cta_sizes(N):
    """Segments in one chunk each: 512 and 1024 threads with 24 and 32 places, full and barely started."""
    _rank_many_segments(N)


@pytest.mark.parametrize("N", [32769, 40960, 40961, 49152, 49153, 65537])
def test_ranking_of_segments_with_a_short_last_chunk(N):
    """Last chunks of one element, of the most for 8 and for 16 places per thread, and of one more."""
    _rank_many_segments(N)


@pytest.mark.parametrize("N", [1, 1023, 1024, 1030])
@pytest.mark.parametrize("Hkv", [1, 9])
def test_streams_of_the_head_sharded_pass_and_composite(N, Hkv):
    """Rows that allow 16-byte accesses and rows that do not, more heads than one batch of loads.  The sums are taken in
    head order (exact); the added mean is one product and one sum, possibly fused: one rounding more or less."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    L, Bt = 2, 3
    desc = kvc.kvc_desc_init(L, Bt, Hkv, Hkv, 64, N, 1, kvc.F32)
    S = np.random.default_rng(N).random((L, Bt, Hkv, N), dtype=np.float32)
    scores = torch.from_numpy(S).to(dev)
    head_sum = torch.empty((L, Bt, N), dtype=torch.float32, device=dev)
    kvc.kvc_head_sum(desc, scores, head_sum)
    want = np.zeros((L, Bt, N), dtype=np.float32)
    for h in range(Hkv):
        want += S[:, :, h]
    assert np.array_equal(head_sum.cpu().numpy(), want)
    kvc.kvc_add_head_mean(desc, scores, head_sum, 2 * Hkv)
    want_s = S.astype(np.float64) + want[:, :, None].astype(np.float64) / (2 * Hkv)
    assert np.allclose(scores.cpu().numpy(), want_s, rtol=3 * 2.0 ** -24, atol=0)
    kvc.kvc_scale(head_sum, 0.5)
    assert np.array_equal(head_sum.cpu().numpy(), want * np.float32(0.5))
    idx = torch.empty((L, Bt, Hkv, N), dtype=torch.int32, device=dev)
    comp = torch.empty((L, Bt, N), dtype=torch.float32, device=dev)
    ws = torch.empty(kvc.kvc_workspace_size(desc, 0), dtype=torch.uint8, device=dev)
    kvc.kvc_compose(desc, scores, idx, comp, ws)
    torch.cuda.synchronize()
    s = scores.cpu().numpy()
    Pz.assert_rank_exact(s, idx.cpu().numpy())
    Pz.assert_compose_exact(s, idx.cpu().numpy(), comp.cpu().numpy(), desc.agg_head)


@pytest.mark.parametrize("N", [31, 16385, 262144, 262145])
def test_position_order_with_the_bitmap_in_either_memory(N):
    """Marks in shared memory (up to 262144 tokens) and in the workspace; more words than threads, a partial last word."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    L, Hkv = 2, 2
    desc = kvc.kvc_desc_init(L, 1, Hkv, Hkv, 64, N, 1, kvc.F32)
    g = np.random.default_rng(N)
    perm = np.stack([np.stack([g.permutation(N) for _ in range(Hkv)]) for _ in range(L)])[:, None].astype(np.int32)
    n_keep = np.array([[N // 3, N - 1]], dtype=np.int32)
    idx = torch.from_numpy(perm.copy()).to(dev)
    ws = torch.empty(kvc.kvc_workspace_size(desc, 0), dtype=torch.uint8, device=dev)
    kvc.kvc_order_kept(desc, idx, torch.from_numpy(n_keep).to(dev), ws)
    torch.cuda.synchronize()
    got = idx.cpu().numpy()
    for l in range(L):
        n = int(n_keep[0, l])
        want = perm[l, 0].copy()
        want[:, :n] = np.sort(want[:, :n], axis=-1)
        assert np.array_equal(got[l, 0], want)


@pytest.mark.parametrize("L,Hkv,N", [(1, 2, 65536), (2, 4, 32768), (2, 4, 16384)])
def test_ranking_into_arrays_that_start_on_four_bytes(L, Hkv, N):
    """Segments of several chunks (eight, four and two: the last merge writes the caller's idx): scores, idx and composite
    need the alignment of their elements only."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    desc = kvc.kvc_desc_init(L, 1, Hkv, Hkv, 64, N, 1, kvc.F32)
    n = L * Hkv * N
    S = np.random.default_rng(N).random(n, dtype=np.float32)
    S[: n // 2] = np.round(S[: n // 2] * 7) / 8
    scores = torch.empty(n + 1, dtype=torch.float32, device=dev)[1:]
    idx_buf = torch.full((n + 2,), -1, dtype=torch.int32, device=dev)
    comp_buf = torch.full((L * N + 2,), -1.0, dtype=torch.float32, device=dev)
    idx, comp = idx_buf[1:n + 1], comp_buf[1:L * N + 1]
    assert [t.data_ptr() % 16 for t in (scores, idx, comp)] == [4, 4, 4]
    scores.copy_(torch.from_numpy(S))
    ws = torch.empty(kvc.kvc_workspace_size(desc, 0), dtype=torch.uint8, device=dev)
    kvc.kvc_compose(desc, scores, idx, comp, ws)
    torch.cuda.synchronize()
    S, got = S.reshape(L, 1, Hkv, N), idx_buf.cpu().numpy()
    assert got[0] == -1 and got[-1] == -1
    Pz.assert_rank_exact(S, got[1:-1].reshape(S.shape))
    got_c = comp_buf.cpu().numpy()
    assert got_c[0] == -1 and got_c[-1] == -1
    Pz.assert_compose_exact(S, got[1:-1].reshape(S.shape), got_c[1:-1].reshape(L, 1, N), desc.agg_head)


@pytest.mark.parametrize("L,Hq,Hkv,w,N", [
    (1, 2, 1, 1, 4096), (1, 2, 1, 1, 4097),        # the statistics of four chunks in one piece, of five in slices
    (2, 6, 3, 3, 9000),                            # six rows: a second CTA of rows in every slice
    (1, 4, 1, 160, 20001),                         # 640 rows, 160 CTAs: slices of three chunks, the last one shorter
    (1, 2, 1, 1, 380929), (1, 2, 1, 1, 1050000),   # slices of one chunk; the log-sum-exp of more chunks than a warp
    (1, 1, 1, 2, 114687), (1, 1, 1, 2, 114688),    # few rows: kept logits, and the two sweeps from here on
    (1, 1, 1, 4, 360448), (1, 1, 1, 5, 360448),    # ... the most rows for the sweeps, and one more
])
def test_scoring_of_long_contexts_on_the_cuda_cores(L, Hq, Hkv, w, N):
    cfg = W.WorkloadConfig("long", L, Hq, Hkv, 64, N, w, dtype="f32", elem_std=1.0, hh_frac=0.0)
    dev, wl, desc = _setup(cfg)
    out = alloc_outputs(desc, 1, wl.k[0].dtype, dev)
    kvc.kvc_score(desc, wl.q, wl.k, out.scores, out.workspace)
    torch.cuda.synchronize()
    Pz.assert_scores_close(out.scores.cpu().numpy(), Pz.oracle_scores(wl, desc))


@pytest.mark.parametrize("G,w", [(1, 6), (1, 7), (2, 2), (3, 1)])
def test_few_rows_of_bf16_with_an_explicit_map(G, w):
    """Two units of 131072 tokens: up to 6 rows of one query head, 2 of two heads go to the two sweeps."""
    import ctypes
    N, Hkv = 131072, 2
    cfg = W.WorkloadConfig("few", 1, G * Hkv, Hkv, 64, N, w, dtype="bf16", elem_std=1.0, hh_frac=0.0)
    dev, wl, desc = _setup(cfg)
    members = (ctypes.c_int32 * (G * Hkv))(*[(j + 1) % Hkv for j in range(G * Hkv)])
    desc.q_to_kv = ctypes.cast(members, ctypes.POINTER(ctypes.c_int32))
    assert not kvc.kvc_score_uses_tensor_cores(desc)
    out = alloc_outputs(desc, 1, wl.k[0].dtype, dev)
    kvc.kvc_score(desc, wl.q, wl.k, out.scores, out.workspace)
    torch.cuda.synchronize()
    Pz.assert_scores_close(out.scores.cpu().numpy(), Pz.oracle_scores(wl, desc))


@pytest.mark.parametrize("dtype,w", [("bf16", 16), ("bf16", 200), ("f32", 16)])
def test_positions_far_behind_the_context_mask_nothing(dtype, w):
    """The largest position there is gives what the first one behind the context gives, bit for bit (full tiles and a partial one)."""
    cfg = W.WorkloadConfig("far", 1, 4, 2, 64, 333, w, dtype=dtype, elem_std=1.0)
    dev, wl, desc = _setup(cfg, q_pos0=333)
    out = alloc_outputs(desc, 1, wl.k[0].dtype, dev)
    kvc.kvc_score(desc, wl.q, wl.k, out.scores, out.workspace)
    want = out.scores.clone()
    for q_pos0 in (2 ** 40, 2 ** 63 - 1):
        desc.q_pos0 = q_pos0
        kvc.kvc_score(desc, wl.q, wl.k, out.scores, out.workspace)
        torch.cuda.synchronize()
        assert torch.equal(out.scores, want)
    Pz.assert_scores_close(want.cpu().numpy(), Pz.oracle_scores(wl, desc))


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("Hq,Hkv,w,d,N,L,batch,q_pos0,scale,pairs", [
    # in pairs (on 148 SMs)
    (136, 8, 128, 128, 1024, 6, 4, 5000, 0.0, 2),    # seventeen row tiles: the last work unit has one; whole runs, no mask
    (152, 8, 128, 128, 6400, 2, 2, 6300, 0.0, 2),    # nineteen row tiles, the mask in the last tile
    (36, 2, 8, 128, 8192, 24, 4, None, 0.0, 2),      # sixteen heads of 8 rows in the first row tile, two in the second
    (18, 2, 16, 128, 8192, 24, 4, None, 0.0, 2),     # eight heads of 16 rows, one
    (14, 2, 32, 128, 6528, 32, 4, 6450, 0.0, 2),     # four heads of 32 rows, three
    (16, 4, 64, 128, 6400, 20, 3, None, 2.0, 2),     # logits more than 40 nats above a run's first: the references move
    (4, 2, 300, 128, 8192, 8, 4, 8150, 0.0, 2),      # long windows: three row tiles per head, the last one short
    (6, 3, 200, 64, 2048, 32, 4, 5000, 4.0, 2),      # heads of 64, two row tiles per head
    (2, 1, 200, 64, 40000, 8, 1, None, 0.0, 2),      # the mask in three of 313 tiles
    # one at a time: the mask, or the end of the context, in more than a fiftieth of the tiles
    (16, 8, 128, 128, 5, 64, 8, None, 0.0, 1),       # contexts of five tokens
    (16, 8, 128, 128, 129, 64, 8, None, 0.0, 1),     # of a tile and a token
    (88, 8, 128, 128, 777, 8, 4, 300, 0.0, 1),
    (36, 2, 8, 128, 640, 80, 10, None, 0.0, 1),
    (18, 2, 16, 128, 640, 80, 10, None, 0.0, 1),
    (14, 2, 32, 128, 1537, 64, 8, 0, 0.0, 1),        # row m sees tokens up to m only
    (16, 4, 64, 128, 1500, 64, 4, None, 2.0, 1),
    (4, 2, 300, 128, 700, 64, 6, 5000, 0.0, 1),
    (6, 3, 200, 64, 2049, 32, 4, None, 4.0, 1),
    (6, 3, 200, 64, 2049, 32, 4, 5000, 4.0, 1),
])
def test_row_tiles_in_pairs_give_the_scores_of_one_at_a_time(Hq, Hkv, w, d, N, L, batch, q_pos0, scale, pairs):
    """Large problems take the row tiles of a KV head two at a time over the same keys, small ones one at a time: the scores of
    all layers together are, bit for bit, those of every layer by itself (which the parity tests hold against the oracle)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(7)
    q = [torch.randn((batch, Hq, w, d), generator=gen, device=dev).to(torch.bfloat16) for _ in range(L)]
    k = [torch.randn((batch, Hkv, N, d), generator=gen, device=dev).to(torch.bfloat16) for _ in range(L)]

    def scores(layers, b, group, row_tiles):
        desc = binding.kvc_desc_init(len(layers), len(b), Hq, Hkv, d, N, w, binding.BF16)
        desc.scale = scale
        desc.agg_group = group
        if q_pos0 is not None:
            desc.q_pos0 = q_pos0
        assert kvc.kvc_score_uses_tensor_cores(desc)
        if _sms() == 148:
            assert kvc.kvc_debug_score_plan(desc, 148)["row_tiles"] == row_tiles
        out = torch.empty((len(layers), len(b), Hkv, N), device=dev)
        ws = torch.empty(kvc.kvc_workspace_size(desc, 0), dtype=torch.uint8, device=dev)
        kvc.kvc_score(desc, [q[i][b] for i in layers], [k[i][b] for i in layers], out, ws)
        return out

    for group in (kvc.AGG_MEAN, kvc.AGG_MAX):
        together = scores(list(range(L)), list(range(batch)), group, pairs)
        for i in range(0, L, max(1, L // 6)):
            b = i % batch
            alone = scores([i], [b], group, 1)
            assert torch.isfinite(alone).all()
            assert torch.equal(together[i, b].view(torch.int32), alone[0, 0].view(torch.int32)), (i, b)


# pairs, beside: row tiles per work unit, and whether the norms' CTAs are in the scoring launch (on 148 SMs)
@pytest.mark.parametrize("L,batch,Hkv,d,N,w,pad,pairs,beside", [
    (3, 2, 5, 128, 17, 4, 0, 1, True),         # fewer blocks of rows than warps that take them
    (2, 3, 4, 64, 1033, 32, 64, 1, True),      # rows apart in memory, a short last block per segment
    (24, 4, 8, 128, 515, 16, 0, 1, True),      # many segments per warp
    (1, 1, 2, 128, 40007, 32, 128, 1, True),   # one long segment after the other
    (20, 2, 4, 128, 2100, 130, 0, 1, True),
    (40, 2, 8, 128, 2560, 128, 64, 2, True),   # row tiles in pairs beside the norms
    (28, 1, 4, 128, 3200, 500, 0, 2, True),    # ... of a long window
    (16, 1, 8, 128, 4096, 500, 0, 2, False),   # row tiles in pairs, the norms in their own kernel
])
def test_value_norms_beside_the_scoring(L, batch, Hkv, d, N, w, pad, pairs, beside):
    """The norms that the scoring launch takes along: weighted scores are the plain ones times the norms of the value rows (the
    norm's squares are added in fp32 with errors below 1e-6)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(3)

    def rand(*shape):
        return torch.randn(shape, generator=gen, device=dev).to(torch.bfloat16)

    q = [rand(batch, 2 * Hkv, w, d) for _ in range(L)]
    k = [rand(batch, Hkv, N, d + pad)[..., :d] for _ in range(L)]
    v = [(rand(batch, Hkv, N, d + pad) * (1 + i))[..., :d] for i in range(L)]
    desc = binding.kvc_desc_init(L, batch, 2 * Hkv, Hkv, d, N, w, binding.BF16)
    desc.augment_head_mean = 0
    desc.q_pos0 = N
    for i, s in enumerate(k[0].stride()[:3]):
        desc.kv_stride[i] = s
    assert kvc.kvc_score_uses_tensor_cores(desc)
    plain, weighted = (torch.empty((L, batch, Hkv, N), device=dev) for _ in range(2))
    kvc.kvc_score(desc, q, k, plain, torch.empty(kvc.kvc_workspace_size(desc, 0), dtype=torch.uint8, device=dev))
    desc.value_norm = 1
    if _sms() == 148:
        plan = kvc.kvc_debug_score_plan(desc, 148)
        assert plan["row_tiles"] == pairs and (plan["norm_ctas"] > 0) == beside
    ws = torch.full((kvc.kvc_workspace_size(desc, 0),), 0xff, dtype=torch.uint8, device=dev)
    kvc.kvc_score_weighted(desc, q, k, v, weighted, ws)
    want = torch.stack([p.double() * x.double().norm(dim=-1) for p, x in zip(plain, v)])
    assert torch.isfinite(weighted).all()
    assert ((weighted.double() - want).abs() <= 1e-6 * want.abs()).all()
