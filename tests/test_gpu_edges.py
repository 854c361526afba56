"""GPU parity at the sizes where the kernels' own cuts fall: ends of tiles, chunks and register blocks, remainders, the
smallest and the largest of each range.  Tolerances are those of the kernels' own test files (scores: 1e-4 relative, a
bound on a few fp32 roundings of the exponent's argument; everything else exact)."""
import numpy as np
import pytest

import oracle
from helpers import cu_of, rand_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,L,W,Hq,Hkv,d", [
    ((1,), 1, 1, 1, 1, 64),                                # one key, one row
    ((127,), 1, 32, 8, 2, 128), ((128,), 1, 32, 8, 2, 128), ((129,), 1, 32, 8, 2, 128),     # ends of a key tile
    ((384, 1, 128, 5), 3, 32, 4, 1, 64),                   # tile multiples beside single keys; a CTA per tile
    ((130,) * 40, 8, 16, 8, 2, 64),                        # 1280 tiles: every CTA's range crosses several sequences
    ((2560,), 1, 48, 8, 2, 128),                           # R = 192: two row blocks, the second one partial
    ((2560, 700), 1, 65, 20, 4, 64),                       # R = 325: three row blocks over three warpgroups
    ((1300,), 2, 33, 16, 1, 64),                           # R = 528: five row blocks, a warpgroup takes two of a tile
    ((700, 130, 900), 8, 38, 32, 8, 128),                  # R = 152, a few segments per CTA: records of several rows merged together
    ((19000,), 1, 8, 8, 8, 64),                            # 8 x 149 tiles: one more per KV head than there are SMs
])
def test_score_at_the_cuts(lens, L, W, Hq, Hkv, d):
    import gpu_ops
    rng = np.random.default_rng(11)
    cu = cu_of(lens)
    q, k = rand_bf16(rng, (L, len(lens), W, Hq, d)), rand_bf16(rng, (L, int(cu[-1]), Hkv, d))
    want = oracle.score(q, k, cu).astype(np.float64)
    got = gpu_ops.score(q, k, cu)
    assert np.all(np.abs(got - want) <= 1e-4 * np.abs(want) + 1e-30)


@pytest.mark.parametrize("ks,d,Hkv", [
    ((1,), 128, 1), ((63,), 128, 3), ((64,), 128, 2), ((65,), 128, 2), ((127,), 64, 2), ((128,), 64, 2), ((129,), 64, 3),
    ((0, 64, 0, 1, 200), 128, 2),                          # empty rows at and between the cuts of a CTA's entries
    ((5,) * 32, 64, 2), ((3,) * 33, 128, 1), ((2,) * 70, 64, 2),         # 32 sequences and more: the two ways of the search
])
@pytest.mark.parametrize("counted", [False, True])
def test_pack_at_the_cuts(ks, d, Hkv, counted):
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(12)
    L, lens = 2, tuple(k + 3 for k in ks)
    cu, ck = cu_of(lens), cu_of(ks)
    T, K = int(cu[-1]), int(ck[-1])
    kc, vc = rand_bf16(rng, (L, T, Hkv, d)), rand_bf16(rng, (L, T, Hkv, d))
    sel = np.zeros((L, Hkv, K), dtype=np.int32)
    cnt = np.zeros((L, len(ks), Hkv), dtype=np.int32)
    want_k, want_v = np.full((L, K * Hkv, d), 0x5555, np.uint16), np.full((L, K * Hkv, d), 0x5555, np.uint16)
    for l in range(L):
        for b, n in enumerate(lens):
            for g in range(Hkv):
                sel[l, g, ck[b]:ck[b + 1]] = np.sort(rng.choice(n, ks[b], replace=False))
                cnt[l, b, g] = rng.integers(0, ks[b] + 1) if counted else ks[b]
                for j in range(cnt[l, b, g]):
                    r, t = ck[b] * Hkv + g * ks[b] + j, cu[b] + sel[l, g, ck[b] + j]
                    want_k[l, r], want_v[l, r] = kc[l, t, g], vc[l, t, g]
    if counted:
        pk, pv = (gpu_ops.Guarded((L, K * Hkv, d), torch.int16, 0x5555) for _ in range(2))
        st = gpu_ops.status_word()
        sg.sg_pack_kv_counted(gpu_ops.shape_of(L, Hkv, Hkv, d, 1, cu), gpu_ops.dev(kc), gpu_ops.dev(vc), gpu_ops.dev(sel),
                              gpu_ops.dev(ck), K, gpu_ops.dev(cnt), pk.view, pv.view, st)
        got_k, got_v = pk.numpy(), pv.numpy()
        assert gpu_ops.read_status(st) == 0
    else:
        got_k, got_v = gpu_ops.pack_kv(kc, vc, cu, sel, ck)
    assert np.array_equal(got_k, want_k) and np.array_equal(got_v, want_v)


@pytest.mark.parametrize("ks", [(31,), (32,), (33,), (1024, 1025, 0, 1), (8191,), (8192,), (8193,), (20000, 7)])
def test_split_at_the_cuts(ks):
    from test_gpu_split import make, run_gpu
    idx, mask, cu, ck = make(13, tuple(k + 5 for k in ks), ks, 2, (0.1, 0.5, 0.4))
    for reorder in (True, False):
        want = oracle.split_index(idx, mask, cu, ck, reorder=reorder)
        for a, b in zip(run_gpu(idx, mask, cu, ck, reorder), want):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("lens,ks", [
    ((300,), (256,)), ((300,), (257,)), ((1100,), (1024,)), ((1100,), (1025,)), ((2500,), (2048,)), ((2500,), (2049,)),   # ends of the CTA sizes
    ((5000,), (4096,)), ((5000,), (4097,)),
    ((1300, 40, 1), (1024, 0, 1)), ((3000,) + (100,) * 60, (2900,) + (0,) * 60),      # a row longer than the CTA was chosen for
    ((700,) * 30, (90,) * 30),
])
def test_split_cta_sizes(lens, ks):
    from test_gpu_split import make, run_gpu
    idx, mask, cu, ck = make(17, lens, ks, 3, (0.1, 0.5, 0.4))
    for reorder in (True, False):
        want = oracle.split_index(idx, mask, cu, ck, reorder=reorder)
        for a, b in zip(run_gpu(idx, mask, cu, ck, reorder), want):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [5, 4093, 4096, 8189, 8190, 8192, 16383, 16384, 32765, 32768])
def test_select_rows_off_the_16_byte_boundary(n):
    """Rows that start 0 to 3 values behind a 16-byte boundary, up to the longest of every kernel variant; values from
    all different to a handful, so that the last interval holds from one key to thousands."""
    import gpu_ops
    rng = np.random.default_rng(17)
    for lead, steps in ((0, 1e9), (1, 2000.0), (2, 100.0), (3, 1.0)):
        lens, ks = (lead, n, 2, n), (min(lead, 1), max(1, n // 10), 1, n - 1)
        cu, ck = cu_of(lens), cu_of(ks)
        x = (np.round(rng.standard_normal((1, 2, int(cu[-1]))) * steps) / steps).astype(np.float32)
        want = oracle.select_topk(x, cu, ck)
        assert np.array_equal(gpu_ops.select_topk(x, cu, ck), want)


@pytest.mark.parametrize("n", [1, 31, 4096, 4097, 8192, 8193, 16385, 32768, 32769])
def test_threshold_at_the_cuts(n):
    """Row lengths at the ends of every kernel variant; caps that bind, that are met exactly and that are the whole row."""
    from test_gpu_threshold import run
    rng = np.random.default_rng(14)
    x = np.round(rng.standard_normal((2, 2, n)) * 8).astype(np.float32) / 4                # many ties
    x[0, 0, n // 2] = -np.inf
    above = int((x[1, 0] > x[1, 0].max() - 1.5).sum())
    for cap in sorted({1, min(above, n), min(above + 1, n), max(1, above - 1), n}):
        run(x, (n,), (cap,), 1.5)
    run(np.full((1, 1, n), -np.inf, np.float32), (n,), (n,), 1.0)                           # nothing exceeds -inf


@pytest.mark.parametrize("lens,Hkv,d,M,n_sel", [
    ((640,), 3, 128, 64, 64), ((641, 1, 90), 2, 64, 64, 9), ((5,), 1, 64, 8, 1),      # a list no longer than the layer's blocks
])
@pytest.mark.parametrize("head_major", [False, True])
def test_push_by_list(lens, Hkv, d, M, n_sel, head_major):
    from test_gpu_push import run_case
    run_case(15, lens, Hkv, d, M, 2, n_sel, head_major)


@pytest.mark.parametrize("lens,L,W,Hq,Hkv,d", [
    ((33000,), 1, 4, 8, 8, 128),                           # 67.6 MB of keys, one layer: every KV head is cut over many CTAs
    ((20000, 3, 14001), 2, 16, 16, 8, 128),                # ragged, 139 MB of keys, a part of three keys between long ones
    ((130000,), 2, 8, 4, 4, 64),                           # 133 MB of keys, long rows of 64-element heads
])
def test_score_keys_beyond_l2(lens, L, W, Hq, Hkv, d):
    """Calls with half of L2 to more than all of it in keys; the call is repeated on the same workspace, whose words then
    hold the first call's records."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(16)
    cu = cu_of(lens)
    T = int(cu[-1])
    q, k = rand_bf16(rng, (L, len(lens), W, Hq, d)), rand_bf16(rng, (L, T, Hkv, d))
    want = oracle.score(q, k, cu).astype(np.float64)
    shp = gpu_ops.shape_of(L, Hq, Hkv, d, W, cu)
    ws, st = sg.alloc_workspace(sg.SG_OP_SCORE, shp), gpu_ops.status_word()
    dq, dk = gpu_ops.dev(q), gpu_ops.dev(k)
    for _ in range(2):
        imp = gpu_ops.Guarded((L, Hkv, T), torch.float32, -7.0)
        sg.sg_score(shp, dq, dk, imp.view, ws, st)
        assert np.all(np.abs(imp.numpy() - want) <= 1e-4 * np.abs(want) + 1e-30)
    assert gpu_ops.read_status(st) == 0


# Lists that give the eight warps of a CTA none to several slices of 16, cut one entry to either side, the packed part ending
# on, behind and before a slice boundary.
RING_KS = (0, 1, 15, 16, 127, 129, 256, 383, 511, 640, 769, 1023)


@pytest.mark.parametrize("ks,nls,Hq,Hkv,d", [
    (RING_KS, tuple(reversed(RING_KS)), 32, 8, 128),              # one CTA per pair, rings of three
    (RING_KS, tuple(reversed(RING_KS)), 64, 8, 64),               # G = 8
    (RING_KS, tuple(reversed(RING_KS)), 72, 8, 128),              # G = 9: two tiles of query rows, rings of six
    (RING_KS, tuple(reversed(RING_KS)), 128, 8, 64),              # G = 16
    (tuple(4 * k for k in RING_KS), (0,) * 12, 32, 8, 128), # packed rows only, 1024 and more on average: rings of six
    (tuple(4 * k for k in RING_KS), (0,) * 12, 16, 8, 64),
    ((1500,) * 20, RING_KS[:10] * 2, 32, 8, 128),                 # the same, long ones: eight warps
    ((767,) * 10 + (770,), (0,) * 11, 32, 8, 128), ((769,) * 11, (0,) * 11, 32, 8, 128),   # packed only, to either side of six slices per warp
    ((1535,) * 8, (0,) * 8, 32, 8, 128), ((1537,) * 8, (0,) * 8, 32, 8, 128),     # the same for clusters of two
    ((1100,) * 19, (0,) * 19, 32, 8, 128), ((1023,) * 19, (0,) * 19, 32, 8, 128),  # packed only, up to one and a half CTAs per SM
    ((1100,) * 28, (0,) * 28, 32, 8, 128), ((1100,) * 19, (0,) * 19, 32, 8, 64),   # ... and what keeps eight warps
])
def test_decode_rings(ks, nls, Hq, Hkv, d):
    """Against the oracle on inputs where one dropped or misplaced row shows (tolerances: see test_gpu_decode_sentinel)."""
    from test_gpu_decode_sentinel import build_sentinel, check
    check(build_sentinel(3, tuple(a + b + 5 for a, b in zip(ks, nls)), ks, nls, Hq, Hkv, d))


def test_decode_rings_of_short_lists():
    """More pairs than SMs, four warps.  Values of N(0, 1): the sentinels of a three-entry list average to 20, where bf16
    rounding alone (2^-9 relative, of the weights and of the output) is beyond the absolute tolerance."""
    from test_gpu_decode import build, compare
    nls = RING_KS[:10] * 2
    compare(build(3, tuple(n + 8 for n in nls), (3,) * 20, nls, 32, 8, 128))


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("where,at", [
    ("query", 4), ("query", 6), ("query", 31), ("query", 127),             # row of the block: exponentials on either pipe
    ("key", 5), ("key", 6), ("key", 262), ("key", 1279), ("key", 1299),    # the same for keys; the last ones are not seen by all rows
])
@pytest.mark.parametrize("W,launches", [(32, 1), (32, 2), (13, 1), (13, 2)])               # 128 query rows; 52, which stand twice
def test_score_non_finite_input_marks_its_part(value, where, at, W, launches):
    """A NaN or an infinity in one query or key makes every importance of its (layer, KV head, sequence) NaN, wherever it
    stands, and changes nothing else.  sg_score takes one kernel for such a shape, sg_score_static always two."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(14)
    L, lens, Hq, Hkv, d = 2, (700, 1300), 8, 2, 128
    G, l, b, g = Hq // Hkv, 1, 1, 1
    at = at % (G * W) if where == "query" else at
    cu = cu_of(lens)
    q = gpu_ops.dev(rand_bf16(rng, (L, 2, W, Hq, d))).view(torch.bfloat16)
    k = gpu_ops.dev(rand_bf16(rng, (L, int(cu[-1]), Hkv, d))).view(torch.bfloat16)
    shp = gpu_ops.shape_of(L, Hq, Hkv, d, W, cu)
    ws, st = sg.alloc_workspace(sg.SG_OP_SCORE, shp), gpu_ops.status_word()
    clean, got = (torch.empty((L, Hkv, int(cu[-1])), dtype=torch.float32, device="cuda") for _ in range(2))
    assert sg.sg_testing_score_cluster(shp) > 0
    score = (lambda out: sg.sg_score(shp, q, k, out, ws, st)) if launches == 1 else (lambda out: sg.sg_score_static(shp, q, k, out, st))
    score(clean)
    if where == "query":
        q[l, b, at // G, g * G + at % G, 3] = value
    else:
        k[l, int(cu[b]) + at, g, 3] = value
    score(got)
    assert gpu_ops.read_status(st) == 0
    part = torch.zeros_like(got, dtype=torch.bool)
    part[l, g, int(cu[b]):int(cu[b + 1])] = True
    assert bool(got[part].isnan().all())
    assert torch.equal(got[~part], clean[~part]) and bool(clean.isfinite().all())


@pytest.mark.parametrize("B", [1, 2, 32, 33])
@pytest.mark.parametrize("counted", [False, True])
def test_pack_total_above_the_prefix_array(B, counted):
    """A host total larger than cu_k[B] is flagged; the entries that belong to no row are skipped, the others packed."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(15)
    k, more, Hkv, d = 9, 200, 1, 128                       # one KV head: the rows of the surplus lie behind all others
    cu, ck = cu_of((12,) * B), cu_of((k,) * B)
    K = B * k
    kc = rand_bf16(rng, (1, 12 * B, Hkv, d))
    sel = np.tile(np.arange(k, dtype=np.int32), B + more)[None, None, :K + more].copy()
    pk, pv = (gpu_ops.Guarded((1, (K + more) * Hkv, d), torch.int16, 0x5555) for _ in range(2))
    shp, st = gpu_ops.shape_of(1, Hkv, Hkv, d, 1, cu), gpu_ops.status_word()
    args = [shp, gpu_ops.dev(kc), gpu_ops.dev(kc), gpu_ops.dev(sel), gpu_ops.dev(ck), K + more]
    if counted:
        sg.sg_pack_kv_counted(*args, torch.full((1, B, Hkv), k, dtype=torch.int32, device="cuda"), pk.view, pv.view, st)
    else:
        sg.sg_pack_kv(*args, pk.view, pv.view, st)
    assert gpu_ops.read_status(st) == 1 << sg.SG_ERR_INVALID
    want = np.concatenate([kc[0, 12 * b:12 * b + k, 0] for b in range(B)])
    for got in (pk.numpy(), pv.numpy()):
        assert np.array_equal(got[0, :K], want) and np.all(got[0, K:] == 0x5555)


@pytest.mark.parametrize("call", ["prefill", "prefill_layer", "select_pack"])
@pytest.mark.parametrize("L,lens,Hkv", [
    (1, (900,), 2), (1, (900, 40, 300), 2),                # one kernel for scoring, selection and packing
    (8, (400,), 20), (8, (400, 30), 10),                   # 160 rows: selection and packing in one kernel
    (1, (20000, 9000), 4),                                 # the calls one by one
])
def test_selection_total_above_the_prefix_array(call, L, lens, Hkv):
    """The same through the calls that select and pack: the status bit of sg_pack_kv, and every row of the prefix array right."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(19)
    W, d, more = 8, 64, 50
    if call == "prefill_layer":
        L = 1
    ks = tuple(max(1, n // 7) for n in lens)
    cu, ck = cu_of(lens), cu_of(ks)
    T, Kb = int(cu[-1]), int(ck[-1])
    K = Kb + more
    q, k, v = rand_bf16(rng, (L, len(lens), W, Hkv, d)), rand_bf16(rng, (L, T, Hkv, d)), rand_bf16(rng, (L, T, Hkv, d))
    x = rng.standard_normal((L, Hkv, T)).astype(np.float32)
    shp, st, d_ck = gpu_ops.shape_of(L, Hkv, Hkv, d, W, cu), gpu_ops.status_word(), gpu_ops.dev(ck)
    imp, sel = gpu_ops.dev(x), torch.full((L, Hkv, K), -99, dtype=torch.int32, device="cuda")
    pk, pv = (gpu_ops.Guarded((L, K * Hkv, d), torch.int16, 0x5555) for _ in range(2))
    ws = sg.alloc_workspace(sg.SG_OP_SCORE, shp)
    if call == "prefill":
        sg.prefill(shp, gpu_ops.dev(q), gpu_ops.dev(k), gpu_ops.dev(v), imp, ws, d_ck, K, sel, pk.view, pv.view, st)
    elif call == "prefill_layer":
        sg.prefill_layer(shp, 0, gpu_ops.dev(q), gpu_ops.dev(k), gpu_ops.dev(v), imp, ws, d_ck, K, sel, pk.view, pv.view, st)
    else:
        sg.sg_select_pack_kv(shp, imp, d_ck, K, gpu_ops.dev(k), gpu_ops.dev(v), sel, pk.view, pv.view, st)
    got_k, got_v = pk.numpy(), pv.numpy()
    assert gpu_ops.read_status(st) == 1 << sg.SG_ERR_INVALID
    sel = sel.cpu().numpy()
    want = oracle.select_topk(imp.cpu().numpy(), cu, ck)
    assert np.array_equal(sel[:, :, :Kb], want) and np.all(sel[:, :, Kb:] == -99)
    want_k, want_v = oracle.pack_kv(k, v, cu, want, ck)
    for got, rows in ((got_k, want_k), (got_v, want_v)):
        assert np.array_equal(got[:, :Kb * Hkv], rows) and np.all(got[:, Kb * Hkv:] == 0x5555)


@pytest.mark.parametrize("lens,L,W,Hq,Hkv,d", [
    # such a part as a CTA's second, third and fourth segment, between segments that the helper merges: 384 rows, 1024 rows
    ((12478, 16, 31, 15649, 31, 99, 84, 17425, 94, 32, 10011, 52, 89, 84), 1, 24, 16, 1, 128),
    ((18982, 60, 13, 5233, 43, 29, 21, 3168, 45, 53, 64), 2, 64, 16, 1, 64),
    ((20000, 1, 1, 20000, 1, 1, 20000), 1, 64, 16, 1, 64),
    ((5000, 5000, 60, 5000), 3, 100, 8, 1, 64),            # 800 rows, the last block partial
    ((700, 20, 3, 900), 1, 128, 16, 4, 64),                # 512 rows, a tile or two per CTA: none
])
def test_score_long_parts_behind_short_segments(lens, L, W, Hq, Hkv, d):
    """Parts over many CTAs whose records the epilogue warps merge themselves, at any place of a CTA's segments."""
    import gpu_ops
    rng = np.random.default_rng(18)
    cu = cu_of(lens)
    q, k = rand_bf16(rng, (L, len(lens), W, Hq, d)), rand_bf16(rng, (L, int(cu[-1]), Hkv, d))
    want = oracle.score(q, k, cu).astype(np.float64)
    for _ in range(3):
        got = gpu_ops.score(q, k, cu)
        assert np.all(np.abs(got - want) <= 1e-4 * np.abs(want) + 1e-30)
