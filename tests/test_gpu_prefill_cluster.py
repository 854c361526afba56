"""GPU: scoring, selection and packing in one kernel (a cluster of CTAs per layer, sequence and KV head).

Scores against the two-launch form (sg_score_static always takes it) and the oracle; the index against the oracle's selection on
the GPU's own scores, and the packed rows against its gather: whole values, exact.  Shapes at the edges of key tiles, of the query
row blocks, of the cluster sizes and of the budgets.
"""
import numpy as np
import pytest

import oracle
from helpers import cu_of, rand_bf16

pytestmark = pytest.mark.gpu


def run(lens, L, W, Hq, Hkv, d, budgets, seed=0, k_h=None, max_seqlen=None, pad_heads=0, one_kernel=True):
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(seed)
    cu, ck = cu_of(lens), cu_of(budgets)
    T, K = int(cu[-1]), int(ck[-1])
    q_h = rand_bf16(rng, (L, len(lens), W, Hq, d))
    k_h = rand_bf16(rng, (L, T, Hkv, d)) if k_h is None else k_h
    v_h = rand_bf16(rng, (L, T, Hkv, d))
    wide = [np.concatenate([x, rand_bf16(rng, (L, T, pad_heads, d))], axis=2) if pad_heads else x for x in (k_h, v_h)]
    shp = gpu_ops.shape_of(L, Hq, Hkv, d, W, cu, layer_stride=T * (Hkv + pad_heads) * d, token_stride=(Hkv + pad_heads) * d)
    if max_seqlen is not None:
        shp.max_seqlen = max_seqlen
    cluster = sg.sg_testing_score_cluster(shp)
    assert (cluster > 0) == one_kernel
    q, k, v = (gpu_ops.dev(x) for x in (q_h, *wide))
    st, ws = gpu_ops.status_word(), sg.alloc_workspace(sg.SG_OP_SCORE, shp)
    imp = gpu_ops.Guarded((L, Hkv, T), torch.float32, -7.0)
    sel = gpu_ops.Guarded((L, Hkv, K), torch.int32, -99)
    pk, pv = (gpu_ops.Guarded((L, K * Hkv, d), torch.int16, 77) for _ in range(2))
    sg.prefill(shp, q, k, v, imp.view, ws, gpu_ops.dev(ck), K, sel.view, pk.view, pv.view, st)
    alone, two = (torch.full((L, Hkv, T), -7.0, dtype=torch.float32, device="cuda") for _ in range(2))
    sg.sg_score(shp, q, k, alone, ws)
    sg.sg_score_static(shp, q, k, two)
    got = imp.numpy()
    for other in (alone.cpu().numpy(), two.cpu().numpy()):
        assert np.all(np.abs(got - other) <= 1e-5 * np.abs(other) + 1e-30)     # the same sums, or fp32 sums in another order
    if any(k > n for k, n in zip(budgets, lens)):                       # outside the oracle's contract: the two calls
        two_st, other = gpu_ops.status_word(), [torch.full_like(x.view, 5) for x in (sel, pk, pv)]
        sg.sg_select_topk(shp, imp.view, gpu_ops.dev(ck), K, other[0], None, two_st)
        sg.sg_pack_kv(shp, k, v, other[0], gpu_ops.dev(ck), K, other[1], other[2], two_st)
        for x, y in zip((sel, pk, pv), other):
            assert np.array_equal(x.numpy().view(y.cpu().numpy().dtype), y.cpu().numpy())
        assert gpu_ops.read_status(two_st) == gpu_ops.read_status(st)
        return cluster, got, q_h, k_h, cu, gpu_ops.read_status(st)
    sel_o = oracle.select_topk(got, cu, ck)
    assert np.array_equal(sel.numpy(), sel_o)
    pk_o, pv_o = oracle.pack_kv(k_h, v_h, cu, sel_o, ck)
    assert np.array_equal(pk.numpy(), pk_o) and np.array_equal(pv.numpy(), pv_o)
    return cluster, got, q_h, k_h, cu, gpu_ops.read_status(st)


@pytest.mark.parametrize("lens,L,W,Hq,Hkv,d,budgets", [
    ((8192,), 1, 32, 32, 8, 128, (820,)),                       # ten CTAs per part, seven tiles each, some loaded twice
    ((1024,), 1, 16, 8, 2, 64, (128,)),                         # a tile per CTA, half of the query rows are padding
    ((8191, 4097), 1, 16, 8, 2, 128, (100, 4096)),              # tails of one key less and one more; most keys kept
    ((1, 5, 127, 128, 129, 300), 1, 16, 8, 2, 64, (1, 2, 127, 64, 3, 299)),       # prompts shorter than the window
    ((2000,), 2, 40, 16, 2, 128, (1,)),                         # 320 query rows: three row blocks
    ((900,), 1, 32, 16, 1, 64, (90,)),                          # 512 query rows: four row blocks
    ((1500, 40), 1, 24, 16, 2, 128, (0, 40)),                   # 192 rows; an empty budget and a whole prompt
    ((700,), 1, 5, 6, 2, 64, (33,)),                            # 15 rows
    ((640, 10), 1, 64, 16, 2, 64, (64, 9)),                     # 512 rows; nine keys of ten
    ((15000,), 1, 16, 16, 4, 128, (2000,)),                     # sixteen CTAs, eight tiles each, two of them held at a time
    ((14000,), 1, 16, 8, 2, 128, (2000,)),                      # ... seven
    ((100,) * 18, 1, 16, 8, 8, 64, (10,) * 18),                 # 144 parts of one CTA
    ((7000, 3000, 200), 2, 16, 4, 2, 64, (700, 2999, 1)),       # clusters whose CTAs have from none to five tiles
])
def test_prefill_in_one_kernel(lens, L, W, Hq, Hkv, d, budgets):
    cluster, got, q_h, k_h, cu, status = run(lens, L, W, Hq, Hkv, d, budgets)
    assert status == 0
    want = oracle.score(q_h, k_h, cu)
    assert np.all(np.abs(got - want) <= 1e-4 * np.abs(want) + 1e-30)


# (query rows, tiles of the longest prompt's CTAs, ...): where the launches one by one are faster, they are taken
@pytest.mark.parametrize("lens,L,W,Hq,Hkv,d,one_kernel", [
    ((8192,), 1, 32, 32, 8, 128, True), ((10000,), 1, 32, 32, 8, 128, True), ((8192,), 2, 32, 32, 8, 128, False),
    ((15000,), 1, 16, 8, 2, 128, False),                        # two parts, eight tiles
    ((100,) * 7 + (2048,), 1, 32, 32, 8, 128, False), ((100,) * 7 + (1790,), 1, 32, 32, 8, 128, True),
    ((100,) * 7 + (2048,), 1, 32, 16, 8, 64, True),             # 64 rows, heads of 64
    ((2040, 100) * 4, 1, 32, 32, 8, 128, True),
    ((100,) * 7 + (1270,), 1, 64, 32, 8, 128, False), ((100,) * 7 + (900,), 1, 64, 32, 8, 128, True),      # 256 rows
    ((1270, 100) * 4, 1, 64, 32, 8, 128, True),
    ((100,) * 20 + (1900,), 1, 64, 16, 2, 64, False),           # 512 rows
])
def test_where_one_kernel_pays(lens, L, W, Hq, Hkv, d, one_kernel):
    """The route, and the same results on either."""
    assert run(lens, L, W, Hq, Hkv, d, tuple(max(1, n // 9) for n in lens), one_kernel=one_kernel)[-1] == 0


def test_prefill_in_one_kernel_from_a_wider_cache():
    assert run((900, 333), 2, 16, 8, 2, 128, (90, 33), pad_heads=3)[-1] == 0


def test_ties_go_to_the_lower_position():
    """Keys of three kinds only, in blocks: every importance occurs many times, on both sides of every CTA's range."""
    rng = np.random.default_rng(3)
    kinds = rand_bf16(rng, (3, 1, 2, 64))
    k_h = kinds[rng.integers(0, 3, 3000)].transpose(1, 0, 2, 3).copy()
    for budget in (1, 700, 1500, 2900):
        assert run((3000,), 1, 16, 8, 2, 64, (budget,), k_h=k_h)[-1] == 0


def test_more_candidates_than_are_ranked_directly():
    """Thousands of keys within a few roundings of one another: the interval is narrowed more than once."""
    rng = np.random.default_rng(4)
    k_h = np.broadcast_to(rand_bf16(rng, (1, 1, 2, 64)), (1, 4000, 2, 64)).copy()
    k_h[0, ::7] = rand_bf16(rng, (572, 2, 64), 0.01)
    k_h[0, 5] = rand_bf16(rng, (2, 64), 4.0)
    run((4000,), 1, 16, 8, 2, 64, (2000,), k_h=k_h)


def test_budget_above_the_prompt_and_empty_sequence():
    import paper_2607_28150_b200.binding as sg
    status = run((200, 0, 1000), 1, 16, 8, 2, 64, (230, 7, 100))[-1]
    assert status == (1 << sg.SG_ERR_INVALID) | (1 << sg.SG_ERR_INDEX)


def test_non_finite_key_marks_its_part_only():
    rng = np.random.default_rng(5)
    k_h = rand_bf16(rng, (1, 3000, 2, 128))
    k_h[0, 1234, 1, 17] = 0x7fc0
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    cu = cu_of((2000, 1000))
    shp = gpu_ops.shape_of(1, 8, 2, 128, 16, cu)
    assert sg.sg_testing_score_cluster(shp) > 0
    imp = torch.zeros((1, 2, 3000), device="cuda")
    sg.sg_score(shp, gpu_ops.dev(rand_bf16(rng, (1, 2, 16, 8, 128))), gpu_ops.dev(k_h), imp, sg.alloc_workspace(sg.SG_OP_SCORE, shp))
    nan = torch.isnan(imp[0])
    assert bool(nan[1, :2000].all()) and not bool(nan[0].any()) and not bool(nan[1, 2000:].any())


def test_longest_sequence_above_what_max_seqlen_promised():
    """Scores stay right (the tiles that do not fit are loaded again); the selection flags the row, as the calls one by one do."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(6)
    lens, budgets = (3000, 100), (300, 10)
    cu, ck = cu_of(lens), cu_of(budgets)
    q_h, k_h, v_h = rand_bf16(rng, (1, 2, 16, 8, 64)), rand_bf16(rng, (1, 3100, 2, 64)), rand_bf16(rng, (1, 3100, 2, 64))
    shp = gpu_ops.shape_of(1, 8, 2, 64, 16, cu)
    shp.max_seqlen = 300
    assert sg.sg_testing_score_cluster(shp) > 0
    imp = torch.zeros((1, 2, 3100), device="cuda")
    sel = torch.zeros((1, 2, 310), dtype=torch.int32, device="cuda")
    pk, pv = (torch.ones((1, 620, 64), dtype=torch.int16, device="cuda") for _ in range(2))
    st = gpu_ops.status_word()
    sg.prefill(shp, gpu_ops.dev(q_h), gpu_ops.dev(k_h), gpu_ops.dev(v_h), imp, sg.alloc_workspace(sg.SG_OP_SCORE, shp), gpu_ops.dev(ck), 310,
               sel, pk, pv, st)
    assert gpu_ops.read_status(st) == (1 << sg.SG_ERR_INVALID) | (1 << sg.SG_ERR_INDEX)
    want = oracle.score(q_h, k_h, cu)
    assert np.all(np.abs(imp.cpu().numpy() - want) <= 1e-4 * np.abs(want) + 1e-30)
    sel = sel.cpu().numpy()
    assert np.all(sel[:, :, :300] == -1) and np.array_equal(sel[:, :, 300:], oracle.select_topk(imp.cpu().numpy(), cu, ck)[:, :, 300:])
    assert not pk[0, :600].any() and not pv[0, :600].any()


def test_expired_wait_ends_cleanly_and_the_next_call_is_correct():
    """One part's statistics are withheld and every wait limited to 10 ms: the cluster gives up and says so."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(7)
    cu, ck = cu_of((2000, 500)), cu_of((200, 50))
    q_h, k_h = rand_bf16(rng, (1, 2, 16, 8, 128)), rand_bf16(rng, (1, 2500, 2, 128))
    q, k = gpu_ops.dev(q_h), gpu_ops.dev(k_h)
    shp = gpu_ops.shape_of(1, 8, 2, 128, 16, cu)
    assert sg.sg_testing_score_cluster(shp) > 0
    ws, imp = sg.alloc_workspace(sg.SG_OP_SCORE, shp), torch.zeros((1, 2, 2500), device="cuda")
    sel = torch.zeros((1, 2, 250), dtype=torch.int32, device="cuda")
    pk, pv = (torch.zeros((1, 500, 128), dtype=torch.int16, device="cuda") for _ in range(2))
    for fault in (True, False):
        st = gpu_ops.status_word()
        try:
            if fault:
                sg.sg_testing_score_fault(withhold_unit=1, wait_limit_ms=10)
            sg.prefill(shp, q, k, k, imp, ws, gpu_ops.dev(ck), 250, sel, pk, pv, st)
            torch.cuda.synchronize()
        finally:
            sg.sg_testing_score_fault(-1, 0)
        assert gpu_ops.read_status(st) == ((1 << sg.SG_ERR_TIMEOUT) if fault else 0)
    want = oracle.score(q_h, k_h, cu)
    assert np.all(np.abs(imp.cpu().numpy() - want) <= 1e-4 * np.abs(want) + 1e-30)


def test_expired_wait_leaves_no_earlier_rows():
    """The entries and packed rows of the parts that gave up are -1 and zero, not those of the buffers' previous prompt; the others are right."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(8)
    lens, budgets, Hkv, d = (2000, 500, 90), (200, 50, 90), 2, 64        # the last one keeps the whole prompt
    cu, ck = cu_of(lens), cu_of(budgets)
    T, K = int(cu[-1]), int(ck[-1])
    q_h, k_h, v_h = rand_bf16(rng, (1, 3, 16, 8, d)), rand_bf16(rng, (1, T, Hkv, d)), rand_bf16(rng, (1, T, Hkv, d))
    shp, st = gpu_ops.shape_of(1, 8, Hkv, d, 16, cu), gpu_ops.status_word()
    assert sg.sg_testing_score_cluster(shp) > 0
    imp = torch.zeros((1, Hkv, T), device="cuda")
    sel = gpu_ops.Guarded((1, Hkv, K), torch.int32, 3)
    pk, pv = (gpu_ops.Guarded((1, K * Hkv, d), torch.int16, 77) for _ in range(2))
    try:
        sg.sg_testing_score_fault(withhold_unit=1, wait_limit_ms=10)
        sg.prefill(shp, gpu_ops.dev(q_h), gpu_ops.dev(k_h), gpu_ops.dev(v_h), imp, sg.alloc_workspace(sg.SG_OP_SCORE, shp), gpu_ops.dev(ck), K,
                   sel.view, pk.view, pv.view, st)
        torch.cuda.synchronize()
    finally:
        sg.sg_testing_score_fault(-1, 0)
    assert gpu_ops.read_status(st) == 1 << sg.SG_ERR_TIMEOUT
    want = oracle.select_topk(imp.cpu().numpy(), cu, ck)
    want_k, want_v = oracle.pack_kv(k_h, v_h, cu, want, ck)
    want[0, 1] = -1
    for b, n in enumerate(budgets):
        lost = slice(int(ck[b]) * Hkv + n, int(ck[b]) * Hkv + 2 * n)      # KV head 1
        want_k[0, lost], want_v[0, lost] = 0, 0
    assert np.array_equal(sel.numpy(), want) and np.array_equal(pk.numpy(), want_k) and np.array_equal(pv.numpy(), want_v)


def test_calls_right_behind_one_that_gave_up():
    """What the CTAs of a part have sent one another has landed when the part ends, also where one of them did not send: calls queued
    directly behind, whose CTAs take over the shared memory, are right."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(9)
    cu, ck = cu_of((2000,)), cu_of((200,))
    q, k = gpu_ops.dev(rand_bf16(rng, (1, 1, 16, 32, 64))), gpu_ops.dev(rand_bf16(rng, (1, 2000, 8, 64)))
    shp = gpu_ops.shape_of(1, 32, 8, 64, 16, cu)
    assert sg.sg_testing_score_cluster(shp) > 1
    ws, d_ck = sg.alloc_workspace(sg.SG_OP_SCORE, shp), gpu_ops.dev(ck)

    def call():
        out = [torch.zeros((1, 8, 2000), device="cuda"), torch.zeros((1, 8, 200), dtype=torch.int32, device="cuda"),
               torch.zeros((1, 1600, 64), dtype=torch.int16, device="cuda"), torch.zeros((1, 1600, 64), dtype=torch.int16, device="cuda")]
        st = gpu_ops.status_word()
        sg.prefill(shp, q, k, k, out[0], ws, d_ck, 200, out[1], out[2], out[3], st)
        return out, st

    want, st = call()
    assert gpu_ops.read_status(st) == 0
    for unit in (0, 3, 7, 3):
        try:
            sg.sg_testing_score_fault(withhold_unit=unit, wait_limit_ms=2)
            bad, bad_st = call()
            sg.sg_testing_score_fault(-1, 0)
            after = [call() for _ in range(3)]
        finally:
            sg.sg_testing_score_fault(-1, 0)
        assert gpu_ops.read_status(bad_st) == 1 << sg.SG_ERR_TIMEOUT
        assert bool((bad[1][0, unit] == -1).all()) and not bad[2][0, 200 * unit:200 * unit + 200].any()
        for got, st in after:
            assert gpu_ops.read_status(st) == 0 and all(torch.equal(x, y) for x, y in zip(got, want))


@pytest.mark.parametrize("max_seqlen", [300, 2999, 3000])
def test_single_sequence_above_what_max_seqlen_promised(max_seqlen):
    """As the calls one by one: flagged, no entries, zero rows, where the selection chosen from max_seqlen cannot hold the row."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(10)
    cu, ck = cu_of((3000,)), cu_of((300,))
    q, k = gpu_ops.dev(rand_bf16(rng, (1, 1, 16, 8, 64))), gpu_ops.dev(rand_bf16(rng, (1, 3000, 2, 64)))
    shp, d_ck = gpu_ops.shape_of(1, 8, 2, 64, 16, cu), gpu_ops.dev(ck)
    shp.max_seqlen = max_seqlen
    ws = sg.alloc_workspace(sg.SG_OP_SCORE, shp)
    results = []
    for together in (True, False):
        imp, st = torch.zeros((1, 2, 3000), device="cuda"), gpu_ops.status_word()
        sel = torch.zeros((1, 2, 300), dtype=torch.int32, device="cuda")
        pk, pv = (torch.ones((1, 600, 64), dtype=torch.int16, device="cuda") for _ in range(2))
        if together:
            sg.prefill(shp, q, k, k, imp, ws, d_ck, 300, sel, pk, pv, st)
        else:
            sg.sg_score(shp, q, k, imp, ws, st)
            sg.sg_select_topk(shp, imp, d_ck, 300, sel, None, st)
            sg.sg_pack_kv(shp, k, k, sel, d_ck, 300, pk, pv, st)
        results.append((sel, pk, pv, gpu_ops.read_status(st)))
    for x, y in zip(results[0][:3], results[1][:3]):
        assert torch.equal(x, y)
    flagged = (1 << sg.SG_ERR_INVALID) | (1 << sg.SG_ERR_INDEX)
    assert results[0][3] == results[1][3] == (flagged if max_seqlen == 300 else 0)
