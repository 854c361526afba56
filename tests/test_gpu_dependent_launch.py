"""GPU: ordering of calls that are launched programmatically dependent on one another.

`sg_sparse_decode_attn` lets the next kernel in the stream start while it runs and writes its output at its very end, so it
serves as the producer that a following call must wait for: a long list (few sequences, a million index entries each, all
within a few rows of the cache) keeps it running for several hundred microseconds on half of the SMs, and the
following call's kernels are placed beside it at once.
"""
import numpy as np
import pytest

from helpers import cu_of, rand_bf16

pytestmark = pytest.mark.gpu


class SlowProducer:
    """One attention call of `rows` sequences with `heads` heads: out bf16 [rows][heads][d], written after `entries` index
    entries per list have been attended."""

    def __init__(self, rows, heads, d, entries=1 << 20, tokens=64, seed=0):
        import torch
        import gpu_ops
        rng = np.random.default_rng(seed)
        cu = cu_of((tokens,) * rows)
        self.shape = gpu_ops.shape_of(1, heads, heads, d, 1, cu)
        self.q = gpu_ops.dev(rand_bf16(rng, (rows, heads, d)))
        self.k = gpu_ops.dev(rand_bf16(rng, (rows * tokens, heads, d)))
        self.v = gpu_ops.dev(rand_bf16(rng, (rows * tokens, heads, d)))
        self.nloc = rows * entries
        self.idx = torch.randint(0, tokens, (heads, self.nloc), dtype=torch.int32, device="cuda")
        self.cu_nloc = torch.arange(rows + 1, dtype=torch.int32, device="cuda") * entries
        self.cu_k = torch.zeros(rows + 1, dtype=torch.int32, device="cuda")
        self.out = torch.zeros((rows, heads, d), dtype=torch.int16, device="cuda")

    def __call__(self):
        import paper_2607_28150_b200.binding as sg
        sg.sg_sparse_decode_attn(self.shape, self.q, None, None, self.cu_k, 0, self.k, self.v, self.idx, self.cu_nloc, self.nloc, self.out)


@pytest.mark.parametrize("launches", [1, 2])
@pytest.mark.parametrize("late", ["keys", "queries"])
def test_score_waits_for_a_producer_that_lets_it_start_early(late, launches):
    """One sequence and few key tiles leave SMs free for both scoring kernels while the producer of the keys, or of the
    window queries, is still running: neither may read them before it has ended.  sg_score takes one kernel for such a shape,
    sg_score_static always two."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(21)
    heads, d, n = 2, 128, 4
    W = n if late == "queries" else 2
    make = SlowProducer(n, heads, d)
    T = 300 if late == "queries" else n
    k = gpu_ops.dev(rand_bf16(rng, (1, T, heads, d))) if late == "queries" else make.out.view(1, n, heads, d)
    q = make.out.view(1, 1, W, heads, d) if late == "queries" else gpu_ops.dev(rand_bf16(rng, (1, 1, W, heads, d)))
    shp = gpu_ops.shape_of(1, heads, heads, d, W, cu_of((T,)))
    ws = sg.alloc_workspace(sg.SG_OP_SCORE, shp)
    assert sg.sg_testing_score_cluster(shp) > 0

    def call(imp, st):
        if launches == 1:
            sg.sg_score(shp, q, k, imp, ws, st)
        else:
            sg.sg_score_static(shp, q, k, imp, st)

    def score():
        imp, st = torch.full((1, heads, T), -1.0, dtype=torch.float32, device="cuda"), gpu_ops.status_word()
        call(imp, st)
        return imp, st

    early, _ = score()                                    # on the zeros that the producer will overwrite
    torch.cuda.synchronize()
    for _ in range(3):
        make.out.zero_()
        imp, st = torch.full((1, heads, T), -1.0, dtype=torch.float32, device="cuda"), gpu_ops.status_word()
        torch.cuda.synchronize()
        make()
        call(imp, st)
        assert gpu_ops.read_status(st) == 0
        want, _ = score()                                 # again, when everything has been written
        assert torch.equal(imp, want) and not torch.allclose(want, early, rtol=1e-3)


@pytest.mark.parametrize("late", ["keys", "values", "queries"])
def test_prefill_waits_for_a_producer_that_lets_it_start_early(late):
    """The same for the kernel that also selects and packs."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(24)
    heads, d, n = 2, 128, 4
    make = SlowProducer(n, heads, d)
    T, W = (300, n) if late == "queries" else (n, 2)
    made = {"keys": make.out.view(1, n, heads, d), "values": make.out.view(1, n, heads, d), "queries": make.out.view(1, 1, n, heads, d)}[late]
    k, v = (made if late == name else gpu_ops.dev(rand_bf16(rng, (1, T, heads, d))) for name in ("keys", "values"))
    q = made if late == "queries" else gpu_ops.dev(rand_bf16(rng, (1, 1, W, heads, d)))
    K = T - 1
    shp, ck = gpu_ops.shape_of(1, heads, heads, d, W, cu_of((T,))), gpu_ops.dev(cu_of((K,)))
    ws = sg.alloc_workspace(sg.SG_OP_SCORE, shp)
    assert sg.sg_testing_score_cluster(shp) > 0

    def prefill():
        out = [torch.full((1, heads, T), -1.0, device="cuda"), torch.full((1, heads, K), -9, dtype=torch.int32, device="cuda")]
        out += [torch.full((1, K * heads, d), 5, dtype=torch.int16, device="cuda") for _ in range(2)]
        st = gpu_ops.status_word()
        torch.cuda.synchronize()
        return out, st, lambda: sg.prefill(shp, q, k, v, out[0], ws, ck, K, out[1], out[2], out[3], st)

    def finished():
        out, st, run = prefill()
        run()
        assert gpu_ops.read_status(st) == 0
        return out

    make.out.zero_()
    early = finished()                                     # on the zeros that the producer will overwrite
    for _ in range(3):
        make.out.zero_()
        got, st, run = prefill()
        make()
        run()
        assert gpu_ops.read_status(st) == 0
        want = finished()                                  # again, when everything has been written
        assert all(torch.equal(x, y) for x, y in zip(got, want))
        assert not all(torch.equal(x, y) for x, y in zip(want, early))


def test_pass_2_of_scoring_waits_as_long_as_pass_1_takes():
    """More (layer, sequence, KV head) parts than the fixed scratch of sg_score_static holds at full width: pass 1 runs for
    several milliseconds on a few CTAs while those of pass 2 are set up beside it.  Their bounded waits, shortened to one
    millisecond, count from the end of pass 1."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    B, n, heads, G, d, W = 252, 3000, 8, 8, 64, 64        # 2016 parts of 512 rows: records of 4 KB, 8 MB hold 32 more
    cu = cu_of((n,) * B)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    q = torch.randn((1, B, W, heads * G, d), generator=gen, device="cuda", dtype=torch.bfloat16)
    k = torch.randn((1, B * n, heads, d), generator=gen, device="cuda", dtype=torch.bfloat16)
    shp = gpu_ops.shape_of(1, heads * G, heads, d, W, cu)
    imp = torch.full((1, heads, B * n), -1.0, dtype=torch.float32, device="cuda")
    want, st, st2 = torch.empty_like(imp), gpu_ops.status_word(), gpu_ops.status_word()
    sg.sg_score(shp, q, k, want, sg.alloc_workspace(sg.SG_OP_SCORE, shp), st2)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    try:
        sg.sg_testing_score_fault(-1, 1)
        a.record()
        sg.sg_score_static(shp, q, k, imp, st)
        b.record()
        torch.cuda.synchronize()
    finally:
        sg.sg_testing_score_fault(-1, 0)
    assert a.elapsed_time(b) > 4.0                        # else the limit would not have been exceeded
    assert gpu_ops.read_status(st) == 0 and gpu_ops.read_status(st2) == 0
    # the same sums, cut at other places: a few roundings of fp32 partial sums
    assert torch.all((imp - want).abs() <= 1e-5 * want.abs() + 1e-30)


@pytest.mark.parametrize("late", ["packed rows", "queries"])
def test_two_lane_attention_waits_for_a_producer_that_lets_it_start_early(late):
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(22)
    heads, d, n = 2, 128, 4
    make = SlowProducer(n, heads, d)                       # out [n][heads][d]: n packed rows of each of the heads, or n sequences' queries
    B = n if late == "queries" else 1
    rows = make.out if late == "packed rows" else gpu_ops.dev(rand_bf16(rng, (B * 3, heads, d)))
    q = make.out if late == "queries" else gpu_ops.dev(rand_bf16(rng, (B, heads, d)))
    per = 3 if late == "queries" else n                    # packed rows per list
    packed = rows.view(B * per * heads, d)
    cu_cap = torch.arange(B + 1, dtype=torch.int32, device="cuda") * per
    shp = gpu_ops.shape_of(1, heads, heads, d, 1, cu_of((8,) * B))
    count = torch.full((B, heads), per, dtype=torch.int32, device="cuda")
    none, skip = torch.zeros(B + 1, dtype=torch.int32, device="cuda"), torch.zeros((B, heads), dtype=torch.int32, device="cuda")
    out, want = (torch.zeros((B, heads, d), dtype=torch.int16, device="cuda") for _ in range(2))

    def attend(o):
        sg.sg_sparse_decode_attn_counted(shp, q, packed, packed, cu_cap, B * per, count, None, None, None, none, 0, o, local_skip=skip)

    attend(out)
    torch.cuda.synchronize()
    early = out.clone()                                    # on the zeros that the producer will overwrite
    for _ in range(3):
        make.out.zero_()
        torch.cuda.synchronize()
        make()
        attend(out)
        torch.cuda.synchronize()
        attend(want)                                       # again, when everything has been written
        torch.cuda.synchronize()
        assert torch.equal(out, want) and not torch.equal(want, early)


def test_attention_directly_behind_packing_reads_the_packed_rows():
    """The rows that sg_pack_kv has just written are inputs of the next call, whose kernel reads them without waiting."""
    import torch
    import gpu_ops
    import paper_2607_28150_b200.binding as sg
    rng = np.random.default_rng(23)
    Hq, Hkv, d, N, K = 32, 8, 128, 4096, 800
    cu, ck = gpu_ops.dev(cu_of((N,))), gpu_ops.dev(cu_of((K,)))
    shp = gpu_ops.shape_of(1, Hq, Hkv, d, 1, cu_of((N,)))
    caches = [tuple(gpu_ops.dev(rand_bf16(rng, (1, N, Hkv, d))) for _ in range(2)) for _ in range(2)]
    sel = torch.stack([torch.randperm(N, device="cuda")[:K].sort().values for _ in range(Hkv)]).int()[None].contiguous()
    q = gpu_ops.dev(rand_bf16(rng, (1, Hq, d)))
    none = torch.zeros(2, dtype=torch.int32, device="cuda")
    pk, pv = (torch.zeros((1, K * Hkv, d), dtype=torch.int16, device="cuda") for _ in range(2))
    outs = torch.zeros((402, 1, Hq, d), dtype=torch.int16, device="cuda")
    for i in range(402):
        if i < 2:
            torch.cuda.synchronize()
        sg.sg_pack_kv(shp, *caches[i % 2], sel, ck, K, pk, pv)
        if i < 2:
            torch.cuda.synchronize()                       # the first two are the references
        sg.sg_sparse_decode_attn(shp, q, pk[0], pv[0], ck, K, None, None, None, none, 0, outs[i])
    torch.cuda.synchronize()
    assert not torch.equal(outs[0], outs[1])
    assert torch.equal(outs[2::2], outs[0].expand(200, 1, Hq, d)) and torch.equal(outs[3::2], outs[1].expand(200, 1, Hq, d))
