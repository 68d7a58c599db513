"""Edge sizes of individual kernels: remainders of their tiles, the smallest and the largest of a dispatch rule's
range, each against the oracle or an exact reordering of the input."""
import numpy as np
import pytest

from oracle import feplb_oracle as O
from paper_2604_19654_b200 import build as B
from paper_2604_19654_b200 import feplb as F
from paper_2604_19654_b200 import workloads as W

from gpu_utils import DeviceCase
from test_gpu_backward import _close, _run_backward
from test_gpu_parity import _check_forward, _ffn_case, _random_workload_wm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


@pytest.mark.parametrize("E,d,f", [(1, 128, 64), (3, 384, 64), (2, 128, 320), (5, 640, 192)])
def test_transpose_partial_tiles(E, d, f):
    """128 x 128 tiles with a remainder of 64 in either direction, and matrices smaller than one tile."""
    import torch
    case = DeviceCase(W.get_workload("cfg1").with_(E=E, R=1, K=1, T=8, d=d, f=f))
    w1t, w3t = (torch.zeros(E, d, f, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    w2t = torch.zeros(E, f, d, dtype=torch.bfloat16, device="cuda")
    case.ctx.transpose_weights(case.d_w1, case.d_w3, case.d_w2, w1t, w3t, w2t)
    for got, src in ((w1t, case.w1), (w3t, case.w3), (w2t, case.w2)):
        assert np.array_equal(F.bf16_bits(got), src.transpose(0, 2, 1))
    case.close()


@pytest.mark.parametrize("form", [F.FORM_SINGLE, F.FORM_PAIR])
@pytest.mark.parametrize("E,d,f,rows", [
    (2, 128, 64, [1, 130]),            # one narrow N tile in both passes
    (3, 384, 192, [257, 0, 31]),       # a full and a narrow N tile in both passes
    (2, 640, 320, [128, 129]),         # two full and one narrow
    (2, 1920, 704, [90, 300]),         # many of each, the ring wraps
])
def test_expert_ffn_narrow_last_n_tile(E, d, f, rows, form):
    """Widths that are not multiples of the N tile: f % 128 = 64 (pass 1) and d % 256 = 128 (pass 2)."""
    _ffn_case(E, d, f, rows, form=form)


@pytest.mark.parametrize("T,K,E,R,A", [
    (1, 1, 2, 1, 1),              # one slot
    (13, 7, 24, 3, 128),          # padding rows written by CTAs without rows of their own
    (1024, 1, 8, 2, 1),           # one chunk of 32 slots per warp, full
    (1025, 1, 256, 4, 1),         # two chunks; the most experts
    (2731, 3, 16, 2, 128),        # 8193 slots: the three-launch front
    (2730, 3, 16, 2, 128),        # 8190: the last one-launch front
    (300, 32, 64, 4, 1),          # largest top-k, 9600 slots
    (250, 32, 64, 4, 1),          # ... and 8000
    (100, 2, 257, 1, 1),          # more experts than the one-launch front takes
])
def test_forward_front_range(T, K, E, R, A):
    """Routing and gather of small batches in one launch, and the sizes next to its range."""
    w = W.get_workload("cfg1").with_(T=T, K=K, E=E, R=R, d=128, f=64, tau=1, max_num_dyn=2)
    case = DeviceCase(w, row_align=A)
    _check_forward(case, sample=None if T < 300 else 100)
    case.close()


def test_forward_front_skips_ids_out_of_range():
    """A slot with an expert id outside [0, E) gets row -1 and contributes nothing; the rest is routed as without it."""
    import torch
    w = W.get_workload("cfg1").with_(T=70, d=128, f=64)
    case = DeviceCase(w)
    ids = case.ids.copy()
    ids[3, 0], ids[69, 1] = w.E, -5
    case.ctx.moe_forward(case.d_x, torch.from_numpy(ids).cuda(), case.d_gates, case.d_w1, case.d_w3, case.d_w2, case.buf)
    with pytest.raises(F.FeplbError) as ei:
        case.ctx.check_status()
    assert ei.value.code == F.E_RANGE
    flat = ids.ravel()
    valid = (flat >= 0) & (flat < w.E)
    rows = np.full(flat.size, -1)
    rows[np.flatnonzero(valid)[np.argsort(flat[valid], kind="stable")]] = np.arange(valid.sum())
    assert np.array_equal(case.buf.slot_to_row.cpu().numpy().ravel(), rows)
    assert np.array_equal(case.buf.counts.cpu().numpy(), np.bincount(flat[valid], minlength=w.E))
    assert np.all(case.buf.row_to_token.cpu().numpy()[valid.sum():] == -1)
    case.close()


def test_forward_orders_agree():
    """The order without a wait for the plan and the two orders that run the planner's table: the same integers and,
    row for row, the same products."""
    w = W.get_workload("cfg2").with_(T=300, d=256, f=128)
    case = DeviceCase(w)
    got = []
    for merged in (-1, 1, 0):
        case.ctx.set_launch_merging(merged)
        p, _ = _check_forward(case)
        got.append((p.moves, F.bf16_bits(case.buf.out).copy()))
    assert got[0][0] == got[1][0] == got[2][0] and len(got[0][0]) > 0
    assert np.array_equal(got[0][1], got[1][1]) and np.array_equal(got[0][1], got[2][1])
    case.close()


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 6, 7, 8, 9, 17])
def test_combine_every_batch_size(K):
    """Top-k around the row batches of the combine (2, 4, 6, 8 rows, then several batches of 8), a ragged last slice."""
    import torch
    T, d = 77, 640
    rng = np.random.default_rng(K)
    ctx = F.Context(F.make_config(T, K, 32, 1, d, 64))
    y = W.f32_to_bf16_bits(rng.standard_normal((T * K, d)).astype(np.float32))
    s2r = rng.permutation(T * K).astype(np.int32).reshape(T, K)
    gates = rng.random((T, K)).astype(np.float32)
    out = torch.zeros(T, d, dtype=torch.bfloat16, device="cuda")
    ctx.combine(F.bf16_tensor(y), torch.from_numpy(s2r).cuda(), torch.from_numpy(gates).cuda(), out)
    ref = O.combine(W.bf16_bits_to_f64(y), s2r, gates)
    mag = O.combine(np.abs(W.bf16_bits_to_f64(y)), s2r, gates)
    got = W.bf16_bits_to_f64(F.bf16_bits(out))
    # one bf16 rounding (2^-9 relative) and K fp32 additions (K * 2^-24 of the sum of magnitudes)
    assert np.all(np.abs(got - ref) <= 2.0 ** -8 * np.abs(ref) + 2.0 ** -19 * mag)
    ctx.close()


def test_expert_ffn_few_rows():
    """Groups around the 32 rows below which a tile loads a smaller box of A."""
    _ffn_case(6, 256, 128, [31, 32, 33, 1, 160, 161], form=F.FORM_SINGLE)      # 160 = 128 + 32, 161 = 128 + 33


@pytest.mark.parametrize("pair", [0, 3])
@pytest.mark.parametrize("d,f", [(640, 192), (384, 320), (1152, 704)])
def test_backward_overhanging_n_tile(d, f, pair):
    """Widths whose last 256-column tile of the backward GEMMs overhangs (192, 640, 704, 1152), and ones that keep
    128-column tiles (320, 384)."""
    w = W.get_workload("cfg2").with_(T=150, E=6, R=2, K=3, d=d, f=f, dyn=2, max_num_dyn=2, tau=8)
    case, bwd, dw, ref, _, _ = _run_backward(w, pair=pair)
    for got, want, what in zip((*dw, bwd.d_gates), (ref[2], ref[3], ref[4], ref[1]), ("dw1", "dw3", "dw2", "dgates")):
        _close(got.cpu().numpy().astype(np.float64)[: len(want)], want, what)
    _close(W.bf16_bits_to_f64(F.bf16_bits(bwd.d_x)), ref[0], "dx")
    case.close()


@pytest.mark.parametrize("T,K,E,R", [(1, 1, 2, 1), (700, 3, 48, 3), (4097, 4, 60, 5), (1500, 8, 1024, 16), (20000, 2, 8, 2)])
def test_route_hist_and_dispatch_repeat(T, K, E, R):
    """The histogram's accumulators are left zero (the second call counts other ids from scratch); dispatch from one CTA
    to many, few and many experts per scanning thread."""
    import torch
    w = W.get_workload("cfg1").with_(T=T, K=K, E=E, R=R, d=128, f=64)
    cfg = F.config_from_workload(w)
    ctx, buf = F.Context(cfg), F.Buffers(cfg)
    x = W.gen_activations(w, 0)
    for seed in (1, 2):
        ids = np.random.default_rng(seed).integers(0, E, size=(T, K)).astype(np.int32)
        d_ids = torch.from_numpy(ids).cuda()
        ctx.route_hist(d_ids, buf.counts, buf.rank_load)
        ctx.dispatch(F.bf16_tensor(x), d_ids, buf.counts, buf.x_perm, buf.slot_to_row, buf.row_to_token)
        ctx.check_status()
        counts, load = O.route_hist(ids, E, R)
        assert np.array_equal(buf.counts.cpu().numpy(), counts) and np.array_equal(buf.rank_load.cpu().numpy(), load)
        s2r, r2t, _, n = O.permute(ids, E, 1)
        assert np.array_equal(buf.slot_to_row.cpu().numpy(), s2r) and np.array_equal(buf.row_to_token.cpu().numpy()[:n], r2t)
        assert np.array_equal(F.bf16_bits(buf.x_perm)[:n], O.gather_rows(x, r2t))
    ctx.close()


def test_route_topk_signed_zeros_and_extremes():
    """-0 and +0 tie (lower id first); largest, smallest and subnormal magnitudes keep their order."""
    import torch
    row = np.array([0.0, -0.0, 3.4e38, -3.4e38, 1e-42, -1e-42, -0.0, 0.0], np.float32)
    logits = np.stack([row, row[::-1], np.roll(row, 3)])
    ctx = F.Context(F.make_config(3, 8, 8, 1, 128, 64))
    ids = torch.zeros(3, 8, dtype=torch.int32, device="cuda")
    gates = torch.zeros(3, 8, device="cuda")
    ctx.route_topk(torch.from_numpy(logits.copy()).cuda(), ids, gates)
    assert np.array_equal(ids.cpu().numpy(), O.route_topk(logits, 8)[0])
    ctx.close()


@pytest.mark.parametrize("T,K,E,d,f,A", [
    (4096, 2, 8, 1024, 64, 1),        # four ranges of 1024 tokens
    (5000, 3, 16, 1024, 64, 128),     # boundaries at multiples of 1024 tokens, padding rows, a ragged last range
    (3000, 6, 24, 1920, 192, 1),      # boundaries at multiples of 512 tokens
    (2049, 1, 8, 3072, 64, 1),        # ranges of 1024 and 1025 tokens
])
def test_host_forward_in_token_ranges(T, K, E, d, f, A):
    """Batches whose host copies dominate are processed in token ranges; every buffer and the plan equal those of the
    whole-batch path (device-resident forward) bit for bit."""
    import torch
    w = W.get_workload("cfg1").with_(T=T, K=K, E=E, d=d, f=f, tau=1)
    case = DeviceCase(w, row_align=A)
    p0 = case.ctx.moe_forward(case.d_x, case.d_ids, case.d_gates, case.d_w1, case.d_w3, case.d_w2, case.buf)
    case.ctx.check_status()
    n = int(p0.groups[-1][1] + p0.groups[-1][2])
    names = ("counts", "rank_load", "slot_to_row", "row_to_token", "x_perm", "y_perm", "out")
    want = {k: getattr(case.buf, k).clone() for k in names}
    live = case.buf.row_to_token[:n] >= 0
    for k in names:
        getattr(case.buf, k).fill_(3)
    host = [t.cpu().pin_memory() for t in (case.d_x, case.d_ids, case.d_gates)]
    dev = [torch.zeros_like(t) for t in (case.d_x, case.d_ids, case.d_gates)]
    out = torch.zeros(T, d, dtype=torch.bfloat16).pin_memory()
    before = case.ctx.launch_count()
    p1 = case.ctx.moe_forward_host(*host, *dev, case.d_w1, case.d_w3, case.d_w2, case.buf, out, want_plan=True)
    case.ctx.check_status()
    assert case.ctx.launch_count() - before >= 11                            # 3 + 4 per range: at least two ranges
    assert case.ctx.forward_path() & F.PATH_RANGES
    assert (p1.moves, p1.groups) == (p0.moves, p0.groups)
    assert torch.equal(out, want["out"].cpu())
    for k in names:
        got = getattr(case.buf, k)
        if k in ("x_perm", "y_perm"):
            assert torch.equal(got[:n][live], want[k][:n][live]), k
        else:
            assert torch.equal(got, want[k]), k
    case.close()


@pytest.mark.parametrize("form", [F.FORM_SINGLE, F.FORM_PAIR, F.FORM_WEIGHT_M])
@pytest.mark.parametrize("E,R,split", [(16, 4, 0), (16, 4, 1), (6, 3, 1), (64, 2, 0)])
def test_table_brought_over_by_the_gather(E, R, split, form):
    """The planner's table on the device before the GEMM (merged into the home table, whole experts and several pieces of
    one) and after its start (planner held back): the same integers and the same rows bit for bit."""
    w = W.get_workload("cfg4").with_(T=3000, K=4, E=E, R=R, d=256, f=128, dyn=3, max_num_dyn=4, tau=8, routing="dirichlet", alpha=0.3)
    case = DeviceCase(w, split=split, split_granule=64)
    case.ctx.set_gemm_form(form)
    case.ctx.set_launch_merging(1)
    case.ctx.set_timeline(True)

    def early():
        t = case.ctx.get_timeline()
        return t["dev_counts_to_static_end_us"] == t["dev_counts_to_static_start_us"]

    for attempt in range(100):                                   # a busy host can be late by itself
        for _ in range(4):                                       # the planner thread is up before the last one's counts are
            p0 = case.ctx.moe_forward(case.d_x, case.d_ids, case.d_gates, case.d_w1, case.d_w3, case.d_w2, case.buf)
        if early():
            break
    assert early()
    out = F.bf16_bits(case.buf.out).copy()
    case.ctx.set_planner_timing(planner_delay_us=2000)
    p1, _ = _check_forward(case, sample=200)
    assert not early()
    assert p0.groups == p1.groups and len(p0.moves) > 0
    assert np.array_equal(F.bf16_bits(case.buf.out), out)
    case.close()


@pytest.mark.parametrize("seed", range(6))
def test_merged_orders_of_random_shapes_beyond_the_one_launch_front(seed):
    """Random layers of more than 8192 slots, whole or split experts, the table brought over by the gather (or found later, on
    a busy host) and, with the planner held back, certainly late: equal to the oracle and to each other."""
    w, A, split, _ = _random_workload_wm(seed)
    w = w.with_(T=8192 // w.K + 1 + seed * 100)
    case = DeviceCase(w, mb=seed, row_align=A, split=1 - split, split_granule=128 if A == 128 else 16)
    case.ctx.set_gemm_form((F.FORM_SINGLE, F.FORM_PAIR, F.FORM_WEIGHT_M)[seed % 3])
    case.ctx.set_launch_merging(1)
    p0, _ = _check_forward(case, sample=60)
    out = F.bf16_bits(case.buf.out).copy()
    case.ctx.set_planner_timing(planner_delay_us=1000)
    p1, _ = _check_forward(case, sample=10)
    assert p0.groups == p1.groups and np.array_equal(F.bf16_bits(case.buf.out), out)
    case.close()


@pytest.mark.parametrize("T,merged,path", [
    (48, 1, F.PATH_MERGED | F.PATH_SINGLE),                     # T rows per expert on average: below 64
    (60, 0, F.PATH_WEIGHT_M | F.PATH_SINGLE),                   # four launches, static | dynamic
    (700, 0, F.PATH_WEIGHT_M),
    (800, 0, F.PATH_WEIGHT_M | F.PATH_PAIR),                    # above 768; the one dynamic expert of a rank has more than 512 rows
    (60, -1, F.PATH_HOME_TABLE | F.PATH_SINGLE),
    (700, -1, F.PATH_HOME_TABLE | F.PATH_WEIGHT_M),
])
def test_form_rule_of_large_weights(T, merged, path):
    """Shapes from which the weights-on-M form is chosen (3 Mi elements per matrix): below, inside and above its range of
    rows per expert, in every launch order."""
    w = W.get_workload("cfg2").with_(T=T, E=2, R=2, K=2, d=2048, f=1536, dyn=1, max_num_dyn=1, tau=1)
    case = DeviceCase(w)
    assert case.ctx.forward_path() == 0
    case.ctx.set_launch_merging(merged)
    _check_forward(case, sample=40)
    assert case.ctx.forward_path() == path | F.PATH_SMALL_FRONT
    case.close()


@pytest.mark.parametrize("T,K,E,d,f,path", [
    (1024, 2, 16, 256, 128, F.PATH_HOME_TABLE | F.PATH_SMALL_FRONT | F.PATH_SINGLE),      # 128 rows per expert, a short FFN
    (2048, 2, 16, 256, 128, F.PATH_HOME_TABLE | F.PATH_SMALL_FRONT | F.PATH_PAIR),        # 256 rows per expert: two-CTA tiles
    (2047, 1, 16, 4096, 2048, F.PATH_HOME_TABLE | F.PATH_SMALL_FRONT | F.PATH_WEIGHT_M),  # below 128 rows per expert
    (2048, 1, 16, 4096, 2048, F.PATH_MERGED | F.PATH_SMALL_FRONT | F.PATH_WEIGHT_M),      # 128, and an FFN of 230 us
    (6144, 1, 8, 4096, 2048, F.PATH_SMALL_FRONT | F.PATH_WEIGHT_M | F.PATH_PAIR),         # 768: four launches
])
def test_order_rule(T, K, E, d, f, path):
    """The launch order on both sides of its lines."""
    import torch
    ctx, buf = (c(F.make_config(T, K, E, 2, d, f, dyn=1, tau=1)) for c in (F.Context, F.Buffers))
    rng = torch.Generator(device="cuda").manual_seed(1)
    z = lambda *s: torch.zeros(*s, dtype=torch.bfloat16, device="cuda")       # noqa: E731
    ids = torch.rand(T, E, generator=rng, device="cuda").topk(K, dim=1)[1].int()
    w = z(E, f, d), z(E, f, d), z(E, d, f)
    ctx.moe_forward(z(T, d), ids, torch.ones(T, K, device="cuda"), *w, buf)
    ctx.check_status()
    assert ctx.forward_path() == path
    groups = torch.zeros(E, 5, dtype=torch.int32, device="cuda")
    ctx.home_groups(buf.counts, None, groups)
    for form in (F.FORM_SINGLE, F.FORM_PAIR):
        ctx.set_gemm_form(form)
        ctx.expert_ffn(buf.x_perm, *w, groups, E, buf.h_scratch, buf.y_perm)       # not a forward
    ctx.check_status()
    assert ctx.forward_path() == path
    ctx.close()


@pytest.mark.parametrize("A", [1, 128])
@pytest.mark.parametrize("T", [300, 2730, 2731])
def test_dispatch_takes_the_segments_from_the_counts(T, A):
    """Counts that disagree with the ids: one rule on both sides of the one-launch front's range (8190 and 8193 slots).  The
    caller's counts give the segments, clamped to the buffer; a slot whose row would lie behind it gets -1."""
    import torch
    K, E = 3, 16
    cfg = F.make_config(T, K, E, 2, 128, 64, row_align=A)
    ctx, buf, cap = F.Context(cfg), F.Buffers(cfg), F.s_pad(cfg)
    ids = np.random.default_rng(T).integers(0, E, size=(T, K)).astype(np.int32)
    flat = ids.ravel()
    true = np.bincount(flat, minlength=E)
    rank = np.empty(flat.size, np.int64)
    for e in range(E):
        rank[flat == e] = np.arange(true[e])
    x, d_ids = torch.zeros(T, 128, dtype=torch.bfloat16, device="cuda"), torch.from_numpy(ids).cuda()
    for delta in ({3: 1}, {15: 5}, {0: -2}, {2: -10 ** 6}, {1: 2 ** 30, 2: 2 ** 30, 3: 2 ** 30}, {5: 1000, 9: -7}):
        counts = true.copy()
        for e, dv in delta.items():
            counts[e] = dv if abs(dv) >= 10 ** 6 else counts[e] + dv
        seg = np.maximum(counts, 0)
        off = np.concatenate([[0], np.cumsum((seg + A - 1) // A * A)[:-1]])
        rows = np.minimum(off, cap)[flat] + rank
        rows[rows >= cap] = -1
        ctx.dispatch(x, d_ids, torch.from_numpy(counts.astype(np.int32)).cuda(), buf.x_perm, buf.slot_to_row, buf.row_to_token)
        with pytest.raises(F.FeplbError) as ei:
            ctx.check_status()
        assert ei.value.code == F.E_DEVICE
        assert np.array_equal(buf.slot_to_row.cpu().numpy().ravel(), rows), delta
    ctx.close()


def test_host_times_of_a_forward_in_token_ranges():
    """feplb_get_timeline after a host-buffer forward in token ranges: this call's host times, none left by another."""
    import torch
    w = W.get_workload("cfg1").with_(T=4096, K=2, E=8, d=1024, f=64, tau=1)
    case = DeviceCase(w)
    case.ctx.moe_forward(case.d_x, case.d_ids, case.d_gates, case.d_w1, case.d_w3, case.d_w2, case.buf)
    host = [t.cpu().pin_memory() for t in (case.d_x, case.d_ids, case.d_gates)]
    out = torch.zeros(w.T, w.d, dtype=torch.bfloat16).pin_memory()
    torch.cuda.synchronize()
    before = case.ctx.launch_count()
    case.ctx.moe_forward_host(*host, case.d_x, case.d_ids, case.d_gates, case.d_w1, case.d_w3, case.d_w2, case.buf, out)
    ranges = (case.ctx.launch_count() - before - 3) // 4                     # 3 launches for the batch, 4 per range
    t = case.ctx.get_timeline()
    assert ranges > 1 and t["ffn_launches"] == 2 * ranges
    assert 0 < t["host_enqueue_static_done_us"] <= t["host_counts_ready_us"] <= t["host_plan_done_us"]
    assert t["host_plan_done_us"] <= t["host_upload_enqueued_us"] <= t["host_join_us"] <= t["host_return_us"]
    case.close()


@pytest.mark.parametrize("form", [F.FORM_PAIR, F.FORM_WEIGHT_M])
def test_pass_times_do_not_overlap(form):
    """The two passes' own times fit into the interval between the events around their launches: a CTA of pass 2 that is
    resident but still waits for pass 1 does not count."""
    w = W.get_workload("cfg2")
    case = DeviceCase(w)
    case.ctx.set_gemm_form(form)
    case.ctx.set_launch_merging(1)
    case.ctx.set_timeline(True)
    slack = []
    for _ in range(15):
        case.ctx.moe_forward(case.d_x, case.d_ids, case.d_gates, case.d_w1, case.d_w3, case.d_w2, case.buf, want_plan=False)
        t = case.ctx.get_timeline()
        slack.append(t["dev_static_ffn_us"] - t["dev_ffn_pass1_us"] - t["dev_ffn_pass2_us"])
    case.ctx.check_status()
    assert np.median(slack) > 0, slack
    case.close()


def test_late_planner_does_not_hold_the_gather_up():
    """The CTA that waits for the planner's table gives up when the rows are copied, after 8 us at least (here the copies take
    about 3): with the planner held back, the interval between the events around the gather is about 17 us -- the 8,
    one more look across PCIe and the launch -- against 11 with the table on time and 23 with a fixed wait of 15 us."""
    w = W.get_workload("cfg1").with_(T=3000, K=4, E=16, R=4, d=256, f=128, tau=1)
    case = DeviceCase(w)
    case.ctx.set_launch_merging(1)
    case.ctx.set_planner_timing(planner_delay_us=200)
    case.ctx.set_timeline(True)
    gather = []
    for _ in range(15):
        case.ctx.moe_forward(case.d_x, case.d_ids, case.d_gates, case.d_w1, case.d_w3, case.d_w2, case.buf, want_plan=False)
        gather.append(case.ctx.get_timeline()["dev_dispatch_us"])
    case.ctx.check_status()
    assert np.median(gather) < 20, gather
    case.close()
