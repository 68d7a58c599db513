"""The forms of the expert FFN at the edges of their tiles, against the oracle: segments around the row counts at which a
tile changes its shape, weights in either order in memory, widths that leave the last weight block or K block
half empty."""
import numpy as np
import pytest
import torch

from oracle import feplb_oracle as O
from paper_2604_19654_b200 import build as B
from paper_2604_19654_b200 import feplb as F
from paper_2604_19654_b200 import workloads as W

from gpu_utils import DeviceCase, assert_close, upload_groups
from test_gpu_parity import _check_forward

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def _run(rows, d, f, form, w3_first=False, same=False, preact=False, detail=None):
    """One forward whose expert e has rows[e] rows (top-1), through the variants `detail` (None: any); returns the context's
    launch path."""
    E, T = len(rows), sum(rows)
    w = W.get_workload("cfg1").with_(T=T, E=E, K=1, R=1, d=d, f=f, dyn=0)
    ids = np.repeat(np.arange(E, dtype=np.int32), rows)[np.random.default_rng(T).permutation(T)].reshape(T, 1)
    gates = np.ones((T, 1), np.float32)
    x = W.gen_activations(w, 0)
    w1, w3, w2 = W.gen_weights(w)
    pair = torch.empty(2, E, f, d, dtype=torch.bfloat16, device="cuda")          # one allocation: the order is known
    d_w1, d_w3 = (pair[1], pair[0]) if w3_first else (pair[0], pair[0] if same else pair[1])
    d_w1.copy_(F.bf16_tensor(w1))
    if same:
        w3 = w1
    else:
        d_w3.copy_(F.bf16_tensor(w3))
    cfg = F.config_from_workload(w)
    ctx, buf = F.Context(cfg), F.Buffers(cfg)
    if form is not None:
        ctx.set_gemm_form(form)
    ab = torch.full((T, 2 * f), 7.0, dtype=torch.bfloat16, device="cuda")
    if preact:
        ctx.set_preact_buffer(ab)
    buf.h_scratch.fill_(float("nan"))
    buf.y_perm.fill_(float("nan"))
    ctx.moe_forward(F.bf16_tensor(x), torch.from_numpy(ids).cuda(), torch.from_numpy(gates).cuda(), d_w1, d_w3, F.bf16_tensor(w2), buf)
    ctx.check_status()
    assert_close(W.bf16_bits_to_f64(F.bf16_bits(buf.out)), O.moe_layer(x, ids, gates, w1, w3, w2, E), f"{rows} {d} {f} {form}")
    if preact:
        x64, order = W.bf16_bits_to_f64(x), np.argsort(ids[:, 0], kind="stable")
        for e in np.flatnonzero(rows):
            xe, got = x64[order][ids[order, 0] == e], W.bf16_bits_to_f64(F.bf16_bits(ab))[:T][ids[order, 0] == e]
            assert_close(got[:, :f], xe @ W.bf16_bits_to_f64(w1[e]).T, "a")
            assert_close(got[:, f:], xe @ W.bf16_bits_to_f64(w3[e]).T, "b")
    path = ctx.forward_path()
    assert detail is None or ctx.forward_detail() == detail
    ctx.close()
    return path


def _zeros(T, K, E, d, f):
    """Context, buffers and inputs of a layer of zeros, tokens spread evenly at random: for what a forward does, not what it computes."""
    z = lambda *s: torch.zeros(*s, dtype=torch.bfloat16, device="cuda")       # noqa: E731
    cfg = F.make_config(T, K, E, 1, d, f, dyn=1, tau=1)
    ids = torch.rand(T, E, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda").topk(K, dim=1)[1].int()
    return F.Context(cfg), F.Buffers(cfg), (z(T, d), ids, torch.ones(T, K, device="cuda")), (z(E, f, d), z(E, f, d), z(E, d, f))


@pytest.mark.parametrize("w3_first", [False, True])
@pytest.mark.parametrize("d,f", [(256, 128), (384, 320), (128, 64)])
def test_pair_form_tiles_of_128_and_256_rows(d, f, w3_first):
    """Segments around the multiples of 64 and 128 rows in 256-row tiles; f = 320: N tiles half empty."""
    path = _run([1, 32, 63, 64, 65, 96, 127, 128, 129, 255, 256, 257, 384, 385], d, f, F.FORM_PAIR, w3_first, detail=0)
    assert path & F.PATH_PAIR


@pytest.mark.parametrize("w3_first", [False, True])
@pytest.mark.parametrize("d,f,n_experts", [(384, 320, 25), (1152, 1856, 14)])
def test_deep_stages_and_tiles_of_128_rows(d, f, n_experts, w3_first):
    """Tiles of at most 128 rows go through the 128-row MMA, 64 rows per CTA; K blocks and N tiles half empty in either pass;
    saved pre-activations."""
    rows = [1, 32, 63, 64, 65, 96, 127, 128, 129, 255, 256, 257, 384, 385]
    rows += [0] * (n_experts - len(rows))
    assert _run(rows, d, f, F.FORM_PAIR, w3_first, preact=True, detail=F.DETAIL_DEEP_STAGES) & F.PATH_PAIR


@pytest.mark.parametrize("T,E,d,f,deep", [
    (1024, 16, 2048, 1024, 1), (1024, 16, 2048, 960, 0),          # 2 Mi elements
    (1600, 25, 1024, 512, 1), (1600, 24, 1024, 512, 0),           # 25 experts
    (6400, 25, 1024, 256, 0), (6400, 25, 128, 512, 0),            # a short pass
    (7424, 16, 1024, 512, 1), (7168, 16, 1024, 512, 0),           # 37 row blocks of 4 tiles: two waves of 74 clusters
    (24472, 8, 768, 832, 1), (24472, 8, 640, 832, 0),             # which a short first pass does without
])
def test_rule_of_deep_stages(T, E, d, f, deep):
    ctx, buf, args, w = _zeros(T, 1, E, d, f)
    ctx.set_gemm_form(F.FORM_PAIR)
    ctx.moe_forward(*args, *w, buf)
    assert ctx.forward_detail() == (F.DETAIL_DEEP_STAGES if deep else 0) and ctx.forward_path() & F.PATH_PAIR
    ctx.check_status()
    ctx.close()


@pytest.mark.parametrize("form", [F.FORM_PAIR, None])
def test_weights_in_one_buffer(form):
    """W1 and W3 the same tensor: no map covers both side by side, the launches go without."""
    _run([1, 40, 64, 65, 130], 256, 128, form, same=True)


@pytest.mark.parametrize("rows,fallback", [([1, 40, 64, 65, 130], F.PATH_SINGLE), ([300, 257, 256], F.PATH_PAIR)])
def test_weights_on_m_asked_for_with_weights_in_one_buffer(rows, fallback):
    forms = F.PATH_SINGLE | F.PATH_PAIR | F.PATH_WEIGHT_M
    assert _run(rows, 256, 128, F.FORM_WEIGHT_M) & forms == F.PATH_WEIGHT_M
    assert _run(rows, 256, 128, F.FORM_WEIGHT_M, same=True) & forms == fallback


@pytest.mark.parametrize("w3_first", [False, True])
def test_weights_on_m_units_of_any_width(w3_first):
    """d = 7.5 x 256, f = 13.5 x 128: the second CTA's half of the last weight block lies past the width, the last K block of
    pass 2 is half empty; segments around the multiples of 32 and 256 rows; saved pre-activations."""
    rows = [1, 31, 32, 33, 64, 65, 128, 129, 200, 255, 256, 257, 300]
    assert _run(rows, 1920, 1728, None, w3_first, preact=True) & F.PATH_WEIGHT_M


HALF_UNITS = W.get_workload("cfg2").with_(E=8, R=4, K=2, d=1920, f=1728, dyn=2, max_num_dyn=2, tau=1)   # 7.5 and 13.5 weight blocks


@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("T", [600, 4100])
def test_weights_on_m_late_table_at_half_units(T, split):
    """The planner's table taken up inside the launch where the last weight block is half empty, behind either front."""
    case = DeviceCase(HALF_UNITS.with_(T=T), mb=1, split=split)
    case.ctx.set_planner_timing(planner_delay_us=1000)
    p, _ = _check_forward(case, sample=60)
    assert len(p.moves) > 0 and any(g[4] for g in p.groups)
    assert case.ctx.forward_path() & (F.PATH_WEIGHT_M | F.PATH_MERGED) == F.PATH_WEIGHT_M | F.PATH_MERGED
    case.close()


def test_weights_on_m_receive_slots_at_half_units():
    """Migrated experts' weights from their receive slots, W3 in front of W1 at home: the rows of the relabelled experts, also from
    home weights of zeros."""
    w = HALF_UNITS.with_(T=600)
    weights = W.gen_weights(w)
    base = DeviceCase(w, mb=1, weights=weights)
    p0, _ = _check_forward(base, sample=60)
    case = DeviceCase(w, mb=1, weights=weights, phase2_copy=1)
    pair = torch.empty(2, *case.d_w1.shape, dtype=torch.bfloat16, device="cuda")
    pair[0], pair[1] = case.d_w3, case.d_w1
    case.d_w1, case.d_w3 = pair[1], pair[0]
    p1, _ = _check_forward(case, sample=60)
    assert p1.moves == p0.moves and len(p1.moves) > 0
    assert case.ctx.forward_path() == F.PATH_SMALL_FRONT | F.PATH_WEIGHT_M
    assert torch.equal(case.buf.out.view(torch.int16), base.buf.out.view(torch.int16))
    dst, first = p1.moves[0][2], {}
    for e, src, to, rows in p1.moves:                                  # move i takes the next slot of its destination
        first.setdefault(to, e)
    e = first[dst]
    _, row, rows, _, _ = next(g for g in p1.groups if g[0] == e and g[3] == dst)
    want = case.buf.y_perm[row:row + rows].clone()
    pair.zero_()
    case.buf.y_perm[row:row + rows] = 7.0
    groups = upload_groups([(e, row, rows, dst, 2 + dst * w.max_num_dyn)])
    case.ctx.expert_ffn(case.buf.x_perm, case.d_w1, case.d_w3, torch.zeros_like(case.d_w2), groups, 1, case.buf.h_scratch, case.buf.y_perm)
    case.ctx.check_status()
    assert torch.equal(case.buf.y_perm[row:row + rows].view(torch.int16), want.view(torch.int16))
    base.close()
    case.close()


@pytest.mark.parametrize("w3_first", [False, True])
@pytest.mark.parametrize("d,f,rows,units", [
    (256, 320, [1, 15, 16, 17, 31, 32, 33, 40], F.DETAIL_UNITS_32),          # one wave of units of 32 rows
    (1024, 1024, [1, 15, 16, 17, 33, 63, 64, 65] + [0] * 14, F.DETAIL_UNITS_64),
    (1920, 576, [1, 16, 31, 32, 33, 64, 65, 127, 128, 129], F.DETAIL_UNITS_128),      # K blocks half empty
])
def test_units_for_few_rows_per_expert(d, f, rows, units, w3_first):
    """Segments around the multiples of 16 rows and of a unit, in each size of the units that the rule picks; saved
    pre-activations."""
    assert _run(rows, d, f, None, w3_first, preact=True, detail=units) & F.PATH_SINGLE


@pytest.mark.parametrize("d,f,rows,units", [
    (2048, 1024, [33, 2] + [1] * 28 + [0] * 2, F.DETAIL_UNITS_32),           # 496 units in both passes
    (2048, 1024, [65, 64, 63] + [1] * 26 + [0] * 3, F.DETAIL_UNITS_64),      # 480
    (1024, 2048, [129, 128, 127] + [3] * 28 + [0], F.DETAIL_UNITS_128),      # 1024 and 256
])
def test_several_units_per_cta_for_few_rows(d, f, rows, units):
    """More than three units for each of 148 CTAs, and more K blocks than stages: the accumulators and the ring go round, and
    the weights loaded ahead of the first unit are followed by ordinary loads; saved pre-activations."""
    assert _run(rows, d, f, None, preact=True, detail=units) & F.PATH_SINGLE


@pytest.mark.parametrize("T,K,E,d,f,units", [
    (1, 8, 24, 6144, 1216, 0),                     # 152 units of long weights: a wave and four
    (1, 7, 24, 6144, 1216, F.DETAIL_UNITS_32),     # 133
    (5, 8, 64, 3584, 640, 0),                      # 31 experts of 10 blocks
    (10, 8, 64, 3584, 640, F.DETAIL_UNITS_32),     # 47
    (34, 3, 32, 4224, 320, F.DETAIL_UNITS_32),     # 31 of 5: 1.04 waves if the routing is even
    (30, 8, 128, 2048, 192, 0),
    (30, 8, 128, 1920, 192, F.DETAIL_UNITS_32),    # shorter units
    (96, 2, 96, 2048, 192, 0),                     # units of 64 rows
    (1280, 1, 128, 128, 768, 0),                   # 10 rows per expert of a narrow layer
    (1279, 1, 128, 128, 768, F.DETAIL_UNITS_64),
    (240, 1, 24, 128, 768, F.DETAIL_UNITS_64),     # two waves
])
def test_rule_of_few_rows_per_expert(T, K, E, d, f, units):
    """Single-CTA tiles of token rows where a second wave of units would be nearly empty, or a unit is its fixed costs."""
    ctx, buf, args, w = _zeros(T, K, E, d, f)
    ctx.moe_forward(*args, *w, buf)
    assert ctx.forward_detail() == units and ctx.forward_path() & F.PATH_SINGLE
    ctx.check_status()
    ctx.close()


@pytest.mark.parametrize("T,K,E,d,f,detail", [
    (32, 4, 32, 2048, 1024, F.DETAIL_UNITS_32),
    (16, 4, 16, 128, 64, F.DETAIL_UNITS_32),
    (2048, 1, 16, 2048, 1024, 0),                  # 128 rows per expert
])
def test_detail_of_the_last_forward(T, K, E, d, f, detail):
    """What a forward reports; asking for a form, or a call on a table of one's own, does not change it afterwards."""
    ctx, buf, args, w = _zeros(T, K, E, d, f)
    assert ctx.forward_detail() == 0
    ctx.moe_forward(*args, *w, buf)
    assert ctx.forward_detail() == detail
    ctx.set_gemm_form(F.FORM_SINGLE)
    groups = torch.zeros(E, 5, dtype=torch.int32, device="cuda")
    ctx.home_groups(buf.counts, None, groups)
    ctx.expert_ffn(buf.x_perm, *w, groups, E, buf.h_scratch, buf.y_perm)
    assert ctx.forward_detail() == detail
    ctx.moe_forward(*args, *w, buf)
    assert ctx.forward_detail() == 0
    ctx.check_status()
    ctx.close()


@pytest.mark.parametrize("d,f,rows,form", [
    (128, 64, [300, 200, 280], F.PATH_PAIR),              # 256 rows per expert and more: two-CTA tiles ...
    (128, 64, [300, 200, 364], F.PATH_SINGLE),            # ... and from 288 single-CTA tiles again for small weights
    (2048, 1536, [900, 641, 768], F.PATH_WEIGHT_M),       # weights on M up to 1280 rows per expert
    (2048, 1536, [1281, 1279, 1280], F.PATH_PAIR),
    (1024, 512, [300, 257, 280], F.PATH_PAIR),            # too few units of weights on M
])
def test_forms_of_larger_batches(d, f, rows, form):
    path = _run(rows, d, f, None)
    assert path & (F.PATH_SINGLE | F.PATH_PAIR | F.PATH_WEIGHT_M) == form


@pytest.mark.parametrize("rows,order", [
    ([191] * 8, F.PATH_MERGED),                # an FFN of more than 150 us behind the one-launch front: 192 rows per expert
    ([192] * 8, F.PATH_HOME_TABLE),
    ([640, 0, 1, 128, 300, 255, 200, 12], F.PATH_HOME_TABLE),
])
def test_order_behind_the_one_launch_front(rows, order):
    path = _run(rows, 4096, 4096, None)
    assert path & (F.PATH_MERGED | F.PATH_HOME_TABLE | F.PATH_SMALL_FRONT) == order | F.PATH_SMALL_FRONT
