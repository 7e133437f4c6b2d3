"""The retention from ranked lists against the one-kernel form, bit for bit, through the C ABI (needs a B200)."""
import re

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2502_11494_b200 import dart  # noqa: E402
from test_gpu_parity import BAND_CASES, RETENTION_SHAPES, _band_inputs, run_gpu  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = BAND_CASES + [("gaussian", s) for s in RETENTION_SHAPES] + [
    # (kind, (B, S, d, vis_offset, n_vis, P, Kp))
    ("gaussian", (1, 300, 64, 1, 257, 1, 257)),           # one block of 256 entries and one entry more, one pivot
    ("gaussian", (40, 700, 64, 40, 576, 8, 520)),         # 256 threads per list; 90 % kept: the bins reach the row's upper end
    ("gaussian", (200, 300, 64, 40, 255, 8, 100)),        # 128 threads per list
    ("gaussian", (1, 16400, 64, 3, 16384, 2, 4098)),      # the longest row and the longest lists
    ("gaussian", (1, 3000, 64, 0, 2880, 1000, 2000)),     # 1000 pivots: several rounds of staging
    ("equal tokens", (3, 1500, 64, 10, 1402, 32, 1402)),
    # values per thread: 8, 16, 24 and 32, rows of one quarter more or less, with 64, 128 and 256 threads per list
    ("gaussian", (150, 600, 64, 3, 512, 8, 60)), ("gaussian", (150, 600, 64, 3, 513, 8, 60)),
    ("gaussian", (150, 2100, 64, 3, 2048, 8, 300)), ("gaussian", (150, 2100, 64, 3, 2049, 8, 1900)),
    ("gaussian", (150, 3200, 64, 3, 3072, 8, 9)), ("gaussian", (150, 3200, 64, 3, 3075, 8, 700)),
    ("gaussian", (150, 4200, 64, 3, 4097, 8, 600)), ("gaussian", (150, 6200, 64, 3, 6146, 8, 600)),
]


@pytest.mark.parametrize("kind,shape", CASES, ids=lambda v: v if isinstance(v, str) else "x".join(map(str, v)))
def test_ranked_lists_make_the_same_selections(kind, shape):
    B, S, d, vo, nv, P, Kp = shape
    k, h = _band_inputs(kind, B, S, d, vo, nv, P, seed=17 + sum(shape))
    a = run_gpu(k, h, vo, nv, P, Kp, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_SERIAL)
    b = run_gpu(k, h, vo, nv, P, Kp, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_RANKED)
    c = run_gpu(k, h, vo, nv, P, Kp, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_RANKED, debug=False)
    assert all(np.array_equal(x, y) for x, y in zip(a[:3], b[:3]))
    assert all(np.array_equal(x, y) for x, y in zip(a[:3], c[:3]))      # without the per-step outputs
    assert all(np.array_equal(a[3][n], b[3][n], equal_nan=(n == "eps")) for n in a[3])


@pytest.mark.parametrize("shape", [
    # (B, S, d, vis_offset, n_vis, P, Kp): up to two lists per SM, short rows and long ones; up to eight; rows that take more threads than the rule's
    (1, 1040, 64, 3, 1024, 8, 90), (1, 1040, 64, 3, 1025, 8, 90), (37, 1600, 64, 3, 1537, 8, 700), (38, 1600, 64, 3, 1536, 8, 700), (37, 1600, 64, 3, 1537, 8, 1008), (38, 1600, 64, 3, 1536, 8, 1009),
    (148, 600, 64, 3, 576, 8, 300), (149, 600, 64, 3, 576, 8, 300), (1, 6200, 64, 3, 6145, 3, 2000), (40, 6200, 64, 3, 6144, 8, 200), (40, 6200, 64, 3, 6145, 8, 200),
    (1, 12300, 64, 3, 8193, 2, 100), (1, 12300, 64, 3, 12288, 2, 4000), (1, 12300, 64, 3, 12289, 2, 4000),
], ids=lambda v: "x".join(map(str, v)))
def test_ranked_lists_at_the_lines_between_threads_per_list(shape):
    B, S, d, vo, nv, P, Kp = shape
    k, h = _band_inputs("gaussian", B, S, d, vo, nv, P, seed=23 + sum(shape))
    a = run_gpu(k, h, vo, nv, P, Kp, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_SERIAL, debug=False)
    b = run_gpu(k, h, vo, nv, P, Kp, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_RANKED, debug=False)
    assert all(np.array_equal(x, y) for x, y in zip(a[:3], b[:3]))


def _captured(call):
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    graph.enable_debug_mode()
    with torch.cuda.graph(graph):
        call()
    return graph


def _waits_for_words(graph, path):
    graph.debug_dump(str(path))
    return re.search(r"gather_kernelILb0ELb([01])E", path.read_text()).group(1) == "1"


@pytest.mark.parametrize("kept", [257, 256, 255, 90])
def test_rows_handed_to_the_gather_word_by_word(kept, tmp_path):
    """Both sides of the line (20 packed rows per SM), one context through several calls, a refused call and a replayed one among them."""
    B, d, vo, nv, P = 4, 128, 11, 1216, 5
    S = nv + 5 * torch.cuda.get_device_properties(0).multi_processor_count - 256       # 256 kept: just the line's rows
    bits = lambda t: t.view(torch.int16) if t.dtype == torch.bfloat16 else t
    g = torch.Generator(device="cuda").manual_seed(kept)
    k = torch.randint(-15, 16, (B, S, d), generator=g, device="cuda", dtype=torch.int8).bfloat16()
    h = torch.randn((B, S, d), generator=g, device="cuda").bfloat16()
    bad = torch.zeros((B, P), dtype=torch.int32, device="cuda")             # the same pivot five times
    pos = (torch.randperm(B * S, generator=g, device="cuda") + 7).view(B, S).contiguous()
    ref, ctx = dart.Dart(B, S, d, P, 800), dart.Dart(B, S, d, P, 800)
    want = ref.reduce(h, k, vo, nv, P, kept, pos_in=pos, opts=dart.dart_opts(path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_SERIAL))
    for n in (kept, kept + 1, 0, kept):
        if n == 0:
            ctx.reduce(h, k, vo, nv, P, kept, opts=dart.dart_opts(pivots_in=bad.data_ptr()))
            torch.cuda.synchronize()
            assert ctx.status() == dart.DART_ERR_CHECK
        else:
            got = ctx.reduce(h, k, vo, nv, P, n, pos_in=pos)
    torch.cuda.synchronize()
    assert ctx.status() == dart.DART_OK
    assert all(torch.equal(bits(a), bits(b)) for a, b in zip(want, got))
    for t in got:
        t.zero_()
    torch.cuda.synchronize()
    graph = _captured(lambda: ctx.reduce(h, k, vo, nv, P, kept, pos_in=pos, out=got))
    assert _waits_for_words(graph, tmp_path / "graph.dot") == (kept <= 256)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert ctx.status() == dart.DART_OK
    assert all(torch.equal(bits(a), bits(b)) for a, b in zip(want, got))
    del graph
    ctx.close()
    ref.close()


@pytest.mark.parametrize("captured", ["before", "behind"])
def test_words_that_come_after_the_limit_are_not_the_next_calls(captured, tmp_path):
    """A wait for a row's word of a microsecond, which ends before 400 pivots have taken their turns: the rows are copied all the same,
    and a call on new contents - a graph captured before, replayed, or a call made after one was captured - finds no word of that call's."""
    B, S, d, vo, nv, P, Kp = 1, 16100, 64, 40, 16000, 400, 2600
    bits = lambda t: t.view(torch.int16) if t.dtype == torch.bfloat16 else t
    g = torch.Generator(device="cuda").manual_seed(5)
    draw = lambda: (torch.randint(-15, 16, (B, S, d), generator=g, device="cuda", dtype=torch.int8).bfloat16(),
                    torch.randn((B, S, d), generator=g, device="cuda").bfloat16())
    plain = dart.dart_opts(path=dart.DART_PATH_STAGED)
    ref, ctx = dart.Dart(B, S, d, P, Kp), dart.Dart(B, S, d, P, Kp)
    want = lambda: ref.reduce(h, k, vo, nv, P, Kp, opts=dart.dart_opts(path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_SERIAL))
    same = lambda a, b: all(torch.equal(bits(x), bits(y)) for x, y in zip(a, b))
    k, h = draw()
    got = ctx.reduce(h, k, vo, nv, P, Kp, opts=plain)
    torch.cuda.synchronize()
    capture = lambda: _captured(lambda: ctx.reduce(h, k, vo, nv, P, Kp, out=got, opts=plain))
    if captured == "before":
        graph = capture()
    late = ctx.reduce(h, k, vo, nv, P, Kp, opts=dart.dart_opts(path=dart.DART_PATH_STAGED, wait_limit=1))
    torch.cuda.synchronize()
    first, right = ctx.status(), same(late, want())
    if captured == "behind":
        graph = capture()
    assert _waits_for_words(graph, tmp_path / "graph.dot")
    later = []
    for _ in range(3):
        for t, n in zip((k, h), draw()):
            t.copy_(n)
        if captured == "before":
            graph.replay()
        else:
            ctx.reduce(h, k, vo, nv, P, Kp, out=got, opts=plain)
        later.append(same(got, want()))
        assert ctx.status() == dart.DART_OK
    assert later == [True] * 3
    assert first == dart.DART_OK and right
    del graph
    ctx.close()
    ref.close()


@pytest.mark.parametrize("kind,shape", [("gaussian", (3, 333, 264, 17, 301, 7, 60)), ("equal tokens", (2, 700, 64, 10, 640, 16, 200)),
                                        ("gaussian", (260, 130, 64, 5, 100, 3, 90)), ("gaussian", (2, 3000, 64, 0, 2880, 128, 640))],
                         ids=lambda v: v if isinstance(v, str) else "x".join(map(str, v)))
def test_ranked_lists_with_independent_pivots(kind, shape):
    B, S, d, vo, nv, P, Kp = shape
    k, h = _band_inputs(kind, B, S, d, vo, nv, P, seed=19 + sum(shape))
    got = []
    for retention in (dart.DART_RETAIN_SERIAL, dart.DART_RETAIN_RANKED):
        cu = torch.zeros(B + 1, dtype=torch.int32, device="cuda")
        ctx = dart.Dart(B, S, d, P, Kp)
        oh, oi, op, dbg = ctx.reduce(h, k, vo, nv, P, Kp, debug=True, opts=dart.dart_opts(
            path=dart.DART_PATH_STAGED, retention=retention, rule=dart.DART_RULE_UNION, cu_seqlens=cu.data_ptr()))
        torch.cuda.synchronize()
        assert ctx.status() == dart.DART_OK
        ctx.close()
        n = int(cu[-1])
        got.append([oh.view(-1, d)[:n].view(torch.int16), oi.view(-1)[:n], op.view(-1)[:n], cu, dbg["keep"], dbg["owner"],
                    dbg["eps"].view(torch.int32)])
    assert all(torch.equal(x, y) for x, y in zip(*got))


@pytest.mark.parametrize("n,P", [(1, 1), (5, 5), (2048, 8), (2049, 100), (4096, 1024), (4097, 33), (8195, 7), (12289, 1000), (16384, 1), (16385, 40)])
@pytest.mark.parametrize("values", ["distinct", "few", "equal", "one infinite"])
def test_ranked_pivots(n, P, values):
    """Scores that are exact in any order of summation (sums of 64 small whole numbers): a stable sort is the answer."""
    B, vo = 3, 2
    g = torch.Generator(device="cuda").manual_seed(n + P)
    keys = torch.randint(-127, 128, (B, n + 5, 64), generator=g, device="cuda").bfloat16()
    if values == "few":
        keys[:, :, 2:] = 1
        keys[:, :, :2] %= 5
    elif values == "equal":
        keys[:] = 3
    elif values == "one infinite":
        keys[:, vo + n // 2, 5] = float("inf")
    got = torch.full((B, P), -1, dtype=torch.int32, device="cuda")
    assert dart.dart_pivots_static(keys.data_ptr(), B, n + 5, 64, vo, n, P, got.data_ptr(), 0, None) == dart.DART_OK
    torch.cuda.synchronize()
    score = keys[:, vo:vo + n].float().abs().sum(-1)
    want = torch.sort(score, dim=1, descending=True, stable=True).indices[:, :P]
    assert torch.equal(got.long(), want)


@pytest.mark.parametrize("P,m", [(3, 3), (32, 33), (100, 200), (128, 511), (100, 639), (100, 641), (8, 72), (9, 640), (9, 641), (33, 640), (1, 31), (1, 33), (2, 640)])
@pytest.mark.parametrize("kind", ["gaussian", "same pivots"])
def test_turns_over_lists_of_every_length(kind, P, m):
    """Quotas and lists on both sides of the rule's lines; pivots that rank the tokens alike make every turn walk past the others' picks."""
    k, h = _band_inputs(kind, 3, 900, 64, 20, 850, P, seed=P + m)
    a = run_gpu(k, h, 20, 850, P, P + m, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_SERIAL)
    b = run_gpu(k, h, 20, 850, P, P + m, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_RANKED, debug=False)
    assert all(np.array_equal(x, y) for x, y in zip(a[:3], b[:3]))


@pytest.mark.parametrize("B", [1, 150])
def test_only_the_pivots_are_kept(B):
    k, h = _band_inputs("gaussian", B, 400, 64, 20, 350, 40, seed=B)
    a = run_gpu(k, h, 20, 350, 40, 40, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_SERIAL)
    b = run_gpu(k, h, 20, 350, 40, 40, path=dart.DART_PATH_STAGED)
    assert all(np.array_equal(x, y) for x, y in zip(a[:3], b[:3]))
    assert all(np.array_equal(a[3][n], b[3][n], equal_nan=(n == "eps")) for n in a[3])


@pytest.mark.parametrize("rule", [dart.DART_RULE_QUOTAS, dart.DART_RULE_UNION], ids=["quotas", "independent"])
@pytest.mark.parametrize("retention", range(6))
def test_more_samples_than_a_grid_has_rows(rule, retention):
    """65535 is the most a grid's second dimension takes: the forms that count samples there give way to those that do not."""
    B, S, d, vo, nv, P, Kp = 65537, 20, 64, 2, 16, 2, 6
    k, _ = _band_inputs("gaussian", B, S, d, vo, nv, P, seed=7)
    S_out = S - nv + Kp
    got = []
    for parts in ([(0, B)], [(0, 40000), (40000, B)]):
        rows, lengths = [], []
        ctx = dart.Dart(B, S, d, P, Kp)
        for lo, hi in parts:
            cu = torch.zeros(hi - lo + 1, dtype=torch.int32, device="cuda")
            opts = dart.dart_opts(retention=retention, rule=rule, cu_seqlens=cu.data_ptr() if rule == dart.DART_RULE_UNION else None)
            oh, oi, op = ctx.reduce(k[lo:hi], None, vo, nv, P, Kp, opts=opts)
            torch.cuda.synchronize()
            assert ctx.status() == dart.DART_OK
            n = int(cu[-1]) if rule == dart.DART_RULE_UNION else (hi - lo) * S_out
            rows.append((oh.view(-1, d)[:n].view(torch.int16), oi.view(-1)[:n], op.view(-1)[:n]))
            lengths.append(cu.diff())
        ctx.close()
        got.append([torch.cat(x) for x in zip(*rows)] + [torch.cat(lengths)])
    assert all(torch.equal(x, y) for x, y in zip(*got))


@pytest.mark.parametrize("kind", ["gaussian", "equal tokens"])
@pytest.mark.parametrize("n,less", [(576, 0), (2880, 0), (2880, 1), (2880, 40), (2881, 100), (2883, 300), (4100, 4), (300, 0)])
def test_lists_of_nearly_all_tokens(kind, n, less):
    """The last pivots' lists take nearly every token: what the guessed threshold leaves out goes to the last bin."""
    B, S, d, vo, P, Kp = 9, n + 9, 64, 4, 8, n - less
    k, h = _band_inputs(kind, B, S, d, vo, n, P, seed=n + less)
    a = run_gpu(k, h, vo, n, P, Kp, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_SERIAL)
    b = run_gpu(k, h, vo, n, P, Kp, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_RANKED)
    assert all(np.array_equal(x, y) for x, y in zip(a[:3], b[:3]))
    assert all(np.array_equal(a[3][m], b[3][m], equal_nan=(m == "eps")) for m in a[3])


@pytest.mark.parametrize("kind", ["gaussian", "equal tokens"])
def test_keeping_everything_takes_no_longer_than_the_other_forms(kind):
    """AUTO with n_keep == n_vis (it took 4 times as long as the bands while the last lists were ordered by counting)."""
    B, n, P = 32, 2880, 8
    k, h = _band_inputs(kind, B, n, 64, 0, n, P, seed=3)
    ctx = dart.Dart(B, n, 64, P, n)
    dart.dart_profile_enable(ctx.handle, True)
    ms = {}
    for retention in (dart.DART_RETAIN_AUTO, dart.DART_RETAIN_BANDS, dart.DART_RETAIN_AUTO, dart.DART_RETAIN_BANDS):
        for _ in range(5):
            ctx.reduce(h, k, 0, n, P, n, opts=dart.dart_opts(path=dart.DART_PATH_STAGED, retention=retention))
        ms[retention] = dart.dart_profile_read(ctx.handle)[1]["retain"][0]
    ctx.close()
    assert ms[dart.DART_RETAIN_AUTO] < 2 * ms[dart.DART_RETAIN_BANDS], ms


@pytest.mark.parametrize("n,P", [(5, 5), (576, 8), (576, 575), (1000, 1000), (2049, 100), (4096, 33), (16384, 3), (16385, 3)])
@pytest.mark.parametrize("n_nan", [1, 3])
def test_scores_that_are_not_numbers_rank_last(n, P, n_nan):
    """Inputs are meant to be finite; a score that is not a number comes behind all that are, whatever the sample's length."""
    B, vo = 2, 2
    g = torch.Generator(device="cuda").manual_seed(n + P)
    keys = torch.randint(-127, 128, (B, n + 5, 64), generator=g, device="cuda").bfloat16()
    for i in range(n_nan):
        keys[:, vo + (n - 1) * (i + 1) // n_nan, 7 * i] = float("nan") * (-1) ** i
    score = keys[:, vo:vo + n].float().abs().sum(-1).nan_to_num(nan=-1.0)
    want = torch.sort(score, dim=1, descending=True, stable=True).indices[:, :P]
    got = torch.full((B, P), -1, dtype=torch.int32, device="cuda")
    assert dart.dart_pivots_static(keys.data_ptr(), B, n + 5, 64, vo, n, P, got.data_ptr(), 0, None) == dart.DART_OK
    torch.cuda.synchronize()
    assert torch.equal(got.long(), want)
    if P <= 32 and n <= 8192:
        ctx = dart.Dart(B, n + 5, 64, P, P)
        dbg = ctx.reduce(keys, None, vo, n, P, P, debug=True, opts=dart.dart_opts(path=dart.DART_PATH_FLOW))[3]
        torch.cuda.synchronize()
        assert ctx.status() == dart.DART_OK and torch.equal(dbg["pivot_idx"].long(), want)
        ctx.close()


def test_similarities_that_are_not_numbers():
    k, h = _band_inputs("gaussian", 3, 900, 64, 20, 850, 9, seed=4)
    k[0, 30, 3] = float("inf")      # a pivot (its score is the largest): its own similarities are 0 / inf or inf / inf
    k[1, 40:60] = float("inf")
    k[2, 500, 9] = float("nan")
    a = run_gpu(k, h, 20, 850, 9, 300, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_SERIAL)
    b = run_gpu(k, h, 20, 850, 9, 300, path=dart.DART_PATH_STAGED, retention=dart.DART_RETAIN_RANKED)
    assert all(np.array_equal(x, y) for x, y in zip(a[:3], b[:3]))
    assert np.array_equal(a[3]["keep"], b[3]["keep"]) and np.array_equal(a[3]["owner"], b[3]["owner"])
