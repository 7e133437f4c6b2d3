"""The flow path (both reads of a row a few microseconds apart, pivots published word by word) against the oracle,
through the C ABI (needs a B200)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import parity  # noqa: E402
from paper_2502_11494_b200 import dart, workloads as W  # noqa: E402
from test_gpu_parity import _np, compare, gaussian, run_gpu  # noqa: E402

pytestmark = pytest.mark.gpu
FLOW = dart.DART_PATH_FLOW

# (B, S, d, vis_offset, n_vis, P, Kp): row groups of 64, pivot tiles of 8/16/32, one to sixteen column slices
SHAPES = [
    (1, 16, 64, 0, 16, 1, 1),             # one group, one atom, one slice; most SMs hold nothing
    (2, 50, 64, 3, 40, 32, 40),           # more pivots than groups of 16 selecting threads hold tokens; everything kept
    (3, 200, 128, 7, 64, 8, 20),          # exactly one row group
    (3, 200, 192, 7, 65, 9, 20),          # one row more; three atoms over two slices
    (2, 333, 320, 17, 301, 7, 60),        # five atoms over four slices
    (1, 700, 4096, 40, 576, 8, 64),       # sixteen slices
    (40, 700, 1088, 40, 576, 17, 64),     # 17 atoms, the widest pivot tile
    (2, 3000, 4096, 40, 2880, 16, 320),
    (1, 3300, 256, 9, 3073, 5, 200),      # one token more than the selecting threads ask for at once
    (2, 8200, 64, 4, 8192, 3, 700),       # the longest sample
    (1, 9000, 192, 5, 4097, 32, 500),     # a last row group of one row
    (3, 80, 8192, 2, 70, 12, 30),         # the widest rows
    (300, 40, 64, 1, 33, 4, 9),           # more samples than SMs
    (3, 400, 1024, 5, 301, 7, 60),        # two rows to a scoring task, the last task of one row
    (2, 9, 1024, 3, 1, 1, 1), (3, 80, 1024, 2, 65, 20, 40), (5, 300, 1024, 9, 128, 16, 30),
]


@pytest.mark.parametrize("given", [0, 1, 2], ids=["by score", "given", "given, text tokens among them"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_flow_matches_the_oracle(oracle, shape, given):
    B, S, d, vo, nv, P, Kp = shape
    k, h = gaussian(B, S, d, seed=1300 + sum(shape))
    ctx = dart.Dart(B, S, d, P, Kp)
    opts, piv = dart.dart_opts(path=FLOW), None
    if given:
        g = torch.Generator(device="cuda").manual_seed(5)
        n, opts.text_pivots = (nv, 0) if given == 1 else (S, 1)
        piv = torch.rand((B, n), generator=g, device="cuda").topk(P, dim=1).indices.to(torch.int32)
        piv = (piv - (vo if given == 2 else 0)).contiguous()
        opts.pivots_in = piv.data_ptr()
    try:
        for tune in (0, 0x1001, 0x10000):   # default; the least window and one slot; one slice where it fits
            opts.tune = tune
            try:
                res = ctx.reduce(h, k, vo, nv, P, Kp, debug=True, opts=opts)
            except dart.DartError as e:     # one slice of wide rows does not fit shared memory beside the ring
                assert tune == 0x10000 and d > 1024 and e.code == dart.DART_ERR_UNSUPPORTED
                continue
            torch.cuda.synchronize()
            assert ctx.status() == dart.DART_OK, dart.dart_status_detail(ctx.handle)
            if tune == 0:
                kb, hb = W.bits(k), W.bits(h)
                ora = oracle.reduce(hb, kb, vo, nv, P, Kp, pivots_in=None if piv is None else piv.cpu().numpy(),
                                    text_pivots=given == 2)
                rep = parity.check_batch(ora, kb, hb, vo, nv, P, Kp, _np(res[0]), _np(res[1]), _np(res[2]),
                                         dbg={n: _np(v) for n, v in res[3].items()}, pivots_given=given > 0, text_pivots=given == 2)
                assert rep.exact >= rep.above_margin
                assert rep.max_rel_l1 < 5e-5 and rep.max_rel_l2 < 5e-5 and rep.max_abs_sim < 2e-5
                first = res
            else:
                assert torch.allclose(res[3]["sim"], first[3]["sim"], rtol=0, atol=4e-5)   # each within 2e-5 of the oracle
                assert torch.equal(res[3]["pivot_idx"], first[3]["pivot_idx"]) and torch.equal(res[3]["l1"], first[3]["l1"])
    finally:
        ctx.close()


@pytest.mark.parametrize("B,n,d,P,flow", [
    (2, 300, 960, 8, True), (2, 300, 960, 17, False),          # rows of fewer than 1024 columns: never, up to 16 pivots
    (16, 2048, 512, 16, True), (5, 6554, 512, 16, False),      # ... up to 64 rows per column
    (5, 819, 64, 1, True), (5, 820, 64, 1, False), (40, 1700, 1024, 16, True),
    (3, 333, 1024, 17, False), (2, 500, 1024, 32, True),       # 1000 rows and more of 1024 columns
    (8, 1000, 1024, 25, True), (9, 1000, 1024, 25, False),     # ... up to 8000
    (60, 1000, 1024, 24, True), (9, 1401, 1024, 17, False),    # ... up to 60000 with up to 24 pivots and 1400 tokens
    (8, 1024, 2048, 32, True), (9, 1000, 2048, 32, False),     # 4 rows per column
    (12, 1000, 3072, 20, True), (13, 1000, 3072, 20, False), (4, 3000, 5120, 32, True),   # up to 12000
    (1, 100, 4096, 24, True), (50, 300, 2048, 24, True), (50, 400, 2048, 24, False),      # pairs of tiles half empty
    (50, 300, 5120, 24, False), (20, 700, 8192, 17, True),     # rows too wide for the other tensor-core kernels
], ids=lambda v: str(v))
def test_which_path_auto_takes(B, n, d, P, flow):
    """Both sides of every line of the rule; keys whose sums are exact in any order, so that the other paths give the same bits."""
    g = torch.Generator(device="cuda").manual_seed(B + n + d)
    k = torch.randint(-15, 16, (B, n + 9, d), generator=g, device="cuda", dtype=torch.int8).bfloat16()
    outs = []
    for path in (dart.DART_PATH_AUTO, dart.DART_PATH_STAGED):
        ctx = dart.Dart(B, n + 9, d, P, P + 40)
        dart.dart_profile_enable(ctx.handle, True)
        outs.append(ctx.reduce(k, None, 4, n, P, P + 40, opts=dart.dart_opts(path=path)))
        torch.cuda.synchronize()
        assert ctx.status() == dart.DART_OK
        launched = {name for name, (_, c) in dart.dart_profile_read(ctx.handle)[1].items() if c}
        assert ("flow" in launched) == (flow and path == dart.DART_PATH_AUTO), launched
        ctx.close()
    assert all(torch.equal(a, b) for a, b in zip(*outs))


@pytest.mark.parametrize("P", [17, 32])
@pytest.mark.parametrize("d", [4608, 4672, 5120, 8192])
def test_flow_takes_wide_rows_with_many_pivots_in_large_contexts(oracle, d, P):
    """The widest pivot tiles of the widest rows need eight slices, whose shares the workspace has to hold however large it is."""
    B, S, vo, nv, Kp = 2, 300, 7, 280, 60
    k, h = gaussian(B, S, d, seed=d + P)
    ctx = dart.Dart(600, S, d, P, Kp)     # 3000 row groups
    try:
        res = ctx.reduce(h, k, vo, nv, P, Kp, debug=True, opts=dart.dart_opts(path=FLOW))
        torch.cuda.synchronize()
        assert ctx.status() == dart.DART_OK
    finally:
        ctx.close()
    kb, hb = W.bits(k), W.bits(h)
    rep = parity.check_batch(oracle.reduce(hb, kb, vo, nv, P, Kp), kb, hb, vo, nv, P, Kp, _np(res[0]), _np(res[1]), _np(res[2]),
                             dbg={n: _np(v) for n, v in res[3].items()})
    assert rep.exact >= rep.above_margin and rep.max_abs_sim < 2e-5


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("P", [1, 5, 8, 13, 16, 31])
@pytest.mark.parametrize("nsl", [1, 2, 4, 8, 16])
def test_flow_shares_of_every_number_of_slices(nsl, P, given):
    """Keys whose sums are exact in any order: the similarities added up from the slices' shares equal the plain kernels' bit for bit."""
    B, n, d, Kp = 5, 131, 1024, P + 40                # row groups of 64, 64 and 3 rows
    g = torch.Generator(device="cuda").manual_seed(nsl + P)
    k = torch.randint(-15, 16, (B, n + 9, d), generator=g, device="cuda", dtype=torch.int8).bfloat16()
    piv = torch.rand((B, n), generator=g, device="cuda").topk(P, dim=1).indices.to(torch.int32).contiguous()
    outs = []
    for path in (FLOW, dart.DART_PATH_STAGED):
        ctx = dart.Dart(B, n + 9, d, P, Kp)
        o = dart.dart_opts(path=path, tune=nsl << 16 if path == FLOW else 0, pivots_in=piv.data_ptr() if given else None)
        oh, oi, op, dbg = ctx.reduce(k, None, 4, n, P, Kp, opts=o, debug=True)
        torch.cuda.synchronize()
        assert ctx.status() == dart.DART_OK
        ctx.close()
        outs.append((oh.view(torch.int16), oi, op, dbg["sim"]))
    assert all(torch.equal(a, b) for a, b in zip(*outs))


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("nsl,P,n,B", [(1, 8, 400, 300), (2, 16, 389, 300), (4, 8, 131, 430), (4, 31, 200, 360), (8, 13, 400, 140), (16, 8, 131, 330)])
def test_flow_many_items_of_every_number_of_slices(nsl, P, n, B, given):
    """Tens of items and, from four slices on, of samples per SM: the mailboxes, the pivots' ring and the pivot buffers go round several
    times (as above, bit for bit)."""
    d, Kp = 1024, P + 20
    g = torch.Generator(device="cuda").manual_seed(nsl + P)
    k = torch.randint(-15, 16, (B, n + 3, d), generator=g, device="cuda", dtype=torch.int8).bfloat16()
    piv = torch.rand((B, n), generator=g, device="cuda").topk(P, dim=1).indices.to(torch.int32).contiguous()
    outs = []
    for path in (FLOW, dart.DART_PATH_STAGED):
        ctx = dart.Dart(B, n + 3, d, P, Kp)
        o = dart.dart_opts(path=path, tune=nsl << 16 if path == FLOW else 0, pivots_in=piv.data_ptr() if given else None)
        oh, oi, op, dbg = ctx.reduce(k, None, 2, n, P, Kp, opts=o, debug=True)
        torch.cuda.synchronize()
        assert ctx.status() == dart.DART_OK
        ctx.close()
        outs.append((oh.view(torch.int16), oi, op, dbg["sim"]))
    assert all(torch.equal(a, b) for a, b in zip(*outs))


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("nsl,P,n,B", [(0, 16, 4096, 21), (4, 8, 64, 1300), (8, 3, 1001, 90)])
def test_flow_scorers_wait_for_the_second_pass(nsl, P, n, B, given):
    """Batches of more than 640 MB of keys, whose scorers are held back to some 50 MB beyond their SM's second pass."""
    d, Kp = 4096, P + 20
    assert B * n * d * 2 > 640 << 20
    g = torch.Generator(device="cuda").manual_seed(nsl + P)
    k = torch.randint(-15, 16, (B, n + 3, d), generator=g, device="cuda", dtype=torch.int8).bfloat16()
    piv = torch.rand((B, n), generator=g, device="cuda").topk(P, dim=1).indices.to(torch.int32).contiguous()
    outs = []
    for path in (FLOW, dart.DART_PATH_STAGED):
        ctx = dart.Dart(B, n + 3, d, P, Kp)
        o = dart.dart_opts(path=path, tune=nsl << 16 if path == FLOW else 0, pivots_in=piv.data_ptr() if given else None)
        oh, oi, op, dbg = ctx.reduce(k, None, 2, n, P, Kp, opts=o, debug=True)
        torch.cuda.synchronize()
        assert ctx.status() == dart.DART_OK
        ctx.close()
        outs.append((oh.view(torch.int16), oi, op, dbg["sim"]))
    assert all(torch.equal(a, b) for a, b in zip(*outs))


@pytest.mark.parametrize("norm_kind,smallest", [(1, 1), (2, 0), (2, 1)])
def test_flow_ranking_variants(oracle, norm_kind, smallest):
    k, h = gaussian(3, 500, 256, seed=77)
    rep = compare(oracle, k, h, 20, 444, 6, 90, path=FLOW, norm_kind=norm_kind, smallest=smallest)
    assert rep.exact >= rep.above_margin and rep.max_abs_sim < 2e-5


def test_flow_equal_scores_rank_the_lower_index_first(oracle):
    """Rows that are copies of each other tie in score: the list above the selection's floor holds every token."""
    k, h = gaussian(2, 1300, 128, seed=78)
    k[:, 10:1300] = k[:, 10:11] * 0.5         # all vision rows but the first equal; the first one larger
    k[:, 10] = k[:, 11] * 2
    oh, oi, op, dbg = run_gpu(k, h, 10, 1290, 5, 40, path=FLOW)
    assert np.array_equal(dbg["pivot_idx"], np.tile(np.arange(5, dtype=np.int32), (2, 1)))


@pytest.mark.parametrize("n_vis", [128, 384, 385, 640, 641, 1024, 1025, 8192])
@pytest.mark.parametrize("P", [1, 5, 32])
@pytest.mark.parametrize("values", ["equal", "four values", "half at the top"])
def test_flow_many_equal_scores(values, P, n_vis):
    """More tokens at the selection's floor than its list holds (384 entries up to 1024 tokens, 640 beyond).  Scores are sums of 64
    small whole numbers, exact in any order: a stable sort is the answer, in time that does not grow with the square of the ties."""
    B, vo = 5, 3
    g = torch.Generator(device="cuda").manual_seed(n_vis + P)
    keys = torch.randint(-9, 10, (B, n_vis + 5, 64), generator=g, device="cuda").bfloat16()
    if values == "equal":
        keys[:] = 3
    elif values == "four values":
        keys[:] = keys[:, :1].abs() + torch.randint(1, 5, (B, n_vis + 5, 1), generator=g, device="cuda")
    else:
        keys[:, vo + n_vis // 2:vo + n_vis] = 9
    score = keys[:, vo:vo + n_vis].float().abs().sum(-1)
    ctx = dart.Dart(B, n_vis + 5, 64, P, P)
    for smallest in (0, 1):
        dbg = ctx.reduce(keys, None, vo, n_vis, P, P, debug=True, opts=dart.dart_opts(path=FLOW, pivot_smallest=smallest))[3]
        torch.cuda.synchronize()
        assert ctx.status() == dart.DART_OK
        want = torch.sort(score, dim=1, descending=not smallest, stable=True).indices[:, :P]
        assert torch.equal(dbg["pivot_idx"].long(), want)
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = {FLOW: [], dart.DART_PATH_STAGED: []}    # the staged path selects by radix passes whatever the scores
    for path in list(times) * 5:                      # (the best of five: the host may pause between launches)
        start.record()
        for _ in range(4):
            ctx.reduce(keys, None, vo, n_vis, P, P, opts=dart.dart_opts(path=path))
        end.record()
        torch.cuda.synchronize()
        times[path].append(start.elapsed_time(end))
    assert min(times[FLOW]) < 3 * min(times[dart.DART_PATH_STAGED]), times   # quadratic: 20 times as long at 8192 equal scores
    ctx.close()


@pytest.mark.parametrize("shape", [(1, 64, 64, 0, 64, 33, 40), (1, 8300, 64, 0, 8193, 2, 8), (1, 64, 96, 0, 64, 2, 8)],
                         ids=["33 pivots", "8193 tokens", "d not a multiple of 64"])
def test_flow_says_what_it_does_not_take(shape):
    B, S, d, vo, nv, P, Kp = shape
    k, h = gaussian(B, S, d, seed=79)
    ctx = dart.Dart(B, S, d, P, Kp)
    with pytest.raises(dart.DartError) as e:
        ctx.reduce(h, k, vo, nv, P, Kp, opts=dart.dart_opts(path=FLOW))
    assert e.value.code == dart.DART_ERR_UNSUPPORTED
    ctx.close()


@pytest.mark.parametrize("withhold,where", [(1, 90), (2, 102)], ids=["a row's word never published", "an item's shares never counted in"])
def test_flow_expired_waits_are_reported_not_hung(withhold, where):
    """The warp that waits for what is withheld gives up within its limit and says so, every other wait ends too, and the next call on
    the same context succeeds, as does a graph captured before."""
    w = W.LLAVA15_B64.with_(B=3)
    k, h = W.make_batch(w, device="cuda")
    shape = (w.vis_offset, w.n_vis, w.n_pivot, w.n_keep)
    ctx = dart.Dart(w.B, w.S, w.d, w.n_pivot, w.n_keep)
    out = ctx.reduce(h, k, *shape, opts=dart.dart_opts(path=FLOW))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.reduce(h, k, *shape, out=out, opts=dart.dart_opts(path=FLOW))
    ctx.reduce(h, k, *shape, opts=dart.dart_opts(path=FLOW, wait_limit=20000, test_withhold_pivots=withhold))      # 20 ms limit
    torch.cuda.synchronize()
    assert ctx.status() == dart.DART_ERR_TIMEOUT
    rc, detail = dart.dart_status_detail(ctx.handle)
    assert rc == dart.DART_OK and detail[0] == where, detail
    k, h = k.copy_(k.flip(0)), h.copy_(h.flip(0))
    graph.replay()
    good = ctx.reduce(h, k, *shape, opts=dart.dart_opts(path=FLOW))
    torch.cuda.synchronize()
    assert ctx.status() == dart.DART_OK
    ref = run_gpu(k, h, *shape, path=dart.DART_PATH_STAGED, debug=False)
    for got in (out, good):
        assert np.array_equal(got[1].cpu().numpy(), ref[1]) and np.array_equal(W.bits(got[0]), ref[0])
    del graph
    ctx.close()


def _calls(seed, n):
    """A mixed bag of calls within the maxima (6, 900, 256, 32, 700): batch sizes, lengths, pivots, paths, rules."""
    rng = np.random.default_rng(seed)
    for i in range(n):
        nv = int(rng.choice([rng.integers(1, 70), rng.integers(64, 800)]))
        P = int(rng.integers(1, min(nv, 32) + 1))
        path = int(rng.choice([FLOW, FLOW, FLOW, dart.DART_PATH_AUTO, dart.DART_PATH_TWO_PASS, dart.DART_PATH_FUSED, dart.DART_PATH_STAGED]))
        yield dict(B=int(rng.integers(1, 7)), vo=int(rng.integers(0, 50)), nv=nv, after=int(rng.integers(0, 50)), P=P,
                   Kp=int(rng.integers(P, min(nv, 700) + 1)), path=path, given=bool(rng.integers(0, 3) == 0), union=bool(rng.integers(0, 4) == 0),
                   retention=int(rng.choice([dart.DART_RETAIN_AUTO, dart.DART_RETAIN_RANKED])), seed=1000 * seed + i)


def _inputs(c, d):
    k, h = gaussian(c["B"], c["vo"] + c["nv"] + c["after"], d, seed=c["seed"])
    g = torch.Generator(device="cuda").manual_seed(c["seed"])
    piv = torch.rand((c["B"], c["nv"]), generator=g, device="cuda").topk(c["P"], dim=1).indices.to(torch.int32).contiguous()
    S_out = c["vo"] + c["after"] + c["Kp"]
    out = (torch.zeros((c["B"], S_out, d), dtype=torch.bfloat16, device="cuda"), torch.zeros((c["B"], S_out), dtype=torch.int32, device="cuda"),
           torch.zeros((c["B"], S_out), dtype=torch.int64, device="cuda"))
    cu = torch.zeros(c["B"] + 1, dtype=torch.int32, device="cuda")
    opts = dart.dart_opts(path=c["path"], retention=c["retention"], pivots_in=piv.data_ptr() if c["given"] else None,
                          rule=dart.DART_RULE_UNION if c["union"] else dart.DART_RULE_QUOTAS, cu_seqlens=cu.data_ptr() if c["union"] else None)
    return dict(k=k, h=h, piv=piv, out=out, cu=cu, opts=opts)


@pytest.mark.parametrize("seed", range(6))
def test_one_context_through_changing_calls(seed):
    """The words and counters that a call leaves behind are the next call's, whatever its tensors, batch, length, pivots and path:
    forty different calls on one context, nothing between them, against a context of its own for each."""
    d, calls = 256, list(_calls(seed, 40))
    bags = [_inputs(c, d) for c in calls]
    shared = dart.Dart(6, 900, d, 32, 700)
    torch.cuda.synchronize()
    for c, x in zip(calls, bags):
        shared.reduce(x["h"], x["k"], c["vo"], c["nv"], c["P"], c["Kp"], out=x["out"], opts=x["opts"])
    torch.cuda.synchronize()
    assert shared.status() == dart.DART_OK, dart.dart_status_detail(shared.handle)
    shared.close()
    for c, x in zip(calls, bags):
        y = _inputs(c, d)
        ctx = dart.Dart(c["B"], c["vo"] + c["nv"] + c["after"], d, c["P"], c["Kp"])
        ctx.reduce(x["h"], x["k"], c["vo"], c["nv"], c["P"], c["Kp"], out=y["out"], opts=y["opts"])
        torch.cuda.synchronize()
        assert ctx.status() == dart.DART_OK
        ctx.close()
        n = int(y["cu"][-1]) if c["union"] else None      # rows beyond the packed ones are not written
        assert torch.equal(x["cu"], y["cu"]), c
        for a, b in zip(x["out"], y["out"]):
            a, b = (a.view(-1, d) if a.dim() == 3 else a.view(-1), b.view(-1, d) if b.dim() == 3 else b.view(-1))
            assert torch.equal(a[:n], b[:n]), c


def test_a_graph_replays_on_new_contents_between_other_calls():
    """A captured call reads what its input buffers hold when it is replayed, and finds its words as it expects them after eager
    calls of other shapes on the same context."""
    d, s, g = 256, torch.cuda.Stream(), torch.cuda.CUDAGraph()
    c = dict(B=5, vo=7, nv=600, after=30, P=8, Kp=90, path=FLOW, given=False, union=False, retention=0, seed=1)
    others = list(_calls(77, 6))
    x = _inputs(c, d)
    ctx = dart.Dart(6, 900, d, 32, 700)
    with torch.cuda.stream(s):
        ctx.reduce(x["h"], x["k"], c["vo"], c["nv"], c["P"], c["Kp"], out=x["out"], opts=x["opts"], stream=s)
        s.synchronize()
        g.capture_begin()
        ctx.reduce(x["h"], x["k"], c["vo"], c["nv"], c["P"], c["Kp"], out=x["out"], opts=x["opts"], stream=s)
        g.capture_end()
        for i, o in enumerate(others):
            y = _inputs(dict(o, union=False), d)
            ctx.reduce(y["h"], y["k"], o["vo"], o["nv"], o["P"], o["Kp"], out=y["out"], opts=y["opts"], stream=s)
            fresh = _inputs(dict(c, seed=100 + i), d)
            x["k"].copy_(fresh["k"])
            x["h"].copy_(fresh["h"])
            g.replay()
            s.synchronize()
            assert ctx.status() == dart.DART_OK
            got = [t.clone() for t in x["out"]]
            own = dart.Dart(c["B"], 637, d, 8, 90)
            own.reduce(fresh["h"], fresh["k"], c["vo"], c["nv"], c["P"], c["Kp"], out=fresh["out"], opts=fresh["opts"], stream=s)
            s.synchronize()
            own.close()
            assert all(torch.equal(a, b) for a, b in zip(got, fresh["out"]))
    ctx.close()
