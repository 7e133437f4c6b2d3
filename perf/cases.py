"""The reductions that a user of this package runs, as cases whose time can be measured.

A case is one call of :meth:`Dart.reduce` by a serving engine that keeps a context and its own output buffers:
key states and hidden states of one batch in, packed hidden rows, indices and position ids out.

Values.  The tokens are those of ``workloads`` (clusters, crops, drifting frames, a few outlying norms).  The key
states then go through an int8 cache with one power-of-two scale per token, as a quantised KV cache gives them back.
On that grid every sum of the step (norms, squares, dot products) is exact in fp32 in whatever order it is taken: two
correct implementations select the same tokens and the outputs, all of them copies or whole numbers, agree bit for
bit.  (With unquantised keys about one sample in two hundred has two tokens closer to each other than the rounding
of the sums, which a packed output turns into shifted rows; what rounding does there is checked against the fp64
oracle by the tests.)
"""
import math

import torch

from paper_2502_11494_b200 import dart, workloads

_QUOTAS, _GIVEN, _UNION = "quotas", "given", "union"


def _case(B, n_before, n_vis, n_after, d, n_pivot, n_keep, kind="cluster", mode=_QUOTAS, **more):
    return dict(B=B, n_before=n_before, n_vis=n_vis, n_after=n_after, d=d, n_pivot=n_pivot, n_keep=n_keep, kind=kind,
                mode=mode, **more)


def _of(w, mode=_QUOTAS, **more):
    return _case(w.B, w.n_before, w.n_vis, w.n_after, w.d, w.n_pivot, w.n_keep, w.kind, mode, **more)


def listed():
    W = workloads
    big = W.SWEEP_B256
    cases = {
        # one image of one request: nothing but latency and launches
        "image_b1": _of(W.LLAVA15_B1),
        # one high-resolution image of one request, the setting of the paper's efficiency study
        "highres_b1": _of(W.LLAVA_NEXT_B8.with_(B=1, n_pivot=8)),
        # the control step of 16 environments of a vision-language-action model
        "action_b16": _of(W.VLA_B16),
        # a batched prefill of ordinary images
        "image_b64": _of(W.LLAVA15_B64),
        # a few high-resolution requests, 16 pivots
        "highres_b8": _of(W.LLAVA_NEXT_B8),
        # video: long samples, another row width, 32 pivots
        "video_b4": _of(W.VIDEO_B4),
        # audio: half of the tokens are kept, which moves more rows than it drops
        "audio_b8": _of(W.AUDIO_B8),
        # sizes that nothing divides, a short text before and a long one after
        "ragged_b5": _case(5, 13, 1237, 171, 2048, 7, 173),
        # the large batch of the bandwidth sweep, the paper's setting of 8 pivots and 320 tokens
        "highres_b256": _of(big),
        # the same batch with the most pivots and the largest budget
        "highres_b256_p128": _of(big.with_(n_pivot=128, n_keep=640)),
        # pivots ranked by the caller (attention scores): one pass over the keys
        "given_b32": _of(big.with_(B=32), _GIVEN),
        # independent pivots, packed without padding for variable-length attention
        "union_b64": _of(W.LLAVA15_B64.with_(n_keep=128), _UNION),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Batches of 1 to 256 samples of 128 to 5000 tokens, 1 to 128 pivots, 10 to 80 % of the tokens kept."""
    n_vis = _log_uniform(rng, 128, 5000)
    d = rng.choice((1024, 2048, 3072, 3584, 4096, 4096, 5120))
    n_before, n_after = rng.randint(1, 64), rng.randint(5, 200)
    n_keep = max(8, int(n_vis * math.exp(rng.uniform(math.log(0.1), math.log(0.8)))))
    n_pivot = 8 if rng.random() < 0.5 else min(n_keep, _log_uniform(rng, 1, 128))
    mode = rng.choice((_QUOTAS,) * 5 + (_GIVEN, _UNION))
    one = work(_case(1, n_before, n_vis, n_after, d, n_pivot, n_keep))["bytes"]
    B = _log_uniform(rng, 1, min(256, int(7.5e9 / one)))  # no more than the large batch moves
    return _case(B, n_before, n_vis, n_after, d, n_pivot, n_keep, "cluster", mode)


def _through_int8(x):
    """bf16 rows -> int8 with a power-of-two scale per row (no finer than 1/16) -> bf16, in place."""
    f = x.float()
    scale = torch.exp2(torch.ceil(torch.log2(f.abs().amax(dim=1, keepdim=True) / 127.0))).clamp_(min=0.0625)
    x.copy_((f / scale).round_().clamp_(-127, 127).mul_(scale))


def prepare(case, seed):
    B, n_vis, d, P, Kp = case["B"], case["n_vis"], case["d"], case["n_pivot"], case["n_keep"]
    more = {"cluster": dict(centres_lo=max(4, n_vis // 36), centres_hi=max(4, n_vis // 6)),
            "crops": dict(n_crops=5, shared_frac=0.3),
            "video": dict(n_frames=100 if n_vis % 100 == 0 else 32, drift=0.05)}[case["kind"]]
    w = workloads.Workload("case", seed, B, case["n_before"], n_vis, case["n_after"], d, P, Kp, case["kind"], **more)
    dev = torch.device("cuda", torch.cuda.current_device())
    keys = torch.empty((B, w.S, d), dtype=torch.bfloat16, device=dev)
    hidden = torch.empty_like(keys)
    for b in range(B):
        k, h = workloads.make_sample(w, b, dev)
        keys[b].copy_(k)
        hidden[b].copy_(h)
        _through_int8(keys[b])
    state = {"keys": keys, "hidden": hidden, "w": w, "opts": None}
    state["ctx"] = dart.Dart(B, w.S, d, P, Kp, device=dev.index)
    # the engine's output buffers (with independent pivots fewer rows than these may be written)
    state["out"] = (torch.zeros((B, w.S_out, d), dtype=torch.bfloat16, device=dev),
                    torch.zeros((B, w.S_out), dtype=torch.int32, device=dev),
                    torch.zeros((B, w.S_out), dtype=torch.int64, device=dev))
    if case["mode"] == _GIVEN:
        g = torch.Generator(device=dev).manual_seed(seed)
        attention = torch.rand((B, n_vis), generator=g, device=dev)
        state["pivots"] = attention.topk(P, dim=1).indices.to(torch.int32).contiguous()
        state["opts"] = dart.dart_opts(pivots_in=state["pivots"].data_ptr())
    elif case["mode"] == _UNION:
        state["cu_seqlens"] = torch.zeros(B + 1, dtype=torch.int32, device=dev)
        state["opts"] = dart.dart_opts(rule=dart.DART_RULE_UNION, cu_seqlens=state["cu_seqlens"].data_ptr())
    return state


def run(state):
    w = state["w"]
    out = state["ctx"].reduce(state["hidden"], state["keys"], w.vis_offset, w.n_vis, w.n_pivot, w.n_keep, out=state["out"],
                              opts=state["opts"])
    return out + ((state["cu_seqlens"],) if "cu_seqlens" in state else ())


def work(case):
    """The key rows once, the kept hidden rows read and written, indices and position ids; one dot product per pivot and token."""
    B, n_vis, d, P = case["B"], case["n_vis"], case["d"], case["n_pivot"]
    S_out = case["n_before"] + case["n_after"] + case["n_keep"]
    return {"bytes": B * (2 * d * n_vis + 4 * d * S_out + 12 * S_out), "flops": 2.0 * B * P * n_vis * d}


def tolerance(case):
    return "exact"
