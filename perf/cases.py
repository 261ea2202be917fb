"""The work a user of this library has it do, as timed cases over the range of sizes it serves.

Everything goes through the binding `paper_2607_21599_b200.api`, as an inference program calls it: tensors, parameters
and the workspace are made once, `run` makes the calls of one pass.  The attention shapes are those of the repository's
own workloads (28/4, 32/8 and 40/8 query/key heads of 128 channels, contexts of 1k to 136k document tokens, questions of
some tens of tokens, 5 % to 30 % of the document tokens recomputed).

Kinds of pass (`case["kind"]`):
  layer     one transformer layer (`daf_layer`): selection from importance scores, or positions given, gather and cache
            update, both attention stages, fused rows -- what a prefill does for every layer
  fp8       the same from an offline cache stored in fp8 (`daf_layer_fp8`)
  prefill   every layer of a context: positions ranked once from the K/V of three signal layers (`daf_select_from_kv`),
            then all layers from those positions
  select    the first step of a prefill alone: the signal of three layers, the ranking, gather and cache update
  question  a further question against a context whose cache is already repaired (`daf_qd_attn`)
  full      full recomputation (`daf_full_causal_attn`), the path a program falls back to without an offline cache
  host      one layer whose tensors live in pinned host memory (`daf_layer_host`)
"""
import math

import torch

from paper_2607_21599_b200 import api

HEADS = {"28/4": (28, 4), "32/8": (32, 8), "40/8": (40, 8)}
D = 128
DOC = 512                # tokens of one document: importance and deviation cluster by document
SIGNAL_LAYERS = 3
Q_IN_PLACE_K = 16384     # from this many important tokens on the header's advice is to pass no packed Q buffer


def _case(kind, heads, L_d, L_q, r=0.0, layers=1, n_sig=1, given=False, scatter=False):
    return {"kind": kind, "heads": heads, "L_d": L_d, "L_q": L_q, "r": r, "layers": layers, "n_sig": n_sig,
            "given": given, "scatter": scatter}


def listed():
    def named(name, *a, **kw):
        return dict(_case(*a, **kw), name=name)

    return [
        # the smallest context of the workloads, positions reused from an earlier layer: launches and host time count
        named("layer_1k_given", "layer", "28/4", 1024, 32, 0.15, given=True),
        # a short multi-document question
        named("layer_6k", "layer", "28/4", 6144, 64, 0.15),
        # odd sizes, three rows of scores, rows scattered to their positions (a program that keeps an [N, ...] buffer)
        named("layer_11k_ragged_scatter", "layer", "40/8", 11003, 77, 0.20, n_sig=3, scatter=True),
        # the middle of the benchmark's range
        named("layer_16k", "layer", "32/8", 16384, 128, 0.10),
        # the benchmark's headline shape
        named("layer_32k", "layer", "28/4", 32768, 128, 0.20),
        # the longest context evaluated: everything is tensor-core time
        named("layer_136k", "layer", "28/4", 139264, 128, 0.30),
        # offline cache kept in fp8
        named("layer_fp8_16k", "fp8", "32/8", 16384, 128, 0.10),
        # a whole prefill of a short context: 28 layers one behind the other
        named("prefill_6k_28_layers", "prefill", "28/4", 6144, 64, 0.15, layers=28),
        # ranking from K/V: memory-bound
        named("select_from_kv_32k", "select", "28/4", 32768, 128, 0.20),
        # the next question of a conversation over the same documents
        named("question_32k", "question", "28/4", 32768, 64),
        # no offline cache: everything recomputed
        named("full_16k", "full", "32/8", 16384, 128),
        # tensors in pinned host memory
        named("layer_host_6k", "host", "28/4", 6144, 64, 0.15),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    largest = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(["layer"] * 6 + ["fp8", "prefill", "select", "question", "full", "host"])
        heads = rng.choice(sorted(HEADS))
        L_q = _log_uniform(rng, 16, 256)
        r = round(rng.uniform(0.05, 0.30), 3)
        hi = {"layer": 139264, "fp8": 65536, "prefill": 8192, "select": 65536, "question": 139264, "full": 32768, "host": 16384}[kind]
        L_d = _log_uniform(rng, 1024, hi)
        layers = rng.randint(4, 32) if kind == "prefill" else 1
        if kind in ("question", "full"):
            r = 0.0
        c = _case(kind, heads, L_d, L_q, r, layers,
                  n_sig=rng.choice([1, 3]) if kind in ("layer", "fp8", "host") else 1,
                  given=kind == "layer" and rng.random() < 0.3,
                  scatter=kind in ("layer", "fp8", "prefill") and rng.random() < 0.3)
        if work(c)["flops"] <= largest:
            return c


def _normal(shape, g):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).to(torch.bfloat16)


def _token_spread(n, g):
    """How far a token's fresh state is from its offline one: lognormal per token, larger in a fifth of the documents."""
    docs = torch.rand((n + DOC - 1) // DOC, generator=g, device="cuda") < 0.2
    hot = docs.repeat_interleave(DOC)[:n].float()
    return torch.exp(0.5 * torch.randn(n, generator=g, device="cuda") + 1.2 * hot)


def _scores(n_sig, n, g):
    """Importance signals: positive, heavy-tailed, clustered by document, every signal layer with noise of its own."""
    s = _token_spread(n, g).square()
    return (s * torch.exp(0.3 * torch.randn(n_sig, n, generator=g, device="cuda"))).contiguous()


def _offline(fresh, n, spread, g):
    """The offline document rows: the fresh ones with the token's deviation, and room for the question rows."""
    kv = torch.zeros_like(fresh)
    for lo in range(0, n, 8192):
        hi = min(n, lo + 8192)
        noise = torch.randn(fresh[lo:hi].shape, generator=g, device="cuda")
        kv[lo:hi] = (fresh[lo:hi].float() + 0.3 * spread[lo:hi, None, None] * noise).to(torch.bfloat16)
    return kv


class _State:
    pass


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s = _State()
    s.kind, s.n_sig = case["kind"], case["n_sig"]
    Hq, Hkv = HEADS[case["heads"]]
    L_d, L_q, r, layers = case["L_d"], case["L_q"], case["r"], case["layers"]
    N = L_d + L_q
    s.p = api.make_params(L_d, L_q, r, Hq, Hkv, D, fuse_mode=1 if case["scatter"] else 0)
    s.k = k = api.daf_num_important(L_d, r)
    s.L_d = L_d

    def rows(*shape):
        return torch.empty(shape, dtype=torch.bfloat16, device="cuda")

    if s.kind == "full":
        s.q, s.kf, s.vf = _normal((N, Hq, D), g), _normal((N, Hkv, D), g), _normal((N, Hkv, D), g)
        s.n, s.hidden = N, rows(N, Hq, D)
        s.ws = api.alloc_workspace(s.p)
        return s
    if s.kind == "question":
        s.q, s.kv_k, s.kv_v = _normal((L_q, Hq, D), g), _normal((N, Hkv, D), g), _normal((N, Hkv, D), g)
        s.hidden, s.stride = rows(L_q, Hq, D), Hq * D * 2
        s.ws = api.alloc_workspace(s.p)
        return s

    spread = _token_spread(L_d, g)
    lay = (layers,) if s.kind == "prefill" else ()
    s.q, s.kf, s.vf = _normal(lay + (N, Hq, D), g), _normal(lay + (N, Hkv, D), g), _normal(lay + (N, Hkv, D), g)
    s.idx = torch.empty(k, dtype=torch.int32, device="cuda")
    s.given = None
    s.scores = None if s.kind in ("prefill", "select") else _scores(s.n_sig, L_d, g)
    if case["given"]:
        s.given = torch.sort(torch.topk(s.scores[0], k).indices).values.to(torch.int32)
        s.scores = None

    if s.kind == "host":
        kv_k, kv_v = _offline(s.kf, L_d, spread, g), _offline(s.vf, L_d, spread, g)

        def pinned(t):
            h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
            h.copy_(t)
            return h

        s.q, s.kf, s.vf, s.kv_k, s.kv_v, s.scores = (pinned(t) for t in (s.q, s.kf, s.vf, kv_k, kv_v, s.scores))
        s.hidden = torch.empty((k + L_q, Hq, D), dtype=torch.bfloat16, pin_memory=True)
        s.idx = torch.empty(k, dtype=torch.int32, pin_memory=True)
        s.arena = torch.zeros(api.daf_layer_host_arena_bytes(s.p), dtype=torch.uint8, device="cuda")
        return s

    if s.kind == "fp8":
        def stored(fresh):
            x = _offline(fresh, L_d, spread, g)[:L_d].float()
            scale = x.abs().amax(dim=(0, 2)) / 448.0
            return (x / scale[None, :, None]).to(torch.float8_e4m3fn).view(torch.uint8), scale

        (s.k8, s.k_scale), (s.v8, s.v_scale) = stored(s.kf), stored(s.vf)
        s.kv_k, s.kv_v = torch.zeros_like(s.kf), torch.zeros_like(s.vf)
    elif s.kind == "prefill":
        s.kv_k = torch.stack([_offline(x, L_d, spread, g) for x in s.kf])
        s.kv_v = torch.stack([_offline(x, L_d, spread, g) for x in s.vf])
        # the K/V as they were stored offline: the layers' own caches are repaired in place
        s.sig_k = [s.kv_k[l].clone() for l in range(1, 1 + SIGNAL_LAYERS)]
        s.sig_v = [s.kv_v[l].clone() for l in range(1, 1 + SIGNAL_LAYERS)]
    else:
        s.kv_k, s.kv_v = _offline(s.kf, L_d, spread, g), _offline(s.vf, L_d, spread, g)
    if s.kind == "select":
        s.sig_kf = [_normal((N, Hkv, D), g) for _ in range(SIGNAL_LAYERS)]
        s.sig_vf = [_normal((N, Hkv, D), g) for _ in range(SIGNAL_LAYERS)]
        s.sig_k = [_offline(x, L_d, spread, g) for x in s.sig_kf]
        s.sig_v = [_offline(x, L_d, spread, g) for x in s.sig_vf]
        s.sums = torch.empty(L_d, dtype=torch.float32, device="cuda")
    s.q_pack = rows(k, Hq, D) if k < Q_IN_PLACE_K or s.kind == "select" else None
    s.k_pack, s.v_pack = rows(k, Hkv, D), rows(k, Hkv, D)
    if s.kind != "select":
        s.hidden = torch.zeros(lay + ((N if case["scatter"] else k + L_q), Hq, D), dtype=torch.bfloat16, device="cuda")
    if s.kind == "prefill":
        s.layer_views = [tuple(t[l] for t in (s.q, s.kf, s.vf, s.kv_k, s.kv_v, s.hidden)) for l in range(layers)]
        s.idx_layer = torch.empty_like(s.idx)
    s.ws = api.alloc_workspace(s.p)
    return s


def run(s):
    if s.kind == "layer":
        api.check(api.daf_layer(s.p, s.scores, s.n_sig, s.given, s.q, s.kf, s.vf, s.kv_k, s.kv_v, s.idx, s.q_pack,
                                s.k_pack, s.v_pack, s.hidden, None, s.ws), "daf_layer")
        return s.hidden, s.idx, s.kv_k, s.kv_v
    if s.kind == "fp8":
        api.check(api.daf_layer_fp8(s.p, s.scores, s.n_sig, None, s.q, s.kf, s.vf, s.k8, s.v8, s.k_scale, s.v_scale,
                                    s.kv_k, s.kv_v, s.idx, s.q_pack, s.k_pack, s.v_pack, s.hidden, None, s.ws),
                  "daf_layer_fp8")
        return s.hidden, s.idx, s.kv_k, s.kv_v
    if s.kind == "prefill":
        for l, (q, kf, vf, kv_k, kv_v, hidden) in enumerate(s.layer_views):
            if l == 0:
                # ranked by the signal layers; this call also prepares the first layer's packed rows and cache
                api.check(api.daf_select_from_kv(s.p, [s.layer_views[i][1] for i in range(1, 1 + SIGNAL_LAYERS)],
                                                 [s.layer_views[i][2] for i in range(1, 1 + SIGNAL_LAYERS)], s.sig_k,
                                                 s.sig_v, q, kf, vf, kv_k, kv_v, s.idx, s.q_pack, s.k_pack, s.v_pack,
                                                 None, s.ws), "daf_select_from_kv")
                api.check(api.daf_imp_qd_attn(s.p, s.q_pack, q, s.k_pack, s.v_pack, q[s.L_d:], kv_k, kv_v, s.idx,
                                              hidden, s.ws), "daf_imp_qd_attn")
            else:
                api.check(api.daf_layer(s.p, None, 1, s.idx, q, kf, vf, kv_k, kv_v, s.idx_layer, s.q_pack, s.k_pack,
                                        s.v_pack, hidden, None, s.ws), "daf_layer")
        return s.hidden, s.idx, s.kv_k, s.kv_v
    if s.kind == "select":
        api.check(api.daf_select_from_kv(s.p, s.sig_kf, s.sig_vf, s.sig_k, s.sig_v, s.q, s.kf, s.vf, s.kv_k, s.kv_v,
                                         s.idx, s.q_pack, s.k_pack, s.v_pack, s.sums, s.ws), "daf_select_from_kv")
        return s.idx, s.sums, s.q_pack, s.k_pack, s.v_pack, s.kv_k, s.kv_v
    if s.kind == "question":
        api.check(api.daf_qd_attn(s.p, s.q, s.kv_k, s.kv_v, s.hidden, s.stride, None, None, s.ws), "daf_qd_attn")
        return s.hidden
    if s.kind == "full":
        api.check(api.daf_full_causal_attn(s.p, s.n, s.q, s.kf, s.vf, s.hidden, None, s.ws), "daf_full_causal_attn")
        return s.hidden
    api.check(api.daf_layer_host(s.p, s.scores, s.n_sig, None, s.q, s.kf, s.vf, s.kv_k, s.kv_v, 1, s.hidden, s.idx,
                                 s.arena), "daf_layer_host")
    return s.hidden, s.idx, s.kv_k, s.kv_v


def work(case):
    """Bytes: the rows a pass has to read and the rows it has to leave, each once (packed copies count where they are a
    result, not where they are an intermediate).  Flops: 4 * 128 per query head and visible (query, key) pair."""
    Hq, Hkv = HEADS[case["heads"]]
    L_d, L_q, layers = case["L_d"], case["L_q"], case["layers"]
    N, k = L_d + L_q, api.daf_num_important(L_d, case["r"])
    q_row, kv_row = Hq * D * 2, 2 * Hkv * D * 2      # a K row and a V row
    pairs = {"full": N * (N + 1) // 2, "select": 0}.get(
        case["kind"], k * (k + 1) // 2 + L_q * L_d + L_q * (L_q + 1) // 2)
    flops = 4.0 * D * Hq * pairs * layers
    if case["kind"] == "full":
        return {"bytes": N * (2 * q_row + kv_row), "flops": flops}
    if case["kind"] == "question":
        return {"bytes": L_q * 2 * q_row + N * kv_row, "flops": flops}
    signal = SIGNAL_LAYERS * 2 * L_d * kv_row
    if case["kind"] == "select":
        return {"bytes": signal + 4 * (L_d + k) + k * 2 * q_row + k * 3 * kv_row + L_q * 2 * kv_row, "flops": 0}
    # fresh rows of the important and the question tokens, the offline document rows that stay, outputs
    fresh = (k + L_q) * (q_row + kv_row)
    cache = (L_d - k) * kv_row * (1.5 if case["kind"] == "fp8" else 1)
    out = (k + L_q) * (q_row + kv_row) + 4 * k
    scores = 0 if case["given"] or case["kind"] == "prefill" else 4 * case["n_sig"] * L_d
    total = (fresh + cache + out + scores) * layers
    if case["kind"] == "prefill":
        total += signal
    return {"bytes": total, "flops": flops}


def tolerance(case):
    """Positions and copied rows are exact; what is computed is bf16 attention rows or fp32 sums."""
    if case["kind"] == "select":
        # fp32 sums of 6 * Hkv * 128 squares: 4e-8 from the same sums in 64 bits; another order shows up to about 1e-7
        return {"rel": 4e-7, "differ": 0.0}
    # rows against softmax attention in 64 bits on the same inputs: rel 1.8e-3 to 2.4e-3 (P and the result are rounded
    # to bf16, the latter alone gives 1.6e-3), max 0.010 to 0.032
    return {"rel": 1e-2, "max": 0.13, "differ": 0.0}
