"""What this library is measured on: the work its users have it do, through its public entry points.

Kinds of cases, from the life of a model on this library:

  encode       offline weight encoder, one matrix (every matrix of a model once; all of them for each format of a search)
  join, split  exact bf16 matrix from speculation + verification data (what verification without a bf16 copy does before
               every projection), and the encoder of the verification data
  prefill      Engine.prefill: the prompt(s) through the target model
  kv_prompt    cass_kv_build_codebook: exponent codebooks and compressed records of the whole prompt, every layer
  kv_append    cass_kv_append: further tokens of one layer into both caches
  gemv         stand-alone draft GEMV, 1 to 8 vectors, both weight formats
  project      stand-alone verification projection, 1 to 64 rows
  attend       stand-alone draft attention over the compressed cache
  verify       one cass_verify call with its logits (what sampled decoding and scoring use)
  decode       one step of Engine.generate: gamma drafts, verification, acceptance, read-back (gamma = 0: plain greedy)
  sample       the sampled form of acceptance: two softmax calls and cass_accept_sampling

Weights are 0.02 x Student-t(4) with 1 % of the input channels x20, K and V are N(0, 1) with 2 % of K's channels x10.
Models are the benchmark's shapes with fewer layers, so that several fit one GPU; layers cost the same whatever their number.
"""
from __future__ import annotations

import math
import types

import torch

from paper_2605_26558_b200 import binding as B
from paper_2605_26558_b200 import engine

DEV = "cuda"
SHAPES = {
    "tiny": dict(hidden=256, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=688, vocab=1024),
    "llama8b": dict(hidden=4096, n_q_heads=32, n_kv_heads=8, head_dim=128, ffn=14336, vocab=128256),
    "qwen": dict(hidden=5120, n_q_heads=40, n_kv_heads=8, head_dim=128, ffn=13824, vocab=152064),
}
MATRIX_MAX = 28672 * 4096          # values of the largest matrix of a drawn case


def listed():
    return [
        # smallest projection of the tiny model: launch latency is all there is
        dict(name="gemv_tiny_gate_up", kind="gemv", rows=1376, cols=256, n_vec=1, mode=1, p=400, t=4),
        # the projection that holds most of an 8B layer, batch 1: the method's hot loop
        dict(name="gemv_8b_gate_up", kind="gemv", rows=28672, cols=4096, n_vec=1, mode=1, p=400, t=4),
        # low-batch serving with the other weight format, a projection with many column segments
        dict(name="gemv_mx_qwen_down_x8", kind="gemv", rows=5120, cols=13824, n_vec=8, mode=2, p=400, t=4),
        # verification of gamma + 1 = 5 rows, a small matrix of an 8B layer
        dict(name="project_8b_qkv_5rows", kind="project", n=6144, k=4096, rows=5),
        # one layer of an 8B model, middle of a reasoning-length decode
        dict(name="attend_8b_4k", kind="attend", heads="llama8b", positions=4095, batch=1, kv_mode=1),
        # a prompt becomes compressed cache before the first draft
        dict(name="kv_prompt_8b_2000", kind="kv_prompt", heads="llama8b", layers=2, tokens=2000, batch=1, kv_mode=1),
        # offline encoder on the widest rows of an 8B layer
        dict(name="encode_8b_down", kind="encode", rows=4096, cols=14336, mode=1, p=400, t=4),
        # rebuilding a projection for verification without a bf16 copy
        dict(name="join_8b_qkv", kind="join", rows=6144, cols=4096, p=400, t=4),
        # time to first token
        dict(name="prefill_8b_1000", kind="prefill", shape="llama8b", layers=4, tokens=1000, batch=1),
        # scoring pass of four sequences with their drafts
        dict(name="verify_qwen_4x5", kind="verify", shape="qwen", layers=2, context=2000, batch=4, gamma=4),
        # the headline: one speculative step at batch 1
        dict(name="decode_8b_gamma4", kind="decode", shape="llama8b", layers=8, context=1000, batch=1, gamma=4, mode=1,
             kv_mode=1, graph=True),
        # sampled acceptance of four sequences over an 8B model's vocabulary
        dict(name="sample_8b_4x5", kind="sample", vocab=128256, batch=4, gamma=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _matrix(rng):
    cols = _log_int(rng, 256, 14336)
    rows = _log_int(rng, 256, min(32768, MATRIX_MAX // cols))
    return rows, cols


def _model(rng):
    """A shape and its number of layers; the tiny model is drawn less often than the two that people serve."""
    shape = rng.choice(("tiny", "llama8b", "llama8b", "qwen"))
    return shape, (2 if shape == "tiny" else rng.randint(2, 4) if shape == "llama8b" else rng.randint(2, 3))


def draw(rng):
    kind = rng.choice(("gemv", "gemv", "project", "attend", "kv_prompt", "kv_append", "encode", "join", "split", "prefill",
                       "verify", "decode", "sample"))
    if kind == "gemv":
        rows, cols = _matrix(rng)
        mode = rng.choice((1, 1, 2))
        # the format search runs the unary format with every truncation from 0 to 5 bits; 4 is the default
        t = rng.choice((4, 4, 4, 0, 1, 2, 3, 5)) if mode == 1 else 4
        return dict(kind=kind, rows=rows, cols=cols, n_vec=rng.choice((1, 1, 1, 2, 4, 8)), mode=mode,
                    p=rng.choice((400, 400, 300, 500, 600)), t=t)
    if kind == "project":
        rows, cols = _matrix(rng)
        return dict(kind=kind, n=rows, k=max(256, cols // 8 * 8), rows=_log_int(rng, 1, 64))
    if kind == "attend":
        batch = rng.choice((1, 1, 2, 4, 8))
        return dict(kind=kind, heads=rng.choice(("tiny", "llama8b", "llama8b", "qwen")), positions=_log_int(rng, 64, 32000 // batch),
                    batch=batch, kv_mode=rng.choice((1, 1, 2)))
    if kind == "kv_prompt":
        batch = rng.choice((1, 1, 2, 4, 8))
        return dict(kind=kind, heads=rng.choice(("tiny", "llama8b", "qwen")), layers=rng.randint(1, 4),
                    tokens=_log_int(rng, 16, 4096 // batch), batch=batch, kv_mode=rng.choice((1, 1, 2)))
    if kind == "kv_append":
        return dict(kind=kind, heads=rng.choice(("tiny", "llama8b", "qwen")), start=_log_int(rng, 64, 4096),
                    tokens=_log_int(rng, 1, 2048), kv_mode=rng.choice((1, 1, 2)))
    if kind == "encode":
        rows, cols = _matrix(rng)
        return dict(kind=kind, rows=rows, cols=cols, mode=rng.choice((1, 1, 2)), p=rng.choice((400, 400, 300, 500, 600)), t=4)
    if kind in ("join", "split"):
        rows, cols = _matrix(rng)
        return dict(kind=kind, rows=rows, cols=cols, p=rng.choice((400, 400, 300, 500, 600)), t=rng.choice((4, 4, 4, 2, 3, 5)))
    if kind == "prefill":
        shape, layers = _model(rng)
        batch = rng.choice((1, 1, 2, 4, 8))
        return dict(kind=kind, shape=shape, layers=layers, tokens=_log_int(rng, 16, 1000 // batch), batch=batch)
    if kind == "sample":
        return dict(kind=kind, vocab=_log_int(rng, 1024, 152064), batch=rng.randint(1, 8), gamma=rng.randint(1, 7))
    shape, layers = _model(rng)
    batch = rng.choice((1, 1, 1, 2, 4, 8))
    gamma = rng.choice((2, 4, 4, 6)) if kind == "decode" else rng.choice((0, 2, 4, 6))
    case = dict(kind=kind, shape=shape, layers=layers, context=_log_int(rng, 64, 8192 // batch), batch=batch, gamma=gamma)
    if kind == "decode":
        if rng.random() < 0.25:
            case["gamma"] = 0          # plain greedy decoding
        case.update(mode=rng.choice((1, 1, 2)), kv_mode=rng.choice((1, 1, 2)), graph=rng.choice((True, True, False)))
    return case


# ---- inputs ----------------------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _normal(g, *size):
    return torch.randn(*size, generator=g, device=DEV, dtype=torch.float32)


def _weight(g, rows, cols):
    """bf16 [rows][cols]: 0.02 x Student-t with 4 degrees of freedom, 1 % of the columns x20."""
    w = _normal(g, rows, cols)
    chi2 = _normal(g, rows, cols).square_()
    for _ in range(3):
        n = _normal(g, rows, cols)
        chi2.addcmul_(n, n)
    w.div_(chi2.mul_(0.25).sqrt_()).mul_(0.02)
    w[:, torch.randperm(cols, generator=g, device=DEV)[: max(1, cols // 100)]] *= 20.0
    return w.to(torch.bfloat16)


def _kv(g, tokens, heads, dim):
    k, v = _normal(g, tokens, heads, dim), _normal(g, tokens, heads, dim)
    k[:, :, torch.randperm(dim, generator=g, device=DEV)[: max(1, dim // 50)]] *= 10.0
    return k.to(torch.bfloat16), v.to(torch.bfloat16)


def _i32(n=1):
    return torch.zeros(n, dtype=torch.int32, device=DEV)


def _bytes(n):
    return torch.zeros(n, dtype=torch.uint8, device=DEV)


def _encoded(g, rows, cols, fmt):
    """A matrix, its calibration norms, and the buffers that the encoder takes, blob made."""
    w = _weight(g, rows, cols)
    act = _normal(g, cols).abs_().add_(0.5)
    bound, ws_bytes = B.cass_encoded_weight_bytes(fmt, rows, cols)
    s = types.SimpleNamespace(fmt=fmt, w=w, act=act, blob=_bytes(bound), ws=_bytes(ws_bytes), status=_i32())
    B.cass_encode_weights(fmt, w, act, s.blob, s.ws, s.status)
    s.info = B.cass_weight_blob_info(s.blob)
    return s


def _engine(g, shape, layers, context, batch, gamma, fmt):
    """An engine of that shape whose caches hold `context` positions of every layer and sequence."""
    wt = {"layers": []}
    h, d = shape.hidden, shape.head_dim
    ones = torch.ones(h, dtype=torch.bfloat16, device=DEV)
    for _ in range(layers):
        wt["layers"].append(dict(wqkv=_weight(g, (shape.n_q_heads + 2 * shape.n_kv_heads) * d, h), wo=_weight(g, h, shape.n_q_heads * d),
                                 wgu=_weight(g, 2 * shape.ffn, h), wd=_weight(g, h, shape.ffn), norm_attn=ones, norm_ffn=ones))
    wt.update(embed=_weight(g, shape.vocab, h), lm_head=_weight(g, shape.vocab, h), norm_final=ones)
    max_seq = (context + 64 + 255) // 256 * 256
    return engine.Engine(shape, wt, fmt=fmt, max_seq=max_seq, gamma_max=max(gamma, 1), batch=batch)


def _fill(g, eng, tokens):
    """`tokens` synthetic positions in both caches of every layer and sequence; codebooks from the first of them."""
    s, first = eng.shape, min(tokens, 512)
    rest = []
    for layer in range(s.n_layers):
        for b in range(eng.batch):
            k, v = _kv(g, tokens, s.n_kv_heads, s.head_dim)
            B.cass_kv_append(eng.session, layer, k, v, 0, tokens, B.KV_BF16, seq=b)
            rest.append((layer, b, k[first:], v[first:]))
    B.cass_kv_build_codebook(eng.session, first)
    for layer, b, k, v in rest:
        if tokens > first:
            B.cass_kv_append(eng.session, layer, k, v, first, tokens - first, B.KV_COMPRESSED, seq=b)
    B.cass_set_len(eng.session, tokens)


def _shape(name, layers):
    return types.SimpleNamespace(n_layers=layers, rope_theta=1e4, rms_eps=1e-5, **SHAPES[name])


def _kv_engine(g, heads, layers, tokens, batch, kv_mode):
    """An engine with the heads of that shape and next to no weights: what the KV entry points need."""
    shape = _shape(heads, layers)
    shape.hidden, shape.ffn, shape.vocab = 256, 256, 256
    return _engine(g, shape, layers, tokens, batch, 4, B.default_format(kv_mode=kv_mode))


def _view(eng, ptr, n, dtype=torch.int32):
    """The n elements that a cass_kv_query pointer leads to, as a view of the session's memory."""
    o, size = ptr - eng.mem.data_ptr(), torch.empty(0, dtype=dtype).element_size()
    return eng.mem[o: o + n * size].view(dtype)


def _records(eng, layers, batch):
    """The compressed caches of some layers and sequences: fixed parts, exponent arenas, offsets, codebooks."""
    out, s, seq_len = [], eng.shape, eng.desc.max_seq
    for layer in layers:
        for b in batch:
            for kind in (0, 1):
                v = B.cass_kv_query(eng.session, layer, kind, 0, seq=b)
                out += [_view(eng, v.fixed, s.n_kv_heads * ((seq_len + 31) // 32) * v.fixed_words_per_token * 32),
                        _view(eng, v.arena, s.n_kv_heads * v.arena_words), _view(eng, v.offsets, s.n_kv_heads * (seq_len + 1)),
                        _view(eng, v.codebook, 256, torch.uint8)]
    return out


def _cache_rows(eng, layers, batch, lo, hi):
    """Positions lo..hi-1 of the bf16 caches of some layers and sequences."""
    row, out = eng.shape.n_kv_heads * eng.shape.head_dim, []
    for layer in layers:
        for b in batch:
            for kind in (0, 1):
                v = B.cass_kv_query(eng.session, layer, kind, 0, seq=b)
                out.append(_view(eng, v.k_or_v_bf16, hi * row, torch.bfloat16)[lo * row:])
    return out


def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    if kind == "encode":
        # the encoder's user holds the matrix and buffers of the sizes that the library names; the blob is not made yet
        fmt = B.default_format(w_p=case["p"], w_t=case["t"], mode=case["mode"])
        bound, ws_bytes = B.cass_encoded_weight_bytes(fmt, case["rows"], case["cols"])
        s = types.SimpleNamespace(fmt=fmt, w=_weight(g, case["rows"], case["cols"]), act=_normal(g, case["cols"]).abs_().add_(0.5),
                                  blob=_bytes(bound), ws=_bytes(ws_bytes), status=_i32())
    elif kind in ("join", "split"):
        s = _encoded(g, case["rows"], case["cols"], B.default_format(w_p=case["p"], w_t=case["t"]))
        s.vdata = _bytes(B.cass_verification_data_bytes(s.info))
        if kind == "join":
            B.cass_encode_verification_data(s.blob, s.info, s.w, s.vdata)
            s.out = torch.zeros_like(s.w)
    elif kind == "gemv":
        s = _encoded(g, case["rows"], case["cols"], B.default_format(w_p=case["p"], w_t=case["t"], mode=case["mode"]))
        s.x = _normal(g, case["n_vec"], case["cols"]).to(torch.bfloat16)
        s.partial = torch.zeros(case["n_vec"] * s.info.n_seg * s.info.n_rowblocks * 32, device=DEV)
        s.y = torch.zeros(case["n_vec"], case["rows"], device=DEV)
        s.w = s.act = s.ws = None
    elif kind == "project":
        n, k, rows = case["n"], case["k"], case["rows"]
        s = types.SimpleNamespace(w=_weight(g, n, k), status=_i32(), scratch=_bytes(B.cass_verify_gemm_scratch_bytes(n, k)),
                                  x=_normal(g, 16 if rows <= 16 else 32 if rows <= 32 else 64, k).to(torch.bfloat16),
                                  y=torch.zeros(rows, n, device=DEV))
    elif kind == "sample":
        v, b, gm = case["vocab"], case["batch"], case["gamma"]
        # logits spread as a trained model's are: most of the probability on some hundred tokens; the draft is the target, disturbed
        p = _normal(g, b, gm + 1, v).mul_(3.0)
        q = p[:, :gm].add(_normal(g, b, gm, v)).contiguous()
        drawn = torch.multinomial(torch.softmax(q.view(b * gm, v), dim=1), 1, generator=g).to(torch.int32).view(b, gm)
        rand = lambda *n: torch.rand(*n, generator=g, device=DEV)  # noqa: E731
        s = types.SimpleNamespace(p_logits=p, q_logits=q, p=torch.zeros_like(p), q=torch.zeros_like(q), drafts=drawn, r=rand(b, gm),
                                  u=rand(b), n_acc=_i32(b), out=_i32(b * (gm + 1)), nxt=_i32(b))
    elif kind in ("attend", "kv_prompt", "kv_append"):
        heads, batch = case["heads"], case.get("batch", 1)
        total = case["positions"] + 1 if kind == "attend" else case["tokens"] if kind == "kv_prompt" else case["start"] + case["tokens"]
        eng = _kv_engine(g, heads, case.get("layers", 1), total, batch, case["kv_mode"])
        s, sh = types.SimpleNamespace(eng=eng), eng.shape
        if kind == "kv_prompt":
            for layer in range(sh.n_layers):
                for b in range(batch):
                    B.cass_kv_append(eng.session, layer, *_kv(g, total, sh.n_kv_heads, sh.head_dim), 0, total, B.KV_BF16, seq=b)
            eng.n_prompt = total
            s.out = _records(eng, range(sh.n_layers)[-2:], range(batch)[-2:])
        elif kind == "kv_append":
            _fill(g, eng, case["start"])
            s.k, s.v = _kv(g, case["tokens"], sh.n_kv_heads, sh.head_dim)
            s.out = _records(eng, (0,), (0,)) + _cache_rows(eng, (0,), (0,), case["start"], total)
        else:
            _fill(g, eng, total)
            B.cass_set_len(eng.session, case["positions"])
            s.q = _normal(g, batch, sh.n_q_heads, sh.head_dim).to(torch.bfloat16)
            s.o = torch.zeros_like(s.q)
    elif kind == "prefill":
        eng = _engine(g, _shape(case["shape"], case["layers"]), case["layers"], case["tokens"], case["batch"], 4, B.default_format())
        s = types.SimpleNamespace(eng=eng, prompt=torch.randint(0, eng.shape.vocab, (case["batch"], case["tokens"]), generator=g,
                                                               device=DEV, dtype=torch.int32))
        s.out = _cache_rows(eng, range(case["layers"]), range(case["batch"])[-2:], 0, case["tokens"])
    else:
        fmt = B.default_format(mode=case.get("mode", 1), kv_mode=case.get("kv_mode", 1))
        eng = _engine(g, _shape(case["shape"], case["layers"]), case["layers"], case["context"], case["batch"], case["gamma"], fmt)
        _fill(g, eng, case["context"])
        n = case["batch"] * (case["gamma"] + 1)
        s = types.SimpleNamespace(eng=eng, toks=torch.randint(0, eng.shape.vocab, (n,), generator=g, device=DEV, dtype=torch.int32))
        if kind == "verify":
            s.targ, s.logits = _i32(n), torch.zeros(n, eng.shape.vocab, device=DEV)
            s.out = _cache_rows(eng, range(case["layers"]), range(case["batch"])[-2:], case["context"], case["context"] + case["gamma"] + 1)
        else:
            s.first = s.toks[: case["batch"]].clone()
            eng.encode_weights(None)
            eng.generate(0, case["gamma"], use_graph=case["graph"])
            # of the rows that a step writes, the first alone does not depend on what was drafted
            s.out = _cache_rows(eng, range(case["layers"]), range(case["batch"])[-2:], case["context"], case["context"] + 1)
    s.case = case
    return s


# ---- one pass --------------------------------------------------------------------------------------------------------

def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "encode":
        B.cass_encode_weights(s.fmt, s.w, s.act, s.blob, s.ws, s.status)
        return s.blob
    if kind == "join":
        B.cass_decode_full(s.blob, s.info, s.vdata, s.out)
        return s.out
    if kind == "split":
        B.cass_encode_verification_data(s.blob, s.info, s.w, s.vdata)
        return s.vdata
    if kind == "gemv":
        if case["n_vec"] == 1:
            B.cass_draft_gemv(s.blob, s.info, s.x, s.partial, None, s.y, s.status)
        else:
            B.cass_draft_gemv_batch(s.blob, s.info, s.x, case["n_vec"], s.partial, None, s.y, s.status)
        return s.y
    if kind == "project":
        B.cass_verify_gemm(s.w, s.x, case["rows"], s.scratch, None, s.y, s.status)
        return s.y
    if kind == "attend":
        B.cass_draft_attention(s.eng.session, 0, s.q, s.o)
        return s.o
    if kind == "kv_prompt":
        s.eng.build_kv_codebook()
        return s.out
    if kind == "kv_append":
        B.cass_kv_append(s.eng.session, 0, s.k, s.v, case["start"], case["tokens"], B.KV_BF16 | B.KV_COMPRESSED)
        return s.out
    if kind == "prefill":
        return s.eng.prefill(s.prompt), s.out
    if kind == "verify":
        B.cass_verify(s.eng.session, s.toks, case["gamma"], s.targ, s.logits)
        return s.logits, s.out
    if kind == "sample":
        b, gm, v = case["batch"], case["gamma"], case["vocab"]
        B.cass_softmax(s.p_logits, b * (gm + 1), v, 1.0, s.p)
        B.cass_softmax(s.q_logits, b * gm, v, 1.0, s.q)
        B.cass_accept_sampling(None, b, s.drafts, s.p, s.q, v, s.r, s.u, gm, s.n_acc, s.out, s.nxt)
        return s.p, s.q, s.n_acc, s.out, s.nxt
    # every pass rolls back to the same context and decodes one step from there, as a server does with a new request
    # that shares a prompt
    B.cass_set_len(s.eng.session, case["context"])
    s.eng.set_next_tokens(s.first)
    s.eng.generate(1, case["gamma"], use_graph=case["graph"])
    return s.eng.out_tokens[: s.toks.numel()], s.eng.n_acc[: case["batch"]], s.out


# ---- what a pass cannot do without -----------------------------------------------------------------------------------

def _spec_bytes(values, p=400, t=4, mode=1):
    """Speculation data of that many weights: a bitmap bit each, and per kept one a field and about 1.9 code bits
    (Cassandra-2: a 32nd of an exponent byte)."""
    return values * (1 + (1 - p / 1000) * (8 - t + (1.9 if mode == 1 else 0.25))) / 8


def _kv_bytes(positions, sh, kv_mode):
    """Compressed K and V records of one layer: bitmap, fields, about 1.9 code bits or a 32nd of an exponent byte each."""
    return 2 * positions * sh.n_kv_heads * sh.head_dim * (1 + 0.6 * 4 + (0.6 * 1.9 if kv_mode == 1 else 0.25)) / 8


def _weights(sh):
    d = sh.head_dim
    layer = sh.hidden * ((sh.n_q_heads + 2 * sh.n_kv_heads) * d + sh.n_q_heads * d + 3 * sh.ffn)
    return sh.n_layers * layer, sh.vocab * sh.hidden


def _target_pass(sh, batch, rows, context, logit_rows):
    """Bytes and operations of the target model over `rows` rows of each sequence behind `context` positions."""
    layers, head = _weights(sh)
    kv_row = 2 * sh.n_layers * sh.n_kv_heads * sh.head_dim * 2
    seen = rows * context + rows * (rows + 1) / 2
    return dict(bytes=2 * (layers + head) + batch * (context + rows) * kv_row,
                flops=2 * batch * (rows * layers + logit_rows * head) + 4 * batch * seen * sh.n_layers * sh.n_q_heads * sh.head_dim)


def work(case):
    kind = case["kind"]
    if kind in ("encode", "join", "split", "gemv"):
        values, p, t = case["rows"] * case["cols"], case["p"], case["t"]
        spec, kept = _spec_bytes(values, p, t, case.get("mode", 1)), (1 - p / 1000) * values
        rest = kept * t / 8 + 2 * (values - kept)
        if kind == "encode":
            return dict(bytes=2 * values + spec, flops=values)
        if kind == "split":
            return dict(bytes=2 * values + values / 8 + rest, flops=0)
        if kind == "join":
            return dict(bytes=2 * values + spec + rest, flops=0)
        return dict(bytes=spec + case["n_vec"] * (2 * case["cols"] + 4 * case["rows"]), flops=2 * kept * case["n_vec"])
    if kind == "project":
        return dict(bytes=2 * case["n"] * case["k"] + case["rows"] * (2 * case["k"] + 4 * case["n"]), flops=2 * case["n"] * case["k"] * case["rows"])
    if kind == "sample":
        values = case["vocab"] * case["batch"] * (2 * case["gamma"] + 1)
        return dict(bytes=8 * values + 8 * case["vocab"] * case["batch"], flops=4 * values)
    if kind in ("attend", "kv_prompt", "kv_append"):
        sh, batch = _shape(case["heads"], case.get("layers", 1)), case.get("batch", 1)
        row = 2 * 2 * sh.n_kv_heads * sh.head_dim
        if kind == "attend":
            n = batch * (case["positions"] + 1)
            return dict(bytes=_kv_bytes(n, sh, case["kv_mode"]) + batch * 4 * sh.n_q_heads * sh.head_dim, flops=4 * n * sh.n_q_heads * sh.head_dim)
        n = batch * sh.n_layers * case["tokens"]
        return dict(bytes=n * row * (1 if kind == "kv_prompt" else 2) + _kv_bytes(n, sh, case["kv_mode"]), flops=n * row / 2)
    sh = _shape(case["shape"], case["layers"])
    if kind == "prefill":
        return _target_pass(sh, case["batch"], case["tokens"], 0, 1)
    w = _target_pass(sh, case["batch"], case["gamma"] + 1, case["context"], case["gamma"] + 1)
    if kind == "verify":
        w["bytes"] += 4 * case["batch"] * (case["gamma"] + 1) * sh.vocab
        return w
    layers, head = _weights(sh)
    for i in range(case["gamma"]):
        seen = case["batch"] * (case["context"] + i + 1)
        w["bytes"] += _spec_bytes(layers + head, mode=case["mode"]) + sh.n_layers * _kv_bytes(seen, sh, case["kv_mode"])
        w["flops"] += 2 * 0.6 * case["batch"] * (layers + head) + 4 * seen * sh.n_layers * sh.n_q_heads * sh.head_dim
    return w


def tolerance(case):
    kind = case["kind"]
    if kind in ("gemv", "project"):
        return {"rel": 1e-5}                                   # exact products of bf16 values, 32-bit sums
    if kind == "attend":
        return {"rel": 5e-3, "max": 2e-2}                      # bf16 results
    if kind in ("prefill", "verify", "decode"):
        # bf16 activations between operators: one that rounds the other way moves a layer's output through an outlier
        # column by some per cent of its size at worst
        return {"rel": 1e-2, "max": 0.3}
    if kind == "sample":
        return {"rel": 1e-5}                                   # 32-bit sums over the vocabulary
    return "exact"
