"""Performance cases of the dynamic-vocabulary path, through the public binding.

A case is one call sequence that a serving or scoring program makes over and over:

  step      one decode step of a batch (joint logits, selection, codebook update, hyper-encoder for
            both caches).  A session decodes ``steps`` tokens; then the program takes up the next
            request on the same prompts: the codebook is rebuilt from the prompts' codes
            (decompression), the cache rows of the prompts' entries are still there.
  filtered  the same step with top-k / top-p sampling: stored logits, filtered sample, codebook
            update, hyper-encoder, next input embedding as calls of their own.
  start     a request's prompts: compression, hyper-embedding of every entry for both caches, input
            embeddings of the compressed prompts.
  score     the same and then the joint logits at every compressed position with the logit of the
            position's next code (negative log-likelihood of a prompt batch).
  rows      joint logits for a chunk of compressed positions under causal visibility.
  text      compression of texts and decompression of the codes back into base tokens.

Shapes are those of ``synth_inputs.WORKLOADS`` or lie around them.  Token streams come from
``synth_inputs.token_stream``; weights are N(0, 0.02), gains about 1, hidden states N(0, 1), drawn on
the GPU from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2506_01084_b200 import binding as zb
from paper_2506_01084_b200 import synth_inputs as si

PHI3 = dict(V=32064, d=3072, dtype="bf16", M=3, zipf=1.1, copy_p=0.3, seg_min=4, seg_max=16)
LLAMA3 = dict(V=128256, d=4096, dtype="bf16", M=3, zipf=1.2, copy_p=0.4, seg_min=4, seg_max=32)
LONG = dict(V=128256, d=4096, dtype="bf16", M=5, zipf=1.0, copy_p=0.6, seg_min=8, seg_max=64)
TINY = dict(V=512, d=64, dtype="fp32", M=3, zipf=1.1, copy_p=0.3, seg_min=4, seg_max=16)
STEP = dict(kind="step", steps=256, select="argmax", tied=False, ffn=True, next_embed=True, finished=False)
HIDDEN_BANK = 64          # blocks of hidden rows a decode session cycles through


def listed():
    return [
        # the fp32 parity configuration: the smallest call there is, launches and host time count
        dict(STEP, name="step_tiny_fp32", **TINY, B=1, T=256, cap=256, steps=64),
        # one user at a terminal: a single sequence, a small head, sampled
        dict(STEP, name="step_one_user", **PHI3, B=1, T=600, cap=2048, select="gumbel"),
        # the small decode configuration of the benchmark
        dict(STEP, name="step_phi3_b8", **PHI3, B=8, T=2048, cap=2048, next_embed=False),
        # the ordinary serving batch: the benchmark's default workload
        dict(STEP, name="step_llama3_b32", **LLAMA3, B=32, T=4096, cap=4096, steps=512, next_embed=False),
        # long repetitive contexts, ragged codebooks, longer entries, sampled
        dict(STEP, name="step_long_b4", **LONG, B=4, T=32768, cap=16384, steps=512, select="gumbel"),
        # a throughput batch beyond the decode kernel's 32 rows, one table for both sides, an eighth of
        # the sequences already finished
        dict(STEP, name="step_tied_b90", **PHI3, B=90, T=500, cap=1024, tied=True, finished=True),
        # sampling as chat services configure it: top-k and nucleus on stored logits
        dict(kind="filtered", name="filtered_b16", **LLAMA3, B=16, T=512, cap=1024, steps=256, top_k=50, top_p=0.9),
        # time to first token of one short request
        dict(kind="start", name="start_short", **PHI3, B=1, T=333, cap=2048),
        # prompts of the small configuration arriving together
        dict(kind="start", name="start_phi3_b8", **PHI3, B=8, T=2048, cap=2048),
        # a chunk of positions to be scored (chunked evaluation, verification of drafted codes)
        dict(kind="rows", name="rows_700", **LLAMA3, B=5, N=700, cap=4096),
        # 16 of the prompts of the prompt-scoring configuration, fp16 weight copies lent
        dict(kind="score", name="score_16_prompts", **dict(LLAMA3, M=4), B=16, T=8192, cap=8192, half=True),
        # long texts through compression and back
        dict(kind="text", name="text_long_b4", **LONG, B=4, T=32768, cap=16384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: vocabulary and width from small models to the largest table, batch
    sizes over their logarithm, any prompt length."""
    kind = rng.choice(["step", "step", "step", "filtered", "start", "start", "rows", "score", "text"])
    copy_p = round(rng.uniform(0.2, 0.6), 2)
    seg_min = rng.randint(3, 8)
    c = dict(kind=kind, V=_log_int(rng, 4000, 128256), d=128 * rng.randint(8, 32), dtype="bf16", M=rng.randint(2, 5),
             zipf=round(rng.uniform(1.0, 1.3), 2), copy_p=copy_p, seg_min=seg_min, seg_max=seg_min * rng.randint(2, 8))
    if kind == "step":
        c.update(STEP, B=_log_int(rng, 1, 128), T=_log_int(rng, 64, 2048), cap=rng.choice([1024, 2048, 3000]),
                 select=rng.choice(["argmax", "gumbel"]), tied=rng.random() < 0.3, ffn=rng.random() < 0.85,
                 next_embed=rng.random() < 0.5, finished=rng.random() < 0.2)
        if rng.random() < 0.15:
            c.update(dtype="fp32", V=_log_int(rng, 256, 2048), d=8 * rng.randint(5, 16), B=rng.randint(1, 4),
                     T=_log_int(rng, 64, 512), cap=512, steps=64)
    elif kind == "filtered":
        c.update(B=_log_int(rng, 1, 32), T=_log_int(rng, 64, 512), cap=1024, steps=256,
                 top_k=rng.choice([0, 20, 50, 200]), top_p=rng.choice([1.0, 0.95, 0.9, 0.8]))
    elif kind == "start":
        c.update(B=_log_int(rng, 1, 16), T=_log_int(rng, 40, 2048), cap=2048)
    elif kind == "rows":
        c.update(M=rng.randint(2, 4), B=_log_int(rng, 1, 16), N=_log_int(rng, 33, 2600), cap=4096)
    elif kind == "score":
        c.update(M=rng.randint(2, 4), B=_log_int(rng, 2, 16), T=_log_int(rng, 512, 6000), cap=4096, half=rng.random() < 0.5)
    else:
        c.update(B=_log_int(rng, 1, 64), cap=rng.choice([1024, 4096, 8192, 16384]))
        c["T"] = min(_log_int(rng, 200, 32768), 131072 // c["B"])
    return c


# ---- inputs ------------------------------------------------------------------------------------
def _dtype(case):
    return torch.float32 if case["dtype"] == "fp32" else torch.bfloat16


def _heads(case):
    return case["d"] // 128 if case["d"] >= 128 and case["d"] % 128 == 0 else 4 if case["d"] % 16 == 0 else 2


def _dff(case):
    return 4 * case["d"] if case.get("ffn", True) else 0


def _layers():
    return 2


def _tokens(case, B, T, seed):
    return np.stack([si.token_stream(case["V"], T, case["zipf"], case["copy_p"], case["seg_min"], case["seg_max"],
                                     seed * 1000003 + b) for b in range(B)])


class _Draw:
    """Values of one seed, drawn on the GPU in fp32 and rounded to the storage type."""

    def __init__(self, case, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))
        self.dt = _dtype(case)

    def normal(self, shape, std, mean=0.0):
        out = torch.empty(shape, dtype=self.dt, device="cuda")
        flat = out.view(-1)
        for i in range(0, flat.numel(), 1 << 27):
            n = min(1 << 27, flat.numel() - i)
            flat[i:i + n] = torch.randn(n, generator=self.g, device="cuda") * std + mean
        return out

    def encoder(self, case):
        d, dff = case["d"], _dff(case)
        t = [self.normal((case["M"], d), 0.02)]
        for _ in range(_layers()):
            t += [self.normal((d,), 0.1, 1.0), self.normal((d,), 0.05)]
            t += [self.normal((3 * d, d), 0.02), self.normal((3 * d,), 0.05), self.normal((d, d), 0.02), self.normal((d,), 0.05)]
            t += [self.normal((d,), 0.1, 1.0), self.normal((d,), 0.05)]
            w = max(dff, 8)                                    # attention-only layers ignore the last slots
            t += [self.normal((w, d), 0.02), self.normal((w,), 0.05), self.normal((d, w), 0.02), self.normal((d,), 0.05)]
        return zb.encoder_weights(t)


class _Session:
    """Model side (tables, encoders), codebook handle, caches and prompts of one program."""

    def __init__(self, case, seed, T, encoders=True):
        B, cap, d = case["B"], case["cap"], case["d"]
        r = _Draw(case, seed)
        self.case, self.seed, self.draw, self.T = case, seed, r, T
        self.tied = bool(case.get("tied", False))
        self.cb = zb.Codebook(zb.make_config(case["V"], d, case["M"], cap, B, case["dtype"], _layers(), _heads(case),
                                             _dff(case), int(self.tied)))
        self.tok = torch.from_numpy(_tokens(case, B, T, seed)).cuda()
        self.codes = torch.zeros(B, T, dtype=torch.int32, device="cuda")
        self.clen = torch.zeros(B, dtype=torch.int32, device="cuda")
        if encoders:
            self.W_E = r.normal((case["V"], d), 0.02)
            self.W_U = self.W_E if self.tied else r.normal((case["V"], d), 0.02)
            self.enc_E = r.encoder(case)
            self.enc_U = self.enc_E if self.tied else r.encoder(case)
            self.E_h = torch.zeros(B, cap, d, dtype=r.dt, device="cuda")
            self.U_h = self.E_h if self.tied else torch.zeros_like(self.E_h)

    def encode(self, after=None):
        zb.z2z_lzw_encode(self.cb, self.tok, None, self.codes, self.clen, after)

    def embed(self):
        zb.z2z_hyper_embed(self.cb, zb.CACHE_EMBED, self.W_E, self.enc_E, None, None, -1, self.E_h, None)
        if not self.tied:
            zb.z2z_hyper_embed(self.cb, zb.CACHE_UNEMBED, self.W_U, self.enc_U, None, None, -1, self.U_h, None)

    def caches(self):
        return {"E_h": self.E_h} if self.tied else {"E_h": self.E_h, "U_h": self.U_h}

    def positions(self):
        """(sequence, index) of every compressed position, in order."""
        lens = self.clen.cpu().to(torch.int64)
        seq = torch.repeat_interleave(torch.arange(len(lens)), lens)
        start = torch.cumsum(lens, 0) - lens
        return seq.cuda(), (torch.arange(len(seq)) - start[seq]).cuda()


def _i32(*shape, fill=0):
    return torch.full(shape, fill, dtype=torch.int32, device="cuda")


def _f32(*shape):
    return torch.zeros(*shape, dtype=torch.float32, device="cuda")


def prepare(case, seed):
    kind, B, d = case["kind"], case["B"], case["d"]
    if kind == "rows":
        s = _Session(case, seed, 4 * -(-case["N"] // B) + 64)
        after = torch.zeros_like(s.codes)
        s.encode(after)
        s.embed()
        seq, idx = s.positions()
        share = [case["N"] * (b + 1) // B - case["N"] * b // B for b in range(B)]        # the last positions of each
        keep = torch.cat([(seq == b).nonzero().view(-1)[-n:] if n else seq.new_zeros(0) for b, n in enumerate(share)])
        seq, idx = seq[keep], idx[keep]
        s.row_seq = seq.to(torch.int32)
        s.nvis = after[seq, idx].contiguous()
        s.targets = s.codes[seq, (idx + 1).clamp(max=s.T - 1)].contiguous()
        _rows_out(s, case["N"])
        return s
    s = _Session(case, seed, case["T"], encoders=kind != "text")
    s.encode()
    if kind == "text":
        s.out_tok = torch.zeros_like(s.tok)
        s.out_len = _i32(B)
        return s
    if kind in ("start", "score"):
        seq, idx = s.positions()
        s.row_seq = seq.to(torch.int32)
        if kind == "start":
            s.flat = seq * s.T + idx
            s.x = torch.zeros(B * s.T, d, dtype=s.draw.dt, device="cuda")       # room for any number of codes
            return s
        s.flat_next = seq * s.T + (idx + 1).clamp(max=s.T - 1)
        _rows_out(s, len(seq), B * s.T)
        if case["half"]:
            n = zb.encoder_half_bytes(s.cb.cfg)
            buf = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
            zb.z2z_set_encoder_half_scratch(s.cb, buf[(-buf.data_ptr()) % 256:][:n])
        return s
    s.embed()
    s.prompt_codes, s.prompt_lens = s.codes.clone(), s.clen.clone()
    s.replayed, s.replayed_len = torch.zeros_like(s.tok), _i32(B)
    s.n_prompt = zb.z2z_status(s.cb)[1].cuda()
    s.hidden = s.draw.normal((HIDDEN_BANK, B, d), 1.0)
    s.at = 0
    s.next_codes, s.new_entry = _i32(B), _i32(B)
    s.x = torch.zeros(B, d, dtype=s.draw.dt, device="cuda")
    if kind == "step":
        s.lse, s.selected = _f32(B), _i32(B)
        s.forced = None
        if case["finished"]:
            s.forced = _i32(B, fill=zb.CODE_SELECTED)
            s.forced[3::8] = zb.CODE_NONE
    else:
        s.n = s.n_prompt.clone()
        s.logits = _f32(B, case["V"] + case["cap"])
        s.lse, s.argmax, s.maxl = _f32(B), _i32(B), _f32(B)
    return s


def _rows_out(s, N, room=0):
    n = max(N, room)
    s.hidden = s.draw.normal((N, s.case["d"]), 1.0)
    s.lse, s.argmax, s.maxl, s.tlogit = _f32(n), _i32(n), _f32(n), _f32(n)


# ---- one pass ------------------------------------------------------------------------------------
def _next_request(s):
    """After ``steps`` steps: a new session on the same prompts, rebuilt from their codes."""
    zb.z2z_codebook_init(s.cb)
    zb.z2z_lzw_decode(s.cb, s.prompt_codes, s.prompt_lens, zb.DECODE_REPLAY, s.replayed, s.replayed_len)


def _run_step(s):
    c = s.case
    if s.at and s.at % c["steps"] == 0:
        _next_request(s)
    zb.z2z_decode_step(s.cb, s.hidden[s.at % HIDDEN_BANK], s.W_E, s.W_U, s.enc_E, s.enc_U, s.E_h, s.U_h,
                       zb.SELECT_GUMBEL if c["select"] == "gumbel" else zb.SELECT_ARGMAX, 0.8, s.seed, s.at, s.forced,
                       s.next_codes, s.selected, s.lse, s.new_entry, None, None, s.x if c["next_embed"] else None)
    s.at += 1
    out = {"next": s.next_codes, "selected": s.selected, "lse": s.lse, "entry": s.new_entry, **s.caches()}
    if c["next_embed"]:
        out["x"] = s.x
    return out


def _run_filtered(s):
    c = s.case
    if s.at and s.at % c["steps"] == 0:
        _next_request(s)
        s.n = s.n_prompt.clone()
    zb.z2z_dynamic_logits(s.cb, s.hidden[s.at % HIDDEN_BANK], None, None, s.W_U, s.U_h, zb.SELECT_ARGMAX, 1.0, 0, 0, None,
                          s.lse, s.argmax, s.maxl, logits_debug=s.logits)
    zb.z2z_sample_filtered(s.logits, s.n + c["V"], c["top_k"], c["top_p"], 0.8, s.seed, s.at, s.next_codes)
    zb.z2z_lzw_step(s.cb, s.next_codes, None, s.new_entry)
    made = (s.new_entry >= 0).to(torch.int32)
    zb.z2z_hyper_embed(s.cb, zb.CACHE_EMBED, s.W_E, s.enc_E, s.n, made, c["B"], s.E_h, None)
    zb.z2z_hyper_embed(s.cb, zb.CACHE_UNEMBED, s.W_U, s.enc_U, s.n, made, c["B"], s.U_h, None)
    s.n = s.n + made
    zb.z2z_embed_lookup(s.cb, s.next_codes, None, s.W_E, s.E_h, s.x)
    s.at += 1
    return {"next": s.next_codes, "entry": s.new_entry, "logits": s.logits, "lse": s.lse, "argmax": s.argmax, "x": s.x,
            **s.caches()}


def _run_start(s):
    zb.z2z_codebook_init(s.cb)
    s.encode()
    s.embed()
    zb.z2z_embed_lookup(s.cb, s.codes.view(-1)[s.flat], s.row_seq, s.W_E, s.E_h, s.x[:len(s.flat)])
    return {"codes": s.codes, "lens": s.clen, "x": s.x, **s.caches()}


def _run_score(s):
    zb.z2z_codebook_init(s.cb)
    s.encode()
    s.embed()
    targets = s.codes.view(-1)[s.flat_next]
    zb.z2z_dynamic_logits(s.cb, s.hidden, s.row_seq, None, s.W_U, s.U_h, zb.SELECT_ARGMAX, 1.0, 0, 0, targets, s.lse,
                          s.argmax, s.maxl, None, s.tlogit)
    return {"codes": s.codes, "lens": s.clen, "lse": s.lse, "argmax": s.argmax, "max": s.maxl, "target": s.tlogit,
            **s.caches()}


def _run_rows(s):
    zb.z2z_dynamic_logits(s.cb, s.hidden, s.row_seq, s.nvis, s.W_U, s.U_h, zb.SELECT_ARGMAX, 1.0, 0, 0, s.targets, s.lse,
                          s.argmax, s.maxl, None, s.tlogit)
    return {"lse": s.lse, "argmax": s.argmax, "max": s.maxl, "target": s.tlogit}


def _run_text(s):
    zb.z2z_codebook_init(s.cb)
    s.encode()
    zb.z2z_codebook_init(s.cb)
    zb.z2z_lzw_decode(s.cb, s.codes, s.clen, zb.DECODE_REPLAY, s.out_tok, s.out_len)
    return {"codes": s.codes, "lens": s.clen, "tokens": s.out_tok, "token_lens": s.out_len}


_RUN = {"step": _run_step, "filtered": _run_filtered, "start": _run_start, "score": _run_score, "rows": _run_rows,
        "text": _run_text}


def run(state):
    return _RUN[state.case["kind"]](state)


# ---- what a pass cannot do without ------------------------------------------------------------------
def work(case):
    """Every table row, weight and cache row that the pass needs once, every result once.  The number
    of entries and codes of a prompt is taken from what such streams give on average: about 0.4 codes
    and 0.17 entries of 2.5 tokens per base token."""
    kind, V, d, B = case["kind"], case["V"], case["d"], case["B"]
    es = 4 if case["dtype"] == "fp32" else 2
    sides = 1 if case.get("tied", False) else 2
    enc_params = _layers() * (4 * d * d + 2 * d * _dff(case))
    T = case.get("T") or 4 * -(-case["N"] // B) + 64
    codes = 0.4 * B * T
    entries = B * min(case["cap"], 0.17 * T)
    if kind == "text":
        return {"bytes": 4 * (2 * B * T + 2 * codes) + entries * (4 * case["M"] + 9), "flops": 0}
    if kind == "rows":
        return {"bytes": es * d * (V + entries + case["N"]) + 16 * case["N"], "flops": 2.0 * d * case["N"] * (V + entries / B)}
    if kind in ("step", "filtered"):
        rows = B * 0.7 * 2.5                                   # base tokens of the entries a step creates
        b = es * d * (V + entries + B) + sides * es * enc_params + sides * es * d * (rows + B)
        if kind == "filtered":
            b += 2 * 4 * B * (V + entries / B)                 # logits written and read once
        return {"bytes": b, "flops": 2.0 * d * (B * V + entries) + 2.0 * sides * enc_params * rows}
    b = 4 * (B * T + codes) + sides * es * (enc_params + 2 * d * entries) + 2 * es * d * codes
    f = 2.0 * sides * enc_params * entries * 2.5
    if kind == "score":
        b += es * d * V
        f += 2.0 * d * codes * (V + entries / B)
    return {"bytes": b, "flops": f}


def tolerance(case):
    """Codes and tokens are exact.  Measured between the tensor-core kernels and the CUDA-core kernels
    (other sums, fp32 activations) on the same inputs: cache rows differ by 4e-4, an element by one bf16
    step (7.8e-3 of its value); logits, log-sum-exp and maxima over rows that differ like that by 2e-4 and
    2.9e-3.  About four times that; a near tie may change an argmax."""
    if case["kind"] == "text":
        return "exact"
    if case["dtype"] == "fp32":
        return {"rel": 2e-5, "max": 5e-4, "differ": 0.005}
    if case["kind"] == "rows":
        return {"rel": 2e-4, "max": 4e-3, "differ": 0.005}
    return {"rel": 2e-3 if case.get("half") else 1.6e-3, "max": 3.2e-2, "differ": 0.005}
