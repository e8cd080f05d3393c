"""Hyper-encoder passes at the row counts where the linear-layer kernel, its activation box or its row blocks
change: one entry, capacities around 128, 256 and 512 packed rows (also with few of them live), the switch
to whole output tiles, a rest behind full passes; odd multiples of 128 as width (half a tile of 256 weight
rows); a session whose very first pass is captured into a graph.  Against the fp64 oracle.  Full-size decode
passes of some hundred rows are held to the rounding of their sums, against fp64 on the GPU."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import hyper_encoder as ohe
from oracle import lzw as olzw
from paper_2506_01084_b200 import binding as zb
from paper_2506_01084_b200 import synth_inputs as si
from tests._harness import Pair, TOL, f64

pytestmark = pytest.mark.gpu


def _pair(d, dff, M, B, T, cap, seed, tied=0, dtype="bf16", tensor_cores=1):
    w = si.Workload("rows", V=2000, d=d, dtype=dtype, B=B, T=T, M=M, cap=cap, zipf_s=1.0, copy_p=0.5, seg_min=4,
                    seg_max=14, steps=2, tied=tied, enc_layers=2, enc_heads=max(d // 128, 1), enc_dff=dff)
    p = Pair(w, seed, tensor_cores=tensor_cores)
    p.gpu_encode()
    for b in range(w.B):
        p.oracle.books[b].encode(p.tokens[b].tolist())
    return w, p


def _check(w, p, got, first, count):
    enc = [f64(t) for t in p.enc_E]
    table = f64(p.W_E)
    for b in range(w.B):
        for k in {first[b], first[b] + count[b] - 1, first[b] + count[b] // 2} if count[b] else ():
            want = ohe.hyper_embed([p.oracle.books[b].entries[k]], table, enc, w.heads)[0]
            assert np.abs(got[b, k].double().cpu().numpy() - want).max() <= TOL
        mask = torch.ones(w.cap, dtype=torch.bool)
        mask[first[b]:first[b] + count[b]] = False
        assert torch.all(got[b].cpu()[mask] == -5)            # no other row is touched


@pytest.mark.parametrize("bound", ["exact", "count", "loose"])
@pytest.mark.parametrize("d,dff,M,total", [(128, 384, 3, 1), (256, 512, 3, 42), (256, 512, 3, 43), (384, 640, 8, 16),
                                           (128, 256, 3, 85), (384, 1152, 3, 86), (256, 512, 3, 171), (256, 256, 4, 224),
                                           (256, 256, 4, 225), (128, 384, 2, 512), (128, 128, 3, 1050),
                                           (256, 384, 3, 112), (384, 256, 3, 230), (128, 256, 3, 290)])
def test_embedding_a_range_of_entries(d, dff, M, total, bound):
    B = 3
    w, p = _pair(d, dff, M, B, T=max(400, 6 * total), cap=1400, seed=total)
    n = [p.oracle.books[b].n() for b in range(B)]
    count = [total - 2 * (total // 3), total // 3, total // 3]
    first = [1, 0, 2]
    assert all(n[b] >= first[b] + count[b] for b in range(B))
    i32 = lambda x: torch.tensor(x, dtype=torch.int32, device=p.dev)
    got = torch.full((B, w.cap, d), -5.0, dtype=torch.bfloat16, device=p.dev)
    f32 = torch.full((B, w.cap, d), -5.0, dtype=torch.float32, device=p.dev)
    lim = {"exact": -1, "count": total, "loose": total + 300}[bound]
    zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, i32(first), i32(count), lim, got, f32)
    st, _ = zb.z2z_status(p.cb)
    assert all(int(s) & zb.ST_WAIT_TIMEOUT == 0 for s in st)
    _check(w, p, f32, first, count)
    assert torch.equal(got[0, first[0]].cpu(), f32[0, first[0]].cpu().bfloat16())


@pytest.mark.parametrize("B,tied", [(43, 0), (90, 1), (128, 0)])
def test_decode_step_of_a_large_batch_captured_first(B, tied):
    w, p = _pair(256, 512, 3, B, T=64, cap=64, seed=B, tied=tied)
    hid = si.make_hidden(w, B, 3).to(p.dev)
    nxt, new = (torch.zeros(B, dtype=torch.int32, device=p.dev) for _ in range(2))
    lse = torch.zeros(B, device=p.dev)
    forced = torch.tensor([(31 * b + 7) % w.V for b in range(B)], dtype=torch.int32, device=p.dev)
    forced[::5] = zb.CODE_NONE
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()                     # nothing of this session has run an encoder pass yet
    with torch.cuda.graph(graph):
        zb.z2z_decode_step(p.cb, hid, p.g_WE, p.g_WU, p.g_encE, p.g_encU, p.E_h, p.U_h, zb.SELECT_ARGMAX, 1.0, 0, 0,
                           forced, nxt, None, lse, new, p.E_f32, p.U_f32)
    graph.replay()
    torch.cuda.synchronize()
    enc = [f64(t) for t in p.enc_E]
    table = f64(p.W_E)
    for b in range(B):
        want = -1 if b % 5 == 0 else p.oracle.books[b].step(int(forced[b]))
        assert int(new[b]) == want
        if want >= 0 and b % 7 < 2:
            row = ohe.hyper_embed([p.oracle.books[b].entries[want]], table, enc, w.heads)[0]
            assert np.abs(p.E_f32[b, want].double().cpu().numpy() - row).max() <= TOL


def _node_types(graph):
    """Types of the nodes of a captured graph (0: kernel, 1: copy, 2: set)."""
    rt = ctypes.CDLL("libcudart.so.12")
    n = ctypes.c_size_t(0)
    g = ctypes.c_void_p(graph.raw_cuda_graph())
    assert rt.cudaGraphGetNodes(g, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(g, nodes, ctypes.byref(n)) == 0
    types = []
    for x in nodes:
        t = ctypes.c_int(-1)
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(x), ctypes.byref(t)) == 0
        types.append(t.value)
    return types


@pytest.mark.parametrize("B,tied", [(2, 0), (43, 1), (90, 0), (150, 0)])
def test_steps_captured_first_hold_no_clear(B, tied):
    """Neither the first step of a new session nor of one that starts again, nor a bounded call of one entry per
    sequence, captures anything but kernels; what the session start itself captures clears when it runs."""
    w, p = _pair(256, 512, 3, B, T=64, cap=64, seed=B, tied=tied)
    hid = si.make_hidden(w, B, 3).to(p.dev)
    nxt = torch.zeros(B, dtype=torch.int32, device=p.dev)

    def step():
        zb.z2z_decode_step(p.cb, hid, p.g_WE, p.g_WU, p.g_encE, p.g_encU, p.E_h, p.U_h, zb.SELECT_ARGMAX, 1.0, 0, 0,
                           None, nxt, None, None, None, p.E_f32, p.U_f32)
        zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, None, None, B, p.E_h, p.E_f32)

    for again in (False, True):
        if again:
            zb.z2z_codebook_init(p.cb)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph):
            step()
        assert set(_node_types(graph)) == {0}
        step()


@pytest.mark.parametrize("after_eager_steps", [False, True])
def test_a_graph_replays_over_a_session_that_starts_again(after_eager_steps):
    """The workspace holds anything when the session starts, and other rows exist in every replay."""
    B = 40
    w, p = _pair(256, 512, 3, B, T=64, cap=96, seed=B)
    hid = si.make_hidden(w, B, 3).to(p.dev)
    nxt, new, forced = (torch.zeros(B, dtype=torch.int32, device=p.dev) for _ in range(3))
    lse = torch.zeros(B, device=p.dev)

    def step():
        zb.z2z_decode_step(p.cb, hid, p.g_WE, p.g_WU, p.g_encE, p.g_encU, p.E_h, p.U_h, zb.SELECT_ARGMAX, 1.0, 0, 0,
                           forced, nxt, None, lse, new, p.E_f32, p.U_f32)

    if after_eager_steps:
        step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    p.cb.workspace.fill_(0x42)                                  # (48.6 as fp32)
    zb.z2z_codebook_init(p.cb)
    books = [olzw.Codebook(w.V, w.M, w.cap) for _ in range(B)]
    for t in range(5):
        codes = [(b + 31 * t) % w.V if t == 0 or (b + t) % (5 - t) == 0 else zb.CODE_NONE for b in range(B)]
        forced.copy_(torch.tensor(codes, dtype=torch.int32))
        graph.replay()
        want = [-1 if z == zb.CODE_NONE else books[b].step(z) for b, z in enumerate(codes)]
        assert new.cpu().tolist() == want
        made = [b for b in range(B) if want[b] >= 0][::3]
        for f32, W, enc in ((p.E_f32, p.W_E, p.enc_E), (p.U_f32, p.W_U, p.enc_U)):
            if made:
                rows = ohe.hyper_embed([books[b].entries[want[b]] for b in made], f64(W), [f64(x) for x in enc], w.heads)
                got = torch.stack([f32[b, want[b]] for b in made]).double().cpu().numpy()
                assert np.abs(got - rows).max() <= TOL


def test_a_captured_session_start_clears_when_it_runs():
    w, p = _pair(256, 512, 3, 3, T=64, cap=64, seed=3)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        zb.z2z_codebook_init(p.cb)
    # the graph has not run: the words of the result matrix may hold anything a failed pass left there
    p.cb.workspace.fill_(0xff)
    hid = si.make_hidden(w, 3, 3).to(p.dev)
    nxt, new = (torch.zeros(3, dtype=torch.int32, device=p.dev) for _ in range(2))
    graph.replay()
    for t, codes in enumerate(([5, 6, 7], [8, 9, 10])):
        zb.z2z_decode_step(p.cb, hid, p.g_WE, p.g_WU, p.g_encE, p.g_encU, p.E_h, p.U_h, zb.SELECT_ARGMAX, 1.0, 0, t,
                           torch.tensor(codes, dtype=torch.int32, device=p.dev), nxt, None, torch.zeros(3, device=p.dev), new,
                           p.E_f32, p.U_f32)
    assert new.cpu().tolist() == [0, 0, 0]
    want = ohe.hyper_embed([(5, 8), (6, 9), (7, 10)], f64(p.W_E), [f64(t) for t in p.enc_E], w.heads)
    assert np.abs(p.E_f32[:, 0].double().cpu().numpy() - want).max() <= TOL


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("B,tied", [(8, 0), (60, 0), (100, 1)])
def test_steps_without_an_entry_between_steps_that_create_some(B, tied, captured):
    """A pass without a row leaves the result matrix and the caches alone: all sequences sit out, or feed a code
    that makes no entry, then some create one, in the middle of the batch or everywhere."""
    w, p = _pair(256, 512, 3, B, T=64, cap=96, seed=B, tied=tied)
    i32 = lambda x: torch.tensor(x, dtype=torch.int32, device=p.dev)
    hid = si.make_hidden(w, B, 3).to(p.dev)
    nxt, new, forced = (torch.zeros(B, dtype=torch.int32, device=p.dev) for _ in range(3))
    lse = torch.zeros(B, device=p.dev)
    none = [zb.CODE_NONE] * B
    some = [(41 * b + 3) % w.V if b % 3 == 1 else zb.CODE_NONE for b in range(B)]
    every = [(57 * b + 9) % w.V for b in range(B)]
    plan = [none, some, none, none, every, some, every]           # (the second `some` and `every` repeat codes)

    def step():
        zb.z2z_decode_step(p.cb, hid, p.g_WE, p.g_WU, p.g_encE, p.g_encU, p.E_h, p.U_h, zb.SELECT_ARGMAX, 1.0, 0, 0,
                           forced, nxt, None, lse, new, p.E_f32, p.U_f32)

    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    if captured:
        forced.copy_(i32(none))
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            step()
    sides = [(p.E_f32, p.W_E, p.enc_E), (p.U_f32, p.W_U, p.enc_U)][:1 if tied else 2]
    for codes in plan:
        forced.copy_(i32(codes))
        before = [f32.clone() for f32, _, _ in sides]
        graph.replay() if captured else step()
        want = [-1 if z == zb.CODE_NONE else p.oracle.books[b].step(z) for b, z in enumerate(codes)]
        assert new.cpu().tolist() == want
        for (f32, W, enc), old in zip(sides, before):
            made = [b for b in range(B) if want[b] >= 0]
            mask = torch.ones(B, w.cap, dtype=torch.bool, device=p.dev)
            for b in made:
                mask[b, want[b]] = False
            assert torch.equal(f32[mask], old[mask])
            for b in made[::7]:
                row = ohe.hyper_embed([p.oracle.books[b].entries[want[b]]], f64(W), [f64(t) for t in enc], w.heads)[0]
                assert np.abs(f32[b, want[b]].double().cpu().numpy() - row).max() <= TOL


@pytest.mark.parametrize("M,d,dff", [(2, 128, 256), (3, 384, 384), (5, 128, 128)])
def test_whole_prompts_in_passes_cut_by_rows(M, d, dff):
    """Every entry of a call of several passes, so that those on both sides of a cut are among them."""
    w, p = _pair(d, dff, M, B=3, T=9000, cap=3000, seed=M)
    n = [p.oracle.books[b].n() for b in range(w.B)]
    assert sum(len(e) for b in range(w.B) for e in p.oracle.books[b].entries) > 2 * 1024 * M       # more than one pass holds
    zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, None, None, -1, p.E_h, p.E_f32)
    enc = [f64(t) for t in p.enc_E]
    for b in range(w.B):
        want = ohe.hyper_embed(p.oracle.books[b].entries, f64(p.W_E), enc, w.heads)
        assert np.abs(p.E_f32[b, :n[b]].double().cpu().numpy() - want).max() <= TOL
        assert torch.all(p.E_f32[b, n[b]:] == 0)


@pytest.mark.parametrize("d,dff", [(1024, 4096), (384, 1152), (2560, 768)])
@pytest.mark.parametrize("total", [16, 40, 43, 85, 86, 200])
def test_a_bounded_call_gives_the_same_bits_every_time(d, dff, total):
    """Sessions whose passes hold 1024 rows or more: on one CTA per tile, on pairs, in several row blocks; the
    pairs with eight (d = 1024) and six (2560) clusters per tile."""
    w, p = _pair(d, dff, 3, B=2, T=900, cap=600, seed=total)
    i32 = lambda x: torch.tensor(x, dtype=torch.int32, device=p.dev)
    count = [total // 2, total - total // 2]
    assert all(p.oracle.books[b].n() >= count[b] for b in range(2))
    first = None
    for _ in range(10):
        f32 = torch.full((2, w.cap, d), -5.0, dtype=torch.float32, device=p.dev)
        zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, i32([0, 0]), i32(count), total, p.E_h, f32)
        first = f32 if first is None else first
        assert torch.equal(f32, first)
    _check(w, p, first, [0, 0], count)


@pytest.mark.parametrize("d,dff,dtype,tensor_cores", [(256, 512, "bf16", 1), (384, 512, "bf16", 0), (320, 640, "fp32", 1),
                                                      (64, 128, "fp32", 1)])
def test_entries_beyond_the_bound_stay_due(d, dff, dtype, tensor_cores):
    """On the tensor cores, on the tiled CUDA-core kernels (bf16, fp32) and with narrow models."""
    w, p = _pair(d, dff, 3, B=3, T=500, cap=400, seed=8, dtype=dtype, tensor_cores=tensor_cores)
    n = [p.oracle.books[b].n() for b in range(w.B)]
    p.E_f32.fill_(-5)
    done = 0
    for bound in (20, n[0] + n[1] // 2 - 20, sum(n)):          # inside the first and second sequence, then the rest
        zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, None, None, bound, p.E_h, p.E_f32)
        done = min(done + bound, sum(n))
        assert [int((p.E_f32[b, :, 0] != -5).sum()) for b in range(3)] == [
            max(0, min(n[b], done - sum(n[:b]))) for b in range(3)]
    enc = [f64(t) for t in p.enc_E]
    for b in range(w.B):
        want = ohe.hyper_embed(p.oracle.books[b].entries, f64(p.W_E), enc, w.heads)
        assert np.abs(p.E_f32[b, :n[b]].double().cpu().numpy() - want).max() <= TOL


def _encode64(t, table, tok, heads, layers):
    """Hyper-embedding of one phrase in fp64 on the GPU (tensors in ABI order, fp64)."""
    d, L = table.shape[1], len(tok)
    ln = lambda z, i: torch.nn.functional.layer_norm(z, (d,), t[i], t[i + 1], 1e-5)
    x = table[tok].double() + t[0][:L]
    for o in range(1, 1 + 12 * layers, 12):
        q, k, v = (ln(x, o) @ t[o + 2].T + t[o + 3]).view(L, 3, heads, d // heads).unbind(1)
        a = torch.softmax(torch.einsum("ihc,jhc->hij", q, k) / (d // heads) ** 0.5, -1)
        x = x + torch.einsum("hij,jhc->ihc", a, v).reshape(L, d) @ t[o + 4].T + t[o + 5]
        x = x + torch.nn.functional.gelu(ln(x, o + 6) @ t[o + 8].T + t[o + 9]) @ t[o + 10].T + t[o + 11]
    return x.mean(0)


@pytest.mark.parametrize("d,M,B,tied,bound", [(4096, 3, 128, 0, 2.0e-5), (3072, 5, 128, 0, 1.6e-5), (4096, 3, 256, 1, 2.0e-5),
                                              (3072, 3, 310, 1, 1.6e-5)])
def test_sums_of_a_decode_pass_of_some_hundred_rows(d, M, B, tied, bound):
    """Every row of the pass's capacity is live.  The tensor cores add 16 products to a sum at a time and lose
    low bits each time, so that the error grows with the additions an accumulator takes: with one product per
    weight and a chain over all of K = 4 d the rows were off by 1.8e-5 of their rms at d = 4096 and by 1.4e-5 at
    d = 3072, with both operand parts in one chain by 2.5e-5 to 4.3e-5 and 2.1e-5 to 3.2e-5.  Bound: the former
    and an eighth for other inputs."""
    V, layers, cap, heads, dev = 2000, 2, 16, d // 128, "cuda:0"
    g = torch.Generator(device=dev)
    g.manual_seed(d + M)

    def normal(shape, std, mean=0.0):
        return (torch.randn(shape, generator=g, device=dev) * std + mean).bfloat16()

    def encoder():
        t = [normal((M, d), 0.02)]
        for _ in range(layers):
            t += [normal((d,), 0.1, 1.0), normal((d,), 0.05), normal((3 * d, d), 0.02), normal((3 * d,), 0.05)]
            t += [normal((d, d), 0.02), normal((d,), 0.05), normal((d,), 0.1, 1.0), normal((d,), 0.05)]
            t += [normal((4 * d, d), 0.02), normal((4 * d,), 0.05), normal((d, 4 * d), 0.02), normal((d,), 0.05)]
        return t

    sides = 1 if tied else 2
    W = [normal((V, d), 0.02) for _ in range(sides)]
    enc = [encoder() for _ in range(sides)]
    ew = [zb.encoder_weights(t) for t in enc]
    cache = [torch.zeros(B, cap, d, dtype=torch.bfloat16, device=dev) for _ in range(sides)]
    f32 = [torch.zeros(B, cap, d, device=dev) for _ in range(2)]
    cb = zb.Codebook(zb.make_config(V, d, M, cap, B, "bf16", layers, heads, 4 * d, tied), dev)
    codes = lambda f: torch.tensor([f(b) for b in range(B)], dtype=torch.int32, device=dev)
    zb.z2z_lzw_step(cb, codes(lambda b: b), None, None)
    for k in range(M - 2):                               # a, a a, a a a: the previous phrase grows to M - 1 tokens
        zb.z2z_lzw_step(cb, codes(lambda b: V + k), None, None)
    nxt, new = (torch.zeros(B, dtype=torch.int32, device=dev) for _ in range(2))
    lse = torch.zeros(B, device=dev)
    zb.z2z_decode_step(cb, normal((B, d), 1.0), W[0], W[-1], ew[0], ew[-1], cache[0], cache[-1], zb.SELECT_ARGMAX, 1.0, 0, 0,
                       codes(lambda b: 1000 + b), nxt, None, lse, new, f32[0], f32[1])
    assert new.cpu().tolist() == [M - 2] * B             # B * M rows: every entry is M tokens long
    for side in range(sides):
        t = [x.double() for x in enc[side]]
        err, ref = [], []
        for b in range(0, B, 8):
            want = _encode64(t, W[side], [b] * (M - 1) + [1000 + b], heads, layers)
            ref.append(want)
            err.append(f32[side][b, M - 2].double() - want)
        err, ref = torch.stack(err), torch.stack(ref)
        assert float(err.pow(2).mean().sqrt() / ref.pow(2).mean().sqrt()) <= bound


@pytest.mark.parametrize("B,tied", [(3, 0), (130, 0), (3, 1)])
def test_entries_left_out_by_a_bound_stay_due_through_decode_steps(B, tied):
    """The decode step's own launch (up to 128 sequences) and its separate ones, per side."""
    w, p = _pair(128, 256, 3, B=B, T=120, cap=200, seed=B + tied, tied=tied)
    n = [p.oracle.books[b].n() for b in range(w.B)]
    assert min(n) > 8
    sides = ((zb.CACHE_EMBED, p.g_WE, p.g_encE, p.E_h, p.E_f32, p.enc_E, p.W_E),
             (zb.CACHE_UNEMBED, p.g_WU, p.g_encU, p.U_h, p.U_f32, p.enc_U, p.W_U))[:1 if tied else 2]
    for which, table, enc, cache, f32, _, _ in sides:          # cut inside the second sequence; the other side later
        zb.z2z_hyper_embed(p.cb, which, table, enc, None, None, n[0] + 4 + which, cache, f32)
    nxt, new = (torch.zeros(B, dtype=torch.int32, device=p.dev) for _ in range(2))
    lse = torch.zeros(B, device=p.dev)
    for t in range(2):
        forced = torch.tensor([(37 * b + 911 * t + 5) % w.V for b in range(B)], dtype=torch.int32, device=p.dev)
        zb.z2z_decode_step(p.cb, si.make_hidden(w, B, t).to(p.dev), p.g_WE, p.g_WU, p.g_encE, p.g_encU, p.E_h, p.U_h,
                           zb.SELECT_ARGMAX, 1.0, 0, t, forced, nxt, None, lse, new, p.E_f32, p.U_f32)
        for b in range(B):
            p.oracle.books[b].step(int(forced[b]))
    for which, table, enc, cache, f32, host, W in sides:
        zb.z2z_hyper_embed(p.cb, which, table, enc, None, None, -1, cache, f32)
        for b in range(0, B, max(1, B // 8)):
            want = ohe.hyper_embed(p.oracle.books[b].entries, f64(W), [f64(x) for x in host], w.heads)
            assert np.abs(f32[b, :len(want)].double().cpu().numpy() - want).max() <= TOL
        f32.fill_(-5)                                          # nothing is due any more
        zb.z2z_hyper_embed(p.cb, which, table, enc, None, None, -1, cache, f32)
        assert torch.all(f32 == -5)


def test_decode_steps_settle_what_was_embedded_by_range():
    """A program that embeds its prompts by given ranges: after a decode step only newer entries are due."""
    w, p = _pair(128, 256, 3, B=3, T=120, cap=200, seed=5)
    n = [p.oracle.books[b].n() for b in range(w.B)]
    i32 = lambda x: torch.tensor(x, dtype=torch.int32, device=p.dev)
    zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, i32([0] * 3), i32(n), sum(n), p.E_h, p.E_f32)
    nxt, new = (torch.zeros(3, dtype=torch.int32, device=p.dev) for _ in range(2))
    zb.z2z_decode_step(p.cb, si.make_hidden(w, 3, 1).to(p.dev), p.g_WE, p.g_WU, p.g_encE, p.g_encU, p.E_h, p.U_h,
                       zb.SELECT_ARGMAX, 1.0, 0, 0, i32([7, 8, 9]), nxt, None, torch.zeros(3, device=p.dev), new, p.E_f32, p.U_f32)
    _, m = zb.z2z_status(p.cb)
    zb.z2z_lzw_step(p.cb, i32([1007, 1008, 1009]), None, new)
    assert new.cpu().tolist() == m.tolist()
    p.E_f32.fill_(-5)
    zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, None, None, 3, p.E_h, p.E_f32)
    for b in range(3):
        assert torch.all(p.E_f32[b, int(m[b])] != -5) and torch.all(p.E_f32[b, :int(m[b])] == -5)


@pytest.mark.parametrize("B,bound", [(37, 200), (37, 64), (700, 1000), (5, 1)])
def test_short_list_of_ranges(B, bound):
    """Calls whose offsets, list and row map come from one launch: ranges that start before the first entry, end behind
    the last one or are empty, over one and several warps of sequences, and a bound below what they hold."""
    w, p = _pair(128, 128, 3, B, T=60, cap=40, seed=B)
    n = [p.oracle.books[b].n() for b in range(B)]
    first = [(5 * b) % 7 - 2 for b in range(B)]
    count = [[0, 2, -3, 1, 400][b % 5] if B < 100 else [0, 1, 2, 0, -1][b % 5] for b in range(B)]
    lo = [min(max(f, 0), k) for f, k in zip(first, n)]
    size = [min(max(c, 0), k - f) for c, k, f in zip(count, n, lo)]
    left = bound
    for b in range(B):
        size[b] = min(size[b], left)
        left -= size[b]
    f32 = torch.full((B, w.cap, 128), -5.0, device=p.dev)
    i32 = lambda x: torch.tensor(x, dtype=torch.int32, device=p.dev)
    zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, i32(first), i32(count), bound, p.E_h, f32)
    got = f32.double().cpu().numpy()
    enc, table = [f64(t) for t in p.enc_E], f64(p.W_E)
    for b in range(B):
        assert np.all(got[b, :lo[b]] == -5) and np.all(got[b, lo[b] + size[b]:] == -5)
        if size[b]:
            want = ohe.hyper_embed(p.oracle.books[b].entries[lo[b]:lo[b] + size[b]], table, enc, w.heads)
            assert np.abs(got[b, lo[b]:lo[b] + size[b]] - want).max() <= TOL


@pytest.mark.parametrize("d,dff,total", [(2560, 768, 40), (2560, 768, 80), (384, 512, 200)])
def test_bounded_calls_without_an_entry_between_calls_that_embed(d, dff, total):
    """Calls whose ranges are empty leave nothing behind, in the caches or in the scratch of the calls around them: on one
    CTA per tile and on pairs, with weights for more than the load ring (d = 2560), in several row blocks.  (That they
    stream no weights is not seen here; only their time shows it.)"""
    w, p = _pair(d, dff, 3, B=2, T=900, cap=600, seed=total)
    i32 = lambda x: torch.tensor(x, dtype=torch.int32, device=p.dev)
    some = [total // 2 - 3, total - total // 2]
    assert all(p.oracle.books[b].n() >= total - total // 2 for b in range(2))
    want = None
    for count in ([0, 0], some, [0, 0], [0, 0], some):
        f32 = torch.full((2, w.cap, d), -5.0, dtype=torch.float32, device=p.dev)
        zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, i32([3, 0]), i32(count), total, p.E_h, f32)
        if count == some:
            want = f32 if want is None else want
            assert torch.equal(f32, want)
        else:
            assert torch.all(f32 == -5)
    _check(w, p, want, [3, 0], some)
    st, _ = zb.z2z_status(p.cb)
    assert all(int(x) & zb.ST_WAIT_TIMEOUT == 0 for x in st)


def test_exact_call_beside_joint_logits_on_another_stream():
    """The two calls share no scratch: the input side of a prompt may be embedded while positions are scored."""
    w, p = _pair(256, 512, 3, B=4, T=3000, cap=1200, seed=3)
    n = sum(p.oracle.books[b].n() for b in range(w.B))
    assert n * 2 > 2048                                        # more than one pass
    zb.z2z_hyper_embed(p.cb, zb.CACHE_UNEMBED, p.g_WU, p.g_encU, None, None, -1, p.U_h, None)
    N = 20000
    hid = torch.randn(N, w.d, device=p.dev).to(torch.bfloat16)
    seq = (torch.arange(N, device=p.dev) % w.B).sort().values.to(torch.int32)
    first = torch.zeros(w.B, dtype=torch.int32, device=p.dev)
    count = torch.full((w.B,), w.cap, dtype=torch.int32, device=p.dev)       # clipped to what there is

    def logits():
        lse = torch.zeros(N, device=p.dev)
        zb.z2z_dynamic_logits(p.cb, hid, seq, None, p.g_WU, p.U_h, zb.SELECT_ARGMAX, 1.0, 0, 0, None, lse, None, None)
        return lse

    def embed():
        f32 = torch.zeros_like(p.E_f32)
        zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, first, count, -1, p.E_h, f32)
        return f32

    want_lse, want_rows = logits(), embed()
    torch.cuda.synchronize()
    other = torch.cuda.Stream()
    for _ in range(5):
        with torch.cuda.stream(other):
            lse = [logits() for _ in range(3)]
        rows = [embed() for _ in range(3)]
        torch.cuda.synchronize()
        assert all(torch.equal(x, want_lse) for x in lse) and all(torch.equal(x, want_rows) for x in rows)


@pytest.mark.parametrize("M,heads", [(2, 2), (4, 2), (7, 2), (3, 1)])
def test_rows_that_are_alike_share_the_first_layers_products(M, heads):
    """A pass of more than 512 rows computes q, k, v once per (base token, position); a short one does not.  The same
    bits, on both attention kernels (merge sizes up to 4 with heads of up to 128 columns, and others)."""
    w = si.Workload("alike", V=40, d=256, dtype="bf16", B=3, T=2500, M=M, cap=900, zipf_s=1.0, copy_p=0.5, seg_min=4, seg_max=14,
                    steps=2, enc_layers=2, enc_heads=heads, enc_dff=512)
    p = Pair(w, 5)
    p.gpu_encode()
    n = zb.z2z_status(p.cb)[1].tolist()
    assert 512 < int(sum(n)) and min(n) > 40
    i32 = lambda x: torch.tensor(x, dtype=torch.int32, device=p.dev)
    f32 = torch.full((3, w.cap, 256), -5.0, device=p.dev)
    zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, i32([0] * 3), i32(n), -1, p.E_h, f32)
    part = torch.full((3, w.cap, 256), -5.0, device=p.dev)
    last = [k - 17 for k in n]
    zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, i32(last), i32([17] * 3), -1, p.E_h, part)
    for b in range(3):
        assert torch.equal(f32[b, last[b]:n[b]], part[b, last[b]:n[b]])
        assert torch.all(f32[b, n[b]:] == -5)


def test_exact_rows_do_not_depend_on_the_rest_of_the_call():
    """A few entries alone, in a call of one pass and in a call of several: the same bits."""
    w, p = _pair(256, 512, 3, B=3, T=3000, cap=1400, seed=12)
    n = [p.oracle.books[b].n() for b in range(w.B)]
    assert sum(n) > 1100
    rows = []
    for count in ([5, 0, 9], [200, 30, 100], n):
        f32 = torch.full((3, w.cap, 256), -5.0, device=p.dev)
        i32 = lambda x: torch.tensor(x, dtype=torch.int32, device=p.dev)
        zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, i32([0] * 3), i32(count), -1, p.E_h, f32)
        rows.append(f32)
    assert torch.equal(rows[0][0, :5], rows[2][0, :5]) and torch.equal(rows[0][2, :9], rows[2][2, :9])
    for b, c in enumerate([200, 30, 100]):
        assert torch.equal(rows[1][b, :c], rows[2][b, :c])
