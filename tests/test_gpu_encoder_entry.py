"""The one-launch hyper-encoder pass of narrow models against the fp64 oracle: widths that are no
multiple of the lanes that share an output, one to eight heads, single rows and rows of the largest merge
size, layers without a feed-forward block, no layers at all, the largest width it takes, both dtypes, and
decode steps with one and two encoders; and the number of entries from which the tiled kernels take over."""
import pytest
import torch

from paper_2506_01084_b200 import binding as zb
from paper_2506_01084_b200 import synth_inputs as si
from tests._harness import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,dff,M,layers,dtype,tied", [
    (8, 1, 8, 2, 1, "fp32", False), (40, 5, 160, 8, 2, "fp32", False), (64, 4, 256, 3, 2, "fp32", True),
    (72, 2, 24, 5, 3, "fp32", False), (104, 8, 416, 4, 2, "fp32", False), (128, 4, 0, 3, 2, "fp32", False),
    (256, 2, 1024, 8, 1, "fp32", False), (56, 7, 224, 3, 0, "fp32", False), (88, 2, 352, 4, 2, "bf16", False)])
def test_narrow_encoder_pass(d, heads, dff, M, layers, dtype, tied):
    w = si.Workload("narrow", V=300, d=d, dtype=dtype, B=3, T=200, M=M, cap=150, zipf_s=1.1, copy_p=0.6,
                    seg_min=4, seg_max=12, steps=3, tied=tied, enc_layers=layers, enc_heads=heads, enc_dff=dff, enc_ffn=int(dff > 0))
    p = Pair(w, seed=d + M)
    p.gpu_encode()
    p.oracle.prefill([p.tokens[b].tolist() for b in range(w.B)])
    for which, table, enc, cache, f32 in ((zb.CACHE_EMBED, p.g_WE, p.g_encE, p.E_h, p.E_f32),
                                          (zb.CACHE_UNEMBED, p.g_WU, p.g_encU, p.U_h, p.U_f32)):
        zb.z2z_hyper_embed(p.cb, which, table, enc, None, None, -1, cache, f32)
    # fp32 sums over at most 1024 terms: 2e-5, the bound the fp32 sessions are held to elsewhere;
    # bf16 tables and weights enter exactly, activations stay fp32
    for b in range(w.B):
        p.check_cache_rows(b, 0, p.oracle.books[b].n(), tol=2e-5)
    hid = si.make_hidden(w, 3 * w.B, 9).view(3, w.B, w.d).to(p.dev)
    nxt = torch.zeros(w.B, dtype=torch.int32, device=p.dev)
    lse = torch.zeros(w.B, dtype=torch.float32, device=p.dev)
    new = torch.zeros(w.B, dtype=torch.int32, device=p.dev)
    forced = torch.zeros(w.B, dtype=torch.int32, device=p.dev)
    for t in range(3):
        forced.copy_(torch.tensor([(17 * t + 5 * b) % w.V for b in range(w.B)], dtype=torch.int32))
        zb.z2z_decode_step(p.cb, hid[t], p.g_WE, p.g_WU, p.g_encE, p.g_encU, p.E_h, p.U_h, zb.SELECT_ARGMAX, 1.0, 0, t,
                           forced, nxt, None, lse, new, p.E_f32, p.U_f32)
        onew = p.oracle.advance(nxt.cpu().tolist())
        assert new.cpu().tolist() == onew
        for b in range(w.B):
            if onew[b] >= 0:
                p.check_cache_rows(b, onew[b], onew[b] + 1, tol=2e-5)


@pytest.mark.parametrize("d,most", [(64, 96), (192, 96), (200, 72), (256, 72)])
def test_many_entries_take_the_tiled_kernels(d, most):
    """One launch for as many entries as are quicker that way; a whole prompt reads the weights once per tile."""
    w = si.Workload("narrow", V=300, d=d, dtype="fp32", B=2, T=700, M=3, cap=300, zipf_s=1.0, copy_p=0.3,
                    seg_min=4, seg_max=12, steps=1, enc_layers=2, enc_heads=4, enc_dff=64)
    p = Pair(w, seed=d)
    p.gpu_encode()
    p.oracle.prefill([p.tokens[b].tolist() for b in range(w.B)])
    n = [p.oracle.books[b].n() for b in range(w.B)]
    assert sum(n) > 2 * most + 1
    rest = sum(n) - 2 * most - 1
    for bound, one in ((most, True), (most + 1, False), (rest, rest <= most)):
        zb.z2z_profile_read(p.cb)
        zb.z2z_hyper_embed(p.cb, zb.CACHE_EMBED, p.g_WE, p.g_encE, None, None, bound, p.E_h, p.E_f32)
        assert (zb.z2z_profile_read(p.cb)[1]["encoder_gemm"] == 1) == one
    zb.z2z_hyper_embed(p.cb, zb.CACHE_UNEMBED, p.g_WU, p.g_encU, None, None, -1, p.U_h, p.U_f32)
    for b in range(w.B):
        p.check_cache_rows(b, 0, n[b], tol=2e-5)


def test_decode_step_of_a_large_narrow_batch():
    w = si.Workload("narrow", V=300, d=64, dtype="fp32", B=140, T=40, M=3, cap=60, zipf_s=1.1, copy_p=0.6,
                    seg_min=4, seg_max=12, steps=2, enc_layers=2, enc_heads=4, enc_dff=256)
    p = Pair(w, seed=2)
    p.gpu_encode()
    p.oracle.prefill([p.tokens[b].tolist() for b in range(w.B)])
    hid = si.make_hidden(w, 2 * w.B, 9).view(2, w.B, w.d).to(p.dev)
    nxt, new = (torch.zeros(w.B, dtype=torch.int32, device=p.dev) for _ in range(2))
    for t in range(2):
        forced = torch.tensor([(17 * t + 5 * b) % w.V for b in range(w.B)], dtype=torch.int32, device=p.dev)
        zb.z2z_decode_step(p.cb, hid[t], p.g_WE, p.g_WU, p.g_encE, p.g_encU, p.E_h, p.U_h, zb.SELECT_ARGMAX, 1.0, 0, t,
                           forced, nxt, None, torch.zeros(w.B, device=p.dev), new, p.E_f32, p.U_f32)
        onew = p.oracle.advance(nxt.cpu().tolist())
        assert new.cpu().tolist() == onew
        for b in range(w.B):
            if onew[b] >= 0:
                p.check_cache_rows(b, onew[b], onew[b] + 1, tol=2e-5)
