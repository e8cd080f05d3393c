"""Calls right behind z2z_upload_rows, which lets the next kernel of the stream start before it has written anything:
tables that are no operand of a decode step of up to 32 rows are read as the stream orders it.  The uploaded
tensors are small enough for all blocks of the upload to be resident at once, so that whoever reads ahead of its
dependency wait reads the old values."""
import pytest
import torch

from paper_2506_01084_b200 import binding as zb

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _rnd(seed, *shape, std=1.0):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return (torch.randn(*shape, generator=g, device=DEV) * std).to(torch.bfloat16)


def _uploaded_ahead(table, call):
    """`call` on what `table` holds, and again right behind the upload of it over other values."""
    held = table.cpu().pin_memory()
    want = call()
    torch.cuda.synchronize()
    for _ in range(3):
        table.zero_()
        torch.cuda.synchronize()
        zb.z2z_upload_rows(held, table)
        got = call()
        torch.cuda.synchronize()
        assert all(torch.equal(g, w) for g, w in zip(got, want))


# 40 and 128 rows: five and four stages; a vocabulary whose shares are even (three granules of 32 per SM and more),
# and one where the CTAs share W_U and hypertokens
@pytest.mark.parametrize("V", [4000, 14400])
@pytest.mark.parametrize("B", [40, 128])
@pytest.mark.parametrize("step", [False, True])
def test_batch_logits_behind_an_upload_of_the_table(V, B, step):
    d, cap = 128, 8
    cb = zb.Codebook(zb.make_config(V, d, 2, cap, B, "bf16", 0, 1, 8), DEV)
    hid, Uh = _rnd(1, B, d), _rnd(2, B, cap, d, std=0.05)
    WU = _rnd(3, V, d, std=0.05)
    none = torch.full((B,), zb.CODE_NONE, dtype=torch.int32, device=DEV)
    pos = zb.encoder_weights([_rnd(4, 2, d)])

    def call():
        lse = torch.zeros(B, device=DEV)
        best, nxt = (torch.zeros(B, dtype=torch.int32, device=DEV) for _ in range(2))
        if step:                                         # every sequence sits out: the codebooks stay as they are
            zb.z2z_decode_step(cb, hid, WU, WU, pos, pos, Uh, Uh, zb.SELECT_ARGMAX, 1.0, 0, 0, none, nxt, best, lse)
        else:
            zb.z2z_dynamic_logits(cb, hid, None, None, WU, Uh, zb.SELECT_ARGMAX, 1.0, 0, 0, None, lse, best, None)
        return lse, best

    _uploaded_ahead(WU, call)


# max_entries 30: one launch for list, offsets and row map; 1100: offsets, list and map apart; several row blocks
@pytest.mark.parametrize("bound", [30, 1100])
def test_bounded_embedding_behind_an_upload_of_the_weights(bound):
    V, d, dff, cap, B = 500, 256, 512, 600, 2
    cb = zb.Codebook(zb.make_config(V, d, 2, cap, B, "bf16", 2, 2, dff), DEV)
    tok = torch.randperm(V, generator=torch.Generator().manual_seed(1))[:2 * 40].to(torch.int32).view(B, 40).to(DEV)
    codes, lens = torch.zeros_like(tok), torch.zeros(B, dtype=torch.int32, device=DEV)
    zb.z2z_lzw_encode(cb, tok, None, codes, lens)
    shapes = [(2, d)] + 2 * [(d,), (d,), (3 * d, d), (3 * d,), (d, d), (d,), (d,), (d,), (dff, d), (dff,), (d, dff), (d,)]
    sizes = [torch.Size(s).numel() for s in shapes]
    flat = _rnd(5, sum(sizes), std=0.05)                 # one tensor holds them all
    enc = zb.encoder_weights([t.view(s) for t, s in zip(flat.split(sizes), shapes)])
    table = _rnd(6, V, d)
    first = torch.zeros(B, dtype=torch.int32, device=DEV)
    count = torch.full((B,), 15, dtype=torch.int32, device=DEV)

    def call():
        rows = torch.zeros(B, cap, d, dtype=torch.bfloat16, device=DEV)
        zb.z2z_hyper_embed(cb, zb.CACHE_EMBED, table, enc, first, count, bound, rows)
        return (rows,)

    _uploaded_ahead(flat, call)


# what stands between the upload and the call that may read ahead of the kernel right before it
@pytest.mark.parametrize("between", ["lookup", "update", "embed", "positions", "batch"])
def test_decode_logits_behind_another_call_behind_an_upload(between):
    V, d, cap, B = 14400, 128, 600, 40
    cb = zb.Codebook(zb.make_config(V, d, 2, cap, B, "bf16", 0, 1, 8), DEV)
    WE, WU = _rnd(1, V, d), _rnd(2, V, d, std=0.05)
    Eh, Uh, hid = (_rnd(3 + i, *s) for i, s in enumerate([(B, cap, d), (B, cap, d), (48, d)]))
    x, lse48, pos = torch.zeros_like(hid), torch.zeros(48, device=DEV), zb.encoder_weights([_rnd(7, 2, d)])
    code = torch.arange(B, dtype=torch.int32, device=DEV)
    off = torch.zeros(B, dtype=torch.uint8, device=DEV)
    zero = torch.zeros(B, dtype=torch.int32, device=DEV)
    seq = torch.arange(48, dtype=torch.int32, device=DEV) % 3
    args = (zb.SELECT_ARGMAX, 1.0, 0, 0, None)

    def call():
        if between == "lookup":
            zb.z2z_embed_lookup(cb, code, None, WE, Eh, x)
        elif between == "update":
            zb.z2z_lzw_step(cb, code, off, None)
        elif between == "embed":
            zb.z2z_hyper_embed(cb, zb.CACHE_EMBED, WE, pos, zero, zero, 8, Eh)
        elif between == "positions":                     # more rows than sequences
            zb.z2z_dynamic_logits(cb, hid, seq, None, WE, Uh, *args, lse48, None, None)
        else:
            zb.z2z_dynamic_logits(cb, hid[:B], None, None, WE, Uh, *args, lse48, None, None)
        lse, best = torch.zeros(8, device=DEV), torch.zeros(8, dtype=torch.int32, device=DEV)
        zb.z2z_dynamic_logits(cb, hid[:8], None, None, WU, Uh, *args, lse, best, None)
        return lse, best

    _uploaded_ahead(WU, call)
