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
