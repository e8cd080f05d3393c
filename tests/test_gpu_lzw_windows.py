"""Windowed LZW parse and replay at the sizes where a window can go wrong: its edges (128 positions,
matches that cross them), tiny alphabets in which most windows end early because a phrase repeats
inside them, codebooks that fill up inside a window, both homes of the table (shared memory up to 16384
entries, global memory beyond), sessions that continue, codes that name no entry.  Bit-exact."""
import numpy as np
import pytest
import torch

from oracle import lzw as olzw
from paper_2506_01084_b200 import binding as zb

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _session(V, M, cap, B):
    return zb.Codebook(zb.make_config(V, 8, M, cap, B, "fp32", 0, 1, 8), DEV)


def _stream(rng, V, T, kind):
    if kind == "run":                                   # one token over and over: every code names the newest entry
        return np.full(T, V - 1, dtype=np.int32)
    if kind == "period":
        return np.resize(rng.integers(0, V, size=max(2, min(37, T))), T).astype(np.int32)
    return rng.integers(0, V, size=T).astype(np.int32)


def _check_books(cb, books):
    st, n = zb.z2z_status(cb)
    for b, ob in enumerate(books):
        cons, ln = zb.z2z_codebook_read(cb, b)
        assert int(n[b]) == ob.n()
        assert [tuple(int(x) for x in cons[k, :int(ln[k])]) for k in range(ob.n())] == ob.entries
        assert int(st[b]) == ob.status


def _encode(cb, rows, T):
    B = len(rows)
    toks = np.zeros((B, T), dtype=np.int32)
    for b, r in enumerate(rows):
        toks[b, :len(r)] = r
    codes = torch.full((B, T), -7, dtype=torch.int32, device=DEV)
    after = torch.full((B, T), -7, dtype=torch.int32, device=DEV)
    clen = torch.zeros(B, dtype=torch.int32, device=DEV)
    lens = torch.tensor([len(r) for r in rows], dtype=torch.int32, device=DEV)
    zb.z2z_lzw_encode(cb, torch.from_numpy(toks).to(DEV), lens, codes, clen, after)
    return codes.cpu().numpy(), clen.cpu().numpy(), after.cpu().numpy()


@pytest.mark.parametrize("kind", ["random", "run", "period"])
@pytest.mark.parametrize("V,M,cap", [(2, 8, 4096), (3, 2, 300), (7, 5, 16384), (50, 3, 70), (1000, 8, 16385), (40, 4, 0)])
def test_windows_match_the_oracle(V, M, cap, kind):
    rng = np.random.default_rng(V * 131 + M)
    lens = [0, 1, 7, 127, 128, 129, 135, 136, 255, 256, 263, 1000, 2049]
    B, T = len(lens), max(lens)
    cb = _session(V, M, cap, B)
    books = [olzw.Codebook(V, M, cap) for _ in range(B)]
    streams = [[] for _ in range(B)]
    texts = [[] for _ in range(B)]
    for part in range(2):                               # the second call continues from the first one's codebooks
        rows = [_stream(rng, V, L, kind) for L in lens]
        codes, clen, after = _encode(cb, rows, T)
        for b in range(B):
            want, want_after = books[b].encode(rows[b].tolist())
            assert codes[b, :clen[b]].tolist() == want
            assert after[b, :clen[b]].tolist() == want_after
            assert np.all(codes[b, clen[b]:] == -7) and np.all(after[b, clen[b]:] == -7)
            streams[b] += want
            texts[b] += rows[b].tolist()
        _check_books(cb, books)
    # replay of both parts in two calls, with an oracle that takes one online update per code
    rb = [olzw.Codebook(V, M, cap) for _ in range(B)]
    cb2 = _session(V, M, cap, B)
    for lo, hi in ((0, 0.4), (0.4, 1.0)):
        part = [s[int(len(s) * lo):int(len(s) * hi)] for s in streams]
        Tc = max(max(len(s) for s in part), 1)
        c = np.full((B, Tc), -1, dtype=np.int32)
        for b, s in enumerate(part):
            c[b, :len(s)] = s
            for z in s:
                rb[b].step(z)
                if rb[b].status & olzw.BAD_TOKEN:       # (two greedy parses back to back need not replay as one)
                    break
        T_out = M * Tc
        out = torch.full((B, T_out), -9, dtype=torch.int32, device=DEV)
        olen = torch.zeros(B, dtype=torch.int32, device=DEV)
        zb.z2z_lzw_decode(cb2, torch.from_numpy(c).to(DEV),
                          torch.tensor([len(s) for s in part], dtype=torch.int32, device=DEV), zb.DECODE_REPLAY, out, olen)
        for b, s in enumerate(part):
            want, _ = olzw.expand(rb[b], s if not rb[b].status & olzw.BAD_TOKEN else s[:int(olen[b])])
            if not rb[b].status & olzw.BAD_TOKEN:
                assert out[b, :int(olen[b])].cpu().tolist() == want
        if any(r.status & olzw.BAD_TOKEN for r in rb):
            return
    _check_books(cb2, rb)


@pytest.mark.parametrize("cap", [200, 16385])
def test_replay_stops_at_a_code_without_entry_anywhere_in_a_window(cap):
    rng = np.random.default_rng(5)
    V, M = 20, 4
    x = rng.integers(0, V, size=900).tolist()
    good, _, _ = olzw.encode(x, V, M, cap)
    cuts = [0, 1, 2, 63, 127, 128, 129, 200, len(good) - 1]
    B = len(cuts)
    cb = _session(V, M, cap, B)
    c = np.tile(np.asarray(good, dtype=np.int32), (B, 1))
    books = []
    for b, at in enumerate(cuts):
        ob = olzw.Codebook(V, M, cap)
        for z in good[:at]:
            ob.step(z)
        c[b, at] = V + ob.n() + 1 if b % 2 else -3      # beyond the next entry; negative
        ob.step(int(c[b, at]))
        books.append(ob)
    out = torch.full((B, 1000), -9, dtype=torch.int32, device=DEV)
    olen = torch.zeros(B, dtype=torch.int32, device=DEV)
    zb.z2z_lzw_decode(cb, torch.from_numpy(c).to(DEV), None, zb.DECODE_REPLAY, out, olen)
    _check_books(cb, books)
    for b, at in enumerate(cuts):
        want, _ = olzw.expand(books[b], good[:at])
        assert out[b, :int(olen[b])].cpu().tolist() == want
