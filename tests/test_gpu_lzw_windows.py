"""Windowed LZW parse and replay at the sizes where a window can go wrong: its edges (256 positions, 64 in
a batch of more than two sequences per SM; matches that cross them; the ring of tokens, twice as long), tiny
alphabets in which most windows end early because a phrase repeats inside them, codebooks that fill up
inside a window, both homes of the table (shared memory while it fits, global memory for larger codebooks
and short calls), sessions that continue, codes that name no entry.  Bit-exact."""
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


def _check_books(cb, books, copies=1):
    st, n = zb.z2z_status(cb)
    for c in range(1, copies):                          # the same counts and status everywhere, the last copy's entries too
        k = len(books)
        assert torch.equal(st[c * k:(c + 1) * k], st[:k]) and torch.equal(n[c * k:(c + 1) * k], n[:k])
    for b, ob in list(enumerate(books)) + [((copies - 1) * len(books) + b, ob) for b, ob in enumerate(books) if copies > 1]:
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


def _accepts(book, z):
    """One online update; whether the code named an entry (the status bit of an earlier one stays)."""
    before, book.status = book.status, book.status & ~olzw.BAD_TOKEN
    book.step(z)
    ok = not book.status & olzw.BAD_TOKEN
    book.status |= before
    return ok


LENS = [0, 1, 7, 63, 64, 65, 71, 72, 73, 127, 128, 129, 135, 136, 255, 256, 257, 263, 264, 265, 511, 512, 513, 520, 1000, 2049]


@pytest.mark.parametrize("kind", ["random", "run", "period"])
@pytest.mark.parametrize("copies", [1, 12])             # 26 and 312 sequences
@pytest.mark.parametrize("V,M,cap", [(2, 8, 4096), (3, 2, 300), (7, 5, 16384), (50, 3, 70), (1000, 8, 16385), (40, 4, 0)])
def test_windows_match_the_oracle(V, M, cap, copies, kind):
    rng = np.random.default_rng(V * 131 + M)
    n, T = len(LENS), max(LENS)
    B = n * copies
    cb = _session(V, M, cap, B)
    books = [olzw.Codebook(V, M, cap) for _ in range(n)]
    streams = [[] for _ in range(n)]
    for part in range(2):                               # the second call continues from the first one's codebooks
        rows = [_stream(rng, V, L, kind) for L in LENS]
        codes, clen, after = _encode(cb, rows * copies, T)
        for c in range(1, copies):
            for x in (codes, clen, after):
                assert np.array_equal(x[c * n:(c + 1) * n], x[:n])
        for b in range(n):
            want, want_after = books[b].encode(rows[b].tolist())
            assert codes[b, :clen[b]].tolist() == want
            assert after[b, :clen[b]].tolist() == want_after
            assert np.all(codes[b, clen[b]:] == -7) and np.all(after[b, clen[b]:] == -7)
            streams[b] += want
    _check_books(cb, books, copies)
    # replay of both parts in two calls, with an oracle that takes one online update per code (two greedy
    # parses back to back need not replay as one: such a stream ends at the first code without an entry)
    rb = [olzw.Codebook(V, M, cap) for _ in range(n)]
    cb2 = _session(V, M, cap, B)
    for lo, hi in ((0, 0.4), (0.4, 1.0)):
        part = [s[int(len(s) * lo):int(len(s) * hi)] for s in streams]
        Tc = max(max(len(s) for s in part), 1)
        c = np.full((n, Tc), -1, dtype=np.int32)
        taken = []
        for b, s in enumerate(part):
            c[b, :len(s)] = s
            taken.append(next((i for i, z in enumerate(s) if not _accepts(rb[b], z)), len(s)))
        out = torch.full((B, M * Tc), -9, dtype=torch.int32, device=DEV)
        olen = torch.zeros(B, dtype=torch.int32, device=DEV)
        zb.z2z_lzw_decode(cb2, torch.from_numpy(np.tile(c, (copies, 1))).to(DEV),
                          torch.tensor([len(s) for s in part] * copies, dtype=torch.int32, device=DEV), zb.DECODE_REPLAY, out, olen)
        out, olen = out.cpu().numpy(), olen.cpu().numpy()
        for c in range(1, copies):
            assert np.array_equal(out[c * n:(c + 1) * n], out[:n]) and np.array_equal(olen[c * n:(c + 1) * n], olen[:n])
        for b, s in enumerate(part):
            want, _ = olzw.expand(rb[b], s[:taken[b]])
            assert out[b, :olen[b]].tolist() == want
    _check_books(cb2, rb, copies)


@pytest.mark.parametrize("copies", [1, 40])             # 9 and 360 sequences: blocks of 512 and 128 threads
@pytest.mark.parametrize("cap", [1600, 16385])          # table in shared and in global memory
def test_entries_around_one_per_thread(cap, copies):
    """What a call has made is written back one entry per thread or four at a time."""
    sizes, V, M = [1, 127, 128, 129, 511, 512, 513, 514, 1500], 5000, 3
    rows = [np.random.default_rng(b).permutation(V)[:k + 1].astype(np.int32) for b, k in enumerate(sizes)]
    cb = _session(V, M, cap, len(rows) * copies)
    books = [olzw.Codebook(V, M, cap) for _ in rows]
    codes, clen, _ = _encode(cb, rows * copies, max(sizes) + 1)
    for b, r in enumerate(rows):
        assert codes[b, :clen[b]].tolist() == books[b].encode(r.tolist())[0] and books[b].n() == sizes[b]
    _check_books(cb, books, copies)
    cb2 = _session(V, M, cap, len(rows) * copies)
    out, olen = torch.zeros(codes.shape, dtype=torch.int32, device=DEV), torch.zeros(len(codes), dtype=torch.int32, device=DEV)
    zb.z2z_lzw_decode(cb2, torch.from_numpy(codes).to(DEV), torch.from_numpy(clen).to(DEV), zb.DECODE_REPLAY, out, olen)
    for b, r in enumerate(rows * copies):
        assert out[b, :olen[b]].tolist() == r.tolist()
    _check_books(cb2, books, copies)


@pytest.mark.parametrize("B", [3, 400])
@pytest.mark.parametrize("T", [1, 20, 63, 64, 65])
def test_short_calls_use_the_table_in_place(T, B):
    """A codebook of 16384 entries has 32768 slots: calls of fewer than 64 tokens do not bring them in.  Short and
    longer calls take turns on the same codebooks."""
    V, M, cap = 9, 4, 16384
    rng = np.random.default_rng(T)
    cb = _session(V, M, cap, B)
    books = [olzw.Codebook(V, M, cap) for _ in range(3)]
    for L in (200, T, T, 300, T):
        rows = [_stream(rng, V, L, k) for k in ("random", "run", "period")]
        codes, clen, _ = _encode(cb, [rows[b % 3] for b in range(B)], L)
        for b in range(3):
            assert codes[b, :clen[b]].tolist() == books[b].encode(rows[b].tolist())[0]
    _check_books(cb, [books[b % 3] for b in range(min(B, 12))])


@pytest.mark.parametrize("copies", [1, 16])            # 20 and 320 sequences
@pytest.mark.parametrize("cap", [200, 16384, 16385])
def test_replay_stops_at_a_code_without_entry_anywhere_in_a_window(cap, copies):
    rng = np.random.default_rng(5)
    V, M = 200, 4
    x = rng.integers(0, V, size=1200).tolist()
    good, _, _ = olzw.encode(x, V, M, cap)
    cuts = [0, 1, 2, 62, 63, 64, 65, 127, 128, 129, 191, 192, 200, 255, 256, 257, 511, 512, 513, len(good) - 1]
    assert len(good) > 514
    cuts = cuts * copies
    B = len(cuts)
    cb = _session(V, M, cap, B)
    c = np.tile(np.asarray(good, dtype=np.int32), (B, 1))
    books = []
    for b, at in enumerate(cuts):
        if b >= B // copies:
            books.append(books[b % (B // copies)])
            c[b] = c[b % (B // copies)]
            continue
        ob = olzw.Codebook(V, M, cap)
        for z in good[:at]:
            ob.step(z)
        c[b, at] = V + ob.n() + 1 if b % 2 else -3      # beyond the next entry; negative
        ob.step(int(c[b, at]))
        books.append(ob)
    out = torch.full((B, 1300), -9, dtype=torch.int32, device=DEV)
    olen = torch.zeros(B, dtype=torch.int32, device=DEV)
    zb.z2z_lzw_decode(cb, torch.from_numpy(c).to(DEV), None, zb.DECODE_REPLAY, out, olen)
    _check_books(cb, books)
    out, olen = out.cpu().numpy(), olen.cpu().numpy()
    for b, at in enumerate(cuts):
        want, _ = olzw.expand(books[b], good[:at])
        assert out[b, :olen[b]].tolist() == want
