"""Joint logits at the sizes where the CTA-pair kernel's split can go wrong: every number of rows around a
change of the rows per CTA or of the row tiles, vocabularies that end inside a granule of 64, widths that
are no multiple of 256 (also for decode batches of up to 32 rows), sequences with 0, 1, 63 .. 65 and 300
visible entries, rows without an owner, targets in and outside of what a row sees.  Against fp64 sums."""
import numpy as np
import pytest
import torch

from paper_2506_01084_b200 import binding as zb

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _session(V, d, B, cap, counts, seed):
    """Codebooks of exactly the given sizes: runs of distinct pairs compressed as prompts."""
    cb = zb.Codebook(zb.make_config(V, d, 2, cap, B, "bf16", 0, 1, 8), DEV)
    T = 2 * max(max(counts), 1) + 2
    tok = np.zeros((B, T), dtype=np.int32)
    lens = []
    for b, n in enumerate(counts):
        seen, row = set(), [b % V]
        rng = np.random.default_rng(seed + b)
        while len(seen) < n:                             # a walk whose every step is a pair not seen before
            c = int(rng.integers(0, V))
            if (row[-1], c) not in seen:
                seen.add((row[-1], c))
                row.append(c)
        tok[b, :len(row)] = row
        lens.append(len(row))
    codes = torch.zeros(B, T, dtype=torch.int32, device=DEV)
    clen = torch.zeros(B, dtype=torch.int32, device=DEV)
    zb.z2z_lzw_encode(cb, torch.from_numpy(tok).to(DEV), torch.tensor(lens, dtype=torch.int32, device=DEV), codes, clen, None)
    _, n = zb.z2z_status(cb)
    assert [int(x) for x in n] == list(counts)
    return cb


@pytest.mark.parametrize("B", [33, 90, 128, 200])
@pytest.mark.parametrize("V,d", [(1003, 192), (4097, 1152)])
def test_sampled_batch_of_one_row_per_sequence(V, d, B):
    """Gumbel-max over every column, in and beyond the batch kernel's 128 rows: the sample has to be the
    argmax of the perturbed scores, which the oracle draws column by column."""
    from oracle import logits as olg
    counts = [(7 * b) % 70 for b in range(B)]
    cap, T, seed, step = 80, 0.9, 77, 5
    cb = _session(V, d, B, cap, counts, 4)
    g = torch.Generator(device=DEV)
    g.manual_seed(B + V)
    rnd = lambda *s, std: (torch.randn(*s, generator=g, device=DEV) * std).to(torch.bfloat16)
    hid, WU, Uh = rnd(B, d, std=1.0), rnd(V, d, std=0.05), rnd(B, cap, d, std=0.05)
    lse, mx = torch.zeros(B, device=DEV), torch.zeros(B, device=DEV)
    am, sm = torch.zeros(B, dtype=torch.int32, device=DEV), torch.zeros(B, dtype=torch.int32, device=DEV)
    zb.z2z_dynamic_logits(cb, hid, None, None, WU, Uh, zb.SELECT_GUMBEL, T, seed, step, None, lse, am, mx, sm)
    h, w, u = hid.double().cpu().numpy(), WU.double().cpu().numpy(), Uh.double().cpu().numpy()
    for r in range(B):
        l = np.concatenate([w @ h[r], u[r, :counts[r]] @ h[r]])
        choice, scores, gap = olg.select(l, 1, T, seed, step, r)
        # a score is a logit (error below 1e-4 here) plus noise in fp32 (error below 1e-5 at |g| < 20)
        assert scores[int(sm[r])] >= scores[choice] - 5e-4
        assert abs(float(lse[r]) - (l.max() + np.log(np.exp(l - l.max()).sum()))) < 1e-4


@pytest.mark.parametrize("V,d,B", [(257, 192, 33), (1000, 1152, 47), (257, 64, 128), (14100, 192, 47), (14300, 64, 70)])
def test_batch_with_hypertokens_of_every_job_size(V, d, B):
    """Jobs of 1 to 8 granules of 32 hypertokens: boxes of one, two and four k-blocks, of which the last one ends
    beyond the width, on the group of 8 hidden rows that holds the sequence's; vocabularies on both sides of
    three granules of 32 columns per CTA, from which the shares are even; stored logits too."""
    sizes = [0, 1, 31, 32, 33, 64, 65, 96, 97, 128, 129, 160, 161, 255, 256, 257, 300]
    counts = [sizes[(5 * b) % len(sizes)] for b in range(B)]
    cap = 300
    cb = _session(V, d, B, cap, counts, 8)
    g = torch.Generator(device=DEV)
    g.manual_seed(B)
    rnd = lambda *s, std: (torch.randn(*s, generator=g, device=DEV) * std).to(torch.bfloat16)
    hid, WU, Uh = rnd(B, d, std=1.0), rnd(V, d, std=0.05), rnd(B, cap, d, std=0.05)
    for b in range(B):
        Uh[b, counts[b]:] = float("nan")                     # rows that are no entries are loaded at most
    lse, mx = torch.zeros(B, device=DEV), torch.zeros(B, device=DEV)
    am = torch.zeros(B, dtype=torch.int32, device=DEV)
    out = torch.full((B, V + cap), -7.0, device=DEV)
    zb.z2z_dynamic_logits(cb, hid, None, None, WU, Uh, zb.SELECT_ARGMAX, 1.0, 0, 0, None, lse, am, mx, logits_debug=out)
    st, _ = zb.z2z_status(cb)
    assert all(int(s) & zb.ST_WAIT_TIMEOUT == 0 for s in st)
    for r in range(B):
        l = torch.cat([WU.double() @ hid[r].double(), Uh[r, :counts[r]].double() @ hid[r].double()])
        tol = 2e-5 * (1 + float(l.abs().max()))
        assert float((out[r, :V + counts[r]].double() - l).abs().max()) < tol
        assert torch.all(out[r, V + counts[r]:] == -7)
        assert abs(float(lse[r]) - float(torch.logsumexp(l, 0))) < tol
        assert float(l.max() - l[int(am[r])]) < 2 * tol and abs(float(mx[r]) - float(l.max())) < tol


@pytest.mark.parametrize("select", [0, 1])
@pytest.mark.parametrize("given", ["no", "one", "several"])
@pytest.mark.parametrize("N", [33, 70, 128])
@pytest.mark.parametrize("granules,d", [(0.5, 448), (3, 448), (8.5, 448), (19.3, 320)])
def test_batch_with_several_column_jobs_per_cta(granules, d, N, given, select):
    """Even shares of W_U: three granules of 32 columns per CTA (the fewest that are dealt so), one job of 256 columns
    and a rest, two of them and a rest; more k-blocks than the ring has stages (five up to 40 rows, four at
    128); behind them the hypertokens.  Below three granules one share of both.  Rows in the order of their sequences, or given
    with them, their limits and targets: one per sequence, or several, in one group of 8 rows, in several, or of none."""
    from oracle import logits as olg
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    V = 32 * int(granules * sms) - (5 if granules > 3 else 0)
    assert ((V + 31) // 32 >= 3 * sms) == (granules >= 3)
    sizes = [0, 1, 33, 64, 100, 129, 256, 300]
    B, cap, T, seed, step = N + 2, 300, 0.9, 77, 5
    counts = [sizes[(3 * b) % len(sizes)] for b in range(B)]
    cb = _session(V, d, B, cap, counts, 9)
    g = torch.Generator(device=DEV)
    g.manual_seed(N + V)
    rnd = lambda *s, std: (torch.randn(*s, generator=g, device=DEV) * std).to(torch.bfloat16)
    hid, WU, Uh = rnd(N, d, std=1.0), rnd(V, d, std=0.05), rnd(B, cap, d, std=0.05)
    for b in range(B):
        Uh[b, counts[b]:] = float("nan")                     # rows that are no entries are loaded at most
    seq = nvis = tgt = tl = None
    own, vis = list(range(N)), counts[:N]
    if given != "no":
        seq = torch.randperm(B, generator=g, device=DEV)[:N].to(torch.int32)
        if given == "several":
            seq = torch.arange(N, device=DEV, dtype=torch.int32) // 3
            seq[::7] = seq[::7].flip(0)
            seq[5], seq[6] = -1, B
        nvis = torch.randint(0, cap + 1, (N,), generator=g, device=DEV, dtype=torch.int32)
        tgt = torch.randint(0, V + cap, (N,), generator=g, device=DEV, dtype=torch.int32)
        tgt[::3] = V + torch.arange(N, device=DEV, dtype=torch.int32)[::3]
        tl = torch.zeros(N, device=DEV)
        own = seq.tolist()
        vis = [min(v, counts[o]) if 0 <= o < B else 0 for v, o in zip(nvis.tolist(), own)]
    lse, mx = torch.zeros(N, device=DEV), torch.zeros(N, device=DEV)
    am, sm = (torch.full((N,), -9, dtype=torch.int32, device=DEV) for _ in range(2))
    out = None if select else torch.full((N, V + cap), -7.0, device=DEV)
    zb.z2z_dynamic_logits(cb, hid, seq, nvis, WU, Uh, select, T, seed, step, tgt, lse, am, mx, sm if select else None, tl, out)
    st, _ = zb.z2z_status(cb)
    assert all(int(s) & zb.ST_WAIT_TIMEOUT == 0 for s in st)
    base = hid.double() @ WU.double().T
    for r in range(N):
        if not 0 <= own[r] < B:
            continue                                         # a row without an owner sees nothing
        l = torch.cat([base[r], Uh[own[r], :vis[r]].double() @ hid[r].double()])
        tol = 2e-5 * (1 + float(l.abs().max()))              # fp32 sums of d products, as below
        assert abs(float(lse[r]) - float(torch.logsumexp(l, 0))) < tol
        assert abs(float(mx[r]) - float(l.max())) < tol and float(l.max() - l[int(am[r])]) < 2 * tol
        if tgt is not None and int(tgt[r]) < len(l):
            assert abs(float(tl[r]) - float(l[int(tgt[r])])) < tol
        elif tgt is not None:
            assert torch.isnan(tl[r])
        if out is not None:
            assert float((out[r, :len(l)].double() - l).abs().max()) < tol and torch.all(out[r, len(l):] == -7)
        if select and r % 8 in (0, 5):
            # a score is a logit (error below 1e-4 here) plus noise in fp32 (error below 1e-5 at |g| < 20)
            choice, scores, _ = olg.select(l.cpu().numpy(), 1, T, seed, step, r)
            assert scores[int(sm[r])] >= scores[choice] - 5e-4


@pytest.mark.parametrize("N", [1, 31, 32, 33, 64, 65, 96, 128, 129, 192, 193, 256, 257, 511, 700])
@pytest.mark.parametrize("V,d", [(4097, 192), (1000, 1152), (130, 2176)])
def test_joint_logits_against_fp64(V, d, N):
    counts = [0, 1, 63, 64, 65, 300]
    B, cap = len(counts), 320
    cb = _session(V, d, B, cap, counts, 3)
    g = torch.Generator(device=DEV)
    g.manual_seed(N * 7 + V)
    rnd = lambda *s, std: (torch.randn(*s, generator=g, device=DEV) * std).to(torch.bfloat16)
    hid, WU, Uh = rnd(N, d, std=1.0), rnd(V, d, std=0.05), rnd(B, cap, d, std=0.05)
    seq = torch.randint(0, B, (N,), generator=g, device=DEV, dtype=torch.int32).sort().values
    nvis = torch.randint(0, cap, (N,), generator=g, device=DEV, dtype=torch.int32)
    if N > 40:
        seq[N // 2] = -1                                  # a row without an owner sees nothing
    tgt = torch.randint(0, V + cap, (N,), generator=g, device=DEV, dtype=torch.int32)
    out = dict(lse=torch.zeros(N, device=DEV), am=torch.zeros(N, dtype=torch.int32, device=DEV),
               mx=torch.zeros(N, device=DEV), tl=torch.zeros(N, device=DEV))
    zb.z2z_dynamic_logits(cb, hid, seq, nvis, WU, Uh, zb.SELECT_ARGMAX, 1.0, 0, 0, tgt, out["lse"], out["am"], out["mx"],
                          None, out["tl"])
    st, _ = zb.z2z_status(cb)
    assert all(int(s) & zb.ST_WAIT_TIMEOUT == 0 for s in st)
    h, w, u = hid.double(), WU.double(), Uh.double()
    for r in range(N):
        s = int(seq[r])
        if s < 0:
            continue
        vis = min(int(nvis[r]), counts[s])
        l = torch.cat([w @ h[r], u[s, :vis] @ h[r]])
        # fp32 sums of d products of size std 0.05: relative 2^-24 sqrt(d) of their 2-norm, well under 2e-5
        assert abs(float(out["lse"][r]) - float(torch.logsumexp(l, 0))) < 2e-5 * (1 + float(l.abs().max()))
        assert abs(float(out["mx"][r]) - float(l.max())) < 2e-5 * (1 + float(l.abs().max()))
        assert float(l.max() - l[int(out["am"][r])]) < 4e-5 * (1 + float(l.abs().max()))
        t = int(tgt[r])
        if t < V + vis:
            assert abs(float(out["tl"][r]) - float(l[t])) < 2e-5 * (1 + float(l.abs().max()))
        else:
            assert torch.isnan(out["tl"][r])


@pytest.mark.parametrize("N", [33, 100, 128])
def test_a_batch_given_with_its_sequences_takes_the_batch_kernel(N):
    """In order, in another order, a part of the batch, several rows of one sequence: the same kernels as without
    d_row_seq (counted by their launches), and the right logits."""
    V, d, B, cap = 1003, 256, 128, 80
    counts = [(7 * b) % 70 for b in range(B)]
    cb = _session(V, d, B, cap, counts, 6)
    g = torch.Generator(device=DEV)
    g.manual_seed(N)
    rnd = lambda *s, std: (torch.randn(*s, generator=g, device=DEV) * std).to(torch.bfloat16)
    hid, WU, Uh = rnd(N, d, std=1.0), rnd(V, d, std=0.05), rnd(B, cap, d, std=0.05)
    order = torch.randperm(B, generator=g, device=DEV)[:N].to(torch.int32)
    seqs = [None, torch.arange(N, device=DEV, dtype=torch.int32), order, order // 3]
    launches = []
    for seq in seqs:
        lse = torch.zeros(N, device=DEV)
        zb.z2z_profile_read(cb)
        zb.z2z_dynamic_logits(cb, hid, seq, None, WU, Uh, zb.SELECT_ARGMAX, 1.0, 0, 0, None, lse, None, None)
        launches.append(zb.z2z_profile_read(cb)[1])
        own = list(range(N)) if seq is None else seq.tolist()
        for r in range(0, N, 5):
            l = torch.cat([WU.double() @ hid[r].double(), Uh[own[r], :counts[own[r]]].double() @ hid[r].double()])
            assert abs(float(lse[r]) - float(torch.logsumexp(l, 0))) < 2e-5 * (1 + float(l.abs().max()))
    assert all(x == launches[0] for x in launches)


def test_overflowed_logit_keeps_its_row_a_number():
    N = 100
    cb = _session(300, 256, N, 8, [1] * N, 5)
    hid = torch.ones(N, 256, dtype=torch.bfloat16, device=DEV)
    WU = torch.zeros(300, 256, dtype=torch.bfloat16, device=DEV)
    WU[77] = 3e38                                         # one column of +inf, the others 0
    Uh = torch.zeros(N, 8, 256, dtype=torch.bfloat16, device=DEV)
    lse, mx = torch.zeros(N, device=DEV), torch.zeros(N, device=DEV)
    am = torch.zeros(N, dtype=torch.int32, device=DEV)
    zb.z2z_dynamic_logits(cb, hid, None, None, WU, Uh, zb.SELECT_ARGMAX, 1.0, 0, 0, None, lse, am, mx)
    assert torch.all(torch.isposinf(lse)) and torch.all(torch.isposinf(mx)) and torch.all(am == 77)


@pytest.mark.parametrize("N,B", [(33, 33), (100, 100), (40, 5), (200, 200), (300, 5), (2100, 5)])
@pytest.mark.parametrize("select", [0, 1])
@pytest.mark.parametrize("which", ["two_inf", "first_neg_inf", "many_neg_inf", "all_neg_inf"])
def test_overflowed_logits_leave_the_sum_a_number(N, B, select, which):
    """Overflowed columns anywhere, beyond the decode kernel's 32 rows: several of +inf give +inf, those of -inf add
    nothing, a row of nothing else is -inf, however the columns are split."""
    V, d = 1000, 128
    cb = _session(V, d, B, 8, [1] * B, 5)
    hid = torch.ones(N, d, dtype=torch.bfloat16, device=DEV)
    WU = torch.zeros(V, d, dtype=torch.bfloat16, device=DEV)
    WU[:, 0] = torch.arange(V, device=DEV).fmod(7).to(torch.bfloat16)
    Uh = torch.zeros(B, 8, d, dtype=torch.bfloat16, device=DEV)
    cols = {"two_inf": [77, 500], "first_neg_inf": [0, 1, 2], "many_neg_inf": list(range(250, 420)) + list(range(900, V)),
            "all_neg_inf": list(range(V))}[which]
    WU[cols] = 3e38 if which == "two_inf" else -3e38
    if which == "all_neg_inf":
        Uh[:] = -3e38
    seq = None if N == B else (torch.arange(N, device=DEV) * B // N).to(torch.int32)
    lse, mx = torch.zeros(N, device=DEV), torch.zeros(N, device=DEV)
    am, sm = torch.zeros(N, dtype=torch.int32, device=DEV), torch.zeros(N, dtype=torch.int32, device=DEV)
    zb.z2z_dynamic_logits(cb, hid, seq, None, WU, Uh, select, 1.0, 1, 2, None, lse, am, mx, sm if select else None)
    l = torch.cat([WU[:, 0].double(), torch.zeros(1, dtype=torch.float64, device=DEV)])
    l[cols] = float("inf") if which == "two_inf" else float("-inf")
    if which == "all_neg_inf":
        l[-1] = float("-inf")
    want = float(torch.logsumexp(l, 0))
    assert torch.all(mx == float(l.max())) and torch.all(am == int(l.argmax()))
    assert torch.all(lse == want) if abs(want) == float("inf") else torch.all((lse - want).abs() < 1e-5 * (1 + abs(want)))
