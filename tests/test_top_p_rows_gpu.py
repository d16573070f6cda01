"""massv_sample_top_p where its row-per-cluster kernel can go wrong: one entry, slices with a ragged last group, rows that
start off a 16-byte boundary, a last CTA with few entries or none, every cluster size, ties cut between two CTAs, the
longest row that fits, and the first one that does not (the one-CTA kernel)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _check(z, u, T, top_p, allow=0):
    import paper_2505_10526_b200 as mv
    rows, vocab = z.shape
    tok = torch.full((rows,), -5, dtype=torch.int32, device="cuda")
    pad = torch.full((rows * vocab + 8,), -1.0, device="cuda")
    q = pad[4:4 + rows * vocab].view(rows, vocab)
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    mv.massv_sample_top_p(z, u, tok, T, top_p, q, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert float(pad[:4].max()) == -1.0 and float(pad[4 + rows * vocab:].max()) == -1.0
    ref = oracle.sample_top_p(z.cpu().numpy(), u.cpu().numpy(), T, top_p)
    qg, tg = q.cpu().double().numpy(), tok.cpu().numpy()
    moved = 0
    for r in range(rows):
        same = np.array_equal(qg[r] > 0, ref["q"][r] > 0)
        # fp32 weights against fp64 ones: the mass at which the prefix stops is known to about 1e-6 of the total
        if not same and ref["margin_set"][r] < 1e-5:
            moved += 1
            continue
        assert same, (r, int((qg[r] > 0).sum()), int(ref["nucleus_size"][r]))
        assert np.abs(qg[r] - ref["q"][r]).max() < 1e-4
        assert tg[r] == ref["token"][r] or ref["margin_sample"][r] < 1e-5, (r, tg[r], ref["token"][r])
    assert moved <= allow
    tok2 = torch.empty_like(tok)
    mv.massv_sample_top_p(z, u, tok2, T, top_p, None, status)        # without the distribution, and again: the same tokens
    assert torch.equal(tok, tok2)


@pytest.mark.parametrize("rows,vocab", [(1, 1), (2, 3), (1, 4095), (3, 4097), (1, 8192), (150, 1021), (40, 21 * 1024), (37, 21 * 1024 + 1),
                                        (18, 43009), (1, 131071), (9, 152064), (2, 48 * 1024 * 8), (2, 48 * 1024 * 8 + 1)])
def test_sizes(rows, vocab):
    g = torch.Generator(device="cuda").manual_seed(vocab)
    z = torch.randn((rows, vocab), generator=g, device="cuda") * 4.0
    z[:, vocab // 2:vocab // 2 + vocab // 8] = -float("inf")
    _check(z, torch.rand((rows,), generator=g, device="cuda"), 0.8, 0.9, allow=1 + rows // 16)


@pytest.mark.parametrize("vocab,shift", [(8192, 1), (50264, 2), (152064, 3)])
def test_rows_off_the_alignment(vocab, shift):
    g = torch.Generator(device="cuda").manual_seed(vocab)
    z = torch.randn((3 * vocab + 4,), generator=g, device="cuda")[shift:shift + 3 * vocab].view(3, vocab)
    _check(z, torch.rand((3,), generator=g, device="cuda"), 1.0, 0.7, allow=1)


@pytest.mark.parametrize("top_p", [0.25, 0.5, 0.75, 1.0])
def test_ties_over_several_ctas(top_p):
    """Two levels of logit only: the prefix stops among equal weights, at an index that every CTA has to agree on.  The
    weights are powers of two, so all masses are exact and the last member is known."""
    vocab, rows = 65536, 4
    z = torch.full((rows, vocab), -30.0, device="cuda")
    for r in range(rows):
        z[r, torch.randperm(vocab, generator=torch.Generator().manual_seed(r))[:8192].cuda()] = 3.0
    import paper_2505_10526_b200 as mv
    u = torch.tensor([0.0, 0.3, 0.7, 0.9999], device="cuda")
    tok = torch.empty((rows,), dtype=torch.int32, device="cuda")
    q = torch.empty_like(z)
    # temperature 33 ln 2: the lower level weighs 2^-1 ... of the upper at T = 33 / ln 2 / 40: mass 57344 * 2^-40 of 8192
    T = 33.0 * 1.4426950408889634 / 40.0
    mv.massv_sample_top_p(z, u, tok, T, top_p, q, None)
    torch.cuda.synchronize()
    for r in range(rows):
        heavy = torch.nonzero(z[r] > 0).flatten()
        members = torch.nonzero(q[r] > 0).flatten()
        # the light entries weigh 57,344 * 2^-40 = 5e-8 of one heavy one: at top_p below 1 the prefix ends inside the heavy ones, one
        # more than top_p * 8192 where the light mass tips the ceiling; at 1 it takes everything
        if top_p < 1.0:
            k = members.numel()
            assert k in (int(top_p * 8192), int(top_p * 8192) + 1)
            assert torch.equal(members, heavy[:k])
            assert int(tok[r]) == int(heavy[int(float(u[r]) * k)])
        else:
            assert members.numel() == vocab


def test_rows_without_a_finite_logit():
    import paper_2505_10526_b200 as mv
    z = torch.randn((5, 60000), device="cuda")
    z[3] = -float("inf")
    tok = torch.full((5,), -5, dtype=torch.int32, device="cuda")
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    mv.massv_sample_top_p(z, torch.full((5,), 0.5, device="cuda"), tok, 1.0, 0.9, None, status)
    torch.cuda.synchronize()
    assert int(status.item()) == -1 and int(tok[3]) == 0 and int(tok.min()) >= 0


@pytest.mark.parametrize("vocab", [8192, 50264, 152064])
def test_rows_come_out_the_same_in_calls_of_any_size(vocab):
    """The number of rows decides how many CTAs share a row, and with it the grouping of the fp64 sums: the set of tokens is exact (integer
    masses), the normalisation may differ in its last bit, and a draw only where u falls on a step of the CDF."""
    import paper_2505_10526_b200 as mv
    g = torch.Generator(device="cuda").manual_seed(vocab)
    z = 4.0 * torch.randn((150, vocab), generator=g, device="cuda")
    u = torch.rand((150,), generator=g, device="cuda")

    def run(rows, top_p):
        tok, q = torch.empty((rows,), dtype=torch.int32, device="cuda"), torch.empty((rows, vocab), device="cuda")
        mv.massv_sample_top_p(z[:rows], u[:rows], tok, 0.9, top_p, q, None)
        return tok, q

    for top_p in (0.8, 1.0):
        tok, q = run(150, top_p)
        for rows in (1, 5, 16, 40, 90):
            t, p = run(rows, top_p)
            assert torch.equal(p > 0, q[:rows] > 0)
            assert float(((p - q[:rows]).abs() / q[:rows].clamp_min(1e-30)).max()) <= 2.0 ** -22
            cdf = torch.cumsum(q[:rows].double(), -1)
            at = t.long().clamp_min(1)
            gap = torch.minimum((cdf.gather(-1, t.long()[:, None])[:, 0] - u[:rows]).abs(), (cdf.gather(-1, (at - 1)[:, None])[:, 0] - u[:rows]).abs())
            assert bool(((t == tok[:rows]) | (gap < 1e-6)).all())


@pytest.mark.parametrize("std", [0.01, 0.3, 1.5, 8.0])
@pytest.mark.parametrize("top_p", [0.05, 0.6, 0.97, 1.0])
def test_levels(std, top_p):
    """From rows whose first level holds thousands of entries in a bin to rows that need one level, thresholds among the heavy and
    among the light entries, and the whole row (there entries below 2^-44 of the largest, 5e4 * 2^-44 = 3e-9 of the mass, are left out)."""
    g = torch.Generator(device="cuda").manual_seed(int(100 * std) + int(100 * top_p))
    z = std * torch.randn((5, 50264), generator=g, device="cuda")
    z[1, ::3] = -float("inf")
    z[2, 100:] = -float("inf")
    _check(z, torch.rand((5,), generator=g, device="cuda"), 1.0, top_p, allow=5 if top_p == 1.0 else 2)


@pytest.mark.parametrize("rows,vocab", [(1, 262144), (3, 262144), (2, 393216), (2, 400000)])
def test_the_whole_row_whatever_its_mass(rows, vocab):
    """top_p = 1 takes every entry that has mass, also where the row's mass in units of 2^-44 has more bits than a double: flat rows with
    five entries of 2^-40, 80 units in all, less than half a step of the double next to the row's sum of 2^62."""
    import paper_2505_10526_b200 as mv
    T = 1.4426950408889634                       # weights 2^(z - max)
    z = torch.zeros((rows, vocab), device="cuda")
    g = torch.Generator(device="cuda").manual_seed(vocab)
    at = torch.stack([torch.randperm(vocab, generator=g, device="cuda")[:5] for _ in range(rows)])
    z.scatter_(1, at, -40.0)
    tok = torch.empty((rows,), dtype=torch.int32, device="cuda")
    q = torch.empty_like(z)
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    mv.massv_sample_top_p(z, torch.full((rows,), 0.5, device="cuda"), tok, T, 1.0, q, status)
    assert int(status.item()) == 0
    assert bool((q > 0).all())
