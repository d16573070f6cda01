"""The warp-MMA kernel at head_dim 256, its balanced schedule (pairs cut between CTAs, ranges of several pairs, every number of row
groups, windows) and the chunk grid where the rule keeps it; lengths from zero, ragged ends; against attention in 64 bits on the
same bf16 values."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def _inputs(batch, gamma, q_heads, kv_heads, lens, seed, max_pages=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    R, d = gamma + 1, 256
    max_pages = max_pages or (max(lens) + R + 15) // 16
    n_pages = batch * max_pages + 2
    bf = dict(dtype=torch.bfloat16, device="cuda", generator=g)
    table = torch.randperm(n_pages, generator=g, device="cuda")[:batch * max_pages].view(batch, max_pages).to(torch.int32)
    return dict(q=torch.randn((batch, R, q_heads, d), **bf), k_new=torch.randn((batch, R, kv_heads, d), **bf),
                v_new=torch.randn((batch, R, kv_heads, d), **bf), k_pages=torch.randn((n_pages, kv_heads, 16, d), **bf),
                v_pages=torch.randn((n_pages, kv_heads, 16, d), **bf), page_table=table.contiguous(),
                seq_lens=torch.tensor(lens, dtype=torch.int32, device="cuda"))


def _reference(w, window):
    B, R, hq, d = w["q"].shape
    hkv = w["k_new"].shape[2]
    G = hq // hkv
    out, lse = torch.empty((B, R, hq, d), device="cuda"), torch.empty((B, R, hq), device="cuda")
    for b, n in enumerate(w["seq_lens"].tolist()):
        pages = w["page_table"][b].long()
        k, v = (torch.cat([w[p][pages].transpose(0, 1).reshape(hkv, -1, d)[:, :n], w[x][b].transpose(0, 1)], dim=1).double()
                for p, x in (("k_pages", "k_new"), ("v_pages", "v_new")))
        q = w["q"][b].double().view(R, hkv, G, d).permute(1, 0, 2, 3).reshape(hkv, R * G, d)
        s = q @ k.transpose(1, 2) / math.sqrt(d)
        pos, row = torch.arange(n + R, device="cuda"), n + torch.arange(R, device="cuda").repeat_interleave(G)
        hidden = pos[None] > row[:, None]
        if window:
            hidden |= pos[None] <= row[:, None] - window
        s.masked_fill_(hidden[None], -math.inf)
        out[b] = (torch.softmax(s, -1) @ v).view(hkv, R, G, d).permute(1, 0, 2, 3).reshape(R, hq, d)
        lse[b] = torch.logsumexp(s, -1).view(hkv, R, G).permute(1, 0, 2).reshape(R, hq)
    return out, lse


@pytest.mark.parametrize("batch,gamma,q_heads,kv_heads,lo,hi,window", [
    (1, 5, 2, 1, 0, 0, 0), (3, 0, 4, 4, 31, 33, 0), (2, 5, 16, 8, 9000, 9100, 0), (48, 5, 16, 8, 100, 1500, 0), (40, 3, 16, 8, 700, 2000, 512),
    (64, 1, 8, 8, 0, 100, 0), (20, 3, 32, 4, 0, 900, 0), (24, 5, 32, 4, 300, 900, 0), (9, 7, 8, 1, 5, 2500, 0), (30, 7, 16, 2, 600, 1800, 300),
    (150, 2, 4, 2, 0, 700, 0), (5, 5, 16, 8, 2000, 3000, 1)])
def test_against_fp32(batch, gamma, q_heads, kv_heads, lo, hi, window):
    import paper_2505_10526_b200 as mv
    g = torch.Generator().manual_seed(batch + hi)
    lens = torch.randint(lo, hi + 1, (batch,), generator=g).tolist()
    w = _inputs(batch, gamma, q_heads, kv_heads, lens, seed=hi + gamma)
    want, want_lse = _reference(w, window)
    desc = mv.attn_desc(batch, gamma, q_heads, kv_heads, 256, w["page_table"].shape[1], w["k_pages"].shape[0], window=window)
    ws = mv.alloc_workspace(mv.massv_verify_attn_workspace_size(desc), "cuda")
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")

    def run():
        out = torch.full_like(w["q"], float("nan"))
        f32 = torch.full(out.shape, float("nan"), device="cuda")
        lse = torch.full(out.shape[:3], float("nan"), device="cuda")
        mv.massv_verify_attn(desc, w["q"], w["k_new"], w["v_new"], w["k_pages"], w["v_pages"], w["page_table"], w["seq_lens"], out, f32, lse, ws, status)
        return out, f32, lse

    out, f32, lse = run()
    again = run()
    assert int(status.item()) == 0
    # softmax weights carry bf16's rounding, at most 2^-8 each: 4e-3 of a row's norm for independent values, and another 2^-8 for the
    # bf16 output; the weights' sum is taken before the rounding.  (One position of 9,000 too many or too few is 1e-4 of the sum.)
    assert float((f32 - want).abs().max()) < 1e-2 and float((out.float() - want).abs().max()) < 3e-2
    assert float(((f32 - want).norm(dim=-1) / want.norm(dim=-1)).max()) < 4e-3 and float(((out.float() - want).norm(dim=-1) / want.norm(dim=-1)).max()) < 8e-3
    assert float((lse - want_lse).abs().max()) < 2e-5
    assert all(torch.equal(a, b) for a, b in zip((out, f32, lse), again))
    for b, n in enumerate(lens):                          # the block's rows are in their slots
        for j in range(gamma + 1):
            page, at = int(w["page_table"][b, (n + j) // 16]), (n + j) % 16
            assert torch.equal(w["k_pages"][page, :, at], w["k_new"][b, j]) and torch.equal(w["v_pages"][page, :, at], w["v_new"][b, j])


@pytest.mark.parametrize("batch,gamma,q_heads,kv_heads,hi", [(300, 5, 16, 8, 40), (300, 0, 8, 8, 90), (300, 3, 32, 4, 30), (200, 7, 8, 1, 60), (260, 7, 16, 2, 25)])
def test_many_short_pairs_per_cta(batch, gamma, q_heads, kv_heads, hi):
    """Contexts far below the page table's capacity: a CTA's range is many pairs of one to three tiles, so every stage of its ring
    is patched (block rows, zeros past the end) and refilled with another pair's query rows or tiles over and over."""
    import paper_2505_10526_b200 as mv
    g = torch.Generator().manual_seed(batch + hi)
    lens = torch.randint(0, hi + 1, (batch,), generator=g).tolist()
    w = _inputs(batch, gamma, q_heads, kv_heads, lens, seed=hi + gamma, max_pages=40)
    want, want_lse = _reference(w, 0)
    desc = mv.attn_desc(batch, gamma, q_heads, kv_heads, 256, 40, w["k_pages"].shape[0])
    ws = mv.alloc_workspace(mv.massv_verify_attn_workspace_size(desc), "cuda")
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    first = None
    for _ in range(5):
        out = torch.full_like(w["q"], float("nan"))
        f32 = torch.full(out.shape, float("nan"), device="cuda")
        lse = torch.full(out.shape[:3], float("nan"), device="cuda")
        mv.massv_verify_attn(desc, w["q"], w["k_new"], w["v_new"], w["k_pages"], w["v_pages"], w["page_table"], w["seq_lens"], out, f32, lse, ws, status)
        assert int(status.item()) == 0
        # an output row is a sum of w_i v_i whose weights carry bf16's rounding, at most 2^-8 each: 4e-3 of the row's norm for independent values
        assert float(((f32 - want).norm(dim=-1) / want.norm(dim=-1)).max()) < 4e-3
        # the weights' sum is taken before that rounding: fp32 scores of a few units, fp32 exponentials
        assert float((lse - want_lse).abs().max()) < 2e-5
        first = out if first is None else first
        assert torch.equal(out, first)


@pytest.mark.parametrize("batch,gamma,q_heads,kv_heads,lo,hi,window", [(32, 5, 16, 8, 2048, 8192, 0), (32, 5, 16, 8, 2048, 8192, 1024), (16, 5, 32, 8, 1000, 4000, 0)])
def test_long_rows_are_as_exact_as_in_chunks(batch, gamma, q_heads, kv_heads, lo, hi, window):
    """The error against 64 bits is that of the softmax weights' rounding to bf16, 2^-8 / sqrt(3) rms at a significand of one.  A
    reference that leaves only a prefix's maxima exact gives 0.8 of it (1.43e-3 to 1.47e-3 of the norm on these shapes, the more the
    fewer cuts a context has); with the largest weight of every 16 positions exact the rest carries 1.0e-3 however it is cut."""
    import paper_2505_10526_b200 as mv
    g = torch.Generator().manual_seed(batch + hi)
    lens = torch.randint(lo, hi + 1, (batch,), generator=g).tolist()
    w = _inputs(batch, gamma, q_heads, kv_heads, lens, seed=hi + gamma)
    want, want_lse = _reference(w, window)
    for chunk in (0, 768):
        desc = mv.attn_desc(batch, gamma, q_heads, kv_heads, 256, w["page_table"].shape[1], w["k_pages"].shape[0], window=window, kv_chunk=chunk)
        ws = mv.alloc_workspace(mv.massv_verify_attn_workspace_size(desc), "cuda")
        out = torch.empty_like(w["q"])
        f32 = torch.empty(out.shape, device="cuda")
        lse = torch.empty(out.shape[:3], device="cuda")
        mv.massv_verify_attn(desc, w["q"], w["k_new"], w["v_new"], w["k_pages"], w["v_pages"], w["page_table"], w["seq_lens"], out, f32, lse, ws, None)
        assert float((f32 - want).norm() / want.norm()) < 1.2e-3
        assert float((lse - want_lse).abs().max()) < 2e-5


@pytest.mark.parametrize("batch,gamma,q_heads,kv_heads,long_at", [(70, 5, 16, 8, (3, 40)), (33, 1, 8, 4, (32,)), (41, 5, 32, 4, (0, 20)), (300, 7, 16, 2, (150,)), (9, 7, 8, 1, (4,))])
def test_a_few_long_contexts_among_very_short_ones(batch, gamma, q_heads, kv_heads, long_at):
    """Cuts that fall inside a long pair, between pairs of one tile, and among the units that stand for a pair's set-up; one sequence
    has no room for its block and is skipped."""
    import paper_2505_10526_b200 as mv
    lens = [b % 3 for b in range(batch)]
    for i, b in enumerate(long_at):
        lens[b] = 2500 + 700 * i
    w = _inputs(batch, gamma, q_heads, kv_heads, lens, seed=batch)
    full = batch // 2 + 3
    capacity = w["page_table"].shape[1] * 16
    want, want_lse = _reference(w, 0)
    w["seq_lens"][full] = capacity - gamma                       # one position short of room
    desc = mv.attn_desc(batch, gamma, q_heads, kv_heads, 256, w["page_table"].shape[1], w["k_pages"].shape[0])
    ws = mv.alloc_workspace(mv.massv_verify_attn_workspace_size(desc), "cuda").fill_(0xff)
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    out = torch.full_like(w["q"], 7.0)
    f32 = torch.full(out.shape, 7.0, device="cuda")
    lse = torch.full(out.shape[:3], 7.0, device="cuda")
    mv.massv_verify_attn(desc, w["q"], w["k_new"], w["v_new"], w["k_pages"], w["v_pages"], w["page_table"], w["seq_lens"], out, f32, lse, ws, status)
    assert int(status.item()) == -3
    assert bool((out[full] == 7.0).all()) and bool((f32[full] == 7.0).all())
    rest = [b for b in range(batch) if b != full]
    assert float(((f32 - want).norm(dim=-1) / want.norm(dim=-1))[rest].max()) < 4e-3        # 2^-8 per weight
    assert float((lse - want_lse)[rest].abs().max()) < 2e-5
