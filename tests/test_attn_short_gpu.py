"""The tcgen05 kernel with one CTA per (sequence, KV head) pair, which short page tables take: the longest table of the rule and the
first beyond it for few and many pairs, one position, ragged ends, windows; against attention in 64 bits on the same bf16 values."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def _reference(w, window):
    B, R, hq, d = w["q"].shape
    hkv = w["k_new"].shape[2]
    G = hq // hkv
    out = torch.empty((B, R, hq, d), dtype=torch.float64, device="cuda")
    for b, n in enumerate(w["seq_lens"].tolist()):
        pages = w["page_table"][b].long()
        k, v = (torch.cat([w[p][pages].transpose(0, 1).reshape(hkv, -1, d)[:, :n], w[x][b].transpose(0, 1)], dim=1).double()
                for p, x in (("k_pages", "k_new"), ("v_pages", "v_new")))
        s = w["q"][b].double().view(R, hkv, G, d).permute(1, 0, 2, 3).reshape(hkv, R * G, d) @ k.transpose(1, 2) / math.sqrt(d)
        pos, row = torch.arange(n + R, device="cuda"), n + torch.arange(R, device="cuda").repeat_interleave(G)
        hidden = pos[None] > row[:, None]
        if window:
            hidden |= pos[None] <= row[:, None] - window
        s.masked_fill_(hidden[None], -math.inf)
        out[b] = (torch.softmax(s, -1) @ v).view(hkv, R, G, d).permute(1, 0, 2, 3).reshape(R, hq, d)
    return out


@pytest.mark.parametrize("batch,gamma,q_heads,kv_heads,pages,window", [
    (1, 0, 1, 1, 1, 0), (1, 5, 4, 1, 16, 0), (1, 5, 4, 1, 17, 0), (3, 3, 16, 8, 20, 0), (3, 3, 16, 8, 21, 0), (12, 5, 28, 4, 24, 0), (24, 5, 28, 4, 32, 0),
    (24, 5, 28, 4, 33, 0), (64, 7, 8, 8, 32, 0), (2, 1, 64, 2, 12, 0), (40, 2, 12, 4, 100, 100), (40, 2, 12, 4, 255, 300), (5, 6, 9, 1, 200, 40),
    # the bounds of the rule: 16 and 48 pairs, one wave of CTAs and the first pair beyond, whole pairs per range, two waves
    (15, 5, 7, 1, 16, 0), (16, 5, 7, 1, 16, 0), (47, 1, 3, 1, 20, 0), (48, 1, 3, 1, 20, 0), (37, 1, 8, 8, 32, 0), (99, 0, 3, 3, 24, 0), (99, 0, 3, 3, 28, 0), (64, 1, 8, 8, 12, 0), (149, 0, 4, 4, 24, 0)])
@pytest.mark.parametrize("d", [64, 128])
def test_against_64_bits(batch, gamma, q_heads, kv_heads, pages, window, d):
    import paper_2505_10526_b200 as mv
    R = gamma + 1
    g = torch.Generator(device="cuda").manual_seed(batch + pages + d)
    n_pages = batch * pages + 2
    bf = dict(dtype=torch.bfloat16, device="cuda", generator=g)
    lens = torch.randint(0, pages * 16 - R + 1, (batch,), generator=g, device="cuda").to(torch.int32)
    lens[0] = pages * 16 - R                                 # a full table, and an empty context where there is another sequence
    if batch > 1:
        lens[1] = 0
    w = dict(q=torch.randn((batch, R, q_heads, d), **bf), k_new=torch.randn((batch, R, kv_heads, d), **bf), v_new=torch.randn((batch, R, kv_heads, d), **bf),
             k_pages=torch.randn((n_pages, kv_heads, 16, d), **bf), v_pages=torch.randn((n_pages, kv_heads, 16, d), **bf),
             page_table=torch.randperm(n_pages, generator=g, device="cuda")[:batch * pages].view(batch, pages).to(torch.int32).contiguous(), seq_lens=lens)
    want = _reference(w, window)
    desc = mv.attn_desc(batch, gamma, q_heads, kv_heads, d, pages, n_pages, window=window)
    ws = mv.alloc_workspace(mv.massv_verify_attn_workspace_size(desc), "cuda").fill_(0xff)
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    out = torch.full_like(w["q"], float("nan")); f32 = torch.full(out.shape, float("nan"), device="cuda")
    mv.massv_verify_attn(desc, w["q"], w["k_new"], w["v_new"], w["k_pages"], w["v_pages"], w["page_table"], w["seq_lens"], out, f32, None, ws, status)
    assert int(status.item()) == 0
    # softmax weights rounded to bf16: at most 2^-8 each, 4e-3 of a row's norm for independent values; another 2^-8 for the bf16 output
    assert float(((f32 - want).norm(dim=-1) / want.norm(dim=-1)).max()) < 4e-3 and float(((out.double() - want).norm(dim=-1) / want.norm(dim=-1)).max()) < 8e-3
    for b, n in enumerate(lens.tolist()):                    # the block's rows are in their slots
        for j in range(R):
            page, at = int(w["page_table"][b, (n + j) // 16]), (n + j) % 16
            assert torch.equal(w["k_pages"][page, :, at], w["k_new"][b, j]) and torch.equal(w["v_pages"][page, :, at], w["v_new"][b, j])


@pytest.mark.parametrize("batch,q_heads,kv_heads,base,longer,window", [
    (32, 16, 8, 1500, 500, 1024), (37, 16, 8, 1000, 0, 0), (32, 16, 8, 1000, 128, 0), (32, 16, 8, 1000, 1000, 0), (18, 32, 8, 1100, 300, 512), (64, 16, 4, 700, 64, 0),
    (1, 16, 8, 520, 0, 512)])
@pytest.mark.parametrize("d", [64, 128, 256])
def test_a_pair_per_cta(batch, q_heads, kv_heads, base, longer, window, d):
    """Windows and equal lengths, where the balanced schedule of head_dim 256 gives every pair a CTA, one sequence longer by less and by
    more than the slack, a sequence without room for its block (skipped, and reported)."""
    import paper_2505_10526_b200 as mv
    gamma, R = 5, 6
    g = torch.Generator(device="cuda").manual_seed(batch + base + d)
    pages = (base + longer + R + 15) // 16
    n_pages = batch * pages
    bf = dict(dtype=torch.bfloat16, device="cuda", generator=g)
    lens = torch.full((batch,), base, dtype=torch.int32, device="cuda")
    lens[batch // 2] += longer
    skipped = batch > 8
    w = dict(q=torch.randn((batch, R, q_heads, d), **bf), k_new=torch.randn((batch, R, kv_heads, d), **bf), v_new=torch.randn((batch, R, kv_heads, d), **bf),
             k_pages=torch.randn((n_pages, kv_heads, 16, d), **bf), v_pages=torch.randn((n_pages, kv_heads, 16, d), **bf),
             page_table=torch.randperm(n_pages, generator=g, device="cuda").view(batch, pages).to(torch.int32).contiguous(), seq_lens=lens)
    want = _reference(w, window)
    if skipped:
        lens[3] = pages * 16
    desc = mv.attn_desc(batch, gamma, q_heads, kv_heads, d, pages, n_pages, window=window)
    ws = mv.alloc_workspace(mv.massv_verify_attn_workspace_size(desc), "cuda").fill_(0xff)
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    outs = []
    for _ in range(2):
        out = torch.full_like(w["q"], float("nan")); f32 = torch.full(out.shape, float("nan"), device="cuda")
        mv.massv_verify_attn(desc, w["q"], w["k_new"], w["v_new"], w["k_pages"], w["v_pages"], w["page_table"], w["seq_lens"], out, f32, None, ws, status)
        outs.append(f32)
    keep = [b for b in range(batch) if not (skipped and b == 3)]
    assert (int(status.item()) != 0) == skipped
    # as above
    assert float(((outs[0][keep] - want[keep]).norm(dim=-1) / want[keep].norm(dim=-1)).max()) < 4e-3
    assert torch.equal(outs[0][keep], outs[1][keep])
    assert not skipped or bool(outs[0][3].isnan().all())


@pytest.mark.parametrize("step", [-9.0, -5.9, -3.0, 3.0, 5.9, 9.0])
@pytest.mark.parametrize("batch,kv_heads,pages,window", [(1, 4, 12, 0), (24, 4, 32, 0), (24, 4, 32, 300), (1025, 2, 120, 0)])
@pytest.mark.parametrize("d", [64, 128])
def test_scores_that_fall_or_rise_from_tile_to_tile(batch, kv_heads, pages, window, step, d):
    """Tile maxima that move by `step` binary orders from one tile of 64 positions to the next, over the one-piece route (3 and 8 tiles) and,
    with more sequences than the balanced schedule takes, over 30 tiles in one run: the weights' reference goes with them, and what it
    has left behind must stay in range."""
    import paper_2505_10526_b200 as mv
    gamma, R, G = 1, 2, 2
    g = torch.Generator(device="cuda").manual_seed(batch + pages + d)
    n_pages = batch * pages
    bf = dict(dtype=torch.bfloat16, device="cuda", generator=g)
    table = torch.randperm(n_pages, generator=g, device="cuda").view(batch, pages).to(torch.int32).contiguous()
    # q = 8 in every element, so a key of constant x scores 8 d x / sqrt(d) log2(e) binary orders; the line through zero in the middle
    tile = torch.arange(pages, device="cuda") // 4
    level = ((tile - tile[-1] / 2.0) * step / (8.0 * math.sqrt(d) * math.log2(math.e))).repeat(batch)
    keys = 0.02 * torch.randn((n_pages, kv_heads, 16, d), device="cuda", generator=g)
    keys[table.view(-1).long()] += level[:, None, None, None]
    w = dict(q=torch.full((batch, R, kv_heads * G, d), 8.0, dtype=torch.bfloat16, device="cuda"),
             k_new=torch.full((batch, R, kv_heads, d), float(level[-1]), dtype=torch.bfloat16, device="cuda"), v_new=torch.randn((batch, R, kv_heads, d), **bf),
             k_pages=keys.to(torch.bfloat16), v_pages=torch.randn((n_pages, kv_heads, 16, d), **bf), page_table=table,
             seq_lens=torch.full((batch,), pages * 16 - R, dtype=torch.int32, device="cuda"))
    del keys
    want = _reference(w, window)
    desc = mv.attn_desc(batch, gamma, kv_heads * G, kv_heads, d, pages, n_pages, window=window)
    ws = mv.alloc_workspace(mv.massv_verify_attn_workspace_size(desc), "cuda").fill_(0xff)
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    out = torch.full_like(w["q"], float("nan")); f32 = torch.full(out.shape, float("nan"), device="cuda")
    mv.massv_verify_attn(desc, w["q"], w["k_new"], w["v_new"], w["k_pages"], w["v_pages"], w["page_table"], w["seq_lens"], out, f32, None, ws, status)
    assert int(status.item()) == 0
    # as above: weights rounded to bf16, each by at most 2^-9
    assert float(((f32 - want).norm(dim=-1) / want.norm(dim=-1)).max()) < 4e-3


@pytest.mark.parametrize("d", [64, 128, 256])
def test_a_window_longer_than_any_context(d):
    """A window of 2^31 - 1 positions hides nothing, and takes the route of no window."""
    import paper_2505_10526_b200 as mv
    batch, gamma, q_heads, kv_heads, pages = 3, 3, 8, 4, 256
    R, n_pages = gamma + 1, batch * pages
    g = torch.Generator(device="cuda").manual_seed(d)
    bf = dict(dtype=torch.bfloat16, device="cuda", generator=g)
    w = dict(q=torch.randn((batch, R, q_heads, d), **bf), k_new=torch.randn((batch, R, kv_heads, d), **bf), v_new=torch.randn((batch, R, kv_heads, d), **bf),
             k_pages=torch.randn((n_pages, kv_heads, 16, d), **bf), v_pages=torch.randn((n_pages, kv_heads, 16, d), **bf),
             page_table=torch.randperm(n_pages, generator=g, device="cuda").view(batch, pages).to(torch.int32).contiguous(),
             seq_lens=torch.tensor([pages * 16 - R, 2000, 77], dtype=torch.int32, device="cuda"))
    outs, launches = [], []
    for window in (0, 2 ** 31 - 1, pages * 16):
        desc = mv.attn_desc(batch, gamma, q_heads, kv_heads, d, pages, n_pages, window=window)
        ws = mv.alloc_workspace(mv.massv_verify_attn_workspace_size(desc), "cuda")
        out = torch.empty_like(w["q"])
        before = mv.massv_launch_count()
        mv.massv_verify_attn(desc, w["q"], w["k_new"], w["v_new"], w["k_pages"], w["v_pages"], w["page_table"], w["seq_lens"], out, None, None, ws, None)
        launches.append(mv.massv_launch_count() - before)
        outs.append(out)
    assert launches[0] == launches[1] == launches[2]
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
