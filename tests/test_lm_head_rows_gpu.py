"""The LM head at the edges of its row tiles (16-column chunks of single CTAs, 64-column jobs of CTA pairs, the two sub-tiles above 256 rows) and of the way
it deals the vocabulary out: one band, bands that take a pair per sub-tile and the first count that does not, left-over bands,
ragged ends; logits against 64 bits, greedy tokens against the logits' own argmax, probabilities from the merged statistics."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,gamma", [(1, 0), (17, 0), (11, 2), (48, 0), (49, 0), (16, 3), (13, 4), (16, 5), (43, 2), (32, 5), (51, 4), (64, 3), (257, 0), (68, 3), (64, 5), (77, 4), (100, 3), (73, 6), (64, 7)])
@pytest.mark.parametrize("vocab", [8, 264, 9472, 9480, 18944, 19208, 40008])
def test_rows(batch, gamma, vocab):
    import paper_2505_10526_b200 as mv
    K, R = 192, gamma + 1
    g = torch.Generator(device="cuda").manual_seed(batch * 7 + vocab)
    hidden = (5.0 * torch.randn((batch, R, K), generator=g, device="cuda")).to(torch.bfloat16)
    w = (0.05 * torch.randn((vocab, K), generator=g, device="cuda")).to(torch.bfloat16)
    exact = torch.matmul(hidden.view(-1, K).double(), w.double().t()).view(batch, R, vocab)
    drafts = exact[:, :gamma].argmax(-1).to(torch.int32).contiguous()          # every draft is right: the extra token is row gamma's
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    tokens = torch.empty((batch, R), dtype=torch.int32, device="cuda"); lens = torch.empty((batch,), dtype=torch.int32, device="cuda")
    for T in (0.0, 1.0):
        logits = torch.full((batch, R, vocab), float("nan"), device="cuda")
        probs = torch.full((batch, R, vocab), float("nan"), device="cuda") if T > 0 else None
        q = torch.full((batch, gamma, vocab), 1e-9, device="cuda")
        desc = mv.accept_desc(batch, gamma, K, vocab, T)
        ws = mv.alloc_workspace(mv.massv_accept_workspace_size(desc), "cuda").fill_(0xff)
        mv.massv_accept(desc, hidden, w, drafts, q if T > 0 else None, torch.full((batch, gamma), 0.5, device="cuda") if T > 0 else None,
                        torch.full((batch, R), 0.5, device="cuda") if T > 0 else None, tokens, lens, logits, probs, ws, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        # fp32 sums of 192 products of size about 0.25: 1e-5
        assert float((logits.double() - exact).abs().max()) < 1e-4
        assert lens.tolist() == [R] * batch
        if T == 0:
            assert torch.equal(tokens[:, gamma].long(), logits[:, gamma].argmax(-1))
            assert torch.equal(tokens[:, :gamma], logits[:, :gamma].argmax(-1).to(torch.int32))
        else:
            assert float((probs.double() - torch.softmax(exact, -1)).abs().max()) < 1e-4


@pytest.mark.parametrize("batch,gamma", [(1, 5), (16, 3), (16, 5), (40, 5), (50, 5), (100, 4)])        # 6, 64, 96, 240, 300, 500 token rows
@pytest.mark.parametrize("std,shift,T", [(5.0, 0.0, 1.0), (5.0, 100.0, 1.0), (20.0, 0.0, 0.1), (5.0, -400.0, 0.3)])
def test_sums_of_exponentials(batch, gamma, std, shift, T):
    """The largest probability of a row is 1 / sum exp((z - max) / T), so its relative error is the sum's: terms of a few 2^-24 (one
    product, one exponential), added 32 at a time, by tiles and by slots.  1.5e-6 is twice what a chain of a dozen fp32 sums gives."""
    import paper_2505_10526_b200 as mv
    K, R, vocab = 256, gamma + 1, 40008
    g = torch.Generator(device="cuda").manual_seed(batch + gamma)
    hidden = (std / 0.05 / 16.0 * torch.randn((batch, R, K), generator=g, device="cuda")).to(torch.bfloat16)
    w = (0.05 * torch.randn((vocab, K), generator=g, device="cuda")).to(torch.bfloat16)
    hidden[:, :, 0], w[:, 0] = shift, 1.0                   # every logit moved by the same amount
    q = torch.full((batch, gamma, vocab), 1e-9, device="cuda")
    desc = mv.accept_desc(batch, gamma, K, vocab, T)
    ws = mv.alloc_workspace(mv.massv_accept_workspace_size(desc), "cuda")
    logits, probs = torch.empty((batch, R, vocab), device="cuda"), torch.empty((batch, R, vocab), device="cuda")
    tokens = torch.empty((batch, R), dtype=torch.int32, device="cuda"); lens = torch.empty((batch,), dtype=torch.int32, device="cuda")
    mv.massv_accept(desc, hidden, w, torch.zeros((batch, gamma), dtype=torch.int32, device="cuda"), q, torch.full((batch, gamma), 0.5, device="cuda"),
                    torch.full((batch, R), 0.5, device="cuda"), tokens, lens, logits, probs, ws, None)
    worst = 0.0
    for b in range(batch):
        top = torch.softmax(logits[b].double() / T, dim=-1).max(-1).values
        worst = max(worst, float((probs[b].max(-1).values.double() / top - 1).abs().max()))
    print("worst", worst)
    assert worst < 1.5e-6


@pytest.mark.parametrize("hidden_size", [64, 128, 320, 832, 1088])
@pytest.mark.parametrize("batch", [1, 40, 64, 200, 256])
def test_k_blocks(batch, hidden_size):
    """A ring stage holds two blocks of 64 hidden elements: one block in all, full stages, a last stage with one block, rings that wrap
    inside a tile and across tiles.  fp32 sums of K products of size 0.25 or less, in any order: below K * 2^-24 * sqrt(K) * 0.25."""
    import paper_2505_10526_b200 as mv
    vocab = 40008
    g = torch.Generator(device="cuda").manual_seed(hidden_size + batch)
    hidden = (5.0 * torch.randn((batch, 1, hidden_size), generator=g, device="cuda")).to(torch.bfloat16)
    w = (0.05 * torch.randn((vocab, hidden_size), generator=g, device="cuda")).to(torch.bfloat16)
    exact = torch.matmul(hidden.view(-1, hidden_size).double(), w.double().t()).view(batch, 1, vocab)
    logits = torch.full((batch, 1, vocab), float("nan"), device="cuda")
    tokens = torch.empty((batch, 1), dtype=torch.int32, device="cuda"); lens = torch.empty((batch,), dtype=torch.int32, device="cuda")
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    desc = mv.accept_desc(batch, 0, hidden_size, vocab, 0.0)
    ws = mv.alloc_workspace(mv.massv_accept_workspace_size(desc), "cuda").fill_(0xff)
    mv.massv_accept(desc, hidden, w, torch.zeros((batch, 0), dtype=torch.int32, device="cuda"), None, None, None, tokens, lens, logits, None, ws, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert float((logits.double() - exact).abs().max()) < hidden_size ** 1.5 * 2 ** -24 * 0.25 + 1e-5
    assert torch.equal(tokens[:, 0].long(), logits[:, 0].argmax(-1))
