"""Logits that are NaN or +inf: the row's outcome stays inside the vocabulary and is reported where there is nothing to compare, and
the other sequences come out as without it; every way the LM head deals its rows out, every acceptance path, top-p and TVD."""
import pytest
import torch

pytestmark = pytest.mark.gpu

ROWS = [(1, 5), (16, 5), (40, 5), (50, 5), (100, 4), (3, 0), (64, 0)]        # 6, 96, 240, 300, 500 token rows; one row a sequence


def _inputs(batch, gamma, vocab, T, seed=3):
    K, R = 128, gamma + 1
    g = torch.Generator(device="cuda").manual_seed(seed)
    hidden = (20.0 * torch.randn((batch, R, K), generator=g, device="cuda")).to(torch.bfloat16)
    w = (0.02 * torch.randn((vocab, K), generator=g, device="cuda")).to(torch.bfloat16)
    z = torch.matmul(hidden.view(-1, K), w.t()).float().view(batch, R, vocab)
    q = torch.softmax(z[:, :gamma] + 0.5 * torch.randn((batch, gamma, vocab), generator=g, device="cuda"), dim=-1).contiguous()
    drafts = z[:, :gamma].argmax(-1).to(torch.int32).contiguous()
    u = torch.rand((batch, 2 * R), generator=g, device="cuda")
    return hidden, w, drafts, q, u[:, :gamma].contiguous(), u[:, R:].contiguous()


def _accept(inputs, T):
    import paper_2505_10526_b200 as mv
    hidden, w, drafts, q, ua, us = inputs
    batch, R, K = hidden.shape
    desc = mv.accept_desc(batch, R - 1, K, w.shape[0], T)
    ws = mv.alloc_workspace(mv.massv_accept_workspace_size(desc), "cuda").fill_(0xff)
    tokens = torch.full((batch, R), -9, dtype=torch.int32, device="cuda")
    lens = torch.full((batch,), -9, dtype=torch.int32, device="cuda")
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    s = T > 0
    mv.massv_accept(desc, hidden, w, drafts, q if s else None, ua if s else None, us if s else None, tokens, lens, None, None, ws, status)
    torch.cuda.synchronize()
    return tokens, lens, int(status.item())


@pytest.mark.parametrize("T", [0.0, 1.0])
@pytest.mark.parametrize("batch,gamma", ROWS)
def test_a_hidden_state_that_has_gone_nan(batch, gamma, T):
    vocab = 40008
    inputs = _inputs(batch, gamma, vocab, T)
    clean_tokens, clean_lens, status = _accept(inputs, T)
    assert status == 0
    hit = batch // 2
    inputs[0][hit, 0] = float("nan")
    tokens, lens, status = _accept(inputs, T)
    assert status == -1                                     # MASSV_ERR_INVALID_ARG
    assert int(lens[hit]) == 1 and int(tokens[hit, 0]) == 0 and all(t == -1 for t in tokens[hit, 1:].tolist())
    rest = [b for b in range(batch) if b != hit]
    assert torch.equal(tokens[rest], clean_tokens[rest]) and torch.equal(lens[rest], clean_lens[rest])


@pytest.mark.parametrize("T", [0.0, 1.0])
@pytest.mark.parametrize("batch,gamma", ROWS)
def test_an_infinite_logit(batch, gamma, T):
    """One weight row so large that every logit of one vocabulary entry overflows, in one sequence only."""
    vocab, at = 9480, 4321
    inputs = _inputs(batch, gamma, vocab, T)
    hit = batch // 2
    inputs[0][:, :, 0] = 0.0
    inputs[0][hit, :, 0] = 1.0e4
    inputs[1][:, 0] = 0.0
    clean_tokens, clean_lens, _ = _accept(inputs, T)
    inputs[1][at, 0] = 3.0e38
    tokens, lens, status = _accept(inputs, T)
    if T == 0:
        n = int(lens[hit]) - 1
        assert status == 0 and n == 0 and int(tokens[hit, 0]) == at
    else:
        assert status == -1 and 0 <= int(tokens[hit, int(lens[hit]) - 1]) < vocab
    rest = [b for b in range(batch) if b != hit]
    assert torch.equal(tokens[rest], clean_tokens[rest]) and torch.equal(lens[rest], clean_lens[rest])


@pytest.mark.parametrize("T", [0.0, 1.0])
def test_a_nan_row_in_vocabulary_shards(T):
    from paper_2505_10526_b200.sharded import ShardedAccept, run_lockstep
    batch, gamma, world, Vs = 5, 3, 4, 2048
    hidden, w, drafts, q, ua, us = _inputs(batch, gamma, world * Vs, T)
    hidden[2, 0] = float("nan")
    ranks = [ShardedAccept(batch, gamma, hidden.shape[2], Vs, T, world, r) for r in range(world)]
    kw = [dict(hidden=hidden, lm_head_shard=w[r * Vs:(r + 1) * Vs].contiguous(), draft_tokens=drafts) for r in range(world)]
    if T > 0:
        for r in range(world):
            kw[r].update(draft_probs_shard=q[:, :, r * Vs:(r + 1) * Vs].contiguous(), u_accept=ua, u_sample=us)
    for tokens, lens in run_lockstep(ranks, kw):
        assert int(lens[2]) == 1 and int(tokens[2, 0]) == 0
        assert int(tokens.max()) < world * Vs
    assert all(int(r.dev_status.item()) == -1 for r in ranks)


@pytest.mark.parametrize("rows,vocab", [(1, 2000), (40, 2000), (3, 60000), (70, 152064), (2, 400000)])
def test_top_p(rows, vocab):
    import paper_2505_10526_b200 as mv
    g = torch.Generator(device="cuda").manual_seed(vocab)
    z = 4.0 * torch.randn((rows, vocab), generator=g, device="cuda")
    u = torch.rand((rows,), generator=g, device="cuda")

    def run():
        tok = torch.full((rows,), -5, dtype=torch.int32, device="cuda")
        status = torch.zeros((1,), dtype=torch.int32, device="cuda")
        mv.massv_sample_top_p(z, u, tok, 1.0, 0.9, None, status)
        torch.cuda.synchronize()
        return tok, int(status.item())

    clean, status = run()
    assert status == 0
    hit = rows // 2
    rest = [r for r in range(rows) if r != hit]
    for value in (float("inf"), float("nan")):
        saved = z[hit].clone()
        if value == value:
            z[hit, vocab // 3] = value                       # nothing finite to weigh the others against
        else:
            z[hit] = value
        tok, status = run()
        assert status == -1 and int(tok[hit]) == 0 and torch.equal(tok[rest], clean[rest])
        z[hit] = saved


@pytest.mark.parametrize("batch,gamma,vocab", [(1, 1, 1024), (3, 2, 50264), (64, 7, 20488)])
def test_tvd(batch, gamma, vocab):
    import paper_2505_10526_b200 as mv
    g = torch.Generator(device="cuda").manual_seed(vocab)
    z = 4.0 * torch.randn((batch, gamma + 1, vocab), generator=g, device="cuda")
    q = torch.softmax(z[:, :gamma] + torch.randn((batch, gamma, vocab), generator=g, device="cuda"), dim=-1).contiguous()
    desc = mv.accept_desc(batch, gamma, 64, vocab, 1.0)
    ws = mv.alloc_workspace(mv.massv_tvd_workspace_size(desc), "cuda")
    clean, tvd = torch.empty((2, batch, gamma), device="cuda")
    mv.massv_tvd(desc, z, q, clean, None, ws, None)
    for value in (float("nan"), float("inf")):
        keep = float(z[batch // 2, 0, vocab // 2])
        z[batch // 2, 0, vocab // 2] = value
        mv.massv_tvd(desc, z, q, tvd, None, ws, None)
        z[batch // 2, 0, vocab // 2] = keep
        bad = torch.isnan(tvd)
        assert bool(bad[batch // 2, 0]) and int(bad.sum()) == 1
        assert torch.equal(tvd[~bad], clean[~bad])
