"""massv_accept at T > 0 where its one-launch kernel (a cluster per sequence) can go wrong: one group of entries, segments that
are ragged or empty, every cluster size and the batch at which the next smaller one or the persistent draw takes over, draws at
both ends of the row, a drafter equal to the target (no residual mass), and the distribution output.  The reference decides in
64 bits from the call's own logits."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _call(batch, gamma, vocab, T, u_accept, u_sample, q=None, seed=0, probs=False):
    import paper_2505_10526_b200 as mv
    K, R = 128, gamma + 1
    g = torch.Generator(device="cuda").manual_seed(seed)
    hidden = (20.0 * torch.randn((batch, R, K), generator=g, device="cuda")).to(torch.bfloat16)
    w = (0.02 * torch.randn((vocab, K), generator=g, device="cuda")).to(torch.bfloat16)
    z = torch.matmul(hidden.view(-1, K), w.t()).float().view(batch, R, vocab)
    if q is None:
        q = torch.softmax((z[:, :gamma] + 0.5 * torch.randn((batch, gamma, vocab), generator=g, device="cuda")) / T, dim=-1)
    drafts = torch.multinomial(q.reshape(-1, vocab), 1, generator=g).view(batch, gamma).to(torch.int32) if gamma else torch.zeros((batch, 0), dtype=torch.int32, device="cuda")
    q = q.contiguous()
    desc = mv.accept_desc(batch, gamma, K, vocab, T)
    ws = mv.alloc_workspace(mv.massv_accept_workspace_size(desc), "cuda")
    out = dict(tokens=torch.full((batch, R), -9, dtype=torch.int32, device="cuda"), lens=torch.full((batch,), -9, dtype=torch.int32, device="cuda"),
               logits=torch.empty((batch, R, vocab), device="cuda"), probs=torch.full((batch, R, vocab), -1.0, device="cuda") if probs else None)
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    u_accept = u_accept.expand(batch, gamma).contiguous() if u_accept.dim() < 2 else u_accept
    u_sample = u_sample.expand(batch, R).contiguous() if u_sample.dim() < 2 else u_sample
    for _ in range(2):          # twice, so that nothing left in the workspace matters
        mv.massv_accept(desc, hidden, w, drafts, q, u_accept, u_sample, out["tokens"], out["lens"], out["logits"], out["probs"], ws, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return dict(out, q=q, drafts=drafts, u_accept=u_accept, u_sample=u_sample)


def _check(r, gamma, T):
    p = torch.softmax(r["logits"].double() / T, dim=-1)
    for b in range(p.shape[0]):
        n = 0
        close = False
        while n < gamma:
            x = int(r["drafts"][b, n])
            lhs, rhs = float(r["u_accept"][b, n]) * float(r["q"][b, n, x]), float(p[b, n, x])
            close = close or abs(lhs - rhs) < 1e-5 * max(lhs, rhs)      # fp32 against 64 bits
            if not lhs < rhs:
                break
            n += 1
        if close:
            continue
        assert int(r["lens"][b]) == n + 1
        assert r["tokens"][b, :n].tolist() == r["drafts"][b, :n].tolist() and all(t == -1 for t in r["tokens"][b, n + 1:].tolist())
        mass = (p[b, n] - r["q"][b, n].double()).clamp_min(0) if n < gamma else p[b, n]
        # fp32 masses: an entry is known to about 3e-7 of p, and where p and q all but cancel, the residual to that of its total
        total = float(mass.sum())
        if total < 1e-4:
            continue
        cdf = torch.cumsum(mass, 0) / total
        tok, u = int(r["tokens"][b, n]), float(r["u_sample"][b, n])
        lo = float(cdf[tok - 1]) if tok else 0.0
        slack = 2e-6 / total
        assert lo - slack <= u <= float(cdf[tok]) + slack, (b, n, tok, lo, u, float(cdf[tok]))
    if r["probs"] is not None:
        assert float((r["probs"].double() - p).abs().max()) < 1e-5


@pytest.mark.parametrize("batch,gamma,vocab", [(1, 0, 8), (1, 5, 8), (2, 3, 72), (3, 0, 4088), (3, 2, 4104), (1, 1, 8200), (28, 1, 16384), (29, 1, 16392),
                                               (56, 2, 10008), (57, 2, 10008), (112, 0, 4096), (113, 0, 4096), (128, 3, 1024), (7, 3, 50264),
                                               (28, 0, 152064), (29, 0, 152064), (2, 7, 262144), (13, 1, 262144)])
def test_sizes(batch, gamma, vocab):
    g = torch.Generator(device="cuda").manual_seed(batch + vocab)
    _check(_call(batch, gamma, vocab, 0.8, torch.rand((batch, gamma), generator=g, device="cuda"), torch.rand((batch, gamma + 1), generator=g, device="cuda"),
                 seed=vocab, probs=True), gamma, 0.8)


@pytest.mark.parametrize("vocab", [64, 5000, 152064])
@pytest.mark.parametrize("u", [0.0, 0.99999994])
def test_ends_of_the_row(vocab, u):
    r = _call(3, 0, vocab, 1.0, torch.zeros((), device="cuda"), torch.full((), u, device="cuda"), seed=5)
    _check(r, 0, 1.0)
    assert r["tokens"].min() >= 0 and r["tokens"].max() < vocab


@pytest.mark.parametrize("vocab", [1000, 152064])
def test_no_residual_mass(vocab):
    """q twice the largest p everywhere: whatever is rejected leaves no residual, so the draw falls back to p itself."""
    q = torch.full((2, 2, vocab), 2.0, device="cuda")
    r = _call(2, 2, vocab, 1.0, torch.full((), 0.999, device="cuda"), torch.full((), 0.4, device="cuda"), q=q, seed=9)
    p = torch.softmax(r["logits"].double(), dim=-1)
    assert r["lens"].tolist() == [1, 1]
    for b in range(2):
        cdf = torch.cumsum(p[b, 0], 0)
        tok = int(r["tokens"][b, 0])
        assert (float(cdf[tok - 1]) if tok else 0.0) - 2e-6 <= 0.4 <= float(cdf[tok]) + 2e-6


@pytest.mark.parametrize("batch,gamma,vocab", [(3, 2, 10008), (5, 0, 50264), (300, 0, 4096), (128, 2, 65536), (150, 1, 32000)])
def test_distribution_in_place_of_the_logits(batch, gamma, vocab):
    """probs_out in the buffer of logits_out: the tokens are drawn before the row is overwritten."""
    import paper_2505_10526_b200 as mv
    K, R, T = 128, gamma + 1, 0.8
    g = torch.Generator(device="cuda").manual_seed(vocab)
    hidden = (20.0 * torch.randn((batch, R, K), generator=g, device="cuda")).to(torch.bfloat16)
    w = (0.02 * torch.randn((vocab, K), generator=g, device="cuda")).to(torch.bfloat16)
    q = torch.softmax(4.0 * torch.randn((batch, gamma, vocab), generator=g, device="cuda"), dim=-1).contiguous()
    drafts = torch.randint(0, vocab, (batch, gamma), generator=g, device="cuda", dtype=torch.int32)
    ua, us = torch.rand((batch, gamma), generator=g, device="cuda"), torch.rand((batch, R), generator=g, device="cuda")
    desc = mv.accept_desc(batch, gamma, K, vocab, T)
    ws = mv.alloc_workspace(mv.massv_accept_workspace_size(desc), "cuda")
    res = []
    for shared in (False, True, True):
        logits = torch.empty((batch, R, vocab), device="cuda")
        probs = logits if shared else torch.empty_like(logits)
        tokens = torch.empty((batch, R), dtype=torch.int32, device="cuda"); lens = torch.empty((batch,), dtype=torch.int32, device="cuda")
        mv.massv_accept(desc, hidden, w, drafts, q, ua, us, tokens, lens, logits, probs, ws, None)
        res.append((tokens, lens, probs))
    for other in res[1:]:
        assert all(torch.equal(a, b) for a, b in zip(res[0], other))
