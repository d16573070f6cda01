"""massv_tvd where its kernels can go wrong: one short slice, ragged last slices and CTAs without an entry, every cluster
size, slices longer than the registers hold, slices without a finite logit, the streamed passes with rows that end inside a
CTA's run and the first vocabulary that does not fit a cluster; with and without the acceptance call's statistics."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _reference(z, q, T):
    tvd, acc = [], []
    for zr, qr in zip(z, q):                              # one sequence at a time: the copies in 64 bits stay small
        p = torch.softmax(zr.double() / T, dim=-1)
        tvd.append(0.5 * (p - qr.double()).abs().sum(-1))
        acc.append(torch.minimum(p, qr.double()).sum(-1))
    return torch.stack(tvd), torch.stack(acc)


@pytest.mark.parametrize("batch,gamma,vocab", [(1, 1, 8), (2, 3, 1032), (40, 5, 4096), (3, 2, 10240), (3, 2, 10248), (64, 7, 20488),
                                               (33, 5, 8200), (41, 7, 16392), (30, 5, 152064), (2, 1, 152064), (9, 5, 163848), (2, 2, 262144),
                                               (1, 1, 25 * 1024 * 16), (1, 2, 25 * 1024 * 16 + 8), (3, 5, 1000008)])
@pytest.mark.parametrize("T", [1.0, 0.7])
def test_sizes(batch, gamma, vocab, T):
    import paper_2505_10526_b200 as mv
    g = torch.Generator(device="cuda").manual_seed(vocab + gamma)
    z = 4.0 * torch.randn((batch, gamma + 1, vocab), generator=g, device="cuda")
    z[:, :, :vocab // 3] = -float("inf")                  # whole slices without a finite logit
    q = torch.softmax(z[:, :gamma] + torch.randn((batch, gamma, vocab), generator=g, device="cuda"), dim=-1).contiguous()
    desc = mv.accept_desc(batch, gamma, 64, vocab, T)
    ws = mv.alloc_workspace(mv.massv_tvd_workspace_size(desc), "cuda")
    out = torch.full((2, batch * gamma + 8), -7.0, device="cuda")
    tvd, acc = out[0, 4:4 + batch * gamma].view(batch, gamma), out[1, 4:4 + batch * gamma].view(batch, gamma)
    mv.massv_tvd(desc, z, q, tvd, acc, ws, None)
    want_tvd, want_acc = _reference(z[:, :gamma], q, T)
    # p carries the rounding of one exponential and one product (a few 2^-24 of itself), the sums are double: 1e-6 of a total of 2
    assert float((tvd.double() - want_tvd).abs().max()) < 2e-6 and float((acc.double() - want_acc).abs().max()) < 2e-6
    assert float(out[:, :4].max()) == -7.0 and float(out[:, 4 + batch * gamma:].max()) == -7.0
    again = torch.empty_like(tvd)
    mv.massv_tvd(desc, z, q, again, None, ws, None)
    assert torch.equal(again, tvd)


@pytest.mark.parametrize("batch,gamma,vocab", [(3, 2, 1024), (4, 5, 10248), (2, 3, 152064), (60, 3, 50264)])
def test_with_the_acceptance_calls_statistics(batch, gamma, vocab):
    import paper_2505_10526_b200 as mv
    K, R = 256, gamma + 1
    g = torch.Generator(device="cuda").manual_seed(vocab)
    hidden = (15.0 * torch.randn((batch, R, K), generator=g, device="cuda")).to(torch.bfloat16)
    w = (0.02 * torch.randn((vocab, K), generator=g, device="cuda")).to(torch.bfloat16)
    q = torch.softmax(4.0 * torch.randn((batch, gamma, vocab), generator=g, device="cuda"), dim=-1).contiguous()
    desc = mv.accept_desc(batch, gamma, K, vocab, 1.0)
    ws = mv.alloc_workspace(mv.massv_accept_workspace_size(desc), "cuda")
    tokens = torch.zeros((batch, R), dtype=torch.int32, device="cuda"); lens = torch.zeros((batch,), dtype=torch.int32, device="cuda")
    logits = torch.empty((batch, R, vocab), device="cuda")
    mv.massv_accept(desc, hidden, w, torch.zeros((batch, gamma), dtype=torch.int32, device="cuda"), q, torch.full((batch, gamma), 0.5, device="cuda"),
                    torch.full((batch, R), 0.5, device="cuda"), tokens, lens, logits, None, ws, None)
    ws2 = mv.alloc_workspace(mv.massv_tvd_workspace_size(desc), "cuda")
    tvd = torch.empty((batch, gamma), device="cuda"); acc = torch.empty_like(tvd)
    mv.massv_tvd_after_accept(desc, logits, q, ws, tvd, acc, ws2, None)
    want_tvd, want_acc = _reference(logits[:, :gamma], q, 1.0)
    # the statistics are the LM head's fp32 sums: up to 152,064 terms in blocks, about 1e-6 of the total
    assert float((tvd.double() - want_tvd).abs().max()) < 1e-5 and float((acc.double() - want_acc).abs().max()) < 1e-5
