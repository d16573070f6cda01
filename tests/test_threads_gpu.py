"""Calls of different sizes from several host threads, each on its own stream and workspaces: kernel attributes are the process's, so
no call may change one that another thread's launch depends on."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def _attention(mv, batch, gamma, head_dim, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    R, pages = gamma + 1, 60
    bf = dict(dtype=torch.bfloat16, device="cuda", generator=g)
    q, k, v = torch.randn((batch, R, 4, head_dim), **bf), torch.randn((batch, R, 2, head_dim), **bf), torch.randn((batch, R, 2, head_dim), **bf)
    kp, vp = torch.randn((batch * pages, 2, 16, head_dim), **bf), torch.randn((batch * pages, 2, 16, head_dim), **bf)
    table = torch.arange(batch * pages, dtype=torch.int32, device="cuda").view(batch, pages)
    lens = torch.full((batch,), 50, dtype=torch.int32, device="cuda")
    desc = mv.attn_desc(batch, gamma, 4, 2, head_dim, pages, batch * pages)
    ws = mv.alloc_workspace(mv.massv_verify_attn_workspace_size(desc), "cuda")
    out = torch.empty_like(q)
    return lambda: mv.massv_verify_attn(desc, q, k, v, kp, vp, table, lens, out, None, None, ws, None), lambda: [out]


def _acceptance(mv, batch, gamma, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    R, K, V = gamma + 1, 1024, 4096
    hidden = torch.randn((batch, R, K), generator=g, device="cuda").to(torch.bfloat16)
    w = torch.randn((V, K), generator=g, device="cuda").to(torch.bfloat16)
    drafts = torch.zeros((batch, gamma), dtype=torch.int32, device="cuda")
    desc = mv.accept_desc(batch, gamma, K, V, 0.0)
    ws = mv.alloc_workspace(mv.massv_accept_workspace_size(desc), "cuda")
    tokens, lens = torch.empty((batch, R), dtype=torch.int32, device="cuda"), torch.empty((batch,), dtype=torch.int32, device="cuda")
    return lambda: mv.massv_accept(desc, hidden, w, drafts, None, None, None, tokens, lens, None, None, ws, None), lambda: [tokens, lens]


def _work(mv, i):
    """Pairs of calls that go to the same kernel with different amounts of shared memory."""
    if i < 4:
        return _attention(mv, (1, 900, 64, 700)[i], 5, 256, i)
    return _acceptance(mv, *((16, 5), (42, 5), (50, 5), (60, 4), (64, 7), (80, 4))[i - 4], i)


def test_two_sizes_of_one_kernel_at_a_time():
    import paper_2505_10526_b200 as mv
    n = 10
    alone = []
    for i in range(n):
        call, results = _work(mv, i)
        call()
        torch.cuda.synchronize()
        alone.append([t.clone() for t in results()])
    errors, got = [], [None] * n

    def body(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                call, results = _work(mv, i)
                for _ in range(300):
                    call()
                torch.cuda.current_stream().synchronize()
                got[i] = results()
        except Exception as e:          # the main thread reports it
            errors.append((i, e))

    threads = [threading.Thread(target=body, args=(i,)) for i in range(n)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i in range(n):
        assert all(torch.equal(a, b) for a, b in zip(alone[i], got[i])), i
