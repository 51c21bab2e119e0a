"""Calls that follow each other on a stream: every kernel may be launched while
the one before it still runs, and must see all of its results."""
import pytest
import torch

from gpu_util import dev

pytestmark = pytest.mark.gpu


def chain(sync, dtype, B, L, V, d, rounds):
    """Rounds of dependent calls, each reading what the one before it (a call of
    the library or a torch kernel) has just written; all results."""
    from paper_2608_02625_gb300 import binding as Bn
    dv = dev()
    g = torch.Generator(device=dv).manual_seed(B * L + V)
    i32, f32 = torch.int32, torch.float32
    Hq, Hkv, D = 4, 2, 64
    q = torch.randn(B, L, Hq, D, device=dv, generator=g).to(dtype)
    kv = torch.randn(B, L, Hkv, D, device=dv, generator=g).to(dtype)
    w = (torch.randn(V, d, device=dv, generator=g) * d ** -0.5).to(torch.bfloat16)
    n = torch.full((B,), L, dtype=i32, device=dv)
    p = torch.full((B,), L // 4, dtype=i32, device=dv)
    prm = Bn.RefineParams(0.2, -1, 0.2, V, p, n)
    tok = torch.randint(0, V, (B, L), dtype=i32, device=dv, generator=g)
    msk = (torch.rand(B, L, device=dv, generator=g) < 0.3).to(torch.uint8)
    new = [torch.empty_like(tok), torch.empty_like(msk), torch.empty_like(n)]
    rows = [torch.empty(B, L, dtype=t, device=dv) for t in (i32, f32, f32)]
    lm = [torch.empty(B * L, dtype=t, device=dv) for t in (i32, f32, f32)]
    prob = torch.empty(B, L, dtype=f32, device=dv)
    ws = torch.zeros(B, dtype=i32, device=dv)
    lws = torch.empty(Bn.dlm_lmhead_workspace_bytes(B * L), dtype=torch.uint8, device=dv)
    out, out2 = torch.empty_like(q), torch.empty_like(q)
    seen = []

    def step(*tensors):
        if sync:
            torch.cuda.synchronize()
        seen.extend(t.clone() for t in tensors)

    for r in range(rounds):
        Bn.dlm_bidir_attn(q, kv, kv, n, out)
        step(out)
        Bn.dlm_attn_masked(out, kv, kv, n, p, 1, 16, out2)
        Bn.dlm_bidir_attn(out2, kv, kv, n, out)
        step(out2, out)
        hidden = out.reshape(B * L, Hq * D)[:, :d].to(torch.bfloat16)
        Bn.dlm_lmhead_confidence(hidden, w, *lm, lws)
        Bn.dlm_lmhead_confidence(hidden, w, *lm, lws)
        step(*lm)
        x = (hidden.float() @ w.float().T * 4).to(dtype).view(B, L, V)
        Bn.dlm_vocab_confidence(x, *rows)
        Bn.dlm_token_prob(x, tok, rows[2], prob)
        Bn.dlm_refine_update_ranked(tok, msk, rows[0], rows[1], prob, prm, *new)
        step(*rows, prob, *new)
        Bn.dlm_refine_step(x, new[0], new[1], prm, *rows, tok, msk, new[2], ws)
        Bn.dlm_refine_step(x, tok, msk, prm, *rows, tok, msk, new[2], ws)
        Bn.dlm_refine_update(tok, msk, rows[0], rows[1], prm, *new)
        step(*rows, tok, msk, *new)
        q.mul_(0.5).add_(out)
    torch.cuda.synchronize()
    assert Bn.device_error(clear=True) == 0
    return seen


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("B,L,V", [(1, 16, 40), (3, 130, 2001), (40, 64, 333), (2, 700, 70001)])
def test_results_do_not_depend_on_waiting_between_calls(dtype, B, L, V):
    waited = chain(True, dtype, B, L, V, 64, 3)
    for _ in range(3):
        for a, b in zip(chain(False, dtype, B, L, V, 64, 3), waited):
            assert torch.equal(a, b)
