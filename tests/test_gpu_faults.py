"""GPU tests of faults that were found and mended: each one failed on the code that had the fault."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def long_context_state(n=131071, Hq=32, Hkv=8, d=128):
    import torch
    from paper_2510_05688_b200 import binding as vb
    gen = torch.Generator(device="cuda").manual_seed(3)
    pages = (n + 15) // 16
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.bfloat16)
    q, kc, vc = rand(1, Hq, d), rand(pages, Hkv, 16, d), rand(pages, Hkv, 16, d)
    table = torch.randperm(pages, generator=gen, device="cuda").to(torch.int32)[None].contiguous()
    lens = torch.tensor([n], dtype=torch.int32, device="cuda")
    plan = vb.Plan(batch=1, num_q_heads=Hq, num_kv_heads=Hkv, head_dim=d, max_blocks_per_seq=pages, num_blocks=pages,
                   max_seq_len=n, dtype=vb.DTYPE_BF16)
    plan.set_params(base_rate=0.025, topk_frac=0.025)
    return plan, q, kc, vc, table, lens


def test_pages_of_the_score_pass_are_read_before_they_are_replaced():
    # The score kernel's ring slots are refilled by asynchronous copies while the walk kernel runs on the same SMs: a
    # refill overtook the reads of a page's last elements about once in three steps of this size.  Every score of every
    # step against the plain product (the workspace begins with the scores), and the outputs of all steps are the same.
    import torch
    plan, q, kc, vc, table, lens = long_context_state()
    Hq, n, d, Hkv = 32, 131071, 128, 8
    npad = (n + 31) // 32 * 32
    scores = plan.workspace[:Hq * npad * 4].view(torch.float32).view(Hq, npad)[:, :n]
    want = torch.empty(Hq, n, device="cuda")
    for g in range(Hkv):
        keys = kc[table[0].long(), g].reshape(-1, d)[:n].float()
        want[4 * g:4 * g + 4] = (q[0, 4 * g:4 * g + 4].double() @ keys.double().T / d ** 0.5).float()
    out, first = torch.empty_like(q), None
    for step in range(60):
        plan.decode(q, kc, vc, table, lens, 128, 128, 0, 0.05, 0.05, 3, out)
        torch.cuda.synchronize()
        # fp32 sums of 128 products of about unit size: 2e-5 is the bound of the other tests, a wrong element moves 0.1
        assert float((scores - want).abs().max()) < 1e-3, step
        first = out.clone() if first is None else first
        assert torch.equal(out, first), step
    assert plan.last_status() == 0
