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


def test_pivot_behind_walk_entries_that_are_all_members():
    # 60 of 100 middle tokens are top-k and the base walk begins with 24 to 31 of them: its first residual token lies
    # behind the entries that were laid out ahead (24 here), but below position 32.  The residual rows are all alike, so
    # around the right pivot (one of them) both variances are exactly zero, and so are the budgets; around a top-k row
    # they are rounding errors of its weight.
    from oracle import vattn_oracle as O
    from helpers import run_gpu
    from paper_2510_05688_b200 import synth
    H, d, n, sink, window, k = 8, 64, 112, 4, 8, 60
    case = synth.make_case("pivot", dtype="bf16", B=1, Hq=H, Hkv=H, d=d, seq_lens=[n], sink=sink, window=window, k=k,
                           eps=0.05, delta=0.05, seed=77, gen_seed=1, params=dict(base_rate=0.08))
    q = case.values(case.q)
    K, V = np.zeros((H, n, d), np.float32), np.ones((H, n, d), np.float32)
    for h in range(H):
        order = sink + O.walk_order(n - sink - window, O.walk_round_keys(case.seed, 0, h, 0, 0, 0))
        first = 24 + h                                     # the walk position of the first residual token
        members = np.concatenate([order[:first], order[first + 100 - k:]])
        assert len(members) == k
        K[h, members] = (3.1 + 0.37 * h) * np.sqrt(d) * q[0, h] / (q[0, h] @ q[0, h])
        V[h, members] = 1.5 + 0.25 * h
    pages = n // 16
    to_pages = lambda x: x.reshape(H, pages, 16, d).transpose(1, 0, 2, 3)
    case.k_cache, case.v_cache = case.k_cache.copy(), case.v_cache.copy()
    case.k_cache[case.block_table[0, :pages]] = synth.f32_to_bf16_bits(to_pages(K))
    case.v_cache[case.block_table[0, :pages]] = synth.f32_to_bf16_bits(to_pages(V))
    out, dbg, plan = run_gpu(case)
    assert (dbg["topk_cnt"] == k).all() and (dbg["base_cnt"] == 3).all() and plan.last_status() == 0
    assert (dbg["stats"][0, :, 1:3] == 0.0).all()
    assert (dbg["budgets"][0, :, :3] == 0).all()


@pytest.mark.parametrize("stop", [1, 2, 3, 4])
def test_recorded_step_after_a_step_that_was_cut_short(stop):
    # a caller's graph carries no clearing of the step's counters: the measurement aid, called between two replays with
    # another query, left a used-up unit counter and the maxima of its own scores to the next replay
    import torch
    from paper_2510_05688_b200 import binding as vb
    from paper_2510_05688_b200 import synth
    case = synth.make_case("cut", dtype="bf16", B=6, Hq=8, Hkv=2, d=128, seq_lens=[9000, 20000, 700, 30000, 1, 8191], sink=4,
                           window=8, k=100, eps=0.05, delta=0.05, seed=5, gen_seed=6,
                           heavy=dict(R=12, c1=5.0, alpha=(0.75, 1.25)), params=dict(base_rate=0.05))
    dev = vb.case_to_device(case)
    plan = vb.plan_for_case(case)
    plan.set_params(**case.params)
    q1, q2 = dev["q"], 60.0 * dev["q"].flip(1)       # (far larger scores)
    q, out = q1.clone(), torch.empty_like(q1)
    stream = torch.cuda.Stream()

    def step():
        plan.decode(q, dev["k_cache"], dev["v_cache"], dev["block_table"], dev["seq_lens"], case.sink, case.window, case.k,
                    case.eps, case.delta, case.seed, out, stream=stream)

    step()
    torch.cuda.synchronize()
    want = out.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        step()
    for _ in range(2):
        q.copy_(q2)
        torch.cuda.synchronize()
        plan.set_stop_after(stop)
        step()
        plan.set_stop_after(0)
        torch.cuda.synchronize()
        q.copy_(q1)
        out.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
    assert plan.last_status() == 0


def test_plans_that_take_turns_on_one_workspace():
    # two plans of other shapes on the same memory: each finds the other's scores and lists where its own counters are
    # (unit counters and maxima that are not zero), whichever ran last, through both entry points, and when one is gone
    import torch
    from helpers import out_values, run_oracle
    from paper_2510_05688_b200 import binding as vb
    from paper_2510_05688_b200 import synth
    kw = dict(d=64, sink=4, window=8, k=16, eps=0.05, delta=0.05, seed=1, params=dict(base_rate=0.05))
    cases = [synth.make_case("a", dtype="bf16", B=3, Hq=8, Hkv=2, seq_lens=[5000, 333, 0], gen_seed=1, **kw),
             synth.make_case("b", dtype="bf16", B=2, Hq=4, Hkv=4, seq_lens=[900, 2500], gen_seed=2, **kw)]
    want = [out_values(c, run_oracle(c)[0]) for c in cases]
    devs = [vb.case_to_device(c) for c in cases]
    plans = [vb.Plan(batch=c.batch, num_q_heads=c.num_q_heads, num_kv_heads=c.num_kv_heads, head_dim=64,
                     max_blocks_per_seq=c.max_blocks_per_seq, num_blocks=c.num_blocks, max_seq_len=c.max_blocks_per_seq * 16,
                     dtype=vb.DTYPE_BF16, alloc_workspace=False) for c in cases]
    need = max(p.workspace_bytes() for p in plans)
    mem = torch.empty(need + 4096, dtype=torch.uint8, device="cuda")
    plans[0].set_workspace(mem.data_ptr(), need)
    plans[1].set_workspace(mem.data_ptr() + 4096, need)              # (overlapping, not the same address)
    pinned = [{x: dv[x].cpu().pin_memory() for x in ("q", "block_table", "seq_lens")} for dv in devs]
    stream = torch.cuda.Stream()

    def run(i, host):
        c, dv, p = cases[i], devs[i], plans[i]
        p.set_params(**c.params)
        scalars = (c.sink, c.window, c.k, c.eps, c.delta, c.seed)
        torch.cuda.synchronize()
        if host:
            out = torch.empty_like(pinned[i]["q"]).pin_memory()
            for _ in range(3):
                p.decode_host(pinned[i]["q"], dv["k_cache"], dv["v_cache"], pinned[i]["block_table"], pinned[i]["seq_lens"],
                              *scalars, out, stream=stream)
        else:
            out = torch.empty_like(dv["q"])
            p.decode(dv["q"], dv["k_cache"], dv["v_cache"], dv["block_table"], dv["seq_lens"], *scalars, out)
        torch.cuda.synchronize()
        got = out_values(c, out.view(torch.int16).cpu().numpy().view(np.uint16))
        assert np.abs(got - want[i]).max() <= 2e-2, (i, host)

    for host in (False, True, False):
        for i in (0, 1, 0, 0, 1, 1):
            run(i, host)
    del plans[1]                                                     # (its counters are still lying there)
    run(0, False)
    run(0, True)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("padded", [False, True])
def test_cache_that_a_32_bit_row_index_does_not_cover(dtype, padded):
    # such plans were refused: a bound on the page numbers that bounds nothing (2^31 - 1), and page and token strides whose
    # common divisor is the 16 bytes of their alignment
    import torch
    from helpers import assert_parity, run_gpu, run_oracle
    from paper_2510_05688_b200 import binding as vb
    from paper_2510_05688_b200 import synth
    Hq, Hkv, d = 8, 2, 64
    case = synth.make_case("rows", dtype=dtype, B=2, Hq=Hq, Hkv=Hkv, d=d, seq_lens=[3000, 129], sink=4, window=8, k=100, eps=0.05,
                           delta=0.05, seed=5, gen_seed=6, heavy=dict(R=12, c1=5.0, alpha=(0.75, 1.25)), params=dict(base_rate=0.05))
    dev, nblk = vb.case_to_device(case), case.num_blocks
    strides = (0, 0, 0)
    if padded:
        align = 8 if dtype == "bf16" else 4
        st = d + align
        sh = 16 * st
        strides = (Hkv * sh + align, sh, st)
        assert np.gcd(strides[0], st) == align
        for name in ("k_cache", "v_cache"):
            buf = torch.full((nblk * strides[0],), 7.0, dtype=dev[name].dtype, device="cuda")
            torch.as_strided(buf, (nblk, Hkv, 16, d), (*strides, 1)).copy_(dev[name])
            dev[name] = buf
    plan = vb.Plan(batch=2, num_q_heads=Hq, num_kv_heads=Hkv, head_dim=d, max_blocks_per_seq=case.max_blocks_per_seq,
                   num_blocks=2 ** 31 - 1, max_seq_len=case.max_blocks_per_seq * 16, kv_strides=strides,
                   dtype=vb.DTYPE_BF16 if dtype == "bf16" else vb.DTYPE_FP32)
    for mode in (dict(), dict(gather_mode=1)):
        out_ref, det = run_oracle(case, **mode)
        got, dbg, _ = run_gpu(case, plan=plan, dev=dev, **mode)
        assert_parity(case, got, dbg, det, out_ref)
    assert plan.last_status() == 0
