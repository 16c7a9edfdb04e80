"""GPU parity at the sizes where the step's kernels change over: candidate bounds and their list, sections of the row
kernels, shared grids, the hand-over from whatever ran before on the stream.  Index sets, budgets and counts bit-exact
against the oracle, outputs within the tolerances of test_gpu_parity.py (derived there)."""
import numpy as np
import pytest

from paper_2510_05688_b200 import synth
from helpers import assert_parity, out_values, run_gpu, run_oracle
from test_gpu_parity import check, small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,heads,kv", [
    (2315, 4, 2),        # middle range of 2,303 tokens: the whole of it fits the candidate list
    (2316, 4, 2), (2317, 4, 2), (4096 + 12, 4, 2),
    (16385, 4, 2),       # 1024 threads from here on (512 below)
    (32768, 2, 1), (32769, 2, 1),
    (131072 + 1, 1, 1),  # more than 4,096 samples at every 32nd token: every 64th
])
def test_candidate_bound_sizes(n, heads, kv):
    case = small("bf16", [n], Hq=heads, Hkv=kv, k=max(16, n // 40), params=dict(base_rate=0.01))
    _, dbg, _, plan = check(case)
    assert plan.last_status() == 0
    assert (dbg["paths"] & 17 != 0).all()              # the usual selection, not its general case


@pytest.mark.parametrize("B,Hq", [(37, 4), (149, 1), (37, 8), (297, 1), (160, 8)])
def test_head_counts_of_the_selection_and_the_walk(B, Hq):
    # 296 | 297 heads: other block sizes of the selection on plans for short sequences; 1,280 heads share 1,184 walk CTAs
    lens = [(37 * i) % 700 + 1 for i in range(B)]
    check(small("bf16", lens, Hq=Hq, Hkv=1, d=64, k=9))


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("bf16", 64), ("fp32", 128), ("fp32", 64)])
def test_sections_of_the_row_kernels(dtype, d):
    # budgets around whole sections (256 entries) and batches; top-k sets and base samples likewise
    case = small(dtype, [3000, 1400], Hq=4, Hkv=2, d=d, k=244, params=dict(base_rate=0.1))
    for budget in (1, 255, 256, 257, 512, 513, 1100):
        check(case, force_budget=budget)
    for k in (243, 245, 500):
        check(small(dtype, [2600], Hq=2, Hkv=1, d=d, k=k, params=dict(base_rate=0.25)))


def test_many_heads_with_shares_of_whole_sections():
    # 128 heads: four statistics CTAs per kind share whole sections; 249 + 4 + 8 deterministic rows and more
    for k in (243, 244, 245, 600):
        check(small("bf16", [2900 + 7 * i for i in range(16)], Hq=8, Hkv=2, d=64, k=k, params=dict(base_rate=0.09)))


@pytest.mark.parametrize("B,Hq", [(4, 4), (17, 1), (8, 4), (11, 3), (32, 4), (43, 3), (40, 4), (23, 7),
                                  (37, 5), (62, 3), (74, 5), (53, 7), (64, 8)])
def test_head_counts_of_the_gather_and_the_statistics(B, Hq):
    # 16 | 17, 32 | 33 heads: other chunk counts and the other decomposition of the gather; 160 | 161 and 512: its least
    # chunk (128, 256, 512 rows); 128 | 129: rows per statistics CTA
    lens = [(53 * i) % 500 + 300 for i in range(B - 1)] + [1200]
    case = small("bf16", lens, Hq=Hq, Hkv=1, d=64, k=9)
    for budget in (129, 257, 513):
        check(case, force_budget=budget)


@pytest.mark.parametrize("d", [64, 128])
def test_infinite_key_elements(d):
    # an infinite K element whose score is -inf for the head that sees it: weight 0, everything else untouched.  The
    # statistics take the converting path for such a cache.
    case = small("bf16", [900], Hq=2, Hkv=2, d=d, heavy=None)
    q = synth.bf16_bits_to_f32(case.q)
    tok = 500
    page = case.block_table[0, tok // 16]
    case.k_cache = case.k_cache.copy()
    for g in range(2):
        case.k_cache[page, g, tok % 16, 3] = 0xFF80 if q[0, g, 3] > 0 else 0x7F80
    out_ref, det = run_oracle(case)
    out, dbg, plan = run_gpu(case)
    for (b, h), r in det.items():
        kk = int(dbg["topk_cnt"][b, h])
        assert np.array_equal(dbg["topk_idx"][b, h, :kk], r["I_t"])
        assert tuple(int(x) for x in dbg["budgets"][b, h]) == tuple(r["budgets"])
    assert np.abs(out_values(case, out) - out_values(case, out_ref)).max() <= 2e-2


def test_step_waits_for_the_kernels_in_front():
    # the step's first kernel is launched before its predecessor on the stream has finished: queries and lengths that
    # a long kernel writes right before the call are the ones that count, on every call of a loop
    import torch
    from paper_2510_05688_b200 import binding as vb
    case = small("bf16", [3000, 2000], Hq=8, Hkv=2)
    dev = vb.case_to_device(case)
    plan = vb.plan_for_case(case)
    plan.set_params(**case.params)
    gen = torch.Generator(device="cuda").manual_seed(1)
    qs = [torch.randn(dev["q"].shape, generator=gen, device="cuda").bfloat16() for _ in range(6)]
    lens = [torch.tensor([3000 - 100 * i, 500 + 250 * i], dtype=torch.int32, device="cuda") for i in range(6)]
    big = torch.randn(4096, 4096, device="cuda")

    def step(entry, q, l):
        o = torch.empty_like(q)
        if entry == "dense":
            plan.dense_decode(q, dev["k_cache"], dev["v_cache"], dev["block_table"], l, o)
        else:
            plan.decode(q, dev["k_cache"], dev["v_cache"], dev["block_table"], l, case.sink, case.window, case.k,
                        case.eps, case.delta, case.seed, o)
        return o

    for entry in ("sparse", "dense"):
        want = []
        for i in range(6):
            torch.cuda.synchronize()
            want.append(step(entry, qs[i], lens[i]))
        torch.cuda.synchronize()
        q, l, got = torch.zeros_like(qs[0]), torch.zeros_like(lens[0]), []
        for i in range(6):
            torch.mm(big, big)                         # (long enough for the next launches to queue up behind it)
            l.copy_(lens[i])
            q.copy_(qs[i])
            got.append(step(entry, q, l))
        torch.cuda.synchronize()
        assert all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(want, got)), entry


def test_plans_and_partial_steps_in_turn_on_one_stream():
    # two plans in turn; a step cut short by the measurement aid leaves nothing behind for the next one
    import torch
    from paper_2510_05688_b200 import binding as vb
    cases = [small("bf16", [700, 333, 0], Hq=4, Hkv=2), small("fp32", [900], Hq=4, Hkv=2, d=64)]
    devs = [vb.case_to_device(c) for c in cases]
    plans = [vb.plan_for_case(c) for c in cases]
    want = [run_oracle(c) for c in cases]
    for p, c in zip(plans, cases):
        p.set_params(**c.params)
    for rep in range(3):
        for p, c, dv, (ref, det) in zip(plans, cases, devs, want):
            out = torch.empty_like(dv["q"])
            args = (dv["q"], dv["k_cache"], dv["v_cache"], dv["block_table"], dv["seq_lens"], c.sink, c.window, c.k,
                    c.eps, c.delta, c.seed)
            for stop in ((1, 3, 4) if rep == 1 else ()):
                p.set_stop_after(stop)
                p.decode(*args, torch.empty_like(out))
                p.set_stop_after(0)
            p.decode(*args, out)
            torch.cuda.synchronize()
            got = out.view(torch.int16).cpu().numpy().view(np.uint16) if c.dtype == "bf16" else out.cpu().numpy()
            diff = np.abs(out_values(c, got) - out_values(c, ref))
            assert diff.max() <= (2e-2 if c.dtype == "bf16" else 1e-5 * np.abs(out_values(c, ref)).max()), rep
            assert p.last_status() == 0


@pytest.mark.parametrize("dtype,n", [("bf16", 2400), ("bf16", 33000), ("fp32", 5000), ("bf16", 131073)])
@pytest.mark.parametrize("offset", [5.0, 40.0])
def test_logits_with_a_common_offset(dtype, n, offset):
    # queries and keys share a component: every logit is the offset and a little, so the sample's keys crowd into one bin
    # of the top 12 bits and the bound comes from the next 12
    case = small(dtype, [n], Hq=2, Hkv=1, d=64, k=n // 40, key_std=0.1, heavy=None, params=dict(base_rate=0.02))
    a = np.sqrt(offset * 8.0 / 64.0)
    store = synth.f32_to_bf16_bits if dtype == "bf16" else (lambda x: x.astype(np.float32))
    case.q, case.k_cache = store(case.values(case.q) + np.float32(a)), store(case.values(case.k_cache) + np.float32(a))
    _, dbg, det, plan = check(case)
    assert det[(0, 0)]["m"] > 0.6 * offset and plan.last_status() == 0
    assert (dbg["paths"] & 17 != 0).all()


@pytest.mark.parametrize("dtype,n,k", [("bf16", 131073, 20000), ("bf16", 40000, 17000), ("fp32", 33000, 15000), ("bf16", 20000, 12000)])
def test_top_k_sets_around_the_candidate_list(dtype, n, k):
    # more members than the list of 16,384 candidates takes (or may take): the general selection with a threshold; 12,000
    # of 20,000 tokens: the usual one with an almost full list
    _, dbg, _, plan = check(small(dtype, [n], Hq=2, Hkv=1, d=64, k=k, params=dict(base_rate=0.02)))
    assert plan.last_status() == 0
    assert ((dbg["paths"] & 17 != 0) == (n == 20000)).all()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("eps", [0.07, 0.03])
def test_lists_from_laid_out_walk_entries(dtype, eps):
    # half of the tokens are top-k: more than 1,024 marked entries in the final sample's array, so every budget is served
    # from a list, inside the array (8 base budgets) and beyond it
    case = small(dtype, [12000], Hq=2, Hkv=1, d=64, k=6000, key_std=0.1, heavy=None, eps=eps, delta=eps)
    _, dbg, det, plan = check(case)
    for r in det.values():
        assert r["b0"] < r["b"] < 8 * r["b0"] if eps == 0.07 else 8 * r["b0"] < r["b"] < r["n_s"]
    assert plan.last_status() == 0


@pytest.mark.parametrize("B,Hq", [(8, 16), (37, 5), (62, 3), (37, 10), (53, 7)])
def test_statistics_ctas_per_head(B, Hq):
    # 128 and 185 heads: four CTAs per kind and head; 186, 370: two; 371: one; with rows for more than four of either kind
    # (256 rows each, 64 up to 128 heads)
    case = small("bf16", [4000 - 3 * i for i in range(B)], Hq=Hq, Hkv=1, d=64, k=1300, params=dict(base_rate=0.45))
    _, dbg, _, _ = check(case)
    assert (dbg["topk_cnt"] > 4 * 256).all() and (dbg["base_cnt"] > 4 * 256).all()


@pytest.mark.parametrize("B,Hq,tokens", [(37, 2, 16400), (15, 5, 16400), (15, 5, 65536), (15, 5, 65552), (37, 4, 65552), (149, 1, 65552)])
def test_block_sizes_of_the_selection(B, Hq, tokens):
    # 1,024 threads above 16,384 tokens up to 74 heads, above 65,536 up to 148; 512 otherwise (the plan's longest sequence
    # decides, whatever the sequences are now)
    lens = [(389 * i) % 3000 + 1 for i in range(B)]
    check(small("bf16", lens, Hq=Hq, Hkv=1, d=64, k=60, max_blocks=tokens // 16))


def test_paths_tell_where_the_bound_came_from():
    # 75 heads on a plan for up to 65,536 tokens run 512 threads (every 32nd token up to there); 1 head runs 1,024
    lens = [700] * 14 + [65536]
    _, dbg, plan = run_gpu(small("bf16", lens, Hq=5, Hkv=1, d=64, k=100))
    assert (dbg["paths"] & 17 == 1).all() and plan.last_status() == 0
    _, dbg, plan = run_gpu(small("bf16", [700] * 148 + [70000], Hq=1, Hkv=1, d=64, k=100))       # (149 heads: 512 threads)
    assert (dbg["paths"][:148] & 17 == 1).all() and (dbg["paths"][148] & 17 == 16).all()
    _, dbg, plan = run_gpu(small("bf16", [700, 70000], Hq=1, Hkv=1, d=64, k=100))
    assert (dbg["paths"] & 17 == 1).all()


@pytest.mark.parametrize("dtype,B,Hq,Hkv,d,max_len", [
    ("fp32", 1, 1, 1, 64, None), ("bf16", 1, 16, 2, 128, None), ("bf16", 2, 8, 8, 64, None), ("bf16", 17, 1, 1, 128, None),
    ("fp32", 4, 8, 2, 64, 8192), ("fp32", 4, 8, 2, 64, 8208), ("fp32", 4, 8, 2, 64, 16384), ("fp32", 4, 8, 2, 64, 16400),
    ("fp32", 4, 8, 2, 128, 2048), ("fp32", 4, 8, 2, 128, 16384), ("fp32", 11, 3, 3, 64, None), ("bf16", 1, 4, 1, 128, 16384), ("bf16", 1, 1, 1, 64, 16400),
    ("bf16", 1, 8, 2, 128, 16384), ("bf16", 1, 16, 4, 128, 8192), ("bf16", 1, 16, 4, 128, 8208), ("fp32", 1, 1, 1, 128, 8192), ("fp32", 1, 1, 1, 128, 8208)])
def test_rows_of_a_head_in_one_kernel_and_in_two(dtype, B, Hq, Hkv, d, max_len):
    # 16 | 17 heads, 32 | 33 fp32 heads of 64 elements and 16,384 | 16,385 tokens, a head's sampled rows of up to 16,384 and 4 MB
    # and all heads' of up to 16 Mi elements: one kernel for statistics, budget and gather, or two (which the measurement aids always
    # take).  Empty and one-token rows, no middle range, budgets up to the whole residual, nested samples, fewer rows than CTAs.
    from paper_2510_05688_b200 import binding as vb
    lens = ([1501, 0, 1, 13] + [(97 * i) % 900 + 40 for i in range(B)])[:B]
    case = small(dtype, lens, Hq=Hq, Hkv=Hkv, d=d, k=37, params=dict(base_rate=0.03))
    fused = B * Hq <= (32 if dtype == "fp32" and d == 64 and (max_len or 0) <= 16384 else 16)
    width = 16 * case.max_blocks_per_seq if max_len is None else max_len
    if width > 16 * case.max_blocks_per_seq:
        table = np.zeros((B, (width + 15) // 16), case.block_table.dtype)
        table[:, :case.max_blocks_per_seq] = case.block_table
        case.block_table = table
    for over in ({}, dict(force_budget=1), dict(force_budget=700), dict(force_budget=1 << 20), dict(nested_base=1), dict(base_rate=0.9)):
        out_ref, det = run_oracle(case, **over)
        for two in (False, True):
            plan = vb.plan_for_case(case, max_seq_len=width)
            plan.set_profiling(two)
            out, dbg, _ = run_gpu(case, plan=plan, **over)
            sampled = min(over.get("force_budget", width), width)
            one = (fused and not two and 4 + 8 + 37 + over.get("base_rate", 0.03) * width <= 4096 and sampled <= 16384
                   and sampled * d * (2 if dtype == "bf16" else 4) <= 4 << 20 and B * Hq * sampled * d <= 16 << 20)
            assert plan.last_launch_count() == (4 if one else 5)
            assert_parity(case, out, dbg, det, out_ref)
            assert plan.last_status() == 0
            plain, _, _ = run_gpu(case, debug=False, plan=plan, **over)
            assert np.array_equal(plain, out)


@pytest.mark.parametrize("heads,k", [(2, 1500), (17, 1500), (2, 1110), (2, 1000)])
def test_budgets_beyond_the_walk_array_with_many_members_there(heads, k):
    # more members of I_t at walk positions beyond the array than a list of 1,024 holds: the budget counts them all
    case = small("bf16", [9000], Hq=heads, Hkv=1, d=64, k=k, eps=0.1, delta=0.1, params=dict(base_rate=0.01))
    out, dbg, det, plan = check(case)
    b0 = det[(0, 0)]["b0"]
    far = [r["b"] for r in det.values() if 8 * b0 < r["b"] < r["n_s"]]
    assert far                                          # (beyond the array, short of the whole residual)
    assert plan.last_status() == 0
    for mode in (1, 2):
        check(case, mode=mode)


@pytest.mark.parametrize("dtype,heads,d", [("bf16", 3, 128), ("bf16", 3, 64), ("fp32", 2, 64), ("fp32", 2, 128), ("bf16", 17, 128),
                                           ("bf16", 40, 64), ("fp32", 33, 64)])
@pytest.mark.parametrize("n", [4120, 8250])
def test_budgets_far_beyond_the_walk_array(dtype, heads, d, n):
    # nearly all of the sample at computed walk entries, with |M| just above a power of two: several of them per lane in stages
    # of either size, chunks that begin in the array, behind it, and at the end of one another's; one kernel for the rows and two
    case = small(dtype, [n, n - 77, 900], Hq=heads, Hkv=1, d=d, k=150, eps=0.13, delta=0.2, params=dict(base_rate=0.004))
    out, dbg, det, plan = check(case)
    far = [r["b"] for r in det.values() if 16 * r["b0"] < r["b"] < r["n_s"]]
    assert far
    assert plan.last_status() == 0
    check(case, gather_mode=1)


@pytest.mark.parametrize("dtype,d,max_len", [("bf16", 128, 4000), ("bf16", 64, 4000), ("fp32", 64, 4000), ("fp32", 128, 4000), ("bf16", 128, 30000)])
def test_lists_of_few_heads(dtype, d, max_len):
    # more than 1,024 members of I_t in the final sample's walk array: every budget short of the whole residual is served from a
    # list, which one of the head's CTAs writes for the others (the plan of 4,000 tokens) or the last CTA of the statistics (30,000)
    import oracle.vattn_oracle as O
    from paper_2510_05688_b200 import binding as vb
    case = small(dtype, [4000, 3990], Hq=2, Hkv=1, d=d, k=2000, eps=0.03, delta=0.03, params=dict(base_rate=0.1))
    if max_len > 4000:
        table = np.zeros((2, max_len // 16), case.block_table.dtype)
        table[:, :case.max_blocks_per_seq] = case.block_table
        case.block_table = table
    for over in (dict(force_budget=1500), dict(), dict(mode=2)):
        out_ref, det = run_oracle(case, **over)
        for (b, h), r in det.items():
            mlen = r["n"] - case.sink - case.window
            order = np.array(O.walk_order(mlen, O.walk_round_keys(case.seed, b, h, 0, 0, 1)))
            member = np.zeros(mlen, bool)
            member[np.asarray(r["I_t"]) - case.sink] = True
            laid = over.get("force_budget", 8 * r["b0"])                  # residual tokens in the array, at least
            marked = int(np.searchsorted(np.cumsum(~member[order]), laid)) - laid
            assert marked > 1024 and 0 < r["b"] < r["n_s"]
        plan = vb.plan_for_case(case, max_seq_len=max_len)
        out, dbg, _ = run_gpu(case, plan=plan, **over)
        assert plan.last_launch_count() == (4 if max_len == 4000 else 5)
        assert_parity(case, out, dbg, det, out_ref)
        plain, _, plan = run_gpu(case, debug=False, plan=plan, **over)
        assert np.array_equal(plain, out)
        assert plan.last_status() == 0


@pytest.mark.parametrize("dtype,heads,n,k,eps,over", [
    ("bf16", 2, 9000, 1500, 0.01, {}), ("bf16", 17, 9000, 1500, 0.01, {}), ("fp32", 2, 9000, 1500, 0.01, {}),
    ("bf16", 40, 3000, 100, 0.03, {}), ("fp32", 1, 3000, 100, 0.1, dict(force_budget=1 << 20)),
    ("bf16", 2, 3000, 100, 0.03, dict(gather_mode=1))])
def test_infinite_value_elements_of_top_k_tokens(dtype, heads, n, k, eps, over):
    # members of I_t belong to the deterministic sums alone.  Where the gather meets them on the final sample's walk (laid out,
    # beyond the array, in token order) they weigh nothing, whatever their rows hold: an infinity stays one
    case = small(dtype, [n], Hq=heads, Hkv=1, d=64, k=k, eps=eps, delta=eps, params=dict(base_rate=0.01, mode=1))
    _, det = run_oracle(case, **over)
    case.v_cache = case.v_cache.copy()
    for e, tok in enumerate(det[(0, 0)]["I_t"][:48]):
        case.v_cache[case.block_table[0, tok // 16], 0, tok % 16, e] = 0x7F80 if dtype == "bf16" else np.inf
    with np.errstate(invalid="ignore"):
        out_ref, det = run_oracle(case, **over)
    out, dbg, plan = run_gpu(case, **over)
    assert all(r["b"] == int(dbg["dyn_cnt"][b, h]) for (b, h), r in det.items())
    ref, got = out_values(case, out_ref), out_values(case, out)
    assert np.isposinf(ref[0, 0, :48]).all() and np.isfinite(ref[..., 48:]).all()
    assert np.array_equal(np.isposinf(ref), np.isposinf(got)) and not np.isnan(got).any()
    fin = np.isfinite(ref)
    assert np.abs(got[fin] - ref[fin]).max() <= (2e-2 if dtype == "bf16" else 1e-4)      # (as for infinite keys; fp32 sums)
