"""GPU tests of the two further forms of the compact cache (section 2.2.2 as driven during prefill, section
2.1's decode cache): compaction inside the layer's own buffer, and gather into a paged cache through a
block table.  Both are bit-exact against the oracle's gather on the same indices."""
import numpy as np
import pytest
import torch

import oracle
from paper_2503_17922_b200 import binding
from paper_2503_17922_b200 import workloads as wl

import parity_util as pu

pytestmark = pytest.mark.gpu


def _case(**kw):
    base = dict(name="cache-forms", dtype="bf16", batch=2, n_layers=2, gamma=2, n_q_heads=8, n_kv_heads=2,
                head_dim=128, max_seqlen=1337, l_obs=16, window=8, top_p=4, budget_frac=0.2, n_planted=5, config_id=12)
    base.update(kw)
    return wl.scaled(wl.llama8b_single_group(), **base)


def _indices(w, grp, prob, pattern):
    """Window lists chosen by the test (ascending, k per sequence): 'selected' = the oracle's selection;
    'shift' = windows 1..k (every output window lies on the source of the next slot); 'tail' = the last k
    windows (the longest moves, ragged last window included); 'front' = windows 0..k-1 (nothing moves)."""
    if pattern == "selected":
        ref = oracle.select_leader(grp["q_obs"], grp["k_layers"][0], **pu.oracle_kwargs(w, grp))
        return np.ascontiguousarray(ref["window_idx"], dtype=np.int32)
    idx = np.full((w.batch, w.n_kv_heads, prob.k_max), -1, dtype=np.int32)
    for b in range(w.batch):
        n = int(grp["seqlens"][b])
        kw = oracle.num_windows(n, w.l_obs, w.window)
        k = oracle.num_selected(n, w.l_obs, w.window, int(grp["budgets"][b]))
        for h in range(w.n_kv_heads):
            if pattern == "shift":
                lo = 1 if k < kw else 0
            elif pattern == "tail":
                lo = kw - k
            elif pattern == "run":      # half of them a run from window 2 on, the rest spread over what follows
                half = min(k // 2, kw - 2) if kw > 2 else 0
                rest = np.random.Generator(np.random.Philox(key=h)).permutation(np.arange(2 + half, kw))[: k - half]
                if half + len(rest) == k:
                    idx[b, h, :k] = np.concatenate([np.arange(2, 2 + half), np.sort(rest)])
                    continue
                lo = 0
            else:
                lo = 0
            idx[b, h, :k] = np.arange(lo, lo + k)
    return idx


@pytest.mark.parametrize("pattern", ["selected", "shift", "tail", "front"])
@pytest.mark.parametrize("case", [
    dict(),                                                    # dense [B, H_kv, N, d]
    dict(layout="bnhd", window=16, max_seqlen=777),            # token-major rows
    dict(ragged=True, batch=3, max_seqlen=900),                # packed [T, H_kv, d]
    dict(dtype="f32", head_dim=64, n_q_heads=4, l_obs=8),
    dict(budget_frac=0.9, max_seqlen=2100),                    # most rows kept: many batches per unit, short moves
    dict(budget_frac=None, budget_tokens=10 ** 6),             # everything kept: nothing moves
], ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()) or "base")
def test_compaction_in_place(case, pattern):
    case = dict(case)
    layout, budgets = case.pop("layout", "bhnd"), case.pop("budgets", None)
    w = _case(**case)
    grp = wl.make_group(w, 0)
    if budgets is not None:
        grp["budgets"] = np.array(budgets, dtype=np.int32)
    prob = binding.Problem(dtype=w.dtype, batch=w.batch, n_q_heads=w.n_q_heads, n_kv_heads=w.n_kv_heads,
                           head_dim=w.head_dim, l_obs=w.l_obs, window=w.window, task=w.task, top_p=w.top_p,
                           max_seqlen=w.max_seqlen, budgets=grp["budgets"], cu_seqlens=grp["cu_seqlens"],
                           kv_layout=layout)
    idx = _indices(w, grp, prob, pattern)

    def dev(x):
        return binding.to_device(np.ascontiguousarray(x.transpose(0, 2, 1, 3)) if layout == "bnhd" else x)
    ks = [dev(x) for x in grp["k_layers"]]
    vs = [dev(x) for x in grp["v_layers"]]
    before = [binding.to_host_bits(t) for t in ks + vs]
    binding.wkv_compact_kv_inplace(prob, ks, vs, torch.from_numpy(idx).cuda())
    torch.cuda.synchronize()
    kw_ = dict(n_kv_heads=w.n_kv_heads, l_obs=w.l_obs, window=w.window, max_seqlen=w.max_seqlen,
               budgets=grp["budgets"], keep_max=prob.keep_max, cu_seqlens=grp["cu_seqlens"], fill=0)
    moved = 0
    for layer in range(w.gamma):
        for src, got_t, old in ((grp["k_layers"][layer], ks[layer], before[layer]),
                                (grp["v_layers"][layer], vs[layer], before[w.gamma + layer])):
            exp = oracle.gather_layer(src, idx, **kw_)                  # dense [B, H_kv, keep_max, d]
            got = binding.to_host_bits(got_t)
            for b in range(w.batch):
                n = int(grp["seqlens"][b])
                n_r = max(n - w.l_obs, 0)
                k = oracle.num_selected(n, w.l_obs, w.window, int(grp["budgets"][b]))
                for h in range(w.n_kv_heads):
                    kept = sum(min((int(i) + 1) * w.window, n_r) - int(i) * w.window for i in idx[b, h, :k]) + min(w.l_obs, n)
                    if grp["cu_seqlens"] is not None:
                        lo = int(grp["cu_seqlens"][b])
                        unit_rows, old_rows = got[lo:lo + n, h], old[lo:lo + n, h]
                    elif layout == "bnhd":
                        unit_rows, old_rows = got[b, :n, h], old[b, :n, h]
                    else:
                        unit_rows, old_rows = got[b, h, :n], old[b, h, :n]
                    np.testing.assert_array_equal(unit_rows[:kept], exp[b, h, :kept])
                    # rows behind the compact cache are leftovers: each still equals some row of the old tensor
                    # at the same position (never written) - the kernel writes nothing at or beyond kept
                    np.testing.assert_array_equal(unit_rows[kept:], old_rows[kept:])
                    moved += int((unit_rows[:kept] != old_rows[:kept]).any())
    if pattern in ("shift", "tail", "selected") and case.get("budget_tokens") is None:
        assert moved > 0


@pytest.mark.parametrize("pool_layout", ["heads-outer", "token-major"])
@pytest.mark.parametrize("case", [
    dict(),
    dict(ragged=True, batch=3, max_seqlen=900, window=16),
    dict(dtype="f32", head_dim=64, n_q_heads=4, l_obs=8),
], ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()) or "base")
def test_gather_into_a_paged_cache(case, pool_layout):
    """Pages of 24 rows (not a multiple of the window length, so windows straddle pages), a block table
    that scatters every sequence's pages over the pool, one table for all layers and for K and V."""
    w = _case(**case)
    grp = wl.make_group(w, 0)
    prob = binding.Problem.from_workload(w)
    ref = oracle.select_leader(grp["q_obs"], grp["k_layers"][0], **pu.oracle_kwargs(w, grp))
    idx = np.ascontiguousarray(ref["window_idx"], dtype=np.int32)
    ps = 24
    max_pages = -(-prob.keep_max // ps)
    num_pages = w.batch * max_pages + 5
    g = np.random.Generator(np.random.Philox(key=99))
    table = g.permutation(num_pages)[: w.batch * max_pages].reshape(w.batch, max_pages).astype(np.int32)
    H, d = w.n_kv_heads, w.head_dim
    tdt = torch.float32 if w.dtype == "f32" else torch.bfloat16
    if pool_layout == "heads-outer":
        shape, strides = (num_pages, H, ps, d), (H * ps * d, ps * d, d)
    else:
        shape, strides = (num_pages, ps, H, d), (ps * H * d, d, H * d)
    ks = [binding.to_device(x) for x in grp["k_layers"]]
    vs = [binding.to_device(x) for x in grp["v_layers"]]
    pools = [[torch.empty(shape, dtype=tdt, device="cuda") for _ in range(w.gamma)] for _ in range(2)]
    for t in pools[0] + pools[1]:
        t.view(torch.uint8).fill_(pu.FILL_BYTE)
    binding.wkv_gather_kv_paged(prob, ks, vs, torch.from_numpy(idx).cuda(), pools[0], pools[1],
                                torch.from_numpy(table).cuda(), ps, num_pages, *strides)
    torch.cuda.synchronize()
    fill = pu.fill_pattern(w.dtype)
    kw_ = dict(n_kv_heads=H, l_obs=w.l_obs, window=w.window, max_seqlen=w.max_seqlen, budgets=grp["budgets"],
               keep_max=prob.keep_max, cu_seqlens=grp["cu_seqlens"], fill=fill)
    for layer in range(w.gamma):
        for src, pool in ((grp["k_layers"][layer], pools[0][layer]), (grp["v_layers"][layer], pools[1][layer])):
            exp = oracle.gather_layer(src, idx, **kw_)                  # dense [B, H, keep_max, d], fill behind kept
            got = binding.to_host_bits(pool)
            want = np.empty(got.shape, dtype=got.dtype)                 # the pool as the definition of the layout gives it
            want.view(np.uint32 if w.dtype == "f32" else np.uint16)[...] = fill
            for b in range(w.batch):
                for h in range(H):
                    kept = int(ref["kept_len"][b, h])
                    for r in range(kept):
                        page, slot = int(table[b, r // ps]), r % ps
                        if pool_layout == "heads-outer":
                            want[page, h, slot] = exp[b, h, r]
                        else:
                            want[page, slot, h] = exp[b, h, r]
            np.testing.assert_array_equal(got, want)


def test_paged_cache_argument_checks():
    w = _case()
    grp = wl.make_group(w, 0)
    prob = binding.Problem.from_workload(w)
    z = torch.zeros(64, dtype=torch.int32, device="cuda")
    t = [torch.zeros(8, dtype=torch.bfloat16, device="cuda")]
    with pytest.raises(binding.WkvError) as e:          # two pages of 24 rows cannot hold keep_max rows
        binding.wkv_gather_kv_paged(prob, t, None, z, [torch.zeros(8, dtype=torch.bfloat16, device="cuda")], None,
                                    z.view(2, 32)[:, :2].contiguous(), 24, 10, 24 * 128 * 2, 24 * 128, 128)
    assert e.value.status == 2


@pytest.mark.parametrize("pattern", ["shift", "tail"])
@pytest.mark.parametrize("case", [
    dict(batch=1, max_seqlen=9000, budget_frac=0.9),                       # eight blocks per unit, four batches
    dict(batch=1, n_q_heads=4, n_kv_heads=1, max_seqlen=257, budget_frac=0.5),   # fewer rows than eight blocks' threads
    dict(batch=9, max_seqlen=2500, n_layers=4, gamma=4, budget_frac=0.6),  # 144 (unit, tensor) pairs: one block each
], ids=["clusters-of-8", "few-rows", "no-cluster"])
def test_compaction_in_place_over_cluster_sizes(case, pattern):
    """A unit spread over a cluster of blocks: several batches in a row, fewer rows than threads, and one block."""
    test_compaction_in_place(case, pattern)


@pytest.mark.parametrize("pattern", ["selected", "shift", "tail", "front"])
@pytest.mark.parametrize("case", [
    # 40 (sequence, head) pairs x 4 tensors: one block each, so that few rows are already several batches
    dict(max_seqlen=16 + 8 * 400 + 3, budget_frac=0.45),                   # short last window, nearly half retained: long chains
    dict(max_seqlen=16 + 8 * 420 + 1, budget_frac=0.3),                    # last window of one token
    dict(l_obs=61, window=16, max_seqlen=3000, budget_frac=0.3),           # observation rows over four windows, not aligned
    dict(l_obs=64, window=8, max_seqlen=2500, budget_frac=0.3),            # ... over eight
    dict(window=7, max_seqlen=3200, budget_frac=0.2, l_obs=5),
    dict(window=200, max_seqlen=5000, budget_frac=0.3, n_planted=2),       # windows of several pieces
    dict(layout="bnhd", max_seqlen=3001, budget_frac=0.4, dtype="f32", head_dim=64, l_obs=8),
    dict(ragged=True, max_seqlen=4000, budget_frac=0.3),
], ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()))
def test_compaction_in_place_by_chains(case, pattern):
    """More rows than one batch and at most half of the windows retained: every chain of slots that read one another's
    windows, and the stretch that the observation rows overwrite, in all the ways they can meet."""
    test_compaction_in_place(dict(batch=20, n_q_heads=4, n_kv_heads=2) | case, pattern)


@pytest.mark.parametrize("pattern", ["shift", "tail"])
def test_compaction_in_place_of_rows_wider_than_a_block_moves_at_once(pattern):
    """Rows of 80 KB (the entry point takes up to 128 KB) in 136 (unit, tensor) pairs, which get one block each as far as
    occupancy goes: a block moves 64 KB at once."""
    test_compaction_in_place(dict(batch=34, n_layers=1, gamma=1, n_q_heads=2, n_kv_heads=2, head_dim=40960, max_seqlen=20,
                                  l_obs=2, window=3, top_p=2, budget_frac=0.8, n_planted=0), pattern)


@pytest.mark.parametrize("pattern", ["shift", "run", "tail"])
@pytest.mark.parametrize("case", [
    dict(batch=1, n_layers=1, gamma=1, window=16, l_obs=32, max_seqlen=20805, budget_frac=0.5),   # clusters of sixteen
    dict(batch=8, n_layers=4, gamma=4, max_seqlen=6001, budget_frac=0.2),       # two blocks per pair, several free stretches
    dict(batch=3, ragged=True, max_seqlen=4000, budgets=[3600, 300, 17]),       # a sequence that keeps nine tenths beside others
    dict(batch=20, head_dim=96, max_seqlen=3001, budget_frac=0.3),              # rows whose vectors do not divide a batch
    dict(batch=1, n_q_heads=4, n_kv_heads=1, head_dim=64, window=1, l_obs=3, top_p=1, max_seqlen=30000,
         budgets=[13000]),                                                      # a list longer than shared memory takes
], ids=["clusters-of-16", "two-blocks", "nine-tenths", "ragged-vectors", "long-list"])
def test_compaction_in_place_by_free_stretches(case, pattern):
    """Runs of retained windows with a spread rest behind them: batches that need a barrier, stretches that need none, and
    every change from one to the other."""
    test_compaction_in_place(dict(n_q_heads=4, n_kv_heads=2, n_planted=0) | case, pattern)


def test_compaction_time_depends_on_the_number_of_rows_only():
    """8 heads x 65,536 keys, 12 % retained: windows that all move by one place must not take longer than spread ones.
    What is measured differs by a fifth; the bound of three allows for a disturbed run."""
    H, n, omega, alpha, d = 8, 65536, 16, 32, 128
    prob = binding.Problem(dtype="bf16", batch=1, n_q_heads=32, n_kv_heads=H, head_dim=d, l_obs=alpha, window=omega, task=0,
                           top_p=8, max_seqlen=n, budgets=[n * 12 // 100])
    kw, k = prob.kw_max, prob.k_max
    rng = np.random.Generator(np.random.Philox(key=5))
    lists = {"spread": np.stack([np.sort(rng.permutation(kw)[:k]) for _ in range(H)]),
             "by one": np.tile(np.arange(1, k + 1), (H, 1)),
             "run": np.tile(np.concatenate([np.arange(3, 3 + k // 2), kw - np.arange(k - k // 2, 0, -1)]), (H, 1))}
    t = [torch.zeros((1, H, n, d), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    us = {}
    for name, rows in lists.items():
        idx = torch.from_numpy(rows[None].astype(np.int32)).cuda()
        samples = []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                binding.wkv_compact_kv_inplace(prob, t[:1], t[1:], idx)
            b.record()
            torch.cuda.synchronize()
            samples.append(a.elapsed_time(b))
        us[name] = sorted(samples)[len(samples) // 2]
    assert us["by one"] < 3 * us["spread"] and us["run"] < 3 * us["spread"], us


def test_a_list_that_misses_the_last_window_stays_inside_the_tensors():
    """Everything is to be kept, but the list holds no window (nothing has been selected into it yet): the observation rows
    keep their place, in the packed cache and inside the buffer, and nothing is written behind the sequence."""
    H, n, alpha, omega, d, guard = 2, 61, 7, 8, 64, 16                     # 54 review rows: seven windows, the last of six
    prob = binding.Problem(dtype="bf16", batch=1, n_q_heads=4, n_kv_heads=H, head_dim=d, l_obs=alpha, window=omega, task=0,
                           top_p=4, max_seqlen=n, budgets=[1000], cu_seqlens=[0, n])
    assert prob.k_max == prob.kw_max == 7
    idx = torch.full((1, H, 7), -1, dtype=torch.int32, device="cuda")
    k = torch.randn((n + guard, H, d), device="cuda").to(torch.bfloat16)
    before = k.clone()
    out = torch.full((n + guard, H, d), -3.0, dtype=torch.bfloat16, device="cuda")
    binding.wkv_gather_kv(prob, [k], None, idx, [out], None, cu_seqlens_out=torch.tensor([0, n], dtype=torch.int32, device="cuda"))
    binding.wkv_compact_kv_inplace(prob, [k], None, idx)
    torch.cuda.synchronize()
    assert torch.equal(k, before)
    assert torch.equal(out[n - alpha:n], before[n - alpha:n])
    assert bool((out[:n - alpha] == -3.0).all()) and bool((out[n:] == -3.0).all())


def test_a_refused_launch_is_reported_once():
    """More (sequence, head) pairs than a grid takes: the gather reports it, and the next call is none the worse."""
    prob = binding.Problem(dtype="bf16", batch=65536, n_q_heads=1, n_kv_heads=1, head_dim=8, l_obs=1, window=1, task=0, top_p=1,
                           max_seqlen=2, budgets=[2] * 65536)
    k = torch.zeros((65536, 1, 2, 8), dtype=torch.bfloat16, device="cuda")
    idx = torch.zeros((65536, 1, 1), dtype=torch.int32, device="cuda")
    with pytest.raises(binding.WkvError) as e:
        binding.wkv_gather_kv(prob, [k], None, idx, [torch.zeros_like(k)], None, keep_capacity=2)
    assert e.value.status == 8
    binding.wkv_probe_ex2_rate(torch.zeros(4, dtype=torch.float32, device="cuda"), 1, 32, 1)
    torch.cuda.synchronize()


@pytest.mark.parametrize("inplace", [False, True])
@pytest.mark.parametrize("layout", ["bhnd", "bnhd"])
def test_rows_that_the_kernel_in_front_writes(layout, inplace):
    """A gather or compaction fetches rows into L2 before the kernel in front has ended; what it then reads is what that
    kernel wrote.  Here a gather writes the keys that the next call takes rows from, at odd sizes and with a short last
    window, several times back to back."""
    B, H, n, d, alpha, omega, k = 2, 3, 4999, 128, 8, 16, 60
    rows = k * omega + alpha
    rng = np.random.default_rng(5)

    def problem(length, layout):
        return binding.Problem(dtype="bf16", batch=B, n_q_heads=H, n_kv_heads=H, head_dim=d, l_obs=alpha, window=omega, task=0,
                               top_p=omega, max_seqlen=length, budgets=[rows] * B, kv_layout=layout)

    first, second = problem(n, layout), problem(rows, "bhnd")
    assert first.k_max == k and second.k_max == k
    kw = -(-(n - alpha) // omega)
    idx = np.stack([np.stack([np.sort(rng.permutation(kw)[:k]) for _ in range(H)]) for _ in range(B)]).astype(np.int32)
    idx[0, 0, -1] = kw - 1                                 # the short last window
    again = np.tile(np.arange(k, dtype=np.int32), (B, H, 1))
    again[:, :, 7:] = -1                                   # of the compact rows: the first seven windows and the last rows
    shape = (B, H, n, d) if layout == "bhnd" else (B, n, H, d)
    idx_d, again_d = torch.from_numpy(idx).cuda(), torch.from_numpy(again).cuda()
    for seed in range(4):
        src = torch.randn(shape, dtype=torch.bfloat16, device="cuda", generator=torch.Generator("cuda").manual_seed(seed))
        mid = torch.zeros((B, H, rows, d), dtype=torch.bfloat16, device="cuda")
        out = torch.zeros_like(mid)
        binding.wkv_gather_kv(first, [src], [src], idx_d, [mid], [torch.empty_like(mid)], keep_capacity=rows)
        if inplace:
            binding.wkv_compact_kv_inplace(second, [mid], None, again_d)
        else:
            binding.wkv_gather_kv(second, [mid], [mid], again_d, [out], [torch.empty_like(out)], keep_capacity=rows)
        got = (mid if inplace else out).float().cpu()
        full = (src if layout == "bhnd" else src.transpose(1, 2)).float().cpu()
        for b in range(B):
            for h in range(H):
                taken = torch.cat([full[b, h, w * omega:min((w + 1) * omega, n - alpha)] for w in idx[b, h, :7]])
                assert torch.equal(got[b, h, :7 * omega], taken)


