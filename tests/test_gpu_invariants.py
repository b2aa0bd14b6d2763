"""What has to hold whatever the timing, the order of the calls and the number of threads: plans that do not depend on when
a warp arrives, caches that do not disturb one another, state that a refused call leaves as it was, and work lists that hold
every item once and are balanced."""
import heapq
import threading

import numpy as np
import pytest
import torch

from oracle import gkv_oracle as O
from paper_2608_23599_b200 import workloads as W
import parity_util as U

pytestmark = pytest.mark.gpu


def _binding():
    from paper_2608_23599_b200 import binding as B
    return B


def _gqa(ctx, batch=1, n_kv=1, group=1, room=128, **kw):
    return W.Workload("invariant", 70, 1, batch, n_kv * group, n_kv, 128, 128, ctx, ctx + room, n_heavy=0, **kw)


# ---- allocator -----------------------------------------------------------------------------------------
@pytest.mark.parametrize("n_closed,monotone", [(65, 1), (65, 0), (700, 1), (700, 0), (2100, 1)])
def test_device_plans_do_not_depend_on_timing(n_closed, monotone):
    """Two CTAs' worth of streams per SM (up to 1024 threads each) make their plans again and again: every plan equals the
    first, and the streams' plans equal the host allocator's."""
    B = _binding()
    batch, n_kv = (37, 8) if n_closed < 1000 else (5, 8)
    T = 64 * n_closed + 9
    w = _gqa(T, batch, n_kv, policy=W.POLICY_RD, rd_budget_bpv=4.0, retire_after=64)
    cfg = B.config_from_workload(w)
    cfg.monotone_in_age = monotone
    g = B.Cache(cfg)
    gen = torch.Generator(device=g.device)
    gen.manual_seed(n_closed)
    k = torch.randn((1, T, n_kv, 128), generator=gen, device=g.device).to(torch.bfloat16).expand(batch, -1, -1, -1).contiguous()
    mass = torch.softmax(3 * torch.randn((batch, n_kv, T), generator=gen, device=g.device), -1)
    g.gkv_append_demote(0, k, k, token_mass=mass)
    first, ms, rg, miss = g.gkv_debug_device_plan(0)
    for _ in range(30):
        again, _, _, miss2 = g.gkv_debug_device_plan(0)
        assert np.array_equal(first, again) and miss == miss2
    for b, h in ((0, 0), (batch - 1, n_kv - 1), (batch // 2, 3)):
        prev = g.gkv_debug_export_levels(0, b, h).astype(np.int8)
        want, _ = B.gkv_debug_replan_levels(g.cfg, 9, ms[b, h], rg[b, h], prev)
        assert np.array_equal(first[b, h], want), (b, h)


# ---- threads ---------------------------------------------------------------------------------------------
def _in_two_threads(work):
    """work(side, meet) for side 0 and 1, each in a thread with a stream of its own; meet() lets the two go on together."""
    errors, barrier = [], threading.Barrier(2, timeout=60)

    def body(side):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                work(side, barrier.wait)
                torch.cuda.current_stream().synchronize()
        except Exception as e:      # noqa: BLE001
            errors.append((side, e))
            barrier.abort()

    threads = [threading.Thread(target=body, args=(side,)) for side in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_lists_of_two_long_contexts_made_by_two_threads():
    """Contexts whose work lists need more shared memory than a kernel has without asking, a different amount each: the
    lists are remade again and again (a block closes), and every read equals the one of a cache worked on alone."""
    B = _binding()
    sizes, rounds = (140_000, 300_000), 40

    def decode(side, outs, meet=lambda: None):
        w = _gqa(sizes[side], room=64 * (rounds + 1), stair_tokens=(64, 64, 64, -1))
        gen = torch.Generator(device="cuda")
        gen.manual_seed(side)
        k = torch.randn((1, w.ctx, 1, 128), generator=gen, device="cuda").to(torch.bfloat16)
        q = torch.randn((1, 1, 128), generator=gen, device="cuda").to(torch.bfloat16)
        cache = B.Cache(B.config_from_workload(w))
        cache.gkv_append_demote(0, k, k)
        row = k[:, :1].contiguous()
        for r in range(rounds):
            for _ in range(64):
                cache.gkv_append_demote(0, row, row)
            out = torch.empty((1, 1, 128), dtype=torch.float32, device="cuda")
            meet()
            cache.gkv_decode_attn(0, q, out)
            outs[side].append(out)
        torch.cuda.current_stream().synchronize()
        cache.close()

    alone, both = ([], []), ([], [])
    for side in range(2):
        decode(side, alone)
    _in_two_threads(lambda side, meet: decode(side, both, meet))
    for side in range(2):
        assert len(both[side]) == rounds
        for r in range(rounds):
            assert torch.equal(alone[side][r], both[side][r]), (side, r)


def test_plans_of_two_sizes_made_by_two_threads():
    """Allocations whose breakpoints need more shared memory than a kernel has without asking, a different amount each."""
    B = _binding()
    sizes = (1700, 4095)

    def plans(side, out, meet=lambda: None):
        w = _gqa(64 * sizes[side] + 5, policy=W.POLICY_RD, rd_budget_bpv=4.0, retire_after=64)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(side)
        k = torch.randn((1, w.ctx, 1, 128), generator=gen, device="cuda").to(torch.bfloat16)
        mass = torch.softmax(3 * torch.randn((1, 1, w.ctx), generator=gen, device="cuda"), -1)
        cache = B.Cache(B.config_from_workload(w))
        cache.gkv_append_demote(0, k, k, token_mass=mass)
        out[side] = []
        for _ in range(40):
            meet()
            out[side].append(cache.gkv_debug_device_plan(0)[0])
        cache.close()

    alone, both = [None, None], [None, None]
    for side in range(2):
        plans(side, alone)
    _in_two_threads(lambda side, meet: plans(side, both, meet))
    for side in range(2):
        assert all(np.array_equal(p, alone[side][0]) for p in both[side])


# ---- a refused ingest ---------------------------------------------------------------------------------------
def _smallest_arena(B, cfg):
    """Fewest bytes that a cache of this configuration is made in: its metadata and one exact block."""
    lo, hi = 4096, B.gkv_query_arena_bytes(cfg)
    while hi - lo > 256:
        mid = (lo + hi) // 2
        try:
            B.Cache(cfg, arena_bytes=mid).close()
            hi = mid
        except B.GkvError:
            lo = mid
    return hi


@pytest.mark.parametrize("policy", ["rd", "staircase", "latent"])
def test_refused_ingest_leaves_the_layer_empty(policy):
    """A prompt that the arena has no room for, first; then the same calls as on a cache that never saw it: single tokens
    (an observing read and, where there are pages, a read by list: both look at residual rows), or a prompt that fits."""
    B = _binding()
    latent = policy == "latent"
    if latent:
        w = W.Workload("refused", 71, 1, 2, 16, 1, 576, 512, 2000, 2200, v_aliases_k=1, stair_tokens=(64, 64, -1, 0), n_heavy=0,
                       softmax_scale=0.07)
    else:
        w = _gqa(2000, 2, 2, 4, room=200, page_tokens=64, residual_fraction=0.1,
                 **(dict(policy=W.POLICY_RD, rd_budget_bpv=5.0, retire_after=64) if policy == "rd" else dict(stair_tokens=(64, 64, 64, -1))))
    cfg = B.config_from_workload(w)
    small = _smallest_arena(B, cfg) + (14 * 73728 if latent else 20 * 32768)
    assert small < B.gkv_query_arena_bytes(cfg)
    data = W.make_layer(w, 0, "cuda")
    mass = None if latent else torch.softmax(3 * torch.randn((2, 2, 2000), device="cuda"), -1)

    def ingest(cache, n):
        return cache.gkv_append_demote(0, data["k"][:, :n].contiguous(), None if latent else data["v"][:, :n].contiguous(),
                                       token_mass=None if latent else mass[:, :, :n].contiguous())

    def reads(cache, first, n):
        got = []
        for t in range(first, first + n):
            cache.gkv_append_demote(0, data["k"][:, t:t + 1].contiguous(), None if latent else data["v"][:, t:t + 1].contiguous())
            out = torch.empty((2, w.n_q_heads, w.d_v), device="cuda")
            cache.gkv_decode_attn(0, data["q"], out)
            got.append(out)
            if latent or t % 9:
                continue
            out, m = torch.empty_like(out), torch.empty((2, 2, -(-(t + 1) // 64)), device="cuda")
            cache.gkv_decode_attn_observe(0, data["q"], out, None, m)
            got += [out, m, torch.from_numpy(cache.gkv_debug_export_mass(0))]
            n_pages = (t + 1) // 64
            pages = torch.arange(n_pages, dtype=torch.int32, device="cuda").expand(2, 2, -1).contiguous()
            out = torch.empty_like(out)
            cache.gkv_decode_attn(0, data["q"], out, page_idx=pages, n_sel=n_pages)
            got.append(out)
        torch.cuda.synchronize()
        bits = cache.gkv_bits_report(0)
        return got, (bits.values, bits.resident_bits, bits.residual_bits, cache.last_report_status)

    fits = 300
    for calls in (lambda c: reads(c, 0, 150), lambda c: (ingest(c, fits), reads(c, fits, 40))[1]):
        fresh, used = B.Cache(cfg), B.Cache(cfg, arena_bytes=small)
        for _ in range(2):                         # (what the first refusal took has come back)
            with pytest.raises(B.GkvError) as e:
                ingest(used, 2000)
            assert e.value.status == B.ERR_ARENA_TOO_SMALL
        assert used.gkv_ctx_len(0) == 0
        (a, bits_a), (b, bits_b) = calls(fresh), calls(used)
        assert bits_a == bits_b
        for i, (x, y) in enumerate(zip(a, b)):
            assert torch.equal(x, y), i


# ---- precision of the latent read -----------------------------------------------------------------------------
@pytest.mark.parametrize("seed", [0, 1])
@pytest.mark.parametrize("stair,bound", [((0, 0, -1, 0), 4.4e-5), ((0, -1, 0, 0), 4.6e-6)])
def test_latent_read_loses_no_bit_to_the_largest_probability(stair, bound, seed):
    """Contexts of one rung that give every group of warps two half blocks, one of them its first.  The value MMAs add 16
    products and cut the sum off at a fixed distance below the exponent of the largest one: with a probability of exactly 1
    in a unit that is one bit higher than with all of them below 1.  Relative error, 4 and 8 bits: 6.5e-5 - 6.8e-5 and
    5.9e-6 - 6.3e-6 with the 1, half as much of that bit without (3.1e-5 - 3.3e-5 and 3.4e-6 - 3.6e-6); the bounds lie a
    third above the latter."""
    B = _binding()
    w = W.Workload("latent_error", 72 + seed, 1, 2, 16, 1, 576, 512, 9472, 9600, v_aliases_k=1, stair_tokens=stair, n_heavy=0,
                   softmax_scale=1.0 / 192.0 ** 0.5, n_outlier=8, outlier_gain=6.0)
    data = W.make_layer(w, 0, "cpu")
    ocache, g = O.GradedCache(U.oracle_config(w)), B.Cache(B.config_from_workload(w))
    U.ingest_both(w, 0, data, ocache, g)
    out, _, want, _ = U.decode_both(ocache, g, 0, data["q"])
    rel = np.linalg.norm(out.double().cpu().numpy() - want) / np.linalg.norm(want)
    assert rel <= bound, rel


# ---- work lists -------------------------------------------------------------------------------------------------
def _mixed_plan(rs, shape, n, levels=(16, 8, 4, 2, 1, 1)):
    """Runs of 1 to 24 blocks of one rung, rungs at random."""
    plan = np.empty(shape + (n,), dtype=np.int8)
    for at in np.ndindex(shape):
        i = 0
        while i < n:
            m = int(rs.randint(1, 25))
            plan[at][i:i + m] = rs.choice(np.array(levels, dtype=np.int8))
            i += m
    return plan


def _check_lists(rows, levels, n_res, head_groups):
    """Every tile of every closed block, the partial block and every residual group once per head group; whole runs of
    centroid blocks; and no warp with more than 1.02 times what the fullest one has when the units are dealt one by one,
    longest first, to the least laden warp."""
    n = levels.shape[1]
    for hg in range(levels.shape[0] * head_groups):
        mine = rows[rows[:, 1] == hg]
        lv = levels[hg // head_groups]
        groups = -(-int(n_res[hg // head_groups]) // 16)
        tiles = np.zeros(n + 1 + groups, dtype=np.int64)
        for t in range(4):
            one = mine[(mine[:, 3] >> t & 1 == 1) & (mine[:, 4] == 1)]
            np.add.at(tiles, one[:, 2], 1 << (4 * t))
        for _, _, item, mask, run, _ in mine[mine[:, 4] > 1]:
            assert mask == 15 and np.all(lv[item:item + run] == 1) and item // 16 == (item + run - 1) // 16
            tiles[item:item + run] += 0x1111
        assert np.all(tiles == 0x1111), (hg, np.nonzero(tiles != 0x1111)[0][:8])
        warps = np.unique(mine[:, 0])
        load = np.zeros(int(mine[:, 0].max()) + 1, dtype=np.int64)
        np.add.at(load, mine[:, 0], mine[:, 5])
        heap = [0] * len(warps)
        for cost in np.sort(mine[:, 5])[::-1]:
            heapq.heapreplace(heap, heap[0] + int(cost))
        assert load.max() <= 1.02 * max(heap), (hg, int(load.max()), max(heap))


@pytest.mark.parametrize("batch,n_kv,group,T,residual,fixed", [
    (1, 1, 1, 70, 0.0, None), (2, 2, 8, 13_100, 0.0, None), (2, 1, 8, 27_300, 0.0, None), (4, 1, 8, 16_750, 0.0, None),
    (1, 2, 8, 16_384, 0.01, None), (4, 8, 4, 32_763, 0.10, "newest"), (8, 8, 4, 16_384, 0.10, "newest"), (2, 1, 4, 6000, 0.05, "newest"),
    (2, 1, 5, 3000, 0.05, "newest"), (3, 2, 3, 2500, 0.03, None), (3, 8, 4, 16_400, 0.0, "4 bits"),
    (12, 8, 4, 4000, 0.0, "4 bits"), (6, 4, 8, 16_400, 0.0, "4 bits"), (1, 1, 4, 140_000, 0.02, None)])
def test_work_lists_are_complete_and_balanced(batch, n_kv, group, T, residual, fixed):
    B = _binding()
    w = _gqa(T, batch, n_kv, group, policy=W.POLICY_EXTERNAL, residual_fraction=residual)
    rs = np.random.RandomState(T)
    plan = _mixed_plan(rs, (batch, n_kv), T // 64)
    if fixed == "4 bits":                           # equal streams, whose warps round up to more than a wave of CTAs
        plan[:] = 4
    elif fixed:                                     # 256 exact tokens, centroids, exact residual rows
        plan[:] = 1
        plan[..., -4:] = 16
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T)
    k = torch.randn((batch, T, n_kv, 128), generator=gen, device="cuda").to(torch.bfloat16)
    mass = torch.softmax(torch.randn((batch, n_kv, T), generator=gen, device="cuda"), -1) if residual else None
    g = B.Cache(B.config_from_workload(w))
    g.gkv_append_demote(0, k, k, token_mass=mass, level_plan=plan)
    q = torch.randn((batch, n_kv * group, 128), generator=gen, device="cuda").to(torch.bfloat16)
    out = torch.empty((batch, n_kv * group, 128), device="cuda")
    with pytest.raises(B.GkvError):
        g.gkv_debug_export_units(0)                  # none made yet
    n_res = [len(g.gkv_debug_export_residual(0, b, h)) for b in range(batch) for h in range(n_kv)]
    levels = plan.reshape(batch * n_kv, -1).astype(np.int64)
    for observe in (False, True):                    # parts of blocks in small workloads; whole blocks
        if observe:
            m = torch.empty((batch, n_kv, -(-T // 64)), device="cuda")
            g.gkv_decode_attn_observe(0, q, out, None, m)
            assert torch.allclose(m.sum(-1), torch.ones((), device="cuda"), atol=2e-3)      # residual rows in their blocks
        else:
            g.gkv_decode_attn(0, q, out)
        rows = g.gkv_debug_export_units(0)
        _check_lists(rows, levels, n_res, -(-group // 4))
        assert rows[:, 0].max() < 148 * 16           # one wave of CTAs


@pytest.mark.parametrize("levels", [(16,), (16, 8, 4, 2)])
@pytest.mark.parametrize("n_closed", [3125, 45_200])
def test_long_context_lists(n_closed, levels):
    """One stream whose work list needs more shared memory than a kernel has without asking, and one that is longer than the
    units whose warps are kept in shared memory (it is dealt without a look at what a warp has): every block once, and, of
    exact blocks, the read against the one by page list, which has no work lists.  Both sum exact products in fp32: 1e-4 of
    the output is ten times what they differ by, and a block left out or read twice changes it by 1 / sqrt(blocks) = 5e-3."""
    B = _binding()
    T = 64 * n_closed + 33
    w = _gqa(T, room=64, page_tokens=64, policy=W.POLICY_EXTERNAL)
    plan = _mixed_plan(np.random.RandomState(n_closed), (1, 1), n_closed, levels)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n_closed)
    k = torch.randn((1, T, 1, 128), generator=gen, device="cuda", dtype=torch.bfloat16)
    q = (0.25 * torch.randn((1, 1, 128), generator=gen, device="cuda")).to(torch.bfloat16)
    g = B.Cache(B.config_from_workload(w))
    g.gkv_append_demote(0, k, k, level_plan=plan)
    del k
    out, listed = torch.empty((1, 1, 128), device="cuda"), torch.empty((1, 1, 128), device="cuda")
    g.gkv_decode_attn(0, q, out)
    rows = g.gkv_debug_export_units(0)
    assert np.array_equal(np.sort(rows[:, 2]), np.arange(n_closed + 1)) and np.all(rows[:, 3] == 15)
    assert 147 * 16 < len(np.unique(rows[:, 0])) <= 148 * 16      # about one wave of warps
    if levels == (16,):
        pages = torch.arange(n_closed, dtype=torch.int32, device="cuda").reshape(1, 1, -1)
        g.gkv_decode_attn(0, q, listed, page_idx=pages, n_sel=n_closed)
        torch.cuda.synchronize()
        assert float((out - listed).norm() / listed.norm()) < 1e-4


# ---- the finish of an observing read ---------------------------------------------------------------------------
@pytest.mark.parametrize("n_kv,n_res", [(9, 500), (9, 501), (10, 500), (11, 455)])
def test_observing_read_of_a_full_gpu_with_residual_rows(n_kv, n_res):
    """On both sides of the lines (500 rows of a stream, 5000 in all) beyond which the finish waits for the read's end: calls
    one behind another, without a wait between them, give the same bits as one alone, and every stream's masses add up
    to 1 (fp32 sums of 158 positive masses of relative error 1e-3 at most: 2e-3)."""
    B = _binding()
    T = 10_033
    w = _gqa(T, 1, n_kv, 4, policy=W.POLICY_STAIRCASE, stair_tokens=(64, 0, -1, 0), residual_fraction=(n_res + 0.5) / T)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n_res)
    k = torch.randn((1, T, n_kv, 128), generator=gen, device="cuda").to(torch.bfloat16)
    mass = torch.softmax(torch.randn((1, n_kv, T), generator=gen, device="cuda"), -1)
    g = B.Cache(B.config_from_workload(w))
    g.gkv_append_demote(0, k, k, token_mass=mass)
    q = torch.randn((1, n_kv * 4, 128), generator=gen, device="cuda").to(torch.bfloat16)
    out = torch.empty((1, n_kv * 4, 128), device="cuda")
    m = [torch.full((1, n_kv, -(-T // 64)), -1.0, device="cuda") for _ in range(5)]
    c = [torch.full((1, n_kv * 4), -1.0, device="cuda") for _ in range(5)]
    for i in range(5):
        g.gkv_decode_attn_observe(0, q, out, None, m[i], c[i])
        if i == 0:
            torch.cuda.synchronize()
    assert [len(g.gkv_debug_export_residual(0, 0, h)) for h in range(n_kv)] == [n_res] * n_kv
    assert g.gkv_debug_export_units(0)[:, 0].max() >= 65 * 16
    assert torch.allclose(m[0].sum(-1), torch.ones((), device="cuda"), atol=2e-3) and float(m[0].min()) >= 0.0
    assert all(torch.equal(m[0], x) for x in m[1:]) and all(torch.equal(c[0], x) for x in c[1:]) and float(c[0].min()) > 0.0


# ---- page-locked host memory -----------------------------------------------------------------------------------
def _centroid_cache(B, layers, batch, ctx):
    return B.Cache(B.make_config(layers, batch, 32, 8, 128, 128, ctx, stair_tokens=(0, 0, 0, 0)))


def test_host_memory_of_a_large_cache_is_kept_and_given_back():
    """The block tables of 32 layers x 64 streams x 131,072 tokens (67 MB): kept after the cache is gone, given back on
    request or when eight caches of another size have come and gone; a cache in use keeps its own."""
    B = _binding()
    table = 32 * 64 * (131_072 // 64) * 16
    B.gkv_release_host_memory()
    _centroid_cache(B, 32, 8, 131_072).close()
    assert table <= B.gkv_release_host_memory() < 1.25 * table
    assert B.gkv_release_host_memory() == 0
    live = _centroid_cache(B, 2, 1, 1024)
    assert B.gkv_release_host_memory() == 0
    k = torch.randn((1, 130, 8, 128), device="cuda").to(torch.bfloat16)
    out = torch.empty((1, 32, 128), device="cuda")
    live.gkv_append_demote(0, k, k)
    live.gkv_decode_attn(0, torch.zeros((1, 32, 128), dtype=torch.bfloat16, device="cuda"), out)
    torch.cuda.synchronize()
    want = k.float().mean(1).repeat_interleave(4, 1)      # equal weights; two centroids of 64 tokens (bf16) and two tokens
    assert torch.allclose(out, want, atol=2.0 ** -9)
    live.close()
    _centroid_cache(B, 32, 8, 131_072).close()
    for _ in range(9):
        _centroid_cache(B, 2, 1, 1024).close()
    assert B.gkv_release_host_memory() < table


def test_host_memory_that_is_kept_is_bounded():
    B = _binding()
    B.gkv_release_host_memory()
    caches = [_centroid_cache(B, 32, b, 131_072) for b in (2, 3, 5, 8, 12, 16)]      # 18 to 140 MB each
    for c in caches:
        c.close()
    assert B.gkv_release_host_memory() <= 320 << 20


def test_host_memory_is_given_back_while_other_threads_make_caches():
    B = _binding()

    def work(side, meet):
        meet()
        for i in range(40):
            _centroid_cache(B, 2, 1 + (i + side) % 3, 2048).close()
            if i % 4 == side:
                B.gkv_release_host_memory()

    _in_two_threads(work)
    assert B.gkv_release_host_memory() <= 4 << 20
    assert B.gkv_release_host_memory() == 0
