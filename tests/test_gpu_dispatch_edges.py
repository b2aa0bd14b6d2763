"""The sizes at which a kernel or a dispatch rule changes: selection lists around the number of keys a thread
holds, page scorer shapes, clusters of one to eight CTAs, work lists that share CTAs, device allocator sizes,
parameters outside the fp16 range and NaN in the bulk encoder, signed zeros in page boxes, latent batches around one wave of
CTAs, and caches that hand their page-locked block on between threads."""
import dataclasses
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


def _gqa(ctx, batch=1, n_kv=1, group=1, **kw):
    return W.Workload("edge", 60, 1, batch, n_kv * group, n_kv, 128, 128, ctx, ctx + 128, n_heavy=0, **kw)


# ---- page scores and selection ----------------------------------------------------------------------
@pytest.mark.parametrize("n_pages", [4, 64, 68, 4096, 4100, 16384, 16388, 32768, 32772])
def test_selection_around_the_lengths_that_change_its_kernel(n_pages):
    """One stream of n_pages 16-token pages whose keys are small integers, so that many scores are equal: scores against
    the sequential fp32 rule, selected pages against a stable sort, for one page, an eighth and all of them."""
    B = _binding()
    T = 16 * n_pages + 3
    w = _gqa(T, group=2, page_tokens=16, stair_tokens=(64, 0, 0, 0))
    g = B.Cache(B.config_from_workload(w))
    gen = torch.Generator(device=g.device)
    gen.manual_seed(n_pages)
    k = torch.randint(-2, 3, (1, T, 1, 128), generator=gen, device=g.device).to(torch.bfloat16)
    q = torch.randint(-1, 2, (1, 2, 128), generator=gen, device=g.device).to(torch.bfloat16)
    g.gkv_append_demote(0, k, k)
    score = g.gkv_debug_export_scores(0, q)[0, 0]
    pages = k[0, : 16 * n_pages, 0].float().reshape(n_pages, 16, 128)
    lo, hi, qf = pages.amin(1), pages.amax(1), q[0].float()
    acc = torch.zeros((2, n_pages), device=g.device)
    for d in range(128):
        acc = acc + qf[:, d: d + 1] * torch.where(qf[:, d: d + 1] >= 0, hi[:, d], lo[:, d])
    assert np.array_equal(score, torch.maximum(acc[0], acc[1]).cpu().numpy())
    order = np.argsort(-score, kind="stable")
    for n_sel in sorted({1, max(1, n_pages // 8), n_pages}):
        out = torch.full((1, 1, n_sel), -1, dtype=torch.int32, device=g.device)
        assert g.gkv_quest_select(0, q, 16 * n_sel, out) == n_sel
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy()[0, 0], np.sort(order[:n_sel])), n_sel


def test_box_of_signed_zeros_takes_the_sign_of_the_first():
    """Pages whose smallest or largest key is a zero of either sign: the box holds the page's first zero, bit for bit."""
    B = _binding()
    T = 640
    w = _gqa(T, page_tokens=16, stair_tokens=(-1, 0, 0, 0))
    g = B.Cache(B.config_from_workload(w))
    rs = np.random.RandomState(3)
    bits = np.where(rs.rand(T, 128) < 0.5, 0x0000, 0x8000).astype(np.uint16)
    bits[:, 32:64] = np.where(rs.rand(T, 32) < 0.3, 0x3f80, bits[:, 32:64])      # zeros and ones: the minimum is a zero
    bits[:, 64:96] = np.where(rs.rand(T, 32) < 0.3, 0xbf80, bits[:, 64:96])      # zeros and minus ones: the maximum is
    k = torch.from_numpy(bits.view(np.int16)).to(g.device).view(torch.bfloat16).reshape(1, T, 1, 128)
    g.gkv_append_demote(0, k, k)
    lo, hi = g.gkv_debug_export_boxes(0, 0, 0)
    val = (bits.astype(np.uint32) << 16).view(np.float32).reshape(T // 16, 16, 128)
    raw = bits.reshape(T // 16, 16, 128)
    first = lambda ext: np.take_along_axis(raw, np.argmax(val == ext[:, None], axis=1)[:, None], axis=1)[:, 0]   # noqa: E731
    assert np.array_equal(lo, first(val.min(1))) and np.array_equal(hi, first(val.max(1)))


# ---- work lists --------------------------------------------------------------------------------------
@pytest.mark.parametrize("batch,n_kv,group,T", [
    (1, 1, 1, 70), (1, 1, 8, 200), (1, 2, 4, 1000), (2, 1, 5, 2500), (2, 2, 4, 4100), (3, 6, 2, 1500), (5, 4, 6, 700),
    (37, 4, 1, 130), (38, 4, 1, 130), (1, 1, 4, 9000)])
def test_work_lists_from_one_cta_to_shared_ctas(batch, n_kv, group, T):
    """Random plans with centroid runs of every length: one CTA per head group, clusters of two to eight, more head groups
    than SMs, and streams that share CTAs; the read, and the observing read, which takes whole blocks only."""
    B = _binding()
    w = _gqa(T, batch, n_kv, group, policy=W.POLICY_EXTERNAL)
    data = W.make_layer(w, 0, "cpu")
    rs = np.random.RandomState(T + batch)
    plan = np.empty((batch, n_kv, T // 64), dtype=np.int8)
    for b in range(batch):
        for h in range(n_kv):
            i = 0
            while i < T // 64:
                n = int(rs.randint(1, 25))
                plan[b, h, i:i + n] = rs.choice(np.array([16, 8, 4, 2, 1, 1], dtype=np.int8))
                i += n
    ocache, g = O.GradedCache(U.oracle_config(w)), B.Cache(B.config_from_workload(w))
    U.ingest_both(w, 0, data, ocache, g, level_plan=plan)
    out, lse, o_out, o_lse = U.decode_both(ocache, g, 0, data["q"])
    U.assert_outputs_close(out, o_out, "read")
    assert np.max(np.abs(lse.cpu().numpy() - o_lse)) < 5e-3
    mass = torch.empty((batch, n_kv, -(-T // 64)), dtype=torch.float32, device=g.device)
    out2 = torch.empty_like(out)
    g.gkv_decode_attn_observe(0, data["q"].to(g.device), out2, None, mass)
    torch.cuda.synchronize()
    U.assert_outputs_close(out2, o_out, "observing read")
    assert np.allclose(mass.cpu().numpy().sum(-1), 1.0, atol=2e-3)
    again = torch.empty_like(out)
    g.gkv_decode_attn(0, data["q"].to(g.device), again)
    assert torch.equal(again, out2)              # the same lists until a block closes


@pytest.mark.parametrize("ctas", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("batch,group", [(2, 3), (3, 1), (2, 8)])
def test_clusters_of_every_size(ctas, batch, group):
    """Lists of half blocks for one warp each, so many that a head group gets a cluster of `ctas` CTAs, whose shares of the channels
    are even for two, four and eight only: the read and the observing read, and the same bits back to back."""
    B = _binding()
    blocks = 8 * ctas - 6                        # two units each, and four of the tail: half a CTA below ctas * 16
    w = _gqa(64 * blocks + 50, batch, 1, group, policy=W.POLICY_EXTERNAL)
    data = W.make_layer(w, 0, "cpu")
    ocache, g = O.GradedCache(U.oracle_config(w)), B.Cache(B.config_from_workload(w))
    plan = np.random.RandomState(ctas).choice(np.array([8, 4, 2], dtype=np.int8), size=(batch, 1, blocks))
    U.ingest_both(w, 0, data, ocache, g, level_plan=plan)
    out, lse, o_out, o_lse = U.decode_both(ocache, g, 0, data["q"])
    units = g.gkv_debug_export_units(0)
    first = [units[units[:, 1] == hg, 0].min() for hg in range(batch * (1 if group <= 4 else 2))]
    assert first == [16 * ctas * hg for hg in range(len(first))]        # a head group's warps begin with a cluster, 16 to a CTA
    U.assert_outputs_close(out, o_out, f"{ctas} CTAs")
    assert np.max(np.abs(lse.cpu().numpy() - o_lse)) < 5e-3
    q = data["q"].to(g.device)
    again = [torch.empty_like(out) for _ in range(20)]
    for o in again:
        g.gkv_decode_attn(0, q, o)
    assert all(torch.equal(o, out) for o in again)
    mass = torch.empty((batch, 1, blocks + 1), dtype=torch.float32, device=g.device)
    g.gkv_decode_attn_observe(0, q, out, None, mass)
    U.assert_outputs_close(out, o_out, "observing read")
    assert np.allclose(mass.cpu().numpy().sum(-1), 1.0, atol=2e-3)
    g.gkv_bits_report(0)                         # (raises if a wait ran out)


@pytest.mark.parametrize("streams", [15, 22, 25, 30, 40, 74, 75])
def test_page_lists_over_clusters_of_every_size(streams):
    """A page list is read by as many CTAs per head group as fill the GPU once, 148 / streams and at most eight, as a cluster where it has
    room for all."""
    B = _binding()
    T, n_sel = 64 * 9 + 5, 6
    w = _gqa(T, streams, 1, 2, page_tokens=64, stair_tokens=(128, 128, 128, 64))
    data = W.make_layer(w, 0, "cpu")
    ocache, g = O.GradedCache(U.oracle_config(w)), B.Cache(B.config_from_workload(w))
    U.ingest_both(w, 0, data, ocache, g)
    rs = np.random.RandomState(streams)
    pages = np.stack([np.sort(rs.permutation(9)[:n_sel]) for _ in range(streams)]).astype(np.int32)[:, None]
    out, lse, o_out, o_lse = U.decode_both(ocache, g, 0, data["q"], torch.from_numpy(pages).to(g.device), n_sel,
                                           [[pages[b, 0]] for b in range(streams)])
    U.assert_outputs_close(out, o_out, f"{streams} streams")
    assert np.max(np.abs(lse.cpu().numpy() - o_lse)) < 5e-3
    g.gkv_bits_report(0)


@pytest.mark.parametrize("batch,T", [(1, 65), (2, 333), (9, 300), (148, 70), (149, 70)])
def test_latent_batches_around_one_wave_of_ctas(batch, T):
    B = _binding()
    w = W.Workload("edge_latent", 61, 1, batch, 16, 1, 576, 512, T, T + 128, v_aliases_k=1, stair_tokens=(64, 64, 128, 0),
                   softmax_scale=1.0 / 192.0 ** 0.5, n_outlier=8, outlier_gain=6.0, n_heavy=0)
    data = W.make_layer(w, 0, "cpu")
    ocache, g = O.GradedCache(U.oracle_config(w)), B.Cache(B.config_from_workload(w))
    U.ingest_both(w, 0, data, ocache, g)
    for step in range(3):                        # the tail grows into new 16-row units
        out, lse, o_out, o_lse = U.decode_both(ocache, g, 0, data["q"])
        U.assert_outputs_close(out, o_out, f"latent batch {batch}, step {step}")
        assert np.max(np.abs(lse.cpu().numpy() - o_lse)) < 5e-3
        for i in range(11):
            tok = W.make_decode_tokens(w, 0, 100 * step + i, "cpu")
            ocache.append_demote(0, U.f32(tok["k"]), None)
            g.gkv_append_demote(0, tok["k"].to(g.device), None)


# ---- allocator and encoder ---------------------------------------------------------------------------
@pytest.mark.parametrize("n_closed", [1, 2, 3, 31, 33, 1023, 1025, 4095, 4097])
def test_ingest_plan_equals_host_allocator(n_closed):
    """The plan of a bulk ingest (made on the device up to 4095 blocks) against the host-only entry point on the same
    masses and ranges."""
    B = _binding()
    T = 64 * n_closed + 7
    w = _gqa(T, n_kv=2, policy=W.POLICY_RD, rd_budget_bpv=5.0, retire_after=128)
    g = B.Cache(B.config_from_workload(w))
    gen = torch.Generator(device=g.device)
    gen.manual_seed(n_closed)
    k = torch.randn((1, T, 2, 128), generator=gen, device=g.device).to(torch.bfloat16)
    mass = torch.softmax(3 * torch.randn((1, 2, T), generator=gen, device=g.device), -1)
    g.gkv_append_demote(0, k, k, token_mass=mass)
    _, ms, rg, _ = g.gkv_debug_device_plan(0)
    for h in range(2):
        want, _ = B.gkv_debug_plan_levels(g.cfg, n_closed, 7, ms[0, h], rg[0, h])
        assert np.array_equal(g.gkv_debug_export_levels(0, 0, h), want), h


@pytest.mark.parametrize("level", [8, 4, 2])
def test_bulk_encoder_with_parameters_outside_the_fp16_range(level):
    """Blocks whose scale or zero point saturates beside ordinary ones (the two go through different code): the stored
    state against the oracle, bit for bit."""
    B = _binding()
    T = 256
    w = _gqa(T, policy=W.POLICY_EXTERNAL)
    data = W.make_layer(w, 0, "cpu")
    for name, sign in (("k", 1.0), ("v", -1.0)):
        x = data[name].float()
        x[0, 3, 0, 5] = sign * 3e38              # a scale and, negative, a zero point beyond 65504
        x[0, 70, 0, 60:64] = -1e6
        x[0, 71, 0, 100] = 1e-30                 # a range that fp16 scales cannot express
        x[0, 130:194] = sign * 7e4               # constant blocks beyond the range
        data[name] = x.to(torch.bfloat16)
    ocache, g = O.GradedCache(U.oracle_config(w)), B.Cache(B.config_from_workload(w))
    with np.errstate(over="ignore", invalid="ignore"):
        U.ingest_both(w, 0, data, ocache, g, level_plan=np.full((1, 1, T // 64), level, dtype=np.int8))
    U.assert_state_equal(ocache, g, 0)


# ---- caches one after another -------------------------------------------------------------------------
def test_caches_of_two_threads_hand_on_their_host_blocks():
    """Two threads, each with a stream of its own, make, use and release caches of changing size; every read equals the
    one of the same cache made alone."""
    B = _binding()
    shapes = [(1, 200), (2, 1500), (1, 5000), (4, 300), (1, 200), (2, 1500)]

    def request(i, side):
        batch, T = shapes[i]
        w = dataclasses.replace(_gqa(T, batch, 2, 4, stair_tokens=(64, 128, 256, 512)), config_id=60 + side)
        data = W.make_layer(w, i, "cuda")
        cache = B.Cache(B.config_from_workload(w))
        out = torch.empty((batch, 8, 128), dtype=torch.float32, device=cache.device)
        cache.gkv_append_demote(0, data["k"], data["v"])
        for s in range(70):
            cache.gkv_append_demote(0, data["k"][:, s: s + 1].contiguous(), data["v"][:, s: s + 1].contiguous())
            cache.gkv_decode_attn(0, data["q"], out)
        torch.cuda.current_stream().synchronize()
        cache.close()
        return out.cpu()

    alone = {(i, side): request(i, side) for i in range(len(shapes)) for side in range(2)}
    got, errors = {}, []

    def work(side):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for i in range(len(shapes)):
                    got[(i, side)] = request(i, side)
        except Exception as e:      # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(side,)) for side in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for key, want in alone.items():
        assert torch.equal(got[key], want), key


@pytest.mark.parametrize("T", [2, 17, 64 + 16, 3 * 64 + 33, 9 * 64 + 63])
def test_latent_steps_of_one_to_four_units(T):
    """148 sequences, so that one CTA walks a whole sequence: random levels put one to four units of a kind into a step of the
    read kernel, switch between code and row operands, and end with a tail of one to four units."""
    B = _binding()
    w = W.Workload("edge_mla", 61, 1, 148, 16, 1, 576, 512, T, T + 64, v_aliases_k=1, n_outlier=8, outlier_gain=6.0, n_heavy=0,
                   softmax_scale=1.0 / 192 ** 0.5, policy=W.POLICY_EXTERNAL)
    oc = O.GradedCache(U.oracle_config(w))
    g = B.Cache(B.config_from_workload(w))
    data = W.make_layer(w, 0, "cpu")
    rs = np.random.RandomState(T)
    plan = rs.choice(np.array([16, 8, 8, 4, 4, 1], dtype=np.int8), size=(w.batch, 1, T // 64))
    U.ingest_both(w, 0, data, oc, g, level_plan=plan)
    out, lse, o_out, o_lse = U.decode_both(oc, g, 0, data["q"])
    U.assert_outputs_close(out, o_out, f"latent steps T {T}")
    assert np.max(np.abs(lse.cpu().numpy() - o_lse)) < 5e-3
    assert g.gkv_bits_report(0).resident_bits == oc.bits_report(0)["resident_bits"]
    g.close()


def _mixed_plan(w, seed, levels=(16, 8, 4, 2, 1)):
    rs = np.random.RandomState(seed)
    return rs.choice(np.array(levels, dtype=np.int8), size=(w.batch, w.n_kv_heads, w.ctx // 64))


@pytest.mark.parametrize("T", [2048 + 5, 33000, 66000, 140000])
def test_final_merge_of_a_few_to_many_rows(T):
    """One stream over the whole GPU: its partial rows are merged 32 at a time, in one pass or several."""
    B = _binding()
    w = _gqa(T, group=3, policy=W.POLICY_EXTERNAL)
    data = W.make_layer(w, 0, "cpu")
    ocache, g = O.GradedCache(U.oracle_config(w)), B.Cache(B.config_from_workload(w))
    U.ingest_both(w, 0, data, ocache, g, level_plan=_mixed_plan(w, T, (16, 8, 4, 4, 2)))
    out, lse, o_out, o_lse = U.decode_both(ocache, g, 0, data["q"])
    U.assert_outputs_close(out, o_out, f"T {T}")
    assert np.max(np.abs(lse.cpu().numpy() - o_lse)) < 5e-3
    again = torch.empty_like(out)
    g.gkv_decode_attn(0, data["q"].to(g.device), again)
    torch.cuda.synchronize()
    assert torch.equal(out, again)


@pytest.mark.parametrize("batch", [4, 5, 10, 18, 19])
def test_latent_batches_around_the_slices_of_the_merge(batch):
    """The merge of the CTAs' rows takes 64, 128, 256 or 512 channels to a block, by the number of sequences."""
    B = _binding()
    T = 64 * 9 + 33
    w = W.Workload("edge_latent", 61, 1, batch, 16, 1, 576, 512, T, T + 128, v_aliases_k=1, stair_tokens=(128, 128, 192, 0),
                   softmax_scale=1.0 / 192.0 ** 0.5, n_outlier=8, outlier_gain=6.0, n_heavy=0)
    data = W.make_layer(w, 0, "cpu")
    ocache, g = O.GradedCache(U.oracle_config(w)), B.Cache(B.config_from_workload(w))
    U.ingest_both(w, 0, data, ocache, g)
    out, lse, o_out, o_lse = U.decode_both(ocache, g, 0, data["q"])
    U.assert_outputs_close(out, o_out, f"latent batch {batch}")
    assert np.max(np.abs(lse.cpu().numpy() - o_lse)) < 5e-3


@pytest.mark.parametrize("spread", [1.0, 3e-5, 2e-6])
def test_bulk_encoder_with_and_without_codes_to_clamp(spread):
    """Groups whose scale is a subnormal fp16 number, rounded by up to a half, have values beyond the last code; the others do not
    and take the shorter arithmetic.  Every rung, stored bits against the oracle's."""
    B = _binding()
    T = 64 * 12
    w = _gqa(T, n_kv=2, policy=W.POLICY_EXTERNAL)
    data = W.make_layer(w, 0, "cpu")
    for name in ("k", "v"):
        data[name][:, T // 3:] *= spread           # (mixed: a warp takes one form or the other for all its groups)
    ocache, g = O.GradedCache(U.oracle_config(w)), B.Cache(B.config_from_workload(w))
    U.ingest_both(w, 0, data, ocache, g, level_plan=np.tile(np.array([8, 4, 2], dtype=np.int8), (1, 2, 4)))
    U.assert_state_equal(ocache, g, 0)


@pytest.mark.parametrize("level", [8, 4, 2])
@pytest.mark.parametrize("share", [1 / 4096, 0.02])
def test_bulk_encoder_keeps_a_nan_to_itself(level, share):
    """NaN among ordinary values (alone in a warp's tile, or many): the extremes pass over it and its code is 0.  Codes, scales and zero points
    against the same rows 4 bytes off, which go through the encoder of demotions; the codes of all numbers also against the
    quantiser's rule."""
    B = _binding()
    T = 64 * 6
    w = _gqa(T, n_kv=2, policy=W.POLICY_EXTERNAL)
    rs = np.random.RandomState(level)
    plan = np.full((1, 2, T // 64), level, dtype=np.int8)
    rows, caches = {}, []
    for name in ("k", "v"):
        x = rs.randn(T, 2, 128).astype(np.float32)
        x[rs.rand(*x.shape) < share] = np.nan
        x[5, 0, 2] = x[6, 1, 3] = x[69, 0, 5] = np.nan          # either half of a register
        x[:, :, 8] *= -1e4                                      # a neighbour far from the others
        x[128:160, 0, 40] = np.nan                              # a group of nothing else
        rows[name] = torch.from_numpy(x).to(torch.bfloat16).reshape(1, T, 2, 128)
    for shift in (0, 2):
        g = B.Cache(B.config_from_workload(w))
        args = []
        for name in ("k", "v"):
            flat = torch.zeros(T * 256 + 8, dtype=torch.bfloat16, device=g.device)
            flat[shift: shift + T * 256] = rows[name].to(g.device).reshape(-1)
            args.append(flat[shift: shift + T * 256].view(1, T, 2, 128))
        g.gkv_append_demote(0, *args, level_plan=plan)
        caches.append(g)
    for h in range(2):
        for blk in range(T // 64):
            for which, name in ((B.TENSOR_K, "k"), (B.TENSOR_V, "v")):
                got, want = (g.gkv_debug_export_block(0, 0, h, blk, which) for g in caches)
                for part in ("scale", "zero", "codes"):
                    assert np.array_equal(got[part], want[part]), (name, h, blk, part)
                s, z = (got[part].view(np.float16).astype(np.float32) for part in ("scale", "zero"))
                x = rows[name][0, 64 * blk: 64 * blk + 64, h].float().numpy()
                s, z = (np.repeat(p, 32, axis=0 if name == "k" else 1) for p in (s, z))
                with np.errstate(divide="ignore", invalid="ignore"):
                    code = np.clip(np.rint((x - z) * np.where(s > 0, np.float32(1) / s, np.float32(0))), 0, 2 ** level - 1)
                assert np.array_equal(got["codes"], np.where(np.isnan(x), 0, code)), (name, h, blk)
