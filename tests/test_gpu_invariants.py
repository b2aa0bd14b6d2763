"""What has to hold whatever the timing, the order of the calls and the number of threads: plans that do not depend on when
a warp arrives, caches that do not disturb one another, state that a refused call leaves as it was, and work lists that hold
every item once and are balanced."""
import numpy as np
import pytest
import torch

from paper_2608_23599_b200 import workloads as W

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
