"""The warp-per-query matching of the per-pair schedule at the edges of its
steps, against the oracle (match lists entry for entry: every result is an
integer, so the tolerance is zero)."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_parity import ch, gpu_run, oparams, oracle_codes  # noqa: F401

pytestmark = pytest.mark.gpu


def _compare(ch, orc, s, pairs, pk):  # noqa: F811
    ctx, ds, off, got, _ = gpu_run(ch, s, pairs, schedule=0, **pk)
    po = oparams(orc, pk)
    mu, codes, buckets = oracle_codes(orc, s.desc, s.R, po)
    eoff, emt = orc.match_pairs(s.desc, s.img_off, codes, buckets, pairs, po, F=s.F, kpts=s.kpts)
    assert np.array_equal(off, eoff)
    assert np.array_equal(got, emt)
    return ctx, ds, off, got


@pytest.mark.parametrize("pk", [dict(bits_per_table=0, n_tables=1, top_k=10), dict(bits_per_table=2, n_tables=8, top_k=32),
                                dict(bits_per_table=1, n_tables=3, top_k=2, tau=50), dict(top_k=4, code_bits=64),
                                dict(bits_per_table=4, n_tables=4, top_k=11, epi_px=40.0)])
def test_per_pair_candidate_steps(ch, orc, pk):  # noqa: F811
    """No candidate, one, fewer than k, one under and over a lane step (32) and a load step (128), many; pairs
    overlap in one chain of launches, which a graph capture repeats."""
    sizes = [0, 1, 2, 31, 33, 127, 129, 700]
    s = synth.random_set(616, sizes)
    n = len(sizes)
    pairs = np.array([(i, k) for i in range(n) for k in range(n)], np.uint32)
    if "epi_px" in pk:
        rng = np.random.default_rng(616)
        s.kpts = (rng.random((s.desc.shape[0], 2)) * 300.0).astype(np.float32)
        s.F = rng.standard_normal((len(pairs), 9)) * [1e-3, 1e-3, 1, 1e-3, 1e-3, 1, 1, 1, 1e2]
    ctx, ds, off, got = _compare(ch, orc, s, pairs, pk)
    plan = ch.cashash_plan_create(ctx, ds, pairs)
    cap = int(s.sizes()[pairs[:, 0]].sum())
    moff = torch.zeros(len(pairs) + 1, dtype=torch.int64, device="cuda")
    mt = torch.zeros((cap, 2), dtype=torch.int32, device="cuda")
    F = None if s.F is None else torch.from_numpy(np.ascontiguousarray(s.F)).cuda()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ch.cashash_match_plan(ctx, plan, moff, mt, cap, F=F, stream=torch.cuda.current_stream().cuda_stream)
    for _ in range(2):
        moff.zero_()
        g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(moff.cpu().numpy().astype(np.uint64), off)
    assert np.array_equal(mt[:int(off[-1])].cpu().numpy().view(np.uint32), got)
    plan.close()
    ctx.close()


def test_per_pair_largest_pairs(ch, orc):  # noqa: F811
    """Both sides of the rule that leaves pairs of many queries with long buckets to the thread-per-query kernel,
    one after the other in one call."""
    s = synth.random_set(617, [32768, 32769, 2100])
    pk = dict(bits_per_table=1, n_tables=2)  # 2,100 candidates per query
    ctx, *_ = _compare(ch, orc, s, np.array([[0, 2], [1, 2], [2, 2], [2, 1]], np.uint32), pk)
    ctx.close()


@pytest.mark.parametrize("flags", [0, 1])
def test_plans_of_a_few_pairs(ch, orc, flags):  # noqa: F811
    """One to four pairs around the rule that gives a few pairs a warp per query: kept plans under every kernel, and
    calls that make their plan for one match, on a stream of their own that nothing orders with the others."""
    sizes = [900, 0, 1, 2500]
    s = synth.random_set(618, sizes)
    pk = dict(schedule=1, flags=flags)
    p = ch.cashash_default_params(**pk)
    ctx = ch.cashash_create(p, s.R)
    ds = ch.DeviceSet(p, s.img_off, s.desc, s.kpts)
    ch.cashash_build_codes(ctx, ds)
    torch.cuda.synchronize()
    po = oparams(orc, pk)
    mu, codes, buckets = oracle_codes(orc, s.desc, s.R, po)
    side = torch.cuda.Stream()
    for pairs in ([[0, 3]], [[3, 0], [0, 1]], [[0, 3], [1, 1], [2, 3]], [[0, 3], [3, 0], [3, 3], [2, 0]]):
        pairs = np.array(pairs, np.uint32)
        eoff, emt = orc.match_pairs(s.desc, s.img_off, codes, buckets, pairs, po)
        cap = int(s.sizes()[pairs[:, 0]].sum())
        moff = torch.zeros(len(pairs) + 1, dtype=torch.int64, device="cuda")
        mt = torch.zeros((cap, 2), dtype=torch.int32, device="cuda")

        def check():
            assert ch.cashash_sync_status(ctx) == ch.CASHASH_OK
            off = moff.cpu().numpy().astype(np.uint64)
            assert np.array_equal(off, eoff)
            assert np.array_equal(mt[:int(off[-1])].cpu().numpy().view(np.uint32), emt)
            moff.zero_()
            mt.zero_()
            torch.cuda.synchronize()

        torch.cuda.synchronize()
        for _ in range(3):
            ch.cashash_match_pairs(ctx, ds, pairs, moff, mt, cap, stream=side.cuda_stream)
            check()
        plan = ch.cashash_plan_create(ctx, ds, pairs)
        few = len(pairs) * (1 + flags) <= 3
        assert ch.cashash_plan_get_tuning(plan)["kernel"] == (ch.CASHASH_KERNEL_WARP if few else ch.CASHASH_KERNEL_JOIN)
        for kernel in (0, ch.CASHASH_KERNEL_JOIN, ch.CASHASH_KERNEL_QUERY, ch.CASHASH_KERNEL_WARP, 0):
            if kernel:
                ch.cashash_plan_set_tuning(plan, kernel, 0, 0)
            ch.cashash_match_plan(ctx, plan, moff, mt, cap)
            check()
        plan.close()
    ctx.close()
