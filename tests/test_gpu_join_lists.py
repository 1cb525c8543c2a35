"""The survivor lists of the bucket join where points repeat in them (a point met
through several tables is listed for each), against the oracle (match lists
entry for entry: every result is an integer, so the tolerance is zero), and
what such lists leave to the exact fallback."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_parity import ch, gpu_run, oparams, oracle_codes  # noqa: F401

pytestmark = pytest.mark.gpu


def clustered_set(seed, sizes, group):
    """Images of near copies of a few descriptors, `group` of each per image: a query shares most buckets with
    its group, so these candidates stand in its list once for every table."""
    rng = np.random.default_rng(seed)
    base = synth.sift_like(rng, (max(sizes) + group - 1) // group)
    imgs = [synth.noisy_copy(rng, np.repeat(base, group, axis=0)[:n], 2.0)[rng.permutation(n)] for n in sizes]
    n = len(sizes)
    pairs = np.array([(i, k) for i in range(n) for k in range(n)], np.uint32)
    return synth.ImageSet(np.concatenate(imgs), np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64), pairs,
                          synth.projection_matrix(seed))


@pytest.mark.parametrize("kernel", ["join", "join_tc"])
@pytest.mark.parametrize("group", [3, 7, 9])
@pytest.mark.parametrize("pk", [dict(n_tables=8, top_k=3), dict(n_tables=8, top_k=4), dict(n_tables=6, top_k=10),
                                dict(n_tables=8, bits_per_table=7, top_k=5), dict(n_tables=8, bits_per_table=4, top_k=11),
                                dict(n_tables=2, bits_per_table=1, top_k=32, tau=40), dict(n_tables=1, bits_per_table=5)])
def test_lists_with_repeats(ch, orc, pk, group, kernel):  # noqa: F811
    """Lists whose repeats exceed the two spare entries (with 8 bits they are read a second time, with fewer read
    by the dropping insertion at once), k below and at the instantiation's, fewer distinct points than k."""
    s = clustered_set(1200 + group, [200, 333, 64], group)
    tuning = (ch.CASHASH_KERNEL_JOIN if kernel == "join" else ch.CASHASH_KERNEL_JOIN_TC, 4 if kernel == "join" else 0, 0)
    ctx, ds, off, got, _ = gpu_run(ch, s, s.pairs, tuning=tuning, schedule=1, **pk)
    po = oparams(orc, pk)
    mu, codes, buckets = oracle_codes(orc, s.desc, s.R, po)
    eoff, emt = orc.match_pairs(s.desc, s.img_off, codes, buckets, s.pairs, po)
    assert np.array_equal(off, eoff)
    assert np.array_equal(got, emt)
    ctx.close()


@pytest.mark.parametrize("bits", [4, 8])
def test_repeats_stay_in_the_join(ch, bits):  # noqa: F811
    """Short codes, and 8 bits with images of near copies, where most listed points repeat: few queries may be left
    to the fallback, whose time (as much as the join's or more when repeats left queries to it, 7 % without) is held
    below a third of the join's."""
    s = synth.random_set(1300, [1000] * 12) if bits == 4 else clustered_set(1301, [1000] * 12, 2)
    pairs = np.array([(i, k) for i in range(12) for k in range(12) if i != k] * 3, np.uint32)
    p = ch.cashash_default_params(schedule=1, n_tables=8 if bits == 4 else 6, bits_per_table=bits, top_k=10)
    ctx = ch.cashash_create(p, s.R)
    ds = ch.DeviceSet(p, s.img_off, s.desc, s.kpts)
    ch.cashash_build_codes(ctx, ds)
    plan = ch.cashash_plan_create(ctx, ds, pairs)
    assert ch.cashash_plan_get_tuning(plan)["kernel"] == ch.CASHASH_KERNEL_JOIN
    cap = 1000 * len(pairs)
    moff = torch.zeros(len(pairs) + 1, dtype=torch.int64, device="cuda")
    mt = torch.zeros((cap, 2), dtype=torch.int32, device="cuda")
    ch.cashash_set_profiling(ctx, True)
    ratio = []
    for _ in range(8):
        ch.cashash_match_plan(ctx, plan, moff, mt, cap)
        assert ch.cashash_sync_status(ctx) == ch.CASHASH_OK
        ms = ch.cashash_get_stats(ctx)["ms_stage"]
        ratio.append(ms["fallback"] / ms["match"])
    plan.close()
    ctx.close()
    assert min(ratio[3:]) < 1.0 / 3.0
