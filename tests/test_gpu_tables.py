"""The lookup tables of sets whose images and chunks sort in one launch or in
two, through the matching that reads them (the per-query kernel the chunk
tables, the others the image tables), against the oracle, entry for entry."""
import numpy as np
import pytest

import synth
from test_gpu_parity import ch, gpu_run, oparams, oracle_codes  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pk", [dict(), dict(bits_per_table=0, n_tables=1), dict(bits_per_table=1, n_tables=8)])
@pytest.mark.parametrize("sizes", [[1, 0, 511, 512, 513], [3968, 3969, 31], [13653, 200], [13654, 200]])
def test_tables_of_one_and_two_launches(ch, orc, pk, sizes):  # noqa: F811
    """Fewer features than a CTA has threads or warps, a full chunk and one more, the line of the rule; one bucket
    for all features, two, and 256."""
    s = synth.random_set(919, sizes)
    n = len(sizes)
    pairs = np.array([(i, k) for i in range(n) for k in range(n) if min(sizes[i], sizes[k]) < 1000], np.uint32)
    pk = dict(schedule=1, **pk)
    po = oparams(orc, pk)
    mu, codes, buckets = oracle_codes(orc, s.desc, s.R, po)
    eoff, emt = orc.match_pairs(s.desc, s.img_off, codes, buckets, pairs, po)
    for kernel in (ch.CASHASH_KERNEL_WARP, ch.CASHASH_KERNEL_QUERY):
        ctx, ds, off, got, _ = gpu_run(ch, s, pairs, tuning=(kernel, 0, 0), **pk)
        assert np.array_equal(off, eoff)
        assert np.array_equal(got, emt)
        ctx.close()
