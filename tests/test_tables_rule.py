"""The rule that sorts image and chunk tables in one launch, at its line."""
import ctypes as C
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from test_gpu_parity import ch, gpu_run, oparams, oracle_codes  # noqa: E402,F401

LINE = 13640  # largest image whose tables sort together with the chunks'


def sort_smem(n):  # bytes: 16 warps' histograms, 16-bit index and bucket of each feature
    return 16 * 256 * 4 + (n + 7) // 8 * 8 * 3


def test_one_launch_while_four_ctas_fit():
    """Four CTAs of an SM's 228 KB, each with its dynamic and 32 static bytes (in steps of 128) and the system's KB."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_1805_08995_gb300 as ch
    rule = C.CDLL(os.path.abspath(ch.LIB_PATH))["_ZN3chx17tables_one_launchEj"]
    rule.argtypes, rule.restype = [C.c_uint32], C.c_bool
    four = [n for n in range(65536) if 4 * ((sort_smem(n) + 32 + 127) // 128 * 128 + 1024) <= 228 * 1024]
    assert max(four) == LINE
    assert rule(0) and rule(LINE) and not rule(LINE + 1) and not rule(65535)


def test_warps_per_cta():
    """Many CTAs of small images take 8 warps; few CTAs, and large images, 16."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_1805_08995_gb300 as ch
    rule = C.CDLL(os.path.abspath(ch.LIB_PATH))["_ZN3chx12tables_warpsEjmi"]
    rule.argtypes, rule.restype = [C.c_uint32, C.c_uint64, C.c_int], C.c_int
    assert [rule(n, t, 152) for n, t in ((64, 24000), (64, 153), (64, 152), (4096, 1200), (4097, 1200), (1, 0))] == \
        [8, 8, 16, 8, 16, 16]


@pytest.mark.gpu
@pytest.mark.parametrize("pk", [dict(), dict(bits_per_table=0, n_tables=1), dict(bits_per_table=1, n_tables=8)])
@pytest.mark.parametrize("top", [4096, 4097])
def test_tables_of_many_small_images(ch, orc, pk, top):  # noqa: F811
    """Both numbers of warps on images around a warp's and a CTA's threads, empty ones among them, and one of two
    chunks, through the warp kernel (image tables) and the per-query kernel (chunk tables), against the oracle."""
    sizes = [0, 1, 31, 33, 255, 256, 257, 300, 513] * 22 + [top]
    s = synth.random_set(921, sizes)
    n = len(sizes)
    pairs = np.array([(i, (7 * i + 3) % n) for i in range(0, n, 3)] + [(n - 1, 8), (8, n - 1)], np.uint32)
    po = oparams(orc, pk)
    mu, codes, buckets = oracle_codes(orc, s.desc, s.R, po)
    eoff, emt = orc.match_pairs(s.desc, s.img_off, codes, buckets, pairs, po)
    for kernel in (ch.CASHASH_KERNEL_WARP, ch.CASHASH_KERNEL_QUERY, ch.CASHASH_KERNEL_JOIN):
        ctx, ds, off, got, _ = gpu_run(ch, s, pairs, tuning=(kernel, 0, 0), schedule=1, **pk)
        assert np.array_equal(off, eoff) and np.array_equal(got, emt)
        ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("pk", [dict(), dict(bits_per_table=1, n_tables=8)])
@pytest.mark.parametrize("n", [LINE, LINE + 1])
def test_tables_at_the_line(ch, orc, pk, n):  # noqa: F811
    """The image tables through the warp kernel, the chunk tables through the per-query kernel, against the oracle."""
    s = synth.random_set(920, [n, 200])
    pairs = np.array([[0, 1], [1, 0], [1, 1]], np.uint32)
    po = oparams(orc, pk)
    mu, codes, buckets = oracle_codes(orc, s.desc, s.R, po)
    eoff, emt = orc.match_pairs(s.desc, s.img_off, codes, buckets, pairs, po)
    for kernel in (ch.CASHASH_KERNEL_WARP, ch.CASHASH_KERNEL_QUERY):
        ctx, ds, off, got, _ = gpu_run(ch, s, pairs, tuning=(kernel, 0, 0), schedule=1, **pk)
        assert (off == eoff).all() and got.shape == emt.shape and (got == emt).all()
        ctx.close()
