"""The rounding bound of the projection: its factor against a derivation in exact arithmetic, and rows of R
whose small terms are as large as the split allows, against doubles."""
import os
import re
from fractions import Fraction as Q

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")

from test_gpu_parity import ch, oparams, oracle_codes  # noqa: E402,F401

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1805_08995_gb300", "csrc")


def test_bound_factor_covers_a_truncating_adder():
    """alpha, in units of max(2^s ||R_b||, 256) ||x||, for the three-term split: 16 MMAs of 16 products each into the
    second accumulator, in each of which the 16 products and the accumulator are aligned to the largest of them and
    cut off below its 24th bit, and so is their sum; all partial sums are at most S = sum x (|mid| + |lo|)."""
    src = open(os.path.join(CSRC, "codes.cu")).read()
    m = re.search(r"r\.alpha = \(float\)\(0x1p-(\d+) \* fmax\(nr, 256\.0\)", src)
    alpha = Q(1, 2 ** int(m.group(1)))
    root128 = Q(11314, 1000)                      # sqrt(128) rounded up; sum x <= sqrt(128) ||x||
    S = (1024 + Q(1, 2)) * root128                # |mid| <= 1024, |lo| <= 1/2
    cut = 16 * (16 + 1 + 1) * Q(1, 2 ** 23) * S / 2 ** 11 / 256
    split = Q(1, 2 ** 23) * root128 / 256         # what the three terms leave of R
    add = Q(1, 2 ** 24) * (1 + 2 * cut + split)   # A + 2^-11 B rounded
    sub = Q(1, 2 ** 24) * (1 + 2 * cut + split)   # minus c rounded (the share of |c| is in beta)
    assert split + cut + add + sub < alpha
    # the first accumulator is exact: integers below 2^24
    assert 128 * 255 * 512 < 2 ** 24


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
def test_rows_of_one_large_entry_and_half_steps(ch, orc, precision):  # noqa: F811
    """Rows scaled to one entry of 256 and the rest close to half a step of the first term, of one sign, of
    alternating signs, and at larger whole numbers; full and random descriptors.  Bits equal the oracle's, and the
    approximation stays inside its bound."""
    s = synth.random_set(1515, [900, 1100])
    rng = np.random.default_rng(1515)
    s.desc[:100] = 255
    s.desc[100:200] = rng.integers(0, 2, (100, 128)) * 255
    s.desc[200:300, ::2] = 255
    R = np.array(s.R, np.float64)
    half = 0.5 - rng.random(128) * 2.0 ** -12
    for b, row in enumerate([half, -half, half * (-1.0) ** np.arange(128), half + rng.integers(0, 200, 128),
                             -half - 128.0, np.full(128, 0.5 - 2.0 ** -23), np.full(128, 0.5 + 2.0 ** -23)]):
        for k, at in enumerate((0, 77)):
            R[2 * b + k] = row * 2.0 ** (k - 3)
            R[2 * b + k, at] = 256.0 * 2.0 ** (k - 3)
    s.R = R
    pk = dict(precision=precision)
    ctx = ch.cashash_create(ch.cashash_default_params(**pk), R)
    ds = ch.DeviceSet(ctx.params, s.img_off, s.desc, s.kpts)
    po = oparams(orc, pk)
    mu, codes, buckets = oracle_codes(orc, s.desc, R, po)
    ch.cashash_build_codes(ctx, ds)
    assert ch.cashash_sync_status(ctx) == ch.CASHASH_OK
    assert np.array_equal(ds.codes_np(), codes)
    assert np.array_equal(ds.buckets_np(po.n_tables), buckets)
    approx, bound = ch.cashash_projection_bounds(ctx, ds, 0, ds.n)
    v = orc.projections(s.desc, mu, R, 176)
    err = np.abs(approx.cpu().numpy().astype(np.float64) - v)
    assert (err <= bound.cpu().numpy()).all()
    ctx.close()
