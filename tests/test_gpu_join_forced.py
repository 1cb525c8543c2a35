"""Cases of one to three pairs, where the band's and the degenerate sets'
decisions are worked out, through the bucket join: plans of so few pairs take
the warp-per-query kernel by default, so here the join is forced."""
import pytest

import test_gpu_parity as cases
from test_gpu_parity import ch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(params=["join", "join_tc"])
def forced(request, ch, monkeypatch):  # noqa: F811
    """check_case of the batched schedule, with the kernel forced and its plan asked for it."""
    kernel = ch.CASHASH_KERNEL_JOIN if request.param == "join" else ch.CASHASH_KERNEL_JOIN_TC
    tuning = (kernel, 4 if request.param == "join" else 0, 0)
    check, ran = cases.check_case, []

    def check_case(ch, orc, s, pairs, **pk):
        assert pk.setdefault("schedule", 1) == 1 and pk.pop("tuning", None) is None
        ran.append(len(pairs))
        return check(ch, orc, s, pairs, tuning=tuning, **pk)

    monkeypatch.setattr(cases, "check_case", check_case)
    yield
    assert ran


def test_band_edge_decisions(ch, orc, forced):  # noqa: F811
    cases.test_band_edge_decisions(ch, orc, 1)


@pytest.mark.parametrize("case", ["huge_coordinates", "large_F", "infinite_point", "nan_point", "huge_F"])
def test_band_threshold_fallbacks(ch, orc, forced, case):  # noqa: F811
    cases.test_band_threshold_fallbacks(ch, orc, case)


def test_identical_and_degenerate_descriptors(ch, orc, forced):  # noqa: F811
    cases.test_identical_and_degenerate_descriptors(ch, orc)


def test_one_pair_workload(ch, orc, forced):  # noqa: F811
    s = cases.synth.config0()
    cases.check_case(ch, orc, s, s.pairs)
