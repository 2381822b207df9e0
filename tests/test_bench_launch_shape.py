"""bench.py reports the launch shape that its timed kernel has, and says when an
option cannot change it."""
import re
import sys

import pytest

ROOT = __file__.rsplit("/", 2)[0]


@pytest.fixture(scope="module")
def bench():
    sys.path.insert(0, ROOT)
    import bench
    return bench


def _constant(unit, name):
    text = open("%s/paper_2511_19633_gb300/csrc/%s" % (ROOT, unit)).read()
    return int(re.search(r"constexpr int %s = (\d+);" % name, text).group(1))


def test_reported_shape_is_the_kernels(bench):
    shape = bench.timed_launch_shape(True)
    assert shape["events_in_flight_per_sm"] == _constant("shower_mixed.cu", "kSlots")
    shape = bench.timed_launch_shape(False)
    assert shape["threads_per_block"] == _constant("shower_fp64.cu", "kThreads")
    assert shape["blocks_per_sm"] == _constant("shower_fp64.cu", "kMinBlocks")
    assert shape["events_in_flight_per_sm"] == (shape["blocks_per_sm"] * shape["threads_per_block"]
                                                // _constant("shower_fp64.cu", "kG"))


def test_options_without_effect_are_named(bench):
    class Args:
        pass

    args = Args()
    for k, v in bench.SHAPE_OPTIONS.items():
        setattr(args, k, v)
    assert bench.shape_options_given(args) == []
    args.veto_bps, args.block = 3, 128
    assert bench.shape_options_given(args) == ["--block", "--veto-bps"]
