"""The autotuner's cache: a set tuned again gets the configuration it got the
first time, and another set of about the same size is tuned on its own."""
import re

import numpy as np
import pytest

import lbm_workloads as wl
import paper_1904_02471_gb300 as pkg

pytestmark = pytest.mark.gpu

VMAX4 = 2.33441421833897723932


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available()
    from paper_1904_02471_gb300 import build
    build.build()
    torch.cuda.init()
    return torch.cuda.get_device_properties(0).multi_processor_count


def _tuned(nx, ny, scheme="rk3", record=0):
    """Tile index or rows and grid of an FD lattice's group, from the report, and
    its populations after four steps."""
    dt = 0.3 / nx / VMAX4
    B = pkg.Batch([pkg.make_spec("fd", 4, nx, ny, 2 * dt, dt, 0.0, "fp32", scheme=scheme)])
    B.init(0, *wl.taylor_green(nx, ny, 0.01))
    if record:
        B.record(0, record, 100)
    rep = B.tune(2)
    B.step(4)
    f, ser = B.populations(0), B.series(0)
    B.close()
    return rep, int(re.search(r"grid=(\d+)", rep).group(1)), f, ser


def test_a_larger_set_is_not_held_to_a_smaller_ones_blocks(gpu):
    """128 x 65 and 128 x 127 have the same size to a factor of two; the grid is one
    block per SM, two, or one per tile of the set itself."""
    for ny in (65, 127):
        rep, grid, _, _ = _tuned(128, ny)
        m = re.search(r"tile=32x(\d+)", rep)
        assert m, rep   # not taken from another set
        items = 4 * -(-ny // int(m.group(1)))
        assert grid in {min(items, k * gpu) for k in (1, 2)} | {items}, rep


@pytest.mark.parametrize("record", [0, 1, 7])
def test_the_same_set_gets_the_same_configuration(record):
    first = _tuned(640, 333, record=record)
    second = _tuned(640, 333, record=record)
    assert "cached" not in first[0] and "cached" in second[0]
    assert first[1] == second[1]
    assert np.array_equal(first[2], second[2])
    steps = list(range(0, 4, record)) if record else []
    assert [o["step"] for o in first[3]] == [o["step"] for o in second[3]] == steps
