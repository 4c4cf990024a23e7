"""The kinetic sums of the observables hold what FP64 sums of the particles'
FP32 values hold: the last bit of a sum, and sums beyond the FP32 range."""
import numpy as np
import pytest

import paper_1311_0402_gb300 as dpd
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _observe(x, v, box, through_buffer):
    g = dpd.Sim(box, [[25.0]], 4.5, 1.0, 1.0, 1.0, 0.01)
    g.set_state(x, v)
    if through_buffer:
        buf = dpd.ObsBuffer(1)
        g.observables_async(buf, 0)
        g.sync()
        o = buf.get(0)
    else:
        o = g.observables()
    g.close()
    return o


def _isolated(k):
    """k^3 particles two cutoffs apart."""
    return 2.0 * np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5, (2.0 * k,) * 3


# exact in FP64 (a 1 followed by 52 bits at most), whatever the order: the
# expected values are equal, not close
@pytest.mark.parametrize("through_buffer", [False, True])
@pytest.mark.parametrize("k", [3, 4, 7])
def test_sums_keep_the_bits_of_fp64(k, through_buffer):
    need_gpu()
    x, box = _isolated(k)
    v = np.zeros((k ** 3, 3))
    v[:3, 0] = 1.0, 2.0 ** -26, 2.0 ** -51
    v[-2:, 1] = -2.0, 2.0 ** -50
    o = _observe(x, v, box, through_buffer)
    assert o["momentum"][0] == 1.0 + 2.0 ** -26 + 2.0 ** -51
    assert o["momentum"][1] == -2.0 + 2.0 ** -50
    assert o["momentum"][2] == 0.0
    w = np.zeros((k ** 3, 3))
    w[:3, 2] = 1.0, 2.0 ** -13, 2.0 ** -25
    assert _observe(x, w, box, through_buffer)["kinetic"] == 0.5 * (1.0 + 2.0 ** -26 + 2.0 ** -50)


@pytest.mark.parametrize("k", [4, 7])
def test_sums_beyond_the_fp32_range(k):
    """|v|^2 of each particle fits FP32, their sum does not."""
    need_gpu()
    x, box = _isolated(k)
    v = 1.0e19 * np.where(np.arange(3 * k ** 3) % 2, 1.0, -1.0).reshape(-1, 3)
    o = _observe(x, v, box, False)
    s = (v.astype(np.float32).astype(np.float64) ** 2).sum()
    assert abs(o["kinetic"] - 0.5 * s) < 1e-12 * s
    assert abs(o["temperature"] - s / (3 * k ** 3 - 3)) < 1e-12 * o["temperature"]
    assert np.array_equal(o["momentum"], v.astype(np.float32).astype(np.float64).sum(0))
