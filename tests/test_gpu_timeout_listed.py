"""A copy that times out in the search of listed tiles: the CTA leaves without
searching live units in shared memory that the copy may still write.  The call
reports the timeout, what records there are belong to the plane, and the next
search is complete."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def spd():
    import paper_1611_09704_gb300 as m
    m.build()
    m.load()
    return m


def test_timeout_among_listed_tiles(spd):
    from paper_1611_09704_gb300.binding import SPD_ERR_TIMEOUT, debug_set_copy_wait
    # rows of dense tiles between rows of noise with live units
    x = synth.ska_like(256, 20000, n_pulses=40, drift_amp=0.0, mean=0.0, sd=1.0, device=DEV,
                       seed=5).data
    x[::2] += 1.5
    widths, thr, cap = list(range(1, 33)), 6.0, 1 << 22

    def records():
        out, res, _ = spd.search(x, widths, thr, cap)
        count, status = spd.read_result(res)
        return np.sort(spd.candidates_to_numpy(out, count), order=["dm", "sample"]), status

    want, status = records()
    assert status == 0 and np.unique(want["dm"] % 2).size == 2
    try:
        debug_set_copy_wait(20_000_000, 32)
        got, status = records()
    finally:
        debug_set_copy_wait()
    assert status == SPD_ERR_TIMEOUT and got.size < want.size
    assert np.isin(got, want).all()
    again, status = records()
    assert status == 0 and np.array_equal(again, want)
