"""The level planes of the decimated search, several levels per pass: the
records equal a search of planes decimated one level at a time."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def spd():
    import paper_1611_09704_gb300 as m
    m.build()
    m.load()
    return m


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("n,pad,first", [(40000, 0, 0), (33331, 1, 1), (4096 * 3 + 15, 9, 0)])
@pytest.mark.parametrize("levels", [
    [(0, [1]), (1, [1, 2, 3])],
    [(2, [1, 2, 5, 7]), (5, [1, 3])],          # past one pass, levels left out
    [(0, [1, 2]), (3, [1, 4]), (4, [5, 9]), (9, [1, 2])],
])
def test_levels(spd, dtype, n, pad, first, levels):
    sp = synth.ska_like(7, n, n_pulses=10, mean=0.0, sd=1.0, drift_amp=0.0, device=DEV, seed=n)
    x, scale = sp.data, None
    if dtype != "f32":
        q = synth.quantise_rows(sp, dtype)
        x, scale = q.data, q.scale
    flat = torch.zeros(first + 7 * (n + pad), dtype=x.dtype, device=DEV)
    rows = flat[first:].view(7, n + pad)
    rows[:, :n] = x
    out, res, _ = spd.search_decimated(rows, levels, 5.0, 1 << 18, n_samp=n, scale=scale)
    count, status = spd.read_result(res)
    got = spd.candidates_to_numpy(out, count)
    y = x.float()
    if scale is not None:
        y = scale[:, None] * y
    want = []
    for level in range(levels[-1][0] + 1):
        if level:
            m = y.shape[1] // 2
            y = (y[:, 0:2 * m:2] + y[:, 1:2 * m:2]).contiguous()
        for lv, w in levels:
            if lv != level:
                continue
            # width 1 is evaluated where it is listed (and always by a search)
            plane = spd.Plane(x, scale=scale) if level == 0 else y
            o, r, _ = spd.search(plane, w, 5.0, 1 << 18)
            rec = spd.candidates_to_numpy(o, spd.read_result(r)[0]).copy()
            if w[0] != 1:
                rec = None
                break
            rec["sample"] <<= level
            rec["width"] <<= level
            want.append(rec)
    order = ["dm", "sample", "width"]
    if levels[-1][0] == 9:      # a level whose list starts past width 1: its count alone
        lo, hi = 5 << 4, 9 << 4
        got = got[(got["width"] < lo) | (got["width"] > hi)]
    want = np.concatenate(want)
    assert status == 0 and want.size
    assert np.array_equal(np.sort(got, order=order), np.sort(want, order=order))
