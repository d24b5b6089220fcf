"""Runs of one search give the same bits, with more live units than tiles to
search whole.  A start's rounding can depend on whether its tile is searched
whole or by single units (a spike in each tile makes the two skip different
width groups), so that choice must not depend on the order of arrival."""
import ctypes

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


def test_repeated_searches_are_equal(spd):
    widths = list(range(1, 17)) + list(range(24, 257, 8))
    thr, n_dm, n = 7.0, 8192, 3056
    x = synth.noise_plane(n_dm, n, mean=3.0, device=DEV, seed=11)
    msd = spd.msd(x)
    r = torch.arange(n_dm, device=DEV)[:, None]
    t = torch.arange(n, device=DEV)
    x[:, 5] += 1e5
    for k in range(2):      # two pulses of 30 to 35 samples a row: some 9 live units
        w = 30 + (r * 37 + 11 * k) % 6
        at = 300 + 1300 * k + (r * 101) % 100
        x += torch.where((t >= at) & (t < at + w), 8.0 / w.sqrt(), 0.0)
    prm, keep = spd.binding._params(widths, thr, 0, 0, 0)
    ws = torch.empty(spd.binding.load().spd_detect_workspace_bytes(
        ctypes.byref(spd.Plane(x).c()), ctypes.byref(prm)), dtype=torch.uint8, device=DEV)
    first = None
    for _ in range(20):
        out, res = spd.detect(x, msd, widths, thr, 1 << 21, workspace=ws)
        count, status = spd.read_result(res)
        assert status == 0 and 20 * n_dm < count <= 1 << 21
        out = out[:count]
        out = out[torch.argsort(out[:, 0].long() * n + out[:, 1])]
        if first is None:
            first = out
        assert first.shape == out.shape and torch.equal(first, out)
