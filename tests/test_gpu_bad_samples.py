"""Starts next to a sample that is not finite, given the statistics of clean
data: a window that holds it has no SNR, and every start is found by its other
windows.  One row per place of the sample in a unit of 16 starts and distance of
a spike before it; the expected records come from plain FP64 sums."""
import ctypes

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
AT, THR = 2000, 6.0
LISTS = {"8": list(range(1, 9)), "32": list(range(1, 33)), "8-step": [1, 2, 8, 16, 24, 32, 40],
         "far": [1, 2, 3, 20, 900]}


@pytest.fixture(scope="module")
def spd():
    import paper_1611_09704_gb300 as m
    m.build()
    m.load()
    return m


def _rows(value, n):
    """(rows with the sample, the sample's place in each, clean rows)"""
    x = synth.noise_plane(16 * 15, n, device=DEV, seed=7).clamp_(-3, 3)
    place = AT + torch.arange(240, device=DEV) // 15
    dist = 1 + torch.arange(240, device=DEV) % 15
    r = torch.arange(240, device=DEV)
    x[r, place - dist] = 12.0
    x[r, place + 40 + dist] = 12.0
    clean = x.clone()
    x[r, place] = value
    return x, place.cpu().numpy(), clean


def _records(spd, x, msd, widths):
    """Which samples are records: screened, and every tile."""
    prm, keep = spd.binding._params(widths, THR, 0, 0, 0)
    nb = spd.binding.load().spd_detect_workspace_bytes(ctypes.byref(spd.Plane(x).c()),
                                                       ctypes.byref(prm))
    for room in (nb, nb - 1):
        ws = torch.empty(nb, dtype=torch.uint8, device=DEV)[:room]
        out, res = spd.detect(x, msd, widths, THR, 1 << 20, workspace=ws)
        count, status = spd.read_result(res)
        assert status == 0
        got = np.zeros(x.shape, dtype=bool)
        rec = spd.candidates_to_numpy(out, count)
        got[rec["dm"], rec["sample"]] = True
        yield got


def _expected(x, place, msd, widths, starts):
    """Best SNR of each row's starts over the windows inside the row without the sample."""
    y = x.double().cpu().numpy() - msd["mean"][0]
    n = x.shape[1]
    best = np.full((x.shape[0], len(starts)), -np.inf)
    for r, bad in enumerate(place):
        v = y[r].copy()
        v[bad] = 0.0
        c = np.concatenate(([0.0], np.cumsum(v)))
        for w in widths:
            for k, d in enumerate(starts):
                s = bad + d
                if s + w <= n and not s <= bad < s + w:
                    best[r, k] = max(best[r, k], (c[s + w] - c[s]) / np.sqrt(w) / msd["sd"][0])
    return best


def _check(spd, value, name, starts, n):
    widths = LISTS[name]
    x, place, clean = _rows(value, n)
    msd = spd.msd(clean)
    best = _expected(x, place, spd.msd_to_numpy(msd), widths, starts)
    assert (best >= THR).any(axis=1).any()
    for got in _records(spd, x, msd, widths):
        have = np.stack([got[r, place[r] + np.asarray(starts)] for r in range(x.shape[0])])
        sure = np.abs(best - THR) > 1e-3
        assert np.array_equal(have[sure], (best >= THR)[sure])


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("name", LISTS)
def test_starts_before_the_sample(spd, value, name):
    # close to the row end: fewer units follow the sample than make a tile worth
    # searching whole
    _check(spd, value, name, list(range(-48, 0)), 2190)


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("name", LISTS)
def test_starts_after_the_sample(spd, value, name):
    # every unit after the sample's own, in tiles that are searched whole
    _check(spd, value, name, list(range(16, 64)), 4400)


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("n", [2190, 4400])
def test_starts_after_the_sample_in_its_unit(spd, value, n):
    """Found by widths to 16; wider ones may miss them."""
    x, place, clean = _rows(value, n)
    r = torch.arange(x.shape[0], device=DEV)
    x[r, torch.from_numpy(place).to(DEV) + 3] = 12.0
    msd = spd.msd(clean)
    best = _expected(x, place, spd.msd_to_numpy(msd), list(range(1, 17)), list(range(1, 16)))
    for got in _records(spd, x, msd, list(range(1, 33))):
        have = np.stack([got[r, place[r] + np.arange(1, 16)] for r in range(x.shape[0])])
        assert have[best >= THR + 1e-3].all()
