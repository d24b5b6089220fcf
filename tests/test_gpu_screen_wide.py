"""The screen at wide width lists, whose tiles are searched whole from few live
units on: one, two and up to sixteen pulses per tile, against the search of every
tile.  Integer samples and a spacing of the pulses that leaves every sum exact,
so the records are equal bit for bit."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
LISTS = {"256": [1, 2, 3] + list(range(8, 257, 8)), "700": [1, 5, 100, 700],
         "2048": [1, 2, 3, 500, 2048], "4096": [1, 100, 4000, 4096]}


@pytest.fixture(scope="module")
def spd():
    import paper_1611_09704_gb300 as m
    m.build()
    m.load()
    return m


@pytest.mark.parametrize("name", LISTS)
def test_pulses_per_tile(spd, name):
    widths, thr, n_dm, n = LISTS[name], 7.0, 340, 9000
    # statistics of data of mean 0 and sd 1
    msd = spd.msd((torch.arange(2048, device=DEV) % 2 * 2.0 - 1.0).view(2, 1024))
    x = (torch.arange(n, device=DEV) % 2 * 2.0 - 1.0).repeat(n_dm, 1)
    r, t = torch.arange(n_dm, device=DEV)[:, None], torch.arange(n, device=DEV)
    # a pulse of height 10 every 3000 / k samples, k = 0 .. 16 by row
    k = r % 17
    step = torch.where(k > 0, 3000 // k.clamp(min=1), 2 * n)
    x += torch.where((t % step == 7) & (t < k * step), 10.0, 0.0)
    prm, keep = spd.binding._params(widths, thr, 0, 0, 0)
    nb = spd.binding.load().spd_detect_workspace_bytes(ctypes.byref(spd.Plane(x).c()),
                                                       ctypes.byref(prm))
    got = []
    for room in (nb, nb - 1):      # screened, and every tile
        ws = torch.empty(nb, dtype=torch.uint8, device=DEV)[:room]
        out, res = spd.detect(x, msd, widths, thr, 1 << 20, workspace=ws)
        count, status = spd.read_result(res)
        assert status == 0 and n_dm < count <= 1 << 20
        out = out[:count]
        got.append(out[torch.argsort(out[:, 0].long() * n + out[:, 1])])
    assert got[0].shape == got[1].shape and torch.equal(got[0], got[1])
