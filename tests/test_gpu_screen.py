"""The screened search against the search of every tile: the same records, bit
for bit (a start's SNR comes out of the same operations either way).  A
workspace one byte short of the screen's piece gives the unscreened search."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
W46 = list(range(1, 17)) + list(range(24, 257, 8))
LISTS = {"32": list(range(1, 33)), "46": W46, "512": list(range(1, 513)),
         "16": list(range(1, 33)) + list(range(48, 257, 16)),
         "odd": [3, 5, 20, 22, 51, 100, 301, 1000, 2000], "far": [1, 100, 4000, 4096]}


@pytest.fixture(scope="module")
def spd():
    import paper_1611_09704_gb300 as m
    m.build()
    m.load()
    return m


def _both(spd, x, widths, thr, cap=1 << 20, **kw):
    sig = {k: v for k, v in kw.items() if k in ("sigma_mode", "scope", "nmax_sigma")}
    pl = {k: v for k, v in kw.items() if k not in sig}
    nb = spd.search_workspace_bytes(x, widths, thr, **kw)
    got = []
    for n in (nb, nb - 1):
        ws = torch.full((nb,), 0x5A, dtype=torch.uint8, device=DEV)[:n]
        out, res, _ = spd.search(x, widths, thr, cap, workspace=ws, **sig, **pl)
        count, status = spd.read_result(res)
        assert count <= cap
        got.append((status, np.sort(spd.candidates_to_numpy(out, count),
                                    order=["dm", "sample", "width"])))
    return got


@pytest.mark.parametrize("name", LISTS)
@pytest.mark.parametrize("n_samp,stride", [(1, 1), (17, 20), (255, 255), (3792, 3792), (3793, 3800),
                                           (4017, 4017), (30011, 30016)])
def test_sizes_and_width_lists(spd, name, n_samp, stride):
    sp = synth.ska_like(6, n_samp, n_pulses=6, mean=3.0, sd=1.0, drift_amp=0.5, drift_period=9000,
                        device=DEV, seed=n_samp, stride=stride)
    for scope in (0, 1):
        (s0, a), (s1, b) = _both(spd, sp.data, LISTS[name], 4.0, n_samp=n_samp, scope=scope)
        assert s0 == s1 and np.array_equal(a, b)
        assert n_samp < 3000 or a.size


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("stride", [9000, 9004, 9001])     # 16-byte, 8-byte and 2-byte steps
def test_stored_types(spd, dtype, stride):
    sp = synth.ska_like(5, 9000, n_pulses=8, drift_amp=0.0, device=DEV, seed=5)
    q = synth.quantise_rows(sp, dtype)
    x = torch.zeros((5, stride), dtype=q.data.dtype, device=DEV)
    x[:, :9000] = q.data
    off = torch.linspace(-3, 3, 5, device=DEV)
    for kw in ({}, {"offset": off}, {"sigma_mode": spd.SIGMA_LINEAR_EXCESS}):
        (s0, a), (s1, b) = _both(spd, x, W46, 4.0, n_samp=9000, scale=q.scale, **kw)
        assert s0 == s1 == 0 and a.size and np.array_equal(a, b)


@pytest.mark.parametrize("thr", [-1.0, 0.0, 1.0, 50.0])
def test_thresholds(spd, thr):
    x = synth.ska_like(3, 20000, n_pulses=4, device=DEV, seed=8).data
    (s0, a), (s1, b) = _both(spd, x, W46, thr)
    assert s0 == s1 == 0 and np.array_equal(a, b)
    assert a.size == 0 or thr < 50


def test_more_live_units_than_the_list_holds(spd):
    """14 lone spikes per tile: few enough for the list of units, too many of
    them for its room, so the last tiles are searched whole."""
    n_dm, widths = 32, [1, 2]
    halo = (widths[-1] + 47) // 16 + 1
    tile = 16 * (256 - halo)
    n = 25 * tile
    x = synth.noise_plane(n_dm, n, device=DEV, seed=3).clamp_(-4, 4)
    at = torch.arange(n, device=DEV)
    x[:, ((at % tile) % 272 == 12) & ((at % tile) < 14 * 272)] = 12.0
    (s0, a), (s1, b) = _both(spd, x, widths, 8.0)
    assert s0 == s1 == 0 and a.size >= n_dm * 25 * 14 and np.array_equal(a, b)


def test_samples_that_are_not_finite(spd):
    """A sample that is not finite hides no start whose windows avoid it."""
    x = synth.noise_plane(4, 12000, device=DEV, seed=4)
    x[:, 8000:8010] += 9.0
    clean = x.clone()
    for r, v in enumerate((float("nan"), float("inf"), float("-inf"))):
        x[r, 3000] = v
    msd = spd.msd(clean)
    widths = list(range(1, 33))
    got = []
    for y in (x, clean):
        out, res = spd.detect(y, msd, widths, 6.0, 1 << 16)
        count, status = spd.read_result(res)
        got.append(spd.candidates_to_numpy(out, count))
    away = lambda r: np.sort(r[np.abs(r["sample"] - 3000) > 40], order=["dm", "sample"])
    assert away(got[1]).size and np.array_equal(away(got[0]), away(got[1]))
