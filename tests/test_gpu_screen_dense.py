"""Planes most of whose tiles are full of candidates: below, at and above the
part at which all tiles are searched instead of the listed ones, with the rest
empty or holding single pulses; and thresholds that no bound can use.  The
records are those of the search without a screen."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
W46 = list(range(1, 17)) + list(range(24, 257, 8))


@pytest.fixture(scope="module")
def spd():
    import paper_1611_09704_gb300 as m
    m.build()
    m.load()
    return m


def _both(spd, x, widths, thr, **kw):
    nb, n = spd.search_workspace_bytes(x, widths, thr, **kw), x.shape[1]
    got = []
    for room in (nb, nb - 1):      # with a screen, and without
        ws = torch.empty(nb, dtype=torch.uint8, device=DEV)[:room]
        out, res, _ = spd.search(x, widths, thr, x.numel(), workspace=ws, **kw)
        count, status = spd.read_result(res)
        assert status == 0 and count <= x.numel()
        out = out[:count]
        got.append(out[torch.argsort(out[:, 0].long() * n + out[:, 1])])
    return got


# of 5120 tiles (enough for chunks of more than one): 14/16 .. 16/16
@pytest.mark.parametrize("full", [4480, 4799, 4800, 4801, 5120])
@pytest.mark.parametrize("scope", [0, 1])
def test_part_of_the_tiles(spd, full, scope):
    tile = 16 * (256 - ((W46[-1] + 47) // 16 + 1))
    n_dm, n = 1280, 4 * tile
    x = synth.noise_plane(n_dm, n, mean=2.0, device=DEV, seed=full)
    g = torch.Generator(device=DEV).manual_seed(full)
    rest = torch.randperm(4 * n_dm, generator=g, device=DEV)[:4 * n_dm - full]
    up = torch.ones(4 * n_dm, device=DEV)
    up[rest] = 0.0
    # one half period of a square wave per 512 samples: every unit sees a rise
    wave = torch.sign(torch.sin(torch.arange(n, device=DEV) * (3.14159265 / 256)))
    x += 2.0 * wave * up.view(n_dm, 4).repeat_interleave(tile, 1)
    at = rest[::2]
    x[at // 4, (at % 4) * tile + 1000] += 30.0      # a pulse in every second other tile
    a, b = _both(spd, x, W46, 6.0, scope=scope)
    assert a.shape == b.shape and torch.equal(a, b) and a.shape[0] > n_dm * n // 8


@pytest.mark.parametrize("thr", [-3.0, 0.0, 1e-30, 0.5])
def test_thresholds_without_bounds(spd, thr):
    x = synth.noise_plane(400, 4000, device=DEV, seed=8)
    a, b = _both(spd, x, list(range(1, 9)), thr)
    assert a.shape == b.shape and torch.equal(a, b) and a.shape[0] > x.numel() // 4
