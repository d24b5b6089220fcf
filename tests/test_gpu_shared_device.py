"""The search of listed tiles while another stream keeps all but one place of
the device busy, so that single CTAs take listed tiles one after the other:
the records are those of the search of every tile."""
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


def test_listed_tiles_beside_another_stream(spd):
    widths, thr = list(range(1, 17)), 6.0
    tile = 16 * (256 - ((widths[-1] + 47) // 16 + 1))     # starts per tile
    n_dm, n = 96, 24 * tile
    x = synth.noise_plane(n_dm, n, device=DEV, seed=3)
    msd = spd.msd(x)
    at = torch.arange(n, device=DEV)
    x[:, (at // tile) % 2 == 1] += 12.0          # every second tile full of candidates
    x += (at % 977).to(torch.float32) * 1e-3     # no two tiles alike
    prm, keep = spd.binding._params(widths, thr, 0, 0, 0)
    nb = spd.binding.load().spd_detect_workspace_bytes(ctypes.byref(spd.Plane(x).c()),
                                                       ctypes.byref(prm))
    out = torch.zeros((n_dm * n, 4), dtype=torch.int32, device=DEV)
    res = torch.empty(16, dtype=torch.uint8, device=DEV)

    def records(ws, stream=None):
        if stream is None:
            spd.detect(x, msd, widths, thr, out.shape[0], out=out, result=res, workspace=ws)
        else:
            with torch.cuda.stream(stream):
                spd.detect(x, msd, widths, thr, out.shape[0], out=out, result=res, workspace=ws)
        torch.cuda.synchronize()
        count, status = spd.read_result(res)
        assert status == 0 and count <= out.shape[0]
        r = out[:count].to(torch.int64)
        return r[torch.argsort(r[:, 0] * n + r[:, 1])]

    ws = torch.empty(nb, dtype=torch.uint8, device=DEV)
    want = records(ws[:nb - 1])                  # no room for the screen: every tile
    # one tile per CTA on all but one of 304 places, some 40 launches in a row
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    bg = synth.noise_plane(1, 3776 * (2 * sms - 1), device=DEV, seed=9)
    bg_msd, bg_widths = spd.msd(bg), list(range(1, 257))
    planes = spd.boxcar_snr(bg, bg_msd, bg_widths)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(20):
        with torch.cuda.stream(b):
            for _ in range(40):
                spd.boxcar_snr(bg, bg_msd, bg_widths, snr_out=planes[0], width_out=planes[1])
        got = records(ws, a)
        assert got.shape == want.shape and torch.equal(got, want)
