"""Plane output with halos of 33 to 64 blocks, where the last one or two warps
of a CTA hold no starts and reach the end of a tile long before the others:
runs of several tiles per CTA, rows at vector boundaries and not, against the
FP64 oracle (every sample's SNR and width)."""
import math

import numpy as np
import pytest

import oracle
import synth
from tests import _parity as P

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
LISTS = {"1-512": list(range(1, 513)), "to 968": list(range(1, 17)) + list(range(24, 969, 16))}


@pytest.fixture(scope="module")
def spd():
    import paper_1611_09704_gb300 as m
    m.build()
    m.load()
    return m


@pytest.mark.parametrize("name", LISTS)
@pytest.mark.parametrize("n,pad,dtype", [(120000, 0, "f32"), (120001, 0, "f32"),
                                         (120001, 0, "f16")])
def test_plane_with_idle_warps(spd, name, n, pad, dtype):
    widths, n_dm = LISTS[name], 22        # 740 tiles and more: two or three per CTA
    sp = synth.ska_like(n_dm, n, n_pulses=6, mean=5.0, sd=2.0, drift_amp=1.0, drift_period=30000,
                        device=DEV, seed=n + len(widths), stride=n + pad)
    x, scale = sp.data, None
    if dtype != "f32":
        q = synth.quantise_rows(sp, dtype)
        x, scale = q.data, q.scale
    op = oracle.Plane(synth.to_host_numpy(x), dtype=dtype, n_samp=n,
                      scale=None if scale is None else scale.cpu().numpy())
    m = spd.msd(x, 0, n_samp=n, scale=scale)
    snr, w = spd.boxcar_snr(x, m, widths, n_samp=n, scale=scale)
    mean, sd, sdn, tab = oracle.msd_and_sigma(op, widths, 0, 0, 0)
    best, win = oracle.boxcar_snr(op, mean, sd, tab, widths, 0)

    def sigma_of(e, v):
        return math.sqrt(v) * float(np.atleast_1d(sd)[e])

    P.check_plane(snr.cpu().numpy(), spd.widths_to_numpy(w), best, win, op, mean, sigma_of)
