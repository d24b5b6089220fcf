"""Plane output at the edges of its tiles and width groups, against the FP64
oracle (every sample's SNR and width)."""
import math

import numpy as np
import pytest
import torch

import oracle
import synth
from tests import _parity as P

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
LISTS = {"1": [1], "1-32": list(range(1, 33)), "w46": list(range(1, 17)) + list(range(24, 257, 8)),
         "step16": list(range(1, 33)) + list(range(48, 193, 16)), "1-200": list(range(1, 201)),
         "unaligned": [2, 3, 7] + list(range(13, 62, 8)) + [99, 100, 301],
         "wide": [1, 50, 1000, 1016, 1024]}


@pytest.fixture(scope="module")
def spd():
    import paper_1611_09704_gb300 as m
    m.build()
    m.load()
    return m


@pytest.mark.parametrize("name", LISTS)
@pytest.mark.parametrize("n,pad,dtype,scope", [
    (1, 0, "f32", 0), (23, 1, "f32", 0), (3776, 0, "f32", 0), (3785, 7, "f16", 1),
    (9000, 0, "bf16", 0), (9001, 3, "f32", 1),
])
def test_tiles(spd, name, n, pad, dtype, scope):
    widths = LISTS[name]
    sp = synth.ska_like(3, n, n_pulses=4, mean=5.0, sd=2.0, drift_amp=1.0, drift_period=3000,
                        device=DEV, seed=n + len(widths), stride=n + pad)
    x, scale = sp.data, None
    if dtype != "f32":
        q = synth.quantise_rows(sp, dtype)
        x, scale = q.data, q.scale
    op = oracle.Plane(synth.to_host_numpy(x), dtype=dtype, n_samp=n,
                      scale=None if scale is None else scale.cpu().numpy())
    m = spd.msd(x, scope, n_samp=n, scale=scale)
    snr, w = spd.boxcar_snr(x, m, widths, scope=scope, n_samp=n, scale=scale)
    if n == 1:        # one sample has no sd
        if scope == 0 and float(x[:, 0].float().std()) > 0:
            assert torch.isfinite(snr).all() and (spd.widths_to_numpy(w) == 1).all()
        return
    mean, sd, sdn, tab = oracle.msd_and_sigma(op, widths, 0, scope, 0)
    best, win = oracle.boxcar_snr(op, mean, sd, tab, widths, scope)

    def sigma_of(e, v):
        return math.sqrt(v) * float(np.atleast_1d(sd)[e])

    P.check_plane(snr.cpu().numpy(), spd.widths_to_numpy(w), best, win, op, mean, sigma_of,
                  scope=scope)


def test_degenerate_rows(spd):
    x = synth.noise_plane(3, 5000, device=DEV, seed=2)
    x[1] = 7.0
    m = spd.msd(x, 1)
    snr, w = spd.boxcar_snr(x, m, [1, 2, 3], scope=1)
    assert torch.isnan(snr[1]).all() and (w[1] == 0).all()
    assert torch.isfinite(snr[0]).all() and torch.isfinite(snr[2]).all()
