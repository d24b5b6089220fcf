"""Clusters that run through many loads of a warp: breaks of exactly the gap and of
one sample more at every place of a load, equal peaks in several lanes and loads,
and signed zeros, against the oracle's walk along the whole row."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.test_gpu_cluster import _compare

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def spd():
    import paper_1611_09704_gb300 as m
    m.build()
    m.load()
    return m


@pytest.mark.parametrize("gap", [1, 7, 30, 31, 32, 100, 600])
@pytest.mark.parametrize("every", [1, 3])       # every sample a candidate, or every third
def test_runs_with_breaks(spd, gap, every):
    n = 20000
    snr = torch.zeros((96, n), device=DEV)
    g = torch.Generator(device=DEV).manual_seed(gap)
    snr[:, ::every] = torch.randint(7, 12, (96, (n + every - 1) // every), generator=g,
                                    device=DEV).to(torch.float32)
    for r in range(96):                          # one break a row, around sample 5000
        at = 5000 + 11 * r
        snr[r, at:at + max(gap, every) + r % 3] = 0.0
    width = torch.randint(1, 300, (96, n), generator=g, device=DEV).to(torch.int16)
    out, res = spd.cluster_rows(snr, width, 7.0, gap, 1 << 21)
    count, status = spd.read_result(res)
    want = oracle.cluster_rows(synth.to_host_numpy(snr),
                               synth.to_host_numpy(width).view(np.uint16), 7.0, gap)
    assert status == 0 and count == want.size <= 1 << 21
    _compare(spd.clusters_to_numpy(out, count), want)


def test_equal_and_signed_zero_peaks(spd):
    n = 9000
    snr = torch.full((4, n), -1.0, device=DEV)
    snr[0, 100:8000] = -0.0                      # the first of equal peaks, of either sign
    snr[0, 3000:7000] = 0.0
    snr[1, 100:8000] = 0.0
    snr[1, 3000:7000] = -0.0
    snr[2, 700:8500:5] = 3.0                     # the same peak in every load
    snr[3] = float("-inf")
    width = (torch.arange(4 * n, device=DEV) % 500).view(4, n).to(torch.int16)
    for thr in (-0.5, 0.0, -2.0):
        out, res = spd.cluster_rows(snr, width, thr, 40, 1 << 16)
        count, status = spd.read_result(res)
        want = oracle.cluster_rows(synth.to_host_numpy(snr),
                                   synth.to_host_numpy(width).view(np.uint16), thr, 40)
        assert status == 0 and count == want.size
        _compare(spd.clusters_to_numpy(out, count), want)
