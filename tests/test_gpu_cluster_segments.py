"""Clusters across the segments a row is cut into (4096 samples and up): every
field equal to the oracle's walk along the whole row."""
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


@pytest.mark.parametrize("n_samp", [4096, 4097, 8191, 12288, 30001])
@pytest.mark.parametrize("thr,gap", [
    (9.0, 1),        # many short clusters
    (9.0, 60),       # long ones, over several segments
    (2.0, 30),       # one per row
    (9.5, 5),        # no candidate at all
    (9.0, 5000),     # a gap longer than the shortest segment
])
def test_segments_match_the_oracle(spd, n_samp, thr, gap):
    snr, width = synth.snr_plane(3, n_samp, device=DEV, seed=n_samp + gap)
    snr[1, 4000:4096] = 0.0           # a quiet stretch up to a boundary
    snr[1, 4096:4097] = 9.0
    snr[2, 100:8000] = 0.0            # and one over a whole segment
    out, res = spd.cluster_rows(snr, width, thr, gap, 1 << 16)
    count, status = spd.read_result(res)
    want = oracle.cluster_rows(synth.to_host_numpy(snr),
                               synth.to_host_numpy(width).view(np.uint16), thr, gap)
    assert status == 0 and count == want.size
    _compare(spd.clusters_to_numpy(out, count), want)
