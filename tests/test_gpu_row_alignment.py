"""16-bit planes whose rows start on 8-byte but not on 16-byte boundaries: the
bulk copies of the search need 16, so such rows take plain loads and give the
records and planes of the same values at a padded stride."""
import numpy as np
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


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("stride,first", [(17740, 0), (20000, 4), (9004, 4)])
def test_rows_at_odd_8_byte_steps(spd, dtype, stride, first):
    n_dm, n = 5, stride - 8
    widths = list(range(1, 17)) + list(range(24, 129, 8))
    sp = synth.ska_like(n_dm, n, n_pulses=6, mean=0.0, sd=1.0, drift_amp=0.0, device=DEV, seed=31)
    q = synth.quantise_rows(sp, dtype)
    wide = (stride + 15) // 8 * 8          # rows of whole 16-byte pieces
    padded = torch.zeros((n_dm, wide), dtype=q.data.dtype, device=DEV)
    padded[:, :n] = q.data[:, :n]
    flat = torch.zeros(n_dm * stride + 16, dtype=q.data.dtype, device=DEV)
    odd = flat[first:first + n_dm * stride].view(n_dm, stride)
    odd[:, :n] = q.data[:, :n]
    got = []
    for x in (odd, padded):
        out, res, msd = spd.search(x, widths, 6.0, 1 << 16, n_samp=n, scale=q.scale)
        count, status = spd.read_result(res)
        assert status == 0 and 0 < count < 1 << 16
        snr, w = spd.boxcar_snr(x, msd, widths, n_samp=n, scale=q.scale)
        got.append((np.sort(spd.candidates_to_numpy(out, count), order=["dm", "sample"]),
                    snr.cpu().numpy(), spd.widths_to_numpy(w)))
    for a, b in zip(*got):
        assert np.array_equal(a, b)
