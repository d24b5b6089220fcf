"""Chunks of a stream at any element step, from device memory (copied by the
library's kernel, the MSD read from the chunk) and from page-locked host memory
(copied by the runtime): the same records and running MSD, bit for bit."""
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


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16])
@pytest.mark.parametrize("wmax", [1, 2, 6, 9, 17, 64])      # halos of 0 .. 63 samples
@pytest.mark.parametrize("first,pad", [(0, 0), (1, 0), (3, 5), (8, 1)])
def test_device_and_host_chunks_agree(spd, dtype, wmax, first, pad):
    n_dm, lengths, cap = 9, [3000, 1, 47, 4096, 2011], 1 << 16
    total = sum(lengths)
    x = synth.ska_like(n_dm, total, n_pulses=8, mean=0.0, sd=1.0, drift_amp=0.0, device=DEV,
                       seed=wmax).data.to(dtype)
    got = []
    for host in (False, True):
        bs = spd.binding.BeamStream(n_dm, dtype, list(range(1, wmax + 1)), 4.0, device=DEV)
        ws = torch.empty(bs.workspace_bytes(max(lengths)), dtype=torch.uint8, device=DEV)
        rec, msds, a = [], [], 0
        for k, n in enumerate(lengths + [0]):
            out = torch.empty((cap, 4), dtype=torch.int32, device=DEV)
            res = torch.empty(16, dtype=torch.uint8, device=DEV)
            msd = torch.empty(40, dtype=torch.uint8, device=DEV)
            if n:
                flat = torch.full((first + n_dm * (n + pad),), 99.0, dtype=dtype, device=DEV)
                rows = flat[first:].view(n_dm, n + pad)
                rows[:, :n] = x[:, a:a + n]
                if host:
                    rows = flat.cpu().pin_memory()[first:].view(n_dm, n + pad)
                bs.push(rows, out, cap, res, ws, msd_out=msd, n_samp=n)
                msds.append(msd.cpu().numpy().tobytes())
                a += n
            else:
                bs.flush(out, cap, res, ws)
            count, status = spd.read_result(res)
            assert status == 0 and count <= cap
            rec.append(np.sort(spd.candidates_to_numpy(out, count), order=["dm", "sample"]))
        got.append((rec, msds))
    assert sum(r.size for r in got[0][0]) and got[0][1] == got[1][1]
    for p, q in zip(got[0][0], got[1][0]):
        assert np.array_equal(p, q)
