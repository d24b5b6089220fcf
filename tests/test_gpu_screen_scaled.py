"""The screen over ranges with and without a scale in one launch, at lists that
reach one, two and more than two rounds of blocks: the records of the search
without a screen, bit for bit."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("wmax", [32, 128, 300, 700])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_scaled_and_plain_ranges_share_a_launch(dtype, wmax):
    import paper_1611_09704_gb300 as spd
    spd.build()
    spd.load()
    specs = []
    for i, n_samp in enumerate((9000, 3776, 12344, 16)):
        p = synth.ska_like(4, n_samp, n_pulses=5, mean=3.0, sd=1.0, drift_amp=0.2,
                           drift_period=4000, device=DEV, seed=i).data
        x = p if dtype == "f32" else p.to(torch.float16)
        sc = {} if i % 2 == 0 else {"scale": torch.linspace(0.5, 2.0, 4, device=DEV)}
        specs.append(spd.RangeSpec(spd.Plane(x, **sc), list(range(1, wmax + 1)), 4.0,
                                   dm_offset=100 * i))
    need = spd.search_batched_workspace_bytes(specs)
    got = []
    for n in (need, need - 1):      # one byte short of the screen's piece: no screen
        ws = torch.zeros(need, dtype=torch.uint8, device=DEV)[:n]
        out, res, _ = spd.search_batched(specs, 1 << 20, workspace=ws)
        count, status = spd.read_result(res)
        assert status == 0
        got.append(np.sort(spd.candidates_to_numpy(out, count), order=["dm", "sample", "width"]))
    assert got[0].size and np.array_equal(got[0], got[1])
