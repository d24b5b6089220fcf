"""De-dispersion where a block of trials is not full, in each shape of CTA, and
the middle shape between its limits: against the FP64 oracle, with channels read
from shared and from global memory."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def spd():
    import paper_1611_09704_gb300 as m
    m.build()
    m.load()
    return m


@pytest.mark.parametrize("n_out,n_dm", [
    (160000, 3),      # 4 outputs of 16 trials per thread, 3 of them there
    (52000, 33),      # the last block's one trial
    (8200, 243),      # 2 of 16
    (30000, 17),      # and one trial
    (1500, 5),        # 1 of 4, and one
])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_blocks_that_are_not_full(spd, n_out, n_dm, dtype):
    n_chan = 11
    rs = np.random.default_rng([n_out, n_dm])
    d = np.sort(rs.integers(0, 60, (n_dm, n_chan)), axis=0).astype(np.int32)
    d[:, 3] = rs.integers(0, 700, n_dm)          # no two differences alike
    d[:, 6] = rs.integers(0, 5000, n_dm)         # wider than a staged window
    n = n_out + int(d.max())
    x = synth.noise_plane(n_chan, n, mean=1.0, device=DEV, seed=n)
    scale = None
    if dtype != "f32":
        q = synth.quantise_rows(synth.SynthPlane(x, n), dtype)
        x, scale = q.data, q.scale
    out = torch.full((n_dm + 1, n_out + 1), 7.0, device=DEV)
    spd.dedisperse(spd.Plane(x, scale=scale), torch.from_numpy(d).to(DEV), n_out, out=out[:n_dm])
    got = out.cpu().numpy().astype(np.float64)
    assert (got[n_dm] == 7.0).all() and (got[:, n_out] == 7.0).all()
    op = oracle.Plane(synth.to_host_numpy(x), dtype=dtype,
                      scale=None if scale is None else scale.cpu().numpy())
    want = oracle.dedisperse(op, d, n_out)
    mag = oracle.dedisperse(oracle.Plane(np.abs(op.values()).astype(np.float32)), d, n_out)
    # FP32 sums: a few ulp of the running magnitude per channel
    assert np.all(np.abs(got[:n_dm, :n_out] - want) <= 2e-7 * n_chan * mag + 1e-30)
