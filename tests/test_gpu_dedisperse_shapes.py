"""De-dispersion in each shape of CTA (by the plane's size) against the FP64
oracle: pairs of channels summed by delay differences, channels one by one,
rows at any element step, and 16-bit storage with scale and offset."""
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


def _delays(kind, n_dm, n_chan, rs):
    if kind == "plasma":      # neighbouring trials: few differences per pair
        return synth.dispersion_delays(n_chan, np.linspace(0, 60, n_dm))
    if kind == "random":      # no two trials alike
        return rs.integers(0, 700, (n_dm, n_chan)).astype(np.int32)
    d = rs.integers(0, 40, (n_dm, n_chan)).astype(np.int32)     # "mixed"
    d[:, ::3] = 7             # some channels without spread
    d[:, 5] = rs.integers(0, 1500, n_dm)     # one wider than a staged window
    return d


@pytest.mark.parametrize("n_out,n_dm", [
    (20481, 245),     # 4 outputs of 16 trials per thread
    (10300, 243),     # 2 of 16
    (1500, 19),       # 1 of 4
])
@pytest.mark.parametrize("kind", ["plasma", "random", "mixed"])
@pytest.mark.parametrize("dtype,first,pad", [("f32", 0, 0), ("f32", 1, 3), ("f16", 0, 0),
                                             ("bf16", 3, 5)])
def test_shapes_match_the_oracle(spd, n_out, n_dm, kind, dtype, first, pad):
    n_chan = 131 if n_dm < 20 else 17        # over one chunk of channels; odd
    rs = np.random.default_rng([n_out, n_chan, len(kind)])
    d = _delays(kind, n_dm, n_chan, rs)
    n = n_out + int(d.max())
    x = synth.noise_plane(n_chan, n, mean=1.0, device=DEV, seed=n)
    scale = offset = None
    if dtype != "f32":
        q = synth.quantise_rows(synth.SynthPlane(x, n), dtype)
        x, scale = q.data, q.scale
        offset = torch.linspace(-1, 1, n_chan, device=DEV)
    # rows `pad` elements apart, the first one `first` elements into the buffer
    flat = torch.full((first + n_chan * (n + pad) + 8,), float("nan"), dtype=x.dtype, device=DEV)
    rows = flat[first:first + n_chan * (n + pad)].view(n_chan, n + pad)
    rows[:, :n] = x
    out = torch.full((n_dm, n_out + 3), 7.0, device=DEV)
    spd.dedisperse(spd.Plane(rows, n_samp=n, scale=scale, offset=offset),
                   torch.from_numpy(d).to(DEV), n_out, out=out)
    got = out.cpu().numpy().astype(np.float64)
    assert (got[:, n_out:] == 7.0).all()
    op = oracle.Plane(synth.to_host_numpy(x), dtype=dtype,
                      scale=None if scale is None else scale.cpu().numpy(),
                      offset=None if offset is None else offset.cpu().numpy())
    want = oracle.dedisperse(op, d, n_out)
    mag = oracle.dedisperse(oracle.Plane(np.abs(op.values()).astype(np.float32)), d, n_out)
    # FP32 sums: a few ulp of the running magnitude per channel
    assert np.all(np.abs(got[:, :n_out] - want) <= 2e-7 * n_chan * mag + 1e-30)
