"""FP64 log likelihood on grids that start far below the band where the data weigh:
the leading phase term there exceeds the phases in the band by up to ten decades,
and a point's phases must not take their rounding from it. Against the oracle, at
the parity tests' 1e-9 of max(|log L|, 1); about an injection of SNR 30 log L passes
through zero, and <h|h>/2 (450) is its size. The oracle itself is within 2e-10 of
80-bit arithmetic on these inputs."""
import numpy as np
import pytest

import gwinputs as gi
from test_gpu_parity import FP64_RTOL, problem, sampler_from

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f0", [20.0, 5.0, 1.0, 0.1, 0.01])
@pytest.mark.parametrize("N,df", [(4095, 0.25), (16001, 1 / 16)])
def test_low_start(gw, f0, N, df):
    """Up to about 1 kHz, the second grid with tiles where it starts at 1 Hz or above."""
    import torch
    w, pb, th = problem("c4", f0=f0, N=N, df=df)
    near = np.tile(th, (24, 1))
    near[1:, gi.P_TC] += np.linspace(-1e-3, 1e-3, 23)
    near[1:, gi.P_PHIC] += np.linspace(-2.0, 2.0, 23)
    want = pb.loglike_theta(near)
    with sampler_from(gw, pb, 0, n_live=8) as sp:
        got = sp.eval_lnl_theta(torch.tensor(near, device="cuda")).cpu().numpy()
        assert np.max(np.abs(got - want)) < FP64_RTOL * 450.0
        if f0 >= 0.1:       # below, the oracle's own rounding reaches 1e-9 of prior draws' log L
            u = gi.unit_cube(11, 24, pb.dim)
            a, b = sp.eval_lnl(u), pb.loglike(u)
            assert np.max(np.abs(a - b) / np.maximum(1.0, np.abs(b))) < FP64_RTOL


@pytest.mark.parametrize("f0", [20.0, 1.0, 0.1])
def test_low_start_relative_binning(gw, f0):
    """The coarse bins' phases, differences from the fiducial point's, likewise."""
    import oracle
    w, pb, th = problem("c4", f0=f0, N=16001, df=1 / 16)
    rb = oracle.RelativeBinning(pb, th, B=300)
    u = gi.unit_cube(11, 24, pb.dim)
    want = rb.loglike(u)
    with sampler_from(gw, pb, 0, n_live=8, coarse_bins=300, theta_fid=th) as sp:
        got = sp.eval_lnl(u)
    assert np.max(np.abs(got - want) / np.maximum(1.0, np.abs(want))) < FP64_RTOL
