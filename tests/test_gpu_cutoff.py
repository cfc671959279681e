"""The cutoff index (the last bin at or below f_ISCO) on grids whose frequencies are
many bins from zero, where a single-precision frequency spans several bins."""
import math

import numpy as np
import pytest

import gwinputs as gi
import oracle
from test_gpu_parity import FP64_RTOL, MIXED_ATOL, sampler_from

pytestmark = pytest.mark.gpu


def narrow_band(f0, df, N):
    """One ideal detector, noise of unit weight per bin, chirp masses whose f_ISCO lies about f0."""
    kind, lo, hi = gi._prior_11(mc=(0.5, 60.0))
    f = f0 + np.arange(N) * df
    psd = np.ones((1, N))
    data = gi.noise(3, psd, df) * 1e-2
    lo[gi.P_DL], hi[gi.P_DL] = 1.0, 2.0
    return oracle.Problem(f0=f0, df=df, psd=psd, data=data, ideal=True, kind=kind, lo=lo, hi=hi), f


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("f0,df,N", [(1000.0, 1e-6, 4001), (300.0, 1e-6, 4001), (1500.0, 2.0 ** -20, 4001),
                                     (2000.0, 2.0 ** -10, 4001), (20.0, 2.0 ** -9, 1 << 20)])
def test_cutoff_index(gw, f0, df, N, precision):
    """f_ISCO between two bins: about the first, the last and random ones."""
    import torch
    pb, f = narrow_band(f0, df, N)
    rng = np.random.default_rng(1)
    js = np.concatenate([[-1, 0, 1, N - 3, N - 2, N - 1], rng.integers(0, N, 60)])
    th = np.zeros((js.size, gi.NPARAM))
    th[:, gi.P_Q], th[:, gi.P_COSI], th[:, gi.P_TC] = 0.8, 0.3, 0.01
    eta = 0.8 / 1.8 ** 2
    fisco = f0 + (js + rng.uniform(0.2, 0.8, js.size)) * df
    th[:, gi.P_MC] = eta ** 0.6 / (6.0 ** 1.5 * math.pi * 4.925490947641267e-6 * fisco)
    # a distance that puts the largest <h|h> at 100
    th[:, gi.P_DL] = 1.0
    th[:, gi.P_DL] = math.sqrt(max(pb.snr2(t) for t in th[:30])) / 10.0
    want = pb.loglike_theta(th)
    assert np.ptp(want) > 1.0
    with sampler_from(gw, pb, precision, n_live=8) as sp:
        got = sp.eval_lnl_theta(torch.tensor(th, device="cuda")).cpu().numpy()
    if precision == 0:
        assert np.max(np.abs(got - want) / np.maximum(1.0, np.abs(want))) < FP64_RTOL
    else:
        assert np.max(np.abs(got - want)) < MIXED_ATOL
