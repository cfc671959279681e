"""Tables rebuilt in place by set_data, and node tiles against the library's own bin-by-bin sums."""
import numpy as np
import pytest

import gwinputs as gi
from test_gpu_parity import problem, sampler_from

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name,over,coarse", [("c1", {}, 0), ("c1", {"N": 20001, "df": 1 / 32}, 0),
                                              ("c4", {"N": 60001, "df": 1 / 256}, 0),
                                              ("c4", {"N": 60001, "df": 1 / 256}, 200)])
def test_set_data_equals_a_fresh_sampler(gw, name, over, coarse, precision):
    """Data of other amplitudes (detector by detector from 1e-3 to 1e3 of the first), then the first again: scales,
    weights, every level of node weights and the coarse bins' summary data are those of a sampler made with them."""
    w, pb, th = problem(name, **over)
    rb = dict(coarse_bins=coarse, theta_fid=th) if coarse else {}
    a = pb.data()
    b = np.roll(a, 11, axis=1) * np.geomspace(1e-3, 1e3, a.shape[0])[:, None]
    u = gi.unit_cube(5, 200, pb.dim)
    with sampler_from(gw, pb, precision, n_live=8, **rb) as sp:
        first = sp.eval_lnl(u)
        sp.set_data(b)
        second = sp.eval_lnl(u)
        live_u, live_logl = sp.live()
        sp.set_data(a)
        assert np.array_equal(sp.eval_lnl(u), first)
    with sampler_from(gw, pb, precision, n_live=8, data=b, **rb) as sp:
        assert np.array_equal(sp.eval_lnl(u), second)
        assert np.array_equal(sp.eval_lnl(live_u), live_logl)
    assert not np.any(first == second)


@pytest.mark.parametrize("name,over,rms", [("c1", {"N": 20001, "df": 1 / 32}, 1.3e-14), ("c2", {}, 1.3e-14),
                                           ("c4", {"N": 60001, "df": 1 / 256}, 1e-12),
                                           ("c4", {"N": 200001, "df": 1 / 256, "n_det": 4}, 1e-12)])
def test_tiles_against_bins(gw, name, over, rms):
    """The same points in a sampler whose t_c prior lies elsewhere, outside whose tiles' box they are summed
    bin by bin. The bin sums' error is some 1.3e-14 (chirp masses of 10 or more) or 1e-12 (1.1 or more) of the weights'
    norm over draws (test_fx_blocks.py's ranges); times |G_d| that norm is sqrt(2 <h|h>) for noise alone, and a
    signal adds at most |<d|h>|. Two sums, five standard deviations; the tiles' interpolation adds 1e-15."""
    import torch
    w, pb, th = problem(name, **over)
    theta = np.concatenate([pb.theta(gi.unit_cube(6, 100, pb.dim)), th[None]])
    t = torch.tensor(theta, device="cuda")
    lo, hi = pb.lo.copy(), pb.hi.copy()
    lo[gi.P_TC] += 10.0
    hi[gi.P_TC] += 10.0
    with sampler_from(gw, pb, 0, n_live=8) as tiles, sampler_from(gw, pb, 0, n_live=8, lo=lo, hi=hi) as bins:
        a, b = tiles.eval_lnl_theta(t).cpu().numpy(), bins.eval_lnl_theta(t).cpu().numpy()
    hh = np.array([pb.snr2(x) for x in theta])
    assert np.all(np.abs(a - b) <= 5.0 * np.sqrt(2.0) * rms * (np.sqrt(2.0 * hh) + np.abs(b + 0.5 * hh)))
    assert np.count_nonzero(a != b) > 50       # the tiles were taken
