"""FP64 form on the GPU at the sizes where its tiles, segments and coarse-bin
passes can go wrong, against the oracle; tolerance as in the parity tests (1e-9
of max(|log L|, 1): phases of up to 1.4e4 rad rounded at 1e-16 each)."""
import math

import numpy as np
import pytest

import gwinputs as gi
import oracle
from test_gpu_parity import FP64_RTOL, problem, pts_for, sampler_from

pytestmark = pytest.mark.gpu


def close(got, want):
    return np.max(np.abs(got - want) / np.maximum(1.0, np.abs(want))) < FP64_RTOL


def ending_at(pb, base, j):
    """Parameters whose f_ISCO lies 0.3 of a bin above grid frequency j."""
    t = base.copy()
    eta = t[gi.P_Q] / (1 + t[gi.P_Q]) ** 2
    f = pb.f0 + (j + 0.3) * pb.df
    t[gi.P_MC] = eta ** 0.6 / (6.0 ** 1.5 * math.pi * 4.925490947641267e-6 * f)
    return t


@pytest.mark.parametrize("n_det", [1, 2, 3, 4])
def test_cutoffs_about_tile_edges(gw, n_det):
    """Cutoffs one bin either side of multiples of every tile length, at a tile's
    last and first bins, at the grid's ends; inside the prior and (masses below 10
    or above 40, t_c beyond 0.1 s) outside the tiles' box."""
    import torch
    w, pb, th = problem("c1", N=20001, df=1 / 32, n_det=n_det)
    js = [-1, 0, 1] + [m + o for m in (64, 640, 1024, 1536, 2048, 3072, 4096, 8192) for o in (-2, -1, 0, 1, 63, 64)]
    theta = [ending_at(pb, th, j) for j in js] + [th.copy()]
    for t in list(theta[::7]):
        t2 = t.copy()
        t2[gi.P_TC] = 0.35
        theta.append(t2)
    theta = np.array(theta)
    want = pb.loglike_theta(theta)
    with sampler_from(gw, pb, 0, n_live=8) as sp:
        got = sp.eval_lnl_theta(torch.tensor(theta, device="cuda")).cpu().numpy()
        u = pts_for(pb, th, count=61)
        assert close(sp.eval_lnl(u), pb.loglike(u))
        # outside the unit cube
        u = gi.unit_cube(5, 7, pb.dim) * 0.2 + 1.01
        u[:, 1] = 0.5       # the mass ratio stays below 1
        u[:, 10] = 0.5      # and the sine of the declination
        assert close(sp.eval_lnl(u), pb.loglike(u))
    assert close(got, want)


@pytest.mark.parametrize("over,cutoff", [({"N": 4097, "df": 1 / 256}, True), ({"N": 60001, "df": 1 / 256}, True),
                                         ({"N": 60001, "df": 1 / 256}, False), ({"N": 16384, "df": 1 / 64}, False)])
def test_low_mass_grids(gw, over, cutoff):
    w, pb, th = problem("c4", **over)
    if not cutoff:
        pb, th = oracle.make_problem(gi.workload("c4", **over), cutoff=False)
    u = pts_for(pb, th, count=16)
    with sampler_from(gw, pb, 0, n_live=8) as sp:
        assert close(sp.eval_lnl(u), pb.loglike(u))


def test_batch_sizes_and_nan(gw):
    """One to a few thousand points give the same values in every batch; a NaN coordinate gives NaN
    for its point alone."""
    w, pb, th = problem("c1", N=20001, df=1 / 32)
    u = gi.unit_cube(3, 2500, pb.dim)
    with sampler_from(gw, pb, 0, n_live=8) as sp:
        full = sp.eval_lnl(u)
        for m in (1, 2, 3, 5, 64, 305, 609, 1217):
            assert np.array_equal(sp.eval_lnl(u[:m]), full[:m])
        v = u[:9].copy()
        v[4, 7] = np.nan
        got = sp.eval_lnl(v)
    assert np.isnan(got[4]) and np.array_equal(np.delete(got, 4), np.delete(full[:9], 4))


@pytest.mark.parametrize("bins", [1, 2, 30, 31, 32, 62, 63, 95, 700])
@pytest.mark.parametrize("n_det", [1, 3, 4])
def test_coarse_bin_counts(gw, bins, n_det):
    """Passes of 31 coarse bins: counts about their multiples, cutoffs among them."""
    w, pb, th = problem("c1", n_det=n_det)
    rb = oracle.RelativeBinning(pb, th, B=bins)
    u = pts_for(pb, th, count=33)
    with sampler_from(gw, pb, 0, n_live=8, coarse_bins=bins, theta_fid=th) as sp:
        assert close(sp.eval_lnl(u), rb.loglike(u))
