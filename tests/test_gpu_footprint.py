"""The server's estimate of an analysis' device memory against what its context takes."""
import pytest

import gwinputs as gi
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name,over,coarse", [("c4", {"N": 300000, "df": 1 / 256, "n_det": 3}, 0),
                                              ("c4", {"N": 400000, "df": 1 / 256, "n_det": 1}, 0),
                                              ("c2", {"N": 300000, "df": 1 / 256, "n_det": 4}, 0),
                                              ("c2", {"N": 200000, "df": 1 / 8, "n_det": 2}, 0),
                                              ("c4", {"N": 300000, "df": 1 / 256, "n_det": 3}, 400)])
def test_estimate_covers_the_context(gw, name, over, coarse, precision):
    """From what one running analysis takes from the device's free memory: the estimate is no
    smaller (up to the 2 MB granules of some 40 buffers) and at most 1.6 times as large (node rows are
    counted at their largest)."""
    import torch
    w = gi.workload(name, n_live=16, k=8, **over)
    pb, th = oracle.make_problem(w)
    args = dict(kind=pb.kind, lo=pb.lo, hi=pb.hi, data=pb.data(), psd=pb.psd, f0=pb.f0, df=pb.df, pos=pb.pos,
                xarm=pb.xarm, yarm=pb.yarm, n_live=16, k=8, steps_per_dim=1, dlogz_stop=-1.0, seed=1)
    if coarse:
        args.update(coarse_bins=coarse, theta_fid=th)
    with gw.Server(precision=precision, max_iter=1000) as srv:
        first = srv.submit(**args)       # loads the kernels, and makes the server's own buffers
        srv.tick()
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        rid = srv.submit(**args)
        srv.tick()
        torch.cuda.synchronize()
        taken = free - torch.cuda.mem_get_info()[0]
        st = srv.poll(rid)
        assert st["state"] == gw.NS_REQ_RUNNING
        srv.cancel(rid)
        srv.cancel(first)
    assert taken > 40e6
    assert taken - 40e6 <= st["footprint"] <= 1.6 * taken, (taken, st["footprint"])
