"""A failed host allocation inside ns_init: the call reports NS_ERR_OOM and gives back
all device memory. A small library whose operator new throws once, when asked to,
stands in for a host without memory."""
import os
import shutil
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

SHIM = r"""
#include <cstdlib>
#include <new>
static std::size_t least = 0;
extern "C" void fail_next(std::size_t n) { least = n; }     // the next allocation of n bytes or more
extern "C" int armed() { return least != 0; }
void *operator new(std::size_t n) {
    if (least && n >= least) {
        least = 0;
        throw std::bad_alloc();
    }
    void *p = std::malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }
"""

PROGRAM = r"""
import ctypes, sys
shim = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
shim.fail_next.argtypes = [ctypes.c_size_t]
sys.path[:0] = [sys.argv[2], sys.argv[2] + "/tests"]
import torch
import paper_2509_24949_gb300 as g
from test_gpu_parity import problem, sampler_from
w, pb, th = problem("c1", N=20001, df=1 / 32, n_det=1)
sampler_from(g, pb, 0, n_live=8).close()
free = []
for i in range(41):
    shim.fail_next(150000)
    try:
        sampler_from(g, pb, 0, n_live=8).close()
    except g.GWNSError as e:
        assert "allocation" in str(e), e
    else:
        raise SystemExit("no failure reported")
    assert not shim.armed()
    torch.cuda.synchronize()
    free.append(torch.cuda.mem_get_info()[0])
print(free[0] - free[-1])
"""


def test_prior_draws_buffer(gw, tmp_path):
    """The draws that choose the node tiles: 1024 coefficient sets, 220 kB, on the device and the host.
    Forty failures would leave 8.8 MB behind."""
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "shim.cpp").write_text(SHIM)
    lib = str(tmp_path / "shim.so")
    subprocess.run([cxx, "-O1", "-shared", "-fPIC", "-o", lib, str(tmp_path / "shim.cpp")], check=True)
    r = subprocess.run([sys.executable, "-c", PROGRAM, lib, ROOT], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0, r.stdout + r.stderr
    assert int(r.stdout.split()[-1]) <= 4 << 20
