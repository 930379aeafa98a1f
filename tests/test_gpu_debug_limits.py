"""The bounds-checked build's checks themselves: with a limit set below a buffer's size (the buffer is as large
as ever, so nothing is at risk), every kind of access of the strip and the tile kernels beyond it is
reported as ROEAM_E_BOUNDS: the source, U^n, the result, and residuals into the state's layout and into
the allocation-free call's scratch. (In a child process: a process loads one libroeam.)"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r'''
import ctypes as C
import sys
import numpy as np
sys.path.insert(0, ROOT); sys.path.insert(0, ROOT + "/tests")
from paper_1711_09272_gb300 import build, roeam as R
lib = R.load_library(build.build(debug=True))
import workloads as W

SRC, UN, DST = range(3)
def spec(ni, nj):
    return W.GridSpec(ni=ni, nj=nj, dx=0.1, dy=0.1, params=W.SchemeParams(m_ref=0.4))

def limit(b, buffer, n):
    lib.roeam_debug_limit(C.c_void_p(b.handle), C.c_int(buffer), C.c_longlong(n))

def refused(b, call):
    try:
        call()
        b.check()
    except R.RoeamError as e:
        assert e.status == R.ROEAM_E_BOUNDS, e
        return True
    return False

checked = 0
for prec in (64, 32):
    for count in (1, 2):
        specs = [spec(40, 30), spec(33, 21)][:count]
        with R.Batch(specs, precision=prec) as b:
            b.set_states([W.random_smooth_state(s, seed=3, mach=0.3) for s in specs])
            out = np.empty((4, specs[-1].nj, specs[-1].ni))
            step = lambda: b.step(dt_fixed=1e-4, nsteps=1)
            stages = lambda: [b.stage(s, 1e-4) for s in range(3)]
            residual = lambda: R.roeam_flux_residual(b.handle, count - 1, None)
            noalloc = lambda: R.roeam_flux_residual_noalloc(b.handle, count - 1, out)
            norm = lambda: b.residual_norm(count - 1)
            cells = sum(64 * s.nj for s in specs)          # pitched rows of 64 cells of four values
            last = 4 * cells - 4 * 64 * 3                  # all but the last three rows
            room = 4 * 64 * (specs[-1].nj - 3)             # of the scratch: the same of one grid
            cases = [(SRC, last, step), (DST, last, step), (SRC, last, stages), (UN, last, stages), (DST, last, stages),
                     (SRC, last, residual), (DST, last, residual), (SRC, last, noalloc), (DST, room, noalloc), (SRC, last, norm)]
            if prec == 64:                                 # (FP32 steps in rectangles hold U^n on chip)
                cases.append((UN, last, step))
            for buffer, n, call in cases:
                limit(b, buffer, n)
                assert refused(b, call), (prec, count, buffer, call)
                limit(b, buffer, -1)
                b.set_states([W.random_smooth_state(s, seed=3, mach=0.3) for s in specs])
                assert not refused(b, call), (prec, count, buffer, call)
                checked += 1
print("limits ok", checked)
'''


def test_every_access_is_checked():
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + SCRIPT], cwd=ROOT, capture_output=True,
                       text=True, timeout=1200)
    assert r.returncode == 0, (r.stdout[-2000:], r.stderr[-3000:])
    assert "limits ok" in r.stdout
