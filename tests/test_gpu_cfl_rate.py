"""The first FP32-flux step's time step where FP32 cannot bound a node's rate: metrics whose squares
are subnormal, dropped or infinite, reciprocal volumes beyond FP32, a node of negative pressure.

The node of the largest rate stands where a false bound of another node, or of its own, would leave it
out: late in the sweep (the warps take a second turn of 32 nodes by then) and beside nodes of the other
kind.  Bar: a metric is a difference of products of coordinates up to 160 cells across, about ten
roundings of 160 x 1.1e-16 each on either side, so 1e-12 relative on dt."""
import ctypes
import math

import numpy as np
import pytest
import torch

from oracle import jz_oracle as O
from paper_2003_08746_gb300 import workloads as W
from parity import oracle_grid

pytestmark = pytest.mark.gpu

SHAPE = (64, 160, 66)                 # 21120 turns of 32 nodes for at most 9728 warps


@pytest.fixture(scope="module")
def jz():
    from paper_2003_08746_gb300 import build, jz as J
    build.build()
    J.load()
    assert torch.cuda.is_available()
    return J


def _grid(h, vary, flat):
    """Box of spacing h, h / flat along i; vary: along i the spacing goes over 0.9 .. 1.1 of that and back."""
    g = W.box_grid(*SHAPE, h=h)
    if vary:
        i = np.arange(SHAPE[0])
        g.xyz[0] += h * 0.1 * SHAPE[0] / (2 * math.pi) * np.sin(2 * math.pi * i / SHAPE[0])
    g.xyz[0] /= flat
    g.period[0] /= flat
    return g


# spacing, uneven or not, flat cells, i of the fastest node and its sound speed; a node of negative pressure beside it or not
CASES = {
    "subnormal squares": (1e-11, False, 1, 40, 1.0047, False),
    "squares dropped": (1e-12, False, 1, 40, 1.0047, False),
    "volumes about 1 / FLT_MAX": ((350 / 3.4028e38) ** (1.0 / 3.0), True, 350, 4, 1.5, False),
    "squares about FLT_MAX": (0.98 * 3.4028e38 ** 0.25, True, 1, 33, 1.2, False),
    "negative pressure": (0.2, False, 1, 40, 1.2, True),
}


@pytest.mark.parametrize("case", list(CASES))
def test_first_step_rate_beyond_fp32(jz, case):
    h, vary, flat, i, a, negative = CASES[case]
    g, prm = _grid(h, vary, flat), W.box_params()
    q = W.random_state(g, seed=1, amp=0.0)
    j, k = 150, 60
    q[4, k, j, i] += (a * a - 1.0) / (1.4 * 0.4)              # p = a^2 / gamma at rho = 1
    if negative:
        q[:, k, j, i + 1] = (1.0, 8.0, 0.0, 0.0, 0.9 * 32.0)
    c, og = O.Consts(prm), oracle_grid(g)
    _, u, v, w, _, T = O.primitives(og.pad(torch.from_numpy(q)), c)
    lam = O.spectral_radii(og, u, v, w, T)
    rate = O.real((lam[0] + lam[1] + lam[2]) * og.invV)
    best = np.nanmax(rate.numpy())                            # a node without a real sound speed has no rate
    assert rate[k, j, i].item() == best
    grid = jz.Grid.from_workload(g)
    s = jz.Solver(grid, prm, jz.JZ_PREC_FP32FLUX)
    s.set_state(q, 0.0)
    s.step(1, False)
    # the time after the step: FP32 fluxes cannot carry such cells, so the state's own check may report
    # it (the figures are filled in all the same)
    st = jz.jz_step_stats()
    rc = jz.load().jz_rk_step(s.h, 0, ctypes.byref(st))
    s.close()
    grid.close()
    assert rc in (jz.JZ_OK, jz.JZ_ERR_NONFINITE)
    assert abs(st.t * best / c.cfl - 1.0) <= 1e-12, st.t * best / c.cfl
