"""Sizes and parameters at the edges of the kernels' tiles, roles and rules, against the oracle.

Bars: the state after a few steps is held to the forms' bars (1e-12 relative L2 for the FP64 and
pair forms, 1e-5 for the FP32-flux form); a time step is one division of an FP64 rate, a maximum
of sums of a dozen FP64 operations, so 1e-13."""
import ctypes
import dataclasses

import numpy as np
import pytest
import torch

from oracle import jz_oracle as O
from paper_2003_08746_gb300 import workloads as W
from parity import field_errors, oracle_grid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def jz():
    from paper_2003_08746_gb300 import build, jz as J
    build.build()
    J.load()
    assert torch.cuda.is_available()
    return J


def _noise(g, seed, amp):
    z = dict(base_u=(0, 0, 0))
    return W.random_state(g, seed=seed, amp=amp, **z) - W.random_state(g, seed=seed, amp=0.0, **z)


def _against_oracle(jz, g, q, prm, form, nsteps, tol):
    grid = jz.Grid.from_workload(g)
    s = jz.Solver(grid, prm, form)
    s.set_state(q, 0.1)
    st = s.step(nsteps)
    ref, t, dts, _ = O.run(oracle_grid(g), torch.from_numpy(q), O.Consts(prm), nsteps, t0=0.1)
    e2, _ = field_errors(s.get_state(), ref.numpy())
    s.close()
    grid.close()
    assert e2.max() <= tol, e2
    return st, t, dts


# whole (5, 3) and fractional exponents of the isentropes; the smallest jets (every azimuthal image
# of a node is a ghost, the far field two rows from the axis), odd extents, more than one block per role
@pytest.mark.parametrize("gamma", [1.4, 5.0 / 3.0, 1.3])
@pytest.mark.parametrize("shape", [(4, 4, 4), (5, 4, 6), (9, 19, 20), (131, 6, 4)])
@pytest.mark.parametrize("form,tol", [("FP64", 1e-12), ("FP64PAIR", 1e-12), ("FP32FLUX", 1e-5)])
def test_jet_boundaries_and_ghosts(jz, shape, gamma, form, tol):
    g = W.jet_grid(*shape)
    prm = dataclasses.replace(W.jet_params(seed=3), gamma=gamma)
    q = W.jet_state(g, gamma=gamma) + _noise(g, 7, 2e-3)
    _against_oracle(jz, g, q, prm, getattr(jz, "JZ_PREC_" + form), 3, tol)


# tile edges of the marching pair kernels (30 and 31 nodes along i, 8 and 7 along j) and the chunks
# along k, down to one plane
@pytest.mark.parametrize("shape", [(28, 6, 1), (29, 7, 2), (30, 8, 3), (31, 9, 33), (32, 15, 5), (61, 16, 4), (63, 22, 34)])
def test_pair_tiles(jz, shape):
    g = W.box_grid(*shape, h=0.21)
    _against_oracle(jz, g, W.random_state(g, seed=9, amp=0.05), W.box_params(), jz.JZ_PREC_FP64PAIR, 2, 1e-12)


# a box's update writes its ghosts: extents under two (several images of a node along an axis), and
# blocks and chunks that hold one edge, both or none
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 1, 3), (3, 5, 2), (4, 2, 1), (1, 40, 3), (37, 3, 12), (5, 17, 70)])
@pytest.mark.parametrize("form", ["FP64", "FP64PAIR"])
def test_box_ghosts(jz, shape, form):
    g = W.box_grid(*shape, h=0.21)
    st, t, _ = _against_oracle(jz, g, W.random_state(g, seed=4, amp=0.05), W.box_params(), getattr(jz, "JZ_PREC_" + form), 3,
                               1e-12)
    assert abs(st.t - t) <= 1e-12 * t


# the first FP32-flux step's rate: its maximum anywhere in a turn of 32 nodes, ties everywhere,
# supersonic flow (pressure the small rest of e), and cells too small for FP32 bounds
@pytest.mark.parametrize("case", ["noise", "uniform", "hypersonic", "tiny", "jet", "one"])
def test_first_step_rate(jz, case):
    if case == "jet":
        g, prm = W.jet_grid(67, 21, 10), W.jet_params(seed=2)
        q = W.jet_state(g) + _noise(g, 5, 2e-3)
    else:
        shape = (1, 1, 1) if case == "one" else (65, 9, 7)
        g, prm = W.box_grid(*shape, h=1e-14 if case == "tiny" else 0.2), W.box_params()
        u = (25.0, 0.3, -0.2) if case == "hypersonic" else (0.3, 0.1, -0.1)
        q = W.random_state(g, seed=6, amp=0.0 if case == "uniform" else 0.02, base_u=u)
    og = oracle_grid(g)
    dt = O.cfl_dt(og, torch.from_numpy(q), O.Consts(prm)).item()
    grid = jz.Grid.from_workload(g)
    s = jz.Solver(grid, prm, jz.JZ_PREC_FP32FLUX)
    s.set_state(q, 0.0)
    s.step(1, False)
    # the time after the step; FP32 fluxes cannot carry the tiny cells, so the state's own check may
    # report that one (the figures are filled in all the same)
    st = jz.jz_step_stats()
    rc = jz.load().jz_rk_step(s.h, 0, ctypes.byref(st))
    s.close()
    grid.close()
    assert rc == jz.JZ_OK or (case == "tiny" and rc == jz.JZ_ERR_NONFINITE)
    assert abs(st.t - dt) <= 1e-13 * dt


# the adjoint's three ways to the stage states: all kept, kept per checkpoint segment, recomputed; which
# one is taken depends on the free memory, the gradient does not (sums with atomics: 1e-12, as between
# checkpoint intervals)
def test_adjoint_with_little_memory(jz):
    g, prm = W.jet_grid(128, 96, 64), W.jet_params(seed=4)
    grid = jz.Grid.from_workload(g)
    s = jz.Solver(grid, prm, jz.JZ_PREC_FP64PAIR)
    s.set_state(W.jet_state(g) + _noise(g, 3, 1e-3), 0.0)
    A = np.asarray(prm.forcing_amp)
    state = 5 * 8 * 132 * 100 * 68                                # bytes of one padded state
    base = (10 + 5 + 3 * 12 + 2) * state // 5                     # the adjoint arrays
    n, ck = 12, 4
    torch.cuda.empty_cache()
    J0, g0 = jz.jz_adjoint_step(s.h, A, n, ck, 0.75)              # all kept
    for leave in (base + (n * 5 + 4) * state, base + 20 * state):  # not twice all; not twice a segment's
        free = torch.cuda.mem_get_info()[0]
        hold = torch.empty(int(free - leave), dtype=torch.uint8, device="cuda")
        J, gr = jz.jz_adjoint_step(s.h, A, n, ck, 0.75)
        del hold
        torch.cuda.empty_cache()
        assert abs(J - J0) <= 1e-12 * abs(J0)
        assert np.abs(gr - g0).max() <= 1e-12 * np.abs(g0).max()
    s.close()
    grid.close()


# copies in and out, whole and with part of a warp to a row: a copy is exact
@pytest.mark.parametrize("ni", [1, 2, 3, 8, 9, 17, 31, 32, 33, 67])
@pytest.mark.parametrize("form", ["FP64PAIR", "FP32FLUX"])
def test_state_round_trip(jz, ni, form):
    g = W.box_grid(ni, 7, 5, h=0.2)
    q = W.random_state(g, seed=ni, amp=0.05)
    grid = jz.Grid.from_workload(g)
    s = jz.Solver(grid, W.box_params(), getattr(jz, "JZ_PREC_" + form))
    s.set_state(q, 0.0)
    assert np.array_equal(s.get_state(), q)
    s.close()
    grid.close()
