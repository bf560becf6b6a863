"""Memory of jz_adjoint_step: what it may take, and what it does when it cannot have it."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2003_08746_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def jz():
    from paper_2003_08746_gb300 import build, jz as J
    build.build()
    J.load()
    assert torch.cuda.is_available()
    return J


def _solver(jz, shape, form="FP64PAIR"):
    g, prm = W.jet_grid(*shape), W.jet_params(seed=4)
    z = dict(base_u=(0, 0, 0))
    q = W.jet_state(g) + W.random_state(g, seed=3, amp=1e-3, **z) - W.random_state(g, seed=3, amp=0.0, **z)
    grid = jz.Grid.from_workload(g)
    s = jz.Solver(grid, prm, getattr(jz, "JZ_PREC_" + form))
    s.set_state(q, 0.0)
    return grid, s, np.asarray(prm.forcing_amp)


# runs whose states no device holds (the counts at the end of an int's range): an error, and the solver goes on
@pytest.mark.parametrize("every", [1, 2**30, 2**31 - 1])
def test_more_steps_than_memory(jz, every):
    grid, s, A = _solver(jz, (24, 16, 8))
    J0, g0 = jz.jz_adjoint_step(s.h, A, 4, 2, 0.75)
    with pytest.raises(jz.JzError) as e:
        jz.jz_adjoint_step(s.h, A, 2**31 - 1, every, 0.75)
    assert e.value.code == jz.JZ_ERR_OOM
    J, g = jz.jz_adjoint_step(s.h, A, 4, every, 0.75)
    # sums with atomics, as between checkpoint intervals
    assert abs(J - J0) <= 1e-12 * abs(J0) and np.abs(g - g0).max() <= 1e-12 * np.abs(g0).max()
    s.close()
    grid.close()


SHAPE = (128, 96, 64)
STATE = 5 * 8 * 132 * 100 * 68                       # bytes of one padded state


def _gradient(jz, s, A, n, every):
    """J, dJ/dA and the forward stages advanced for them (launches of the kernel with the face fluxes)."""
    launches = (ctypes.c_longlong * 10)()
    jz.load().jz_profile_read(s.h, None, launches)
    J, g = jz.jz_adjoint_step(s.h, A, n, every, 0.75)
    jz.load().jz_profile_read(s.h, None, launches)
    return J, g, launches[2]


# the three ways to the stage states, the last segment shorter than the others: all kept, kept per segment
# (segments but the last advanced twice), four stages of every step once more
@pytest.mark.parametrize("form", ["FP64", "FP64PAIR"])
def test_ways_to_the_stage_states(jz, form):
    grid, s, A = _solver(jz, SHAPE, form)
    n, every = 7, 3
    torch.cuda.empty_cache()
    J0, g0, stages = _gradient(jz, s, A, n, every)
    assert stages == 5 * n
    # free memory left: 32 times less than all the states; room for the segment's states, its stage states over half of it
    for leave, expect in ((300 * STATE, 5 * n + 5 * 6), (27 * STATE, 5 * n + 5 * 6 + 4 * n)):
        hold = torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")
        J, g, stages = _gradient(jz, s, A, n, every)
        del hold
        torch.cuda.empty_cache()
        assert stages == expect
        # sums with atomics, as between checkpoint intervals
        assert abs(J - J0) <= 1e-12 * abs(J0) and np.abs(g - g0).max() <= 1e-12 * np.abs(g0).max()
    s.close()
    grid.close()


# more states than 1/32 of the free memory holds: the caller's interval decides (a program may allocate beside the call)
def test_interval_bounds_memory(jz):
    grid, s, A = _solver(jz, SHAPE)
    torch.cuda.empty_cache()
    n, every = torch.cuda.mem_get_info()[0] // 32 // (5 * STATE) + 1, 4
    _, _, stages = _gradient(jz, s, A, n, every)
    assert stages == 5 * n + 5 * ((n - 1) // every * every)
    s.close()
    grid.close()
