"""Memory of jz_adjoint_step: what it may take, and what it does when it cannot have it."""
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
