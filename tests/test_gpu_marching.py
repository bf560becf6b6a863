"""The marching kernels over several planes per thread block, with a shorter last chunk, against the
oracle: grids just large enough for the chunk rules of a 152-SM device to take more than one plane (the
shapes of test_gpu_edges.py take one).  Planes per block, remainder in brackets:

  shape        flux kernel  faces kernel  fused FP32-flux kernel
  33 x 17 x 99     2 (1)        1            2 (1)     (jet: 98 planes)
  60 x 16 x 131    3 (1)        1            2 (1)     whole tiles of 30 x 8
  61 x 17 x 131    3 (1)        1            4 (3)     one node into the next tile
  97 x 95 x 81     3 (2)        2 (1)        5 (1)
  97 x 95 x 149    5 (1)        3 (2)        7 (2)
  97 x 95 x 152    5 (4)        3 (2)        7 (5)

A box's step covers the update that writes its ghosts, a jet's the update followed by the boundary kernel,
the residual the output of the right-hand side.  Bars: the forms' own (state 1e-12 and 1e-5 relative L2,
residual 1e-11 and 2e-4)."""
import functools

import pytest
import torch

from oracle import jz_oracle as O
from paper_2003_08746_gb300 import workloads as W
from parity import field_errors, oracle_grid

pytestmark = pytest.mark.gpu

BARS = {"FP64PAIR": (1e-12, 1e-11), "FP32FLUX": (1e-5, 2e-4)}


@pytest.fixture(scope="module")
def jz():
    from paper_2003_08746_gb300 import build, jz as J
    build.build()
    J.load()
    assert torch.cuda.is_available()
    return J


@functools.lru_cache(maxsize=1)
def _reference(topology, shape):
    if topology == "box":
        g, prm = W.box_grid(*shape, h=0.21), W.box_params()
        q = W.random_state(g, seed=9, amp=0.05)
    else:
        g, prm = W.jet_grid(*shape), W.jet_params(seed=3)
        z = dict(base_u=(0, 0, 0))
        q = W.jet_state(g) + W.random_state(g, seed=7, amp=2e-3, **z) - W.random_state(g, seed=7, amp=0.0, **z)
    og, c, Q = oracle_grid(g), O.Consts(prm), torch.from_numpy(q)
    state, t, _, _ = O.run(og, Q, c, 2, t0=0.1)
    return g, prm, q, O.residual(og, Q, c).numpy(), state.numpy(), float(t)


@pytest.mark.parametrize("topology,shape", [
    ("box", (33, 17, 99)), ("box", (60, 16, 131)), ("box", (61, 17, 131)), ("box", (97, 95, 81)), ("box", (97, 95, 149)),
    ("jet", (33, 17, 98)), ("jet", (97, 95, 152))])
@pytest.mark.parametrize("form", ["FP64PAIR", "FP32FLUX"])
def test_planes_per_block(jz, topology, shape, form):
    g, prm, q, res, state, t = _reference(topology, shape)
    bar_state, bar_res = BARS[form]
    grid = jz.Grid.from_workload(g)
    s = jz.Solver(grid, prm, getattr(jz, "JZ_PREC_" + form))
    e_res, _ = field_errors(s.residual(q), res)
    s.set_state(q, 0.1)
    st = s.step(2)
    e_state, _ = field_errors(s.get_state(), state)
    s.close()
    grid.close()
    print(f"{topology} {shape} {form}: residual {e_res.max():.2e}, state {e_state.max():.2e}")
    assert e_state.max() <= bar_state, e_state
    assert e_res.max() <= bar_res, e_res
    assert abs(st.t - t) <= bar_state * t
