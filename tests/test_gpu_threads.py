"""Solvers stepped from several host threads at once, each on its own stream: the states are those of a
solver alone, bit for bit (a step reduces by maxima only).  The first steps of a process fill what the
library asks the device for once, so the threads start in a fresh one."""
import subprocess
import sys

import pytest
import torch

from conftest import ROOT

pytestmark = pytest.mark.gpu

RUN = """
import threading
import numpy as np, torch
from paper_2003_08746_gb300 import jz, workloads as W
jz.load()
torch.cuda.init()
cases = [(f, W.jet_grid(40, 20, 16) if n % 2 else W.box_grid(33, 17, 9, h=0.2), n)
         for n, f in enumerate((jz.JZ_PREC_FP64PAIR, jz.JZ_PREC_FP64PAIR, jz.JZ_PREC_FP32FLUX, jz.JZ_PREC_FP32FLUX,
                                jz.JZ_PREC_FP64, jz.JZ_PREC_FP64))]

def work(case, out, wait):
    form, g, n = case
    prm, q = (W.jet_params(seed=n), W.jet_state(g)) if n % 2 else (W.box_params(), W.random_state(g, seed=n, amp=0.05))
    torch.cuda.set_device(0)
    st = torch.cuda.Stream()
    wait()
    grid = jz.Grid.from_workload(g)
    s = jz.Solver(grid, prm, form, stream=st.cuda_stream)
    s.set_state(q, 0.0)
    s.step(5)
    out[n] = s.get_state()
    s.close()
    grid.close()

together, alone = {}, {}
bar = threading.Barrier(len(cases))
ts = [threading.Thread(target=work, args=(c, together, bar.wait)) for c in cases]
[t.start() for t in ts]
[t.join() for t in ts]
for c in cases:
    work(c, alone, lambda: None)
assert len(together) == len(cases)
assert all(np.array_equal(together[n], alone[n]) for n in alone)
print("same states")
"""


def test_threads_match_alone():
    from paper_2003_08746_gb300 import build
    build.build()
    assert torch.cuda.is_available()
    r = subprocess.run([sys.executable, "-c", RUN], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same states" in r.stdout, r.stdout + r.stderr
