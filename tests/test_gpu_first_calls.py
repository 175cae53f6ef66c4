"""The first call of a process that needs no handle loads the kernels it can run, of every radius but
not the batched launches, so that later calls of any radius load nothing, also within a caller's
capture."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SETUP = """
import sys, time
sys.path.insert(0, %r)
import torch
from paper_1306_2461_gb300 import of
I1 = (torch.arange(60 * 80, device="cuda") * 7919 %% 251).to(torch.uint8).view(60, 80)
I2 = I1.roll(1, 1).contiguous()
u, v = torch.empty(60, 80, device="cuda"), torch.empty(60, 80, device="cuda")
x = torch.ones(5, 60, 80, device="cuda")
plan = lambda r: of.Plan.make(60, 80, 1, r, 2)
def noalloc(r): of.compute_noalloc(plan(r), I1, I2, u, v)
def sums(r): return of.window_sums(x, r)
def create(r): return of.Flow(plan(r))
torch.cuda.synchronize()
""" % ROOT


def run(code):
    r = subprocess.run([sys.executable, "-c", SETUP + code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return r.stdout


def test_first_calls_load_what_they_run():
    # fresh processes; all kernels of every radius take eleven times as long as those of one
    t = {n: float(run(f"t0 = time.perf_counter(); {n}(4); torch.cuda.synchronize(); print(time.perf_counter() - t0)"))
         for n in ("create", "sums", "noalloc")}
    print(t)
    assert t["sums"] < t["create"] and t["noalloc"] < 6 * t["create"]


@pytest.mark.parametrize("mode", ["global", "thread_local"])
def test_first_use_of_a_radius_in_a_capture(mode):
    out = run(f"""
noalloc(4); sums(4); torch.cuda.synchronize()
g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
with torch.cuda.graph(g, stream=s, capture_error_mode={mode!r}):
    noalloc(9)
    w = sums(11)
u.fill_(7.0); v.fill_(7.0)
g.replay(); torch.cuda.synchronize()
got = [t.clone() for t in (u, v, w)]
noalloc(9)
want = [u, v, sums(11)]
torch.cuda.synchronize()
print(all(torch.equal(a, b) for a, b in zip(got, want)) and float(want[2].max()) == 23 * 23)
""")
    assert out.strip() == "True"
