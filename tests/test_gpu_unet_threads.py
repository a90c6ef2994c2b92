"""Networks in several host threads, each on a stream of its own: the same results
as alone, from the first launch on (a fresh process: nothing is set up yet)."""
import subprocess
import sys

import pytest

from .conftest import ROOT

pytestmark = pytest.mark.gpu

CODE = """
import threading
import numpy as np, torch
import paper_2407_12399_gb300 as tsf
shapes = [(16, 20, 16), (24, 24, 24), (8, 12, 132), (32, 16, 20)]
rng = np.random.default_rng(3)
f = [rng.random(s, dtype=np.float32) for s in shapes]
torch.cuda.init()
streams = [torch.cuda.Stream() for _ in shapes]
nets = [tsf.UNet(seed=k, stream=streams[k]) for k in range(len(shapes))]
got, start = [None] * len(nets), threading.Barrier(len(nets))
def work(k):
    start.wait()
    got[k] = [(nets[k].forward(f[k], 0.05), *nets[k].gradients(f[k], 0.9 * f[k], 0.05)) for _ in range(3)]
threads = [threading.Thread(target=work, args=(k,)) for k in range(len(nets))]
[t.start() for t in threads]
[t.join() for t in threads]
for k, net in enumerate(nets):
    want = (net.forward(f[k], 0.05), *net.gradients(f[k], 0.9 * f[k], 0.05))
    for run in got[k]:
        assert np.array_equal(run[0], want[0]) and run[1] == want[1] and np.array_equal(run[2], want[2]), k
print("same")
"""


def test_networks_in_several_threads_give_what_each_gives_alone():
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stdout + r.stderr
