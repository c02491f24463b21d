"""Host threads that use the library at the same time, each with its own trees and stream."""
import os
import subprocess
import sys
import threading

import pytest
import torch

from workloads import Workload, make_inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2509_06040_b200 import binding
    return binding


FIRST_CALLS = """
import threading, sys
import torch
import __graft_entry__
__graft_entry__.build()
from paper_2509_06040_b200 import binding as B
from paper_2509_06040_b200.session import TreeSession
from workloads import Workload, make_inputs
w = Workload(name="threads", n_trees=1, tokens=300, channels=64, T=1, K=1, splits=(), sigma=0.3, velocity="mlp", reward="mixture", hidden=1024)
inp, sessions = make_inputs(w), [TreeSession(w) for _ in range(8)]
for s in sessions:
    s.upload_inputs(inp)
    s.init()
    s.v.fill_(float("nan"))
torch.cuda.synchronize()
together, errors = threading.Barrier(len(sessions)), []
def work(s):
    try:
        with torch.cuda.stream(torch.cuda.Stream()):
            together.wait()
            B.velocity_mlp(s.tree, s.packed, w.hidden, s.v)      # the process's first launch of the stage
    except Exception as e:
        errors.append(e)
threads = [threading.Thread(target=work, args=(s,)) for s in sessions]
[t.start() for t in threads]
[t.join() for t in threads]
torch.cuda.synchronize()
assert not errors, errors
assert all(torch.equal(s.v, sessions[0].v) for s in sessions)
print("same bits")
"""


def test_first_velocity_calls_of_several_threads():
    """The stage asks its device once how many clusters fit; threads that get there together all launch the same split."""
    out = subprocess.run([sys.executable, "-c", FIRST_CALLS], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and "same bits" in out.stdout, out.stderr[-2000:]


def test_whole_tree_rollouts_of_different_depth_in_two_threads(B):
    """Trees whose open forks take 96 and 64 KB of shared memory, rolled out over and over by two threads: no launch is refused
    and each tree comes out as on its own."""
    from paper_2509_06040_b200.session import TreeSession
    sessions = []
    for splits in ((1, 2, 3, 4, 5, 6), (1, 2, 3, 4)):           # three trees an SM: no fork is dealt out to the grid
        w = Workload(name="threads", n_trees=444, tokens=9, channels=4, T=splits[-1] + 1, K=2, splits=splits, sigma=0.3, velocity="linear",
                     reward="neg_mse_mu", branch_corr_s=2.0)
        s = TreeSession(w)
        s.upload_inputs(make_inputs(w))
        s.rollout()
        sessions.append(s)
    torch.cuda.synchronize()
    alone = [s.latents.clone() for s in sessions]
    together, errors = threading.Barrier(2), []

    def work(s):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                together.wait()
                for _ in range(1000):
                    s.rollout()
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in sessions]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for s, ref in zip(sessions, alone):
        assert torch.equal(s.latents, ref)
