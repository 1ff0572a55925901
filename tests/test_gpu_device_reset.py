"""A program may reset the device between simulators (cudaDeviceReset ends its own CUDA context only): what the library
keeps for later simulators -- page-locked blocks, copiers, kernel attributes, the address of its static array -- is made
anew, and the second half of the program gets what the first got."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
import ctypes, glob, os, sys
import numpy as np
import torch
from paper_2009_05766_b200 import binding

def runtime():
    near = os.path.join(os.path.dirname(os.path.dirname(torch.__file__)), "nvidia", "cuda_runtime", "lib", "libcudart.so*")
    for path in sorted(glob.glob(near)) + ["libcudart.so.12", "/usr/local/cuda/lib64/libcudart.so.12"]:
        try:
            return ctypes.CDLL(path)
        except OSError:
            pass
    raise SystemExit("no CUDA runtime library")

def run(M, d, rounds, links=False):
    rng = np.random.default_rng(M)
    P = rng.random((M, M)) + 0.05
    np.fill_diagonal(P, 0.0)
    P /= P.sum(axis=1, keepdims=True)
    g = binding.Netmax(M=M, d=d, lr=0.1, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, seed=3, policy_K=2, policy_R=2)
    if links:
        s = np.triu(np.exp(rng.uniform(0.0, 4.0, (M, M))), 1)
        g.set_policy(link_speed_gbps=s + s.T)
    g.round(rounds)
    out = [g.read_replicas(), g.peer_trace(), *g.telemetry(), g.read_columns_static([0, d - 1]), g.get_policy()[0]]
    g.close()
    return out

def all_of_them():
    # short vectors, tiles of long ones, tiles that fill a CTA's shared memory, a policy change on the device
    return [run(4, 1000, 5), run(8, 400_003, 20), run(600, 64, 30), run(330, 64, 3, links=True)]

first = all_of_them()
assert runtime().cudaDeviceReset() == 0
second = all_of_them()
for a, b in zip(first, second):
    for k, (x, y) in enumerate(zip(a, b)):
        if k in (2, 3):  # telemetry: sums whose order may differ from run to run
            np.testing.assert_allclose(x, y, rtol=1e-9)
        else:
            assert x.shape == y.shape and (x == y).all()
print("fine")
"""


def test_simulators_work_after_a_device_reset():
    done = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0 and done.stdout.strip() == "fine", (done.returncode, done.stdout, done.stderr[-2000:])
