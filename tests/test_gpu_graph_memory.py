"""A device without the memory that a captured graph takes: evaluations, spectra
and the tuner run by direct launches.  The runtime's answer is faked (a
preloaded function in its place), so no memory is taken."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = """
static int calls;
int fake_calls(void) { return calls; }
int %s(void* a, void* b, unsigned long long f) { (void)a; (void)b; (void)f; ++calls; return 2; } /* cudaErrorMemoryAllocation */
"""

RUN = """
import ctypes, hashlib, json, sys
import torch
from paper_2602_14016_gb300 import api, synthetic
import numpy as np
ctx = api.Context(api.Config(n=64, nsteps=4, dt=1e-3, nu=1e-3, px=4, every=2, kernels=[api.KernelSpec("identity", 0.0)] * 20))
chosen, ms = ctx.autotune(2)
ctx.set_plan(0)
ctx.set_graphs(True)
w = torch.from_numpy(np.stack([synthetic.random_vorticity_hat(64, b) for b in range(20)])).cuda()
s = ctx.control_from_omega(w)
ctx.set_observations(torch.ones((20, ctx.nt, 16, 2), dtype=torch.float64, device="cuda"))
out = list(ctx.cost_grad(s)) + list(ctx.cost_grad(s)) + list(ctx.adjoint_spectra(s, w, 2)) + list(ctx.adjoint_spectra(s, w, 2))
h = hashlib.sha256(b"".join(t.cpu().numpy().tobytes() for t in out)).hexdigest()
lib = ctypes.CDLL(None)
print(json.dumps({"hash": h, "calls": lib.fake_calls() if len(sys.argv) > 1 else 0, "ms": ms, "launches": ctx.launches}))
"""


def run(tmp_path, name=None):
    env = dict(os.environ, PYTHONPATH=ROOT)
    args = [sys.executable, "-c", RUN]
    if name:
        src, lib = tmp_path / f"{name}.c", tmp_path / f"{name}.so"
        src.write_text(FAKE % name)
        subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(src)], check=True)
        env["LD_PRELOAD"] = str(lib)
        args.append("fake")
    p = subprocess.run(args, env=env, cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    return json.loads(p.stdout.strip().splitlines()[-1])


def test_evaluations_go_on_without_memory_for_a_graph(tmp_path):
    want = run(tmp_path)
    for name in ("cudaGraphInstantiate", "cudaGraphUpload", "cudaGraphLaunch"):
        got = run(tmp_path, name)
        assert got["calls"] > 0 and all(t > 0 for t in got["ms"])
        assert got["hash"] == want["hash"] and got["launches"] == want["launches"]
