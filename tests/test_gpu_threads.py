"""Several host threads, each with a context and a stream of its own, make the library's first calls in a
process at once: what a kernel's first use sets up is there for all of them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import threading
import torch
import workloads as wl
from paper_1812_05264_gb300 import api
N, kinds = 8, [(388, False), (132, False), (256, False), (100, True)]
sys_ = []
for s, fp64 in kinds:
    wk = wl.fcc_cu(20, kT=0.5, n_probes=s, jitter=0.05)
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    ctx = api.Context()
    H = api.assemble_H(ctx, api.Model.from_workload(wk, "cuda"), pos, api.build_neighbors(ctx, pos, wk.cutoff))
    sys_.append((H, *api.spectral_bounds(ctx, H)))
torch.cuda.synchronize()
out, start = [None] * N, threading.Barrier(N)
def work(i):
    (s, fp64), (H, lo, hi) = kinds[i % len(kinds)], sys_[i % len(kinds)]
    c = api.Context(stream=torch.cuda.Stream())
    start.wait()
    try:
        out[i] = api.chebyshev_moments(c, H, lo, hi, 3, s, 24, fp64).cpu()
    except Exception as e:
        out[i] = e
ts = [threading.Thread(target=work, args=(i,)) for i in range(N)]
[t.start() for t in ts]
[t.join() for t in ts]
for i, m in enumerate(out):
    assert torch.is_tensor(m), m
    (s, fp64), (H, lo, hi) = kinds[i % len(kinds)], sys_[i % len(kinds)]
    assert torch.equal(m, api.chebyshev_moments(api.Context(), H, lo, hi, 3, s, 24, fp64).cpu()), i
"""


@pytest.mark.parametrize("trial", [0, 1])
def test_first_calls_from_many_threads(trial):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
