"""Grids whose copy in shared memory, with the kernel's own, passes the 48 KB that need no larger limit (3056 to 3072 points),
and the sizes around, each as the first call of a process."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import numpy as np, torch
from oracle import gwc_oracle as G
from paper_2412_17132_gb300 import gwc
n, eta, n_t, t_max = {n}, 1e-3, 1024, 500.0
eps = torch.linspace(-10.5, 3.0, 12, dtype=torch.float64, device="cuda")
o_ov = torch.zeros((8, 20), dtype=torch.float64, device="cuda")
o_core = torch.zeros((12, 1, 8), dtype=torch.float64, device="cuda")
ctx = gwc.Context(eps, 2, [0], o_ov, o_core, prec="fp64", n_t=n_t, t_max=t_max, eta=eta)
w = np.linspace(-{top}, 0.2, n)
im = np.where(w < 0, 0.01 * np.minimum(1.0, (w / 0.3) ** 2), 0.0)
a, _ = ctx.cumulant_spectrum(torch.as_tensor(w, device="cuda")[None], torch.as_tensor(im, device="cuda")[None])
ctx.sync()
ref = G.gwc_spectrum(w, im, eta, n_t, t_max)[1]
assert np.max(np.abs(a[0].cpu().numpy() - ref)) <= 1e-10 * np.max(np.abs(ref))
"""


# a largest frequency that goes by blocks, and one that takes the direct sum
@pytest.mark.parametrize("n,top", [(3008, 0.9), (3055, 0.9), (3057, 0.9), (3072, 0.9), (3072, 1.5), (3073, 1.5), (8192, 1.5)])
def test_grid_sizes_around_the_shared_memory_limit(n, top):
    r = subprocess.run([sys.executable, "-c", CODE.format(n=n, top=top)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
