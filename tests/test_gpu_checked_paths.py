"""The bounds-mode build over the paths that tests/test_gpu_checked.py leaves out: batches with
headroom, incremental re-embedding, the vertex gradient and the LBM step run clean, and a link
whose cell lies outside the level becomes EMB_ERR_BOUNDS instead of an access."""
from __future__ import annotations

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import sys
sys.path.insert(0, sys.argv[1]); sys.path.insert(0, sys.argv[1] + "/tests")
import numpy as np, torch
import paper_2512_01251_gb300 as P
from paper_2512_01251_gb300 import _lib
assert _lib.LIB_PATH.endswith("libemb_check.so"), _lib.LIB_PATH
from synth import bump, populations, workload
from test_gpu_incremental import changed_extent
w = workload("star_112k")
v, t = w.build_mesh()
dv, dt = torch.from_numpy(v), torch.from_numpy(t)
E = P.embed(dv, dt, w.R, w.levels, w.band, 27)
m = P.emb_mesh_create(dv, dt, w.R)
b = P.emb_batch_create([m], [w.levels], [w.band], [27], headroom=20)
P.emb_batch_run(b)
r = P.emb_batch_results(b, 0)
assert torch.equal(r["links"]["cell"], E.links["cell"]) and torch.equal(r["masks"][-1], E.masks[-1])
assert P.emb_status_get() == P.EMB_OK
n = len(E.links["q"])
gq = torch.ones(n, device="cuda")
L = E.links
g = P.emb_cutlinks_backward(E.mesh, E.forest, L["cell"], L["dir"], L["q"], L["tri"], gq)
nblk = len(E.masks[-1])
pop = torch.from_numpy(populations(64 * nblk, seed=1, lattice=27)).cuda()
P.emb_lbm_step(E.forest, 27, L, 1.2, pop)
assert P.emb_status_get() == P.EMB_OK
far = L["cell"].clone()
k = n // 2
far[k] = 64 * nblk + 64 * 5
h = P.emb_cutlinks_backward(E.mesh, E.forest, far, L["dir"], L["q"], L["tri"], gq)
assert P.emb_status_get() == -8  # EMB_ERR_BOUNDS
keep = torch.arange(n, device="cuda") != k
cut = [x[keep].contiguous() for x in (L["cell"], L["dir"], L["q"], L["tri"], gq)]
ref = P.emb_cutlinks_backward(E.mesh, E.forest, *cut)
assert torch.allclose(h, ref, rtol=1e-5, atol=1e-6 * float(ref.abs().max()))  # the link was left out
assert P.emb_status_get() == P.EMB_OK
v2, moved = bump(v, (0.2, 1.0, 0.3), 0.97, 900)
P.reembed_window(E, torch.from_numpy(v2).cuda(), changed_extent(v, v2, t, moved, w.R), w.band)
assert P.emb_status_get() == P.EMB_OK
F = P.embed(torch.from_numpy(v2), dt, w.R, w.levels, w.band, 27)
assert all(torch.equal(E.links[x], F.links[x]) for x in ("cell", "dir", "q", "tri"))
print("bounds mode ok")
'''


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_bounds_mode_build_runs_clean_on_the_other_paths():
    from paper_2512_01251_gb300 import build as B
    B.build(check=True)
    env = dict(os.environ, EMB_LIBRARY="check")
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], env=env, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0 and "bounds mode ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
