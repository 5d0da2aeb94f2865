"""Triangle and block counts around the tiles of the scans (16,384 triangles, 4,096 blocks),
of the filter and of the refine kernel (32 triangles), and x-rows of blocks that span
several warps of the row scan.  Every output against the oracle's sorted-line tier."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import compare_full, gpu_embed
from synth.meshes import axis_box, radial_star

pytestmark = pytest.mark.gpu
G = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# 2 n_phi (n_theta - 1) triangles: 16,380, 16,384 and 16,386 (and one of 32 k + 2)
@pytest.mark.parametrize("n_theta,n_phi,R,levels", [(92, 90, 8, 2), (65, 128, 16, 2), (4, 2731, 8, 3), (4, 11, 5, 2)])
def test_triangle_tiles(orc, n_theta, n_phi, R, levels):
    v, t = radial_star(n_theta, n_phi, 4, lambda l: 0.05 / l ** 2, seed=n_phi)
    assert len(t) == 2 * n_phi * (n_theta - 1)
    _, g = gpu_embed(v, t, R, levels, 2, 19)
    compare_full(g, orc.embed_lines(v, t, R, levels, 2, 19), levels)


# rows of 31 to 72 root blocks: shorter than, as long as, and longer than a warp's 32
@pytest.mark.parametrize("R", [31, 32, 48, 72])
def test_long_rows(orc, R):
    v, t = axis_box([G // 16 + 3, G // 3 + 1, G // 3 - 5], [15 * G // 16 - 7, G // 2 + 9, G // 2 - 1])
    v, t = np.asarray(v, dtype=np.float32), np.asarray(t, dtype=np.int32)
    _, g = gpu_embed(v, t, R, 0, 2, 27)
    compare_full(g, orc.embed_lines(v, t, R, 0, 2, 27), 0)
