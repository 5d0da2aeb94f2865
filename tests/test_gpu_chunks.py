"""Few large triangles on fine grids: their lines and candidate blocks are cut into chunks
for whole warps (the number of chunks grows with the items, small ones first in a small
mesh), and their plane offsets need more than 64 bits on the coarse side of the line
between the two.  Every output against the oracle's sorted-line tier."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import compare_full, gpu_embed
from synth.meshes import axis_box, octahedron

pytestmark = pytest.mark.gpu
G = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# lines a face: a few (below the lower line of 8), tens, hundreds, thousands; radii above and
# below 2^18, the extent up to which the plane offsets fit 64 bits
@pytest.mark.parametrize("R,levels,radii", [
    (2, 1, (G // 4 + 3, G // 4 + 7, G // 3 + 1)), (4, 2, (G // 4 + 3, G // 5, G // 3 + 1)),
    (3, 3, (G // 4 + 3, G // 5, G // 3 + 1)), (8, 3, (G // 4 + 3, G // 4 - 1, G // 4 + 1)),
    (16, 2, ((1 << 17) - 3, (1 << 17) - 1, 1 << 17)), (12, 3, ((1 << 16) + 5, (1 << 17) + 1, 1 << 16)),
])
def test_octahedron(orc, R, levels, radii):
    v, t = octahedron([G // 2 + 5, G // 2 - 3, G // 2 + 9], radii)
    v, t = np.asarray(v, dtype=np.float32), np.asarray(t, dtype=np.int32)
    _, g = gpu_embed(v, t, R, levels, 2, 27)
    compare_full(g, orc.embed_lines(v, t, R, levels, 2, 27), levels)


def test_box_with_many_lines_a_face(orc):
    """4,096 lines a triangle and more candidate blocks than 16 chunks of 64 hold."""
    v, t = axis_box([G // 4 + 11] * 3, [3 * G // 4 - 7] * 3)
    v, t = np.asarray(v, dtype=np.float32), np.asarray(t, dtype=np.int32)
    _, g = gpu_embed(v, t, 16, 2, 2, 19)
    compare_full(g, orc.embed_lines(v, t, 16, 2, 2, 19), 2)
