"""The link kernel's line test beyond the 32-bit gate, where the signs of the Pluecker values
come from float values with an error bound: edges that pass the line at a few units over
offsets of 2^14 to 2^25 (values around the bound and at zero), against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import predicate_cases as PC

pytestmark = pytest.mark.gpu
N = 200_000
DIRS = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
                 (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
                 (0, 1, -1), (0, -1, 1), (1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1),
                 (-1, 1, 1), (1, -1, -1)], dtype=np.int64)


@pytest.mark.parametrize("lo,hi,near", [(14, 16, 0), (14, 18, 2), (16, 22, 8), (20, 25, 2), (20, 25, 200), (14, 25, 5000)])
def test_edges_close_to_the_line(orc, lo, hi, near):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_01251_gb300 as P
    rng = np.random.default_rng(1000 * lo + 10 * hi + near)
    h = (1 << rng.integers(13, 19, N)).astype(np.int64)
    half = h // 2
    ncell = PC.TOP // h
    Pt = (2 * np.floor(rng.random((N, 3)) * ncell[:, None]).astype(np.int64) + 1) * half[:, None]
    dirs = rng.integers(1, 27, N).astype(np.int64)
    c = DIRS[dirs]
    assert np.array_equal(DIRS, np.array(P.emb_directions()))
    size = np.exp2(rng.uniform(lo, hi, (N, 3))).astype(np.int64)
    # two vertices along the line, one on either side of the link, a few units beside it; the
    # third anywhere
    jit = rng.integers(-near, near + 1, (N, 2, 3))
    ab = np.stack([size[:, :1], -size[:, 1:2]], 1) * c[:, None, :] + jit
    far = rng.integers(-1, 2, (N, 1, 3)) * size[:, 2][:, None, None] + rng.integers(-near, near + 1, (N, 1, 3))
    tri = PC._clip(Pt[:, None, :] + np.concatenate([ab, far], 1)).reshape(N, 9)
    q = np.zeros((N, 15), dtype=np.int64)
    q[:, 0:9], q[:, 9:12], q[:, 12], q[:, 13] = tri, Pt, dirs, h
    hit, t = orc.each_segment(tri, Pt, dirs, h)
    got, gq = P.emb_probe_predicates(P.EMB_PROBE_PAIR, torch.from_numpy(q))
    got, gq = got.cpu().numpy(), gq.cpu().numpy().astype(np.float64)
    bad = np.nonzero(got != hit)[0]
    assert len(bad) == 0, (len(bad), q[bad[:3]].tolist())
    sel = hit == 1
    assert sel.sum() >= 10
    assert np.abs(gq[sel] - t[sel]).max() <= 2e-6
