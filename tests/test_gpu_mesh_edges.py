"""The watertight check of emb_mesh_create: closed, open, doubled and degenerate triangle
lists, in any numbering, where a few vertices hold most edges (the edge table's overflow,
and its second size), and with many vertices that no triangle uses."""
from __future__ import annotations

import numpy as np
import pytest

from synth.meshes import icosphere

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _bipyramid(n):
    """Two apexes over a rim of n vertices: 2n triangles, 3n edges, 2n of them at the apexes."""
    r = np.arange(n)
    nx = (r + 1) % n
    up = np.stack([np.full(n, n), r, nx], 1)
    down = np.stack([np.full(n, n + 1), nx, r], 1)
    return n + 2, np.concatenate([up, down]).astype(np.int32)


def _sphere(spare=0):
    v, t = icosphere(3)
    return len(v) + spare, np.asarray(t, dtype=np.int32)


def _status(nv, t, **kw):
    import torch

    import paper_2512_01251_gb300 as P
    v = torch.full((nv, 3), 0.5, dtype=torch.float32, device="cuda")
    try:
        P.emb_mesh_create(v, torch.from_numpy(np.ascontiguousarray(t)), 2, **kw).close()
    except P.EmbError as e:
        return e.code
    return P.EMB_OK


CASES = {"sphere": _sphere(), "spare_vertices": _sphere(10000), "rim_5": _bipyramid(5), "rim_4001": _bipyramid(4001),
         "rim_40000": _bipyramid(40000), "rim_131072": _bipyramid(1 << 17)}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("renumber", [False, True])
def test_watertight(name, renumber):
    import paper_2512_01251_gb300 as P
    nv, t = CASES[name]
    rng = np.random.default_rng(len(t))
    if renumber:
        t = rng.permutation(nv).astype(np.int32)[t][rng.permutation(len(t))]
    assert _status(nv, t) == P.EMB_OK
    for k in (0, len(t) // 2, len(t) - 1):
        assert _status(nv, np.delete(t, k, 0)) == P.EMB_ERR_NOT_WATERTIGHT  # an open edge
        assert _status(nv, np.concatenate([t, t[k:k + 1]])) == P.EMB_ERR_NOT_WATERTIGHT  # a face twice
        turned = t.copy()
        turned[k] = turned[k, ::-1]
        assert _status(nv, turned) == P.EMB_ERR_NOT_WATERTIGHT  # a face the wrong way round
        assert _status(nv, turned, check_watertight=False) == P.EMB_OK
        pinched = t.copy()
        pinched[k, 1] = pinched[k, 0]
        assert _status(nv, pinched) == P.EMB_ERR_NOT_WATERTIGHT  # an edge from a vertex to itself
        outside = t.copy()
        outside[k, 2] = nv
        assert _status(nv, outside) == P.EMB_ERR_BAD_INPUT
        outside[k, 2] = -1
        assert _status(nv, outside) == P.EMB_ERR_BAD_INPUT
