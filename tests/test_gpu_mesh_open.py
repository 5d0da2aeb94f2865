"""The watertight check on lists with up to twice the edges of a closed one, all of them open:
unindexed triangles, and every pair of a few vertices once."""
from __future__ import annotations

import numpy as np
import pytest

from test_gpu_mesh_edges import _status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _soup(n):
    """n triangles that share no vertex (an unindexed list): 3n edges, all open."""
    return 3 * n, np.arange(3 * n, dtype=np.int32).reshape(n, 3)


def _every_pair_once(n):
    """Bose's triple system on 3n points (n odd): every pair of points in one triangle, so
    3n (3n - 1) / 2 edges at few vertices, all open."""
    i, j = np.triu_indices(n, 1)
    mean = (i + j) * ((n + 1) // 2) % n
    x = np.arange(n)
    t = [np.stack([x, x + n, x + 2 * n], 1)]
    t += [np.stack([i + k * n, j + k * n, mean + (k + 1) % 3 * n], 1) for k in range(3)]
    return 3 * n, np.concatenate(t).astype(np.int32)


OPEN = {"soup_1": _soup(1), "soup_4096": _soup(4096), "soup_100000": _soup(100000), "pairs_201": _every_pair_once(67),
        "pairs_651": _every_pair_once(217)}


@pytest.mark.parametrize("name", list(OPEN))
@pytest.mark.parametrize("renumber", [False, True])
def test_open_lists_with_more_edges_than_a_closed_one(name, renumber):
    import paper_2512_01251_gb300 as P
    nv, t = OPEN[name]
    if renumber:
        rng = np.random.default_rng(len(t))
        t = rng.permutation(nv).astype(np.int32)[t][rng.permutation(len(t))]
    assert _status(nv, t) == P.EMB_ERR_NOT_WATERTIGHT
    assert _status(nv, t, check_watertight=False) == P.EMB_OK
