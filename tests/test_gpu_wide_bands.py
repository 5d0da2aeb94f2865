"""Near-wall bands wider than the domain: every block of every refined level is flagged, as
for a band that just covers it.  The dilation in frame units, (band - 1/2) h, is a multiple of
2^32 less half a cell or more in these cases, so that it does not survive 32 bits."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import compare_full, gpu_embed
from synth.meshes import icosphere

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _small():
    g = float(1 << 20)
    v, t = icosphere(1)
    v = np.asarray(v, dtype=np.float64)
    v = (v - v.mean(0)) * 0.1 + [0.3, 0.6, 0.4]
    return (np.round(v * g) / g).astype(np.float32), np.asarray(t, dtype=np.int32)


@pytest.mark.parametrize("R,levels,band", [(8, 1, 1 << 17), (8, 2, 1 << 18), (3, 1, 1 << 20), (16, 2, 1 << 20), (4, 1, 1 << 14)])
def test_band_wider_than_the_domain(orc, R, levels, band):
    import torch

    import paper_2512_01251_gb300 as P
    v, t = _small()
    cover = 4 * R << levels  # cells across the domain
    o = orc.embed_lines(v, t, R, levels, cover, 19)
    assert all(np.all(o["flags"][L] == 1) for L in range(levels))
    few = orc.embed_lines(v, t, R, levels, 2, 19)
    assert len(few["blocks"][-1]) < len(o["blocks"][-1])  # a narrow band leaves blocks out
    _, g = gpu_embed(v, t, R, levels, band, 19)
    compare_full(g, o, levels)
    assert P.emb_status_get() == P.EMB_OK
    m = P.emb_mesh_create(torch.from_numpy(v), torch.from_numpy(t), R)
    b = P.emb_batch_create([m], [levels], [band], [19])
    P.emb_batch_run(b)
    r = P.emb_batch_results(b, 0)
    np.testing.assert_array_equal(r["masks"][-1].cpu().numpy().view(np.uint64), o["masks"][-1])
    np.testing.assert_array_equal(r["links"]["cell"].cpu().numpy(), o["links"]["cell"])
    assert P.emb_status_get() == P.EMB_OK
