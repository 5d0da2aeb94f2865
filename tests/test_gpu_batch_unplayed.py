"""Counts and results of a batch with headroom before its first replay: the root level and
nothing else, whatever the buffers held before."""
from __future__ import annotations

import numpy as np
import pytest

from synth import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_before_the_first_replay():
    import torch

    import paper_2512_01251_gb300 as P
    w = workload("star_1k")
    v, t = w.build_mesh()
    for _ in range(4):  # freed buffers of one batch are those of the next
        m = P.emb_mesh_create(torch.from_numpy(v), torch.from_numpy(t), w.R)
        b = P.emb_batch_create([m], [w.levels], [w.band], [19], headroom=20)
        assert P.emb_batch_counts(b, 0) == ([w.R ** 3] + [0] * w.levels, 0)
        r = P.emb_batch_results(b, 0)
        assert [len(x) for x in r["masks"]] == [w.R ** 3] + [0] * w.levels
        assert all(len(r["links"][k]) == 0 for k in ("cell", "dir", "q", "tri"))
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            P.emb_batch_run(b, s)
        s.synchronize()
        E = P.embed(torch.from_numpy(v), torch.from_numpy(t), w.R, w.levels, w.band, 19)
        blocks, n = P.emb_batch_counts(b, 0)
        assert n == len(E.links["q"]) and blocks == [len(x) for x in E.masks]
        np.testing.assert_array_equal(P.emb_batch_results(b, 0)["links"]["cell"].cpu().numpy(), E.links["cell"].cpu().numpy())
        assert P.emb_status_get() == P.EMB_OK
        b.close()
