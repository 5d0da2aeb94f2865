"""The vertex gradient at a q next to the link's crossing: the hit point lies where the given q
puts it, however close.  Triangles much smaller than a cell, so that a shift along the link
moves the barycentric weights by several times its size."""
from __future__ import annotations

import numpy as np
import pytest

from synth.meshes import radial_star

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("R,levels", [(2, 0), (3, 0), (1, 1)])
@pytest.mark.parametrize("shift", [0.0, 2.0 ** -21, -2.0 ** -21, 2.0 ** -23, -2.0 ** -22, "ulp"])
def test_gradient_next_to_the_crossing(orc, R, levels, shift):
    import torch

    import paper_2512_01251_gb300 as P
    v, t = radial_star(65, 64, 6, lambda l: 0.05 / l ** 2, seed=12)
    E = P.embed(torch.from_numpy(v), torch.from_numpy(t), R, levels, 2, 27)
    o = orc.embed_lines(v, t, R, levels, 2, 27)
    L = E.links
    q = L["q"].cpu().numpy()
    assert len(q) > 200
    q = np.nextafter(q, np.float32(2)) if shift == "ulp" else (q + np.float32(shift)).astype(np.float32)
    gq = np.random.default_rng(3).standard_normal(len(q)).astype(np.float32)
    lk = dict(o["links"], q=q.astype(np.float64))
    if shift == 0.0:
        lk["q"] = o["links"]["q"]  # the table's q: the crossing itself
    ref = orc.grad_verts_from_gq(lk, gq.astype(np.float64), o["X"], t, R, levels, o["blocks"][-1], len(v))
    _, nrm, _, _, _, _, c, h = orc.dq_dverts(lk, o["X"], t, R, levels)
    size = np.zeros((len(v), 3))
    b = np.abs(gq[:, None].astype(np.float64) * nrm / (h * np.einsum("ij,ij->i", nrm, c))[:, None])
    for j in range(3):
        np.add.at(size, t[lk["tri"], j], b)
    g = P.emb_cutlinks_backward(E.mesh, E.forest, L["cell"], L["dir"], torch.from_numpy(q).cuda(), L["tri"],
                                torch.from_numpy(gq).cuda()).cpu().numpy().astype(np.float64)
    assert P.emb_status_get() == P.EMB_OK
    # one rounding to FP32; the terms and their sums carry 40 bits or more
    assert np.all(np.abs(g - ref) <= 2.0 ** -23 * np.abs(ref) + 2.0 ** -32 * size)
