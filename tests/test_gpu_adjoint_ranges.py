"""The force, dF/dq and the vertex gradient where their fast arithmetic ends: populations
and weights of any magnitude (zeros, infinities and NaN among them), a q that is not the
link's crossing, thousands of links at one vertex, link counts around a tile, and the same
bits from run to run.  References in FP64."""
from __future__ import annotations

import numpy as np
import pytest

from synth import workload
from synth.meshes import octahedron

pytestmark = pytest.mark.gpu
G = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.fixture(scope="module")
def body(orc):
    import torch

    import paper_2512_01251_gb300 as P
    w = workload("star_1k")
    v, t = w.build_mesh()
    E = P.embed(torch.from_numpy(v), torch.from_numpy(t), w.R, w.levels, w.band, 27)
    o = orc.embed_lines(v, t, w.R, w.levels, w.band, 27)
    partner = orc.partner_cells(w.R, w.levels, o["blocks"][-1], o["masks"][-1], o["links"]["cell"], o["links"]["dir"])
    return w, v, t, E, o, partner


def _call(E, pop, gF, q=None):
    import torch

    import paper_2512_01251_gb300 as P
    L = E.links
    q = L["q"] if q is None else q
    F = P.emb_mex_force(E.forest, 27, L["cell"], L["dir"], q, pop)
    gq = P.emb_mex_force_backward(E.forest, 27, L["cell"], L["dir"], q, pop, torch.from_numpy(gF))
    return F.cpu().numpy().astype(np.float64), gq.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("spread", [0, 12, 30])
def test_force_over_magnitudes(orc, body, spread):
    """Populations 2^-spread .. 2^spread (30: beyond the float pairs' range once squared by
    the weights below): each dF/dq to FP32 rounding, the force to that of its terms."""
    import torch
    w, v, t, E, o, partner = body
    rng = np.random.default_rng(spread)
    ncell = 64 * len(o["blocks"][-1])
    pop = (rng.standard_normal((27, ncell)) * np.exp2(rng.uniform(-2 * spread, 2 * spread, (27, ncell)))).astype(np.float32)
    pop[:, rng.integers(0, ncell, ncell // 8)] = 0.0
    gF = np.array([0.3, -1.2e-3, 0.7e3], dtype=np.float32)
    lk = dict(o["links"], q=E.links["q"].cpu().numpy().astype(np.float64))
    F, gq = _call(E, torch.from_numpy(pop).cuda(), gF)
    c = orc.directions()[lk["dir"]].astype(np.float64)
    ref = orc.mex_force_dq(lk, pop.astype(np.float64), partner) @ gF.astype(np.float64)
    # one rounding to FP32 (2^-24), and 2^-40 of the products for the pairs
    mag = np.abs(c * gF.astype(np.float64)).sum(1) * np.abs(orc.mex_force_dq(lk, np.abs(pop).astype(np.float64), partner)).max(1)
    assert np.all(np.abs(gq - ref) <= 2.0 ** -23 * np.abs(ref) + 2.0 ** -40 * mag + 1e-37)
    F_ref = orc.mex_force(lk, pop.astype(np.float64), partner)
    scale = orc.mex_force(dict(lk), np.abs(pop).astype(np.float64), partner)
    total = sum(np.abs(x) for x in orc._link_pops(lk, np.abs(pop).astype(np.float64), partner)[1:4]).sum()
    assert np.all(np.isfinite(scale))
    assert np.all(np.abs(F - F_ref) <= 2.0 ** -23 * np.abs(F_ref) + 2.0 ** -38 * 8 * total)


def test_force_not_finite(orc, body):
    """NaN and infinite populations reach exactly the links that read them."""
    import torch
    w, v, t, E, o, partner = body
    ncell = 64 * len(o["blocks"][-1])
    pop = np.random.default_rng(1).standard_normal((27, ncell)).astype(np.float32)
    lk = dict(o["links"], q=E.links["q"].cpu().numpy().astype(np.float64))
    k = np.random.default_rng(2).integers(0, len(lk["cell"]), 12)
    pop[lk["dir"][k[:4]], lk["cell"][k[:4]]] = np.inf
    pop[lk["dir"][k[4:8]], lk["cell"][k[4:8]]] = -np.inf
    pop[lk["dir"][k[8:]], lk["cell"][k[8:]]] = np.nan
    gF = np.array([0.3, -1.2, 0.7], dtype=np.float32)
    with np.errstate(invalid="ignore"):
        c, f_i, f_o, f_p, has = orc._link_pops(lk, pop.astype(np.float64), partner)
        lo = lk["q"] < 0.5
        g = np.where(lo, np.where(has, 2 * (f_i - f_p), 0.0), (f_o - f_i) / (2 * lk["q"] ** 2))
        ref = (c @ gF.astype(np.float64)) * g
    F, gq = _call(E, torch.from_numpy(pop).cuda(), gF)
    np.testing.assert_allclose(gq, ref, rtol=1e-6, atol=1e-6)
    assert np.all(np.isnan(F))


def _grad(E, gq, q=None, n=None):
    import torch

    import paper_2512_01251_gb300 as P
    L = E.links
    q = L["q"] if q is None else torch.from_numpy(q).cuda()
    cut = [x[:n].contiguous() for x in (L["cell"], L["dir"], q, L["tri"], torch.from_numpy(gq).cuda())]
    g = P.emb_cutlinks_backward(E.mesh, E.forest, *cut)
    assert torch.equal(torch.nan_to_num(g), torch.nan_to_num(P.emb_cutlinks_backward(E.mesh, E.forest, *cut)))
    assert P.emb_status_get() == P.EMB_OK
    return g.cpu().numpy().astype(np.float64)


def _ref(orc, lk, gq, o, t, R, levels, nv, n=None):
    lk = {k: np.asarray(x)[:n] for k, x in lk.items() if k in ("cell", "dir", "q", "tri")}
    gq = gq.astype(np.float64)[:n]
    ref = orc.grad_verts_from_gq(lk, gq, o["X"], t, R, levels, o["blocks"][-1], nv)
    # the size of the summed terms: one link at a time would be |gq| |dq/dV|
    _, nrm, _, _, _, _, c, h = orc.dq_dverts(lk, o["X"], t, R, levels)
    size = np.zeros((nv, 3))
    b = np.abs(gq[:, None] * nrm / (h * np.einsum("ij,ij->i", nrm, c))[:, None])
    for j in range(3):
        np.add.at(size, t[lk["tri"], j], b)
    return ref, size


@pytest.mark.parametrize("spread", [0, 20, 60])
def test_gradient_over_magnitudes(orc, body, spread):
    w, v, t, E, o, partner = body
    rng = np.random.default_rng(spread + 5)
    n = len(o["links"]["q"])
    gq = (rng.standard_normal(n) * np.exp2(rng.uniform(-spread, spread, n))).astype(np.float32)
    gq[::7] = 0.0
    ref, size = _ref(orc, o["links"], gq, o, t, w.R, w.levels, len(v))
    g = _grad(E, gq)
    assert np.all(np.abs(g - ref) <= 2.0 ** -23 * np.abs(ref) + 2.0 ** -22 * size)


@pytest.mark.parametrize("n", [0, 1, 31, 256, 511, 512, 513, 1024, 1025])
def test_gradient_link_counts(orc, body, n):
    w, v, t, E, o, partner = body
    gq = np.random.default_rng(n).standard_normal(len(o["links"]["q"])).astype(np.float32)
    ref, size = _ref(orc, o["links"], gq, o, t, w.R, w.levels, len(v), n)
    assert np.all(np.abs(_grad(E, gq, n=n) - ref) <= 2.0 ** -23 * np.abs(ref) + 2.0 ** -22 * size)


def test_gradient_at_another_q(orc, body):
    """A q that is not the link's crossing moves the hit point along the link."""
    w, v, t, E, o, partner = body
    rng = np.random.default_rng(9)
    n = len(o["links"]["q"])
    gq = rng.standard_normal(n).astype(np.float32)
    q = rng.uniform(0.0, 1.0, n).astype(np.float32)
    ref, size = _ref(orc, dict(o["links"], q=q.astype(np.float64)), gq, o, t, w.R, w.levels, len(v))
    # barycentric weights reach the link's length over the triangle's height here
    assert np.all(np.abs(_grad(E, gq, q=q) - ref) <= 1e-5 * (np.abs(ref) + size))


def test_gradient_not_finite(orc, body):
    w, v, t, E, o, partner = body
    n = len(o["links"]["q"])
    gq = np.zeros(n, dtype=np.float32)
    k = np.random.default_rng(3).integers(0, n, 3)
    gq[k] = [np.nan, np.inf, -np.inf]
    g = _grad(E, gq)
    touched = np.zeros(len(v), dtype=bool)
    touched[t[o["links"]["tri"][k]].reshape(-1)] = True
    assert not np.any(np.isfinite(g[touched])) and np.all(g[~touched] == 0.0)


def test_gradient_many_links_per_vertex(orc):
    """Eight faces on a fine grid: every vertex takes a third of the terms of four faces."""
    import torch

    import paper_2512_01251_gb300 as P
    v, t = octahedron([G // 2 + 3, G // 2 - 5, G // 2 + 1], [G // 4 + 11, G // 5, G // 3 - 7])
    v, t = np.asarray(v, dtype=np.float32), np.asarray(t, dtype=np.int32)
    E = P.embed(torch.from_numpy(v), torch.from_numpy(t), 4, 3, 2, 27)
    o = orc.embed_lines(v, t, 4, 3, 2, 27)
    n = len(o["links"]["q"])
    assert n > 20000
    gq = np.random.default_rng(8).standard_normal(n).astype(np.float32)
    ref, size = _ref(orc, o["links"], gq, o, t, 4, 3, len(v))
    g = _grad(E, gq)
    # each term's own error is FP32-sized; independent, they add up to far less than this
    assert np.all(np.abs(g - ref) <= 2.0 ** -23 * np.abs(ref) + 2.0 ** -24 * size)
