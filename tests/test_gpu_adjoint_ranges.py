"""The force and dF/dq where their fast arithmetic ends: populations of any magnitude
(zeros, infinities and NaN among them).  References in FP64."""
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
