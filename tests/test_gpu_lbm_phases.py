"""The passes of an LBM step called one by one (phases 1, 2, 4 and 3, 6, 5): streaming moves
populations and changes none, the boundary pass writes the linked ones, and the passes in turn
give the oracle's step, as the fused whole step does."""
from __future__ import annotations

import numpy as np
import pytest

from synth import populations, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("name,lattice,omega", [("icosphere_320", 19, 1.3), ("star_4k_r3", 27, 1.7)])
def test_phases_one_by_one(orc, name, lattice, omega):
    import torch

    import paper_2512_01251_gb300 as P
    w = workload(name)
    v, t = w.build_mesh()
    E = P.embed(torch.from_numpy(v), torch.from_numpy(t), w.R, w.levels, w.band, lattice)
    o = orc.embed(v, t, w.R, w.levels, w.band, lattice)
    blocks, masks, links = o["blocks"][-1], o["masks"][-1], o["links"]
    pop = populations(64 * len(blocks), seed=5, u=(0.03, 0.02, -0.01), noise=0.05, lattice=lattice)
    solid = ((masks[:, None] >> np.arange(64, dtype=np.uint64)) & np.uint64(1)).reshape(-1).astype(bool)
    pop[:, solid] = 0.0
    d = torch.from_numpy(pop).cuda()

    def step(phases, pre, out=None):
        r = P.emb_lbm_step(E.forest, lattice, E.links, omega, d, out=out, pre=pre, phases=phases)
        assert P.emb_status_get() == P.EMB_OK
        return r

    # streaming: each population from its source, bit for bit
    src = orc.lbm_sources(w.R, w.levels, blocks, masks, lattice)
    moved = np.zeros_like(pop)
    for i in range(lattice):
        moved[i] = np.where(src[i] >= 0, pop[i, np.maximum(src[i], 0)], np.where(src[i] == -2, pop[i], np.float32(0)))
    moved[:, solid] = 0.0
    pre = torch.full_like(d, float("nan"))
    step(1, pre)
    np.testing.assert_array_equal(pre.cpu().numpy(), moved)
    # the boundary pass: the linked populations by the linear rule, no other one
    step(2, pre)
    _, f_i, f_opp, f_p, has = orc._link_pops(links, pop.astype(np.float64), orc.partner_cells(w.R, w.levels, blocks, masks, links["cell"], links["dir"]))
    inc = orc.bouzidi_incoming(links["q"], f_i, f_p, f_opp, has)
    opp = np.array([orc.opposite(int(x)) for x in links["dir"]])
    got = pre.cpu().numpy()
    at = (opp, links["cell"])
    # q within 2e-6 of the oracle's, float arithmetic of a few roundings
    assert np.all(np.abs(got[at] - inc) <= 1e-6 + 2e-5 * np.abs(inc))
    rest = np.ones(pop.shape, dtype=bool)
    rest[at] = False
    np.testing.assert_array_equal(got[rest], moved[rest])
    # collision, and the whole
    out = step(4, pre).cpu().numpy().astype(np.float64)
    ref = orc.lbm_step(w.R, w.levels, blocks, masks, links, pop.astype(np.float64), omega, lattice)
    assert np.all(np.abs(out - ref) <= 1e-6 + 2e-5 * np.abs(ref))
    both = torch.empty_like(d)
    step(3, both)
    assert torch.equal(both, pre)
    np.testing.assert_array_equal(step(4, both).cpu().numpy().astype(np.float64), out)
    stream = torch.empty_like(d)
    step(1, stream)
    np.testing.assert_array_equal(step(6, stream).cpu().numpy().astype(np.float64), out)
    # streaming and collision alone (5) leave the boundary pass out: other values at linked cells only
    plain = step(5, torch.empty_like(d)).cpu().numpy().astype(np.float64)
    cells = np.zeros(pop.shape[1], dtype=bool)
    cells[links["cell"]] = True
    np.testing.assert_array_equal(plain[:, ~cells], out[:, ~cells])
    assert np.any(plain[:, cells] != out[:, cells])
    whole = step(7, torch.empty_like(d)).cpu().numpy().astype(np.float64)
    assert np.all(np.abs(whole - out) <= 1e-7 + 4e-6 * np.abs(out))  # the same rules, contracted otherwise
