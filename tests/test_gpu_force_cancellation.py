"""The force where its terms cancel: the sums and the terms carry FP64's 53 bits, so what is left
of them is right to 2^-51 of the summed magnitudes.  References in exact rationals."""
from __future__ import annotations

from fractions import Fraction

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
    return E, o, partner


def _exact(orc, cell, d, q, partner, pop):
    """(F, sum |m|) of the links, exactly."""
    C = orc.directions()
    F, total = [Fraction(0)] * 3, Fraction(0)
    for k in range(len(cell)):
        qq, f_i = Fraction(float(q[k])), Fraction(float(pop[d[k], cell[k]]))
        if qq < Fraction(1, 2):
            g = f_i if partner[k] < 0 else 2 * qq * f_i + (1 - 2 * qq) * Fraction(float(pop[d[k], partner[k]]))
        else:
            f_o = Fraction(float(pop[orc.opposite(int(d[k])), cell[k]]))
            g = (f_i + (2 * qq - 1) * f_o) / (2 * qq)
        F = [F[x] + int(C[d[k]][x]) * (f_i + g) for x in range(3)]
        total += abs(f_i + g)
    return F, total


def _force(E, cell, d, q, pop):
    import torch

    import paper_2512_01251_gb300 as P
    c, dd, qq = torch.from_numpy(cell.astype(np.int32)).cuda(), torch.from_numpy(d.astype(np.uint8)).cuda(), torch.from_numpy(q).cuda()
    p = torch.from_numpy(pop).cuda()
    fixed = torch.empty(3, dtype=torch.float32, device="cuda")
    P.emb_mex_force_noalloc(E.forest, 27, c, dd, qq, p, fixed)
    return [x.cpu().numpy().astype(np.float64) for x in (P.emb_mex_force(E.forest, 27, c, dd, qq, p), fixed)]


def _check(orc, E, cell, d, q, partner, pop):
    ref, total = _exact(orc, cell, d, q, partner, pop)
    for F in _force(E, cell, d, q, pop):
        for x in range(3):
            err = abs(Fraction(float(F[x])) - ref[x])
            assert err <= Fraction(1, 1 << 24) * abs(ref[x]) + Fraction(1, 1 << 51) * total, (x, float(err), float(total))


@pytest.mark.parametrize("side", ["below", "above"])
@pytest.mark.parametrize("seed", range(12))
def test_two_links_against_each_other(orc, body, side, seed):
    """Opposite links with the same q next to 1/2 and populations one ulp apart: the force is
    about 2^-44 of each term."""
    E, o, partner = body
    rng = np.random.default_rng(seed)
    cell, d = np.asarray(o["links"]["cell"]), np.asarray(o["links"]["dir"])
    has = np.flatnonzero(partner >= 0)
    for _ in range(200):
        i = rng.choice(has)
        j = rng.choice(has[d[has] == orc.opposite(int(d[i]))])
        if len({int(cell[i]), int(cell[j]), int(partner[i]), int(partner[j])}) == 4:
            break
    k = np.array([i, j])
    steps = int(rng.integers(1, 16))
    q = np.float32(0.5)
    for _ in range(steps):
        q = np.nextafter(q, np.float32(0 if side == "below" else 1))
    pop = np.zeros((27, 64 * len(o["blocks"][-1])), dtype=np.float32)
    f_i, f = np.float32(rng.uniform(0.5, 2)), np.float32(rng.uniform(0.5, 2))
    pop[d[k], cell[k]] = f_i
    two = np.array([f, np.nextafter(f, np.float32(4))])
    if side == "below":
        pop[d[k], partner[k]] = two
    else:
        pop[[orc.opposite(int(x)) for x in d[k]], cell[k]] = two
    _check(orc, E, cell[k], d[k], np.array([q, q], dtype=np.float32), partner[k], pop)


def test_uniform_populations_around_a_closed_body(orc, body):
    """The lattice's weights in every cell: the force of a body in a fluid at rest."""
    E, o, partner = body
    w = orc.lattice_weights(27).astype(np.float32)
    pop = np.repeat(w[:, None], 64 * len(o["blocks"][-1]), 1)
    cell, d = np.asarray(o["links"]["cell"]), np.asarray(o["links"]["dir"])
    _check(orc, E, cell, d, E.links["q"].cpu().numpy(), partner, pop)
