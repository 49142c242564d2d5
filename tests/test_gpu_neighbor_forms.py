"""Neighbour build (a warp per receiver, 32 bins at a time) and the reductions per
structure (512 atoms a block) at the sizes where their loops can go wrong."""

import numpy as np
import pytest

import oracle
from synth import MODEL_TINY, normal_weights, random_structure
from gpu_common import edge_set, get_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pbc", [(1, 1, 1), (1, 0, 1), (0, 0, 1), (0, 0, 0)])
@pytest.mark.parametrize("n,edges", [(1, (3.1, 2.6, 4.0)), (33, (6.0, 5.2, 9.0)), (70, (17.0, 8.0, 5.1))])
def test_bins_in_range_and_open_directions(n, edges, pbc):
    """27 to 225 bins in range (several turns of 32), several images of a bin, open
    directions with atoms outside the cell, a skewed cell."""
    rng = np.random.default_rng(n)
    cell = np.diag(edges) + np.array([[0, 0, 0], [0.9, 0, 0], [-0.4, 0.7, 0]])
    pos = rng.uniform(-0.6, 1.6, (n, 3)) @ cell
    model = get_model(MODEL_TINY)
    dst, src, sh = model.neighbors(pos, cell, pbc)
    od, os_, osh = oracle.neighbor_list_bruteforce(pos, cell, MODEL_TINY.r_cut, [bool(p) for p in pbc])
    assert edge_set(dst, src, sh, pos, cell, MODEL_TINY.r_cut) == edge_set(od, os_, osh, pos, cell, MODEL_TINY.r_cut)
    assert len(dst) == len(set(zip(dst, src, map(tuple, sh))))


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_energy_and_virial_of_supercells(prec):
    """Supercells of 1, 511, 512, 513 and 1,025 atoms: n copies of a base cell have n
    times its energy and virial (atoms see the same surroundings; the sums are FP64,
    so what is left is FP32 rounding of the coordinates: 1e-6 an atom, 1e-5 of W)."""
    spec = MODEL_TINY
    model = get_model(spec)
    w = normal_weights(oracle.n_params(spec))
    for counts, reps in (({"Si": 1}, (1, 1, 1)), ({"Si": 24, "O": 49}, (7, 1, 1)), ({"Si": 3, "O": 5}, (4, 4, 4)),
                         ({"Si": 6, "O": 13}, (3, 3, 3)), ({"Si": 14, "O": 27}, (5, 5, 1))):
        s = random_structure(counts, 2.3, 1.6, seed=len(reps) + reps[0])
        n = int(np.prod(reps))
        shifts = np.stack(np.meshgrid(*[np.arange(r) for r in reps], indexing="ij"), -1).reshape(-1, 3) @ s.cell
        pos = (s.pos[None] + shifts[:, None]).reshape(-1, 3)
        E, F, W = model.evaluate(pos, s.cell * np.array(reps)[:, None], np.tile(s.species, n), precision=prec)
        Eo, Fo, Wo, *_ = oracle.energy_forces_virial(spec, w, s.species, s.pos, s.cell)
        e_tol, w_tol = (1e-6, 1e-5) if prec == "fp32" else (1e-5, 5e-3)
        assert abs(E - n * Eo) <= e_tol * len(pos)
        assert np.linalg.norm(W - n * Wo) <= w_tol * n * max(np.linalg.norm(Wo), 1e-12)
        assert np.linalg.norm(F - np.tile(Fo, (n, 1))) <= w_tol * max(np.sqrt(n) * np.linalg.norm(Fo), 1e-4)
