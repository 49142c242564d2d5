"""The streaming forward convolution (radial weights into tensor memory, sums per
receiver over groups of four edges) through whole evaluations, against the FP64
oracle, where its layout can go wrong: receivers without edges, groups with one
to three empty slots, fewer chunks than helper warps, fewer receivers than CTAs,
every number of paths and tiles a block kind and degree gives.  The adjoint over
pairs reads blocked rows of dE/dm and takes the scalars 64 channels at a time with
a remainder of 32; "odd" has both.

Tolerances: FP32 1e-5 of the forces' norm, as everywhere for that path (sums of
some thousand products at 2^-24 each); BF16 5e-3 (operands at 2^-9)."""

import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2402_03789_gb300 import _lib
from synth import ModelSpec, MODEL_SEVENNET0, benchmark_model, random_structure
from gpu_common import errors, get_model

pytestmark = pytest.mark.gpu

WIDE = ModelSpec(n_species=3, n_layers=2, mul=(32, 96, 64), avg_num_neigh=34.0)
SPECS = {"sevennet0": MODEL_SEVENNET0, "l2_32": benchmark_model(3, 32, 2), "l3_32": benchmark_model(3, 32, 3),
         "uneven": WIDE, "odd": ModelSpec(n_species=3, n_layers=3, mul=(96, 32, 64), avg_num_neigh=34.0)}


def _gas(n, box, seed):
    """Atoms far apart on a line plus one cluster of 2..5: degrees 0 to 4."""
    rng = np.random.default_rng(seed)
    pos = [rng.uniform(0, box, 3)]
    while len(pos) < n:
        p = pos[-1] + np.array([1.9, 0.3, -0.2]) if len(pos) % 5 else rng.uniform(0, box, 3)
        d = np.array(pos) - p
        d -= box * np.round(d / box)
        if (d * d).sum(1).min() > 1.2:
            pos.append(p)
    return np.array(pos), np.eye(3) * box, rng.integers(0, 3, n).astype(np.int32)


def _check(spec, pos, cell, species, prec):
    from synth import normal_weights
    model = get_model(spec)
    E, F, W = model.evaluate(pos, cell, species, precision=prec)
    Eo, Fo, Wo, *_ = oracle.energy_forces_virial(spec, normal_weights(oracle.n_params(spec)), species, pos, cell)
    e, f, w = errors(E, F, W, Eo, Fo, Wo, len(pos))
    print(f"{prec}: E {e:.1e} F {f:.1e} W {w:.1e}")
    assert f <= (1e-5 if prec == "fp32" else 5e-3) and e <= (1e-6 if prec == "fp32" else 1e-5)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("name", list(SPECS))
def test_sparse_receivers(name, prec):
    pos, cell, species = _gas(37, 34.0, 5)
    _check(SPECS[name], pos, cell, species, prec)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("name,counts", [("sevennet0", {"Si": 2, "O": 3}), ("l2_32", {"Si": 50, "O": 101}),
                                         ("l3_32", {"Si": 21, "O": 40}), ("uneven", {"N": 31, "O": 60}), ("odd", {"Si": 11, "O": 20})])
def test_dense_cells(name, counts, prec):
    s = random_structure(counts, 2.4, 1.5, seed=11)
    _check(SPECS[name], s.pos, s.cell, s.species, prec)


def test_single_atom_and_isolated_atoms():
    spec = SPECS["sevennet0"]
    cell = np.eye(3) * 30.0
    for pos in (np.zeros((1, 3)), np.array([[0.0, 0, 0], [15.0, 15, 15]])):
        E, F, W = get_model(spec).evaluate(pos, cell, np.zeros(len(pos), np.int32), precision="bf16")
        assert np.isfinite(E) and np.abs(F).max() == 0 and np.abs(W).max() == 0


def _set_wait_limit(model, cycles):
    model.lib.sn_test_set_wait_limit(model.handle, ctypes.c_uint32(cycles))


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_waits_that_run_out_end_the_call(prec):
    """With no time for any wait, the first one that is not over at once gives up: every
    warp must leave its pipeline together and the call report it (status ETIMEDOUT), and
    the tensor memory must be free for the next call, which gives the same bits as before."""
    s = random_structure({"N": 31, "O": 60}, 2.4, 1.5, seed=11)
    model = get_model(WIDE)
    before = model.evaluate(s.pos, s.cell, s.species, precision=prec)
    try:
        _set_wait_limit(model, 0)
        with pytest.raises(RuntimeError) as err:
            model.evaluate(s.pos, s.cell, s.species, precision=prec)
        assert err.value.status == _lib.ETIMEDOUT
    finally:
        _set_wait_limit(model, 4000000000)
    after = model.evaluate(s.pos, s.cell, s.species, precision=prec)
    assert after[0] == before[0] and np.array_equal(after[1], before[1]) and np.array_equal(after[2], before[2])


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_messages_of_a_timed_out_forward_are_nan(prec):
    """A block whose waits ran out hands on NaN, not partial sums or what an earlier call
    left: the energy on the device is NaN, and the status is still the timeout's."""
    s = random_structure({"N": 31, "O": 60}, 2.4, 1.5, seed=11)
    model = get_model(WIDE)
    pos = torch.tensor(s.pos, dtype=torch.float64, device="cuda")
    args = ([0, s.n_atoms], s.cell[None], torch.tensor(s.species, dtype=torch.int32, device="cuda"), pos, prec)
    out = model.evaluate_batch_dev(*args)
    assert all(torch.isfinite(t).all() for t in out)
    try:
        _set_wait_limit(model, 0)
        with pytest.raises(RuntimeError) as err:
            model.evaluate_batch_dev(*args, out=out)
    finally:
        _set_wait_limit(model, 4000000000)
    torch.cuda.synchronize()
    assert err.value.status == _lib.ETIMEDOUT
    assert torch.isnan(out[0]).all()
