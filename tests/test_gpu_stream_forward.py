"""The streaming forward convolution (radial weights into tensor memory, sums per
receiver over groups of four edges) through whole evaluations, against the FP64
oracle, where its layout can go wrong: receivers without edges, groups with one
to three empty slots, fewer chunks than helper warps, fewer receivers than CTAs,
every number of paths and tiles a block kind and degree gives.  The adjoint over
pairs reads blocked rows of dE/dm and takes the scalars 64 channels at a time with
a remainder of 32; "odd" has both.

Tolerances: FP32 1e-5 of the forces' norm, as everywhere for that path (sums of some
thousand products at 2^-24 each); BF16 5e-3 (operands at 2^-9).  The virial is a sum
over edges, W = -sum g_e (x) d_e, that may cancel to a small part of its terms: with
edge gradients within the same tolerance its error is at most that times sum |g_e| |d_e|."""

import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2402_03789_gb300 import _lib
from synth import ModelSpec, MODEL_SEVENNET0, benchmark_model, normal_weights, random_structure
from gpu_common import errors, get_model

pytestmark = pytest.mark.gpu

WIDE = ModelSpec(n_species=3, n_layers=2, mul=(32, 96, 64), avg_num_neigh=34.0)
SPECS = {"sevennet0": MODEL_SEVENNET0, "l2_32": benchmark_model(3, 32, 2), "l3_32": benchmark_model(3, 32, 3),
         # degree 1: chunked in both precisions (rows of gradients below 4,096 bytes), streaming in
         # BF16 alone (below 7,000), streaming in both
         "l1_32": ModelSpec(n_species=3, n_layers=3, mul=(32, 32), avg_num_neigh=34.0),
         "l1_64": ModelSpec(n_species=3, n_layers=3, mul=(64, 64), avg_num_neigh=34.0),
         "l1_96": ModelSpec(n_species=3, n_layers=3, mul=(96, 96), avg_num_neigh=34.0),
         "uneven": WIDE, "odd": ModelSpec(n_species=3, n_layers=3, mul=(96, 32, 64), avg_num_neigh=34.0)}


def _gas(n, isolated, box, seed):
    """Chains of one to five atoms in random places, and atoms alone (farther than every cutoff)."""
    rng = np.random.default_rng(seed)
    pos = [rng.uniform(0, box, 3)]

    def nearest(p):
        d = np.array(pos) - p
        d -= box * np.round(d / box)
        return (d * d).sum(1).min()

    while len(pos) < n:
        p = pos[-1] + np.array([1.9, 0.3, -0.2]) if len(pos) % 5 else rng.uniform(0, box, 3)
        if nearest(p) > 1.2:
            pos.append(p)
    while len(pos) < n + isolated:
        p = rng.uniform(0, box, 3)
        if nearest(p) > 5.2 ** 2:
            pos.insert(rng.integers(len(pos)), p)
    return np.array(pos), np.eye(3) * box, rng.integers(0, 3, n + isolated).astype(np.int32)


def _virial_terms(spec, pos, cell, species, edges):
    """sum |g_e| |d_e| over the edges, g_e = dE/dd_e of the oracle."""
    dst, src, shift = (torch.as_tensor(a) for a in edges)
    p = torch.as_tensor(pos)
    d = (p[src] - p[dst] + shift.double() @ torch.as_tensor(cell)).requires_grad_()
    wd = oracle.param_layout(spec).unpack(normal_weights(oracle.n_params(spec)))
    g, = torch.autograd.grad(oracle.model_energy(spec, wd, species, d, dst, src, len(pos)).sum(), d)
    return float((g.norm(dim=1) * d.detach().norm(dim=1)).sum())


def _check(spec, pos, cell, species, prec):
    model = get_model(spec)
    E, F, W = model.evaluate(pos, cell, species, precision=prec)
    Eo, Fo, Wo, _, edges = oracle.energy_forces_virial(spec, normal_weights(oracle.n_params(spec)), species, pos, cell)
    e, f, _ = errors(E, F, W, Eo, Fo, Wo, len(pos))
    w = np.linalg.norm(W - Wo) / _virial_terms(spec, pos, cell, species, edges)
    print(f"{prec}: E {e:.1e} F {f:.1e} W {w:.1e}")
    tol = 1e-5 if prec == "fp32" else 5e-3
    assert f <= tol and w <= tol and e <= (1e-6 if prec == "fp32" else 1e-5)


def _dirty(spec, prec):
    """An evaluation of 61 atoms with some 50 edges each: what it leaves in the message rows
    must not show in a later call."""
    s = random_structure({"Si": 21, "O": 40}, 2.4, 1.5, seed=11)
    get_model(spec).evaluate(s.pos, s.cell, s.species, precision=prec)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("name", list(SPECS))
def test_sparse_receivers(name, prec):
    spec = SPECS[name]
    pos, cell, species = _gas(37, 9, 40.0, 5)
    dst, *_ = oracle.neighbor_list(pos, cell, spec.r_cut)
    degree = np.bincount(dst, minlength=len(pos))
    assert (degree == 0).sum() >= 9 and {1, 2, 3} <= set(degree % 4)
    _dirty(spec, prec)
    _check(spec, pos, cell, species, prec)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("name,counts", [("sevennet0", {"Si": 2, "O": 3}), ("l2_32", {"Si": 50, "O": 101}),
                                         ("l3_32", {"Si": 21, "O": 40}), ("l1_32", {"Si": 21, "O": 40}),
                                         ("l1_64", {"Si": 21, "O": 40}), ("l1_96", {"Si": 21, "O": 40}),
                                         ("uneven", {"N": 31, "O": 60}), ("odd", {"Si": 11, "O": 20})])
def test_dense_cells(name, counts, prec):
    s = random_structure(counts, 2.4, 1.5, seed=11)
    _check(SPECS[name], s.pos, s.cell, s.species, prec)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("name", ["sevennet0", "l3_32", "l1_96"])
def test_single_atom_and_isolated_atoms(name, prec):
    """No edges at all: messages of zero, so the self-connection's energy."""
    spec = SPECS[name]
    cell = np.eye(3) * 30.0
    for pos in (np.zeros((1, 3)), np.array([[0.0, 0, 0], [15.0, 15, 15]])):
        sp = np.arange(len(pos), dtype=np.int32)
        _dirty(spec, prec)
        E, F, W = get_model(spec).evaluate(pos, cell, sp, precision=prec)
        Eo, *_ = oracle.energy_forces_virial(spec, normal_weights(oracle.n_params(spec)), sp, pos, cell)
        assert abs(E - Eo) <= (1e-6 if prec == "fp32" else 1e-5) * len(pos)
        assert np.abs(F).max() == 0 and np.abs(W).max() == 0


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
