"""Edge capacity overflow and its retry.  The asynchronous neighbour build writes
into preallocated edge arrays (64 per atom at first) and reports on the device
when a structure needs more; the evaluation then runs again with the count the
device reported, and a serving batch reruns through the same path.  A dense
cell (about 95 neighbours per atom within 5 A) forces both."""

import time

import numpy as np
import pytest

import oracle
from synth import MODEL_SEVENNET0, benchmark_model, normal_weights, random_structure
from gpu_common import errors

pytestmark = pytest.mark.gpu


def _dense():
    s = random_structure({"Si": 20, "O": 40}, 6.0, 1.0, seed=71)
    dst, _, _ = oracle.neighbor_list(s.pos, s.cell, MODEL_SEVENNET0.r_cut)
    assert len(dst) / s.n_atoms > 64          # beyond the first capacity
    return s


def test_dense_cell_is_retried_with_more_edge_room():
    import paper_2402_03789_gb300 as sn
    spec = MODEL_SEVENNET0
    w = normal_weights(oracle.n_params(spec))
    s = _dense()
    model = sn.SevenNet(spec, w)              # a fresh workspace
    E, F, W = model.evaluate(s.pos, s.cell, s.species, "fp32")
    Eo, Fo, Wo, *_ = oracle.energy_forces_virial(spec, w, s.species, s.pos, s.cell)
    e_pa, f_rel, w_rel = errors(E, F, W, Eo, Fo, Wo, s.n_atoms)
    assert e_pa <= 1e-6 and f_rel <= 1e-5 and w_rel <= 1e-5, (e_pa, f_rel, w_rel)
    model.close()


def test_server_reruns_a_batch_beyond_its_slot_capacity():
    import paper_2402_03789_gb300 as sn
    spec = MODEL_SEVENNET0
    w = normal_weights(oracle.n_params(spec))
    s = _dense()
    model = sn.SevenNet(spec, w)
    E, F, W = model.evaluate(s.pos, s.cell, s.species, "fp32")
    # a slot of 64 atoms (about 51 KB each for this model): its 4,096 edges are fewer than the cell needs
    srv = sn.Server(model, hbm_budget_bytes=3_300_000, n_streams=1, max_batch_structs=4, precision="fp32")
    t = srv.submit(s.pos, s.cell, s.species)
    r, t0 = None, time.time()
    while r is None and time.time() - t0 < 60:
        r = srv.poll(t)
        time.sleep(0.001)
    assert r is not None
    assert r["energy"] == E and np.array_equal(r["forces"], F) and np.array_equal(r["virial"], W)
    srv.close()
    model.close()


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_server_memory_stays_within_its_budget(prec):
    """The slots' allocations against the budget, for a model whose rows of gradients
    (7,168 bytes an atom) are smaller than the FP32 hidden activations of 32 pairs that
    share their memory (8,192).  Each of the about 45 allocations of a slot may round up to 2 MiB."""
    import torch
    import paper_2402_03789_gb300 as sn
    spec = benchmark_model(5, 32, 2)
    model = sn.SevenNet(spec, normal_weights(oracle.n_params(spec)))
    s = random_structure({"Si": 20, "O": 40}, 2.2, 1.6, seed=31)
    model.evaluate(s.pos, s.cell, s.species, prec)            # its own workspace and kernels
    budget, slots = 12 << 30, 2
    free = torch.cuda.mem_get_info()[0]
    srv = sn.Server(model, hbm_budget_bytes=budget, n_streams=slots, max_batch_structs=32, precision=prec)
    used = free - torch.cuda.mem_get_info()[0]
    srv.close()
    model.close()
    assert 0.97 * budget <= used <= budget + slots * 45 * (2 << 20)


def test_call_after_one_that_ran_out_of_memory():
    """24,000 atoms with 600 MB of device memory left (they need 1.2 GB) end with ENOMEM
    half way through the workspace; a small call after that allocates again what the
    failed one had given back, and gives the bits of before."""
    import torch
    import paper_2402_03789_gb300 as sn
    spec = MODEL_SEVENNET0
    model = sn.SevenNet(spec, normal_weights(oracle.n_params(spec)))
    s = random_structure({"Si": 64, "O": 128}, 2.2, 1.6, seed=5)
    before = model.evaluate(s.pos, s.cell, s.species, "fp32")
    rng = np.random.default_rng(0)
    k = 29                                        # a lattice of 24,389 sites, 2.6 A apart
    pos = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3) * 2.6
    species = rng.integers(0, 3, len(pos)).astype(np.int32)
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - (600 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(sn.SevenNetError) as err:
            model.evaluate(pos, np.eye(3) * (2.6 * k), species, "fp32")
        assert err.value.status == -2
        after = model.evaluate(s.pos, s.cell, s.species, "fp32")
    finally:
        del filler
        torch.cuda.empty_cache()
    assert after[0] == before[0] and np.array_equal(after[1], before[1]) and np.array_equal(after[2], before[2])
    model.close()


def test_hidden_activations_that_do_not_fit_leave_the_chunked_forward():
    """A list of some 100 edges an atom, where the pairs' FP32 hidden activations (129 edges of
    room: 16.5 KB an atom) are larger than the gradients whose memory they share (7.2 KB):
    with memory for the gradients alone the call still runs, in the chunked kernels."""
    import dataclasses
    import torch
    import paper_2402_03789_gb300 as sn
    spec = dataclasses.replace(benchmark_model(3, 32, 2), r_cut=7.0)
    w = normal_weights(oracle.n_params(spec))
    rng = np.random.default_rng(3)
    k = 28
    grid = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)
    pos, cell = (grid + rng.uniform(-0.16, 0.16, grid.shape)) * 2.4, np.eye(3) * (2.4 * k)
    species = rng.integers(0, 3, len(pos)).astype(np.int32)
    torch.cuda.empty_cache()

    def run():
        model = sn.SevenNet(spec, w)
        first = model.lib.sevennet_launch_count()
        out = model.evaluate(pos, cell, species, "fp32")
        return model, out, model.lib.sevennet_launch_count() - first

    free = torch.cuda.mem_get_info()[0]
    model, (E1, F1, W1), n1 = run()
    used = free - torch.cuda.mem_get_info()[0]
    model.close()
    short = len(pos) * (16500 - 7200) // 2
    filler = torch.empty(torch.cuda.mem_get_info()[0] - used + short, dtype=torch.uint8, device="cuda")
    try:
        model, (E2, F2, W2), n2 = run()
        model.close()
    finally:
        del filler
        torch.cuda.empty_cache()
    assert n2 < n1                                # no hidden layers once per pair, no groups of four
    e_pa, f_rel, w_rel = errors(E2, F2, W2, E1, F1, W1, len(pos))
    assert e_pa <= 1e-6 and f_rel <= 1e-5 and w_rel <= 1e-5
