"""The unordered-pair sums where their scratch is not to be had: fewer tile offsets a launch, then the
row-by-row kernel, never an error that the row kernel would not give.

The fallback to the row kernel gives that kernel's bits; several launches add the columns of the same
tiles in another order: a few hundred tiles x 2^-47 as in test_pairsum_sym_gpu.py, 1e-9 of the sums."""
import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10

pytestmark = pytest.mark.gpu
FP64, MIXED = vv10.VV10_FP64, vv10.VV10_MIXED_TF32X3
SCRATCH = 7  # device allocations of a first energy call: E, U, W, block sums, energy, sums, then the scratch


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    return torch.device("cuda", 0)


def engine(g, dev):
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev, torch.float64)
    eng = vv10.VV10(0)
    eng.prepare(T(g.coords), T(g.weights), T(g.rho), T(g.grad_rho))
    return eng


def rows(eng, prec, on):
    """Fix the row kernel's own default shape, or go back to automatic."""
    vv10.vv10_set_tiles(eng.h, 3 * (prec == FP64), (1 if prec == FP64 else 2) if on else 0, 0)


@pytest.mark.parametrize("prec,n", [(MIXED, 11000), (FP64, 5000)], ids=["mixed", "fp64"])
def test_no_scratch_at_all(dev, prec, n):
    eng = engine(synth.random_points(n, seed=n), dev)
    try:
        vv10.vv10_debug_inject(eng.h, vv10.VV10_DEBUG_FAIL_ALLOC, SCRATCH)
        e, vr, vg = eng.energy_potential(prec)
        assert vv10.vv10_last_error(eng.h) == ""
        rows(eng, prec, True)
        e_rows, vr_rows, vg_rows = eng.energy_potential(prec)
        assert e == e_rows and torch.equal(vr, vr_rows) and torch.equal(vg, vg_rows)
        rows(eng, prec, False)  # room again: the unordered pairs
        e2, vr2, vg2 = eng.energy_potential(prec)
        for a, b in ((vr2, vr), (vg2, vg)):
            assert float((a - b).norm()) <= 1e-9 * float(b.norm())
    finally:
        eng.close()


def test_scratch_for_fewer_offsets(dev):
    g = synth.random_points(130_000, seed=5, spread=6.0)
    eng = engine(g, dev)
    try:
        launches = lambda: vv10.vv10_profile_read(eng.h)["pair_sums_EUW"][1]
        launches()
        vv10.vv10_debug_inject(eng.h, vv10.VV10_DEBUG_FAIL_ALLOC, SCRATCH)
        e, vr, vg = eng.energy_potential(MIXED)
        assert launches() > 1
        e1, vr1, vg1 = eng.energy_potential(MIXED)  # now with the scratch that was refused
        assert launches() == 1 and abs(e - e1) <= 1e-9 * abs(e1)
        for a, b in ((vr, vr1), (vg, vg1)):
            assert float((a - b).norm()) <= 1e-9 * float(b.norm())
    finally:
        eng.close()


@pytest.mark.parametrize("prec,n", [(MIXED, 11000), (FP64, 5000)], ids=["mixed", "fp64"])
def test_captured_without_scratch(dev, prec, n):
    """A call that never ran outside the capture but for the row kernel's buffers."""
    g = synth.random_points(n, seed=n)
    eng = engine(g, dev)
    vr, vg = (torch.zeros(g.n, dtype=torch.float64, device=dev) for _ in range(2))
    try:
        rows(eng, prec, True)
        _, vr_rows, vg_rows = eng.energy_potential(prec)
        rows(eng, prec, False)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            vv10.vv10_energy_potential(eng.h, prec, vr, vg, torch.cuda.current_stream(), False)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(vr, vr_rows) and torch.equal(vg, vg_rows)
    finally:
        eng.close()


@pytest.mark.parametrize("first,prec,later", [(5000, FP64, 4000), (4000, MIXED, 4000)], ids=["smaller", "fp64"])
def test_graph_survives_a_small_fp64_system(dev, first, prec, later):
    """The small FP64 kernel's partials, larger than a 5,000-point system's or an FP32 call's, leave the
    buffer in place that a captured call uses; prepared again as at the capture, it replays its bits."""
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev, torch.float64)
    a, b = synth.random_points(first, seed=1), synth.random_points(later, seed=2)
    da, db = ([T(x) for x in (g.coords, g.weights, g.rho, g.grad_rho)] for g in (a, b))
    eng = vv10.VV10(0)
    try:
        assert eng.prepare(*da) == first
        _, vr_ref, vg_ref = eng.energy_potential(prec)
        vr, vg = torch.zeros_like(vr_ref), torch.zeros_like(vg_ref)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            vv10.vv10_energy_potential(eng.h, prec, vr, vg, torch.cuda.current_stream(), False)
        eng.prepare(*db)
        eng.energy_potential(FP64)
        eng.prepare(*da)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(vr, vr_ref) and torch.equal(vg, vg_ref)
    finally:
        eng.close()
