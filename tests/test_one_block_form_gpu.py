"""The FP32 form with one block per SM, which serves P1 and P2 meshes whose largest cell has more gather slots
than the blocks with several cells per SM take (from about 130 and 320 nodes): against the oracle, under every
schedule that belongs to it, and in batches whose other members run the other form.

The FP32 rows of M_i^-1 tell the forms apart: handles on this form carry them from the start, others
from the first request for the tensor-memory form on.  Tolerances are the reduced-precision bar of the other
FP32 tests (relative L2 <= 1e-5); schedules and neighbours change no bit of a cell's result.
"""
import numpy as np
import pytest

from inputs import states
from inputs.lattice import split_cube_lattice
from inputs.voronoi import periodic_voronoi
from tests.harness import Pair, rel_l2, rel_l2_fields

FP32_TOL = 1e-5
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def afe():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2605_00619_gb300 import afe as a
    a.lib()
    return a


def _params(afe, N, **over):
    return afe.afe_default_params(N, precision=afe.AFE_FP32, picard_tol=1e-6, cfl=0.1, **over)


def _carries_rows(afe, h):
    before = afe.afe_device_bytes(h)
    afe.afe_set_predictor_variant(h, 1)
    afe.afe_set_predictor_variant(h, 0)
    return afe.afe_device_bytes(h) == before


def _handle(afe, pm, N, **over):
    h = afe.create_from_polymesh(pm, _params(afe, N, **over))
    x = afe.afe_get_node_coords(h)
    afe.afe_set_state(h, states.density_wave(x, amp=0.1, vel=(0.5, -0.3, 0.2)))
    return h


# cubes with split edges: 8 sub-tets per edge part and direction, S / 2 + 3 nodes at P1, 5 S / 2 + 5 at P2
@pytest.mark.parametrize("N,splits,nodes", [(1, (11, 11, 10), 131), (2, (6, 5, 5), 325), (2, (8, 8, 8), 485)])
def test_large_cells_against_the_oracle(afe, N, splits, nodes):
    pr = Pair(split_cube_lattice((2, 1, 1), splits, d=0.5), _params(afe, N))
    plan = afe.afe_plan_info(pr.h)
    assert plan.fp32_shared == 1 and plan.max_nodes == nodes
    u0 = states.density_wave(pr.om.node_coords(), amp=0.1, vel=(0.5, -0.3, 0.2))
    pr.set_state(u0)
    dts = []
    for _ in range(2):
        info = pr.oracle_step()
        dts.append(info.dt)
        assert pr.lib_step(info.dt) == 0
    ref = pr.lib_state()
    assert rel_l2_fields(ref, pr.u) <= FP32_TOL
    for sched in (dict(cost_order=1), dict(narrow=1), dict(ring_cap=1), dict(cost_order=1, narrow=1, ring_cap=2)):
        afe.afe_set_schedule(pr.h, **sched)
        pr.set_state(u0)
        for dt in dts:
            assert pr.lib_step(dt) == 0
        np.testing.assert_array_equal(pr.lib_state(), ref, err_msg=str(sched))
    assert _carries_rows(afe, pr.h)
    pr.close()


def test_the_next_smaller_cells_take_the_other_form(afe):
    for N, splits, nodes in ((1, (11, 10, 10), 127), (2, (5, 5, 5), 305)):
        h = _handle(afe, split_cube_lattice((2, 1, 1), splits, d=0.5), N)
        assert afe.afe_plan_info(h).max_nodes == nodes and not _carries_rows(afe, h)
        afe.afe_mesh_destroy(h)


def _members(afe, N):
    splits = [(6, 5, 5), (8, 8, 8)] if N == 2 else [(11, 11, 10), (12, 12, 12)]
    visc = dict(equations=afe.AFE_NAVIER_STOKES, mu=0.01, kappa=-1.0, visc_dt_subtet=1)
    return [_handle(afe, split_cube_lattice((2, 1, 1), splits[0], d=0.5), N), _handle(afe, periodic_voronoi(3), N),
            _handle(afe, split_cube_lattice((3, 1, 1), splits[1], d=0.5), N, **visc),
            _handle(afe, periodic_voronoi(4), N, limiter=1, visc_dt_subtet=1), _handle(afe, periodic_voronoi(3), N, **visc)]


@pytest.mark.parametrize("sched", [{}, dict(cost_order=1), dict(cost_order=1, narrow=1, ring_cap=1)])
@pytest.mark.parametrize("N", [1, 2])
def test_batches_of_both_forms(afe, N, sched):
    """One predictor and one corrector launch per form: every member equals stepping it alone, bit for bit."""
    alone, mem = _members(afe, N), _members(afe, N)
    for h in alone:
        for _ in range(3):
            afe.afe_step(h, 0.0)
    b = afe.afe_batch_create(mem)
    before = afe.afe_batch_info(b)[2]
    afe.afe_batch_step_async(b, 0.0, 1, False)
    afe.afe_batch_sync(b, len(mem))
    # flags; means, limiter, time step, predictor and corrector per form, face fluxes
    assert afe.afe_batch_info(b)[2] - before == 1 + 2 + 1 + 2 + 2 + 1
    afe.afe_batch_set_schedule(b, **sched)
    afe.afe_batch_step_async(b, 0.0, 2, True)
    afe.afe_batch_sync(b, len(mem))
    afe.afe_batch_destroy(b)
    for i, (h, m) in enumerate(zip(alone, mem)):
        np.testing.assert_array_equal(afe.afe_get_state(m), afe.afe_get_state(h), err_msg=f"member {i}")
    assert [_carries_rows(afe, h) for h in mem] == [True, False, True, False, False]
    for h in alone + mem:
        afe.afe_mesh_destroy(h)


def test_autotuned_batch_of_both_forms(afe):
    """The candidates include the tensor-memory form for all members, whose rows the others then form."""
    alone, mem = _members(afe, 2), _members(afe, 2)
    for h in alone:
        for _ in range(2):
            afe.afe_step(h, 0.0)
    b = afe.afe_batch_create(mem)
    sched, best, default = afe.afe_batch_autotune(b, 2)
    assert 0 < best <= default * 1.0001
    afe.afe_batch_step_async(b, 0.0, 2, True)
    afe.afe_batch_sync(b, len(mem))
    afe.afe_batch_destroy(b)
    for i, (h, m) in enumerate(zip(alone, mem)):
        if sched.variant == 0:
            np.testing.assert_array_equal(afe.afe_get_state(m), afe.afe_get_state(h), err_msg=f"member {i}")
        else:
            assert rel_l2(afe.afe_get_state(m), afe.afe_get_state(h)) <= FP32_TOL
    for h in alone + mem:
        afe.afe_mesh_destroy(h)
