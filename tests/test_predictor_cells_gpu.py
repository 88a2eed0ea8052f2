"""The FP32 predictor with several cells in flight per SM: sizes at the edges of its tiles, lists
and chunks against the oracle, and its two block shapes against each other.

Tolerances are the reduced-precision bar of the other FP32 tests (relative L2 <= 1e-5); the block
shape, the launch it runs in and its neighbours change no bit of a cell's result.
"""
import numpy as np
import pytest

from inputs import states
from inputs.lattice import split_cube_lattice
from inputs.voronoi import periodic_voronoi
from tests.harness import Pair, rel_l2_fields

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


# cubes with split edges: 24 sub-tets and 15 nodes (one 16-row tile) at N = 1 up to 72 sub-tets and 511
# nodes at N = 3 (gather slots past the first of each thread; the cell centre's list is 24 long, one
# thread's, or longer, shared by a warp)
@pytest.mark.parametrize("visc", [False, True])
@pytest.mark.parametrize("splits", [(1, 1, 1), (2, 1, 1), (3, 2, 2), (3, 3, 3)])
@pytest.mark.parametrize("N", [1, 2, 3])
def test_cell_sizes_against_the_oracle(afe, N, splits, visc):
    pm = split_cube_lattice((2, 1, 1), splits, d=0.5)
    over = dict(equations=afe.AFE_NAVIER_STOKES, mu=0.01, kappa=-1.0, visc_dt_subtet=1) if visc else {}
    p = afe.afe_default_params(N, precision=afe.AFE_FP32, picard_tol=1e-6, cfl=0.1, **over)
    pr = Pair(pm, p)
    assert afe.afe_plan_info(pr.h).fp32_shared == 1
    pr.set_state(states.density_wave(pr.om.node_coords(), amp=0.1, vel=(0.5, -0.3, 0.2)))
    for _ in range(2):
        info = pr.oracle_step()
        assert pr.lib_step(info.dt) == 0
    assert rel_l2_fields(pr.lib_state(), pr.u) <= FP32_TOL
    pr.close()


@pytest.mark.parametrize("N", [1, 2, 3])
def test_block_shapes_agree_bit_for_bit(afe, N):
    """A mesh of few cells alone (more warps per cell) and in a batch of many (fewer), where a
    limited explosion's viscous cells take the other kernel."""
    pm, big = periodic_voronoi(4), periodic_voronoi(7)

    def handle(mesh, **over):
        p = afe.afe_default_params(N, precision=afe.AFE_FP32, picard_tol=1e-6, cfl=0.1, **over)
        h = afe.create_from_polymesh(mesh, p)
        x = afe.afe_get_node_coords(h)
        u = states.spherical_riemann(x, centre=(0.5, 0.5, 0.5), radius=0.25, alpha0=0.1) if over else \
            states.density_wave(x)
        afe.afe_set_state(h, u)
        return h

    alone = [handle(pm), handle(pm, limiter=1, visc_dt_subtet=1)]
    for h in alone:
        for _ in range(3):
            afe.afe_step(h, 0.0)
    mem = [handle(pm), handle(pm, limiter=1, visc_dt_subtet=1), handle(big)]
    b = afe.afe_batch_create(mem)
    afe.afe_batch_step_async(b, 0.0, 3, True)
    afe.afe_batch_sync(b, len(mem))
    afe.afe_batch_destroy(b)
    for h, m in zip(alone, mem):
        np.testing.assert_array_equal(afe.afe_get_state(m), afe.afe_get_state(h))
    for h in alone + mem:
        afe.afe_mesh_destroy(h)


def test_a_batch_keeps_every_members_form(afe):
    """Cells too large for two blocks per SM (623 nodes) beside small ones: each member's result is
    that of stepping it alone, bit for bit."""
    def handles():
        out = []
        for pm in (split_cube_lattice((2, 1, 1), (4, 4, 3), d=0.5), periodic_voronoi(3),
                   split_cube_lattice((3, 1, 1), (4, 4, 3), d=0.5), periodic_voronoi(4)):
            p = afe.afe_default_params(3, precision=afe.AFE_FP32, picard_tol=1e-6, cfl=0.1)
            h = afe.create_from_polymesh(pm, p)
            afe.afe_set_state(h, states.density_wave(afe.afe_get_node_coords(h), amp=0.1))
            out.append(h)
        return out

    alone, mem = handles(), handles()
    for h in alone:
        for _ in range(3):
            afe.afe_step(h, 0.0)
    b = afe.afe_batch_create(mem)
    afe.afe_batch_step_async(b, 0.0, 1, False)
    afe.afe_batch_sync(b, len(mem))
    afe.afe_batch_set_schedule(b, cost_order=1)
    afe.afe_batch_step_async(b, 0.0, 2, True)
    afe.afe_batch_sync(b, len(mem))
    afe.afe_batch_destroy(b)
    for h, m in zip(alone, mem):
        np.testing.assert_array_equal(afe.afe_get_state(m), afe.afe_get_state(h))
    for h in alone + mem:
        afe.afe_mesh_destroy(h)


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("N", [1, 3])
def test_a_new_handle_is_complete_on_any_stream(afe, N, bits):
    """Creation leaves no set-up work behind on its stream: a handle moved to another stream at once steps
    like one that was waited for, bit for bit."""
    import torch
    pm = periodic_voronoi(6)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    p = afe.afe_default_params(N, precision=afe.AFE_FP32 if bits == 32 else afe.AFE_FP64,
                               picard_tol=1e-6 if bits == 32 else 1e-12, cfl=0.1)
    ref = afe.create_from_polymesh(pm, p)
    u = states.density_wave(afe.afe_get_node_coords(ref))
    du = torch.from_numpy(u).cuda()
    torch.cuda.synchronize()
    afe.afe_set_state(ref, u)
    assert afe.afe_step(ref, 0.0) == 0
    for _ in range(3):
        h = afe.create_from_polymesh(pm, p, a.cuda_stream)
        afe.afe_set_stream(h, b.cuda_stream)
        afe.afe_set_state_device(h, du.data_ptr())
        assert afe.afe_step(h, 0.0) == 0
        np.testing.assert_array_equal(afe.afe_get_state(h), afe.afe_get_state(ref))
        afe.afe_mesh_destroy(h)
    afe.afe_mesh_destroy(ref)
