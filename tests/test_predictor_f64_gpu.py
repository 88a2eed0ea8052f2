"""The FP64 predictor whose M_i^-1 product is formed from digits on the tensor cores: sizes at the
edges of its tiles, lists and chunks against the oracle (the FP64 bar of the other tests, a relative
L-infinity of 1e-11), badly scaled states, and states that are not finite.
"""
import numpy as np
import pytest

from inputs import states
from inputs.lattice import split_cube_lattice
from inputs.voronoi import periodic_voronoi
from tests.harness import Pair, rel_l2_fields, rel_linf

FP64_TOL = 1e-11
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def afe():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2605_00619_gb300 import afe as a
    a.lib()
    return a


# one 16-row tile (15 nodes) up to 32 tiles: one, two and five chunks of 112 columns; cells of 623 nodes
# beyond its shared memory (the global-scratch kernel)
@pytest.mark.parametrize("visc", [False, True])
@pytest.mark.parametrize("N,splits", [(1, (1, 1, 1)), (1, (3, 3, 3)), (2, (1, 1, 1)), (2, (3, 2, 2)), (3, (1, 1, 1)),
                                      (3, (3, 3, 3)), (3, (4, 4, 3))])
def test_cell_sizes_against_the_oracle(afe, N, splits, visc):
    pm = split_cube_lattice((2, 1, 1), splits, d=0.5)
    over = dict(equations=afe.AFE_NAVIER_STOKES, mu=0.01, kappa=-1.0, visc_dt_subtet=1) if visc else {}
    pr = Pair(pm, afe.afe_default_params(N, cfl=0.1, **over))
    pr.set_state(states.density_wave(pr.om.node_coords(), amp=0.1, vel=(0.5, -0.3, 0.2)))
    info = pr.oracle_step()
    assert pr.lib_step(info.dt) == 0
    assert rel_linf(pr.lib_state(), pr.u) <= FP64_TOL
    pr.close()


@pytest.mark.parametrize("rho,speed,p", [(1.2, 30.0, 1e5), (1e-6, 1e4, 1e-2), (1e6, 1e-3, 1.0)])
def test_scales_of_the_variables(afe, rho, speed, p):
    """Right-hand sides whose variables lie many powers of two apart (each has its own scale)."""
    pm = periodic_voronoi(3)
    pr = Pair(pm, afe.afe_default_params(2, cfl=0.1))
    x = pr.om.node_coords()
    w = 1 + 0.1 * np.sin(2 * np.pi * x.sum(axis=1))
    pr.set_state(states.primitive_to_conserved(rho * w, speed * np.stack([w, 2 - w, w * 0 + 1], 1), p * (2 - w)))
    info = pr.oracle_step()
    # a supersonic case whose new pressure is negative somewhere, in the oracle too, is reported so
    r, _, q = states.conserved_to_primitive(pr.u)
    admissible = np.isfinite(pr.u).all() and (r > 0).all() and (q > 0).all()
    assert pr.lib_step(info.dt, check=False) in ((0, 5) if admissible else (afe.AFE_ENONFINITE,))
    if admissible:
        assert rel_l2_fields(pr.lib_state(), pr.u) <= FP64_TOL
    pr.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_state_that_is_not_finite_is_reported(afe, bad):
    pm = periodic_voronoi(3)
    h = afe.create_from_polymesh(pm, afe.afe_default_params(2, cfl=0.1, picard_max=8))
    u = states.density_wave(afe.afe_get_node_coords(h))
    u[7, 4] = bad
    afe.afe_set_state(h, u)
    assert afe.afe_step(h, 1e-4, check=False) == afe.AFE_ENONFINITE
    # the other cells that do not touch the bad one keep finite states
    v = afe.afe_get_state(h)
    ptr = afe.afe_node_ptr(h, pm.n_cells)
    assert not np.isfinite(v[ptr[0]:ptr[1]]).all() and np.isfinite(v).any()
    afe.afe_mesh_destroy(h)
