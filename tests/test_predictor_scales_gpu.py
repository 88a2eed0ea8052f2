"""The FP32 form on cells with sub-tets of very different size, and at lengths far from one.

The predictor and the corrector multiply by M_i^-1 in pairs of 16-bit values, whose exponent range is
a small part of FP32's: what keeps every row of a graded matrix, and every scale of a mesh, at full
precision are the powers of two that rows, columns and variables are scaled by.
"""
import numpy as np
import pytest

from inputs import states
from inputs.lattice import split_cube_lattice
from tests.harness import rel_l2_fields

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


def _thin_lattice(eps):
    """Two cubes whose edges along x are split close to their lower end: next to every split point lies a
    fan sub-tet that is eps as long in x as its neighbours.  Returns the mesh and its sub-tets' volumes."""
    pm = split_cube_lattice((2, 1, 1), (2, 1, 1), d=0.5)
    x = pm.xyz[:, 0]
    mid = np.isin(np.round(x / 0.25).astype(int), (1, 3)) & np.isin(pm.xyz[:, 1], (0.0, 0.5)) & np.isin(pm.xyz[:, 2], (0.0, 0.5))
    assert mid.sum() == 8
    pm.xyz[mid, 0] += (2 * eps - 1) * 0.25
    v = pm.xyz[pm.subtet_vtx]
    return pm, np.abs(np.linalg.det(v[:, 1:] - v[:, :1])) / 6


@pytest.mark.parametrize("eps", [1e-4, 1e-9])
@pytest.mark.parametrize("N", [2, 3])
def test_cells_with_thin_sub_tets(afe, N, eps):
    """The update of the nodes that touch no thin sub-tet against the FP64 form's, whose own error is that of
    64 bits.  FP32 rounding of the fluxes (6e-8 of up to 3.5) enters the update through derivatives (at most
    2 N^2 over a sub-tet's length of 0.25) and the scaled mass matrix (condition 17, its root bounds the L2
    error): 6e-5 at N = 3, against an update of about 0.2 per entry, 3e-4.  The bar is 1e-3.  (The update over
    dt resolves 64 bits of the state to 1e-5 at the smaller dt.)"""
    pm, vol = _thin_lattice(eps)
    du, keep = {}, None
    for prec in (afe.AFE_FP64, afe.AFE_FP32):
        p = afe.afe_default_params(N, precision=prec, picard_tol=1e-6 if prec == afe.AFE_FP32 else 1e-12, cfl=0.1)
        h = afe.create_from_polymesh(pm, p)
        if prec == afe.AFE_FP32:
            assert afe.afe_plan_info(h).fp32_shared == 1
        x = afe.afe_get_node_coords(h)
        u0 = states.density_wave(x, amp=0.1, vel=(0.5, -0.3, 0.2))
        afe.afe_set_state(h, u0)
        assert afe.afe_step(h, 1e-2 * eps) == 0
        du[prec] = (afe.afe_get_state(h) - u0) / (1e-2 * eps)
        # nodes in a thin sub-tet lie within its thickness of the triangle (centre, face centre, corner)
        touch = np.zeros(len(x), bool)
        for t in pm.subtet_vtx[vol < 1e-2 * vol.max()]:
            w = pm.xyz[t[:3]]
            lam = np.linalg.lstsq(np.vstack([w.T, np.ones(3)]), np.vstack([x.T, np.ones(len(x))]), rcond=None)[0]
            touch |= (lam > -1e-3).all(0) & (np.abs(w.T @ lam - x.T).max(0) < 2 * eps)
        assert keep is None or (keep == ~touch).all()
        keep = ~touch
        afe.afe_mesh_destroy(h)
    assert keep.sum() >= 10
    a, b = du[afe.AFE_FP32][keep], du[afe.AFE_FP64][keep]
    assert np.linalg.norm(a - b) <= 1e-3 * np.linalg.norm(b)


@pytest.mark.parametrize("k", [-36, 44])
@pytest.mark.parametrize("N", [1, 2, 3])
def test_length_scales(afe, N, k):
    """Lengths and the time step times 2^k: every term of the scheme scales by a power of two (those of M_i^-1
    by 2^-3k: its largest is 2^118 to 2^123, and 2^-122 to 2^-117), so the states agree to the bar of the
    other FP32 tests; the update itself is 1e-3 of the state and more."""
    out = []
    for s in (1.0, 2.0 ** k):
        pm = split_cube_lattice((2, 1, 1), (2, 1, 1), d=0.5 * s)
        p = afe.afe_default_params(N, precision=afe.AFE_FP32, picard_tol=1e-6, cfl=0.1)
        h = afe.create_from_polymesh(pm, p)
        u0 = states.density_wave(afe.afe_get_node_coords(h) / s, amp=0.1, vel=(0.5, -0.3, 0.2))
        afe.afe_set_state(h, u0)
        for _ in range(4):
            assert afe.afe_step(h, 2e-3 * s) == 0
        out.append(afe.afe_get_state(h))
        afe.afe_mesh_destroy(h)
    assert rel_l2_fields(out[0], u0) > 1e-3
    assert rel_l2_fields(out[1], out[0]) <= FP32_TOL
