"""The small kernels of a step at the states and sizes where they can go wrong."""
import numpy as np
import pytest

from inputs import states
from inputs.lattice import split_cube_lattice
from inputs.voronoi import periodic_voronoi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def afe():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2605_00619_gb300 import afe as a
    a.lib()
    return a


def _bound(u, gamma=1.4):
    u = u[np.isfinite(u[:, 0])]
    rho, v, p = states.conserved_to_primitive(u, gamma)
    return (np.linalg.norm(v, axis=1) + np.sqrt(gamma * p / rho)).max()


# density scale, velocity scale, pressure scale: from rest to a kinetic energy that leaves the
# pressure 1e-13 of the total, and values outside FP32's range
@pytest.mark.parametrize("scales", [(1, 0, 1), (1, 1, 1), (1, 1e3, 1), (1, 1e5, 1e-3), (1e-9, 10, 1e-6), (1e40, 1, 1e41),
                                    (1, 1e-40, 1), (1e-42, 1, 1e-42)])
@pytest.mark.parametrize("N", [1, 3])
def test_time_step_is_the_fp64_maximum(afe, N, scales):
    """dt is inversely proportional to the largest bound over all nodes, evaluated in FP64: on one
    mesh dt times the bound is the same for every state (to the rounding of its operations)."""
    pm = periodic_voronoi(3)
    h = afe.create_from_polymesh(pm, afe.afe_default_params(N, precision=afe.AFE_FP32, picard_tol=1e-6))
    n = afe.afe_num_nodes(h)
    rng = np.random.default_rng(3)

    def dt_times_bound(u):
        afe.afe_set_state(h, u)
        return afe.afe_compute_dt(h) * _bound(u)

    ref = dt_times_bound(states.primitive_to_conserved(np.ones(n), np.zeros((n, 3)), np.ones(n)))
    for _ in range(3):
        r, s, q = scales
        u = states.primitive_to_conserved(r * rng.uniform(0.5, 2, n), s * rng.normal(size=(n, 3)), q * rng.uniform(0.5, 2, n))
        p = states.conserved_to_primitive(u)[2]
        if (p <= 0).any():  # rounding of the total energy: inadmissible, and reported
            with pytest.raises(afe.AfeError):
                dt_times_bound(u)
            continue
        # p = (gamma - 1) (E - m^2 / 2 rho) is rounded to 2^-52 of E on either side (products may be
        # fused), which moves c = sqrt(gamma p / rho) by up to sqrt(gamma 2^-51 E / rho)
        tol = 1e-12 + np.sqrt(1.4 * 2.0 ** -51 * u[:, 4] / u[:, 0]).max() / _bound(u)
        assert abs(dt_times_bound(u) / ref - 1) <= tol
    u = states.primitive_to_conserved(np.ones(n), rng.normal(size=(n, 3)), np.ones(n))
    for bad in (np.nan, -1.0, np.inf):
        w = u.copy()
        w[n // 2, 0] = bad
        if bad == np.inf:  # the bound as it is written is 0 there: no report, the other nodes decide
            assert abs(dt_times_bound(w) / ref - 1) <= 1e-12
            continue
        afe.afe_set_state(h, w)
        with pytest.raises(afe.AfeError):
            afe.afe_compute_dt(h)
    afe.afe_mesh_destroy(h)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_every_launch_of_the_bound_starts_from_zero(afe, precision):
    """The CFL launch's last block sets dt and the clock and leaves the maximum at zero: neither a bound
    read before a step nor a faster state stepped before reaches the next step's dt."""
    pm = periodic_voronoi(3)
    prec = afe.AFE_FP32 if precision == "fp32" else afe.AFE_FP64
    p = afe.afe_default_params(1, precision=prec, picard_tol=1e-6 if precision == "fp32" else 1e-12, cfl=0.3)
    h, g = afe.create_from_polymesh(pm, p), afe.create_from_polymesh(pm, p)
    n = afe.afe_num_nodes(h)

    def state(speed):
        return states.primitive_to_conserved(np.ones(n), np.full((n, 3), speed), np.ones(n))

    afe.afe_set_state(h, state(100.0))
    fast = afe.afe_compute_dt(h)
    afe.afe_cfl_pieces(h, 2)
    afe.afe_set_state(h, state(1.0))
    afe.afe_set_state(g, state(1.0))
    slow = afe.afe_compute_dt(g)
    assert slow > 10 * fast
    afe.afe_step_async(h, 0.0, 1)
    assert afe.afe_sync(h) == 0
    assert afe.afe_get_stats(h).t == afe.afe_get_stats(h).dt == slow
    afe.afe_step_async(h, slow / 2, 2)
    assert afe.afe_sync(h) == 0
    assert afe.afe_get_stats(h).t == pytest.approx(2 * slow, rel=2.0**-51)  # two roundings
    for m in (h, g):
        afe.afe_mesh_destroy(m)


# gamma - 1 far from a power of two and down to 1e-4, where gamma in FP32 has lost it to 4 digits
@pytest.mark.parametrize("gamma", [1.0001, 1.001, 1.005, 5.0 / 3.0])
@pytest.mark.parametrize("first", ["hot", "fast"])
def test_time_step_over_gamma_and_kinds_of_nodes(afe, gamma, first):
    """Nodes whose bound is nearly all sound speed beside nodes whose bound is nearly all velocity, one kind
    ahead of the other by 1e-5: whatever their order, dt is that of the largest FP64 bound, to the rounding of
    its operations (a few 2^-53; the bar is that of the uniform states above), and the same in every run."""
    pm = periodic_voronoi(3)
    h = afe.create_from_polymesh(pm, afe.afe_default_params(2, precision=afe.AFE_FP32, picard_tol=1e-6, gamma=gamma))
    n = afe.afe_num_nodes(h)
    rng = np.random.default_rng(11)
    one = states.primitive_to_conserved(np.ones(n), np.zeros((n, 3)), np.ones(n), gamma)
    afe.afe_set_state(h, one)
    ref = afe.afe_compute_dt(h) * _bound(one, gamma)
    for _ in range(3):
        hot = rng.random(n) < 0.5
        speed = np.where(hot, 1.0, 1.0 - 1e-5) if first == "hot" else np.where(hot, 1.0 - 1e-5, 1.0)
        speed *= 1 - 1e-6 * rng.random(n)
        mach = np.where(hot, 1e-3, 20.0)  # |v| / c
        c = speed / (1 + mach)
        d = rng.normal(size=(n, 3))
        rho = rng.uniform(0.5, 2, n)
        u = states.primitive_to_conserved(rho, (mach * c / np.linalg.norm(d, axis=1))[:, None] * d, rho * c * c / gamma,
                                          gamma)
        afe.afe_set_state(h, u)
        dts = {afe.afe_compute_dt(h) for _ in range(5)}
        assert len(dts) == 1
        assert abs(dts.pop() * _bound(u, gamma) / ref - 1) <= 1e-12
    afe.afe_mesh_destroy(h)


# values whose products leave FP32's range though they themselves do not
@pytest.mark.parametrize("rho,c", [(1e-19, 1.0), (1e-21, 1.0), (1e-24, 1.0), (1e-24, 1e5), (1e12, 1e-21), (1e25, 1e-27)])
def test_time_step_of_small_products(afe, rho, c):
    """Fast cold nodes (|v| = 3 c) among hot ones at rest (c' = 2 c), densities down to 1e-24: dt is that of the
    largest FP64 bound, to the rounding of its operations (the pressure is a tenth of the total energy or
    more: a few 2^-52)."""
    pm = periodic_voronoi(3)
    h = afe.create_from_polymesh(pm, afe.afe_default_params(2, precision=afe.AFE_FP32, picard_tol=1e-6))
    n = afe.afe_num_nodes(h)
    rng = np.random.default_rng(13)
    one = states.primitive_to_conserved(np.ones(n), np.zeros((n, 3)), np.ones(n))
    afe.afe_set_state(h, one)
    ref = afe.afe_compute_dt(h) * _bound(one)
    for _ in range(3):
        hot = rng.random(n) < 0.5
        d = rng.normal(size=(n, 3))
        d /= np.linalg.norm(d, axis=1)[:, None]
        cs = np.where(hot, 2.0, 1.0) * c * rng.uniform(0.9, 1, n)
        r = rho * rng.uniform(0.5, 2, n)
        u = states.primitive_to_conserved(r, np.where(hot, 0.0, 3.0 * c)[:, None] * d, r * cs * cs / 1.4)
        afe.afe_set_state(h, u)
        assert abs(afe.afe_compute_dt(h) * _bound(u) / ref - 1) <= 1e-12
    afe.afe_mesh_destroy(h)
