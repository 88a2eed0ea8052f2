"""Device memory of handles: what the tensor-core forms keep of M_i^-1 takes the place of what the other forms
read, it does not come on top of it, so that a pool of slots with a fixed budget holds no fewer."""
import numpy as np
import pytest

from inputs import states
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


# bytes of the same handles when the predictor read FP64 rows and kept its coefficients in global memory
@pytest.mark.parametrize("N,k,rows_alone", [(1, 16, 173409210), (2, 11, 361215064), (3, 8, 788863260)])
def test_digits_replace_the_fp64_rows(afe, N, k, rows_alone):
    h = afe.create_from_polymesh(periodic_voronoi(k), afe.afe_default_params(N))
    bytes_ = afe.afe_device_bytes(h)
    print(f"P{N} FP64: {bytes_} bytes, rows alone {rows_alone}")
    assert bytes_ <= rows_alone
    afe.afe_mesh_destroy(h)


def _handle(afe, pm, N):
    p = afe.afe_default_params(N, precision=afe.AFE_FP32, picard_tol=1e-6, cfl=0.1)
    h = afe.create_from_polymesh(pm, p)
    afe.afe_set_state(h, states.density_wave(afe.afe_get_node_coords(h)))
    return h


def _row_bytes(afe, h, pm):
    """FP32 rows of M_i^-1 as the one-block and tensor-memory forms read them (16-byte rows, padded)."""
    n = np.diff(afe.afe_node_ptr(h, pm.n_cells))
    return int((4 * ((n * ((n + 15) // 16 * 16 + 8) + 31) // 32 * 32)).sum())


# bytes of the same handles when M_i^-1 was kept as FP32 rows alone
@pytest.mark.parametrize("N,rows_alone", [(1, 5071804), (2, 20214068), (3, 98315172)])
def test_split_pairs_replace_the_rows(afe, N, rows_alone):
    pm = periodic_voronoi(6)
    h = _handle(afe, pm, N)
    bytes_ = afe.afe_device_bytes(h)
    print(f"P{N}: {bytes_} bytes, rows alone {rows_alone}")
    assert bytes_ <= rows_alone
    # the tensor-memory form's rows are formed when it is asked for, and are the handle's from then on
    afe.afe_set_predictor_variant(h, 1)
    assert afe.afe_device_bytes(h) == bytes_ + _row_bytes(afe, h, pm)
    afe.afe_set_predictor_variant(h, 0)
    afe.afe_set_schedule(h, variant=1)
    assert afe.afe_device_bytes(h) == bytes_ + _row_bytes(afe, h, pm)
    afe.afe_mesh_destroy(h)


@pytest.mark.parametrize("N", [1, 2, 3])
def test_rows_formed_late_are_those_of_set_up(afe, N):
    """A batch switched to the tensor-memory form after steps in the other one, against members switched before
    they joined a batch: bit for bit."""
    meshes = [periodic_voronoi(3), periodic_voronoi(4)]
    late, early = ([_handle(afe, pm, N) for pm in meshes] for _ in range(2))
    b = afe.afe_batch_create(late)
    afe.afe_batch_step_async(b, 0.0, 2, True)
    afe.afe_batch_sync(b, 2)
    afe.afe_batch_set_schedule(b, variant=1)
    afe.afe_batch_step_async(b, 0.0, 2, True)
    afe.afe_batch_sync(b, 2)
    afe.afe_batch_destroy(b)
    for h in early:
        for _ in range(2):
            afe.afe_step(h, 0.0)
        afe.afe_set_predictor_variant(h, 1)
    b = afe.afe_batch_create(early)
    afe.afe_batch_step_async(b, 0.0, 2, False)
    afe.afe_batch_sync(b, 2)
    afe.afe_batch_destroy(b)
    for x, y in zip(late, early):
        np.testing.assert_array_equal(afe.afe_get_state(x), afe.afe_get_state(y))
    for h in late + early:
        afe.afe_mesh_destroy(h)
