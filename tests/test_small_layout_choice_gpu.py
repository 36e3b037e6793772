"""Small handles in 16-bit storage: the tile layout they are created in can be
chosen, found by the autotuner and read back."""
import numpy as np
import pytest

from paper_2403_16122_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_2403_16122_gb300 import build
    from paper_2403_16122_gb300 import lbm as mod

    build.build()
    mod.load()
    return mod


def _drop(lbm, storage, n=128):
    p, phi0, T0 = inputs.sessile(nx=n, ny=n, R=0.25 * n, theta_deg=75.0)
    return lbm.Lattice([p], storage=getattr(lbm, "LBM_STORE_" + storage)).init(phi0, T0)


@pytest.mark.parametrize("storage", ["FP16", "BF16"])
def test_16bit_tiles_can_be_chosen(lbm, storage):
    """TILE (32, 4) in 16-bit storage is the kernel such a handle is created in:
    the same bits. The other tile shapes stay refused, and so does the
    persistent form."""
    a, b = _drop(lbm, storage), _drop(lbm, storage)
    b.set_kernel(lbm.LBM_KERNEL_TILE, 32, 4)
    assert b.kernel == (lbm.LBM_KERNEL_TILE, 32, 4, 0)
    for u, v in zip(a.step(25).get_state(), b.step(25).get_state()):
        assert np.array_equal(u, v)
    assert a.observables() == b.observables()
    for shape in ((32, 8), (64, 4), (32, 16), (32, 5)):
        with pytest.raises(lbm.LbmError):
            b.set_kernel(lbm.LBM_KERNEL_TILE, *shape)
    with pytest.raises(lbm.LbmError):
        b.set_exec(lbm.LBM_EXEC_PERSISTENT, 4)
    # and on a lattice of more than two waves of tiles
    c, d = _drop(lbm, storage, 512), _drop(lbm, storage, 512)
    c.set_kernel(lbm.LBM_KERNEL_TILE, 32, 4).step(3)
    d.step(3)
    # a stored value may round to the other neighbour (2^-13, 2^-10 apart) a step
    tol = 3 * (2.0 ** -13 if storage == "FP16" else 2.0 ** -10)
    for u, v in zip(c.get_state(), d.get_state()):
        assert np.abs(u - v).max() <= tol


@pytest.mark.parametrize("storage", ["FP16", "BF16"])
def test_autotuner_keeps_small_16bit_lattices_in_tiles(lbm, storage):
    """A step of 128 x 128 sites takes a third of the time in tiles."""
    a = _drop(lbm, storage)
    a.autotune(steps=50)
    assert a.kernel == (lbm.LBM_KERNEL_TILE, 32, 4, 0)
    b = _drop(lbm, storage).set_kernel(*a.kernel)
    assert b.kernel == a.kernel


@pytest.mark.parametrize("storage", ["FP32", "FP16", "BF16"])
def test_step_kernel_is_what_runs(lbm, storage):
    """kernel reports the chosen layout, step_kernel the one that steps: tiles
    on a small handle as it was created, and only there. Handing it to a second
    handle gives the same bits; the persistent form and a chosen layout run as
    they are reported."""
    a = _drop(lbm, storage)
    assert a.kernel[0] == lbm.LBM_KERNEL_STAGED
    assert a.step_kernel == (lbm.LBM_KERNEL_TILE, 32, 4, 0)
    b = _drop(lbm, storage).set_kernel(*a.step_kernel)
    assert b.kernel == b.step_kernel == a.step_kernel
    for u, v in zip(a.step(10).get_state(), b.step(10).get_state()):
        assert np.array_equal(u, v)
    a.set_exec(lbm.LBM_EXEC_PERSISTENT, 4)
    assert a.step_kernel == a.kernel
    a.set_exec(lbm.LBM_EXEC_LAUNCH)
    assert a.step_kernel[0] == lbm.LBM_KERNEL_TILE
    a.set_kernel(lbm.LBM_KERNEL_STAGED, 4, 0, 168)
    assert a.step_kernel == a.kernel
    big = _drop(lbm, storage, 512)
    assert big.step_kernel == big.kernel and big.kernel[0] == lbm.LBM_KERNEL_STAGED
    p, _, _ = inputs.stefan(nx=64)  # walls in x
    if storage == "FP32":
        lat = lbm.Lattice([p])
        assert lat.step_kernel == lat.kernel == (lbm.LBM_KERNEL_TILE, 32, 4, 0)


def test_failed_change_of_form_leaves_the_handle_as_it_was(lbm):
    """To the persistent form a small handle rebuilds its tables, which waits for
    the stream: an error while the stream is being captured. The handle then
    steps on as before, on the same tables."""
    import ctypes

    import torch

    s = torch.cuda.Stream()
    p, phi0, T0 = inputs.sessile(nx=96, ny=64, R=24.0)
    a, b = (lbm.Lattice([p], stream=s).init(phi0, T0).step(3) for _ in range(2))
    cu = ctypes.CDLL("libcuda.so.1")
    stream, graph = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p()
    torch.cuda.synchronize()
    assert cu.cuStreamBeginCapture_v2(stream, 1) == 0  # of this thread
    with pytest.raises(lbm.LbmError) as e:
        a.set_exec(lbm.LBM_EXEC_PERSISTENT, 4)
    assert e.value.code == lbm.LBM_ECUDA
    assert cu.cuStreamEndCapture(stream, ctypes.byref(graph)) != 0  # the capture is void
    assert a.exec[:2] == b.exec[:2] and a.step_kernel == b.step_kernel
    for u, v in zip(a.step(20).get_state(), b.step(20).get_state()):
        assert np.array_equal(u, v)
    assert a.observables() == b.observables()
    assert a.freezing() == b.freezing()
    a.set_exec(lbm.LBM_EXEC_PERSISTENT, 4)
    assert a.step_kernel[0] == lbm.LBM_KERNEL_STAGED
    a.step(9)
    assert a.observables()["nonfinite"] == 0.0
