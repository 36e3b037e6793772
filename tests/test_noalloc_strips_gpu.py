"""lbm_step_noalloc in strips (lattices periodic in x of more than two waves of
tiles) and in tiles against another tile kernel of a handle, on the same state,
every column of it."""
import numpy as np
import pytest
from test_zz_no_alloc import _blocked, _unblocked

from paper_2403_16122_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    from paper_2403_16122_gb300 import build, lbm

    build.build()
    lbm.load()
    return torch, lbm


def _noalloc_step(env, p, pops, aux, pitch):
    """One lbm_step_noalloc from a host state: (P, A, record)."""
    torch, lbm = env
    L = p["Cp"] * (p["T_m"] - p["T_w"]) / p["Ste"]
    P, A = (torch.from_numpy(v).cuda() for v in _blocked(pops, aux, L, pitch))
    Po, Ao = torch.zeros_like(P), torch.zeros_like(A)
    rec = torch.full((lbm.LBM_OBS_COUNT,), -1.0, dtype=torch.float64, device="cuda")
    lbm.lbm_step_noalloc(p, P.data_ptr(), A.data_ptr(), Po.data_ptr(), Ao.data_ptr(), pitch,
                         rec.data_ptr(), torch.cuda.current_stream().cuda_stream)
    return Po.cpu().numpy(), Ao.cpu().numpy(), dict(zip(lbm.OBS_NAMES, rec.cpu().numpy()))


@pytest.mark.parametrize("nx,ny", [(500, 420), (512, 512), (1500, 131)])
def test_record_is_summed_in_64_bits(env, nx, ny):
    """Without phase change phi and H of a site are plain sums of its
    populations, taken in one order by every kernel: the same FP32 values in
    strips and in tiles. Their sums over the sites are FP64 in both (the tiles'
    from one value a thread), so the records differ by the order of fewer than
    2^18 positive FP64 terms in trees at most 600 deep: 600 x 2^-53 < 1e-13. A
    row summed in FP32 would be off by some 1e-9."""
    torch, lbm = env
    p, phi0, T0 = inputs.sessile(nx=nx, ny=ny, R=0.3 * ny, theta_deg=80.0)
    p = dict(p, dirichlet_y_lo=0)
    lat = lbm.Lattice([p]).set_kernel(lbm.LBM_KERNEL_TILE, 32, 8).init(phi0, T0 + 0.1).step(5)
    pops, aux = lat.get_state()
    want = lat.step(1).observables()
    lat.close()
    _, _, got = _noalloc_step(env, p, pops, aux, (nx + 31) // 32 * 32)
    assert want["solid"] == got["solid"] == 0.0
    for k in ("volume", "enthalpy"):
        assert got[k] == pytest.approx(want[k], rel=1e-13), k


# strips (whole and ragged last strips, a pitch wider than they need), then
# tiles: two waves at most, walls in x, more 32 x 4 tiles than partial slots
LAYOUTS = [(500, 420, 1, 512), (500, 420, 1, 576), (512, 512, 1, 512), (1501, 131, 1, 1568),
           (483, 430, 1, 512), (100, 90, 1, 128), (450, 400, 0, 480), (1000, 1100, 0, 1024)]


@pytest.mark.parametrize("nx,ny,px,pitch", LAYOUTS)
def test_every_column_matches_other_tiles(env, nx, ny, px, pitch):
    """Two steps against a handle in 64 x 4 tiles, which no allocation-free step
    uses: layouts agree within 1e-6, in every column, the ragged last strip and
    the wall columns included, and the padding is never written."""
    torch, lbm = env
    p = inputs.params(nx=nx, ny=ny, periodic_x=px, periodic_y=0, dirichlet_y_lo=1,
                      dirichlet_y_hi=ny % 2, dirichlet_x_hi=1 - px, theta_deg=60.0)
    phi0, T0 = inputs.random_state(p, seed=nx + pitch)
    L = p["Cp"] * (p["T_m"] - p["T_w"]) / p["Ste"]
    lat = lbm.Lattice([p]).set_kernel(lbm.LBM_KERNEL_TILE, 64, 4).init(phi0, T0).step(2)
    for call in range(2):
        pops, aux = lat.get_state()
        want = lat.step(1)
        Po, Ao, rec = _noalloc_step(env, p, pops, aux, pitch)
        got = _unblocked(Po, Ao, L, nx, ny, pitch)
        for a, b in zip(got, want.get_state()):
            assert np.abs(a - b).max() <= 1e-6, call
        pad = Po.reshape(ny, pitch // 32, 768)[:, (nx + 31) // 32:]
        assert not pad.any()
        obs = want.observables(check=False)
        for k in ("volume", "solid", "enthalpy", "mass", "condensed_mass", "solid_col", "solid_row"):
            assert rec[k] == pytest.approx(obs[k], rel=1e-6, abs=1e-6), (call, k)
        assert rec["umax"] == pytest.approx(obs["umax"], rel=1e-3, abs=1e-6)
    lat.close()
