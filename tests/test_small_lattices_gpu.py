"""The layouts that are chosen by size, at the sizes where they can go wrong:
handles of small lattices run in 32 x 4 tiles (FP32 and 16-bit storage),
lbm_step_noalloc takes tiles or strips, the observable reduction sums 64
partials a CTA, and FP32 checkpoints are converted on the device. Each is
compared with another layout of the same step, which the oracle tests hold."""
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


def _state(lbm, p, phi0, T0, storage, kernel, steps):
    lat = lbm.Lattice([p], storage=storage).init(phi0, T0)
    if kernel:
        lat.set_kernel(*kernel)
    lat.step(steps)
    out = lat.get_state(), lat.observables(check=False)
    lat.close()
    return out


# one site, one tile, ragged tiles one site wide or high, several tiles
SIZES = [(3, 3), (32, 4), (33, 5), (31, 9), (65, 4), (96, 64), (129, 70)]


@pytest.mark.parametrize("py", [0, 1])
@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_small_handle_in_tiles_matches_strips(lbm, storage, nx, ny, py):
    """One step of a small handle as lbm_create lays it out against the same
    step in staged strips. FP32: the layouts agree to rounding (1.5e-7 after one
    step; the bar of one step from a common state is 2e-6). 16-bit storage: a
    value may round to the other neighbour; deviations stay below 0.25 in these
    fields, where neighbours are 2^-13 apart in FP16 and 2^-10 in BF16."""
    st = {"fp32": lbm.LBM_STORE_FP32, "fp16": lbm.LBM_STORE_FP16, "bf16": lbm.LBM_STORE_BF16}[storage]
    tol = {"fp32": 2e-6, "fp16": 2.0 ** -13, "bf16": 2.0 ** -10}[storage]
    p = inputs.params(nx=nx, ny=ny, periodic_x=1, periodic_y=py, dirichlet_y_lo=1 - py,
                      theta_deg=65.0, st_mask_liquid=1)
    phi0, T0 = inputs.random_state(p, seed=nx + 100 * ny)
    (a, oa) = _state(lbm, p, phi0, T0, st, None, 1)
    (b, ob) = _state(lbm, p, phi0, T0, st, (lbm.LBM_KERNEL_STAGED, 4, 0, 168), 1)
    assert np.abs(a[0] - b[0]).max() <= tol
    assert np.abs(a[1] - b[1]).max() <= tol
    for k in ("volume", "mass", "enthalpy", "condensed_mass"):
        assert oa[k] == pytest.approx(ob[k], rel=1e-6, abs=1e-6), k


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_rows_chosen_for_a_batch_change_no_bit(lbm, storage):
    """Uneven lattices, together more than two waves of tiles (staged strips):
    the chosen rows per item against 2, 16 and more rows than a lattice has."""
    st = lbm.LBM_STORE_FP32 if storage == "fp32" else lbm.LBM_STORE_FP16
    cases = [inputs.sessile(300, 280, 70.0, theta_deg=80.0), inputs.sessile(251, 303, 60.0),
             inputs.sessile(96, 64, 16.0, theta_deg=120.0)]
    want = None
    for rows in (None, 2, 16, 400):
        lat = lbm.Lattice([c[0] for c in cases], storage=st)
        for k, (_, phi0, T0) in enumerate(cases):
            lat.init(phi0, T0, inst=k)
        if rows:
            lat.set_kernel(lbm.LBM_KERNEL_STAGED, 4, rows, 168)
        assert lat.kernel[0] == lbm.LBM_KERNEL_STAGED and lat.kernel[2] >= 2
        lat.step(9)
        got = [lat.get_state(k) for k in range(3)], lat.observables_all()
        lat.close()
        if want is None:
            want = got
            continue
        for (a, b), (c, d) in zip(want[0], got[0]):
            assert np.array_equal(a, c) and np.array_equal(b, d)
        np.testing.assert_allclose(got[1], want[1], rtol=1e-6, atol=1e-6)


@pytest.mark.parametrize("nx,ny", [(32, 4), (32, 256), (32, 260), (1024, 520)])
def test_reduction_over_one_or_more_ctas(lbm, nx, ny):
    """1, 64, 65 and 4160 tiles (one partial, one CTA, two CTAs, more CTAs than
    one pass combines) against the strips' partials of the same step."""
    p = inputs.params(nx=nx, ny=ny, periodic_x=1, periodic_y=0, dirichlet_y_lo=1, theta_deg=70.0)
    phi0, T0 = inputs.random_state(p, seed=3)
    got = {}
    for kern in ((lbm.LBM_KERNEL_TILE, 32, 4), (lbm.LBM_KERNEL_STAGED, 4, 0, 168)):
        lat = lbm.Lattice([p]).init(phi0, T0).set_kernel(*kern)
        lat.step(3)
        lat.step(2)
        got[kern[0]] = lat.observables(check=False), lat.freezing(), lat.solid_profile()
        lat.close()
    (oa, fa, pa), (ob, fb, pb) = got.values()
    for k in ("volume", "solid", "mass", "enthalpy", "condensed_mass", "solid_col", "solid_row"):
        assert oa[k] == pytest.approx(ob[k], rel=1e-6, abs=1e-5), k
    assert oa["umax"] == pytest.approx(ob["umax"], rel=1e-3)
    assert fa["step"] == fb["step"] == 5
    assert fa["mdot_integral"] == pytest.approx(fb["mdot_integral"], rel=1e-5, abs=1e-6)
    assert np.abs(pa - pb).max() <= 2e-5 * ny


@pytest.mark.parametrize("nx,ny,px", [(100, 90, 1), (500, 420, 1), (1500, 9, 1), (450, 400, 0),
                                      (1000, 1100, 0)])
def test_noalloc_layouts(lbm, nx, ny, px):
    """Small tiles, strips, flat strips, more tiles than two waves, and more
    32 x 4 tiles than there are partial slots: two steps through
    lbm_step_noalloc on copies of a handle's buffers against the handle's."""
    import torch

    p = inputs.params(nx=nx, ny=ny, periodic_x=px, periodic_y=0, dirichlet_y_lo=1,
                      dirichlet_x_hi=1 - px, theta_deg=60.0)
    phi0, T0 = inputs.random_state(p, seed=nx)
    lat = lbm.Lattice([p])
    nb = ny * ((nx + 31) // 32)
    size = nb * (768 + 320) * 4

    def buffers(k):  # the state buffers are the tail of the workspace
        at = lat.workspace.numel() - (2 - k) * size
        w = lat.workspace[at:at + size].view(torch.float32)
        return w[:nb * 768], w[nb * 768:]

    lat.init(phi0, T0).step(2)  # an even number of steps: buffer 0 is current
    bufs = [tuple(v.clone() for v in buffers(0)) for _ in range(2)]
    d_obs = torch.zeros(lbm.LBM_OBS_COUNT, dtype=torch.float64, device="cuda")
    pitch = (nx + 31) // 32 * 32
    for k in range(2):
        (Pi, Ai), (Po, Ao) = bufs[k], bufs[k ^ 1]
        lbm.lbm_step_noalloc(p, Pi.data_ptr(), Ai.data_ptr(), Po.data_ptr(), Ao.data_ptr(), pitch,
                             d_obs.data_ptr(), torch.cuda.current_stream().cuda_stream)
    lat.step(2)
    want = buffers(0)
    full = nx // 32  # whole blocks: the padding of the last one holds nothing
    # (nor do the last 64 of a block's 320 own-site floats)
    for got, ref, n, used in ((bufs[0][0], want[0], 768, 768), (bufs[0][1], want[1], 320, 256)):
        d = (got - ref).view(ny, pitch // 32, n)[:, :full, :used]
        assert d.abs().max().item() <= 1e-6
    obs = lat.observables(check=False)
    for j, k in enumerate(lbm.OBS_NAMES):
        if k in ("volume", "solid", "enthalpy", "mass", "condensed_mass", "solid_col", "solid_row"):
            assert d_obs[j].item() == pytest.approx(obs[k], rel=1e-6, abs=1e-5), k
    lat.close()


@pytest.mark.parametrize("nx,ny", [(3, 3), (33, 7), (64, 5), (95, 40)])
def test_checkpoint_round_trip_of_ragged_lattices(lbm, nx, ny):
    """lbm_get_state returns what lbm_set_state was given, rounded to FP32, with
    h_0 rounded in its shifted form."""
    p = inputs.params(nx=nx, ny=ny, periodic_x=0, periodic_y=1, dirichlet_x_lo=1)
    rng = np.random.default_rng(nx)
    pops = rng.standard_normal((27, ny, nx))
    aux = rng.standard_normal((5, ny, nx))
    lat = lbm.Lattice([p]).init(np.full((ny, nx), 0.5), np.zeros((ny, nx)))
    lat.set_state(pops, aux)
    got_p, got_a = lat.get_state()
    lat.close()
    L = p["Cp"] * (p["T_m"] - p["T_w"]) / p["Ste"]
    fl = aux[0].astype(np.float32).astype(np.float64)
    want = pops.astype(np.float32).astype(np.float64)
    want[9] = (pops[9] - L * fl).astype(np.float32).astype(np.float64) + L * fl
    assert np.array_equal(got_a, aux.astype(np.float32).astype(np.float64))
    keep = np.arange(27) != 9
    assert np.array_equal(got_p[keep], want[keep])
    # one ulp of the shifted value where the device's fused product rounds apart
    assert np.abs(got_p[9] - want[9]).max() <= 2e-6
