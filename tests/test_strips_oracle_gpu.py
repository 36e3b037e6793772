"""The row-staged strips against the FP64 oracle and their own bitwise
properties, chosen explicitly: the lattices of the oracle tests are small
enough that a handle as it is created steps them in tiles. Bars and lengths are
those of the tests of the default layout."""
import numpy as np
import pytest
from parity_util import compare_state, gpu_run, oracle_run
from test_batched_parity_gpu import _batch
from test_fp16_proxy_gpu import _golden

from paper_2403_16122_gb300 import inputs

pytestmark = pytest.mark.gpu

STAGED = (2, 4, 0, 168)  # LBM_KERNEL_STAGED


@pytest.fixture(scope="module")
def lbm():
    from paper_2403_16122_gb300 import build
    from paper_2403_16122_gb300 import lbm as mod

    build.build()
    mod.load()
    assert STAGED[0] == mod.LBM_KERNEL_STAGED
    return mod


def _store(lbm, name):
    return {"fp32": lbm.LBM_STORE_FP32, "fp16": lbm.LBM_STORE_FP16,
            "bf16": lbm.LBM_STORE_BF16}[name]


def _strips(cases, steps, storage=0, kernel=STAGED):
    lat = gpu_run([c[0] for c in cases], [c[1:] for c in cases], 0, storage=storage)
    lat.set_kernel(*kernel)
    assert lat.step_kernel[0] == kernel[0]
    return lat.step(steps) if steps else lat


PER_PHASE = dict(Cp_ratio_sl=0.5, k_ratio_sl=3.8, Cp_ratio_gl=1.0, k_ratio_gl=0.04)


@pytest.mark.parametrize("case", ["sessile", "bubbles", "buoyancy", "per_phase", "top_wall"])
def test_fp32_strips_match_oracle(lbm, oracle_mod, case):
    """1000 steps within 1e-5 (500 with bubbles, 100 with per-phase properties:
    see the tests of the default layout), observables within 1e-5 relative."""
    steps = 1000
    if case == "sessile":
        c = inputs.sessile(nx=100, ny=70, R=24.0, theta_deg=70.0)
    elif case == "bubbles":
        c, steps = inputs.bubbles_drop(n=96, n_bub=2, r_lo=4.0, r_hi=6.0, seed=9), 500
    elif case == "buoyancy":
        c = inputs.column_bubbles(l=24, g=1e-3)
    elif case == "per_phase":
        c, steps = inputs.sessile(nx=96, ny=64, R=24.0, theta_deg=100.0, **PER_PHASE), 100
    else:  # cold top wall, adiabatic bottom
        p, phi0, T0 = inputs.sessile(nx=96, ny=64, R=40.0, theta_deg=120.0)
        c = dict(p, dirichlet_y_lo=0, dirichlet_y_hi=1), phi0, T0
    o = oracle_run(oracle_mod, *c, steps)
    lat = _strips([c], steps)
    compare_state(lat.get_state(), o.get_state())
    if case == "per_phase":
        lat.step(900)
        o.step(900)
    got, want = lat.observables(), o.observables()
    for k in ("volume", "solid", "enthalpy", "solid_col"):
        assert got[k] == pytest.approx(want[k], rel=1e-5, abs=1e-6), k
    lat.close()


@pytest.mark.parametrize("case", ["sessile", "bubbles"])
@pytest.mark.parametrize("storage", ["fp16", "bf16"])
def test_16bit_strips_match_oracle_observables(lbm, oracle_mod, storage, case):
    """The reduced-precision bar after 2000 steps: volume and solidified amount
    within 1 %, centre front height within 0.5 lattice units."""
    c = inputs.sessile(nx=96, ny=64, R=24.0, theta_deg=100.0) if case == "sessile" else \
        inputs.bubbles_drop(n=96, n_bub=2, r_lo=4.0, r_hi=6.0, seed=21)
    o = oracle_run(oracle_mod, *c, 2000)
    lat = _strips([c], 2000, _store(lbm, storage))
    got, want = lat.observables(), o.observables()
    assert got["volume"] == pytest.approx(want["volume"], rel=0.01)
    assert got["solid"] == pytest.approx(want["solid"], rel=0.01)
    assert abs(got["solid_col"] - want["solid_col"]) <= 0.5
    assert got["nonfinite"] == 0.0
    lat.close()


@pytest.mark.parametrize("walls", ["top", "both"])
@pytest.mark.parametrize("storage,kernel", [
    ("fp16", "created"), ("fp16", "staged"), ("fp16", "strip"), ("fp16", "block"),
    ("bf16", "created"), ("bf16", "staged"), ("bf16", "block")])
def test_16bit_one_step_at_a_cold_top_wall(lbm, oracle_mod, storage, kernel, walls):
    """One step from the oracle's state after 200 steps with a Dirichlet wall at
    the top (and at the bottom too): the bars of the same test at the bottom
    wall, 5e-5 (FP16) and 4e-4 (BF16); a wrong sign or reference of a bounced h is
    some 0.05 off."""
    p, phi0, T0 = inputs.sessile(nx=80, ny=60, R=35.0, theta_deg=120.0)
    p = dict(p, dirichlet_y_lo=int(walls == "both"), dirichlet_y_hi=1)
    o = oracle_run(oracle_mod, p, phi0, T0, 200)
    pops, aux = o.get_state()
    lat = gpu_run([p], [(phi0, T0)], 0, storage=_store(lbm, storage))
    if kernel != "created":
        lat.set_kernel(*{"staged": STAGED, "strip": (lbm.LBM_KERNEL_STRIP, 4, 16, 168),
                         "block": (lbm.LBM_KERNEL_BLOCK, 4, 0, 168)}[kernel])
    lat.set_state(pops, aux)
    lat.step(1)
    o.step(1)
    tol = 5e-5 if storage == "fp16" else 4e-4
    for got, want in zip(lat.get_state(), o.get_state()):
        assert np.abs(got - want).max() < tol
    lat.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_bubble_drop_256_in_strips_20000_steps(lbm, storage):
    gold = _golden()
    p, phi0, T0 = inputs.bubbles_drop(n=256)
    lat = _strips([(p, phi0, T0)], 0, _store(lbm, storage))
    for step in sorted(gold):
        lat.step(step - lat.step_count)
        ob, g = lat.observables(), gold[step]
        front, rel = (0.01, 1e-4) if storage == "fp32" else (0.5, 0.01)
        assert abs(ob["solid_col"] - g["solid_col"]) <= front, step
        assert ob["solid"] == pytest.approx(g["solid"], rel=rel), step
        assert ob["volume"] == pytest.approx(g["volume"], rel=rel), step
    if storage == "fp32":
        assert lat.freezing()["mdot_integral"] == pytest.approx(gold[20000]["mdot_integral"], rel=1e-4)
    lat.close()


@pytest.mark.parametrize("mode", ["launch", "graph"])
def test_batch_in_strips_matches_oracle_1000_steps(lbm, oracle_mod, mode):
    cases = _batch()
    lat = _strips(cases, 0)
    lat.set_exec(lbm.LBM_EXEC_GRAPH if mode == "graph" else lbm.LBM_EXEC_LAUNCH, 64)
    lat.step(1000)
    for k, c in enumerate(cases):
        o = oracle_run(oracle_mod, *c, 1000)
        compare_state(lat.get_state(k), o.get_state())
    lat.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_strips_bit_for_bit(lbm, storage):
    """In strips, lattices of a batch equal the same lattices alone, and graph
    replay equals launches, bit for bit."""
    st = _store(lbm, storage)
    cases = inputs.batched_sweep(n_inst=3, seed=3, sizes=(40, 64, 96))
    batch = _strips(cases, 60, st)
    replay = _strips(cases, 0, st)
    replay.set_exec(lbm.LBM_EXEC_GRAPH, 16)
    replay.step(60)
    assert np.array_equal(batch.observables_all(), replay.observables_all())
    for k, c in enumerate(cases):
        one = _strips([c], 60, st)
        for a, b, d in zip(batch.get_state(k), one.get_state(), replay.get_state(k)):
            assert np.array_equal(a, b) and np.array_equal(a, d)
        one.close()
    batch.close()
    replay.close()
