"""GPU parity: the CUDA path through the C ABI against the FP64 CPU oracle on the
same seeded inputs, element by element.

FP64 bar: max |f_gpu - f_oracle| <= 1e-12 max |f_oracle| (relative, max norm), the
target of 1e-12 after 1000 steps.  FP32 deviation storage: the error budget of
single precision, stated per quantity below (unit round-off 6e-8 per operation,
accumulated over the steps run).
"""
import os

import numpy as np
import pytest

import oracle
from theory import maxwell

pytestmark = pytest.mark.gpu

LAT = {  # binding constant -> oracle constant
    0: oracle.D2Q9, 1: oracle.D3Q19, 2: oracle.D2Q13, 3: oracle.D2Q25,
}


def pair(lbm, lattice, shape, *, stencil=0, coll=0, G=-5.0, tau=1.0, psi=0, T_over_Tc=0.0,
         precision=0, s=(1.64, 1.54, 1.9), path=0):
    nz, ny, nx = shape
    dom = lbm.Domain(nx, ny, nz, lattice=lattice, stencil=stencil, collision=coll, G=G, tau=tau,
                     psi=psi, T_over_Tc=T_over_Tc, precision=precision,
                     s_e=s[0], s_eps=s[1], s_q=s[2], path=path)
    order = stencil
    ref = oracle.Sim(LAT[lattice], nx, ny, nz, stencil=order, psi=psi, T_over_Tc=T_over_Tc, G=G,
                     tau=tau, coll=coll, s_e=s[0], s_eps=s[1], s_q=s[2])
    return dom, ref


def rel_max(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("path", [1, 2])
def test_config_d2q9_64_fp64_1000_steps(lbm, path):
    """D2Q9 BGK tau = 1, FP64, 64x64, psi = 1 - exp(-rho), G = -5, 4th-order stencil,
    droplet R = 16 (rho_l = 2.0, rho_g = 0.15, width 2): 1000 steps, both schedules."""
    dom, ref = pair(lbm, lbm.LBM_D2Q9, (1, 64, 64), path=path)
    for d in (dom, ref):
        d.init_droplet(2.0, 0.15, 16.0, 2.0)
    dom.step(1000)
    ref.step(1000)
    assert rel_max(dom.get_f(), ref.get_f()) <= 1e-12
    og, oo = dom.observables(), ref.observables()
    for k in ("rho_l", "rho_g", "mass"):
        assert og[k] == pytest.approx(oo[k], rel=1e-12)
    for k in ("max_u", "mean_u", "dp"):
        assert og[k] == pytest.approx(oo[k], rel=1e-10)
    assert og["step"] == 1000


@pytest.mark.parametrize("precision", [0, 1])
def test_bitwise_reproducible(lbm, precision):
    outs = []
    for _ in range(2):
        dom = lbm.Domain(70, 50, precision=precision)
        dom.init_droplet(2.0, 0.15, 12.0, 2.0)
        dom.step(333)
        outs.append((dom.get_f(), dom.observables()))
        dom.close()
    assert np.array_equal(outs[0][0], outs[1][0])
    assert outs[0][1] == outs[1][1]


CASES_2D = [(lat, st, coll) for lat, st, coll in
            [(0, 4, 0), (0, 6, 0), (0, 8, 0), (0, 10, 0), (0, 4, 1), (0, 8, 1), (0, 10, 1),
             (2, 0, 0), (2, 10, 0), (3, 0, 0), (3, 4, 0), (3, 10, 0)]]


@pytest.mark.parametrize("lattice,stencil,coll", CASES_2D)
def test_2d_ragged_domain_matches_oracle(lbm, lattice, stencil, coll):
    """37 x 29: two tiles in x (one ragged), four in y (one ragged)."""
    tau = {0: 0.8, 2: 11 / 12, 3: 19 / 24}[lattice]
    dom, ref = pair(lbm, lattice, (1, 29, 37), stencil=stencil, coll=coll, tau=tau)
    for d in (dom, ref):
        d.init_droplet(1.9, 0.15, 8.0, 2.0)
    dom.step(150)
    ref.step(150)
    assert rel_max(dom.get_f(), ref.get_f()) <= 1e-12


@pytest.mark.parametrize("lattice,stencil", [(0, 4), (0, 8), (0, 10), (2, 0), (3, 0)])
def test_exact_difference_forcing_matches_oracle(lbm, lattice, stencil):
    """BGK with the exact-difference forcing of the paper's runs, FP64, on the
    ragged 37 x 29 box, against the oracle to 1e-12."""
    tau = {0: 0.8, 2: 11 / 12, 3: 19 / 24}[lattice]
    dom, ref = pair(lbm, lattice, (1, 29, 37), stencil=stencil, coll=lbm.LBM_BGK_EDM, tau=tau)
    for d in (dom, ref):
        d.init_droplet(1.9, 0.15, 8.0, 2.0)
    dom.step(150)
    ref.step(150)
    assert rel_max(dom.get_f(), ref.get_f()) <= 1e-12
    assert dom.observables()["max_u"] == pytest.approx(ref.observables()["max_u"], rel=1e-9)


def test_exact_difference_forcing_fp32_and_3d(lbm):
    """FP32 deviation storage with the exact-difference forcing stays within the
    FP32 budget of the oracle; a 3-D lattice is refused."""
    dom, ref = pair(lbm, lbm.LBM_D2Q9, (1, 64, 64), stencil=4, coll=lbm.LBM_BGK_EDM, precision=1)
    for d in (dom, ref):
        d.init_droplet(2.0, 0.15, 16.0, 2.0)
    dom.step(300)
    ref.step(300)
    assert rel_max(dom.get_f(), ref.get_f()) <= 2e-4
    with pytest.raises(lbm.LbmError):
        lbm.Domain(16, 16, 16, lattice=lbm.LBM_D3Q19, collision=lbm.LBM_BGK_EDM)


@pytest.mark.parametrize("T_over_Tc", [0.9, 0.8])
def test_peng_robinson_exact_difference_matches_oracle(lbm, T_over_Tc):
    """The paper's configuration: P-R psi with the exact-difference forcing,
    on D2Q25 (lattice as stencil) at T/Tc = 0.9 and 0.8."""
    rv, rl = maxwell(T_over_Tc)
    dom, ref = pair(lbm, lbm.LBM_D2Q25, (1, 40, 40), stencil=0, psi=1, T_over_Tc=T_over_Tc, G=-1.0,
                    tau=19 / 24, coll=lbm.LBM_BGK_EDM)
    for d in (dom, ref):
        d.init_droplet(rl, rv, 10.0, 3.0)
    dom.step(200)
    ref.step(200)
    assert rel_max(dom.get_f(), ref.get_f()) <= 1e-12


@pytest.mark.parametrize("stencil,coll", [(4, 0), (6, 0), (4, 1), (6, 1)])
def test_3d_ragged_domain_matches_oracle(lbm, stencil, coll):
    dom, ref = pair(lbm, lbm.LBM_D3Q19, (11, 20, 37), stencil=stencil, coll=coll, tau=0.9,
                    s=(1.2, 1.4, 1.7))
    for d in (dom, ref):
        d.init_droplet(1.9, 0.15, 5.0, 2.0)
    dom.step(60)
    ref.step(60)
    assert rel_max(dom.get_f(), ref.get_f()) <= 1e-12


@pytest.mark.parametrize("lattice,stencil", [(0, 4), (0, 8), (3, 0)])
def test_peng_robinson_matches_oracle(lbm, lattice, stencil):
    """T/Tc = 0.9 (density ratio ~10); at 0.8 the Guo-forced tau = 1 droplet
    diverges on both sides alike."""
    rv, rl = maxwell(0.9)
    dom, ref = pair(lbm, lattice, (1, 40, 40), stencil=stencil, psi=1, T_over_Tc=0.9, G=-1.0,
                    tau=1.0)
    for d in (dom, ref):
        d.init_droplet(rl, rv, 10.0, 3.0)
    dom.step(200)
    ref.step(200)
    assert rel_max(dom.get_f(), ref.get_f()) <= 1e-12
    assert dom.observables()["dp"] == pytest.approx(ref.observables()["dp"], rel=1e-9)


def test_fp32_shifted_error_budget(lbm):
    """FP32 deviation storage on the 64x64 droplet, 1000 steps, against the FP64
    oracle.  Budget: each population sees ~40 float operations per step at unit
    round-off u = 6e-8; accumulated as a random walk over n = 1000 steps that is
    40 u sqrt(n) ~ 8e-5 relative, and at most 40 u n ~ 2.4e-3 if every error
    added up.  The bar is 2e-4 relative on populations and densities, 2e-5
    absolute on dp (a difference of two pressures ~0.4), 1e-2 relative on max|u|
    (a small velocity, ~5e-3, that carries the absolute error of the momenta),
    and 1e-6 relative on the mass (a sum of 4096 independent round-offs)."""
    dom, ref = pair(lbm, lbm.LBM_D2Q9, (1, 64, 64), precision=1)
    for d in (dom, ref):
        d.init_droplet(2.0, 0.15, 16.0, 2.0)
    dom.step(1000)
    ref.step(1000)
    err_f = rel_max(dom.get_f(), ref.get_f())
    og, oo = dom.observables(), ref.observables()
    print(f"FP32 vs FP64 oracle after 1000 steps: f {err_f:.2e}, rho_l {og['rho_l'] / oo['rho_l'] - 1:.2e}, "
          f"rho_g {og['rho_g'] / oo['rho_g'] - 1:.2e}, dp {og['dp'] - oo['dp']:.2e}, "
          f"max_u {og['max_u'] / oo['max_u'] - 1:.2e}")
    assert err_f <= 2e-4
    assert og["rho_l"] == pytest.approx(oo["rho_l"], rel=2e-4)
    assert og["rho_g"] == pytest.approx(oo["rho_g"], rel=2e-4)
    assert og["mass"] == pytest.approx(oo["mass"], rel=1e-6)
    assert abs(og["dp"] - oo["dp"]) <= 2e-5
    assert og["max_u"] == pytest.approx(oo["max_u"], rel=1e-2)


def test_fp32_d3q19_error_budget(lbm):
    dom, ref = pair(lbm, lbm.LBM_D3Q19, (24, 24, 24), precision=1)
    for d in (dom, ref):
        d.init_droplet(2.0, 0.15, 7.0, 2.0)
    dom.step(200)
    ref.step(200)
    assert np.abs(dom.fields()["rho"] - ref.fields()["rho"]).max() <= 2e-5
    assert dom.observables()["max_u"] == pytest.approx(ref.observables()["max_u"], rel=1e-3)


def test_minimum_size_flat_and_zero_steps(lbm):
    dom, ref = pair(lbm, lbm.LBM_D2Q9, (1, 8, 8))
    for d in (dom, ref):
        d.init_flat(1.9, 0.15, 2.0, 0)
    dom.step(0)
    assert rel_max(dom.get_f(), ref.get_f()) <= 1e-15
    dom.step(40)
    ref.step(40)
    assert rel_max(dom.get_f(), ref.get_f()) <= 1e-12
    assert dom.observables()["thickness"] == ref.observables()["thickness"]


def test_set_get_populations_roundtrip_and_from_rho(lbm):
    rng = np.random.default_rng(1906)
    dom, ref = pair(lbm, lbm.LBM_D2Q25, (1, 33, 41), stencil=0, tau=19 / 24)
    rho0 = rng.uniform(0.2, 1.9, size=(1, 33, 41))
    dom.init_from_rho(rho0)
    ref.init_from_rho(rho0)
    assert np.array_equal(dom.get_f(), ref.get_f())
    f = ref.get_f() * (1 + 1e-3 * rng.standard_normal(ref.get_f().shape))
    dom.set_f(f)
    assert np.array_equal(dom.get_f(), f)
    ref.set_f(f)
    dom.step(30)
    ref.step(30)
    assert rel_max(dom.get_f(), ref.get_f()) <= 1e-12


def test_checkpoint_resume_bit_identical(lbm, tmp_path):
    a = lbm.Domain(48, 40, precision=1)
    a.init_droplet(2.0, 0.15, 10.0, 2.0)
    a.step(50)
    path = str(tmp_path / "ck.bin")
    a.save(path)
    a.step(70)
    b = lbm.Domain(48, 40, precision=1)
    b.load(path)
    b.step(70)
    assert np.array_equal(a.get_f(), b.get_f())
    assert a.observables() == b.observables()


def test_nonfinite_input_reported(lbm):
    dom = lbm.Domain(16, 16)
    rho = np.full(256, 1.0)
    rho[37] = np.nan
    dom.init_from_rho(rho)
    with pytest.raises(lbm.LbmError) as e:
        dom.observables()
    assert e.value.code == lbm.LBM_ENONFINITE


def test_run_to_steady_flat_interface(lbm):
    dom = lbm.Domain(128, 8, G=-5.0, tau=1.0)
    dom.init_flat(1.89, 0.12, 4.0, 0)
    steps, ok = dom.run_to_steady(1e-10, 60000, 1)
    assert ok and 0 < steps < 60000
    o = dom.observables()
    # the rule stops when max|u| changes by < 1e-10 per step: a slowly decaying
    # residual remains (~1e-5 here), and the densities are already at coexistence
    assert o["max_u"] < 1e-4
    assert o["rho_l"] == pytest.approx(1.888, rel=2e-3)
    dom.step(2000)
    assert dom.observables()["max_u"] < o["max_u"]


def test_torch_allocator_and_stream(lbm):
    import torch
    s = torch.cuda.Stream()
    dom = lbm.Domain(64, 64, stream=s, torch_alloc=True)
    alloc = dom._alloc
    assert alloc.calls >= 6 and alloc.live >= 6  # buffers came from torch's allocator
    dom.init_droplet(2.0, 0.15, 16.0, 2.0)
    dom.step(20)
    ref = lbm.Domain(64, 64)
    ref.init_droplet(2.0, 0.15, 16.0, 2.0)
    ref.step(20)
    assert np.array_equal(dom.get_f(), ref.get_f())
    dom.close()
    assert alloc.live == 0


def test_full_size_d3q19_256_fp32_against_oracle(lbm):
    """The benchmark's workload at full size: D3Q19, FP32 deviations, 256^3,
    psi = 1 - exp(-rho), G = -5, 4th-order stencil, droplet R = 40.  Two steps
    are compared cell by cell with the FP64 oracle; mass is then checked over a
    longer run (conserved to the FP32 budget)."""
    n = 256
    dom, ref = pair(lbm, lbm.LBM_D3Q19, (n, n, n), precision=1)
    for d in (dom, ref):
        d.init_droplet(2.0, 0.15, 40.0, 2.0)
    dom.step(2)
    ref.step(2)
    rg = dom.fields()["rho"]
    rr = ref.fields()["rho"]
    assert np.abs(rg - rr).max() <= 2e-6
    del ref
    m0 = dom.observables()["mass"]
    dom.step(100)
    assert dom.observables()["mass"] == pytest.approx(m0, rel=1e-6)


@pytest.mark.parametrize("coll,stencil,schedule", [(0, 4, "onepass_rowp2_256x3_s2_np"),
                                                  (1, 4, "onepass_rowp2_256x3_s2_np"),
                                                  (0, 6, "onepass_rowr_w256x3_s1_np"),
                                                  (1, 6, "onepass_rowr_w256x3_s1_np"),
                                                  (0, 6, "onepass_rowc_w256x3_s2"),
                                                  (1, 6, "onepass_rowc_w256x3_s2")])
def test_full_size_headline_schedule_populations_against_oracle(lbm, coll, stencil, schedule):
    """The benchmark's schedule at the benchmark's size, populations compared
    cell by cell: D3Q19, FP32 deviations, 256^3, psi = 1 - exp(-rho), G = -5,
    4th-order stencil, droplet R = 40, with the packed-pair whole-row kernel
    (three rows per item, no producer warp) pinned, BGK and MRT; and the
    6th-order stencil on the radius-2 whole-row kernel (one stage) and on the
    carried-density kernel, BGK and MRT.  At this
    size every block walks several items, so the copy sequence runs on across
    item boundaries.  After three steps every population lies within 2e-6 of
    the largest (FP32 storage of deviations of size ~0.3, rounded at 2^-24)."""
    n = 256
    dom = lbm.Domain(n, n, n, lattice=lbm.LBM_D3Q19, stencil=stencil, precision=1, G=-5.0, tau=1.0,
                     collision=coll)
    dom.set_schedule(schedule)
    dom.init_droplet(2.0, 0.15, 40.0, 2.0)
    dom.step(3)
    f_gpu = dom.get_f()
    dom.close()
    ref = oracle.Sim(oracle.D3Q19, n, n, n, stencil=stencil, G=-5.0, tau=1.0, coll=coll)
    ref.init_droplet(2.0, 0.15, 40.0, 2.0)
    ref.step(3)
    f_ref = ref.get_f()
    del ref
    err = np.abs(f_gpu - f_ref).max() / np.abs(f_ref).max()
    assert err <= 2e-6, err


@pytest.mark.parametrize("schedule", ["onepass_rowc_w256x3_s2", "onepass_rowc_w256x2_s3"])
def test_carried_density_restarts_on_every_state_change(lbm, tmp_path, schedule):
    """The carried-density schedules take psi from a density that the step
    before wrote for them.  Every change of the state must start that density
    again from the populations: populations set from the host, a checkpoint
    loaded, another schedule run in between.  A stale carry would give psi of
    the state before the change, far outside the FP32 budget checked here."""
    nz, ny, nx = 12, 13, 64
    ref = oracle.Sim(oracle.D3Q19, nx, ny, nz, stencil=6, G=-5.0, tau=0.9)
    ref.init_droplet(1.9, 0.15, 4.0, 2.0)
    ref.step(4)
    f4 = ref.get_f()
    snaps = {}
    for t in (10, 13, 15):
        ref.step(t - ref.step_count)
        snaps[t] = ref.get_f()
    dom = lbm.Domain(nx, ny, nz, lattice=lbm.LBM_D3Q19, stencil=6, precision=1, G=-5.0, tau=0.9)
    dom.set_schedule(schedule)
    dom.init_droplet(1.7, 0.2, 3.0, 2.0)  # another state first, so that a carry of it exists
    dom.step(3)
    dom.set_f(f4)
    dom.step(6)
    assert rel_max(dom.get_f(), snaps[10]) <= 1e-5
    ck = str(tmp_path / "state.bin")
    dom.save(ck)
    dom.step(5)
    dom.load(ck)
    dom.step(3)
    assert rel_max(dom.get_f(), snaps[13]) <= 1e-5
    dom.set_schedule("two_pass")
    dom.step(1)
    dom.set_schedule(schedule)
    dom.step(1)
    assert rel_max(dom.get_f(), snaps[15]) <= 1e-5
    dom.close()


@pytest.mark.parametrize("lattice,shape,stencil,coll,precision", [
    (0, (1, 29, 37), 10, 1, 0),
    (0, (1, 40, 300), 4, 0, 1),
    (2, (1, 29, 37), 0, 0, 0),
    (3, (1, 33, 41), 8, 0, 1),
    (1, (11, 20, 37), 6, 1, 0),
    (1, (24, 17, 40), 4, 0, 1),
])
def test_one_pass_matches_two_pass(lbm, lattice, shape, stencil, coll, precision):
    """The one-pass schedule (psi recomputed in a shared-memory ring) and the
    two-pass schedule (psi buffer + TMA tiles) do the same arithmetic."""
    nz, ny, nx = shape
    doms = [lbm.Domain(nx, ny, nz, lattice=lattice, stencil=stencil, collision=coll, tau=0.9,
                       precision=precision, path=path) for path in (1, 2)]
    for d in doms:
        d.init_droplet(1.9, 0.15, min(nx, ny) / 4, 2.0)
        d.step(57)
    a, b = doms[0].get_f(), doms[1].get_f()
    # FP32: the packed-pair kernels order their float operations differently
    assert np.abs(a - b).max() <= (1e-13 if precision == 0 else 1e-5) * np.abs(a).max()


def test_one_pass_ragged_3d_against_oracle(lbm):
    """Chunk and tile edges: 3-D sizes that are not multiples of the 32x8 tile or
    of the 16-slab chunk, marching across the periodic z boundary."""
    dom, ref = pair(lbm, lbm.LBM_D3Q19, (35, 13, 45), stencil=6, tau=0.8, path=2)
    for d in (dom, ref):
        d.init_droplet(1.9, 0.15, 5.0, 2.0)
    dom.step(40)
    ref.step(40)
    assert rel_max(dom.get_f(), ref.get_f()) <= 1e-12


@pytest.mark.parametrize("lattice,shape,stencil,precision,coll", [
    (1, (40, 24, 70), 4, 1, 0),    # 3-D FP32 hot path: every compiled variant
    (1, (12, 10, 128), 4, 1, 0),   # nx = 128 and 256: the whole-row staged variants too
    (1, (9, 10, 256), 4, 1, 0),
    (1, (9, 10, 256), 4, 1, 1),    # MRT on the packed-pair whole-row kernels
    (1, (9, 10, 200), 4, 1, 0),    # runtime row lengths: 200 (three rows per item), ragged rows
    (1, (8, 11, 300), 4, 1, 1),    # 300 (two rows per item), MRT
    (1, (8, 9, 136), 4, 1, 1),     # 136: every run-time width, MRT
    (1, (8, 9, 420), 4, 1, 0),     # 420 (one row per item)
    (1, (21, 19, 37), 6, 1, 0),
    (1, (13, 11, 64), 6, 1, 0),    # radius-2 whole-row kernels (ragged rows and chunks)
    (1, (13, 11, 64), 6, 1, 1),    # MRT with the 6th-order stencil (carried-density kernels)
    (1, (10, 13, 96), 6, 1, 0),    # groups of one row (13 = 4 * 3 + 1 = 6 * 2 + 1): both frames on one row
    (1, (20, 16, 33), 4, 0, 0),
    (1, (13, 11, 256), 4, 0, 1),
    (0, (1, 45, 300), 4, 1, 0),
    (0, (1, 45, 300), 4, 1, 1),    # MRT on the packed-pair segment kernels
    (0, (1, 70, 520), 8, 1, 0),    # radius-2 stencil: every segment variant, ragged tiles and chunks
    (0, (1, 70, 520), 8, 1, 1),
    (0, (1, 37, 260), 10, 1, 0),   # radius 3, the widest halo the segment staging takes
    (0, (1, 37, 260), 10, 1, 1),
    (0, (1, 33, 70), 10, 0, 0),
    (3, (1, 37, 150), 0, 1, 0),
])
def test_every_schedule_variant_matches_oracle(lbm, lattice, shape, stencil, precision, coll):
    """Pin each schedule the autotuner could pick and compare with the oracle
    (FP64: 1e-12; FP32: against the two-pass FP32 result to 1e-6)."""
    nz, ny, nx = shape
    probe = lbm.Domain(nx, ny, nz, lattice=lattice, stencil=stencil, precision=precision, collision=coll)
    names = [k for k in probe.schedule_report() if k != "chosen"]
    probe.close()
    ref = oracle.Sim(LAT[lattice], nx, ny, nz, stencil=stencil, G=-5.0, tau=0.9, coll=coll)
    ref.init_droplet(1.9, 0.15, min(nx, ny) / 4, 2.0)
    ref.step(23)
    f_ref = ref.get_f()
    results = {}
    for name in names:
        dom = lbm.Domain(nx, ny, nz, lattice=lattice, stencil=stencil, precision=precision, tau=0.9,
                         collision=coll)
        dom.set_schedule(name)
        dom.init_droplet(1.9, 0.15, min(nx, ny) / 4, 2.0)
        dom.step(23)
        results[name] = dom.get_f()
        dom.close()
        tol = 1e-12 if precision == 0 else 1e-5
        assert rel_max(results[name], f_ref) <= tol, name
    # FP32 variants order their float operations differently (packed pairs,
    # regrouped sums), so they agree with each other within the FP32 budget
    base = results["two_pass"]
    for name, f in results.items():
        assert np.abs(f - base).max() <= (1e-13 if precision == 0 else 1e-5) * np.abs(base).max(), name


def test_persistent_row_kernel_bitwise_at_full_size(lbm):
    """At 256^3 the persistent whole-row kernel hands every block several items
    (896 items over one block per SM), so its producer runs on from one item
    into the next.  It performs the same arithmetic as the kernel that starts
    every item afresh: after 10 steps the populations are bit-identical."""
    out = {}
    for name in ("onepass_rowp256x2_s2", "onepass_row256x2_zauto_s2_prod"):
        dom = lbm.Domain(256, 256, 256, lattice=lbm.LBM_D3Q19, stencil=4, precision=1, G=-5.0, tau=1.0)
        dom.set_schedule(name)
        dom.init_droplet(2.0, 0.15, 40.0, 2.0)
        dom.step(10)
        out[name] = dom.get_f()
        dom.close()
    a, b = out.values()
    assert np.array_equal(a, b)


@pytest.mark.parametrize("lattice,shape,stencil,coll", [
    (0, (1, 8, 8), 4, 0),      # the smallest box: the halo wraps round more than once per tile
    (0, (1, 33, 31), 10, 1),   # one cell short of and past a tile, radius 3, MRT
    (0, (1, 17, 65), 8, 2),    # exact-difference forcing, rows and columns past a tile
    (2, (1, 15, 33), 0, 2),
    (3, (1, 32, 64), 10, 0),   # reach 2, whole tiles
])
def test_tile_schedules_at_tile_edges(lbm, lattice, shape, stencil, coll):
    """The 2-D tile schedules at their edges against the oracle (FP32 budget of the
    schedule comparison above: 1e-5 after 23 steps)."""
    nz, ny, nx = shape
    probe = lbm.Domain(nx, ny, nz, lattice=lattice, stencil=stencil, precision=1, collision=coll)
    names = [k for k in probe.schedule_report() if k.startswith("tile")]
    probe.close()
    assert len(names) >= 2
    ref = oracle.Sim(LAT[lattice], nx, ny, nz, stencil=stencil, G=-5.0, tau=0.9, coll=coll)
    ref.init_droplet(1.9, 0.15, min(nx, ny) / 4, 2.0)
    ref.step(23)
    for name in names:
        dom = lbm.Domain(nx, ny, nz, lattice=lattice, stencil=stencil, precision=1, tau=0.9, collision=coll)
        dom.set_schedule(name)
        dom.init_droplet(1.9, 0.15, min(nx, ny) / 4, 2.0)
        dom.step(23)
        assert rel_max(dom.get_f(), ref.get_f()) <= 1e-5, name
        dom.close()


@pytest.mark.parametrize("lattice,shape,coll,top", [
    (0, (1, 8, 9), 0, 17.0),     # densities on both sides of the table's end (15.5)
    (0, (1, 64, 76), 1, 2.0),    # 4864 cells: the last size of the early launch
    (0, (1, 60, 82), 0, 2.0),    # 4920: past it
    (0, (1, 389, 401), 1, 2.0),  # 155,989: blocks of more than one warp, a ragged last one
    (2, (1, 9, 11), 2, 17.0),
    (3, (1, 13, 9), 2, 17.0),
    (1, (9, 11, 10), 1, 17.0),
])
def test_fp64_kernels_at_their_edges(lbm, lattice, shape, coll, top):
    """FP64 step where its psi table ends and its launch shape changes, against the oracle:
    3 steps from densities spread over [0.1, top] stay within 1e-12 (operations of 1e-16
    each, some hundreds in a row)."""
    dom, ref = pair(lbm, lattice, shape, coll=coll, G=-0.5, path=1)
    rho = 0.1 + (top - 0.1) * np.random.default_rng(5).random(shape)
    for d in (dom, ref):
        d.init_from_rho(rho)
        d.step(3)
    assert rel_max(dom.get_f(), ref.get_f()) <= 1e-12
    dom.close()


@pytest.mark.parametrize("shape,coll", [
    ((8, 8, 8), 0),       # the smallest box: the halo wraps round in every tile
    ((9, 11, 9), 1),      # odd rows: every alignment of a row occurs, the last pair has one cell
    ((8, 13, 86), 1),     # rows of 8-byte alignment
    ((10, 9, 139), 0),    # the longest odd rows of the five-row tile
    ((8, 9, 231), 1),     # and of the three-row tile, buffer ends off 16 bytes
    ((161, 16, 12), 0),   # items of several chunks along z
])
def test_unaligned_row_schedules(lbm, shape, coll):
    """Whole-row schedules for rows that start on no 16-byte boundary against the oracle
    (FP32 budget of the schedule comparison above: 1e-5 after 23 steps)."""
    nz, ny, nx = shape
    probe = lbm.Domain(nx, ny, nz, lattice=lbm.LBM_D3Q19, stencil=4, precision=1, collision=coll)
    names = [k for k in probe.schedule_report() if k.startswith("onepass_rowu")]
    probe.close()
    assert names
    ref = oracle.Sim(LAT[lbm.LBM_D3Q19], nx, ny, nz, stencil=4, G=-5.0, tau=0.9, coll=coll)
    ref.init_droplet(1.9, 0.15, min(nx, ny, nz) / 4, 2.0)
    ref.step(23)
    for name in names:
        dom = lbm.Domain(nx, ny, nz, lattice=lbm.LBM_D3Q19, stencil=4, precision=1, tau=0.9, collision=coll)
        dom.set_schedule(name)
        dom.init_droplet(1.9, 0.15, min(nx, ny, nz) / 4, 2.0)
        dom.step(23)
        assert rel_max(dom.get_f(), ref.get_f()) <= 1e-5, name
        dom.close()


@pytest.mark.parametrize("lattice,shape,stencil,names", [
    (0, (1, 80, 260), 4, ["onepass_128_z16_b2_smem", "onepass_256_z16_b3_smem", "onepass_256_z16_b3_reg",
                          "onepass_async_256_z16_b2", "onepass_x2_256_z16_b2_smem", "onepass_seg256_z64_s8",
                          "onepass_seg256_z64_s6", "onepass_seg128_z64_s8", "onepass_seg512_z64_s6"]),
    (0, (1, 70, 133), 10, ["onepass_128_z16_b2_smem", "onepass_256_z16_b3_smem", "onepass_async_256_z16_b2"]),
    (2, (1, 66, 130), 6, ["onepass_128_z16_b2_smem", "onepass_256_z16_b3_smem", "onepass_x2_256_z16_b2_smem"])])
def test_untimed_2d_schedules_can_still_be_pinned(lbm, lattice, shape, stencil, names):
    """Schedule names that programs pinned before tiles took over: the step is bitwise
    that of the two-pass schedule (every one-cell form shares its arithmetic, and the
    packed pairs round where it does), but for the march that holds a row in registers,
    which the compiler contracts differently: 40 operations a step, 30 steps."""
    nz, ny, nx = shape
    outs = {}
    for name in ["two_pass"] + names:
        dom = lbm.Domain(nx, ny, nz, lattice=lattice, stencil=stencil, G=-5.0, tau=0.9, precision=1)
        dom.init_droplet(2.0, 0.15, 16.0, 2.5)
        dom.set_schedule(name)
        dom.step(30)
        outs[name] = dom.get_f()
        dom.close()
    for name in names:
        if name.endswith("_reg"):
            assert rel_max(outs[name], outs["two_pass"]) <= 40 * 30 * 2.0 ** -24, name
        else:
            assert np.array_equal(outs[name], outs["two_pass"]), name


@pytest.mark.parametrize("side", [24, 64])
def test_tuned_step_of_a_small_box_is_not_slower_than_two_pass(lbm, side):
    """The schedule that the tuner picks, in calls of many steps (replayed graphs), against
    the two-pass schedule pinned: where launches take most of a trial's time, the tuner
    picked one that is 1.2 (64^3) to 1.6 (24^3) times as slow."""
    import torch

    stream = torch.cuda.Stream()
    ms = {}
    for name in ("two_pass", None):
        dom = lbm.Domain(side, side, side, lattice=1, G=-5.0, tau=0.93, precision=1, stream=stream)
        dom.init_droplet(2.0, 0.15, side / 4, 2.0)
        if name:
            dom.set_schedule(name)
        else:
            dom.schedule_report()
        dom.step(64)
        best = float("inf")
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record(stream)
            dom.step(128)
            b.record(stream)
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        ms[name] = best
        dom.close()
    assert ms[None] <= 1.1 * ms["two_pass"], ms


@pytest.mark.parametrize("lattice,shape,radius", [(0, (1, 40, 48), 1), (3, (1, 40, 48), 2), (1, (12, 16, 20), 1)])
def test_fp64_domain_takes_two_population_buffers_and_psi(lbm, monkeypatch, lattice, shape, radius):
    """Device memory of an FP64 domain: two buffers of its populations, psi with its
    ghosts, and what does not grow with the cells; stepping takes no more."""
    nz, ny, nx = shape
    sizes = []

    class Counting(lbm.TorchAllocator):
        def _alloc(self, nbytes, ctx):
            sizes.append(nbytes)
            return super()._alloc(nbytes, ctx)

    monkeypatch.setattr(lbm, "TorchAllocator", Counting)
    dom = lbm.Domain(nx, ny, nz, lattice=lattice, G=-5.0, precision=0, torch_alloc=True)
    psi = 8 * ((nx + 8 + 3) // 4 * 4) * (ny + 2 * radius) * (nz + (2 * radius if nz > 1 else 0))
    assert sizes[:3] == [8 * dom.Q * dom.N] * 2 + [psi]
    dom.init_droplet(2.0, 0.15, 4.0 if nz > 1 else 12.0, 2.0)
    taken = len(sizes)
    dom.step(20)
    assert len(sizes) == taken
    dom.close()
