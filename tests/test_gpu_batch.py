"""Batched sweep (many independent D2Q9 domains in one persistent kernel and a
CUDA graph) against the FP64 oracle, domain by domain, and against
single-domain runs of the library."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

DOMAINS = [
    dict(nx=64, ny=64, G=-5.0, tau=1.0, stencil=4, rho_l=2.0, rho_g=0.15, R=16.0, width=2.0),
    dict(nx=96, ny=80, G=-4.8, tau=0.8, stencil=6, rho_l=1.8, rho_g=0.2, R=20.0, width=2.0),
    dict(nx=37, ny=45, G=-5.5, tau=0.6, stencil=10, rho_l=2.2, rho_g=0.1, R=9.0, width=2.0),
    dict(nx=128, ny=64, G=-5.2, tau=1.0, stencil=8, rho_l=2.0, rho_g=0.13, R=14.0, width=3.0),
    dict(nx=70, ny=33, G=-4.6, tau=0.7, stencil=4, rho_l=1.6, rho_g=0.22, R=10.0, width=2.0),
]


def oracle_run(d, steps):
    s = oracle.Sim(oracle.D2Q9, d["nx"], d["ny"], stencil=d["stencil"], G=d["G"], tau=d["tau"])
    s.init_droplet(d["rho_l"], d["rho_g"], d["R"], d["width"])
    s.step(steps)
    return s


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-5)])
def test_batch_matches_oracle_per_domain(lbm, precision, tol):
    b = lbm.Batch(DOMAINS, precision=precision)
    b.step(120)
    for i, d in enumerate(DOMAINS):
        ref = oracle_run(d, 120)
        f_ref = ref.get_f()
        f = b.get_f(i)
        assert np.abs(f - f_ref).max() <= tol * np.abs(f_ref).max(), i
        o = b.observables()[i]
        oo = ref.observables()
        assert o["mass"] == pytest.approx(oo["mass"], rel=1e-12 if precision == 0 else 1e-6)
        assert o["max_u"] == pytest.approx(oo["max_u"], rel=1e-9 if precision == 0 else 1e-2)
        assert o["rho_l"] == pytest.approx(oo["rho_l"], rel=1e-12 if precision == 0 else 1e-4)
    b.close()


def test_batch_odd_steps_and_bitwise_repeat(lbm):
    outs = []
    for _ in range(2):
        b = lbm.Batch(DOMAINS[:3], precision=1)
        b.step(31)
        b.step(8)
        outs.append([b.get_f(i) for i in range(3)])
        b.close()
    for a, c in zip(*outs):
        assert np.array_equal(a, c)
    ref = oracle_run(DOMAINS[2], 39)
    assert np.abs(outs[0][2] - ref.get_f()).max() <= 1e-5 * np.abs(ref.get_f()).max()


def test_batch_run_to_steady_retires_domains(lbm):
    doms = [dict(nx=48, ny=48, G=-5.0, tau=1.0, stencil=4, rho_l=1.93, rho_g=0.16, R=r, width=2.0)
            for r in (8.0, 12.0)]
    doms.append(dict(nx=64, ny=64, G=-5.0, tau=0.7, stencil=8, rho_l=1.93, rho_g=0.16, R=16.0, width=2.0))
    b = lbm.Batch(doms, precision=0)
    steps, obs, ok = b.run_to_steady(1e-9, 200000, 50)
    assert ok
    assert all(s % 50 == 0 and 0 < s < 200000 for s in steps)
    # each domain stopped where a single-domain run with the same rule stops
    for i, d in enumerate(doms):
        dom = lbm.Domain(d["nx"], d["ny"], G=d["G"], tau=d["tau"], stencil=d["stencil"])
        dom.init_droplet(d["rho_l"], d["rho_g"], d["R"], d["width"])
        s1, ok1 = dom.run_to_steady(1e-9, 200000, 50)
        # the same rule on the same FP64 trajectory stops at the same check; a
        # last-bit difference between kernels may move a borderline stop by one check
        assert ok1 and abs(s1 - steps[i]) <= 50
        o1 = dom.observables()
        assert obs[i]["max_u"] == pytest.approx(o1["max_u"], rel=1e-10 if s1 == steps[i] else 1e-3)
        assert obs[i]["mass"] == pytest.approx(o1["mass"], rel=1e-12)
    b.close()


def test_batch_fp32_steady_agrees_with_fp64(lbm):
    """The sweep's acceptance: FP32 batched steady max|u| within 5% of FP64."""
    doms = [dict(nx=64, ny=64, G=g, tau=t, stencil=o, rho_l=2.0, rho_g=0.15, R=r, width=2.0)
            for g, t, o, r in ((-5.0, 1.0, 4, 14.0), (-4.6, 0.8, 6, 12.0), (-5.4, 0.8, 10, 18.0))]
    b32 = lbm.Batch(doms, precision=1)
    b64 = lbm.Batch(doms, precision=0)
    s32, o32, ok32 = b32.run_to_steady(1e-10, 200000, 100)
    s64, o64, ok64 = b64.run_to_steady(1e-10, 200000, 100)
    assert ok32 and ok64
    for a, c in zip(o32, o64):
        assert a["max_u"] == pytest.approx(c["max_u"], rel=0.05)
        assert a["rho_l"] == pytest.approx(c["rho_l"], rel=1e-3)


def test_batch_rejects_unsupported(lbm):
    d = dict(DOMAINS[0])
    p = lbm.lbm_params_default()
    p.lattice = lbm.LBM_D3Q19
    p.nz = 16
    with pytest.raises(lbm.LbmError):
        lbm.lbm_batch_create([p], [2.0, 0.15, 8.0, 2.0])
    del d


def test_batch_retires_diverged_domain(lbm):
    """G = -5.4 at tau = 0.6 with the 10th-order stencil diverges under BGK; the
    batch retires it (max_u = inf) and the stable domain still converges."""
    doms = [dict(nx=64, ny=64, G=-5.4, tau=0.6, stencil=10, rho_l=2.0, rho_g=0.15, R=18.0, width=2.0),
            dict(nx=48, ny=48, G=-5.0, tau=1.0, stencil=4, rho_l=1.93, rho_g=0.16, R=10.0, width=2.0)]
    b = lbm.Batch(doms, precision=0)
    steps, obs, ok = b.run_to_steady(1e-9, 200000, 50)
    assert ok
    assert obs[0]["max_u"] == float("inf")
    assert np.isfinite(obs[1]["max_u"]) and obs[1]["max_u"] < 1e-2


def test_batch_autotuner_reports_and_every_shape_is_bitwise_equal(lbm):
    """The tile shapes perform the same per-cell arithmetic: every shape gives
    the same bits after the same steps, and the autotuner (which times them on a
    saved copy of the state) leaves the state where it was."""
    rep = None
    outs = {}
    b = lbm.Batch(DOMAINS, precision=1)
    rep = b.schedule_report()
    assert rep["chosen"] in rep and len(rep) >= 5
    b.step(17)
    outs["auto"] = [b.get_f(i) for i in range(len(DOMAINS))]
    b.close()
    for name in [k for k in rep if k != "chosen"]:
        b = lbm.Batch(DOMAINS, precision=1)
        b.set_schedule(name)
        b.step(17)
        outs[name] = [b.get_f(i) for i in range(len(DOMAINS))]
        b.close()
    for name, fs in outs.items():
        for a, c in zip(fs, outs["auto"]):
            assert np.array_equal(a, c), name
    ref = oracle_run(DOMAINS[1], 17)
    assert np.abs(outs["auto"][1] - ref.get_f()).max() <= 1e-5 * np.abs(ref.get_f()).max()
    b = lbm.Batch(DOMAINS[:1], precision=0)
    with pytest.raises(lbm.LbmError):
        b.set_schedule("no_such_shape")
    b.close()


STAGED_DOMAINS = [
    dict(nx=64, ny=64, G=-5.0, tau=1.0, stencil=4, rho_l=2.0, rho_g=0.15, R=16.0, width=2.0),
    dict(nx=96, ny=80, G=-4.8, tau=0.8, stencil=6, rho_l=1.8, rho_g=0.2, R=20.0, width=2.0),
    dict(nx=68, ny=45, G=-5.5, tau=0.6, stencil=10, rho_l=2.2, rho_g=0.1, R=9.0, width=2.0),
    dict(nx=132, ny=70, G=-5.2, tau=1.0, stencil=8, rho_l=2.0, rho_g=0.13, R=14.0, width=3.0),
]


def test_batch_staged_shapes_match_oracle_and_each_other(lbm):
    """Bulk-copy staged shapes (FP32, every nx a multiple of 4; ragged tiles and
    row chunks): each matches the oracle per domain and the plain tiled shape
    bit for bit; an FP64 batch refuses them."""
    b = lbm.Batch(STAGED_DOMAINS, precision=1)
    names = [k for k in b.schedule_report() if k != "chosen"]
    b.close()
    staged = [n for n in names if n.startswith("staged")]
    assert len(staged) >= 3
    outs = {}
    for name in ["tile64_rows16"] + staged:
        b = lbm.Batch(STAGED_DOMAINS, precision=1)
        b.set_schedule(name)
        b.step(41)
        outs[name] = [b.get_f(i) for i in range(len(STAGED_DOMAINS))]
        b.close()
    for name in staged:
        for a, c in zip(outs[name], outs["tile64_rows16"]):
            assert np.array_equal(a, c), name
    for i, d in enumerate(STAGED_DOMAINS):
        ref = oracle_run(d, 41).get_f()
        assert np.abs(outs[staged[0]][i] - ref).max() <= 1e-5 * np.abs(ref).max(), i
    b = lbm.Batch(STAGED_DOMAINS, precision=0)
    with pytest.raises(lbm.LbmError):
        b.set_schedule(staged[0])
    b.close()


RESIDENT_DOMAINS = STAGED_DOMAINS + [
    dict(nx=8, ny=8, G=-4.5, tau=1.0, stencil=10, rho_l=1.4, rho_g=0.3, R=2.0, width=2.0),    # bands of 4 rows
    dict(nx=38, ny=45, G=-5.5, tau=0.6, stencil=10, rho_l=2.2, rho_g=0.1, R=9.0, width=2.0),  # odd rows, 19 pairs
    dict(nx=70, ny=33, G=-4.6, tau=0.7, stencil=4, rho_l=1.6, rho_g=0.22, R=10.0, width=2.0),
    dict(nx=256, ny=256, G=-5.0, tau=0.8, stencil=10, rho_l=2.0, rho_g=0.15, R=60.0, width=2.0),  # 16 blocks
    dict(nx=192, ny=190, G=-4.9, tau=1.0, stencil=8, rho_l=2.0, rho_g=0.15, R=40.0, width=2.0),   # uneven bands
    dict(nx=500, ny=20, G=-4.9, tau=0.9, stencil=6, rho_l=2.0, rho_g=0.15, R=6.0, width=2.0),
]


@pytest.mark.parametrize("doms", [RESIDENT_DOMAINS, RESIDENT_DOMAINS[4:5], RESIDENT_DOMAINS[7:9]])
def test_batch_resident_shape_is_bitwise_the_tiled_one(lbm, doms):
    """The cluster-resident shape against the tiled one after odd and even numbers
    of steps (the state changes pools), bit for bit, with few domains (spread over
    more blocks) and many; odd nx and FP64 are refused."""
    outs = {}
    for name in ("tile64_rows16", "resident_cluster"):
        b = lbm.Batch(doms, precision=1)
        b.set_schedule(name)
        b.step(7)
        first = [b.get_f(i) for i in range(len(doms))]
        b.step(12)
        outs[name] = (first, [b.get_f(i) for i in range(len(doms))])
        b.close()
    for a, c in zip(*outs.values()):
        for i, (x, y) in enumerate(zip(a, c)):
            assert np.array_equal(x, y), i
    for bad, precision in ((DOMAINS[2:3], 1), (doms, 0)):
        b = lbm.Batch(bad, precision=precision)
        with pytest.raises(lbm.LbmError):
            b.set_schedule("resident_cluster")
        b.close()


MIXED_SIDES = [64, 96, 128, 192, 256] * 8


def mixed_domains():
    return [dict(nx=n, ny=n, G=-5.0 + 0.01 * i, tau=0.9, R=0.2 * n, stencil=(4, 6, 8, 10)[i % 4], rho_l=2.0,
                 rho_g=0.15, width=2.0) for i, n in enumerate(MIXED_SIDES)]


def test_batch_single_steps_do_not_pay_for_long_calls(lbm):
    """The tuned batch takes a call of one step about as fast as a pinned per-step shape
    (a resident call loads and stores every domain and forks a stream per cluster size:
    3.7 times as slow), and long calls by the faster of the two, whatever came before."""
    import time

    import torch

    def per_step(b, n, calls):
        best = float("inf")
        for _ in range(5):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(calls):
                b.step(n)
            torch.cuda.synchronize()
            best = min(best, (time.perf_counter() - t) / (n * calls))
        return best

    times = {}
    for name in (None, "tile128_rows16", "resident_cluster"):
        b = lbm.Batch(mixed_domains(), precision=1)
        if name:
            b.set_schedule(name)
        b.step(2)
        times[name] = (per_step(b, 1, 100), per_step(b, 2, 50), per_step(b, 128, 4))
        b.close()
    for auto, tile, resident in zip(*times.values()):
        assert auto <= 1.3 * min(tile, resident), times


def resting(n, k):
    """Domains of one density: steady at the first check."""
    return [dict(nx=n, ny=n, G=-4.5, tau=1.0, stencil=4, rho_l=0.7, rho_g=0.7, R=n / 4, width=2.0) for _ in range(k)]


def test_batch_resident_survivors_spread_over_freed_sms(lbm):
    """149 of 150 domains retire at the first check: the last one then runs about as
    fast as alone, on as many SMs (it stayed on one, among clusters without work)."""
    import time

    import torch

    drop = dict(nx=64, ny=64, G=-5.0, tau=1.0, stencil=4, rho_l=2.0, rho_g=0.15, R=16.0, width=2.0)
    times = []
    for doms in ([drop], [drop] + resting(64, 149)):
        b = lbm.Batch(doms, precision=1)
        b.set_schedule("resident_cluster")
        steps, _, ok = b.run_to_steady(1e-12, 400, 100)
        assert not ok and list(steps) == [400] + [100] * (len(doms) - 1)
        torch.cuda.synchronize()
        t = time.perf_counter()
        b.run_to_steady(1e-12, 4000, 100)
        times.append(time.perf_counter() - t)
        b.close()
    assert times[1] <= 2.0 * times[0], times


def test_batch_resident_steady_runs_bitwise_like_the_tiled_shape(lbm):
    """Clusters of several sizes, forked and joined inside the captured steady block,
    while domains retire at different checks; then plain steps of what is left, and a
    call longer than one launch takes (4096 steps) from an odd number of steps on."""
    doms = [RESIDENT_DOMAINS[k] for k in (0, 1, 6, 8, 9)] + resting(48, 6) + resting(256, 2)
    doms.append(dict(nx=40, ny=44, G=-5.0, tau=1.0, stencil=4, rho_l=1.93, rho_g=0.16, R=9.0, width=3.0))
    outs = {}
    for name in ("tile64_rows16", "resident_cluster"):
        b = lbm.Batch(doms, precision=1)
        b.set_schedule(name)
        b.step(3)
        steps, obs, ok = b.run_to_steady(2e-7, 1200, 100)
        again = b.run_to_steady(2e-7, 600, 50)
        b.step(5)
        outs[name] = (list(steps), obs, ok, list(again[0]), again[1], [b.get_f(i) for i in range(len(doms))])
        b.close()
    a, c = outs.values()
    assert a[:5] == c[:5]
    assert len(set(a[0])) >= 3, a[0]  # retired at different checks
    for i, (x, y) in enumerate(zip(a[5], c[5])):
        assert np.array_equal(x, y), i
    long = [dict(nx=8, ny=8, G=-4.5, tau=1.0, stencil=s, rho_l=1.4, rho_g=0.3, R=2.0, width=2.0) for s in (4, 10)]
    long.append(dict(nx=16, ny=20, G=-4.5, tau=1.0, stencil=6, rho_l=1.4, rho_g=0.3, R=4.0, width=2.0))
    fs = []
    for name in ("tile32_rows8", "resident_cluster"):
        b = lbm.Batch(long, precision=1)
        b.set_schedule(name)
        b.step(7)
        b.step(4097 + 2)
        fs.append([b.get_f(i) for i in range(len(long))])
        b.close()
    for x, y in zip(*fs):
        assert np.array_equal(x, y)


def test_batch_steady_run_takes_its_own_tolerance(lbm):
    """A second run with the same check interval and a looser tolerance retires by that
    tolerance (the captured check kept the first run's)."""
    b = lbm.Batch(DOMAINS[:1], precision=0)
    steps, _, ok = b.run_to_steady(1e-14, 200, 100)
    assert not ok and steps[0] == 200
    steps, _, ok = b.run_to_steady(1.0, 400, 100)
    assert ok and steps[0] == 300
    b.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_batch_state_io_needs_no_memory(lbm, precision):
    """Reading and writing populations works when the allocator has nothing left, takes
    nothing from it, and leaves every domain, running or retired, as it was."""
    b = lbm.Batch(DOMAINS + resting(40, 1), precision=precision, torch_alloc=True)
    b.step(3)
    steps, _, _ = b.run_to_steady(1e-9, 100, 50)
    assert steps[-1] < steps[0]  # the resting domain has retired
    alloc, live = b._alloc, b._alloc.live
    torch = alloc._torch

    class Spent:
        class cuda:
            @staticmethod
            def caching_allocator_alloc(*a):
                raise MemoryError

            caching_allocator_delete = staticmethod(torch.cuda.caching_allocator_delete)

    alloc._torch = Spent
    fs = [b.get_f(i) for i in range(b.n)]
    for i, f in enumerate(fs):
        b.set_f(i, f)
    for i, f in enumerate(fs):
        assert np.array_equal(b.get_f(i), f), i
    assert alloc.live == live
    b.step(5)
    assert np.array_equal(b.get_f(b.n - 1), fs[-1]) and not np.array_equal(b.get_f(0), fs[0])
    b.close()
    assert alloc.live == 0
