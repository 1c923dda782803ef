"""Round-off of the FP64 kernels, measured against extended precision (numpy's
longdouble) from the same state, tables and parameters (weights, c_s^2, force weights
times c_s^2, 2 / (G c_s^2), each rounded to double).

The kernels regroup the printed formulas; a regrouping that rounds a shared factor
once too often is off in the same direction in every cell and step.  The measure is
the plain form: the printed formulas, term by term, in double precision.
"""
import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

LD = np.longdouble


def _pr_parameters(T_over_Tc):
    """T and alpha(T) of the Peng-Robinson EOS as the library forms them (double)."""
    eta = 0.25
    for _ in range(60):
        step = (((eta + 1.0) * eta + 1.0) * eta - 1.0 / 3.0) / ((3.0 * eta + 2.0) * eta + 1.0)
        eta -= step
        if abs(step) < 1e-17:
            break
    d = 1.0 + 2.0 * eta - eta * eta
    tc = 2.0 * (2.0 / 49.0) * (eta / (2.0 / 21.0)) * (1.0 + eta) * (1.0 - eta) * (1.0 - eta) / (d * d)
    k = 0.37464 + 1.54226 * 0.344 - 0.26992 * 0.344 * 0.344
    s = 1.0 + k * (1.0 - math.sqrt(T_over_Tc))
    return T_over_Tc * tc, s * s


class Plain:
    """The step as printed (Guo or exact-difference forcing, BGK) in one number type."""

    def __init__(self, real, lattice, stencil, T_over_Tc, G, tau, exact_difference):
        self.real = real
        c, w, cs2 = oracle.lattice_table(lattice)
        self.c, self.w, self.cs2 = c, [real(v) for v in w], real(cs2)
        dim = 3 if lattice == oracle.D3Q19 else 2
        e, we = oracle.stencil_table(dim, stencil)
        self.force = [(tuple(v), real(q * cs2)) for v, q in zip(e, we)]
        self.pr = [real(v) for v in _pr_parameters(T_over_Tc)] if T_over_Tc else None
        self.G, self.omega, self.edm = real(G), real(1.0 / tau), exact_difference
        self.K = real(2.0 / (G * cs2))  # a parameter like the weights: rounded once to double

    def psi(self, r):
        if self.pr is None:
            return -np.expm1(-r)
        T, alpha = self.pr
        a, b = self.real(2.0 / 49.0), self.real(2.0 / 21.0)
        p = r * T / (1 - b * r) - a * alpha * r * r / (1 + 2 * b * r - b * b * r * r)
        return np.sqrt(self.K * (p - self.cs2 * r))

    def step(self, f):
        s, w = self.cs2, self.omega
        rho = sum(f)
        j = [sum(int(v[k]) * x for x, v in zip(f, self.c)) for k in range(3)]
        psi = self.psi(rho)
        F = [np.zeros_like(psi) for _ in range(3)]
        for e, q in self.force:
            shifted = np.roll(psi, (-e[2], -e[1], -e[0]), (0, 1, 2))
            for k in range(3):
                if e[k]:
                    F[k] = F[k] + q * int(e[k]) * shifted
        F = [-self.G * psi * x for x in F]

        def eq(b, u):
            cu = sum(int(self.c[b][k]) * u[k] for k in range(3))
            return self.w[b] * rho * (1 + cu / s + cu * cu / (2 * s * s) - sum(x * x for x in u) / (2 * s))

        out = []
        if self.edm:
            u = [x / rho for x in j]
            v = [(x + y) / rho for x, y in zip(j, F)]
            for b in range(len(f)):
                out.append((1 - w) * f[b] - (1 - w) * eq(b, u) + eq(b, v))
        else:
            u = [(x + y / 2) / rho for x, y in zip(j, F)]
            uF = sum(x * y for x, y in zip(u, F))
            for b in range(len(f)):
                cu = sum(int(self.c[b][k]) * u[k] for k in range(3))
                cF = sum(int(self.c[b][k]) * F[k] for k in range(3))
                out.append(f[b] - w * (f[b] - eq(b, u))
                           + (1 - w / 2) * self.w[b] * ((cF - uF) / s + cu * cF / (s * s)))
        return [np.roll(x, (int(v[2]), int(v[1]), int(v[0])), (0, 1, 2)) for x, v in zip(out, self.c)]

    def run(self, f, steps):
        f = [x.astype(self.real) for x in f]
        for _ in range(steps):
            f = self.step(f)
        return np.stack(f)


@pytest.mark.parametrize("lattice,shape,stencil,T_over_Tc,G,tau,coll,steps", [
    (oracle.D2Q25, (1, 60, 60), 8, 0.9, -1.0, 1.0, 2, 60),
    (oracle.D2Q25, (1, 60, 60), 8, 0.95, -1.0, 1.0, 2, 60),
    (oracle.D2Q9, (1, 64, 64), 4, 0.0, -4.8, 0.9, 0, 100),
    (oracle.D3Q19, (26, 28, 24), 4, 0.0, -4.8, 0.9, 0, 40),
])
def test_fp64_step_is_as_accurate_as_the_plain_form(lbm, lattice, shape, stencil, T_over_Tc, G, tau, coll, steps):
    """RMS error over the populations, mean of two droplets, at most 1.25 times the plain
    form's: two means of the same round-off spread by some 20%."""
    nz, ny, nx = shape
    mine, plain = [], []
    for k in range(2):
        dom = lbm.Domain(nx, ny, nz, lattice=lattice, stencil=stencil, collision=coll, G=G, tau=tau,
                         psi=1 if T_over_Tc else 0, T_over_Tc=T_over_Tc, precision=0)
        rl, rg = {0.0: (2.0, 0.15), 0.9: (5.91, 0.58), 0.95: (4.93, 1.013)}[T_over_Tc]
        dom.init_droplet(rl, rg, min(nx, ny) * (0.22 + 0.05 * k), 4.0 if T_over_Tc else 2.5)
        f0 = dom.get_f()
        dom.step(steps)
        f = dom.get_f()
        dom.close()
        args = (lattice, stencil, T_over_Tc, G, tau, coll == 2)
        ref = Plain(LD, *args).run(f0, steps)
        norm = float(np.sqrt((ref * ref).sum()))
        mine.append(float(np.sqrt(((f - ref) ** 2).sum())) / norm)
        plain.append(float(np.sqrt(((Plain(np.float64, *args).run(f0, steps) - ref) ** 2).sum())) / norm)
    assert np.mean(mine) <= 1.25 * np.mean(plain), (mine, plain)


def test_fp64_psi_at_low_density(lbm):
    """psi = 1 - exp(-rho) for 1/128 <= rho < 1/64, through the force of a rest state:
    columns [tiny, r, r], so that at the first r only psi(r) pulls and the velocity is
    G psi(r)^2 c_s^2 / (2 r) with nothing cancelled.  RMS error at most 1.25 times that of
    the same expression in double precision with the C library's expm1."""
    n = 2048
    rng = np.random.default_rng(3)
    rho = np.zeros((1, 8, 3 * n))
    rho[:, :, 0::3] = 1e-14
    rho[:, :, 1::3] = rho[:, :, 2::3] = rng.uniform(1.0 / 128, 1.0 / 64, n)
    dom = lbm.Domain(3 * n, 8, G=-5.0, tau=1.0, precision=0)
    dom.init_from_rho(rho)
    got = dom.fields()
    f = dom.get_f()[:, 0, 0]
    dom.close()
    # the density that psi is taken of: the populations by opposite pairs
    pairs = f[0].copy()
    for b in range(1, 9, 2):
        pairs += f[b] + f[b + 1]

    def velocity(real):
        r = got["rho"][0, 0].astype(real)
        psi = -np.expm1(-pairs.astype(real))
        d = psi[2::3] - psi[0::3]
        w1, w2 = real((1.0 / 3.0) * (1.0 / 3.0)), real((1.0 / 12.0) * (1.0 / 3.0))
        return real(5.0) * psi[1::3] * (w1 * d + w2 * d + w2 * d) / 2 / r[1::3]

    ref = velocity(LD)

    def rms(u):
        return float(np.sqrt((((u - ref) / ref) ** 2).mean()))

    assert rms(got["u"][0, 0, 1::3, 0]) <= 1.25 * rms(velocity(np.float64))


@pytest.mark.parametrize("lattice", [oracle.D2Q9, oracle.D2Q13, oracle.D2Q25, oracle.D3Q19])
@pytest.mark.parametrize("rho", [3e-307, 3e-308])
def test_fp64_populations_below_the_normal_range(lbm, lattice, rho):
    """A rest state so thin that the outer populations are subnormal: each is a product
    rounded to a multiple of 2^-1074, so a step moves a population by at most 2^-1074 per
    operation on it (20) besides the round-off of the normal ones."""
    shape = (8, 8, 8) if lattice == oracle.D3Q19 else (1, 8, 8)
    dom = lbm.Domain(*shape[::-1], lattice=lattice, G=-5.0, tau=1.0, precision=0)
    dom.init_from_rho(np.full(shape, rho))
    f0 = dom.get_f()
    dom.step(2)
    f = dom.get_f()
    dom.close()
    _, w, _ = oracle.lattice_table(lattice)
    assert np.abs(f0 - (w * rho)[:, None, None, None]).max() <= 2 * 5e-324
    assert np.abs(f - f0).max() <= 40 * 5e-324 + 1e-14 * rho


@pytest.mark.parametrize("lattice,shape,stencil,coll", [
    (oracle.D2Q9, (1, 96, 128), 4, 0), (oracle.D2Q9, (1, 96, 128), 8, 1), (oracle.D2Q13, (1, 96, 128), 6, 0),
    (oracle.D3Q19, (34, 36, 44), 4, 0), (oracle.D3Q19, (34, 36, 44), 4, 1), (oracle.D3Q19, (34, 36, 44), 6, 0)])
@pytest.mark.parametrize("tau", [0.8, 0.9])
def test_fp32_schedules_share_one_round_off(lbm, lattice, shape, stencil, coll, tau):
    """Every FP32 schedule rounds the collision's large terms at the same places, so its
    RMS error against an FP64 run, mean of six droplets, is the two-pass schedule's
    within 6% (the order of the small terms differs).  omega is exact in single
    precision at tau = 0.8 and off by 5e-8 at 0.9, where 1 - omega has to match it."""
    nz, ny, nx = shape
    names, err = None, {}
    for k in range(6):
        par = (2.0 - 0.02 * k, 0.15, min(v for v in shape if v > 1) * (0.2 + 0.016 * k), 2.0 + 0.15 * k)
        args = dict(lattice=lattice, stencil=stencil, collision=coll, G=-5.1 + 0.06 * k, tau=tau)
        dom = lbm.Domain(nx, ny, nz, precision=0, **args)
        dom.init_droplet(*par)
        dom.step(80)
        ref = dom.get_f()
        dom.close()
        dom = lbm.Domain(nx, ny, nz, precision=1, **args)
        dom.init_droplet(*par)
        f0 = dom.get_f()
        names = names or [n for n in dom.schedule_report() if n != "chosen"]
        for name in names:
            dom.set_f(f0)
            dom.set_schedule(name)
            dom.step(80)
            err.setdefault(name, []).append(np.linalg.norm(dom.get_f() - ref) / np.linalg.norm(ref))
        dom.close()
    two_pass = np.mean(err["two_pass"])
    off = {n: np.mean(v) / two_pass for n, v in err.items() if not np.mean(v) <= 1.06 * two_pass}
    assert not off, off


@pytest.mark.parametrize("lattice,stencil,coll", [
    (oracle.D2Q9, 4, 0), (oracle.D2Q9, 10, 0), (oracle.D2Q9, 8, 1), (oracle.D2Q13, 6, 0), (oracle.D2Q25, 8, 0)])
def test_fp32_schedules_of_a_plane_are_bitwise_alike(lbm, lattice, stencil, coll):
    outs = {}
    dom = lbm.Domain(132, 70, lattice=lattice, stencil=stencil, collision=coll, G=-5.0, tau=0.87, precision=1)
    dom.init_droplet(2.0, 0.15, 18.0, 2.5)
    f0 = dom.get_f()
    # (the march that holds a row in registers is compiled with other contractions)
    for name in [n for n in dom.schedule_report() if n != "chosen" and not n.endswith("_reg")]:
        dom.set_f(f0)
        dom.set_schedule(name)
        dom.step(60)
        outs[name] = dom.get_f()
    dom.close()
    assert len(outs) >= 2 and np.isfinite(outs["two_pass"]).all()
    for name, f in outs.items():
        assert np.array_equal(f, outs["two_pass"]), name
