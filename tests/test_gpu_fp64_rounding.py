"""Rounding of the FP64 operators where a smooth field's differences are far
smaller than the field: the rows difference a field before they combine it with
another or scale it, so that a row's rounding error is of its terms' size, not
of the fields'.  Each bound counts roundings of the terms (u = 2^-53) and was
set from that count.

The diffusion flux of N_c and N_p, sum over a cell's faces of (m + m_q)
((mu_q - mu) + alpha (p_q - p)), at rest with c = c^n = 1 and mobility 1: every
other term of the two rows is then exactly zero.  A face takes two differences,
one product each and two additions, the sum two more operations: at most 8 u of
sum 2 (|mu_q - mu| + alpha |p_q - p|).  Grids: one on each side of the sizes
that change the residual's launch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
LD = np.longdouble


@pytest.fixture(scope="module")
def qn():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_06606_gb300 import qnsch
    return qnsch


# fluid 1 is 100 times lighter: alpha = 99; M = 1, eta = 1
KW = dict(rho1=0.01, rho2=1.0, eta1=1.0, eta2=1.0, Re=10.0, We=1e6, Pe=1.0, Cn=1.0, eps_mob=1.0,
          eta_st=1.0)


def resting(m1, m2):
    """c = 1, no flow, smooth mu near 1 and p of size 10."""
    x, y = np.meshgrid((np.arange(m1) + 0.5) / m1, (np.arange(m2) + 0.5) / m1)
    return dict(c=np.ones((m2, m1)), mu=1.0 + 0.25 * np.sin(2 * np.pi * x + 1.0) * np.cos(3.0 * y),
                p=10.0 * np.cos(2 * np.pi * x) * np.sin(5.0 * y + 0.3),
                u=np.zeros((m2, m1 + 1)), v=np.zeros((m2 + 1, m1)))


def faces(a, px):
    """a's differences to the east, west, north and south neighbours (0 across a
    wall) in extended precision."""
    a = a.astype(LD)
    e = np.concatenate([a, a[:, :1] if px else a[:, -1:]], axis=1)
    w = np.concatenate([a[:, -1:] if px else a[:, :1], a], axis=1)
    n, s = np.concatenate([a, a[-1:]]), np.concatenate([a[:1], a])
    return [e[:, 1:] - a, w[:, :-1] - a, n[1:] - a, s[:-1] - a]


def flux(f, alpha, px):
    """The flux sum with m = 1, and the sum of its terms' sizes."""
    dm, dp = faces(f["mu"], px), faces(f["p"], px)
    return (2 * sum(a + alpha * b for a, b in zip(dm, dp)),
            2 * sum(abs(a) + alpha * abs(b) for a, b in zip(dm, dp)))


@pytest.mark.parametrize("scheme", [0, 1], ids=["primitive", "projection"])
@pytest.mark.parametrize("m1,m2,px", [(1024, 32, False), (512, 66, True), (1024, 64, True),
                                      (1024, 2048, False)])
def test_flux_of_the_residual(qn, m1, m2, px, scheme):
    if scheme and m2 == 2048:
        m2 = 1024
    s = qn.Solver(m1, m2, periodic_x=px, scheme=scheme, levels=1, **KW)
    f = resting(m1, m2)
    s.set_fields(f)
    s.begin_step(1.0)
    r, _ = s.residual()
    s.close()
    alpha, dif = LD((1.0 - 0.01) / 0.01), 0.5 * float(m1) ** 2
    F, size = flux(f, alpha, px)
    assert np.all(abs(r["c"].astype(LD) - dif * F) <= 8 * U * dif * size)
    if not scheme:  # the projection method's N_p holds the pressure's own gradient too
        assert np.all(abs(r["p"].astype(LD) - alpha * dif * F) <= 9 * U * alpha * dif * size)


@pytest.mark.parametrize("team", [0, 1 << 20], ids=["one_lane", "four_lanes"])
@pytest.mark.parametrize("px", [False, True])
def test_flux_of_the_ch_visit(qn, px, team):
    """One CH visit at the same state: the Newton step of the 2x2 system in
    extended precision.  R_c carries the flux's error, R_mu = rho mu one
    rounding, and the solve's products and reciprocal 8 u of the terms that they
    form (kappa: those of the determinant, over it)."""
    m1, m2 = 1024, 32
    s = qn.Solver(m1, m2, periodic_x=px, levels=1, ch_team_max=team, **KW)
    f = resting(m1, m2)
    s.set_fields(f)
    s.begin_step(1.0)
    s.smooth_ch(0)
    g = s.get_iterate()
    s.close()
    a = (1.0 - 0.01) / 0.01
    alpha, rho, h2 = LD(a), LD(1.0 / (a + 1.0)), LD(m1) ** 2
    K = Lam = LD(1e-6)
    F, size = flux(f, alpha, px)
    mu = f["mu"].astype(LD)
    open_ = np.full((m2, m1), 4.0)
    open_[0] -= 1
    open_[-1] -= 1
    if not px:
        open_[:, 0] -= 1
        open_[:, -1] -= 1
    J00, J01, J11 = rho, h2 * open_, rho
    J10 = -alpha * rho ** 2 * mu - K / 8 * 2 * rho - Lam / 8 * h2 * open_ * 4 * rho
    R0, R1 = -0.5 * h2 * F, rho * mu
    det = J00 * J11 - J01 * J10
    kappa = (J00 * J11 + abs(J01 * J10)) / abs(det)
    dc, dm = (J11 * R0 - J01 * R1) / det, (J00 * R1 - J10 * R0) / det
    d0, d1 = 8 * U * 0.5 * h2 * size, 2 * U * abs(R1)
    bc = (J11 * d0 + J01 * d1 + 8 * U * (abs(J11 * R0) + J01 * abs(R1))) / abs(det)
    bm = (J00 * d1 + abs(J10) * d0 + 8 * U * (J00 * abs(R1) + abs(J10 * R0))) / abs(det)
    bc += 8 * U * kappa * abs(dc) + 2 * U * abs(1 - dc)
    bm += 8 * U * kappa * abs(dm) + 2 * U * abs(mu - dm)
    j, i = np.meshgrid(np.arange(1, m2 + 1), np.arange(1, m1 + 1), indexing="ij")
    own = (i + j) % 2 == 0
    assert np.all(abs(g["c"].astype(LD) - (1 - dc))[own] <= bc[own])
    assert np.all(abs(g["mu"].astype(LD) - (mu - dm))[own] <= bm[own])


@pytest.mark.parametrize("m2", [32, 64])
def test_rows_of_the_intermediate_velocity(qn, m2):
    """The projection method's momentum rows from rest (no convection) with
    density and viscosity uniform: rho x / dt and the viscous fluxes, away from
    the walls.  The time term takes at most 6 roundings, a viscous flux 8 from its
    difference to the row."""
    m1, a = 1024, (1.0 - 0.01) / 0.01
    s = qn.Solver(m1, m2, periodic_x=True, scheme=1, levels=1, **KW)
    f = resting(m1, m2)
    s.set_fields(f)
    s.begin_step(1.0)
    x, y = np.arange(m1 + 1) / m1, (np.arange(m2) + 0.5) / m1
    f["u"] = np.sin(2 * np.pi * x + 0.3)[None, :] * np.cos(3.0 * y)[:, None]
    f["u"][:, 0] = f["u"][:, m1]
    f["v"][1:-1] = (np.cos(2 * np.pi * (x[1:] - 0.5 / m1) + 0.4)[None, :]
                    * np.sin(3.0 * np.arange(1, m2) / m1 + 0.2)[:, None])
    s.set_iterate(f)
    r, _ = s.residual()
    s.close()
    rho, hv = LD(1.0 / (a + 1.0)), LD(0.1) * LD(m1) ** 2
    u, v = f["u"][:, 1:].astype(LD), f["v"].astype(LD)  # u of edges 1 .. m1

    def row(c, dr, dl, dp, dm, br, bl):
        n = rho * c - hv * ((dr - dl) + (dp - dm) + ((dr + br) - (dl + bl)) / 3)
        size = abs(dr) + abs(dl) + abs(dp) + abs(dm) + (abs(dr) + abs(br) + abs(dl) + abs(bl)) / 3
        return n, U * (6 * rho * abs(c) + 8 * hv * size)

    east, west = np.roll(u, -1, 1), np.roll(u, 1, 1)
    b = v[1:] - v[:-1]  # v across the cells of each row
    i = slice(1, -1)    # rows away from the walls
    n, tol = row(u[i], (east - u)[i], (u - west)[i], u[2:] - u[i], u[i] - u[:-2],
                 np.roll(b, -1, 1)[i], b[i])
    assert np.all(abs(r["u"][i, 1:].astype(LD) + n) <= tol)
    i = slice(2, -2)
    c = v[i]
    b = u - west        # u across the cells of each row
    n, tol = row(c, v[3:-1] - c, c - v[1:-3], (np.roll(v, -1, 1) - v)[i], (v - np.roll(v, 1, 1))[i],
                 b[2:-1], b[1:-2])
    assert np.all(abs(r["v"][i].astype(LD) + n) <= tol)


# --- densities: 1 / (0.5 c + 0.5) for rho1 = 1, rho2 = 2, whose argument rounds
# once wherever it is formed, so the division's result is known to the last bit
# (a reciprocal within 0.51 ulp differs in 3 of 10^4 arguments)
def samples(n):
    c = np.random.default_rng(12).random(n)
    return c, 1.0 / (0.5 * c + 0.5)


def test_density_of_the_rows_is_the_divisions(qn):
    """With no viscosity to speak of, no flow at c^n and u = 1 in the iterate, the
    x row of a uniform grid line is its rho(c).  A denominator of zero gives an
    infinite density, and no other line notices."""
    m2 = 65536
    c, rho = samples(m2)
    s = qn.Solver(4, m2, periodic_x=True, levels=1, rho1=1.0, rho2=2.0, Re=1e300)
    f = s.zeros()
    f["c"][:] = c[:, None]
    s.set_fields(f)
    s.begin_step(1.0)
    f["u"][:] = 1.0
    s.set_iterate(f)
    r, _ = s.residual()
    assert np.array_equal(r["u"][:, 1:], -np.repeat(rho[:, None], 4, axis=1))
    lines = [7, 40000]
    f["c"][lines] = -1.0
    s.set_iterate(f)
    r, _ = s.residual()
    s.close()
    rho[lines] = np.inf
    assert np.array_equal(r["u"][:, 1:], -np.repeat(rho[:, None], 4, axis=1))


def test_density_of_the_mass_is_the_divisions(qn):
    """Eight equal cells, h^2 = 1/16: the mass is rho / 2."""
    c, rho = samples(20000)
    s = qn.Solver(4, 2, periodic_x=True, rho1=1.0, rho2=2.0)
    f, got = s.zeros(), np.empty_like(c)
    for k, x in enumerate(c):
        f["c"][:] = x
        s.set_fields(f)
        got[k] = s.mass()[0]
    s.close()
    assert np.array_equal(got, 0.5 * rho)


def test_density_of_the_allocation_free_mass_is_the_divisions(qn):
    """One cell a call, h = 1: the mass is rho."""
    import torch
    c, rho = samples(20000)
    d = torch.from_numpy(c).cuda()
    out = torch.zeros((c.size, 2), dtype=torch.float64, device="cuda")
    for k in range(c.size):
        qn.mass_noalloc(d[k:k + 1].view(1, 1), 1.0, 1.0, 2.0, out[k])
    torch.cuda.synchronize()
    assert np.array_equal(out[:, 0].cpu().numpy(), rho)


@pytest.mark.parametrize("m1,m2,px", [(737, 5, False), (96, 144, True), (49, 1000, False)])
def test_divergence_is_the_differences_divided_by_h(qn, m1, m2, px):
    s = qn.Solver(m1, m2, periodic_x=px, levels=1)
    rng = np.random.default_rng(3)
    f = {k: rng.standard_normal(v.shape) for k, v in s.zeros().items()}
    f["v"][[0, -1]] = 0.0
    f["u"][:, 0] = f["u"][:, -1] if px else 0.0
    if not px:
        f["u"][:, -1] = 0.0
    s.set_fields(f)
    d = (f["u"][:, 1:] - f["u"][:, :-1]) / s.h + (f["v"][1:] - f["v"][:-1]) / s.h
    assert np.array_equal(s.divergence(), d)
    g = s.diagnostics()
    s.close()
    assert (g["div_max"], g["div_expansion"], g["div_compression"]) == (
        np.max(abs(d)), max(d.max(), 0.0), max((-d).max(), 0.0))


def test_projection_constant_rounds_once(qn):
    """From rest with density 1 and pressures of 0 and 1 in turn, the projected
    velocity is dt / (M h) and nothing else: 1/h, 1/M and 1/dt as they are held,
    their product rounded once."""
    from fractions import Fraction
    rng = np.random.default_rng(8)
    for m1 in range(4, 124, 2):
        dt, M = rng.uniform(1e-4, 1e-3), rng.uniform(0.01, 0.05)
        s = qn.Solver(m1, 2, periodic_x=True, scheme=1, levels=1, M=M)
        f = s.zeros()
        f["c"][:] = 1.0
        s.set_fields(f)
        s.begin_step(dt)
        f["p"][:, 1::2] = 1.0
        s.set_iterate(f)
        s.commit_step()
        u = s.get_fields()["u"][:, 1:]
        k = float(Fraction(1.0 / s.h) * Fraction(1.0 / M) / Fraction(1.0 / dt))
        s.close()
        assert np.array_equal(u, np.where(np.arange(m1) % 2, k, -k) + np.zeros((2, 1))), m1
