"""The FP64 hexahedron kernels' fixed-point line operators (csrc/fr_hexfx.cuh)
where numbers of very different size meet in an element: stretched elements,
whose metric terms differ by the aspect ratio, and fields that span many powers
of two.  The reference is the 50-digit right-hand side of brute_mp.

Tolerance, per point and variable: FP64 rounds every operation of the chain
traces -> (gradients -> their traces) -> fluxes -> transformed flux -> jumps ->
divergence, about 60 of them along the longest path (a sum of N + 2 <= 7 terms
at four places, 10 operations in each flux, 3 in each metric product, the
interface flux and the scaling by 1/J), each by at most 2^-53 of the magnitudes
that enter it.  ``_magnitudes`` carries those magnitudes (the same chain on
absolute values, nothing cancelling) to the result: B.  Independent roundings
then add up to about sqrt(60) 2^-53 B; the bound is twice that, 16 * 2^-53 B.
"""
import numpy as np
import pytest

import paper_2408_16509_gb300 as fr
from oracle.fr import FRSystem
from oracle.mesh import FRMesh as OracleMesh

pytestmark = pytest.mark.gpu
GAMMA, MU, PR = 1.4, 0.05, 0.71


@pytest.fixture(scope="module", autouse=True)
def built():
    fr.build()


def _magnitudes(o, u, ns):
    """B [ne][nu][5]: the right-hand side's chain on absolute values."""
    m, t = o.m, "hex"
    el = m.el[t]
    M0, D, L, S = (np.abs(a) for a in (el.M0, el.D, el.LIFT, m.S_u[t]))
    nrm, J = np.abs(el.fpts_norm), m.detJ[t]

    def physics(ua, ut):
        """Magnitudes of pressure and Euler flux (..., 3, 5) from those of
        the state, ua; divisors are the true values, ut."""
        r = ut[..., 0]
        amp = ua[..., 0] / r  # the density's own rounding, by which all scale
        p = (GAMMA - 1) * (ua[..., 4] + 0.5 * (ua[..., 1:4] ** 2).sum(-1) / r) * amp
        v = ua[..., 1:4] / r[..., None] * amp[..., None]
        F = v[..., :, None] * ua[..., None, :]
        F[..., 4] += v * p[..., None]
        for j in range(3):
            F[..., j, 1 + j] += p
        return p, v, F

    def viscous(ua, ut, g):
        r = ut[..., 0]
        _, v, _ = physics(ua, ut)
        d = (g[..., 1:4] + g[..., :1] * v[..., None, :]) / r[..., None, None]
        e = ua[..., 4] / r
        ge = (g[..., 4] + g[..., 0] * e[..., None]) / r[..., None] + (d * v[..., None, :]).sum(-1)
        tau = MU * (d + np.swapaxes(d, -1, -2)
                    + (2 / 3) * np.trace(d, axis1=-2, axis2=-1)[..., None, None] * np.eye(3))
        F = np.zeros_like(g)
        F[..., 1:4] = tau
        F[..., 4] = (tau * v[..., None, :]).sum(-1) + MU * GAMMA / PR * ge
        return F

    if m.family == "gll":  # (traces are solution points)
        M0 = np.where(M0 > 0.5, 1.0, 0.0)
        uf = np.einsum("fz,ezv->efv", M0, u)
    else:
        uf = np.einsum("fz,ezv->efv", el.M0, u)
    ua, ufa = np.abs(u), np.einsum("fz,ezv->efv", M0, np.abs(u))
    flat = [a.reshape(-1, 5) for a in (uf, ufa)]
    other = np.empty(len(flat[0]), int)
    other[m.pair_l], other[m.pair_r] = m.pair_r, m.pair_l
    xf, xfa = (a[other].reshape(uf.shape) for a in flat)
    # jumps: of rounded sums, or of stored values
    jump = np.abs(xf - uf) if m.family == "gll" else ufa + xfa
    _, _, F = physics(ua, u)
    pl, vl, Fl = physics(ufa, uf)
    px, vx, Fx = physics(xfa, xf)
    n = np.abs(m.fn_all).reshape(*uf.shape[:2], 3)
    mag = m.fm_all.reshape(uf.shape[:2])

    def wave(ua_, ut, p, v):
        pt = (GAMMA - 1) * (ut[..., 4] - 0.5 * (ut[..., 1:4] ** 2).sum(-1) / ut[..., 0])
        c = np.sqrt(GAMMA * pt / ut[..., 0])
        return (v * n).sum(-1) + c * (1 + p / pt + ua_[..., 0] / ut[..., 0])
    lam = np.maximum(wave(ufa, uf, pl, vl), wave(xfa, xf, px, vx))
    fc = 0.5 * ((Fl + Fx) * n[..., None]).sum(-2) + 0.5 * lam[..., None] * jump
    if ns:
        du = 0.5 * jump
        gr = np.stack([np.einsum("zv,evk->ezk", D[d], ua)
                       + np.einsum("zf,efk->ezk", L, nrm[None, :, d, None] * du)
                       for d in range(3)], axis=2)
        g = np.einsum("ezij,ezik->ezjk", S, gr) / J[..., None, None]
        gf = np.einsum("fz,ezjk->efjk", M0, g)
        gx = gf.reshape(-1, 3, 5)[other].reshape(gf.shape)
        F = F + viscous(ua, u, g)
        fv = viscous(ufa, uf, gf) + viscous(xfa, xf, gx)
        fc = fc + 0.5 * (fv * n[..., None]).sum(-2)
    ft = np.einsum("ezij,ezjk->ezik", S, F)
    fn = np.einsum("fd,fz,ezdk->efk", nrm, M0, ft)
    div = sum(np.einsum("zv,evk->ezk", D[d], ft[:, :, d]) for d in range(3))
    div = div + np.einsum("zf,efk->ezk", L, mag[..., None] * fc + fn)
    return div / J[..., None]


def _rotation():
    q, _ = np.linalg.qr(np.random.default_rng(5).normal(size=(3, 3)))
    return q * np.sign(np.linalg.det(q))


def _worst(p, family, physics, A, n, u):
    """Largest error of the library's right-hand side in units of 2^-53 B."""
    from brute_mp import BruteFR, spec_for  # needs mpmath
    spec = spec_for(A, n)
    g = fr.FRMesh(spec, p, physics=physics, mu=MU, prandtl=PR, family=family)
    g.set_variant("sumfact")
    g.set_solution({"hex": u})
    got = g.rhs()["hex"]
    N = p + 1

    def key(e, z):
        return ((e % n[0], e // n[0] % n[1], e // (n[0] * n[1])),
                z % N, z // N % N, z // (N * N))
    brute = BruteFR(p, A, n, gamma=GAMMA, mu=MU, pr=PR, dps=40, family=family)
    ref = brute.rhs({key(e, z): u[e, z] for e in range(len(u)) for z in range(N ** 3)}, physics)
    # the difference is taken at 40 digits: only its size matters afterwards
    err = np.array([[[float(ref[key(e, z)][k] - float(got[e, z, k])) for k in range(5)]
                     for z in range(N ** 3)] for e in range(len(u))])
    o = FRSystem(OracleMesh(spec, p, family=family), physics, gamma=GAMMA, mu=MU, pr=PR)
    B = _magnitudes(o, u, physics == "ns")
    return float((np.abs(err) / (2.0 ** -53 * np.maximum(B, 1e-300))).max())


def _line(p, family):
    from brute_mp import gauss_points, lobatto_points
    return np.array([float(x) for x in (lobatto_points if family == "gll"
                                        else gauss_points)(p + 1)])


def _sheet(p, family, n, R):
    """Smooth flow within the planes of a sheet of elements: nothing varies or
    moves across it."""
    x = _line(p, family)
    N = p + 1
    ne = n[0] * n[1] * n[2]
    e = np.arange(ne)[:, None]
    z = np.arange(N ** 3)[None, :]
    X = np.pi * (2 * (e % n[0]) + 1 + x[z % N]) / n[0]
    Y = np.pi * (2 * (e // n[0] % n[1]) + 1 + x[z // N % N]) / n[1]
    rho = 1.0 + 0.2 * np.sin(X + 0.3) * np.cos(Y)
    v = np.stack([0.4 + 0.3 * np.sin(Y), 0.3 * np.cos(X + 0.5) - 0.2, 0 * X], axis=-1) @ R.T
    pr = 1.0 + 0.1 * np.cos(X - Y)
    E = pr / (GAMMA - 1) + 0.5 * rho * (v ** 2).sum(-1)
    return np.concatenate([rho[..., None], rho[..., None] * v, E[..., None]], axis=-1)


@pytest.mark.parametrize("p", [2, 3, 4])
@pytest.mark.parametrize("family", ["gl", "gll"])
@pytest.mark.parametrize("physics", ["euler", "ns"])
@pytest.mark.parametrize("aspect", [1.0, 1e2, 1e4])
@pytest.mark.parametrize("rotated", [False, True])
def test_stretched_elements(p, family, physics, aspect, rotated):
    pytest.importorskip("mpmath")
    R = _rotation() if rotated else np.eye(3)
    n = (2, 2, 1)
    A = R @ np.diag([1.0, 1.0, 1.0 / aspect])
    assert _worst(p, family, physics, A, n, _sheet(p, family, n, R)) < 16.0


@pytest.mark.parametrize("p", [2, 3, 4])
@pytest.mark.parametrize("physics", ["euler", "ns"])
@pytest.mark.parametrize("bits", [8, 20])
def test_range_within_an_element(p, physics, bits):
    # density and pressure fall by 2^bits from one end of an element to the
    # other (Gauss-Lobatto points: the faces' values are solution points)
    pytest.importorskip("mpmath")
    n, N = (2, 1, 1), p + 1
    x = _line(p, "gll")
    e = np.arange(2)[:, None]
    z = np.arange(N ** 3)[None, :]
    s = x[z % N] * np.where(e == 0, 1.0, -1.0)
    w = 2.0 ** (-0.5 * bits * (1.0 + s))
    rng = np.random.default_rng(p)
    rho = w * (1.0 + 0.1 * rng.uniform(-1, 1, w.shape))
    v = 0.3 * rng.uniform(-1, 1, (*w.shape, 3))
    E = w / (GAMMA - 1) + 0.5 * rho * (v ** 2).sum(-1)
    u = np.concatenate([rho[..., None], rho[..., None] * v, E[..., None]], axis=-1)
    assert _worst(p, "gll", physics, np.diag([0.5, 0.6, 0.7]), n, u) < 16.0


@pytest.mark.parametrize("p", [2, 3, 4])
def test_gauss_lobatto_traces_are_the_end_points(p):
    # the traces that the volume kernel leaves for the next step are the
    # solution's end points bit for bit: a step from them equals a step from
    # traces formed anew
    rng = np.random.default_rng(11)
    n, N = (3, 2, 2), p + 1
    rho = np.exp2(rng.uniform(-4, 4, (12, N ** 3)))
    v = rng.normal(size=(12, N ** 3, 3))
    E = rho / (GAMMA - 1) + 0.5 * rho * (v ** 2).sum(-1)
    u = np.concatenate([rho[..., None], rho[..., None] * v, E[..., None]], axis=-1)
    from frinputs import box_hex
    g = fr.FRMesh(box_hex(n, perturb=0.1), p, physics="ns", mu=0.01, prandtl=PR, family="gll")
    g.set_variant("sumfact")
    g.set_solution({"hex": u})
    g.rk_step("rk4", 1e-6, 1)
    mid = g.get_solution()
    g.rk_step("rk4", 1e-6, 1)
    on = g.get_solution()["hex"]
    g.set_solution(mid)
    g.rk_step("rk4", 1e-6, 1)
    assert np.array_equal(on, g.get_solution()["hex"])
