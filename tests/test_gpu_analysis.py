"""The analysis kernels at the sizes where their blocking can go wrong: lattices of one site in a direction, bins
shared by a whole warp, one warp's worth of bins and the largest bin count, tables that do not fit, and sums over
fewer and more rows than a block has threads -- against plain NumPy in FP64 on the library's own densities."""
import numpy as np
import pytest

import sc_synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2112_02574_gb300 import binding

    return binding


def run(B, shape, storage="F32", steps=3, **kw):
    f = S.droplet(shape[::-1], tuple(s // 2 for s in shape), min(shape) / 4 + 1, n_in=0.85, n_out=0.15,
                  amplitude=1e-2, seed=11)
    sim = B.Simulation(B.make_params(shape, storage=getattr(B, f"SC_STORE_{storage}"), G=2.5, psi_self=B.SC_PSI_EXP,
                                     **kw), *f)
    sim.step(steps)
    return sim


def shift(a, v):
    return np.roll(a, (-v[2], -v[1], -v[0]), (0, 1, 2))


def tensor(n, G, G_self, stencil):
    """Eq. sm:pt on [z, y, x] fields: {mu, nu} -> field."""
    W = {1: 1 / 6, 2: 1 / 12} if stencil == 0 else {1: 2 / 15, 2: 1 / 15, 3: 1 / 60, 4: 1 / 120}
    r = range(-1, 2) if stencil == 0 else range(-2, 3)
    vs = [(x, y, z) for x in r for y in r for z in r if x * x + y * y + z * z in W]
    psi = [np.exp(-1.0 / a) for a in n]
    P = {}
    for p in range(3):
        for q in range(p, 3):
            C = [sum(W[sum(c * c for c in v)] * v[p] * v[q] * shift(a, v) for v in vs) for a in (*n, *psi)]
            P[p, q] = ((n[0] + n[1]) / 3 if p == q else 0.0) + (
                G * (n[0] * C[1] + n[1] * C[0]) + G_self[0] * psi[0] * C[2] + G_self[1] * psi[1] * C[3]) / 6
    return P


@pytest.mark.parametrize("G_self", [(0.0, 0.0), (-0.4, 0.0), (-0.4, 0.1)])
@pytest.mark.parametrize("stencil", [0, 1])
@pytest.mark.parametrize("shape", [(40, 9, 7), (33, 5, 12), (64, 64, 6)])
def test_profiles(B, shape, stencil, G_self):
    sim = run(B, shape, stencil=stencil, G_self=G_self)
    nx, ny, nz = shape
    n = [a.cpu().numpy().reshape(nz, ny, nx) for a in sim.moments(with_u=False)[:2]]
    P = tensor(n, 2.5, G_self, stencil)
    # FP64 sums of at most N terms of order one: rtol 1e-12
    rows = sim.profile(B.SC_PROFILE_PLANAR_Z, (0.0, 0.0, 0.0), 1.0, nz).cpu().numpy()
    want = np.stack([np.arange(nz), P[2, 2].mean((1, 2)), 0.5 * (P[0, 0] + P[1, 1]).mean((1, 2)), n[0].mean((1, 2)),
                     n[1].mean((1, 2)), np.full(nz, nx * ny)], 1)
    np.testing.assert_allclose(rows, want, rtol=1e-12)
    c = (nx // 2 + 0.25, ny // 2, nz // 2)
    for width, bins in ((0.5, 6), (0.7, 40), (0.125, 4096)):  # a power of two, a quotient, one warp's largest bins
        rows = sim.profile(B.SC_PROFILE_RADIAL, c, width, bins).cpu().numpy()
        d = []
        for m, L in enumerate(shape):
            x = np.arange(L) - c[m]
            x = x - L * np.floor(x / L + 0.5)
            d.append(np.broadcast_to(x.reshape([-1 if 2 - m == k else 1 for k in range(3)]), (nz, ny, nx)))
        r = np.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        e = [np.where(r > 0, x / np.where(r > 0, r, 1.0), 0.0) for x in d]
        PN = sum((2 if p != q else 1) * e[p] * e[q] * P[p, q] for p, q in P)
        tr = P[0, 0] + P[1, 1] + P[2, 2]
        PN = np.where(r > 0, PN, tr / 3)
        PT = np.where(r > 0, 0.5 * (tr - PN), tr / 3)
        b = np.floor(r / width).astype(int).ravel()
        keep = b < bins
        cnt = np.bincount(b[keep], minlength=bins)[:bins]
        np.testing.assert_array_equal(rows[:, 5], cnt)
        for k, v in enumerate((r, PN, PT, *n)):
            s = np.bincount(b[keep], weights=v.ravel()[keep], minlength=bins)[:bins]
            np.testing.assert_allclose(rows[:, k], s / np.maximum(cnt, 1), rtol=1e-11, atol=1e-13)


@pytest.mark.parametrize("storage", ["F32", "F16", "BF16", "F64"])
@pytest.mark.parametrize("shape,lattice", [((20, 13, 17), 1), ((7, 1, 1), 1), ((5, 6, 1), 1), ((37, 29, 1), 0)])
def test_densities_velocity_and_totals(B, storage, shape, lattice):
    G_self = (-0.4, 0.1)
    sim = run(B, shape, storage, lattice=lattice, G_self=G_self, tau=(1.0, 0.9))
    nx, ny, nz = shape
    f = sim.populations().cpu().numpy().reshape(2, -1, nz, ny, nx)  # FP64, component by direction
    nA, nB, u = (t.cpu().numpy() for t in sim.moments())
    cs = np.array([[0, 0, 0]] + [s * np.array(v) for v in
                   (([(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)])
                    if lattice else [(1, 0, 0), (0, 1, 0), (1, 1, 0), (1, -1, 0)]) for s in (1, -1)])
    n = f.sum(1)
    # 19 populations of one rounding each against sums exact to FP64: a few ulp of the density
    np.testing.assert_allclose(np.stack([nA, nB]).reshape(n.shape), n, rtol=1e-14)
    w = {1: 1 / 6, 2: 1 / 12} if lattice else {1: 1 / 3, 2: 1 / 12}
    grad = lambda a: [sum(w[int(c @ c)] * c[m] * shift(a, c) for c in cs[1:]) for m in range(3)]
    psi = np.exp(-1.0 / n)
    F = [[-2.5 / 3 * n[J] * g - G_self[J] / 3 * psi[J] * h for g, h in zip(grad(n[1 - J]), grad(psi[J]))] for J in (0, 1)]
    want = np.stack([(np.einsum("i,jizyx->zyx", cs[:, m].astype(float), f) + 0.5 * (F[0][m] + F[1][m])) / (n[0] + n[1])
                     for m in range(3)])
    np.testing.assert_allclose(u.reshape(want.shape), want, rtol=0, atol=1e-14)
    tot = sim.totals().cpu().numpy()
    np.testing.assert_allclose(tot[:2], n.sum((1, 2, 3)), rtol=1e-13)
    np.testing.assert_allclose(tot[2:], np.einsum("im,jizyx->m", cs.astype(float), f), rtol=0, atol=1e-13 * n.sum())


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("nbins", [2, 31, 256, 257, 600])
def test_surface_of_tension_minimum(B, dim, nbins):
    """Rows with empty bins among them, more and fewer than the kernel's 256 threads, and grids of few and many
    samples: the trapezoid and the grid minimum against NumPy."""
    import torch

    rng = np.random.default_rng(nbins)
    rows = np.zeros((nbins, 6))
    rows[:, 0] = (np.arange(nbins) + 0.3) * 0.5
    rows[:, 2] = 0.3 + 0.02 * np.tanh(rows[:, 0] - nbins / 6) + 1e-3 * rng.standard_normal(nbins)
    rows[:, 5] = rng.integers(0, 3, nbins)
    rows[[0, nbins - 1], 5] = 1
    rows[rows[:, 5] == 0, :5] = 0.0
    pio = np.array([0.36, 0.30])
    full = rows[rows[:, 5] > 0]
    r, pt = full[:, 0], full[:, 2]
    g = r ** (dim - 1) * pt
    C = pio[1] * r[-1] ** dim / dim - np.sum(0.5 * (g[1:] + g[:-1]) * np.diff(r))
    dP = pio[0] - pio[1]
    sig = lambda R: dP * R / dim + C / R ** (dim - 1)
    for lo, hi, step in ((0.01, nbins * 0.5, 0.01), (0.2, 1.0, 0.4), (0.5, 2.0, 1e-4)):
        out = torch.empty(8, dtype=torch.float64, device="cuda")
        B.sc_sigma_minimum(torch.tensor(rows, device="cuda"), torch.tensor(pio, device="cuda"), dim, lo, hi, step, out)
        o = out.cpu().numpy()
        ng = int(np.floor((hi - lo) / step + 0.5)) + 1
        R = lo + step * np.arange(ng)
        k = min(max(int(np.argmin(sig(R))), 1), ng - 2)
        y0, y1, y2 = sig(R[k - 1]), sig(R[k]), sig(R[k + 1])
        off = 0.5 * (y0 - y2) / (y0 - 2 * y1 + y2)
        # sums of up to 600 terms of order r^2: 600 ulp of the largest; the parabola divides differences of
        # neighbouring samples, 1e-16 sigma against their curvature
        scale = np.abs(g).max() * r[-1]
        assert abs(o[1] - C) < 600 * 2.3e-16 * scale
        tol = (1 + abs(off)) * 1e-13 * max(abs(y1), abs(C) / lo ** (dim - 1)) / abs(y0 - 2 * y1 + y2) * step + 600 * 2.3e-16 * scale / abs(C) * hi
        assert abs(o[4] - (R[k] + off * step)) < tol + 1e-12, (o[4], R[k] + off * step)
        np.testing.assert_allclose(o[[0, 6, 7]], [dP, *pio], rtol=1e-15)
