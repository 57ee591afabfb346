"""The sigma[R] grid search where the minimum lies inside the grid (rows of a droplet: P_T dips at the interface, so
C > 0), with every output checked: coarse and fine grids, samples tied to the last bits, pressures outside the range
of the FP32 screen, and an all-zero sigma."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.3e-16


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2112_02574_gb300 import binding

    return binding


def droplet(dim, nbins, scale):
    """Rows (some of them empty) and pressures; the FP64 dP, C and the error C may have (600 ulp of its two parts)."""
    rng = np.random.default_rng(nbins)
    r = (np.arange(nbins) + 0.3) * 0.5
    R0, pio = r[-1] / 2, scale * np.array([0.36, 0.30])
    rows = np.zeros((nbins, 6))
    rows[:, 0] = r
    rows[:, 2] = pio[1] - scale * 0.02 * np.exp(-((r - R0) / 2) ** 2) * (1 + 0.1 * rng.random(nbins))
    rows[:, 5] = rng.integers(0, 4, nbins)
    rows[[0, nbins // 2, nbins - 1], 5] = 1
    rows[rows[:, 5] == 0, :5] = 0.0
    full = rows[rows[:, 5] > 0]
    x, g = full[:, 0], full[:, 0] ** (dim - 1) * full[:, 2]
    out = pio[1] * x[-1] ** dim / dim
    C = out - np.sum(0.5 * (g[1:] + g[:-1]) * np.diff(x))
    return rows, pio, pio[0] - pio[1], C, 600 * EPS * abs(out)


def search(B, rows, pio, dim, lo, hi, step):
    import torch

    out = torch.empty(8, dtype=torch.float64, device="cuda")
    B.sc_sigma_minimum(torch.tensor(rows, device="cuda"), torch.tensor(pio, device="cuda"), dim, lo, hi, step, out)
    return out.cpu().numpy()


# scales of 1e+-30 leave the FP32 screen's range: every sample in FP64
@pytest.mark.parametrize("scale", [1.0, 1e30, 1e-30])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("nbins", [40, 256, 600])
def test_interior_minimum(B, dim, nbins, scale):
    rows, pio, dP, C, dC = droplet(dim, nbins, scale)
    Rs = (6 * C / dP) ** (1 / 3) if dim == 3 else (2 * C / dP) ** 0.5
    assert C > 0 and 2.0 < Rs < 0.5 * nbins - 2.0
    sig = lambda R: dP * R / dim + C / R ** (dim - 1)
    fine = max(1.0, Rs / 8)
    for lo, hi, step in ((0.01, 0.5 * nbins, 0.01), (Rs - fine, Rs + fine, 2e-4), (Rs / 2, 2 * Rs, 1.5 * Rs / 300000),
                         (0.37, 0.5 * nbins, 0.173)):
        o = search(B, rows, pio, dim, lo, hi, step)
        ng = int(np.floor((hi - lo) / step + 0.5)) + 1
        R = lo + step * np.arange(ng)
        k = int(np.argmin(sig(R)))
        assert 10 < k < ng - 10 or step == 0.173 and 3 < k < ng - 4
        y0, y1, y2 = sig(R[k - 1]), sig(R[k]), sig(R[k + 1])
        den = y0 - 2 * y1 + y2
        Rg = R[k] + 0.5 * (y0 - y2) / den * step
        # a sample is good to 4 ulp; the vertex moves by its error over the curvature, with C, and, where the search
        # takes the other of two samples tied to that error, by the cubic term of sigma
        tol = 4 * (4 * EPS * y1) / abs(den) * step + Rs * dC / C + 4 * step**2 / Rs
        assert abs(o[4] - Rg) < tol, (lo, hi, step, o[4], Rg, tol)
        best = sig(Rs)
        # sigma at the vertex: 4 ulp, the error of C, and the parabola against sigma (fourth order in step / R)
        assert abs(o[5] - best) < 16 * EPS * best + 4 * dC / Rs ** (dim - 1) + best * (step / Rs) ** 3
        assert abs(o[1] - C) < dC
        np.testing.assert_allclose(o[[0, 6, 7]], [dP, *pio], rtol=1e-15)
        np.testing.assert_allclose(o[2], Rs, rtol=dC / C + 1e-14)
        np.testing.assert_allclose(o[3], dP * Rs / (2 if dim == 3 else 1), rtol=dC / C + 1e-14)


@pytest.mark.parametrize("dim", [2, 3])
def test_samples_tied_to_the_last_bits(B, dim):
    """10 000 samples within 5e-6 of the minimum, whose sigma differ in the last bits only: any of them may win."""
    rows, pio, dP, C, dC = droplet(dim, 256, 1.0)
    o = search(B, rows, pio, dim, 1.0, 100.0, 0.01)
    Rs = o[2]
    best = dP * Rs / dim + o[1] / Rs ** (dim - 1)
    t = search(B, rows, pio, dim, Rs - 5e-6, Rs + 5e-6, 1e-9)
    assert abs(t[4] - Rs) < 2e-5
    assert abs(t[5] - best) < 16 * EPS * best


@pytest.mark.parametrize("dim", [2, 3])
def test_exact_ties_take_the_lowest_sample(B, dim):
    """sigma = 0 everywhere: sample 0, moved to 1 for the parabola, which has no curvature."""
    rows = np.zeros((50, 6))
    rows[:, 0] = np.arange(50) * 0.5
    rows[:, 5] = 1
    for ng in (3, 40, 1000):
        o = search(B, rows, np.zeros(2), dim, 1.0, 1.0 + 0.125 * (ng - 1), 0.125)
        np.testing.assert_array_equal(o[[0, 1, 4, 5]], [0.0, 0.0, 1.125, 0.0])
