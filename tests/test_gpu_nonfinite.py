"""Densities and velocity of a state that holds infinities or NaN: what FP64 sums of its populations give."""
import numpy as np
import pytest

import sc_synth as S

pytestmark = pytest.mark.gpu

INF, NAN = float("inf"), float("nan")


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2112_02574_gb300 import binding

    return binding


@pytest.mark.parametrize("storage", ["F32", "F16", "BF16"])
@pytest.mark.parametrize("lattice", [1, 0])
@pytest.mark.parametrize("values", [(INF,), (-INF,), (INF, -INF), (NAN,), (INF, 1.0, NAN)])
def test_sums_with_infinite_terms(B, storage, lattice, values):
    import torch

    nx, ny, nz = shape = (9, 8, 7 if lattice else 1)
    f0 = S.droplet(shape[::-1], (4, 4, 3), 2.5, n_in=0.85, n_out=0.15, amplitude=1e-2, seed=5)
    sim = B.Simulation(B.make_params(shape, lattice=lattice, storage=getattr(B, f"SC_STORE_{storage}")), *f0)
    sim.step(2)
    raw = sim.state()
    elem = {"F32": torch.float32, "F16": torch.float16, "BF16": torch.bfloat16}[storage]
    n_el = 2 * sim.Q * sim.N
    g = raw[: n_el * (torch.finfo(elem).bits // 8)].view(elem).view(sim.Q, nz, ny, nx, 2)
    # directions 1, 3, 5, ... of component B, from the sites whose populations arrive at (4, 4, z): one density
    cs = [(1, 0, 0), (0, 1, 0), (0, 0, 1)] if lattice else [(1, 0, 0), (0, 1, 0), (1, 1, 0)]
    z = nz // 2
    for k, (v, c) in enumerate(zip(values, cs)):
        g[1 + 2 * k, (z - c[2]) % nz, 4 - c[1], 4 - c[0], 1] = v
    sim.set_state(raw)
    with np.errstate(all="ignore"):
        f = sim.populations().cpu().numpy().reshape(2, sim.Q, nz, ny, nx)
        n = f.sum(1)
        nA, nB, u = (t.cpu().numpy() for t in sim.moments())
        np.testing.assert_allclose(np.stack([nA, nB]).reshape(n.shape), n, rtol=1e-14)
        assert np.isfinite(n).sum() == n.size - 1
        half = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
        if not lattice:
            half = [(1, 0, 0), (0, 1, 0), (1, 1, 0), (1, -1, 0)]
        j = np.zeros((3, nz, ny, nx))
        for i, c in enumerate(half):
            for m in range(3):
                if c[m]:
                    j[m] += c[m] * (f[:, 1 + 2 * i] - f[:, 2 + 2 * i]).sum(0)
        # the force (Eq. sc_force) at zero couplings: the differences across the site times zero
        F = np.zeros_like(j)
        shift = lambda a, c: np.roll(a, (-c[2], -c[1], -c[0]), (0, 1, 2))
        for c in half:
            for m in range(3):
                if c[m]:
                    F[m] += 0.0 * sum(shift(a, c) - shift(a, [-x for x in c]) for a in n)
        ok = np.isfinite(n.sum(0))
        np.testing.assert_allclose(u.reshape(j.shape)[:, ok], ((j + F) / n.sum(0))[:, ok], rtol=1e-12, atol=1e-14)
