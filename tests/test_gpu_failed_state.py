"""A lattice that fails everywhere at once, in every step kernel: the status is reported once and cleared."""
import pytest

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


@pytest.mark.parametrize("shape,kw", [((40, 33, 31), {}), ((40, 33, 31), dict(stencil=1, storage=1)), ((32, 32, 32), dict(storage=3)),
                                      ((40, 32, 32), dict(variant=2)), ((40, 33, 31), dict(variant=1)),
                                      ((64, 64, 1), dict(lattice=0)), ((64, 64, 1), dict(lattice=0, storage=3))])
def test_nan_everywhere(B, shape, kw):
    import torch

    n = shape[0] * shape[1] * shape[2]
    f = torch.full((n,), 0.5, dtype=torch.float64, device="cuda")
    sim = B.Simulation(B.make_params(shape, G=2.5, G_self=(-0.4, 0.0), **kw), f, f)
    good = sim.populations()
    sim.set_populations(torch.full_like(good, float("nan")))
    sim.step(2)
    with pytest.raises(B.ScError) as e:
        sim.sync()
    assert e.value.status == B.SC_ENAN
    sim.sync()  # reported once
    sim.set_populations(good)
    sim.step(2)
    sim.sync()
