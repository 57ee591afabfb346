"""D2Q9 lattices on both sides of the size above which tau = 1 steps are plain launches with read-only loads: the stored
bits are those of the batched kernel, which every size shares."""
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


@pytest.mark.parametrize("storage,side", [("F32", 424), ("F32", 425), ("BF16", 424), ("BF16", 425), ("F16", 894),
                                          ("F16", 895)])
def test_lone_equals_batched(B, storage, side):
    import torch

    gen = torch.Generator(device="cuda")
    gen.manual_seed(side)
    a = 0.3 + 0.4 * torch.rand(side * side, generator=gen, dtype=torch.float64, device="cuda")
    p = B.make_params((side, side, 1), lattice=B.SC_D2Q9, G=2.5, G_self=(-0.4, 0.1), storage=getattr(B, f"SC_STORE_{storage}"))
    lone, batch = B.Simulation(p, a, 1.0 - a), B.Batch([p], [(a, 1.0 - a)])
    lone.step(37)  # single steps and a replayed run
    batch.step(37)
    assert torch.equal(lone.state(), batch.members[0].state())
