"""Steps recorded into a caller's CUDA graph: replays advance the state as eager steps do, and what is read after a
replay is the state it left.  (Runs of 32 steps are graph launches of the library's own, which a capture refuses.)"""
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


def field(shape):
    return S.droplet(shape[::-1], tuple(s // 2 for s in shape), min(s for s in shape if s > 1) / 4, n_in=0.85, n_out=0.15,
                     amplitude=1e-3, seed=3)


CASES = [((24, 20, 18), dict(G_self=(-0.4, 0.1)), 3), ((24, 20, 18), dict(stencil=1, storage=1), 3),
         ((40, 33, 1), dict(lattice=0), 1), ((40, 33, 1), dict(lattice=0, storage=3), 4), ((32, 16, 16), dict(variant=2), 2)]


@pytest.mark.parametrize("shape,kw,variant", CASES)
def test_replayed_steps(B, shape, kw, variant, nsteps=2):
    import torch

    stream = torch.cuda.Stream()
    p, f = B.make_params(shape, G=2.5, **kw), field(shape)
    sim = B.Simulation(p, *f, stream=stream)
    assert sim.step_config["variant"] == variant
    sim.step(34)  # in step with the eager runs
    sim.sync()
    nA, nB = (torch.empty(sim.N, dtype=torch.float64, device="cuda") for _ in range(2))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        sim.step(nsteps)
    eager = B.Simulation(p, *f)
    eager.step(34)
    for _ in range(3):
        with torch.cuda.stream(stream):
            graph.replay()
        B.sc_moments(sim.ctx, nA, nB, None)
        sim.sync()
        eager.step(nsteps)
        want = eager.moments(with_u=False)
        eager.sync()
        np.testing.assert_array_equal(nA.cpu().numpy(), want[0].cpu().numpy())
        np.testing.assert_array_equal(nB.cpu().numpy(), want[1].cpu().numpy())
        np.testing.assert_array_equal(sim.state().cpu().numpy(), eager.state().cpu().numpy())


def test_replayed_batch_steps(B):
    import torch

    stream = torch.cuda.Stream()
    shapes = [(24, 20, 18), (97, 96, 95)]
    make = lambda **kw: B.Batch([B.make_params(s, G=2.5, G_self=(-0.4, 0.0)) for s in shapes], [field(s) for s in shapes], **kw)
    batch, eager = make(stream=stream), make()
    batch.step(2)
    eager.step(2)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        batch.step(2)
    for _ in range(2):
        with torch.cuda.stream(stream):
            graph.replay()
        eager.step(2)
        torch.cuda.synchronize()
        for a, b in zip(batch.members, eager.members):
            for x, y in zip(a.moments(with_u=False)[:2], b.moments(with_u=False)[:2]):
                torch.cuda.synchronize()
                assert torch.equal(x, y)
