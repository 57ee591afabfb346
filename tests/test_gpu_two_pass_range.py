"""The two-pass step over the rest of its default range, bit for bit against the one-pass generic kernel: moments that
do not stay in L2, self couplings above the small-lattice register budget, psi = n, byte offsets beyond 2^31, and
batches with the extended stencil or in BF16."""
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


def densities(shape, seed):
    import torch

    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n = shape[0] * shape[1] * shape[2]
    a = 0.3 + 0.4 * torch.rand(n, generator=gen, dtype=torch.float64, device="cuda")
    return a, 1.0 - a


def final_state(B, shape, steps, seed, want, **kw):
    sim = B.Simulation(B.make_params(shape, G=2.5, **kw), *densities(shape, seed))
    assert sim.step_config["variant"] == want
    sim.step(steps)
    out = sim.state()
    sim.sync()
    return out


@pytest.mark.parametrize("shape,storage,kw", [
    # more moments than the 140 MiB that are kept in L2
    ((192, 192, 192), "F16", {}),
    ((192, 192, 192), "BF16", {}),
    ((177, 176, 175), "F32", dict(G_self=(-0.4, 0.1))),
    ((176, 176, 176), "F16", dict(G_self=(0.0, -0.3))),
    ((168, 168, 168), "F32", dict(stencil=1)),
    ((136, 136, 136), "F64", {}),
    # a self coupling on more than 300 000 sites, whose moments are kept
    ((64, 64, 256), "F32", dict(stencil=1, G_self=(-0.4, 0.0))),
    ((64, 64, 256), "F16", dict(stencil=1, G_self=(-0.4, 0.0))),
    ((64, 64, 256), "BF16", dict(stencil=1, G_self=(-0.4, 0.0))),
    ((97, 65, 101), "F32", dict(G_self=(-0.4, 0.1))),
    # both sides of 300 000 sites
    ((100, 60, 50), "F32", dict(G_self=(-0.4, 0.1))),
    ((100, 61, 50), "F32", dict(G_self=(-0.4, 0.1))),
    # psi = n
    ((64, 48, 40), "F32", dict(G_self=(-0.3, 0.2), psi_self=0)),
    ((33, 32, 31), "F16", dict(G_self=(-0.3, 0.0), psi_self=0, stencil=1)),
    ((33, 32, 31), "F64", dict(G_self=(-0.3, 0.2), psi_self=0)),
    # 16 bytes a site of densities and psi: offsets pass 2^31
    ((512, 512, 516), "BF16", dict(G_self=(-0.4, 0.1))),
])
def test_two_passes_equal_one(B, shape, storage, kw):
    import torch

    kw = dict(kw, storage=getattr(B, f"SC_STORE_{storage}"))
    two = final_state(B, shape, 3, 17, 3, **kw)
    one = final_state(B, shape, 3, 17, 1, variant=1, **kw)
    assert torch.equal(two, one)


@pytest.mark.parametrize("storage,stencil,psi", [("F32", 1, 1), ("F16", 1, 1), ("BF16", 1, 0), ("F64", 1, 1), ("BF16", 0, 1)])
def test_batches(B, storage, stencil, psi):
    import torch

    shapes = [(4, 5, 6), (25, 25, 25), (97, 96, 95), (32, 8, 9), (64, 64, 40)]
    kws = [dict(storage=getattr(B, f"SC_STORE_{storage}"), stencil=stencil, psi_self=psi,
                G_self=(0.0, 0.0) if k == 3 else (-0.4, 0.1 * k)) for k in range(len(shapes))]
    batch = B.Batch([B.make_params(s, G=2.5, **kw) for s, kw in zip(shapes, kws)],
                    [densities(s, 70 + k) for k, s in enumerate(shapes)])
    assert B.sc_batch_variant(batch.handle) == 4
    batch.step(34)  # a replayed run and two single steps
    for k, (s, kw) in enumerate(zip(shapes, kws)):
        assert torch.equal(batch.members[k].state(), final_state(B, s, 34, 70 + k, 1, variant=1, **kw)), s
