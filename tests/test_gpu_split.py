"""The two-pass step (the library's choice for small, odd, E6 and FP64 lattices with tau = 1) against the
one-pass generic kernel, bit for bit: both compute the same expressions in the same order."""
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


def field(shape, seed):
    c = tuple(s // 2 for s in shape)
    return S.droplet(shape[::-1], c, min(shape) / 4, n_in=0.85, n_out=0.15, amplitude=1e-3, seed=seed)


# the smallest sides, sites short of and just past a block of 128, odd and uneven sides, a staged-size lattice
SHAPES = [(4, 4, 4), (5, 4, 6), (4, 32, 1 * 4), (43, 3 + 1, 7), (33, 17, 9), (64, 12, 10)]


@pytest.mark.parametrize("storage", ["F32", "F16", "BF16", "F64"])
@pytest.mark.parametrize("stencil", ["E4", "E6"])
@pytest.mark.parametrize("G_self", [(0.0, 0.0), (-0.4, 0.1)])
def test_two_passes_equal_one(B, storage, stencil, G_self):
    for k, shape in enumerate(SHAPES):
        kw = dict(stencil=getattr(B, f"SC_FORCE_{stencil}"), psi_self=B.SC_PSI_EXP, G=2.5, G_self=G_self,
                  storage=getattr(B, f"SC_STORE_{storage}"))
        f = field(shape, 900 + k)
        two = B.Simulation(B.make_params(shape, **kw), *f)
        one = B.Simulation(B.make_params(shape, variant=1, **kw), *f)
        assert two.step_config["variant"] == 3 and one.step_config["variant"] == 1
        for n in (3, 34):  # single steps, and a replayed run of 32
            two.step(n)
            one.step(n)
        two.sync()
        one.sync()
        assert two.launches == 37
        np.testing.assert_array_equal(two.state().cpu().numpy(), one.state().cpu().numpy())


def test_one_pass_kernels_keep_what_two_passes_cannot_take(B):
    kw = dict(G=2.5, psi_self=B.SC_PSI_EXP)
    for shape, extra, variant in (((3, 8, 8), {}, 1), ((8, 8, 3), {}, 1), ((16, 16, 16), dict(tau=(1.0, 0.9)), 1),
                                  ((16, 16, 1), dict(lattice=B.SC_D2Q9), 1), ((32, 32, 32), dict(tile_y=8), 2),
                                  ((32, 32, 32), dict(variant=2), 2), ((192, 192, 192), {}, 2)):
        sim = B.Simulation(B.make_params(shape, **kw, **extra), *field(shape, 7))
        assert sim.step_config["variant"] == variant, (shape, extra)
        sim.step(2)
        sim.sync()


@pytest.mark.parametrize("storage", ["F32", "F16", "F64"])
def test_two_pass_batch_members_equal_lone_runs(B, storage):
    st = getattr(B, f"SC_STORE_{storage}")
    ps, fs = [], []
    for k, shape in enumerate([(4, 5, 6), (16, 16, 16), (25, 25, 25), (32, 8, 9)]):
        kw = dict(G=2.5, G_self=(0.0, 0.0) if k % 2 else (-0.4, 0.1), psi_self=B.SC_PSI_EXP, storage=st)
        ps.append((shape, kw))
        fs.append(field(shape, 40 + k))
    batch = B.Batch([B.make_params(s, **kw) for s, kw in ps], fs)
    assert B.sc_batch_variant(batch.handle) == 4
    batch.step(35)
    batch.retire(1)
    batch.step(33)
    for k, ((shape, kw), f) in enumerate(zip(ps, fs)):
        lone = B.Simulation(B.make_params(shape, variant=1, **kw), *f)
        lone.step(35 if k == 1 else 68)
        batch.members[k].sync()
        np.testing.assert_array_equal(batch.members[k].state().cpu().numpy(), lone.state().cpu().numpy())


def test_two_pass_batch_takes_the_staged_launch_forms_when_asked(B):
    shapes = [(32, 32, 32), (40, 16, 12)]
    fs = [field(s, 60 + k) for k, s in enumerate(shapes)]
    ps = [B.make_params(s, G=2.5, psi_self=B.SC_PSI_EXP) for s in shapes]
    batch = B.Batch(ps, fs)
    ref = B.Batch(ps, fs)
    batch.persistent = False  # no persistent launch in use: nothing changes
    assert B.sc_batch_variant(batch.handle) == 4
    batch.step(33)
    batch.persistent = True
    assert B.sc_batch_variant(batch.handle) == 3 and batch.staged
    batch.step(33)
    batch.persistent = False
    assert B.sc_batch_variant(batch.handle) == 2
    batch.step(2)
    ref.step(68)
    for a, b in zip(batch.members, ref.members):
        np.testing.assert_array_equal(a.state().cpu().numpy(), b.state().cpu().numpy())


def test_two_pass_batch_groups(B):
    """Members above the group size step alone, the others in groups; a retired member changes the groups."""
    shapes = [(96, 96, 96), (20, 12, 10), (92, 92, 92), (97, 91, 90), (31, 31, 31)]
    fs = [field(s, 80 + k) for k, s in enumerate(shapes)]
    kw = dict(G=2.5, G_self=(-0.4, 0.0), psi_self=B.SC_PSI_EXP)
    batch = B.Batch([B.make_params(s, **kw) for s in shapes], fs)
    batch.step(33)
    batch.retire(0)
    batch.step(32)
    for k, (s, f) in enumerate(zip(shapes, fs)):
        lone = B.Simulation(B.make_params(s, variant=1, **kw), *f)
        lone.step(33 if k == 0 else 65)
        np.testing.assert_array_equal(batch.members[k].state().cpu().numpy(), lone.state().cpu().numpy())


@pytest.mark.parametrize("tau", [(1.0, 1.0), (1.0, 0.9)])
@pytest.mark.parametrize("psi,G_self", [("N", (0.0, 0.0)), ("EXP", (-0.4, 0.1)), ("EXP", (0.0, -0.3))])
def test_d2q9_fp64_thread_per_component_equals_tiles(B, tau, psi, G_self):
    """The small-lattice D2Q9 FP64 kernel (tiles of 32 x 1) against the tiled one, bit for bit: partial tiles, one
    row, one column, and both sides of the size rule (304 blocks)."""
    kw = dict(lattice=B.SC_D2Q9, psi_self=getattr(B, f"SC_PSI_{psi}"), storage=B.SC_STORE_F64, G=2.5, G_self=G_self, tau=tau)
    for k, (nx, ny) in enumerate([(64, 64), (31, 7), (33, 1), (1, 40), (65, 101), (32, 304), (32, 305)]):
        f = S.droplet((1, ny, nx), (nx // 2, ny // 2, 0), min(nx, ny) / 4 + 1, n_in=0.85, n_out=0.15, amplitude=1e-3, seed=k)
        a = B.Simulation(B.make_params((nx, ny, 1), **kw), *f)
        b = B.Simulation(B.make_params((nx, ny, 1), tile_y=4, **kw), *f)
        assert a.step_config["tile_y"] == (1 if (nx + 31) // 32 * ny <= 304 else 4)
        for n in (3, 34):
            a.step(n)
            b.step(n)
        a.sync()
        b.sync()
        np.testing.assert_array_equal(a.state().cpu().numpy(), b.state().cpu().numpy())
