"""Host logic of contexts and batches when a CUDA call fails, on a fake runtime (no GPU): what stays valid after the
error, and which launches follow."""
import ctypes

import pytest

import fake_gpu


@pytest.fixture(scope="module")
def B():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2112_02574_gb300 import binding

    return binding


@pytest.fixture(scope="module")
def lib(B, tmp_path_factory):
    return fake_gpu.load(B, str(tmp_path_factory.mktemp("fake")))


@pytest.fixture
def L(lib):
    lib.fake_reset()
    yield lib
    lib.fake_reset()


def fields_computed(L):
    return sum("fields_kernel" in c for c in fake_gpu.calls(L))


def test_two_pass_step_that_fails_half_way_leaves_no_fields_behind(B, L):
    """The moments overwrite the space of the cached fields: after a step whose collision launch fails, the fields are
    computed again from the (unchanged) populations."""
    c = fake_gpu.Context(L, B.make_params((16, 16, 16), G=2.5))
    assert c.status == B.SC_OK and c.moments() == B.SC_OK
    L.fake_reset()
    assert c.moments() == B.SC_OK and fields_computed(L) == 0  # cached
    L.fake_fail(b"kernel", 1)  # the moments are launched, the collision is not
    assert L.sc_step(c.ctx, 1) == B.SC_ECUDA
    assert ["moments" in n for n in fake_gpu.calls(L)] == [True]
    assert L.sc_kernel_launches(c.ctx) == 0
    assert c.moments() == B.SC_OK and fields_computed(L) == 1


def test_batch_step_that_fails_is_not_counted(B, L):
    """A step that fails between the groups of a two-pass batch is not counted, and run again from the same buffers (a
    step reads one buffer and writes the other); no member's fields are taken from before it."""
    b = fake_gpu.Batch(L, [B.make_params((96, 96, 96), G=2.5), B.make_params((16, 16, 16), G=2.5)])
    assert b.status == B.SC_OK and L.sc_batch_variant(b.handle) == 4
    m = [b.member(k) for k in range(2)]
    keep, out = fake_gpu.buffer(16 * 96**3)
    for x in m:
        assert L.sc_moments(x, out, out, None) == B.SC_OK
    L.fake_reset()
    L.fake_fail(b"kernel", 5)  # one step (two groups of two launches), then the second's first group only
    assert L.sc_batch_step(b.handle, 3) == B.SC_ECUDA
    assert L.sc_batch_launches(b.handle) == 1
    assert [L.sc_kernel_launches(x) for x in m] == [1, 1]
    before = fields_computed(L)
    for x in m:
        assert L.sc_moments(x, out, out, None) == B.SC_OK
    assert fields_computed(L) == before + 2
    assert L.sc_batch_step(b.handle, 2) == B.SC_OK
    assert L.sc_batch_launches(b.handle) == 3
    assert [L.sc_kernel_launches(x) for x in m] == [3, 3]


def test_batch_run_that_fails_is_not_counted(B, L):
    b = fake_gpu.Batch(L, [B.make_params((16, 16, 16), G=2.5)])
    L.fake_fail(b"cudaGraphLaunch", 1)
    assert L.sc_batch_step(b.handle, 96) == B.SC_ECUDA
    assert L.sc_batch_launches(b.handle) == 32
    assert L.sc_kernel_launches(b.member(0)) == 32


def test_two_pass_batch_without_a_graph_steps_with_plain_launches(B, L):
    """Where the capture of a run fails, creating the batch and retiring a member succeed and whole runs go out as
    plain launches (two per group and step), as a lone context's do."""
    params = [B.make_params((16, 16, 16), G=2.5), B.make_params((96, 96, 96), G=2.5)]
    for call in (b"cudaStreamCreateWithFlags", b"cudaStreamBeginCapture", b"kernel", b"cudaGraphInstantiate"):
        L.fake_reset()
        whole = fake_gpu.Batch(L, params)
        assert whole.status == B.SC_OK
        L.fake_fail(call, 0)
        assert L.sc_batch_retire(whole.handle, 0) == B.SC_OK
        L.fake_reset()
        assert L.sc_batch_step(whole.handle, 34) == B.SC_OK
        assert len(fake_gpu.calls(L)) == 2 * 34 and "graph launch" not in fake_gpu.calls(L)
        assert L.sc_batch_launches(whole.handle) == 34
        L.sc_batch_destroy(whole.handle)
    for call in (b"cudaStreamCreateWithFlags", b"cudaGraphInstantiate"):
        L.fake_reset()
        L.fake_fail(call, 0)
        b = fake_gpu.Batch(L, params)
        assert b.status == B.SC_OK and L.sc_batch_variant(b.handle) == 4
        L.fake_reset()
        assert L.sc_batch_step(b.handle, 32) == B.SC_OK
        assert len(fake_gpu.calls(L)) == 4 * 32


def test_failed_persistent_build_keeps_the_two_passes(B, L):
    """SC_EUNSUPPORTED leaves the batch as it was; the form changes when the persistent launch has been built."""
    b = fake_gpu.Batch(L, [B.make_params((32, 32, 32), G=2.5), B.make_params((40, 16, 12), G=2.5)])
    assert b.status == B.SC_OK and L.sc_batch_variant(b.handle) == 4
    L.fake_fail(b"cudaGraphInstantiate", 0)
    assert L.sc_batch_set_persistent(b.handle, 1) == B.SC_EUNSUPPORTED
    assert b"persistent" in L.sc_last_error()
    assert L.sc_batch_variant(b.handle) == 4
    L.fake_reset()
    assert L.sc_batch_step(b.handle, 33) == B.SC_OK
    assert [("split" in c) for c in fake_gpu.calls(L)] == [False, True, True]  # a replayed run, then one step
    assert L.sc_batch_set_persistent(b.handle, 1) == B.SC_OK and L.sc_batch_variant(b.handle) == 3
    # from here on the batch is a staged one: without the persistent launch it takes one launch per step
    assert L.sc_batch_set_persistent(b.handle, 0) == B.SC_OK and L.sc_batch_variant(b.handle) == 2


def test_fields_after_a_captured_step_are_computed_anew(B, L):
    """A step recorded into a caller's graph runs again at every replay, which the library does not see: the fields it
    leaves (the moments are in their space) are never taken for the cached ones."""
    c = fake_gpu.Context(L, B.make_params((16, 16, 16), G=2.5))
    L.fake_capturing(1)
    assert L.sc_step(c.ctx, 2) == B.SC_OK
    L.fake_capturing(0)
    for k in range(3):  # with a replay before each
        L.fake_reset()
        assert c.moments() == B.SC_OK and fields_computed(L) == 1, k
    b = fake_gpu.Batch(L, [B.make_params((16, 16, 16), G=2.5)])
    out = fake_gpu.buffer(32 * 16**3)
    L.fake_capturing(1)
    assert L.sc_batch_step(b.handle, 2) == B.SC_OK
    L.fake_capturing(0)
    for k in range(2):
        L.fake_reset()
        assert L.sc_moments(b.member(0), out[1], out[1], None) == B.SC_OK and fields_computed(L) == 1, k


# bytes a site that the moments of the two-pass step need beyond the space of the FP64 fields
GROWTH = [("F32", (0.0, 0.0), 0), ("F32", (-0.4, 0.0), 8), ("BF16", (0.0, 0.2), 8), ("F64", (0.0, 0.0), 32),
          ("F64", (-0.4, 0.1), 48)]


@pytest.mark.parametrize("storage,G_self,grown", GROWTH)
def test_workspace_of_one_pass_is_enough(B, L, storage, G_self, grown):
    """Only a context that steps in two passes asks for the room of the moments, and one that is given a workspace
    without it steps in one pass; with less it is refused."""
    shape, N = (32, 16, 16), 32 * 16 * 16
    kw = dict(G=2.5, G_self=G_self, storage=getattr(B, f"SC_STORE_{storage}"))
    size = lambda **more: B.sc_workspace_bytes(B.make_params(shape, **kw, **more))
    one, two = size(variant=1), size()
    assert two - one == grown * N and size(variant=2) == one and size(tau=(1.0, 0.9)) == one

    def variant(c):
        v = (ctypes.c_int32 * 8)()
        assert L.sc_step_config(c.ctx, v, 8) == B.SC_OK
        return v[0]

    p = B.make_params(shape, **kw)
    c = fake_gpu.Context(L, p)
    assert c.status == B.SC_OK and variant(c) == 3
    c = fake_gpu.Context(L, p, one)
    assert c.status == B.SC_OK and variant(c) == (2 if grown else 3)
    assert L.sc_step(c.ctx, 3) == B.SC_OK and c.moments() == B.SC_OK
    assert fake_gpu.Context(L, p, one - 1).status == B.SC_ENOMEM
    host, ws = fake_gpu.buffer(64 * N), fake_gpu.buffer(one)
    h = [ctypes.c_void_p(host[1].value + 8 * N * k) for k in range(4)]
    for nbytes, want in ((one, B.SC_OK), (one - 1, B.SC_ENOMEM)):
        assert L.sc_run_host(ctypes.byref(p), h[0], h[1], 2, h[2], h[3], ws[1], nbytes, None) == want
        assert L.sc_run_host_sigma(ctypes.byref(p), h[0], h[1], 2, None, 0.5, 4, h[2], h[3], host[1], ws[1], nbytes,
                                   None) == want


@pytest.mark.parametrize("storage,G_self,grown", GROWTH)
def test_batch_workspace_of_one_pass_is_enough(B, L, storage, G_self, grown):
    shapes = [(32, 16, 16), (40, 32, 8)]
    kw = dict(G=2.5, G_self=G_self, storage=getattr(B, f"SC_STORE_{storage}"))
    ps = [B.make_params(s, **kw) for s in shapes]
    one = B.sc_batch_workspace_bytes([B.make_params(s, variant=2, **kw) for s in shapes])
    two = B.sc_batch_workspace_bytes(ps)
    assert two - one >= grown * sum(x * y * z for x, y, z in shapes)
    assert L.sc_batch_variant(fake_gpu.Batch(L, ps).handle) == 4
    b = fake_gpu.Batch(L, ps, one)
    assert b.status == B.SC_OK and L.sc_batch_variant(b.handle) == 3
    assert L.sc_batch_step(b.handle, 33) == B.SC_OK
    assert fake_gpu.Batch(L, ps, one - 256).status == B.SC_ENOMEM


@pytest.mark.parametrize("shape,more,want", [
    ((64, 64, 1), {}, (4, 1, 128)),                   # a thread per site and component: blocks of 32 x 1 sites
    ((64, 64, 1), dict(tile_y=1), (1, 1, 128)),       # the same tile asked for: the generic kernel
    ((64, 64, 1), dict(variant=1), (1, 4, 32)),
    ((512, 512, 1), {}, (1, 4, 2048)),
    ((64, 64, 1), dict(storage=0), (1, 4, 32)),
])
def test_step_config_names_the_small_d2q9_kernel(B, L, shape, more, want):
    c = fake_gpu.Context(L, B.make_params(shape, **{**dict(lattice=B.SC_D2Q9, storage=B.SC_STORE_F64, G=2.5), **more}))
    v = (ctypes.c_int32 * 8)()
    assert L.sc_step_config(c.ctx, v, 8) == B.SC_OK
    assert (v[0], v[1], v[5]) == want
    L.fake_reset()
    assert L.sc_step(c.ctx, 1) == B.SC_OK
    assert [("lanes" in n) for n in fake_gpu.calls(L)] == [want[0] == 4]


@pytest.mark.parametrize("storage,tau,side,dependent", [
    ("F32", 1.0, 424, True), ("F32", 1.0, 425, False), ("BF16", 1.0, 424, True), ("BF16", 1.0, 425, False),
    ("F16", 1.0, 894, True), ("F16", 1.0, 895, False), ("F32", 0.9, 1024, True), ("F64", 1.0, 1024, True)])
def test_large_d2q9_lattices_take_plain_launches(B, L, storage, tau, side, dependent):
    c = fake_gpu.Context(L, B.make_params((side, side, 1), lattice=B.SC_D2Q9, tau=(tau, tau), G=2.5,
                                          storage=getattr(B, f"SC_STORE_{storage}")))
    L.fake_reset()
    assert L.sc_step(c.ctx, 1) == B.SC_OK
    assert [n.endswith("(dependent)") for n in fake_gpu.calls(L)] == [dependent]


@pytest.mark.parametrize("storage,psi,shape,passes", [
    # FP32: 4.7 M sites, 33 M with psi
    ("F32", False, (160, 160, 160), 2), ("F32", False, (168, 168, 168), 1), ("F32", True, (320, 320, 320), 2),
    ("F32", True, (324, 324, 324), 1),
    # 16-bit without psi: full tiles up to 28 M sites, one x tile up to 4 M, partial tiles further
    ("F16", False, (288, 288, 288), 2), ("BF16", False, (320, 320, 320), 1), ("F16", False, (512, 512, 512), 1),
    ("F16", False, (32, 360, 360), 2), ("F16", False, (32, 400, 400), 1), ("BF16", False, (336, 336, 336), 2),
    ("F16", False, (496, 496, 496), 1), ("F16", False, (36, 1200, 1200), 2),
    # with psi
    ("F16", True, (512, 512, 512), 2), ("BF16", True, (640, 640, 640), 2),
    # planes too large for two of them to stay in L2, unless the lattice is small or a few planes thick
    ("F16", True, (1024, 1024, 120), 1), ("F16", True, (1024, 1024, 16), 2), ("F16", False, (1024, 1024, 16), 1),
    ("F16", False, (1024, 1024, 8), 2), ("F32", True, (768, 768, 48), 1), ("F32", True, (512, 512, 64), 2),
    # what the staged kernel cannot take
    ("F32", False, (321, 320, 320), 2), ("F16", False, (518, 512, 512), 2),
])
def test_lone_lattices_take_two_passes_where_they_gain(B, L, storage, psi, shape, passes):
    c = fake_gpu.Context(L, B.make_params(shape, G=2.5, G_self=(-0.4 if psi else 0.0, 0.0),
                                          storage=getattr(B, f"SC_STORE_{storage}")))
    assert c.status == B.SC_OK
    v = (ctypes.c_int32 * 8)()
    assert L.sc_step_config(c.ctx, v, 8) == B.SC_OK
    assert v[0] == passes + 1 if passes == 2 else v[0] == 2


def test_large_batch_members_take_their_lone_kernel(B, L):
    """A 16-bit member that steps alone in a two-pass batch does so as a lone lattice of its parameters would: one staged
    launch a step where that one would not take two passes.  In FP32 it takes two passes at any size."""
    for storage, staged in (("F16", True), ("F32", False)):
        kw = dict(G=2.5, storage=getattr(B, f"SC_STORE_{storage}"))
        b = fake_gpu.Batch(L, [B.make_params(s, **kw) for s in ((16, 16, 16), (32, 400, 400), (96, 96, 96))])
        assert b.status == B.SC_OK and L.sc_batch_variant(b.handle) == 4
        L.fake_reset()
        assert L.sc_batch_step(b.handle, 1) == B.SC_OK
        two = ["split_moments", "split_collide"]
        kinds = ("split_moments_batched", "split_collide_batched", *two, "step_staged")
        assert [next(k for k in kinds if k in n) for n in fake_gpu.calls(L)] == [
            *kinds[:2], *(["step_staged"] if staged else two), *two]
        assert L.sc_batch_retire(b.handle, 1) == B.SC_OK
        L.fake_reset()
        assert L.sc_batch_step(b.handle, 1) == B.SC_OK
        assert not any("staged" in n for n in fake_gpu.calls(L)) and len(fake_gpu.calls(L)) == 4
