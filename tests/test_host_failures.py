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
