"""Host side of the library without a GPU: which device memory belongs to, who waits for what, what happens when an
allocation fails.  Two pretended devices (tests/fake_cudart.cpp); kernels do not run, they only report sizes."""
import pytest

from tests import fake_device


@pytest.fixture(scope="module")
def so(tmp_path_factory):
    return fake_device.build(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def fake(so):
    return fake_device.Fake(so)


def test_sizes_read_while_another_device_is_current(fake):
    """Sample on device 1, then on device 0, then ask for the sizes of the first object: what its context needs is made on
    device 1, and no block changes its device."""
    ctx1, ctx0 = fake.context(1), fake.context(0)
    fake.report(PHI=5000, PSI=6000, EDGES=900)
    rc, on1 = fake.sample(ctx1, 100)
    assert rc == 0
    rc, on0 = fake.sample(ctx0, 100)
    assert rc == 0
    live0 = fake.lib.fake_live(0)
    assert fake.lib.fake_current() == 0
    assert fake.nnz(on1) == (0, 5000) and fake.nnz(on1, 2) == (0, 6000)
    assert fake.lib.fake_live(0) == live0
    fake.report(EDGES=90000)                      # grows what was made above
    assert fake.sample(ctx1, 100, on1)[0] == 0
    fake.lib.fake_set_current(0)
    assert fake.nnz(on1)[0] == 0
    assert fake.sample(ctx0, 100, on0)[0] == 0
    assert fake.sample(ctx1, 100, on1)[0] == 0    # its launches find their memory on device 1
    assert fake.errors() == 0
    for h in (on0, on1):
        assert fake.lib.grf_features_free(h) == 0
    for c in (ctx0, ctx1):
        assert fake.lib.grf_ctx_destroy(c) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0 and fake.lib.fake_live(1) == 0
