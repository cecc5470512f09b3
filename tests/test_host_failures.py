"""Allocation failures that a caller recovers from, on the host (no GPU)."""
import pytest

import fakecuda

OOM, CUDA = 4, 3


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    return fakecuda.load(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def fake(library):
    library.fake_reset()
    yield library
    library.fake_reset()


def test_a_failed_allocation_is_reported_once(fake):
    """The call that it fails says so; the next one, with memory again, works."""
    h = fakecuda.Handle(fake)
    try:
        fake.fake_fail_in(0)
        assert h.objective() == OOM
        assert h.objective() == 0
    finally:
        h.close()


def test_tv_prox_after_a_failed_allocation(fake):
    """Whichever of its allocations fails, the call says so, and the next one
    ends up with every buffer that a handle without a failure has."""
    h = fakecuda.Handle(fake)
    bare = fake.fake_live()
    assert h.prox_tv() == 0 and fake.fake_launches(b"fgp_march") == 1
    need = fake.fake_live() - bare
    h.close()
    assert need >= 4  # barrier words, flags and both dual buffers
    for n in range(need):
        h = fakecuda.Handle(fake)
        try:
            before = fake.fake_launches(b"fgp_")
            fake.fake_fail_in(n)
            assert h.prox_tv() in (OOM, CUDA)
            assert fake.fake_launches(b"fgp_") == before
            assert h.prox_tv() == 0
            assert fake.fake_live() - bare == need, n
            assert fake.fake_launches(b"fgp_march") == before + 1
        finally:
            h.close()
