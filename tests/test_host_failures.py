"""Allocation failures that a caller recovers from, on the host (no GPU)."""
import pytest

import fakecuda

OOM = 4


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
