"""Allocation failures that a caller recovers from, and the limits of what is
accepted, on the host (no GPU)."""
import pytest

import fakecuda

OOM, CUDA, UNSUPPORTED = 4, 3, 7


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


# a scan whose spectrum of the BF16 kernel takes more memory than the tensor-core
# operator for BF16, and that one more than the operator for FP8
SCAN = dict(X=40, Y=40, Z=60, T=200)


def _largest(fake, precision, pinned):
    """The largest array that a handle allocates to be used at the precision."""
    h = fakecuda.Handle(fake, **SCAN)
    if pinned:
        h.pin()
    fake.fake_largest()
    assert h.precision(precision) == 0
    h.close()
    return fake.fake_largest()


@pytest.mark.parametrize("first", ["fp32", "fp8"])
def test_bf16_without_memory_for_its_spectrum(fake, first):
    """The tensor-core kernels serve BF16 then, and the transforms again once
    the precision is selected with enough memory."""
    limit = _largest(fake, "bf16", False) - 1
    assert limit >= _largest(fake, "bf16", True)
    h = fakecuda.Handle(fake, **SCAN)
    try:
        assert h.precision(first) == 0
        fake.fake_limit(limit)
        assert h.precision("bf16") == 0, fake.swopt_last_error()
        n = fake.fake_launches(b"spec_kernel"), fake.fake_launches(b"tc_conv_kernel")
        assert h.forward() == 0 and h.adjoint() == 0
        assert fake.fake_launches(b"spec_kernel") == n[0]
        assert fake.fake_launches(b"tc_conv_kernel") == n[1] + 2
        fake.fake_limit(2**63)
        assert h.precision("bf16") == 0
        assert h.forward() == 0 and h.adjoint() == 0
        assert fake.fake_launches(b"spec_kernel") == n[0] + 2
        assert fake.fake_launches(b"tc_conv_kernel") == n[1] + 2
    finally:
        h.close()


def test_former_precision_serves_on_after_a_failed_selection(fake):
    limit = _largest(fake, "fp8", True)
    assert limit < _largest(fake, "bf16", True)
    h = fakecuda.Handle(fake, **SCAN)
    try:
        h.pin()
        assert h.precision("fp8") == 0
        fake.fake_limit(limit)
        assert h.precision("bf16") == OOM and b"cudaMalloc" in fake.swopt_last_error()
        n = fake.fake_launches(b"tc_conv_kernel")
        assert h.forward() == 0 and h.adjoint() == 0, fake.swopt_last_error()
        assert fake.fake_launches(b"tc_conv_kernel") == n + 2
    finally:
        h.close()


@pytest.mark.parametrize("P,N,served", [(1, 1, True), (8, 1, True), (1, 8, False)])
def test_workspaces_and_their_limit(fake, P, N, served):
    """8 GB per workspace for the states' planes, or the direct kernels serve; with
    more species than states the depths of all species (256 pairs on 9 tiles of
    256 x 256), and no more than that."""
    fake.fake_largest()
    h = fakecuda.Handle(fake, X=700, Y=700, Z=512, T=4, N=N, P=P, k=1, cycle=N)
    try:
        largest = fake.fake_largest()
        assert largest == 8 * 9 * 256**2 * 256 * P if served else largest <= 8.1e9
        n = fake.fake_launches(b"spec_kernel")
        assert h.forward() == 0
        assert (fake.fake_launches(b"spec_kernel") > n) == served
    finally:
        h.close()


@pytest.mark.parametrize("kw,geometry,takes", [
    (dict(T=256), "window", True), (dict(T=257), "window", False),
    (dict(Z=256, T=8), "depths", True), (dict(Z=257, T=8), "depths", False)])
@pytest.mark.parametrize("resync", ["bf16", "bf16x3"])
def test_resync_precisions_that_the_tensor_cores_refuse(fake, kw, geometry, takes, resync):
    """A refined FP32 solve refuses a resync precision where selecting it is
    refused, although the transforms would serve it."""
    h = fakecuda.Handle(fake, **kw)
    try:
        for _ in range(2):
            st = h.fista_init(step=0.1, lambda_tv=0.0, refine_every=2, refine_precision=resync)
            assert st == (0 if takes else UNSUPPORTED)
        assert h.precision(resync) == st
        assert h.fista_init(step=0.1, lambda_tv=0.0, refine_every=2, refine_precision="fp32") == 0
    finally:
        h.close()
