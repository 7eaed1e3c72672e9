"""Each translation unit has its own device error flag: the check must read every one that a wait can raise."""

from test_host_launches import libs, run  # noqa: F401


def test_every_unit_that_waits_is_read(libs):  # noqa: F811
    """Each unit's flag, raised alone in the stand-in runtime, is reported once and cleared.  Units without a wait
    register no flag."""
    run("""
assert fk.flags >= 4  # element-wise kernels, GEMM, attention and the self-test
assert lib.acid_check_device_error() == A.ACID_OK
for unit in range(fk.flags):
    fk.raised = unit
    assert lib.acid_check_device_error() == A.ACID_ERR_TIMEOUT, unit
    assert lib.acid_check_device_error() == A.ACID_OK, unit
""", *libs)
