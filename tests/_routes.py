"""Calls by way of one of the two row kernels."""


def streaming(e3):
    """Makes a row call go through the streaming kernel, whatever its size: the test hook, armed for a tile behind the call's last one,
    stalls nothing."""
    def through(call, *args, **kwargs):
        e3.e3_test_arm_stall(1 << 40, 2_000_000_000)
        return call(*args, **kwargs)
    return through
