"""Which of the two row kernels a call takes, and calls by way of the streaming kernel whatever their size."""
import torch


def short(e3, rows, V, dtype, sampler=-1, masked=False):
    """Blocks per row of the kernel of short calls on this device, 0 where the call takes the streaming kernel."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return e3.e3_test_row_blocks(e3.E3_F32 if dtype == torch.float32 else e3.E3_BF16, rows, V, sampler, masked, sms)


class Streaming:
    """The binding, with every row call sent to the streaming kernel: the test hook, armed for a tile behind the call's last one, stalls
    nothing.  A stall that a test has armed itself stays as it is."""

    def __init__(self, e3):
        self._e3, self._armed = e3, False

    def __getattr__(self, name):
        return getattr(self._e3, name)

    def e3_test_arm_stall(self, tile, wait_ns):
        self._e3.e3_test_arm_stall(tile, wait_ns)
        self._armed = True

    def _through(self, call, args, kwargs):
        if not self._armed:
            self._e3.e3_test_arm_stall(1 << 40, 2_000_000_000)
        self._armed = False
        try:
            return call(*args, **kwargs)
        finally:
            self._e3.e3_test_arm_stall(-1, 0)

    def e3_sample(self, *args, **kwargs):
        return self._through(self._e3.e3_sample, args, kwargs)

    def e3_token_logp_entropy(self, *args, **kwargs):
        return self._through(self._e3.e3_token_logp_entropy, args, kwargs)
