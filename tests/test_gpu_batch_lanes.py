"""One batched launch whose members are few markers each and many together:
the interpolation then takes one lane per marker, where each member alone
takes eight.  The members (pulling, reading the node moments, with the node
cache; FP32 and 16-bit; with and without walls) must still have exactly the
results of the same box in a batch of its own."""
import pytest

from tests.gpu_helpers import require_cuda
from tests.test_gpu_batch_forms import advance, assert_same, make_member

pytestmark = pytest.mark.gpu

KINDS = [("fc", "f32", False), ("ibm", "f32", False), ("fc_inside", "f32", False),
         ("fc", "f32", True), ("fc", "f16dev", True), ("fc_inside", "bf16dev", False)]


@pytest.mark.parametrize("moments", [0, 1])
def test_members_of_a_large_launch_equal_the_member_alone(moments):
    require_cuda()
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    M = 50 * sms + 1                  # alone: eight lanes; two together: one
    assert M <= 8192                  # (the members can be recorded)

    def member(q):
        return make_member(*KINDS[q // 2], moments=moments, seed=40 + q, count=M)

    mix = advance([member(q) for q in range(2 * len(KINDS))], "batched")
    for q in range(2 * len(KINDS)):
        assert_same(mix[q], advance([member(q)], "batched")[0])
