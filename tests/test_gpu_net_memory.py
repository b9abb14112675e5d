"""What a network holds on the device."""
import gc

import pytest

torch = pytest.importorskip("torch")

from paper_1801_04577_gb300.net import Net  # noqa: E402

pytestmark = pytest.mark.gpu


def held(in_ch, **kw):
    gc.collect()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    net = Net(kw["G"], in_ch, 3, kw["base"], kw["levels"], kw["batch"], seed=1)
    used = before - torch.cuda.mem_get_info()[0]
    net.close()
    return used


def test_operand_tensors_take_the_place_of_fp32_activations():
    """Up to eight input channels the convolutions read operand tensors (2 bytes
    a value, for activations and gradients each, beside FP32 gradients and skip
    connections), with nine they gather from FP32 activations and gradients (4
    bytes each).  The operands' borders, 3 % of half of it, are less than the
    input's share, so the former must not hold more (with the upsampled part of
    the skip tensors in FP32, or partial sums that nothing reads, it held 9 % more)."""
    kw = dict(G=128, base=8, levels=3, batch=64)
    held(8, **kw)  # the library's own first allocations
    assert held(8, **kw) <= held(9, **kw)
