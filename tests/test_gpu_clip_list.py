"""stage_clip over many tensors per launch: sizes at the edges of the chunks and of the 16-byte accesses, both
element types in one stage, unaligned and empty tensors, more tensors than one launch takes, overlapping ones."""

import numpy as np
import pytest
import torch

from oracle import dp_oracle as dp
from paper_2607_13332_b200 import binding, dp_ops
from oracle.metrics import max_rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [
    [1, 7, 8, 0, 8191, 8192, 8193, 16384, 16385, 3 * 16384 + 5], [16384 * 2400 + 3, 1, 40000], list(range(1, 131))])
def test_many_tensors_per_launch(sizes):
    g = torch.Generator(device="cuda").manual_seed(len(sizes))
    grads = []
    for i, n in enumerate(sizes):               # every third tensor unaligned, both types
        dt = torch.float32 if i % 2 else torch.bfloat16
        t = torch.randn(n + 1, device="cuda", generator=g).to(dt)
        grads.append(t[1:] if i % 3 == 0 else t[:n])
    before = [t.double().cpu().numpy() for t in grads]
    expect, norm, coef = dp.stage_clip(before, 0.5)
    norm2 = float(dp_ops.stage_clip(grads, 0.5).item())
    assert coef < 1.0 and abs(norm2 - norm * norm) <= 1e-6 * norm * norm   # squares summed four (eight) at a time in fp32
    for t, e in zip(grads, expect):
        # one rounding of the coefficient and one of the product
        assert max_rel_err(t.double().cpu().numpy(), e) <= (2.0**-22 if t.dtype == torch.float32 else 2.0**-8)
    kept = [t.clone() for t in grads]
    dp_ops.stage_clip(grads, 10.0)              # inside the budget: untouched
    assert all(torch.equal(a, b) for a, b in zip(grads, kept))


def test_overlapping_tensors_and_errors():
    a = torch.full((1000,), 2.0, device="cuda")
    s = dp_ops.stage_clip([a, a[:100]], 1.0)    # counted twice and scaled twice, as one tensor after the other is
    assert abs(float(s.item()) - 4400.0) < 1e-2
    coef = 1.0 / (np.sqrt(4400.0) + 1e-6)
    assert abs(float(a[0]) - 2 * coef * coef) < 1e-6 and abs(float(a[999]) - 2 * coef) < 1e-6
    s = torch.zeros(1, dtype=torch.float64, device="cuda")
    for tensors, thr, status in ((binding.clip_list([0], [4], [0]), 1.0, binding.SSN_ERR_NULL),
                                 (binding.clip_list([a.data_ptr()], [4], [9]), 1.0, binding.SSN_ERR_DTYPE),
                                 (binding.clip_list([a.data_ptr()], [-1], [0]), 1.0, binding.SSN_ERR_SHAPE),
                                 (binding.clip_list([a.data_ptr()], [4], [0]), 0.0, binding.SSN_ERR_SHAPE)):
        with pytest.raises(binding.SsnError) as e:
            binding.stage_clip_scale_list(tensors, s.data_ptr(), thr)
        assert e.value.status == status
    binding.stage_clip_sumsq_list(binding.clip_list([], [], []), s.data_ptr())
    torch.cuda.synchronize()
    assert float(s.item()) == 0.0


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n", [0, 1, 4097])
def test_one_tensor_alone(n, dt):
    """A single tensor takes the launches without a list, to the same result."""
    t = torch.randn(n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(n)).to(dt)
    before = t.double().cpu().numpy()
    expect, norm, _ = dp.stage_clip([before], 0.01)
    norm2 = float(dp_ops.stage_clip([t], 0.01).item())
    assert abs(norm2 - norm * norm) <= 1e-6 * norm * norm
    if n:
        assert max_rel_err(t.double().cpu().numpy(), expect[0]) <= (2.0**-22 if dt == torch.float32 else 2.0**-8)
