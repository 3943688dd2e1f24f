"""The torch-facing codec object: every call sees what is attached to it now."""

import pytest
import torch

from paper_2607_13332_b200 import synth
from tests.harness import Codec

pytestmark = pytest.mark.gpu


def _codec(seed, d=256, k=16):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return Codec(synth.F32, torch.randn((d, k), device="cuda", generator=g))


def test_a_replaced_c_codec_is_used_by_every_call():
    codec, other = _codec(1), _codec(2)
    codec.c = other.c
    X, Z = torch.randn((33, 256), device="cuda"), torch.randn((33, 16), device="cuda")
    for call in (lambda c: c.compress(X), lambda c: c.decompress(Z), lambda c: c.grad_project(X), lambda c: c.grad_project_wire(X)):
        assert torch.equal(call(codec), call(other))
