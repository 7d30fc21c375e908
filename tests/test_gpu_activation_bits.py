"""The MLP activations of the forward epilogue, bit for bit.  Every E5M2 code times every E4M3 code (infinities and NaN among
them) is an exact accumulator; three dequantisation factors spread them over the range in which the activation bends.
The digests are those of the scalar form, one binary32 operation after another: rewriting it for speed moves no rounding."""
import hashlib

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

FACTORS = (1.0, 0.0137, 3.1e-4)
# stored bf16 outputs, FP8 copies and amax of the three factors, in this order
DIGESTS = {
    "gelu": "7aa98a82facf9534bc3f4e0f787f9fb62c8621ef724885729648fed54388e648",
    "gelu_tanh": "f36583745a8f38de96d904c957bfabd2d96f61654c64bac07dd0f6af58c3c20f",
    "swiglu": "f94051e4d387d1dc2697c0206f02b228c717558413bfb3cf2d89e8670f45c63a",
}


@pytest.fixture(scope="module")
def tw():
    from paper_2511_23225_b200 import binding
    binding.lib()
    return binding


def outputs(tw, act):
    """[(y, copy, amax)] for the three factors; rows: E5M2 codes, columns: E4M3 codes."""
    code = torch.arange(256, dtype=torch.uint8, device="cuda")
    x = torch.zeros((256, 16), dtype=torch.uint8, device="cuda")
    x[:, 0] = code
    rows = 512 if act == "swiglu" else 256
    w = torch.zeros((rows, 16), dtype=torch.uint8, device="cuda")
    w[:256, 0] = code
    if act == "swiglu":
        w[256:, 0] = 0x38 + (code & 7)     # the up rows: 1 to 1.875
    kind = {"gelu": tw.ACT_GELU, "gelu_tanh": tw.ACT_GELU_TANH, "swiglu": tw.ACT_SWIGLU}[act]
    one, res = torch.ones(1, device="cuda"), []
    for f in FACTORS:
        amax = torch.zeros(1, device="cuda")
        q = torch.zeros((256, 256), dtype=torch.uint8, device="cuda")
        y = tw.fp8_linear_fwd_act(x, w, one, one * f, kind, fmt_x=tw.E5M2, out_amax=amax, out_q=q, q_scale=one * 3.0)
        res.append((y, q, amax))
    torch.cuda.synchronize()
    assert tw.read_device_status() == 0
    return res


def digest(res):
    h = hashlib.sha256()
    for y, q, amax in res:
        for t in (y.view(torch.int16), q, amax.view(torch.int32)):
            h.update(np.ascontiguousarray(t.cpu().numpy()).tobytes())
    return h.hexdigest()


@pytest.mark.parametrize("act", sorted(DIGESTS))
def test_every_product_of_two_codes_keeps_its_bits(tw, act):
    assert digest(outputs(tw, act)) == DIGESTS[act]


def test_infinities_and_nan_follow_the_definition(tw):
    """v Phi(v): infinity at +infinity, NaN at -infinity (infinity times zero) and at NaN; v / (1 + exp(-v)) the same."""
    plus, minus, nan, one = 0x7C, 0xFC, 0x7F, 0x38      # rows: E5M2 codes; column: E4M3 1.0
    for act in sorted(DIGESTS):
        y = outputs(tw, act)[0][0]
        assert y[plus, one].item() == float("inf")
        assert torch.isnan(y[minus, one]) and torch.isnan(y[nan, one])
        assert y[0, one].item() == 0.0
