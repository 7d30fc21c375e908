"""Tiles of the CTA-pair kernels narrower than 256 columns (64, 128, 192; chosen from the shape): products against the
oracle at the edges of tiles, for every operand layout and epilogue.  Bounds: one bf16 rounding (2^-8 relative) of the FP64
product, plus binary32 accumulation (2^-24 per term, K terms, of the sum of magnitudes)."""
import numpy as np
import pytest
import torch

from oracle import tweo_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tw():
    from paper_2511_23225_b200 import binding
    return binding


def _codes(shape, seed):
    g = torch.Generator().manual_seed(seed)
    return torch.randint(0, 256, shape, generator=g, dtype=torch.uint8) & 0xB7   # finite E4M3 codes, both signs, below 2


def _f64(q):
    return q.view(torch.float8_e4m3fn).double()


def _close(y, ref, mag, K):
    err = (y.double().cpu() - ref).abs()
    assert (err <= ref.abs() * 2.0 ** -8 + mag * K * 2.0 ** -24).all(), float((err - ref.abs() * 2.0 ** -8).max())


# widths the rule gives these (148 SMs): 64, 128, 192 and 256; ragged rows, columns and contractions
SHAPES = [(512, 256, 1024), (300, 144, 208), (130, 1024, 1040), (1000, 1024, 1008), (4096, 768, 784), (2300, 3072, 784),
          (700, 2048, 8208), (257, 400, 272)]


@pytest.mark.parametrize("M,K,N", SHAPES)
def test_products_match_float64(tw, M, K, N):
    xq, wq, dyq = _codes((M, K), 1), _codes((N, K), 2), _codes((M, N), 3)
    one = torch.ones(1, device="cuda")
    x, w, dy = xq.cuda(), wq.cuda(), dyq.cuda()
    X, W, D = _f64(xq), _f64(wq), _f64(dyq)
    y = tw.fp8_linear_fwd(x, w, one, one)
    _close(y, X @ W.T, X.abs() @ W.abs().T, K)
    dx, dw = tw.fp8_linear_bwd(dy, x, w, one, one, one, fmt_dy=tw.E4M3)
    _close(dx, D @ W, D.abs() @ W.abs(), N)
    _close(dw, D.T @ X, D.abs().T @ X.abs(), M)
    dx1 = tw.fp8_linear_bwd_dgrad(dy, w, one, one, fmt_dy=tw.E4M3)   # the single product, the same bits
    assert torch.equal(dx1, dx)
    # fused outputs: amax and codes of the stored values, bit for bit
    am, q, sc = torch.zeros(1, device="cuda"), torch.zeros((M, N), dtype=torch.uint8, device="cuda"), torch.full((1,), 0.37, device="cuda")
    y2 = tw.fp8_linear_fwd(x, w, one, one, out_amax=am, out_q=q, q_scale=sc)
    assert torch.equal(y2, y) and float(am) == float(y.float().abs().max())
    codes = orc.quantize_bf16(y.view(torch.int16).cpu().numpy().view(np.uint16), orc.E4M3, 0.37)
    assert np.array_equal(q.cpu().numpy(), codes[0] if isinstance(codes, tuple) else codes)
    assert tw.read_device_status() == 0


@pytest.mark.parametrize("M,K,N", [(1200, 512, 2064), (3000, 256, 1040), (2000, 1024, 272)])
def test_integer_product_is_exact(tw, M, K, N):
    g = torch.Generator().manual_seed(4)
    x, w = (torch.randint(-127, 128, s, generator=g, dtype=torch.int8) for s in ((M, K), (N, K)))
    one = torch.full((1,), 127.0, device="cuda")
    y = tw.int8_linear(x.cuda(), one, w.cuda(), one)
    ref = (x.double() @ w.double().T).float().to(torch.bfloat16)   # 1 / 127^2 and 127^2 cancel to one binary32 rounding each
    assert ((y.cpu().double() - ref.double()).abs() <= ref.double().abs() * 2.0 ** -7).all()


@pytest.mark.parametrize("act", ["ACT_GELU", "ACT_GELU_TANH"])
@pytest.mark.parametrize("M,K,N", [(2000, 768, 3088), (300, 256, 272)])
def test_activation_equals_the_one_of_a_wider_launch(tw, act, M, K, N):
    """Every row is the same whatever the launch it is part of: 20 times the rows take tiles of 256 columns."""
    one = torch.full((1,), 0.05, device="cuda")
    x, w = _codes((M, K), 5).cuda(), _codes((N, K), 6).cuda()
    y = tw.fp8_linear_fwd_act(x, w, one, one, getattr(tw, act))
    big = tw.fp8_linear_fwd_act(x.repeat(20, 1), w, one, one, getattr(tw, act))
    assert torch.equal(big.view(20, M, N), y.expand(20, M, N))
