"""A product whose weight operand the call just before it writes, without a host synchronisation in between: the few-token
kernel starts while that call is still running and must not take the weight's former contents.  Every step writes other codes
into the same buffer.  Reference: the same product on a copy of the codes, after everything has completed (the products do
not depend on timing)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

STEPS = 12


@pytest.fixture(scope="module")
def tw():
    from paper_2511_23225_b200 import binding
    binding.lib()
    return binding


def i8(shape, seed):
    return torch.randint(-127, 128, shape, generator=torch.Generator().manual_seed(seed), dtype=torch.int8).cuda()


def run(tw, weight_of, product):
    """weight_of(step) enqueues the call that writes the weight and returns it; product(w) is checked for every step."""
    torch.cuda.synchronize()
    got = []
    for s in range(STEPS):
        w = weight_of(s)
        got.append((product(w), w.clone()))
    torch.cuda.synchronize()
    assert tw.read_device_status() == 0
    for s, (y, w) in enumerate(got):
        torch.cuda.synchronize()
        assert torch.equal(y, product(w)), f"step {s} used other codes"
        assert s == 0 or not torch.equal(w, got[s - 1][1])


# tokens: the narrow ring, and (above 128) the wide one with a ragged last tile
@pytest.mark.parametrize("M", [1, 16, 128, 300])
@pytest.mark.parametrize("writer", ["int8_linear_q8", "residual_add_q8", "residual_add_q8_rows", "absmax_rows", "absmax_tensor",
                                    "linear_behind_an_addition"])
def test_integer_linear_behind_the_call_that_writes_its_weight(tw, writer, M):
    N, K, C = 1024, 1024, 2048           # weight [N, K]; C: the contraction of the linear that writes it
    one = torch.ones(1, device="cuda")
    rows = torch.rand(N, generator=torch.Generator().manual_seed(9)).cuda() + 0.5
    src, mat = [i8((N, C), 20 + s) for s in range(STEPS)], i8((K, C), 3)
    a, b = [i8((N, K), 50 + s) for s in range(STEPS)], i8((N, K), 4)
    act = [torch.randn((N, K), generator=torch.Generator().manual_seed(80 + s)).to(torch.bfloat16).cuda() for s in range(STEPS)]
    x, w = i8((M, K), 7), torch.zeros((N, K), dtype=torch.int8, device="cuda")
    other = torch.zeros_like(w)
    big = one * 60.0

    def weight_of(s):
        if writer in ("int8_linear_q8", "linear_behind_an_addition"):
            tw.int8_linear_q8(src[s], one, mat, one, big, yq=w)
            if writer == "linear_behind_an_addition":   # does not touch w, but starts early itself
                tw.residual_add_q8_rows(a[s], rows, b, rows, yq=other)
            return w
        if writer == "residual_add_q8":
            tw.residual_add_q8(a[s], one, b, one, one * 2.0, yq=w)
            return w
        if writer == "residual_add_q8_rows":
            tw.residual_add_q8_rows(a[s], rows, b, rows, yq=w)
            return w
        return tw.absmax_quantize(act[s], granularity=tw.GRAN_ROW if writer == "absmax_rows" else tw.GRAN_TENSOR)[0]

    run(tw, weight_of, lambda v: tw.int8_linear(x, one, v, rows))


@pytest.mark.parametrize("M", [1, 16, 128])
@pytest.mark.parametrize("writer", ["fp4_quantize", "copy"])
def test_packed_weight_linear_behind_the_call_that_writes_its_weight(tw, writer, M):
    N, K = 2048, 2048
    one = torch.ones(1, device="cuda")
    ws = [torch.randn((N, K), generator=torch.Generator().manual_seed(30 + s)).to(torch.bfloat16).cuda() for s in range(STEPS)]
    packed = [tw.fp4_quantize(w, carriers=False).q4.view(N, K // 2) for w in ws]
    x = torch.randint(0, 0x70, (M, K), generator=torch.Generator().manual_seed(5), dtype=torch.uint8).cuda()
    out = tw.QuantizedFP4(torch.zeros(N * K // 2, dtype=torch.uint8, device="cuda"), None, *(torch.ones(1, device="cuda") for _ in range(3)))

    def weight_of(s):
        if writer == "fp4_quantize":
            tw.fp4_quantize(ws[s], carriers=False, out=out)
        else:
            out.q4.copy_(packed[s].view(-1))
        return out.q4.view(N, K // 2)

    run(tw, weight_of, lambda w: tw.fp4_weight_linear(x, one, w, one))


# the product behind the call's own cast loads its weight at once: the call before has to have completed by then
@pytest.mark.parametrize("M", [1, 16, 128, 300])
def test_static_4_bit_linear_behind_the_cast_of_its_weight(tw, M):
    N, K = 2048, 4096
    one = torch.ones(1, device="cuda")
    ws = [torch.randn((N, K), generator=torch.Generator().manual_seed(40 + s)).to(torch.bfloat16).cuda() for s in range(STEPS)]
    x = torch.randn((M, K), generator=torch.Generator().manual_seed(6)).to(torch.bfloat16).cuda()
    out = tw.QuantizedFP4(None, torch.zeros((N, K), dtype=torch.uint8, device="cuda"), *(torch.ones(1, device="cuda") for _ in range(3)))
    buf = tw.new_workspace(tw.OP_W8A8, M, N, K)
    run(tw, lambda s: tw.fp4_quantize(ws[s], packed=False, out=out).q8, lambda w: tw.w4a4_static_gemm(x, one, w, one, ws=buf))


@pytest.mark.parametrize("M", [1, 16, 128, 300])
@pytest.mark.parametrize("call", ["fwd", "dgrad", "w8a8_codes", "w8a8_bf16"])
def test_fp8_product_behind_the_cast_of_its_weight(tw, call, M):
    N, K = 2048, 4096
    one = torch.ones(1, device="cuda")
    ws = [torch.randn((N, K), generator=torch.Generator().manual_seed(60 + s)).to(torch.bfloat16).cuda() for s in range(STEPS)]
    out = tw.Quantized(torch.zeros((N, K), dtype=torch.uint8, device="cuda"), *(torch.ones(1, device="cuda") for _ in range(3)), None, tw.E4M3)
    g = torch.Generator().manual_seed(8)
    xb, buf = torch.randn((M, K), generator=g).to(torch.bfloat16).cuda(), tw.new_workspace(tw.OP_W8A8, M, N, K)
    xq, dy = (torch.randint(0, 0x70, (M, c), generator=g, dtype=torch.uint8).cuda() for c in (K, N))
    product = {"fwd": lambda w: tw.fp8_linear_fwd(xq, w, one, one), "dgrad": lambda w: tw.fp8_linear_bwd_dgrad(dy, w, one, one),
               "w8a8_codes": lambda w: tw.w8a8_static_gemm(xq, one, w, one, ws=buf), "w8a8_bf16": lambda w: tw.w8a8_static_gemm(xb, one, w, one, ws=buf)}[call]
    run(tw, lambda s: tw.quantize_per_tensor(ws[s], out=out).q, product)
