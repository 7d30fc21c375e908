"""Static W8A8 on few bf16 activations, cast in the product's kernel: the same bits as the product of the codes that the
cast of its own gives (one kernel, one split, one order of sums), for token counts, contractions and widths at the edges."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tw():
    from paper_2511_23225_b200 import binding
    binding.lib()
    return binding


# one to four groups of 16 tokens; one k-block, a ragged last one, slices of 1, 4, 16, 26 and 27 k-blocks; ragged widths
@pytest.mark.parametrize("M", [1, 7, 15, 16, 17, 31, 32, 33, 48, 49, 64])
@pytest.mark.parametrize("K,N", [(16, 16), (112, 144), (4096, 1040), (3344, 272), (8192, 8192), (6656, 12000), (6800, 12000), (8208, 4096)])
def test_same_bits_as_the_cast_of_its_own(tw, M, K, N):
    g = torch.Generator(device="cuda").manual_seed(M * 7 + K)
    x = torch.randn((M, K), device="cuda", generator=g).to(torch.bfloat16)
    flat = x.view(-1)
    flat[0], flat[-1], flat[K // 2] = 1e30, -float("inf"), -0.0   # saturated
    w = torch.randint(0, 256, (N, K), dtype=torch.uint8, device="cuda", generator=g) & 0xB7   # finite codes of both signs
    sx, sw = torch.full((1,), 97.0, device="cuda"), torch.full((1,), 0.125, device="cuda")
    ws = tw.new_workspace(tw.OP_W8A8, M, N, K).fill_(255)
    y = [tw.w8a8_static_gemm(x, sx, w, sw, ws=ws) for _ in range(3)]
    codes = tw.quantize_per_tensor(x, tw.E4M3, tw.SCALE_GIVEN, scale=sx).q
    ref = tw.w8a8_static_gemm(codes, sx, w, sw, ws=ws)
    assert tw.read_device_status() == 0
    assert all(torch.equal(t, ref) for t in y)
    x[0, K - 1] = float("nan")
    bad = tw.w8a8_static_gemm(x, sx, w, sw, ws=ws)
    assert torch.equal(bad[1:], ref[1:]) and torch.isnan(bad[0].float()).all()


def test_weights_and_activations_written_just_before(tw):
    """A chain of calls, each on operands that the kernel before it wrote."""
    M, K, N = 8, 4096, 4096
    one = torch.ones(1, device="cuda")
    ws = tw.new_workspace(tw.OP_W8A8, M, N, K)
    w = [torch.randint(0, 256, (N, K), dtype=torch.uint8, device="cuda") & 0xB7 for _ in range(3)]
    x = [torch.randn((M, K), device="cuda").to(torch.bfloat16) for _ in range(3)]
    want = [tw.w8a8_static_gemm(a, one, b, one, ws=ws) for a, b in zip(x, w)]
    torch.cuda.synchronize()
    wb, xb, got = torch.empty_like(w[0]), torch.empty_like(x[0]), []
    for _ in range(20):
        for a, b in zip(x, w):
            wb.copy_(b)
            xb.copy_(a)
            got.append(tw.w8a8_static_gemm(xb, one, wb, one, ws=ws))
    torch.cuda.synchronize()
    assert all(torch.equal(t, want[i % 3]) for i, t in enumerate(got))
