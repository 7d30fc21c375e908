"""The few-token product kernel at the edges of its splits: token tiles, slices of the contraction, ragged widths, and the
data gradient's operand layout.  Reference: the exact product of the decoded codes.  An output may differ from it by its
one bf16 rounding (2^-8 of the value) and by the binary32 accumulation, held to 1e-4 of the largest output like
every product of this library."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tw():
    from paper_2511_23225_b200 import binding
    binding.lib()
    return binding


def codes(shape, seed, fmt=torch.float8_e4m3fn, std=60.0):
    x = torch.randn(shape, generator=torch.Generator().manual_seed(seed)) * std
    return x.clamp(-448, 448).to(fmt)


def close(got, ref):
    got = got.double().cpu()
    assert torch.all((got - ref).abs() <= ref.abs() * 2.0 ** -8 + 1e-4 * ref.abs().max())


# tokens: one and two tiles, whole and ragged ones; contractions of one block, of an odd width, and long enough for eight slices
@pytest.mark.parametrize("M,K,N", [(1, 16, 16), (17, 1040, 144), (128, 4096, 272), (129, 2064, 528), (256, 4096, 1040), (257, 4096, 128),
                                   (300, 1024, 4096), (520, 8208, 400), (777, 3344, 880)])
def test_static_linear_matches_the_product_of_the_codes(tw, M, K, N):
    x, w = codes((M, K), M + K), codes((N, K), N, std=30.0)
    sx, sw = torch.full((1,), 16.0), torch.full((1,), 0.125)
    y = tw.w8a8_static_gemm(x.view(torch.uint8).cuda(), sx.cuda(), w.view(torch.uint8).cuda(), sw.cuda())
    again = tw.w8a8_static_gemm(x.view(torch.uint8).cuda(), sx.cuda(), w.view(torch.uint8).cuda(), sw.cuda())
    torch.cuda.synchronize()
    assert tw.read_device_status() == 0 and torch.equal(y, again)
    close(y, x.double() @ w.double().T * (0.125 / 16.0))


# the form inference takes: bf16 activations, whose cast the product overlaps (its weight is loaded while the cast runs)
@pytest.mark.parametrize("M,K,N", [(1, 4096, 1040), (128, 1040, 272), (129, 2064, 528), (257, 4096, 128), (300, 4096, 4096), (777, 3344, 880)])
def test_static_linear_on_bf16_activations(tw, M, K, N):
    x = torch.randn((M, K), generator=torch.Generator().manual_seed(M * 3 + K)).to(torch.bfloat16)
    w, s = codes((N, K), N, std=30.0), 100.0
    sx, sw = torch.full((1,), s), torch.full((1,), 0.125)
    y = tw.w8a8_static_gemm(x.cuda(), sx.cuda(), w.view(torch.uint8).cuda(), sw.cuda())
    again = tw.w8a8_static_gemm(x.cuda(), sx.cuda(), w.view(torch.uint8).cuda(), sw.cuda())
    torch.cuda.synchronize()
    assert tw.read_device_status() == 0 and torch.equal(y, again)
    xq = (x.float() * s).clamp(-448, 448).to(torch.float8_e4m3fn)
    close(y, xq.double() @ w.double().T * (0.125 / s))


# integer sums are exact: the two scales and the bf16 rounding are all that may differ (three roundings of 2^-24, one of 2^-8)
@pytest.mark.parametrize("M,K,N", [(1, 16, 16), (128, 4096, 272), (129, 2064, 528), (257, 4096, 128), (300, 4096, 4096), (777, 3344, 880)])
def test_integer_linear_matches_the_product_of_the_codes(tw, M, K, N):
    g = torch.Generator().manual_seed(M + K + N)
    x, w = (torch.randint(-127, 128, shape, generator=g, dtype=torch.int8) for shape in ((M, K), (N, K)))
    sx, sw = torch.rand(M, generator=g) + 0.5, torch.rand(N, generator=g) + 0.5
    y = tw.int8_linear(x.cuda(), sx.cuda(), w.cuda(), sw.cuda())
    torch.cuda.synchronize()
    assert tw.read_device_status() == 0
    ref = (x.double() @ w.double().T) * (sx.double()[:, None] / 127.0) * (sw.double() / 127.0)
    assert torch.all((y.double().cpu() - ref).abs() <= ref.abs() * (2.0 ** -8 + 2.0 ** -21))


def test_static_linear_into_rows_that_allow_no_wide_stores(tw):
    M, K, N = 5, 512, 144
    x, w = codes((M, K), 3), codes((N, K), 4)
    one = torch.ones(1, device="cuda")
    y = torch.zeros((M, N + 3), dtype=torch.bfloat16, device="cuda")
    tw.w8a8_static_gemm(x.view(torch.uint8).cuda(), one, w.view(torch.uint8).cuda(), one, y=y[:, 1:N + 1])
    torch.cuda.synchronize()
    close(y[:, 1:N + 1], x.double() @ w.double().T)
    assert not y[:, 0].any() and not y[:, N + 1:].any()


@pytest.mark.parametrize("M,N,K", [(1, 16, 16), (16, 400, 528), (100, 5760, 272), (128, 1024, 4096), (128, 144, 128)])
def test_few_token_data_gradient(tw, M, N, K):
    dy, w = codes((M, N), M + N, torch.float8_e5m2, 2.0), codes((N, K), K, std=30.0)
    one = torch.ones(1, device="cuda")
    dx = tw.fp8_linear_bwd_dgrad(dy.view(torch.uint8).cuda(), w.view(torch.uint8).cuda(), one, one)
    torch.cuda.synchronize()
    assert tw.read_device_status() == 0
    close(dx, dy.double() @ w.double())


def test_first_calls_from_several_threads():
    """The split of a process's first few-token products, asked for by eight threads at once, each on a stream of its own."""
    import subprocess
    import sys
    code = """
import threading
import torch
from paper_2511_23225_b200 import binding as tw
x = torch.randint(0, 0x70, (8, 4096), dtype=torch.uint8, device="cuda")
w = torch.randint(0, 0x70, (4096, 4096), dtype=torch.uint8, device="cuda")
one, out, gate = torch.ones(1, device="cuda"), [None] * 8, threading.Barrier(8)
torch.cuda.synchronize()
def work(i):
    with torch.cuda.stream(torch.cuda.Stream()):
        gate.wait()
        out[i] = tw.fp8_linear_fwd(x[i:i + 1], w, one, one)
        torch.cuda.current_stream().synchronize()
ts = [threading.Thread(target=work, args=(i,)) for i in range(8)]
[t.start() for t in ts]
[t.join() for t in ts]
assert tw.read_device_status() == 0
for i in range(8):
    assert torch.equal(out[i], tw.fp8_linear_fwd(x[i:i + 1], w, one, one))
print("same")
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split() == ["same"], r.stderr[-2000:]
