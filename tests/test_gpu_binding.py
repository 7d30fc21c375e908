"""What the calls of the native marshalling module accept and refuse."""
import collections
import types

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tw():
    from paper_2511_23225_b200 import binding
    binding.lib()
    return binding


def codes(shape, seed):
    return torch.randint(0, 0x70, shape, generator=torch.Generator().manual_seed(seed), dtype=torch.uint8).cuda()


@pytest.mark.parametrize("kind", [dict, collections.OrderedDict, collections.UserDict, types.MappingProxyType, lambda d: collections.ChainMap({}, d),
                                  lambda d: collections.defaultdict(lambda: None, d)])
def test_a_grouped_problem_is_any_mapping(tw, kind):
    x, w, one = codes((256, 256), 1), codes((384, 256), 2), torch.ones(1, device="cuda")
    y, amax, copy = torch.zeros((256, 384), dtype=torch.bfloat16, device="cuda"), torch.zeros(1, device="cuda"), torch.zeros((256, 384), dtype=torch.uint8, device="cuda")
    problem = dict(product=tw.PRODUCT_FWD, xq=x, wq=w, sx_inv=one, sw_inv=one, out=y, out_amax=amax, out_q=copy, q_scale=one)
    tw.fp8_linear_group([kind(problem)])
    torch.cuda.synchronize()
    assert torch.equal(y, tw.fp8_linear_fwd(x, w, one, one)) and amax.item() == y.float().abs().max().item() and copy.any()
    for missing in ("product", "out"):
        if kind is dict or kind is collections.UserDict:
            with pytest.raises(KeyError):
                tw.fp8_linear_group([kind({k: v for k, v in problem.items() if k != missing})])
    with pytest.raises(TypeError):
        tw.fp8_linear_group([kind({**problem, "wq": w.cpu()})])


def test_a_single_cast_writes_into_storage_of_any_type(tw):
    x = torch.randn(4096, generator=torch.Generator().manual_seed(3)).to(torch.bfloat16).cuda()
    ref = tw.quantize_per_tensor(x)
    for qt in (torch.uint8, torch.int8, torch.float8_e4m3fn):
        cell = lambda: torch.zeros(1, dtype=torch.int32, device="cuda")
        out = tw.Quantized(torch.zeros(4096, dtype=qt, device="cuda"), torch.zeros(1, device="cuda"), cell(), cell(), cell(), tw.E4M3)
        assert tw.quantize_per_tensor(x, out=out) is out
        torch.cuda.synchronize()
        assert torch.equal(out.q.view(torch.uint8), ref.q) and torch.equal(out.scale, ref.scale)
        assert torch.equal(out.amax.view(torch.float32), ref.amax) and torch.equal(out.scale_inv.view(torch.float32), ref.scale_inv)
        assert out.sat_count.item() == 0
        if qt == torch.int8:
            with pytest.raises(TypeError):        # a batch states what it takes
                tw.quantize_per_tensor_batch([x], [out])
        out.q = out.q.cpu()
        with pytest.raises(TypeError):
            tw.quantize_per_tensor(x, out=out)


def test_a_required_workspace_is_storage_of_any_type(tw):
    def both(op, call, *shape):
        ws = tw.new_workspace(op, *shape)
        ref = call(ws)
        got = call(torch.zeros(ws.numel(), dtype=torch.int32, device="cuda"))
        torch.cuda.synchronize()
        assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(ref, got))
        with pytest.raises(TypeError):
            call(ws.cpu())

    x, f = (torch.randn((16, 256), generator=torch.Generator().manual_seed(s)).to(torch.bfloat16).cuda() for s in (1, 2))
    w, one = codes((272, 256), 3), torch.ones(1, device="cuda")
    record = lambda: tw.Quantized(torch.zeros(x.shape, dtype=torch.uint8, device="cuda"), *(torch.zeros(1, device="cuda") for _ in range(3)), None, tw.E4M3)
    both(tw.OP_QUANTIZE, lambda ws: [tw.quantize_per_tensor_batch([x], [record()], ws=ws)[0].q])
    both(tw.OP_LOSS, lambda ws: [tw.loss_fwd_bwd([x, f], ws=ws)[0]], x.numel(), 2)
    both(tw.OP_W8A8, lambda ws: [tw.w8a8_static_gemm(x, one, w, one, ws=ws)], 16, 272, 256)
    both(tw.OP_BLOCK_OUTPUT, lambda ws: tw.block_output_fused(x, f, ws=ws)[:4])


def test_an_output_that_does_not_fit_is_an_out_of_memory_error(tw):
    """Under a limit of the allocator's own, so that the device is not driven out of memory."""
    x = torch.zeros((4096, 8192), dtype=torch.bfloat16, device="cuda")
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (1 << 20)) / total)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            tw.absmax_quantize(x, granularity=tw.GRAN_ROW)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    q, s = tw.absmax_quantize(x, granularity=tw.GRAN_ROW)
    torch.cuda.synchronize()
    assert not q.any() and s.shape == (4096,)
