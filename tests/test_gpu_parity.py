"""GPU parity: the CUDA path (through the C ABI) against the CPU oracle on identical seeded inputs.

Bars: dequantized weights and quantized activation codes bit-exact; matmul outputs within
1e-3 relative Frobenius error, both sides rounded to bf16 (accumulating 16-bit products in
FP32 instead of FP64 moves a result across a bf16 rounding boundary only rarely; one such
flip costs 2^-8 relative on one element).
"""
import numpy as np
import pytest
import torch

from oracle import razer_oracle as ro
from paper_2501_04052_b200 import inputs

from _util import (blocks_agree, elementwise_report, oracle_quantized_weights, oracle_reference, rel_fro_bits, rows_with_edge_tiles,
                   sample_rows, to_dev)

pytestmark = pytest.mark.gpu
TOL = 1e-3


@pytest.fixture(scope="module")
def b():
    from paper_2501_04052_b200 import binding
    return binding


def _pack(b, codes, scales, d32, sv_mag=(5.0, 8.0), remap_code=0x8):
    N, K = codes.shape[0], codes.shape[1] * 2
    desc = b.make_desc(N, K, d32, sv_mag=sv_mag, remap_code=remap_code)
    packed = b.razer_pack_layout(desc, to_dev(codes), to_dev(scales))
    return desc, packed


# ------------------------------------------------------------------ dequant (bit-exact)

@pytest.mark.parametrize("N,K,seed", [(1024, 1024, 0), (200, 80, 3), (1, 16, 4), (129, 4160, 5)])
def test_dequant_bit_exact_oracle_quantized(b, N, K, seed):
    w, codes, scales, d32 = oracle_quantized_weights(N, K, seed)
    desc, packed = _pack(b, codes, scales, d32)
    d1 = b.razer_dequant(desc, packed, fp32=False).cpu()
    d2 = b.razer_dequant(desc, packed, fp32=True).cpu().numpy()
    want1 = ro.dequant_d1(codes, scales)
    want2 = ro.dequant_d2(codes, scales, np.float32(d32))
    assert np.array_equal(inputs.bf16_to_bits(d1), ro.f64_to_bf16_bits(want1.astype(np.float64)))
    assert np.array_equal(d2.view(np.uint32), want2.view(np.uint32))


@pytest.mark.parametrize("remap_code", [0x8, 0x0])
@pytest.mark.parametrize("sv_mag", [(5.0, 8.0), (5.0, 7.0), (5.0, 9.0), (2.5, 12.0)])
def test_dequant_bit_exact_random_codes(b, remap_code, sv_mag):
    """Uniform random codes and metadata exercise every special value, both zero codes,
    subnormal scales and zero blocks."""
    N, K = 300, 1104
    codes, scales = inputs.random_codes(N, K, seed=11, scale_lo=0, scale_hi=64, zero_block_frac=0.05)
    codes, scales = codes.numpy(), scales.numpy()
    desc, packed = _pack(b, codes, scales, 0.0123, sv_mag=sv_mag, remap_code=remap_code)
    d1 = b.razer_dequant(desc, packed, fp32=False).cpu()
    d2 = b.razer_dequant(desc, packed, fp32=True).cpu().numpy()
    want1 = ro.dequant_d1(codes, scales, sv_mag=sv_mag, remap_code=remap_code)
    want2 = ro.dequant_d2(codes, scales, np.float32(0.0123), sv_mag=sv_mag, remap_code=remap_code)
    assert np.array_equal(inputs.bf16_to_bits(d1), ro.f64_to_bf16_bits(want1.astype(np.float64)))
    assert np.array_equal(d2.view(np.uint32), want2.view(np.uint32))


# ------------------------------------------------------------------ GEMV / skinny GEMM

def _check_matmul(b, fn, desc, packed, codes, scales, d32, x, rows=None, **kw):
    """Two calls on one workspace must agree bit for bit; the result must meet the relative Frobenius bar and,
    element by element, lie within half a bf16 unit of the exact value plus the FP32 accumulation allowance."""
    op = b.OP_GEMV if fn is b.razer_gemv else b.OP_GEMM
    ws = b.alloc_workspace(desc, x.shape[0], op, "cuda")
    y = fn(desc, packed, x.cuda(), workspace=ws)
    b.razer_workspace_status(ws)            # synchronizes; raises if a device wait gave up
    y2 = fn(desc, packed, x.cuda(), workspace=ws)   # the workspace is left ready for the next call
    b.razer_workspace_status(ws)
    assert torch.equal(y, y2), "second call with the same workspace differs"
    xb = inputs.bf16_to_bits(x)
    if rows is None:
        ref, y64, mag = oracle_reference(xb, codes, scales, np.float32(d32), **kw)
        got = y
    else:
        ref, y64, mag = oracle_reference(xb, codes[rows], scales[rows], np.float32(d32), **kw)
        got = y[:, torch.from_numpy(rows).cuda()]
    err = rel_fro_bits(got, ref)
    assert err <= TOL, f"relative Frobenius error {err:.3e}"
    bad, differ, total = elementwise_report(got, ref, y64, mag)
    print(f"[parity] {tuple(x.shape)} x {tuple(codes.shape)}: rel fro {err:.2e}, {differ} of {total} outputs differ from "
          f"the oracle's bf16, {bad} outside the element-wise bound")
    assert bad == 0, f"{bad} of {total} outputs outside 2^-8 |y| + 2^-20 sum|x w|"
    return err


def test_gemv_config1_student_t(b):
    """Workload config 1: N=K=1024, Student-t x 0.02 weights from seed 0, M=1."""
    w, codes, scales, d32 = oracle_quantized_weights(1024, 1024, 0, outliers=0.0)
    desc, packed = _pack(b, codes, scales, d32)
    x = inputs.activations(1, 1024, 0)
    _check_matmul(b, b.razer_gemv, desc, packed, codes, scales, d32, x)


@pytest.mark.parametrize("N,K", [(4096, 4096), (11008, 4096), (4096, 11008)])
def test_gemv_config2_llama7b_shapes(b, N, K):
    w, codes, scales, d32 = oracle_quantized_weights(N, K, 1)
    desc, packed = _pack(b, codes, scales, d32)
    x = inputs.activations(1, K, 1)
    _check_matmul(b, b.razer_gemv, desc, packed, codes, scales, d32, x)


@pytest.mark.parametrize("M", [1, 2, 3, 4, 7, 16, 33, 64])
def test_gemv_ragged_shapes_random_codes(b, M):
    N, K = 333, 2064                      # N not a multiple of the row tile, K not of the k chunk
    codes, scales = inputs.random_codes(N, K, seed=20 + M, zero_block_frac=0.02)
    codes, scales = codes.numpy(), scales.numpy()
    desc, packed = _pack(b, codes, scales, 0.004)
    x = inputs.activations(M, K, 20 + M)
    _check_matmul(b, b.razer_gemv, desc, packed, codes, scales, 0.004, x)


@pytest.mark.parametrize("compiled", [True, False])
def test_both_ways_into_the_library(b, monkeypatch, compiled):
    """The compiled part of the binding and ctypes: the same results, and what one refuses the other refuses in the same way."""
    if compiled:
        assert b._call is not None
    else:
        monkeypatch.setattr(b, "_call", None)
    N, K = 300, 528
    codes, scales = inputs.random_codes(N, K, seed=5)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.01)
    for M, fn, op in ((3, b.razer_gemv, b.OP_GEMV), (20, b.razer_gemv, b.OP_GEMV), (70, b.razer_gemm, b.OP_GEMM)):
        x, ws = inputs.activations(M, K, M).cuda(), b.alloc_workspace(desc, M, op, "cuda")
        y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
        assert fn(desc, packed, x, y, ws) is y
        assert torch.equal(y, fn(desc, packed, x))                                        # buffers allocated by the binding
        assert torch.equal(y, fn(desc, packed, torch.nn.Parameter(x, requires_grad=False), workspace=ws))
        with torch.cuda.stream(torch.cuda.Stream()):
            other = fn(desc, packed, x, torch.empty_like(y), ws)
            torch.cuda.current_stream().synchronize()
        assert torch.equal(y, other)
        for bad in (x.float(), x[:, :-16], x.t().contiguous().t(), x.cpu()):
            with pytest.raises(AssertionError):
                fn(desc, packed, bad, y, ws)
        with pytest.raises(IndexError):
            fn(desc, packed, x.reshape(-1), y, ws)
        for args, code in (((desc, packed, x, y, ws[:256]), b.ERR_WORKSPACE), ((desc, None, x, y, ws), b.ERR_INVALID_ARG),
                           ((b.make_desc(N, K, -1.0), packed, x, y, ws), b.ERR_INVALID_ARG)):
            with pytest.raises(b.RazerError) as e:
                fn(*args)
            assert e.value.code == code
    xh, yh = inputs.activations(2, K, 9).pin_memory(), torch.empty((2, N), dtype=torch.bfloat16).pin_memory()
    xd, yd, ws = torch.empty((2, K), dtype=torch.bfloat16, device="cuda"), torch.empty((2, N), dtype=torch.bfloat16, device="cuda"), b.alloc_workspace(desc, 2, b.OP_GEMV, "cuda")
    b.razer_gemv_host(desc, packed, xh, yh, xd, yd, ws)
    assert torch.equal(yh, b.razer_gemv(desc, packed, xh.cuda()).cpu())
    with pytest.raises(AssertionError):
        b.razer_gemv_host(desc, packed, xh.cuda(), yh, xd, yd, ws)


@pytest.mark.parametrize("M", [9, 16, 17, 32, 33])
@pytest.mark.parametrize("N,K", [(260, 208), (4200, 256), (1030, 1040), (130, 9232), (2300, 5008)])
def test_gemv_both_decodes_up_to_32_tokens(b, M, N, K):
    """Launches of one item a CTA to some twenty, on either side of where weights are decoded by table rather than in registers."""
    codes, scales = inputs.random_codes(N, K, seed=M + K, scale_lo=0, scale_hi=64, zero_block_frac=0.02)
    codes, scales = codes.numpy(), scales.numpy()
    for sv_mag, remap_code in (((5.0, 8.0), 0x8), ((2.5, 12.0), 0x0)):
        desc, packed = _pack(b, codes, scales, 0.004, sv_mag=sv_mag, remap_code=remap_code)
        _check_matmul(b, b.razer_gemv, desc, packed, codes, scales, 0.004, inputs.activations(M, K, M), rows=sample_rows(N, 200, M), sv_mag=sv_mag,
                      remap_code=remap_code)


def test_compiled_call_takes_plain_arguments_only(b):
    """What the compiled part answers itself, and what it hands on (None)."""
    N, K, M = 300, 528, 3
    codes, scales = inputs.random_codes(N, K, seed=6)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.01)
    x, y, ws = inputs.activations(M, K, 1).cuda(), torch.zeros((M, N), dtype=torch.bfloat16, device="cuda"), b.alloc_workspace(desc, M, b.OP_GEMV, "cuda")
    want = b._matmul(b.lib().razer_gemv, desc, packed, x, None, None, b.OP_GEMV)
    plain = (b._GEMV, b.RazerDesc, desc, packed, x, y, ws)
    assert b._call.matmul(*plain) == 0 and torch.equal(y, want)
    assert b._call.matmul(*plain[:6], ws[:256]) == b.ERR_WORKSPACE

    class Sub(torch.Tensor):
        pass

    class Other(b.RazerDesc):
        pass
    for at, other in ((0, None), (2, None), (2, Other()), (3, None), (4, x.float()), (4, x.cpu()), (4, x.as_subclass(Sub)), (4, x[0]), (4, x[:, :-16]),
                      (5, None), (5, y.as_subclass(Sub)), (5, y.to_sparse()), (6, None), (6, 7)):
        args = list(plain)
        args[at] = other
        assert b._call.matmul(*args) is None, (at, other)
    assert b._call.matmul(*plain[:6]) is None
    # a subclass goes the other way, with the same result
    assert torch.equal(b.razer_gemv(desc, packed, x.as_subclass(Sub), y, ws).as_subclass(torch.Tensor), want)
    xh, yh = x.cpu().pin_memory(), torch.zeros((M, N), dtype=torch.bfloat16).pin_memory()
    host = (b._GEMV_HOST, b.RazerDesc, desc, packed, xh, yh, x, y, ws)
    assert b._call.gemv_host(*host) == 0 and torch.equal(yh, want.cpu())
    for at, other in ((4, x), (5, y), (4, xh.as_subclass(Sub)), (4, torch.tensor(1.0)), (6, None), (8, None)):
        args = list(host)
        args[at] = other
        assert b._call.gemv_host(*args) is None, (at, other)
    for bad in ((x, yh), (xh, y)):
        with pytest.raises(AssertionError):
            b.razer_gemv_host(desc, packed, *bad, x, y, ws)


def test_activations_with_trailing_axes_of_one(b):
    """x's first two axes are its rows and columns; further ones of length one (a view of a caller's layout) change nothing."""
    codes, scales = inputs.random_codes(300, 528, seed=33)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.01)
    x = inputs.activations(3, 528, 33).cuda()
    want = b.razer_gemv(desc, packed, x)
    for view in ((3, 528, 1), (3, 528, 1, 1)):
        assert torch.equal(b.razer_gemv(desc, packed, x.view(view)), want) and torch.equal(b.razer_gemm(desc, packed, x.view(view)), want)


@pytest.mark.parametrize("sv_mag,remap_code", [((5.0, 7.0), 0x8), ((5.0, 9.0), 0x0), ((2.5, 12.0), 0x8)])
def test_gemv_other_special_values(b, sv_mag, remap_code):
    N, K = 256, 1024
    codes, scales = inputs.random_codes(N, K, seed=31)
    codes, scales = codes.numpy(), scales.numpy()
    desc, packed = _pack(b, codes, scales, 0.01, sv_mag=sv_mag, remap_code=remap_code)
    x = inputs.activations(4, K, 31)
    _check_matmul(b, b.razer_gemv, desc, packed, codes, scales, 0.01, x, sv_mag=sv_mag, remap_code=remap_code)


@pytest.mark.parametrize("M,N,K", [(4, 8192, 8192), (16, 8192, 8192), (64, 8192, 8192),
                                   (4, 28672, 8192), (16, 28672, 8192), (4, 8192, 28672), (16, 8192, 28672),
                                   (64, 8192, 28672)])
def test_skinny_config3_full_size_sampled_rows(b, M, N, K):
    """Workload config 3 (skinny GEMM) at full size: random RaZeR codes, a sample of output columns checked
    one by one against the oracle."""
    codes, scales = inputs.random_codes(N, K, seed=40)
    codes, scales = codes.numpy(), scales.numpy()
    desc, packed = _pack(b, codes, scales, 0.002)
    x = inputs.activations(M, K, 40 + M)
    rows = rows_with_edge_tiles(N, 192, 41)
    _check_matmul(b, b.razer_gemv, desc, packed, codes, scales, 0.002, x, rows=rows)


def test_skinny_config3_full_size_every_output(b):
    """M = 64 against 28672 x 8192: every one of the 1.8 M outputs of the full-size launch is compared with the
    oracle (computed in chunks of weight rows), so every CTA stripe and tile boundary is covered."""
    M, N, K = 64, 28672, 8192
    codes, scales = inputs.random_codes(N, K, seed=42)
    codes, scales = codes.numpy(), scales.numpy()
    desc, packed = _pack(b, codes, scales, 0.002)
    x = inputs.activations(M, K, 43)
    _check_matmul(b, b.razer_gemv, desc, packed, codes, scales, 0.002, x)


def test_skinny_config3_oracle_quantized(b):
    w, codes, scales, d32 = oracle_quantized_weights(2048, 8192, 2)
    desc, packed = _pack(b, codes, scales, d32)
    for M in (4, 16, 64):
        x = inputs.activations(M, 8192, 50 + M)
        _check_matmul(b, b.razer_gemv, desc, packed, codes, scales, d32, x)


# ------------------------------------------------------------------ prefill GEMM

@pytest.mark.parametrize("M,N,K", [(256, 512, 1024), (130, 200, 464), (2048, 1024, 4096), (100, 300, 1040),
                                   (128, 640, 2048), (65, 129, 4160)])
def test_gemm_oracle_quantized(b, M, N, K):
    w, codes, scales, d32 = oracle_quantized_weights(N, K, 3, outliers=0.0)
    desc, packed = _pack(b, codes, scales, d32)
    x = inputs.activations(M, K, 60, outlier_channel_frac=0.01)
    _check_matmul(b, b.razer_gemm, desc, packed, codes, scales, d32, x)


@pytest.mark.parametrize("N,K", [(14336, 4096), (4096, 14336)])
def test_gemm_config4_full_size_sampled_rows(b, N, K):
    codes, scales = inputs.random_codes(N, K, seed=70)
    codes, scales = codes.numpy(), scales.numpy()
    desc, packed = _pack(b, codes, scales, 0.002)
    x = inputs.activations(2048, K, 70, outlier_channel_frac=0.01)
    rows = rows_with_edge_tiles(N, 96, 71)
    _check_matmul(b, b.razer_gemm, desc, packed, codes, scales, 0.002, x, rows=rows)


def test_gemm_config4_full_size_every_output(b):
    """M = 2048 against 4096 x 14336 (the shape whose stripes cut every output tile): all 8.4 M outputs."""
    M, N, K = 2048, 4096, 14336
    codes, scales = inputs.random_codes(N, K, seed=72)
    codes, scales = codes.numpy(), scales.numpy()
    desc, packed = _pack(b, codes, scales, 0.002)
    x = inputs.activations(M, K, 73, outlier_channel_frac=0.01)
    _check_matmul(b, b.razer_gemm, desc, packed, codes, scales, 0.002, x)


@pytest.mark.parametrize("M,N,K", [(9, 108, 1344), (9, 137, 64), (17, 672, 3264), (150, 132, 64), (33, 1049, 1904), (33, 3914, 80),
                                   (65, 666, 1920), (65, 2299, 80), (100, 4750, 3376), (100, 5457, 80), (300, 2323, 3456),
                                   (333, 3093, 4704), (150, 4968, 80), (200, 3116, 3392), (512, 3178, 4480), (400, 5620, 80),
                                   (2048, 19000, 80)])
def test_gemm_token_tiles_and_partitions(b, M, N, K):
    """Every token tile of the tcgen05 kernel (16, 32, 64, 96, 128, 192, 256) with tiles that stay on one CTA and tiles cut evenly
    among several CTAs, the two widest in stripes too, as the host picks them for these sizes; ragged in every dimension."""
    codes, scales = inputs.random_codes(N, K, seed=74)
    codes, scales = codes.numpy(), scales.numpy()
    desc, packed = _pack(b, codes, scales, 0.002)
    x = inputs.activations(M, K, 75, outlier_channel_frac=0.01)
    _check_matmul(b, b.razer_gemm, desc, packed, codes, scales, 0.002, x, rows=rows_with_edge_tiles(N, 96, 76))


@pytest.mark.parametrize("M,N,K", [(9, 18962, 784), (17, 19058, 784), (33, 18977, 784), (65, 9731, 4112), (97, 6274, 4112),
                                   (9, 19381, 272), (17, 19681, 272), (33, 19519, 272), (65, 19086, 288), (97, 19109, 336), (129, 19373, 192),
                                   (200, 19098, 384)])
def test_gemm_stripes_and_several_whole_tiles(b, M, N, K):
    """The other partitions: stripes over all SMs that begin and end inside tiles of 4 to 17 items, for each of the five narrower token
    tiles, and two or three whole tiles to a CTA for all seven."""
    codes, scales = inputs.random_codes(N, K, seed=78)
    codes, scales = codes.numpy(), scales.numpy()
    desc, packed = _pack(b, codes, scales, 0.002)
    x = inputs.activations(M, K, 79, outlier_channel_frac=0.01)
    _check_matmul(b, b.razer_gemm, desc, packed, codes, scales, 0.002, x, rows=rows_with_edge_tiles(N, 128, 80))


@pytest.mark.parametrize("M,N,K", [(10, 68, 2272), (10, 20463, 80), (27, 17668, 64), (30, 3999, 10992), (498, 132, 3200), (19, 19597, 80),
                                   (58, 6003, 1008), (37, 21233, 64), (50, 3999, 8208), (80, 5003, 1008), (454, 157, 3184), (124, 9731, 4112),
                                   (255, 21336, 64), (197, 5385, 64), (194, 3379, 3168), (20, 11003, 1040), (129, 19010, 528), (250, 4071, 8208)])
def test_gemm_more_token_tiles_and_partitions(b, M, N, K):
    """Tiles and partitions that the sizes above leave out: 16 and 32 tokens decoded in registers with cut tiles and with several tiles to a CTA, by
    table likewise, 64 to 256 tokens with whole, cut and several tiles, 128 and 192 in stripes."""
    codes, scales = inputs.random_codes(N, K, seed=M, zero_block_frac=0.02)
    codes, scales = codes.numpy(), scales.numpy()
    desc, packed = _pack(b, codes, scales, 0.002)
    x = inputs.activations(M, K, 77, outlier_channel_frac=0.01)
    _check_matmul(b, b.razer_gemm, desc, packed, codes, scales, 0.002, x, rows=rows_with_edge_tiles(N, 96, 76))


def test_gemm_sixteen_tokens_keep_three_partial_sums_apart(b):
    """Up to 16 tokens, three items of 256 columns in a row are summed apart and added up once per tile (a third of the
    additions in a chain).  All weights are 1, and a tile's four items contribute 2^30, 1, 1 + m and -2^30: FP32 sums in one chain
    lose the two in the middle (a unit of 2^30 in FP32 is 128), sums apart lose nothing, so y is exact.  148 row tiles of 1024
    columns stay whole on a CTA each; the 16 rows beyond make a tile whose parts several CTAs hold, some without all three."""
    M, K = 16, 1024
    x = torch.zeros((M, K), dtype=torch.bfloat16)
    x[:, 5], x[:, 256 + 5], x[:, 512 + 5], x[:, 768 + 5] = 2.0 ** 30, 1.0, 1.0 + torch.arange(M), -2.0 ** 30
    want = (2.0 + torch.arange(M)).to(torch.bfloat16).cuda()[:, None]
    for N in (148 * 128, 148 * 128 + 16):
        codes = torch.full((N, K // 2), 0x22, dtype=torch.uint8)              # 1.0
        scales = torch.full((N, K // 16), 0x38, dtype=torch.uint8)            # x 1.0
        desc, packed = _pack(b, codes.numpy(), scales.numpy(), 1.0)
        y = b.razer_gemm(desc, packed, x.cuda())
        if N == 148 * 128:
            assert torch.equal(y, want.expand(M, N))
        x1 = inputs.activations(M, K, 77)
        y1 = b.razer_gemm(desc, packed, x1.cuda())
        ref = x1.double().sum(1)
        assert torch.all((y1.cpu().double() - ref[:, None]).abs() <= 2.0 ** -8 * ref.abs()[:, None] + 2.0 ** -20 * x1.double().abs().sum(1)[:, None])


# ------------------------------------------------------------------ activation quantization / W4A4

@pytest.mark.parametrize("M,K,seed", [(256, 8192, 80), (7, 48, 81), (33, 1040, 82)])
def test_quant_act_bit_exact(b, M, K, seed):
    x = inputs.activations(M, K, seed, outlier_channel_frac=0.01)
    codes, scales, ts = b.razer_quant_act(x.cuda())
    torch.cuda.synchronize()
    want_c, want_s, want_d, dbg = ro.quantize_act(inputs.bf16_to_bits(x), return_debug=True)
    assert np.float32(ts.item()) == want_d
    got_s, got_c = scales.cpu().numpy(), codes.cpu().numpy()
    assert np.array_equal(got_s & 0x7F, want_s & 0x7F)
    # metadata and codes must agree except where the two candidates' errors tie within rounding
    blk_ok, right = blocks_agree(x.float().numpy(), want_d, (got_c, got_s), (want_c, want_s), dbg["near_tie"], 16, ro.SCALE_E4M3_META1, (5.0, 5.0))
    assert np.all(right) and blk_ok.mean() > 0.999
    # the decode kernel inverts the GPU's own codes exactly like the oracle's decoder
    d1 = b.razer_decode_act(codes, scales).cpu()
    want1 = ro.dequant_d1(got_c, got_s, scale_fmt=ro.SCALE_E4M3_META1, sv_mag=(5.0,))
    assert np.array_equal(inputs.bf16_to_bits(d1), ro.f64_to_bf16_bits(want1.astype(np.float64)))


def test_quant_act_given_scale_and_zero_input(b):
    x = inputs.activations(8, 256, 83)
    given = torch.tensor([0.05], dtype=torch.float32)
    codes, scales, ts = b.razer_quant_act(x.cuda(), tensor_scale=given.cuda())
    want_c, want_s, want_d = ro.quantize_act(inputs.bf16_to_bits(x), tensor_scale=np.float32(0.05))
    assert ts.item() == np.float32(0.05)
    assert np.array_equal(scales.cpu().numpy(), want_s) and np.array_equal(codes.cpu().numpy(), want_c)
    z = torch.zeros((4, 64), dtype=torch.bfloat16)
    codes, scales, ts = b.razer_quant_act(z.cuda())
    assert ts.item() == 1.0 and not codes.any() and not scales.any()


@pytest.mark.parametrize("M,K", [(64, 16368), (64, 16384), (129, 8208), (1100, 4096)])
def test_quant_act_computed_scale_large(b, M, K):
    """Below, at and above the size from which the tensor maximum has a launch of its own: the scale is that of Eq. 1, everything
    else is what the same scale gives when it is handed in, and the scratch is zero again; one that was not is reported."""
    x = inputs.activations(M, K, 85).cuda()
    x[M - 1, K - 1] = -37.5 * x.abs().max().float()       # the maximum is the last element
    want = torch.tensor([float(np.float32(x.abs().max().float().item()) / np.float32(448.0 * 6.0))], dtype=torch.float32).cuda()
    for sv in (5.0, 0.0):
        scratch = torch.zeros(2, dtype=torch.int32, device="cuda")
        for _ in range(3):                                # back to back on one scratch
            codes, scales, ts = b.razer_quant_act(x, sv_mag=sv, scratch=scratch)
        assert torch.equal(ts.reshape(-1), want) and not scratch.any()
        for got, given in zip((codes, scales), b.razer_quant_act(x, sv_mag=sv, tensor_scale=want)):
            assert torch.equal(got, given)
    # zeroed buffers: the alignment gap between codes and scale factors belongs to neither
    act, act_given = torch.zeros((2, b.razer_fp4_act_bytes(M, K)), dtype=torch.uint8, device="cuda")
    _, ts = b.razer_quant_act_fp4(x, act_fp4=act, scratch=scratch)
    b.razer_quant_act_fp4(x, tensor_scale=want, act_fp4=act_given)
    assert torch.equal(act, act_given) and torch.equal(ts.reshape(-1), want) and not scratch.any()
    if M * K >= 1 << 20:
        for dirty in (1, 7):
            scratch = torch.tensor([0, dirty], dtype=torch.int32, device="cuda")
            assert torch.isnan(b.razer_quant_act(x, scratch=scratch)[2]).all()


@pytest.mark.parametrize("log2_scale", [None, -80, -58, -50, -40, 0, 80])
@pytest.mark.parametrize("sv_mag", [5.0, 8.0, None])
def test_quant_act_extreme_magnitudes(b, log2_scale, sv_mag):
    """Rows from bf16 subnormals to 2^100, zero blocks among them, against the oracle: the blocks that the kernel's short form
    cannot take go through the plain procedure, with the same decisions.  At the scales -58 to -40 the step alone and the
    largest elements alone are within the short form's range, but the quotient is not (FP32 infinity)."""
    M, K = 60, 272
    x = inputs.activations(M, K, 84).float() * torch.pow(2.0, torch.linspace(-132, 100, M))[:, None]
    x[5, 32:64] = 0.0
    x = x.to(torch.bfloat16)
    ts = None if log2_scale is None else torch.tensor([2.0 ** log2_scale])
    codes, scales, out = b.razer_quant_act(x.cuda(), sv_mag=sv_mag or 0.0, tensor_scale=None if ts is None else ts.cuda())
    with np.errstate(all="ignore"):
        want_c, want_s, want_d, dbg = ro.quantize_act(inputs.bf16_to_bits(x), sv_mag=sv_mag and (sv_mag,), return_debug=True,
                                                      tensor_scale=None if ts is None else np.float32(ts.item()))
    assert np.float32(out.item()) == want_d
    ok = blocks_agree(x.float().numpy(), want_d, (codes.cpu().numpy(), scales.cpu().numpy()), (want_c, want_s), dbg["near_tie"], 16,
                      ro.SCALE_E4M3_META1, sv_mag and (sv_mag, sv_mag))[1]
    assert np.all(ok), np.argwhere(~ok)[:5].tolist()
    # prepared for the FP4 matmul: the same decisions, so a product with the same operand in the interchange format is the same
    if sv_mag is None and ts is not None:
        desc, packed = _pack(b, *(t.numpy() for t in inputs.random_codes(64, K, seed=7)), 0.01)
        act, ats = b.razer_quant_act_fp4(x.cuda(), tensor_scale=ts.cuda())
        assert torch.equal(b.razer_gemm_w4a4_fp4(desc, packed, act, ats, M).view(torch.int16),
                           b.razer_gemm_w4a4(desc, packed, codes, scales, ats, use_native_fp4=True).view(torch.int16))


@pytest.mark.parametrize("block,aware", [(16, False), (16, True), (32, False), (128, True)])
def test_quant_weight_any_alignment(b, block, aware):
    """A weight tensor on a 16-byte boundary that is not a 32-byte one gives what the same tensor gives on a 256-byte boundary."""
    N, K = 131, 384
    w = inputs.student_t_weights(N, K, 9, outlier_frac=0.01).cuda()
    buf = torch.empty(N * K + 4, device="cuda")
    off = buf[4:].view(N, K).copy_(w)
    assert off.data_ptr() % 32 == 16 and w.data_ptr() % 32 == 0
    for got, want in zip(b.razer_quant_weight(off, block=block, scale_aware=aware), b.razer_quant_weight(w, block=block, scale_aware=aware)):
        assert torch.equal(got, want)


@pytest.mark.parametrize("block,aware", [(16, False), (16, True), (64, False), (128, True)])
def test_quant_weight_extreme_magnitudes(b, block, aware):
    """The same for the weight quantizer, at a given tensor scale that puts some rows' steps outside the short form."""
    N, K = 70, 384
    w = inputs.student_t_weights(N, K, 8, outlier_frac=0.01) * torch.pow(2.0, torch.linspace(-140, 100, N))[:, None]
    w[3, 128:256] = 0.0
    for log2_scale in (-70, -58, -50, -40, -4, 70):        # -58 to -40: only the quotient leaves the short form's range
        ts = torch.tensor([2.0 ** log2_scale])
        codes, scales, _ = b.razer_quant_weight(w.cuda(), tensor_scale=ts.cuda(), block=block, scale_aware=aware)
        with np.errstate(all="ignore"):
            quantize = ro.quantize_scale_aware if aware else ro.quantize_weight
            want_c, want_s, _, dbg = quantize(w.numpy(), tensor_scale=np.float32(ts.item()), block=block, return_debug=True)
        ok = blocks_agree(w.numpy(), ts.item(), (codes.cpu().numpy(), scales.cpu().numpy()), (want_c, want_s), dbg["near_tie"], block,
                          ro.SCALE_E3M3_META2, (5.0, 8.0), own_scales=aware)[1]
        assert np.all(ok), (log2_scale, np.argwhere(~ok)[:5].tolist())


@pytest.mark.parametrize("N,K", [(16, 1024), (17, 1040), (31, 2032), (1, 2064), (4737, 512), (4737, 528), (4600, 528), (300, 8192)])
def test_dequant_spans_and_unaligned_output(b, N, K):
    """Widths at and around the chunks that a CTA lays out (four or sixteen, by the tensor's size) or decodes (sixteen) at a time, and
    outputs that are not 16-byte aligned."""
    codes, scales = inputs.random_codes(N, K, seed=12, scale_lo=0, scale_hi=64, zero_block_frac=0.05)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.0123)
    want1 = ro.f64_to_bf16_bits(ro.dequant_d1(codes.numpy(), scales.numpy()).astype(np.float64))
    want2 = ro.dequant_d2(codes.numpy(), scales.numpy(), np.float32(0.0123))
    for off in (0, 1):
        o1 = torch.empty(N * K + 1, dtype=torch.bfloat16, device="cuda")[off:off + N * K]
        o2 = torch.empty(N * K + 1, dtype=torch.float32, device="cuda")[off:off + N * K]
        for out, fp32 in ((o1, 0), (o2, 1)):
            b._check(b.lib().razer_dequant(desc, packed.data_ptr(), out.data_ptr(), fp32, None))
        torch.cuda.synchronize()
        assert np.array_equal(inputs.bf16_to_bits(o1.cpu()).reshape(N, K), want1)
        assert np.array_equal(o2.cpu().numpy().view(np.uint32).reshape(N, K), want2.view(np.uint32))


@pytest.mark.parametrize("offset_bytes", [16, 32, 48])
def test_outputs_aligned_to_16_or_32_bytes(b, offset_bytes):
    """Decoded weights and activations are stored 32 bytes at a time where the output is aligned to that, 16 where not."""
    N, K = 37, 2064
    codes, scales = inputs.random_codes(N, K, seed=13, scale_lo=0, scale_hi=64, zero_block_frac=0.05)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.0123)
    want = {0: b.razer_dequant(desc, packed, fp32=False), 1: b.razer_dequant(desc, packed, fp32=True)}
    for fp32, dtype in ((0, torch.bfloat16), (1, torch.float32)):
        size = 4 if fp32 else 2
        buf = torch.full((N * K + 64,), 7.0, dtype=dtype, device="cuda")
        out = buf[offset_bytes // size:][:N * K]
        b._check(b.lib().razer_dequant(desc, packed.data_ptr(), out.data_ptr(), fp32, None))
        torch.cuda.synchronize()
        assert torch.equal(out.view(N, K), want[fp32])
        assert bool((buf[:offset_bytes // size] == 7).all()) and bool((buf[offset_bytes // size + N * K:] == 7).all())
    ac, as_, _ = b.razer_quant_act(inputs.activations(19, K, 3).cuda())
    ref = b.razer_decode_act(ac, as_)
    buf = torch.full((19 * K + 64,), 7.0, dtype=torch.bfloat16, device="cuda")
    out = buf[offset_bytes // 2:][:19 * K]
    b._check(b.lib().razer_decode_act(ac.data_ptr(), as_.data_ptr(), 19, K, 5.0, out.data_ptr(), None))
    torch.cuda.synchronize()
    assert torch.equal(out.view(19, K), ref) and bool((buf[offset_bytes // 2 + 19 * K:] == 7).all()) and bool((buf[:offset_bytes // 2] == 7).all())


@pytest.mark.parametrize("N,K,seed,sv_mag,remap_code", [(1024, 1024, 0, (5.0, 8.0), 0x8), (200, 80, 3, (5.0, 8.0), 0x8),
                                                         (129, 4160, 5, (5.0, 9.0), 0x0), (300, 528, 6, (2.5, 12.0), 0x8)])
def test_quant_weight_bit_exact(b, N, K, seed, sv_mag, remap_code):
    """GPU weight quantizer against the oracle's (Sec. 4.2: E3M3 block scale, four special values): tensor scale,
    scale codes, metadata and element codes, bit for bit except where two candidates' errors tie within rounding."""
    w = inputs.student_t_weights(N, K, seed, outlier_frac=0.001)
    codes, scales, ts = b.razer_quant_weight(w.cuda(), sv_mag=sv_mag, remap_code=remap_code)
    torch.cuda.synchronize()
    want_c, want_s, want_d, dbg = ro.quantize_weight(w.numpy(), sv_mag=sv_mag, remap_code=remap_code, return_debug=True)
    assert np.float32(ts.item()) == want_d
    got_s, got_c = scales.cpu().numpy(), codes.cpu().numpy()
    assert np.array_equal(got_s & 0x3F, want_s & 0x3F)
    blk_ok, right = blocks_agree(w.numpy(), want_d, (got_c, got_s), (want_c, want_s), dbg["near_tie"], 16, ro.SCALE_E3M3_META2, sv_mag, remap_code)
    assert np.all(right) and blk_ok.mean() > 0.999
    # the GPU's codes go through the pack and dequant kernels like any others
    desc, packed = _pack(b, got_c, got_s, float(ts.item()), sv_mag=sv_mag, remap_code=remap_code)
    d2 = b.razer_dequant(desc, packed, fp32=True).cpu().numpy()
    want2 = ro.dequant_d2(got_c, got_s, np.float32(ts.item()), sv_mag=sv_mag, remap_code=remap_code)
    assert np.array_equal(d2.view(np.uint32), want2.view(np.uint32))
    # and the quantization error is the format's: a few percent of the tensor's norm
    assert np.linalg.norm(d2 - w.numpy()) / np.linalg.norm(w.numpy()) < 0.12


@pytest.mark.parametrize("block", [16, 32, 64, 128])
@pytest.mark.parametrize("sv_mag,remap_code", [((5.0, 8.0), 0x8), ((3.5, 6.5), 0x0), ((2.5, 12.0), 0x8)])
def test_quant_weight_ties_between_candidates(b, block, sv_mag, remap_code):
    """Scaled elements on a grid of eighths: every error is exact in FP32, candidates tie often, and elements sit exactly on the ends of the
    intervals that a special value takes, so codes, signs and special values must be the first minimum's without exception.  Every other row
    saturates its scale code, with elements up to 9.25 steps; a few blocks are zero."""
    N, K = 96, 1152
    gen = torch.Generator().manual_seed(block)
    w = torch.randint(-40, 41, (N, K), generator=gen).float()
    w = torch.where(torch.rand((N, K), generator=gen) < 0.6, torch.round(w / 4) * 4, w)
    w.view(N, -1, block)[:, :, 3] = 48.0                       # block maximum: 6 steps
    w.view(N, -1, block)[1::2, ::2, 5] = -74.0                 # or 9.25
    w.view(N, -1, block)[::7, 1] = 0.0
    w = w / 8
    w[1::2] *= 1.875
    given = torch.tensor([1.0])
    codes, scales, _ = b.razer_quant_weight(w.cuda(), sv_mag=sv_mag, remap_code=remap_code, tensor_scale=given.cuda(), block=block)
    want_c, want_s, _ = ro.quantize_weight(w.numpy(), sv_mag=sv_mag, remap_code=remap_code, tensor_scale=np.float32(1.0), block=block)
    assert np.array_equal(scales.cpu().numpy(), want_s) and np.array_equal(codes.cpu().numpy(), want_c)


def _weights_like(b, got, w, d32, block, sv_mag=(5.0, 8.0), remap_code=0x8):
    """Codes and scale bytes of the GPU against the oracle's at tensor scale d32, near-ties aside."""
    want_c, want_s, _, dbg = ro.quantize_weight(w, sv_mag=sv_mag, remap_code=remap_code, tensor_scale=np.float32(d32), block=block, return_debug=True)
    got_c, got_s = got[0].cpu().numpy(), got[1].cpu().numpy()
    assert np.array_equal(got_s & 0x3F, want_s & 0x3F)
    ok, right = blocks_agree(w, np.float32(d32), (got_c, got_s), (want_c, want_s), dbg["near_tie"], block, ro.SCALE_E3M3_META2, sv_mag, remap_code)
    assert np.all(right), f"{int((~right).sum())} of {right.size} blocks"
    return ok.mean()


@pytest.mark.parametrize("block", [16, 32, 64, 128])
@pytest.mark.parametrize("clip", [0.5, 0.1, 0.01, 1e-4])
def test_quant_weight_given_scale_that_clips(b, block, clip):
    """A tensor scale below the tensor's own: elements go beyond 6 steps, up to the point where every block saturates (0.01) and where the
    short form's bound decides nothing any more (1e-4)."""
    N, K = 130, 2048
    w = inputs.student_t_weights(N, K, 31, outlier_frac=0.001)
    d32 = np.float32(float(w.abs().max()) / 11.25 * clip)
    got = b.razer_quant_weight(w.cuda(), tensor_scale=torch.tensor([float(d32)]).cuda(), block=block)
    assert _weights_like(b, got, w.numpy(), d32, block) > 0.99


@pytest.mark.parametrize("block", [16, 32, 64, 128])
@pytest.mark.parametrize("scale", [2.0**-50, 2.0**45])
def test_quant_weight_far_from_one(b, block, scale):
    """Whole tensors near the ends of the range that the short form takes."""
    w = inputs.student_t_weights(70, 1024, 32, outlier_frac=0.001) * scale
    d32 = ro.quantize_weight(w.numpy(), block=block)[2]
    assert _weights_like(b, b.razer_quant_weight(w.cuda(), block=block), w.numpy(), d32, block) > 0.999


@pytest.mark.parametrize("block,N,K", [(16, 1, 16), (16, 3, 528), (16, 1300, 2048), (32, 1300, 2048), (64, 40, 1088), (128, 1300, 2048), (128, 7, 128)])
@pytest.mark.parametrize("sv_mag,remap_code", [((5.0, 8.0), 0x8), ((2.5, 12.0), 0x0)])
def test_quant_weight_undecided_blocks(b, block, N, K, sv_mag, remap_code):
    """Weights on a coarse grid, where a good part of the blocks is left to the error sums: none, a few and more than a warp at a time, over one
    and over several turns of the grid, some with a NaN or an infinity, some zero.  Steps are powers of two and errors exact, so the first
    minimum is the answer without exception."""
    gen = torch.Generator().manual_seed(N + block)
    w = torch.randint(-12, 13, (N, K), generator=gen).float() / 2
    w.view(N, -1, block)[:, :, 3] = 6.0                        # block maximum: 6 steps of one
    blocks = w.view(-1, block)
    if blocks.shape[0] > 64:
        blocks[5::11] = 0.0
    codes, scales, _ = b.razer_quant_weight(w.cuda(), sv_mag=sv_mag, remap_code=remap_code, tensor_scale=torch.ones(1, device="cuda"), block=block)
    want_c, want_s, _ = ro.quantize_weight(w.numpy(), sv_mag=sv_mag, remap_code=remap_code, tensor_scale=np.float32(1.0), block=block)
    assert np.array_equal(scales.cpu().numpy(), want_s) and np.array_equal(codes.cpu().numpy(), want_c)
    # blocks with a NaN or an infinity leave the others as they are, whichever of a block's lanes holds it
    odd = torch.randint(0, blocks.shape[0], (max(1, blocks.shape[0] // 9),), generator=gen)
    at = torch.randint(0, block, odd.shape, generator=gen)
    blocks[odd, at] = torch.where(torch.rand(odd.shape, generator=gen) < 0.5, float("nan"), float("inf"))
    c2, s2, _ = b.razer_quant_weight(w.cuda(), sv_mag=sv_mag, remap_code=remap_code, tensor_scale=torch.ones(1, device="cuda"), block=block)
    keep = np.ones(blocks.shape[0], bool)
    keep[odd.numpy()] = False
    assert np.array_equal(s2.cpu().numpy().reshape(-1)[keep], want_s.reshape(-1)[keep])
    assert np.array_equal(c2.cpu().numpy().reshape(-1, block // 2)[keep], want_c.reshape(-1, block // 2)[keep])


def test_quant_weight_maxima_back_to_back(b):
    """The quantizer starts up while the maximum ahead of it is still being taken: every call of a stream has its own tensor's scale."""
    gen = torch.Generator().manual_seed(9)
    ws = [torch.randn((n, 4096), generator=gen) * 4.0 ** i for i, n in enumerate((700, 3, 64, 2000))]
    want = [np.float32(np.float32(w.abs().max()) / np.float32(11.25)) for w in ws]
    dev = [w.cuda() for w in ws]
    out = [b.razer_quant_weight(dev[i % 4])[2] for i in range(400)]
    got = torch.cat(out).cpu().numpy()
    assert np.array_equal(got, np.array([want[i % 4] for i in range(400)], dtype=np.float32))


@pytest.mark.parametrize("block", [16, 32, 64, 128])
@pytest.mark.parametrize("sv_mag,remap_code", [((4.5, 8.0), 0x8), ((7.0, 10.0), 0x0), ((5.0, 2.5), 0x8), ((2.5, 5.0), 0x0)])
def test_quant_weight_other_magnitudes_bit_exact(b, block, sv_mag, remap_code):
    """Magnitudes outside the short cut of the usual ones (the first not halfway between FP4 values, or the second below 6): continuous weights,
    near-ties aside, and weights on a grid of eighths at a scale of one, where every error is exact."""
    w = inputs.student_t_weights(129, 1152, 40, outlier_frac=0.001)
    got = b.razer_quant_weight(w.cuda(), sv_mag=sv_mag, remap_code=remap_code, block=block)
    d32 = ro.quantize_weight(w.numpy(), sv_mag=sv_mag, remap_code=remap_code, block=block)[2]
    assert np.float32(got[2].item()) == d32 and _weights_like(b, got, w.numpy(), d32, block, sv_mag, remap_code) > 0.999
    gen = torch.Generator().manual_seed(block)
    w = torch.randint(-40, 41, (96, 1152), generator=gen).float()
    w.view(96, -1, block)[:, :, 3] = 48.0
    w.view(96, -1, block)[::5, 1] = 0.0
    w = w / 8
    codes, scales, _ = b.razer_quant_weight(w.cuda(), sv_mag=sv_mag, remap_code=remap_code, tensor_scale=torch.ones(1, device="cuda"), block=block)
    want_c, want_s, _ = ro.quantize_weight(w.numpy(), sv_mag=sv_mag, remap_code=remap_code, tensor_scale=np.float32(1.0), block=block)
    assert np.array_equal(scales.cpu().numpy(), want_s) and np.array_equal(codes.cpu().numpy(), want_c)


@pytest.mark.parametrize("block", [32, 64, 128])
def test_larger_blocks_quantize_pack_and_multiply(b, block):
    """Block sizes 32 / 64 / 128 (Sec. 5's block-size study, Sec. 4.3's deployment size): the GPU weight quantizer
    against the oracle's bit for bit (near-ties aside), the packed form's dequantization bit-exact, the decode
    GEMV and the tensor-core GEMM within the matmul bars."""
    N, K = 260, 2048
    w = inputs.student_t_weights(N, K, 160 + block, outlier_frac=0.001)
    codes, scales, ts = b.razer_quant_weight(w.cuda(), block=block)
    torch.cuda.synchronize()
    want_c, want_s, want_d, dbg = ro.quantize_weight(w.numpy(), block=block, return_debug=True)
    assert np.float32(ts.item()) == want_d and tuple(scales.shape) == (N, K // block)
    got_s, got_c = scales.cpu().numpy(), codes.cpu().numpy()
    assert np.array_equal(got_s & 0x3F, want_s & 0x3F)
    blk_ok, right = blocks_agree(w.numpy(), want_d, (got_c, got_s), (want_c, want_s), dbg["near_tie"], block, ro.SCALE_E3M3_META2, (5.0, 8.0))
    assert np.all(right) and blk_ok.mean() > 0.999
    desc = b.make_desc(N, K, float(ts.item()), block=block)
    packed = b.razer_pack_layout(desc, codes, scales)
    d2 = b.razer_dequant(desc, packed, fp32=True).cpu().numpy()
    want2 = ro.dequant_d2(got_c, got_s, np.float32(ts.item()), block=block)
    assert np.array_equal(d2.view(np.uint32), want2.view(np.uint32))
    for M, fn in ((1, b.razer_gemv), (40, b.razer_gemv), (130, b.razer_gemm)):
        x = inputs.activations(M, K, 170 + M)
        _check_matmul(b, fn, desc, packed, got_c, got_s, float(ts.item()), x, block=block)


@pytest.mark.parametrize("N,K,seed,sv_mag,block", [(512, 1024, 21, (5.0, 8.0), 16), (200, 2048, 22, (7.0, 10.0), 32),
                                                    (130, 528, 23, (2.5, 5.0), 16)])
def test_quant_weight_scale_aware_bit_exact(b, N, K, seed, sv_mag, block):
    """Scale-aware special-value selection (Eq. 6-7 with the scale of Eq. 2 chosen together with v) on the GPU
    against the oracle's: same scale codes and metadata, same element codes, near-ties aside; the result decodes
    through the unchanged kernels and is no worse than the plain selection's."""
    w = inputs.student_t_weights(N, K, seed, outlier_frac=0.001)
    codes, scales, ts = b.razer_quant_weight(w.cuda(), sv_mag=sv_mag, block=block, scale_aware=True)
    torch.cuda.synchronize()
    want_c, want_s, want_d, dbg = ro.quantize_scale_aware(w.numpy(), sv_mag=sv_mag, block=block, return_debug=True)
    assert np.float32(ts.item()) == want_d
    got_s, got_c = scales.cpu().numpy(), codes.cpu().numpy()
    blk_ok, right = blocks_agree(w.numpy(), want_d, (got_c, got_s), (want_c, want_s), dbg["near_tie"], block, ro.SCALE_E3M3_META2, sv_mag,
                                 own_scales=True)
    assert np.all(right) and blk_ok.mean() > 0.999
    desc = b.make_desc(N, K, float(ts.item()), sv_mag=sv_mag, block=block)
    packed = b.razer_pack_layout(desc, codes, scales)
    d2 = b.razer_dequant(desc, packed, fp32=True).cpu().numpy()
    want2 = ro.dequant_d2(got_c, got_s, np.float32(ts.item()), sv_mag=sv_mag, block=block)
    assert np.array_equal(d2.view(np.uint32), want2.view(np.uint32))
    c0, s0, t0 = b.razer_quant_weight(w.cuda(), sv_mag=sv_mag, block=block)
    plain = ro.dequant_d2(c0.cpu().numpy(), s0.cpu().numpy(), np.float32(t0.item()), sv_mag=sv_mag, block=block)
    e_aware, e_plain = np.linalg.norm(d2 - w.numpy()), np.linalg.norm(plain - w.numpy())
    if max(sv_mag) > 6.0:
        assert e_aware < e_plain
    else:
        assert np.array_equal(got_c, c0.cpu().numpy()) and np.array_equal(got_s, s0.cpu().numpy())
    x = inputs.activations(3, K, seed + 100)
    _check_matmul(b, b.razer_gemv, desc, packed, got_c, got_s, float(ts.item()), x, sv_mag=sv_mag, block=block)


def test_quant_weight_given_scale_and_zero_input(b):
    w = inputs.student_t_weights(16, 256, 7)
    given = torch.tensor([0.01], dtype=torch.float32)
    codes, scales, ts = b.razer_quant_weight(w.cuda(), tensor_scale=given.cuda())
    want_c, want_s, want_d = ro.quantize_weight(w.numpy(), tensor_scale=np.float32(0.01))
    assert ts.item() == np.float32(0.01)
    assert np.array_equal(scales.cpu().numpy(), want_s) and np.array_equal(codes.cpu().numpy(), want_c)
    z = torch.zeros((4, 64), dtype=torch.float32)
    codes, scales, ts = b.razer_quant_weight(z.cuda())
    assert ts.item() == 1.0 and not codes.any() and not scales.any()
    codes, scales, ts = b.razer_quant_weight(z.cuda(), remap_code=0x0)      # the true zero is then code 0x8
    assert ts.item() == 1.0 and bool((codes == 0x88).all()) and not scales.any()
    with pytest.raises(b.RazerError) as e:
        b.razer_quant_weight(w.cuda(), sv_mag=(5.0, 6.0))                   # 6 is an FP4 value, not an allowed special value
    assert e.value.code == b.ERR_UNSUPPORTED


@pytest.mark.parametrize("M,N,K", [(256, 1024, 8192), (17, 200, 464), (8, 300, 2048), (13, 520, 1040)])
def test_w4a4_oracle_quantized(b, M, N, K):
    """Workload config 5, W4A4 (rows of N sampled down to keep the oracle quantizer quick)."""
    w, wc, ws, wd = oracle_quantized_weights(N, K, 4)
    desc, packed = _pack(b, wc, ws, wd)
    x = inputs.activations(M, K, 90, outlier_channel_frac=0.01)
    ac, as_, ats = b.razer_quant_act(x.cuda())
    y = b.razer_gemm_w4a4(desc, packed, ac, as_, ats)
    torch.cuda.synchronize()
    ref = ro.matmul_w4a4(ac.cpu().numpy(), as_.cpu().numpy(), np.float32(ats.item()), wc, ws, np.float32(wd))
    err = rel_fro_bits(y, ref)
    assert err <= TOL, f"relative Frobenius error {err:.3e}"


def _w4a4_native_check(b, desc, packed, wc, ws, wd, ac, as_, ats, rows=None, **kw):
    """Two-pass block-scaled FP4 path against the oracle's W4A4 matmul: relative Frobenius bar and the
    element-wise bound of the other matmul kernels (FP32 accumulation of exact products)."""
    M = ac.shape[0]
    wsb = b.alloc_workspace(desc, M, b.OP_GEMM_W4A4, "cuda")
    y = b.razer_gemm_w4a4(desc, packed, ac, as_, ats, workspace=wsb, use_native_fp4=True)
    b.razer_workspace_status(wsb)
    y2 = b.razer_gemm_w4a4(desc, packed, ac, as_, ats, workspace=wsb, use_native_fp4=True)
    b.razer_workspace_status(wsb)
    assert torch.equal(y, y2), "second call with the same workspace differs"
    acn, asn = ac.cpu().numpy(), as_.cpu().numpy()
    if rows is not None:
        wc, ws, y = wc[rows], ws[rows], y[:, torch.from_numpy(rows).cuda()]
    da = ro.dequant_d1(acn, asn, scale_fmt=ro.SCALE_E4M3_META1, sv_mag=(5.0, 5.0)).astype(np.float64)
    dw = ro.dequant_d1(wc, ws, **kw).astype(np.float64)
    scale = float(np.float32(wd)) * float(np.float32(ats.item()))
    y64 = scale * (da @ dw.T)
    mag = abs(scale) * (np.abs(da) @ np.abs(dw).T)
    ref = ro.f64_to_bf16_bits(y64)
    if kw.get("remap_code", 0x8) == 0x8:            # (the oracle's W4A4 matmul takes one remapped code for both operands)
        assert np.array_equal(ref, ro.matmul_w4a4(acn, asn, np.float32(ats.item()), wc, ws, np.float32(wd),
                                                  sv_mag_w=kw.get("sv_mag", (5.0, 8.0))))
    err = rel_fro_bits(y, ref)
    bad, differ, total = elementwise_report(y, ref, y64, mag)
    print(f"[parity] native FP4 {tuple(ac.shape)} x {tuple(wc.shape)}: rel fro {err:.2e}, {differ} of {total} differ, {bad} out of bound")
    assert err <= TOL and bad == 0


@pytest.mark.parametrize("M,N,K,sv_mag,remap_code", [(256, 512, 8192, (5.0, 8.0), 0x8), (17, 200, 464, (5.0, 8.0), 0x8),
                                                    (130, 300, 2048, (2.5, 12.0), 0x0), (13, 520, 1040, (7.0, 10.0), 0x8),
                                                    (300, 260, 272, (5.0, 8.0), 0x8)])
def test_w4a4_native_fp4_two_pass(b, M, N, K, sv_mag, remap_code):
    """App. D.3: RaZeR weights as B_main + B_comp on the block-scaled FP4 tensor-core path, activations in plain
    NVFP4 (quantized on the GPU with no special value, checked against the oracle's Eq. 1-3)."""
    w = inputs.student_t_weights(N, K, 300 + M, outlier_frac=0.001).numpy()
    wc, ws, wd = ro.quantize_weight(w, sv_mag=sv_mag, remap_code=remap_code)
    desc = b.make_desc(N, K, float(wd), sv_mag=sv_mag, remap_code=remap_code)
    packed = b.razer_pack_layout(desc, torch.from_numpy(wc).cuda(), torch.from_numpy(ws).cuda())
    x = inputs.activations(M, K, 301, outlier_channel_frac=0.01)
    ac, as_, ats = b.razer_quant_act(x.cuda(), sv_mag=0.0)
    torch.cuda.synchronize()
    want_c, want_s, want_d = ro.quantize_act(inputs.bf16_to_bits(x), sv_mag=None)
    assert np.float32(ats.item()) == want_d
    assert np.array_equal(ac.cpu().numpy(), want_c) and np.array_equal(as_.cpu().numpy(), want_s)
    _w4a4_native_check(b, desc, packed, wc, ws, wd, ac, as_, ats, sv_mag=sv_mag, remap_code=remap_code)


@pytest.mark.parametrize("nt,M", [(128, 300), (256, 40), (256, 300)])
def test_w4a4_native_fp4_forced_token_tile(b, monkeypatch, nt, M):
    """Both token-tile widths of the FP4 kernel at token counts the host would give to the other one."""
    monkeypatch.setenv("RAZER_FP4_NT", str(nt))
    N, K = 390, 2320                                                   # ragged row tile, 9.06 stages
    w = inputs.student_t_weights(N, K, 310 + nt, outlier_frac=0.001).numpy()
    wc, ws, wd = ro.quantize_weight(w)
    desc = b.make_desc(N, K, float(wd))
    packed = b.razer_pack_layout(desc, torch.from_numpy(wc).cuda(), torch.from_numpy(ws).cuda())
    x = inputs.activations(M, K, 311, outlier_channel_frac=0.01)
    ac, as_, ats = b.razer_quant_act(x.cuda(), sv_mag=0.0)
    _w4a4_native_check(b, desc, packed, wc, ws, wd, ac, as_, ats)


@pytest.mark.parametrize("M,N,K", [(16, 1000, 1024), (64, 300, 4112), (100, 19000, 336), (2000, 1100, 528), (250, 600, 8208),
                                   (333, 4090, 5520), (140, 260, 80), (2, 16, 16), (9, 18962, 784), (129, 1180, 4320), (129, 9826, 4624),
                                   (129, 9355, 112), (129, 19374, 288)])
def test_w4a4_native_fp4_token_tiles_and_partitions(b, M, N, K):
    """Both token tiles of the FP4 kernel with one or two tiles to a CTA, tiles cut evenly among several, and stripes, as the host
    picks them for these sizes."""
    wc, ws = inputs.random_codes(N, K, seed=99)
    wc, ws = wc.numpy(), ws.numpy()
    desc, packed = _pack(b, wc, ws, 0.002)
    x = inputs.activations(M, K, 99, outlier_channel_frac=0.01)
    ac, as_, ats = b.razer_quant_act(x.cuda(), sv_mag=0.0)
    _w4a4_native_check(b, desc, packed, wc, ws, 0.002, ac, as_, ats, rows=rows_with_edge_tiles(N, 64, 98))


@pytest.mark.parametrize("M,N,K", [(256, 512, 8192), (17, 200, 464), (300, 260, 1040), (130, 390, 2320)])
def test_w4a4_fp4_prepared_operand_matches_the_interchange_route(b, M, N, K):
    """razer_quant_act_fp4 + razer_gemm_w4a4_fp4 (the quantizer writes the tensor core's operand layout itself)
    against razer_quant_act(sv_mag = 0) + razer_gemm_w4a4(use_native_fp4): same tensor scale, bit-identical outputs,
    and the outputs within the matmul bars of the oracle's W4A4 result.  The operand buffer starts as garbage: the
    quantizer has to write its padding too."""
    w = inputs.student_t_weights(N, K, 320 + M, outlier_frac=0.001).numpy()
    wc, ws, wd = ro.quantize_weight(w)
    desc = b.make_desc(N, K, float(wd))
    packed = b.razer_pack_layout(desc, torch.from_numpy(wc).cuda(), torch.from_numpy(ws).cuda())
    x = inputs.activations(M, K, 321, outlier_channel_frac=0.01).cuda()
    ac, as_, ats = b.razer_quant_act(x, sv_mag=0.0)
    wsb = b.alloc_workspace(desc, M, b.OP_GEMM_W4A4, "cuda")
    y_ref = b.razer_gemm_w4a4(desc, packed, ac, as_, ats, workspace=wsb, use_native_fp4=True).clone()
    b.razer_workspace_status(wsb)
    buf = torch.full((b.razer_fp4_act_bytes(M, K),), 0xA5, dtype=torch.uint8, device="cuda")
    act, ats2 = b.razer_quant_act_fp4(x, act_fp4=buf)
    assert ats2.item() == ats.item()
    wsb2 = b.alloc_workspace(desc, M, b.OP_GEMM_W4A4, "cuda")
    y = b.razer_gemm_w4a4_fp4(desc, packed, act, ats2, M, workspace=wsb2)
    b.razer_workspace_status(wsb2)
    assert torch.equal(y, y_ref)
    given = torch.tensor([0.01], dtype=torch.float32, device="cuda")          # a given tensor scale: no grid rendezvous
    act3, ats3 = b.razer_quant_act_fp4(x, tensor_scale=given)
    ac3, as3, _ = b.razer_quant_act(x, sv_mag=0.0, tensor_scale=given)
    y3 = b.razer_gemm_w4a4_fp4(desc, packed, act3, ats3, M, workspace=wsb2)
    y3_ref = b.razer_gemm_w4a4(desc, packed, ac3, as3, ats3, workspace=wsb, use_native_fp4=True)
    assert torch.equal(y3, y3_ref)
    _w4a4_native_check(b, desc, packed, wc, ws, wd, ac, as_, ats)


def test_w4a4_native_fp4_decodes_bit_exactly(b):
    """One-hot NVFP4 activations (code 1.0, block scale 1.0) through the two-pass path: y[m, n] is the tensor
    scale times one decoded weight, exact whatever the accumulation order, so main + comp is checked bit for bit."""
    N, K, TS = 300, 1104, 0.25
    for remap_code, sv_mag, seed in [(0x8, (5.0, 8.0), 211), (0x0, (2.5, 12.0), 212)]:
        codes, scales = inputs.random_codes(N, K, seed=seed, scale_lo=0, scale_hi=64, zero_block_frac=0.05)
        codes, scales = codes.numpy(), scales.numpy()
        want = ro.dequant_d1(codes, scales, sv_mag=sv_mag, remap_code=remap_code).astype(np.float64) * TS
        want_bits = ro.f64_to_bf16_bits(want)
        desc = b.make_desc(N, K, TS, sv_mag=sv_mag, remap_code=remap_code)
        packed = b.razer_pack_layout(desc, torch.from_numpy(codes).cuda(), torch.from_numpy(scales).cuda())
        M = 160                                                        # two token tiles, the second ragged
        wsb = b.alloc_workspace(desc, M, b.OP_GEMM_W4A4, "cuda")
        one = torch.ones(1, dtype=torch.float32, device="cuda")
        got = torch.empty((N, K), dtype=torch.bfloat16, device="cuda")
        as_ = torch.full((M, K // 16), 0x38, dtype=torch.uint8, device="cuda")      # E4M3 1.0 everywhere
        ar = torch.arange(M, device="cuda")
        for k0 in range(0, K, M):
            m = min(M, K - k0)
            ac = torch.zeros((M, K // 2), dtype=torch.uint8, device="cuda")
            kk = k0 + ar[:m]
            ac[ar[:m], kk // 2] = torch.where(kk % 2 == 0, 0x02, 0x20).to(torch.uint8)   # FP4 code of 1.0
            y = b.razer_gemm_w4a4(desc, packed, ac, as_, one, workspace=wsb, use_native_fp4=True)
            got[:, k0:k0 + m] = y[:m].t()
        b.razer_workspace_status(wsb)
        got_bits = inputs.bf16_to_bits(got.cpu())
        g = np.where((got_bits & 0x7FFF) == 0, 0, got_bits)
        wv = np.where((want_bits & 0x7FFF) == 0, 0, want_bits)
        bad = np.argwhere(g != wv)
        assert bad.size == 0, (remap_code, sv_mag, len(bad), bad[:5].tolist())


def test_w4a4_native_fp4_config5_full_size_sampled_rows(b):
    M, N, K = 256, 8192, 8192
    wc, ws = inputs.random_codes(N, K, seed=97)
    wc, ws = wc.numpy(), ws.numpy()
    desc, packed = _pack(b, wc, ws, 0.002)
    x = inputs.activations(M, K, 97, outlier_channel_frac=0.01)
    ac, as_, ats = b.razer_quant_act(x.cuda(), sv_mag=0.0)
    _w4a4_native_check(b, desc, packed, wc, ws, 0.002, ac, as_, ats, rows=sample_rows(N, 128, 98))


def test_w4a4_config5_full_size_sampled_rows(b):
    M, N, K = 256, 8192, 8192
    wc, ws = inputs.random_codes(N, K, seed=95)
    wc, ws = wc.numpy(), ws.numpy()
    desc, packed = _pack(b, wc, ws, 0.002)
    x = inputs.activations(M, K, 95, outlier_channel_frac=0.01)
    ac, as_, ats = b.razer_quant_act(x.cuda())
    y = b.razer_gemm_w4a4(desc, packed, ac, as_, ats)
    torch.cuda.synchronize()
    rows = sample_rows(N, 128, 96)
    ref = ro.matmul_w4a4(ac.cpu().numpy(), as_.cpu().numpy(), np.float32(ats.item()), wc[rows], ws[rows],
                         np.float32(0.002))
    err = rel_fro_bits(y[:, torch.from_numpy(rows).cuda()], ref)
    assert err <= TOL, f"relative Frobenius error {err:.3e}"


@pytest.mark.parametrize("M,N,K", [(2048, 14336, 4096), (64, 11008, 4096), (24, 4096, 11008), (128, 11008, 4096)])
def test_repeated_launches_are_bit_identical(b, M, N, K):
    """The same call repeated many times must return the same bits.  The tcgen05 kernel once let a dequant
    group mistake a weight load that was still in flight for the next load of the same stage (the loads of a
    ring complete in any order, and a group does not watch the stages of the items it skips): about one launch
    in a thousand of the first shape then produced a wrong partial tile at the start of a CTA's stripe."""
    codes, scales = inputs.random_codes(N, K, seed=140)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.002)
    x = inputs.activations(M, K, 141, outlier_channel_frac=0.01).cuda()
    op, fn = (b.OP_GEMV, b.razer_gemv) if M <= 64 else (b.OP_GEMM, b.razer_gemm)
    ws = b.alloc_workspace(desc, M, op, "cuda")
    y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    fn(desc, packed, x, y, ws)
    first = y.clone()
    differing = 0
    for _ in range(1500):
        fn(desc, packed, x, y, ws)
        differing += int(not torch.equal(y, first))
    b.razer_workspace_status(ws)
    assert differing == 0, f"{differing} of 1500 launches differ from the first"
    rows = sample_rows(N, 64, 142)
    ref = ro.matmul_w4a16(inputs.bf16_to_bits(x.cpu()), codes.numpy()[rows], scales.numpy()[rows], np.float32(0.002))
    assert rel_fro_bits(first[:, torch.from_numpy(rows).cuda()], ref) <= TOL


@pytest.mark.parametrize("M,N,K", [(256, 8192, 8192), (2048, 4096, 4096), (100, 11008, 4096)])
def test_repeated_fp4_launches_are_bit_identical(b, M, N, K):
    """The block-scaled FP4 matmul repeated many times on one workspace must return the same bits: three rings, two
    producer warps, sixteen remap warps and partial tiles combined across CTAs leave room for a rare ordering fault."""
    codes, scales = inputs.random_codes(N, K, seed=150)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.002)
    x = inputs.activations(M, K, 151, outlier_channel_frac=0.01).cuda()
    act, ats = b.razer_quant_act_fp4(x)
    ws = b.alloc_workspace(desc, M, b.OP_GEMM_W4A4, "cuda")
    y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    b.razer_gemm_w4a4_fp4(desc, packed, act, ats, M, y=y, workspace=ws)
    first = y.clone()
    differing = 0
    for _ in range(1000):
        b.razer_gemm_w4a4_fp4(desc, packed, act, ats, M, y=y, workspace=ws)
        differing += int(not torch.equal(y, first))
    b.razer_workspace_status(ws)
    assert differing == 0, f"{differing} of 1000 launches differ from the first"


# ------------------------------------------------------------------ host-buffer entry point, errors

@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("M,N,K", [(2, 512, 1024), (40, 300, 528)])
def test_gemv_host_entry_point(b, pinned, M, N, K):
    """Host x in, host y out.  Pinned y takes the kernel's stores directly, pageable y goes through the staging
    buffer; (2, 512, 1024) runs on the register-fragment kernel, (40, 300, 528) on the tcgen05 kernel."""
    codes, scales = inputs.random_codes(N, K, seed=97)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.01)
    x = inputs.activations(M, K, 97)
    y = torch.full((M, N), float("nan"), dtype=torch.bfloat16)
    if pinned:
        x, y = x.pin_memory(), y.pin_memory()
    xs = torch.empty((M, K), dtype=torch.bfloat16, device="cuda")
    ys = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    ws = b.alloc_workspace(desc, M, b.OP_GEMV, "cuda")
    for _ in range(2):
        b.razer_gemv_host(desc, packed, x, y, xs, ys, ws)
        y_dev = b.razer_gemv(desc, packed, x.cuda())
        assert torch.equal(y, y_dev.cpu())
        y.fill_(float("nan"))


@pytest.mark.parametrize("M,N,K,offset", [(1, 300, 528, 0), (2, 300, 528, 4), (64, 256, 2048, 0), (64, 256, 2064, 0)])
def test_gemv_host_routes_of_x(b, M, N, K, offset):
    """x fetched by a kernel, or copied because it is not on a 16-byte boundary or larger than 256 KB; new values in the same host
    buffer on the second call; a status that an earlier call left in the workspace is reported."""
    codes, scales = inputs.random_codes(N, K, seed=99)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.01)
    buf = torch.empty(M * K + offset, dtype=torch.bfloat16).pin_memory()
    x = buf[offset:].view(M, K)
    y = torch.empty((M, N), dtype=torch.bfloat16).pin_memory()
    xs, ys = torch.empty((M, K), dtype=torch.bfloat16, device="cuda"), torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    ws = b.alloc_workspace(desc, M, b.OP_GEMV, "cuda")
    for seed in (99, 100):
        x.copy_(inputs.activations(M, K, seed))
        b.razer_gemv_host(desc, packed, x, y, xs, ys, ws)
        assert torch.equal(y, b.razer_gemv(desc, packed, x.cuda()).cpu())
    ws[:4] = torch.tensor([7, 0, 0, 0], dtype=torch.uint8)
    with pytest.raises(b.RazerError) as e:
        b.razer_gemv_host(desc, packed, x, y, xs, ys, ws)
    assert e.value.code == b.ERR_DEVICE_TIMEOUT and "7" in str(e.value)


_FAILED_CALL_CHECK = r"""
import sys, torch
sys.path.insert(0, sys.argv[1])
from paper_2501_04052_b200 import binding as b, inputs
codes, scales = (t.cuda() for t in inputs.random_codes(256, 256, seed=1))
desc = b.make_desc(256, 256, 0.01)
ws = b.alloc_workspace(desc, 1, b.OP_GEMV, "cuda")
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.stream(torch.cuda.Stream()):
    g.capture_begin()
    try:
        b.razer_workspace_status(ws)          # waits for the stream, which a stream that is being captured refuses
        print("not refused")
    except b.RazerError as e:
        assert e.code == b.ERR_CUDA
    try:
        g.capture_end()
    except Exception:
        pass
packed = b.razer_pack_layout(desc, codes, scales)
d1 = b.razer_dequant(desc, packed, fp32=False)
b.razer_workspace_status(ws)
print("ok")
"""


def test_a_failed_call_is_reported_once():
    """A CUDA error that one call has returned is not found again by the next call's check of its own launch."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _FAILED_CALL_CHECK, root], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr


@pytest.mark.parametrize("which", ["x", "y"])
def test_gemv_host_buffer_pinned_in_part(b, which):
    """Only the first of a buffer's two pages is registered: no kernel may touch the other one.  The call copies instead, which
    either works or is an error of the copy, and the next call is as good as ever."""
    N = K = 4096                                                     # 8 KB of x and of y
    codes, scales = inputs.random_codes(N, K, seed=101)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.01)
    room = torch.empty(3 * 2048 * 2, dtype=torch.bfloat16)
    page = room[(-room.data_ptr() % 4096) // 2:][:4096].view(1, 4096)
    x, y = inputs.activations(1, K, 101).pin_memory(), torch.empty((1, N), dtype=torch.bfloat16).pin_memory()
    xs, ys = torch.empty((1, K), dtype=torch.bfloat16, device="cuda"), torch.empty((1, N), dtype=torch.bfloat16, device="cuda")
    ws = b.alloc_workspace(desc, 1, b.OP_GEMV, "cuda")
    want = b.razer_gemv(desc, packed, x.cuda()).cpu()
    page.copy_(x)
    cudart = torch.cuda.cudart()
    assert page.data_ptr() % 4096 == 0 and int(cudart.cudaHostRegister(page.data_ptr(), 4096, 0)) == 0
    try:
        try:
            b.razer_gemv_host(desc, packed, page if which == "x" else x, page if which == "y" else y, xs, ys, ws)
            assert torch.equal(page if which == "y" else y, want)
        except b.RazerError as e:
            assert e.code == b.ERR_CUDA and "copy" in str(e)
        torch.cuda.synchronize()
        b.razer_gemv_host(desc, packed, x, y, xs, ys, ws)
        assert torch.equal(y, want)
    finally:
        torch.cuda.synchronize()
        cudart.cudaHostUnregister(page.data_ptr())


def test_workspace_too_small_is_an_error(b):
    N, K = 512, 4096
    codes, scales = inputs.random_codes(N, K, seed=98)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.01)
    need = b.razer_workspace_bytes(desc, 1, b.OP_GEMV)
    if need > 256:
        x = inputs.activations(1, K, 98).cuda()
        tiny = torch.empty(256, dtype=torch.uint8, device="cuda")
        with pytest.raises(b.RazerError) as e:
            b.razer_gemv(desc, packed, x, workspace=tiny)
        assert e.value.code == b.ERR_WORKSPACE


def test_one_workspace_serves_all_shapes_and_token_counts_in_turn(b):
    """A workspace prepared once serves any decode calls one after another: what the partial sums of one shape or kernel leave
    behind must not be where another one has its arrival counters.  (66000 rows: more row tiles than the counters of the
    small-batch kernel once took, so that its partial sums lay on the counters of the larger token counts.)"""
    cases, sizes = [], []
    for i, (N, K) in enumerate([(1024, 4096), (66000, 512), (2000, 8192)]):
        codes, scales = inputs.random_codes(N, K, seed=180 + i)
        desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.002)
        for M in (2, 16, 7, 64):
            x = inputs.activations(M, K, 190 + i).cuda()
            cases.append((desc, packed, x, b.razer_gemv(desc, packed, x)))    # a workspace of its own
            sizes.append(b.razer_workspace_bytes(desc, M, b.OP_GEMV))
    ws = torch.empty(max(sizes), dtype=torch.uint8, device="cuda")
    b.razer_workspace_init(ws)
    for step in (1, 5, 7):                                                    # three orders of the twelve calls
        for i in range(len(cases)):
            desc, packed, x, want = cases[(i * step) % len(cases)]
            assert torch.equal(b.razer_gemv(desc, packed, x, workspace=ws), want)
    b.razer_workspace_status(ws)


def test_workspace_sized_for_the_largest_batch(b):
    """Sized once for 512 tokens, a workspace serves every kernel and token tile below, in any order, with unchanged results."""
    N, K = 4096, 4096
    codes, scales = inputs.random_codes(N, K, seed=270)
    desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.002)
    ws = torch.zeros(b.razer_workspace_bytes(desc, 512, b.OP_GEMM), dtype=torch.uint8, device="cuda")
    xs = {M: inputs.activations(M, K, 271).cuda() for M in (512, 200, 1, 96, 16, 333, 128, 8, 33, 160, 64, 24, 256)}
    want = {M: b.razer_gemm(desc, packed, x) for M, x in xs.items()}
    for M in [*xs, *reversed(xs)]:
        assert torch.equal(b.razer_gemm(desc, packed, xs[M], workspace=ws), want[M]), M
    b.razer_workspace_status(ws)


def test_one_workspace_serves_both_w4a4_routes_in_turn(b):
    """The same for the weight-activation matmul: exact route, FP4 route and prepared operand, with M and K falling and rising; what
    one call keeps behind the status word and the counters (partial sums, decoded or re-laid-out activations) is nothing to the
    next, and the status word is the kernels' own after every route."""
    cases, sizes = [], []
    for i, (M, N, K) in enumerate([(256, 8192, 2048), (128, 4096, 8192), (16, 1000, 1040), (300, 390, 2320), (4, 512, 4096), (65, 4096, 4096)]):
        codes, scales = inputs.random_codes(N, K, seed=280 + i)
        desc, packed = _pack(b, codes.numpy(), scales.numpy(), 0.002)
        x = inputs.activations(M, K, 290 + i).cuda()
        exact, plain = b.razer_quant_act(x), b.razer_quant_act(x, sv_mag=0.0)
        act, ats = b.razer_quant_act_fp4(x)
        for fn in (lambda ws, a=(desc, packed, *exact): b.razer_gemm_w4a4(*a, workspace=ws),
                   lambda ws, a=(desc, packed, *plain): b.razer_gemm_w4a4(*a, workspace=ws, use_native_fp4=True),
                   lambda ws, a=(desc, packed, act, ats, M): b.razer_gemm_w4a4_fp4(*a, workspace=ws)):
            cases.append((fn, fn(None)))                                      # a workspace of its own
        sizes.append(b.razer_workspace_bytes(desc, M, b.OP_GEMM_W4A4))
    ws = torch.empty(max(sizes), dtype=torch.uint8, device="cuda")
    b.razer_workspace_init(ws)
    for step in (1, 5, 7, 11):                                                # four orders of the eighteen calls
        for i in range(len(cases)):
            fn, want = cases[(i * step) % len(cases)]
            assert torch.equal(fn(ws), want), (step, i)
            b.razer_workspace_status(ws)
    ws.zero_()
    cases[0][0](ws)                                                           # exact route, M = 256
    assert not ws[:4].any()


def test_weights_written_just_ahead_of_the_matmul_are_seen(b):
    """Stream-ordering contract of the header: the matmul kernels start reading the packed weights before the kernel
    directly ahead of them is known to have finished (programmatic dependent launch).  What is guaranteed: weights
    written by razer_pack_layout or by a device-to-device copy queued directly ahead of the matmul are the ones read.
    Two different tensors go alternately into ONE packed buffer, each time followed at once by the GEMV."""
    N, K = 4096, 4096
    desc = b.make_desc(N, K, 0.002)
    sets, want = [], []
    x = inputs.activations(1, K, 7).cuda()
    ws = b.alloc_workspace(desc, 1, b.OP_GEMV, "cuda")
    for s in range(2):
        c, sc = inputs.random_codes(N, K, seed=400 + s)
        sets.append((c.cuda(), sc.cuda()))
        p = b.razer_pack_layout(desc, *sets[-1])
        want.append(b.razer_gemv(desc, p, x, workspace=ws).clone())
    assert not torch.equal(want[0], want[1])
    packed = torch.empty_like(p)
    y = torch.empty_like(want[0])
    keep = [b.razer_pack_layout(desc, *sets[s]) for s in range(2)]
    bad = 0
    for i in range(300):
        s = i & 1
        if i % 3 == 0:
            packed.copy_(keep[s])                                       # device-to-device copy
        else:
            b.razer_pack_layout(desc, sets[s][0], sets[s][1], packed)   # the library's own writer
        b.razer_gemv(desc, packed, x, y, ws)
        bad += int(not torch.equal(y, want[s]))
    b.razer_workspace_status(ws)
    assert bad == 0, f"{bad} of 300 launches read stale weights"


# ------------------------------------------------------------------ alternative kernels (chosen by environment)

_ALT_KERNEL_CHECK = r"""
import sys, numpy as np, torch
sys.path.insert(0, sys.argv[1])
from oracle import razer_oracle as ro
from paper_2501_04052_b200 import binding as b, inputs
for (M, N, K, seed) in [(1, 1000, 4160, 1), (5, 333, 2064, 2), (16, 640, 1024, 3), (8, 384, 8192, 4), (2, 6000, 1088, 5),
                        (1, 4096, 4096, 6), (3, 8200, 1024, 7), (2, 11008, 2048, 8), (1, 50, 16, 9), (8, 5000, 144, 10)]:
    codes, scales = inputs.random_codes(N, K, seed=seed, scale_lo=0, scale_hi=64, zero_block_frac=0.02)
    codes, scales = codes.numpy(), scales.numpy()
    desc = b.make_desc(N, K, 0.004, sv_mag=(5.0, 9.0))
    packed = b.razer_pack_layout(desc, torch.from_numpy(codes).cuda(), torch.from_numpy(scales).cuda())
    x = inputs.activations(M, K, seed)
    ws = b.alloc_workspace(desc, M, b.OP_GEMV, "cuda")
    y = b.razer_gemv(desc, packed, x.cuda(), workspace=ws)
    b.razer_workspace_status(ws)
    ref = ro.matmul_w4a16(inputs.bf16_to_bits(x), codes, scales, np.float32(0.004), sv_mag=(5.0, 9.0))
    err = ro.rel_frobenius(inputs.bf16_to_bits(y.cpu()), ref)
    assert err <= 1e-3, (M, N, K, err)
print("ok")
"""


@pytest.mark.parametrize("kernel,extra_env", [
    ("umma", {}), ("simt", {}), ("stream", {}),
    # the decode kernel's partitions, each forced on every shape: whole units only / units cut along K and combined
    # through the workspace, with one or two 16-row strips per unit
    ("stream", {"RAZER_STREAM_SPLIT": "0", "RAZER_STREAM_TM": "1"}),
    ("stream", {"RAZER_STREAM_SPLIT": "0", "RAZER_STREAM_TM": "2"}),
    ("stream", {"RAZER_STREAM_SPLIT": "1", "RAZER_STREAM_TM": "1"}),
    ("stream", {"RAZER_STREAM_SPLIT": "1", "RAZER_STREAM_TM": "2"}),
])
def test_alternative_kernels_match_the_oracle(kernel, extra_env):
    """RAZER_KERNEL pins the matmul entry points to one kernel (the tcgen05 kernel, the TMA-fed
    register-fragment kernel wherever it can run (M <= 8), or the CUDA-core kernel) instead of the
    per-shape choice; it is read once per process, so the check runs in a child process."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, RAZER_KERNEL=kernel, **extra_env)
    r = subprocess.run([sys.executable, "-c", _ALT_KERNEL_CHECK, root], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr


@pytest.mark.parametrize("sw,tm,spw,split", [(1, 1, 1, 1), (1, 1, 2, 0), (1, 2, 1, 1), (1, 2, 2, 1), (1, 4, 1, 0), (1, 4, 1, 1),
                                             (2, 1, 1, 0), (2, 1, 2, 1), (2, 2, 1, 1), (2, 2, 2, 0)])
def test_decode_kernel_unit_shapes(sw, tm, spw, split):
    """Every unit shape of the decode kernel (warps along the rows, strips per warp, chunks per warp and stage), each forced on
    shapes that fill no unit, end inside a chunk, and leave stages and pieces ragged."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, RAZER_KERNEL="stream", RAZER_STREAM_SW=str(sw), RAZER_STREAM_TM=str(tm), RAZER_STREAM_SPW=str(spw),
               RAZER_STREAM_SPLIT=str(split))
    r = subprocess.run([sys.executable, "-c", _ALT_KERNEL_CHECK, root], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr


_DEPENDENT_EDGES = r"""
import ctypes, sys, torch
sys.path.insert(0, sys.argv[1])
from paper_2501_04052_b200 import binding as b, inputs
N = K = 1024
codes, scales = (t.cuda() for t in inputs.random_codes(N, K, seed=1))
desc = b.make_desc(N, K, 0.01)
packed = b.razer_pack_layout(desc, codes, scales)
x = inputs.activations(1024, K, 2).cuda()                 # 2^20 elements: the quantizer takes two launches
scratch = torch.zeros(2, dtype=torch.int32, device="cuda")
ws = b.alloc_workspace(desc, 1024, b.OP_GEMM_W4A4, "cuda")
def calls():
    q = b.razer_quant_act(x, sv_mag=0.0, scratch=scratch)
    y = [b.razer_gemm_w4a4(desc, packed, *q, workspace=ws, use_native_fp4=f) for f in (False, True)]
    act, ts = b.razer_quant_act_fp4(x, scratch=scratch)
    y.append(b.razer_gemm_w4a4_fp4(desc, packed, act, ts, 1024, workspace=ws))
    y.append(b.razer_gemv(desc, packed, x[:4], workspace=ws))
    return y
want = calls()
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph(keep_graph=True)
with torch.cuda.graph(g):
    got = calls()
get_edges, graph, n = ctypes.CDLL("libcuda.so.1").cuGraphGetEdges_v2, ctypes.c_void_p(int(g.raw_cuda_graph())), ctypes.c_size_t(0)
assert get_edges(graph, None, None, None, ctypes.byref(n)) == 0 and n.value >= 8
ends, data = [(ctypes.c_void_p * n.value)() for _ in range(2)], (ctypes.c_ubyte * 8 * n.value)()   # data: from port, to port, type
assert get_edges(graph, *ends, data, ctypes.byref(n)) == 0
g.instantiate()
g.replay()
torch.cuda.synchronize()
assert all(torch.equal(a, c) for a, c in zip(got, want))
print(sum(e[2] != 0 for e in data), n.value)
"""


@pytest.mark.parametrize("pdl", ["0", "1"])
def test_dependent_launch_switch(pdl):
    """RAZER_PDL=0 turns programmatic dependent launch off in every kernel: a graph of the calls that use it has ordinary edges only.
    Without it every launch of those calls follows the one ahead by a programmatic edge, and the results are the same."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _DEPENDENT_EDGES, root], env=dict(os.environ, RAZER_PDL=pdl), capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    programmatic, edges = map(int, r.stdout.split())
    assert programmatic == (0 if pdl == "0" else edges), r.stdout


def test_back_to_back_dependent_launches(b):
    """The matmul kernels start their weight stream while the preceding kernel of the stream still runs
    (programmatic dependent launch) and must read activations, workspace and outputs only after it has
    finished.  A chain y1 = W1 x, y2 = W2 y1, y3 = W1 y2 with shared workspace, launched back to back many
    times, is compared with the same chain computed by the oracle."""
    N = K = 2048
    M = 3
    c1, s1 = inputs.random_codes(N, K, seed=131)
    c2, s2 = inputs.random_codes(N, K, seed=132)
    c1, s1, c2, s2 = c1.numpy(), s1.numpy(), c2.numpy(), s2.numpy()
    d1, p1 = _pack(b, c1, s1, 0.002)
    d2, p2 = _pack(b, c2, s2, 0.002)
    x = inputs.activations(M, K, 133)
    ws = b.alloc_workspace(d1, M, b.OP_GEMV, "cuda")
    xd = x.cuda()
    bufs = [torch.empty((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    outs = []
    for rep in range(20):
        b.razer_gemv(d1, p1, xd, bufs[0], ws)
        b.razer_gemv(d2, p2, bufs[0], bufs[1], ws)
        b.razer_gemv(d1, p1, bufs[1], bufs[2], ws)
        outs.append(bufs[2].clone())
    b.razer_workspace_status(ws)
    y1 = ro.matmul_w4a16(inputs.bf16_to_bits(x), c1, s1, np.float32(0.002))
    y2 = ro.matmul_w4a16(y1, c2, s2, np.float32(0.002))
    y3 = ro.matmul_w4a16(y2, c1, s1, np.float32(0.002))
    for o in outs:
        assert torch.equal(o, outs[0]), "a repetition of the chain differs"
    # three chained bf16 roundings: allow a few times the single-product bar
    assert rel_fro_bits(outs[0], y3) <= 5e-3
    assert rel_fro_bits(bufs[0], y1) <= TOL
