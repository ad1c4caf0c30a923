"""GPU parity: every conversion entry point, through the C ABI, bit-exact against the CPU oracle."""
import numpy as np
import pytest
import torch

import paper_2409_16626_b200 as H
import workloads as W
from oracle import hif8_oracle as O

from gpu_util import NP_OF, dev_empty, to_dev, workspace

pytestmark = pytest.mark.gpu

MODES = [H.RND_TA, H.RND_HR, H.RND_SSR, H.RND_TE, H.RND_SR]
FLAGSETS = [0, H.FLAG_SATURATE, H.FLAG_NAN_TO_ZERO, H.FLAG_SATURATE | H.FLAG_NAN_TO_ZERO]


def gpu_encode(src_bits, dtype, offset_in=0, offset_out=0, **kw):
    n = src_bits.size
    if offset_in:
        item = src_bits.dtype.itemsize
        raw = torch.empty(n * item + offset_in + 16, dtype=torch.uint8, device="cuda")
        raw[offset_in:offset_in + n * item] = torch.from_numpy(src_bits.view(np.uint8).copy()).cuda()
        src_ptr, keep = raw.data_ptr() + offset_in, raw
    else:
        keep = to_dev(src_bits)
        src_ptr = keep.data_ptr()
    _, dptr, rb = dev_empty(n, np.uint8, offset_out)
    H.hif8_encode(src_ptr, dtype, dptr, n, **kw)
    torch.cuda.synchronize()
    return rb()


def assert_same(got, want, src=None):
    if not np.array_equal(got, want):
        bad = np.nonzero(got != want)[0]
        i = bad[0]
        msg = f"{bad.size} mismatches; first at {i}: got {got[i]:#x} want {want[i]:#x}"
        if src is not None:
            msg += f" src {src.reshape(-1)[i]:#x}"
        raise AssertionError(msg)


# ----------------------------------------------------------------------------- decode
@pytest.mark.parametrize("dtype", [H.F32, H.BF16, H.F16])
@pytest.mark.parametrize("scale_exp", [0, 5, -7, 126, -126, 20, -20])
def test_decode_all_codes(dtype, scale_exp):
    codes = np.tile(np.arange(256, dtype=np.uint8), 37)[: 256 * 37 - 5]      # several tiles and a ragged tail
    d = to_dev(codes)
    _, ptr, rb = dev_empty(codes.size, NP_OF[dtype])
    H.hif8_decode(d, ptr, dtype, codes.size, scale_exp)
    torch.cuda.synchronize()
    assert_same(rb(), O.decode(codes, dtype, scale_exp))


@pytest.mark.parametrize("dtype", [H.F32, H.BF16, H.F16])
def test_decode_large_random_and_misaligned(dtype):
    codes = W.random_codes(3_000_011, seed=21, finite_only=False)
    want = O.decode(codes, dtype, 3)
    for off_in, off_out in [(0, 0), (3, 0), (0, 4), (1, 2)]:
        raw = torch.empty(codes.size + 32, dtype=torch.uint8, device="cuda")
        raw[off_in:off_in + codes.size] = torch.from_numpy(codes).cuda()
        item = np.dtype(NP_OF[dtype]).itemsize
        _, ptr, rb = dev_empty(codes.size, NP_OF[dtype], off_out * item if off_out else 0)
        H.hif8_decode(raw.data_ptr() + off_in, ptr, dtype, codes.size, 3)
        torch.cuda.synchronize()
        assert_same(rb(), want)


# ----------------------------------------------------------------------------- encode, exhaustive 16-bit
@pytest.mark.parametrize("dtype", [H.BF16, H.F16])
@pytest.mark.parametrize("mode", MODES)
def test_encode_exhaustive_16bit(dtype, mode):
    bits = W.all_u16()
    for flags in FLAGSETS:
        want = O.encode(bits, dtype, 0, mode, flags, seed=1, quick=False)
        assert_same(gpu_encode(bits, dtype, scale_exp=0, rnd=mode, flags=flags, seed=1), want, bits)
    for se in (3, -9, 14, -30, 100, -100, 126, 110):  # the last two bring subnormal BF16 sources into range
        want = O.encode(bits, dtype, se, mode, 0, seed=7, quick=True)
        assert_same(gpu_encode(bits, dtype, scale_exp=se, rnd=mode, seed=7), want, bits)


# ----------------------------------------------------------------------------- encode, FP32
def f32_cases():
    special = np.array([0x00000000, 0x80000000, 0x7F800000, 0xFF800000, 0x7FC00000, 0xFFC00000, 0x7F800001,
                        0xFF800001, 0x7FFFFFFF, 0x00000001, 0x807FFFFF, 0x00800000, 0x7F7FFFFF, 0x47200000,
                        0x471FFFFF, 0x47400000, 0x473FFFFF, 0x34000000, 0x33FFFFFF, 0x34800000, 0x347FFFFF],
                       dtype=np.uint32)
    return {
        "normal": W.normal_f32(1_000_003, seed=1234).view(np.uint32),
        "loguniform": W.loguniform_f32(1_000_003, seed=3456).view(np.uint32),
        "bits": np.concatenate([special, W.random_bits_f32(500_000, seed=9).view(np.uint32)]),
    }


@pytest.mark.parametrize("mode", MODES)
def test_encode_f32(mode):
    for name, bits in f32_cases().items():
        for se, flags in [(0, 0), (0, 3), (7, 0), (-5, 1), (126, 0), (-126, 2), (110, 0)]:
            want = O.encode(bits, O.F32, se, mode, flags, seed=42, quick=True)
            got = gpu_encode(bits, H.F32, scale_exp=se, rnd=mode, flags=flags, seed=42)
            assert_same(got, want, bits)


def test_encode_f32_subnormal_sources_with_large_scale():
    bits = np.concatenate([np.arange(1, 1 << 16, dtype=np.uint32), (np.arange(1 << 12, dtype=np.uint32) << 11) | 0x400,
                           np.arange(0x7F0000, 0x810000, dtype=np.uint32)])
    bits = np.concatenate([bits, bits | 0x80000000]).astype(np.uint32)
    for mode in MODES:
        for se in (126, 120, 104, 103):
            want = O.encode(bits, O.F32, se, mode, 0, seed=3, quick=True)
            assert_same(gpu_encode(bits, H.F32, scale_exp=se, rnd=mode, seed=3), want, bits)


@pytest.mark.parametrize("mode", [H.RND_HR, H.RND_SSR])
@pytest.mark.parametrize("scale_exp", [-126, -40, 0, 3, 60, 126])
def test_encode_f32_thresholds_at_the_edges_of_every_binade(mode, scale_exp):
    # the first and last values of every binade of the scaled magnitude (carries into the next one, the binades below the format's
    # range, overflow), with the source bits that are the threshold at 0, 1, 2, the middle and their largest value
    e = np.arange(1, 255, dtype=np.uint32)[:, None, None]
    top = np.array([0, 1, 2, 255, 256, 257, 509, 510, 511], dtype=np.uint32)[None, :, None] << 14
    low = np.array([0, 1, 2, 3, 8191, 8192, 8193, 16381, 16382, 16383], dtype=np.uint32)[None, None, :]
    bits = ((e << 23) | top | low).reshape(-1)
    bits = np.concatenate([bits, bits | np.uint32(0x80000000)]).astype(np.uint32)
    want = O.encode(bits, O.F32, scale_exp, mode, 0, quick=True)
    assert_same(gpu_encode(bits, H.F32, scale_exp=scale_exp, rnd=mode), want, bits)


@pytest.mark.parametrize("mode", [H.RND_TA, H.RND_SR, H.RND_HR, H.RND_SSR])
def test_encode_ragged_sizes_and_misaligned_pointers(mode):
    base = W.loguniform_f32(5000, seed=5, lo_exp=-26, hi_exp=17).view(np.uint32)
    for n in (1, 3, 4, 15, 16, 17, 1023, 1024, 1025, 4097):
        bits = base[:n]
        want = O.encode(bits, O.F32, 0, mode, 0, seed=11, quick=True)
        for off_in, off_out in [(0, 0), (4, 0), (0, 1), (8, 3)]:
            assert_same(gpu_encode(bits, H.F32, offset_in=off_in, offset_out=off_out, rnd=mode, seed=11), want)
    b16 = W.normal_bf16(4099, seed=6)
    want = O.encode(b16, O.BF16, 2, mode, 0, seed=11, quick=True)
    for off_in, off_out in [(0, 0), (2, 0), (0, 5), (6, 1)]:
        assert_same(gpu_encode(b16, H.BF16, offset_in=off_in, offset_out=off_out, scale_exp=2, rnd=mode, seed=11), want)
    assert H.hif8_encode(0, H.F32, 0, 0) == 0


def test_encode_sizes_around_the_groups_per_block_steps():
    # Large tensors give a block two, three or four groups of vectors (grid-stride) and skip the bounds checks of groups
    # that lie wholly inside the tensor: sizes just below and above each step, with ragged vector and element tails,
    # every element compared
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    wave, per_group = sms * 8, 256 * 4 * 4                    # resident blocks per wave; FP32 elements per group
    base = W.loguniform_f32(1 << 22, seed=77, lo_exp=-26, hi_exp=17).view(np.uint32)
    for groups in (2, 3, 4):
        for n in (groups * wave * per_group - 4099, groups * wave * per_group + 3 * per_group + 1027):
            bits = np.resize(base, n)
            d_src = to_dev(bits)
            for mode in (H.RND_TA, H.RND_HR) + ((H.RND_SR,) if groups == 2 else ()):
                _, dptr, rb = dev_empty(n, np.uint8)
                H.hif8_encode(d_src, H.F32, dptr, n, 3, mode, 0, 21)
                torch.cuda.synchronize()
                assert np.array_equal(rb(), O.encode(bits, O.F32, 3, mode, 0, seed=21, quick=True))
    # the BF16 fake-quant kernels (rounding on the bit pattern) take the same grid rule
    n = 4 * wave * 256 * 4 * 8 + 8 * 1024 + 13
    b16 = np.resize(W.llm_activation_bf16(512, 4096, seed=5).reshape(-1), n)
    d = to_dev(b16)
    for mode in (H.RND_TA, H.RND_HR):
        _, dptr, rb = dev_empty(n, np.uint16)
        H.hif8_fake_quant(d, dptr, H.BF16, n, 0, 4, mode, 0, 9)
        torch.cuda.synchronize()
        assert np.array_equal(rb(), O.fake_quant(b16, O.BF16, 4, mode, 0, seed=9, quick=True))


def test_encode_sr_index_is_the_element_offset():
    # the threshold of element i depends on (seed, i) only: a long tensor and a slice of it differ
    bits = np.full(100_000, np.float32(1.03).view(np.uint32), dtype=np.uint32)
    full = gpu_encode(bits, H.F32, rnd=H.RND_SR, seed=5)
    assert_same(full, O.encode(bits, O.F32, 0, O.SR, 0, seed=5, quick=True))
    assert 0.2 < np.mean(full == full.max()) < 0.3          # F = 0.24
    other = gpu_encode(bits, H.F32, rnd=H.RND_SR, seed=6)
    assert np.any(other != full)


# ----------------------------------------------------------------------------- amax + scale + encode
@pytest.mark.parametrize("dtype", [H.F32, H.BF16, H.F16])
def test_amax_scale_encode_jit_and_delayed(dtype):
    n = 2_000_003
    if dtype == H.F32:
        src = W.normal_f32(n, seed=1234).view(np.uint32).copy()
        src[[5, 77]] = [0x7F800000, 0x7FC00000]              # Inf / NaN do not take part in amax
    elif dtype == H.BF16:
        src = W.llm_activation_bf16(n // 1000 + 1, 1000, seed=2345).reshape(-1)[:n].copy()
        src[[5, 77]] = [0x7F80, 0x7FC1]
    else:
        src = W.normal_f32(n, seed=77, std=3.0).astype(np.float16).view(np.uint16).copy()
        src[[5, 77]] = [0xFC00, 0x7E01]
    ws, wsb = workspace()
    d_src = to_dev(src)
    outs = torch.zeros(4, dtype=torch.int32, device="cuda")
    for target in (14, 3):
        amax, se = O.amax_scale(src, dtype, target)
        for mode in (H.RND_TA, H.RND_HR):
            _, dptr, rb = dev_empty(n, np.uint8)
            H.hif8_amax_scale_encode(d_src, dtype, dptr, n, target, mode, 0, 0, None, outs[0:1], outs[1:2], outs[2:3],
                                     ws, wsb)
            torch.cuda.synchronize()
            o = outs.cpu().numpy()
            assert o[0:1].view(np.float32)[0] == np.float32(amax) and o[1] == se
            assert o[2:3].view(np.float32)[0] == np.float32(2.0) ** se
            assert_same(rb(), O.encode(src, dtype, se, mode, 0, quick=True), src)
    # delayed scaling: exponent given on the device, amax of this tensor still reported
    amax, _ = O.amax_scale(src, dtype, 14)
    d_se = torch.tensor([5], dtype=torch.int32, device="cuda")
    outs.zero_()
    _, dptr, rb = dev_empty(n, np.uint8)
    H.hif8_amax_scale_encode(d_src, dtype, dptr, n, 14, H.RND_TA, 0, 0, d_se, outs[0:1], outs[1:2], outs[2:3], ws, wsb)
    torch.cuda.synchronize()
    o = outs.cpu().numpy()
    assert o[0:1].view(np.float32)[0] == np.float32(amax) and o[1] == 5 and o[2:3].view(np.float32)[0] == 32.0
    assert_same(rb(), O.encode(src, dtype, 5, O.TA, 0, quick=True), src)


@pytest.mark.parametrize("dtype", [H.F32, H.BF16, H.F16])
@pytest.mark.parametrize("mode", MODES)
def test_scaled_conversions_of_small_tensors(dtype, mode):
    """The one-launch form: no, one and several vectors per thread, tails, 1 to 16 blocks and the sizes where their number doubles;
    a source that is not 16-byte aligned takes the general path and gives the same."""
    pv = 4 if dtype == H.F32 else 8
    ws, wsb = workspace()
    outs = torch.zeros(4, dtype=torch.int32, device="cuda")
    for i, n in enumerate([1, pv - 1, pv, 511 * pv + 3, 1024 * pv, 1024 * pv + 1, 1025 * pv, 4096 * pv + 2, 8192 * pv + pv - 1,
                           8193 * pv, 16384 * pv - 1, 16384 * pv + pv - 1, 16385 * pv]):
        if dtype == H.F32:
            src = W.loguniform_f32(n, seed=i, lo_exp=-30, hi_exp=20).view(np.uint32).copy()
        else:
            src = (W.normal_bf16(n, seed=i) if dtype == H.BF16 else W.normal_f32(n, seed=i).astype(np.float16).view(np.uint16)).copy()
        specials = {H.F32: [0x7F800000, 0xFFC00001], H.BF16: [0x7F80, 0xFFC1], H.F16: [0xFC00, 0x7E01]}[dtype]
        if n > 100:
            src[[3, n - 1]] = specials                       # Inf / NaN do not take part in amax
        flags = FLAGSETS[i % 4]
        amax, se = O.amax_scale(src, dtype, 14)
        want, want_fq = O.encode(src, dtype, se, mode, flags, seed=9, quick=True), O.fake_quant(src, dtype, se, mode, flags, seed=9, quick=True)
        d_src = to_dev(src)
        shifted = torch.empty(n * src.itemsize + 16, dtype=torch.uint8, device="cuda")
        shifted[4:4 + n * src.itemsize] = torch.from_numpy(src.view(np.uint8)).cuda()
        for source in (d_src, shifted.data_ptr() + 4):
            _, dptr, rb = dev_empty(n, np.uint8)
            H.hif8_amax_scale_encode(source, dtype, dptr, n, 14, mode, flags, 9, None, outs[0:1], outs[1:2], outs[2:3], ws, wsb)
            torch.cuda.synchronize()
            o = outs.cpu().numpy()
            assert o[0:1].view(np.float32)[0] == np.float32(amax) and o[1] == se and o[2:3].view(np.float32)[0] == np.float32(2.0) ** se
            assert_same(rb(), want, src)
        buf = d_src.clone()
        H.hif8_fake_quant(buf, buf, dtype, n, 1, 14, mode, flags, 9, outs[0:1], outs[1:2], ws, wsb)
        torch.cuda.synchronize()
        o = outs.cpu().numpy()
        assert o[0:1].view(np.float32)[0] == np.float32(amax) and o[1] == se
        assert_same(buf.cpu().numpy().view(NP_OF[dtype]), want_fq, src)


@pytest.mark.parametrize("dtype", [H.F32, H.BF16, H.F16])
@pytest.mark.parametrize("fq,mode", [(0, H.RND_TA), (0, H.RND_HR), (0, H.RND_SR), (1, H.RND_TA), (1, H.RND_HR)])
def test_scaled_conversions_at_the_limits_of_the_launch_forms(dtype, fq, mode):
    """The last size of the one-launch form and the first above it, one cluster of the two-launch form and a little more, its last
    size with fewer and more clusters, its limit and the first size above; the largest element first, last, in the middle and in the tail."""
    pv = 4 if dtype == H.F32 else 8
    one = (1 << 17) if mode == H.RND_SR else (3 << 16) if fq else (1 << 18) if mode != H.RND_TA else (11 << 15) if dtype == H.F32 else (1 << 19)
    two = (24 << 20) // (4 if dtype == H.F32 else 2)
    cluster = 32768 * pv
    sizes = [one, one + 1, 9 * cluster + pv - 1, 18 * cluster, 18 * cluster + pv, two + pv - 1, two + pv]  # (from 19 clusters on they are not doubled)
    ws, wsb = workspace()
    outs = torch.zeros(4, dtype=torch.int32, device="cuda")
    np_t = {H.F32: np.float32, H.BF16: np.uint16, H.F16: np.float16}[dtype]
    for i, n in enumerate(sizes):
        base = W.normal_bf16(n, seed=i) if dtype == H.BF16 else W.normal_f32(n, seed=i).astype(np_t)
        src = base.view(np.uint32 if dtype == H.F32 else np.uint16).copy()
        at = [0, n - 1, n // 2, (n // pv) * pv - 1][i % 4]
        src[at] = {H.F32: 0x42F00000, H.BF16: 0x42F0, H.F16: 0x5780}[dtype]  # 120
        amax, se = O.amax_scale(src, dtype, 14)
        assert amax == 120.0
        d_src = to_dev(src)
        if fq:
            out = torch.empty(n, dtype=torch.int32 if dtype == H.F32 else torch.int16, device="cuda")
            assert H.hif8_fake_quant(d_src, out, dtype, n, 1, 14, mode, 0, 9, outs[0:1], outs[1:2], ws, wsb) == 0
            torch.cuda.synchronize()
            assert_same(out.cpu().numpy().view(src.dtype), O.fake_quant(src, dtype, se, mode, 0, seed=9, quick=True), src)
        else:
            _, dptr, rb = dev_empty(n, np.uint8)
            assert H.hif8_amax_scale_encode(d_src, dtype, dptr, n, 14, mode, 0, 9, None, outs[0:1], outs[1:2], outs[2:3], ws, wsb) == 0
            torch.cuda.synchronize()
            assert_same(rb(), O.encode(src, dtype, se, mode, 0, seed=9, quick=True), src)
        o = outs.cpu().numpy()
        assert o[0:1].view(np.float32)[0] == 120.0 and o[1] == se


def test_amax_alone():
    ws, wsb = workspace()
    out = torch.zeros(1, dtype=torch.float32, device="cuda")
    for dtype, src in [(H.F32, W.loguniform_f32(1_000_003, seed=4).view(np.uint32)), (H.BF16, W.normal_bf16(300_001, seed=5)),
                       (H.F16, W.normal_f32(70_001, seed=6).astype(np.float16).view(np.uint16)),
                       (H.F32, np.array([0x7FC00000, 0xFF800000, 0x80000000], np.uint32))]:
        for _ in range(2):
            H.hif8_amax(to_dev(src), dtype, src.size, out, ws, wsb)
            torch.cuda.synchronize()
            assert float(out.item()) == O.amax_scale(src, dtype, 14)[0]


def test_amax_degenerate_tensors():
    ws, wsb = workspace()
    outs = torch.zeros(4, dtype=torch.int32, device="cuda")
    for src, want_se in [(np.zeros(1000, np.uint32), 0), (np.full(999, 0x7FC00000, np.uint32), 0),
                         (np.full(17, 0x00000003, np.uint32), 126), (np.full(5, 0x7F7FFFFF, np.uint32), 14 - 127)]:
        amax, se = O.amax_scale(src, O.F32, 14)
        assert se == want_se
        _, dptr, rb = dev_empty(src.size, np.uint8)
        H.hif8_amax_scale_encode(to_dev(src), H.F32, dptr, src.size, 14, H.RND_TA, 0, 0, None, outs[0:1], outs[1:2], None,
                                 ws, wsb)
        torch.cuda.synchronize()
        o = outs.cpu().numpy()
        assert o[0:1].view(np.float32)[0] == np.float32(amax) and o[1] == se
        assert_same(rb(), O.encode(src, O.F32, se, O.TA, 0, quick=True))


# ----------------------------------------------------------------------------- fake-quant
@pytest.mark.parametrize("dtype", [H.F32, H.BF16, H.F16])
@pytest.mark.parametrize("mode", MODES)
def test_fake_quant(dtype, mode):
    n = 300_007
    if dtype == H.F32:
        src = np.concatenate([W.loguniform_f32(n, seed=8, lo_exp=-30, hi_exp=20).view(np.uint32),
                              W.random_bits_f32(20_000, seed=10).view(np.uint32)])
    elif dtype == H.BF16:
        src = np.concatenate([W.llm_activation_bf16(301, 1000, seed=2345).reshape(-1), W.all_u16()])
    else:
        src = np.concatenate([W.normal_f32(n, seed=8).astype(np.float16).view(np.uint16), W.all_u16()])
    d_src = to_dev(src)
    for se, flags in [(0, 0), (6, 3), (-3, 0), (125, 0), (-125, 0)]:
        _, dptr, rb = dev_empty(src.size, NP_OF[dtype])
        H.hif8_fake_quant(d_src, dptr, dtype, src.size, 0, se, mode, flags, 9)
        torch.cuda.synchronize()
        assert_same(rb(), O.fake_quant(src, dtype, se, mode, flags, seed=9, quick=True), src)
    # fused amax, in place
    ws, wsb = workspace()
    outs = torch.zeros(2, dtype=torch.int32, device="cuda")
    amax, se = O.amax_scale(src, dtype, 14)
    buf = d_src.clone()
    H.hif8_fake_quant(buf, buf, dtype, src.size, 1, 14, mode, 0, 9, outs[0:1], outs[1:2], ws, wsb)
    torch.cuda.synchronize()
    o = outs.cpu().numpy()
    assert o[0:1].view(np.float32)[0] == np.float32(amax) and o[1] == se
    got = buf.cpu().numpy().view(NP_OF[dtype])
    assert_same(got, O.fake_quant(src, dtype, se, mode, 0, seed=9, quick=True), src)


def test_fake_quant_bf16_standard_sr_many_thresholds_per_pattern():
    # the in-place kernel's standard SR: every BF16 pattern at 32 positions (32 different Philox words each), several
    # scales and seeds, both options; the last positions run through the scalar tail
    src = np.tile(W.all_u16(), 32)[:-3]
    d_src = to_dev(src)
    for se, flags, seed in [(0, 0, 1), (5, 3, 2), (-20, 0, 3), (14, 1, 0xDEADBEEF12345678), (30, 2, 5)]:
        _, dptr, rb = dev_empty(src.size, np.uint16)
        H.hif8_fake_quant(d_src, dptr, H.BF16, src.size, 0, se, H.RND_SR, flags, seed)
        torch.cuda.synchronize()
        assert_same(rb(), O.fake_quant(src, O.BF16, se, O.SR, flags, seed=seed, quick=True), src)


@pytest.mark.parametrize("mode,omode", [(H.RND_TA, O.TA), (H.RND_TE, O.TE), (H.RND_HR, O.HR), (H.RND_SSR, O.SSR), (H.RND_SR, O.SR)])
def test_fake_quant_bf16_in_place_scale_edges_and_tails(mode, omode):
    # the in-place kernel rounds BF16 with per-exponent constants (packed BF16 arithmetic except for round half away):
    # scales at which a constant leaves the BF16 range or subnormal sources come into range, every pattern; then ragged,
    # misaligned pieces
    src = W.all_u16()
    d_src = to_dev(src)
    for se in (14, -30, 100, 101, 104, 111, 112, 120, 122, 126, -100, -105, -110, -120, -126):
        _, dptr, rb = dev_empty(src.size, np.uint16)
        H.hif8_fake_quant(d_src, dptr, H.BF16, src.size, 0, se, mode, 0, 0)
        torch.cuda.synchronize()
        assert_same(rb(), O.fake_quant(src, O.BF16, se, omode, 0, quick=True), src)
    part = W.llm_activation_bf16(7, 1000, seed=5).reshape(-1)
    for n, off in [(1, 0), (7, 0), (8, 0), (9, 2), (1025, 0), (4099, 6), (6999, 2)]:
        piece = part[:n]
        raw = torch.zeros(2 * n + 32, dtype=torch.uint8, device="cuda")
        raw[off:off + 2 * n] = torch.from_numpy(piece.view(np.uint8).copy()).cuda()
        out = torch.zeros(2 * n + 32, dtype=torch.uint8, device="cuda")
        H.hif8_fake_quant(raw.data_ptr() + off, out.data_ptr() + off, H.BF16, n, 0, 5, mode, 3, 0)
        torch.cuda.synchronize()
        got = out[off:off + 2 * n].cpu().numpy().view(np.uint16)
        assert_same(got, O.fake_quant(piece, O.BF16, 5, omode, 3, quick=True), piece)


# ----------------------------------------------------------------------------- full sizes: sampled outputs
def test_config2_full_size():
    # FP32 4096x4096 N(0,1): per-tensor scaled encode + decode, every element (neighbour-pair oracle), and a strided
    # sample plus both ends through the oracle's scan of all 256 codes
    x = W.normal_f32((4096, 4096), seed=1234).reshape(-1)
    n = x.size
    ws, wsb = workspace()
    outs = torch.zeros(4, dtype=torch.int32, device="cuda")
    d_src = to_dev(x)
    codes = torch.empty(n, dtype=torch.uint8, device="cuda")
    back = torch.empty(n, dtype=torch.int32, device="cuda")
    H.hif8_amax_scale_encode(d_src, H.F32, codes, n, 14, H.RND_TA, 0, 0, None, outs[0:1], outs[1:2], outs[2:3], ws, wsb)
    torch.cuda.synchronize()
    amax, se = O.amax_scale(x, O.F32, 14)
    assert int(outs[1]) == se
    H.hif8_decode(codes, back, H.F32, n, se)
    torch.cuda.synchronize()
    got_codes = codes.cpu().numpy()
    want_codes = O.encode(x, O.F32, se, O.TA, 0, quick=True)
    assert_same(got_codes, want_codes)
    assert_same(back.cpu().numpy().view(np.uint32), O.decode(want_codes, O.F32, se))
    idx = np.unique(np.concatenate([np.arange(0, n, 53), np.arange(0, 70000), np.arange(n - 70000, n)]))
    assert_same(got_codes[idx], O.encode(x[idx], O.F32, se, O.TA, 0, quick=False))


def test_f32_full_sweep_all_2_32_patterns():
    # every FP32 encoding, unscaled, round-half-away: 64 slices of 2^26 patterns generated from the index
    n = 1 << 26
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    ar = torch.arange(n, dtype=torch.int64, device="cuda")
    for chunk in range(64):
        first = chunk << 26
        d = (ar + first).to(torch.int32) if first < (1 << 31) else (ar + (first - (1 << 32))).to(torch.int32)
        H.hif8_encode(d, H.F32, out, n, 0, H.RND_TA)
        torch.cuda.synchronize()
        want = O.encode_f32_range(first, n, 0, O.TA, 0, 0, quick=True)
        got = out.cpu().numpy()
        if not np.array_equal(got, want):
            i = int(np.nonzero(got != want)[0][0])
            raise AssertionError(f"pattern {first + i:#010x}: got {got[i]:#x} want {want[i]:#x}")


@pytest.mark.parametrize("mode", [H.RND_HR, H.RND_SSR, H.RND_TE, H.RND_SR])
def test_f32_full_sweep_other_modes(mode):
    # every FP32 encoding of either sign in every other rounding mode, 64 slices of 2^26 patterns
    n = 1 << 26
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    ar = torch.arange(n, dtype=torch.int64, device="cuda")
    for chunk in range(64):
        first = chunk << 26
        d = (ar + first).to(torch.int32) if first < (1 << 31) else (ar + (first - (1 << 32))).to(torch.int32)
        H.hif8_encode(d, H.F32, out, n, 0, mode, 0, 77)
        torch.cuda.synchronize()
        want = O.encode_f32_range(first, n, 0, mode, 0, 77, quick=True)
        got = out.cpu().numpy()
        if not np.array_equal(got, want):
            i = int(np.nonzero(got != want)[0][0])
            raise AssertionError(f"pattern {first + i:#010x}: got {got[i]:#x} want {want[i]:#x}")


@pytest.mark.parametrize("mode", [H.RND_TA, H.RND_HR, H.RND_SSR, H.RND_TE, H.RND_SR])
def test_generated_f32_patterns_sweep_with_both_options(mode):
    # hif8_encode_f32_patterns: the whole FP32 range without a source tensor, here with SATURATE and NaN -> 0 switched on
    # (Section 3: the two options), against the oracle; plus equality with hif8_encode on a slice, wrap-around of the
    # pattern counter, an unaligned destination and a ragged length
    n = 1 << 26
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    omode = {H.RND_TA: O.TA, H.RND_HR: O.HR, H.RND_SSR: O.SSR, H.RND_TE: O.TE, H.RND_SR: O.SR}[mode]
    for chunk in range(64):
        first = chunk << 26
        H.hif8_encode_f32_patterns(first, out, n, 0, mode, 3, 91)
        torch.cuda.synchronize()
        want = O.encode_f32_range(first, n, 0, omode, 3, 91, quick=True)
        got = out.cpu().numpy()
        if not np.array_equal(got, want):
            i = int(np.nonzero(got != want)[0][0])
            raise AssertionError(f"pattern {first + i:#010x}: got {got[i]:#x} want {want[i]:#x}")
    first, m = 0xFFFFFF00, 1003                              # wraps through 0xFFFFFFFF -> 0, scaled, ragged, misaligned
    raw, ptr, readback = dev_empty(m, np.uint8, offset_bytes=3)
    H.hif8_encode_f32_patterns(first, ptr, m, 5, mode, 0, 7)
    bits = ((np.arange(m, dtype=np.uint64) + first) & 0xFFFFFFFF).astype(np.uint32)
    src = to_dev(bits)
    ref = torch.empty(m, dtype=torch.uint8, device="cuda")
    H.hif8_encode(src, H.F32, ref, m, 5, mode, 0, 7)
    torch.cuda.synchronize()
    assert np.array_equal(readback(), ref.cpu().numpy())
    assert np.array_equal(readback(), O.encode(bits, O.F32, 5, omode, 0, seed=7, quick=True))


@pytest.mark.parametrize("rnd", [H.RND_TA, H.RND_HR, H.RND_TE])
@pytest.mark.parametrize("dtype", [H.F32, H.BF16, H.F16])
@pytest.mark.parametrize("groups", [1184, 1185, 1184 * 5 // 4 + 1, 2 * 1184 - 1, 2 * 1184, 5 * 1184 + 3, 10 * 1184 - 5, 14 * 1184])
def test_conversions_whatever_the_number_of_blocks(groups, dtype, rnd):
    # Blocks of a launch come from how often the groups of a tensor fill the device: on both sides of those lines, every code and value is the one
    # that the tensor's pieces, which are one group a block, have; nothing in front of or behind the results is written.
    pv = 4 if dtype == H.F32 else 8
    n = groups * 1024 * pv - 3
    t = {H.F32: torch.float32, H.BF16: torch.bfloat16, H.F16: torch.float16}[dtype]
    gen = torch.Generator(device="cuda").manual_seed(groups)
    x = (torch.randn(n, generator=gen, device="cuda") * 3).to(t)
    x[12345] = 77.0
    exp, amax = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(1, device="cuda")
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    guard, piece = 256, 1000 * 1024 * pv

    def fresh(like):
        return torch.full((n + 2 * guard,), 0x5A, dtype=torch.uint8, device="cuda") if like is None else torch.full((n + 2 * guard,), 9.0, dtype=t, device="cuda")

    def check(out, want):
        assert torch.equal(out[guard:guard + n].view(torch.uint8), want.view(torch.uint8))
        assert bool((out[:guard] == (0x5A if out.dtype == torch.uint8 else 9.0)).all()) and bool((out[guard + n:] == (0x5A if out.dtype == torch.uint8 else 9.0)).all())

    H.hif8_amax(x, dtype, n, amax, ws, 256)
    assert float(amax) == 77.0
    codes, values = torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty(n, dtype=t, device="cuda")
    for scale_exp in (8, None):  # 14 - floor(log2 77) = 8: a given exponent, and the one worked out from the amax
        for a in range(0, n, piece):
            m = min(piece, n - a)
            H.hif8_encode(x[a:], dtype, codes[a:], m, 8, rnd)
            H.hif8_fake_quant(x[a:], values[a:], dtype, m, 0, 8, rnd)
        out, back = fresh(None), fresh(t)
        if scale_exp is None:
            H.hif8_amax_scale_encode(x, dtype, out[guard:], n, 14, rnd, 0, 0, None, amax, exp, None, ws, 256)
            H.hif8_fake_quant(x, back[guard:], dtype, n, 1, 14, rnd, 0, 0, None, None, ws, 256)
            assert int(exp) == 8
        else:
            H.hif8_encode(x, dtype, out[guard:], n, scale_exp, rnd)
            H.hif8_fake_quant(x, back[guard:], dtype, n, 0, scale_exp, rnd)
        check(out, codes)
        check(back, values)
    out = fresh(None)
    amax.zero_()
    H.hif8_amax_scale_encode(x, dtype, out[guard:], n, 14, rnd, 0, 0, exp, amax, None, None, ws, 256)  # encodes with the exponent and measures
    check(out, codes)
    assert float(amax) == 77.0


@pytest.mark.parametrize("dtype", [H.F32, H.BF16, H.F16])
def test_scaled_conversions_in_flight_together_share_a_workspace(dtype):
    # Calls of all launch forms one behind the other in a stream, with one workspace and no wait in between: every result is the one the
    # call gives by itself.
    t = {H.F32: torch.float32, H.BF16: torch.bfloat16, H.F16: torch.float16}[dtype]
    gen = torch.Generator(device="cuda").manual_seed(int(dtype) + 1)
    ws, wsb = workspace()
    calls = []
    for i, n in enumerate([700, 9000, 1_300_001, 150_000, 2_100_000, 2_100_000, 500_003, 40_000, 4_000_000, 1_000_000, 6_500_000, 80_000, 3_000_003, 1_700_000]):
        x = (torch.randn(n + 1, generator=gen, device="cuda") * 2.0 ** (i % 7 - 3)).to(t)
        x[n // 2] = 3.0 * 2.0 ** (i % 9)  # every call has another scale
        src = x[1:] if i == 4 else x[:n]  # (off its alignment: the general path)
        rnd = [H.RND_TA, H.RND_HR, H.RND_SSR, H.RND_TE, H.RND_SR][i % 5]
        calls.append((src, n, rnd, i % 3 == 2, torch.empty(n, dtype=t, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda"),
                      torch.zeros(1, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")))

    def run(c):
        src, n, rnd, fq, values, codes, amax, exp = c
        if fq:
            assert H.hif8_fake_quant(src, values, dtype, n, 1, 14, rnd, 0, 5, amax, exp, ws, wsb) == 0
        else:
            assert H.hif8_amax_scale_encode(src, dtype, codes, n, 14, rnd, 0, 5, None, amax, exp, None, ws, wsb) == 0
        return (values if fq else codes), amax, exp

    alone = []
    for c in calls:
        out = run(c)
        torch.cuda.synchronize()
        alone.append([o.view(torch.uint8).clone() for o in out])
    for order in (range(len(calls)), reversed(range(len(calls)))):
        for c in calls:
            for o in c[4:]:
                o.zero_()
        torch.cuda.synchronize()
        order = list(order)
        outs = {i: run(calls[i]) for i in order}
        torch.cuda.synchronize()
        for i in order:
            for got, want in zip(outs[i], alone[i]):
                assert torch.equal(got.view(torch.uint8), want), (i, calls[i][1:4])


def test_one_launch_form_beside_the_work_of_another_stream():
    # The cluster of a just-in-time call waits for room of its own: it gets it, and its results, while another stream keeps the device busy.
    n = 11 << 15  # the largest the form takes: sixteen blocks of all the shared memory it asks for
    x = torch.randn(n, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    x[n - 2] = -96.0
    big = torch.randn(1 << 25, device="cuda")
    junk = torch.empty_like(big)
    ws, wsb = workspace()
    codes = torch.empty(n, dtype=torch.uint8, device="cuda")
    outs = [(torch.empty(n, dtype=torch.uint8, device="cuda"), torch.zeros(1, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")) for _ in range(20)]
    H.hif8_encode(x, H.F32, codes, n, 14 - 6)
    busy = torch.cuda.Stream()
    torch.cuda.synchronize()
    before = H.hif8_launch_count()
    for _ in range(40):
        H.hif8_fake_quant(big, junk, H.F32, big.numel(), 0, 3, H.RND_HR, stream=busy)
    between = H.hif8_launch_count()
    for out, amax, exp in outs:
        H.hif8_amax_scale_encode(x, H.F32, out, n, 14, H.RND_TA, 0, 0, None, amax, exp, None, ws, wsb)
    assert between - before == 40 and H.hif8_launch_count() - between == 20  # one launch a call
    torch.cuda.synchronize()
    for out, amax, exp in outs:
        assert torch.equal(out, codes) and float(amax) == 96.0 and int(exp) == 8


@pytest.mark.parametrize("dtype", [H.F32, H.BF16, H.F16])
@pytest.mark.parametrize("n", [600_003, 2_600_005])
def test_scaled_conversions_of_middle_sizes_with_specials_in_place_and_misaligned(n, dtype):
    # The two-launch form: the largest magnitude is negative, beside Inf and NaN of either sign, which do not count; fake-quant into its own source;
    # and a destination off its alignment, where a conversion element by element reads the words that the amax launch left.
    sign, inf = {H.F32: (1 << 31, 0x7F800000), H.BF16: (1 << 15, 0x7F80), H.F16: (1 << 15, 0x7C00)}[dtype]
    np_t = {H.F32: np.float32, H.F16: np.float16}.get(dtype)
    src = W.normal_bf16(n, seed=4) if dtype == H.BF16 else W.normal_f32(n, seed=4).astype(np_t).view(NP_OF[dtype])
    src = src.view(NP_OF[dtype]).copy()
    src[n // 3] = sign | {H.F32: 0x42F00000, H.BF16: 0x42F0, H.F16: 0x5780}[dtype]  # -120
    src[[5, n // 2, n - 1, 77]] = inf, sign | inf, inf + 1, sign | (inf + 1)
    amax, se = O.amax_scale(src, dtype, 14)
    assert amax == 120.0
    ws, wsb = workspace()
    outs = torch.zeros(4, dtype=torch.int32, device="cuda")
    for rnd in (H.RND_TA, H.RND_HR):
        for offset in (0, 1):
            outs.zero_()
            _, dptr, rb = dev_empty(n, np.uint8, offset)
            assert H.hif8_amax_scale_encode(to_dev(src), dtype, dptr, n, 14, rnd, 0, 0, None, outs[0:1], outs[1:2], outs[2:3], ws, wsb) == 0
            torch.cuda.synchronize()
            assert_same(rb(), O.encode(src, dtype, se, rnd, 0, quick=True), src)
            assert outs[0:1].view(torch.float32).item() == 120.0 and outs[1].item() == se
        buf = to_dev(src)
        assert H.hif8_fake_quant(buf, buf, dtype, n, 1, 14, rnd, 0, 0, outs[0:1], outs[1:2], ws, wsb) == 0
        torch.cuda.synchronize()
        assert_same(buf.cpu().numpy().view(NP_OF[dtype]), O.fake_quant(src, dtype, se, rnd, 0, quick=True), src)


@pytest.mark.parametrize("rnd", [H.RND_SSR, H.RND_SR])
@pytest.mark.parametrize("dtype", [H.F32, H.BF16, H.F16])
@pytest.mark.parametrize("groups", [1184, 1185, 2 * 1184 + 7, 3 * 1184 + 1, 10 * 1184 - 5, 14 * 1184])
def test_stochastic_conversions_whatever_the_number_of_blocks(groups, dtype, rnd):
    # Random words belong to elements, whichever block converts them: all codes and values are those of the element-by-element path, which a source
    # and destination off their alignment take.
    pv = 4 if dtype == H.F32 else 8
    n = groups * 1024 * pv - 3
    t = {H.F32: torch.float32, H.BF16: torch.bfloat16, H.F16: torch.float16}[dtype]
    shifted = torch.empty(n + 1, dtype=t, device="cuda")
    x = (torch.randn(n, generator=torch.Generator(device="cuda").manual_seed(groups), device="cuda") * 3).to(t)
    x[54321] = -77.0
    shifted[1:] = x
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    amax, exp = torch.zeros(1, device="cuda"), torch.full((1,), 8, dtype=torch.int32, device="cuda")
    state = torch.empty(H.SCALE_STATE_BYTES, dtype=torch.uint8, device="cuda")
    want_codes, want = torch.empty(n + 1, dtype=torch.uint8, device="cuda"), torch.empty(n + 1, dtype=t, device="cuda")
    H.hif8_encode(shifted[1:], dtype, want_codes[1:], n, 8, rnd, 0, 11)
    H.hif8_fake_quant(shifted[1:], want[1:], dtype, n, 0, 8, rnd, 0, 11)
    for call in ("encode", "jit", "measure", "delayed"):
        codes = torch.zeros(n, dtype=torch.uint8, device="cuda")
        amax.zero_()
        if call == "encode":
            H.hif8_encode(x, dtype, codes, n, 8, rnd, 0, 11)
        elif call == "jit":
            H.hif8_amax_scale_encode(x, dtype, codes, n, 14, rnd, 0, 11, None, amax, None, None, ws, 256)
        elif call == "measure":
            H.hif8_amax_scale_encode(x, dtype, codes, n, 14, rnd, 0, 11, exp, amax, None, None, ws, 256)
        else:
            H.hif8_scale_state_init(state, 1)
            H.hif8_delayed_scale_encode(x, dtype, codes, n, rnd, 0, 11, state, 1)  # measures: exponent 8 from the next call on
            H.hif8_delayed_scale_encode(x, dtype, codes, n, rnd, 0, 11, state, 0)
            assert int(state[:4].view(torch.int32)) == 8
        assert torch.equal(codes, want_codes[1:])
        assert call in ("encode", "delayed") or float(amax) == 77.0
    for use_amax in (0, 1):
        back = torch.zeros(n, dtype=t, device="cuda")
        H.hif8_fake_quant(x, back, dtype, n, use_amax, 14 if use_amax else 8, rnd, 0, 11, None, None, ws, 256)
        assert torch.equal(back.view(torch.uint8), want[1:].clone().view(torch.uint8))
