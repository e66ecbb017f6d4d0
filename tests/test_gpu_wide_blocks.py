"""The wide rotate-quantize loop (b = 64, 128, 256; symmetric E4M3 and E2M3 codes,
asymmetric E4M3 codes, 8-bit split planes) against the general loop on the same
rows, which writes packed nibbles (and, given clip bounds that never bind, 8-bit
codes): both form every output by the same sums in the same order, so codes,
scales, bounds and rotated rows agree bit for bit (a zero code may be written as
either zero).  Few elements of short rows go to the general loop on both sides; the
last test has enough of them."""
import numpy as np
import pytest
import torch

from paper_2509_24416_gb300 import clq

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
E4M3_INT = {0x00: 0, 0x38: 1, 0x40: 2, 0x44: 3, 0x48: 4, 0x4A: 5, 0x4C: 6, 0x4E: 7, 0x50: 8}


def _lut():
    t = torch.full((256,), 99, dtype=torch.int16)
    for byte, v in E4M3_INT.items():
        t[byte] = v
        t[byte | 0x80] = -v
    return t.to(DEV)


def _nibbles(p):
    lo, hi = (p & 15).to(torch.int16), (p >> 4).to(torch.int16)
    q = torch.stack([lo, hi], dim=2).reshape(p.shape[0], -1)
    return torch.where(q >= 8, q - 16, q)


def _planes(q, K):
    """Integer codes of split planes: bytes of 16 h and of l."""
    lut = torch.full((256,), 9999, dtype=torch.int32)
    for v in range(-128, 129):
        a = abs(v)
        f, x = np.frexp(float(a)) if a else (0.0, 0)
        m = (f * 2 - 1) * 8
        if a and m == int(m):
            lut[((x - 1 + 7) << 3) | int(m) | (0x80 if v < 0 else 0)] = v
    lut[0x00] = lut[0x80] = 0
    v = lut.to(DEV)[q.long()]
    hi, lo = v[:, :K], v[:, K:]
    assert bool((hi % 16 == 0).all()) and int(lo.min()) >= -8 and int(lo.max()) <= 7
    return hi + lo


def _rows(M, K, dtype, seed):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(M, K, generator=g)
    x[:, torch.randperm(K, generator=g)[:3]] *= 40
    x[M // 2] = 0  # a zero row
    x[M - 1, :] = 0
    x[M - 1, K // 3] = -1e-7 if dtype == torch.float16 else -1e-39  # a spike in the subnormals
    if M > 2:
        x[1] = 5.0  # every block sums to one large value and zeros
    return x.to(dtype).to(DEV)


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("b,K", [(64, 64), (64, 192), (64, 1152), (128, 128), (128, 1152), (128, 4736),
                                 (256, 256), (256, 1280), (256, 12288), (128, 16384)])
@pytest.mark.parametrize("M", [1, 7, 300])
def test_wide_equals_general(b, K, M, dtype):
    X = _rows(M, K, dtype, b + K + M)
    perm = torch.randperm(K, generator=torch.Generator().manual_seed(K)).to(torch.int32).to(DEV)
    shifted = torch.empty(K + 1, dtype=torch.int32, device=DEV)[1:].copy_(perm)  # 4-byte aligned
    wide = torch.zeros(M, K + 8, dtype=dtype, device=DEV)
    wide[:, :K] = X
    lut = _lut()
    want, s_want, rot_want = clq.rotate_quant_act(X, perm, b, with_rot=True)
    want = _nibbles(want)
    a_want, d_want, l_want = clq.rotate_quant_act_asym(X, perm, b, codes=clq.CLQ_CODES_INT4_PACKED)
    a_want = _nibbles(a_want)
    for p in (perm, shifted):
        for x in (X, wide[:, :K]):
            q, s = clq.rotate_quant_act(x, p, b, clq.CLQ_CODES_E4M3)
            assert torch.equal(lut[q.long()], want) and torch.equal(s, s_want)
            q, d, lo = clq.rotate_quant_act_asym(x, p, b)
            assert torch.equal(lut[q.long()], a_want)
            assert torch.equal(d, d_want) and torch.equal(lo, l_want)
            if K % 128 == 0:
                q, s = clq.rotate_quant_act(x, p, b, clq.CLQ_CODES_E2M3)
                packed = clq.convert_codes(q, K, clq.CLQ_CODES_INT4_PACKED)
                assert torch.equal(_nibbles(packed), want) and torch.equal(s, s_want)
    # 8-bit symmetric codes: weight preparation with a clip takes the general loop
    S8 = clq.CLQ_CODES_E4M3_SPLIT
    clip = torch.full((M,), 3e38, device=DEV)
    q8_want, s8_want, rot8 = clq.prepare_weights(X, perm, b, clip=clip, codes=S8, with_rot=True)
    assert torch.equal(rot8, rot_want)
    v8_want = _planes(q8_want, K)
    for p in (perm, shifted):
        q8, s8 = clq.rotate_quant_act(wide[:, :K], p, b, S8)
        assert torch.equal(s8, s8_want)
        assert torch.equal(_planes(q8, K), v8_want)
    qa, da, la = clq.rotate_quant_act_asym(X, perm, b, codes=S8)
    x64 = rot_want.double()
    lo, span = x64.amin(1, keepdim=True), x64.amax(1, keepdim=True) - x64.amin(1, keepdim=True)
    ratio = torch.where(span > 0, (x64 - lo) / span.clamp(min=1e-300) * 255, torch.zeros_like(x64))
    codes = _planes(qa, K).double() + 128
    assert torch.equal(la, l_want)
    # delta: 2 ulp (2.5e-7), or one step 2^-149 of the subnormal grid, times 255
    assert bool(((da.double() * 255 - span[:, 0]).abs()
                 <= 2.5e-7 * span[:, 0] + 255 * 2.0 ** -149).all())
    # 8-bit ratios reach 255: fp32 keeps them within 1e-4 (tests/parity_utils.py)
    assert bool(((codes - ratio).abs() <= 0.5 + 1e-4).all())
    q, s, rot = clq.rotate_quant_act(X, perm, b, clq.CLQ_CODES_E4M3, with_rot=True)
    assert torch.equal(rot, rot_want) and torch.equal(lut[q.long()], want)
    assert clq.device_status() == 0
    assert np.isfinite(s.cpu().numpy()).all()


def _small_rows(M, K, b, spans, seed):
    """bf16 rows whose rotated values span about spans[i % len(spans)]."""
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(M, K, generator=g, dtype=torch.float64)
    s = torch.tensor(spans, dtype=torch.float64)[torch.arange(M) % len(spans)]
    return (x * (s / (7 * b ** 0.5))[:, None]).to(torch.bfloat16).to(DEV)


@pytest.mark.parametrize("b,K", [(32, 1152), (64, 1152), (128, 1152), (256, 1280)])
def test_asym_small_spans(b, K):
    """Asymmetric codes of rows whose span is normal but so small that (2^n - 1) /
    span passes the largest float (spans below 4.4e-38 with 4 bits, 7.5e-37 with 8),
    and of rows around that range, in both loops."""
    X = _small_rows(64, K, b, [1.3e-38, 2e-38, 4e-38, 5e-38, 1e-37, 3e-37, 7e-37, 8e-37, 3e-36], b)
    perm = torch.randperm(K, generator=torch.Generator().manual_seed(K)).to(torch.int32).to(DEV)
    lut = _lut()
    for codes, bits in ((clq.CLQ_CODES_INT4_PACKED, 4), (clq.CLQ_CODES_E4M3, 4),
                        (clq.CLQ_CODES_E4M3_SPLIT, 8)):
        q, d, lo, rot = clq.rotate_quant_act_asym(X, perm, b, codes=codes, with_rot=True)
        x64 = rot.double()
        span = x64.amax(1, keepdim=True) - x64.amin(1, keepdim=True)
        small = (2 ** bits - 1) * 2.0 ** -128  # below: the reciprocal's product overflows
        assert bool(((span > 2.0 ** -126) & (span < small)).any())
        assert bool((span > small).any())
        got = (_nibbles(q) if codes == clq.CLQ_CODES_INT4_PACKED else
               lut[q.long()] if codes == clq.CLQ_CODES_E4M3 else _planes(q, K)).double()
        ratio = (x64 - x64.amin(1, keepdim=True)) / span * (2 ** bits - 1)
        # a quotient and its product with 2^n - 1: fp32 keeps ratios up to 255 within 1e-4
        assert bool(((got + 2 ** (bits - 1) - ratio).abs() <= 0.5 + 1e-4).all())
        assert torch.equal(lo.double(), x64.amin(1))
        # as above: 2 ulp, or one step of the subnormal grid
        assert bool(((d.double() * (2 ** bits - 1) - span[:, 0]).abs()
                     <= 2.5e-7 * span[:, 0] + (2 ** bits - 1) * 2.0 ** -149).all())
    assert clq.device_status() == 0


@pytest.mark.parametrize("b,K", [(64, 4736), (128, 4736), (256, 1280)])
def test_split_subnormal_scales(b, K):
    """8-bit codes of rows with a subnormal scale (|x| up to 127 * 2^-126 = 1.5e-36):
    the nearest integer to the fp32 quotient by that scale, in the general loop
    (reached through a clip that never binds) and in the wide one."""
    M = 300
    X = _small_rows(M, K, b, [1e-38, 1e-37, 5e-37, 1e-36], K)
    perm = torch.randperm(K, generator=torch.Generator().manual_seed(b)).to(torch.int32).to(DEV)
    S8 = clq.CLQ_CODES_E4M3_SPLIT
    q, s, rot = clq.rotate_quant_act(X, perm, b, S8, with_rot=True)
    assert bool(((s > 0) & (s < 2.0 ** -126)).all())
    want = torch.round((rot.double() / s.double()[:, None]).float()).to(torch.int32)
    assert torch.equal(_planes(q, K), want)
    clip = torch.full((M,), 3e38, device=DEV)
    q, s_want = clq.prepare_weights(X, perm, b, clip=clip, codes=S8)
    assert torch.equal(s, s_want) and torch.equal(_planes(q, K), want)
    assert clq.device_status() == 0


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("b,K,M", [(64, 1152, 700), (128, 128, 5000), (128, 1152, 700),
                                   (256, 256, 2500), (256, 1280, 700)])
def test_wide_equals_general_many_rows(b, K, M, dtype):
    """Short rows, which the wide loop takes from some 600 thousand elements on in every
    layout (fewer go to the general loop)."""
    test_wide_equals_general(b, K, M, dtype)
