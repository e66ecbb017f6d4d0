"""The GEMM at the edges of its tiles: CTA pairs share 256-row tiles, 256, 192,
128 or 64 columns wide, each warp storing 32 x 32 blocks (N % 8 == 0) or
copying them out by column pairs.  Rows and columns one below, at and one above
those sizes, in every execution layout, against the oracle: accumulators bit for
bit, outputs within half an ulp of the output format plus the fp32 epilogue's
rounding (tests/parity_utils.py)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_24416_gb300 import clq
from parity_utils import check_output_elementwise

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
SETTINGS = {"e4m3": (4, 4, None), "e2m3": (4, 4, clq.CLQ_CODES_E2M3), "w4a8": (8, 4, None),
            "w8a8": (8, 8, None)}


def _values(t, layout, K):
    """Integer codes of an array, through the library-independent E4M3 table."""
    e4m3 = {0x00: 0, 0x80: 0}
    for v in range(1, 129):
        f, x = np.frexp(float(v))
        m = (f * 2 - 1) * 8
        if m == int(m):
            e4m3[((x - 1 + 7) << 3) | int(m)] = v
            e4m3[((x - 1 + 7) << 3) | int(m) | 0x80] = -v
    lut = np.full(256, 999, np.int64)
    for k, v in e4m3.items():
        lut[k] = v
    q = lut[t.cpu().numpy()]
    assert np.abs(q).max() <= 128
    return q if layout == clq.CLQ_CODES_E4M3 else q[:, :K] + q[:, K:]


@pytest.mark.parametrize("setting", sorted(SETTINGS))
@pytest.mark.parametrize("M,N,K", [(1, 1, 128), (127, 31, 128), (129, 33, 384), (255, 191, 256),
                                   (257, 193, 128), (256, 255, 1152), (300, 257, 128), (31, 1003, 256),
                                   (128, 192, 896), (385, 250, 256)])
def test_tile_edges(setting, M, N, K):
    a_bits, w_bits, w_codes = SETTINGS[setting]
    dtype = "f16" if (M + N) % 2 == 0 else "bf16"
    td = torch.float16 if dtype == "f16" else torch.bfloat16
    g = torch.Generator().manual_seed(M * 7919 + N * 31 + K)
    b = 128
    X = torch.randn(M, K, generator=g).to(td).to(DEV)
    W = (0.05 * torch.randn(N, K, generator=g)).to(td).to(DEV)
    bias = torch.randn(N, generator=g).to(td).to(DEV) if N % 3 else None
    perm = torch.randperm(K, generator=g).to(torch.int32).to(DEV)
    layer = clq.PreparedLinear.from_weight(W, perm, b, bias=bias, a_bits=a_bits, w_bits=w_bits,
                                           w_codes=w_codes)
    Xq, s_x = clq.rotate_quant_act(X, perm, b, layer.act_codes)
    # one guard row behind Y: nothing may be written past the last row
    buf = torch.full(((M + 1) * N,), 7.0, dtype=td, device=DEV)
    Y, acc = clq.linear(Xq, s_x, layer.We, layer.s_w, b, K, bias, out_dtype=td,
                        Y=buf[:M * N].view(M, N), with_acc=True)
    assert clq.device_status() == 0
    assert bool((buf[M * N:] == 7.0).all())
    we = layer.We if w_codes is None else clq.convert_codes(layer.We, K, clq.CLQ_CODES_E4M3)
    xe = Xq if w_codes is None else clq.convert_codes(Xq, K, clq.CLQ_CODES_E4M3)
    qx = _values(xe, clq.codes_layout(xe, K), K)
    qw = _values(we, clq.codes_layout(we, K), K)
    want = oracle.int_gemm(qx, qw)
    assert np.array_equal(acc.cpu().numpy().astype(np.int64), want)
    sx, sw = s_x.cpu().numpy(), layer.s_w.cpu().numpy()
    bb = None if bias is None else bias.float().cpu().numpy()
    y64 = want * sx.astype(np.float64)[:, None] * sw.astype(np.float64)[None, :] / b
    if bb is not None:
        y64 = y64 + bb[None, :]
    check_output_elementwise(Y.float().cpu().numpy(), y64, want, sx, sw, b, bb, dtype)


@pytest.mark.parametrize("setting", sorted(SETTINGS) + ["asym"])
@pytest.mark.parametrize("M,N,K", [(4001, 2051, 1152), (2600, 2504, 896), (4601, 1501, 1152),
                                   (300, 8195, 256)])
def test_tile_widths(setting, M, N, K):
    """Shapes for which the launcher takes 256, 128, 192 and 64 columns (where the
    setting has them), several tiles a unit, against fp64 products of the codes on
    the GPU (integers, so exact)."""
    a_bits, w_bits, w_codes = SETTINGS.get(setting, (4, 4, None))
    g = torch.Generator(device=DEV).manual_seed(M)
    b = 128
    X = torch.randn(M, K, generator=g, device=DEV).half()
    W = (0.05 * torch.randn(N, K, generator=g, device=DEV)).half()
    bias = torch.randn(N, generator=g, device=DEV).half()
    perm = torch.randperm(K, generator=g, device=DEV).to(torch.int32)
    layer = clq.PreparedLinear.from_weight(W, perm, b, bias=bias, a_bits=a_bits, w_bits=w_bits,
                                           w_codes=w_codes)
    if setting == "asym":
        Xq, s_x, lo = clq.rotate_quant_act_asym(X, perm, b)
        wsum = clq.weight_code_sums(layer.We, K)
        Y, acc = clq.linear_asym(Xq, s_x, lo, layer.We, layer.s_w, wsum, b, K, bias, with_acc=True)
    else:
        Xq, s_x = clq.rotate_quant_act(X, perm, b, layer.act_codes)
        Y, acc = clq.linear(Xq, s_x, layer.We, layer.s_w, b, K, bias, with_acc=True)
    assert clq.device_status() == 0

    def codes(t):
        if w_codes is not None:
            t = clq.convert_codes(t, K, clq.CLQ_CODES_E4M3)
        q = torch.from_numpy(_values(t, clq.codes_layout(t, K), K))
        return q.to(DEV).double()

    qx, qw = codes(Xq), codes(layer.We)
    want = qx @ qw.t()
    assert torch.equal(acc.double(), want)
    scale = layer.s_w.double()[None, :] / b
    y64 = want * s_x.double()[:, None] * scale
    size = y64.abs()
    if setting == "asym":
        zp = (lo.double() + 8 * s_x.double())[:, None] * qw.sum(1)[None, :] * scale
        y64 = y64 + zp
        size = size + zp.abs()
    y64 = y64 + bias.double()[None, :]
    size = size + bias.double().abs()[None, :]
    # half an ulp of fp16, three fp32 roundings of the terms, the smallest subnormal
    err = (Y.double() - y64).abs()
    assert bool((err <= 2.0 ** -11 * y64.abs() + 1e-6 * size + 2.0 ** -24).all())


@pytest.mark.parametrize("K", [1024, 7936, 7968, 16384])
@pytest.mark.parametrize("M,N", [(130, 40), (3000, 3000)])
def test_w8a8_accumulators_at_their_limit(K, M, N):
    """K at and past the point where W8A8's cross and low products stop sharing an
    accumulator, with the code whose products there are largest (120 = 128 - 8:
    2 * 128 * -8 + 64 a pair) in every place but a few: |acc| up to 14400 K."""
    def split(q):
        h = torch.div(q + 8, 16, rounding_mode="floor")
        lut = torch.zeros(257, dtype=torch.uint8, device=DEV)
        for v in range(-128, 129):
            a = abs(v)
            f, x = np.frexp(float(a)) if a else (0.0, 0)
            m = (f * 2 - 1) * 8
            if a and m == int(m):
                lut[v + 128] = ((x - 1 + 7) << 3) | int(m) | (0x80 if v < 0 else 0)
        return torch.cat([lut[(16 * h + 128).long()], lut[(q - 16 * h + 128).long()]], dim=1)

    g = torch.Generator(device=DEV).manual_seed(K)
    qx = torch.full((M, K), 120, dtype=torch.int32, device=DEV)
    qw = torch.full((N, K), 120, dtype=torch.int32, device=DEV)
    qx[:, :5] = torch.randint(-127, 128, (M, 5), generator=g, device=DEV, dtype=torch.int32)
    qw[1::2] = -qw[1::2]
    ones = torch.ones(M, device=DEV), torch.ones(N, device=DEV)
    Y, acc = clq.linear(split(qx), ones[0], split(qw), ones[1], 32, K, None, with_acc=True)
    want = qx.double() @ qw.double().t()
    assert torch.equal(acc.double(), want)
    assert clq.device_status() == 0


@pytest.mark.parametrize("w_codes", [None, clq.CLQ_CODES_E2M3])
@pytest.mark.parametrize("M,N,K", [(1900, 4600, 1152), (2200, 4701, 640), (9700, 1152, 1152),
                                   (8322, 1160, 1152), (700, 1400, 9344), (300, 10241, 9344),
                                   (300, 10240, 9344)])
def test_fused_wide_tiles_match_separate(M, N, K, w_codes):
    """The one-kernel layer on the wide tiles that CTA pairs share, with a last pair
    whose second CTA has no rows or few and ragged columns: the separate kernels'
    output bit for bit, twice over one workspace.  At K = 9344 the sequential form, on
    pairs and, where those take a round more, on single CTAs."""
    g = torch.Generator(device=DEV).manual_seed(N)
    b = 64
    X = torch.randn(M, K, generator=g, device=DEV).half()
    W = (0.05 * torch.randn(N, K, generator=g, device=DEV)).half()
    bias = torch.randn(N, generator=g, device=DEV).half()
    perm = torch.randperm(K, generator=g, device=DEV).to(torch.int32)
    layer = clq.PreparedLinear.from_weight(W, perm, b, bias=bias, w_codes=w_codes)
    ws = clq.fused_workspace(M, K, DEV)
    want = layer(X)
    for _ in range(2):
        assert torch.equal(layer(X, fused=True, workspace=ws), want)
    assert clq.device_status() == 0


@pytest.mark.parametrize("setting", sorted(SETTINGS) + ["asym", "asym_w4a8", "asym_w8a8"])
@pytest.mark.parametrize("M,N,K", [(300, 10241, 4608), (300, 10008, 8064), (12, 11013, 2304)])
def test_single_cta_tiles(setting, M, N, K):
    """Shapes whose rounds of 256-row tiles would come out so coarse, or whose rows are
    so few, that the launcher takes single CTAs, on both sides of the K up to which
    W8A8 has two accumulators: products exact, outputs as in test_tile_widths."""
    a_bits, w_bits, w_codes = SETTINGS.get(setting.replace("asym_", ""), (4, 4, None))
    asym = setting.startswith("asym")
    g = torch.Generator(device=DEV).manual_seed(M + N)
    b = 128
    X = torch.randn(M, K, generator=g, device=DEV).bfloat16()
    W = (0.05 * torch.randn(N, K, generator=g, device=DEV)).bfloat16()
    bias = torch.randn(N, generator=g, device=DEV).bfloat16()
    perm = torch.randperm(K, generator=g, device=DEV).to(torch.int32)
    layer = clq.PreparedLinear.from_weight(W, perm, b, bias=bias, a_bits=a_bits, w_bits=w_bits,
                                           w_codes=w_codes)
    kw = dict(out_dtype=torch.bfloat16, with_acc=True,
              Y=torch.full((M + 1, N), 7.0, dtype=torch.bfloat16, device=DEV)[:M])
    guard = kw["Y"].as_strided((N,), (1,), M * N)  # the row behind Y
    if asym:
        codes = clq.CLQ_CODES_E4M3 if a_bits == 4 else clq.CLQ_CODES_E4M3_SPLIT
        Xq, s_x, lo = clq.rotate_quant_act_asym(X, perm, b, codes)
        wsum = clq.weight_code_sums(layer.We, K)
        Y, acc = clq.linear_asym(Xq, s_x, lo, layer.We, layer.s_w, wsum, b, K, bias, **kw)
    else:
        Xq, s_x = clq.rotate_quant_act(X, perm, b, layer.act_codes)
        Y, acc = clq.linear(Xq, s_x, layer.We, layer.s_w, b, K, bias, **kw)
    assert clq.device_status() == 0 and bool((guard == 7.0).all())

    def codes64(t):
        if w_codes is not None:
            t = clq.convert_codes(t, K, clq.CLQ_CODES_E4M3)
        return torch.from_numpy(_values(t, clq.codes_layout(t, K), K)).to(DEV).double()

    qx, qw = codes64(Xq), codes64(layer.We)
    want = qx @ qw.t()
    assert torch.equal(acc.double(), want)
    scale = layer.s_w.double()[None, :] / b
    y64 = want * s_x.double()[:, None] * scale
    size = y64.abs()
    if asym:
        zp = (lo.double() + (8 if a_bits == 4 else 128) * s_x.double())[:, None] \
            * qw.sum(1)[None, :] * scale
        y64, size = y64 + zp, size + zp.abs()
    y64 = y64 + bias.double()[None, :]
    size = size + bias.double().abs()[None, :]
    # half an ulp of bf16, three fp32 roundings of the terms
    assert bool(((Y.double() - y64).abs() <= 2.0 ** -8 * y64.abs() + 1e-6 * size + 2.0 ** -126).all())
