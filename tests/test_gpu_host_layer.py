"""A layer's plain call (one native step) against the same layer with its
buffers passed in (the Python path, two C calls): bit-identical outputs over
the forms it accepts, and the same errors for what both refuse."""
import pytest
import torch

from paper_2509_24416_gb300 import clq

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
P, E, C = clq.CLQ_CODES_INT4_PACKED, clq.CLQ_CODES_E4M3, clq.CLQ_CODES_E2M3


def _layer(K=1152, N=96, dtype=torch.float16, bias=True, **kw):
    g = torch.Generator().manual_seed(K + N)
    W = (0.02 * torch.randn(N, K, generator=g)).to(dtype).to(DEV)
    bi = torch.randn(N, generator=g).to(dtype).to(DEV) if bias else None
    return clq.PreparedLinear.from_weight(W, torch.randperm(K, generator=g), 64, bias=bi, **kw)


def _buffers(layer, X):
    M, N = X.shape[0], layer.We.shape[0]
    return dict(Y=torch.empty((M, N), dtype=X.dtype, device=DEV),
                Xq=torch.empty((M, clq.codes_width(layer.act_codes, layer.K)), dtype=torch.uint8,
                               device=DEV),
                s_x=torch.empty(M, dtype=torch.float32, device=DEV))


@pytest.mark.parametrize("kw", [{}, dict(w_codes=C), dict(w_codes=P), dict(w_codes=P, a_codes=P),
                                dict(a_codes=P), dict(a_bits=8), dict(a_bits=8, w_bits=8)])
@pytest.mark.parametrize("dtype,bias", [(torch.float16, True), (torch.bfloat16, False)])
@pytest.mark.parametrize("M", [1, 5, 333])
def test_matches_python_path(kw, dtype, bias, M):
    layer = _layer(dtype=dtype, bias=bias, **kw)
    X = torch.randn(M, 1152, device=DEV).to(dtype)
    assert torch.equal(layer(X), layer(X, **_buffers(layer, X)))
    wide = torch.randn(M, 1152 + 64, device=DEV).to(dtype)
    for Xs in (wide[:, 64:], wide[:, :1152]):  # strided rows
        assert torch.equal(layer(Xs), layer(Xs, **_buffers(layer, Xs)))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        Y1 = layer(X)
    Y2 = layer(X, stream=side, **_buffers(layer, X))
    torch.cuda.synchronize()
    assert torch.equal(Y1, Y2)


def test_empty_and_refused_calls():
    layer = _layer()
    Y = layer(torch.empty((0, 1152), dtype=torch.float16, device=DEV))
    assert Y.shape == (0, 96) and Y.dtype == torch.float16
    with pytest.raises(TypeError):
        layer(torch.randn(4, 1152, device=DEV))
    with pytest.raises(TypeError):  # bias of another type than the output
        layer(torch.randn(4, 1152, device=DEV).bfloat16())
    with pytest.raises(ValueError):
        layer(torch.randn(4, 2, 1152, device=DEV).half())
    with pytest.raises(ValueError):
        layer(torch.randn(1152, 4, device=DEV).half().t())
    with pytest.raises(ValueError):  # K of another layer
        layer(torch.randn(4, 1024, device=DEV).half())
    assert clq.device_status() == 7  # its rotate-quant met swap indexes past 1024
    with pytest.raises(clq.ClqError) as e:  # row stride not a multiple of 8
        layer(torch.randn(4, 1156, device=DEV).half()[:, :1152])
    assert e.value.status == 3
    layer.b = 48
    with pytest.raises(clq.ClqError) as e:
        layer(torch.randn(4, 1152, device=DEV).half())
    assert e.value.status == 2 and "clq_rotate_quant_act" in str(e.value)
    assert clq.device_status() == 0


def _pool(t):
    """Handle of the stream whose allocator pool holds t."""
    at = t.data_ptr()
    for seg in torch.cuda.memory_snapshot():
        if seg["address"] <= at < seg["address"] + seg["total_size"]:
            return seg["stream"]
    return None


@pytest.mark.parametrize("kw", [{}, dict(a_bits=8), dict(w_codes=P)])
def test_explicit_stream_owns_its_buffers(kw):
    """layer(X, stream=side) without buffers, behind a busy side stream and in front
    of work on the current stream that takes blocks of the same sizes."""
    layer = _layer(N=1152, **kw)
    X = torch.randn(2048, 1152, device=DEV).half()
    want = layer(X)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for fused in (False, True)[:1 if kw.get("a_bits") else 2]:
        got = []
        for _ in range(4):
            with torch.cuda.stream(side):
                torch.cuda._sleep(2000000)  # about a millisecond
            got.append(layer(X, fused=fused, stream=side))
            assert _pool(got[-1]) == side.cuda_stream
            for n in (want.numel() * 2, X.numel(), 2 * X.numel(), 4 * 2048):
                torch.full((n,), 0x7F, dtype=torch.uint8, device=DEV)
        torch.cuda.synchronize()
        assert all(torch.equal(y, want) for y in got)


def test_calibrate_on_a_stream():
    g = torch.Generator(device=DEV).manual_seed(3)
    W = torch.randn(96, 1152, generator=g, device=DEV).half()
    calib = torch.randn(4, 64, 1152, generator=g, device=DEV).half()
    side = torch.cuda.Stream()
    for grid in (None, (0.0, 0.01)):
        want, iw = clq.PreparedLinear.calibrate(W, calib, 64, clip_grid=grid)
        torch.cuda._sleep(2000000)  # the inputs may still be in the making
        c2 = calib * 1
        got, ig = clq.PreparedLinear.calibrate(W * 1, c2, 64, clip_grid=grid, stream=side)
        assert torch.equal(got.We, want.We) and torch.equal(got.s_w, want.s_w)
        assert torch.equal(ig["perm"], iw["perm"]) and torch.equal(ig["scores"], iw["scores"])
        assert _pool(got.We) == side.cuda_stream
    assert clq.device_status() == 0
