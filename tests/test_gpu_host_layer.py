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
