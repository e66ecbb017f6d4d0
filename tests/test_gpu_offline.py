"""Offline kernels at their edges: the column-swap vector built on the device
against the host builder, and the word-wise code conversions against the formats'
definitions for every byte value."""
import numpy as np
import pytest
import torch

from paper_2509_24416_gb300 import clq

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
P, E = clq.CLQ_CODES_INT4_PACKED, clq.CLQ_CODES_E4M3


@pytest.mark.parametrize("K", [1, 2, 3, 31, 1000, 1023, 1024, 1025, 1152, 3072, 16383, 16384])
@pytest.mark.parametrize("kind", ["random", "ties", "equal", "special"])
def test_device_permutation_matches_host(K, kind):
    rng = np.random.default_rng(K)
    s = {"random": lambda: rng.standard_normal(K),
         "ties": lambda: rng.integers(0, 4, K),
         "equal": lambda: np.full(K, 1.5),
         "special": lambda: rng.choice([0.0, -0.0, np.inf, 1e-45, -1.0, 3e38, -np.inf], K)}[kind]()
    s = torch.from_numpy(s.astype(np.float32))
    perm, bad = clq.build_permutation_device(s.to(DEV))
    assert torch.equal(perm.cpu(), clq.build_permutation(s)) and int(bad) == 0
    s[K // 2] = float("nan")
    perm, bad = clq.build_permutation_device(s.to(DEV))
    assert int(bad) == 1 and torch.equal(perm.cpu(), torch.arange(K, dtype=torch.int32))
    with pytest.raises(clq.ClqError):
        clq.build_permutation(s)


def test_device_permutation_refuses(monkeypatch):
    with pytest.raises(clq.ClqError) as e:
        clq.build_permutation_device(torch.zeros(16385, device=DEV))
    assert e.value.status == 2
    with pytest.raises(clq.ClqError) as e:
        clq.build_permutation_device(torch.zeros(0, device=DEV))
    assert e.value.status == 1
    W = torch.randn(64, 128, device=DEV).half()
    calib = torch.randn(1, 4, 128, device=DEV).half()
    monkeypatch.setattr(clq, "outlier_scores", lambda *a, **k: torch.full((128,), float("nan"),
                                                                          device=DEV))
    with pytest.raises(clq.ClqError) as e:
        clq.PreparedLinear.calibrate(W, calib, 32)
    assert e.value.status == 1 and "clq_build_permutation" in str(e.value)
    assert clq.device_status() == 0


def test_convert_every_byte():
    K = 32
    every = torch.arange(256, dtype=torch.uint8)
    # packed -> E4M3: each byte value in each of 16 places among valid codes
    packed = torch.full((256, 16), 0x71, dtype=torch.uint8)
    packed[torch.arange(256), torch.arange(256) % 16] = every
    out = clq.convert_codes(packed.to(DEV), K, E).cpu().numpy()
    lo, hi = packed.numpy() & 15, packed.numpy() >> 4
    q = np.stack([lo, hi], 2).reshape(256, K).astype(np.int64)
    q = np.where(q >= 8, q - 16, q)
    want = np.where(q == -8, 0, q)  # -8 is written as 0 and reported
    mag = np.array([0x00, 0x38, 0x40, 0x44, 0x48, 0x4A, 0x4C, 0x4E])
    assert np.array_equal(out, mag[np.abs(want)] | np.where(want < 0, 0x80, 0))
    assert clq.device_status() == 9
    # E4M3 -> packed: every byte value; one past +-7 is written as 0 and reported,
    # a fraction truncates
    e4 = torch.full((256, K), 0xC8, dtype=torch.uint8)  # -4
    e4[torch.arange(256), torch.arange(256) % K] = every
    out = clq.convert_codes(e4.to(DEV), K, P).cpu().numpy()
    b = e4.numpy().astype(np.int64)
    ex, m = (b >> 3) & 15, b & 7
    v = np.where(ex == 0, 0.0, (8 + m) * 2.0 ** (ex - 10.0))
    v = np.trunc(v) * np.where(b & 0x80, -1, 1)
    v = np.where(np.abs(v) > 7, 0, v).astype(np.int64)
    got = np.stack([out & 15, out >> 4], 2).reshape(256, K).astype(np.int64)
    assert np.array_equal(np.where(got >= 8, got - 16, got), v)
    assert clq.device_status() == 9
    # whole valid arrays there and back, no report
    codes = torch.randint(0, 256, (77, 576), dtype=torch.uint8)
    codes[(codes & 15) == 8] = 0x17
    codes[(codes >> 4) == 8] = 0x19
    there = clq.convert_codes(codes.to(DEV), 1152, E)
    assert torch.equal(clq.convert_codes(there, 1152, P).cpu(), codes)
    assert torch.equal(there, clq.expand_weights(codes.to(DEV)))
    assert clq.device_status() == 0


@pytest.mark.parametrize("K,b", [(1152, 128), (12288, 64), (1152, 32)])
def test_device_permutation_feeds_the_next_call(K, b):
    """A vector built on the device into a buffer that held another one, and read by
    the very next call on the stream: each rotate-quant loop and the one-kernel
    layer give what they give for the finished vector."""
    g = torch.Generator(device=DEV).manual_seed(K)
    X = torch.randn(300, K, generator=g, device=DEV).half()
    W = (0.05 * torch.randn(64, K, generator=g, device=DEV)).half()
    scores = [torch.rand(K, generator=g, device=DEV) for _ in range(4)]
    perms = [clq.build_permutation_device(s)[0] for s in scores]
    layers = [clq.PreparedLinear.from_weight(W, p, b) for p in perms]
    ws = clq.fused_workspace(300, K, DEV)
    calls = [lambda p, i, c=c: clq.rotate_quant_act(X, p, b, c)
             for c in (P, E, clq.CLQ_CODES_E4M3_SPLIT)]
    calls.append(lambda p, i: clq.rotate_quant_act_asym(X, p, b))
    calls.append(lambda p, i: (clq.fused_linear(X, p, b, layers[i].We, layers[i].s_w,
                                                workspace=ws),))
    torch.cuda.synchronize()
    want = [[call(perms[i], i) for i in range(4)] for call in calls]
    torch.cuda.synchronize()
    perm = perms[3].clone()
    bad = torch.zeros(1, dtype=torch.int32, device=DEV)
    st = torch.cuda.current_stream().cuda_stream
    for j, call in enumerate(calls):
        for n in range(20):
            i = n % 4
            assert clq.clq_build_permutation_device(scores[i].data_ptr(), K, perm.data_ptr(),
                                                    bad.data_ptr(), st) == 0
            got = call(perm, i)
            assert all(torch.equal(a, w) for a, w in zip(got, want[j][i]))
    assert clq.device_status() == 0
