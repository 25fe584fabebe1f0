"""Codes on their way to the multiply: every code and zero point at every place of a packed word, and activations far from one."""
import numpy as np
import pytest
import torch

from paper_2606_11357_b200 import binding as tf
from paper_2606_11357_b200 import workloads as wl
import gpu_util as gu

pytestmark = pytest.mark.gpu

# GEMV up to 8 tokens, GEMV up to 16, GEMM
KINDS = [("gemv", 8), ("gemv", 16), ("gemm", 32)]


def _linear(kind, bits, blob, a, K, N, group):
    M = a.shape[0]
    y = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
    op = (2 if kind == "gemm" else 0) + (bits == 8)
    ws = torch.zeros(tf.tf_workspace_size(op, M, K, N), dtype=torch.uint8, device="cuda")
    name = f"tf_{kind}_w{bits}a16"
    if group < 128:
        getattr(tf, name + "_grouped")(blob, a, y, M, K, N, group, ws)
    else:
        getattr(tf, name)(blob, a, y, M, K, N, ws)
    assert tf.tf_device_status(ws) == 0
    return y


@pytest.mark.parametrize("group", [128, 64, 32])
@pytest.mark.parametrize("kind,M", KINDS)
def test_every_code_and_zero_point_comes_out_exactly(kind, M, group):
    """Scale 1, one-hot activations: y is a row of q - z, whole numbers that bf16 holds, so nothing may differ."""
    K, N = 128, 1024
    k, n = np.meshgrid(np.arange(K), np.arange(N), indexing="ij")
    q = ((n // 64 + k) % 16).astype(np.uint8)                       # a column meets every code, a strip's 64 columns ...
    z = ((np.arange(N)[None, :] + 5 * np.arange(K // group)[:, None]) % 16).astype(np.uint8)      # ... every zero point
    blob = torch.from_numpy(tf.tf_pack_awq(wl.awq_pack_words(q), np.ones((K // group, N), np.float16), wl.awq_pack_words(z), K, N, group)).cuda()
    for first in range(0, K, M):
        a = torch.zeros((M, K), dtype=torch.bfloat16, device="cuda")
        a[torch.arange(M), first + torch.arange(M)] = 1.0
        y = _linear(kind, 4, blob, a, K, N, group)
        rows = np.arange(first, first + M)
        want = q[rows].astype(np.int64) - z[rows // group]
        assert np.array_equal(y.float().cpu().numpy().astype(np.int64), want)


@pytest.mark.parametrize("kind,M", KINDS)
def test_every_int8_value_comes_out_exactly(kind, M):
    K, N = 128, 512
    k, n = np.meshgrid(np.arange(K), np.arange(N), indexing="ij")
    w = ((n + 3 * k) % 256 - 128).astype(np.int8)
    blob = torch.from_numpy(tf.tf_pack_w8(w, np.ones((1, N), np.float16), K, N)).cuda()
    for first in range(0, K, M):
        a = torch.zeros((M, K), dtype=torch.bfloat16, device="cuda")
        a[torch.arange(M), first + torch.arange(M)] = 1.0
        y = _linear(kind, 8, blob, a, K, N, 128)
        assert np.array_equal(y.float().cpu().numpy().astype(np.int64), w[first:first + M])


@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("kind,M", [("gemv", 3), ("gemv", 16), ("gemm", 50)])
def test_a_power_of_two_goes_through_unchanged(kind, M, bits):
    """Activations times 2^e give the same results times 2^e, bit for bit: every step scales exactly as long as no number of the
    way leaves the normal range (products are at least 2^-14 2^-6 2^-80, sums at most 2^100 2^20)."""
    K, N = 1024, 264
    p = (wl.make_w4 if bits == 4 else wl.make_w8)(M, K, N, seed=40 + M)
    a = gu.to_device_bf16(p.a_bf16).float()
    a = torch.where(a.abs() < 2.0 ** -14, torch.zeros_like(a), a)
    blob = torch.from_numpy(gu.pack(p)).cuda()
    plain = _linear(kind, bits, blob, a.bfloat16(), K, N, 128).double()
    for e in (-80, 100):
        y = _linear(kind, bits, blob, (a * 2.0 ** e).bfloat16(), K, N, 128).double()
        assert torch.equal(y, plain * 2.0 ** e)


@pytest.mark.parametrize("value", [1.9921875, -1.9921875, 1.0078125])
@pytest.mark.parametrize("M,K,N", [(1, 512, 128), (2, 512, 128), (1, 6144, 14400), (1, 1024, 19008)])
def test_integer_path_at_the_ends_of_its_ranges(M, K, N, value):
    """Codes and zero points 0 and 15 against activations that are all the same number: the largest sums that the integers of a tile
    reach, in the forms with and without kept pieces.  Scale 2^-6, so every sum of a tile and over K is exact in fp32 and only the
    store rounds."""
    n = np.arange(N)
    q = np.broadcast_to(np.where(n & 1, 15, 0).astype(np.uint8), (K, N))
    z = np.broadcast_to(np.where(n & 2, 15, 0).astype(np.uint8), (K // 128, N))
    blob = torch.from_numpy(tf.tf_pack_awq(wl.awq_pack_words(q), np.full((K // 128, N), 2.0 ** -6, np.float16), wl.awq_pack_words(z), K, N)).cuda()
    a = torch.full((M, K), value, dtype=torch.bfloat16, device="cuda")
    y = _linear("gemv", 4, blob, a, K, N, 128)
    want = (q[0].astype(np.float64) - z[0]) * 2.0 ** -6 * value * K
    assert torch.equal(y, torch.from_numpy(want).to(torch.bfloat16).cuda().expand(M, N))
