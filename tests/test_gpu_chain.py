"""Chains of dependent GEMVs on one stream (Section 4.6: operators are dispatched in sequence, each consuming
the output of the one before it).

Every kernel of the library lets its successor on the stream start early (programmatic dependent launch) and a
half-SM GEMV becomes resident beside its predecessor.  The successor may fetch weights at once but must not read
activations before the predecessor has completed.  These tests make the window as wide as it gets -- a long
first call, a second call whose activations ARE the first call's output, intermediates pre-filled with NaN on the
same stream -- for every launch plan of the GEMV, and check every result against the oracle applied to the bits
the previous call actually produced."""
import numpy as np
import pytest
import torch

import gpu_util as gu
from paper_2606_11357_b200 import binding as tf
from paper_2606_11357_b200 import workloads as wl

pytestmark = pytest.mark.gpu

_WEIGHTS = {}


def weights(K, N, seed):
    """(problem with M = 16 activations, device blob), cached per shape: the 30 MB matrices take a moment to draw."""
    key = (K, N, seed)
    if key not in _WEIGHTS:
        p = wl.make_w4(16, K, N, seed=seed)
        _WEIGHTS[key] = (p, torch.from_numpy(gu.pack(p)).cuda())
    return _WEIGHTS[key]


def with_activations(problem, a_bits):
    """The same weights as `problem` with other activations (a shallow copy: the oracle reads, never writes)."""
    import copy
    q = copy.copy(problem)
    q.a_bf16 = a_bits
    q.M = a_bits.shape[0]
    return q


def plan_kind(M, K, N):
    p = tf.tf_gemv_plan(4, M, K, N)
    return "cluster" if p["cluster"] > 1 else ("whole" if p["full"] else "half")


# dims = layer widths d0 -> d1 -> d2 (-> d3); `plans` = the launch plan each call of the chain must take, so that
# a change of the planning heuristics cannot silently move a case to another code path
CHAINS = [
    ((4096, 14336, 4096), 1, ("half", "half")),
    ((4096, 14336, 4096), 2, ("half", "half")),
    ((4096, 14336, 4096), 4, ("whole", "whole")),
    ((4096, 14336, 4096), 8, ("whole", "whole")),
    ((4096, 4096, 1024), 1, ("half", "half")),
    ((4096, 4096, 1024), 8, ("whole", "whole")),
    ((4096, 14336, 4096, 1024), 1, ("half", "half", "half")),
    ((4096, 14336, 4096, 1024), 4, ("whole", "whole", "whole")),
    ((4096, 14336, 4096), 16, ("whole", "whole")),
    ((4096, 4096, 1024), 16, ("cluster", "cluster")),
    ((4096, 32768, 1024), 2, ("whole", "half")),            # a long integer-path range: whole SM, 16 warps, piece table
    ((5120, 18432, 1024), 1, ("whole", "half")),            # the same without the table
    ((1024, 32768, 1024), 2, ("half", "half")),            # two tokens with the piece table, then without
    ((384, 14336, 4096), 1, ("half", "half")),
]


@pytest.mark.parametrize("dims,M,plans", CHAINS, ids=[f"{'x'.join(map(str, d))}-M{m}" for d, m, _ in CHAINS])
def test_gemv_chain_consumes_previous_output(dims, M, plans):
    layers = [weights(dims[i], dims[i + 1], seed=2000 + i) for i in range(len(dims) - 1)]
    assert tuple(plan_kind(M, dims[i], dims[i + 1]) for i in range(len(layers))) == plans
    a0_bits = layers[0][0].a_bf16[:M].copy()
    a0 = gu.to_device_bf16(a0_bits)
    ys = [torch.empty((M, dims[i + 1]), dtype=torch.bfloat16, device="cuda") for i in range(len(layers))]
    ws = torch.zeros(tf.tf_workspace_size(tf.TF_OP_GEMV_W4A16, M, 4096, 4096), dtype=torch.uint8, device="cuda")
    for rep in range(4):                                   # an early read shows up intermittently
        for y in ys:
            y.fill_(float("nan"))                          # on the stream, right before the chain
        x = a0
        for (p, blob), y in zip(layers, ys):
            tf.tf_gemv_w4a16(blob, x, y, M, p.K, p.N, ws)
            x = y
        assert tf.tf_device_status(ws) == 0
        torch.cuda.synchronize()
        outs = [gu.bits_of(y) for y in ys]
        if rep == 0:
            first = outs
            x_bits = a0_bits
            for (p, _), out in zip(layers, outs):
                gu.check_against_oracle(with_activations(p, x_bits), out)
                x_bits = out
        else:                                              # deterministic: later repetitions must give the same bits
            for o, f in zip(outs, first):
                assert np.array_equal(o, f)


def test_gemm_then_half_sm_gemv_chain():
    """A whole-SM kernel (the GEMM) followed by two half-SM GEMVs that each consume the previous result."""
    M = 2
    (p1, b1), (p2, b2), (p3, b3) = weights(4096, 4096, 2100), weights(4096, 14336, 2101), weights(14336, 4096, 2102)
    a0_bits = p1.a_bf16[:M].copy()
    a0 = gu.to_device_bf16(a0_bits)
    y1 = torch.empty((M, 4096), dtype=torch.bfloat16, device="cuda")
    y2 = torch.empty((M, 14336), dtype=torch.bfloat16, device="cuda")
    y3 = torch.empty((M, 4096), dtype=torch.bfloat16, device="cuda")
    need = max(tf.tf_workspace_size(tf.TF_OP_GEMM_W4A16, M, 4096, 4096), tf.tf_workspace_size(tf.TF_OP_GEMV_W4A16, M, 4096, 4096))
    ws = torch.zeros(need, dtype=torch.uint8, device="cuda")
    for rep in range(3):
        for y in (y1, y2, y3):
            y.fill_(float("nan"))
        tf.tf_gemm_w4a16(b1, a0, y1, M, 4096, 4096, ws)
        tf.tf_gemv_w4a16(b2, y1, y2, M, 4096, 14336, ws)
        tf.tf_gemv_w4a16(b3, y2, y3, M, 14336, 4096, ws)
        assert tf.tf_device_status(ws) == 0
        torch.cuda.synchronize()
        o1, o2, o3 = gu.bits_of(y1), gu.bits_of(y2), gu.bits_of(y3)
        gu.check_against_oracle(with_activations(p1, a0_bits), o1)
        gu.check_against_oracle(with_activations(p2, o1), o2)
        gu.check_against_oracle(with_activations(p3, o2), o3)


def test_w8_integer_path_chain():
    """The W8A16 integer path (1 and 2 tokens) reads its activations in the consumer warps too."""
    M = 2
    p1 = wl.make_w8(M, 4096, 14336, seed=2200)
    p2 = wl.make_w8(M, 14336, 4096, seed=2201)
    assert tf.tf_gemv_plan(8, M, 4096, 14336)["i8"] == 1 and tf.tf_gemv_plan(8, M, 14336, 4096)["i8"] == 1
    b1, b2 = torch.from_numpy(gu.pack(p1)).cuda(), torch.from_numpy(gu.pack(p2)).cuda()
    a0 = gu.to_device_bf16(p1.a_bf16)
    y1 = torch.empty((M, 14336), dtype=torch.bfloat16, device="cuda")
    y2 = torch.empty((M, 4096), dtype=torch.bfloat16, device="cuda")
    ws = torch.zeros(tf.tf_workspace_size(tf.TF_OP_GEMV_W8A16, M, 4096, 4096), dtype=torch.uint8, device="cuda")
    for rep in range(3):
        y1.fill_(float("nan"))
        y2.fill_(float("nan"))
        tf.tf_gemv_w8a16(b1, a0, y1, M, 4096, 14336, ws)
        tf.tf_gemv_w8a16(b2, y1, y2, M, 14336, 4096, ws)
        assert tf.tf_device_status(ws) == 0
        torch.cuda.synchronize()
        o1, o2 = gu.bits_of(y1), gu.bits_of(y2)
        gu.check_against_oracle(p1, o1)
        gu.check_against_oracle(with_activations(p2, o1), o2)


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("kind,M,K,N", [("gemv", 1, 1024, 4096), ("gemv", 4, 2048, 1032), ("gemm", 40, 1024, 4096)])
def test_packing_between_calls(kind, M, K, N, captured):
    """The device packer rewrites one blob between calls that read it, with nothing but the stream to order them, and reads arrays that
    a copy just ahead of it has put there: every result is that of its own weights."""
    problems = [wl.make_w4(M, K, N, seed=60 + i) for i in range(3)]
    sources = [[torch.from_numpy(p.qweight.view(np.int32)).cuda(), torch.from_numpy(p.scales_f16).cuda(), torch.from_numpy(p.qzeros.view(np.int32)).cuda()] for p in problems]
    a = [gu.to_device_bf16(p.a_bf16) for p in problems]
    arrays = [torch.empty_like(t) for t in sources[0]]
    blob = torch.zeros(tf.tf_packed_size(4, K, N, 128), dtype=torch.uint8, device="cuda")
    ys = [torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in problems]
    ws = torch.zeros(tf.tf_workspace_size(tf.TF_OP_GEMV_W4A16 if kind == "gemv" else tf.TF_OP_GEMM_W4A16, M, K, N), dtype=torch.uint8, device="cuda")
    call = tf.tf_gemv_w4a16 if kind == "gemv" else tf.tf_gemm_w4a16

    def chain():
        for i in range(len(problems)):
            for dst, src in zip(arrays, sources[i]):
                dst.copy_(src)
            tf.tf_pack_awq_device(*arrays, K, N, 128, blob)
            for _ in range(2):
                call(blob, a[i], ys[i], M, K, N, ws)

    chain()
    if captured:
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            chain()
        for y in ys:
            y.fill_(float("nan"))
        graph.replay()
    assert tf.tf_device_status(ws) == 0
    for p, y in zip(problems, ys):
        gu.check_against_oracle(p, gu.bits_of(y))


@pytest.mark.parametrize("M,K,N", [(16, 256, 1024), (3, 384, 264), (200, 512, 4096)])
@pytest.mark.parametrize("group", [128, 32])
def test_packing_what_the_call_just_ahead_has_written(M, K, N, group):
    """The packer starts before the GEMV or GEMM ahead of it has ended, and its three arrays are parts of that call's result, rewritten in place
    each time: what it packs is what that call wrote.  (264 columns: rows of 33 words, read one by one.)"""
    rows = K // group
    words = [K * N // 8, (rows * N // 2 + 3) // 4 * 4, (rows * N // 8 + 3) // 4 * 4]           # qweight, scales, qzeros; each 16-byte aligned
    Np = (sum(words) * 2 // M // 64 + 1) * 64                                                # M x Np bf16 results hold them
    kind, Kp = "gemv" if M <= 16 else "gemm", 2048
    p = wl.make_w4(M, Kp, Np, seed=80 + M)
    producer, ws = torch.from_numpy(gu.pack(p)).cuda(), torch.zeros(tf.tf_workspace_size(tf.TF_OP_GEMM_W4A16, M, Kp, Np), dtype=torch.uint8, device="cuda")
    call = tf.tf_gemv_w4a16 if kind == "gemv" else tf.tf_gemm_w4a16
    inputs = [gu.to_device_bf16(p.a_bf16), gu.to_device_bf16(p.a_bf16[:, ::-1].copy()), gu.to_device_bf16(p.a_bf16 ^ np.uint16(0x8000))]
    y = torch.zeros(M, Np, dtype=torch.bfloat16, device="cuda")
    flat = y.view(-1).view(torch.int32)
    q, s, z = flat[:words[0]], flat[words[0]:words[0] + words[1]], flat[words[0] + words[1]:sum(words)]
    blobs = [torch.zeros(tf.tf_packed_size(4, K, N, group), dtype=torch.uint8, device="cuda") for _ in inputs]
    call(producer, inputs[0], y, M, Kp, Np, ws)
    for a, blob in zip(inputs, blobs):
        call(producer, a, y, M, Kp, Np, ws)
        tf.tf_pack_awq_device(q, s, z, K, N, group, blob)
    assert tf.tf_device_status(ws) == 0
    for a, blob in zip(inputs, blobs):
        call(producer, a, y, M, Kp, Np, ws)
        torch.cuda.synchronize()
        words_now = flat.cpu().numpy()
        hq = words_now[:words[0]].view(np.uint32).reshape(K, N // 8)
        hs = words_now[words[0]:words[0] + words[1]].view(np.float16)[:rows * N].reshape(rows, N)
        hz = words_now[words[0] + words[1]:sum(words)].view(np.uint32)[:rows * N // 8].reshape(rows, N // 8)
        assert np.array_equal(tf.tf_pack_awq(hq.copy(), hs.copy(), hz.copy(), K, N, group), blob.cpu().numpy())
