"""Variants of the setup the paper also describes (Section 2.1: per-channel W8A16 scales; group sizes above
128; token counts between the decode and prefill ranges): same kernels, same acceptance rule."""
import numpy as np
import pytest
import torch

from oracle import tilefuse_oracle as orc
from paper_2606_11357_b200 import binding as tf
from paper_2606_11357_b200 import workloads as wl
import gpu_util as gu
from helpers import WORKSPACE_ZERO_BYTES, bf16_bits_to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,M", [("gemv", 1), ("gemv", 16), ("gemm", 40), ("gemm", 300)])
def test_w8_per_channel_scales(kind, M):
    """group_size == K: one scale per output column."""
    K, N = 1024, 712
    p = wl.make_w8(M, K, N, seed=500 + M, group_size=K)
    assert p.scales_f16.shape == (1, N)
    gu.check_against_oracle(p, gu.run(p, kind))


@pytest.mark.parametrize("kind,M,g", [("gemv", 3, 256), ("gemv", 9, 512), ("gemm", 130, 256), ("gemm", 64, 1536)])
def test_w4_group_sizes_above_the_tile(kind, M, g):
    K, N = 1536, 328
    p = wl.make_w4(M, K, N, seed=600 + M, group_size=g)
    gu.check_against_oracle(p, gu.run(p, kind))


def test_unpack_with_group_256_is_bit_exact():
    K, N, g = 1024, 136, 256
    p = wl.make_w4(1, K, N, seed=77, group_size=g)
    blob = torch.from_numpy(gu.pack(p)).cuda()
    q = torch.full((K, N), 0xEE, dtype=torch.uint8, device="cuda")
    z = torch.full((K // g, N), 0xEE, dtype=torch.uint8, device="cuda")
    s = torch.zeros((K // g, N), dtype=torch.float16, device="cuda")
    tf.tf_unpack_w4(blob, q, z, s, K, N, g)
    torch.cuda.synchronize()
    assert np.array_equal(q.cpu().numpy(), orc.unpack_awq(p.qweight))
    assert np.array_equal(z.cpu().numpy(), orc.unpack_awq(p.qzeros))
    assert np.array_equal(s.cpu().numpy().view(np.uint16), p.scales_f16.view(np.uint16))


@pytest.mark.parametrize("M", [17, 33, 100, 129, 255])
def test_medium_token_counts_through_the_gemm(M):
    """Between the decode (<= 16) and prefill ranges the GEMM entry point applies, with smaller token tiles."""
    p = wl.make_w4(M, 2048, 1096, seed=700 + M)
    gu.check_against_oracle(p, gu.run(p, "gemm"))


def test_illegal_group_sizes_are_rejected():
    assert tf.tf_packed_size(4, 1024, 64, 16) == 0          # below the smallest group size
    assert tf.tf_packed_size(8, 1024, 64, 64) == 0          # below the tile's k-extent: 4-bit only
    assert tf.tf_packed_size(4, 1024, 64, 384) == 0         # does not divide K
    assert tf.tf_packed_size(8, 1024, 64, 1024) > 0


@pytest.mark.parametrize("g", [64, 32])
@pytest.mark.parametrize("kind,M,K,N", [("gemv", 1, 1024, 512), ("gemv", 2, 4096, 1024), ("gemv", 7, 512, 200), ("gemv", 16, 2048, 1096),
                                       ("gemv", 3, 4096, 4096), ("gemm", 17, 512, 200), ("gemm", 100, 1024, 328),
                                       ("gemm", 300, 2048, 1096), ("gemm", 130, 4096, 512)])
def test_group_sizes_64_and_32(kind, M, K, N, g):
    """Section 2.2's group-wise quantization with the group sizes below the tile's k-extent: unpack bit-exact, GEMV and
    GEMM within the stated tolerance, through the *_grouped entry points."""
    p = wl.make_w4(M, K, N, seed=1400 + M + g, group_size=g)
    blob = torch.from_numpy(gu.pack(p)).cuda()
    q = torch.full((K, N), 0xEE, dtype=torch.uint8, device="cuda")
    z = torch.full((K // g, N), 0xEE, dtype=torch.uint8, device="cuda")
    s = torch.zeros((K // g, N), dtype=torch.float16, device="cuda")
    tf.tf_unpack_w4(blob, q, z, s, K, N, g)
    torch.cuda.synchronize()
    assert np.array_equal(q.cpu().numpy(), orc.unpack_awq(p.qweight))
    assert np.array_equal(z.cpu().numpy(), orc.unpack_awq(p.qzeros))
    assert np.array_equal(s.cpu().numpy().view(np.uint16), p.scales_f16.view(np.uint16))
    a = gu.to_device_bf16(p.a_bf16)
    guard = 512
    ybuf = torch.full((guard + M * N + guard,), gu.CANARY, dtype=torch.int16, device="cuda")
    y = ybuf[guard:guard + M * N].view(torch.bfloat16).view(M, N)
    op = tf.TF_OP_GEMV_W4A16 if kind == "gemv" else tf.TF_OP_GEMM_W4A16
    ws = torch.zeros(tf.tf_workspace_size(op, M, K, N), dtype=torch.uint8, device="cuda")
    fn = tf.tf_gemv_w4a16_grouped if kind == "gemv" else tf.tf_gemm_w4a16_grouped
    for _ in range(2):
        fn(blob, a, y, M, K, N, g, ws)
    assert tf.tf_device_status(ws) == 0
    raw = ybuf.cpu().numpy().view(np.uint16)
    assert np.all(raw[:guard] == gu.CANARY) and np.all(raw[guard + M * N:] == gu.CANARY), "write outside y"
    gu.check_against_oracle(p, raw[guard:guard + M * N].reshape(M, N))


def test_group_size_mismatch_is_detected_on_the_device():
    """A blob packed with group size 64 given to the default entry point (group size 128), and the other way round:
    the status word says TF_ERR_BLOB and y is untouched."""
    M, K, N = 2, 512, 256
    for g_blob, g_call in ((64, 128), (128, 64), (32, 64)):
        p = wl.make_w4(M, K, N, seed=1500 + g_blob, group_size=g_blob)
        blob = torch.from_numpy(gu.pack(p)).cuda()
        big = torch.zeros(tf.tf_packed_size(4, K, N, 32), dtype=torch.uint8, device="cuda")     # room for the largest tiles
        big[:blob.numel()] = blob
        a = gu.to_device_bf16(p.a_bf16)
        y = torch.full((M, N), -2.0, dtype=torch.bfloat16, device="cuda")
        ws = torch.zeros(tf.tf_workspace_size(tf.TF_OP_GEMV_W4A16, M, K, N), dtype=torch.uint8, device="cuda")
        tf.tf_gemv_w4a16_grouped(big, a, y, M, K, N, g_call, ws)
        assert tf.tf_device_status(ws) == 4
        assert bool((y == -2.0).all())


@pytest.mark.parametrize("kind,M,K,N", [("gemv", 1, 4096, 1024), ("gemv", 16, 4096, 4096), ("gemv", 4, 1536, 328), ("gemv", 3, 14336, 4096),
                                        ("gemm", 300, 2048, 1096), ("gemm", 512, 4096, 640)])
def test_workspace_head_is_left_zero(kind, M, K, N):
    """The status word, the GEMM's flags and the GEMV's partial-sum slots must be zero again after a call, so the
    same workspace serves the next call without being cleared."""
    p = wl.make_w4(M, K, N, seed=900 + M)
    blob = torch.from_numpy(gu.pack(p)).cuda()
    a = gu.to_device_bf16(p.a_bf16)
    y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    op = tf.TF_OP_GEMV_W4A16 if kind == "gemv" else tf.TF_OP_GEMM_W4A16
    ws = torch.zeros(tf.tf_workspace_size(op, M, K, N), dtype=torch.uint8, device="cuda")
    fn = tf.tf_gemv_w4a16 if kind == "gemv" else tf.tf_gemm_w4a16
    for _ in range(3):
        fn(blob, a, y, M, K, N, ws)
    assert tf.tf_device_status(ws) == 0
    assert int(ws[:WORKSPACE_ZERO_BYTES].to(torch.int32).sum().item()) == 0
    gu.check_against_oracle(p, gu.bits_of(y))


@pytest.mark.parametrize("M", [1, 2])
@pytest.mark.parametrize("pattern", ["wide", "tiny_tile", "huge"])
def test_w8_gemv_activation_dynamic_range(M, pattern):
    """W8A16 with 1 or 2 tokens multiplies int8 codes with the activations of a k-tile written as integers on the
    tile's own power-of-two scale; the result must stay inside the acceptance rule whatever the spread of magnitudes
    inside a tile, from tile to tile, or the absolute magnitude."""
    K, N = 2048, 328
    p = wl.make_w8(M, K, N, seed=900 + M)
    rng = np.random.default_rng(901 + M)
    a = rng.standard_normal((M, K)).astype(np.float32)
    if pattern == "wide":            # exponents spread over 40 binades inside every tile
        a *= np.exp2(rng.integers(-30, 11, size=(M, K))).astype(np.float32)
    elif pattern == "tiny_tile":     # whole k-tiles 2^-40 below their neighbours
        a[:, 128:256] *= np.float32(2.0 ** -40)
        a[:, 1024:1152] *= np.float32(2.0 ** -60)
    else:                            # near the top and the bottom of the bf16 range
        a[0] *= np.float32(2.0 ** 100)
        a[M - 1, K // 2:] *= np.float32(2.0 ** -110)
    p.a_bf16 = wl.f32_to_bf16_bits(a)
    gu.check_against_oracle(p, gu.run(p, "gemv"))


@pytest.mark.parametrize("kind,M", [("gemv", 1), ("gemv", 16), ("gemm", 200)])
def test_fused_qkv_blob_from_pack_concat(kind, M):
    """Three weight matrices packed separately, joined with tf_pack_concat, multiplied in one launch: the result
    is the oracle's for the column-concatenated matrix (Section 4.5: fewer, wider operators per token)."""
    K, widths = 1024, (512, 128, 128)
    parts = [wl.make_w4(M, K, n, seed=800 + i) for i, n in enumerate(widths)]
    for p in parts[1:]:
        p.a_bf16 = parts[0].a_bf16
    blobs = [tf.tf_pack_awq(p.qweight, p.scales_f16, p.qzeros, K, p.N) for p in parts]
    whole = wl.Problem("fused_qkv", 4, M, K, sum(widths), 128, 0, parts[0].a_bf16,
                       np.concatenate([p.scales_f16 for p in parts], axis=1),
                       qweight=np.concatenate([p.qweight for p in parts], axis=1),
                       qzeros=np.concatenate([p.qzeros for p in parts], axis=1))
    fused = torch.from_numpy(tf.tf_pack_concat(blobs)).cuda()
    y = gu.run(whole, kind, blob_dev=fused)
    gu.check_against_oracle(whole, y)
    # and column block i of the fused result obeys the acceptance rule of part i on its own
    n0 = 0
    for p in parts:
        gu.check_against_oracle(p, y[:, n0:n0 + p.N].copy())
        n0 += p.N


@pytest.mark.parametrize("bits,K,N,g", [(4, 512, 200, 128), (4, 1024, 328, 256), (8, 384, 136, 128), (8, 512, 64, 512)])
def test_dequant_to_memory_is_bit_exact(bits, K, N, g):
    """The ablation baseline writes w = bf16((q - z) * s) to memory: (q - z) * s is exact in fp32 and in the oracle's
    fp64, so one round-to-nearest-even of the oracle's value must give the same bits."""
    p = wl.make_w4(1, K, N, seed=950 + K, group_size=g) if bits == 4 else wl.make_w8(1, K, N, seed=950 + K, group_size=g)
    blob = torch.from_numpy(gu.pack(p)).cuda()
    guard = 256
    buf = torch.full((guard + K * N + guard,), gu.CANARY, dtype=torch.int16, device="cuda")
    w = buf[guard:guard + K * N].view(torch.bfloat16).view(K, N)
    tf.tf_dequant_bf16(blob, w, bits, K, N)
    torch.cuda.synchronize()
    raw = buf.cpu().numpy().view(np.uint16)
    assert np.all(raw[:guard] == gu.CANARY) and np.all(raw[guard + K * N:] == gu.CANARY), "write outside w"
    ref = (orc.dequant_w4(p.qweight, p.scales_f16, p.qzeros, g) if bits == 4 else orc.dequant_w8(p.w_i8, p.scales_f16, g))
    ref32 = ref.astype(np.float32)
    assert np.array_equal(ref32.astype(np.float64), ref)             # exact in fp32, as claimed
    assert np.array_equal(raw[guard:guard + K * N].reshape(K, N), wl.f32_to_bf16_bits(ref32))


@pytest.mark.parametrize("M", [1, 2, 3])
def test_w8_gemv_non_finite_activation_is_not_hidden(M):
    """An Inf or NaN activation must not come out as a finite number: every output of that token is non-finite
    (NaN on the integer path of 1 and 2 tokens, Inf or NaN on the floating-point path), other tokens are untouched."""
    K, N = 512, 136
    p = wl.make_w8(M, K, N, seed=990 + M)
    clean = gu.run(p, "gemv")
    bits = p.a_bf16.copy()
    bits[0, 300] = 0x7F80                      # +Inf in token 0
    y = gu.run(p, "gemv", a_bits=bits)
    vals = bf16_bits_to_f64(y)
    assert not np.any(np.isfinite(vals[0]))
    if M > 1:
        assert np.array_equal(y[1:], clean[1:])


@pytest.mark.parametrize("first,second,M", [("gemv", "gemv", 16), ("gemv", "gemm", 16), ("gemm", "gemm", 96), ("gemm", "gemv", 8)])
def test_dependent_calls_without_host_sync(first, second, M):
    """The second call multiplies what the first one writes, on the same stream and workspace, with no host
    synchronisation in between.  Both kernels are launched so that they may start before their predecessor has
    finished; they must not read its output early (checked against the oracle applied to the first call's bits)."""
    K1, N1, N2 = 1024, 1024, 520
    p1 = wl.make_w4(M, K1, N1, seed=1001, scale_range=(0.002, 0.004))
    p2 = wl.make_w4(M, N1, N2, seed=1002)
    b1 = torch.from_numpy(gu.pack(p1)).cuda()
    b2 = torch.from_numpy(gu.pack(p2)).cuda()
    a = gu.to_device_bf16(p1.a_bf16)
    y1 = torch.empty((M, N1), dtype=torch.bfloat16, device="cuda")
    y2 = torch.empty((M, N2), dtype=torch.bfloat16, device="cuda")
    ops = {"gemv": (tf.tf_gemv_w4a16, tf.TF_OP_GEMV_W4A16), "gemm": (tf.tf_gemm_w4a16, tf.TF_OP_GEMM_W4A16)}
    need = max(tf.tf_workspace_size(ops[first][1], M, K1, N1), tf.tf_workspace_size(ops[second][1], M, N1, N2))
    ws = torch.zeros(need, dtype=torch.uint8, device="cuda")
    for _ in range(3):                                   # repeated: an early read would show up intermittently
        y1.fill_(float("nan"))
        y2.fill_(float("nan"))
        ops[first][0](b1, a, y1, M, K1, N1, ws)
        ops[second][0](b2, y1, y2, M, N1, N2, ws)
        assert tf.tf_device_status(ws) == 0
        torch.cuda.synchronize()
        gu.check_against_oracle(p1, gu.bits_of(y1))
        p2.a_bf16 = gu.bits_of(y1)
        gu.check_against_oracle(p2, gu.bits_of(y2))


def test_gemv_on_two_streams_with_their_own_workspaces():
    """Calls on different streams may run concurrently when each stream has its own workspace; what the library
    remembers about the last launch per stream only steers overlap and must not affect results."""
    shapes = [(1, 1024, 1024), (16, 1024, 712), (4, 2048, 328), (16, 512, 4096)]
    probs = [wl.make_w4(M, K, N, seed=1100 + i) for i, (M, K, N) in enumerate(shapes)]
    blobs = [torch.from_numpy(gu.pack(p)).cuda() for p in probs]
    acts = [gu.to_device_bf16(p.a_bf16) for p in probs]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    wss = [torch.zeros(tf.tf_workspace_size(tf.TF_OP_GEMV_W4A16, 16, 4096, 4096), dtype=torch.uint8, device="cuda") for _ in range(2)]
    ys = [[torch.empty((p.M, p.N), dtype=torch.bfloat16, device="cuda") for p in probs] for _ in range(2)]
    torch.cuda.synchronize()
    for rep in range(4):
        for i, p in enumerate(probs):
            for s in range(2):                            # the same call alternately on the two streams
                tf.tf_gemv_w4a16(blobs[i], acts[i], ys[s][i], p.M, p.K, p.N, wss[s], stream=streams[s])
    for s in range(2):
        assert tf.tf_device_status(wss[s], stream=streams[s]) == 0
    torch.cuda.synchronize()
    for i, p in enumerate(probs):
        gu.check_against_oracle(p, gu.bits_of(ys[0][i]))
        assert np.array_equal(gu.bits_of(ys[0][i]), gu.bits_of(ys[1][i]))      # same inputs, bit-identical outputs


def test_gemv_and_gemm_share_one_workspace():
    """One workspace of the largest size serves every call of a stream, in any order: the GEMV's partial sums of cut
    strips and the GEMM's flags must not use the same bytes, and both leave the head of it zero."""
    Mv, Mm, K, N = 4, 160, 4096, 4096                       # both shapes cut strips / tiles between CTAs
    pv = wl.make_w4(Mv, K, N, seed=1201)
    pm = wl.make_w4(Mm, K, N, seed=1202)
    bv, bm = torch.from_numpy(gu.pack(pv)).cuda(), torch.from_numpy(gu.pack(pm)).cuda()
    av, am = gu.to_device_bf16(pv.a_bf16), gu.to_device_bf16(pm.a_bf16)
    yv = torch.empty((Mv, N), dtype=torch.bfloat16, device="cuda")
    ym = torch.empty((Mm, N), dtype=torch.bfloat16, device="cuda")
    need = max(tf.tf_workspace_size(tf.TF_OP_GEMV_W4A16, Mv, K, N), tf.tf_workspace_size(tf.TF_OP_GEMM_W4A16, Mm, K, N))
    ws = torch.zeros(need, dtype=torch.uint8, device="cuda")
    for order in ("vm", "mv", "vvm", "mmv"):
        yv.fill_(float("nan"))
        ym.fill_(float("nan"))
        for op in order:
            if op == "v":
                tf.tf_gemv_w4a16(bv, av, yv, Mv, K, N, ws)
            else:
                tf.tf_gemm_w4a16(bm, am, ym, Mm, K, N, ws)
        assert tf.tf_device_status(ws) == 0
        assert int(ws[:WORKSPACE_ZERO_BYTES].to(torch.int32).sum().item()) == 0
        gu.check_against_oracle(pv, gu.bits_of(yv))
        gu.check_against_oracle(pm, gu.bits_of(ym))


def _same_sign_problem(bits, M, K, N, seed):
    """Worst case for rounding: every product a * w has the same sign, so |y| equals the bound sum_k |a_k w_k| and
    nothing cancels -- the output rounding alone may use half of the tolerance, a rounded weight operand the rest."""
    p = wl.make_w4(M, K, N, seed=seed) if bits == 4 else wl.make_w8(M, K, N, seed=seed)
    p.a_bf16 = p.a_bf16 & np.uint16(0x7FFF)                         # a >= 0
    rng = np.random.default_rng(seed + 1)
    if bits == 4:
        z = rng.integers(0, 8, size=(K // 128, N), dtype=np.uint8)
        q = (np.repeat(z, 128, axis=0) + rng.integers(1, 9, size=(K, N), dtype=np.uint8)).astype(np.uint8)   # q > z
        p.qweight, p.qzeros = wl.awq_pack_words(q), wl.awq_pack_words(z)
    else:
        p.w_i8 = np.abs(p.w_i8.astype(np.int16)).clip(1, 127).astype(np.int8)
    return p


@pytest.mark.parametrize("kind,bits,M,K,N", [("gemv", 4, 1, 4096, 1024), ("gemv", 4, 7, 4096, 1024), ("gemv", 4, 16, 2048, 1096),
                                            ("gemv", 8, 2, 4096, 512), ("gemv", 8, 6, 2048, 512)])
def test_same_sign_inputs_gemv_stays_within_the_stated_tolerance(kind, bits, M, K, N):
    """The GEMV keeps the weights exact, so its only rounding of note is the bf16 output: up to 2^-8 of |y| = B,
    which is 0.98 of the stated tolerance when y sits just above a power of two."""
    p = _same_sign_problem(bits, M, K, N, seed=1300 + M)
    gu.check_against_oracle(p, gu.run(p, kind))


@pytest.mark.parametrize("bits,M,K,N", [(4, 200, 4096, 1024), (4, 40, 8192, 512), (8, 130, 4096, 512)])
def test_same_sign_inputs_gemm_stays_within_two_roundings(bits, M, K, N):
    """The GEMM multiplies w = bf16((q - z) * s) (Section 4.1: dequantize once, then the bf16 tensor-core product), so
    in the worst case -- nothing cancels, every weight and the output rounded the same way -- two bf16 roundings add up:
    |err| <= 2 * 2^-8 * B.  The stated tolerance 4e-3 * B is one bf16 rounding (2^-8 = 3.9e-3); it holds with a wide
    margin on the seeded inputs of every configuration (asserted by the parity tests), and this adversarial input is
    held to the two-rounding bound instead, with the observed ratio to the stated tolerance kept below 1.5."""
    p = _same_sign_problem(bits, M, K, N, seed=1300 + M)
    y_bits = gu.run(p, "gemm")
    y_ref, bound = orc.solve(p)
    err = np.abs(bf16_bits_to_f64(y_bits) - y_ref)
    assert np.all(err <= 2.0 * 2.0 ** -8 * bound + 1e-5)
    assert float(np.max(err / (4e-3 * bound + 1e-5))) <= 1.5


@pytest.mark.parametrize("M,K,N,parts", [(1, 4096, 1096, 3), (16, 2048, 4096, 4), (5, 1024, 200, 2)])
def test_column_shards_reassemble_to_the_full_product(M, K, N, parts):
    """Section 4.4: every worker owns distinct output columns and needs nothing from the others.  Each shard's GEMV
    (blob cut out by tf_pack_shard, N = the shard's column count) fills its column range of y; the assembled result
    passes parity against the oracle on the whole matrix."""
    p = wl.make_w4(M, K, N, seed=1600 + M)
    full = gu.pack(p)
    a = gu.to_device_bf16(p.a_bf16)
    y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    ws = torch.zeros(tf.tf_workspace_size(tf.TF_OP_GEMV_W4A16, M, K, N), dtype=torch.uint8, device="cuda")
    for part in range(parts):
        n0, nc = tf.tf_shard_columns(N, part, parts)
        shard = torch.from_numpy(tf.tf_pack_shard(full, part, parts)).cuda()
        y_part = torch.empty((M, nc), dtype=torch.bfloat16, device="cuda")
        tf.tf_gemv_w4a16(shard, a, y_part, M, K, nc, ws)
        y[:, n0:n0 + nc] = y_part
    assert tf.tf_device_status(ws) == 0
    gu.check_against_oracle(p, gu.bits_of(y))
