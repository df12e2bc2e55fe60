"""GPU parity: the CUDA library, called through its C ABI, against the CPU oracle on the same
seeded inputs.  Integer / byte work must be bit-exact; products must satisfy
max|y_gpu - y_ref| <= 5e-3 * max|y_ref|."""
import numpy as np
import pytest
import torch

import oracle
from helpers import lut_max_units, TOL, make_layer, rel_err, tiled_operands
from paper_2407_02891_b200 import binding as bq
from paper_2407_02891_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def gpu_layer(N, K, q, group, layout, codes, alpha, z):
    return bq.pack_layer(N, K, q, group, layout, dev(codes), dev(alpha), dev(z))


def run_gemv(layer, x, plan=None):
    y = torch.full((layer.d.N,), float("nan"), dtype=torch.float16, device=DEV)
    xd = dev(x.reshape(-1))
    if plan is None:
        ws = bq.new_workspace(layer.d, 1)
        bq.gemv(layer.d, layer.packed, layer.alpha, layer.z, xd, y, ws)
    else:
        ws = bq.new_workspace(layer.d, 1, plan)
        bq.gemv_plan(layer.d, plan, layer.packed, layer.alpha, layer.z, xd, y, ws)
    torch.cuda.synchronize()
    return y.cpu().numpy().astype(np.float64)


# ---------------------------------------------------------------------------------------
# packing / repacking: bit-exact
# ---------------------------------------------------------------------------------------

@pytest.mark.parametrize("N,K,q,group", [(16, 32, 3, 32), (16, 32, 3, 0), (40, 1024, 3, 128), (24, 512, 2, 128),
                                         (8, 1536, 4, 128), (72, 512, 1, 0), (13, 96, 3, 32)])
def test_pack_canonical_bit_exact(N, K, q, group):
    p, codes, alpha, z, _ = make_layer(f"pack/{N}x{K}", N, K, q, group)
    L = gpu_layer(N, K, q, group, bq.LAYOUT_CANONICAL, codes, alpha, z)
    assert np.array_equal(L.packed.cpu().numpy(), oracle.pack_canonical(codes, q).ravel())
    assert np.array_equal(L.alpha.cpu().numpy().view(np.uint16), alpha.ravel().view(np.uint16))
    assert np.array_equal(L.z.cpu().numpy().view(np.uint16), z.ravel().view(np.uint16))


@pytest.mark.parametrize("N,K,q,group", [(40, 1024, 3, 128), (24, 512, 2, 128), (8, 1536, 4, 128), (72, 512, 1, 0),
                                         (296, 2048, 3, 128), (64, 1024, 2, 0), (40, 1024, 3, 64), (24, 512, 2, 32),
                                         (8, 1536, 4, 32), (72, 512, 1, 64), (296, 2048, 3, 32), (64, 1024, 4, 64)])
def test_pack_tiled_and_repack_bit_exact(N, K, q, group):
    p, codes, alpha, z, _ = make_layer(f"tile/{N}x{K}", N, K, q, group)
    canon = oracle.pack_canonical(codes, q)
    want_p, want_a, want_z = tiled_operands(canon, alpha, z, group)
    T = gpu_layer(N, K, q, group, bq.LAYOUT_TILED, codes, alpha, z)
    assert T.packed.numel() == want_p.size == bq.packed_bytes(T.d)
    assert np.array_equal(T.packed.cpu().numpy(), want_p)
    if group == 0:
        assert np.array_equal(T.alpha.cpu().numpy().view(np.uint16), want_a.view(np.uint16))
        assert np.array_equal(T.z.cpu().numpy().view(np.uint16), want_z.view(np.uint16))
    else:
        assert T.alpha is None and T.z is None
    # canonical -> tiled via repack gives the same bytes; tiled -> canonical is the inverse
    C = gpu_layer(N, K, q, group, bq.LAYOUT_CANONICAL, codes, alpha, z)
    p2, a2, z2 = bq.empty_operands(T.d, DEV)
    p2.zero_()
    bq.repack(C.d, C.packed, C.alpha, C.z, T.d, p2, a2, z2)
    assert torch.equal(p2, T.packed)
    if group == 0:
        assert torch.equal(a2.view(torch.int16), T.alpha.view(torch.int16))
        assert torch.equal(z2.view(torch.int16), T.z.view(torch.int16))
    p3, a3, z3 = torch.zeros_like(C.packed), torch.zeros_like(C.alpha), torch.zeros_like(C.z)
    bq.repack(T.d, p2, a2, z2, C.d, p3, a3, z3)
    assert np.array_equal(p3.cpu().numpy(), canon.ravel())
    assert np.array_equal(a3.cpu().numpy().view(np.uint16), alpha.ravel().view(np.uint16))
    assert np.array_equal(z3.cpu().numpy().view(np.uint16), z.ravel().view(np.uint16))


# ---------------------------------------------------------------------------------------
# linear-int -> merged binary code: bit-exact codes, alpha, z
# ---------------------------------------------------------------------------------------

def _partitions(n, q):
    out = []

    def rec(i, assign, used):
        if i == n:
            if used == q:
                out.append(list(assign))
            return
        for j in range(min(used + 1, q)):
            rec(i + 1, assign + [j], max(used, j + 1))

    rec(0, [], 0)
    return out


@pytest.mark.parametrize("N,K,group,n,q", [(16, 32, 32, 4, 3), (16, 32, 0, 4, 3), (16, 32, 32, 5, 3),
                                           (64, 512, 128, 5, 2), (16, 32, 32, 3, 2), (24, 256, 64, 4, 4)])
def test_merge_linear_bit_exact(N, K, group, n, q):
    w, S, qbias = synth.linear_int_case(f"merge/n{n}", N, K, group, n)
    d = bq.desc(N, K, q, group)
    G = d.G
    for b2p in _partitions(n, q):
        codes = torch.zeros((N, K), dtype=torch.uint8, device=DEV)
        alpha = torch.zeros((q, N, G), dtype=torch.float16, device=DEV)
        z = torch.zeros((N, G), dtype=torch.float16, device=DEV)
        bq.merge_linear(d, dev(w), dev(S), dev(qbias), n, b2p, codes, alpha, z)
        rc, ra, rz = oracle.merge_linear(w, S, qbias, group, n, b2p)
        assert np.array_equal(codes.cpu().numpy(), rc)
        assert np.array_equal(alpha.cpu().numpy().view(np.uint16), ra.view(np.uint16))
        assert np.array_equal(z.cpu().numpy().view(np.uint16), rz.view(np.uint16))


def test_merge_linear_rounds_general_scales_like_the_oracle():
    """S, qbias with full 11-bit significands: alpha and z need a real rounding to fp16."""
    N, K, group, n, q = 32, 256, 64, 5, 3
    w, _, _ = synth.linear_int_case("merge/general", N, K, group, n)
    G = K // group
    S = (0.002 + 0.03 * synth.uniform("merge/general/S", 0, N * G)).astype(np.float16).reshape(N, G)
    qbias = (synth.normal("merge/general/b", 0, N * G) * 0.1).astype(np.float16).reshape(N, G)
    d = bq.desc(N, K, q, group)
    b2p = [0, 1, 1, 2, 2]
    codes = torch.zeros((N, K), dtype=torch.uint8, device=DEV)
    alpha = torch.zeros((q, N, G), dtype=torch.float16, device=DEV)
    z = torch.zeros((N, G), dtype=torch.float16, device=DEV)
    bq.merge_linear(d, dev(w), dev(S), dev(qbias), n, b2p, codes, alpha, z)
    rc, ra, rz = oracle.merge_linear(w, S, qbias, group, n, b2p)
    assert np.array_equal(codes.cpu().numpy(), rc)
    assert np.array_equal(alpha.cpu().numpy().view(np.uint16), ra.view(np.uint16))
    assert np.array_equal(z.cpu().numpy().view(np.uint16), rz.view(np.uint16))


def test_tiny_case_end_to_end():
    """16 x 32, 4-bit linear codes -> 3 planes -> pack -> product, against the oracle chain."""
    N, K, group, n, q = 16, 32, 32, 4, 3
    w, S, qbias = synth.linear_int_case("tiny/e2e", N, K, group, n)
    x = synth.activations("tiny/e2e", 1, K)
    d = bq.desc(N, K, q, group)
    for b2p in _partitions(n, q):
        codes = torch.zeros((N, K), dtype=torch.uint8, device=DEV)
        alpha = torch.zeros((q, N, 1), dtype=torch.float16, device=DEV)
        z = torch.zeros((N, 1), dtype=torch.float16, device=DEV)
        bq.merge_linear(d, dev(w), dev(S), dev(qbias), n, b2p, codes, alpha, z)
        L = bq.pack_layer(N, K, q, group, bq.LAYOUT_CANONICAL, codes, alpha, z)
        y = run_gemv(L, x)
        rc, ra, rz = oracle.merge_linear(w, S, qbias, group, n, b2p)
        ref = oracle.forward_dequant(rc, ra, rz, x, group)[0]
        assert rel_err(y, ref) <= TOL


# ---------------------------------------------------------------------------------------
# products
# ---------------------------------------------------------------------------------------

@pytest.mark.parametrize("N,K,q,group", [(16, 32, 3, 32), (13, 96, 3, 32), (50, 256, 2, 64), (33, 1024, 4, 0),
                                         (1024, 1024, 3, 128), (7, 2048, 1, 128)])
def test_gemv_generic_kernel(N, K, q, group):
    p, codes, alpha, z, x = make_layer(f"gen/{N}x{K}", N, K, q, group)
    ref = oracle.forward_planes(p, alpha, z, x, group)[0]
    L = gpu_layer(N, K, q, group, bq.LAYOUT_CANONICAL, codes, alpha, z)
    assert rel_err(run_gemv(L, x), ref) <= TOL


LUT_SHAPES = [(1024, 1024, 3, 128), (8, 512, 3, 128), (296, 2048, 3, 128), (1000, 1536, 2, 128),
              (520, 3584, 3, 128), (64, 1024, 1, 128), (136, 1024, 4, 128), (4096, 4096, 3, 128),
              # one scale per row (the paper's granularity)
              (1024, 1024, 2, 0), (8, 512, 3, 0), (296, 2048, 2, 0), (520, 3584, 3, 0), (136, 1024, 4, 0),
              (64, 1024, 1, 0), (2304, 9216, 2, 0)]


@pytest.mark.parametrize("N,K,q,group,B", [
    (1, 32, 1, 32, 1),          # one row, one word
    (17, 96, 3, 32, 2),         # a row beyond the first sixteen; a segment of three words
    (33, 544, 2, 0, 16),        # two windows, the second a single word; K split over a cluster of two
    (40, 480, 4, 96, 5),        # scaling units of three words that straddle segments
    (23, 1120, 3, 160, 1),
    (16, 2048, 3, 64, 9),
    (300, 11008, 3, 128, 1),    # 22 windows over eight blocks
    (48, 11008, 2, 256, 16),    # phases: 16 columns' x does not fit at once
    (5000, 1024, 3, 128, 4),    # more 16-row blocks than two per SM
    (64, 3072, 1, 3072, 3),     # one scaling unit, given as a group
])
def test_canonical_products(N, K, q, group, B):
    """Every scaling-unit form, row and K remainder, cluster split and phase of the canonical kernel.  The bound: one
    rounding to fp16 (2^-11 of the value) plus fp32 sums, far below the other half."""
    p, codes, alpha, z, X = make_layer(f"canon/{N}x{K}q{q}g{group}", N, K, q, group, B)
    ref = oracle.forward_planes(p, alpha, z, X, group)
    L = gpu_layer(N, K, q, group, bq.LAYOUT_CANONICAL, codes, alpha, z)
    Y = torch.full((B, N), float("nan"), dtype=torch.float16, device=DEV)
    bq.gemm_smallbatch(L.d, L.packed, L.alpha, L.z, dev(X), Y, B, None)
    torch.cuda.synchronize()
    assert rel_err(Y.cpu().numpy(), ref) <= 2.0 ** -10
    Y2 = torch.zeros_like(Y)
    bq.gemm_smallbatch(L.d, L.packed, L.alpha, L.z, dev(X), Y2, B, None)
    torch.cuda.synchronize()
    assert torch.equal(Y.view(torch.int16), Y2.view(torch.int16))


@pytest.mark.parametrize("N,K,q,group,B", [(17, 640, 3, 128, 1), (17, 768, 2, 256, 9), (16, 1408, 1, 128, 4), (33, 1792, 4, 256, 2),
                                           (17, 608, 3, 32, 1), (16, 992, 2, 0, 3)])
def test_canonical_products_use_no_scale_but_a_rows_own(N, K, q, group, B):
    """The last window of 512 weights is a partial one: NaN right behind the scales, and in one row's scales, shows in no
    other row.  (alpha and z are views of larger buffers, whose tails are the NaN.)  Bound as above."""
    p, codes, alpha, z, X = make_layer(f"own/{N}x{K}q{q}g{group}", N, K, q, group, B)
    ref = oracle.forward_planes(p, alpha, z, X, group)
    bad = N // 2
    alpha, z = alpha.copy(), z.copy()
    alpha[:, bad], z[bad] = np.nan, np.nan

    def framed(a):
        own = torch.full((a.size + 64,), float("nan"), dtype=torch.float16, device=DEV)
        own[:a.size] = dev(a).reshape(-1)
        return own[:a.size]

    L = gpu_layer(N, K, q, group, bq.LAYOUT_CANONICAL, codes, alpha, z)
    Y = torch.zeros((B, N), dtype=torch.float16, device=DEV)
    bq.gemm_smallbatch(L.d, L.packed, framed(alpha), framed(z), dev(X), Y, B, None)
    torch.cuda.synchronize()
    y, others = Y.cpu().numpy(), np.arange(N) != bad
    assert np.isnan(y[:, bad]).all()
    assert rel_err(y[:, others], ref[:, others]) <= 2.0 ** -10


@pytest.mark.parametrize("group,B", [(32, 1), (32, 9), (0, 1), (0, 9), (256, 2)])
def test_canonical_sums_do_not_drift_along_the_row(group, B):
    """65536 positive terms, one block per 16 rows: whatever a running sum loses at each step adds up.  A segment of 128 is 8 steps
    of the tensor cores, at most 2^-23 each; each warp then adds 64 of them, and the eight warps' sums are added, with roundings
    of 2^-24: 2^-17.5 in all, beside the one rounding to fp16."""
    N, K, L = 1200, 65536, group or 65536
    rng = np.random.default_rng(group + B)
    alpha = rng.uniform(0.25, 1.0, (1, N, K // L)).astype(np.float16)
    X = np.exp2(rng.uniform(-17, -7, (B, K))).astype(np.float16)
    ref = X.astype(np.float64).reshape(B, K // L, L).sum(axis=2) @ alpha[0].astype(np.float64).T
    d = bq.desc(N, K, 1, group, bq.LAYOUT_CANONICAL)
    Y = torch.zeros((B, N), dtype=torch.float16, device=DEV)
    bq.gemm_smallbatch(d, torch.full((N * K // 8,), 255, dtype=torch.uint8, device=DEV), dev(alpha.reshape(-1)),
                       torch.zeros(N * K // L, dtype=torch.float16, device=DEV), dev(X), Y, B, None)
    torch.cuda.synchronize()
    half_step = np.exp2(np.floor(np.log2(ref)) - 11)
    assert (np.abs(Y.cpu().numpy().astype(np.float64) - ref) <= half_step + 2.0 ** -17.5 * ref).all()


@pytest.mark.parametrize("N,K,q,group", LUT_SHAPES)
def test_gemv_lut_kernel_default_plan(N, K, q, group):
    p, codes, alpha, z, x = make_layer(f"lut/{N}x{K}", N, K, q, group)
    ref = oracle.forward_planes(p, alpha, z, x, group)[0]
    L = gpu_layer(N, K, q, group, bq.LAYOUT_TILED, codes, alpha, z)
    assert bq.plan_default(L.d).kernel == 1
    assert rel_err(run_gemv(L, x), ref) <= TOL


@pytest.mark.parametrize("group", [128, 0])
@pytest.mark.parametrize("N,K,q,rb,ks", [(520, 3584, 3, 2, 1), (520, 3584, 3, 2, 7), (520, 3584, 3, 3, 2),
                                         (520, 3584, 3, 65, 3), (520, 3584, 3, 5, 4), (512, 1024, 2, 1, 1),
                                         (512, 1024, 2, 1, 2), (1000, 1536, 2, 125, 3), (1000, 1536, 2, 2, 1),
                                         (1472, 1024, 3, 1, 2), (4000, 512, 2, 3, 1)])
def test_gemv_lut_kernel_explicit_plans(N, K, q, rb, ks, group):
    """Ragged row blocks, one and several windows per block, with and without split-K."""
    p, codes, alpha, z, x = make_layer(f"lutp/{N}x{K}", N, K, q, group)
    ref = oracle.forward_planes(p, alpha, z, x, group)[0]
    L = gpu_layer(N, K, q, group, bq.LAYOUT_TILED, codes, alpha, z)
    assert rel_err(run_gemv(L, x, bq.Plan(1, rb, ks, 0)), ref) <= TOL


def test_gemv_workspace_is_reusable_and_result_deterministic():
    N, K, q = 520, 3584, 3
    p, codes, alpha, z, x = make_layer("lut/reuse", N, K, q, 128)
    L = gpu_layer(N, K, q, 128, bq.LAYOUT_TILED, codes, alpha, z)
    plan = bq.Plan(1, 3, 7, 0)
    ws = bq.new_workspace(L.d, 1, plan)
    xd = dev(x.reshape(-1))
    ys = []
    for _ in range(3):
        y = torch.zeros(N, dtype=torch.float16, device=DEV)
        bq.gemv_plan(L.d, plan, L.packed, L.alpha, L.z, xd, y, ws)
        ys.append(y)
    torch.cuda.synchronize()
    assert torch.equal(ys[0].view(torch.int16), ys[1].view(torch.int16))
    assert torch.equal(ys[0].view(torch.int16), ys[2].view(torch.int16))
    ref = oracle.forward_planes(p, alpha, z, x, 128)[0]
    assert rel_err(ys[2].cpu().numpy(), ref) <= TOL


@pytest.mark.parametrize("layout", [bq.LAYOUT_CANONICAL, bq.LAYOUT_TILED])
def test_gemv_structured_inputs(layout):
    N, K, q, group = 64, 1024, 3, 128
    p, codes, alpha, z, x = make_layer("struct", N, K, q, group)
    W = oracle.dequant(codes, alpha, z, group)
    L = gpu_layer(N, K, q, group, layout, codes, alpha, z)
    # unit vectors return columns of the dequantised matrix (rounded to fp16 once)
    for k in (0, 7, 8, 15, 16, 127, 128, 511, 512, 1023):
        e = np.zeros((1, K), np.float16)
        e[0, k] = 1.0
        y = run_gemv(L, e)
        assert np.abs(y - W[:, k]).max() <= 2.0 ** -10 * np.abs(W[:, k]).max() + 1e-7
    # all planes +1
    ones = np.full_like(codes, (1 << q) - 1)
    L1 = gpu_layer(N, K, q, group, layout, ones, alpha, z)
    ref = oracle.forward_dequant(ones, alpha, z, x, group)[0]
    assert rel_err(run_gemv(L1, x), ref) <= TOL
    # alpha = 0: only the offsets remain
    L0 = gpu_layer(N, K, q, group, layout, codes, np.zeros_like(alpha), z)
    ref = oracle.forward_dequant(codes, np.zeros_like(alpha), z, x, group)[0]
    assert rel_err(run_gemv(L0, x), ref) <= TOL
    # a single non-zero group
    xg = np.zeros((1, K), np.float16)
    xg[0, 384:512] = x[0, 384:512]
    ref = oracle.forward_dequant(codes, alpha, z, xg, group)[0]
    assert rel_err(run_gemv(L, xg), ref) <= TOL
    # negative and zero scales are legal
    a2 = alpha.copy()
    a2[1] = -a2[1]
    a2[2, ::2] = 0
    L2 = gpu_layer(N, K, q, group, layout, codes, a2, z)
    ref = oracle.forward_dequant(codes, a2, z, x, group)[0]
    assert rel_err(run_gemv(L2, x), ref) <= TOL


@pytest.mark.parametrize("layout,N,K,q,group", [(bq.LAYOUT_CANONICAL, 50, 256, 3, 64), (bq.LAYOUT_TILED, 264, 1024, 3, 128),
                                                (bq.LAYOUT_CANONICAL, 16, 32, 3, 32), (bq.LAYOUT_TILED, 64, 512, 2, 0)])
@pytest.mark.parametrize("B", [1, 2, 3, 4, 8, 16])
def test_gemm_smallbatch(layout, N, K, q, group, B):
    p, codes, alpha, z, X = make_layer(f"sb/{N}x{K}", N, K, q, group, B)
    ref = oracle.forward_planes(p, alpha, z, X, group)
    L = gpu_layer(N, K, q, group, layout, codes, alpha, z)
    Y = torch.full((B, N), float("nan"), dtype=torch.float16, device=DEV)
    ws = bq.new_workspace(L.d, B)
    bq.gemm_smallbatch(L.d, L.packed, L.alpha, L.z, dev(X), Y, B, ws)
    torch.cuda.synchronize()
    Yh = Y.cpu().numpy()
    assert rel_err(Yh, ref) <= TOL
    if B > 1:
        # permuting the batch permutes the result bit for bit
        perm = np.roll(np.arange(B), 1)
        Y2 = torch.zeros_like(Y)
        bq.gemm_smallbatch(L.d, L.packed, L.alpha, L.z, dev(X[perm]), Y2, B, ws)
        torch.cuda.synchronize()
        assert np.array_equal(Y2.cpu().numpy().view(np.uint16), Yh[perm].view(np.uint16))


@pytest.mark.parametrize("N,K,q,group,rb,ks,B", [
    (264, 1024, 3, 128, 1, 1, 2),      # 33 units: an odd number, the last pair is a single tile
    (264, 1024, 3, 128, 1, 2, 8),      # split-K, both windows apart
    (264, 2048, 3, 128, 3, 2, 16),     # 11 units per block, two windows per split, wide
    (1408, 1536, 3, 128, 1, 1, 5),     # 176 units: every warp four pairs, three windows
    (1408, 1536, 3, 128, 1, 3, 9),
    (776, 2560, 2, 128, 2, 1, 4),      # 97 units -> 48 + 49
    (776, 2560, 2, 0, 2, 5, 16),       # one scale per row
    (512, 1024, 1, 128, 4, 1, 3),
    (512, 1024, 4, 128, 4, 2, 12),
    (512, 1024, 4, 0, 1, 1, 7),
    (8, 512, 3, 128, 1, 1, 2),         # one unit, one window
    (16, 16384, 3, 128, 1, 1, 16),     # 32 windows in one block
])
def test_small_batch_kernel_explicit_plans(N, K, q, group, rb, ks, B):
    """The tensor-core small-batch kernel under decompositions chosen by the caller."""
    p, codes, alpha, z, X = make_layer(f"mma/{N}x{K}q{q}g{group}", N, K, q, group, B)
    ref = oracle.forward_planes(p, alpha, z, X, group)
    L = gpu_layer(N, K, q, group, bq.LAYOUT_TILED, codes, alpha, z)
    plan = bq.Plan(2, rb, ks, 0)
    ws = bq.new_workspace(L.d, B, plan)
    Y = torch.full((B, N), float("nan"), dtype=torch.float16, device=DEV)
    for _ in range(2):   # the second call finds the counters as the first one left them
        bq.gemm_smallbatch_plan(L.d, plan, L.packed, L.alpha, L.z, dev(X), Y, B, ws)
    torch.cuda.synchronize()
    bq.poll_status()
    assert rel_err(Y.cpu().numpy(), ref) <= TOL
    # through the lookup-table kernel (two columns per pass with group 128, one with per-row scales):
    # the same numbers up to rounding
    p1 = bq.plan_default(L.d, 1)
    Y1 = torch.zeros_like(Y)
    bq.gemm_smallbatch_plan(L.d, p1, L.packed, L.alpha, L.z, dev(X), Y1, B, bq.new_workspace(L.d, B, p1))
    torch.cuda.synchronize()
    bq.poll_status()
    assert rel_err(Y1.cpu().numpy(), ref) <= TOL


@pytest.mark.parametrize("N,K,q,rb,ks,B", [
    (264, 1024, 3, 1, 1, 2),       # 33 units, both windows in one block
    (264, 1024, 3, 1, 2, 2),       # split-K
    (1472, 1536, 3, 1, 3, 2),      # 184 units: every consumer warp eight units
    (776, 2560, 2, 2, 5, 3),       # a pair and a single column
    (512, 1024, 1, 4, 1, 4),
    (512, 1024, 4, 4, 2, 5),
    (8, 512, 3, 1, 1, 2),          # one unit, one window
    (16, 16384, 3, 1, 1, 2),       # 32 windows in one block
])
def test_lookup_kernel_on_column_pairs(N, K, q, rb, ks, B):
    """Plan kernel 1 with group 128 runs two columns per launch (both columns' sums in one table entry)."""
    group = 128
    p, codes, alpha, z, X = make_layer(f"pair/{N}x{K}q{q}", N, K, q, group, B)
    ref = oracle.forward_planes(p, alpha, z, X, group)
    L = gpu_layer(N, K, q, group, bq.LAYOUT_TILED, codes, alpha, z)
    plan = bq.Plan(1, rb, ks, 0)
    ws = bq.new_workspace(L.d, B, plan)
    Y = torch.full((B, N), float("nan"), dtype=torch.float16, device=DEV)
    for _ in range(2):   # the second call finds the counters as the first one left them
        bq.gemm_smallbatch_plan(L.d, plan, L.packed, L.alpha, L.z, dev(X), Y, B, ws)
    torch.cuda.synchronize()
    bq.poll_status()
    Yh = Y.cpu().numpy()
    assert rel_err(Yh, ref) <= TOL
    # each column equals the batch-1 product of that column bit for bit (same table values, same order of sums)
    y1 = torch.zeros(N, dtype=torch.float16, device=DEV)
    ws1 = bq.new_workspace(L.d, 1, plan)
    for b in range(B):
        bq.gemv_plan(L.d, plan, L.packed, L.alpha, L.z, dev(X[b]), y1, ws1)
        torch.cuda.synchronize()
        assert np.array_equal(y1.cpu().numpy().view(np.uint16), Yh[b].view(np.uint16))


@pytest.mark.parametrize("N,K,q,group,rb,ks,B", [
    (1408, 16384, 4, 128, 1, 1, 16),   # phases: 176 units and 32 windows in one block, one ring slot per warp
    (1400, 8704, 4, 0, 1, 1, 9),       # phases of unequal length, an odd number of units, scales per row
    (24, 1536, 2, 0, 1, 1, 16),        # six jobs on sixteen warps: every pair is shared
    (8, 2560, 3, 128, 1, 1, 3),        # one unit, five windows
    (272, 3584, 1, 128, 1, 1, 8),      # 17 pairs x 7 windows: runs that end inside a pair
    (640, 4608, 3, 128, 5, 9, 11),     # nine arrivals per word
])
def test_small_batch_kernel_shares_pairs_and_phases(N, K, q, group, rb, ks, B):
    """Every way the (pair, window) jobs can fall on the warps.  Products are exact, sums fp32: what is left is one rounding
    to fp16 (2^-11 of the value) and sums of K fp32 terms, far below the other half of the bound."""
    p, codes, alpha, z, X = make_layer(f"share/{N}x{K}q{q}", N, K, q, group, B)
    ref = oracle.forward_planes(p, alpha, z, X, group)
    L = gpu_layer(N, K, q, group, bq.LAYOUT_TILED, codes, alpha, z)
    plan = bq.Plan(2, rb, ks, 0)
    ws = bq.new_workspace(L.d, B, plan)
    Y = torch.full((B, N), float("nan"), dtype=torch.float16, device=DEV)
    for _ in range(2):
        bq.gemm_smallbatch_plan(L.d, plan, L.packed, L.alpha, L.z, dev(X), Y, B, ws)
    torch.cuda.synchronize()
    bq.poll_status()
    assert rel_err(Y.cpu().numpy(), ref) <= 2.0 ** -10
    if ws is not None:
        assert not ws.any()                # every word is cleared again


@pytest.mark.parametrize("N,K,q,B", [(1024, 4096, 3, 2), (776, 2560, 2, 3), (8, 512, 1, 2), (4096, 4096, 4, 3)])
def test_two_and_three_columns_with_one_scale_per_row_are_single_products(N, K, q, B):
    """By default: same bits as bcq_gemv on every column, with the workspace of a single product."""
    p, codes, alpha, z, X = make_layer(f"rows23/{N}x{K}q{q}", N, K, q, 0, B)
    L = gpu_layer(N, K, q, 0, bq.LAYOUT_TILED, codes, alpha, z)
    ws = bq.new_workspace(L.d, 1)
    Y = torch.zeros((B, N), dtype=torch.float16, device=DEV)
    bq.gemm_smallbatch(L.d, L.packed, L.alpha, L.z, dev(X), Y, B, ws)
    torch.cuda.synchronize()
    for b in range(B):
        assert np.array_equal(run_gemv(L, X[b]), Y[b].cpu().numpy().astype(np.float64))


def small_batch(N, K, q, group, rb, ks, codes, alpha, z, X):
    B = X.shape[0]
    L = gpu_layer(N, K, q, group, bq.LAYOUT_TILED, codes, alpha, z)
    plan = bq.Plan(2, rb, ks, 0)
    ws = bq.new_workspace(L.d, B, plan)
    Y = torch.zeros((B, N), dtype=torch.float16, device=DEV)
    for _ in range(2):
        bq.gemm_smallbatch_plan(L.d, plan, L.packed, L.alpha, L.z, dev(X), Y, B, ws)
    torch.cuda.synchronize()
    bq.poll_status()
    assert ws is None or not ws.any()
    return Y.cpu().numpy()


def far_apart_sums(N, K, q, B):
    """Groups of 128; in rows 0 .. 5, at the two ends of K: +inf and -inf; an infinity and a large finite sum of the other sign;
    each infinity alone; finite sums of 3.8e9 that cancel to 30000; one of 32000."""
    p, codes, alpha, z, X = make_layer(f"carry/{N}x{K}q{q}", N, K, q, 128, B)
    X = np.random.default_rng(K // 512).integers(400, 600, X.shape).astype(np.float16)
    X[:, -128:] = X[:, :128]
    X[:, -1] -= np.float16(0.5)                       # 60000 times the difference: 30000
    alpha, z = alpha.copy(), np.zeros_like(z)
    alpha[:, :, :4], alpha[:, :, -4:] = 0, 0          # the first and the last 512 weights: offsets only
    z[0, 0], z[0, -1] = np.inf, -np.inf
    z[1, 0], z[1, -1] = np.inf, -60000.0
    z[2, 0] = np.inf
    z[3, -1] = -np.inf
    z[4, 0], z[4, -1] = 60000.0, -60000.0
    z[5, 1] = 0.5
    with np.errstate(invalid="ignore"):
        return codes, alpha, z, X, oracle.forward_planes(p, alpha, z, X, 128)


def check_far_apart_sums(y, ref, cancelled):
    y = y.astype(np.float64)
    assert np.isnan(ref[:, 0]).all() and np.isnan(y[:, 0]).all()
    assert (y[:, 1] == np.inf).all() and (y[:, 2] == np.inf).all() and (y[:, 3] == -np.inf).all()
    assert cancelled < 20000 and np.abs(y[:, 4] - ref[:, 4]).max() <= cancelled
    # fp32 sums, then one rounding to fp16
    assert np.abs(y[:, 5:] - ref[:, 5:]).max() <= 2.0 ** -10 * np.abs(ref[:, 5:]).max()


@pytest.mark.parametrize("N,W,q,ks,rb,B", [(40, 4, 3, 4, 2, 3), (16, 64, 1, 64, 1, 2), (24, 128, 2, 128, 2, 9), (16, 16, 4, 16, 1, 16)])
def test_small_batch_splits_carry_any_partial_sum(N, W, q, ks, rb, B):
    """Infinities, and finite sums beyond what a split-K word holds, in different splits."""
    codes, alpha, z, X, ref = far_apart_sums(N, 512 * W, q, B)
    # row 4's sum may be of the order of 3.8e9 until the last split is added: half an fp32 step, 2^7, per addition
    check_far_apart_sums(small_batch(N, 512 * W, q, 128, rb, ks, codes, alpha, z, X), ref, 2.0 ** 7 * W)


@pytest.mark.parametrize("N,K,q,B", [(24, 4096, 3, 1), (16, 1152, 2, 16), (2500, 1024, 1, 2)])
def test_canonical_products_carry_any_partial_sum(N, K, q, B):
    """The same in the warps and the blocks of a cluster that share a row."""
    codes, alpha, z, X, ref = far_apart_sums(N, K, q, B)
    L = gpu_layer(N, K, q, 128, bq.LAYOUT_CANONICAL, codes, alpha, z)
    Y = torch.zeros((B, N), dtype=torch.float16, device=DEV)
    bq.gemm_smallbatch(L.d, L.packed, L.alpha, L.z, dev(X), Y, B, None)
    torch.cuda.synchronize()
    # two warps may carry row 4's 3.8e9 through all their K / 1024 + 1 segments' q + 1 additions each, then eight warps and blocks
    check_far_apart_sums(Y.cpu().numpy(), ref, 2.0 ** 7 * (2 * (K / 1024 + 1) * (q + 1) + 16))


@pytest.mark.parametrize("N,K,q,group,rb,ks,B", [(40, 2048, 3, 128, 2, 4, 5), (72, 1536, 1, 0, 1, 3, 16), (24, 1024, 4, 0, 1, 2, 3), (1400, 8704, 2, 128, 1, 2, 12)])
def test_small_batch_columns_that_are_not_numbers(N, K, q, group, rb, ks, B):
    """A column of NaN, a column with one infinity, activations of 65504 (sums beyond the split-K words, most of them beyond fp16):
    the other columns' bits are not disturbed, and these come out as the oracle has them."""
    p, codes, alpha, z, X = make_layer(f"nan/{N}x{K}q{q}", N, K, q, group, B)
    clean = small_batch(N, K, q, group, rb, ks, codes, alpha, z, X)
    X = X.copy()
    X[0], X[1, K // 2] = np.nan, np.inf
    X[2] = np.copysign(np.float16(65504.0), X[2])
    with np.errstate(invalid="ignore", over="ignore"):
        ref = oracle.forward_planes(p, alpha, z, X, group)
        want = ref.astype(np.float16).astype(np.float64)
    y = small_batch(N, K, q, group, rb, ks, codes, alpha, z, X)
    assert np.array_equal(y[3:].view(np.uint16), clean[3:].view(np.uint16))
    assert np.isnan(y[0]).all()
    assert np.array_equal(np.isnan(y[1]), np.isnan(want[1])) and np.array_equal(y[1][~np.isnan(want[1])], want[1][~np.isnan(want[1])])
    y2, near = y[2].astype(np.float64), np.abs(np.abs(ref[2]) - 65520.0) < 64.0   # (next to the largest fp16 number either side is right)
    assert np.array_equal(np.isinf(y2[~near]), np.isinf(want[2][~near])) and np.isinf(want[2]).any()
    finite = np.isfinite(y2) & ~near
    assert finite.any() and np.abs(y2 - ref[2])[finite].max() <= 2.0 ** 6


@pytest.mark.parametrize("N,W,q,ks,rb,B", [(48, 16, 3, 16, 3, 2), (16, 64, 1, 64, 1, 11), (128, 8, 2, 4, 2, 8)])
def test_small_batch_splits_keep_small_sums(N, W, q, ks, rb, B):
    """Outputs around 2^-16, below fp16's normal range: the one rounding to a multiple of 2^-24 is all that may be lost.  The
    signed sums of 128 activations are exact in fp32 (multiples of 2^-24 below 1); K / 128 (q + 1) fused multiply-adds to sums
    below 2^-13 lose at most 2^-38 each, the additions of the splits as much."""
    K, group = 512 * W, 128
    p, codes, alpha, z, X = make_layer(f"small/{N}x{K}q{q}", N, K, q, group, B)
    X = (X * np.float16(2.0 ** -19)).astype(np.float16)
    ref = oracle.forward_planes(p, alpha, z, X, group)
    assert 0 < np.abs(ref).max() < 2.0 ** -14
    y = small_batch(N, K, q, group, rb, ks, codes, alpha, z, X).astype(np.float64)
    assert np.abs(y - ref).max() <= 2.0 ** -25 + (K / 128 * (q + 1) + ks) * 2.0 ** -38


def test_small_batch_kernel_structured_inputs():
    """Unit activations pick out single weights: exact values, every (row, k) position distinguishable."""
    N, K, q, group, B = 64, 1024, 3, 128, 16
    p, codes, alpha, z, _ = make_layer("mma/struct", N, K, q, group, B)
    L = gpu_layer(N, K, q, group, bq.LAYOUT_TILED, codes, alpha, z)
    rng = np.random.default_rng(5)
    ks = rng.choice(K, size=B, replace=False)
    X = np.zeros((B, K), np.float16)
    X[np.arange(B), ks] = 1.0
    ref = oracle.forward_planes(p, alpha, z, X, group)     # = column ks[b] of the dequantised matrix
    Y = torch.zeros((B, N), dtype=torch.float16, device=DEV)
    bq.gemm_smallbatch(L.d, L.packed, L.alpha, L.z, dev(X), Y, B, bq.new_workspace(L.d, B))
    torch.cuda.synchronize()
    got = Y.cpu().numpy().astype(np.float64)
    assert np.abs(got - ref).max() <= 2.0 ** -10 * np.abs(ref).max()


def test_gemv_host_buffers():
    N, K, q, group = 520, 3584, 3, 128
    p, codes, alpha, z, x = make_layer("host", N, K, q, group)
    L = gpu_layer(N, K, q, group, bq.LAYOUT_TILED, codes, alpha, z)
    xh = torch.from_numpy(x.reshape(-1).copy()).pin_memory()
    yh = torch.zeros(N, dtype=torch.float16).pin_memory()
    xs = torch.zeros(K, dtype=torch.float16, device=DEV)
    ys = torch.zeros(N, dtype=torch.float16, device=DEV)
    ws = bq.new_workspace(L.d, 1)
    bq.gemv_host(L.d, L.packed, L.alpha, L.z, xh, yh, xs, ys, ws)
    torch.cuda.synchronize()
    ref = oracle.forward_planes(p, alpha, z, x, group)[0]
    assert rel_err(yh.numpy(), ref) <= TOL
    # pageable host buffers take the staged path
    yp = torch.zeros(N, dtype=torch.float16)
    ys.zero_()
    bq.gemv_host(L.d, L.packed, L.alpha, L.z, torch.from_numpy(x.reshape(-1).copy()), yp, xs, ys, ws)
    torch.cuda.synchronize()
    assert np.array_equal(yp.numpy().view(np.uint16), yh.numpy().view(np.uint16))
    assert np.array_equal(ys.cpu().numpy().view(np.uint16), yh.numpy().view(np.uint16))   # staged through y_stage


def test_device_errors_are_reported_not_raised_as_faults():
    """Bad arguments come back as status codes through the binding, with the GPU untouched."""
    d = bq.desc(64, 1000, 3, 128)
    t = torch.zeros(64, dtype=torch.float16, device=DEV)
    with pytest.raises(bq.BcqError) as e:
        bq.gemv(d, t, t, t, t, t)
    assert e.value.status == bq.ERR_UNSUPPORTED_SHAPE
    bq.poll_status()        # no bounded wait ran out in any kernel launched so far


def test_random_shapes_batches_and_plans():
    """Seeded random cases over every kernel of the tiled layout: shapes (1..260 row units, 1..11 windows),
    q, scale granularity, batch, and decompositions (given and default), each against the oracle."""
    rng = np.random.default_rng(240702891)
    for case in range(48):
        q = int(rng.integers(1, 5))
        group = int(rng.choice([0, 128]))
        U, W = int(rng.integers(1, 260)), int(rng.integers(1, 12))
        N, K = 8 * U, 512 * W
        B = int(rng.choice([1, 1, 2, 3, 4, 5, 8, 9, 16]))
        kernel = int(rng.choice([1, 2])) if B >= 2 else 1
        ks = int(rng.integers(1, W + 1))
        rb_min = -(-U // (lut_max_units(q, group, B) if kernel == 1 else 176))
        rb = int(rng.integers(rb_min, min(U, rb_min + 6) + 1))
        p, codes, alpha, z, X = make_layer(f"random/{case}", N, K, q, group, B)
        ref = oracle.forward_planes(p, alpha, z, X, group)
        L = gpu_layer(N, K, q, group, bq.LAYOUT_TILED, codes, alpha, z)
        Y = torch.empty((B, N), dtype=torch.float16, device=DEV)
        for plan in (bq.Plan(kernel, rb, ks, 0), bq.plan_default(L.d, B)):
            ws = bq.new_workspace(L.d, B, plan)
            Y.fill_(float("nan"))
            for _ in range(2):
                bq.gemm_smallbatch_plan(L.d, plan, L.packed, L.alpha, L.z, dev(X), Y, B, ws)
            torch.cuda.synchronize()
            bq.poll_status()
            assert rel_err(Y.cpu().numpy(), ref) <= TOL, (case, N, K, q, group, B, plan.kernel, plan.row_blocks, plan.k_splits)


def _heavy_tailed(kind, K, name):
    """Activations with the outliers LLM hidden states have: fp16, the bulk N(0,1)."""
    x = synth.normal(name + "/x", 0, K)
    u = synth.uniform(name + "/pick", 0, K)
    if kind == "outliers_x50":               # one value in a hundred is fifty times larger
        x = np.where(u < 0.01, 50.0 * x, x)
    elif kind == "spikes_1e2_1e4":           # a few spikes of 1e2 .. 1e4 in every window of 512
        for w in range(K // 512):
            for j, mag in enumerate((1e2, -1e3, 1e4)):
                x[512 * w + int(u[512 * w + j] * 512)] = mag
    elif kind == "near_table_limit":         # one chunk of eight same-sign values whose sum is just below the
        x[8 * 37:8 * 37 + 8] = 8000.0        # largest finite fp16 (64000 < 65504), another with the opposite sign
        x[8 * 101:8 * 101 + 8] = -8000.0
    elif kind == "cancelling":               # large values that cancel inside a chunk: the table entry is small,
        x[8 * 5:8 * 5 + 8] = [3000.0, -3000.0, 2000.0, -2000.0, 1000.0, -1000.0, 0.5, -0.25]   # its terms are not
    return x.astype(np.float16).reshape(1, K)


@pytest.mark.parametrize("group", [128, 0])
@pytest.mark.parametrize("kind", ["outliers_x50", "spikes_1e2_1e4", "near_table_limit", "cancelling"])
def test_gemv_heavy_tailed_activations(kind, group):
    """The lookup tables hold fp16 sums of 8 activations (one rounding each, relative 2^-11): the product
    must stay inside the stated tolerance when the activations have outliers, up to the documented limit
    (every 8-activation sum finite in fp16)."""
    N, K, q = 1024, 4096, 3
    p, codes, alpha, z, _ = make_layer(f"tails/{group}", N, K, q, group)
    x = _heavy_tailed(kind, K, f"tails/{kind}")
    ref = oracle.forward_planes(p, alpha, z, x, group)[0]
    L = gpu_layer(N, K, q, group, bq.LAYOUT_TILED, codes, alpha, z)
    assert bq.plan_default(L.d).kernel == 1
    y = run_gemv(L, x)
    assert np.isfinite(y).all()
    assert rel_err(y, ref) <= TOL
    # two columns per launch build their tables the same way
    if group:
        X = np.concatenate([x, synth.activations("tails/col1", 1, K)])
        Y = torch.zeros((2, N), dtype=torch.float16, device=DEV)
        bq.gemm_smallbatch(L.d, L.packed, L.alpha, L.z, dev(X), Y, 2, bq.new_workspace(L.d, 2))
        torch.cuda.synchronize()
        assert rel_err(Y.cpu().numpy(), oracle.forward_planes(p, alpha, z, X, group)) <= TOL


def test_operands_rewritten_in_place_between_two_products():
    """The products fetch packed operands before they wait for the kernel in front of them; operands
    written by the library's own calls must still be complete.  Pack layer A, multiply, pack layer B into
    the SAME buffers, multiply again at once: the second result is B's, for each way of writing operands."""
    N, K, q, group = 2048, 4096, 3, 128
    pa, ca, aa, za, x = make_layer("inplace/A", N, K, q, group)
    pb, cb, ab, zb, _ = make_layer("inplace/B", N, K, q, group)
    ref_b = oracle.forward_planes(pb, ab, zb, x, group)[0]
    d = bq.desc(N, K, q, group, bq.LAYOUT_TILED)
    dc = d.with_layout(bq.LAYOUT_CANONICAL)
    packed, _, _ = bq.empty_operands(d, DEV)
    xd = dev(x.reshape(-1))
    ws = bq.new_workspace(d, 1)
    ya = torch.zeros(N, dtype=torch.float16, device=DEV)
    yb = torch.zeros(N, dtype=torch.float16, device=DEV)
    codes_a, codes_b = dev(ca), dev(cb)
    canon_b = dev(pb.reshape(-1))
    for how in ("pack", "repack"):
        for _ in range(3):
            bq.pack(d, codes_a, dev(aa), dev(za), packed, None, None)
            bq.gemv(d, packed, None, None, xd, ya, ws)
            if how == "pack":
                bq.pack(d, codes_b, dev(ab), dev(zb), packed, None, None)
            else:
                bq.repack(dc, canon_b, dev(ab), dev(zb), d, packed, None, None)
            bq.gemv(d, packed, None, None, xd, yb, ws)          # no synchronisation in between
        torch.cuda.synchronize()
        bq.poll_status()
        assert rel_err(yb.cpu().numpy(), ref_b) <= TOL, how
