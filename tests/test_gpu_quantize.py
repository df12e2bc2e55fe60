"""bcq_quantize_rtn against the oracle: step-1 integers, S, qbias, packed planes and fused scales,
all bit for bit (the integer is decided in fp64 on both sides, from the stored fp16 S)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import TOL, rel_err, tiled_operands
from paper_2407_02891_b200 import binding as bq
from paper_2407_02891_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def weights(name, N, K, scale=0.05):
    return (scale * synth.normal(name + "/W", 0, N * K)).reshape(N, K).astype(np.float16)


def run(W, q, group, layout, n_bits, b2p, s_factor=1.0, want_int=True):
    N, K = W.shape
    d = bq.desc(N, K, q, group, layout)
    G = 1 if group == 0 else K // group
    Wd = torch.from_numpy(W).to(DEV)
    S = torch.zeros(N * G, dtype=torch.float16, device=DEV)
    qb = torch.zeros(N * G, dtype=torch.float16, device=DEV)
    wi = torch.full((N * K,), 255, dtype=torch.uint8, device=DEV) if want_int else None
    packed, a, z = bq.empty_operands(d, DEV)
    packed.fill_(0xA5)
    bq.quantize_rtn(d, Wd, n_bits, b2p, S, qb, wi, packed, a, z, s_factor)
    torch.cuda.synchronize()
    cpu = lambda t: None if t is None else t.cpu().numpy()
    return cpu(S), cpu(qb), cpu(wi), cpu(packed), cpu(a), cpu(z)


def expected(W, q, group, layout, n_bits, b2p, s_factor=1.0):
    w_int, S, qb = oracle.quantize_rtn(W, group, n_bits, s_factor)
    codes, alpha, z = oracle.merge_linear(w_int, S, qb, group, n_bits, b2p)
    planes = oracle.pack_canonical(codes, q)
    if layout == bq.LAYOUT_TILED:
        packed, a, zz = tiled_operands(planes, alpha, z, group)
    else:
        packed, a, zz = planes.reshape(-1), alpha.reshape(-1), z.reshape(-1)
    return w_int, S, qb, packed, a, zz, (codes, alpha, z)


def same(a, b):
    return np.array_equal(np.asarray(a).reshape(-1).view(np.uint8), np.asarray(b).reshape(-1).view(np.uint8))


@pytest.mark.parametrize("N,K,q,group,layout,n_bits,b2p,s_factor", [
    (16, 32, 3, 32, bq.LAYOUT_CANONICAL, 4, [0, 1, 2, 2], 1.0),          # the tiny 4-bit -> 3-plane case
    (16, 32, 3, 0, bq.LAYOUT_CANONICAL, 4, [0, 1, 1, 2], 1.0),
    (50, 256, 3, 64, bq.LAYOUT_CANONICAL, 4, [0, 1, 2, 2], 1.0),
    (40, 1024, 3, 128, bq.LAYOUT_TILED, 4, [0, 1, 2, 2], 1.0),
    (264, 1536, 3, 128, bq.LAYOUT_TILED, 5, [0, 0, 1, 1, 2], 0.8),       # a re-explored scale: the top clamps
    (264, 1536, 2, 128, bq.LAYOUT_TILED, 5, [0, 0, 1, 1, 1], 1.3),
    (72, 512, 2, 0, bq.LAYOUT_TILED, 3, [0, 1, 1], 1.0),                 # one scale per row
    (24, 4096, 4, 128, bq.LAYOUT_TILED, 4, [0, 1, 2, 3], 1.0),           # q = n: plain linear quantisation
    (13, 96, 1, 32, bq.LAYOUT_CANONICAL, 2, [0, 0], 0.55),
    (8, 36864, 3, 0, bq.LAYOUT_CANONICAL, 8, [0, 0, 0, 1, 1, 1, 2, 2], 1.0),   # long rows, 8-bit step 1
])
def test_quantize_rtn_bit_exact(N, K, q, group, layout, n_bits, b2p, s_factor):
    W = weights(f"q/{N}x{K}/{group}", N, K)
    S, qb, wi, packed, a, z = run(W, q, group, layout, n_bits, b2p, s_factor)
    e_wi, e_S, e_qb, e_packed, e_a, e_z, _ = expected(W, q, group, layout, n_bits, b2p, s_factor)
    assert same(S, e_S) and same(qb, e_qb)
    assert same(wi, e_wi)
    assert same(packed, e_packed)
    if a is not None:
        assert same(a, e_a) and same(z, e_z)


def test_quantize_rtn_structured_weights():
    """Constant groups (S = 0), exact half-way points (ties to even), zeros of both signs."""
    N, K, q, group = 8, 512, 3, 128
    W = weights("q/struct", N, K)
    W[0, :128] = np.float16(0.375)                       # constant group
    W[1, :] = 0.0
    W[1, 5] = np.float16(-0.0)                           # a zero row with a negative zero
    W[2, :8] = [0.0, 7.0, 0.5, 1.5, 2.5, 3.5, 4.5, 6.5]  # with n = 3, S = 1: ties
    W[2, 8:128] = 3.0
    for layout in (bq.LAYOUT_CANONICAL, bq.LAYOUT_TILED):
        S, qb, wi, packed, a, z = run(W, q, group, layout, 3, [0, 1, 2])
        e_wi, e_S, e_qb, e_packed, e_a, e_z, _ = expected(W, q, group, layout, 3, [0, 1, 2])
        assert same(S, e_S) and same(qb, e_qb) and same(wi, e_wi) and same(packed, e_packed)
        if a is not None:
            assert same(a, e_a) and same(z, e_z)
        assert wi.reshape(N, K)[2, :8].tolist() == [0, 7, 0, 2, 2, 4, 4, 6]
        assert np.all(wi.reshape(N, K)[0, :128] == 0) and np.all(wi.reshape(N, K)[1] == 0)


def test_quantize_rtn_without_integer_output_and_product():
    """w_int is optional; the operand that comes out multiplies like the oracle's dequantised matrix."""
    N, K, q, group, n_bits, b2p = 520, 2048, 3, 128, 4, [0, 0, 1, 2]
    W = weights("q/prod", N, K)
    d = bq.desc(N, K, q, group, bq.LAYOUT_TILED)
    S, qb, wi, packed, a, z = run(W, q, group, bq.LAYOUT_TILED, n_bits, b2p, want_int=False)
    assert wi is None
    _, _, _, e_packed, _, _, (codes, alpha, zz) = expected(W, q, group, bq.LAYOUT_TILED, n_bits, b2p)
    assert same(packed, e_packed)
    x = synth.activations("q/prod", 1, K)
    y = torch.zeros(N, dtype=torch.float16, device=DEV)
    bq.gemv(d, torch.from_numpy(packed).to(DEV), None, None, torch.from_numpy(x.reshape(-1)).to(DEV), y,
            bq.new_workspace(d, 1))
    torch.cuda.synchronize()
    ref = oracle.forward_dequant(codes, alpha, zz, x, group)[0]
    assert rel_err(y.cpu().numpy(), ref) <= TOL
    # and stays within the method's own error of the unquantised product.  Per weight: half a step of
    # step 1 (S/2: the range scale reaches both ends of the group exactly), half the largest gap between
    # reachable integers in the rounding of Eq. round (S * gap / 2), and the fp16 rounding of the fused
    # scales (2^-11 of sum_j alpha_j + |z|).  Per row that sums, at worst, against |x|.
    _, reach = oracle.bcchoice(n_bits, b2p)
    gap = float(np.diff(np.sort(reach)).max())
    _, e_S, _ = oracle.quantize_rtn(W, group, n_bits)
    Sd = e_S.astype(np.float64)                                          # [N][G]
    per_weight = 0.5 * Sd * (1.0 + gap) + 2.0 ** -11 * (np.abs(alpha.astype(np.float64)).sum(0) + np.abs(zz.astype(np.float64)))
    ax = np.abs(x[0].astype(np.float64)).reshape(-1, group).sum(1)        # sum |x| per group
    bound = per_weight @ ax
    exact = W.astype(np.float64) @ x[0].astype(np.float64)
    assert (np.abs(ref - exact) <= bound).all()


def test_quantize_rtn_full_size_sampled_rows():
    """OPT-30B projection size: S, qbias of all rows, integers and planes of sampled rows."""
    N, K, q, group, n_bits, b2p = 7168, 7168, 3, 128, 4, [0, 1, 2, 2]
    W = weights("q/full", N, K)
    d = bq.desc(N, K, q, group, bq.LAYOUT_CANONICAL)
    S, qb, wi, packed, a, z = run(W, q, group, bq.LAYOUT_CANONICAL, n_bits, b2p)
    rows = np.array([0, 1, 7, 3583, 3584, 7160, 7167])
    e_wi, e_S, e_qb = oracle.quantize_rtn(W[rows], group, n_bits)
    G = K // group
    assert same(S.reshape(N, G)[rows], e_S) and same(qb.reshape(N, G)[rows], e_qb)
    assert same(wi.reshape(N, K)[rows], e_wi)
    codes, alpha, zz = oracle.merge_linear(e_wi, e_S, e_qb, group, n_bits, b2p)
    planes = oracle.pack_canonical(codes, q)
    assert same(packed.reshape(q, N, K // 8)[:, rows], planes)
    assert same(a.reshape(q, N, G)[:, rows], alpha) and same(z.reshape(N, G)[rows], zz)
    # every row: S is one fp16 rounding away from the range formula, qbias is the minimum
    Wd = W.astype(np.float64).reshape(N, G, group)
    assert np.array_equal(qb.reshape(N, G).astype(np.float64), Wd.min(axis=2))
    exact_S = (Wd.max(axis=2) - Wd.min(axis=2)) / 15
    assert np.all(np.abs(S.reshape(N, G).astype(np.float64) - exact_S) <= exact_S * 2.0 ** -11)


def test_quantize_rtn_rejects_bad_arguments():
    d = bq.desc(16, 64, 3, 32, bq.LAYOUT_CANONICAL)
    t16 = torch.zeros(16 * 64, dtype=torch.float16, device=DEV)
    t8 = torch.zeros(3 * 16 * 8, dtype=torch.uint8, device=DEV)
    sc = torch.zeros(3 * 16 * 2, dtype=torch.float16, device=DEV)
    for kwargs in (dict(n_bits=2, b2p=[0, 1]),            # fewer bits than planes
                   dict(n_bits=4, b2p=[0, 1, 1, 1]),      # plane 2 empty
                   dict(n_bits=4, b2p=[0, 1, 2, 3])):     # plane index out of range
        with pytest.raises(bq.BcqError):
            bq.quantize_rtn(d, t16, kwargs["n_bits"], kwargs["b2p"], sc, sc, None, t8, sc, sc)
    with pytest.raises(bq.BcqError):
        bq.quantize_rtn(d, t16, 4, [0, 1, 2, 2], sc, sc, None, t8, sc, sc, s_factor=0.0)
    with pytest.raises(bq.BcqError):
        bq.quantize_rtn(d, t16, 4, [0, 1, 2, 2], sc, sc, None, t8, None, None)   # canonical needs alpha and z


@pytest.mark.parametrize("N,K,q,group,layout,n_bits,b2p,s_factor", [
    (17, 160, 2, 32, bq.LAYOUT_CANONICAL, 3, [0, 1, 1], 1.0),             # ragged rows and a short last segment
    (9, 384, 3, 96, bq.LAYOUT_CANONICAL, 5, [0, 1, 1, 2, 2], 0.52),       # groups that straddle segments; many clamped
    (8, 4128, 1, 0, bq.LAYOUT_CANONICAL, 7, [0] * 7, 1.0),
    (5, 256, 4, 256, bq.LAYOUT_CANONICAL, 8, [0, 0, 1, 1, 2, 2, 3, 3], 0.7),   # 15 fraction bits
    (16, 512, 3, 64, bq.LAYOUT_TILED, 8, [0, 0, 0, 1, 1, 1, 2, 2], 1.0),
    (24, 1024, 4, 32, bq.LAYOUT_TILED, 6, [0, 1, 1, 2, 2, 3], 0.6),
    (16, 512, 2, 0, bq.LAYOUT_TILED, 4, [0, 0, 1, 1], 1.0),
    (8, 512, 3, 128, bq.LAYOUT_TILED, 7, [0, 0, 1, 1, 1, 2, 2], 1.0),
])
@pytest.mark.parametrize("kind", ["normal", "grid", "offset", "tiny"])
def test_quantize_rtn_where_the_estimate_does_not_decide(N, K, q, group, layout, n_bits, b2p, s_factor, kind):
    """Weights on and next to rounding boundaries (a grid of half steps), ranges far away from zero (the offset is
    thousands of steps), subnormal scales: the integers stay those of the fp64 definition."""
    rng = np.random.default_rng(N * K + n_bits)
    if kind == "normal":
        W = weights(f"q2/{N}x{K}", N, K)
    elif kind == "grid":
        W = (rng.integers(0, 2 ** (n_bits + 1) - 1, (N, K)) * 0.5 - 3).astype(np.float16)
    elif kind == "offset":
        W = (100.0 + rng.integers(0, 5, (N, K)) * 0.0625).astype(np.float16)
    else:
        W = (rng.integers(0, 300, (N, K)) * 2.0 ** -24 + rng.integers(0, 2, (N, 1))).astype(np.float16)
    S, qb, wi, packed, a, z = run(W, q, group, layout, n_bits, b2p, s_factor)
    e_wi, e_S, e_qb, e_packed, e_a, e_z, _ = expected(W, q, group, layout, n_bits, b2p, s_factor)
    assert same(S, e_S) and same(qb, e_qb) and same(wi, e_wi) and same(packed, e_packed)
    if a is not None:
        assert same(a, e_a) and same(z, e_z)


@pytest.mark.parametrize("group", [32, 128, 0])
def test_quantize_rtn_weights_that_are_not_numbers(group):
    """A NaN among finite weights is ignored by the range and becomes integer 0; the others are not disturbed."""
    N, K = 8, 512
    W = weights("q/nan", N, K)
    clean = W.copy()
    W[3, 77] = np.float16(np.nan)
    lo = np.nanargmin(W[3, 64:96])
    clean[3, 77] = W[3, 64 + lo]                      # a value that changes no minimum or maximum
    S, qb, wi, packed, a, z = run(W, 3, group, bq.LAYOUT_TILED, 4, [0, 1, 2, 2])
    e_wi, e_S, e_qb, *_ = expected(clean, 3, group, bq.LAYOUT_TILED, 4, [0, 1, 2, 2])
    assert same(S, e_S) and same(qb, e_qb)
    wi, e_wi = wi.reshape(N, K), e_wi.reshape(N, K).copy()
    assert wi[3, 77] == 0
    e_wi[3, 77] = 0
    assert np.array_equal(wi, e_wi)


@pytest.mark.parametrize("N,K,q,group", [
    (5, 12288, 3, 0),        # a few long rows: a row unit's segments in twelve parts
    (1, 131072, 2, 0),       # the most parts
    (17, 4128, 3, 96),       # short groups, four at a time; parts that share groups, a last segment of 32 weights
    (9, 4608, 2, 1536),      # long groups that parts share
    (8, 2048, 4, 512),       # the longest group that goes four at a time; two parts
    (3, 1056, 1, 352),       # one part, fewer groups than warps
])
def test_quantize_rtn_in_parts(N, K, q, group):
    W = weights(f"q/parts/{N}x{K}", N, K)
    W[N // 2, K // 2] = np.float16(6.0)                # a maximum that one part alone holds
    b2p = [min(i, q - 1) for i in range(5)]
    S, qb, wi, packed, a, z = run(W, q, group, bq.LAYOUT_CANONICAL, 5, b2p)
    e_wi, e_S, e_qb, e_packed, e_a, e_z, _ = expected(W, q, group, bq.LAYOUT_CANONICAL, 5, b2p, 1.0)
    assert same(S, e_S) and same(qb, e_qb) and same(wi, e_wi) and same(packed, e_packed)
    assert same(a, e_a) and same(z, e_z)


@pytest.mark.parametrize("n_bits", [1, 3, 4, 5])
@pytest.mark.parametrize("N,K,group,layout,s_factor", [
    (24, 1024, 128, bq.LAYOUT_TILED, 1.0), (24, 1024, 64, bq.LAYOUT_TILED, 0.6), (17, 1184, 32, bq.LAYOUT_CANONICAL, 1.0), (9, 1152, 0, bq.LAYOUT_CANONICAL, 0.9)])
def test_quantize_rtn_clamps_where_a_weight_lies_beyond_the_top(N, K, group, layout, s_factor, n_bits):
    """Blocks of 32 subnormal weights strewn among ordinary ones, factors of one and below: a quotient beyond the top integer in some
    groups of 32 at 3 and 4 bits and, with the factors below one, in every group.  Integers of up to four bits are looked up in pairs."""
    rng = np.random.default_rng(N + K + n_bits)
    W = weights(f"top/{N}x{K}", N, K)
    small = rng.random((N, K // 32)) < 0.3
    W = np.where(np.repeat(small, 32, axis=1), (rng.integers(0, 24, (N, K)) * 2.0 ** -24).astype(np.float16), W).astype(np.float16)
    q = min(n_bits, 2)
    b2p = [i % q for i in range(n_bits)]
    S, qb, wi, packed, a, z = run(W, q, group, layout, n_bits, b2p, s_factor)
    e_wi, e_S, e_qb, e_packed, e_a, e_z, _ = expected(W, q, group, layout, n_bits, b2p, s_factor)
    assert same(S, e_S) and same(qb, e_qb) and same(wi, e_wi) and same(packed, e_packed)
    if a is not None:
        assert same(a, e_a) and same(z, e_z)


def top_sides(W, S, qb, L, n_bits, lane_wise):
    """(segments of eight rows that hold an integer beyond the top, segments whose largest quotients are below top + 0.4), by the
    definition; the largest of 32 neighbouring weights where lane_wise, of a group otherwise."""
    N, K = W.shape
    G, top = K // L, 2 ** n_bits - 1
    s = np.repeat(S.astype(np.float64).reshape(N, G), L, axis=1)
    t = (W.astype(np.float64) - np.repeat(qb.astype(np.float64).reshape(N, G), L, axis=1)) / np.where(s > 0, s, np.inf)
    run_len = 32 if lane_wise else L
    largest = np.repeat(t.reshape(N, K // run_len, run_len).max(axis=2), run_len, axis=1)
    beyond = within = 0
    for n in range(0, N, 8):
        for k in range(0, K, 128):
            beyond += bool((np.rint(t[n:n + 8, k:k + 128]) > top).any())
            within += bool((largest[n:n + 8, k:k + 128] < top + 0.4).all())
    return beyond, within


@pytest.mark.parametrize("n_bits", [2, 4, 5, 7, 8])
@pytest.mark.parametrize("N,K,group,layout", [
    (24, 1024, 128, bq.LAYOUT_TILED), (24, 1024, 64, bq.LAYOUT_TILED), (17, 1184, 32, bq.LAYOUT_CANONICAL), (12, 1152, 0, bq.LAYOUT_CANONICAL),
    (24, 1536, 192, bq.LAYOUT_CANONICAL)])
@pytest.mark.parametrize("factor", ["one", "line", "low"])
def test_quantize_rtn_segments_with_and_without_integers_beyond_the_top(N, K, group, layout, n_bits, factor):
    """A segment in which no quotient rounds to more than the top integer goes without the comparison with it.  Every second row
    unit holds groups whose range is about 1.45 top of the smallest subnormal number, which is their scale: with a factor of one
    their largest quotients, and no other group's, lie beyond the top.  With a factor just above top / (top + 1/2) the largest quotients
    of ordinary groups lie about where the top integer's cell ends, well below it far beyond."""
    rng = np.random.default_rng(1000 * n_bits + K + group)
    L, top = group or K, 2 ** n_bits - 1
    W = weights(f"sides/{N}x{K}/{n_bits}", N, K)
    reach = top + max(1, 4 * top // 9)        # less than 1.5 top: the scale is rounded down to 2^-24
    for n in range(8, N, 16):
        for r in range(n, min(n + 8, N)):
            for g in range(K // L):
                if rng.random() < 0.3 or (r == n and g % 2 == 0):
                    steps = rng.integers(0, reach + 1, L)
                    steps[rng.permutation(L)[:2]] = 0, reach
                    W[r, g * L:(g + 1) * L] = ((steps - 3) * 2.0 ** -24).astype(np.float16)
    s_factor = {"one": 1.0, "line": 1.0005 * top / (top + 0.5), "low": 0.6}[factor]
    q = min(n_bits, 3)
    b2p = [i % q for i in range(n_bits)]
    e_wi, e_S, e_qb, e_packed, e_a, e_z, _ = expected(W, q, group, layout, n_bits, b2p, s_factor)
    beyond, within = top_sides(W, e_S, e_qb, L, n_bits, L not in (128, 64, 32))
    assert beyond > 0 and (factor != "one" or within > 0)
    for want_int in (True, False):
        S, qb, wi, packed, a, z = run(W, q, group, layout, n_bits, b2p, s_factor, want_int)
        assert same(S, e_S) and same(qb, e_qb) and same(packed, e_packed) and (wi is None or same(wi, e_wi))
        if a is not None:
            assert same(a, e_a) and same(z, e_z)
