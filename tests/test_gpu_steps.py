"""GPU parity of each step of the path against the oracle's restatement of
the same step (oracle.method), through the C ABI.

Tolerances: integer/mask work is bit-exact.  Floating-point steps compute in
FP32 against an FP64 oracle on values of at most 255 gray; a single FP32
operation on such values carries an error of about 255 * 2^-24 = 1.5e-5, so
stencil-sized expressions are compared at 2e-4 (absolute) and the ORAS
iteration, whose local PCG amplifies rounding over its steps, at 1e-3 of the
largest correction plus 2e-4."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import method as M

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module")
def di():
    from paper_2401_06744_gb300 import build as b

    b.build()
    import paper_2401_06744_gb300 as di

    di.load()
    return di


def T(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    if dtype is not None:
        t = t.to(dtype)
    return t.to(DEV)


def N(t):
    torch.cuda.synchronize()
    return t.detach().cpu().numpy()


def _case(h, w, C, d, seed, nan=True):
    g = np.random.default_rng(seed)
    f = g.uniform(0, 255, size=(C, h, w)).astype(np.float32)
    c = (g.random((h, w)) < d).astype(np.uint8)
    if not c.any():
        c[g.integers(h), g.integers(w)] = 1
    fn = f.copy()
    if nan:
        fn[:, c == 0] = np.nan  # never read at unknown pixels
    return f, fn, c


SIZES = [(1, 1), (1, 9), (7, 1), (3, 5), (17, 33), (64, 64), (101, 67), (130, 257), (66, 128), (2, 2)]


@pytest.mark.parametrize("h,w", SIZES)
def test_mask_downsample_bit_exact(di, h, w):
    _, _, c = _case(h, w, 1, 0.15, h * 7 + w)
    cH = di.mask_downsample(T(c))
    assert np.array_equal(N(cH), M.mask_downsample(c))


@pytest.mark.parametrize("h,w", SIZES)
@pytest.mark.parametrize("modified", [True, False])
def test_values_downsample(di, h, w, modified):
    f, fn, c = _case(h, w, 3, 0.3, h * 11 + w)
    cH = M.mask_downsample(c)
    out = N(di.values_downsample(T(c), T(fn), T(cH), modified=modified))
    ref = (M.values_downsample_modified(c, f, cH) if modified
           else M.values_downsample_naive(c, f))
    assert np.isfinite(out).all()
    assert np.abs(out - ref).max() < 2e-4


@pytest.mark.parametrize("h,w", SIZES + [(1080, 1920), (33, 2000)])
@pytest.mark.parametrize("modified", [True, False])
def test_pyramid_level_one_pass_bit_exact(di, h, w, modified):
    # the decoder's one-pass pyramid level: the coarse mask bit-exact with the
    # oracle's 2x2 max pooling, the mask values bit-identical to the separate
    # downsampling step and within rounding of the oracle, the packed words
    # and the unknown count exactly those of the coarse mask
    f, fn, c = _case(h, w, 2, 0.2, h * 5 + w)
    cH, bH, bits, unk = di.pyramid_level(T(c), T(fn), modified=modified)
    cH_ref = M.mask_downsample(c)
    assert np.array_equal(N(cH), cH_ref)
    sep = N(di.values_downsample(T(c), T(fn), T(cH_ref), modified=modified))
    assert np.array_equal(N(bH), sep)
    ref = (M.values_downsample_modified(c, f, cH_ref) if modified
           else M.values_downsample_naive(c, f))
    assert np.abs(N(bH) - ref).max() < 2e-4
    hH, wH = cH_ref.shape
    wpr = (wH + 31) // 32 + 1
    words = N(bits).astype(np.int64) & 0xFFFFFFFF
    known = np.ones((hH, 32 * wpr), dtype=bool)
    known[:, :wH] = cH_ref.astype(bool)
    ref_words = (known.reshape(hH, wpr, 32) * (1 << np.arange(32, dtype=np.int64))).sum(axis=2)
    assert np.array_equal(words, ref_words)
    assert int(N(unk)[0]) == int((cH_ref == 0).sum())
    # masks only
    cH2, bH2, bits2, unk2 = di.pyramid_level(T(c))
    assert bH2 is None and np.array_equal(N(cH2), cH_ref) and np.array_equal(N(bits2), N(bits))


@pytest.mark.parametrize("h,w", SIZES)
def test_residual_and_norm(di, h, w):
    f, fn, c = _case(h, w, 2, 0.1, h * 13 + w)
    g = np.random.default_rng(5)
    u = np.where(c.astype(bool), f, g.uniform(0, 255, f.shape)).astype(np.float32)
    with di.Context() as ctx:
        # b = C f (values off the mask never read) ...
        r, n2 = ctx.residual_norm(T(u), T(fn), T(c), rhs_zero=True)
        ref = M.residual(u, M.rhs(f, c), c)
        assert np.abs(N(r) - ref).max() < 2e-4
        assert np.allclose(N(n2), (ref ** 2).sum(axis=(1, 2)), rtol=1e-5, atol=1e-6)
        # ... and a general right-hand side at unknown pixels
        b = np.where(c.astype(bool), f, g.normal(size=f.shape)).astype(np.float32)
        r, n2 = ctx.residual_norm(T(u), T(b), T(c), rhs_zero=False)
        ref = M.residual(u, b, c)
        assert np.abs(N(r) - ref).max() < 2e-4


@pytest.mark.parametrize("h,w", SIZES)
def test_restrict_residual(di, h, w):
    f, fn, c = _case(h, w, 2, 0.05, h * 17 + w)
    g = np.random.default_rng(6)
    u = np.where(c.astype(bool), f, g.uniform(0, 255, f.shape)).astype(np.float32)
    cH = M.mask_downsample(c)
    rH = N(di.restrict_residual(T(u), T(fn), T(c), T(cH), rhs_zero=True))
    ref = M.restrict_residual(M.residual(u, M.rhs(f, c), c), cH)
    assert np.abs(rH - ref).max() < 1e-3
    b = np.where(c.astype(bool), 0.0, g.normal(size=f.shape)).astype(np.float32)
    u2 = np.where(c.astype(bool), 0.0, g.normal(size=f.shape)).astype(np.float32)
    rH = N(di.restrict_residual(T(u2), T(b), T(c), T(cH), rhs_zero=False))
    ref = M.restrict_residual(M.residual(u2, b, c), cH)
    assert np.abs(rH - ref).max() < 1e-4


@pytest.mark.parametrize("h,w", SIZES)
def test_prolong_both_modes(di, h, w):
    f, fn, c = _case(h, w, 2, 0.2, h * 19 + w)
    H, W = M.coarse_shape(h, w)
    g = np.random.default_rng(7)
    uH = g.uniform(0, 255, (2, H, W)).astype(np.float32)
    out = N(di.prolong(T(uH), T(c), 0, b=T(fn)))
    ref = M.prolong_solution(uH, f, c)
    assert np.abs(out - ref).max() < 1e-4
    assert np.array_equal(out[:, c == 1], f[:, c == 1])  # mask values exact
    u = g.uniform(0, 255, (2, h, w)).astype(np.float32)
    ut = T(u)
    di.prolong(T(uH), T(c), 1, u=ut)
    ref = M.prolong_correct(u, uH, c)
    out = N(ut)
    assert np.abs(out - ref).max() < 1e-4
    assert np.array_equal(out[:, c == 1], u[:, c == 1])


ORAS_CASES = [  # (h, w, block, overlap, iters)
    (32, 32, 32, 6, 8), (70, 95, 32, 6, 8), (77, 61, 16, 4, 6), (61, 77, 16, 2, 5),
    (45, 38, 8, 2, 4), (45, 38, 8, 4, 3), (40, 41, 8, 1, 4), (50, 33, 16, 1, 2),
    (130, 100, 32, 6, 0), (130, 100, 32, 6, 1), (9, 120, 32, 6, 8), (120, 9, 16, 4, 8),
    (70, 96, 32, 2, 8), (130, 100, 32, 2, 10), (33, 35, 32, 2, 4), (70, 95, 32, 3, 8),
]


@pytest.mark.parametrize("h,w,B,o,K", ORAS_CASES)
def test_oras_iteration_matches_oracle_cg(di, h, w, B, o, K):
    f, fn, c = _case(h, w, 2, 0.06, h * 23 + w + B)
    g = np.random.default_rng(8)
    # an iterate that equals b on the mask (cascadic form, b = C f) ...
    u = np.where(c.astype(bool), f, g.uniform(0, 255, f.shape)).astype(np.float32)
    with di.Context(block=B, overlap=o, alpha=0.5) as ctx:
        out = N(ctx.oras_iteration(T(u), T(fn), T(c), K, rhs_zero=True))
        ref = M.oras_iteration(u, M.rhs(f, c), c, B, o, 0.5, ("cg", K))
        scale = np.abs(ref - u).max()
        assert np.abs(out - ref).max() < 1e-3 * scale + 2e-4
        assert np.array_equal(out[:, c == 1], u[:, c == 1])
        # ... and the correction form (zero on the mask, general right-hand side)
        b = np.where(c.astype(bool), 0.0, g.normal(size=f.shape)).astype(np.float32)
        e = np.where(c.astype(bool), 0.0, g.normal(size=f.shape)).astype(np.float32)
        out = N(ctx.oras_iteration(T(e), T(b), T(c), K, rhs_zero=False))
        ref = M.oras_iteration(e, b, c, B, o, 0.5, ("cg", K))
        scale = np.abs(ref - e).max()
        assert np.abs(out - ref).max() < 1e-3 * scale + 1e-5


@pytest.mark.parametrize("B,o", [(32, 6), (16, 4), (8, 2)])
def test_oras_converged_local_solves_match_exact(di, B, o):
    # with enough local PCG steps each block solve is exact: compare with the
    # oracle's direct local solves (Algorithm 2 as printed)
    f, fn, c = _case(48, 53, 1, 0.08, 99 + B)
    g = np.random.default_rng(9)
    u = np.where(c.astype(bool), f, g.uniform(0, 255, f.shape)).astype(np.float32)
    with di.Context(block=B, overlap=o) as ctx:
        out = N(ctx.oras_iteration(T(u), T(fn), T(c), 3 * B * B, rhs_zero=True))
    ref = M.oras_iteration(u, M.rhs(f, c), c, B, o, 0.5, "exact")
    assert np.abs(out - ref).max() < 2e-3


def test_oras_is_deterministic(di):
    f, fn, c = _case(300, 257, 3, 0.05, 5)
    u = np.where(c.astype(bool), f, 100.0).astype(np.float32)
    with di.Context() as ctx:
        a = N(ctx.oras_iteration(T(u), T(fn), T(c), 8, rhs_zero=True))
        b = N(ctx.oras_iteration(T(u), T(fn), T(c), 8, rhs_zero=True))
    assert np.array_equal(a, b)


def test_oras_rejects_aliasing(di):
    f, fn, c = _case(40, 40, 1, 0.1, 1)
    with di.Context() as ctx:
        ut = T(f)
        with pytest.raises(di.DiError):
            ctx.oras_iteration(ut, T(fn), T(c), 4, rhs_zero=True, out=ut)


def _unaligned(a):
    # the same values in a tensor whose data starts 4 bytes past a 16-byte
    # boundary: the block kernel then copies its tiles with cp.async, not TMA
    flat = torch.empty(a.size + 1, dtype=torch.float32, device=DEV)
    v = flat[1:].view(a.shape)
    v.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    assert v.data_ptr() % 16 == 4
    return v


@pytest.mark.parametrize("o,rhs_zero", [(2, True), (6, True), (2, False), (6, False)])
def test_oras_tma_and_cp_async_tiles_agree(di, o, rhs_zero):
    # widths that are multiples of 4 with 16-byte aligned images take the TMA
    # path; the same data 4 bytes off that alignment takes cp.async: identical
    # tiles, identical bits
    h, w = 70, 96
    f, fn, c = _case(h, w, 3, 0.06, 4242 + o)
    g = np.random.default_rng(9)
    u = np.where(c.astype(bool), f, g.uniform(0, 255, f.shape)).astype(np.float32)
    b = fn if rhs_zero else g.uniform(-5, 5, f.shape).astype(np.float32)
    with di.Context(block=32, overlap=o) as ctx:
        a = N(ctx.oras_iteration(T(u), T(b), T(c), 8, rhs_zero=rhs_zero))
        bq = N(ctx.oras_iteration(_unaligned(u), _unaligned(b), T(c), 8, rhs_zero=rhs_zero))
    assert np.array_equal(a, bq)
    assert np.isfinite(a).all()


@pytest.mark.parametrize("h,w", [(64, 96), (31, 130)])
def test_transfers_vector_and_scalar_paths_agree(di, h, w):
    # even widths with 8-byte aligned images take the 8-byte-word paths of the
    # restriction and prolongation, the same data 4 bytes off alignment the
    # scalar paths: identical bits
    f, fn, c = _case(h, w, 2, 0.05, 77 + w)
    g = np.random.default_rng(3)
    u = np.where(c.astype(bool), 0.0, g.normal(size=f.shape)).astype(np.float32)
    b = np.where(c.astype(bool), 0.0, g.normal(size=f.shape)).astype(np.float32)
    cH = T(M.mask_downsample(c))
    ra = N(di.restrict_residual(T(u), T(b), T(c), cH, rhs_zero=False))
    rb = N(di.restrict_residual(_unaligned(u), _unaligned(b), T(c), cH, rhs_zero=False))
    assert np.array_equal(ra, rb)
    H, W = M.coarse_shape(h, w)
    e = g.uniform(-3, 3, (2, H, W)).astype(np.float32)
    ua, ub = T(u), _unaligned(u)
    di.prolong(T(e), T(c), 1, u=ua)
    di.prolong(T(e), T(c), 1, u=ub)
    assert np.array_equal(N(ua), N(ub))
    pa = N(di.prolong(T(e), T(c), 0, b=T(fn)))
    pb = N(di.prolong(T(e), T(c), 0, b=_unaligned(fn)))
    assert np.array_equal(pa, pb)


@pytest.mark.parametrize("h", [5, 31, 32, 33, 61, 62, 63, 77])
@pytest.mark.parametrize("w,o", [(96, 2), (95, 2), (64, 1), (70, 5), (62, 16), (33, 4)])
def test_oras_block_edges(di, h, w, o):
    # blocks clipped at every remainder of the block height, odd strides (tile
    # columns off 8-byte boundaries) and outputs off 8-byte boundaries: against
    # the oracle's K-step CG (the bound of test_oras_iteration_matches_oracle_cg)
    # and the same bits wherever u_out lies
    f, fn, c = _case(h, w, 2, 0.07, 7 * h + w + o)
    g = np.random.default_rng(h + w)
    u = np.where(c.astype(bool), f, g.uniform(0, 255, f.shape)).astype(np.float32)
    with di.Context(block=32, overlap=o, alpha=0.4) as ctx:
        out = N(ctx.oras_iteration(T(u), T(fn), T(c), 6, rhs_zero=True))
        ref = M.oras_iteration(u, M.rhs(f, c), c, 32, o, 0.4, ("cg", 6))
        assert np.abs(out - ref).max() < 1e-3 * np.abs(ref - u).max() + 2e-4
        off = _unaligned(np.zeros_like(u))
        assert np.array_equal(N(ctx.oras_iteration(T(u), T(fn), T(c), 6, rhs_zero=True, out=off)),
                              out)


@pytest.mark.parametrize("h,w", [(9, 17), (31, 33), (32, 95), (36, 64), (63, 40), (101, 130)])
@pytest.mark.parametrize("B,o", [(8, 1), (8, 3), (8, 4), (16, 1), (16, 3), (16, 5), (16, 8)])
def test_oras_shared_pixels_of_small_blocks(di, h, w, B, o):
    # the sums of pixels shared by blocks of 8 and 16, at ragged last blocks and
    # at the edges of a thread's four rows and a warp's 32 columns: against the
    # oracle's K-step CG (the bound of test_oras_iteration_matches_oracle_cg)
    f, fn, c = _case(h, w, 2, 0.07, 3 * h + w + B + o)
    g = np.random.default_rng(h * w)
    u = np.where(c.astype(bool), f, g.uniform(0, 255, f.shape)).astype(np.float32)
    with di.Context(block=B, overlap=o, alpha=0.4) as ctx:
        out = N(ctx.oras_iteration(T(u), T(fn), T(c), 4, rhs_zero=True))
    ref = M.oras_iteration(u, M.rhs(f, c), c, B, o, 0.4, ("cg", 4))
    assert np.abs(out - ref).max() < 1e-3 * np.abs(ref - u).max() + 2e-4


def _quad_tasks(di):
    # local problems up to which a launch takes four warps per problem
    fn = ctypes.CDLL(di.LIB_PATH)["_ZN2di15oras_quad_tasksEv"]
    fn.restype = ctypes.c_int
    return fn()


def _blocks(h, w, o):
    return len(M.axis_blocks(h, 32, o)) * len(M.axis_blocks(w, 32, o))


QUAD_CASES = [  # (h, w, overlap, aligned): up to 608 local problems in one channel, more in four
    (601, 600, 2, True), (500, 601, 6, True), (601, 640, 4, False), (660, 580, 2, False),
    (601, 600, 4, True), (487, 604, 6, True), (481, 320, 16, True),
]


@pytest.mark.parametrize("h,w,o,aligned", QUAD_CASES)
@pytest.mark.parametrize("rhs_zero", [True, False])
def test_oras_few_problems_same_bits(di, h, w, o, aligned, rhs_zero):
    # launches of few local problems take four warps per problem, larger ones two:
    # one channel alone and the same channel among four give the same bits, for
    # the plain iteration and both prolonged starts
    assert _blocks(h, w, o) <= _quad_tasks(di) < 4 * _blocks(h, w, o)
    f, fn, c = _case(h, w, 1, 0.06, h + 3 * w + o)
    g = np.random.default_rng(w)
    H, W = M.coarse_shape(h, w)
    known = c.astype(bool)
    if rhs_zero:
        u = np.where(known, f, g.uniform(0, 255, f.shape)).astype(np.float32)
        b = fn
    else:
        u = np.where(known, 0.0, g.normal(size=f.shape)).astype(np.float32)
        b = np.where(known, 0.0, g.normal(size=f.shape)).astype(np.float32)
    uH = g.uniform(0, 255, size=(1, H, W)).astype(np.float32)
    put = T if aligned else _unaligned
    outs = []
    with di.Context(block=32, overlap=o, alpha=0.3) as ctx:
        for C in (1, 4):
            ub, bb, eb = (np.repeat(a, C, axis=0) for a in (u, b, uH))
            r = [ctx.oras_iteration(put(ub), put(bb), T(c), 7, rhs_zero=rhs_zero),
                 ctx.prolong_oras_iteration(T(eb), put(ub), put(bb), T(c), 7, rhs_zero=rhs_zero),
                 ctx.oras_iteration(put(ub), put(bb), T(c), 400, rhs_zero=rhs_zero)]
            if rhs_zero:
                r.append(ctx.prolong_oras_iteration(T(eb), put(bb), put(bb), T(c), 7, rhs_zero=True,
                                                    mode=0))
            outs.append([N(x) for x in r])
    for a, b4 in zip(*outs):
        assert np.isfinite(a).all()
        for ch in range(4):
            assert np.array_equal(a[0], b4[ch])


@pytest.mark.parametrize("C,o", [(1, 2), (1, 6), (4, 2), (4, 6), (4, 5)])
@pytest.mark.parametrize("rhs_zero", [True, False])
def test_oras_of_a_scaled_image(di, C, o, rhs_zero):
    # the iteration is linear and powers of two are exact, so an image scaled by
    # one has the bits of the image's own result, also where r.r is no normal FP32
    # number any more (at 2^-72; a block with unknown pixels has |r| > 1 gray here,
    # so r.r stays above 2^-149, the smallest of all); one channel takes four warps
    # per local problem, four channels two
    h, w = 500, 600
    f, _, c = _case(h, w, C, 0.06, 77 + o, nan=False)
    g = np.random.default_rng(o)
    known = c.astype(bool)
    u = np.where(known, f, g.uniform(0, 255, f.shape)).astype(np.float32)
    b = g.normal(size=f.shape).astype(np.float32)
    with di.Context(block=32, overlap=o, alpha=0.5) as ctx:
        ref = N(ctx.oras_iteration(T(u), T(b), T(c), 12, rhs_zero=rhs_zero))
        assert np.abs(ref - u).max() > 1
        for e in (20, 40, -20, -40, -60, -66, -72):
            k = np.float32(2.0 ** e)
            out = N(ctx.oras_iteration(T(u * k), T(b * k), T(c), 12, rhs_zero=rhs_zero))
            assert np.array_equal(out, ref * k), e


TWO_WARP_CASES = [  # (h, w, overlap, aligned): last blocks of different heights and widths
    (480, 640, 2, True), (453, 640, 2, False), (461, 641, 2, True), (480, 640, 4, True),
    (437, 652, 4, True), (461, 640, 4, False), (480, 640, 6, True), (431, 604, 6, True),
    (449, 607, 6, True), (453, 600, 6, False), (300, 404, 16, True),
]


@pytest.mark.parametrize("h,w,o,aligned", TWO_WARP_CASES)
@pytest.mark.parametrize("rhs_zero", [True, False])
def test_oras_two_warps_per_problem(di, h, w, o, aligned, rhs_zero):
    # launches of more local problems than take four warps each, through TMA tiles
    # (aligned, w a multiple of 4) and cp.async: the iteration against the oracle's
    # (the bounds of test_oras_iteration_matches_oracle_cg) and both prolonged
    # starts against their two steps (identical bits)
    C, K = 3, 6
    assert C * _blocks(h, w, o) > _quad_tasks(di)
    f, fn, c = _case(h, w, C, 0.06, h + 5 * w + o)
    g = np.random.default_rng(3 * h + w)
    H, W = M.coarse_shape(h, w)
    known = c.astype(bool)
    if rhs_zero:
        u = np.where(known, f, g.uniform(0, 255, f.shape)).astype(np.float32)
        b, ref_b, atol = fn, M.rhs(f, c), 2e-4
    else:
        u = np.where(known, 0.0, g.normal(size=f.shape)).astype(np.float32)
        b = np.where(known, 0.0, g.normal(size=f.shape)).astype(np.float32)
        ref_b, atol = b, 1e-5
    uH = g.normal(scale=4.0, size=(C, H, W)).astype(np.float32)
    put = T if aligned else _unaligned
    with di.Context(block=32, overlap=o, alpha=0.4) as ctx:
        out = N(ctx.oras_iteration(put(u), put(b), T(c), K, rhs_zero=rhs_zero))
        ref = M.oras_iteration(u, ref_b, c, 32, o, 0.4, ("cg", K))
        assert np.abs(out - ref).max() < 1e-3 * np.abs(ref - u).max() + atol
        up = put(u)
        di.prolong(T(uH), T(c), 1, u=up)
        two = N(ctx.oras_iteration(up, put(b), T(c), K, rhs_zero=rhs_zero))
        fused = N(ctx.prolong_oras_iteration(T(uH), put(u), put(b), T(c), K, rhs_zero=rhs_zero))
        assert np.array_equal(fused, two)
        if rhs_zero:
            start = di.prolong(T(uH), T(c), 0, b=put(fn))
            two = N(ctx.oras_iteration(start, put(fn), T(c), K, rhs_zero=True))
            fused = N(ctx.prolong_oras_iteration(T(uH), put(fn), put(fn), T(c), K, rhs_zero=True,
                                                 mode=0))
            assert np.array_equal(fused, two)


@pytest.mark.parametrize("o", [1, 2, 5, 6, 16])
@pytest.mark.parametrize("h,w", [(77, 96), (62, 95)])
def test_oras_fp64_residual_steps(di, h, w, o):
    # FP64 block residuals at even and odd overlaps, with and without a right-hand
    # side: the bounds of test_oras_iteration_matches_oracle_cg
    f, fn, c = _case(h, w, 2, 0.07, h + w + o)
    g = np.random.default_rng(o)
    known = c.astype(bool)
    u = np.where(known, f, g.uniform(0, 255, f.shape)).astype(np.float32)
    e = np.where(known, 0.0, g.normal(size=f.shape)).astype(np.float32)
    b = np.where(known, 0.0, g.normal(size=f.shape)).astype(np.float32)
    with di.Context(block=32, overlap=o, alpha=0.4, refine_fp64=1) as ctx:
        out = N(ctx.oras_iteration(T(u), T(fn), T(c), 6, rhs_zero=True))
        ref = M.oras_iteration(u, M.rhs(f, c), c, 32, o, 0.4, ("cg", 6))
        assert np.abs(out - ref).max() < 1e-3 * np.abs(ref - u).max() + 2e-4
        out = N(ctx.oras_iteration(T(e), T(b), T(c), 6, rhs_zero=False))
        ref = M.oras_iteration(e, b, c, 32, o, 0.4, ("cg", 6))
        assert np.abs(out - ref).max() < 1e-3 * np.abs(ref - e).max() + 1e-5


@pytest.mark.parametrize("w", [16, 48, 64, 112, 4112])
@pytest.mark.parametrize("h", [1, 31, 33, 130])
def test_packed_mask_sixteen_columns_at_a_time(di, h, w):
    # rows of whole 16-byte groups: the unknown count and the solution's mask
    # pixels show the packed words
    f, fn, c = _case(h, w, 1, 0.1, 5 * h + w)
    c[-1, -1] = 1
    fn[:, -1, -1] = f[:, -1, -1]
    with di.Context(max_cycles=2, stop_rule=2) as ctx:
        u, _ = ctx.inpaint(T(fn), T(c))
        assert ctx.stats()["unknowns"] == int((c == 0).sum())
    assert np.array_equal(N(u)[:, c == 1], f[:, c == 1])
    g = np.random.default_rng(3)
    u0 = np.where(c.astype(bool), f, g.uniform(0, 255, f.shape)).astype(np.float32)
    with di.Context(block=32, overlap=2) as ctx:  # the same mask off the 16-byte boundary
        flat = torch.empty(c.size + 1, dtype=torch.uint8, device=DEV)
        co = flat[1:].view(c.shape)
        co.copy_(torch.from_numpy(c))
        a = N(ctx.oras_iteration(T(u0), T(fn), T(c), 5, rhs_zero=True))
        assert np.array_equal(N(ctx.oras_iteration(T(u0), T(fn), co, 5, rhs_zero=True)), a)


@pytest.mark.parametrize("h,w", [(1999, 2003), (1201, 2048), (577, 3333)])
def test_pyramid_level_large_and_odd(di, h, w):
    # four rows of cells per thread: the same bits as the separate steps at
    # ragged rows and columns
    f, fn, c = _case(h, w, 3, 0.05, h + w)
    cH, bH, _, unk = di.pyramid_level(T(c), T(fn))
    cH_ref = M.mask_downsample(c)
    assert np.array_equal(N(cH), cH_ref) and int(N(unk)[0]) == int((cH_ref == 0).sum())
    assert np.array_equal(N(bH), N(di.values_downsample(T(c), T(fn), T(cH_ref))))


@pytest.mark.parametrize("h,w", [(1999, 2003), (1201, 2048), (577, 3333), (700, 1000)])
@pytest.mark.parametrize("C,modified,density", [(1, False, 0.05), (4, False, 0.6), (1, True, 0.6),
                                                (4, True, 0.6)])
def test_pyramid_level_forms(di, h, w, C, modified, density):
    # the naive average (two rows of cells per thread, one on smaller levels; gray
    # by itself) and the weights of mostly known cells: the same bits as the
    # separate steps
    f, fn, c = _case(h, w, C, density, h + w + C)
    cH, bH, _, unk = di.pyramid_level(T(c), T(fn), modified=modified)
    cH_ref = M.mask_downsample(c)
    assert np.array_equal(N(cH), cH_ref) and int(N(unk)[0]) == int((cH_ref == 0).sum())
    assert np.array_equal(N(bH), N(di.values_downsample(T(c), T(fn), T(cH_ref),
                                                        modified=modified)))


@pytest.mark.parametrize("C", [2, 3, 4])
@pytest.mark.parametrize("h,w,aligned", [(1200, 1100, True), (1101, 1203, True), (1200, 1100, False)])
@pytest.mark.parametrize("rhs_zero", [True, False])
def test_restrict_all_channels_of_a_cell(di, h, w, C, aligned, rhs_zero):
    # large levels restrict every channel of a cell in one thread: the same bits
    # as channel by channel
    f, fn, c = _case(h, w, C, 0.05, h + C)
    g = np.random.default_rng(C)
    u = np.where(c.astype(bool), f, g.uniform(0, 255, f.shape)).astype(np.float32)
    b = fn if rhs_zero else g.normal(size=f.shape).astype(np.float32)
    put = T if aligned else _unaligned
    cH = di.mask_downsample(T(c))
    r = N(di.restrict_residual(put(u), put(b), T(c), cH, rhs_zero=rhs_zero))
    for ch in range(C):
        one = N(di.restrict_residual(put(u[ch:ch + 1]), put(b[ch:ch + 1]), T(c), cH,
                                     rhs_zero=rhs_zero))
        assert np.array_equal(r[ch], one[0])


@pytest.mark.parametrize("h,w,C", [(70, 95, 1), (1101, 1203, 3), (1200, 1100, 4)])
@pytest.mark.parametrize("density", [0.7, 1.0])
def test_restrict_of_mostly_known_images(di, h, w, C, density):
    # known cells give 0, the few others what test_restrict_residual says
    f, fn, c = _case(h, w, C, density, h + w)
    cH = M.mask_downsample(c)
    g = np.random.default_rng(6)
    u = np.where(c.astype(bool), f, g.uniform(0, 255, f.shape)).astype(np.float32)
    b = np.where(c.astype(bool), 0.0, g.normal(size=f.shape)).astype(np.float32)
    for rhs, rhs_zero in ((fn, True), (b, False)):
        rH = N(di.restrict_residual(T(u), T(rhs), T(c), T(cH), rhs_zero=rhs_zero))
        ref = M.restrict_residual(M.residual(u, M.rhs(f, c) if rhs_zero else b, c), cH)
        assert np.abs(rH - ref).max() < 1e-3
        assert not rH[:, cH == 1].any()


PRO_CASES = [  # (h, w, overlap, rhs_zero, aligned)
    (70, 96, 2, True, True), (70, 96, 2, False, False), (70, 96, 6, False, True),
    (33, 35, 2, False, True), (130, 100, 2, True, False), (61, 250, 6, True, True),
    (1, 9, 2, False, True), (7, 1, 2, True, True), (3, 5, 6, False, False),
    (17, 33, 2, False, True), (95, 64, 4, False, True), (71, 96, 2, False, True),
    (129, 160, 6, True, True),
]


@pytest.mark.parametrize("h,w,o,rhs_zero,aligned", PRO_CASES)
def test_prolong_oras_iteration_bit_identical_to_two_steps(di, h, w, o, rhs_zero, aligned):
    # the decoder's correction step inside the first post-smoothing iteration
    # (mode 1): the same bits as the prolongation on a copy followed by the
    # plain iteration, through both tile paths (TMA where aligned) and the
    # ragged right and bottom blocks
    C = 3
    f, fn, c = _case(h, w, C, 0.08, 31 * h + w + o)
    g = np.random.default_rng(h + 7 * w)
    H, W = M.coarse_shape(h, w)
    if rhs_zero:
        u = np.where(c.astype(bool), f, g.uniform(0, 255, f.shape)).astype(np.float32)
        b = fn
    else:
        u = np.where(c.astype(bool), 0.0, g.normal(size=f.shape)).astype(np.float32)
        b = np.where(c.astype(bool), 0.0, g.normal(size=f.shape)).astype(np.float32)
    uH = g.normal(scale=4.0, size=(C, H, W)).astype(np.float32)
    put = T if aligned else _unaligned
    with di.Context(block=32, overlap=o) as ctx:
        ut = put(u)
        fused = N(ctx.prolong_oras_iteration(T(uH), ut, put(b), T(c), 8, rhs_zero=rhs_zero))
        assert np.array_equal(N(ut), u)  # u_in is not modified
        up = put(u)
        di.prolong(T(uH), T(c), 1, u=up)
        two = N(ctx.oras_iteration(up, put(b), T(c), 8, rhs_zero=rhs_zero))
    assert np.array_equal(fused, two)
    # and against the oracle's two steps
    start = M.prolong_correct(u.astype(np.float64), uH, c)
    ref = M.oras_iteration(start, M.rhs(f, c) if rhs_zero else b, c, 32, o, 0.5, ("cg", 8))
    scale = np.abs(ref - start).max() + np.abs(start).max() * 1e-5
    assert np.abs(fused - ref).max() < 1e-3 * scale + 2e-4


@pytest.mark.parametrize("h,w,o,aligned", [(70, 96, 2, True), (70, 96, 6, False),
                                           (33, 35, 2, True), (1, 9, 2, True),
                                           (130, 100, 2, False), (61, 250, 4, True)])
def test_prolong_oras_iteration_interpolation_bit_identical(di, h, w, o, aligned):
    # the cascade's step (mode 0): u_in = b (not finite off the mask, where it
    # must not be read), the start is b on the mask and P uH elsewhere
    C = 3
    f, fn, c = _case(h, w, C, 0.08, 17 * h + w + o)
    g = np.random.default_rng(2 * h + w)
    H, W = M.coarse_shape(h, w)
    uH = g.uniform(0, 255, size=(C, H, W)).astype(np.float32)
    put = T if aligned else _unaligned
    with di.Context(block=32, overlap=o) as ctx:
        fused = N(ctx.prolong_oras_iteration(T(uH), put(fn), put(fn), T(c), 8, rhs_zero=True,
                                             mode=0))
        start = di.prolong(T(uH), T(c), 0, b=put(fn))
        two = N(ctx.oras_iteration(start, put(fn), T(c), 8, rhs_zero=True))
    assert np.isfinite(fused).all()
    assert np.array_equal(fused, two)
    s0 = M.prolong_solution(uH, f, c)
    ref = M.oras_iteration(s0, M.rhs(f, c), c, 32, o, 0.5, ("cg", 8))
    assert np.abs(fused - ref).max() < 1e-3 * np.abs(ref - s0).max() + 2e-4


def test_prolong_oras_iteration_4k_rgb(di):
    # the finest level of the bench frames' size (3840 x 2160 x 3): bit-identical
    # to the two steps
    h, w, C = 2160, 3840, 3
    g = torch.Generator(device=DEV).manual_seed(5)
    c = (torch.rand((h, w), generator=g, device=DEV) < 0.04).to(torch.uint8)
    f = torch.rand((C, h, w), generator=g, device=DEV) * 255
    u = torch.where(c.bool(), f, torch.full_like(f, 128.0))
    uH = torch.randn((C, (h + 1) // 2, (w + 1) // 2), generator=g, device=DEV) * 4
    with di.Context(block=32, overlap=2) as ctx:
        fused = ctx.prolong_oras_iteration(uH, u, f, c, 10, rhs_zero=True)
        up = u.clone()
        di.prolong(uH, c, 1, u=up)
        two = ctx.oras_iteration(up, f, c, 10, rhs_zero=True)
    torch.cuda.synchronize()
    assert torch.equal(fused, two)


@pytest.mark.parametrize("kw", [dict(block=32, overlap=3), dict(block=16, overlap=2),
                                dict(block=32, overlap=2, precision=1)])
def test_prolong_oras_iteration_rejects_other_configurations(di, kw):
    f, fn, c = _case(40, 40, 1, 0.1, 3)
    uH = np.zeros((1, 20, 20), np.float32)
    with di.Context(**kw) as ctx:
        with pytest.raises(di.DiError):
            ctx.prolong_oras_iteration(T(uH), T(f), T(fn), T(c), 4, rhs_zero=True)
