"""GPU parity: every CUDA entry point, called through the C-ABI binding, against the fp64 CPU
oracle on the same seeded inputs.

Tolerances:
  * packed bits: bit-exact, except in groups the oracle flags as near-ties (decision margin
    below 2^-20 of mean|w|), where rounding order may legitimately flip a bit;
  * quantizer alpha: |a - a_ref| <= 1e-5 * max(|a_ref|, mean|w_group|);
  * fp32 outputs of fwd / dX / dalpha: max|out - ref| / max|ref| <= 2e-3 (the bound the task
    states for bf16 inputs with fp32 accumulation; the kernels round the scaled weight once to
    fp16 and land near 3e-4; dalpha multiplies exact bf16 values and lands near 3e-7);
  * bf16 outputs: the same bound plus one bf16 rounding (2^-8 relative).
"""
import numpy as np
import pytest

import oracle
import paper_2210_03858_b200 as bcq
from paper_2210_03858_b200 import build as bcq_build
from paper_2210_03858_b200 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = 2e-3


@pytest.fixture(scope="module", autouse=True)
def _built():
    bcq_build.build_library()
    assert torch.cuda.is_available()
    yield
    bcq.check_device()  # raises if a kernel reported an expired wait
    assert bcq.device_timeout_flag() == 0, "a kernel reported an expired wait"


def dev_bf16(a_u16):
    return torch.from_numpy(a_u16.view(np.int16)).cuda().view(torch.bfloat16)


def dev_bits(bits_u32):
    return torch.from_numpy(bits_u32.view(np.int32)).cuda()


def host_bits(t):
    return t.cpu().numpy().view(np.uint32)


def rel_err(out, ref):
    return float(np.abs(out.astype(np.float64) - ref).max() / np.abs(ref).max())


def make_case(seed, n, d_in, d_out, q, g, alt=0, outliers=0.0):
    key = (100, seed, 0)
    W = synth.weights(d_out, d_in, key, outlier_frac=outliers)
    X = synth.activations(n, d_in, key, synth.ROLE_X)
    dY = synth.activations(n, d_out, key, synth.ROLE_DY)
    bits, alpha, sq_err, margin = oracle.quantize(W, q, g, alt_iters=alt)
    return W, X, dY, bits, alpha, sq_err, margin


# --------------------------------------------------------------------------- quantizer

QUANT_CASES = [
    # d_out, d_in, q, g, alt, outliers
    (64, 128, 3, 128, 0, 0.0),
    (37, 1000, 3, 1000, 0, 0.0),      # row-wise, d_in not a multiple of 32
    (50, 1600, 4, 128, 0, 0.0),       # ragged last group (64)
    (24, 1024, 1, 32, 0, 0.0),
    (9, 4096, 2, 4096, 0, 0.0),       # CTA-wide teams
    (3, 20480, 2, 20480, 0, 0.0),
    (5, 8192, 8, 2048, 0, 0.0),
    (40, 512, 2, 128, 5, 1e-3),
    (40, 512, 3, 128, 5, 1e-3),
    (40, 640, 4, 128, 5, 1e-3),
    (16, 1024, 3, 1024, 3, 0.0),
    (6, 2304, 4, 2304, 2, 0.0),
    (12, 200, 5, 200, 1, 0.0),
    (32, 768, 3, 128, 15, 1e-3),      # the 15 alternating rounds of the paper's appendix
    (32, 768, 4, 128, 15, 1e-3),
]


@pytest.mark.parametrize("d_out,d_in,q,g,alt,outl", QUANT_CASES)
def test_quantize_matches_oracle(d_out, d_in, q, g, alt, outl):
    W, _, _, bits_ref, alpha_ref, sq_ref, margin = make_case(d_in + q, 1, d_in, d_out, q, g, alt, outl)
    bits, alpha, sq_err = bcq.quantize(torch.from_numpy(W).cuda(), q, g, alt, want_sq_err=True)
    torch.cuda.synchronize()
    bits, alpha, sq_err = host_bits(bits), alpha.cpu().numpy(), sq_err.cpu().numpy()
    G = oracle.num_groups(d_in, g)
    # padding bits are zero
    total = bits.shape[2] * 32
    kk = np.arange(d_in, total)
    if kk.size:
        assert not ((bits[:, :, kk >> 5] >> (kk & 31).astype(np.uint32)) & 1).any()
    flagged = margin < 2.0 ** -20
    diff_words = bits != bits_ref
    if diff_words.any():
        # every differing bit must sit in a flagged group
        k = np.arange(d_in)
        dbit = ((bits ^ bits_ref)[:, :, k >> 5] >> (k & 31).astype(np.uint32)) & 1
        for c in range(G):
            bad = dbit[:, :, c * g:(c + 1) * g].any(axis=(0, 2))
            assert not (bad & ~flagged[:, c]).any(), "bits differ in a group that is not a near-tie"
    same = ~np.stack([(bits != bits_ref)[:, :, (c * g) >> 5:((min((c + 1) * g, d_in) + 31) >> 5)].any(axis=(0, 2))
                      for c in range(G)], axis=1)
    assert same.mean() > 0.999
    mean_abs = np.stack([np.abs(W[:, c * g:(c + 1) * g]).mean(axis=1) for c in range(G)], axis=1)
    tol = 1e-5 * np.maximum(np.abs(alpha_ref), mean_abs[None])
    ok = np.abs(alpha - alpha_ref) <= tol
    assert ok[:, same].all()
    np.testing.assert_allclose(sq_err[same], sq_ref[same], rtol=1e-6, atol=1e-18)


@pytest.mark.parametrize("alt", [0, 2, 3])
@pytest.mark.parametrize("d_in,g", [(96, 32), (200, 64), (420, 96), (520, 160), (900, 256), (1100, 512), (1023, 1023),
                                    (2050, 2050), (5000, 2528), (8192, 8192), (12001, 12001), (20000, 20000)])
def test_quantize_team_sizes_with_exact_ties(d_in, g, alt):
    # Multiples of 1/64 with many zeros (also -0.0) and repeated magnitudes: every sum the quantizer
    # forms from them is exact in fp64 whatever its order (values below 2, at most 2^15 of them, 24
    # bits each), so ties are ties on both sides and the bits have to be the oracle's, one for one.
    rng = np.random.default_rng(d_in + alt)
    for q in (1, 2, 3, 4) if d_in < 3000 else (3,):
        W = (rng.integers(-6, 7, size=(5, d_in)) / 64.0).astype(np.float32)
        W[0, ::3] = -0.0
        W[1] = 0.0
        W[2, : d_in // 2] = 0.25
        Wd = torch.zeros((5, d_in + 1), dtype=torch.float32, device="cuda")[:, 1:]   # rows not 16-byte aligned
        Wd.copy_(torch.from_numpy(W))
        bits_ref, alpha_ref, sq_ref, _ = oracle.quantize(W, q, g, alt_iters=alt)
        for src in (Wd, torch.from_numpy(W).cuda()):
            bits, alpha, sq = bcq.quantize(src, q, g, alt, want_sq_err=True)
            np.testing.assert_array_equal(host_bits(bits), bits_ref)
            np.testing.assert_allclose(alpha.cpu().numpy(), alpha_ref, rtol=1e-6, atol=1e-9)
            np.testing.assert_allclose(sq.cpu().numpy(), sq_ref, rtol=1e-6, atol=1e-12)


@pytest.mark.parametrize("alt", [2, 3])
@pytest.mark.parametrize("d_in,g", [(100, 32), (420, 96), (260, 128), (700, 256), (900, 512), (1023, 1023), (1582, 1582)])
def test_quantize_alternating_short_and_long_problems(d_in, g, alt):
    # The size of the team depends on how much there is to do: the same five rows alone and repeated past
    # every line (98304 weights per SM at most).  Values as in the test above, so the bits are the oracle's exactly.
    # (Groups of up to 256 are taken by teams with two rounds, with three by lanes on sorted magnitudes.)
    rng = np.random.default_rng(d_in)
    W = (rng.integers(-6, 7, size=(5, d_in)) / 64.0).astype(np.float32)
    W[0, ::3] = -0.0
    W[2, : d_in // 2] = 0.25
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    reps = (99000 if 128 < g <= 512 else 30720) * sms // (5 * -(-d_in // g) * g) + 1
    Wd = torch.from_numpy(W).cuda()
    for q in (1, 2, 3, 4):
        bits_ref, alpha_ref, sq_ref, _ = oracle.quantize(W, q, g, alt_iters=alt)
        for r in (1, reps):
            bits, alpha, sq = bcq.quantize(Wd.repeat(r, 1), q, g, alt, want_sq_err=True)
            np.testing.assert_array_equal(host_bits(bits), np.tile(bits_ref, (1, r, 1)))
            np.testing.assert_allclose(alpha.cpu().numpy(), np.tile(alpha_ref, (1, r, 1)), rtol=1e-6, atol=1e-9)
            np.testing.assert_allclose(sq.cpu().numpy(), np.tile(sq_ref, (r, 1)), rtol=1e-6, atol=1e-12)


@pytest.mark.parametrize("alt", [0, 2])
@pytest.mark.parametrize("d_in,g", [(64, 32), (130, 64), (420, 128), (1000, 1000), (3000, 3000)])
def test_quantize_weights_that_are_not_finite(d_in, g, alt):
    # r >= 0 is false for a NaN whatever its sign bit, and a group with an infinity has NaN residuals from its
    # second plane on: the bits of such groups (and of their neighbours) are the oracle's all the same
    rng = np.random.default_rng(d_in)
    W = (rng.integers(-6, 7, size=(7, d_in)) / 64.0).astype(np.float32)
    W[0, 3], W[1, 5], W[2, 7], W[3, d_in - 1] = np.nan, np.inf, -np.inf, np.float32(-np.nan)
    W[4, 9], W[4, 11], W[5, :] = np.inf, -np.inf, np.nan
    for q in (1, 2, 3, 4):
        bits_ref, alpha_ref, sq_ref, _ = oracle.quantize(W, q, g, alt_iters=alt)
        bits, alpha, sq = bcq.quantize(torch.from_numpy(W).cuda(), q, g, alt, want_sq_err=True)
        np.testing.assert_array_equal(host_bits(bits), bits_ref)
        np.testing.assert_allclose(alpha.cpu().numpy(), alpha_ref, rtol=1e-6, atol=1e-9, equal_nan=True)
        np.testing.assert_allclose(sq.cpu().numpy(), sq_ref, rtol=1e-6, atol=1e-12, equal_nan=True)


@pytest.mark.parametrize("d_in,g", [(64, 32), (256, 64), (640, 128), (1000, 256), (1700, 512), (700, 700), (1500, 1500)])
def test_quantize_a_row_alone_and_among_many(d_in, g):
    # Every (row, group) is a problem of its own: what a row becomes must not depend on how many others are
    # in the call, to the last bit, though the teams that share a group differ in size.
    gen = torch.Generator(device="cuda").manual_seed(d_in)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = (99000 if 128 < g <= 512 else 30720) * sms // (-(-d_in // g) * g) + 1  # past every line between the team sizes
    W = torch.randn((rows, d_in), generator=gen, device="cuda") * 0.02
    pick = slice(rows // 2, rows // 2 + 600)
    for q, alt in ((1, 3), (2, 3), (3, 3), (4, 3), (4, 0), (2, 2), (3, 2), (4, 2), (2, 4)):
        bits, alpha, sq = bcq.quantize(W, q, g, alt, want_sq_err=True)
        b, a, s = bcq.quantize(W[pick].contiguous(), q, g, alt, want_sq_err=True)
        assert torch.equal(b, bits[:, pick]) and torch.equal(a, alpha[:, pick]) and torch.equal(s, sq[pick])


@pytest.mark.parametrize("alt", [3, 15])
@pytest.mark.parametrize("d_in,g", [(32, 32), (64, 64), (130, 64), (288, 96), (420, 128), (256, 256), (1001, 256),
                                    (500, 160), (580, 192), (450, 224)])
def test_quantize_rounds_on_sorted_magnitudes(d_in, g, alt):
    # Values whose sums are exact in fp64 (see above), so that the bits are the oracle's: ties with a scale and with a
    # midpoint, groups of one magnitude, of zeros, with one weight far above the rest, infinities and NaNs; rows
    # that are no multiple of a warp's share, aligned and not, alone and 150 times, and in rows whose padding is not to be read.
    rng = np.random.default_rng(d_in + alt)
    W = (rng.integers(-40, 41, size=(13, d_in)) / 64.0).astype(np.float32)
    W[0, ::3], W[1], W[2] = -0.0, 0.0, np.where(rng.random(d_in) < 0.5, 0.25, -0.25)
    W[3] = rng.integers(-1, 2, size=d_in) * 0.5
    W[4, d_in // 2] = 1024.0
    W[5, 3], W[6, 5], W[7, 7], W[8, :], W[9, [1, 9]] = np.nan, np.inf, -np.inf, np.nan, (np.inf, -np.inf)
    W[10, 0] = np.array([0x7FFFFFFF], np.uint32).view(np.float32)[0]
    odd = torch.zeros((13, d_in + 1), dtype=torch.float32, device="cuda")[:, 1:]
    odd.copy_(torch.from_numpy(W))
    padded = torch.full((13, -(-d_in // 4) * 4 + 4), 7e4, dtype=torch.float32, device="cuda")[:, :d_in]
    padded.copy_(torch.from_numpy(W))
    for q in (2, 3, 4):
        bits_ref, alpha_ref, sq_ref, _ = oracle.quantize(W, q, g, alt_iters=alt)
        for src, r in ((odd, 1), (padded, 1), (torch.from_numpy(W).cuda(), 1), (torch.from_numpy(W).cuda().repeat(150, 1), 150)):
            bits, alpha, sq = bcq.quantize(src, q, g, alt, want_sq_err=True)
            np.testing.assert_array_equal(host_bits(bits), np.tile(bits_ref, (1, r, 1)))
            np.testing.assert_allclose(alpha.cpu().numpy(), np.tile(alpha_ref, (1, r, 1)), rtol=1e-6, atol=1e-9, equal_nan=True)
            np.testing.assert_allclose(sq.cpu().numpy(), np.tile(sq_ref, (r, 1)), rtol=1e-6, atol=1e-12, equal_nan=True)


@pytest.mark.parametrize("d_in,g", [(32, 32), (130, 64), (288, 96), (420, 128), (1001, 256)])
def test_quantize_sorted_rounds_in_blocks_of_four_warps(d_in, g):
    # From 24 warps an SM on, four warps of 32 groups (16 with more than 128 weights) share a block.  The last block's warps
    # past the last group repeat it; its row, the last, is not finite.  What every copy of the rows becomes is what they
    # become alone (which the test above compares with the oracle).
    rng = np.random.default_rng(d_in)
    W = (rng.integers(-40, 41, size=(13, d_in)) / 64.0).astype(np.float32)
    W[0, ::3], W[1] = -0.0, 0.0
    W[4, 3], W[12, [0, d_in - 1]] = np.inf, (np.inf, np.nan)
    Wd = torch.from_numpy(W).cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    G, share = -(-d_in // g), 32 if g <= 128 else 16
    reps = 24 * sms * share // (13 * G) + 1
    while -(-13 * reps * G // share) % 4 == 0:
        reps += 1
    for q in (2, 3, 4):
        one = bcq.quantize(Wd, q, g, 4, want_sq_err=True)
        many = bcq.quantize(Wd.repeat(reps, 1), q, g, 4, want_sq_err=True)
        for a, b, rows in zip(one, many, (1, 1, 0)):
            want = a.repeat((1, reps, 1) if rows else (reps, 1))
            if a.dtype == torch.int32:
                assert torch.equal(want, b)
            else:
                assert torch.equal(want.nan_to_num(nan=1.5, posinf=2.5, neginf=3.5), b.nan_to_num(nan=1.5, posinf=2.5, neginf=3.5))


def test_quantize_strided_input_and_determinism():
    W = synth.weights(48, 384, (101, 0, 0))
    Wp = np.zeros((48, 400), dtype=np.float32)
    Wp[:, :384] = W
    ref_bits, ref_alpha, _, _ = oracle.quantize(W, 3, 128)
    Wd = torch.from_numpy(Wp).cuda()[:, :384]
    b1, a1, _ = bcq.quantize(Wd, 3, 128)
    b2, a2, _ = bcq.quantize(Wd, 3, 128)
    torch.cuda.synchronize()
    assert torch.equal(b1, b2) and torch.equal(a1, a2)
    np.testing.assert_array_equal(host_bits(b1), ref_bits)
    np.testing.assert_array_equal(a1.cpu().numpy(), ref_alpha)


def test_dequantize_matches_oracle():
    for (d_out, d_in, q, g) in ((33, 1000, 3, 1000), (20, 1600, 4, 128), (7, 96, 2, 32)):
        _, _, _, bits, alpha, _, _ = make_case(7, 1, d_in, d_out, q, g)
        out = bcq.dequantize(dev_bits(bits), torch.from_numpy(alpha).cuda(), d_in, g).cpu().numpy()
        ref = oracle.dequantize(bits, alpha, d_in, g)
        np.testing.assert_allclose(out, ref, rtol=1e-6, atol=1e-9)


# --------------------------------------------------------------------------- linear layer

LINEAR_CASES = [
    # n, d_in, d_out, q, g
    (512, 1024, 1024, 3, 1024),    # the single-layer workload: several tiles, row-wise
    (300, 1000, 200, 4, 1000),     # ragged everywhere, row-wise with d_in % 32 != 0
    (257, 1600, 336, 4, 128),      # ragged last group, partial tiles in every dimension
    (64, 256, 128, 1, 32),         # smallest group size
    (130, 320, 384, 2, 96),        # groups not aligned to the tile widths
    (1100, 512, 640, 3, 256),      # more token tiles than one wave of a small grid
    (96, 2048, 256, 8, 512),       # q = 8
]


def _upload(X, dY, bits, alpha):
    return dev_bf16(X), dev_bf16(dY), dev_bits(bits), torch.from_numpy(alpha).cuda()


@pytest.mark.parametrize("n,d_in,d_out,q,g", LINEAR_CASES)
def test_fwd_matches_oracle(n, d_in, d_out, q, g):
    _, X, dY, bits, alpha, _, _ = make_case(n, n, d_in, d_out, q, g)
    Xd, _, bd, ad = _upload(X, dY, bits, alpha)
    ref = oracle.fwd(X, bits, alpha, d_in, g)
    Y = bcq.linear_fwd(Xd, bd, ad, d_in, g)
    Y2 = bcq.linear_fwd(Xd, bd, ad, d_in, g)
    torch.cuda.synchronize()
    assert torch.equal(Y, Y2), "two runs differ"
    assert rel_err(Y.cpu().numpy(), ref) <= TOL
    # bias and bf16 output
    bias = synth.bias(d_out, (100, n, 0))
    Yb = bcq.linear_fwd(Xd, bd, ad, d_in, g, bias=torch.from_numpy(bias).cuda(),
                        out_dtype=torch.bfloat16)
    Yb2 = bcq.linear_fwd(Xd, bd, ad, d_in, g, bias=torch.from_numpy(bias).cuda(),
                         out_dtype=torch.bfloat16)
    refb = ref + bias.astype(np.float64)
    assert torch.equal(Yb, Yb2), "two bf16 runs differ"
    assert rel_err(Yb.float().cpu().numpy(), refb) <= TOL + 2.0 ** -8


@pytest.mark.parametrize("n,d_in,d_out,q,g", LINEAR_CASES)
def test_bwd_x_matches_oracle(n, d_in, d_out, q, g):
    _, X, dY, bits, alpha, _, _ = make_case(n, n, d_in, d_out, q, g)
    _, dYd, bd, ad = _upload(X, dY, bits, alpha)
    ref = oracle.bwd_x(dY, bits, alpha, d_in, g)
    dX = bcq.linear_bwd_x(dYd, bd, ad, d_in, g)
    dX2 = bcq.linear_bwd_x(dYd, bd, ad, d_in, g)
    torch.cuda.synchronize()
    assert torch.equal(dX, dX2)
    assert rel_err(dX.cpu().numpy(), ref) <= TOL
    dXb = bcq.linear_bwd_x(dYd, bd, ad, d_in, g, out_dtype=torch.bfloat16)
    dXb2 = bcq.linear_bwd_x(dYd, bd, ad, d_in, g, out_dtype=torch.bfloat16)
    assert torch.equal(dXb, dXb2), "two bf16 runs differ"
    assert rel_err(dXb.float().cpu().numpy(), ref) <= TOL + 2.0 ** -8


@pytest.mark.parametrize("n,d_in,d_out,q,g", LINEAR_CASES)
def test_bwd_alpha_matches_oracle(n, d_in, d_out, q, g):
    _, X, dY, bits, alpha, _, _ = make_case(n, n, d_in, d_out, q, g)
    Xd, dYd, bd, _ = _upload(X, dY, bits, alpha)
    ref = oracle.bwd_alpha(dY, X, bits, d_in, g)
    dA = bcq.linear_bwd_alpha(dYd, Xd, bd, d_in, g)
    dA2 = bcq.linear_bwd_alpha(dYd, Xd, bd, d_in, g)
    torch.cuda.synchronize()
    assert torch.equal(dA, dA2)
    assert rel_err(dA.cpu().numpy(), ref) <= TOL
    # alpha_1 only, the paper's 1/g scale, accumulate on top of existing values
    out = torch.full_like(dA, 3.0)
    bcq.linear_bwd_alpha(dYd, Xd, bd, d_in, g, plane_mask=1, scale=1.0 / g, accumulate=True, out=out)
    o = out.cpu().numpy()
    assert (o[1:] == 3.0).all()
    assert np.abs(o[0] - 3.0 - ref[0] / g).max() <= TOL * np.abs(ref[0] / g).max() + 1e-6


@pytest.mark.parametrize("n,d_in,d_out,q,g", [(65, 40, 136, 2, 40), (64, 64, 256, 3, 32), (127, 136, 264, 1, 136),
                                              (200, 320, 384, 4, 64), (640, 456, 104, 2, 128)])
def test_bwd_alpha_partial_tiles_of_a_cta_pair(n, d_in, d_out, q, g):
    # last column tiles of 64, 128 and 192 columns (32, 64 and 96 in each CTA of the pair), and row tiles
    # that hold rows for one CTA of the pair only
    _, X, dY, bits, alpha, _, _ = make_case(40 + n, n, d_in, d_out, q, g)
    Xd, dYd, bd, _ = _upload(X, dY, bits, alpha)
    ref = oracle.bwd_alpha(dY, X, bits, d_in, g)
    assert rel_err(bcq.linear_bwd_alpha(dYd, Xd, bd, d_in, g).cpu().numpy(), ref) <= TOL


@pytest.mark.parametrize("mask", [0b1, 0b10, 0b1010, 0b10000000, 0b11010110, 0b11111111])
@pytest.mark.parametrize("n,d_in,d_out,g", [(130, 200, 72, 200), (70, 320, 136, 32)])
def test_bwd_alpha_of_some_planes(n, d_in, d_out, g, mask):
    # planes of the mask are written, the others keep what they held
    q = 8
    _, X, dY, bits, alpha, _, _ = make_case(60 + n, n, d_in, d_out, q, g)
    Xd, dYd, bd, ad = _upload(X, dY, bits, alpha)
    ref = oracle.bwd_alpha(dY, X, bits, d_in, g)
    out = torch.full_like(ad, 7.0)
    bcq.linear_bwd_alpha(dYd, Xd, bd, d_in, g, plane_mask=mask, out=out)
    o = out.cpu().numpy()
    for i in range(q):
        if (mask >> i) & 1:
            assert np.abs(o[i] - ref[i]).max() <= TOL * np.abs(ref).max()
        else:
            assert (o[i] == 7.0).all()


@pytest.mark.parametrize("n", [1, 4, 16, 5])
@pytest.mark.parametrize("d_in,d_out,q,g", [(4096, 1536, 3, 128), (1024, 520, 4, 128), (2048, 256, 3, 2048)])
def test_decode_matches_oracle(n, d_in, d_out, q, g):
    _, X, dY, bits, alpha, _, _ = make_case(n + d_out, n, d_in, d_out, q, g)
    Xd, _, bd, ad = _upload(X, dY, bits, alpha)
    ref = oracle.fwd(X, bits, alpha, d_in, g)
    Y = bcq.linear_decode(Xd, bd, ad, d_in, g)
    Y2 = bcq.linear_decode(Xd, bd, ad, d_in, g)
    torch.cuda.synchronize()
    assert torch.equal(Y, Y2)
    assert rel_err(Y.cpu().numpy(), ref) <= TOL


@pytest.mark.parametrize("n,d_in,d_out,q,g", [c for c in LINEAR_CASES if c[3] <= 4] + [(200, 640, 304, 2, 128),
                                                                                       (300, 1600, 4800, 4, 128)])
def test_prepared_planes_give_the_same_results(n, d_in, d_out, q, g):
    # B is frozen: the planes regrouped once must give, bit for bit, what the per-call regrouping gives
    _, X, dY, bits, alpha, _, _ = make_case(n, n, d_in, d_out, q, g)
    Xd, dYd, bd, ad = _upload(X, dY, bits, alpha)
    pf = bcq.prepare_planes(bcq.OP_FWD, bd, d_in, g)
    px = bcq.prepare_planes(bcq.OP_BWD_X, bd, d_in, g)
    for dt in (torch.float32, torch.bfloat16):
        assert torch.equal(bcq.linear_fwd(Xd, pf, ad, d_in, g, out_dtype=dt), bcq.linear_fwd(Xd, bd, ad, d_in, g, out_dtype=dt))
        assert torch.equal(bcq.linear_bwd_x(dYd, px, ad, d_in, g, out_dtype=dt),
                           bcq.linear_bwd_x(dYd, bd, ad, d_in, g, out_dtype=dt))
    assert rel_err(bcq.linear_fwd(Xd, pf, ad, d_in, g).cpu().numpy(), oracle.fwd(X, bits, alpha, d_in, g)) <= TOL
    assert rel_err(bcq.linear_bwd_x(dYd, px, ad, d_in, g).cpu().numpy(), oracle.bwd_x(dY, bits, alpha, d_in, g)) <= TOL
    # alpha may change between calls (it is what AlphaTuning trains); the prepared planes stay valid
    ad2 = ad * 1.25
    ref2 = oracle.fwd(X, bits, (alpha * np.float32(1.25)).astype(np.float32), d_in, g)
    assert rel_err(bcq.linear_fwd(Xd, pf, ad2, d_in, g).cpu().numpy(), ref2) <= TOL


def test_prepared_planes_need_at_most_four_planes():
    assert bcq.lib().bcq_prepared_bytes(bcq.OP_FWD, 64, 256, 5, 64) == 0
    assert bcq.lib().bcq_prepared_bytes(bcq.OP_BWD_X, 64, 256, 4, 64) > 0
    assert bcq.lib().bcq_prepared_bytes(bcq.OP_DECODE, 64, 256, 4, 64) == 0


# --------------------------------------------------------------------------- tile-schedule corners

@pytest.mark.parametrize("n", [129, 145, 257, 300, 530, 1000])
def test_fwd_and_bwd_x_with_token_counts_between_tile_widths(n):
    # above 128 tokens the token-tile width is any multiple of 16 up to 256, chosen per call: these
    # counts give widths that are not powers of two, ragged last tiles and single tiles wider than n
    d_in, d_out, q, g = 640, 2560, 4, 128
    _, X, dY, bits, alpha, _, _ = make_case(900 + n, n, d_in, d_out, q, g)
    Xd, dYd, bd, ad = _upload(X, dY, bits, alpha)
    ref_y = oracle.fwd(X, bits, alpha, d_in, g)
    ref_dx = oracle.bwd_x(dY, bits, alpha, d_in, g)
    for dt, tol in ((torch.float32, TOL), (torch.bfloat16, TOL + 2.0 ** -8)):
        assert rel_err(bcq.linear_fwd(Xd, bd, ad, d_in, g, out_dtype=dt).float().cpu().numpy(), ref_y) <= tol
        assert rel_err(bcq.linear_bwd_x(dYd, bd, ad, d_in, g, out_dtype=dt).float().cpu().numpy(), ref_dx) <= tol


@pytest.mark.parametrize("n", [1, 17, 31, 32])
def test_fwd_and_bwd_x_with_few_tokens(n):
    # the prefill entry points accept any n >= 1; n <= 32 takes the narrowest token tile
    d_in, d_out, q, g = 640, 384, 3, 128
    _, X, dY, bits, alpha, _, _ = make_case(700 + n, n, d_in, d_out, q, g)
    Xd, dYd, bd, ad = _upload(X, dY, bits, alpha)
    ref_y = oracle.fwd(X, bits, alpha, d_in, g)
    ref_dx = oracle.bwd_x(dY, bits, alpha, d_in, g)
    for dt, tol in ((torch.float32, TOL), (torch.bfloat16, TOL + 2.0 ** -8)):
        assert rel_err(bcq.linear_fwd(Xd, bd, ad, d_in, g, out_dtype=dt).float().cpu().numpy(), ref_y) <= tol
        assert rel_err(bcq.linear_bwd_x(dYd, bd, ad, d_in, g, out_dtype=dt).float().cpu().numpy(), ref_dx) <= tol


@pytest.mark.parametrize("d_in", [64, 128, 192])
def test_many_tiles_per_cta_with_short_k(d_in):
    # 320 output tiles of 128 x 256 on 148 SMs: every persistent CTA walks three tiles, so both
    # accumulators are reused (second phase of their barriers) and, with K this short, the worker
    # warps are far ahead of the tensor core when they reach the last tile's epilogue
    n, d_out, q, g = 4096, 2560, 3, 64
    _, X, dY, bits, alpha, _, _ = make_case(800 + d_in, n, d_in, d_out, q, g)
    Xd, _, bd, ad = _upload(X, dY, bits, alpha)
    ref = oracle.fwd(X, bits, alpha, d_in, g)
    Yb = bcq.linear_fwd(Xd, bd, ad, d_in, g, out_dtype=torch.bfloat16)
    Yb2 = bcq.linear_fwd(Xd, bd, ad, d_in, g, out_dtype=torch.bfloat16)
    assert torch.equal(Yb, Yb2)
    assert rel_err(Yb.float().cpu().numpy(), ref) <= TOL + 2.0 ** -8
    assert rel_err(bcq.linear_fwd(Xd, bd, ad, d_in, g).cpu().numpy(), ref) <= TOL


@pytest.mark.parametrize("n,d_in,d_out,q,g", [(40, 8192, 200, 2, 128), (64, 2112, 264, 4, 64), (17, 1056, 1032, 5, 96),
                                              (5100, 15400, 1000, 3, 15400)])
def test_tiles_cut_along_k(n, d_in, d_out, q, g):
    # Few tiles: every tile in several pieces, one per CTA pair (last pieces shorter).  The last case has 80
    # tiles for 74 pairs: pieces of six tiles first, then a whole tile per pair.  Against a dense fp64
    # product with the dequantized weights (dequantize has its own test against the oracle).
    gen = torch.Generator(device="cuda").manual_seed(n)
    W = torch.randn((d_out, d_in), generator=gen, device="cuda") * 0.02
    bits, alpha, _ = bcq.quantize(W, q, g)
    X = torch.randn((n, d_in), generator=gen, device="cuda").bfloat16()
    bias = torch.randn(d_out, generator=gen, device="cuda")
    ref = (X.double() @ bcq.dequantize(bits, alpha, d_in, g).double().t()).cpu().numpy()
    for dt, tol in ((torch.float32, TOL), (torch.bfloat16, TOL + 2.0 ** -8)):
        Y = bcq.linear_fwd(X, bits, alpha, d_in, g, bias=bias, out_dtype=dt)
        assert torch.equal(Y, bcq.linear_fwd(X, bits, alpha, d_in, g, bias=bias, out_dtype=dt)), "two runs differ"
        assert rel_err(Y.float().cpu().numpy(), ref + bias.double().cpu().numpy()) <= tol
    # the same contraction as an input gradient: the transposed matrix
    bits, alpha, _ = bcq.quantize(W.t().contiguous(), q, 32 if d_out % 32 == 0 else d_out)
    gt = 32 if d_out % 32 == 0 else d_out
    ref = (X.double() @ bcq.dequantize(bits, alpha, d_out, gt).double()).cpu().numpy()
    for dt, tol in ((torch.float32, TOL), (torch.bfloat16, TOL + 2.0 ** -8)):
        dX = bcq.linear_bwd_x(X, bits, alpha, d_out, gt, out_dtype=dt)
        assert torch.equal(dX, bcq.linear_bwd_x(X, bits, alpha, d_out, gt, out_dtype=dt)), "two runs differ"
        assert rel_err(dX.float().cpu().numpy(), ref) <= tol


@pytest.mark.parametrize("k", [8200, 16384, 16392, 24576, 24584, 32760])
def test_pre_pass_of_long_rows(k):
    # rows that a lane holds in eight vectors, in twelve, and those that are read again; each token's largest element
    # in another part of its row.  Against a dense fp64 product, as the forward and as the input gradient.
    n, m, q = 6, 40, 2
    gen = torch.Generator(device="cuda").manual_seed(k)
    W = torch.randn((m, k), generator=gen, device="cuda") * 0.02
    X = torch.randn((n, k), generator=gen, device="cuda").bfloat16()
    for t in range(n):
        X[t, (t + 1) * k // n - 1] = 300.0 * (t + 1)
    bits, alpha, _ = bcq.quantize(W, q, k)
    ref = (X.double() @ bcq.dequantize(bits, alpha, k, k).double().t()).cpu().numpy()
    assert rel_err(bcq.linear_fwd(X, bits, alpha, k, k).cpu().numpy(), ref) <= TOL
    bits, alpha, _ = bcq.quantize(W.t().contiguous(), q, m)
    ref = (X.double() @ bcq.dequantize(bits, alpha, m, m).double()).cpu().numpy()
    assert rel_err(bcq.linear_bwd_x(X, bits, alpha, m, m).cpu().numpy(), ref) <= TOL


@pytest.mark.parametrize("shift", [1, 2, 3])
@pytest.mark.parametrize("d_in,d_out,q,g", [(4096, 600, 3, 32), (96, 24, 2, 96)])
def test_scales_at_any_address(d_in, d_out, q, g, shift):
    # a linear's scales may be a view of a flat array, four bytes aligned: same results as from an allocation of their own
    gen = torch.Generator(device="cuda").manual_seed(d_in + shift)
    bits, alpha, _ = bcq.quantize(torch.randn((d_out, d_in), generator=gen, device="cuda") * 0.02, q, g)
    alpha[q - 1, d_out - 1, -1] = 3.0  # the largest, and it decides the scaling, is the last
    flat = torch.empty(alpha.numel() + 4, device="cuda")
    view = flat[shift:shift + alpha.numel()].view_as(alpha).copy_(alpha)
    X = torch.randn((64, d_in), generator=gen, device="cuda").bfloat16()
    dY = torch.randn((64, d_out), generator=gen, device="cuda").bfloat16()
    assert torch.equal(bcq.linear_fwd(X, bits, view, d_in, g), bcq.linear_fwd(X, bits, alpha, d_in, g))
    assert torch.equal(bcq.linear_bwd_x(dY, bits, view, d_in, g), bcq.linear_bwd_x(dY, bits, alpha, d_in, g))
    assert torch.equal(bcq.linear_decode(X[:3], bits, view, d_in, g), bcq.linear_decode(X[:3], bits, alpha, d_in, g))
    ref = (X.double() @ bcq.dequantize(bits, alpha, d_in, g).double().t()).cpu().numpy()
    assert rel_err(bcq.linear_fwd(X, bits, view, d_in, g).cpu().numpy(), ref) <= TOL


def test_bwd_x_many_tiles_per_cta_with_short_k():
    n, d_in, d_out, q, g = 4096, 2560, 64, 4, 128
    _, X, dY, bits, alpha, _, _ = make_case(811, n, d_in, d_out, q, g)
    _, dYd, bd, ad = _upload(X, dY, bits, alpha)
    ref = oracle.bwd_x(dY, bits, alpha, d_in, g)
    assert rel_err(bcq.linear_bwd_x(dYd, bd, ad, d_in, g, out_dtype=torch.bfloat16).float().cpu().numpy(),
                   ref) <= TOL + 2.0 ** -8
    assert rel_err(bcq.linear_bwd_x(dYd, bd, ad, d_in, g).cpu().numpy(), ref) <= TOL


@pytest.mark.parametrize("k", [256, 257, 320, 384])
def test_many_tiles_per_cta_around_the_shortest_shared_output(k):
    # 4 and 5 stages a tile lie on either side of the line above which the worker warps share the output of a
    # CTA's last tile; 160 tiles for 74 pairs, so accumulators are reused.  Against a dense fp64 product.
    n, m = 4096, 2560
    gen = torch.Generator(device="cuda").manual_seed(k)
    X = torch.randn((n, (k + 7) // 8 * 8), generator=gen, device="cuda").bfloat16()[:, :k]
    W = torch.randn((m, k), generator=gen, device="cuda") * 0.02
    bits, alpha, _ = bcq.quantize(W, 3, k)
    ref = X.double() @ bcq.dequantize(bits, alpha, k, k).double().t()
    bits_t, alpha_t, _ = bcq.quantize(W.t().contiguous(), 3, 128)
    ref_t = X.double() @ bcq.dequantize(bits_t, alpha_t, m, 128).double()
    for dt, tol in ((torch.float32, TOL), (torch.bfloat16, TOL + 2.0 ** -8)):
        for _ in range(3):
            Y = bcq.linear_fwd(X, bits, alpha, k, k, out_dtype=dt)
            assert float((Y.double() - ref).abs().max() / ref.abs().max()) <= tol
            dX = bcq.linear_bwd_x(X, bits_t, alpha_t, m, 128, out_dtype=dt)
            assert float((dX.double() - ref_t).abs().max() / ref_t.abs().max()) <= tol


# --------------------------------------------------------------------------- dynamic range

def _bf16(x):
    return synth.f32_to_bf16_bits(np.asarray(x, dtype=np.float32))


def test_token_with_one_huge_channel():
    # one channel of one token is 1e4 among N(0,1): the per-token power-of-two scale has to keep
    # both the outlier and the ordinary channels inside the fp16 operands' range
    n, d_in, d_out, q, g = 96, 512, 256, 3, 128
    _, X, dY, bits, alpha, _, _ = make_case(900, n, d_in, d_out, q, g)
    Xf = synth.bf16_bits_to_f32(X)
    Xf[5, 77] = 1.0e4
    Xf[40, 300] = -3.0e4
    X = _bf16(Xf)
    Xd, _, bd, ad = _upload(X, dY, bits, alpha)
    ref = oracle.fwd(X, bits, alpha, d_in, g)
    Y = bcq.linear_fwd(Xd, bd, ad, d_in, g).cpu().numpy()
    assert np.isfinite(Y).all()
    # per token, since the two outlier tokens dwarf the others
    for t in (0, 5, 40, 95):
        assert np.abs(Y[t] - ref[t]).max() <= TOL * np.abs(ref[t]).max()
    pack = bcq.decode_pack(bd, ad, d_in, g)
    for nn in (1, 16):
        refd = ref[:nn * 6:6]
        Xs = Xd[:nn * 6:6].contiguous()
        for Yd in (bcq.linear_decode(Xs, bd, ad, d_in, g).cpu().numpy(),
                   bcq.linear_decode_packed(Xs, pack, d_out, d_in, q, g).cpu().numpy()):
            for t in range(nn):
                assert np.abs(Yd[t] - refd[t]).max() <= TOL * np.abs(refd[t]).max()


def test_tiny_output_gradients():
    # dY ~ 1e-6: far below the smallest normal fp16 number unless each token row is rescaled
    n, d_in, d_out, q, g = 200, 384, 256, 4, 128
    _, X, dY, bits, alpha, _, _ = make_case(901, n, d_in, d_out, q, g)
    dY = _bf16(synth.bf16_bits_to_f32(dY) * np.float32(1e-6))
    Xd, dYd, bd, ad = _upload(X, dY, bits, alpha)
    ref = oracle.bwd_x(dY, bits, alpha, d_in, g)
    assert rel_err(bcq.linear_bwd_x(dYd, bd, ad, d_in, g).cpu().numpy(), ref) <= TOL
    ref = oracle.bwd_alpha(dY, X, bits, d_in, g)
    assert rel_err(bcq.linear_bwd_alpha(dYd, Xd, bd, d_in, g).cpu().numpy(), ref) <= TOL


def test_scales_spread_over_4096x_between_rows_and_groups():
    # alpha differs by 2^12 between rows and, inside a row, between groups (also: the first groups
    # of a row are ~1e-6 of the later ones, and the other way round)
    n, d_in, d_out, q, g = 80, 1024, 256, 3, 128
    W = synth.weights(d_out, d_in, (100, 902, 0))
    row_mul = np.float32(2.0) ** -(np.arange(d_out) % 13).astype(np.float32)
    W = W * row_mul[:, None]
    W[64:128, :512] *= np.float32(1e-6)     # tiny first four groups
    W[128:192, 512:] *= np.float32(1e-6)    # tiny last four groups
    W[192:, 256:384] *= np.float32(4096.0)  # one large group in the middle
    X = synth.activations(n, d_in, (100, 902, 0), synth.ROLE_X)
    dY = synth.activations(n, d_out, (100, 902, 0), synth.ROLE_DY)
    bits, alpha, _, _ = oracle.quantize(W.astype(np.float32), q, g)
    Xd, dYd, bd, ad = _upload(X, dY, bits, alpha)
    ref = oracle.fwd(X, bits, alpha, d_in, g)
    # decode, column by column: every weight row has its own magnitude and its own scale
    pack = bcq.decode_pack(bd, ad, d_in, g)
    for nn in (1, 4, 16):
        Xs = Xd[:nn].contiguous()
        for Yd in (bcq.linear_decode(Xs, bd, ad, d_in, g).cpu().numpy(),
                   bcq.linear_decode_packed(Xs, pack, d_out, d_in, q, g).cpu().numpy()):
            assert np.isfinite(Yd).all()
            e = np.abs(Yd - ref[:nn]).max(axis=0) / np.abs(ref).max(axis=0)
            assert e.max() <= TOL
    # the prefill kernels scale all weights by one power of two: rows 2^12 below the largest keep
    # the absolute accuracy of the largest, which the per-tensor metric is about
    assert rel_err(bcq.linear_fwd(Xd, bd, ad, d_in, g).cpu().numpy(), ref) <= TOL
    assert rel_err(bcq.linear_bwd_x(dYd, bd, ad, d_in, g).cpu().numpy(),
                   oracle.bwd_x(dY, bits, alpha, d_in, g)) <= TOL


@pytest.mark.parametrize("n", [1, 2, 4, 7, 16])
@pytest.mark.parametrize("d_in,d_out,q,g", [
    (4096, 1536, 3, 128), (1024, 520, 4, 128), (2048, 256, 3, 2048), (1000, 200, 4, 1000),
    (1600, 336, 4, 128), (320, 384, 2, 96), (256, 128, 1, 32), (2304, 4100, 2, 64),
])
def test_decode_packed_matches_oracle(n, d_in, d_out, q, g):
    _, X, dY, bits, alpha, _, _ = make_case(n + d_out + q, n, d_in, d_out, q, g)
    Xd, _, bd, ad = _upload(X, dY, bits, alpha)
    ref = oracle.fwd(X, bits, alpha, d_in, g)
    pack = bcq.decode_pack(bd, ad, d_in, g)
    Y = bcq.linear_decode_packed(Xd, pack, d_out, d_in, q, g)
    Y2 = bcq.linear_decode_packed(Xd, pack, d_out, d_in, q, g)
    torch.cuda.synchronize()
    assert torch.equal(Y, Y2)
    assert rel_err(Y.cpu().numpy(), ref) <= TOL
    bias = synth.bias(d_out, (100, n, 1))
    Yb = bcq.linear_decode_packed(Xd, pack, d_out, d_in, q, g, bias=torch.from_numpy(bias).cuda(),
                                  out_dtype=torch.bfloat16)
    assert rel_err(Yb.float().cpu().numpy(), ref + bias.astype(np.float64)) <= TOL + 2.0 ** -8


@pytest.mark.parametrize("n,d_in,d_out,q,g", [
    (1, 136, 24, 1, 136), (9, 1000, 40, 2, 1000), (8, 672, 72, 4, 96), (16, 320, 17, 3, 32), (3, 2600, 264, 5, 64),
    (11, 520, 136, 8, 520), (2, 128, 30008, 4, 128), (12, 256, 30000, 3, 64), (16, 16392, 40, 4, 16392),
])
def test_decode_from_planes_and_packs(n, d_in, d_out, q, g):
    # both decode kernels at the edges of their units (16 rows x 128 columns, 8 tokens): ragged rows and
    # columns, groups inside a unit, q > 4, and more row tiles per CTA than its sums have room for.
    # Against a dense fp64 product with the dequantized weights.
    gen = torch.Generator(device="cuda").manual_seed(n * 1000 + d_out)
    W = torch.randn((d_out, d_in), generator=gen, device="cuda") * 0.02
    bits, alpha, _ = bcq.quantize(W, q, g)
    X = torch.randn((n, d_in), generator=gen, device="cuda").bfloat16()
    bias = torch.randn(d_out, generator=gen, device="cuda")
    ref = (X.double() @ bcq.dequantize(bits, alpha, d_in, g).double().t() + bias.double()).cpu().numpy()
    calls = [lambda dt: bcq.linear_decode(X, bits, alpha, d_in, g, bias=bias, out_dtype=dt)]
    if q <= 4:
        pack = bcq.decode_pack(bits, alpha, d_in, g)
        calls.append(lambda dt: bcq.linear_decode_packed(X, pack, d_out, d_in, q, g, bias=bias, out_dtype=dt))
    for call in calls:
        for dt, tol in ((torch.float32, TOL), (torch.bfloat16, TOL + 2.0 ** -8)):
            Y = call(dt)
            assert torch.equal(Y, call(dt)), "two runs differ"
            assert rel_err(Y.float().cpu().numpy(), ref) <= tol


@pytest.mark.parametrize("d_in,d_out,q,g,n", [(1024, 264, 4, 128, 1), (4096, 1000, 3, 64, 3), (512, 2400, 2, 512, 16)])
def test_decode_right_after_packing_into_a_used_buffer(d_in, d_out, q, g, n):
    # the decode kernel may start while the kernels that write its pack are still running: two matrices are
    # packed in turn into one buffer, each decoded at once, and must give what they give from packs of
    # their own
    lib = bcq.lib()
    gen = torch.Generator(device="cuda").manual_seed(d_in)
    X = torch.randn((n, d_in), generator=gen, device="cuda").bfloat16()
    mats, ref = [], []
    for _ in range(2):
        bits, alpha, _ = bcq.quantize(torch.randn((d_out, d_in), generator=gen, device="cuda") * 0.02, q, g)
        mats.append((bits, alpha))
        own = bcq.decode_pack(bits, alpha, d_in, g)
        torch.cuda.synchronize()
        ref.append(bcq.linear_decode_packed(X, own, d_out, d_in, q, g))
    pack = torch.empty(lib.bcq_decode_pack_bytes(d_out, d_in, q, g), dtype=torch.uint8, device="cuda")
    outs = [torch.empty((n, d_out), device="cuda") for _ in range(60)]
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream().cuda_stream
    for i, out in enumerate(outs):
        bits, alpha = mats[i % 2]
        assert lib.bcq_decode_pack(d_out, d_in, q, g, bits.data_ptr(), alpha.data_ptr(), pack.data_ptr(), pack.numel(),
                                   stream) == 0
        bcq.linear_decode_packed(X, pack, d_out, d_in, q, g, out=out)
    for i, out in enumerate(outs):
        assert torch.equal(out, ref[i % 2]), i


@pytest.mark.parametrize("d_in,d_out,q,g", [(100, 40, 2, 100), (2048, 300, 4, 128), (2056, 300, 4, 128), (4104, 2400, 3, 64),
                                            (16384, 512, 4, 128), (16400, 33, 1, 16400), (128, 60000, 1, 64), (2080, 500, 3, 32),
                                            (4096, 512, 4, 128), (6144, 500, 3, 64)])
def test_decode_of_few_tokens_is_decode_of_many(d_in, d_out, q, g):
    # up to two tokens (four, with more than 16 steps of 128 to a CTA) the activations go by way of shared memory, once for the
    # CTA: the same conversion and the same sums, so to the last bit what the first rows of a larger batch get
    # (ragged steps, clusters, several rounds of tiles, tables of two and four groups a step)
    gen = torch.Generator(device="cuda").manual_seed(d_in + d_out)
    bits, alpha, _ = bcq.quantize(torch.randn((d_out, d_in), generator=gen, device="cuda") * 0.02, q, g)
    pack = bcq.decode_pack(bits, alpha, d_in, g)
    X = torch.randn((8, (d_in + 7) // 8 * 8), generator=gen, device="cuda").bfloat16()[:, :d_in]
    X[1] *= 1e-3
    Y = bcq.linear_decode_packed(X, pack, d_out, d_in, q, g)
    ref = (X.double() @ bcq.dequantize(bits, alpha, d_in, g).double().t()).cpu().numpy()
    assert rel_err(Y.cpu().numpy(), ref) <= TOL
    for n in (1, 2, 3, 4, 5):
        assert torch.equal(bcq.linear_decode_packed(X[:n], pack, d_out, d_in, q, g), Y[:n]), n


@pytest.mark.parametrize("d_in,d_out,q,g", [(128, 300, 3, 128), (768, 760, 3, 768), (1608, 4790, 2, 64), (6400, 1600, 1, 6400),
                                            (4096, 512, 3, 64), (3200, 1600, 4, 128), (1408, 6390, 4, 1408), (1280, 4096, 4, 32),
                                            (4480, 1000, 4, 128), (128, 60000, 2, 64), (128, 60000, 4, 64)])
def test_decode_from_planes_two_units_ahead(d_in, d_out, q, g):
    # few units of 16 rows x 128 columns to a warp (none to four; one, two or four CTAs to a tile; two rounds of tiles): with up to
    # three planes and eight tokens the weights are taken two units ahead, else one, with the same sums where a CTA's tiles
    # fit one round.
    # Against a dense fp64 product.
    gen = torch.Generator(device="cuda").manual_seed(d_in + d_out)
    bits, alpha, _ = bcq.quantize(torch.randn((d_out, d_in), generator=gen, device="cuda") * 0.02, q, g)
    X = torch.randn((16, d_in), generator=gen, device="cuda").bfloat16()
    ref = (X.double() @ bcq.dequantize(bits, alpha, d_in, g).double().t()).cpu().numpy()
    Y = bcq.linear_decode(X, bits, alpha, d_in, g)
    assert rel_err(Y.cpu().numpy(), ref) <= TOL
    for n in (1, 8):
        few = bcq.linear_decode(X[:n], bits, alpha, d_in, g)
        assert rel_err(few.cpu().numpy(), ref[:n]) <= TOL
        if d_out < 20000:
            assert torch.equal(few, Y[:n]), n


@pytest.mark.parametrize("n", [1, 9])
@pytest.mark.parametrize("d_in,d_out,q,g", [(4096, 1040, 4, 128), (4224, 1030, 3, 96), (8200, 512, 2, 8200),
                                            (16384, 250, 4, 64), (8192, 16, 6, 128), (4100, 17, 1, 4100)])
def test_decode_of_few_rows_by_clusters(n, d_in, d_out, q, g):
    # few row tiles and a long row: 2, 4 or 8 CTAs share a tile's steps, evenly or not (4224: 33 steps, 8200: 65);
    # 4096 and 1040 rows lie on the lines of the rule.  Against a dense fp64 product.
    gen = torch.Generator(device="cuda").manual_seed(d_in + d_out)
    W = torch.randn((d_out, d_in), generator=gen, device="cuda") * 0.02
    bits, alpha, _ = bcq.quantize(W, q, g)
    X = torch.randn((n, (d_in + 7) // 8 * 8), generator=gen, device="cuda").bfloat16()[:, :d_in]
    bias = torch.randn(d_out, generator=gen, device="cuda")
    ref = (X.double() @ bcq.dequantize(bits, alpha, d_in, g).double().t() + bias.double()).cpu().numpy()
    outs = [[bcq.linear_decode(X, bits, alpha, d_in, g, bias=bias) for _ in range(3)]]
    if q <= 4:
        pack = bcq.decode_pack(bits, alpha, d_in, g)
        outs.append([bcq.linear_decode_packed(X, pack, d_out, d_in, q, g, bias=bias) for _ in range(3)])
    for ys in outs:
        assert torch.equal(ys[0], ys[1]) and torch.equal(ys[0], ys[2]), "runs differ"
        assert rel_err(ys[0].cpu().numpy(), ref) <= TOL


def test_decode_pack_rejects_more_than_four_planes():
    assert bcq.lib().bcq_decode_pack_bytes(64, 256, 5, 64) == 0
    assert bcq.lib().bcq_decode_pack_bytes(64, 256, 4, 64) > 0


def test_strided_activations_and_outputs():
    n, d_in, d_out, q, g = 70, 256, 192, 3, 128
    _, X, dY, bits, alpha, _, _ = make_case(3, n, d_in, d_out, q, g)
    Xd, dYd, bd, ad = _upload(X, dY, bits, alpha)
    Xp = torch.zeros((n, d_in + 8), dtype=torch.bfloat16, device="cuda")
    Xp[:, :d_in] = Xd
    Yp = torch.full((n, d_out + 5), -7.0, dtype=torch.float32, device="cuda")
    bcq.linear_fwd(Xp[:, :d_in], bd, ad, d_in, g, out=Yp[:, :d_out])
    ref = oracle.fwd(X, bits, alpha, d_in, g)
    assert rel_err(Yp[:, :d_out].cpu().numpy(), ref) <= TOL
    assert (Yp[:, d_out:] == -7.0).all()       # nothing written past the row


def test_quantize_then_layer_end_to_end():
    # the whole path on device: W -> (bits, alpha) -> fwd, dX, dalpha, all against the oracle
    n, d_in, d_out, q, g = 256, 512, 384, 3, 128
    W, X, dY, bits_ref, alpha_ref, _, _ = make_case(11, n, d_in, d_out, q, g)
    bits, alpha, _ = bcq.quantize(torch.from_numpy(W).cuda(), q, g)
    np.testing.assert_array_equal(host_bits(bits), bits_ref)
    Xd, dYd = dev_bf16(X), dev_bf16(dY)
    assert rel_err(bcq.linear_fwd(Xd, bits, alpha, d_in, g).cpu().numpy(),
                   oracle.fwd(X, bits_ref, alpha_ref, d_in, g)) <= TOL
    assert rel_err(bcq.linear_bwd_x(dYd, bits, alpha, d_in, g).cpu().numpy(),
                   oracle.bwd_x(dY, bits_ref, alpha_ref, d_in, g)) <= TOL
    assert rel_err(bcq.linear_bwd_alpha(dYd, Xd, bits, d_in, g).cpu().numpy(),
                   oracle.bwd_alpha(dY, X, bits_ref, d_in, g)) <= TOL
