"""Each CUDA kernel, through the C ABI, against the fp64 oracle on the same seeded inputs.
Sizes span several tiles plus ragged tails; tolerances are derived from bf16 storage
(unit round-off u = 2^-9) with fp32 arithmetic inside the kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle  # noqa: E402
from synth.inputs import CONFIGS, make_inputs, round_to_bf16  # noqa: E402
from gpu_common import BF16_U, bf16_dev, f32_dev, i32_dev, rand_bf16, to_np64  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rlx():
    import paper_2609_37916_b200 as pkg
    from paper_2609_37916_b200.build import build
    build()
    return pkg


def assert_close_bf16_out(got, ref, extra_abs=0.0):
    """Output stored in bf16: |err| <= 2u|ref| + small absolute slack for fp32 accumulation."""
    tol = 2 * BF16_U * np.abs(ref) + 1e-5 + extra_abs
    bad = np.abs(got - ref) > tol
    assert not bad.any(), (int(bad.sum()), float(np.abs(got - ref).max()))


# ------------------------------------------------------------------ LayerNorm / embedding / pool
@pytest.mark.parametrize("H", [128, 384, 768, 1024])
@pytest.mark.parametrize("rows", [1, 7, 1000])
def test_layernorm(rlx, H, rows):
    rng = np.random.default_rng(H + rows)
    x = rand_bf16(rng, (rows, H), 2.0) + round_to_bf16(np.float32(0.5))
    x = round_to_bf16(x)
    g = (1 + 0.1 * rng.standard_normal(H)).astype(np.float32)
    b = (0.1 * rng.standard_normal(H)).astype(np.float32)
    got = to_np64(rlx.layernorm(bf16_dev(x), f32_dev(g), f32_dev(b), 1e-12))
    ref = oracle.layernorm(x.astype(np.float64), g, b, 1e-12)
    assert_close_bf16_out(got, ref)


def test_layernorm_constant_row_gives_beta(rlx):
    H = 384
    x = np.full((3, H), 1.5, np.float32)
    b = round_to_bf16(np.linspace(-1, 1, H).astype(np.float32))
    got = to_np64(rlx.layernorm(bf16_dev(x), f32_dev(np.ones(H)), f32_dev(b), 1e-12))
    assert np.array_equal(got, np.broadcast_to(b.astype(np.float64), (3, H)))


@pytest.mark.parametrize("name", ["c0", "c1"])
def test_embed_layernorm_matches_oracle_stage(rlx, name):
    inp = make_inputs(CONFIGS[name], ln_affine_random=True)
    c = inp.cfg
    # hit both ends of the vocabulary
    inp.ids[0, 0], inp.ids[0, 1] = 0, c.vocab - 1
    _, d = oracle.encoder_forward(c, inp.ids, inp.mask, inp.params, [],
                                  compute_all_rows=True, dumps=True)
    p = inp.params
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = rlx.embed_layernorm(i32_dev(inp.ids), bf16_dev(p["word_emb"]), bf16_dev(p["pos_emb"]),
                              bf16_dev(p["type_emb"]), f32_dev(p["emb_ln_g"]), f32_dev(p["emb_ln_b"]),
                              c.seq, c.vocab, c.ln_eps, status=status)
    assert_close_bf16_out(to_np64(got).reshape(c.batch, c.seq, c.hidden), d["x_emb"])
    assert int(status.item()) == 0


def test_embed_out_of_range_id_is_clamped_and_flagged(rlx):
    inp = make_inputs(CONFIGS["c0"])
    c, p = inp.cfg, inp.params
    ids = inp.ids.copy()
    ids[0, 3] = c.vocab + 5
    ids[0, 4] = -2
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    args = (bf16_dev(p["word_emb"]), bf16_dev(p["pos_emb"]), bf16_dev(p["type_emb"]), f32_dev(p["emb_ln_g"]),
            f32_dev(p["emb_ln_b"]), c.seq, c.vocab, c.ln_eps)
    got = rlx.embed_layernorm(i32_dev(ids), *args, status=status)
    assert int(status.item()) == 1
    clamped = inp.ids.copy()
    clamped[0, 3], clamped[0, 4] = c.vocab - 1, 0
    want = rlx.embed_layernorm(i32_dev(clamped), *args)
    assert torch.equal(got, want)


@pytest.mark.parametrize("B,S,H", [(1, 16, 384), (5, 37, 384), (3, 512, 768), (2, 9, 1024), (4, 33, 128)])
def test_pool_l2norm(rlx, B, S, H):
    rng = np.random.default_rng(B * S + H)
    x = rand_bf16(rng, (B, S, H))
    mask = (rng.random((B, S)) < 0.6).astype(np.int32)
    mask[0, :] = 0
    mask[0, S // 2] = 1          # single valid token
    if B > 1:
        mask[1, :] = 0           # empty sequence -> zeros
    got = to_np64(rlx.pool_l2norm(bf16_dev(x), i32_dev(mask)))
    ref = oracle.pool_l2(x.astype(np.float64), mask)
    assert np.abs(got - ref).max() < 2e-6
    if B > 1:
        assert np.array_equal(got[1], np.zeros(H))


@pytest.mark.parametrize("B,S,holes", [(1, 16, 0.0), (7, 130, 0.0), (5, 512, 0.4), (300, 33, 0.3), (64, 128, 0.0)])
def test_pack_sequences_is_bit_exact(rlx, B, S, holes):
    rng = np.random.default_rng(B * S)
    lengths = rng.integers(0, S + 1, size=B)
    lengths[0] = S
    if B > 2:
        lengths[1], lengths[2] = 0, 1
    mask = (np.arange(S)[None, :] < lengths[:, None]).astype(np.int32)
    if holes:
        mask = (mask * (rng.random((B, S)) >= holes)).astype(np.int32)
    dmask = i32_dev(mask)
    for _ in range(2):   # the ticket counter must be left ready for a second launch
        seq_len, seq_start, pos, ticket = rlx.pack_sequences(dmask)
        torch.cuda.synchronize()
        assert int(ticket.item()) == 0
        want_len = mask.astype(bool).sum(1)
        assert np.array_equal(seq_len.cpu().numpy(), want_len)
        assert np.array_equal(seq_start.cpu().numpy(), np.concatenate([[0], np.cumsum(want_len)]))
        got = pos.cpu().numpy()
        for b in range(B):
            assert np.array_equal(got[b, :want_len[b]], np.nonzero(mask[b])[0])


# ------------------------------------------------------------------ GEMM
GEMM_SHAPES = [(128, 64, 64), (16, 1152, 384), (300, 384, 384), (257, 1536, 384), (1000, 384, 1536),
               (129, 768, 768), (4096, 192, 72), (2048, 2304, 768), (9000, 1152, 384), (40000, 384, 384)]
GEMM_IMPLS = [0, 1, 2, 3, 4]
GEMM_IMPL_IDS = ["tcgen05", "simt", "tcgen05_pair", "tcgen05_single", "tcgen05_resident"]


def _impl_applies(impl, N, K):
    if impl == 2:
        return N % 128 == 0          # CTA-pair tiles
    if impl == 4:
        return K <= 384 and (N % 128 == 0 or N % 192 == 0)   # A-resident CTA-pair kernel
    return True


@pytest.mark.parametrize("impl", GEMM_IMPLS, ids=GEMM_IMPL_IDS)
def test_gemm_small_integers_is_bit_exact(rlx, impl):
    """Operands are small integers (exact in bf16, sums exact in fp32): any layout, descriptor or
    indexing mistake shows up as a wrong integer, with no tolerance to hide behind."""
    rng = np.random.default_rng(11)
    for (M, N, K) in [(128, 64, 64), (128, 128, 128), (200, 192, 384), (384, 256, 136), (130, 384, 1536),
                      (700, 1152, 384), (5000, 1536, 320)]:
        if not _impl_applies(impl, N, K):
            continue
        a = rng.integers(-1, 2, size=(M, K)).astype(np.float32)
        w = rng.integers(-1, 2, size=(N, K)).astype(np.float32)
        bias = rng.integers(-8, 9, size=N).astype(np.float32)
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        got = to_np64(rlx.gemm_bf16(bf16_dev(a), bf16_dev(w), f32_dev(bias), impl=impl, status=status))
        ref = a.astype(np.float64) @ w.astype(np.float64).T + bias
        assert int(status.item()) == 0
        assert np.abs(ref).max() < 256  # integers below 2^8 are exact in bf16
        assert np.array_equal(got, ref), (M, N, K, np.abs(got - ref).max())


@pytest.mark.parametrize("impl", GEMM_IMPLS, ids=GEMM_IMPL_IDS)
@pytest.mark.parametrize("epi", [0, 1, 2], ids=["bias", "gelu", "residual"])
@pytest.mark.parametrize("shape", GEMM_SHAPES)
def test_gemm_matches_oracle_linear(rlx, shape, epi, impl):
    M, N, K = shape
    if not _impl_applies(impl, N, K):
        pytest.skip("tile shape of this variant does not divide the problem")
    if impl == 1 and M * N * K > 2e9:
        pytest.skip("bring-up GEMM: large case covered by the tensor-core path")
    rng = np.random.default_rng(M + N + K + epi)
    a = rand_bf16(rng, (M, K))
    w = rand_bf16(rng, (N, K), 0.05)
    bias = (0.1 * rng.standard_normal(N)).astype(np.float32)
    res = rand_bf16(rng, (M, N)) if epi == 2 else None
    got = to_np64(rlx.gemm_bf16(bf16_dev(a), bf16_dev(w), f32_dev(bias),
                                residual=bf16_dev(res) if res is not None else None, epilogue=epi, impl=impl))
    ref = oracle.linear(a.astype(np.float64), w, bias)
    if epi == 1:
        ref = oracle.gelu(ref)
    if epi == 2:
        ref = ref + res.astype(np.float64)
    # fp32 accumulation of K products of magnitude ~|a||w|: error ~ K * 2^-24 * sum|a_k w_k|
    assert_close_bf16_out(got, ref, extra_abs=K * 2.0 ** -24 * 0.2)


@pytest.mark.parametrize("M", [1, 31, 32, 33, 64, 65, 96, 97, 129, 160, 225])
@pytest.mark.parametrize("N,K", [(64, 64), (192, 384), (128, 200), (64, 1600)])   # k-blocks in pairs, an odd number of them, part of one
def test_narrow_tiles_at_the_edges_of_their_row_blocks(rlx, M, N, K):
    """One row to a whole row block in the last one; small integers, so that a row or a k-block out of place is a wrong integer."""
    rng = np.random.default_rng(M + N + K)
    a, w = rng.integers(-1, 2, size=(M, K)).astype(np.float32), rng.integers(-1, 2, size=(N, K)).astype(np.float32)
    bias = rng.integers(-8, 9, size=N).astype(np.float32)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = to_np64(rlx.gemm_bf16(bf16_dev(a), bf16_dev(w), f32_dev(bias), status=status))
    ref = a.astype(np.float64) @ w.astype(np.float64).T + bias
    assert int(status.item()) == 0 and np.abs(ref).max() < 256
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("M,N,K", [(6145, 384, 1536), (7424, 384, 1536), (9473, 384, 1600), (12544, 384, 3072), (5000, 768, 3072),
                                   (3073, 768, 1664)])
@pytest.mark.parametrize("epi", [0, 1, 2])
def test_pair_tiles_of_any_width_give_the_bits_of_single_ones(rlx, M, N, K, epi):
    """Products whose tile width is chosen on the device: one round of tiles of 192 columns, two rounds of 128, an odd number of
    k-blocks, a last row block of one row.  (64 columns: few of the rows exist, see the packed forwards.)  The order along K is the
    same in every tile."""
    rng = np.random.default_rng(M + N + K + epi)
    a, w = bf16_dev(rand_bf16(rng, (M, K))), bf16_dev(rand_bf16(rng, (N, K), 0.05))
    bias = f32_dev((0.1 * rng.standard_normal(N)).astype(np.float32))
    res = bf16_dev(rand_bf16(rng, (M, N))) if epi == 2 else None
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = rlx.gemm_bf16(a, w, bias, residual=res, epilogue=epi, status=status)
    assert int(status.item()) == 0
    assert torch.equal(got, rlx.gemm_bf16(a, w, bias, residual=res, epilogue=epi, impl=3))


@pytest.mark.parametrize("M,H,F", [(256, 384, 256), (300, 384, 1536), (5000, 384, 1536), (40000, 384, 1536), (1000, 256, 512),
                                   (37, 384, 128)])
def test_ffn_fused_matches_oracle(rlx, M, H, F):
    """out = gelu(x W1^T + b1) W2^T + b2 + x in one kernel against the oracle's linear / gelu.  The hidden
    activation is rounded to bf16 once (as the two-kernel form stores it), which the reference mirrors; what
    is left is fp32 accumulation, the bf16 store, the GELU polynomial (6e-6) and rounding flips of hidden
    values (one bf16 ulp of g times |w2| each: fp32-accumulated, polynomial-GELU hidden values land on the other
    side of a rounding boundary for a few per cent of the 1536 terms).  The sharper statement is the second
    one: the two-kernel form of the library, which has its own oracle tests, gives the same bits."""
    rng = np.random.default_rng(M + H + F)
    x = rand_bf16(rng, (M, H))
    w1 = rand_bf16(rng, (F, H), 0.05)
    w2 = rand_bf16(rng, (H, F), 0.05)
    b1 = (0.1 * rng.standard_normal(F)).astype(np.float32)
    b2 = (0.1 * rng.standard_normal(H)).astype(np.float32)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = to_np64(rlx.ffn_fused_bf16(bf16_dev(x), bf16_dev(w1), f32_dev(b1), bf16_dev(w2), f32_dev(b2), status=status))
    assert int(status.item()) == 0
    g = round_to_bf16(oracle.gelu(oracle.linear(x.astype(np.float64), w1, b1)).astype(np.float32))
    ref = oracle.linear(g.astype(np.float64), w2, b2) + x.astype(np.float64)
    assert_close_bf16_out(got, ref, extra_abs=1e-2)
    # same rounding points, same k order: the two-kernel form gives the same bits
    two = rlx.gemm_bf16(rlx.gemm_bf16(bf16_dev(x), bf16_dev(w1), f32_dev(b1), epilogue=1), bf16_dev(w2), f32_dev(b2),
                        residual=bf16_dev(x), epilogue=2)
    assert np.array_equal(to_np64(two), got)
    # the LayerNorm variant normalises the unrounded sums
    gamma = (1 + 0.1 * rng.standard_normal(H)).astype(np.float32)
    beta = (0.1 * rng.standard_normal(H)).astype(np.float32)
    got_ln = to_np64(rlx.ffn_fused_bf16(bf16_dev(x), bf16_dev(w1), f32_dev(b1), bf16_dev(w2), f32_dev(b2), f32_dev(gamma),
                                        f32_dev(beta), 1e-12, status=status))
    assert int(status.item()) == 0
    assert_close_bf16_out(got_ln, oracle.layernorm(ref, gamma, beta, 1e-12), extra_abs=1e-2)


@pytest.mark.parametrize("M,H,F", [(256, 384, 256), (300, 384, 1536), (5000, 384, 1536), (40000, 384, 1536), (1000, 256, 512),
                                   (37, 384, 128)])
def test_layer_tail_matches_oracle(rlx, M, H, F):
    """Out-projection + residual + LayerNorm + feed-forward block + residual + LayerNorm in one kernel against
    the oracle's linear / layernorm / gelu.  The reference mirrors the two bf16 roundings inside (x1 and the
    hidden activation); both LayerNorms see unrounded sums."""
    rng = np.random.default_rng(M + H + F + 1)
    ctx = rand_bf16(rng, (M, H))
    h = rand_bf16(rng, (M, H))
    wo = rand_bf16(rng, (H, H), 0.05)
    w1 = rand_bf16(rng, (F, H), 0.05)
    w2 = rand_bf16(rng, (H, F), 0.05)
    bo, b2 = [(0.1 * rng.standard_normal(H)).astype(np.float32) for _ in range(2)]
    b1 = (0.1 * rng.standard_normal(F)).astype(np.float32)
    g1, g2 = [(1 + 0.1 * rng.standard_normal(H)).astype(np.float32) for _ in range(2)]
    e1, e2 = [(0.1 * rng.standard_normal(H)).astype(np.float32) for _ in range(2)]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = to_np64(rlx.layer_tail_bf16(bf16_dev(ctx), bf16_dev(h), bf16_dev(wo), f32_dev(bo), f32_dev(g1), f32_dev(e1),
                                      bf16_dev(w1), f32_dev(b1), bf16_dev(w2), f32_dev(b2), f32_dev(g2), f32_dev(e2), 1e-12,
                                      status=status))
    assert int(status.item()) == 0
    x1 = round_to_bf16(oracle.layernorm(oracle.linear(ctx.astype(np.float64), wo, bo) + h.astype(np.float64), g1, e1,
                                        1e-12).astype(np.float32)).astype(np.float64)
    g = round_to_bf16(oracle.gelu(oracle.linear(x1, w1, b1)).astype(np.float32)).astype(np.float64)
    ref = oracle.layernorm(oracle.linear(g, w2, b2) + x1, g2, e2, 1e-12)
    # a rounding flip of an x1 value (one bf16 ulp of |x1| ~ 1) moves the result by about that ulp
    assert_close_bf16_out(got, ref, extra_abs=2e-2)
    # the library's own unfused chain: same values up to those flips
    assert np.abs(got - ref).mean() <= 2e-3


def test_ffn_fused_layernorm_rows_with_a_large_mean(rlx):
    """Rows whose mean is 200 times their spread: the row statistics are kept as deviations from a pivot, so the
    variance does not cancel.  Zero weights make the pre-LayerNorm row exactly x + b2."""
    M, H, F = 300, 384, 256
    rng = np.random.default_rng(5)
    x = round_to_bf16((100.0 + 0.5 * rng.standard_normal((M, H))).astype(np.float32))
    zeros = lambda *s: np.zeros(s, np.float32)
    gamma = (1 + 0.1 * rng.standard_normal(H)).astype(np.float32)
    beta = (0.1 * rng.standard_normal(H)).astype(np.float32)
    got = to_np64(rlx.ffn_fused_bf16(bf16_dev(x), bf16_dev(zeros(F, H)), f32_dev(zeros(F)), bf16_dev(zeros(H, F)),
                                     f32_dev(zeros(H)), f32_dev(gamma), f32_dev(beta), 1e-12))
    ref = oracle.layernorm(x.astype(np.float64), gamma, beta, 1e-12)
    assert_close_bf16_out(got, ref, extra_abs=1e-4)


@pytest.mark.parametrize("impl", [0, 1], ids=["cluster", "whole_row"])
@pytest.mark.parametrize("shape", [(128, 384, 384), (300, 384, 1536), (1000, 256, 320), (129, 512, 512),
                                   (20000, 384, 384), (19000, 384, 1536), (2200, 768, 768), (5000, 768, 3072),
                                   (700, 1024, 256), (333, 128, 128), (16, 384, 384)])
def test_gemm_residual_layernorm_fused(rlx, shape, impl):
    M, N, K = shape
    if impl == 1 and N not in (256, 384, 512):
        pytest.skip("whole-row variant: the row must fit in tensor memory")
    rng = np.random.default_rng(M + N + K)
    a = rand_bf16(rng, (M, K))
    w = rand_bf16(rng, (N, K), 0.05)
    bias = (0.1 * rng.standard_normal(N)).astype(np.float32)
    res = rand_bf16(rng, (M, N))
    g = (1 + 0.1 * rng.standard_normal(N)).astype(np.float32)
    b = (0.1 * rng.standard_normal(N)).astype(np.float32)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = to_np64(rlx.gemm_residual_layernorm_bf16(bf16_dev(a), bf16_dev(w), f32_dev(bias), bf16_dev(res), f32_dev(g),
                                                   f32_dev(b), 1e-12, impl=impl, status=status))
    assert int(status.item()) == 0
    ref = oracle.layernorm(oracle.linear(a.astype(np.float64), w, bias) + res.astype(np.float64), g, b, 1e-12)
    # the pre-LayerNorm sum stays in fp32 here (no bf16 round trip), so the plain bf16-output bound holds
    assert_close_bf16_out(got, ref, extra_abs=K * 2.0 ** -24 * 0.5)


@pytest.mark.parametrize("impl", [0, 1], ids=["cluster", "whole_row"])
def test_gemm_residual_layernorm_constant_rows_give_beta(rlx, impl):
    """Zero weights, zero bias and a constant residual row: LayerNorm of a constant row is exactly beta."""
    M, N, K = 200, 384, 384
    a = np.ones((M, K), np.float32)
    w = np.zeros((N, K), np.float32)
    res = np.full((M, N), 1.5, np.float32)
    beta = round_to_bf16(np.linspace(-1, 1, N).astype(np.float32))
    got = to_np64(rlx.gemm_residual_layernorm_bf16(bf16_dev(a), bf16_dev(w), f32_dev(np.zeros(N)), bf16_dev(res),
                                                   f32_dev(np.ones(N)), f32_dev(beta), 1e-12, impl=impl))
    assert np.array_equal(got, np.broadcast_to(beta.astype(np.float64), (M, N)))


# ------------------------------------------------------------------ attention
def _qkv_case(seed, B, S, h, d, gain=1.0, holes=0.0):
    rng = np.random.default_rng(seed)
    H = h * d
    qkv = rand_bf16(rng, (B, S, 3 * H))
    qkv[..., :H] = round_to_bf16(qkv[..., :H] * np.float32(gain))
    lengths = rng.integers(1, S + 1, size=B)
    lengths[0] = S
    if B > 1:
        lengths[1] = 1
    mask = (np.arange(S)[None, :] < lengths[:, None]).astype(np.int32)
    if holes > 0:
        mask = (mask * (rng.random((B, S)) >= holes)).astype(np.int32)
        mask[:, 0] = 1
    return qkv, mask


ATT_CASES = [(1, 16, 12, 32), (3, 128, 12, 32), (2, 129, 4, 32), (2, 1, 2, 32), (3, 200, 3, 64), (2, 512, 2, 64),
             (4, 63, 12, 32), (2, 65, 2, 64)]


@pytest.mark.parametrize("case", ATT_CASES)
@pytest.mark.parametrize("variant", ["plain", "peaky", "holes"])
def test_attention_f32_mode_within_1e4_relative(rlx, case, variant):
    B, S, h, d = case
    qkv, mask = _qkv_case(sum(case), B, S, h, d, gain=6.0 if variant == "peaky" else 1.0,
                          holes=0.3 if variant == "holes" else 0.0)
    got = to_np64(rlx.attention_f32(f32_dev(qkv), i32_dev(mask), h))
    ref = oracle.attention(qkv.astype(np.float64), mask, h, compute_all_rows=True)
    valid = mask != 0
    ref_v, got_v = ref[valid], got[valid]
    # per (sequence, head) scale-relative error and an element-wise bound
    assert np.abs(got_v - ref_v).max() <= 1e-4 * np.abs(ref_v).max()
    # element-wise: relative 1e-4 plus a floor for outputs that cancel to ~0.  fp32 logits carry an
    # absolute rounding error of ~d * 2^-24 * sum|q_c k_c| / sqrt(d), i.e. a relative error of that
    # size in every probability, hence an absolute output error of that size times max|v|.
    vmax = np.abs(qkv[..., 2 * h * d:]).max()
    assert np.all(np.abs(got_v - ref_v) <= 1e-4 * np.abs(ref_v) + 1e-5 * vmax)
    for b in range(B):
        for j in range(h):
            r = ref[b][valid[b]][:, j * d:(j + 1) * d]
            g = got[b][valid[b]][:, j * d:(j + 1) * d]
            assert np.abs(g - r).max() <= 1e-4 * np.abs(r).max()


@pytest.mark.parametrize("case", ATT_CASES)
@pytest.mark.parametrize("variant", ["plain", "peaky", "holes"])
def test_attention_bf16_mode(rlx, case, variant):
    B, S, h, d = case
    qkv, mask = _qkv_case(sum(case) + 1, B, S, h, d, gain=6.0 if variant == "peaky" else 1.0,
                          holes=0.3 if variant == "holes" else 0.0)
    got = to_np64(rlx.attention_bf16(bf16_dev(qkv), i32_dev(mask), h))
    ref = oracle.attention(qkv.astype(np.float64), mask, h, compute_all_rows=True)
    valid = mask != 0
    # probabilities are rounded to bf16 before the PV product and the result is stored in bf16:
    # |err| <= u * (max|v| + |out|) with margin 2
    vmax = np.abs(qkv[..., 2 * h * d:]).max()
    assert np.abs(got[valid] - ref[valid]).max() <= 2 * BF16_U * (vmax + np.abs(ref[valid]).max())
    assert np.all(np.isfinite(got))


PACKED_CASES = [([11], 12, 32), ([128], 2, 32), ([5, 128, 64, 1, 129, 200], 3, 32), ([512, 17, 300], 2, 64),
                ([256, 255, 257, 16, 15], 12, 32), ([130, 1, 511], 1, 64)]


@pytest.mark.parametrize("impl", [0, 1], ids=["tcgen05", "mma_sync"])
@pytest.mark.parametrize("lengths,h,d", PACKED_CASES)
@pytest.mark.parametrize("gain", [1.0, 6.0], ids=["plain", "peaky"])
def test_attention_packed_matches_oracle(rlx, lengths, h, d, gain, impl):
    """Packed rows (what the forward runs): every sequence is a dense block of valid rows.  The oracle
    sees each sequence as a batch-1 problem with an all-ones mask."""
    rng = np.random.default_rng(sum(lengths) + h + d)
    H = h * d
    total = sum(lengths)
    rows = total + 7                                  # a few rows past the last sequence
    qkv = rand_bf16(rng, (rows, 3 * H))
    qkv[:, :H] = round_to_bf16(qkv[:, :H] * np.float32(gain))
    qkv[total:] = np.float32("nan")                   # junk after the last sequence must not leak in
    start = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = to_np64(rlx.attention_packed_bf16(bf16_dev(qkv), i32_dev(start[:-1]), i32_dev(np.array(lengths)),
                                            max(lengths), h, impl=impl, status=status))
    assert int(status.item()) == 0
    vmax = np.abs(qkv[:total, 2 * H:]).max()
    for b, n in enumerate(lengths):
        seq = qkv[start[b]:start[b] + n].astype(np.float64)[None]
        ref = oracle.attention(seq, np.ones((1, n), np.int32), h)[0]
        err = np.abs(got[start[b]:start[b] + n] - ref).max()
        assert np.isfinite(err) and err <= 2 * BF16_U * (vmax + np.abs(ref).max()), (b, n, err)
    assert np.array_equal(got[total:], np.zeros((rows - total, H)))


@pytest.mark.parametrize("impl", [0, 1], ids=["tcgen05", "mma_sync"])
@pytest.mark.parametrize("trend", ["rising", "falling", "spike_last"])
def test_attention_packed_row_maximum_moves_between_key_blocks(rlx, trend, impl):
    """Logits whose level changes by far more than 2^8 from one 64-key block to the next: a running
    maximum that is only corrected when it is exceeded by a margin has to take the correction path
    (rising, spike in the last block) or live with probabilities that underflow (falling)."""
    h, d = 2, 32
    H = h * d
    lengths = [300, 512, 70]
    total = sum(lengths)
    rng = np.random.default_rng(len(trend))
    qkv = rand_bf16(rng, (total, 3 * H))
    start = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    for b, n in enumerate(lengths):
        pos = np.arange(n)
        blk = pos // 64
        level = {"rising": blk * 14.0, "falling": -blk * 14.0,
                 "spike_last": np.where(pos >= n - 3, 40.0, 0.0)}[trend]
        # q = (1, 0, ...) * sqrt(d) makes the logit equal to k's first component
        q = np.zeros((n, H), np.float32)
        q[:, 0::d] = np.sqrt(d)
        k = qkv[start[b]:start[b] + n, H:2 * H].copy()
        k[:, 0::d] = round_to_bf16((level + rng.normal(size=n)).astype(np.float32))[:, None]
        qkv[start[b]:start[b] + n, :H] = round_to_bf16(q)
        qkv[start[b]:start[b] + n, H:2 * H] = k
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = to_np64(rlx.attention_packed_bf16(bf16_dev(qkv), i32_dev(start[:-1]), i32_dev(np.array(lengths)),
                                            max(lengths), h, impl=impl, status=status))
    assert int(status.item()) == 0
    vmax = np.abs(qkv[:, 2 * H:]).max()
    for b, n in enumerate(lengths):
        seq = qkv[start[b]:start[b] + n].astype(np.float64)[None]
        ref = oracle.attention(seq, np.ones((1, n), np.int32), h)[0]
        err = np.abs(got[start[b]:start[b] + n] - ref).max()
        assert np.isfinite(err) and err <= 2 * BF16_U * (vmax + np.abs(ref).max()), (b, n, err)


def test_attention_adversarial_logits(rlx):
    """One dominant key (+30), all-equal logits, and logits so negative that exp underflows."""
    h, d, S = 1, 32, 64
    H = h * d
    for mode in ("dominant", "equal", "underflow"):
        qkv = np.zeros((1, S, 3 * H), np.float32)
        rng = np.random.default_rng(5)
        qkv[..., 2 * H:] = rand_bf16(rng, (1, S, H))
        if mode == "dominant":
            qkv[0, :, :H] = 1.0
            qkv[0, 7, H:2 * H] = round_to_bf16(np.float32(30.0 * np.sqrt(d) / d))
        elif mode == "underflow":
            qkv[0, :, :H] = 1.0
            qkv[0, :, H:2 * H] = -40.0
            qkv[0, 3, H:2 * H] = 0.0
        mask = np.ones((1, S), np.int32)
        ref = oracle.attention(qkv.astype(np.float64), mask, h)
        got32 = to_np64(rlx.attention_f32(f32_dev(qkv), i32_dev(mask), h))
        got16 = to_np64(rlx.attention_bf16(bf16_dev(qkv), i32_dev(mask), h))
        assert np.abs(got32 - ref).max() <= 1e-4 * np.abs(ref).max(), mode
        assert np.abs(got16 - ref).max() <= 4 * BF16_U * np.abs(qkv[..., 2 * H:]).max(), mode


def test_attention_all_masked_sequence_gives_zeros(rlx):
    qkv, mask = _qkv_case(3, 2, 70, 2, 32)
    mask[1, :] = 0
    got = rlx.attention_bf16(bf16_dev(qkv), i32_dev(mask), 2)
    assert torch.count_nonzero(got[1]) == 0
    got32 = rlx.attention_f32(f32_dev(qkv), i32_dev(mask), 2)
    assert torch.count_nonzero(got32[1]) == 0


# ------------------------------------------------------------------ GEMM split along K over a cluster
@pytest.mark.parametrize("M,N,K", [(m, n, k) for m in (1, 31, 33, 64, 97, 128, 129, 300)
                                   for n, k in ((64, 1536), (384, 1536), (192, 1544), (768, 3072))] +
                         [(1000, 384, 1536), (1900, 384, 1544), (897, 384, 3072), (500, 768, 1608)])
def test_gemm_split_along_k(rlx, M, N, K):
    """Few rows and a long contraction, split on request: four CTAs per tile (up to 37 tiles on 148 SMs) or two (the last
    four shapes: 48, 90, 48 and 48 tiles), at the edges of the 32-row units and of uneven k ranges, against the oracle and the one-CTA-per-tile form, twice (the order of the partial sums is
    fixed)."""
    rng = np.random.default_rng(M + N + K)
    a, w = rand_bf16(rng, (M, K)), rand_bf16(rng, (N, K), 0.05)
    bias, res = (0.1 * rng.standard_normal(N)).astype(np.float32), rand_bf16(rng, (M, N))
    for epi in (0, 1, 2):
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        args = (bf16_dev(a), bf16_dev(w), f32_dev(bias), bf16_dev(res) if epi == 2 else None, epi)
        got = rlx.gemm_bf16(*args, impl=5, status=status)
        assert torch.equal(got, rlx.gemm_bf16(*args, impl=5)) and int(status.item()) == 0
        ref = oracle.linear(a.astype(np.float64), w, bias)
        ref = oracle.gelu(ref) if epi == 1 else ref + res if epi == 2 else ref
        assert_close_bf16_out(to_np64(got), ref, extra_abs=K * 2.0 ** -24 * 0.2)
        # the same sums in another order: the fp32 accumulation error (as above, both sides) may flip one bf16 rounding,
        # which moves a value by one ulp, at most 2^-7 of it = 4u
        one = to_np64(rlx.gemm_bf16(*args, impl=3))
        assert (np.abs(to_np64(got) - one) <= 4 * BF16_U * np.abs(one) + 2 * K * 2.0 ** -24 * 0.2).all()
