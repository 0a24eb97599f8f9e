"""End-to-end parity of the CUDA encoder forward (through the C ABI) with the fp64 oracle on the
five benchmark configurations, plus stress variants, edge cases and bitwise properties."""
import dataclasses
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import cosine_rows, i32_dev, to_np64  # noqa: E402
from oracle import oracle  # noqa: E402
from synth.inputs import CONFIGS, EncoderConfig, make_inputs  # noqa: E402

pytestmark = pytest.mark.gpu

# Graded tolerance: cosine >= 0.9995 per embedding and max |err| <= 2e-2.  Honest bf16 error is
# ~100x smaller, so the tests also hold a tighter internal gate that catches subtle mistakes.
COS_MIN, ABS_MAX = 0.9995, 2e-2
COS_TIGHT, ABS_TIGHT = 0.9999, 4e-3


@pytest.fixture(scope="module")
def rlx():
    import paper_2609_37916_b200 as pkg
    from paper_2609_37916_b200.build import build
    build()
    return pkg


def run_gpu(rlx, inp, flags=0, host_io=False, weights=None, enc=None):
    c = inp.cfg
    own = enc is None
    if own:
        enc = rlx.Encoder.from_config(c, flags=flags, max_batch=c.batch, max_seq=c.seq)
    w = weights if weights is not None else rlx.upload_weights(inp.params, inp.layers)
    ws = enc.alloc_workspace(c.batch, c.seq)
    if host_io:
        out = torch.empty((c.batch, c.hidden), dtype=torch.float32).pin_memory()
        enc.forward_host(torch.from_numpy(inp.ids).pin_memory(), torch.from_numpy(inp.mask).pin_memory(), w, out, ws)
        res = out.numpy().astype(np.float64)
    else:
        out = torch.empty((c.batch, c.hidden), dtype=torch.float32, device="cuda")
        enc.forward(i32_dev(inp.ids), i32_dev(inp.mask), w, out, ws)
        torch.cuda.synchronize()
        res = to_np64(out)
    status = enc.last_device_status(ws)
    if own:
        enc.close()
    return res, status


def check(got, ref, lengths, tight=True):
    keep = np.asarray(lengths) > 0
    cos = cosine_rows(got[keep], ref[keep])
    err = np.abs(got - ref).max()
    assert np.all(np.isfinite(got))
    assert cos.min() >= COS_MIN and err <= ABS_MAX, (cos.min(), err)
    if tight:
        assert cos.min() >= COS_TIGHT and err <= ABS_TIGHT, (cos.min(), err)
    assert np.allclose(np.linalg.norm(got[keep], axis=1), 1.0, atol=1e-5)
    return float(cos.min()), float(err)


@pytest.mark.parametrize("name", ["c0", "c1", "c2"])
@pytest.mark.parametrize("mode", ["graph", "eager", "padded", "separate_ln", "separate_ln_eager", "attn_tcgen05", "cluster_ln",
                                  "fold_ln", "fold_ln_eager", "fold_ln_padded", "simt_gemm", "host_io"])
def test_full_config_matches_oracle(rlx, name, mode):
    if mode == "simt_gemm" and name == "c2":
        pytest.skip("bring-up GEMM is covered on c0/c1")
    inp = make_inputs(CONFIGS[name])
    flags = {"graph": 0, "eager": 1, "padded": 8, "separate_ln": 0x400, "separate_ln_eager": 0x401, "attn_tcgen05": 0x20, "cluster_ln": 0x80, "fold_ln": 0x200,
             "fold_ln_eager": 0x201, "fold_ln_padded": 0x208, "simt_gemm": 1 | 2, "host_io": 0}[mode]
    got, status = run_gpu(rlx, inp, flags=flags, host_io=(mode == "host_io"))
    assert status == 0
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    check(got, ref, inp.lengths)


def test_c0_matches_stored_golden(rlx):
    inp = make_inputs(CONFIGS["c0"])
    got, _ = run_gpu(rlx, inp)
    want = np.loadtxt(os.path.join(os.path.dirname(__file__), "golden", "c0_embedding.txt"), comments="#")
    check(got, want.reshape(1, -1), inp.lengths)


@pytest.mark.parametrize("flags", [0, 0x400, 0x20, 0x40, 0x80, 0x200], ids=["default", "separate_ln", "attn_tcgen05", "whole_row_ln", "cluster_ln", "fold_ln"])
@pytest.mark.parametrize("name,sample", [("c3", [0, 1, 100, 255]), ("c4", [0, 63])])
def test_large_config_sampled_sequences_match_oracle(rlx, name, sample, flags):
    """Full-size run in the benchmark's launch configuration; the oracle recomputes a sample of the
    sequences one by one (sequences are independent, so a batch-1 oracle call is the same function)."""
    inp = make_inputs(CONFIGS[name])
    got, status = run_gpu(rlx, inp, flags=flags)
    assert status == 0
    assert np.all(np.isfinite(got))
    assert np.allclose(np.linalg.norm(got, axis=1), 1.0, atol=1e-5)
    # always include the shortest and the longest sequence of the batch
    sample = sorted(set(sample) | {int(np.argmin(inp.lengths)), int(np.argmax(inp.lengths))})
    one = EncoderConfig(**{**inp.cfg.__dict__, "batch": len(sample)})
    ref = oracle.encoder_forward(one, inp.ids[sample], inp.mask[sample], inp.params, inp.layers)
    check(got[sample], ref, inp.lengths[sample])


def test_host_call_pinned_and_pageable_buffers_and_new_contents_between_calls(rlx):
    """rlx_encoder_forward_host with pinned and with pageable host buffers: both give the device call's
    bits, and a second call on the same buffers (the cached graph is replayed) reads what they hold at
    that moment."""
    a = make_inputs(CONFIGS["c1"], num_layers=2)
    c = a.cfg
    w = rlx.upload_weights(a.params, a.layers)
    enc = rlx.Encoder.from_config(c, max_batch=c.batch, max_seq=c.seq)
    ws = enc.alloc_workspace(c.batch, c.seq)
    want = torch.empty((c.batch, c.hidden), dtype=torch.float32, device="cuda")

    def device_result(ids, mask):
        enc.forward(i32_dev(ids), i32_dev(mask), w, want, ws)
        torch.cuda.synchronize()
        return want.cpu().numpy().copy()

    second_ids, second_mask = a.ids[::-1].copy(), a.mask[::-1].copy()   # the batch in reverse order
    for pinned in (True, False):
        ids = torch.from_numpy(a.ids.copy())
        mask = torch.from_numpy(a.mask.copy())
        out = torch.empty((c.batch, c.hidden), dtype=torch.float32)
        if pinned:
            ids, mask, out = ids.pin_memory(), mask.pin_memory(), out.pin_memory()
        enc.forward_host(ids, mask, w, out, ws)
        assert np.array_equal(out.numpy(), device_result(a.ids, a.mask))
        ids.copy_(torch.from_numpy(second_ids))       # same buffers, new contents: the cached graph is replayed
        mask.copy_(torch.from_numpy(second_mask))
        enc.forward_host(ids, mask, w, out, ws)
        assert np.array_equal(out.numpy(), device_result(second_ids, second_mask))
    assert enc.last_device_status(ws) == 0
    enc.close()


@pytest.mark.parametrize("flags", [0x800, 0x801], ids=["graph", "eager"])
def test_token_chunk_scheduling_is_bitwise_the_unchunked_forward(rlx, flags):
    """RLX_FLAG_CHUNKED: 200 sequences x 128 positions (25,600 padded tokens) run as two sub-batches through the
    same workspace; same kernels on fewer rows, so every bit must agree with the single-pass forward."""
    inp = make_inputs(CONFIGS["c2"], batch=200, num_layers=2)
    w = rlx.upload_weights(inp.params, inp.layers)
    whole, status = run_gpu(rlx, inp, weights=w, flags=flags & 1)
    assert status == 0
    parts, status = run_gpu(rlx, inp, weights=w, flags=flags)
    assert status == 0
    assert np.array_equal(whole, parts)
    again, status = run_gpu(rlx, inp, weights=w, flags=flags)      # a second call on a fresh encoder: same bits
    assert status == 0 and np.array_equal(again, parts)


@pytest.mark.parametrize("name", ["c3", "c4"])
def test_large_config_every_sequence_matches_oracle(rlx, name):
    """The two large configurations in the benchmark's launch configuration, EVERY sequence compared
    with the oracle (about 25 s and 100 s of oracle time on 16 host cores)."""
    oracle.set_threads(len(os.sched_getaffinity(0)))
    inp = make_inputs(CONFIGS[name])
    got, status = run_gpu(rlx, inp)
    assert status == 0
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    check(got, ref, inp.lengths)


@pytest.mark.parametrize("name", ["c0", "c1", "c2"])
def test_oracle_on_unrounded_weights_still_within_graded_tolerance(rlx, name):
    """Secondary reading of the weight precision: the oracle consumes the fp32 draws, the GPU their bf16
    roundings (the generator rounds; neither side does).  Weight quantisation then adds to the error,
    which must still clear the graded gate (cosine >= 0.9995, max |err| <= 2e-2); the tight internal
    gate belongs to the primary reading only."""
    rounded = make_inputs(CONFIGS[name])
    raw = make_inputs(CONFIGS[name], fp32_weights=True)
    assert np.array_equal(rounded.ids, raw.ids) and np.array_equal(rounded.mask, raw.mask)
    assert not np.array_equal(rounded.layers[0]["wqkv"], raw.layers[0]["wqkv"])
    got, status = run_gpu(rlx, rounded)
    assert status == 0
    ref = oracle.encoder_forward(raw.cfg, raw.ids, raw.mask, raw.params, raw.layers)
    check(got, ref, raw.lengths, tight=False)


@pytest.mark.parametrize("kw", [dict(qk_gain=8.0), dict(ln_affine_random=True), dict(mask_holes=0.3),
                                dict(qk_gain=8.0, ln_affine_random=True, mask_holes=0.2)],
                         ids=["peaky_softmax", "ln_affine", "mask_holes", "all"])
def test_stress_variants(rlx, kw):
    inp = make_inputs(CONFIGS["c1"], batch=4, seq=96, **kw)
    got, status = run_gpu(rlx, inp)
    assert status == 0
    padded, _ = run_gpu(rlx, inp, flags=8)           # padded layout: same function, other key blocking
    assert np.abs(got - padded).max() <= 2e-3
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    # a peaky softmax amplifies bf16 rounding of q and k: keep the graded gate, relax the internal one
    check(got, ref, inp.lengths, tight=("qk_gain" not in kw))


@pytest.mark.parametrize("B,S", [(1, 1), (3, 17), (2, 127), (2, 129), (1, 512), (5, 64)])
def test_odd_shapes(rlx, B, S):
    lengths = np.random.default_rng(B * 1000 + S).integers(1, S + 1, size=B)
    lengths[0] = S
    inp = make_inputs(CONFIGS["c1"], batch=B, seq=S, num_layers=2, lengths=lengths)
    got, status = run_gpu(rlx, inp)
    assert status == 0
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    check(got, ref, inp.lengths)


@pytest.mark.parametrize("seed", range(12))
def test_random_small_problems_match_oracle(rlx, seed):
    """Randomised sweep over batch, sequence length, valid lengths (incl. 0 and full), holes, LayerNorm
    affine parameters and layer count, each compared with the oracle and between the execution modes."""
    rng = np.random.default_rng(1000 + seed)
    B = int(rng.integers(1, 9))
    S = int(rng.choice([1, 2, 15, 16, 17, 31, 33, 63, 64, 65, 100, 128, 130, 200, 255, 256]))
    L = int(rng.integers(1, 4))
    lengths = rng.integers(0, S + 1, size=B)
    lengths[rng.integers(0, B)] = S
    inp = make_inputs(CONFIGS["c1"], batch=B, seq=S, num_layers=L, lengths=lengths,
                      ln_affine_random=bool(seed % 2), mask_holes=0.25 if seed % 3 == 0 else 0.0,
                      qk_gain=3.0 if seed % 4 == 0 else 1.0)
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    w = rlx.upload_weights(inp.params, inp.layers)
    base, status = run_gpu(rlx, inp, weights=w)
    assert status == 0
    check(base, ref, inp.lengths, tight=(seed % 4 != 0))
    assert np.array_equal(base[inp.lengths == 0], np.zeros_like(base[inp.lengths == 0]))
    for flags in (0x10, 0x100, 1, 0x400, 0x401, 0x420, 0x20, 0x80, 8, 0x408, 0x200, 0x201):   # no PDL, no prefetch, eager, tcgen05 attn, cluster LN, padded, folded LN (graph / eager)
        other, status = run_gpu(rlx, inp, weights=w, flags=flags)
        assert status == 0
        if flags in (0x10, 0x100, 1):
            assert np.array_equal(base, other), hex(flags)     # same kernels, other launch mechanics
        else:
            check(other, ref, inp.lengths, tight=(seed % 4 != 0))


@pytest.mark.parametrize("name,B,S", [("c1", 3, 191), ("c1", 21, 192), ("c1", 22, 192), ("c1", 22, 255), ("c1", 22, 256),
                                      ("c1", 45, 385), ("c4", 1, 256), ("c4", 2, 256), ("c4", 1, 257), ("c4", 64, 128),
                                      ("c4", 63, 129), ("c4", 64, 129)])
def test_attention_kernel_choice_at_its_edges(rlx, name, B, S):
    """Both sides of every line where a forward changes its attention kernel (heads of 32 and of 64), the first, a
    middle and the last sequence against the oracle; the kernel that may be asked for gives the same at that tolerance."""
    lengths = np.random.default_rng(B * 1000 + S).integers(0, S + 1, size=B)
    lengths[0], lengths[-1] = S, S - 1
    inp = make_inputs(CONFIGS[name], batch=B, seq=S, num_layers=2, lengths=lengths)
    pick = sorted({0, B // 2, B - 1})
    ref = oracle.encoder_forward(inp.cfg, inp.ids[pick], inp.mask[pick], inp.params, inp.layers)
    w = rlx.upload_weights(inp.params, inp.layers)
    for flags in (0, 0x20):
        got, status = run_gpu(rlx, inp, weights=w, flags=flags)
        assert status == 0
        check(got[pick], ref, inp.lengths[pick])


@pytest.mark.parametrize("name,B,S", [("c1", 5, 128), ("c1", 6, 128), ("c1", 7, 110), ("c1", 8, 128), ("c1", 9, 120), ("c4", 2, 128),
                                      ("c4", 3, 128), ("c4", 4, 97), ("c4", 6, 128), ("c4", 7, 128), ("c4", 8, 120)])
@pytest.mark.parametrize("full", [False, True])
def test_folded_forward_splits_its_long_contraction(rlx, name, B, S, full):
    """FFN-down of a small folded forward (residual through LayerNorm, row statistics out) on four CTAs per tile, on two, and
    on one, at the first and last row counts of each on 148 SMs, against the oracle; and twice the same bits.  With every
    position valid clusters of four (36 tiles) and of two (84 tiles) take more tiles and fewer CTAs for each."""
    lengths = np.random.default_rng(B * S).integers(1, S + 1, size=B)
    lengths[0] = lengths[-1] = S
    if full:
        lengths[:] = S
    inp = make_inputs(CONFIGS[name], batch=B, seq=S, num_layers=2, lengths=lengths)
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    w = rlx.upload_weights(inp.params, inp.layers)
    got, status = run_gpu(rlx, inp, weights=w)
    assert status == 0
    check(got, ref, inp.lengths)
    again, _ = run_gpu(rlx, inp, weights=w)
    assert np.array_equal(got, again)


@pytest.mark.parametrize("name,hidden,ffn,heads,layers", [("c1", 128, 64, 4, 3), ("c1", 384, 1536, 12, 4), ("c1", 640, 192, 10, 2), ("c4", 768, 3072, 12, 1),
                                                          ("c1", 1024, 64, 16, 3), ("c1", 128, 64, 4, 16), ("c4", 768, 3072, 12, 13)])
def test_folded_weights_by_launch(rlx, name, hidden, ffn, heads, layers):
    """The folded weights of one launch and of two and three (the first two layers', 24 matrices at a time), where a row is less than one
    pass of a warp, a pass and a part, and whole passes; on the side branch of the graph and in front of the eager launches."""
    cfg = dataclasses.replace(CONFIGS[name], hidden=hidden, ffn=ffn, num_heads=heads, num_layers=layers)
    inp = make_inputs(cfg, batch=3, seq=40, num_layers=layers, lengths=np.array([40, 1, 23]), ln_affine_random=True)
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    w = rlx.upload_weights(inp.params, inp.layers)
    got, status = run_gpu(rlx, inp, weights=w)
    assert status == 0
    check(got, ref, inp.lengths)
    eager, _ = run_gpu(rlx, inp, weights=w, flags=1)
    assert np.array_equal(got, eager)


@pytest.mark.parametrize("name,B,S,lengths", [
    ("c1", 1, 1, "full"), ("c1", 1, 128, "full"), ("c1", 1, 16, "ragged"), ("c1", 5, 33, "ragged"),
    ("c1", 12, 128, "full"), ("c1", 13, 128, "ragged"),                    # one head per CTA, two
    ("c1", 40, 3, "ragged"), ("c1", 200, 17, "one"),                       # bins that are full by their number of sequences
    ("c1", 32, 128, "ragged"), ("c1", 33, 125, "ragged"), ("c1", 36, 128, "ragged"), ("c1", 36, 128, "full"), ("c1", 40, 102, "ragged"), ("c1", 192, 32, "ragged"), ("c1", 74, 64, "full"),
    ("c1", 31, 130, "ragged"), ("c1", 41, 65, "ragged"), ("c1", 193, 32, "ragged"), ("c1", 75, 64, "full"), ("c1", 48, 128, "full"),                                            # the last sizes that take it, the first that do not
    ("c4", 1, 128, "full"), ("c4", 7, 120, "ragged"), ("c4", 9, 64, "holes"), ("c4", 64, 31, "ragged"), ("c4", 22, 128, "ragged"),
    ("c4", 45, 64, "full"), ("c4", 128, 32, "ragged"), ("c4", 23, 65, "ragged"), ("c4", 32, 128, "ragged")])
@pytest.mark.parametrize("flags", [0, 0x400])   # LayerNorm folded into the product, and a kernel of its own
def test_projection_and_attention_in_one_kernel_give_the_bits_of_two(rlx, name, B, S, lengths, flags):
    """The instrumented forward (RLX_FLAG_KERNEL_EVENTS) keeps the QKV GEMM and the attention apart.  Bins of several sequences, of
    one, of empty ones, full and nearly full; heads of 32 and of 64."""
    rng = np.random.default_rng(B * 1000 + S)
    n = {"full": np.full(B, S), "one": np.ones(B, int)}.get(lengths, rng.integers(0, S + 1, size=B))
    n[B // 2] = S
    inp = make_inputs(CONFIGS[name], batch=B, seq=S, num_layers=2, lengths=n, ln_affine_random=True, mask_holes=0.2 if lengths == "holes" else 0.0)
    w = rlx.upload_weights(inp.params, inp.layers)
    one, status = run_gpu(rlx, inp, weights=w, flags=flags)
    two, tstatus = run_gpu(rlx, inp, weights=w, flags=flags | 4)
    eager, estatus = run_gpu(rlx, inp, weights=w, flags=flags | 1)
    assert status == 0 and tstatus == 0 and estatus == 0
    assert np.array_equal(one, two) and np.array_equal(one, eager)
    pick = sorted({0, B // 2, B - 1})
    check(one[pick], oracle.encoder_forward(inp.cfg, inp.ids[pick], inp.mask[pick], inp.params, inp.layers), inp.lengths[pick])
    # from pinned host buffers: packing and embedding in one kernel up to 256 positions, apart beyond
    host, hstatus = run_gpu(rlx, inp, weights=w, flags=flags, host_io=True)
    assert hstatus == 0 and np.array_equal(host, one)


@pytest.mark.parametrize("B,S,lengths", [(1, 64, [64]), (1, 64, [0]), (2, 32, [1, 32]), (2, 32, [0, 31]), (4, 16, [16, 3, 0, 16]), (1, 33, [33]),
                                         (1, 16, [11]), (1, 65, [65]), (3, 22, [22, 1, 9])])
def test_attention_output_of_tiny_calls_gives_the_bits_of_its_own_kernel(rlx, B, S, lengths):
    """Up to 64 positions a cluster of the heads goes on to the attention output; the instrumented forward keeps every step apart."""
    inp = make_inputs(CONFIGS["c1"], batch=B, seq=S, num_layers=3, lengths=lengths, ln_affine_random=True)
    w = rlx.upload_weights(inp.params, inp.layers)
    enc = rlx.Encoder.from_config(inp.cfg, max_batch=B, max_seq=S)
    assert enc.launches_per_forward(B, S) == enc.launches_per_forward(1, 1) + (3 if B * S > 64 else 0)   # a kernel less per layer, asked before any forward
    one, status = run_gpu(rlx, inp, weights=w, enc=enc)
    apart, astatus = run_gpu(rlx, inp, weights=w, flags=4)
    eager, estatus = run_gpu(rlx, inp, weights=w, flags=1)
    assert status == 0 and astatus == 0 and estatus == 0
    assert np.array_equal(one, apart) and np.array_equal(one, eager)
    enc.close()


@pytest.mark.parametrize("name,B,S", [("c1", 1, 32), ("c1", 3, 22), ("c1", 7, 128), ("c1", 10, 200), ("c1", 50, 100), ("c1", 130, 256),
                                      ("c4", 1, 128), ("c4", 9, 64)])
def test_launches_per_forward_are_the_kernels_of_a_recorded_one(rlx, name, B, S):
    """The kernel nodes of a forward that the caller records (RLX_FLAG_NO_GRAPH: kernel by kernel into the caller's graph)."""
    from cuda.bindings import runtime as rt
    cfg = dataclasses.replace(CONFIGS[name], num_layers=13 if name == "c4" else 3)
    inp = make_inputs(cfg, batch=B, seq=S, lengths=np.full(B, S))
    w = rlx.upload_weights(inp.params, inp.layers)
    enc = rlx.Encoder.from_config(inp.cfg, max_batch=B, max_seq=S, flags=1)
    ids, mask, ws = i32_dev(inp.ids), i32_dev(inp.mask), enc.alloc_workspace(B, S)
    out = torch.empty((B, cfg.hidden), dtype=torch.float32, device="cuda")
    enc.forward(ids, mask, w, out, ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        enc.forward(ids, mask, w, out, ws)
    def ok(r):
        assert int(r[0]) == 0, r[0]
        return r[1:]
    raw = rt.cudaGraph_t(graph.raw_cuda_graph())
    n = ok(rt.cudaGraphGetNodes(raw))[1]
    nodes = ok(rt.cudaGraphGetNodes(raw, n))[0]
    kernels = sum(ok(rt.cudaGraphNodeGetType(x))[0] == rt.cudaGraphNodeType.cudaGraphNodeTypeKernel for x in nodes)
    assert kernels == enc.launches_per_forward(B, S)
    enc.close()


def test_tiny_calls_one_behind_the_other_hand_their_context_over_each_time(rlx):
    """The heads' CTAs write into each other's operand ring once its owner has read it: hundreds of calls back to back on changing
    inputs, sequences of one row to four groups of 16, every result that of the separate kernels."""
    rng = np.random.default_rng(11)
    base = make_inputs(CONFIGS["c1"], batch=2, seq=32, num_layers=3, lengths=[32, 32], ln_affine_random=True)
    w = rlx.upload_weights(base.params, base.layers)
    enc, apart = (rlx.Encoder.from_config(base.cfg, max_batch=2, max_seq=32, flags=f) for f in (0, 4))
    ws, ws_apart = enc.alloc_workspace(2, 32), apart.alloc_workspace(2, 32)
    ids, mask = torch.empty(2, 32, dtype=torch.int32, device="cuda"), torch.empty(2, 32, dtype=torch.int32, device="cuda")
    out = torch.empty((2, base.cfg.hidden), dtype=torch.float32, device="cuda")
    inputs = [(i32_dev(rng.integers(0, base.cfg.vocab, size=(2, 32))),
               i32_dev(np.arange(32)[None, :] < np.array([[1 + i % 32], [(7 * i) % 33]]))) for i in range(40)]
    want = [apart.forward(a, m, w, torch.empty_like(out), ws_apart) for a, m in inputs]
    got = []
    for i in range(400):
        ids.copy_(inputs[i % 40][0]); mask.copy_(inputs[i % 40][1])
        got.append(enc.forward(ids, mask, w, out, ws).clone())
    assert enc.last_device_status(ws) == 0 and apart.last_device_status(ws_apart) == 0
    assert all(torch.equal(g, want[i % 40]) for i, g in enumerate(got))
    enc.close(); apart.close()


@pytest.mark.parametrize("B,S,lo,hi", [(61, 203, 40, 203), (64, 128, 1, 90), (52, 128, 8, 128), (70, 128, 1, 70)])   # 192, 64, 128 and 64 columns
@pytest.mark.parametrize("flags", [0, 0x200])   # the residual in the epilogue, and normalised there
def test_packed_rows_choose_the_tile_width_and_not_the_result(rlx, B, S, lo, hi, flags):
    """The packed and the padded layout (RLX_FLAG_NO_PACK: 128 columns, 192 from the second on) hand the feed-forward down product other row counts: other
    widths, the same bits."""
    lengths = np.linspace(lo, hi, B).astype(int)
    inp = make_inputs(CONFIGS["c1"], batch=B, seq=S, num_layers=2, lengths=lengths)
    w = rlx.upload_weights(inp.params, inp.layers)
    packed, status = run_gpu(rlx, inp, weights=w, flags=flags)
    padded, pstatus = run_gpu(rlx, inp, weights=w, flags=flags | 8)
    assert status == 0 and pstatus == 0 and np.array_equal(packed, padded)
    pick = [0, B - 1]
    check(packed[pick], oracle.encoder_forward(inp.cfg, inp.ids[pick], inp.mask[pick], inp.params, inp.layers), inp.lengths[pick])


@pytest.mark.parametrize("B,S", [(33, 125), (61, 203), (96, 128), (98, 128)])
def test_calls_beyond_the_folding_line_keep_what_was_promised_for_them(rlx, B, S):
    """Beyond 4096 positions: the bits of the separate LayerNorms, in a workspace sized for them, timed by kernel in the count that
    is announced; the layer tail where RLX_FLAG_FUSED_FFN asks for it, and from 12288 positions on where the device chooses it."""
    inp = make_inputs(CONFIGS["c1"], batch=B, seq=S, num_layers=2, lengths=np.full(B, S), ln_affine_random=True)
    c = inp.cfg
    w = rlx.upload_weights(inp.params, inp.layers)
    apart, _ = run_gpu(rlx, inp, weights=w, flags=0x400)
    got, status = run_gpu(rlx, inp, weights=w)
    assert status == 0 and np.array_equal(got, apart)
    with_tail, _ = run_gpu(rlx, inp, weights=w, flags=0x1400)
    asked, _ = run_gpu(rlx, inp, weights=w, flags=0x1000)
    assert np.array_equal(asked, with_tail) and not np.array_equal(asked, got)
    chosen, _ = run_gpu(rlx, inp, weights=w, flags=0x4000)
    assert np.array_equal(chosen, with_tail if B * S >= 12288 else apart)
    plain, timed = (rlx.Encoder.from_config(c, max_batch=B, max_seq=S, flags=f) for f in (0x400, 4))
    ids, mask, ws = i32_dev(inp.ids), i32_dev(inp.mask), plain.alloc_workspace(B, S)
    out = torch.empty((B, c.hidden), dtype=torch.float32, device="cuda")
    assert np.array_equal(to_np64(timed.forward(ids, mask, w, out, ws)), got)
    assert len(timed.kernel_times(B, S)) == 3 + 7 * 2
    plain.close(); timed.close()


@pytest.mark.parametrize("heads", [2, 4])
@pytest.mark.parametrize("flags", [0, 0x200, 0x400])   # the host's choice, folded LayerNorm, none folded
def test_a_short_last_chunk_takes_the_kernels_of_the_whole_call(rlx, heads, flags):
    """4033 x 256 positions run as 63 sub-batches of 64 sequences and one of a single sequence, a size at which a call of its own
    would fold the LayerNorms, split the long contraction and take another attention kernel."""
    cfg = EncoderConfig("chunks", 1, 128, heads, 1536, 4033, 256, 1, 256, 7)
    inp = make_inputs(cfg)
    w = rlx.upload_weights(inp.params, inp.layers)
    whole, status = run_gpu(rlx, inp, flags=flags, weights=w)
    chunked, cstatus = run_gpu(rlx, inp, flags=flags | 0x800, weights=w)
    assert status == 0 and cstatus == 0
    bad = np.flatnonzero((whole != chunked).any(1))
    assert bad.size == 0, bad


@pytest.mark.parametrize("seed", range(4))
def test_last_layernorm_of_rows_with_a_large_mean(rlx, seed):
    """Rows in front of the last LayerNorm with a mean of 256 deviations: the LayerNorm folded into the pooling keeps its
    fp32 precision.  The layer is set up so that those rows are b2 alone (w2 = 0, ln1 = 0), numbers that bf16 holds exactly.

    Bound: z a and the sum of b are of the size of the mean, 258 deviations, and are rounded to fp32 at most four times in all;
    the embedding is that over the length of the unscaled row, at least sqrt(H)."""
    rng = np.random.default_rng(seed)
    inp = make_inputs(CONFIGS["c1"], batch=3, seq=16, num_layers=1, lengths=[1, 1, 1])
    H, layer = inp.cfg.hidden, inp.layers[0]
    layer["b2"] = (256 + 2 * rng.integers(0, 2, H)).astype(np.float32)
    layer["ln2_b"] = (0.5 * rng.choice((-1.0, 1.0), H)).astype(np.float32)
    layer["ln2_g"] = np.ones(H, np.float32)
    for name in ("w2", "ln1_g", "ln1_b", "b1"):
        layer[name] = np.zeros_like(layer[name])
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    got, status = run_gpu(rlx, inp, flags=0x200)
    assert status == 0
    assert np.abs(got - ref).max() <= 4 * 258 * 2.0 ** -24 / np.sqrt(H), np.abs(got - ref).max()


def test_degenerate_lengths_zero_one_full(rlx):
    inp = make_inputs(CONFIGS["c1"], batch=3, seq=40, num_layers=2, lengths=[0, 1, 40])
    got, status = run_gpu(rlx, inp)
    assert status == 0
    assert np.array_equal(got[0], np.zeros(inp.cfg.hidden))   # no valid token -> zero embedding
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    check(got, ref, inp.lengths)


def test_all_sequences_empty_gives_zero_embeddings(rlx):
    """No valid token anywhere: zero packed rows, every kernel must cope with an empty problem."""
    inp = make_inputs(CONFIGS["c1"], batch=3, seq=33, num_layers=2, lengths=[0, 0, 0])
    for flags in (0, 8, 0x20):
        got, status = run_gpu(rlx, inp, flags=flags)
        assert status == 0
        assert np.array_equal(got, np.zeros_like(got))


def test_vocabulary_ends_and_out_of_range_ids(rlx):
    inp = make_inputs(CONFIGS["c0"])
    inp.ids[0, 0], inp.ids[0, 1] = 0, inp.cfg.vocab - 1
    got, status = run_gpu(rlx, inp)
    assert status == 0
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    check(got, ref, inp.lengths)
    bad = make_inputs(CONFIGS["c0"])
    bad.ids[0, 2] = bad.cfg.vocab + 7
    _, status = run_gpu(rlx, bad)
    assert status == 6  # RLX_ERR_TOKEN_RANGE: clamped and flagged, no fault


def test_padding_invariance_and_determinism_are_bitwise(rlx):
    inp = make_inputs(CONFIGS["c2"], batch=8)
    w = rlx.upload_weights(inp.params, inp.layers)
    a, _ = run_gpu(rlx, inp, weights=w)
    b, _ = run_gpu(rlx, inp, weights=w)
    assert np.array_equal(a, b)                        # run-to-run determinism
    e, _ = run_gpu(rlx, inp, weights=w, flags=1)
    assert np.array_equal(a, e)                        # graph replay == eager launches
    p, _ = run_gpu(rlx, inp, weights=w, flags=8)
    assert np.array_equal(a, p)                        # packed rows == padded layout (prefix masks)
    moved = make_inputs(CONFIGS["c2"], batch=8)
    pad = moved.mask == 0
    assert pad.any()
    moved.ids[pad] = (moved.ids[pad] + 12345) % moved.cfg.vocab
    c, _ = run_gpu(rlx, moved, weights=w)
    assert np.array_equal(a, c)                        # ids under mask 0 do not matter
    perm = np.random.default_rng(0).permutation(8)
    moved.ids, moved.mask = inp.ids[perm], inp.mask[perm]
    d, _ = run_gpu(rlx, moved, weights=w)
    assert np.array_equal(a[perm], d)                  # batch-permutation equivariance


def test_forward_refuses_an_encoder_bound_to_another_device(rlx):
    inp = make_inputs(CONFIGS["c0"])
    c = inp.cfg
    enc = rlx.Encoder.from_config(c, max_batch=1, max_seq=c.seq, device=torch.cuda.device_count())  # not current
    w = rlx.upload_weights(inp.params, inp.layers)
    out = torch.zeros((1, c.hidden), dtype=torch.float32, device="cuda")
    with pytest.raises(rlx.RlxError) as ei:
        enc.forward(i32_dev(inp.ids), i32_dev(inp.mask), w, out, enc.alloc_workspace(1, c.seq))
    assert ei.value.status == 1 and torch.count_nonzero(out) == 0
    enc.close()


def test_graph_cache_reuse_and_new_inputs(rlx):
    """Same encoder object, several calls: the captured graph must be replayed for the same
    pointer set and rebuilt when the buffers or the weights change."""
    inp = make_inputs(CONFIGS["c1"])
    c = inp.cfg
    enc = rlx.Encoder.from_config(c, max_batch=4, max_seq=c.seq)
    w = rlx.upload_weights(inp.params, inp.layers)
    ws = enc.alloc_workspace(1, c.seq)
    ids, mask = i32_dev(inp.ids), i32_dev(inp.mask)
    out = torch.empty((1, c.hidden), dtype=torch.float32, device="cuda")
    ref = oracle.encoder_forward(c, inp.ids, inp.mask, inp.params, inp.layers)
    for _ in range(3):
        out.zero_()
        enc.forward(ids, mask, w, out, ws)
        torch.cuda.synchronize()
        check(to_np64(out), ref, inp.lengths)
    # new contents in the same buffers: replay must read them
    ids2 = inp.ids.copy()
    ids2[0, :4] = [5, 6, 7, 8]
    ids.copy_(torch.from_numpy(ids2))
    enc.forward(ids, mask, w, out, ws)
    torch.cuda.synchronize()
    ref2 = oracle.encoder_forward(c, ids2, inp.mask, inp.params, inp.layers)
    check(to_np64(out), ref2, inp.lengths)
    # different weights -> different result, not a stale graph
    other = make_inputs(CONFIGS["c0"], batch=1, seq=c.seq, num_layers=c.num_layers, lengths=inp.lengths)
    w2 = rlx.upload_weights(other.params, other.layers)
    enc.forward(ids, mask, w2, out, ws)
    torch.cuda.synchronize()
    ref3 = oracle.encoder_forward(c, ids2, inp.mask, other.params, other.layers)
    check(to_np64(out), ref3, inp.lengths)
    enc.close()


@pytest.mark.parametrize("flags", [0x1400, 0x1401], ids=["graph", "eager"])
def test_fused_ffn_forward_against_the_two_kernel_forward(rlx, flags):
    """RLX_FLAG_FUSED_FFN: everything of a layer behind the attention in one kernel.  The products have the
    rounding points and the k order of the separate GEMMs; both LayerNorms work on unrounded sums (two bf16
    roundings fewer per layer), so the embeddings differ from the plain 7-kernel layer's by rounding noise only
    (0x400 keeps LayerNorm folding out of both)."""
    inp = make_inputs(CONFIGS["c2"])
    w = rlx.upload_weights(inp.params, inp.layers)
    plain, status = run_gpu(rlx, inp, weights=w, flags=0x400 | (flags & 1))
    assert status == 0
    fused, status = run_gpu(rlx, inp, weights=w, flags=flags)
    assert status == 0
    assert np.abs(plain - fused).max() <= 2e-3
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    check(fused, ref, inp.lengths)


def test_fused_ffn_is_chosen_from_32768_padded_tokens_on(rlx):
    """Without a flag the one-kernel layer tail takes over at batch*seq >= 32768; RLX_FLAG_NO_FUSED_FFN (0x2000)
    keeps the 7-kernel layer.  Four kernels less per layer, embeddings equal up to rounding noise."""
    inp = make_inputs(CONFIGS["c2"], batch=256, num_layers=2)
    w = rlx.upload_weights(inp.params, inp.layers)
    auto, status = run_gpu(rlx, inp, weights=w, flags=0)
    assert status == 0
    two, status = run_gpu(rlx, inp, weights=w, flags=0x2000)
    assert status == 0
    assert np.abs(auto - two).max() <= 2e-3
    ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
    check(auto, ref, inp.lengths)
    c = inp.cfg
    assert c.batch * c.seq >= 32768
    a = rlx.Encoder.from_config(c, flags=0, max_batch=c.batch, max_seq=c.seq)
    b = rlx.Encoder.from_config(c, flags=0x2000, max_batch=c.batch, max_seq=c.seq)
    assert b.kernels_per_forward(256, 128) - a.kernels_per_forward(256, 128) == 4 * c.num_layers
    assert a.kernels_per_forward(255, 128) == b.kernels_per_forward(255, 128)
    a.close(); b.close()


def test_layer_tail_forward_on_random_shapes(rlx):
    """Random batches (1..40 sequences of 1..512 positions, empty sequences, masks with holes, random LayerNorm
    affine, 1..3 layers) through the forced 3-kernel layer, graph / eager / unpacked: against the oracle, run
    twice for bit-for-bit repeatability."""
    rng = np.random.default_rng(4242)
    for _ in range(10):
        B = int(rng.integers(1, 40))
        S = int(rng.choice([1, 7, 16, 33, 64, 65, 127, 128, 200, 256, 300, 512]))
        L = int(rng.integers(1, 4))
        lengths = rng.integers(0, S + 1, size=B)
        lengths[rng.integers(0, B)] = S
        inp = make_inputs(CONFIGS["c1"], batch=B, seq=S, num_layers=L, lengths=lengths,
                          ln_affine_random=bool(rng.integers(0, 2)), mask_holes=0.2 if rng.integers(0, 3) == 0 else 0.0)
        ref = oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers)
        w = rlx.upload_weights(inp.params, inp.layers)
        for flags in (0x1400, 0x1401, 0x1408):
            enc = rlx.Encoder.from_config(inp.cfg, flags=flags, max_batch=B, max_seq=S)
            assert enc.kernels_per_forward(B, S) == (2 if flags & 8 else 3) + 3 * L
            a, status = run_gpu(rlx, inp, weights=w, enc=enc)
            b, _ = run_gpu(rlx, inp, weights=w, enc=enc)
            enc.close()
            assert status == 0 and np.array_equal(a, b), (B, S, L, hex(flags))
            check(a, ref, inp.lengths, tight=False)


def test_captured_forward_chooses_the_layer_form_on_the_device(rlx):
    """RLX_FLAG_DEVICE_CHOICE (0x4000): from 12288 padded tokens on a captured forward carries both forms of the layer
    behind an IF / ELSE graph node; the packing kernel takes the layer tail when at least 9216 rows are valid.  Same call, same
    shapes, two masks: the dense batch gives bit for bit the forced layer-tail result, the sparse one the
    separate kernels' result."""
    B, S = 100, 128
    for lengths, forced in ((np.full(B, S), 0x1400), (np.full(B, 30), 0x2400)):
        inp = make_inputs(CONFIGS["c2"], batch=B, seq=S, num_layers=2, lengths=lengths)
        w = rlx.upload_weights(inp.params, inp.layers)
        auto, status = run_gpu(rlx, inp, weights=w, flags=0x4400)
        assert status == 0
        ref_path, status = run_gpu(rlx, inp, weights=w, flags=forced)
        assert status == 0
        assert np.array_equal(auto, ref_path), int(lengths.sum())
        again, _ = run_gpu(rlx, inp, weights=w, flags=0x4400)
        assert np.array_equal(auto, again)
        check(auto, oracle.encoder_forward(inp.cfg, inp.ids, inp.mask, inp.params, inp.layers), inp.lengths)
