"""GPU parity: the CUDA library, called through its C ABI, against the CPU checker on the same seeded inputs.

Tolerances: teacher-forced logits within max-abs 1e-4 (fp32 mode) / 3e-2 (bf16 mode); greedy token ids
bit-exact wherever the checker's top-2 logit margin exceeds 0.1."""
import ctypes as C

import numpy as np
import pytest

from paper_2503_05931_b200 import workloads as wl
from tests.helpers import MARGIN, TOL, greedy_compare, oracle_reference, teacher_forced_compare

pytestmark = pytest.mark.gpu

SMALL = dict(n_layers=2, d_model=128, n_heads=2, d_ffn=256, vocab=300, d_enc=128)
MID = dict(n_layers=3, d_model=256, n_heads=4, d_ffn=512, vocab=1000, d_enc=192)


def _binding():
    from paper_2503_05931_b200 import binding
    return binding


def _run_both(w, rows=None, need_tokens=True, label=""):
    """Teacher-forced logits and argmax at every step (this comparison carries the weight: it never stops at a
    near-tie), then the free-running greedy decode up to each utterance's first near-tie.  ``need_tokens``: demand
    that the greedy comparison covered at least one token."""
    b = _binding()
    ref = oracle_reference(w, rows)
    dec = b.decoder_for_workload(w)
    try:
        worst, compared, bad = teacher_forced_compare(dec, w, ref, rows)
        assert compared > 0
        print(f"[parity] {label or w.name} {w.dtype} B={w.batch}: max |logit diff| = {worst:.3e} over {compared} rows x steps")
        assert worst < TOL[w.dtype], f"max |logit diff| {worst:.3e} above {TOL[w.dtype]}"
        assert not bad, f"argmax mismatches at margin > {MARGIN}: {bad[:5]}"
        n_tok, _ = greedy_compare(dec, w, ref, rows)
        print(f"[parity] {label or w.name} {w.dtype}: {n_tok} greedy tokens compared")
        if need_tokens:
            assert n_tok > 0, "the greedy comparison covered no token"
    finally:
        dec.close()
    return worst


def test_config1_tiny_fp32_full():
    """The 2-layer fp32 parity configuration, every logit of every step compared."""
    w = wl.make_workload("cfg1")
    worst = _run_both(w)
    print(f"cfg1 max |logit diff| = {worst:.3e}")


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_ragged_multi_tile(dtype):
    """Lengths that span several attention chunks and GEMM row tiles with ragged tails, d_enc != d_model."""
    enc_lens = [1, 63, 64, 65, 130, 257, 5, 200] + [17] * 62      # 70 rows: more than one 64-row tile
    dec_lens = [1, 2, 70, 66, 5, 33, 64, 65] + [3] * 62
    w = wl.make_custom(MID, enc_lens, dec_lens, dtype=dtype, seed=21, out_std=0.1)
    _run_both(w, rows=[0, 1, 2, 3, 4, 5, 6, 7, 8, 69])


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("shape", [((1,), (1,)), ((1,), (5,)), ((7,), (1,)), ((3, 1, 2), (2, 4, 1))])
def test_degenerate_shapes(dtype, shape):
    enc_lens, dec_lens = shape
    w = wl.make_custom(SMALL, list(enc_lens), list(dec_lens), dtype=dtype, seed=5)
    _run_both(w, need_tokens=False)         # one or two tokens in all: the first may already be a near-tie


def test_random_shapes_fp32():
    rng = np.random.default_rng(77)
    for case in range(6):
        B = int(rng.integers(1, 10))
        w = wl.make_custom(SMALL, rng.integers(1, 71, size=B), rng.integers(1, 41, size=B), dtype="fp32",
                           seed=100 + case)
        _run_both(w, need_tokens=False, label=f"random{case}")


def test_batch_composition_invariance_on_gpu():
    """An utterance's logits do not depend on its batch companions (bit-exact in fp32 mode with the same row tile)."""
    import torch
    b = _binding()
    w = wl.make_custom(SMALL, [9, 30, 4, 66], [6, 6, 6, 6], dtype="fp32", seed=8)
    outs = []
    for rows in ([0, 1, 2, 3], [2], [3, 2, 1]):
        sub = w.subset(rows)
        dec = b.decoder_for_workload(sub)
        dec.precompute_cross_kv(dec.upload_encoder(sub.enc), sub.enc_lens)
        logits = torch.zeros((sub.batch, SMALL["vocab"]), dtype=torch.float32, device="cuda:0")
        toks = torch.full((sub.batch,), 1, dtype=torch.int32, device="cuda:0")
        rec = []
        for t in range(6):
            dec.step(toks, None, logits, None)
            toks.fill_(3 + t)
            rec.append(logits[rows.index(2)].cpu().numpy().copy())
        dec.sync_status()
        dec.close()
        outs.append(np.stack(rec))
    np.testing.assert_allclose(outs[0], outs[1], atol=2e-6)
    np.testing.assert_allclose(outs[0], outs[2], atol=2e-6)


def _eos_case(dtype):
    """A seeded workload and an end-of-sequence id, found by the checker alone, such that some utterance stops
    early and every token up to each utterance's stop is fixed by the checker (top-2 margin > MARGIN)."""
    for seed in range(13, 60):
        w = wl.make_custom(SMALL, [12, 20, 7, 33, 5], [10, 10, 1, 10, 2], dtype=dtype, seed=seed, out_std=0.1)
        free = oracle_reference(w, want_logits=False)
        for u, t in ((1, 3), (0, 2), (3, 5), (2, 1), (4, 6)):
            eos = int(free["next"][u, t])
            cut = oracle_reference(w, want_logits=False, eos=eos)
            fixed = all(np.min(cut["margin"][v, :cut["lens"][v]]) > MARGIN for v in range(w.batch))
            early = cut["lens"] < w.dec_lens
            if fixed and np.any(early) and np.any(~early) and np.min(cut["lens"][early]) >= 3:
                return w, eos, cut
    raise AssertionError("no seeded case found")


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_eos_stops_an_utterance(dtype):
    """With eos enabled an utterance retires right after emitting it (the token is stored and counted) while the
    others run on.  Expectation: the CPU checker's decode with the same end-of-sequence id."""
    b = _binding()
    w, eos, cut = _eos_case(dtype)
    dec = b.decoder_for_workload(w, eos_id=eos)
    dec.precompute_cross_kv(dec.upload_encoder(w.enc), w.enc_lens)
    toks, lens = dec.greedy_decode(w.dec_lens)
    toks, lens = toks.cpu().numpy(), lens.cpu().numpy()
    dec.close()
    stopped_early = 0
    for u in range(w.batch):
        n = int(cut["lens"][u])
        assert lens[u] == n, (u, lens[u], n)
        assert np.array_equal(toks[u, :n], cut["next"][u, :n])
        assert np.all(toks[u, n:] == -1)
        if n < w.dec_lens[u]:
            assert toks[u, n - 1] == eos
            stopped_early += 1
    assert stopped_early > 0


def test_eos_ends_the_decode_early():
    """When every utterance has emitted the end-of-sequence id, the greedy loop stops issuing steps (the host follows
    the device's retired count a few steps behind) instead of replaying all max_len of them."""
    b = _binding()
    for seed in range(13, 80):
        w = wl.make_custom(SMALL, [12, 20, 7, 33, 5], [200] * 5, dtype="bf16", seed=seed, out_std=0.3)
        probe = wl.make_custom(SMALL, [12, 20, 7, 33, 5], [8] * 5, dtype="bf16", seed=seed, out_std=0.3)
        free = oracle_reference(probe, want_logits=False)
        eos = int(free["next"][0, 3])
        cut = oracle_reference(probe, want_logits=False, eos=eos)
        if np.all(cut["lens"] < 8) and all(np.min(cut["margin"][u, :cut["lens"][u]]) > MARGIN for u in range(5)):
            break
    else:
        raise AssertionError("no seeded case found")
    dec = b.decoder_for_workload(w, eos_id=eos)
    try:
        dec.precompute_cross_kv(dec.upload_encoder(w.enc), w.enc_lens)
        before = dec.launch_count()
        toks, lens = dec.greedy_decode(w.dec_lens)
        issued = dec.launch_count() - before
        toks, lens = toks.cpu().numpy(), lens.cpu().numpy()
    finally:
        dec.close()
    assert np.array_equal(lens, cut["lens"])
    for u in range(5):
        n = int(lens[u])
        assert np.array_equal(toks[u, :n], cut["next"][u, :n]) and np.all(toks[u, n:] == -1)
    per_step = 8 * SMALL["n_layers"] + 5
    assert issued < 30 * per_step, issued          # 200 steps would be 4200 launches


def test_handle_reuse_across_batch_sizes():
    """One handle and one pair of output buffers decode batches of 12, 7 and 12 utterances in turn (the step graphs
    recorded for the first batch are replayed for the others): every batch against the checker."""
    import torch
    b = _binding()
    rng = np.random.default_rng(3)
    works = [wl.make_custom(MID, rng.integers(1, 90, size=n), rng.integers(2, 12, size=n), dtype="bf16", seed=71,
                            out_std=0.3) for n in (12, 7, 12)]
    dec = b.Decoder(MID, works[0].weights, "bf16", max_batch=12,
                    max_total_enc_frames=max(int(w.enc_lens.sum()) for w in works),
                    max_enc_len=max(int(w.enc_lens.max()) for w in works), max_dec_len=12)
    toks = torch.empty((12, 12), dtype=torch.int32, device="cuda:0")
    lens = torch.empty(12, dtype=torch.int32, device="cuda:0")
    total = 0
    try:
        for w in works:
            per_batch = 0
            assert all(np.array_equal(a, c) for a, c in zip(w.weights["w_qkv"], works[0].weights["w_qkv"]))
            ref = oracle_reference(w, want_logits=False)
            dec.precompute_cross_kv(dec.upload_encoder(w.enc), w.enc_lens)
            dec.greedy_decode(w.dec_lens, toks, lens)
            got, got_lens = toks.cpu().numpy(), lens.cpu().numpy()
            assert np.array_equal(got_lens[:w.batch], w.dec_lens)
            for u in range(w.batch):
                L = int(w.dec_lens[u])
                assert np.all(got[u, L:] == -1)
                for t in range(L):
                    if ref["margin"][u, t] <= MARGIN:
                        break
                    assert got[u, t] == ref["next"][u, t], (w.batch, u, t)
                    per_batch += 1
            assert per_batch > 0
            total += per_batch
    finally:
        dec.close()
    assert total > 0


LN_CASES = {
    "small": (SMALL, [37, 5, 70, 9], [9, 12, 4, 6]),
    "mid": (MID, [1, 63, 130, 17, 40, 8, 90], [3, 20, 7, 11, 2, 16, 5]),
    "wide": (dict(n_layers=2, d_model=1024, n_heads=16, d_ffn=2048, vocab=900, d_enc=256), [50, 3, 140, 21, 77], [6, 9, 3, 8, 5]),
}


@pytest.mark.parametrize("offset", [0.0, 4.0])
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("case", ["small", "mid", "wide"])
def test_layernorm_parameters_output_bias_and_mean_offset(case, dtype, offset):
    """LayerNorm gains and shifts drawn around 1 and 0 (N(1, 0.3), N(0, 0.3)), an output-projection bias, and
    (offset 4) an embedding table shifted by a constant so that the residual stream's mean dwarfs its spread:
    the folded LayerNorm rstd * ((gamma * x) W^T - mean * c1) + c2 has to survive that cancellation."""
    model, enc_lens, dec_lens = LN_CASES[case]
    w = wl.make_custom(model, enc_lens, dec_lens, dtype=dtype, seed=91, ln_std=0.3, out_bias_std=0.3,
                       embed_offset=offset)
    _run_both(w, need_tokens=False, label=f"ln-{case}-offset{offset:g}")


def test_long_rows_bf16():
    """Decodes far beyond 128 cached positions (the self-attention block loops over its warps' chunks more than
    once) beside a short one, with encoder outputs of up to 500 frames at a batch small enough for the
    cross-attention variant that overlaps its loads: every step of every row against the checker."""
    w = wl.make_custom(MID, [300, 40, 500, 9, 77], [240, 145, 129, 128, 17], dtype="bf16", seed=33, out_std=0.1)
    _run_both(w, label="long-rows")


def test_error_codes():
    import torch
    b = _binding()
    w = wl.make_custom(SMALL, [5, 6], [3, 3], dtype="fp32", seed=2)
    dec = b.decoder_for_workload(w)
    toks = torch.ones(2, dtype=torch.int32, device="cuda:0")
    with pytest.raises(b.AedError) as e:
        dec.step(toks)
    assert e.value.status == b.AED_ERR_STATE
    enc = dec.upload_encoder(w.enc)
    with pytest.raises(b.AedError) as e:
        dec.precompute_cross_kv(enc, [5, 0])
    assert e.value.status == b.AED_ERR_INVALID_ARG
    with pytest.raises(b.AedError) as e:
        dec.precompute_cross_kv(enc, [5, 7])          # beyond max_enc_len = 6
    assert e.value.status == b.AED_ERR_CAPACITY
    with pytest.raises(b.AedError) as e:
        dec.precompute_cross_kv(enc, [5, 6, 1])       # beyond max_batch = 2
    assert e.value.status == b.AED_ERR_CAPACITY
    dec.precompute_cross_kv(enc, w.enc_lens)
    with pytest.raises(b.AedError) as e:
        dec.greedy_decode([3, 4])                     # beyond max_dec_len = 3
    assert e.value.status == b.AED_ERR_CAPACITY
    with pytest.raises(b.AedError) as e:
        dec.greedy_decode([3, 0])
    assert e.value.status == b.AED_ERR_INVALID_ARG
    for _ in range(3):
        dec.step(toks)
    with pytest.raises(b.AedError) as e:
        dec.step(toks)                                # caches are full
    assert e.value.status == b.AED_ERR_CAPACITY
    with pytest.raises(b.AedError) as e:
        dec.greedy_decode([3, 3])                     # not directly after a precompute
    assert e.value.status == b.AED_ERR_STATE
    dec.sync_status()
    # a masked step on an utterance whose cache is full is refused on the device, not written out of bounds
    dec.precompute_cross_kv(enc, w.enc_lens)
    only0 = torch.tensor([1, 0], dtype=torch.uint8, device="cuda:0")
    for _ in range(4):
        dec.step(toks, only0)
    with pytest.raises(b.AedError) as e:
        dec.sync_status()
    assert e.value.status == b.AED_ERR_CAPACITY
    dec.close()
    # creation errors
    bad = dict(SMALL, d_model=96, n_heads=2)          # head_dim 48
    wb = wl.make_custom(bad, [4], [2], seed=1)
    with pytest.raises(b.AedError) as e:
        b.decoder_for_workload(wb)
    assert e.value.status == b.AED_ERR_UNSUPPORTED
    lib = b.load_library()
    assert lib.aed_dec_create(None, None, None) == b.AED_ERR_INVALID_ARG
    assert lib.aed_dec_step(None, None, None, None, None) == b.AED_ERR_INVALID_ARG
    lib.aed_dec_destroy(None)


@pytest.mark.parametrize("batch", [130, 300, 520])
def test_large_batches_bf16(batch):
    """Row counts beyond one MMA tile: N = 256 tiles, two and three row tiles, with rows retiring at different steps."""
    rng = np.random.default_rng(batch)
    enc_lens = rng.integers(1, 90, size=batch)
    dec_lens = rng.integers(1, 9, size=batch)
    dec_lens[:3] = [12, 1, 7]
    w = wl.make_custom(MID, enc_lens, dec_lens, dtype="bf16", seed=40 + batch, out_std=0.1)
    rows = [0, 1, 2, batch // 2, batch - 2, batch - 1] + [int(r) for r in rng.choice(batch, size=6, replace=False)]
    _run_both(w, rows=sorted(set(rows)))


@pytest.mark.parametrize("batch", [20, 130])
def test_projection_stage_ring_reuse(batch, monkeypatch):
    """With a single k-split every projection CTA walks all of its k-blocks (4 for d = 256, 8 for the FFN): two rounds
    of the tcgen05 kernel for the FFN at 20 rows, and the ring of the many-rows kernel, whose stages are refilled while
    earlier ones are still being read, at 130."""
    monkeypatch.setenv("AED_DEC_GEMM_CTAS", "1")
    rng = np.random.default_rng(batch)
    w = wl.make_custom(MID, rng.integers(1, 90, size=batch), rng.integers(1, 7, size=batch), dtype="bf16", seed=batch,
                       out_std=0.1)
    _run_both(w, rows=[0, 1, batch // 2, batch - 1])


@pytest.mark.parametrize("model, batch, ctas", [("odd", 49, None), ("odd", 64, "8"), ("wide_a", 65, None), ("odd", 112, "1"), ("wide_a", 113, "24"),
                                                 ("odd", 128, None)])
def test_projections_of_49_to_128_rows(model, batch, ctas, monkeypatch):
    """The tcgen05 projections: one to five k-blocks per CTA in one round or two, k-splits of unequal length, one to eight
    rows of a k-block per thread, a last row tile of 16 with one row, feature counts that end inside a tile."""
    if ctas:
        monkeypatch.setenv("AED_DEC_GEMM_CTAS", ctas)
    rng = np.random.default_rng(990 + batch)
    w = wl.make_custom({"odd": ODD, "wide_a": WIDE_A}[model], rng.integers(1, 40, size=batch), rng.integers(1, 5, size=batch), dtype="bf16",
                       seed=370 + batch, out_std=0.1, ln_std=0.2, bias_std=0.05)
    _run_both(w, rows=sorted({0, 15, 16, 31, 32, 47, 48, batch // 2, batch - 2, batch - 1}))


def test_config3_shape_sampled_rows():
    """4-layer d=1024 bf16 decoder at batch 128 (shallow-decoder variant), sampled utterances against the checker."""
    w = wl.make_workload("cfg3")
    order = np.argsort(w.dec_lens)
    rows = sorted({int(order[1]), int(order[len(order) // 3]), int(np.argmax(w.enc_lens)), 127})
    rows = [r for r in rows if w.dec_lens[r] <= 60][:4]
    _run_both(w, rows=rows)


def test_config4_shape_sampled_rows():
    """24-layer d=1024 bf16 decoder at batch 512 with uniform durations (the large-batch configuration: 256-row
    projection tiles, rows retiring step by step down to the small-batch path): sampled short utterances against
    the checker, every other utterance of the batch decoding alongside."""
    w = wl.make_workload("cfg4")
    order = np.argsort(w.dec_lens)
    rows = sorted({int(order[0]), int(order[5]), int(order[17]), int(np.argmin(w.enc_lens))})
    rows = [r for r in rows if w.dec_lens[r] <= 24][:4]
    assert rows
    # plus one long row: more than 128 tokens (the looping part of self-attention) over more than 400 frames
    long_rows = [int(r) for r in np.flatnonzero((w.dec_lens > 128) & (w.enc_lens > 400))]
    assert long_rows
    rows = sorted(set(rows + [min(long_rows, key=lambda r: int(w.dec_lens[r]))]))
    _run_both(w, rows=rows)


def test_config2_shape_sampled_rows():
    """24-layer d=1024 bf16 decoder at batch 64 (the benchmark configuration, on both launch paths): a sample of
    utterances is decoded one by one by the checker and compared with the GPU's full-batch run."""
    w = wl.make_workload("cfg2")
    order = np.argsort(w.dec_lens)
    rows = sorted({int(order[0]), int(order[len(order) // 2]), int(order[3]), int(np.argmin(w.enc_lens))})
    # keep the checker's work bounded: drop sampled rows longer than 40 tokens
    rows = [r for r in rows if w.dec_lens[r] <= 40][:4]
    rows = sorted(set(rows + [int(np.argmax(w.dec_lens))]))     # and the longest decode of the batch (131 tokens)
    _run_both(w, rows=rows)


# ---- small batches: every row-tile width of the step projections ------------------------------------------------------

WIDE_A = dict(n_layers=2, d_model=512, n_heads=8, d_ffn=1024, vocab=600, d_enc=256)
WIDE_B = dict(n_layers=1, d_model=1024, n_heads=16, d_ffn=768, vocab=520, d_enc=128)
ODD = dict(n_layers=3, d_model=192, n_heads=3, d_ffn=320, vocab=333, d_enc=64)           # 3 k-blocks, partial feature tiles


@pytest.mark.parametrize("batch", [1, 7, 16, 17, 40, 64])
def test_small_batch_row_counts(batch):
    """Row-tile widths 16, 32 and 64 of the step projections with partly filled tiles, ragged encoder lengths from
    1 frame to several attention chunks, and rows retiring at different steps."""
    rng = np.random.default_rng(900 + batch)
    enc_lens = rng.integers(1, 150, size=batch)
    dec_lens = rng.integers(1, 24, size=batch)
    enc_lens[0], dec_lens[0] = 1, 40              # one frame; longer than two 16-position chunks of the self cache
    w = wl.make_custom(WIDE_A, enc_lens, dec_lens, dtype="bf16", seed=300 + batch, out_std=0.1)
    rows = sorted({0, batch - 1, batch // 2, int(np.argmax(enc_lens))})
    _run_both(w, rows=rows)


@pytest.mark.parametrize("batch", [20, 24, 25, 33, 47, 49])
def test_row_tiles_of_three(batch):
    """Row counts around the steps that cover their rows with three tiles of 8 per CTA: a partly filled third tile, a
    full one, one row beyond, and the same in two row halves (the second one partly filled)."""
    rng = np.random.default_rng(950 + batch)
    w = wl.make_custom(WIDE_A, rng.integers(1, 80, size=batch), rng.integers(1, 6, size=batch), dtype="bf16", seed=330 + batch,
                       out_std=0.1, ln_std=0.2)
    _run_both(w, rows=sorted({0, 7, 16, 19, batch // 2, batch - 1}))


@pytest.mark.parametrize("batch", [3, 4, 5, 11, 12, 13, 20, 21, 28, 29, 36, 37, 44, 45])
def test_row_tiles_of_four(batch):
    """Row counts whose last row tile has at most four rows (high and low planes in one MMA), filled, partly filled and one row
    beyond, alone and in two row halves."""
    rng = np.random.default_rng(1100 + batch)
    w = wl.make_custom(WIDE_A, rng.integers(1, 80, size=batch), rng.integers(1, 6, size=batch), dtype="bf16", seed=510 + batch,
                       out_std=0.1, ln_std=0.2)
    _run_both(w, rows=sorted({0, batch // 2 - 1, batch // 2, max(batch - 5, 0), batch - 4 if batch > 4 else 0, batch - 1}))


@pytest.mark.parametrize("model, batch", [("odd", 49), ("odd", 63), ("odd", 64), ("wide_a", 65), ("odd", 95), ("odd", 97), ("odd", 127), ("wide_b", 128)])
def test_halves_of_a_row_tile(model, batch):
    """Projections on pairs of blocks with half of the rows each: even and odd row counts, tiles of 64, 96 and 128 rows, full and not, and
    feature counts that are an odd number of 128s (the last pair's second block has none)."""
    rng = np.random.default_rng(1200 + batch)
    m = {"wide_a": WIDE_A, "wide_b": WIDE_B, "odd": ODD}[model]
    w = wl.make_custom(m, rng.integers(1, 40, size=batch), rng.integers(1, 4, size=batch), dtype="bf16", seed=530 + batch,
                       out_std=0.1, ln_std=0.2)
    half = (batch + 1) // 2
    _run_both(w, rows=sorted({0, 15, 16, half - 1, half, half + 16, batch - 2, batch - 1}))


@pytest.mark.parametrize("model, batch", [("wide_a", 129), ("wide_b", 65), ("odd", 342), ("odd", 347)])
def test_self_attention_of_many_rows(model, batch):
    """More than 1024 (row, head) pairs, where self-attention takes a warp per pair: just above the line, a last block
    with 1 and 2 of its 8 pairs, blocks that span two rows, and caches that end at and around 16-position chunks."""
    rng = np.random.default_rng(970 + batch)
    dec_lens = rng.integers(1, 6, size=batch)
    dec_lens[:5] = [1, 16, 17, 33, 34]
    m = {"wide_a": WIDE_A, "wide_b": WIDE_B, "odd": ODD}[model]
    w = wl.make_custom(m, rng.integers(1, 30, size=batch), dec_lens, dtype="bf16", seed=340 + batch, out_std=0.1, ln_std=0.2)
    _run_both(w, rows=[0, 1, 2, 3, 4, batch // 2, batch - 1])


@pytest.mark.parametrize("batch, frames", [(80, 40), (160, 40), (160, 300)])
def test_attention_blocks_of_fewer_warps(batch, frames):
    """320 and 640 (row, head) pairs that all reach position 139: self-attention blocks of 4 and 2 warps whose warps take up to
    five 16-position chunks each; 640 pairs of cross-attention with short outputs (4 warps) and with long ones (8)."""
    rng = np.random.default_rng(1010 + batch + frames)
    dec_lens = np.full(batch, 140)
    dec_lens[1] = 129
    w = wl.make_custom(MID, rng.integers(max(1, frames - 20), frames + 1, size=batch), dec_lens, dtype="bf16", seed=410 + batch + frames,
                       out_std=0.1, ln_std=0.2)
    _run_both(w, rows=[0, 1, batch - 1])


@pytest.mark.parametrize("enc_lens", [(1,), (128,), (100, 29), (256,), (200, 57), (384, 1)])
def test_cross_kv_frame_tiles(enc_lens):
    """Encoder frames that fill 1, 2, 3 and 4 tiles of 128 exactly or by one frame (an odd last tile has no partner in
    its pair of blocks), with a feature count that ends inside a 256-wide tile and crosses from keys to values in it."""
    w = wl.make_custom(ODD, list(enc_lens), [3] * len(enc_lens), dtype="bf16", seed=360 + sum(enc_lens), out_std=0.1, ln_std=0.2,
                       bias_std=0.05)
    _run_both(w)


@pytest.mark.parametrize("batch", [18, 70, 83, 131, 163, 259])
def test_equal_row_tiles(batch):
    """Row counts that take one tile of 32, 80 or 96 rows, two of 80, two of 96 with ready-made planes, and two tiles of
    the vocabulary projection, whose 333 entries end inside a tile and inside a lane's four."""
    rng = np.random.default_rng(980 + batch)
    w = wl.make_custom(ODD, rng.integers(1, 20, size=batch), rng.integers(1, 4, size=batch), dtype="bf16", seed=350 + batch,
                       out_std=0.1, ln_std=0.2, out_bias_std=0.1)
    _run_both(w, rows=sorted({0, 15, 16, 17, batch // 2 - 1, batch // 2, batch // 2 + 1, batch - 2, batch - 1}))


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("groups", [[(8, 3)], [(9, 3)], [(4, 2), (5, 4), (3, 7)], [(131, 2), (5, 6)], [(60, 3), (2, 5)]])
def test_rows_of_the_next_step(groups, dtype):
    """Steps around the 8 rows that the bookkeeping kernel embeds itself, and row counts that fall to fewer from one step
    to the next: from 12 over 8 to 3, from ready-made planes (136 rows) and from the tiled projections (62) at once."""
    dec_lens = np.concatenate([[steps] * n for n, steps in groups])
    rng = np.random.default_rng(len(dec_lens))
    rng.shuffle(dec_lens)
    w = wl.make_custom(ODD, rng.integers(1, 20, size=len(dec_lens)), dec_lens, dtype=dtype, seed=370 + len(dec_lens), out_std=0.1, ln_std=0.2)
    _run_both(w, rows=sorted({0, len(dec_lens) - 1} | set(int(u) for u in np.argsort(dec_lens)[-5:])))


@pytest.mark.parametrize("batch", [3, 12, 50, 131])
def test_steps_with_other_buffers(batch, monkeypatch):
    """Steps of the caller's loop of a size that keeps coming are replayed as graphs (enough of them here that the last passes are):
    every call has tokens, logits and choices of its own (or none), and a mask or none, and has to do what the same calls do
    launched kernel by kernel."""
    import torch
    rng = np.random.default_rng(1000 + batch)
    w = wl.make_custom(MID, rng.integers(1, 60, size=batch), [8] * batch, dtype="bf16", seed=400 + batch, out_std=0.1, ln_std=0.2)
    V = MID["vocab"]
    tokens = torch.from_numpy(rng.integers(0, V, size=(6, batch)).astype(np.int32)).cuda()
    mask = torch.from_numpy((rng.random(batch) < 0.6).astype(np.uint8)).cuda()

    def run(graphs, passes, everything):
        monkeypatch.setenv("AED_DEC_NO_GRAPH", "0" if graphs else "1")
        dec = _binding().decoder_for_workload(w)
        enc = dec.upload_encoder(w.enc)
        outs = []
        for _ in range(passes):
            dec.precompute_cross_kv(enc, w.enc_lens)
            for t in range(6):
                logits = torch.full((batch, V), -7.0, device="cuda") if everything or t % 3 != 1 else None
                choice = torch.full((batch,), -1, dtype=torch.int32, device="cuda") if everything or t % 2 == 0 else None
                dec.step(tokens[t].clone(), mask if t in (2, 4) else None, logits, choice)
                outs.append([x.clone() if x is not None else None for x in (logits, choice)])
        dec.sync_status()
        dec.close()
        return outs

    # fp32 sums of split projections come in another order, so logits may differ by `tol`, and choices only where the two best
    # entries are closer than twice that
    tol, decided, choices = 2e-3, 0, 0
    want = run(False, 1, True)
    for i, (logits, choice) in enumerate(run(True, 8, False)):
        full, best = want[i % 6]
        if logits is not None:
            assert torch.equal(logits == -7.0, full == -7.0)
            assert float((logits - full).abs().max()) < tol
        if choice is not None:
            assert torch.equal(choice == -1, best == -1)
            top = full.topk(2, dim=1).values
            sure = (top[:, 0] - top[:, 1] > 2 * tol) & (best != -1)
            assert torch.equal(choice[sure], best[sure])
            decided, choices = decided + int(sure.sum()), choices + int((best != -1).sum())
    assert decided > 0.9 * choices


@pytest.mark.parametrize("dtype, steps", [("bf16", 3), ("bf16", 4), ("bf16", 21), ("fp32", 37)])
def test_several_steps_per_graph(dtype, steps):
    """Greedy decodes of fewer steps than a graph holds, of exactly as many, and across 16-position chunks, with rows that
    retire inside a graph."""
    w = wl.make_custom(ODD, [9, 30, 4], [steps, max(1, steps - 5), 2], dtype=dtype, seed=380 + steps, out_std=0.1, ln_std=0.2)
    _run_both(w)


@pytest.mark.parametrize("model, batch", [("odd", 129), ("wide_a", 193), ("odd", 320), ("wide_b", 321), ("odd", 385)])
def test_plane_projections(model, batch):
    """The row counts at which the projections of many rows change their tiles (two of 96, 128 and 160, three and four of
    128, FFN1 in more), with an odd number of 128-feature tiles and tiles that end inside one."""
    rng = np.random.default_rng(990 + batch)
    m = {"wide_a": WIDE_A, "wide_b": WIDE_B, "odd": ODD}[model]
    w = wl.make_custom(m, rng.integers(1, 20, size=batch), rng.integers(1, 4, size=batch), dtype="bf16", seed=390 + batch, out_std=0.1,
                       ln_std=0.2, bias_std=0.05)
    _run_both(w, rows=sorted({0, 31, 32, 95, 96, batch // 2, batch - 2, batch - 1}))


F32_DEEP = dict(n_layers=2, d_model=320, n_heads=5, d_ffn=1344, vocab=517, d_enc=192)


@pytest.mark.parametrize("heads", [22, 24, 26])
def test_vocabulary_projection_of_wide_models(heads):
    """Few rows and a d_model (1408, 1536, 1664) around the widest that the few-row vocabulary kernel has shared memory for."""
    model = dict(n_layers=1, d_model=64 * heads, n_heads=heads, d_ffn=256, vocab=300, d_enc=128)
    w = wl.make_custom(model, [9, 5, 30], [3, 3, 2], dtype="bf16", seed=690 + heads, out_std=0.1)
    _run_both(w, label=f"d{64 * heads}")


@pytest.mark.parametrize("batch", [16, 17, 63, 64, 65, 80, 128, 129, 256, 257, 300])
def test_vocabulary_projection_of_one_k_block(batch):
    """d_model 64: the ring of the vocabulary projection has one stage, and the accumulator's rows need more room than it
    in tiles of 64 rows and more; row tiles of 16 to 256, one and two of them, on either side of the switch to ready-made planes."""
    model = dict(n_layers=2, d_model=64, n_heads=1, d_ffn=128, vocab=333, d_enc=64)
    rng = np.random.default_rng(600 + batch)
    w = wl.make_custom(model, rng.integers(1, 40, size=batch), rng.integers(1, 4, size=batch), dtype="bf16", seed=601 + batch, out_std=0.4)
    rows = sorted({0, 15, 16, 63, 64, 79, 127, 128, 255, 256, batch - 1} & set(range(batch)))
    _run_both(w, rows=rows, label=f"d64 B={batch}")


@pytest.mark.parametrize("dtype, batch", [("fp32", 3), ("fp32", 12), ("fp32", 21), ("bf16", 3), ("bf16", 12), ("bf16", 40), ("bf16", 70), ("bf16", 131)])
def test_vectors_at_any_element(dtype, batch, monkeypatch):
    """LayerNorm parameters and biases that start one element past a 16-byte boundary."""
    _shift_vectors(monkeypatch)
    rng = np.random.default_rng(620 + batch)
    w = wl.make_custom(MID, rng.integers(1, 60, size=batch), rng.integers(1, 5, size=batch), dtype=dtype, seed=621 + batch, out_std=0.3,
                       ln_std=0.3, out_bias_std=0.1)
    _run_both(w, rows=sorted({0, batch // 2, batch - 1}), label=f"shifted vectors B={batch}")


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_encoder_states_have_to_be_aligned(dtype):
    """Encoder states off a 16-byte boundary are refused by every call that takes them, and the batch of before goes on."""
    import torch
    b = _binding()
    w = wl.make_custom(SMALL, [9, 5], [3, 3], dtype=dtype, seed=630)
    dec = b.decoder_for_workload(w)
    enc = dec.upload_encoder(w.enc)
    dec.precompute_cross_kv(enc, w.enc_lens)
    bad = torch.zeros(enc.numel() + 1, dtype=enc.dtype, device="cuda:0")[1:].view(enc.shape)
    with pytest.raises(b.AedError) as e:
        dec.precompute_cross_kv(bad, w.enc_lens)
    assert e.value.status == b.AED_ERR_INVALID_ARG
    with pytest.raises(b.AedError) as e:
        dec.decode_stream(bad, w.enc_lens, w.dec_lens, 1)
    assert e.value.status == b.AED_ERR_INVALID_ARG
    toks, lens = dec.greedy_decode(w.dec_lens)
    assert np.array_equal(lens.cpu().numpy(), w.dec_lens)
    dec.open_slots(1)
    with pytest.raises(b.AedError) as e:
        dec.admit(0, bad[:9], 3)
    assert e.value.status == b.AED_ERR_INVALID_ARG
    dec.close()


def test_fp32_half_a_million_rows():
    """fp32: more frames, and more rows of a step, than 8-row tiles fit into one extent of a grid (8 * 65535)."""
    import torch
    batch = 8 * 65535 + 21
    model = dict(n_layers=1, d_model=64, n_heads=1, d_ffn=64, vocab=40, d_enc=64)
    w = wl.make_custom(model, [1] * batch, [2] * batch, dtype="fp32", seed=660, out_std=0.3)
    rows = [0, 63, 8 * 65535 - 1, 8 * 65535, batch - 1]
    ref = oracle_reference(w, rows)
    dec = _binding().decoder_for_workload(w)
    worst, compared, bad = teacher_forced_compare(dec, w, ref, rows)
    assert compared == 2 * len(rows) and worst < TOL["fp32"] and not bad, (worst, bad)
    dec.precompute_cross_kv(dec.upload_encoder(w.enc), w.enc_lens)
    toks, lens = dec.greedy_decode(w.dec_lens)
    dec.close()
    assert bool((lens == 2).all())
    got = toks[torch.tensor(rows, device="cuda:0")].cpu().numpy()
    for i in range(len(rows)):
        for t in range(2):
            if ref["margin"][i, t] <= MARGIN:
                break
            assert got[i, t] == ref["next"][i, t]


def _shift_vectors(monkeypatch):
    """Decoders from here on have their LayerNorm parameters and biases one element past a 16-byte boundary."""
    cls = _binding().Decoder
    upload = cls._upload

    def shifted(self, arr):
        arr = np.asarray(arr)
        if arr.ndim != 1:
            return upload(self, arr)
        return upload(self, np.concatenate([np.zeros(1, arr.dtype), arr])) + self.tdtype.itemsize
    monkeypatch.setattr(cls, "_upload", shifted)


@pytest.mark.parametrize("vocab, batch, shift", [(12001, 33, False), (12001, 64, True), (6200, 64, False), (6200, 65, False), (90, 1537, False), (90, 1600, True)])
def test_fp32_tiles_of_many_rows(vocab, batch, shift, monkeypatch):
    """fp32 launches on either side of the rule for 64 x 64 tiles: the vocabulary projection alone (33 to 65 rows), every
    projection of a step (1537 and 1600), with rows and features that fill their last tile by one or not at all, and vectors
    that cannot be read 16 bytes at a time."""
    if shift:
        _shift_vectors(monkeypatch)
    model = dict(n_layers=1, d_model=256, n_heads=4, d_ffn=320, vocab=vocab, d_enc=192)
    rng = np.random.default_rng(670 + batch)
    w = wl.make_custom(model, rng.integers(1, 30, size=batch), rng.integers(1, 4, size=batch), dtype="fp32", seed=671 + batch, out_std=0.1,
                       ln_std=0.3, out_bias_std=0.1)
    _run_both(w, rows=sorted({0, 1, 31, 32, 63, 64, 1535, 1536, batch - 1} & set(range(batch))), label=f"fp32 tiles V={vocab} B={batch}")


@pytest.mark.parametrize("frames", [767, 768, 769, 833])
def test_fp32_cross_kv_frames(frames):
    """fp32 cross-attention keys and values around the rule for tiles (512 features: 768 frames) and past a whole tile."""
    model = dict(n_layers=2, d_model=256, n_heads=4, d_ffn=64, vocab=90, d_enc=192)
    w = wl.make_custom(model, [500, 1, frames - 501], [3, 3, 3], dtype="fp32", seed=680 + frames, out_std=0.3)
    _run_both(w, label=f"{frames} frames")


@pytest.mark.parametrize("frames", [2, 40, 300])
def test_fp32_softmax_weights_below_the_normal_range(frames):
    """fp32: a softmax weight below 2^-126 still counts (here e^-89 times a value of 1e38).  The cross-attention query is the
    constant (8, 0, ...), so the score of a frame is its first encoder value and what it contributes its second one."""
    d = 64
    model = dict(n_layers=1, d_model=d, n_heads=1, d_ffn=64, vocab=50, d_enc=64)
    w = wl.make_custom(model, [frames, frames], [2, 2], dtype="fp32", seed=650, out_std=1.0)
    W = w.weights
    zero = lambda *names: [W[n].__setitem__(0, np.zeros_like(W[n][0])) for n in names]
    zero("w_o", "b_o", "w_q_c", "b_q_c", "w_kv_c", "b_kv_c", "w_o_c", "b_o_c", "w_ff2", "b_ff2")
    W["embed"] = np.zeros_like(W["embed"])
    W["b_q_c"][0][0] = 8.0
    W["w_kv_c"][0][0, 0] = 1.0                        # key dimension 0 = encoder value 0
    W["w_kv_c"][0][d + 1, 1] = 1.0                    # value dimension 1 = encoder value 1
    W["w_o_c"][0][1, 1] = 1.0
    w.enc[:] = 0.0
    for u, at in ((0, frames - 1), (1, frames // 2)):
        w.enc[u * frames:(u + 1) * frames, 0] = -200.0
        w.enc[u * frames, 0] = 0.0
        w.enc[u * frames + at, :2] = (-89.0, 1e38)
    ref = oracle_reference(w)
    assert np.max(np.abs(ref["logits"][0][0])) > 0.1
    dec = _binding().decoder_for_workload(w)
    worst, _, _ = teacher_forced_compare(dec, w, ref)
    dec.close()
    assert worst < TOL["fp32"], worst


@pytest.mark.parametrize("dtype, batch", [("fp32", 3), ("fp32", 12), ("fp32", 21), ("bf16", 3), ("bf16", 21), ("bf16", 70)])
def test_choice_among_special_logits(dtype, batch):
    """The greedy choice is the lowest index of the largest logit, also among negative ones and infinities; a NaN is chosen
    only if nothing else is there."""
    import torch
    b = _binding()
    w = wl.make_custom(SMALL, [7] * batch, [2] * batch, dtype=dtype, seed=640, out_std=0.1, out_bias_std=0.1)
    V = SMALL["vocab"]
    plain = w.weights["b_out"].copy()
    toks = torch.arange(batch, dtype=torch.int32, device="cuda:0") + 3
    nothing = {i: -np.inf for i in range(V)}
    for shift, special in ((0, {5: np.nan, 299: np.nan}), (-64, {5: np.nan, 299: np.nan}), (-64, {5: np.nan, 9: -np.inf}),
                           (0, {7: np.inf, 200: np.inf, 3: np.nan}), (0, nothing), (0, {**nothing, 0: np.nan}),
                           (0, {i: np.nan for i in range(V)})):
        bias = plain + np.float32(shift)
        for i, v in special.items():
            bias[i] = v
        w.weights["b_out"] = bias
        dec = b.decoder_for_workload(w)
        dec.precompute_cross_kv(dec.upload_encoder(w.enc), w.enc_lens)
        logits = torch.zeros((batch, V), dtype=torch.float32, device="cuda:0")
        nxt = torch.full((batch,), -7, dtype=torch.int32, device="cuda:0")
        dec.step(toks, None, logits, nxt)
        z, got = logits.cpu().numpy(), nxt.cpu().numpy()
        dec.close()
        assert np.array_equal(np.isnan(z), np.broadcast_to(np.isnan(bias), z.shape))
        largest = np.max(z, axis=1, where=~np.isnan(z), initial=-np.inf, keepdims=True)
        want = np.argmax(z == largest, axis=1)            # (all NaN: no entry is equal, index 0)
        assert np.array_equal(got, want), (shift, got, want)


@pytest.mark.parametrize("batch", [1, 4, 5, 16, 17, 23])
def test_fp32_row_tiles(batch):
    """Rows around the steps between 4-row and 8-row tiles and one and two features per warp of the fp32 projections, with
    K beyond the weights held ahead, K no multiple of 128 and feature counts that end inside a block."""
    rng = np.random.default_rng(995 + batch)
    w = wl.make_custom(F32_DEEP, rng.integers(1, 40, size=batch), rng.integers(1, 6, size=batch), dtype="fp32", seed=400 + batch, out_std=0.1,
                       ln_std=0.2)
    _run_both(w)


@pytest.mark.parametrize("model", ["wide_b", "odd"])
def test_small_batch_model_shapes(model):
    """d_model 1024 with 16 heads at 64 rows, and a model whose widths are not multiples of 128 (an odd number of
    k-blocks, feature tiles that end inside a tile, a cross-K/V feature count that is not a multiple of 256)."""
    rng = np.random.default_rng(31)
    batch = 64 if model == "wide_b" else 23
    m = WIDE_B if model == "wide_b" else ODD
    w = wl.make_custom(m, rng.integers(1, 200, size=batch), rng.integers(1, 20, size=batch), dtype="bf16", seed=77,
                       out_std=0.1, ln_std=0.2, out_bias_std=0.1)
    _run_both(w, rows=[0, 5, batch // 2, batch - 1])


@pytest.mark.parametrize("seed", range(10))
def test_random_shapes_and_row_counts_bf16(seed):
    """Model widths, k-block counts, row counts and lengths drawn at random: every projection form (warp-level with
    fragments from global memory, with shared-memory planes at one or two row halves, tcgen05, ready-made planes) meets
    k ranges of one, two and four k-blocks, partial feature tiles and partly filled row tiles."""
    rng = np.random.default_rng(1000 + seed)
    heads = int(rng.integers(1, 6))
    d = 64 * heads
    model = dict(n_layers=int(rng.integers(1, 4)), d_model=d, n_heads=heads, d_ffn=64 * int(rng.integers(1, 13)),
                 vocab=int(rng.integers(130, 700)), d_enc=64 * int(rng.integers(1, 5)))
    batch = int(rng.choice([1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 31, 32, 33, 40, 41, 48, 63, 64, 65, 90, 128, 129, 140]))
    enc_lens = rng.integers(1, 160, size=batch)
    dec_lens = rng.integers(1, 7, size=batch)
    w = wl.make_custom(model, enc_lens, dec_lens, dtype="bf16", seed=2000 + seed, out_std=0.1, ln_std=0.2, bias_std=0.05)
    rows = sorted({0, batch - 1, batch // 2, int(np.argmax(dec_lens)), int(np.argmax(enc_lens))})
    _run_both(w, rows=rows, need_tokens=False, label=f"random shape {model} B={batch}")


@pytest.mark.parametrize("model, batch", [("tiny", 1), ("tiny", 5), ("tiny", 9), ("tiny", 28), ("tiny", 29), ("tiny", 57), ("one_head", 7), ("three_heads", 6),
                                          ("odd_vocab", 4)])
def test_fp32_steps_in_one_launch(model, batch):
    """Small fp32 models, whose steps are one launch: clusters with missing rows, clusters of 16 and of 8 blocks and just beyond both, rows embedded
    with the row table (up to 8) and in the launch, widths that leave blocks without features or pairs, caches and encoder outputs on both
    sides of what the warps of a pair take at a time."""
    m = {"tiny": wl.MODELS["tiny"], "one_head": dict(n_layers=2, d_model=64, n_heads=1, d_ffn=64, vocab=301, d_enc=64),
         "three_heads": dict(n_layers=3, d_model=192, n_heads=3, d_ffn=320, vocab=77, d_enc=64),
         "odd_vocab": dict(n_layers=1, d_model=256, n_heads=4, d_ffn=1024, vocab=2999, d_enc=128)}[model]
    rng = np.random.default_rng(1300 + batch)
    enc_lens, dec_lens = rng.integers(1, 80, size=batch), rng.integers(1, 6, size=batch)
    enc_lens[0], dec_lens[0] = 130, 70 if batch < 10 else 9
    w = wl.make_custom(m, enc_lens, dec_lens, dtype="fp32", seed=560 + batch, out_std=0.5, ln_std=0.2, out_bias_std=0.1)
    _run_both(w, rows=sorted({0, batch // 2, max(batch - 5, 0), batch - 1}))


def test_fp32_steps_in_one_launch_and_kernel_by_kernel(monkeypatch):
    """The same steps either way: their sums differ in order alone.  (Each is within 1e-4 of the checker; 2e-6 of logits of size 1 to
    10 is what the two orders of up to 1024 products leave.)"""
    import torch
    w = wl.make_custom(wl.MODELS["tiny"], [20, 33, 60, 7, 41], [6] * 5, dtype="fp32", seed=590, ln_std=0.2, out_bias_std=0.1)
    out = []
    for off in ("0", "1"):
        monkeypatch.setenv("AED_DEC_NO_CLUSTER", off)
        dec = _binding().decoder_for_workload(w)
        dec.precompute_cross_kv(dec.upload_encoder(w.enc), w.enc_lens)
        logits = torch.zeros((w.batch, w.model["vocab"]), dtype=torch.float32, device="cuda:0")
        steps = []
        for t in range(6):
            tokens = (torch.arange(w.batch, dtype=torch.int32, device="cuda:0") * 7 + 3 * t) % w.model["vocab"]
            dec.step(tokens, None, logits, None)
            steps.append(logits.clone())
        dec.sync_status()
        dec.close()
        out.append(torch.stack(steps))
    size = out[0].abs().max().item()
    assert (out[0] - out[1]).abs().max().item() < 2e-6 * max(size, 1.0)
