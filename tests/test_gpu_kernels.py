"""Single kernels at the sizes where they can go wrong: tile edges, remainders, the ends of their ranges."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bpd():
    import paper_1811_03115_b200 as b
    return b


# token tiles of 16..256 rows, K splits over clusters of 1, 2, 4 and 8 CTAs (with a short or an empty last split),
# feature counts that end inside a tile, inside a group of four, or take the scalar stores
@pytest.mark.parametrize("rows,in_f,out_f", [(1, 8, 4), (16, 64, 128), (17, 72, 130), (31, 584, 127), (33, 1024, 512), (96, 640, 1027),
                                             (257, 512, 256), (113, 4096, 516), (300, 2040, 64), (130, 328, 4100)])
def test_wide_projection_at_tile_edges(bpd, rows, in_f, out_f):
    import torch
    g = torch.Generator().manual_seed(rows + in_f)
    x = torch.randn(rows, in_f, generator=g).bfloat16()
    w = (torch.randn(out_f, in_f, generator=g) * 0.05).bfloat16()
    b = (torch.randn(out_f, generator=g) * 0.1).bfloat16()
    want = np.maximum(x.double().numpy() @ w.double().numpy().T + b.double().numpy(), 0)
    got = bpd.bpd_op_linear(x.cuda(), w.cuda(), b.cuda(), relu=True).cpu().numpy()
    np.testing.assert_allclose(got, want, atol=1e-5 * np.sqrt(in_f))
    idx, val = bpd.bpd_op_vocab_argmax(x[:, :1024].contiguous().cuda(), w[:, :1024].contiguous().cuda(), want_val=True)
    logits = x[:, :1024].double().numpy() @ w[:, :1024].double().numpy().T
    picked = logits[np.arange(rows), idx.cpu().numpy()]
    np.testing.assert_allclose(picked, logits.max(-1), atol=1e-4)
    np.testing.assert_allclose(val.cpu().numpy(), logits.max(-1), atol=1e-4)


# row tiles of 8, 16, 32 and 64 rows, K tiles of 64 columns, feature tiles of 32
@pytest.mark.parametrize("rows,in_f,out_f", [(1, 8, 1), (8, 64, 32), (9, 72, 33), (16, 1024, 31), (17, 136, 65), (64, 200, 96), (65, 64, 40),
                                             (129, 520, 7)])
def test_fp32_projection_at_tile_edges(bpd, rows, in_f, out_f):
    import torch
    g = torch.Generator().manual_seed(rows + in_f)
    x = torch.randn(rows, in_f, generator=g)
    w = torch.randn(out_f, in_f, generator=g) * 0.05
    b = torch.randn(out_f, generator=g) * 0.1
    want = x.double().numpy() @ w.double().numpy().T
    got = bpd.bpd_op_linear(x.cuda(), w.cuda(), b.cuda(), relu=True).cpu().numpy()
    np.testing.assert_allclose(got, np.maximum(want + b.double().numpy(), 0), atol=2e-6 * np.sqrt(in_f))
    idx, val = bpd.bpd_op_vocab_argmax(x.cuda(), w.cuda(), want_val=True)
    idx2, val2 = torch.zeros(rows, dtype=torch.int32, device="cuda"), torch.zeros(rows, device="cuda")
    bpd.bpd_op_vocab_argmax_noalloc(x.cuda(), w.cuda(), idx2, val2)
    for i, v in ((idx, val), (idx2, val2)):
        np.testing.assert_allclose(want[np.arange(rows), i.cpu().numpy()], want.max(-1), atol=1e-5)
        np.testing.assert_allclose(v.cpu().numpy(), want.max(-1), atol=1e-5)


# the fp32 top-1 only enqueues, so a program may capture it: replays after the kept scratch of the stream was replaced
# by a larger call's, with eager calls in between, on the stream of the capture and on another
def test_captured_fp32_top1_replays_after_its_stream_saw_larger_calls(bpd):
    import torch
    g = torch.Generator().manual_seed(3)
    w = (torch.randn(1000, 64, generator=g) * 0.05).cuda()
    x = torch.empty(37, 64, device="cuda")
    big = torch.randn(300, 64, generator=g).cuda()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        bpd.bpd_op_vocab_argmax(big[:37], w)                   # loads the kernel, leaves a small scratch kept for this stream
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            idx, val = bpd.bpd_op_vocab_argmax(x, w, want_val=True)
        bpd.bpd_op_vocab_argmax(big, w)
        torch.cuda.synchronize()
        canary = [torch.full((64, n), 7, dtype=torch.uint8, device="cuda") for n in (256, 1024, 4096)]
        torch.cuda.synchronize()
        for on in (s, torch.cuda.Stream()):
            x.copy_(torch.randn(37, 64, generator=g))
            torch.cuda.synchronize()
            with torch.cuda.stream(on):
                graph.replay()
            torch.cuda.synchronize()
            want = x.double().cpu().numpy() @ w.double().cpu().numpy().T
            np.testing.assert_allclose(want[np.arange(37), idx.cpu().numpy()], want.max(-1), atol=1e-5)
            np.testing.assert_allclose(val.cpu().numpy(), want.max(-1), atol=1e-5)
    assert all(bool((c == 7).all()) for c in canary)


# attention of many-row sessions against the oracle's decoder: one chunk and several (96 encoder rows per chunk), query tiles
# of up to 16 rows, sources from one id on, sequences long enough for a second chunk of 256 cached keys, local attention
@pytest.mark.parametrize("batch,k,max_src,tgt,local", [(3, 8, 33, 20, 0), (9, 2, 100, 12, 0), (10, 16, 17, 40, 0), (19, 3, 5, 300, 0), (19, 3, 97, 290, 64)])
def test_many_row_attention_decodes_like_the_oracle(bpd, batch, k, max_src, tgt, local):
    from bpd_inputs import ModelConfig, Workload, make_weights
    from oracle.decode import TransformerScorer
    from oracle.model import parse_blob
    cfg = ModelConfig(1, 2, 256, 4, 256, 300, k, 64, local_q=local, local_m=local // 2)
    w = Workload("attn", cfg, 0.06, 5, 6, 7, batch=batch, src_lo=1, src_hi=max_src, n_decode=tgt)
    blob = make_weights(cfg, 5, 0.06)
    rng = np.random.default_rng(batch)
    lens = rng.integers(1, max_src + 1, batch).astype(np.int32)
    lens[:2] = 1, max_src
    src = rng.integers(2, 300, (batch, max_src)).astype(np.int32)
    model = bpd.Model(blob)
    s = bpd.Session(model, batch, max_src, tgt)
    s.bpd_encode(src, lens)
    model_o, rows = parse_blob(blob), (0, 1, batch - 1)
    scorers = {b: TransformerScorer(model_o, src[b], int(lens[b]), cached=True, capacity=tgt + k + 2) for b in rows}
    inputs = {b: [0] for b in rows}
    for b in rows:
        scorers[b](inputs[b], 1)
    while True:
        r = s.bpd_iteration(k, tgt, want_hidden=True, accept_mode=k << 16)      # minimum block k: every proposal is kept
        for b in rows:
            block = [int(t) for t in r["block"][b]]
            scorers[b](inputs[b] + block, k)
            n = int(r["khat"][b])
            np.testing.assert_allclose(r["hidden"][b].cpu().numpy(), scorers[b].last_hidden, atol=8e-3)     # the cache is bf16
            inputs[b] += block[:n]
        if len(inputs[0]) > tgt:
            break
    s.close()
    model.close()


# the encoder with its layer norms folded into the projections (widths of whole pairs of tiles) and with layer-norm kernels,
# one decoder layer (its own launch of keys and values) and several (one launch), from one encoder row to several token tiles
@pytest.mark.parametrize("batch,max_src,d,n_dec", [(1, 1, 256, 2), (2, 9, 256, 1), (5, 60, 512, 3), (3, 40, 192, 2)])
def test_encoder_feeds_the_decoder_like_the_oracle(bpd, batch, max_src, d, n_dec):
    from bpd_inputs import ModelConfig, make_weights
    from oracle.decode import TransformerScorer
    from oracle.model import parse_blob
    blob = make_weights(ModelConfig(2, n_dec, d, d // 64, 2 * d, 300, 4, 64), 5, 0.06)
    rng = np.random.default_rng(d + batch)
    lens = rng.integers(1, max_src + 1, batch).astype(np.int32)
    lens[-1] = max_src
    src = rng.integers(2, 300, (batch, max_src)).astype(np.int32)
    model = bpd.Model(blob)
    s = bpd.Session(model, batch, max_src, 8)
    s.bpd_encode(src, lens)
    r = s.bpd_iteration(4, 8, want_hidden=True)
    model_o = parse_blob(blob)
    for b in range(batch):
        scorer = TransformerScorer(model_o, src[b], int(lens[b]), cached=True, capacity=14)
        scorer([0], 1)
        scorer([0] + [int(t) for t in r["block"][b]], 4)
        np.testing.assert_allclose(r["hidden"][b].cpu().numpy(), scorer.last_hidden, atol=8e-3)     # the cache is bf16
    s.close()
    model.close()


# With the decoder's self-attention output projections at zero nothing that reaches the hidden states is rounded to the
# cache's bf16: encoder, cross-attention and feed-forward layers carry fp32 throughout (two bf16 planes per activation, three
# in the attention kernels), in every form the layers take.  Rows far from zero mean (64 standard deviations) must cost the
# encoder nothing.  An activation's planes round at 2^-18 of its value, the hidden states are normalised (elements up to
# about 4) and some 15 such roundings lie on the way, so 15 * 4 * 2^-18 = 2.3e-4 at worst; 1e-4 is five times what is
# seen.  Losing a plane costs 2^-9 of a value, uncentred planes of the shifted rows 64 * 2^-18.
@pytest.mark.parametrize("shift", [0, 64])
@pytest.mark.parametrize("batch,k,heads,max_src,tgt,options", [
    (1, 4, 4, 40, 20, {}),                                           # persistent kernel: one short sequence
    (1, 4, 8, 100, 600, {}),                                         # one long
    (2, 4, 4, 40, 20, {}),                                           # several in one set of clusters
    (5, 4, 8, 40, 20, {}),                                           # groups
    (2, 4, 8, 40, 20, {"persistent_layers": 0}),                     # cluster launches
    (2, 4, 4, 40, 20, {"persistent_layers": 0, "cluster_layers": 0}),    # one kernel per projection, few rows
    (24, 4, 8, 97, 20, {}),                                          # many rows, layer-norm kernels in the encoder
    (24, 4, 8, 97, 20, {"fold_layer_norms": 1}),                     # and folded, several token tiles
    (9, 4, 16, 85, 20, {}),                                          # the most rows that are folded, eight tiles of statistics
    (3, 8, 3, 33, 20, {}),                                           # widths without folded layer norms
])
def test_fp32_paths_keep_their_precision(bpd, batch, k, heads, max_src, tgt, options, shift):
    import torch
    from bpd_inputs import ModelConfig, make_weights
    from bpd_inputs.blob import blob_layout
    from oracle.decode import TransformerScorer
    from oracle.model import parse_blob
    cfg = ModelConfig(2, 2, 64 * heads, heads, 128 * heads, 300, k, 64)
    blob = make_weights(cfg, 5, 0.06)
    for name, shape, _, off, nbytes in blob_layout(cfg)[0]:
        if name.endswith("self.wo"):
            blob[off:off + nbytes] = 0
        if name == "src_embed":
            t = torch.from_numpy(blob[off:off + nbytes].view(np.int16)).view(torch.bfloat16)
            t.copy_((t.float() + shift * 0.06).bfloat16())
    rng = np.random.default_rng(batch)
    lens = rng.integers(1, max_src + 1, batch).astype(np.int32)
    lens[-1] = max_src
    src = rng.integers(2, 300, (batch, max_src)).astype(np.int32)
    model = bpd.Model(blob)
    s = bpd.Session(model, batch, max_src, tgt, options=options)
    s.bpd_encode(src, lens)
    r = s.bpd_iteration(k, tgt, want_hidden=True)
    model_o = parse_blob(blob)
    for b in sorted({0, 1, batch - 1} & set(range(batch))):
        scorer = TransformerScorer(model_o, src[b], int(lens[b]), cached=True, capacity=tgt + k + 2)
        scorer([0], 1)
        scorer([0] + [int(t) for t in r["block"][b]], k)
        np.testing.assert_allclose(r["hidden"][b].cpu().numpy(), scorer.last_hidden, atol=1e-4)
    s.close()
    model.close()


# Cross-attention of the persistent kernel takes the encoder's rows in chunks of 8, one per warp: one row, a chunk's edges and
# the edges of a second round of the eight warps; rows staged for groups of sequences, for all sequences (as many as fit), and
# read out of L2; one CTA per SM and two (16 heads).  Tolerance as above (fp32 throughout, the same roundings on the way).
UNSTAGED = {"persistent_layers": 1, "stage_encoder_rows": 0}


@pytest.mark.parametrize("heads,lens,options", [
    (4, (1, 7, 8, 9, 63, 64, 65, 72), {}), (8, (1, 7, 8, 9, 63, 64, 65, 72), {}),
    (4, (63, 64, 72), {}), (8, (1, 7, 8, 9), {}), (8, (63, 64, 65), {}), (16, (1, 7, 8, 9), {}), (16, (63,), {}), (16, (64,), {}),
    (4, (1, 7, 8, 9, 63, 64, 65, 72), UNSTAGED), (8, (1, 7, 8, 9, 63, 64, 65, 72), UNSTAGED),
    (16, (1, 7, 8, 9), UNSTAGED), (16, (63, 64, 65, 72), UNSTAGED)])
def test_source_lengths_around_a_chunk_of_encoder_rows(bpd, heads, lens, options):
    from bpd_inputs import ModelConfig, make_weights
    from bpd_inputs.blob import blob_layout
    from oracle.decode import TransformerScorer
    from oracle.model import parse_blob
    cfg = ModelConfig(2, 2, 64 * heads, heads, 128 * heads, 300, 2, 64)
    blob = make_weights(cfg, 5, 0.06)
    for name, shape, _, off, nbytes in blob_layout(cfg)[0]:
        if name.endswith("self.wo"):
            blob[off:off + nbytes] = 0
    src = np.random.default_rng(heads).integers(2, 300, (len(lens), max(lens))).astype(np.int32)
    model = bpd.Model(blob)
    s = bpd.Session(model, len(lens), max(lens), 20, options=options)
    assert s.layer_path == 2
    s.bpd_encode(src, np.array(lens, np.int32))
    r = s.bpd_iteration(2, 20, want_hidden=True)
    model_o = parse_blob(blob)
    for b in range(len(lens)):
        scorer = TransformerScorer(model_o, src[b], lens[b], cached=True, capacity=24)
        scorer([0], 1)
        scorer([0] + [int(t) for t in r["block"][b]], 2)
        np.testing.assert_allclose(r["hidden"][b].cpu().numpy(), scorer.last_hidden, atol=1e-4)
    s.close()
    model.close()


# Every instantiation of the persistent kernel: width, hidden units per cluster, variant, token tiles.  First with the
# self-attention's output projections at zero, tolerance as above; then whole, over several blocks: a cached key or value is
# off by 2^-9 of itself.  Weights of 0.06 sqrt(256 / d) keep products at 0.96 of their input at every width, hence scores and
# attention outputs at a standard deviation of 0.9; a score is then off by 0.9 * 2^-9 and so is a weight, a value by 2^-9, an
# output by 0.9 * 1.9 * 2^-9 = 3.4e-3, and two layers add up to 6.7e-3.  (At 0.06 the 1024-wide model's scores have a
# deviation of 3.7: four times as much in the scores, four times in the outputs.)
@pytest.mark.parametrize("units", [128, 256])
@pytest.mark.parametrize("heads,batch,k,max_src,tgt,options", [
    (heads, *case) for heads in (4, 8) for case in [
        (2, 3, 20, 20, UNSTAGED), (3, 4, 20, 20, UNSTAGED), (2, 3, 20, 300, UNSTAGED), (2, 7, 20, 300, UNSTAGED),     # general, short and long
        (2, 4, 20, 20, {}), (2, 8, 112, 20, {}),                            # short; too many encoder rows for groups
        (1, 4, 20, 600, {}), (1, 10, 20, 600, {}), (1, 4, 20, 20, {}), (1, 10, 20, 20, {}),      # one long, one short sequence
        (5, 3, 20, 20, {}), (3, 10, 20, 20, {})]                            # groups
] + [(16, 2, 4, 20, 20, UNSTAGED), (16, 1, 2, 20, 300, {"persistent_layers": 1}), (16, 4, 2, 9, 20, {})])
def test_every_shape_of_the_persistent_kernel_scores_like_the_oracle(bpd, heads, batch, k, max_src, tgt, options, units):
    from bpd_inputs import ModelConfig, make_weights
    from bpd_inputs.blob import blob_layout
    from oracle.decode import TransformerScorer
    from oracle.model import parse_blob
    cfg = ModelConfig(1, 2, 64 * heads, heads, units * heads, 300, k, 64)
    rng = np.random.default_rng(batch * k)
    lens = rng.integers(1, max_src + 1, batch).astype(np.int32)
    lens[-1] = max_src
    src = rng.integers(2, 300, (batch, max_src)).astype(np.int32)
    blob = make_weights(cfg, 5, 0.06 * (4 / heads) ** 0.5)
    kept = blob.copy()
    for name, shape, _, off, nbytes in blob_layout(cfg)[0]:
        if name.endswith("self.wo"):
            blob[off:off + nbytes] = 0
    for weights, blocks, atol in ((blob, 1, 1e-4), (kept, 3, 8e-3)):
        model = bpd.Model(weights)
        s = bpd.Session(model, batch, max_src, tgt, options=options)
        no_room = units == 256 and (heads, batch, k, tgt) in ((8, 3, 10, 20), (16, 1, 2, 300))
        assert (s.layer_path == 2) != no_room
        s.bpd_encode(src, lens)
        model_o, rows = parse_blob(weights), sorted({0, batch - 1})
        scorers = {b: TransformerScorer(model_o, src[b], int(lens[b]), cached=True, capacity=tgt + k + 2) for b in rows}
        inputs = {b: [0] for b in rows}
        for b in rows:
            scorers[b](inputs[b], 1)
        for _ in range(blocks):
            r = s.bpd_iteration(k, tgt, want_hidden=True, accept_mode=k << 16)      # minimum block k: every proposal is kept
            for b in rows:
                block = [int(t) for t in r["block"][b]]
                scorers[b](inputs[b] + block, k)
                np.testing.assert_allclose(r["hidden"][b].cpu().numpy(), scorers[b].last_hidden, atol=atol)
                inputs[b] += block[:int(r["khat"][b])]
            if len(inputs[0]) > tgt:
                break
        s.close()
        model.close()


# the persistent layer kernel with groups of sequences: a last group that is full and one that is not, two sequences per
# group and one, one token tile and two, lengths up to the limit of 256 positions, one encoder row and the most (a
# multiple of 8) whose staging tile fits beside the working buffers of each shape: 136, 104 and 48
@pytest.mark.parametrize("batch,k,heads,max_src,tgt", [(3, 4, 4, 61, 30), (8, 4, 4, 9, 251), (5, 3, 8, 1, 20), (2, 10, 8, 33, 40), (4, 16, 8, 24, 48),
                                                       (9, 4, 4, 7, 12), (3, 4, 4, 136, 20), (5, 3, 8, 104, 20), (2, 10, 8, 48, 20)])
def test_groups_of_sequences_decode_like_the_oracle(bpd, batch, k, heads, max_src, tgt):
    from bpd_inputs import ModelConfig, make_weights
    from oracle.decode import TransformerScorer
    from oracle.model import parse_blob
    blob = make_weights(ModelConfig(1, 2, 64 * heads, heads, 128 * heads, 300, k, 64), 5, 0.06)
    rng = np.random.default_rng(batch * k)
    lens = rng.integers(1, max_src + 1, batch).astype(np.int32)
    lens[-1] = max_src
    src = rng.integers(2, 300, (batch, max_src)).astype(np.int32)
    model = bpd.Model(blob)
    s = bpd.Session(model, batch, max_src, tgt)
    assert s.layer_path == 2
    s.bpd_encode(src, lens)
    model_o, rows = parse_blob(blob), sorted({0, 1, batch - 1})
    scorers = {b: TransformerScorer(model_o, src[b], int(lens[b]), cached=True, capacity=tgt + k + 2) for b in rows}
    inputs = {b: [0] for b in rows}
    for b in rows:
        scorers[b](inputs[b], 1)
    while len(inputs[0]) <= tgt:
        r = s.bpd_iteration(k, tgt, want_hidden=True, accept_mode=k << 16)      # minimum block k: every proposal is kept
        for b in rows:
            block = [int(t) for t in r["block"][b]]
            scorers[b](inputs[b] + block, k)
            np.testing.assert_allclose(r["hidden"][b].cpu().numpy(), scorers[b].last_hidden, atol=8e-3)     # the cache is bf16
            inputs[b] += block[:int(r["khat"][b])]
    s.close()
    model.close()
