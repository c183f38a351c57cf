"""End-to-end parity of the translation path (C ABI, sm_103a kernels) against the
CPU oracle: identical token sequences, lengths and beam scores, and bit-exact
intermediate taps (encoder output, cross-attention keys/values, self-attention
cache, decoder output), on the seeded synthetic workloads at full size (sampled
sentences where the oracle is slow) and on small models that span the
configuration space (pre/post-LN, factorised/tied embedding, greedy/beam)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2306_04235_gb300 import mnmt, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MINI = {
    "odd": synth.ModelConfig(2, 2, 192, 3, 384, 300, 192, 1, 1, max_pos=64),   # d = 3 x 64: 4-CTA cluster step
    "pre": synth.ModelConfig(2, 2, 64, 2, 128, 300, 64, 1, 1, max_pos=64),
    "post": synth.ModelConfig(2, 1, 64, 1, 128, 300, 64, 0, 1, max_pos=64),
    "fact": synth.ModelConfig(3, 2, 128, 4, 256, 500, 32, 1, 0, max_pos=96),
    "wide-head": synth.ModelConfig(1, 2, 256, 2, 256, 400, 256, 1, 1, max_pos=64),
}


@pytest.fixture(scope="module")
def stream():
    return torch.cuda.Stream()


def _gpu(blob, ids, lens, beam, max_len, stream, max_batch=None, max_src=None):
    tr = mnmt.Translator(blob, max_batch or ids.shape[0], max_src or ids.shape[1], beam, max_len, stream)
    try:
        out = tr.translate(ids, lens, max_len)
    finally:
        tr.close()
    return out


@pytest.mark.parametrize("kind", list(MINI))
@pytest.mark.parametrize("beam", [1, 3])
def test_small_models_match_oracle(kind, beam, stream):
    cfg = MINI[kind]
    blob = synth.build_blob(cfg, 21, gamma_range=(0.5, 1.5))
    ids, lens = synth.source_batch(cfg.vocab, 5, 1, 40, 22)
    T = 24
    g_ids, g_len, g_sc = _gpu(blob, ids, lens, beam, T, stream)
    o_ids, o_len, o_sc = O.translate(blob, ids, lens, beam, T, n_threads=5)
    assert np.array_equal(g_ids, o_ids)
    assert np.array_equal(g_len, o_len)
    assert np.array_equal(g_sc.view(np.uint32), o_sc.view(np.uint32))


@pytest.mark.parametrize("kind,beam", [("fact", 4), ("pre", 3)])
def test_many_sentences_beam_search_matches_oracle(kind, beam, stream):
    """80 sentences: enough that the cross attention serves all beams of a
    sentence from one block (the batched-beam layout)."""
    cfg = MINI[kind]
    blob = synth.build_blob(cfg, 31, gamma_range=(0.5, 1.5))
    ids, lens = synth.source_batch(cfg.vocab, 80, 1, 30, 32)
    T = 12
    g_ids, g_len, g_sc = _gpu(blob, ids, lens, beam, T, stream)
    o_ids, o_len, o_sc = O.translate(blob, ids, lens, beam, T, n_threads=8)
    assert np.array_equal(g_ids, o_ids)
    assert np.array_equal(g_len, o_len)
    assert np.array_equal(g_sc.view(np.uint32), o_sc.view(np.uint32))


def test_tiny_workload_tokens_and_taps(stream):
    cfg, blob, ids, lens, beam, T = synth.workload_inputs("tiny-b1-s16-greedy16")
    d, H, L = cfg.d_model, cfg.n_heads, cfg.n_dec
    dh = d // H
    tr = mnmt.Translator(blob, 1, ids.shape[1], beam, T, stream)
    try:
        out, olen, _ = tr.translate(ids, lens, T)
        S = ids.shape[1]
        enc = mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_ENC_OUT, 0, np.int8, (1, S, d))
        ck = [mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_CROSS_K, l, np.int8, (1, H, S, dh)) for l in range(L)]
        cv = [mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_CROSS_V, l, np.int8, (1, H, S, dh)) for l in range(L)]
        sk = [mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_SELF_K, l, np.int8, (1, H, T, dh)) for l in range(L)]
        sv = [mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_SELF_V, l, np.int8, (1, H, T, dh)) for l in range(L)]
        dec = mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_DEC_OUT, 0, np.int8, (1, d))
    finally:
        tr.close()
    ref, rlen, _ = O.translate(blob, ids, lens, beam, T)
    assert np.array_equal(out, ref) and np.array_equal(olen, rlen)
    e_q, e_k, e_v = O.encode(blob, ids[0], lens[0], cfg)
    assert np.array_equal(enc[0], e_q)
    for l in range(L):
        assert np.array_equal(ck[l][0].transpose(1, 0, 2).reshape(S, d), e_k[l])
        assert np.array_equal(cv[l][0].transpose(1, 0, 2).reshape(S, d), e_v[l])
    n = int(olen[0])
    tgt = np.concatenate([[cfg.bos_id], out[0, :n - 1]]).astype(np.int32)
    logits, dec_q, self_k, self_v = O.decode_trace(blob, ids[0], lens[0], tgt, cfg, want_cache=True)
    assert np.array_equal(dec, dec_q[n - 1:n])
    for l in range(L):
        assert np.array_equal(sk[l][0, :, :n].transpose(1, 0, 2).reshape(n, d), self_k[l])
        assert np.array_equal(sv[l][0, :, :n].transpose(1, 0, 2).reshape(n, d), self_v[l])


def test_small_batch1_workload_matches_oracle(stream):
    cfg, blob, ids, lens, beam, T = synth.workload_inputs("small-b1-s10to50-greedy64")
    g = _gpu(blob, ids, lens, beam, T, stream)
    o = O.translate(blob, ids, lens, beam, T)
    assert np.array_equal(g[0], o[0]) and np.array_equal(g[1], o[1])


def test_paper_shape_src30_tgt30(stream):
    cfg, blob, ids, lens, beam, T = synth.workload_inputs("small-b1-s30-greedy30")
    g = _gpu(blob, ids, lens, beam, T, stream)
    o = O.translate(blob, ids, lens, beam, T)
    assert np.array_equal(g[0], o[0]) and np.array_equal(g[1], o[1])


def test_small_batched_beam_workload_sampled(stream):
    """Batch 32, beam 4, 128 steps at full size; the oracle checks 4 sentences."""
    cfg, blob, ids, lens, beam, T = synth.workload_inputs("small-b32-s10to80-beam4-t128")
    g_ids, g_len, g_sc = _gpu(blob, ids, lens, beam, T, stream)
    pick = [0, 9, 17, 31]
    o_ids, o_len, o_sc = O.translate(blob, ids[pick], lens[pick], beam, T, n_threads=4)
    assert np.array_equal(g_ids[pick], o_ids)
    assert np.array_equal(g_len[pick], o_len)
    assert np.array_equal(g_sc[pick].view(np.uint32), o_sc.view(np.uint32))


def test_wide_batched_beam_workload_sampled(stream):
    """Batch 128, beam 4, 160 steps at full size; the oracle checks 2 sentences."""
    cfg, blob, ids, lens, beam, T = synth.workload_inputs("wide-b128-s20to128-beam4-t160")
    g_ids, g_len, g_sc = _gpu(blob, ids, lens, beam, T, stream)
    pick = [5, 127]
    o_ids, o_len, o_sc = O.translate(blob, ids[pick], lens[pick], beam, T, n_threads=2)
    assert np.array_equal(g_ids[pick], o_ids)
    assert np.array_equal(g_len[pick], o_len)
    assert np.array_equal(g_sc[pick].view(np.uint32), o_sc.view(np.uint32))


def test_longest_source(stream):
    cfg = synth.MODELS["small-12x2-d256-v32k-e128"]
    blob = synth.build_blob(cfg, 1)
    ids, lens = synth.source_batch(cfg.vocab, 2, 500, 512, 33)
    ids = np.pad(ids, ((0, 0), (0, 512 - ids.shape[1])))
    g = _gpu(blob, ids, lens, 1, 6, stream)
    o = O.translate(blob, ids, lens, 1, 6, n_threads=2)
    assert np.array_equal(g[0], o[0])


@pytest.mark.parametrize("beam", [1, 4])
def test_forced_eos_stops_at_once(beam, stream):
    cfg = MINI["pre"]
    blob = synth.build_blob(cfg, 3, out_bias={cfg.eos_id: 1000.0})
    ids, lens = synth.source_batch(cfg.vocab, 3, 2, 9, 4)
    g_ids, g_len, _ = _gpu(blob, ids, lens, beam, 20, stream)
    assert np.all(g_len == 1) and np.all(g_ids[:, 0] == cfg.eos_id) and np.all(g_ids[:, 1:] == cfg.pad_id)


@pytest.mark.parametrize("kind", list(MINI))
@pytest.mark.parametrize("batch", [1, 3])
def test_cluster_step_models_match_oracle(kind, batch, stream):
    """Every small model shape (pre- and post-LN, factorised and plain
    embedding, tied and untied output, d_h 64 and 128, d = 3 x 64) through
    the single-cluster step: greedy batches of at most 4 rows."""
    cfg = MINI[kind]
    blob = synth.build_blob(cfg, 41, gamma_range=(0.5, 1.5))
    ids, lens = synth.source_batch(cfg.vocab, batch, 1, 40, 42)
    T = 24
    tr = mnmt.Translator(blob, batch, ids.shape[1], 1, T, stream)
    try:
        g_ids, g_len, g_sc = tr.translate(ids, lens, T)
        assert mnmt.mnmt_session_decode_path(tr.session) == 1
    finally:
        tr.close()
    o_ids, o_len, o_sc = O.translate(blob, ids, lens, 1, T, n_threads=3)
    assert np.array_equal(g_ids, o_ids)
    assert np.array_equal(g_len, o_len)
    assert np.array_equal(g_sc.view(np.uint32), o_sc.view(np.uint32))


@pytest.mark.parametrize("seed,bias,rows,lengths", [
    (3, 0.15, None, [23, 1, 40, 40]),
    (3, 0.2, None, [1, 1, 16, 40]),   # one sentence ends on a 16-step graph boundary
    (5, 0.28, None, [1, 1, 24, 40]),
    (3, 0.1, 0, [31]),
    (3, 0.2, 2, [16]),
])
def test_cluster_step_mixed_lengths_match_oracle(seed, bias, rows, lengths, stream):
    """The single-cluster step (greedy, <= 4 rows) with sentences that finish
    at different steps, inside and at the end of a captured run of 16 steps:
    the greedy selection left pending by the vocabulary kernel is applied by
    the next step kernel or by the greedy update that closes the run."""
    cfg = MINI["pre"]
    blob = synth.build_blob(cfg, seed, out_bias={cfg.eos_id: bias})
    ids, lens = synth.source_batch(cfg.vocab, 4, 2, 30, 4)
    if rows is not None:
        ids, lens = ids[rows:rows + 1], lens[rows:rows + 1]
    T = 40
    tr = mnmt.Translator(blob, ids.shape[0], ids.shape[1], 1, T, stream)
    try:
        g_ids, g_len, g_sc = tr.translate(ids, lens, T)
        assert mnmt.mnmt_session_decode_path(tr.session) == 1
    finally:
        tr.close()
    o_ids, o_len, o_sc = O.translate(blob, ids, lens, 1, T, n_threads=4)
    assert o_len.tolist() == lengths
    assert np.array_equal(g_ids, o_ids)
    assert np.array_equal(g_len, o_len)
    assert np.array_equal(g_sc.view(np.uint32), o_sc.view(np.uint32))


@pytest.mark.parametrize("beam", [1, 3])
def test_decode_step_api_matches_translate(beam, stream):
    cfg = MINI["fact"]
    blob = synth.build_blob(cfg, 8)
    ids, lens = synth.source_batch(cfg.vocab, 2, 3, 20, 9)
    T = 12
    o_ids, o_len, o_sc = O.translate(blob, ids, lens, beam, T, n_threads=2)
    tr = mnmt.Translator(blob, 2, ids.shape[1], beam, T, stream)
    try:
        mnmt.mnmt_encode(tr.session, ids, lens, 2, ids.shape[1])
        toks, pars = [], []
        for t in range(T):
            tok, par, sc, done = mnmt.mnmt_decode_step(tr.session, 2 * beam)
            toks.append(tok); pars.append(par)
            if done:
                break
        with pytest.raises(mnmt.MnmtError):
            for _ in range(T + 1):
                mnmt.mnmt_decode_step(tr.session, 2 * beam)
    finally:
        tr.close()
    # backtrack beam 0 of each sentence through the parents
    for b in range(2):
        r = 0
        seq = []
        for t in range(len(toks) - 1, -1, -1):
            seq.append(toks[t][b * beam + r])
            r = pars[t][b * beam + r] if beam > 1 else 0
        seq = seq[::-1]
        n = int(o_len[b])
        assert seq[:n] == list(o_ids[b, :n])


@pytest.mark.parametrize("beam", [1, 3])
def test_queued_decode_steps_match_stepwise_decode(beam, stream):
    """mnmt_decode_steps queues steps without host round trips: the token and
    parent history equals the one of step-by-step decoding, and steps past the
    length limit are not queued."""
    cfg = MINI["fact"]
    blob = synth.build_blob(cfg, 8)
    ids, lens = synth.source_batch(cfg.vocab, 2, 3, 20, 9)
    T, R = 12, 2 * beam
    tr = mnmt.Translator(blob, 2, ids.shape[1], beam, T, stream)
    try:
        mnmt.mnmt_encode(tr.session, ids, lens, 2, ids.shape[1])
        steps = [mnmt.mnmt_decode_step(tr.session, R) for _ in range(T)]
        mnmt.mnmt_encode(tr.session, ids, lens, 2, ids.shape[1])
        assert mnmt.mnmt_decode_steps(tr.session, 5) == 5
        assert mnmt.mnmt_decode_steps(tr.session, 100) == T - 5
        assert mnmt.mnmt_decode_steps(tr.session, 1) == 0
        hist = mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_HISTORY, 0, np.int32, (T, R))
        par = mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_PARENTS, 0, np.int32, (T, R))
    finally:
        tr.close()
    assert np.array_equal(hist, np.stack([s[0] for s in steps]))
    if beam > 1:
        assert np.array_equal(par, np.stack([s[1] for s in steps]))


def test_cluster_step_graph_serves_changing_source_lengths(stream):
    """One session translating sentences of different padded lengths in turn
    (the cluster step keeps its captured graph and only updates the length)."""
    cfg, blob, _, _, beam, T = synth.workload_inputs("small-b1-s10to50-greedy64")
    tr = mnmt.Translator(blob, 1, 50, 1, T, stream)
    try:
        for i, S in enumerate([37, 12, 50, 12, 29]):
            ids, lens = synth.source_batch(cfg.vocab, 1, S, S, 70 + i)
            g_ids, g_len, _ = tr.translate(ids, lens, T)
            assert mnmt.mnmt_session_decode_path(tr.session) == 1
            o_ids, o_len, _ = O.translate(blob, ids, lens, 1, T, n_threads=1)
            assert np.array_equal(g_ids, o_ids) and np.array_equal(g_len, o_len), S
    finally:
        tr.close()


def test_device_pointer_path_equals_host_path(stream):
    cfg = MINI["pre"]
    blob = synth.build_blob(cfg, 5)
    ids, lens = synth.source_batch(cfg.vocab, 4, 2, 30, 6)
    T = 16
    tr = mnmt.Translator(blob, 4, ids.shape[1], 2, T, stream)
    try:
        h = tr.translate(ids, lens, T)
        d_ids, d_lens = torch.from_numpy(ids).cuda(), torch.from_numpy(lens).cuda()
        o_ids = torch.zeros((4, T), dtype=torch.int32, device="cuda")
        o_len = torch.zeros(4, dtype=torch.int32, device="cuda")
        o_sc = torch.zeros(4, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        mnmt.mnmt_translate(tr.session, d_ids, d_lens, 4, ids.shape[1], T, mnmt.DEVICE_PTRS, o_ids, o_len, o_sc)
        stream.synchronize()
        assert np.array_equal(o_ids.cpu().numpy(), h[0]) and np.array_equal(o_len.cpu().numpy(), h[1])
        assert np.array_equal(o_sc.cpu().numpy(), h[2])
    finally:
        tr.close()


def test_bad_inputs_are_rejected(stream):
    cfg = MINI["pre"]
    blob = synth.build_blob(cfg, 5)
    tr = mnmt.Translator(blob, 2, 10, 1, 8, stream)
    try:
        ids = np.full((2, 10), 5, np.int32)
        with pytest.raises(mnmt.MnmtError) as ei:
            tr.translate(ids, np.array([3, 11], np.int32), 8)       # length beyond S_pad
        assert ei.value.code == mnmt.EINVAL
        bad = ids.copy(); bad[1, 2] = cfg.vocab
        with pytest.raises(mnmt.MnmtError):
            tr.translate(bad, np.array([3, 4], np.int32), 8)         # id outside the vocabulary
        with pytest.raises(mnmt.MnmtError):
            tr.translate(np.full((3, 10), 5, np.int32), np.array([3, 4, 5], np.int32), 8)  # batch > capacity
        out = tr.translate(ids, np.array([3, 4], np.int32), 8)      # session still usable
        assert out[0].shape == (2, 8)
    finally:
        tr.close()


def _with_path(cluster: bool):
    import os
    if cluster:
        os.environ.pop("MNMT_DECODE_CLUSTER", None)
    else:
        os.environ["MNMT_DECODE_CLUSTER"] = "0"


@pytest.mark.parametrize("kind", list(MINI))
@pytest.mark.parametrize("B", [1, 3, 4])
def test_cluster_decode_step_matches_oracle(kind, B, stream):
    """Greedy batches of <= 4 sentences run the single-cluster decode step."""
    cfg = MINI[kind]
    blob = synth.build_blob(cfg, 31, gamma_range=(0.5, 1.5))
    ids, lens = synth.source_batch(cfg.vocab, B, 1, 40, 32)
    T = 24
    _with_path(True)
    tr = mnmt.Translator(blob, B, ids.shape[1], 1, T, stream)
    try:
        g_ids, g_len, _ = tr.translate(ids, lens, T)
        assert mnmt.mnmt_session_decode_path(tr.session) == 1
    finally:
        tr.close()
    o_ids, o_len, _ = O.translate(blob, ids, lens, 1, T, n_threads=B)
    assert np.array_equal(g_ids, o_ids) and np.array_equal(g_len, o_len)


@pytest.mark.parametrize("name", ["tiny-b1-s16-greedy16", "small-b1-s10to50-greedy64"])
def test_cluster_and_kernel_paths_bit_identical(name, stream):
    cfg, blob, ids, lens, beam, T = synth.workload_inputs(name)
    d, H, L = cfg.d_model, cfg.n_heads, cfg.n_dec
    dh = d // H
    res = {}
    for cluster in (True, False):
        _with_path(cluster)
        tr = mnmt.Translator(blob, 1, ids.shape[1], beam, T, stream)
        try:
            out = tr.translate(ids, lens, T)
            assert mnmt.mnmt_session_decode_path(tr.session) == int(cluster)
            taps = [mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_DEC_OUT, 0, np.int8),
                    mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_RESID, 0, np.float32)]
            for l in range(L):
                taps.append(mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_SELF_K, l, np.int8))
                taps.append(mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_SELF_V, l, np.int8))
            res[cluster] = (out, taps)
        finally:
            tr.close()
    _with_path(True)
    (o1, t1), (o0, t0) = res[True], res[False]
    assert np.array_equal(o1[0], o0[0]) and np.array_equal(o1[1], o0[1])
    for a, b in zip(t1, t0):
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
    ref = O.translate(blob, ids, lens, beam, T)
    assert np.array_equal(o1[0], ref[0])


def test_bench_workload_uses_cluster_step(stream):
    cfg, blob, ids, lens, beam, T = synth.workload_inputs("small-b1-s10to50-greedy64")
    _with_path(True)
    tr = mnmt.Translator(blob, 1, ids.shape[1], beam, T, stream)
    try:
        mnmt.mnmt_encode(tr.session, ids, lens, 1, ids.shape[1])
        assert mnmt.mnmt_session_decode_path(tr.session) == 1
    finally:
        tr.close()


def _with_tc(on: bool):
    import os
    if on:
        os.environ.pop("MNMT_TC", None)
    else:
        os.environ["MNMT_TC"] = "0"


@pytest.mark.parametrize("kind", list(MINI))
@pytest.mark.parametrize("beam", [1, 4])
def test_tensor_core_rows_match_oracle(kind, beam, stream):
    """Batches of >= 128 decoder rows (and encoder rows) run their linears on
    the tcgen05 kernel: tokens, lengths and scores still equal the oracle's."""
    cfg = MINI[kind]
    blob = synth.build_blob(cfg, 41, gamma_range=(0.5, 1.5))
    B = 160 // beam
    ids, lens = synth.source_batch(cfg.vocab, B, 1, 40, 42)
    T = 20
    _with_tc(True)
    g_ids, g_len, g_sc = _gpu(blob, ids, lens, beam, T, stream)
    o_ids, o_len, o_sc = O.translate(blob, ids, lens, beam, T, n_threads=8)
    assert np.array_equal(g_ids, o_ids)
    assert np.array_equal(g_len, o_len)
    assert np.array_equal(g_sc.view(np.uint32), o_sc.view(np.uint32))


def test_tensor_core_and_imma_paths_bit_identical(stream):
    """The same batched beam workload through the tcgen05 linears and through
    the int8 linears (MNMT_TC=0): identical outputs."""
    cfg, blob, ids, lens, beam, T = synth.workload_inputs("small-b32-s10to80-beam4-t128")
    outs = []
    for on in (True, False):
        _with_tc(on)
        try:
            outs.append(_gpu(blob, ids, lens, beam, T, stream))
        finally:
            _with_tc(True)
    for a, b in zip(*outs):
        assert np.array_equal(a.view(np.uint32) if a.dtype == np.float32 else a,
                              b.view(np.uint32) if b.dtype == np.float32 else b)


@pytest.mark.parametrize("d,H,F,n_dec,beam,B,wq,step", [
    (128, 2, 128, 1, 1, 5, synth.WQ_INT8, [2, 8, 1, 1]),       # 64 FFN columns per CTA, two CTAs, one ragged cluster
    (128, 2, 512, 2, 3, 3, synth.WQ_INT8, [2, 8, 1, 2]),       # sentences straddling warps; 256 columns
    (256, 4, 768, 2, 5, 7, synth.WQ_INT4, [2, 8, 1, 5]),       # 192 columns, 4-bit rows, 5 beams over 4-row chunks
    (384, 6, 768, 1, 4, 9, synth.WQ_INT8, [2, 8, 1, 5]),       # odd factor of d, owned rows of unequal number
    (384, 6, 384, 1, 1, 40, synth.WQ_INT8, [2, 8, 1, 5]),
    (512, 8, 2048, 2, 2, 13, synth.WQ_INT8, [2, 8, 1, 4]),     # K = 2048
    (512, 8, 2048, 1, 4, 33, synth.WQ_INT8, [2, 16, 1, 9]),    # 16 rows per cluster
    (512, 8, 1536, 1, 4, 100, synth.WQ_INT8, [2, 32, 1, 13]),  # 32 rows per cluster
    (512, 8, 2048, 1, 4, 128, synth.WQ_INT8, [2, 16, 2, 32]),  # two heads per CTA, 16 rows
    (512, 8, 1024, 1, 4, 144, synth.WQ_INT8, [2, 16, 2, 36]),  # as many clusters as are resident at once
    (512, 8, 1024, 1, 4, 150, synth.WQ_INT8, [0, 0, 0, 0]),    # more: a kernel per operation
    (512, 8, 1024, 1, 1, 250, synth.WQ_INT8, [0, 0, 0, 0]),    # 32 rows without beams: the same
])
def test_batched_cluster_step_equals_kernel_per_operation(d, H, F, n_dec, beam, B, wq, step, stream, monkeypatch):
    """The batched decode step, in the form named, against the oracle and against
    the kernel-per-operation step, bit for bit: tokens, scores, the last decoder
    output, residual and self cache, over steps that cross a 16-key block, and
    again after the padded source length changes (the captured steps are kept)."""
    cfg = synth.ModelConfig(1, n_dec, d, H, F, 300, d, 1, 1, max_pos=64)
    blob = synth.build_blob(cfg, 91, gamma_range=(0.5, 1.5), wq=wq)
    T, out = 20, {}
    for env in ("1", "0"):
        monkeypatch.setenv("MNMT_DECODE_CLUSTER", env)
        tr = mnmt.Translator(blob, B, 33, beam, T, stream)
        try:
            res = []
            for S, seed in ((33, 5), (18, 6)):
                ids, lens = synth.source_batch(cfg.vocab, B, 1, S, seed)
                ids = np.pad(ids, ((0, 0), (0, S - ids.shape[1])))
                res += list(tr.translate(ids, lens, T))
                assert mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_STEP, 0, np.int32).tolist() == (step if env == "1" else [0] * 4)
                res += [mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_DEC_OUT), mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_RESID, 0, np.uint32),
                        mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_SELF_K, n_dec - 1), mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_SELF_V, 0)]
            out[env] = res
        finally:
            tr.close()
    for a, b in zip(out["1"], out["0"]):
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
    o_ids, o_len, o_sc = O.translate(blob, ids, lens, beam, T, n_threads=16)  # of the second batch
    g_ids, g_len, g_sc = out["1"][7:10]
    assert np.array_equal(g_ids, o_ids) and np.array_equal(g_len, o_len)
    assert np.array_equal(g_sc.view(np.uint32), o_sc.view(np.uint32))


@pytest.mark.parametrize("beam,B,n_dec", [(1, 240, 2), (4, 65, 1), (3, 23, 4)])
def test_batched_cluster_step_with_caches_beyond_l2(beam, B, n_dec, stream, monkeypatch):
    """Sessions whose caches exceed L2 bring a layer's to it ahead of its
    attention: the first step (no own keys yet), sentences of one token, beams
    that straddle clusters, against the kernel-per-operation step."""
    T = 500
    cfg = synth.ModelConfig(1, n_dec, 512, 8, 512, 300, 512, 1, 1, max_pos=512)
    assert (B * beam * T + B * 33) * 2 * 512 * n_dec > 128e6
    blob = synth.build_blob(cfg, 93, gamma_range=(0.5, 1.5))
    ids, lens = synth.source_batch(cfg.vocab, B, 1, 33, 7)
    ids = np.pad(ids, ((0, 0), (0, 33 - ids.shape[1])))
    out = {}
    for env in ("1", "0"):
        monkeypatch.setenv("MNMT_DECODE_CLUSTER", env)
        tr = mnmt.Translator(blob, B, 33, beam, T, stream)
        try:
            out[env] = list(tr.translate(ids, lens, 20)) + [mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_DEC_OUT)]
            assert mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_STEP, 0, np.int32)[0] == (2 if env == "1" else 0)
        finally:
            tr.close()
    for a, b in zip(out["1"], out["0"]):
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))


@pytest.mark.parametrize("V,beam", [(4096, 4), (8192, 2), (8196, 4), (20000, 3), (32768, 5), (5000, 16), (32764, 8)])
@pytest.mark.parametrize("flat", [False, True])
def test_beam_rows_in_registers(V, beam, flat, stream):
    """The beam step that keeps a row's logits in registers: its vocabulary
    limits, every list size, beams that share a 32-byte sector of candidates;
    flat: an output bias that makes hundreds of logits tie (the candidate list
    overflows and the row is scanned in full), with EOS among the first."""
    cfg = synth.ModelConfig(1, 1, 64, 1, 64, V, 64, 1, 1, max_pos=32)
    bias = {i: 40.0 for i in range(0, 900)} if flat else None
    blob = synth.build_blob(cfg, 17, gamma_range=(0.5, 1.5), out_bias=bias)
    if flat:  # equal logits: the tied embedding rows of the biased ids zeroed
        off = 64
        b = bytearray(blob)
        b[off: off + 900 * 64] = bytes(900 * 64)
        blob = bytes(b)
    ids, lens = synth.source_batch(V, 5, 3, 9, 8)
    T = 7
    tr = mnmt.Translator(blob, 5, ids.shape[1], beam, T, stream)
    try:
        g_ids, g_len, g_sc = tr.translate(ids, lens, T)
    finally:
        tr.close()
    o_ids, o_len, o_sc = O.translate(blob, ids, lens, beam, T)
    assert np.array_equal(g_ids, o_ids) and np.array_equal(g_len, o_len)
    assert np.array_equal(g_sc.view(np.uint32), o_sc.view(np.uint32))


@pytest.mark.parametrize("V,beam,B,lo", [(4096, 4, 39, 0), (8192, 5, 31, 0), (8196, 8, 20, 7296), (20000, 16, 10, 19100),
                                         (32764, 4, 39, 31864), (32768, 3, 51, 15934), (32768, 4, 39, 0)])
@pytest.mark.parametrize("flat", [False, True])
def test_beam_rows_two_to_an_sm(V, beam, B, lo, flat, stream):
    """More rows than SMs: blocks of 512 threads, above 8192 entries those from
    16384 on in shared memory; flat: 900 equal logits from id lo on, in either half
    or across both (the list overflows and the row is scanned in full)."""
    cfg = synth.ModelConfig(1, 1, 64, 1, 64, V, 64, 1, 1, max_pos=32)
    bias = {lo + i: 40.0 for i in range(0, 900)} if flat else None
    blob = synth.build_blob(cfg, 19, gamma_range=(0.5, 1.5), out_bias=bias)
    if flat:  # equal logits: the tied embedding rows of the biased ids zeroed
        b = bytearray(blob)
        b[64 + lo * 64: 64 + (lo + 900) * 64] = bytes(900 * 64)
        blob = bytes(b)
    ids, lens = synth.source_batch(V, B, 3, 9, 8)
    T = 5
    tr = mnmt.Translator(blob, B, ids.shape[1], beam, T, stream)
    try:
        g_ids, g_len, g_sc = tr.translate(ids, lens, T)
    finally:
        tr.close()
    o_ids, o_len, o_sc = O.translate(blob, ids, lens, beam, T, n_threads=4)
    assert np.array_equal(g_ids, o_ids) and np.array_equal(g_len, o_len)
    assert np.array_equal(g_sc.view(np.uint32), o_sc.view(np.uint32))


@pytest.mark.parametrize("B,beam,S,cluster", [(2, 1, 9, "1"), (1, 1, 9, "1"), (6, 2, 9, "1"), (3, 4, 9, "0"), (100, 1, 9, "1"), (12, 1, 33, "0")])
def test_infinite_attention_scale(B, beam, S, cluster, stream, monkeypatch):
    """Query and key scales whose product overflows: the codes are all zero, the
    scores 0 * inf, no key has a weight, and every context is the code of 0 -- as
    with large finite scales and zero value codes.  Both encoder attentions, the
    single-cluster, the batched and the kernel-per-operation step."""
    cfg = synth.ModelConfig(1, 2, 128, 2, 256, 300, 128, 1, 1, max_pos=64)
    blob = synth.build_blob(cfg, 23, gamma_range=(0.5, 1.5), cross_gains=synth.NO_GAINS)
    lin = np.float32(synth.activation_scales(cfg)["lin"])

    def scaled(s_qk, s_v):  # every attention block's {s_in, s_q, s_k, s_v, s_ctx, gamma, 0, 0}
        f = np.frombuffer(blob, np.float32).copy()
        at = [i for i in np.nonzero(f[:-8] == lin)[0] if (f[i: i + 4] == lin).all() and not f[i + 5: i + 7].any()]
        assert len(at) == cfg.n_enc + 2 * cfg.n_dec
        for i in at:
            f[i: i + 2], f[i + 2] = s_qk, s_v
        return f.tobytes()

    blobs = {"finite": scaled(1e15, 1e15), "infinite": scaled(1e30, lin)}
    monkeypatch.setenv("MNMT_DECODE_CLUSTER", cluster)
    ids, lens = synth.source_batch(cfg.vocab, B, max(1, S // 2), S, 8)
    ids = np.pad(ids, ((0, 0), (0, S - ids.shape[1])))
    T, out = 6, {}
    for name, b in blobs.items():
        tr = mnmt.Translator(b, B, S, beam, T, stream)
        try:
            out[name] = list(tr.translate(ids, lens, T)) + [mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_ENC_OUT), mnmt.mnmt_debug_tap(tr.session, mnmt.TAP_DEC_OUT)]
        finally:
            tr.close()
    o_ids, o_len, o_sc = O.translate(blobs["finite"], ids, lens, beam, T)
    assert np.array_equal(out["finite"][0], o_ids) and np.array_equal(out["finite"][2].view(np.uint32), o_sc.view(np.uint32))
    for a, b in zip(out["finite"], out["infinite"]):
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))


@pytest.mark.parametrize("beam,B", [(1, 3), (1, 9), (3, 4)])
def test_queued_translations_keep_their_step_limits(beam, B, stream):
    """Two device-pointer translations queued on one session while the stream is
    busy: each runs to its own max_len (the second call's must not reach the
    first), as when they run one after the other."""
    cfg = MINI["fact"]
    tr = mnmt.Translator(synth.build_blob(cfg, 41, gamma_range=(0.5, 1.5)), B, 12, beam, 8, stream)
    try:
        ids, lens = synth.source_batch(cfg.vocab, B, 3, 12, 42)
        ids = np.pad(ids, ((0, 0), (0, 12 - ids.shape[1])))
        refs = [tr.translate(ids, lens, T) for T in (8, 3)]
        d_ids, d_lens = torch.from_numpy(ids).cuda(), torch.from_numpy(lens).cuda()
        outs = [(torch.zeros((B, T), dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda"),
                 torch.zeros(B, device="cuda")) for T in (8, 3)]
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            torch.cuda._sleep(100_000_000)
        for T, o in zip((8, 3), outs):
            mnmt.mnmt_translate(tr.session, d_ids, d_lens, B, 12, T, mnmt.DEVICE_PTRS, *o)
        torch.cuda.synchronize()
        for ref, out in zip(refs, outs):
            for a, b in zip(ref, out):
                assert np.array_equal(a.view(np.uint32), b.cpu().numpy().view(np.uint32))
    finally:
        tr.close()


def test_session_holds_packed_weights_only_where_the_batched_step_can_run(stream, monkeypatch):
    """Lengths above 512, or the step switched off when the session is created:
    no packed decoder weights in the session (and a kernel per operation)."""
    cfg = synth.ModelConfig(1, 2, 256, 4, 1024, 300, 256, 1, 1, max_pos=600)
    packed = cfg.n_dec * (6 * 256 * 256 + 2 * 256 * 1024)
    model = mnmt.mnmt_load_weights(synth.build_blob(cfg, 3), stream)
    ids, lens = synth.source_batch(cfg.vocab, 4, 8, 8, 4)

    def session(T):
        s = mnmt.mnmt_session_create(model, 4, 8, 4, T)
        try:
            mnmt.mnmt_encode(s, ids, lens, 4, ids.shape[1])
            return mnmt.mnmt_session_device_bytes(s), int(mnmt.mnmt_debug_tap(s, mnmt.TAP_STEP, 0, np.int32)[0])
        finally:
            mnmt.mnmt_session_free(s)

    try:
        monkeypatch.setenv("MNMT_DECODE_CLUSTER", "1")
        (with_, kind), (long_, kind_long) = session(512), session(513)
        monkeypatch.setenv("MNMT_DECODE_CLUSTER", "0")
        off, kind_off = session(512)
    finally:
        mnmt.mnmt_model_free(model)
    assert (kind, kind_long, kind_off) == (2, 0, 0)
    assert with_ - off >= packed and with_ - long_ > 0.9 * packed
