"""Sizes at the edges of the kernels' partitions and dispatch rules, against the CPU oracle (needs a B200)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_2608_04991_b200 import binding as rac
    from paper_2608_04991_b200 import synth
    import parity
    rac.load()
    oracle.lib()
    return type("Env", (), dict(orc=oracle, rac=rac, synth=synth, P=parity, dev=torch.device("cuda:0")))


# ------------------------------------------------------------------------------- statistics passes, 1024 channels per warp
@pytest.mark.parametrize("d,g,T", [(32, 32, 1), (1024, 1024, 7), (1056, 32, 9), (2880, 64, 17), (8192, 256, 1025),
                                   (5120, 128, 480)])
def test_statistics_passes_at_partition_edges(env, d, g, T):
    """Widths that leave the last 1024-channel piece full, one lane wide or ragged; token counts below, at and above one
    round of the partition.  The step tables are taken with GIVEN coefficient words, so both sides sum the same binary32
    residuals: the binary32 sums of the device (at most T/8 + 8 terms in one chain, relative error below 1e-5) can move a
    step over at most one binary16 boundary, and only where the exact value lies within 1e-5 of one (a binary16 step is
    4.9e-4 to 9.8e-4 of its value: 1 to 2 % of the channels at the very worst)."""
    s, rac, orc, dev, P = env.synth, env.rac, env.orc, env.dev, env.P
    J = d // g
    gen = s.generator(70 + T, dev)
    scale = s.channel_scale(d, 7, dev)
    X = s.activations(T, d, scale, gen)
    R = s.affine_noisy_reference(X, g, gen)
    rng = np.random.default_rng(T)
    rows = rng.permutation(T).astype(np.int32)
    rows[rng.random(T) < 0.3] = -1
    rows_d = torch.from_numpy(rows).to(dev)
    cuts = np.unique(np.concatenate([[0], rng.integers(0, T + 1, 3), [T]])).astype(np.int32)
    n_seg = cuts.size - 1
    cfg = rac.CodecCfg(d, g, 4, 0, coef_fmt=1)
    so = torch.from_numpy(cuts).to(dev)
    coef = torch.full((n_seg, J), -3, dtype=torch.int32, device=dev)
    seg_of = torch.full((T,), -3, dtype=torch.int32, device=dev)
    st = torch.zeros(1, dtype=torch.int32, device=dev)
    nb = rac.rac_fit_segments_workspace_bytes(cfg, T)
    ws = torch.full((nb + 16,), 0x5A, dtype=torch.uint8, device=dev)
    rac.rac_fit_segments(cfg, X, T, R, T, rows_d, None, None, so, n_seg, coef, seg_of, ws[:nb], nb, st)
    Xb, Rb = s.bf16_bits(X), s.bf16_bits(R)
    o_coef, dg = orc.fit_segments(d, g, Xb, cuts, ref_base=Rb, ref_row=rows, diag=True)
    g_coef = coef.cpu().numpy().view(np.uint32)
    assert np.array_equal(seg_of.cpu().numpy(), np.searchsorted(cuts, np.arange(T), side="right") - 1)
    seg = torch.from_numpy(np.searchsorted(cuts, np.arange(T), side="right") - 1)
    for shift, name, exact in ((0, "alpha", dg["alpha"]), (16, "beta", dg["beta"])):
        a, b = ((g_coef >> shift) & 0xffff).astype(np.uint16), ((o_coef >> shift) & 0xffff).astype(np.uint16)
        m = (a != b) & ~(((a | b) & 0x7fff) == 0)
        if m.any():      # a word that differs is what the optimum rounds to within the fit's evaluation error
            # (the rows are unrelated here: the slope is small against sum|dr*dh| / Sxx, whose binary32 rounding counts)
            mag = float(X.float().abs().max())
            P._check_flips(name, a[m], b[m], exact[m], 4.0 * 2.0 ** -24 * (mag if shift else 64.0))
    step = torch.zeros((2, d), dtype=torch.float32, device=dev)
    inv = torch.zeros_like(step)
    nb = rac.rac_calibrate_workspace_bytes(cfg)
    ws = torch.full((nb + 16,), 0x5A, dtype=torch.uint8, device=dev)
    rac.rac_calibrate_steps_shared(cfg, X, T, R, T, rows_d, None, None, coef, seg_of, 3.0, step, inv, ws[:nb], nb, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and torch.all(ws[nb:] == 0x5A)
    o_step, o_inv = orc.calibrate(d, g, 4, Xb, ref_base=Rb, ref_row=rows, shared_coef=g_coef[seg.numpy()])
    gs = step.cpu().numpy()
    assert np.all(np.abs(gs - o_step) <= np.spacing(o_step.astype(np.float16)).astype(np.float32))
    assert (gs != o_step).sum() <= max(2, 0.02 * gs.size)
    assert np.array_equal(inv.cpu().numpy()[gs == o_step], o_inv[gs == o_step])


# ------------------------------------------------------------------------------- retrieval: chunks of 512 query positions
def _match(env, hist, query, w, K):
    rac, dev = env.rac, env.dev
    h, q = torch.from_numpy(hist).to(dev), torch.from_numpy(query).to(dev)
    N = q.numel()
    nb = rac.rac_match_workspace_bytes(h.numel(), N, K)
    ws = torch.full((nb + 32,), 0x5A, dtype=torch.uint8, device=dev)
    rows = torch.full((N + 8,), 12345, dtype=torch.int32, device=dev)
    cap = N // w + 1
    spans = torch.full((cap + 2, 3), 777, dtype=torch.int32, device=dev)
    n = torch.full((1,), -5, dtype=torch.int32, device=dev)
    rac.rac_match_spans(h, h.numel(), q, N, w, K, rows[:N], spans[:cap], n, ws[:nb], nb)
    torch.cuda.synchronize()
    assert torch.all(rows[N:] == 12345) and torch.all(spans[cap:] == 777) and torch.all(ws[nb:] == 0x5A)
    return rows[:N].cpu().numpy(), spans[:int(n.item())].cpu().numpy()


@pytest.mark.parametrize("N,w,K", [(511, 4, 8), (512, 1, 3), (513, 4, 16), (4096, 5, 8), (4097, 4, 8), (1024 * 512 + 700, 4, 8),
                                   (1500, 3, 0)])
def test_selection_at_chunk_edges(env, N, w, K):
    """Query lengths at the edges of a chunk, of the chunks of one cluster, and of the 1024 chunks that are resolved
    together; spans of one token up to several chunks, some ending exactly at a chunk's end; sets of 3, 8 and 16 starts."""
    rng = np.random.default_rng(N + K)
    hist = rng.integers(0, 3, 3000).astype(np.int32)          # three tokens: every window occurs many times
    hist[500:2500] = rng.integers(0, 500, 2000)
    query = rng.integers(0, 500, N).astype(np.int32)
    i = int(rng.integers(0, 9))
    while i < N:
        L = min(int(rng.choice([1, 5, 40, 511, 512, 1300])), N - i)
        if rng.random() < 0.3 and i % 512:
            L = min(512 - i % 512, N - i)                     # up to the end of the chunk
        j = int(rng.integers(0, hist.size - L + 1))
        query[i:i + L] = hist[j:j + L]
        i += L + int(rng.integers(0, 4))
    rows, spans = _match(env, hist, query, w, K)
    o_rows, o_spans = env.orc.match_spans(hist, query, w, K)
    assert np.array_equal(rows, o_rows) and np.array_equal(spans, o_spans)


def test_one_span_over_many_chunks_and_no_span_at_all(env):
    rng = np.random.default_rng(1)
    hist = rng.integers(0, 30000, 9000).astype(np.int32)
    for query in (hist[100:8100].copy(), rng.integers(40000, 50000, 6000).astype(np.int32)):
        rows, spans = _match(env, hist, query, 4, 8)
        o_rows, o_spans = env.orc.match_spans(hist, query, 4, 8)
        assert np.array_equal(rows, o_rows) and np.array_equal(spans, o_spans)


def test_windows_that_occur_thousands_of_times(env):
    """All threads at one slot and one set of starts at the same time: the sets still end as the K most recent starts."""
    hist = np.zeros(20000, np.int32)
    hist[::17] = 1
    query = np.concatenate([hist[:300], np.full(40, 2, np.int32), hist[17 * 900:17 * 900 + 700]])
    for K in (1, 3, 8, 16):
        rows, spans = _match(env, hist, query, 4, K)
        o_rows, o_spans = env.orc.match_spans(hist, query, 4, K)
        assert np.array_equal(rows, o_rows) and np.array_equal(spans, o_spans)


@pytest.mark.parametrize("N,w,K,live", [(1, 1, 8, 0), (31, 32, 1, 0), (513, 3, 16, 0), (1537, 32, 3, 2000), (4096, 4, 8, 0),
                                        (4097, 4, 8, 3300), (3000, 2, 0, 1000)])
def test_index_and_token_table_at_cluster_edges(env, N, w, K, live):
    """Prompts of one chunk up to the chunks of one cluster and one token more, with intra-sequence references (the table of
    tokens in the cluster's shared memory or in global memory; tokens of every sign, among them -1), requests of all lengths,
    whose ends cut matches off, and windows of one token up to 32.  Every result is exact."""
    rac, dev = env.rac, env.dev
    rng = np.random.default_rng(1000 + N)
    hist = rng.integers(-40, 400, 6000).astype(np.int32)
    cuts = np.unique(np.concatenate([[0, 6000], rng.integers(0, 6000, 12), [700, 701]])).astype(np.int32)
    query = rng.integers(-300, 4000, N).astype(np.int32)
    i = int(rng.integers(0, 9))
    while i < N:
        L = min(int(rng.choice([1, 9, 33, 300, 1300])), N - i)
        j = int(rng.choice(cuts[:-1])) if rng.random() < 0.3 else int(rng.integers(0, 6000 - L + 1))
        L = min(L, 6000 - j)
        query[i:i + L] = hist[j:j + L]
        i += L + int(rng.integers(0, 30))
    cfg = rac.IndexCfg(6000, w, K)
    nb, nws = rac.rac_index_bytes(cfg), rac.rac_index_query_workspace_bytes(N)
    mem = torch.full((nb,), 0x5A, dtype=torch.uint8, device=dev)
    ws = torch.full((nws + 16,), 0x5A, dtype=torch.uint8, device=dev)
    h, q = torch.from_numpy(hist).to(dev), torch.from_numpy(query).to(dev)
    rows = torch.full((N + 4,), 12345, dtype=torch.int32, device=dev)
    spans = torch.full((N // w + 1, 3), 777, dtype=torch.int32, device=dev)
    n = torch.full((1,), -5, dtype=torch.int32, device=dev)
    rac.rac_index_reset(cfg, mem, nb)
    for a, b in zip(cuts, cuts[1:]):
        rac.rac_index_append(cfg, mem, nb, h, int(a), int(b))
    for intra in (True, False):
        rac.rac_index_query_live(cfg, mem, nb, h, 6000, live, q, N, intra, rows[:N], spans, n, ws[:nws], nws)
        o_rows, o_spans = env.orc.match_spans_req(hist, cuts, query, w=w, max_hits=K, intra=intra, first_live=live)
        assert np.array_equal(rows[:N].cpu().numpy(), o_rows)
        assert np.array_equal(spans[:int(n.item())].cpu().numpy(), o_spans)
    assert torch.all(rows[N:] == 12345) and torch.all(ws[nws:] == 0x5A)


def _index_query(env, hist, requests, query, w, K, intra):
    rac, dev = env.rac, env.dev
    N, H = query.size, hist.size
    cfg = rac.IndexCfg(H, w, K)
    nb, nws = rac.rac_index_bytes(cfg), rac.rac_index_query_workspace_bytes(N)
    mem, ws = (torch.full((n,), 0x5A, dtype=torch.uint8, device=dev) for n in (nb, nws))
    h, q = torch.from_numpy(hist).to(dev), torch.from_numpy(query).to(dev)
    rows = torch.full((N,), 12345, dtype=torch.int32, device=dev)
    spans = torch.full((N // w + 1, 3), 777, dtype=torch.int32, device=dev)
    n = torch.full((1,), -5, dtype=torch.int32, device=dev)
    rac.rac_index_reset(cfg, mem, nb)
    for a, b in requests:
        rac.rac_index_append(cfg, mem, nb, h, a, b)
    rac.rac_index_query(cfg, mem, nb, h, H, q, N, intra, rows, spans, n, ws, nws)
    return rows.cpu().numpy(), spans[:int(n.item())].cpu().numpy()


def _edited_copies(N, edit, seed):
    """History: a text, and prefixes of 3 to 9 tokens of its stretches repeated behind it.  Query: stretches of the text with
    single tokens replaced at `edit` and every 12 to 20 from there, so that a match resumes at the same distance."""
    rng = np.random.default_rng(seed)
    text = rng.integers(0, 3000, 2500).astype(np.int32)
    starts = rng.integers(0, 2300, 40)
    tail = np.concatenate([np.concatenate([rng.integers(5000, 9000, 5), text[s:s + int(rng.integers(3, 10))]])
                           for s in np.concatenate([starts, starts, rng.integers(0, 2300, 40)])]).astype(np.int32)
    query = np.empty(0, np.int32)
    while query.size < N:
        s = int(rng.choice(starts))
        part = text[s:s + int(rng.integers(40, 200))].copy()
        part[edit::int(rng.integers(12, 21))] = 20000
        query = np.concatenate([query, rng.integers(10000, 12000, int(rng.integers(0, 32))).astype(np.int32), part])
    return np.concatenate([text, tail]), np.ascontiguousarray(query[:N])


def test_copy_that_resumes_after_a_changed_token(env):
    """The later of two starts matches its window only, the earlier one up to the changed token; behind it the copy goes on at the
    earlier one's distance.  Nothing may reach over the changed token."""
    rng = np.random.default_rng(0)
    A = rng.permutation(2000)[:96].astype(np.int32)
    first = A.copy()
    first[12] = 5000
    cases = [(np.concatenate([first, np.arange(6000, 6005), A[:8], np.arange(7000, 7020)]).astype(np.int32), A)]
    hist = rng.permutation(20000)[:400].astype(np.int32)
    hist[300:304] = hist[100:104]
    query = hist[100:164].copy()
    query[12] = 30000
    cases.append((hist, query))
    for hist, query in cases:
        o_rows, o_spans = env.orc.match_spans(hist, query, 4, 8)
        assert o_spans[0, 2] == 12
        rows, spans = _match(env, hist, query, 4, 8)
        assert np.array_equal(rows, o_rows) and np.array_equal(spans, o_spans)
        rows, spans = _index_query(env, hist, [(0, hist.size)], query, 4, 8, False)
        assert np.array_equal(rows, o_rows) and np.array_equal(spans, o_spans)


@pytest.mark.parametrize("N,K", [(600, 8), (4500, 8), (600, 0)])
@pytest.mark.parametrize("named", [2000, 2990, 2999, 3000, 3500])
def test_query_that_names_other_than_the_indexed_tokens(env, N, K, named):
    """n_hist is where the rows of intra-sequence references begin: a caller may give the rows of its state buffer, more or fewer
    than the tokens in the index.  The candidates are those of the index."""
    rac, dev = env.rac, env.dev
    rng = np.random.default_rng(named + N)
    hist = rng.integers(0, 200, 3000).astype(np.int32)
    cuts = [0, 900, 1970, 2985, 3000]
    query = rng.integers(0, 3000, N).astype(np.int32)
    for i in range(3, N - 40, 43):
        L = int(rng.integers(4, 41))
        j = int(rng.integers(1900, 3000 - L + 1))
        query[i:i + L] = hist[j:j + L]
    query[N - 15:] = hist[2985:]
    cfg = rac.IndexCfg(3500, 3, K)
    nb, nws = rac.rac_index_bytes(cfg), rac.rac_index_query_workspace_bytes(N)
    mem, ws = (torch.full((n,), 0x5A, dtype=torch.uint8, device=dev) for n in (nb, nws))
    h, q = torch.from_numpy(hist).to(dev), torch.from_numpy(query).to(dev)
    rows = torch.full((N,), 12345, dtype=torch.int32, device=dev)
    spans = torch.full((N // 3 + 1, 3), 777, dtype=torch.int32, device=dev)
    n = torch.full((1,), -5, dtype=torch.int32, device=dev)
    rac.rac_index_reset(cfg, mem, nb)
    for a, b in zip(cuts, cuts[1:]):
        rac.rac_index_append(cfg, mem, nb, h, a, b)
    rac.rac_index_query(cfg, mem, nb, h, named, q, N, True, rows, spans, n, ws, nws)
    o_rows, o_spans = env.orc.match_spans_req(hist, cuts, query, w=3, max_hits=K, intra=True)
    o_rows[o_rows >= 3000] += named - 3000
    assert np.array_equal(spans[:int(n.item())].cpu().numpy(), o_spans) and np.array_equal(rows.cpu().numpy(), o_rows)


def test_requests_in_any_order(env):
    """The end of the index is that of its last token, not of the request that came last."""
    rng = np.random.default_rng(12)
    hist = rng.integers(0, 200, 2000).astype(np.int32)
    query = np.concatenate([hist[1700:1760], rng.integers(0, 200, 30), hist[1960:], hist[300:350]]).astype(np.int32)
    o_rows, o_spans = env.orc.match_spans_req(hist, [0, 800, 2000], query, w=3, max_hits=8)
    rows, spans = _index_query(env, hist, [(800, 2000), (0, 800)], query, 3, 8, False)
    assert np.array_equal(rows, o_rows) and np.array_equal(spans, o_spans)


@pytest.mark.parametrize("N", [64, 512, 2048, 4096, 4097])
@pytest.mark.parametrize("w,K", [(1, 8), (3, 2), (4, 3), (4, 8), (4, 16), (8, 8)])
def test_edited_copies(env, N, w, K):
    """Copies with single tokens changed, over windows that occur several times: the first change at 8 to 31 tokens, the copies at
    every alignment to a warp; one history and an index of several requests, with and without intra-sequence references."""
    for edit in (8, 11, 12, 13, 17, 20, 25, 31):
        hist, query = _edited_copies(N, edit, 100 * edit + N + K)
        rows, spans = _match(env, hist, query, w, K)
        o_rows, o_spans = env.orc.match_spans(hist, query, w, K)
        assert np.array_equal(rows, o_rows) and np.array_equal(spans, o_spans)
        cuts = [0, 700, 2500, 2600, hist.size]
        for intra in (False, True):
            rows, spans = _index_query(env, hist, list(zip(cuts, cuts[1:])), query, w, K, intra)
            o_rows, o_spans = env.orc.match_spans_req(hist, cuts, query, w=w, max_hits=K, intra=intra)
            assert np.array_equal(rows, o_rows) and np.array_equal(spans, o_spans)


# ------------------------------------------------------------------------------- encode with outliers in one launch
@pytest.mark.parametrize("d,g,bits,k,T", [
    (64, 32, 4, 2, 9000), (2048, 128, 3, 8, 8000), (2080, 32, 4, 16, 5000), (4096, 64, 2, 8, 5400), (4128, 32, 3, 5, 4100),
    (3072, 64, 4, 8, 6000), (5120, 128, 4, 8, 4100), (5120, 64, 2, 12, 8193), (5152, 32, 4, 8, 2700), (8192, 1024, 4, 1, 2400),
    (8192, 64, 3, 8, 3), (8192, 128, 4, 8, 1024)])
def test_one_launch_outliers_at_shape_edges(env, d, g, bits, k, T):
    """Widths on both sides of every CTA shape, more tokens than four rounds of the record slots (or fewer than CTAs), gathered
    rows with direct tokens, some tokens with many equal residuals (the whole-token path): records equal the oracle's given the
    device's coefficient words."""
    s, rac, orc, dev, P = env.synth, env.rac, env.orc, env.dev, env.P
    gen = s.generator(d + T, dev)
    scale = s.channel_scale(d, 5, dev)
    X = s.activations(T, d, scale, gen)
    R = s.affine_noisy_reference(X, g, gen)
    rng = np.random.default_rng(d)
    rows = np.arange(T, dtype=np.int32)
    rows[rng.random(T) < 0.2] = -1
    equal = rng.random(T) < 0.02                       # reference equal to the token: an all-zero residual
    R[torch.from_numpy(np.flatnonzero(equal)).to(dev)] = X[torch.from_numpy(np.flatnonzero(equal)).to(dev)]
    flat = np.flatnonzero(rng.random(T) < 0.02)        # a few levels only: many equal magnitudes
    X[torch.from_numpy(flat).to(dev)] = torch.sign(X[torch.from_numpy(flat).to(dev)].float()).to(torch.bfloat16)
    cal = min(T, 512)
    step, inv = orc.calibrate(d, g, bits, s.bf16_bits(X[:cal]), ref_base=s.bf16_bits(R[:cal]), ref_row=rows[:cal])
    step_d, inv_d = P.to_dev(step, dev), P.to_dev(inv, dev)
    cfg = rac.CodecCfg(d, g, bits, k)
    pay, st = P.gpu_encode(cfg, X, R, torch.from_numpy(rows).to(dev), None, None, step_d, inv_d)
    assert st == 0
    P.compare_encode(cfg, pay, s.bf16_bits(X), s.bf16_bits(R), rows, None, None, step, inv)
    # with x_hat: the same records, and x_hat equal to the oracle's reconstruction of them
    pay2, xs, st = P.gpu_encode_reconstruct(cfg, X, R, torch.from_numpy(rows).to(dev), None, None, step_d, inv_d)
    assert st == 0 and np.array_equal(pay, pay2)
    o_x = orc.reconstruct(d, g, bits, k, pay, T, ref_base=s.bf16_bits(R), ref_row=rows, step=step, nthreads=orc.max_threads())
    assert np.array_equal(o_x.reshape(-1), s.bf16_bits(xs).reshape(-1))


@pytest.mark.parametrize("d,g,bits,k,T,predictor", [
    (32, 32, 4, 1, 40, False), (32, 32, 2, 16, 40, False), (256, 32, 3, 8, 40, True), (288, 32, 4, 16, 40, False),
    (1536, 64, 3, 4, 60, False), (4096, 128, 4, 8, 700, False),
    (5120, 128, 2, 5, 300, True), (8160, 32, 3, 8, 50, False), (8192, 64, 4, 16, 1200, False)])
def test_many_equal_residuals(env, d, g, bits, k, T, predictor):
    """Tokens whose outliers are looked for in the whole token: all-zero residuals, one magnitude everywhere, magnitudes that rise
    or fall from one piece of channels to the next (the 256 channels of a step, fewer and more), and a few levels at random.  The
    whole call with and without x_hat, and the same tokens through two token lists."""
    s, rac, dev, P = env.synth, env.rac, env.dev, env.P
    gen = s.generator(d + k, dev)
    R = s.activations(T, d, s.channel_scale(d, 5, dev), gen)
    rng = np.random.default_rng(d + k)
    gain, bias = s.predictor_gain_bias(d, 5, dev) if predictor else (None, None)
    X = R.clone() if gain is None else torch.addcmul(bias.float(), gain.float(), R.float()).to(torch.bfloat16)
    rows = np.arange(T, dtype=np.int32)
    sign = torch.tensor([1.0, -1.0], device=dev).repeat(d // 2)         # pairs cancel: the mean of a group is exactly zero
    for t in range(T):
        kind = t % 7                                                    # 0: the (transformed) reference itself
        if kind == 0:
            continue
        piece = int(rng.choice([2, 32, 64, 256, 512]))
        level = torch.arange(d, device=dev) // piece
        if kind == 1:
            level = torch.zeros_like(level)
        elif kind == 3:
            level = level.flip(0) // 2 * 2
        elif kind == 4:
            level = torch.from_numpy(rng.integers(0, 4, d // 2)).to(dev).repeat_interleave(2)
        elif kind == 5:                                                 # zeros, and fewer non-zero channels than outliers
            level = torch.full((d,), -1, device=dev)
            level[-max(1, (k - 1) // 2) * 2:] = 5
            level = level if k > 2 else level.clamp(max=-1)
        elif kind == 6:
            level = torch.ones_like(level)
            level[int(rng.integers(0, d // 2)) * 2] = 9
        X[t] = ((level + 1).float() * 0.25 * sign).to(torch.bfloat16)
        rows[t] = -1
    step = np.full((2, d), 0.125, np.float32)
    rows_d = torch.from_numpy(rows).to(dev)
    cfg = rac.CodecCfg(d, g, bits, k)
    _, pay, _ = P.round_trip_case(cfg, X, R, rows_d, gain, bias, step, 1.0 / step)
    order = rng.permutation(T).astype(np.int32)
    st = torch.zeros(1, dtype=torch.int32, device=dev)
    nws = rac.rac_encode_workspace_bytes(cfg, T)
    ws = torch.empty(nws, dtype=torch.uint8, device=dev)
    step_d, inv_d = P.to_dev(step, dev), P.to_dev(1.0 / step, dev)
    listed = torch.full((pay.size,), 0xA5, dtype=torch.uint8, device=dev)
    xs = torch.full((T, d), -7.0, dtype=torch.bfloat16, device=dev)
    for part in (order[:T // 3], order[T // 3:]):
        rac.rac_encode_reconstruct_list(cfg, X, T, torch.from_numpy(part).to(dev),
                                        torch.tensor([part.size], dtype=torch.int32, device=dev), R, T, rows_d, None, 0, gain, bias,
                                        step_d, inv_d, listed, pay.size, xs, ws, nws, st)
    assert int(st.item()) == 0 and np.array_equal(listed.cpu().numpy(), pay)
    assert torch.equal(xs.view(torch.int16), P.gpu_encode_reconstruct(cfg, X, R, rows_d, gain, bias, step_d, inv_d)[1].view(torch.int16))


@pytest.mark.parametrize("T", [0, 1, 31, 128, 4095, 4096, 4097, 12289, 131072, 128 * 4096 + 1])
def test_split_waves_at_range_edges(env, T):
    """One token up to more ranges than CTAs; mixed rows, all of one wave, and a first row that only the last token reaches."""
    rac, dev = env.rac, env.dev
    rng = np.random.default_rng(T)
    rows = rng.integers(-1, 2000, max(T, 1)).astype(np.int32)
    rows[-1] = 2 ** 31 - 1
    rows_d = torch.from_numpy(rows).to(dev)
    for first in (1000, 0, 2 ** 31 - 1):
        w1, w2 = (torch.full((T + 1,), -9, dtype=torch.int32, device=dev) for _ in range(2))
        n = torch.full((2,), -5, dtype=torch.int32, device=dev)
        rac.rac_split_waves(rows_d, T, first, w1, w2, n)
        o1, o2 = np.flatnonzero(rows[:T] < first), np.flatnonzero(rows[:T] >= first)
        assert n.tolist() == [o1.size, o2.size]
        assert np.array_equal(w1[:o1.size].cpu().numpy(), o1) and np.array_equal(w2[:o2.size].cpu().numpy(), o2)
        assert torch.all(w1[o1.size:] == -9) and torch.all(w2[o2.size:] == -9)


# ------------------------------------------------------------------------------- token lists, one scale per group
@pytest.mark.parametrize("d,bits,kg,T", [(4096, 4, 1, 700), (4096, 8, 2, 40), (5120, 4, 0, 700), (5120, 8, 1, 33), (3072, 4, 4, 50),
                                         (4096, 4, 3, 5)])
def test_listed_tokens_at_compiled_in_widths(env, d, bits, kg, T):
    """Two lists in random order, together all tokens: the widths and outlier counts that are compiled in, one beyond each, one
    token per CTA and several.  The records meet the oracle's, x_hat of both sides is the oracle's reconstruction of them."""
    s, rac, orc, dev, P = env.synth, env.rac, env.orc, env.dev, env.P
    gen = s.generator(T, dev)
    X = s.activations(T, d, s.channel_scale(d, 3, dev), gen)
    R = s.affine_noisy_reference(X, 128, gen)
    rng = np.random.default_rng(T)
    rows = np.arange(T, dtype=np.int32)
    rows[rng.random(T) < 0.2] = -1
    order = rng.permutation(T).astype(np.int32)
    cut = T // 3
    cfg = rac.CodecCfg(d, 128, bits, 0, scale_mode=1, topk_group=kg)
    rec = rac.rac_record_bytes(cfg)
    rows_d, st = torch.from_numpy(rows).to(dev), torch.zeros(1, dtype=torch.int32, device=dev)
    pay = torch.full((T * rec,), 0xA5, dtype=torch.uint8, device=dev)
    xs, xr = (torch.full((T, d), -7.0, dtype=torch.bfloat16, device=dev) for _ in range(2))
    lists = []
    for part in (order[:cut], order[cut:]):
        lst = torch.from_numpy(part).to(dev) if part.size else torch.zeros(1, dtype=torch.int32, device=dev)
        lists.append((lst, torch.tensor([part.size], dtype=torch.int32, device=dev)))
    nws = rac.rac_encode_workspace_bytes(cfg, T)
    ws = torch.empty(max(nws, 16), dtype=torch.uint8, device=dev)
    for lst, cnt in lists:
        rac.rac_encode_reconstruct_list(cfg, X, T, lst, cnt, R, T, rows_d, None, 0, None, None, None, None, pay, T * rec, xs,
                                        ws if nws else None, nws, st)
    for lst, cnt in lists:
        rac.rac_decode_reconstruct_list(cfg, pay, T, lst, cnt, R, T, rows_d, None, 0, None, None, None, xr, st)
    assert int(st.item()) == 0
    p = pay.cpu().numpy()
    P.compare_encode(cfg, p, s.bf16_bits(X), s.bf16_bits(R), rows)
    o_x = orc.reconstruct(d, 128, bits, 0, p, T, ref_base=s.bf16_bits(R), ref_row=rows, nthreads=orc.max_threads(), scale_mode=1,
                          topk_group=kg)
    for x in (xs, xr):
        assert np.array_equal(o_x.reshape(-1), s.bf16_bits(x).reshape(-1))


@pytest.mark.parametrize("d,bits,kg,T,predictor", [(5120, 4, 1, 900, True), (5120, 4, 2, 889, False), (5120, 4, 8, 888, False),
                                                   (4096, 8, 0, 8000, False)])
def test_group_scales_in_calls_of_many_tokens(env, d, bits, kg, T, predictor):
    """Encode with x_hat past the token counts where it reads the reference a second time (and at the last one where it does
    not): direct tokens, a predictor's gain and bias on the reference, several tokens per CTA."""
    s, rac, P = env.synth, env.rac, env.P
    gen = s.generator(d + kg, env.dev)
    X = s.activations(T, d, s.channel_scale(d, 4, env.dev), gen)
    R = s.affine_noisy_reference(X, 128, gen)
    rows = torch.arange(T, dtype=torch.int32, device=env.dev)
    rows[::7] = -1
    gain, bias = s.predictor_gain_bias(d, 4, env.dev) if predictor else (None, None)
    P.round_trip_case(rac.CodecCfg(d, 128, bits, 0, scale_mode=1, topk_group=kg), X, R, rows, gain, bias)


@pytest.mark.parametrize("d", [2048, 4096])
def test_encode_with_x_hat_on_both_sides_of_the_step_registers(env, d):
    """Identity rows without outliers, one token below and above the size from which rows of 4 and 8 KB leave the steps in memory:
    the same records, and x_hat equal to the receiver's."""
    s, rac, P = env.synth, env.rac, env.P
    T = 80_000_000 // d + 1
    gen = s.generator(d, env.dev)
    X = s.activations(T, d, s.channel_scale(d, 4, env.dev), gen)
    R = s.affine_noisy_reference(X, 128, gen)
    step = (X[:2000].float().std(0, unbiased=False) / 7).half().float().clamp(min=2.0 ** -10).repeat(2, 1).contiguous()
    inv = 1.0 / step
    cfg = rac.CodecCfg(d, 128, 4, 0)
    rec = rac.rac_record_bytes(cfg)
    out = []
    for n in (T, T - 1):
        pay, xs, st = P.gpu_encode_reconstruct(cfg, X[:n], R[:n], None, None, None, step, inv)
        xr, st2 = P.gpu_decode(cfg, pay, n, R[:n], None, None, None, step, env.dev)
        assert st == 0 and st2 == 0 and torch.equal(xs.view(torch.int16), xr.view(torch.int16))
        out.append(pay)
    assert np.array_equal(out[0][:(T - 1) * rec], out[1])
    P.compare_encode(cfg, out[0][-64 * rec:], s.bf16_bits(X[-64:]), s.bf16_bits(R[-64:]), None, None, None, step.cpu().numpy(),
                     inv.cpu().numpy())


# ------------------------------------------------------------------------------------------------------------- the fit
@pytest.mark.parametrize("d,g", [(4096, 128), (3584, 64), (2880, 32), (8192, 1024), (5120, 256)])
@pytest.mark.parametrize("mode", [0, 1])
def test_fit_with_means_small_and_large_beside_the_spread(env, d, g, mode):
    """Means of zero, about half of the spread and large beside it (of the reference and of the token), references that say
    nothing about the token, constant and zero groups, all among the groups of one warp and as whole tokens.  Coefficients
    against the oracle's binary64 fit by the protocol's windows; the rest bit for bit."""
    s, rac, P = env.synth, env.rac, env.P
    T, J = 24, d // g
    rng = np.random.default_rng(d + g)
    r = rng.standard_normal((T, J, g))
    h = 0.9 * r + 0.05 * rng.standard_normal((T, J, g))
    kind = rng.integers(0, 8, (T, J))
    kind[:8] = np.arange(8)[:, None]                      # tokens of one kind; the others mixed
    pick = lambda k: (kind == k)[:, :, None]
    r = r + 0.45 * pick(1) + 0.55 * pick(2) + 40.0 * pick(3)
    h = h + 0.40 * pick(1) + 0.50 * pick(2) + 36.0 * pick(3) + 0.5 * pick(4)
    h = np.where(pick(5), rng.standard_normal((T, J, g)) + 0.45, h)      # unrelated
    r = np.where(pick(6), 1.25, np.where(pick(7), 0.0, r))
    X = torch.from_numpy(h.reshape(T, d)).float().to(torch.bfloat16).to(env.dev)
    R = torch.from_numpy(r.reshape(T, d)).float().to(torch.bfloat16).to(env.dev)
    if mode == 0:
        cfg = rac.CodecCfg(d, g, 4, 8)
        step = np.full((2, d), 0.03125, np.float32)
        P.round_trip_case(cfg, X, ref_base=R, step=step, inv_step=(np.float32(1) / step).astype(np.float32))
    else:
        P.round_trip_case(rac.CodecCfg(d, g, 4, 0, scale_mode=1, topk_group=1), X, ref_base=R)


@pytest.mark.parametrize("d,g", [(2880, 32), (3584, 64), (4096, 128), (5120, 256), (8192, 1024)])
@pytest.mark.parametrize("mode", [0, 1])
def test_encoders_fit_by_the_calibrations_centred_sums(env, d, g, mode):
    """The segment fit leaves its centred statistics per token and group (mean r, mean h, Sxx, Sxy) in its workspace.  The
    encoders' coefficient words are those statistics' division and multiply-add, correctly rounded, bit for bit: a fit whose
    sums round in another way flips a word in some ten thousand (its relative difference over the 2^-11 of a binary16 step).
    Means from zero to half of the spread; some tokens without a reference."""
    s, rac, dev = env.synth, env.rac, env.dev
    T, J = 4096, d // g
    rng = np.random.default_rng(d + mode)
    gen = s.generator(g, dev)
    R = torch.randn((T, J, g), device=dev, generator=gen) + torch.rand((T, J, 1), device=dev, generator=gen) * 0.5
    X = 0.9 * R + 0.05 * torch.randn((T, J, g), device=dev, generator=gen)
    X, R = X.to(torch.bfloat16).view(T, d), R.to(torch.bfloat16).view(T, d)
    rows = rng.permutation(T).astype(np.int32)
    rows[::9] = -1
    X = X[torch.from_numpy(np.where(rows >= 0, rows, np.arange(T))).to(dev).long()]      # next to its reference row
    rows_d = torch.from_numpy(rows).to(dev)
    scfg = rac.CodecCfg(d, g, 4, 0, coef_fmt=1)
    nb = rac.rac_fit_segments_workspace_bytes(scfg, T)
    ws = torch.zeros(nb, dtype=torch.uint8, device=dev)
    st = torch.zeros(1, dtype=torch.int32, device=dev)
    rac.rac_fit_segments(scfg, X, T, R, T, rows_d, None, None, torch.tensor([0, T], dtype=torch.int32, device=dev), 1,
                         torch.zeros((1, J), dtype=torch.int32, device=dev), torch.zeros(T, dtype=torch.int32, device=dev), ws, nb, st)
    rbar, hbar, sxx, sxy = np.moveaxis(ws[:16 * T * J].cpu().numpy().view(np.float32).reshape(T, J, 4), 2, 0)
    assert int(st.item()) == 0 and np.all(sxx[rows >= 0] > 1.0)
    ref = (rows >= 0)[:, None]
    a = np.where(ref, sxy / np.where(ref, sxx, np.float32(1)), np.float32(0))
    b = np.where(ref, (hbar - a.astype(np.longdouble) * rbar).astype(np.float32), hbar)
    want = a.astype(np.float16).view(np.uint16) | (b.astype(np.float16).view(np.uint16).astype(np.uint32) << 16)
    step = torch.full((2, d), 0.03125, device=dev)
    cfg = rac.CodecCfg(d, g, 4, 8) if mode == 0 else rac.CodecCfg(d, g, 4, 0, scale_mode=1, topk_group=1)
    rec = rac.rac_record_bytes(cfg)
    pay, st = env.P.gpu_encode(cfg, X, R, rows_d, None, None, *((step, 1 / step) if mode == 0 else (None, None)))
    got = np.ascontiguousarray(pay.reshape(T, rec)[:, :4 * J]).view(np.uint32)
    assert st == 0 and np.array_equal(got, want)


def test_fit_flags_values_that_are_not_finite(env):
    """An infinity or a NaN in the token or in the reference, in one group of one token: the status bit, and the records of all
    other tokens as without it."""
    s, rac, P = env.synth, env.rac, env.P
    d, T = 4096, 6
    gen = s.generator(5, env.dev)
    X = s.activations(T, d, s.channel_scale(d, 5, env.dev), gen)
    R = s.affine_noisy_reference(X, 128, gen)
    step = np.full((2, d), 0.03125, np.float32)
    inv = (np.float32(1) / step).astype(np.float32)
    cfg = rac.CodecCfg(d, 128, 4, 0)
    rec = rac.rac_record_bytes(cfg)
    clean, _, st = P.gpu_encode_reconstruct(cfg, X, R, None, None, None, torch.from_numpy(step).to(env.dev), torch.from_numpy(inv).to(env.dev))
    assert st == 0
    for bad in (float("inf"), float("nan"), -float("inf")):
        for which in (0, 1):
            x, r = X.clone(), R.clone()
            (x, r)[which][3, 777] = bad
            pay, _, st = P.gpu_encode_reconstruct(cfg, x, r, None, None, None, torch.from_numpy(step).to(env.dev), torch.from_numpy(inv).to(env.dev))
            assert st & rac.STATUS_NONFINITE
            keep = [t for t in range(T) if t != 3]
            assert np.array_equal(pay.reshape(T, rec)[keep], clean.reshape(T, rec)[keep])


@pytest.mark.parametrize("bits", [2, 3, 4, 8])
@pytest.mark.parametrize("kg", [0, 1])
def test_group_scales_keep_a_value_that_is_no_number_in_its_channel(env, bits, kg):
    """A reference value that is not finite (slope 0, the mean alone: one residual without a number), and a NaN of the token
    beside given coefficients: the codes of the channels around it are those that the sender's x_hat was formed with, so the
    receiver's x_hat has the same bits everywhere else.  The fit reports the value; with given coefficients nobody looks."""
    s, rac, dev = env.synth, env.rac, env.dev
    d, g, T, at = 4096, 128, 6, 777
    gen = s.generator(bits, dev)
    X = s.activations(T, d, s.channel_scale(d, 5, dev), gen)
    R = s.affine_noisy_reference(X, g, gen)
    words = torch.full((1, d // g), 0x3C00, dtype=torch.int32, device=dev)          # alpha 1, beta 0
    for bad in (float("nan"), float("inf"), -float("inf"), None):
        x, r = X.clone(), R.clone()
        if bad is None:
            x[3, at] = float("nan")
        else:
            r[3, at] = bad
        cfg = rac.CodecCfg(d, g, bits, 0, scale_mode=1, topk_group=kg, coef_fmt=1 if bad is None else 0)
        seg = dict(coef_seg=words, seg_of=torch.zeros(T, dtype=torch.int32, device=dev)) if bad is None else {}
        pay = torch.zeros(T * rac.rac_record_bytes(cfg), dtype=torch.uint8, device=dev)
        xs, xr = torch.zeros_like(X), torch.zeros_like(X)
        st = torch.zeros(1, dtype=torch.int32, device=dev)
        rac.rac_encode_reconstruct_list(cfg, x, T, None, None, r, T, None, None, 0, None, None, None, None, pay, pay.numel(), xs, None, 0,
                                        st, **seg)
        rac.rac_decode_reconstruct_list(cfg, pay, T, None, None, r, T, None, None, 0, None, None, None, xr, st, **seg)
        assert bool(int(st.item()) & rac.STATUS_NONFINITE) == (bad is not None)
        same = xs.view(torch.int16) == xr.view(torch.int16)
        same[3, at] = True
        assert bool(same.all()), (bad, (~same).nonzero()[:8].tolist())


# ------------------------------------------------------------------- one launch with x_hat: teams of one CTA per SM, from a size on
@pytest.mark.parametrize("d,g,bits,k,per_sm,gathered", [
    (5120, 128, 4, 8, 20, True),      # three teams, width compiled in
    (5120, 64, 3, 5, 54, False),
    (4128, 32, 2, 16, 20, True),      # five warps, the last with one lane
    (5120, 32, 4, 16, 20, True),      # three teams and the tables do not fit: the other forms
    (4096, 128, 4, 8, 54, True),      # three teams, width compiled in
    (4096, 256, 3, 8, 54, True),
    (2080, 32, 4, 8, 54, True),       # four teams of three warps, the last with one lane
    (7168, 256, 2, 8, 20, True),      # two teams, the widest
    (5376, 128, 4, 1, 20, False),
    (7168, 128, 4, 8, 20, True),      # two teams do not fit
    (2112, 64, 3, 8, 64, False),      # the lines of up to 96 threads,
    (5120, 128, 4, 8, 160, False),    # of up to 160 with identity rows,
    (4608, 256, 4, 8, 56, True),      # with gathered rows,
    (4896, 32, 2, 4, 40, True),       # and from 4896 channels on
    (5120, 128, 4, 8, 40, True),
])
@pytest.mark.parametrize("table", ["binary16", "binary32"])
def test_encode_in_teams_at_its_first_sizes(env, d, g, bits, k, per_sm, gathered, table):
    """The last token count of the other forms and the first of this one, where a team gets one token more than another: records
    as without x_hat (another kernel) and against the oracle, x_hat equal to the receiver's; steps that binary16 holds, and steps
    that it does not (these stand as binary32 over the second row of inverse steps)."""
    s, rac, P = env.synth, env.rac, env.P
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    T = per_sm * sms
    gen = s.generator(d + bits, env.dev)
    X = s.activations(T, d, s.channel_scale(d, 4, env.dev), gen)
    R = s.affine_noisy_reference(X, g, gen)
    rows = None
    if gathered:
        rows = torch.arange(T, dtype=torch.int32, device=env.dev)
        rows[::5] = -1
    step = torch.stack([torch.full((d,), 0.05, device=env.dev), X[:2000].float().std(0, unbiased=False) * (3.0 / 7)]).clamp(min=2.0 ** -10)
    step = step.half().float() if table == "binary16" else step + step * 2.0 ** -14
    inv = 1.0 / step
    cfg = rac.CodecCfg(d, g, bits, k)
    rec = rac.rac_record_bytes(cfg)
    out = []
    for n in (T, T - 1):
        r = None if rows is None else rows[:n]
        pay, xs, st = P.gpu_encode_reconstruct(cfg, X[:n], R[:n], r, None, None, step, inv)
        plain, st2 = P.gpu_encode(cfg, X[:n], R[:n], r, None, None, step, inv)
        xr, st3 = P.gpu_decode(cfg, pay, n, R[:n], r, None, None, step, env.dev)
        assert st == 0 and st2 == 0 and st3 == 0
        assert np.array_equal(pay, plain) and torch.equal(xs.view(torch.int16), xr.view(torch.int16))
        out.append(pay)
    assert np.array_equal(out[0][:(T - 1) * rec], out[1])
    at = slice(T - 700, T)
    P.compare_encode(cfg, out[0][(T - 700) * rec:], s.bf16_bits(X[at]), s.bf16_bits(R),
                     np.arange(T - 700, T, dtype=np.int32) if rows is None else rows[at].cpu().numpy(), None, None,
                     step.cpu().numpy(), inv.cpu().numpy())


@pytest.mark.parametrize("d,g,k,predictor", [(5120, 128, 8, True), (5120, 64, 8, True), (5120, 128, 5, True), (5120, 32, 8, False), (5376, 128, 8, True)])
def test_encode_with_x_hat_in_two_launches(env, d, g, k, predictor):
    """Gathered rows with direct tokens, one token more than the one-launch form takes at these widths, where a predictor or the
    size of the groups keeps the call from the form in teams: records as without x_hat (another kernel) and against the oracle,
    x_hat equal to the receiver's."""
    s, rac, P = env.synth, env.rac, env.P
    T = 8193
    gen = s.generator(d + g + k, env.dev)
    X = s.activations(T, d, s.channel_scale(d, 4, env.dev), gen)
    R = s.affine_noisy_reference(X, g, gen)
    rows = torch.arange(T, dtype=torch.int32, device=env.dev)
    rows[::5] = -1
    gain, bias = s.predictor_gain_bias(d, 7, env.dev) if predictor else (None, None)
    step = torch.stack([torch.full((d,), 0.0625, device=env.dev), X[:2000].float().std(0, unbiased=False) * (3.0 / 7)]).clamp(min=2.0 ** -10)
    step = step.half().float()
    inv = 1.0 / step
    cfg = rac.CodecCfg(d, g, 4, k)
    rec = rac.rac_record_bytes(cfg)
    pay, xs, st = P.gpu_encode_reconstruct(cfg, X, R, rows, gain, bias, step, inv)
    plain, st2 = P.gpu_encode(cfg, X, R, rows, gain, bias, step, inv)
    xr, st3 = P.gpu_decode(cfg, pay, T, R, rows, gain, bias, step, env.dev)
    assert st == 0 and st2 == 0 and st3 == 0
    assert np.array_equal(pay, plain) and torch.equal(xs.view(torch.int16), xr.view(torch.int16))
    at = slice(T - 300, T)
    gb, bb = (None, None) if gain is None else (s.f16_bits(gain), s.f16_bits(bias))
    P.compare_encode(cfg, pay[(T - 300) * rec:], s.bf16_bits(X[at]), s.bf16_bits(R), rows[at].cpu().numpy(), gb, bb,
                     step.cpu().numpy(), inv.cpu().numpy())


@pytest.mark.parametrize("d,bits,k,per_sm", [(4096, 4, 8, 54), (6144, 3, 5, 20)])
@pytest.mark.parametrize("table", ["binary16", "binary32"])
def test_teams_whose_waits_cannot_complete_give_up(env, d, bits, k, per_sm, table):
    """The give-up path of the form in teams, in its safe shape: every stage announces more bytes than its copies deliver and each
    wait gives up after its polls.  Every team of a CTA sets the status and returns, none waits for another without a bound, and
    the next ordinary call on the stream gives the bits it always gives."""
    s, rac, P, dev = env.synth, env.rac, env.P, env.dev
    T = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + 1
    gen = s.generator(d + bits, dev)
    X = s.activations(T, d, s.channel_scale(d, 4, dev), gen)
    R = s.affine_noisy_reference(X, 128, gen)
    step = torch.full((2, d), 0.0625, device=dev) * (1.0 if table == "binary16" else 1.0 + 2.0 ** -14)
    inv = 1.0 / step
    cfg = rac.CodecCfg(d, 128, bits, k)
    good = P.gpu_encode_reconstruct(cfg, X, R, None, None, None, step, inv)
    assert good[2] == 0
    n = T * rac.rac_record_bytes(cfg)
    out = torch.zeros(n + 2 * T * d, dtype=torch.uint8, device=dev)
    nws = rac.rac_encode_workspace_bytes(cfg, T)
    ws = torch.zeros(max(nws, 16), dtype=torch.uint8, device=dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    rac.rac_selftest_bounded_wait(cfg, 2, X, T, R, T, step, inv, out, out.numel(), ws if nws else None, nws, status)
    torch.cuda.synchronize()
    assert int(status.item()) & rac.STATUS_TIMEOUT
    with pytest.raises(rac.RacError):      # no room for x_hat behind the records
        rac.rac_selftest_bounded_wait(cfg, 2, X, T, R, T, step, inv, out, out.numel() - 1, ws if nws else None, nws, status)
    pay, xs, st = P.gpu_encode_reconstruct(cfg, X, R, None, None, None, step, inv)
    assert st == 0 and np.array_equal(pay, good[0]) and torch.equal(xs, good[1])
