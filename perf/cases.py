"""Workloads of the codec as its users run it, for timing and for comparing results.

A case is a dict of plain values; ``kind`` says which calls one pass makes:

* ``step``     one decode step of ``T`` concurrent sequences, both ends: the sender codes the new states against the
               previous reconstructions and forms its own x_hat, the receiver reconstructs.
* ``prompt``   a prefill uplink: span retrieval over ``n_hist`` history tokens and the encode with the sender's x_hat
               (``ends`` "send"), the rows from the spans and the reconstruction at the receiver (``ends`` "receive"), or
               one after the other ("both").
* ``encode``   a downlink encode: every token against the row of the same number (no retrieval, no x_hat).
* ``decode``   its reconstruction.
* ``mirror``   encode with the sender's x_hat and the receiver's reconstruction, rows of the same number.
* ``turn``     one turn of a conversation whose index was trimmed: the index is rebuilt from the requests that are kept,
               queried with intra-sequence references, and the prompt is coded and reconstructed in two waves.
* ``tune``     one candidate of the offline calibration: (segment fit,) step tables, encode with x_hat, error.

Sizes are those of the tests and of the benchmark, or generic.  Inputs are the seeded stand-ins of ``synth``.
"""
import math

import numpy as np
import torch

from paper_2608_04991_b200 import binding as rac
from paper_2608_04991_b200 import synth

_CODEC = dict(group=128, bits=4, topk=0, scale_mode=0, qgroup=0, topk_group=0, coef_fmt=0)
_CLIP = 3.0
_NGRAM, _HITS = 4, 8


def _case(kind, T, d, **more):
    return {"kind": kind, "T": T, "d": d, **_CODEC, **more}


def listed():
    def named(name, *a, **k):
        return {"name": name, **_case(*a, **k)}
    return [
        # one conversation's decode step: the smallest call, one 4-bit scale per token (the paper's decode mode)
        named("step_1x4096", "step", 1, 4096, scale_mode=1, qgroup=4096, predictor=False, prepared=False),
        # 64 conversations decoding together, static 3-bit table, predictor in front, arguments marshalled once
        named("step_64x3584", "step", 64, 3584, bits=3, predictor=True, prepared=True),
        # a short prompt without outliers, both ends
        named("mirror_128x4096", "mirror", 128, 4096),
        # an ordinary prompt: retrieval over a 32768-token history, 60 % covered, eight outliers per token, both ends
        named("prompt_2048x4096", "prompt", 2048, 4096, topk=8, n_hist=32768, gap=176, ends="both"),
        # a point of the bits x group sweep, each direction by itself
        named("encode_16384x4096", "encode", 16384, 4096, bits=3, group=64, topk=8),
        named("decode_16384x4096", "decode", 16384, 4096, bits=2, topk=8),
        # the quantiser as printed with one outlier per group (the default of the two-endpoint link), ragged token count
        named("mirror_20001x5120", "mirror", 20001, 5120, scale_mode=1, topk_group=1),
        # a conversation's next turn: eight earlier requests in the index, two waves
        named("turn_2048x4096", "turn", 2048, 4096, scale_mode=1, topk_group=1, requests=8),
        # a candidate of the offline calibration
        named("tune_4096x2880", "tune", 4096, 2880, group=64, topk=8),
        # the long-context round trip, leg by leg: uplink with retrieval, its receiver, downlink
        named("prompt_send_131072x5120", "prompt", 131072, 5120, topk=8, n_hist=131072, gap=112, ends="send"),
        named("prompt_receive_131072x5120", "prompt", 131072, 5120, topk=8, n_hist=131072, gap=112, ends="receive"),
        named("encode_131072x5120", "encode", 131072, 5120, topk=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "mirror", "prompt", "prompt", "encode", "decode", "turn", "tune"])
    group = rng.choice([64, 128, 128, 128, 256])
    # widths in use: whole groups, from 1024 to 8192, not only powers of two
    d = group * rng.randint(-(-1024 // group), 8192 // group)
    bits = rng.choice([2, 3, 4, 4])
    c = dict(group=group, bits=bits)
    if kind == "tune":
        c.update(rng.choice([dict(topk=8), dict(topk=0), dict(topk=8, coef_fmt=1), dict(topk=0, coef_fmt=1)]))
    elif kind == "step":
        c.update(rng.choice([dict(topk=0), dict(topk=0), dict(scale_mode=1, bits=rng.choice([4, 8]), qgroup=d)]))
    elif rng.random() < 0.4 or kind == "turn":
        c.update(scale_mode=1, bits=rng.choice([4, 4, 8]), topk_group=rng.choice([0, 1, 1, 2]))
    else:
        c.update(topk=rng.choice([0, 8, 8, 4]))
    most = 131072 * 5120 // d if kind in ("encode", "decode", "prompt") else 131072 * 5120 // (4 * d)
    if kind == "step":
        return _case(kind, _log_int(rng, 1, 512), d, predictor=rng.random() < 0.5, prepared=rng.random() < 0.5, **c)
    if kind == "prompt":
        return _case(kind, _log_int(rng, 64, min(most, 100000)), d, n_hist=_log_int(rng, 4096, 100000),
                     gap=rng.choice([112, 176]), ends=rng.choice(["both", "send", "receive"]), **c)
    if kind == "turn":
        return _case(kind, _log_int(rng, 128, min(most, 8192)), d, requests=rng.randint(2, 12), **c)
    if kind == "tune":
        return _case(kind, _log_int(rng, 512, min(most, 16384)), d, **c)
    return _case(kind, _log_int(rng, 32, min(most, 131072)), d, **c)


# ---------------------------------------------------------------------------------------------------- inputs
def _cfg(c):
    return rac.CodecCfg(c["d"], c["group"], c["bits"], c["topk"], scale_mode=c["scale_mode"], qgroup=c["qgroup"],
                        topk_group=c["topk_group"], coef_fmt=c["coef_fmt"])


def _tables(c, X, R, rows):
    """Step tables from up to 1024 tokens: 3 sigma of the aligned residual over Qmax, rounded up to binary16 (row 0: tokens
    with a reference, row 1: directly coded)."""
    T, d = X.shape
    g, n = c["group"], min(T, 1024)
    x = X[:n].double().view(n, d // g, g)
    ref = torch.ones(n, dtype=torch.bool, device=X.device) if rows is None else rows[:n] >= 0
    r = (R[:n] if rows is None else R[rows[:n].clamp(min=0).long()]).double().view(n, d // g, g) * ref[:, None, None]
    dx, dr = x - x.mean(2, keepdim=True), r - r.mean(2, keepdim=True)
    sxx = (dr * dr).sum(2, keepdim=True)
    a = torch.where(sxx > 1e-12, (dx * dr).sum(2, keepdim=True) / sxx.clamp(min=1e-12), torch.zeros_like(sxx))
    e = (dx - a * dr).view(n, d)
    step = torch.zeros((2, d), dtype=torch.float64, device=X.device)
    qmax = (1 << (c["bits"] - 1)) - 1
    for row, take in ((0, ref), (1, ~ref)):
        if bool(take.any()):
            step[row] = _CLIP * e[take].pow(2).mean(0).sqrt() / qmax
    h = step.to(torch.float16)
    h = torch.where(h.double() < step, (h.view(torch.int16) + 1).view(torch.float16), h)
    st = h.float()
    return st, torch.where(st > 0, 1.0 / st, torch.zeros_like(st))


def _planted(hist, n, gap, rng):
    """A prompt of n tokens: fresh text with copies of stretches of the history, gaps U{0..gap}, lengths U{8..256}."""
    q = synth.zipf_tokens(n, rng)
    i = int(rng.integers(0, gap + 1))
    while i < n:
        L = min(int(rng.integers(8, 257)), n - i, hist.size)
        j = int(rng.integers(0, hist.size - L + 1))
        q[i:i + L] = hist[j:j + L]
        i += L + int(rng.integers(0, gap + 1))
    return q


def _codec_state(c, X, R, rows, dev):
    cfg = _cfg(c)
    T, d = X.shape
    s = dict(c=c, cfg=cfg, T=T, X=X, R=R, rows=rows, step=None, inv=None,
             status=torch.zeros(1, dtype=torch.int32, device=dev), gain=None, bias=None)
    if c["scale_mode"] == 0 and c["kind"] != "tune":
        s["step"], s["inv"] = _tables(c, X, R, rows)
    s["pay"] = torch.zeros(T * rac.rac_record_bytes(cfg), dtype=torch.uint8, device=dev)
    s["nws"] = rac.rac_encode_workspace_bytes(cfg, T)
    s["ws"] = torch.empty(s["nws"], dtype=torch.uint8, device=dev) if s["nws"] else None
    s["xs"] = torch.zeros_like(X)
    s["xr"] = torch.zeros_like(X)
    return s


def _match(s):
    rac.rac_match_spans(s["hist"], s["hist"].numel(), s["query"], s["T"], _NGRAM, _HITS, s["rows"], s["spans"], s["n_spans"],
                        s["mws"], s["mws"].numel())


def _encode_xhat(s):
    rac.rac_encode_reconstruct(s["cfg"], s["X"], s["T"], s["R"], s["R"].shape[0], s["rows"], s["gain"], s["bias"], s["step"],
                               s["inv"], s["pay"], s["pay"].numel(), s["xs"], s["ws"], s["nws"], s["status"])


def _encode(s):
    rac.rac_encode(s["cfg"], s["X"], s["T"], s["R"], s["R"].shape[0], s["rows"], s["gain"], s["bias"], s["step"], s["inv"],
                   s["pay"], s["pay"].numel(), s["ws"], s["nws"], s["status"])


def _decode(s, rows):
    rac.rac_decode_reconstruct(s["cfg"], s["pay"], s["T"], s["R"], s["R"].shape[0], rows, s["gain"], s["bias"], s["step"],
                               s["xr"], s["status"])


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    c, T, d, kind = case, case["T"], case["d"], case["kind"]
    gen = synth.generator(seed, dev)
    rng = np.random.default_rng([seed, 17])
    scale = synth.channel_scale(d, seed, dev)
    if kind == "step":
        prev = synth.activations(T, d, scale, gen)
        X = synth.random_walk_step(prev, gen)
        s = _codec_state(c, X, prev, None, dev)
        if c["predictor"]:
            s["gain"], s["bias"] = synth.predictor_gain_bias(d, seed, dev)
        if c["prepared"]:
            s["calls"] = [
                rac.prepare(rac.rac_encode_reconstruct, s["cfg"], X, T, prev, T, None, s["gain"], s["bias"], s["step"],
                            s["inv"], s["pay"], s["pay"].numel(), s["xs"], s["ws"], s["nws"], s["status"]),
                rac.prepare(rac.rac_decode_reconstruct, s["cfg"], s["pay"], T, prev, T, None, s["gain"], s["bias"],
                            s["step"], s["xr"], s["status"])]
        return s
    if kind in ("encode", "decode", "mirror"):
        X = synth.activations(T, d, scale, gen)
        s = _codec_state(c, X, synth.affine_noisy_reference(X, c["group"], gen), None, dev)
        if kind == "decode":
            _encode(s)
        return s
    if kind == "tune":
        X = synth.activations(T, d, scale, gen)
        s = _codec_state(c, X, synth.affine_noisy_reference(X, c["group"], gen), None, dev)
        s["step"] = torch.zeros((2, d), dtype=torch.float32, device=dev)
        s["inv"] = torch.zeros_like(s["step"])
        s["cws"] = torch.empty(rac.rac_calibrate_workspace_bytes(s["cfg"]), dtype=torch.uint8, device=dev)
        s["err"] = torch.zeros(3, dtype=torch.float64, device=dev)
        s["ews"] = torch.empty(rac.rac_recon_error_workspace_bytes(), dtype=torch.uint8, device=dev)
        if c["coef_fmt"] == 1:
            bounds = list(range(0, T, 64)) + [T]
            s["seg_off"] = torch.tensor(bounds, dtype=torch.int32, device=dev)
            s["coef_seg"] = torch.zeros((len(bounds) - 1, d // c["group"]), dtype=torch.int32, device=dev)
            s["seg_of"] = torch.zeros(T, dtype=torch.int32, device=dev)
            s["fws"] = torch.empty(rac.rac_fit_segments_workspace_bytes(s["cfg"], T), dtype=torch.uint8, device=dev)
        return s
    if kind == "prompt":
        hist = synth.zipf_tokens(c["n_hist"], rng)
        query = _planted(hist, T, c["gap"], rng)
        n_hist = c["n_hist"]
    else:
        reqs = [synth.zipf_tokens(T, rng)]
        for _ in range(c["requests"]):
            reqs.append(_planted(np.concatenate(reqs), T, 112, rng))
        hist, query = np.concatenate(reqs[:-1]), reqs[-1]
        n_hist = hist.size
    # retrieval once, so that the activations of matched tokens can be drawn next to their reference rows
    m = dict(hist=torch.from_numpy(hist).to(dev), query=torch.from_numpy(query).to(dev), T=T,
             rows=torch.zeros(T, dtype=torch.int32, device=dev),
             spans=torch.zeros((T // _NGRAM + 1, 3), dtype=torch.int32, device=dev),
             n_spans=torch.zeros(1, dtype=torch.int32, device=dev),
             mws=torch.empty(rac.rac_match_workspace_bytes(n_hist, T, _HITS), dtype=torch.uint8, device=dev))
    _match(m)
    Hs = synth.activations(n_hist, d, scale, gen)
    X = synth.affine_noisy_target(Hs, m["rows"], c["group"], gen, scale)
    s = _codec_state(c, X, Hs, m["rows"], dev)
    s.update(m)
    if kind == "prompt":
        s["rows_rx"] = torch.zeros_like(s["rows"])
        if c["ends"] == "receive":
            _encode(s)
        return s
    s["bounds"] = [T * r for r in range(c["requests"] + 1)]
    s["icfg"] = rac.IndexCfg(n_hist, _NGRAM, _HITS)
    s["index"] = torch.empty(rac.rac_index_bytes(s["icfg"]), dtype=torch.uint8, device=dev)
    s["qws"] = torch.empty(rac.rac_index_query_workspace_bytes(T), dtype=torch.uint8, device=dev)
    s["w1"], s["w2"] = torch.zeros_like(s["rows"]), torch.zeros_like(s["rows"])
    s["wc"] = torch.zeros(2, dtype=torch.int32, device=dev)
    return s


# ---------------------------------------------------------------------------------------------------- one pass
def run(s):
    c, kind = s["c"], s["c"]["kind"]
    if kind == "step":
        if c["prepared"]:
            for call in s["calls"]:
                call()
        else:
            _encode_xhat(s)
            _decode(s, None)
        return s["pay"], s["xs"], s["xr"], s["status"]
    if kind == "mirror":
        _encode_xhat(s)
        _decode(s, None)
        return s["pay"], s["xs"], s["xr"], s["status"]
    if kind == "encode":
        _encode(s)
        return s["pay"], s["status"]
    if kind == "decode":
        _decode(s, None)
        return s["xr"], s["status"]
    if kind == "prompt":
        out = []
        if c["ends"] != "receive":
            _match(s)
            _encode_xhat(s)
            out += [s["rows"], s["spans"], s["n_spans"], s["pay"], s["xs"]]
        if c["ends"] != "send":
            rac.rac_spans_to_rows(s["spans"], s["n_spans"], s["T"], s["rows_rx"])
            _decode(s, s["rows_rx"])
            out += [s["rows_rx"], s["xr"]]
        return out + [s["status"]]
    if kind == "tune":
        args = (s["cfg"], s["X"], s["T"], s["R"], s["T"], None, None, None)
        out = [s["step"], s["inv"], s["pay"], s["xs"], s["err"], s["status"]]
        if c["coef_fmt"] == 1:
            rac.rac_fit_segments(*args, s["seg_off"], s["seg_off"].numel() - 1, s["coef_seg"], s["seg_of"], s["fws"],
                                 s["fws"].numel(), s["status"])
            rac.rac_calibrate_steps_shared(*args, s["coef_seg"], s["seg_of"], _CLIP, s["step"], s["inv"], s["cws"],
                                           s["cws"].numel(), s["status"])
            rac.rac_encode_reconstruct_list(s["cfg"], s["X"], s["T"], None, None, s["R"], s["T"], None, None, 0, None, None,
                                            s["step"], s["inv"], s["pay"], s["pay"].numel(), s["xs"], s["ws"], s["nws"],
                                            s["status"], coef_seg=s["coef_seg"], seg_of=s["seg_of"])
            out += [s["coef_seg"], s["seg_of"]]
        else:
            rac.rac_calibrate_steps(*args, _CLIP, s["step"], s["inv"], s["cws"], s["cws"].numel(), s["status"])
            _encode_xhat(s)
        rac.rac_recon_error(s["X"], s["xs"], s["T"], c["d"], s["err"], s["ews"], s["ews"].numel())
        return out
    # turn
    n_hist = s["bounds"][-1]
    rac.rac_index_reset(s["icfg"], s["index"], s["index"].numel())
    for a, b in zip(s["bounds"], s["bounds"][1:]):
        rac.rac_index_append(s["icfg"], s["index"], s["index"].numel(), s["hist"], a, b)
    rac.rac_index_query(s["icfg"], s["index"], s["index"].numel(), s["hist"], n_hist, s["query"], s["T"], True, s["rows"],
                        s["spans"], s["n_spans"], s["qws"], s["qws"].numel())
    rac.rac_split_waves(s["rows"], s["T"], n_hist, s["w1"], s["w2"], s["wc"])
    waves = ((s["w1"], s["wc"][0:1]), (s["w2"], s["wc"][1:2]))
    for lst, cnt in waves:
        rac.rac_encode_reconstruct_list(s["cfg"], s["X"], s["T"], lst, cnt, s["R"], n_hist, s["rows"], s["xs"], s["T"], None,
                                        None, s["step"], s["inv"], s["pay"], s["pay"].numel(), s["xs"], s["ws"], s["nws"],
                                        s["status"])
    for lst, cnt in waves:
        rac.rac_decode_reconstruct_list(s["cfg"], s["pay"], s["T"], lst, cnt, s["R"], n_hist, s["rows"], s["xr"], s["T"], None,
                                        None, s["step"], s["xr"], s["status"])
    return s["rows"], s["spans"], s["n_spans"], s["wc"], s["pay"], s["xs"], s["xr"], s["status"]


# ---------------------------------------------------------------------------------------------------- what it takes
def work(case):
    """Bytes and operations of one pass: rows of X, references, records and outputs once each.  A prompt's tokens are taken as
    60 or 70 % referenced, as its gaps make them; a turn's as all referenced."""
    c, T, d, kind = case, case["T"], case["d"], case["kind"]
    rec = rac.rac_record_bytes(_cfg(c))
    row = 2 * d
    table = 4 * d if c["scale_mode"] == 0 else 0
    share = 1.0
    if kind == "prompt":
        share = 132.0 / (132.0 + c["gap"] / 2.0)
    ref = share * T * row
    enc, enc_x, dec = T * (row + rec) + ref + table, T * (2 * row + rec) + ref + 2 * table, T * (rec + row) + ref + table
    e_ops, d_ops = 16.0 * T * d, 5.0 * T * d
    if kind == "encode":
        return {"bytes": enc, "flops": e_ops}
    if kind == "decode":
        return {"bytes": dec, "flops": d_ops}
    if kind in ("step", "mirror"):
        return {"bytes": enc_x + dec, "flops": e_ops + d_ops}
    if kind == "prompt":
        b = f = 0.0
        if c["ends"] != "receive":
            b, f = b + enc_x + 4 * c["n_hist"] + 8 * T, f + e_ops
        if c["ends"] != "send":
            b, f = b + dec + 4 * T, f + d_ops
        return {"bytes": b, "flops": f}
    if kind == "turn":
        return {"bytes": enc_x + dec + 4 * T * c["requests"] + 16 * T, "flops": e_ops + d_ops}
    passes = 3 if c["coef_fmt"] == 1 else 2          # tables (and the segment fit) read X and R, then the encode does
    return {"bytes": (passes - 1) * 2 * T * row + enc_x + 2 * T * row, "flops": passes * 12.0 * T * d}


def tolerance(case):
    """The fit is taken in binary32 and rounded to binary16: an optimum next to a rounding midpoint may go either way when
    the sums run in another order, and the codes next to a boundary follow.  Against the fit taken in binary64: up to 5.1e-5
    of the payload's bytes, 5.4e-5 relative and 0.114 at most in x_hat (18 cases of these ranges); four times that here, or
    four bytes where the payload is so short that one word is more.  A step table rounded up to binary16 may move by one
    step (2^-10) in one of the four heavy channels that make up its norm: half of that, relative."""
    payload = case["T"] * rac.rac_record_bytes(_cfg(case))
    return {"rel": 5e-4 if case["kind"] == "tune" else 2.2e-4, "max": 0.5, "differ": max(2e-4, 4.0 / payload)}
