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
