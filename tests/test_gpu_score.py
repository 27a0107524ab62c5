"""Distillation score on the GPU (Eq. 3) against the oracle, through the C ABI."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2608_18183_b200 import binding, synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _teacher_shape(s, dtype=None):
    """A wider, deeper model over the same vocabulary, grid and classes."""
    return synth.ModelShape(s.n_layers + 1, s.dim * 2, s.n_heads * 2, s.ffn_hidden * 2, s.vocab, s.grid_h, s.grid_w,
                            s.n_classes, dtype or s.dtype)


def test_bikl_rows_match_the_definition():
    import torch
    sh = synth.ModelShape(1, 64, 1, 64, 16384, 4, 4, 3, "bf16")
    ctx = binding.Context(sh, synth.make_weights(sh, 3, target_entropy=None), 2, 4)
    rng = np.random.default_rng(0)
    rows = 37
    s = (rng.normal(size=(rows, sh.vocab)) * 3.0).astype(np.float32)
    t = (0.6 * s + rng.normal(size=(rows, sh.vocab)) * 2.0).astype(np.float32)
    s[1], t[1] = s[1] + 50.0, t[1] - 70.0          # shifted rows: the normalisers cancel
    t[2] = s[2]                                     # equal distributions
    s[3, 5], t[3, 9] = 90.0, 90.0                   # two nearly one-hot rows that disagree
    got = ctx.hbsjd_bikl(G.dev(s), G.dev(t)).cpu().numpy()
    want = O.bikl(s, t)
    # fp32 sums of V terms with ex2.approx exponentials: a few 1e-6 relative on each of the two halves
    assert np.abs(got - want).max() <= 2e-5 * max(1.0, np.abs(want).max()), np.abs(got - want).max()
    np.testing.assert_allclose(got, want, rtol=2e-4, atol=2e-5)
    assert got[2] == 0.0 and want[3] > 40.0
    ctx.hbsjd_destroy()
    # a small vocabulary (fewer entries than threads x 4) and one that needs several chunks per thread
    for V in (256, 32768):
        sh = synth.ModelShape(1, 64, 1, 64, V, 4, 4, 3, "bf16")
        ctx = binding.Context(sh, synth.make_weights(sh, 3, target_entropy=None), 2, 4)
        s = (rng.normal(size=(5, V)) * 2.0).astype(np.float32)
        t = (rng.normal(size=(5, V)) * 2.0).astype(np.float32)
        np.testing.assert_allclose(ctx.hbsjd_bikl(G.dev(s), G.dev(t)).cpu().numpy(), O.bikl(s, t), rtol=2e-4)
        ctx.hbsjd_destroy()


def _score_both(w, tsh, toks, k, lab, max_batch=None):
    timg = synth.make_weights(tsh, 77)
    stu = binding.Context(w.shape, G.weights_for(w), max_batch or len(k), w.window)
    tea = binding.Context(tsh, timg, max_batch or len(k), w.window)
    pos, per, loss = stu.hbsjd_score(tea, G.dev(toks), G.dev(k), G.dev(lab))
    want = O.score(O.Model(w.shape, G.weights_for(w)), O.Model(tsh, timg), toks, k, lab)
    out = (pos.cpu().numpy(), per.cpu().numpy(), loss), want
    stu.hbsjd_destroy()
    tea.hbsjd_destroy()
    return out


def test_score_fp32_models_match_the_oracle():
    w = synth.WORKLOADS["tiny"]
    T, V = w.shape.T, w.shape.vocab
    rng = np.random.default_rng(2)
    B = 5
    toks = rng.integers(0, V, size=(B, T)).astype(np.int32)
    k = np.array([0, 13, T - 1, T, 40], dtype=np.int32)     # T is not a multiple of the chunk for some rows only
    lab = rng.integers(0, w.shape.n_classes, size=B).astype(np.int32)
    (pos, per, loss), (opos, oper, oloss) = _score_both(w, _teacher_shape(w.shape), toks, k, lab)
    assert opos.max() > 0.05                                    # the comparison is not vacuous
    np.testing.assert_allclose(pos, opos, rtol=2e-3, atol=2e-5)
    for b in range(B):
        assert (pos[b, :k[b]] == 0).all()
    np.testing.assert_allclose(per, oper, rtol=5e-4, atol=1e-6)
    assert per[3] == 0.0
    assert abs(loss - oloss) <= 5e-4 * oloss


def test_score_window_that_does_not_divide_the_sequence():
    w = synth.with_shape(synth.WORKLOADS["tiny"], window=7)      # 64 = 9 chunks of 7 + 1
    T, V = w.shape.T, w.shape.vocab
    rng = np.random.default_rng(3)
    toks = rng.integers(0, V, size=(3, T)).astype(np.int32)
    k = np.array([5, 0, 62], dtype=np.int32)
    lab = np.array([1, 2, 3], dtype=np.int32)
    (pos, per, loss), (opos, oper, oloss) = _score_both(w, _teacher_shape(w.shape), toks, k, lab, max_batch=4)
    np.testing.assert_allclose(pos, opos, rtol=2e-3, atol=2e-5)
    assert abs(loss - oloss) <= 5e-4 * oloss


def test_score_bf16_models_within_the_derived_tolerance():
    """bf16 models: each model's logits carry the rounding noise the forward parity tests bound (mean s per logit,
    max tol: the measured noise floor).  With d = s - t, D = 1/2 sum (p - q) d moves under logit noise e_s, e_t by
    1/2 sum (p - q)(e_s - e_t) + 1/2 (Cov_p(e_s, d) - Cov_q(e_t, d)): the first part has rms <= s (|p - q|_2 <=
    sqrt 2), the second rms <= s std(d) (|p|_2, |q|_2 <= 1).  So a position's error has rms <= s (1 + std d); the
    maximum over the positions is held to the same expression with the max-abs logit bound tol in place of s."""
    w = synth.WORKLOADS["small_bf16"]
    tsh = _teacher_shape(w.shape)
    timg = synth.make_weights(tsh, 77)
    T, V = w.shape.T, w.shape.vocab
    rng = np.random.default_rng(4)
    B = 3
    toks = rng.integers(0, V, size=(B, T)).astype(np.int32)
    k = np.array([0, 50, 100], dtype=np.int32)
    lab = rng.integers(0, w.shape.n_classes, size=B).astype(np.int32)
    (pos, per, loss), (opos, oper, oloss) = _score_both(w, tsh, toks, k, lab)
    seq0 = np.concatenate([[0], toks[0, :T - 1]]).astype(np.int32)
    m_s, m_t = O.Model(w.shape, G.weights_for(w)), O.Model(tsh, timg)
    l_s, l_t = m_s.forward_full(int(lab[0]), seq0), m_t.forward_full(int(lab[0]), seq0)
    # s, tol: mean and maximum of the logit noise floor, measured as the oracle against its own diagnostic form (fp32
    # sums, bf16 attention weights, the RMSNorm form both contexts use) on the same sequence, with the factors of
    # the forward parity tests (1.5 on the mean, 2 on a maximum taken over fewer logits than the GPU's)
    s = tol = 0.0
    for m, ref in ((m_s, l_s), (m_t, l_t)):
        m.set_diag(acc_f32=True, attn_w_bf16=True, norm_folded=True)
        try:
            d = np.abs(m.forward_full(int(lab[0]), seq0).astype(np.float64) - ref)
        finally:
            m.set_diag()
        s, tol = max(s, 1.5 * float(d.mean())), max(tol, 2.0 * float(d.max()))
    spread = 1.0 + float((l_s - l_t).std(axis=1).max())
    live = opos > 0
    assert live.sum() == int((T - k).sum())
    err = np.abs(pos - opos)[live]
    assert err.max() <= tol * spread, (err.max(), tol * spread)
    assert err.mean() <= s * spread, (err.mean(), s * spread)
    assert (pos[~live] == 0).all()
    assert abs(loss - oloss) <= s * spread
    # regression guard, looser than what is measured (3e-5 on the loss, 0.13 % mean per position)
    assert abs(loss - oloss) <= 2e-3 * oloss and err.mean() <= 5e-3 * opos[live].mean()
    np.testing.assert_allclose(per, [pos[b, k[b]:].mean() for b in range(B)], rtol=1e-5)


def test_score_of_a_model_against_itself_is_zero_and_the_call_is_repeatable():
    w = synth.WORKLOADS["tiny_bf16"]
    T, V = w.shape.T, w.shape.vocab
    toks, k, lab = synth.make_inputs(w)
    toks = np.random.default_rng(0).integers(0, V, size=toks.shape).astype(np.int32)
    a = binding.Context(w.shape, G.weights_for(w), w.batch, w.window)
    b = binding.Context(w.shape, G.weights_for(w), w.batch, w.window)
    pos, per, loss = a.hbsjd_score(b, G.dev(toks), G.dev(k), G.dev(lab))
    assert float(pos.abs().max()) == 0.0 and loss == 0.0       # same kernels, same inputs: bit-identical logits
    # scoring follows a rollout on the same context and leaves it usable for the next rollout
    out, st = a.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), G.gpu_params(w, 1))
    tsh = _teacher_shape(w.shape)
    tea = binding.Context(tsh, synth.make_weights(tsh, 77), w.batch, w.window)
    r1 = a.hbsjd_score(tea, out, G.dev(k), G.dev(lab))
    out2, _ = a.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), G.gpu_params(w, 1))
    assert bool((out2 == out).all())
    r2 = a.hbsjd_score(tea, out, G.dev(k), G.dev(lab))
    assert bool((r1[0] == r2[0]).all()) and r1[2] == r2[2] and r1[2] > 0
    # misuse is refused before any launch
    with pytest.raises(binding.HbsjdError) as e:
        a.hbsjd_score(a, out, G.dev(k), G.dev(lab))
    assert e.value.code == -1
    bad = out.clone()
    bad[0, 3] = V
    with pytest.raises(binding.HbsjdError) as e:
        a.hbsjd_score(tea, bad, G.dev(k), G.dev(lab))
    assert e.value.code == -1
    for c in (a, b, tea):
        c.hbsjd_destroy()


def test_score_does_not_depend_on_the_chunk():
    """A forward takes as many inputs per image as its 4096 rows hold, in slots of one to four 16-query blocks, the shapes of
    the attention kernel: of 200, 100, 80 and 9 images 16, 32, 48 and all 144 (in slots of 64).  All see the same keys in
    the same order: equal bits (T = 144: three KV pages, ragged last forwards)."""
    w = synth.WORKLOADS["small_bf16"]
    rng = np.random.default_rng(5)
    toks = rng.integers(0, w.shape.vocab, (200, w.shape.T)).astype(np.int32)
    k = rng.integers(0, w.shape.T, 200).astype(np.int32)
    lab = rng.integers(0, w.shape.n_classes, 200).astype(np.int32)
    tsh = synth.ModelShape(2, 384, 6, 512, w.shape.vocab, 12, 12, 10, "bf16")
    stu = binding.Context(w.shape, G.weights_for(w), 200, 4)
    tea = binding.Context(tsh, synth.make_weights(tsh, 77), 200, 4)
    got = {}
    for n in (200, 100, 80, 9):
        pos, per, loss = stu.hbsjd_score(tea, G.dev(toks[:n]), G.dev(k[:n]), G.dev(lab[:n]))
        got[n] = pos.cpu().numpy(), per.cpu().numpy()
        assert (got[n][0][np.arange(w.shape.T)[None] >= k[:n, None]] > 0).all()
    for pos, per in got.values():
        np.testing.assert_array_equal(pos[:9], got[9][0])
        np.testing.assert_array_equal(per[:9], got[9][1])
        np.testing.assert_array_equal(pos, got[200][0][:len(pos)])
    stu.hbsjd_destroy()
    tea.hbsjd_destroy()


@pytest.mark.parametrize("model,batch", [("tiny", 1), ("B", 3)])
def test_score_of_contexts_on_one_stream_and_on_two_is_the_same(model, batch):
    """Contexts that share a stream run side by side inside the call.  The same kernels do the same arithmetic in the
    same order whatever the streams are, so every bit is equal; work of the shared stream before and after the call (the
    tokens it reads, an overwrite of them) is ordered with it; an invalid argument leaves the contexts usable."""
    import torch
    w = synth.WORKLOADS[model]
    w = synth.with_shape(w, shape=dataclasses.replace(w.shape, n_layers=2))
    rng = np.random.default_rng(8)
    toks = rng.integers(0, w.shape.vocab, size=(batch, w.shape.T)).astype(np.int32)
    k = rng.integers(0, w.shape.T // 2, size=batch).astype(np.int32)
    lab = rng.integers(0, w.shape.n_classes, size=batch).astype(np.int32)
    simg, timg = (synth.make_weights(w.shape, s, target_entropy=None) for s in (5, 6))
    out = []
    for streams in ((torch.cuda.Stream(),) * 2, (torch.cuda.Stream(), torch.cuda.Stream()), (None, None)):
        stu, tea = (binding.Context(w.shape, img, batch, w.window, stream=s) for img, s in zip((simg, timg), streams))
        dk, dl, dt = G.dev(k), G.dev(lab), G.dev(toks)
        bad = dk + w.shape.T
        torch.cuda.synchronize()
        with pytest.raises(binding.HbsjdError):
            stu.hbsjd_score(tea, dt, bad, dl)
        for _ in range(2):
            if streams[0] is streams[1]:
                with torch.cuda.stream(streams[0]):
                    dt.fill_(0)
                    dt.copy_(G.dev(toks))
            pos, per, loss = stu.hbsjd_score(tea, dt, dk, dl)
            out.append((pos.cpu().numpy(), per.cpu().numpy(), loss))
        stu.hbsjd_destroy()
        tea.hbsjd_destroy()
    for pos, per, loss in out[1:]:
        assert np.array_equal(pos, out[0][0]) and np.array_equal(per, out[0][1]) and loss == out[0][2]
    assert out[0][2] > 0


def test_score_on_a_high_priority_stream_keeps_its_priority():
    """Contexts that share a stream score side by side, the student on a stream of its own: of the caller's priority, or
    its half would queue behind other work of the device.  With matrix products filling the GPU from a stream of low
    priority, contexts that share a high-priority stream are compared with contexts on two such streams, which
    nothing moves (measured: 1.0 times their time; 2.1 with the student at default priority)."""
    import time

    import torch
    sh = synth.ModelShape(6, 768, 12, 2048, 1024, 16, 16, 10, "bf16")
    imgs = [synth.make_weights(sh, seed, target_entropy=None) for seed in (1, 2)]
    streams = [torch.cuda.Stream(priority=-1) for _ in range(2)]
    toks = torch.randint(0, 1024, (9, 256), device="cuda", dtype=torch.int32)
    zero = torch.zeros(9, device="cuda", dtype=torch.int32)
    x = torch.randn(4096, 4096, device="cuda").bfloat16()
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    times, losses = [], set()
    for second in (0, 1):
        s, t = (binding.Context(sh, img, 9, 16, stream=st) for img, st in zip(imgs, (streams[0], streams[second])))
        one = []
        for _ in range(9):
            for _ in range(600):
                torch.mm(x, x, out=y)
            t0 = time.perf_counter()
            losses.add(s.hbsjd_score(t, toks, zero, zero)[2])
            one.append(time.perf_counter() - t0)
            torch.cuda.synchronize()
        times.append(sorted(one)[4])
        s.hbsjd_destroy()
        t.hbsjd_destroy()
    assert len(losses) == 1
    assert times[0] < 1.5 * times[1], times
