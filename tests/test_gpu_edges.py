"""Edge and degenerate cases of the rollout on the GPU: nothing to generate, one token to generate, one image,
one kept token, no-op guidance, temperature and history offsets the standard workloads do not use, the largest
vocabulary of the verification kernels."""
import subprocess
import sys

import numpy as np
import pytest

from oracle import oracle as O
from paper_2608_18183_b200 import binding, synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _ctx(w, **kw):
    return binding.Context(w.shape, G.weights_for(w), kw.get("max_batch", w.batch), kw.get("max_window", w.window))


def test_nothing_or_one_token_to_generate():
    w = synth.WORKLOADS["tiny"]
    T = w.shape.T
    toks, k, lab = synth.make_inputs(w)
    ctx = _ctx(w)
    # every image already complete: no round runs, the prefix is the result
    kk = np.full_like(k, T)
    out, st = ctx.hbsjd_rollout(G.dev(toks), G.dev(kk), G.dev(lab), G.gpu_params(w, 0))
    assert st["rounds"] == 0 and st["committed"] == 0 and st["image_forwards"] == 0
    np.testing.assert_array_equal(out.cpu().numpy(), toks)
    assert ctx.hbsjd_round() == 0                     # stepping a finished rollout is a no-op
    # one token left, a complete image and an empty prefix side by side: one round finishes the short ones
    kk = np.array([T - 1, T, 0, T - 1], dtype=np.int32)
    out, st = ctx.hbsjd_rollout(G.dev(toks), G.dev(kk), G.dev(lab), G.gpu_params(w, 3, max_rounds=1))
    cur = ctx.hbsjd_get_state()[1]
    assert cur[0] == T and cur[1] == T and cur[3] == T and 1 <= cur[2] <= w.window
    model = O.Model(w.shape, G.weights_for(w))
    r = O.Rollout(model, toks, kk, lab, G.orc_params(w, 3))
    r.round()
    np.testing.assert_array_equal(cur, r.state()[1])
    # the last token of an image is the bonus sample of a window of one input
    full, _ = ctx.hbsjd_rollout(G.dev(toks), G.dev(kk), G.dev(lab), G.gpu_params(w, 3))
    r.run()
    np.testing.assert_array_equal(full.cpu().numpy(), r.tokens())
    ctx.hbsjd_destroy()


def test_single_image_and_context_larger_than_the_call():
    w = synth.WORKLOADS["tiny"]
    toks, k, lab = synth.make_inputs(w)
    big = _ctx(w, max_batch=7, max_window=16)        # limits above the call's batch and window
    one = _ctx(w, max_batch=1)
    model = O.Model(w.shape, G.weights_for(w))
    for b in range(2):
        a, _ = one.hbsjd_rollout(G.dev(toks[b:b + 1]), G.dev(k[b:b + 1]), G.dev(lab[b:b + 1]), G.gpu_params(w, 5))
        c, _ = big.hbsjd_rollout(G.dev(toks[b:b + 1]), G.dev(k[b:b + 1]), G.dev(lab[b:b + 1]), G.gpu_params(w, 5))
        np.testing.assert_array_equal(a.cpu().numpy(), c.cpu().numpy())
        r = O.Rollout(model, toks[b:b + 1], k[b:b + 1], lab[b:b + 1], G.orc_params(w, 5))
        r.run()
        np.testing.assert_array_equal(a.cpu().numpy(), r.tokens())
    one.hbsjd_destroy()
    big.hbsjd_destroy()


def test_one_kept_token_makes_sampling_greedy():
    """top-k = 1 leaves a one-hot distribution: every sample is the argmax, so the probabilistic rollout commits
    the greedy rollout's tokens (ties of the top logit aside: none in these models)."""
    w = synth.WORKLOADS["tiny_bf16"]
    toks, k, lab = synth.make_inputs(w)
    ctx = _ctx(w)
    a, sa = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), G.gpu_params(w, 9, top_k=1))
    g, sg = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), G.gpu_params(w, 9, top_k=1,
                                                                               verify_mode=binding.VERIFY_GREEDY))
    np.testing.assert_array_equal(a.cpu().numpy(), g.cpu().numpy())
    assert sa["rounds"] == sg["rounds"]
    # top-k >= V is no filter
    x, _ = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), G.gpu_params(w, 9, top_k=0))
    y, _ = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), G.gpu_params(w, 9, top_k=w.shape.vocab + 5))
    np.testing.assert_array_equal(x.cpu().numpy(), y.cpu().numpy())
    ctx.hbsjd_destroy()


def test_guidance_with_the_null_class_is_no_guidance():
    """With the null class as the label both branches compute the same logits, so l_u + s (l_c - l_u) = l_c bit
    for bit and the guided rollout equals the unguided one."""
    w = synth.WORKLOADS["tiny_bf16"]
    toks, k, lab = synth.make_inputs(w)
    null = np.full_like(lab, w.shape.n_classes)
    ctx = _ctx(w)
    a, _ = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(null), G.gpu_params(w, 2, cfg_scale=3.5))
    b, _ = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(null), G.gpu_params(w, 2, cfg_scale=1.0))
    np.testing.assert_array_equal(a.cpu().numpy(), b.cpu().numpy())
    ctx.hbsjd_destroy()


@pytest.mark.parametrize("temperature,history", [(0.7, 8), (1.6, 100), (1.0, 1)])
def test_temperature_and_history_offsets_in_lockstep(temperature, history):
    """Temperature other than 1, a history offset beyond the sequence (every history draft falls back to the
    keyed uniform token) and the shortest offset (a draft copies its left neighbour), fp32 model, every round
    compared with the oracle."""
    w = synth.with_shape(synth.WORKLOADS["tiny"], temperature=temperature, history_offset=history)
    toks, k, lab = synth.make_inputs(synth.with_shape(w, prefix=("uniform", 0, 30)))
    model = O.Model(w.shape, G.weights_for(w))
    ctx = _ctx(w)
    rep = G.lockstep(ctx, model, w, toks, k, lab, 11)
    assert rep["max_logit_err"] <= 1e-4 and rep["max_p_err"] <= 1e-6 and rep["replay_mismatch"] == 0
    assert rep["tokens"] == int((w.shape.T - k).sum()) and rep["same"] == rep["tokens"]
    ctx.hbsjd_destroy()


def test_largest_vocabulary_of_the_verification_kernels():
    """V = 32768 (128 KB of probabilities per CTA): probability pipeline against the oracle and one bit-exact
    verification step."""
    import torch
    V = 32768
    sh = synth.ModelShape(1, 64, 1, 64, V, 4, 4, 3, "bf16")
    ctx = binding.Context(sh, synth.make_weights(sh, 3, target_entropy=None), 6, 8)
    rng = np.random.default_rng(0)
    lc = (rng.normal(size=(3, V)) * 3).astype(np.float32)
    lu = (rng.normal(size=(3, V)) * 3).astype(np.float32)
    for kk in (0, 500):
        p = ctx.hbsjd_probs(G.dev(lc), G.dev(lu), 2.0, 0.9, kk).cpu().numpy()
        for r in range(3):
            ref = O.probs(lc[r], lu[r], s=2.0, tau=0.9, k=kk)
            np.testing.assert_array_equal(p[r] > 0, ref > 1e-37)
            assert np.all(np.abs(p[r] - ref) <= 1e-6 + 1e-5 * ref)
    case = G.verify_case(5, B=6, W=8, T=32, V=V, top_k=200)
    d = {n: G.dev(case[n]) for n in ("logits", "q", "cursor", "seq", "delta", "qbase")}
    p_out = torch.zeros_like(d["q"])
    m_out = torch.zeros(6, dtype=torch.int32, device="cuda")
    ctx.hbsjd_verify(G.verify_desc(case, 4, 2), d["logits"], d["q"], p_out, d["cursor"], d["seq"], d["delta"],
                     d["qbase"], m_out)
    p_gpu = p_out.cpu().numpy()
    for b in range(6):
        c = int(case["cursor"][b])
        if c >= case["T"]:
            continue
        n = min(case["W"], case["T"] - c)
        seq, dl = case["seq"][b].copy(), case["delta"][b].copy()
        nc, m, j = O.replay_round(V, case["T"], case["W"], case["H"], False, 4, b, 2, c, seq, dl, p_gpu[b][:n],
                                  case["q"][b], int(case["qbase"][b]))
        assert nc == int(d["cursor"][b]) and m == int(m_out[b])
        np.testing.assert_array_equal(seq[:nc + 1], d["seq"][b].cpu().numpy()[:nc + 1])
    ctx.hbsjd_destroy()


def test_batch_synchronous_progress_matches_the_oracle():
    """Execution mode SYNC (the baseline of the Table 2 ablation): every live image advances by the batch's
    smallest commit.  fp32 model, every round compared with the oracle's synchronous rollout; greedy verification
    still gives the greedy AR tokens."""
    w = synth.WORKLOADS["tiny"]
    T = w.shape.T
    toks, k, lab = synth.make_inputs(synth.with_shape(w, prefix=("uniform", 0, 30)), seed=3)
    model = O.Model(w.shape, G.weights_for(w))
    ctx = _ctx(w)
    for seed in (5, 6):
        orc = O.Rollout(model, toks, k, lab, G.orc_params(w, seed, exec_mode=3))
        ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab),
                          G.gpu_params(w, seed, exec_mode=binding.EXEC_SYNC, max_rounds=0))
        rounds = 0
        while orc.live():
            before = ctx.hbsjd_get_state()[1].copy()
            ctx.hbsjd_round()
            _, m_o, _ = orc.round()
            _, cur, seq, _, _ = ctx.hbsjd_get_state()
            _, o_cur, o_seq, _, _ = orc.state()
            live = before < T
            assert len(set((cur - before)[live].tolist())) == 1        # one pace for the whole batch
            np.testing.assert_array_equal(cur, o_cur)
            for b in range(len(k)):
                np.testing.assert_array_equal(seq[b, :cur[b] + 1], o_seq[b, :o_cur[b] + 1])
            rounds += 1
        out_sync, st_sync = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab),
                                              G.gpu_params(w, seed, exec_mode=binding.EXEC_SYNC))
        out_free, st_free = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab),
                                              G.gpu_params(w, seed, exec_mode=binding.EXEC_FULL))
        assert st_sync["rounds"] == rounds            # (more rounds than independent progress on average, not per seed)
        assert st_sync["committed"] == st_free["committed"] == int((T - k).sum())
        assert st_sync["compact_rounds"] == 0
    g, _ = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab),
                             G.gpu_params(w, 0, exec_mode=binding.EXEC_SYNC, verify_mode=binding.VERIFY_GREEDY))
    ar = model.ar_rollout(toks, k, lab, G.orc_params(w, 0, greedy=True, window=1))
    np.testing.assert_array_equal(g.cpu().numpy(), ar)
    ctx.hbsjd_destroy()


def test_bf16_model_with_head_size_32_and_unsupported_head_sizes():
    """Head size 32 in bf16 runs the fused QKV epilogue with half a rotation table per head and the plain attention
    kernel; head size 128 is refused for bf16 models at creation."""
    sh = synth.ModelShape(2, 128, 4, 256, 512, 6, 6, 5, "bf16")          # dh = 32
    w = synth.Workload("dh32", sh, 3, 8, 2.0, 40, 1.0, 6, ("uniform", 0, 12))
    img = synth.make_weights(sh, 9)
    toks, k, lab = synth.make_inputs(w)
    ctx = binding.Context(sh, img, w.batch, w.window)
    model = O.Model(sh, img)
    rep = G.lockstep(ctx, model, w, toks, k, lab, 3, floor_every_round=True)
    # logits against the noise floor measured on the same windows (the context folds its RMSNorm: factor 1.5 on the
    # mean, measured 1.25; the maximum over these few thousand logits measured 1.43 x the floor's)
    G.check_logits_against_floor(rep, rep["floor_max"], rep["floor_sum"] / rep["floor_n"], "head size 32",
                                 max_factor=1.8, mean_factor=1.5)
    assert rep["max_p_err"] <= 1e-6
    G.check_flips_explained(rep)
    assert rep["same"] >= 0.9 * rep["tokens"]
    ctx.hbsjd_destroy()
    bad = synth.ModelShape(1, 256, 2, 256, 512, 4, 4, 5, "bf16")         # dh = 128
    with pytest.raises(binding.HbsjdError):
        binding.Context(bad, synth.make_weights(bad, 9, target_entropy=None), 2, 4)


def test_images_do_not_depend_on_their_batch_mates():
    """Each image advances on its own: replacing the other images of the batch (here: marking them complete, or
    giving them other prefixes and labels) leaves an image's tokens unchanged (bf16 model, guidance, top-k)."""
    w = synth.WORKLOADS["tiny_bf16"]
    T = w.shape.T
    toks, k, lab = synth.make_inputs(w)
    ctx = _ctx(w)
    ref, _ = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), G.gpu_params(w, 4))
    ref = ref.cpu().numpy()
    keep = [0, 2]
    k2, lab2, toks2 = k.copy(), lab.copy(), toks.copy()
    for b in range(w.batch):
        if b not in keep:
            k2[b] = T if b % 2 else max(0, int(k[b]) - 3)
            lab2[b] = (lab[b] + 1) % w.shape.n_classes
            toks2[b] = (toks[b] + 7) % w.shape.vocab
    for mode in (binding.EXEC_FULL, binding.EXEC_COMPACT):
        out, _ = ctx.hbsjd_rollout(G.dev(toks2), G.dev(k2), G.dev(lab2), G.gpu_params(w, 4, exec_mode=mode))
        out = out.cpu().numpy()
        for b in keep:
            np.testing.assert_array_equal(out[b], ref[b])
    ctx.hbsjd_destroy()


def test_kernel_profile_bins_add_up():
    """Per-class event timing: the GEMM class split by activation rows adds up to the class, every bin that has
    launches has time, FLOPs and algorithmic bytes, and switching the profile off stops the accounting."""
    w = synth.WORKLOADS["small_bf16"]
    toks, k, lab = synth.make_inputs(w)
    ctx = binding.Context(w.shape, G.weights_for(w), w.batch, w.window)
    ctx.hbsjd_profile(True)
    _, st = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), G.gpu_params(w, 3))
    p = ctx.hbsjd_profile_read()
    ctx.hbsjd_profile(False)
    g, bins = p["gemm"], p["gemm_by_rows"]
    assert g["launches"] > 0 and p["attention"]["launches"] > 0 and p["accept"]["launches"] == st["rounds"]
    assert sum(b["launches"] for b in bins.values()) == g["launches"]
    assert abs(sum(b["ms"] for b in bins.values()) - g["ms"]) <= 1e-6 * g["ms"]
    assert abs(sum(b["work"] for b in bins.values()) - g["work"]) <= 1e-9 * g["work"]
    for b in bins.values():
        assert (b["launches"] > 0) == (b["ms"] > 0) == (b["work"] > 0) == (b["bytes"] > 0)
    assert bins["rows>6144"]["launches"] == 0                  # this context has at most 4096 rows per forward
    ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), G.gpu_params(w, 3))
    assert ctx.hbsjd_profile_read()["gemm"]["launches"] == g["launches"]
    ctx.hbsjd_destroy()



@pytest.mark.parametrize("batch,dim,window", [(9000, 128, 20), (5000, 1024, 33), (300, 128, 16)])
def test_batches_beyond_a_ctas_work_list(batch, dim, window):
    """Thousands of images in one forward: the attention kernel's share of the work list does not depend on the batch (a
    table of every slot did not fit beside the key ring above 8300 images), and at 5000 images of 16 heads with guidance
    a CTA has more items (541) than the 512 entries it holds.  An image's tokens do not depend on the others."""
    sh = synth.ModelShape(1, dim, dim // 64, 64, 64, 4, 4, 3, "bf16")
    c = binding.Context(sh, synth.make_weights(sh, 3, target_entropy=None), batch, window)
    rng = np.random.default_rng(batch)
    toks = rng.integers(0, 64, size=(batch, 16)).astype(np.int32)
    k = rng.integers(0, 16, size=batch).astype(np.int32)
    lab = rng.integers(0, 3, size=batch).astype(np.int32)
    few = 150
    p = binding.make_params(window, 4, cfg_scale=2.0, exec_mode=binding.EXEC_FULL, seed=5)
    out, st = c.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), p)
    assert st["committed"] == int((16 - k).sum())
    out2, _ = c.hbsjd_rollout(G.dev(toks[:few]), G.dev(k[:few]), G.dev(lab[:few]), p)
    np.testing.assert_array_equal(out[:few].cpu().numpy(), out2.cpu().numpy())
    c.hbsjd_destroy()


_WAIT = """
import ctypes, sys, time
flags = int(sys.argv[1])
cu = ctypes.CDLL("libcuda.so.1")
dev = ctypes.c_int()
assert cu.cuInit(0) == 0 and cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
assert cu.cuDevicePrimaryCtxSetFlags_v2(dev, flags) == 0
import torch
from paper_2608_18183_b200 import binding, synth
sh = synth.ModelShape(4, 1024, 16, 1024, 256, 16, 16, 3, "bf16")
c = binding.Context(sh, synth.make_weights(sh, 3, target_entropy=None), 600, 32)
g = torch.Generator(device="cuda").manual_seed(1)
toks = torch.randint(0, 256, (600, 256), device="cuda", dtype=torch.int32, generator=g)
k = torch.full((600,), 100, device="cuda", dtype=torch.int32)
lab = torch.zeros_like(k)
p = binding.make_params(32, 16, seed=4, max_rounds=20, exec_mode=binding.EXEC_FULL)
out, _ = c.hbsjd_rollout(toks, k, lab, p)
wall, cpu = time.perf_counter(), time.thread_time()
for _ in range(3):
    c.hbsjd_rollout(toks, k, lab, p, out)
wall, cpu = time.perf_counter() - wall, time.thread_time() - cpu
print(cpu / wall, int(out.long().sum()))
"""


def test_a_process_that_asked_for_blocking_waits_does_not_poll():
    """The schedule flag of the device (4: blocking synchronisation, 2: yield) is the process's choice of how its threads
    wait.  Rounds here take milliseconds and about a tenth of that to enqueue: a thread that blocks is mostly asleep, one
    that polls never is.  The tokens do not depend on it."""
    out = {}
    for flags in (0, 2, 4):
        r = subprocess.run([sys.executable, "-c", _WAIT, str(flags)], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        out[flags] = r.stdout.split()
    assert float(out[4][0]) < 0.5, out
    assert out[0][1] == out[2][1] == out[4][1]


@pytest.mark.parametrize("window,cfg,mode", [(1, 1.0, "COMPACT"), (5, 3.0, "HYBRID"), (13, 1.0, "FULL"), (16, 3.0, "FULL"),
                                             (33, 3.0, "COMPACT")])
def test_windows_of_every_length_side_by_side(window, cfg, mode):
    """The rows of a forward hold the live images' inputs only, one image behind the other: windows cut short by the end of
    the sequence, whole ones, complete images and empty prefixes in one batch, token for token the oracle's."""
    w = synth.WORKLOADS["tiny"]
    T = w.shape.T
    k = np.array([T - 1, T - window, 0, T, T - window + 1, 3, max(0, T - window - 1), T - 2, 17], dtype=np.int32)
    rng = np.random.default_rng(window)
    toks = rng.integers(0, w.shape.vocab, (len(k), T)).astype(np.int32)
    lab = rng.integers(0, w.shape.n_classes, len(k)).astype(np.int32)
    wl = synth.with_shape(w, batch=len(k), window=window, cfg_scale=cfg)
    ctx = _ctx(wl)
    out, st = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab),
                                G.gpu_params(wl, 11, exec_mode=getattr(binding, "EXEC_" + mode), gamma=3))
    r = O.Rollout(O.Model(w.shape, G.weights_for(w)), toks, k, lab, G.orc_params(wl, 11))
    r.run()
    np.testing.assert_array_equal(out.cpu().numpy(), r.tokens())
    assert st["committed"] == sum(T - k)
    ctx.hbsjd_destroy()


@pytest.mark.parametrize("window", [1, 7, 32])
def test_prefixes_and_trajectories_in_several_passes(window):
    """Pre-filling and scoring take an image's inputs in several slots per forward and, beyond the activation rows, in several
    forwards: 40 images of 144 tokens need two to three (pre-filling 2 x 40 x 143 rows at most, scoring 40 x 144, of 4096), the
    same images five at a time one.  A row's arithmetic depends on its own sequence only: same bits."""
    w = synth.with_shape(synth.WORKLOADS["small_bf16"], batch=40, window=window)
    T = w.shape.T
    rng = np.random.default_rng(3)
    toks = rng.integers(0, w.shape.vocab, (40, T)).astype(np.int32)
    k = rng.integers(0, T, 40).astype(np.int32)
    k[:6] = [T - 1, 0, 63, 64, 65, 128]
    lab = rng.integers(0, w.shape.n_classes, 40).astype(np.int32)
    big, teacher = _ctx(w), _ctx(w)
    few, few_teacher = _ctx(w, max_batch=5), _ctx(w, max_batch=5)
    for c in (big, teacher, few, few_teacher):
        c.hbsjd_debug_fold_norm(1)  # one form for contexts of every size
    p = G.gpu_params(w, 0, verify_mode=1)
    out = big.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), p)[0].cpu().numpy()
    pos = big.hbsjd_score(teacher, G.dev(out), G.dev(k), G.dev(lab))[0].cpu().numpy()
    for b in range(0, 40, 5):
        s = slice(b, b + 5)
        got = few.hbsjd_rollout(G.dev(toks[s]), G.dev(k[s]), G.dev(lab[s]), p)[0].cpu().numpy()
        np.testing.assert_array_equal(got, out[s])
        got = few.hbsjd_score(few_teacher, G.dev(out[s]), G.dev(k[s]), G.dev(lab[s]))[0].cpu().numpy()
        np.testing.assert_array_equal(got, pos[s])
    for c in (big, teacher, few, few_teacher):
        c.hbsjd_destroy()


def test_a_batch_beyond_the_slot_tables_has_one_accept_kernel():
    """18000 images are too many slots for the persistent accept kernel's tables in shared memory, the 70 that are live are
    not: Full and Compact execution have to run the same kernel all the same.  Probabilities and state bit for bit."""
    s = synth.ModelShape(1, 64, 1, 64, 1024, 4, 4, 3, "bf16")
    B, W = 18000, 2
    live = np.arange(0, B, 260)
    rng = np.random.default_rng(18000)
    toks = rng.integers(0, s.vocab, (B, s.T)).astype(np.int32)
    k = np.full(B, s.T, dtype=np.int32)
    k[live] = rng.integers(0, s.T - 4, len(live))
    ctx = binding.Context(s, synth.make_weights(s, 3), B, W)
    got = {}
    for mode in (binding.EXEC_FULL, binding.EXEC_COMPACT):
        ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(np.zeros(B, dtype=np.int32)),
                          binding.make_params(W, 4, 1.0, 0.9, 100, seed=5, exec_mode=mode, max_rounds=2))
        got[mode] = [np.concatenate([ctx.hbsjd_debug_read(binding.DBG_PROBS, int(b)) for b in live])] + list(ctx.hbsjd_get_state())
    for full, compact in zip(got[binding.EXEC_FULL], got[binding.EXEC_COMPACT]):
        np.testing.assert_array_equal(full, compact)
    ctx.hbsjd_destroy()


def test_a_small_context_holds_no_logits_that_its_rounds_do_not_need():
    """24 images token by token with a vocabulary of 16384: the rounds have 48 rows.  Pre-filling and scoring take up to 4096
    rows per forward, whose logits alone would be 268 MB; scoring takes them in parts, with the bits of a context that has
    room for more at a time."""
    import torch
    s = synth.ModelShape(2, 64, 1, 64, 16384, 16, 16, 3, "bf16")
    t = synth.ModelShape(2, 128, 2, 128, 16384, 16, 16, 3, "bf16")
    simg, timg = (synth.make_weights(x, 3 + i, target_entropy=None) for i, x in enumerate((s, t)))
    rng = np.random.default_rng(24)
    toks, k, lab = (G.dev(x.astype(np.int32)) for x in (rng.integers(0, s.vocab, (24, s.T)), rng.integers(0, s.T, 24),
                                                        rng.integers(0, 3, 24)))
    wide = binding.Context(s, simg, 24, 32), binding.Context(t, timg, 24, 32)
    assert wide[0].fold_norm  # one form of RMSNorm throughout
    want = wide[0].hbsjd_score(wide[1], toks, k, lab)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    narrow = [binding.Context(s, simg, 24, 1)]
    used = free - torch.cuda.mem_get_info()[0]
    # weights 4.5 MB, keys and values 6 MB, logits and probabilities 6 MB, activations 3 MB, allocation granules
    assert used < 64e6, used
    narrow.append(binding.Context(t, timg, 24, 1))
    for _ in range(2):
        got = narrow[0].hbsjd_score(narrow[1], toks, k, lab)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]) and got[2] == want[2]
        out = [c.hbsjd_rollout(toks, k, lab, binding.make_params(1, 16, 2.0, 1.0, 50, seed=1))[0] for c in (wide[0], narrow[0])]
        assert torch.equal(out[0], out[1])
    for c in (*wide, *narrow):
        c.hbsjd_destroy()


def test_a_context_whose_larger_activations_do_not_fit_takes_the_smaller():
    """Activations for forwards of 4096 rows are for speed only (75 MB here): with 40 MB less free than the context would take
    it is created all the same, and its tokens are the same."""
    import torch
    s = synth.ModelShape(1, 1024, 16, 4096, 64, 48, 48, 3, "bf16")
    img = synth.make_weights(s, 3, target_entropy=None)
    toks = torch.randint(0, 64, (1, s.T), device="cuda", dtype=torch.int32)
    k, lab = (torch.tensor([x], device="cuda", dtype=torch.int32) for x in (2250, 1))
    p = binding.make_params(1, 48, 1.0, 1.0, 0, seed=1)
    out = [torch.empty_like(toks) for _ in range(2)]
    binding.Context(s, img, 1, 1).hbsjd_destroy()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    ctx = binding.Context(s, img, 1, 1)
    ctx.hbsjd_rollout(toks, k, lab, p, out[0])
    taken = before - torch.cuda.mem_get_info()[0]
    ctx.hbsjd_destroy()
    torch.cuda.synchronize()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - taken + 40 * 2 ** 20, dtype=torch.uint8, device="cuda")
    ctx = binding.Context(s, img, 1, 1)
    ctx.hbsjd_rollout(toks, k, lab, p, out[1])
    assert torch.equal(out[0], out[1])
    ctx.hbsjd_destroy()
    del filler
    torch.cuda.empty_cache()


@pytest.mark.parametrize("batch,k_max,passes", [(4, 0, 0), (4, 1, 1), (4, 128, 1), (40, 128, 3)])
def test_prefill_passes_are_the_forwards_that_ran(batch, k_max, passes):
    """Window 1, prefixes of up to 128 tokens: 128 steps of a window, but one forward while the inputs of both branches fit
    4096 rows (of 40 images 51 each do, in slots of 48: 48, 48 and 32 tokens).  A pass runs attention in every layer but the last: counted by the profile."""
    w = synth.with_shape(synth.WORKLOADS["small_bf16"], batch=batch, window=1, cfg_scale=3.0)
    toks, _, lab = synth.make_inputs(w, seed=3, batch=batch)
    k = np.full(batch, k_max, dtype=np.int32)
    k[0] //= 2
    ctx = _ctx(w)
    assert ctx.hbsjd_prefill_passes() == 0
    ctx.hbsjd_profile(True)
    _, st = ctx.hbsjd_rollout(G.dev(toks), G.dev(k), G.dev(lab), G.gpu_params(w, 1, max_rounds=0))
    assert ctx.hbsjd_profile_read()["attention"]["launches"] == passes * (w.shape.n_layers - 1)
    assert ctx.hbsjd_prefill_passes() == passes and st["prefill_forwards"] == k_max
    ctx.hbsjd_destroy()
