"""Probability pipeline kernel (guidance, temperature, top-k with ties, softmax) against the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2608_18183_b200 import binding, synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx16k():
    # any bf16 context with a 16384-entry vocabulary: the pipeline only needs V
    sh = synth.ModelShape(1, 64, 1, 64, 16384, 4, 4, 3, "bf16")
    c = binding.Context(sh, synth.make_weights(sh, 3, target_entropy=None), 2, 4)
    yield c
    c.hbsjd_destroy()


def _check(ctx, lc, lu, s, tau, k):
    import torch
    p = ctx.hbsjd_probs(torch.from_numpy(lc).cuda(), None if lu is None else torch.from_numpy(lu).cuda(), s, tau,
                        k).cpu().numpy()
    for r in range(lc.shape[0]):
        ref = O.probs(lc[r], None if lu is None else lu[r], s=s, tau=tau, k=k)
        # the same support exactly (the threshold is found exactly, ties kept); entries whose probability
        # underflows fp32 may be flushed to zero by expf
        big = ref > 1e-30
        np.testing.assert_array_equal(p[r][big] > 0, ref[big] > 0)
        assert p[r][ref == 0].max(initial=0.0) < 1e-37  # dropped entries are exactly 0; underflow aside
        # ... and the same values up to expf / fp32-sum rounding
        assert np.abs(p[r] - ref).max() <= 1e-6 + 1e-5 * ref.max()
        assert np.all(np.abs(p[r] - ref) <= 1e-6 + 1e-5 * ref)
        assert abs(float(p[r].astype(np.float64).sum()) - 1.0) < 1e-4


@pytest.mark.parametrize("k", [0, 1, 7, 1000, 16383, 16384, 20000])
def test_gaussian_logits(ctx16k, k):
    rng = np.random.default_rng(k)
    lc = (rng.normal(size=(6, 16384)) * 3.5).astype(np.float32)
    lu = (rng.normal(size=(6, 16384)) * 3.5).astype(np.float32)
    _check(ctx16k, lc, None, 1.0, 1.0, k)
    _check(ctx16k, lc, lu, 4.0, 0.7, k)


def test_ties_and_crowded_bins(ctx16k):
    """Heavily tied logits: the k-th value is shared by thousands of entries (all kept), one bin of the
    selection histogram holds nearly everything (the radix fallback runs), and constant rows keep all."""
    rng = np.random.default_rng(1)
    V = 16384
    rows = []
    rows.append(np.round(rng.normal(size=V) * 2).astype(np.float32))           # ~10 distinct values
    rows.append(np.where(rng.random(V) < 0.001, 50.0, rng.normal(size=V) * 1e-3).astype(np.float32))  # outliers
    rows.append(np.full(V, 1.25, dtype=np.float32))                              # constant
    r3 = rng.normal(size=V).astype(np.float32)
    r3[:3000] = r3[5]                                                            # a 3000-way tie
    rows.append(r3)
    r4 = (rng.normal(size=V) * 1e-6 + 7.0).astype(np.float32)                    # adjacent floats
    rows.append(r4)
    rows.append(-np.abs(rng.normal(size=V)).astype(np.float32) * 30)             # negative, wide
    lc = np.stack(rows)
    for k in (1, 5, 1000, 4000, 16000):
        _check(ctx16k, lc, None, 1.0, 1.0, k)


@pytest.mark.parametrize("V", [4096, 4160, 8256, 16384])
def test_more_rows_than_ctas(V):
    """Several rows per CTA of the persistent kernel (V above 4096; 4096 runs the other one), rows of very different
    scale behind one another, so that the threshold guess carried from row to row is often useless; V that leaves
    threads without entries (4160, 8256)."""
    rng = np.random.default_rng(V)
    sh = synth.ModelShape(1, 64, 1, 64, V, 4, 4, 3, "bf16")
    ctx = binding.Context(sh, synth.make_weights(sh, 3, target_entropy=None), 2, 4)
    rows = 311
    scale = 10.0 ** rng.uniform(-3, 1, size=(rows, 1))
    lc = (rng.normal(size=(rows, V)) * scale + rng.normal(size=(rows, 1)) * 5).astype(np.float32)
    lc[::37] = np.round(lc[::37])
    lu = (rng.normal(size=(rows, V)) * scale).astype(np.float32)
    _check(ctx, lc, None, 1.0, 0.9, 500)
    _check(ctx, lc, None, 1.0, 1.0, 0)
    # the oracle rounds the guided logit once, the kernels after each of three steps, which can swap the k-th largest with
    # a neighbour in the narrow rows: with guidance, multiples of 2^-10 below 2^7, on which every fp32 step is exact
    lc, lu = (np.round(np.clip(x, -40, 40) * 1024).astype(np.float32) / 1024 for x in (lc, lu))
    _check(ctx, lc, lu, 2.0, 0.5, 100)
    ctx.hbsjd_destroy()


@pytest.mark.parametrize("V", [4096, 4160, 8192, 16384, 20480])
def test_masked_huge_and_nan_logits(V):
    """Rows as masks leave them, through both kernels (the persistent one runs 4160 to 16384): -inf or the type's lowest
    value in nearly every place, in every other row only (the threshold guess goes from row to row), a span beyond
    fp32 with the threshold inside its upper end, NaN where both branches are masked under guidance, and more NaN than
    V - k, which count among the k largest.  Against the pipeline in 64 bits."""
    import torch
    sh = synth.ModelShape(1, 64, 1, 64, V, 4, 4, 3, "bf16")
    ctx = binding.Context(sh, synth.make_weights(sh, 3, target_entropy=None), 2, 4)
    g = torch.Generator(device="cuda").manual_seed(V)
    rows, low = 300, torch.finfo(torch.float32).min
    base = torch.randn(rows, V, generator=g, device="cuda") * 3
    hide = torch.rand(rows, V, generator=g, device="cuda") < 0.9

    def check(lc, k, lu=None, kept=None):
        p = ctx.hbsjd_probs(lc, lu, 2.0 if lu is not None else 1.0, 1.0, k)
        x = (lc if lu is None else lu + 2.0 * (lc - lu)).double()
        x = x.masked_fill(torch.isnan(x), float("-inf"))
        kth = torch.topk(x, kept or k, dim=-1).values[:, -1:]
        ref = torch.softmax(x.masked_fill(x < kth, float("-inf")), -1)
        assert bool(((p.double() - ref).abs() <= 1e-6 + 1e-5 * ref).all())

    for value in (float("-inf"), low):
        for every in (1, 2):
            lc = base.clone()
            lc[::every][hide[::every]] = value
            check(lc, 1000)
            check(lc, 40)
    lc = base.clone()
    lc[:, 100:107] = 3e38
    lc[:, 107:3000] = -3e38
    for k in (5, 7, 8, 1000):
        check(lc, k)
    masked = [torch.where(hide, float("-inf"), x) for x in (base, base.flip(0))]
    check(masked[0], 200, lu=masked[1])
    lc = base.clone()
    lc[::3, 50:150] = float("nan")
    check(lc[::3].contiguous(), V - 40, kept=V - 140)
    check(lc, 1000)
    ctx.hbsjd_destroy()


@pytest.mark.parametrize("V", [4160, 8256, 12288])
def test_a_low_entry_does_not_cost_the_threshold_guess(V):
    """One entry per row far below the others, as a mask leaves it, in rows whose last chunk is partly or wholly padding. The
    selection starts from a normal fit of a sample that does not see the entry; without the fit it has to cover the row's
    whole range, one bin then holds the rest of the row, and the byte-wise selection runs (12288: 33 us for 100 rows in place
    of 27).  Ten per cent between the two kinds of rows is several times what runs of one kind differ by.  (k = 1500: the
    fit lies below the k-th largest by more than four of its standard errors, so that no row of the hundred misses.)"""
    import torch
    sh = synth.ModelShape(1, 64, 1, 64, V, 4, 4, 3, "bf16")
    ctx = binding.Context(sh, synth.make_weights(sh, 3, target_entropy=None), 2, 4)
    plain = torch.randn(100, V, generator=torch.Generator(device="cuda").manual_seed(V), device="cuda") * 3.5
    masked = plain.clone()
    masked[:, 3000] = -1e6  # (the sample takes entries 0 to 127 of every 4096)
    best = {}
    for _ in range(30):
        for name, x in (("plain", plain), ("masked", masked)):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            p = ctx.hbsjd_probs(x, None, 1.0, 1.0, 1500)
            end.record()
            end.synchronize()
            best[name] = min(best.get(name, 1e9), start.elapsed_time(end))
            if name == "masked":
                assert not bool(p[:, 3000].any())
    print(V, best)
    assert best["masked"] < 1.1 * best["plain"]
    ctx.hbsjd_destroy()
