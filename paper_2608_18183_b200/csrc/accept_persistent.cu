// Probability pipeline + SJD accept test (Eq. 5; greedy Eq. 4) as a persistent kernel, for V <= 16384.
//
// One CTA of 1024 threads per SM walks the (slot, window position) items of the round.  The logits of the NEXT
// item (conditional and unconditional row, 2 x 64 KB at V = 16384) are fetched by two bulk copies into a staging
// area in shared memory, completing on an mbarrier, while the current item is processed entirely in registers:
// thread t owns the float4 groups {c * 4096 + 4 t .. + 3}, c = 0..3 (fewer below 8193 entries), of the vocabulary from the
// guided combination to the normalised probabilities, which go to global memory straight from the registers.
//
// What bounds it: instructions, and the waits at the barriers of an item that one row in flight per SM cannot cover (128
// images x 32 positions, V = 16384, guidance, top-k 1000: 135 million warp instructions, 0.57 issued per clock and
// scheduler, 223 us under the profiler where 805 MB take 123).  What went into the instructions: loops without bounds, no
// branch per entry for histogram and exponential, no divisions in the walk, the look-ups of an item by one thread, short
// code (the unrolled waits alone were a third of it): 174 million and 263 us with them, the whole step 294 -> 255 us.
// Taking the next row in beside the selection of the current one hides the waits but costs what it gains: 1024 threads
// 401 us, 512 threads with twice the entries each 325 (0.43 issued: half the warps, and rows that pass through
// shared memory).
//
//   guided = l_u + s (l_c - l_u); / temperature                                  (Sec. 4.2 "fused guided logits")
//   top-k threshold, ties kept: monotone 1024-bin histogram over [guess, max] of the entries above a normal-fit
//   guess of the k-th largest, bins scanned by all 32 warps, the selected bin's few entries ranked exactly
//   p = softmax in fp32; accept flag of draft z: u < min(1, p(z) / q(z)), point-mass proposal: u < p(z)   (Eq. 5)
//   refreshed-draft candidate ~ p by fixed-point sampling: integer weights floor(p 2^30), chunk totals, then an
//   ordered scan inside the one chunk that holds the target -- the result does not depend on evaluation order
//
// Five block-wide barriers per item in the usual case; warp reductions are single redux instructions on integers wherever the
// quantity is an integer or an order-preserving key.  Every reduction is a fixed tree over a fixed ownership of the vocabulary,
// so a position's probabilities are the same bits whichever CTA computes them, in Full and in Compact execution.
#include "accept_common.cuh"
#include "internal.h"

namespace hbsjd {

namespace {

constexpr int PT = 1024;          // threads per CTA
constexpr int PWARPS = PT / 32;
constexpr int MAX_CH = 4;         // float4 groups per thread, at most
constexpr int CHUNK = PT * 4;     // vocabulary entries per chunk
constexpr unsigned int NONE = 0xFFFFFFFFu;

struct PShared {
    unsigned int hist[SEL_BINS];
    unsigned int cand[SEL_CAP];
    unsigned int redk[2][PWARPS];  // keys of the per-warp minimum / maximum
    float fit[2];                  // sum and sum of squares of the sample the threshold guess is fitted to
    float redsum[PWARPS];
    unsigned int wtot[PWARPS];
    unsigned int csum[MAX_CH][PWARPS];  // fixed-point weight sums per chunk and warp (a row's weights total 2^30)
    unsigned int best[2][PWARPS];    // greedy: largest probability bits, then the lowest index holding them
    unsigned int sel_bin, sel_k, ncand, theta;  // sel_bin / sel_k: state of the radix fallback
    struct Draft {
        int z, is_delta, qrow;  // the draft under test (-1: none), point-mass proposal, row of its proposal (-1: invalid)
    } draft[3];
    uint32_t words[3][4];  // both by item modulo 3: a fast thread may start the next item while others finish this one
    unsigned long long mbar;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait (about one second).
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    unsigned long long t0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (;;) {
#pragma unroll 1  // (short code: see the head of the file)
        for (int it = 0; it < 64; ++it)
            if (mbar_try_wait(bar, parity)) return true;
        unsigned long long t1;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
        if (t1 - t0 > 1000000000ull) return false;
    }
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Bin of x >= lo in the selection histogram over [lo, lo + 1024 / scale]: a monotone map (the integer nearest to
// (x - lo) * scale, read off the mantissa after adding 2^23; values beyond the range fall into the last bin).
// Monotone is all the selection needs; both passes use this same function.
__device__ __forceinline__ uint32_t sel_bits(float x, float lo, float scale) {
    return __float_as_uint(fminf(__fmaf_rn(x - lo, scale, 8388608.0f), 8388608.0f + (float)(SEL_BINS - 1)));
}
__device__ __forceinline__ int sel_bin_of(float x, float lo, float scale) { return (int)(sel_bits(x, lo, scale) & 0x7FFFFFu); }
// Counts x in its bin of the histogram at this shared-memory address if x >= lo: predicated, so that a row's entries cost
// no branches (the exponent bits of 2^23 leave the address by the subtraction).
__device__ __forceinline__ void count_if_above(uint32_t hist, float x, float lo, float scale) {
    const uint32_t at = hist - (0x4B000000u << 2) + (sel_bits(x, lo, scale) << 2);
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ge.f32 p, %1, %2;\n\t"
        "@p red.shared::cta.add.u32 [%0], 1;\n\t}" ::"r"(at),
        "f"(x), "f"(lo)
        : "memory");
}

// Key of the k-th largest of the block's register-resident values by radix select, one byte per pass from the
// top; exact for any input.  Only reached when the histogram's selected bin is too crowded for the exact ranking.
template <int NCH>
__device__ __forceinline__ unsigned int radix_select_regs(const float (&x)[NCH][4], int tid, int V, unsigned int k, PShared& sh) {
    const int lane = tid & 31, wid = tid >> 5;
    unsigned int* hist = sh.hist;  // [256] used
    __syncthreads();
    if (tid == 0) {
        sh.sel_bin = 0u;  // prefix
        sh.sel_k = k;
    }
#pragma unroll 1
    for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        const unsigned int mask = pass == 0 ? 0u : (0xFFFFFFFFu << (shift + 8));
        if (tid < 256) hist[tid] = 0u;
        __syncthreads();
        const unsigned int prefix = sh.sel_bin;
#pragma unroll
        for (int c = 0; c < NCH; ++c)
            if (c * CHUNK + tid * 4 < V) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const unsigned int key = float_key(x[c][e]);
                    if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
                }
            }
        __syncthreads();
        if (wid == 0) {
            unsigned int cnt[8], tot = 0;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                cnt[b] = hist[lane * 8 + b];
                tot += cnt[b];
            }
            unsigned int incl = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int tt = __shfl_down_sync(0xffffffffu, incl, o);
                if (lane + o < 32) incl += tt;
            }
            unsigned int above = incl - tot;
            const unsigned int kk = sh.sel_k;
            if (above < kk && kk <= above + tot) {
#pragma unroll
                for (int b = 7; b >= 0; --b) {
                    if (above != NONE && above < kk && kk <= above + cnt[b]) {
                        sh.sel_bin = prefix | ((unsigned int)(lane * 8 + b) << shift);
                        sh.sel_k = kk - above;
                        above = NONE;
                    } else if (above != NONE) {
                        above += cnt[b];
                    }
                }
            }
        }
        __syncthreads();
    }
    return sh.sel_bin;
}

// PROBS: the probability pipeline alone (hbsjd_probs): item = row of a.logits (and a.logits_u), probabilities to a.pcur;
// st has V, W = 1 and a place for the error code.
// NCH: float4 groups per thread.  Rows are padded to NCH * CHUNK entries with NaN, which every comparison drops, so that the
// loops have no bounds.
template <bool CFG, bool PROBS, int NCH>
__global__ void __launch_bounds__(PT, 1) k_accept_persistent(State st, AcceptArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int V = st.V, W = st.W;
    constexpr int VP = NCH * CHUNK;
    float* stage_c = (float*)smem_raw;
    float* stage_u = stage_c + (CFG ? VP : 0);
    PShared& sh = *(PShared*)(stage_u + VP);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t bar = smem_addr(&sh.mbar);
    const uint32_t row_bytes = (uint32_t)V * 4u;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int v = V + tid; v < VP; v += PT) stage_c[v] = stage_u[v] = __int_as_float(0x7FFFFFFF);
    if (!a.early) pdl_wait();
    __syncthreads();

    // slot tables of the round in shared memory: the item walk below reads them at every step
    // (image and n share a word: n is at most 64, images are far fewer than 2^25)
    int* s_imgn = (int*)(&sh + 1);
    int* s_row = s_imgn + a.S;
    int* s_c = s_row + a.S;
    for (int sidx = tid; !PROBS && sidx < a.S; sidx += PT) {
        s_imgn[sidx] = __ldcg(st.slot_img + sidx) << 7 | __ldcg(st.slot_n + sidx);
        s_row[sidx] = st.first_row(sidx);
        s_c[sidx] = __ldcg(st.slot_c + sidx);
    }
    __syncthreads();
    auto n_of = [&](int slot) { return s_imgn[slot] & 127; };
    auto img_of = [&](int slot) { return (int)((unsigned int)s_imgn[slot] >> 7); };

    // An item is (slot, window position); the walk takes every gridDim.x-th of them, without a division per step.
    struct Item { int slot, i; };
    const int step_slot = (int)gridDim.x / W, step_i = (int)gridDim.x % W;
    auto exists = [&](const Item& it) { return it.slot < a.S; };
    auto missing = [&](const Item& it) { return !PROBS && it.slot < a.S && it.i >= n_of(it.slot); };
    auto next = [&](Item it) {
        do {
            it.slot += step_slot;
            it.i += step_i;
            if (it.i >= W) {
                it.i -= W;
                ++it.slot;
            }
        } while (missing(it));
        return it;
    };
    auto issue = [&](const Item& it) {  // thread 0: both rows of item `it` into the staging area
        const size_t row = PROBS ? (size_t)it.slot : (size_t)s_row[it.slot] + it.i;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                     "r"(CFG ? 2u * row_bytes : row_bytes)
                     : "memory");
        bulk_load(smem_addr(stage_c), a.logits + row * V, row_bytes, bar);
        if (CFG) bulk_load(smem_addr(stage_u), a.logits_u + row * V, row_bytes, bar);
    };
    // The state an item needs besides its logits -- the draft token under test, whether its proposal is a point
    // mass, the proposal row and the proposal's entry q(z) -- sits behind three levels of dependent global loads.
    // One thread looks it up one item ahead, with the item's random words (Philox keyed by image, position, round), while the
    // others are in pass 1; behind the next barrier the thread that owns vocabulary entry z requests q(z).  It also records
    // state that cannot be valid.
    auto look_ahead = [&](const Item& it, uint32_t par) {
        const int slot = it.slot, i = it.i, img = img_of(slot), c = s_c[slot];
        PShared::Draft d = {-1, 0, -1};
        if (i < n_of(slot) - 1) {  // the last input of a window has no draft to verify
            const size_t at = (size_t)img * (st.T + 1) + c + i + 1;
            const int z = __ldcg(st.seq + at), qi = c + i - __ldcg(st.qbase + img);  // row of the previous round's probabilities
            d.is_delta = __ldcg(st.delta + at);
            if (z < 0 || z >= V) {
                atomicExch(&st.counters[CNT_ERROR], ERR_BAD_TOKEN);
            } else {
                d.z = z;
                if (qi >= 0 && qi < st.Wmax) d.qrow = img * st.Wmax + qi;
                else if (!d.is_delta && !a.greedy) atomicExch(&st.counters[CNT_ERROR], ERR_BAD_PROPOSAL_ROW);
            }
        }
        philox4x32_10((uint32_t)img, (uint32_t)(c + i + 1), a.round, 0u, a.seed_lo, a.seed_hi, sh.words[par]);
        sh.draft[par] = d;
    };
    // q(z) for the thread that owns entry z (1 elsewhere)
    auto fetch_qz = [&](uint32_t par) {
        const PShared::Draft d = sh.draft[par];
        float qz = 1.0f;
        if (d.z >= 0 && ((d.z % CHUNK) >> 2) == tid && !d.is_delta && !a.greedy)
            qz = d.qrow < 0 ? INFINITY /* alpha = 0: rejected */ : __ldcg(a.pprev + (size_t)d.qrow * V + d.z);
        return qz;
    };
    Item it = {(int)blockIdx.x / W, (int)blockIdx.x % W};
    if (missing(it)) it = next(it);
    uint32_t phase = 0;
    const bool select = a.top_k > 0 && a.top_k < V;
    float qz = 1.0f;
    uint32_t par = 0;  // item modulo 3: the next item's words and draft are written while some threads may still read the last one's
    if (!PROBS) {
        if (exists(it) && tid == PT - 32) look_ahead(it, 0);
        __syncthreads();
        if (exists(it)) qz = fetch_qz(0);
    }
    // Behind the LM head (a.early) all of the above, three levels of look-ups, lies beside its tail: that kernel lets this
    // one start only after its own wait, so slot tables, drafts and the last round's probabilities are complete (rollouts
    // of 64 B images 0.994 times the time, 24 L images token by token and one L image 0.996).
    pdl_wait();
    pdl_trigger();  // k_commit reads what precedes this kernel before its own wait
    if (exists(it) && tid == 0) issue(it);
    sh.hist[tid] = 0u;  // SEL_BINS == PT
    // threshold guess carried from the previous item of this CTA: lower end and bin scale of the selection histogram
    float g_lo = 0.f, g_scale = 0.f;
    bool have_guess = false;
    __syncthreads();

    while (exists(it)) {
        const Item nxt = next(it);
        const uint32_t par_next = par == 2u ? 0u : par + 1u;
        if (!PROBS && tid == PT - 32 && exists(nxt)) look_ahead(nxt, par_next);
        const int slot = it.slot, i = it.i;
        const bool last = PROBS || i == n_of(slot) - 1;
        const int oidx = PROBS ? slot : img_of(slot) * st.Wmax + i;

        const uint32_t* words = sh.words[par];  // written one item ahead (below), published by the barriers between
        if (tid == 0) sh.ncand = 0u;

        // ---- the item's logits have landed (bounded wait; the threads agree on its outcome at barrier (1))
        const bool ok = mbar_wait_bounded(bar, phase);
        phase ^= 1u;

        // ---- pass 1: guided logits into registers, row statistics
        float x[NCH][4];
        float mn = INFINITY, mx = -INFINITY;
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
            const int v = ch * CHUNK + tid * 4;
            float4 lc = *reinterpret_cast<const float4*>(stage_c + v);
            if (CFG) {
                const float4 lu = *reinterpret_cast<const float4*>(stage_u + v);
                lc.x = __fadd_rn(lu.x, __fmul_rn(a.cfg_scale, __fsub_rn(lc.x, lu.x)));
                lc.y = __fadd_rn(lu.y, __fmul_rn(a.cfg_scale, __fsub_rn(lc.y, lu.y)));
                lc.z = __fadd_rn(lu.z, __fmul_rn(a.cfg_scale, __fsub_rn(lc.z, lu.z)));
                lc.w = __fadd_rn(lu.w, __fmul_rn(a.cfg_scale, __fsub_rn(lc.w, lu.w)));
            }
            if (a.temperature != 1.0f) {  // (here, not in a loop behind: 60 images x 16 positions 107 -> 105 us)
                lc.x = __fdiv_rn(lc.x, a.temperature);
                lc.y = __fdiv_rn(lc.y, a.temperature);
                lc.z = __fdiv_rn(lc.z, a.temperature);
                lc.w = __fdiv_rn(lc.w, a.temperature);
            }
            x[ch][0] = lc.x; x[ch][1] = lc.y; x[ch][2] = lc.z; x[ch][3] = lc.w;
        }
        if (have_guess) {  // selection histogram with the carried guess, verified after the barrier
            const uint32_t hist = smem_addr(sh.hist);
#pragma unroll
            for (int ch = 0; ch < NCH; ++ch)
#pragma unroll
                for (int e = 0; e < 4; ++e) count_if_above(hist, x[ch][e], g_lo, g_scale);
        }
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
            mn = fminf(fminf(mn, x[ch][0]), fminf(fminf(x[ch][1], x[ch][2]), x[ch][3]));
            mx = fmaxf(fmaxf(mx, x[ch][0]), fmaxf(fmaxf(x[ch][1], x[ch][2]), x[ch][3]));
        }
        // minimum / maximum of the row: one warp reduction instruction each on the order-preserving keys
        {
            const unsigned int kmn = __reduce_min_sync(0xffffffffu, float_key(mn));
            const unsigned int kmx = __reduce_max_sync(0xffffffffu, float_key(mx));
            if (lane == 0) {
                sh.redk[0][wid] = kmn;
                sh.redk[1][wid] = kmx;
            }
        }
        // (1) staging read by everyone; partial statistics, histogram zeros and words published
        if (!__syncthreads_and(ok ? 1 : 0)) {
            if (tid == 0) atomicExch(&st.counters[CNT_ERROR], 4);
            break;  // a copy never arrived; nothing else is in flight (the next item's copies are issued below)
        }
        if (tid == 0 && exists(nxt)) issue(nxt);  // the next item's rows stream in behind the rest of this one
        float qz_next = 1.0f;
        if (!PROBS && exists(nxt)) qz_next = fetch_qz(par_next);
        mn = key_float(__reduce_min_sync(0xffffffffu, sh.redk[0][lane]));
        mx = key_float(__reduce_max_sync(0xffffffffu, sh.redk[1][lane]));

        // ---- exact top-k threshold (ties kept).  The selection histogram covers [lo, lo + 1024 / scale] with (lo,
        // scale) from, in turn: the guess carried from this CTA's previous item (the histogram was then filled during
        // pass 1), a normal fit of this row's sample, the row's whole range.  A source whose lower end lies above
        // the k-th largest is detected by the count and the next one is tried; the result is exact whatever the source.
        float thr = -INFINITY;
        if (select) {
            if (!(mx > mn)) {
                thr = mn;  // all entries equal: everything is kept
                if (have_guess) {
                    __syncthreads();
                    sh.hist[tid] = 0u;
                }
                have_guess = false;
            } else {
                const unsigned int k = (unsigned int)a.top_k;
                unsigned int theta = 0u;
                float lo = g_lo, scale = g_scale;
                bool found = false;
#pragma unroll 1
                for (int source = have_guess ? 0 : 1; source < 3; ++source) {
                    if (source > 0) {
                        if (source == 1) {
                            // The sample: warp 0's 128 entries of every chunk (vocabulary order carries no structure),
                            // without the padding, which would make the sums NaN.  Taken here, where a row without
                            // a carried guess needs it, and not in pass 1 of every row (1537 rows: 93.2 -> 92.3 us).
                            if (wid == 0) {
                                float s1 = 0.f, s2 = 0.f;
#pragma unroll
                                for (int ch = 0; ch < NCH; ++ch)
                                    if (ch * CHUNK + tid * 4 < V) {
                                        s1 += (x[ch][0] + x[ch][1]) + (x[ch][2] + x[ch][3]);
                                        s2 += (x[ch][0] * x[ch][0] + x[ch][1] * x[ch][1]) +
                                              (x[ch][2] * x[ch][2] + x[ch][3] * x[ch][3]);
                                    }
                                s1 = warp_sum(s1);
                                s2 = warp_sum(s2);
                                if (lane == 0) {
                                    sh.fit[0] = s1;
                                    sh.fit[1] = s2;
                                }
                            }
                            __syncthreads();
                            int fit_n = 0;
#pragma unroll
                            for (int ch = 0; ch < NCH; ++ch) fit_n += max(0, min(128, V - ch * CHUNK));
                            const float mean = sh.fit[0] / (float)fit_n;
                            const float sd = sqrtf(fmaxf(sh.fit[1] / (float)fit_n - mean * mean, 0.f));
                            lo = topk_guess(mean, sd, a.top_k, V);
                            if (!(lo > mn) || !(lo < mx)) {
                                lo = mn;
                                source = 2;
                            }
                        } else {
                            lo = mn;
                        }
                        scale = (float)SEL_BINS / (mx - lo);
                        if (!(scale > 0.f)) break;  // -inf among the entries, or a span beyond fp32: no bins
#pragma unroll
                        for (int ch = 0; ch < NCH; ++ch)
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                count_if_above(smem_addr(sh.hist), x[ch][e], lo, scale);
                        __syncthreads();  // (2) only without a carried guess
                    }
                    // bins from the top: warp w, lane l looks at bin 1023 - (32 w + l)
                    const unsigned int tot = __reduce_add_sync(0xffffffffu, sh.hist[SEL_BINS - 1 - (wid * 32 + lane)]);
                    if (lane == 0) sh.wtot[wid] = tot;
                    __syncthreads();  // (3)
                    // every warp locates the bin of the k-th largest by itself: first the warp-sized group of bins ...
                    unsigned int winc = sh.wtot[lane];
                    const unsigned int wcnt = winc;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const unsigned int tt = __shfl_up_sync(0xffffffffu, winc, o);
                        if (lane >= o) winc += tt;
                    }
                    const unsigned int wmask = __ballot_sync(0xffffffffu, winc >= k);
                    if (wmask == 0u) {  // fewer than k entries at or above lo: the next source (uniform decision)
                        __syncthreads();
                        sh.hist[tid] = 0u;
                        __syncthreads();
                        continue;
                    }
                    const int wsel = __ffs(wmask) - 1;
                    const unsigned int above_w = __shfl_sync(0xffffffffu, winc - wcnt, wsel);
                    // ... then the bin inside that group
                    const unsigned int bcnt = sh.hist[SEL_BINS - 1 - (wsel * 32 + lane)];
                    unsigned int binc = bcnt;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const unsigned int tt = __shfl_up_sync(0xffffffffu, binc, o);
                        if (lane >= o) binc += tt;
                    }
                    const int lsel = __ffs(__ballot_sync(0xffffffffu, above_w + binc >= k)) - 1;
                    const int bsel = SEL_BINS - 1 - (wsel * 32 + lsel);
                    const unsigned int krem = k - (above_w + __shfl_sync(0xffffffffu, binc - bcnt, lsel));
                    // entries of the selected bin: a two-compare interval test a little wider than the bin, the
                    // exact bin function only inside it (the last bin also takes everything above the range)
                    const float inv_scale = 1.0f / scale;
                    const float c_lo = fmaxf(lo, lo + ((float)bsel - 1.0f) * inv_scale);
                    const float c_hi = bsel == SEL_BINS - 1 ? INFINITY : lo + ((float)bsel + 1.0f) * inv_scale;
#pragma unroll
                    for (int ch = 0; ch < NCH; ++ch) {
                        bool any = false;  // few groups hold one: a branch per group, not per entry
#pragma unroll
                        for (int e = 0; e < 4; ++e) any |= (x[ch][e] >= c_lo) & (x[ch][e] <= c_hi);
                        if (any) {
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (x[ch][e] >= c_lo && x[ch][e] <= c_hi && sel_bin_of(x[ch][e], lo, scale) == bsel) {
                                    const unsigned int sidx = atomicAdd(&sh.ncand, 1u);
                                    if (sidx < (unsigned int)SEL_CAP) sh.cand[sidx] = float_key(x[ch][e]);
                                }
                        }
                    }
                    __syncthreads();  // (5)
                    sh.hist[tid] = 0u;  // every read of the histogram is behind us: clean for the next item's pass 1
                    const int nc = (int)sh.ncand;
                    // the key with (#strictly greater) < krem <= (#greater or equal) is the krem-th largest of the bin
                    if (nc <= 32) {  // the usual case: every warp ranks the few candidates by itself
                        const unsigned int ku = lane < nc ? sh.cand[lane] : 0u;
                        unsigned int gt = 0, ge = 0;
                        for (int w2 = 0; w2 < nc; ++w2) {
                            const unsigned int kw = sh.cand[w2];
                            gt += kw > ku;
                            ge += kw >= ku;
                        }
                        const unsigned int hit = __ballot_sync(0xffffffffu, lane < nc && gt < krem && krem <= ge);
                        theta = __shfl_sync(0xffffffffu, ku, __ffs(hit) - 1);
                    } else if (nc > SEL_CAP) {
                        break;
                    } else {
#pragma unroll 1
                        for (int u = tid; u < nc; u += PT) {
                            const unsigned int ku = sh.cand[u];
                            unsigned int gt = 0, ge = 0;
                            for (int w2 = 0; w2 < nc; ++w2) {
                                const unsigned int kw = sh.cand[w2];
                                gt += kw > ku;
                                ge += kw >= ku;
                            }
                            if (gt < krem && krem <= ge) sh.theta = ku;  // every such thread writes the same key
                        }
                        __syncthreads();  // (6)
                        theta = sh.theta;
                    }
                    found = true;
                    break;
                }
                if (!found) {  // no histogram, a crowded bin, or fewer than k entries that compare (NaN): by the keys
                    theta = radix_select_regs(x, tid, V, k, sh);
                    __syncthreads();
                    sh.hist[tid] = 0u;  // the radix passes used the first 256 bins
                }
                thr = key_float(theta);
                // the next item's guess: a lower end a little below this threshold, a top a little above this maximum
                // (0.1 of the span: a step at 128 images, window 32, top-k 1000 took 310 us with 0.3, 303 with 0.1 and
                // 0.05, 307 with 0.02, where rows start to miss the guess; the rollouts do not care)
                g_lo = thr - 0.1f * (mx - thr);
                g_scale = (float)SEL_BINS / (1.2f * (mx - thr));
                have_guess = mx > thr && g_scale > 0.f && g_lo > -INFINITY;
            }
        }

        // ---- exp and normalisation (ex2.approx and a multiplication by 1/sum: inside the probability tolerance,
        // and every downstream decision uses these very numbers)
        float part = 0.f;
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                // (dropped entries, and those past V, by exp(-inf): no branch around the exponential)
                x[ch][e] = __expf(x[ch][e] >= thr ? x[ch][e] - mx : -INFINITY);
                part += x[ch][e];
            }
        part = warp_sum(part);
        if (lane == 0) sh.redsum[wid] = part;
        __syncthreads();  // (7)
        const float den = warp_sum(sh.redsum[lane]);
        const float inv = 1.0f / den;
        // fixed-point weights floor(p 2^30): the whole row totals 2^30 (1 + 1e-3) at most, so 32-bit sums are exact
        float* pout = a.pcur + (size_t)oidx * V;
        unsigned int wc[NCH];
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
            const int v = ch * CHUNK + tid * 4;
#pragma unroll
            for (int e = 0; e < 4; ++e) x[ch][e] *= inv;
            if (!PROBS) wc[ch] = fixed_weight(x[ch][0]) + fixed_weight(x[ch][1]) + fixed_weight(x[ch][2]) + fixed_weight(x[ch][3]);
            if (v < V) *reinterpret_cast<float4*>(pout + v) = make_float4(x[ch][0], x[ch][1], x[ch][2], x[ch][3]);
        }

        if (PROBS) {
            // the probabilities are all that is wanted
        } else if (a.greedy) {
            // argmax, lowest index on ties: the largest probability bits, then the lowest index that holds them
            unsigned int bb = 0u;
#pragma unroll
            for (int ch = 0; ch < NCH; ++ch)
#pragma unroll
                for (int e = 0; e < 4; ++e) bb = max(bb, __float_as_uint(x[ch][e]));  // p >= 0: bits are ordered
            bb = __reduce_max_sync(0xffffffffu, bb);
            if (lane == 0) sh.best[0][wid] = bb;
            __syncthreads();  // (8)
            bb = __reduce_max_sync(0xffffffffu, sh.best[0][lane]);
            unsigned int bi = NONE;
#pragma unroll
            for (int ch = NCH - 1; ch >= 0; --ch)
#pragma unroll
                for (int e = 3; e >= 0; --e) {
                    const int v = ch * CHUNK + tid * 4 + e;
                    if (v < V && __float_as_uint(x[ch][e]) == bb) bi = (unsigned int)v;
                }
            bi = __reduce_min_sync(0xffffffffu, bi);
            if (lane == 0) sh.best[1][wid] = bi;
            __syncthreads();  // (9)
            bi = __reduce_min_sync(0xffffffffu, sh.best[1][lane]);
            if (tid == 0) {
                const int am = (int)bi;
                a.cand_rep[oidx] = am;
                a.cand_ref[oidx] = am;
                a.flag[oidx] = (!last && sh.draft[par].z == am) ? 1 : 0;
            }
        } else {
            // accept test (Eq. 5) by the owner of entry z
            const int z = sh.draft[par].z;
            if (!last && z < 0 && tid == 0) a.flag[oidx] = 0;  // invalid draft token: rejected
            if (z >= 0 && ((z % CHUNK) >> 2) == tid) {
                // p(z) out of the registers by a masked sum (a computed index would move the row to local memory)
                const int zc = z / CHUNK, ze = z & 3;
                float pz = 0.f;
#pragma unroll
                for (int ch = 0; ch < NCH; ++ch)
#pragma unroll
                    for (int e = 0; e < 4; ++e) pz = __fmaf_rn((ch == zc && e == ze) ? 1.0f : 0.0f, x[ch][e], pz);
                const float alpha = sh.draft[par].is_delta ? pz : fminf(1.0f, __fdiv_rn(pz, qz));
                const float u = (float)(words[0] >> 8) * (1.0f / 16777216.0f);
                a.flag[oidx] = (u < alpha) ? 1 : 0;
            }
            // refreshed draft candidate ~ p (word 2): chunk totals, then the ordered scan inside one chunk
#pragma unroll
            for (int ch = 0; ch < NCH; ++ch) {
                const unsigned int ws = __reduce_add_sync(0xffffffffu, wc[ch]);
                if (lane == 0) sh.csum[ch][wid] = ws;
            }
            __syncthreads();  // (8)
            unsigned int ctot[NCH], S = 0;
#pragma unroll
            for (int ch = 0; ch < NCH; ++ch) {
                ctot[ch] = __reduce_add_sync(0xffffffffu, sh.csum[ch][lane]);
                S += ctot[ch];
            }
            if (S == 0) {
                if (tid == 0) a.cand_ref[oidx] = -1;
            } else {
                const unsigned int target = (unsigned int)(((unsigned long long)words[2] * S) >> 32);  // < S
                unsigned int run = 0, mine = 0, wsel = 0;
                int cs = 0;
                {
                    unsigned int start = 0;
#pragma unroll
                    for (int ch = 0; ch < NCH; ++ch) {  // the chunk whose span of the running sum holds the target
                        if (target >= start && target - start < ctot[ch]) {
                            cs = ch;
                            run = start;
                            mine = wc[ch];
                            wsel = lane < wid ? sh.csum[ch][lane] : 0u;
                        }
                        start += ctot[ch];
                    }
                }
                // The warp whose groups hold it, warps before it counted, then lanes before its thread; the others are done
                const unsigned int wbase = run + __reduce_add_sync(0xffffffffu, wsel);
                if (target >= wbase && target - wbase < sh.csum[cs][wid]) {
                    unsigned int incl = mine;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const unsigned int tt = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += tt;
                    }
                    const unsigned int start = wbase + incl - mine;
                    if (target >= start && target - start < mine) {  // exactly one thread
                        unsigned int r = start;
                        int pick = 3;
                        bool found = false;
#pragma unroll
                        for (int ch = 0; ch < NCH; ++ch)
                            if (ch == cs) {
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    r += fixed_weight(x[ch][e]);
                                    if (!found && r > target) {
                                        pick = e;
                                        found = true;
                                    }
                                }
                            }
                        a.cand_ref[oidx] = cs * CHUNK + tid * 4 + pick;
                    }
                }
            }
        }
        it = nxt;
        par = par_next;
        qz = qz_next;
    }
}

}  // namespace

// Chunks a row is padded to: 1, 2 or 4.
static int row_chunks(int V) { return V <= CHUNK ? 1 : V <= 2 * CHUNK ? 2 : 4; }
static int smem_bytes(bool cfg, int V, int table_slots) {
    return (cfg ? 2 : 1) * row_chunks(V) * CHUNK * (int)sizeof(float) + (int)sizeof(PShared) + 3 * table_slots * (int)sizeof(int);
}

// The slot tables of a round have to fit beside the rows (7000 slots at V = 16384 with guidance, 15600 up to 4096).  The batch
// decides, not the round's slots: the kernels add a row's terms in different orders, and Compact execution, whose slots
// fall with the live images, has to give Full execution's bits.
bool accept_persistent_supported(const State& st) {
    return st.V <= MAX_CH * CHUNK && st.V % 4 == 0 && st.B <= 65536 && smem_bytes(st.nb == 2, st.V, st.B) <= 227 * 1024;
}

template <bool CFG, bool PROBS, int NCH>
static void launch_nch(const State& st, const AcceptArgs& a, int n_sms, Stream& s) {
    static int configured[64] = {0};
    const int bytes = smem_bytes(CFG, st.V, PROBS ? 0 : a.S);
    const int items = a.S * st.W;
    ensure_dynamic_smem(k_accept_persistent<CFG, PROBS, NCH>, bytes, configured);
    launch_k(k_accept_persistent<CFG, PROBS, NCH>, dim3(items < n_sms ? items : n_sms), dim3(PT), bytes, s, st, a);
}

template <bool CFG, bool PROBS>
static void launch(const State& st, const AcceptArgs& a, int n_sms, Stream& s) {
    switch (row_chunks(st.V)) {
        case 1: launch_nch<CFG, PROBS, 1>(st, a, n_sms, s); break;
        case 2: launch_nch<CFG, PROBS, 2>(st, a, n_sms, s); break;
        default: launch_nch<CFG, PROBS, 4>(st, a, n_sms, s);
    }
}

void launch_accept_persistent(const State& st, const AcceptArgs& a, int n_sms, Stream& s) {
    AcceptArgs b = a;
    b.early = a.early && s.late;
    if (st.nb == 2) launch<true, false>(st, b, n_sms, s);
    else launch<false, false>(st, b, n_sms, s);
}

void launch_probs_persistent(const float* lc, const float* lu, int rows, int V, float cfg_scale, float temperature,
                             int top_k, float* p, int32_t* counters, int n_sms, Stream& s) {
    State st{};
    st.V = V;
    st.W = 1;
    st.counters = counters;
    AcceptArgs a{};
    a.logits = lc;
    a.logits_u = lu;
    a.pcur = p;
    a.S = rows;
    a.cfg_scale = cfg_scale;
    a.temperature = temperature;
    a.top_k = top_k;
    if (lu) launch<true, true>(st, a, n_sms, s);
    else launch<false, true>(st, a, n_sms, s);
}

}  // namespace hbsjd
