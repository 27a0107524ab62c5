// Row-wise kernels of the verifier forward (Sec. 4.2 "Batched verification"): slot set-up / compaction,
// embedding gather, RMSNorm, 2D RoPE + paged KV write, reference attention, SwiGLU, CUDA-core GEMM.
#include <cstring>

#include "internal.h"

namespace hbsjd {

// ------------------------------------------------------------------ set-up / compaction (Sec. 4.3)
// One block.  Builds the slot and row tables of the next forward.  Full: slot b = image b with W rows, n = 0 for inactive
// images.  Compact: active images gathered in increasing image order (block-wide exclusive scan), their inputs' rows
// behind one another without gaps (the scan of n).  Pre-filling and scoring (phase 1) take up to `span` inputs per
// image, in as many slots of W as they fill, always gathered: a layer's keys and values are all written before its
// attention reads them, so the slots of one image need not wait for one another.
// Behind an error that the host has not collected yet (it may run one round ahead) no image is active: the state
// stays the failed round's.
__global__ void k_setup(State st, int phase, int compact, int span) {
    pdl_wait();
    pdl_trigger();
    __shared__ int warp_tot[32], warp_rows[32];
    __shared__ int carry, carry_rows, sum_keys;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) carry = carry_rows = sum_keys = 0;
    const int32_t uncollected = __ldcg(st.counters + CNT_ERROR);  // (in flight over the barrier, beside the cursors)
    auto failed = [&] { return phase == 0 && uncollected != 0; };
    __syncthreads();
    for (int base = 0; base < st.B; base += blockDim.x) {
        const int b = base + tid;
        int c = 0, n = 0;
        if (b < st.B) {
            if (phase == 0) {
                c = st.cursor[b];
                if (c < 0 || c > st.T) {  // cannot be valid: record it and leave the image out of the round
                    atomicExch(&st.counters[CNT_ERROR], 16);
                    c = st.T;
                }
                n = c < st.T && !failed() ? min(st.W, st.T - c) : 0;
            } else {
                c = st.pfill[b];
                n = c < st.klen[b] ? min(span, st.klen[b] - c) : 0;
            }
        }
        int act = n > 0, keys = c + n;  // slots
        if (phase != 0) {
            act = (n + st.W - 1) / st.W;
            keys = 0;
            for (int j = 0; j < act; ++j) keys += c + min(n, (j + 1) * st.W);
        }
        if (act) atomicAdd(&sum_keys, keys);
        // exclusive scans of slots and inputs over the block
        int incl = act, incl_rows = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o), tr = __shfl_up_sync(0xffffffffu, incl_rows, o);
            if (lane >= o) {
                incl += t;
                incl_rows += tr;
            }
        }
        if (lane == 31) {
            warp_tot[wid] = incl;
            warp_rows[wid] = incl_rows;
        }
        __syncthreads();
        int before = carry, rows_before = carry_rows;
        for (int w = 0; w < wid; ++w) {
            before += warp_tot[w];
            rows_before += warp_rows[w];
        }
        const int pos = before + incl - act, row0 = rows_before + incl_rows - n;
        if (b < st.B) {
            const bool gather = compact && !failed();
            const int slot = gather ? pos : b;
            for (int j = 0; j < (gather ? act : 1); ++j) {
                st.slot_img[slot + j] = b;
                st.slot_c[slot + j] = c + j * st.W;
                st.slot_n[slot + j] = min(st.W, n - j * st.W);
                if (st.slot_row != nullptr) st.slot_row[slot + j] = (compact ? row0 : b * st.W) + j * st.W;
            }
        }
        if (st.row_pos != nullptr) {
            // the warp writes its images' rows, one image after the other
            for (unsigned int left = __ballot_sync(0xffffffffu, compact ? act > 0 : b < st.B); left; left &= left - 1) {
                const int src = __ffs(left) - 1;
                const int ib = base + wid * 32 + src;
                const int ic = __shfl_sync(0xffffffffu, c, src), in = __shfl_sync(0xffffffffu, n, src);
                const int ir = compact ? __shfl_sync(0xffffffffu, row0, src) : ib * st.W;
                for (int i = lane; i < (compact ? in : st.W); i += 32)
                    if (ir + i < st.R) st.row_pos[ir + i] = i < in ? make_int2(ib, ic + i) : make_int2(-1, 0);
            }
        }
        __syncthreads();
        if (tid == blockDim.x - 1) {
            carry = before + incl;
            carry_rows = rows_before + incl_rows;
        }
        __syncthreads();
    }
    if (st.row_pos != nullptr && compact)  // rows that the host has allowed for and no input takes
        for (int r = carry_rows + tid; r < st.R; r += blockDim.x) st.row_pos[r] = make_int2(-1, 0);
    // slots by context length, longest first (ties by slot index): the attention kernel deals its work items
    // from this list so that every CTA streams about the same number of key blocks
    if (st.slot_sorted != nullptr) {
        __syncthreads();
        const int n_slots = compact && !failed() ? carry : st.B;
        for (int s0 = tid; s0 < n_slots; s0 += blockDim.x) {
            const int n0 = st.slot_n[s0], c0 = st.slot_c[s0], len = n0 > 0 ? c0 + n0 : -1;
            const int row0 = st.first_row(s0), img0 = st.slot_img[s0];  // (in flight beside the two above)
            int rank = 0;
            for (int s1 = 0; s1 < n_slots; ++s1) {
                const int l1 = st.slot_n[s1] > 0 ? st.slot_c[s1] + st.slot_n[s1] : -1;
                rank += (l1 > len) || (l1 == len && s1 < s0);
            }
            st.slot_sorted[rank] = make_int4(row0, n0, c0, img0);
        }
    }
    if (tid == 0) {
        st.counters[CNT_LIVE_SETUP] = carry;
        st.counters[CNT_SLOTS] = compact ? carry : st.B;
        st.counters[CNT_LIVE] = 0;
        st.counters[CNT_SUM_KEYS] = sum_keys;
        st.counters[CNT_SUM_N] = carry_rows;
    }
}

void launch_setup(const State& st, int phase, int compact, Stream& s, int span) {
    launch_k(k_setup, dim3(1), dim3(1024), 0, s, st, phase, phase == 1 ? 1 : compact, span);
}

__global__ void k_noop() {
    pdl_wait();
    pdl_trigger();
}
void launch_noop(Stream& s) { launch_k(k_noop, dim3(1), dim3(32), 0, s); }

// ------------------------------------------------------------------ embedding gather
// hb / ssq (may be null): bf16 copy of the row and its sums of squares per 32-column chunk (what the RMSNorm
// folded into the first projection reads).  Warp w of the block owns chunks w, w + 4, ...; lane l element l.
template <typename TA>
__global__ void __launch_bounds__(128) k_embed(State st, const TA* __restrict__ tok_emb,
                                               const TA* __restrict__ cls_emb, float* __restrict__ h,
                                               bf16* __restrict__ hb, float* __restrict__ ssq) {
    pdl_wait();
    pdl_trigger();
    const int row = blockIdx.x;
    int br;
    const int2 at = st.pos_of(row, br);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float* dst = h + (size_t)row * st.D;
    const TA* src = nullptr;
    if (at.x >= 0) {
        const int img = at.x, s = at.y;
        if (s == 0) {
            const int cls = br ? st.C : st.label[img];
            src = cls_emb + (size_t)cls * st.D;
        } else {
            src = tok_emb + (size_t)st.seq[(size_t)img * (st.T + 1) + s] * st.D;
        }
    }
    for (int chunk = wid; chunk * 32 < st.D; chunk += 4) {
        const int e = chunk * 32 + lane;
        const float v = (src != nullptr && e < st.D) ? to_f<TA>(src[e]) : 0.f;
        if (e < st.D) {
            dst[e] = v;
            if (hb != nullptr) hb[(size_t)row * st.D + e] = __float2bfloat16_rn(v);
        }
        if (ssq != nullptr) {
            const float ss = warp_sum(v * v);
            if (lane == 0) ssq[(size_t)row * (st.D / 32) + chunk] = ss;
        }
    }
}

template <typename TA>
void launch_embed(const State& st, const TA* tok_emb, const TA* cls_emb, float* h, bf16* hb, float* ssq, Stream& s) {
    launch_k(k_embed<TA>, dim3(st.nb * st.R), dim3(128), 0, s, st, tok_emb, cls_emb, h, hb, ssq);
}
template void launch_embed<float>(const State&, const float*, const float*, float*, bf16*, float*, Stream&);
template void launch_embed<bf16>(const State&, const bf16*, const bf16*, float*, bf16*, float*, Stream&);

// ------------------------------------------------------------------ RMSNorm: out = x * rsqrt(mean(x^2)+eps) * g
// One warp per row; the row stays in registers between the two passes (D <= 2048 through the vector path).
// The sum of squares is reduced in a fixed order that depends on D only.
template <typename TA, int VEC_ITERS>
__global__ void __launch_bounds__(256) k_rmsnorm_warp(const float* __restrict__ h, const TA* __restrict__ gain,
                                                      TA* __restrict__ out, int M, int D, float eps) {
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    // gain read four at a time: 32 two-byte loads per thread in their place cost the rollout of 128 L images 2 %
    struct __align__(4 * sizeof(TA)) Gain4 { TA g[4]; };
    pdl_wait();
    pdl_trigger();
    if (row >= M) return;
    const float4* x4 = reinterpret_cast<const float4*>(h + (size_t)row * D);
    float4 v[VEC_ITERS];
    float ss = 0.f;
#pragma unroll
    for (int it = 0; it < VEC_ITERS; ++it) {
        const int idx = it * 32 + lane;
        if (idx * 4 < D) {
            v[it] = x4[idx];
            ss += v[it].x * v[it].x + v[it].y * v[it].y + v[it].z * v[it].z + v[it].w * v[it].w;
        }
    }
    ss = warp_sum(ss);
    const float r = 1.0f / sqrtf(ss / (float)D + eps);
    TA* o = out + (size_t)row * D;
#pragma unroll
    for (int it = 0; it < VEC_ITERS; ++it) {
        const int idx = it * 32 + lane;
        if (idx * 4 < D) {
            const int e = idx * 4;
            const Gain4 gv = reinterpret_cast<const Gain4*>(gain)[idx];
            const float a = v[it].x * r * to_f<TA>(gv.g[0]), b = v[it].y * r * to_f<TA>(gv.g[1]);
            const float c = v[it].z * r * to_f<TA>(gv.g[2]), d = v[it].w * r * to_f<TA>(gv.g[3]);
            if constexpr (sizeof(TA) == 2) {
                __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
                uint2 pk;
                pk.x = *reinterpret_cast<uint32_t*>(&lo);
                pk.y = *reinterpret_cast<uint32_t*>(&hi);
                *reinterpret_cast<uint2*>(o + e) = pk;
            } else {
                *reinterpret_cast<float4*>(o + e) = make_float4(a, b, c, d);
            }
        }
    }
}

template <typename TA>
__global__ void k_rmsnorm(const float* __restrict__ h, const TA* __restrict__ gain, TA* __restrict__ out, int D,
                          float eps) {
    pdl_wait();
    pdl_trigger();
    __shared__ float red[32];
    const int row = blockIdx.x;
    const float* x = h + (size_t)row * D;
    float ss = 0.f;
    for (int e = threadIdx.x; e < D; e += blockDim.x) ss += x[e] * x[e];
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
    const float r = 1.0f / sqrtf(tot / (float)D + eps);
    TA* o = out + (size_t)row * D;
    for (int e = threadIdx.x; e < D; e += blockDim.x) o[e] = from_f<TA>(x[e] * r * to_f<TA>(gain[e]));
}

template <typename TA>
void launch_rmsnorm(const float* h, const TA* gain, TA* out, int M, int D, float eps, Stream& s) {
    if (D % 4 == 0 && D <= 2048) {
        const int grid = (M + 7) / 8;
        if (D <= 512) launch_k(k_rmsnorm_warp<TA, 4>, dim3(grid), dim3(256), 0, s, h, gain, out, M, D, eps);
        else if (D <= 1024) launch_k(k_rmsnorm_warp<TA, 8>, dim3(grid), dim3(256), 0, s, h, gain, out, M, D, eps);
        else if (D <= 1280) launch_k(k_rmsnorm_warp<TA, 10>, dim3(grid), dim3(256), 0, s, h, gain, out, M, D, eps);
        else launch_k(k_rmsnorm_warp<TA, 16>, dim3(grid), dim3(256), 0, s, h, gain, out, M, D, eps);
    } else {
        launch_k(k_rmsnorm<TA>, dim3(M), dim3(128), 0, s, h, gain, out, D, eps);
    }
}
template void launch_rmsnorm<float>(const float*, const float*, float*, int, int, float, Stream&);
template void launch_rmsnorm<bf16>(const float*, const bf16*, bf16*, int, int, float, Stream&);

// ------------------------------------------------------------------ 2D RoPE + KV write
// One thread per (row, rotation pair).  rope_cs: [T][dh/2][2] cos/sin by sequence index.
template <typename TA>
__global__ void k_rope_kv(State st, int layer, const float* __restrict__ qkv,
                          const float* __restrict__ rope_cs, TA* __restrict__ q, KvView kv) {
    pdl_wait();
    pdl_trigger();
    const int row = blockIdx.x;
    int br;
    const int2 at = st.pos_of(row, br);
    const int D = st.D, half = st.dh / 2;
    TA* qo = q + (size_t)row * D;
    if (at.x < 0) {
        for (int pe = threadIdx.x; pe < D / 2; pe += blockDim.x) {
            qo[2 * pe] = from_f<TA>(0.f);
            qo[2 * pe + 1] = from_f<TA>(0.f);
        }
        return;
    }
    const int s = at.y;
    const int crow = br * st.Bmax + at.x;
    const size_t off = kv.offset(layer, crow, s);
    TA* ko = (TA*)kv.k + off;
    TA* vo = (TA*)kv.v + off;
    const float* src = qkv + (size_t)row * 3 * D;
    for (int pe = threadIdx.x; pe < D / 2; pe += blockDim.x) {
        const int e = pe % half;
        const float cs = rope_cs[((size_t)s * half + e) * 2], sn = rope_cs[((size_t)s * half + e) * 2 + 1];
        const float qa = src[2 * pe], qb = src[2 * pe + 1];
        const float ka = src[D + 2 * pe], kb = src[D + 2 * pe + 1];
        qo[2 * pe] = from_f<TA>(qa * cs - qb * sn);
        qo[2 * pe + 1] = from_f<TA>(qa * sn + qb * cs);
        ko[2 * pe] = from_f<TA>(ka * cs - kb * sn);
        ko[2 * pe + 1] = from_f<TA>(ka * sn + kb * cs);
        vo[2 * pe] = from_f<TA>(src[2 * D + 2 * pe]);
        vo[2 * pe + 1] = from_f<TA>(src[2 * D + 2 * pe + 1]);
    }
}

template <typename TA>
void launch_rope_kv(const State& st, int layer, const float* qkv, const float* rope_cs, TA* q, KvView kv, Stream& s) {
    launch_k(k_rope_kv<TA>, dim3(st.nb * st.R), dim3(128), 0, s, st, layer, qkv, rope_cs, q, kv);
}
template void launch_rope_kv<float>(const State&, int, const float*, const float*, float*, KvView, Stream&);
template void launch_rope_kv<bf16>(const State&, int, const float*, const float*, bf16*, KvView, Stream&);

// ------------------------------------------------------------------ reference attention (one warp per row, head)
// Query at sequence index s = c+i attends keys 0..s of its cache row (cached prefix + this round's
// window up to itself).  Two passes with the scores in shared memory; the reduction order depends on s only.
template <typename TA>
__global__ void k_attention_ref(State st, int layer, const TA* __restrict__ q, KvView kv, TA* __restrict__ out) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ float smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int row = blockIdx.x;
    const int head = blockIdx.y * nw + wid;
    if (head >= st.Hh) return;
    int br;
    const int2 at = st.pos_of(row, br);
    const int dh = st.dh;
    TA* o = out + (size_t)row * st.D + head * dh;
    if (at.x < 0) {
        for (int e = lane; e < dh; e += 32) o[e] = from_f<TA>(0.f);
        return;
    }
    float* sc = smem + (size_t)wid * (st.T + dh);
    float* qs = sc + st.T;
    const int s = at.y;
    const int crow = br * st.Bmax + at.x;
    const TA* qv = q + (size_t)row * st.D + head * dh;
    for (int e = lane; e < dh; e += 32) qs[e] = to_f<TA>(qv[e]);
    __syncwarp();
    const float scale = 1.0f / sqrtf((float)dh);
    float mx = -INFINITY;
    for (int t = lane; t <= s; t += 32) {
        const TA* k = (const TA*)kv.k + kv.offset(layer, crow, t) + head * dh;
        // the value row will be wanted behind the softmax: towards L1 meanwhile
        for (int b = 0; b < dh * (int)sizeof(TA); b += 128)
            asm volatile("prefetch.global.L1 [%0];" ::"l"((const char*)kv.v + ((const char*)k - (const char*)kv.k) + b));
        float dot = 0.f;
        constexpr int PER = 16 / (int)sizeof(TA);  // elements per 16-byte load (head sizes are multiples of 16)
#pragma unroll 4
        for (int e = 0; e < dh; e += PER) {
            const uint4 raw = *reinterpret_cast<const uint4*>(k + e);
            TA v[PER];
            memcpy(v, &raw, 16);
#pragma unroll
            for (int x = 0; x < PER; ++x) dot += qs[e + x] * to_f<TA>(v[x]);
        }
        dot *= scale;
        sc[t] = dot;
        mx = fmaxf(mx, dot);
    }
    mx = warp_max(mx);
    float den = 0.f;
    for (int t = lane; t <= s; t += 32) {
        const float p = expf(sc[t] - mx);
        sc[t] = p;
        den += p;
    }
    den = warp_sum(den);
    __syncwarp();
    for (int e = lane; e < dh; e += 32) {
        // the values of one page at a time, sixteen loads in flight; the sum runs over t in order
        float acc = 0.f;
        for (int t0 = 0; t0 <= s; t0 += kv.page) {
            const TA* v = (const TA*)kv.v + kv.offset(layer, crow, t0) + head * dh + e;
            const int cnt = min(kv.page, s + 1 - t0);
#pragma unroll 16
            for (int t = 0; t < cnt; ++t) acc += sc[t0 + t] * to_f<TA>(v[(size_t)t * st.D]);
        }
        o[e] = from_f<TA>(acc / den);
    }
}

template <typename TA>
void launch_attention_ref(const State& st, int layer, const TA* q, KvView kv, TA* out, Stream& s) {
    const int nw = 4;
    dim3 grid(st.nb * st.R, (st.Hh + nw - 1) / nw);
    const size_t smem = (size_t)nw * (st.T + st.dh) * sizeof(float);
    launch_k(k_attention_ref<TA>, dim3(grid), dim3(nw * 32), smem, s, st, layer, q, kv, out);
}
template void launch_attention_ref<float>(const State&, int, const float*, KvView, float*, Stream&);
template void launch_attention_ref<bf16>(const State&, int, const bf16*, KvView, bf16*, Stream&);

// ------------------------------------------------------------------ SwiGLU: act = silu(gate) * up
template <typename TA>
__global__ void k_swiglu(const float* __restrict__ gu, TA* __restrict__ act, int F) {
    pdl_wait();
    pdl_trigger();
    const int row = blockIdx.y;
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= F) return;
    const float g = gu[(size_t)row * 2 * F + f], u = gu[(size_t)row * 2 * F + F + f];
    act[(size_t)row * F + f] = from_f<TA>(g / (1.0f + expf(-g)) * u);
}

template <typename TA>
void launch_swiglu(const float* gu, TA* act, int M, int F, Stream& s) {
    dim3 grid((F + 255) / 256, M);
    launch_k(k_swiglu<TA>, dim3(grid), dim3(256), 0, s, gu, act, F);
}
template void launch_swiglu<float>(const float*, float*, int, int, Stream&);
template void launch_swiglu<bf16>(const float*, bf16*, int, int, Stream&);

// ------------------------------------------------------------------ CUDA-core GEMM (fp32 model)
// C[M,N] (+)= A[M,K] . W[N,K]^T, fp32 accumulation in increasing k, 64x64 tile, 4x4 outputs per thread.
template <typename TA>
__global__ void __launch_bounds__(256) k_gemm_simt(const TA* __restrict__ A, const TA* __restrict__ W,
                                                   float* __restrict__ C, int M, int N, int K, int accumulate) {
    pdl_wait();
    pdl_trigger();
    __shared__ float As[16][64 + 4];
    __shared__ float Bs[16][64 + 4];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    float acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
    for (int k0 = 0; k0 < K; k0 += 16) {
        for (int idx = threadIdx.x; idx < 64 * 16; idx += 256) {
            const int r = idx >> 4, kk = idx & 15;
            const int gm = m0 + r, gn = n0 + r, gk = k0 + kk;
            As[kk][r] = (gm < M && gk < K) ? to_f<TA>(A[(size_t)gm * K + gk]) : 0.f;
            Bs[kk][r] = (gn < N && gk < K) ? to_f<TA>(W[(size_t)gn * K + gk]) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                a[x] = As[kk][ty * 4 + x];
                b[x] = Bs[kk][tx * 4 + x];
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = fmaf(a[x], b[y], acc[x][y]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const int gm = m0 + ty * 4 + x;
        if (gm >= M) continue;
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int gn = n0 + tx * 4 + y;
            if (gn >= N) continue;
            float* c = C + (size_t)gm * N + gn;
            *c = accumulate ? (*c + acc[x][y]) : acc[x][y];
        }
    }
}

// The same product for problems too small to fill the chip with 64 x 64 tiles (the fp32 decoder's rows of a round):
// bound by latency, not by arithmetic, so a CTA of 64 threads takes a 16 x 16 tile, has every operand panel of its
// ring requested before it needs the first (W's before the preceding kernel has finished when W is a model weight)
// and runs one chain of fused multiply-adds per output in increasing k -- the sum of the 64 x 64 kernel, bit for bit.
// A rollout of four images of the two-layer fp32 model (32 rows, N 64..384, K 64 and 192) spent 11.8 us per launch in
// the 64 x 64 kernel and takes 0.57 times the time with this one.
constexpr int SS_T = 16, SS_K = 64, SS_PITCH = SS_K + 4, SS_STAGES = 4;

__global__ void __launch_bounds__(64) k_gemm_simt_small(const float* __restrict__ A, const float* __restrict__ W,
                                                        float* __restrict__ C, int M, int N, int K, int accumulate,
                                                        int w_constant) {
    pdl_trigger();
    __shared__ __align__(16) float As[SS_STAGES][SS_T * SS_PITCH], Ws[SS_STAGES][SS_T * SS_PITCH];
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const int m0 = blockIdx.y * SS_T, n0 = blockIdx.x * SS_T;
    const int panels = (K + SS_K - 1) / SS_K;
    // 16 bytes per thread and step; rows past the edge and columns past K read as zero (size 0: nothing is fetched)
    auto fetch = [&](const float* __restrict__ src, int rows, int r0, float* dst, int p) {
        for (int idx = tid; idx < SS_T * SS_K / 4; idx += 64) {
            const int r = idx / (SS_K / 4), k = p * SS_K + idx % (SS_K / 4) * 4;
            const int row = r0 + r;
            const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + r * SS_PITCH + idx % (SS_K / 4) * 4);
            const bool in = row < rows && k < K;
            const float* from = in ? src + (size_t)row * K + k : src;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(from), "r"(in ? 16 : 0)
                         : "memory");
        }
    };
    if (w_constant)
        for (int p = 0; p < SS_STAGES && p < panels; ++p) fetch(W, N, n0, Ws[p], p);
    pdl_wait();
    for (int p = 0; p < SS_STAGES; ++p) {  // one group per panel, empty ones included, so that the counts below fit
        if (p < panels) {
            if (!w_constant) fetch(W, N, n0, Ws[p], p);
            fetch(A, M, m0, As[p], p);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, old[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
    if (accumulate) {
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                const int gm = m0 + ty + 8 * x, gn = n0 + tx + 8 * y;
                if (gm < M && gn < N) old[x][y] = C[(size_t)gm * N + gn];
            }
    }
    for (int p = 0; p < panels; ++p) {
        asm volatile("cp.async.wait_group %0;" ::"n"(SS_STAGES - 1) : "memory");
        __syncthreads();
        const float* a = As[p % SS_STAGES] + ty * SS_PITCH;
        const float* w = Ws[p % SS_STAGES] + tx * SS_PITCH;
#pragma unroll
        for (int k = 0; k < SS_K; k += 4) {
            float4 av[2], wv[2];
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                av[x] = *reinterpret_cast<const float4*>(a + 8 * x * SS_PITCH + k);
                wv[x] = *reinterpret_cast<const float4*>(w + 8 * x * SS_PITCH + k);
            }
#pragma unroll
            for (int x = 0; x < 2; ++x)
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    acc[x][y] = fmaf(av[x].x, wv[y].x, acc[x][y]);
                    acc[x][y] = fmaf(av[x].y, wv[y].y, acc[x][y]);
                    acc[x][y] = fmaf(av[x].z, wv[y].z, acc[x][y]);
                    acc[x][y] = fmaf(av[x].w, wv[y].w, acc[x][y]);
                }
        }
        __syncthreads();
        if (p + SS_STAGES < panels) {
            fetch(W, N, n0, Ws[p % SS_STAGES], p + SS_STAGES);
            fetch(A, M, m0, As[p % SS_STAGES], p + SS_STAGES);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const int gm = m0 + ty + 8 * x, gn = n0 + tx + 8 * y;
            if (gm < M && gn < N) C[(size_t)gm * N + gn] = accumulate ? old[x][y] + acc[x][y] : acc[x][y];
        }
}

template <typename TA>
void launch_gemm_simt(const TA* A, const TA* W, float* C, int M, int N, int K, int accumulate, int w_constant,
                      Stream& s) {
    if constexpr (sizeof(TA) == 4) {
        // up to four 16 x 16 tiles per SM (they are resident together); beyond that the 64 x 64 kernel has at least 37
        // tiles and reads every operand four times less often
        const long tiles = (long)((M + SS_T - 1) / SS_T) * ((N + SS_T - 1) / SS_T);
        if (K % 4 == 0 && (((uintptr_t)A | (uintptr_t)W) & 15) == 0 && tiles <= 4L * device_sm_count()) {
            launch_early(k_gemm_simt_small, dim3((N + SS_T - 1) / SS_T, (M + SS_T - 1) / SS_T), dim3(64), 0, s, A, W, C, M,
                     N, K, accumulate, w_constant);
            return;
        }
    }
    dim3 grid((N + 63) / 64, (M + 63) / 64);
    launch_k(k_gemm_simt<TA>, dim3(grid), dim3(256), 0, s, A, W, C, M, N, K, accumulate);
}
template void launch_gemm_simt<float>(const float*, const float*, float*, int, int, int, int, int, Stream&);

}  // namespace hbsjd
