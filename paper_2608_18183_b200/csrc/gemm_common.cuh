// Shared pieces of the two bf16 GEMM kernels (gemm_tcgen05.cu, gemm_skinny.cu): the argument block, mbarrier / TMA
// wrappers and the arithmetic of the fused epilogues.  A row's epilogue is one thread's work on 32 consecutive
// columns in both kernels, through the functions below, so that an output element's bits do not depend on which
// kernel computed it.  A sum of two products is spelled out as the fused operation that it is: left to the compiler,
// which of the two is fused could differ from one instantiation to the next.  (One product, as in the sums of squares,
// leaves no choice; spelled out there it cost the 256-wide residual tiles 50 registers and spills.)
#pragma once
#include <cuda.h>

#include "internal.h"

namespace hbsjd {

constexpr int BK = 64;  // 64 bf16 = 128 bytes = one swizzle row

enum { EPI_STORE = 0, EPI_ADD = 1, EPI_SWIGLU = 2, EPI_QKV = 3, EPI_ADDNORM = 4 };

struct GemmArgs {
    float* C;        // STORE / ADD
    bf16* out;       // SWIGLU: [M, N/2];  QKV: q [M, D]
    int M, N, K;
    int32_t* error_flag;
    // RMSNorm folded around the GEMMs (bf16 model): the operand A is the bf16 copy of the UNNORMALISED residual
    // stream and the norm's gain is folded into W, so that norm(x) W^T = r (x W'^T) with the row factor
    // r = rsqrt(mean(x^2) + eps) applied here, in the epilogue, from partial sums of squares
    const float* ssq_in;   // [M][ssq_n] partial sums of squares of A's rows (null: no row factor)
    int ssq_n;             // partials per row = K / 32
    float inv_dim, eps;
    // ADDNORM: C (fp32 residual) += acc, plus what the next GEMM needs
    bf16* hb;              // [M][N] bf16 copy of the updated residual
    float* ssq_out;        // [M][N / 32] sums of squares of the updated residual per 32-column chunk
    int full_tiles;   // CTA pairs: tiles of the walk that are taken whole; the ones behind them go as two halves each
    int w_constant;   // W never changes while the stream runs (model weights): its tiles may be fetched early
    unsigned int acc_wait_ns;  // 0, or a shorter limit for the epilogue's accumulator wait (time-out test)
    // QKV epilogue
    bool early;       // the kernel before triggers late (see pdl_wait)
    State st;
    int layer;
    const float* rope_cs;  // [T][dh/2][2]
    KvView kv;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
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
__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait (about one second unless a shorter limit is given).  Returns false when it gave up or another
// role raised `abort`.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort,
                                          unsigned long long limit_ns = 1000000000ull) {
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = globaltimer_ns();
    const int polls = limit_ns < 1000000ull ? 1 : 128;  // a short limit is checked after every poll
    for (;;) {
        for (int it = 0; it < polls; ++it)
            if (mbar_try(bar, parity)) return true;
        if (*abort) return false;
        if (globaltimer_ns() - t0 > limit_ns) return false;
    }
}


__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// Per-row context of the QKV epilogue: where the token row's q / k / v go.
struct RowDst {
    bool valid;
    int s;        // sequence index (RoPE position)
    size_t kvoff; // element offset of the row's K/V vector in the page pool
};


// Row factor of the folded RMSNorm: the partial sums of squares of this row of A, added in a fixed order.
__device__ __forceinline__ float norm_row_factor(const GemmArgs& g, int row) {
    const float2* pp = reinterpret_cast<const float2*>(g.ssq_in + (size_t)row * g.ssq_n);
    float ss = 0.f;
    for (int v = 0; v < g.ssq_n / 2; ++v) {
        const float2 t = pp[v];
        ss += t.x;
        ss += t.y;
    }
    return 1.0f / sqrtf(__fmaf_rn(ss, g.inv_dim, g.eps));
}

__device__ __forceinline__ RowDst qkv_row(const GemmArgs& g, int row, bool valid) {
    RowDst rd;
    rd.valid = valid;
    rd.s = 0;
    rd.kvoff = 0;
    if (valid) {
        const State& st = g.st;
        int br;
        const int2 at = st.pos_of(row, br);  // (through L2: may be read before the grid wait)
        rd.valid = at.x >= 0;
        if (rd.valid) {
            rd.s = at.y;
            rd.kvoff = g.kv.offset(g.layer, br * st.Bmax + at.x, rd.s);
        }
    }
    return rd;
}

// 16 outputs silu(gate) * up of one chunk: columns (2f, 2f+1) of the accumulator are (gate_f, up_f).  ex2.approx and
// rcp.approx (about 1e-6 relative, far below bf16).
__device__ __forceinline__ void swiglu_chunk(const uint32_t r[32], float rscale, uint32_t o[8]) {
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        const float g0 = __uint_as_float(r[4 * v]) * rscale, u0 = __uint_as_float(r[4 * v + 1]) * rscale;
        const float g1 = __uint_as_float(r[4 * v + 2]) * rscale, u1 = __uint_as_float(r[4 * v + 3]) * rscale;
        o[v] = pack_bf16x2(__fdividef(g0, 1.0f + __expf(-g0)) * u0, __fdividef(g1, 1.0f + __expf(-g1)) * u1);
    }
}

// 16 rotation pairs of one chunk; t[v] = cos, sin of pairs 2v and 2v + 1.
__device__ __forceinline__ void rope_chunk(const uint32_t r[32], float rscale, const float4 t[8], uint32_t o[16]) {
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        const float a0 = __uint_as_float(r[4 * v]) * rscale, b0 = __uint_as_float(r[4 * v + 1]) * rscale;
        const float a1 = __uint_as_float(r[4 * v + 2]) * rscale, b1 = __uint_as_float(r[4 * v + 3]) * rscale;
        o[2 * v] = pack_bf16x2(__fmaf_rn(a0, t[v].x, -(b0 * t[v].y)), __fmaf_rn(a0, t[v].y, b0 * t[v].x));
        o[2 * v + 1] = pack_bf16x2(__fmaf_rn(a1, t[v].z, -(b1 * t[v].w)), __fmaf_rn(a1, t[v].w, b1 * t[v].z));
    }
}

// Residual update of one chunk: r becomes old + r (one fp32 addition per element), the return value is the new chunk's
// sum of squares.
__device__ __forceinline__ float residual_chunk(const float4 old[8], uint32_t r[32]) {
    float ss = 0.f;
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        const float x0 = old[v].x + __uint_as_float(r[4 * v]);
        const float x1 = old[v].y + __uint_as_float(r[4 * v + 1]);
        const float x2 = old[v].z + __uint_as_float(r[4 * v + 2]);
        const float x3 = old[v].w + __uint_as_float(r[4 * v + 3]);
        ss += x0 * x0;
        ss += x1 * x1;
        ss += x2 * x2;
        ss += x3 * x3;
        r[4 * v] = __float_as_uint(x0);
        r[4 * v + 1] = __float_as_uint(x1);
        r[4 * v + 2] = __float_as_uint(x2);
        r[4 * v + 3] = __float_as_uint(x3);
    }
    return ss;
}

__device__ __forceinline__ void plain_chunk(const uint32_t r[32], float rscale, uint32_t o[16]) {
#pragma unroll
    for (int v = 0; v < 16; ++v)
        o[v] = pack_bf16x2(__uint_as_float(r[2 * v]) * rscale, __uint_as_float(r[2 * v + 1]) * rscale);
}

// 32 bytes to a 32-byte aligned address: one whole sector per thread and instruction (two 16-byte stores leave every
// sector half written until the second one arrives, and a warp's rows are too far apart to be merged otherwise).
__device__ __forceinline__ void store_32b(void* dst, const uint32_t* o) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(o[0]), "r"(o[1]), "r"(o[2]),
                 "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7])
                 : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

// ---- few activation rows (gemm_skinny.cu)
// Tile code (rows * 1000 + columns of C per CTA) for a shape, 0 where the tcgen05 kernel is faster.
int skinny_tile_code(int M, int N, int sms);
bool skinny_tile_exists(int code);
// m_rows: row extent of A's tensor map.  Returns 0 or a negative code with a message in err.
int gemm_skinny_launch(int epi, int code, const bf16* A, const bf16* W, const GemmArgs& g, int m_rows, Stream& s,
                       char* err, size_t errlen);

}  // namespace hbsjd
