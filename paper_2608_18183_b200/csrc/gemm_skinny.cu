// bf16 decoder GEMMs for few activation rows: acc[M,N] = A[M,K] . W[N,K]^T with the same fused epilogues as
// gemm_tcgen05.cu, on mma.sync m16n8k16.
//
// What bounds it: the serial chain over K.  The sum of an output element runs over K in steps of 16 in a fixed order
// (the order every GEMM of this library uses, so that a row's bits do not depend on the batch it sits in), and a
// tcgen05.mma takes at least 64 clocks however few rows and columns it has (measured), 5.7 us for K = 2816.  An
// mma.sync step takes 21 clocks as long as an SM runs no more than about eight 16 x 8 tiles, and sums its 16
// products into the accumulator with the same result bit for bit (measured on random operands; the tests compare the
// two kernels), so for tiles this small the legacy instruction is the faster way through K.
//
// Measured, back to back with the weights streaming from HBM, microseconds per launch, tcgen05 kernel -> this one:
// M = 16: N 3072 K 1024 6.1 -> 4.2; N 1024 K 1024 6.0 -> 3.6; N 5632 K 1024 6.7 -> 4.5; N 1024 K 2816 12.6 -> 6.4.
// M = 64: N 3072 K 1024 6.2 -> 5.1; N 1024 K 2816 12.8 -> 7.9; N 1280 K 3456 15.0 -> 9.4.
//
// One CTA per TM x TN tile of C; nothing is persistent.
//   warps 0 .. NW-1  consumers: ldmatrix + mma.sync on a 16-row part of the tile, fragments loaded one k-block ahead;
//                    then the accumulators pass through shared memory so that one thread finishes one row of 32
//                    columns (the unit of the shared epilogue arithmetic and of the partial sums of squares)
//   warp NW          W producer: starts before the grid dependency resolves (weights never change), so the weight
//                    tiles cross HBM and L2 while the previous kernels of the stream run
//   warp NW + 1      A producer: starts once the previous kernel has finished; until then it asks for the weight
//                    tiles that the ring does not hold to be brought to L2
//   warp NW + 2      (epilogues without a residual) collects what the epilogue needs per row: destination, norm
//                    factor, cos / sin
// A copy brings two or four k-blocks (one thread needs about 330 clocks to wait for a stage, arm its barrier and
// issue the copy, whatever its size), and a CTA takes less than half of an SM's shared memory so that the next
// kernel's CTAs are resident, with their weights on the way, while this one runs.
#include <cstdio>

#include "gemm_common.cuh"

namespace hbsjd {

namespace {

template <int TM, int TN, int EPI>
struct SkinnyCfg {
    static constexpr bool RES = EPI == EPI_ADD || EPI == EPI_ADDNORM;
    static constexpr int WM = TM / 16;                    // consumer warps along M, 16 rows each
    static constexpr int WN = TM == 16 ? TN / 16 : 2;     // along N
    static constexpr int NW = WM * WN;
    static constexpr int GN = TN / WN / 16;               // 16-column groups per warp
    static constexpr int HELP = RES ? 0 : 1;              // helper warps
    static constexpr int THREADS = (NW + 2 + HELP) * 32;
    static constexpr int A_BYTES = TM * BK * 2, W_BYTES = TN * BK * 2;  // one k-block
    static constexpr int KG = TN == 32 ? 4 : 2;           // k-blocks per stage
    static constexpr int STAGE_BYTES = KG * (A_BYTES + W_BYTES);
    static constexpr int PITCH = TN + 4;                  // floats per row of the accumulator tile
    static constexpr int ROPE_PITCH = 36;                 // floats per row of a chunk's cos / sin values
    static constexpr int ROW_BYTES = RES ? 0 : TN / 32 * TM * ROPE_PITCH * 4 + 32 * 16;
    static constexpr int FIXED = TM * PITCH * 4 + ROW_BYTES + 16 + 1024;
    static constexpr int MOST = 113 * 1024;               // two CTAs per SM
    static constexpr int STAGES = (MOST - FIXED) / (STAGE_BYTES + 16);
    static constexpr int SMEM = STAGES * (STAGE_BYTES + 16) + FIXED;
    static_assert(NW * 32 >= TN, "one epilogue warp per 32 columns");
    static_assert(STAGES >= 3, "ring depth");
};

__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* map, int x, int y, int z) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(x), "r"(y),
                 "r"(z)
                 : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t r[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// A wait with a limit shorter than the time that mbar_try may sleep (time-out test; in a function of its own: this poll inside
// mbar_wait cost the tcgen05 epilogue 0.5 % of a rollout of six XL images).
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_brief(uint32_t bar, uint32_t parity, volatile uint32_t* abort, uint32_t limit_ns) {
    const unsigned long long t0 = globaltimer_ns();
    while (!mbar_test(bar, parity))
        if (*abort || globaltimer_ns() - t0 > limit_ns) return false;
    return true;
}

template <int TM, int TN, int EPI>
__global__ void __launch_bounds__(SkinnyCfg<TM, TN, EPI>::THREADS, 2)
    k_gemm_skinny(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_w,
                  const GemmArgs g) {
    using cfg = SkinnyCfg<TM, TN, EPI>;
    constexpr int KG = cfg::KG;
    constexpr bool RES = cfg::RES;
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    const uint32_t tile_at = ring + cfg::STAGES * cfg::STAGE_BYTES - raw;  // byte offset of the accumulator tile
    float* acc_tile = (float*)(smem_raw + tile_at);
    float* rope_tile = acc_tile + TM * cfg::PITCH;                            // [TN / 32][TM][ROPE_PITCH]
    size_t* row_off = (size_t*)(rope_tile + TN / 32 * TM * cfg::ROPE_PITCH);  // [32] K/V offset, ~0: row not stored
    float* row_scale = (float*)(row_off + 32);                                // [32]
    const uint32_t full0 = raw + tile_at + TM * cfg::PITCH * 4 + cfg::ROW_BYTES, empty0 = full0 + 8 * cfg::STAGES;
    volatile uint32_t* abort_flag = (volatile uint32_t*)(smem_raw + (empty0 - raw) + 8 * cfg::STAGES);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int N = g.N, tiles_n = N / TN;
    const int m0 = (int)(blockIdx.x / tiles_n) * TM, n0 = (int)(blockIdx.x % tiles_n) * TN;
    const int num_kb = g.K / BK, groups = (num_kb + KG - 1) / KG;

    if (threadIdx.x == 0) {
        for (int s = 0; s < cfg::STAGES; ++s) {
            mbar_init(full0 + 8 * s, 2);        // the two producers, each with its bytes
            mbar_init(empty0 + 8 * s, cfg::NW);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    if (!RES && warp == cfg::NW + 2) {
        // ---------------------------------------------------------------- helper: what the epilogue needs per row
        // (slot tables, page table and rotation table sit behind one another and the norm's partial sums are added
        // in order: all of it off the consumers' path).  The look-ups need nothing of the kernel before this one, so behind a kernel
        // that triggers late they go before the wait.  (24 L images token by token and one L image 0.97 times the time, six
        // XL images 0.986.)
        if (EPI != EPI_QKV || !g.early) pdl_wait();
        const int row = m0 + lane;
        if (lane < TM && row < g.M) {
            if (EPI == EPI_QKV) {
                const RowDst rd = qkv_row(g, row, true);
                row_off[lane] = rd.valid ? rd.kvoff : ~(size_t)0;
                if (rd.valid && n0 < 2 * g.st.D) {
                    const int half = g.st.dh / 2;
                    const float4* tab = reinterpret_cast<const float4*>(g.rope_cs + (size_t)rd.s * half * 2);
#pragma unroll
                    for (int ch = 0; ch < TN / 32; ++ch) {
                        const int at = (((n0 + ch * 32) % g.st.D) % g.st.dh) / 2 >= 16 ? 8 : 0;
                        float4* dst = reinterpret_cast<float4*>(rope_tile + (ch * TM + lane) * cfg::ROPE_PITCH);
#pragma unroll
                        for (int v = 0; v < 8; ++v) dst[v] = tab[at + v];
                    }
                }
            }
            if (EPI == EPI_QKV) pdl_wait();
            row_scale[lane] = g.ssq_in != nullptr ? norm_row_factor(g, row) : 1.0f;
        }
        asm volatile("bar.arrive 1, %0;" ::"n"((cfg::NW + cfg::HELP) * 32) : "memory");
        return;
    }
    if (warp >= cfg::NW) {
        // ---------------------------------------------------------------- producers
        if (lane == 0) {
            const bool is_w = warp == cfg::NW;
            const CUtensorMap* map = is_w ? &map_w : &map_a;
            asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
            if (!is_w && g.w_constant)
                for (int gi = cfg::STAGES; gi < groups; ++gi) tma_prefetch_3d(&map_w, 0, n0, gi * KG);
            if (!is_w || !g.w_constant) pdl_wait();
            const uint32_t bytes = KG * (is_w ? cfg::W_BYTES : cfg::A_BYTES);
            const uint32_t dst0 = ring + (is_w ? KG * cfg::A_BYTES : 0);
            const int y = is_w ? n0 : m0;
            int armed = 0;
            for (int gi = 0; gi < groups; ++gi) {
                const uint32_t st = (uint32_t)gi % cfg::STAGES, ph = ((uint32_t)gi / cfg::STAGES) & 1u;
                if (gi >= cfg::STAGES && !mbar_wait(empty0 + 8 * st, ph ^ 1u, abort_flag)) {
                    *abort_flag = 1;
                    atomicExch(g.error_flag, 7);
                    break;
                }
                // k-blocks past the last one are filled with zeros, so every stage receives the same bytes
                mbar_expect_tx(full0 + 8 * st, bytes);
                tma_load_3d(dst0 + st * cfg::STAGE_BYTES, map, 0, y, gi * KG, full0 + 8 * st);
                ++armed;
            }
            // What this thread has requested must have landed before shared memory is released.  It has, unless
            // somebody gave up: a stage completes with both producers' bytes, or the limit ends the wait.
            const unsigned long long t0 = globaltimer_ns();
            for (int gi = armed > cfg::STAGES ? armed - cfg::STAGES : 0; gi < armed; ++gi)
                while (!mbar_try(full0 + 8 * (gi % cfg::STAGES), (uint32_t)(gi / cfg::STAGES) & 1u))
                    if (globaltimer_ns() - t0 > 1000000000ull) break;
        }
        return;
    }

    // -------------------------------------------------------------------- consumers
    pdl_wait();
    pdl_trigger();  // (late: see pdl_wait)
    const int row = m0 + lane, col = n0 + warp * 32;  // epilogue warp w: columns 32 w .. 32 w + 31 of the tile
    const bool finisher = warp * 32 < TN && lane < TM && row < g.M;
    float4 pre[8];  // old residual values: they travel while the main loop runs
    if (RES && finisher) {
        const float4* hp = reinterpret_cast<const float4*>(g.C + (size_t)row * N + col);
#pragma unroll
        for (int v = 0; v < 8; ++v) pre[v] = hp[v];
    }
    {
        const int wm = warp / cfg::WN, wn = warp % cfg::WN;
        float acc[cfg::GN][2][4];
#pragma unroll
        for (int t = 0; t < cfg::GN; ++t)
#pragma unroll
            for (int h = 0; h < 2; ++h) acc[t][h][0] = acc[t][h][1] = acc[t][h][2] = acc[t][h][3] = 0.f;
        // fragment addresses inside a k-block tile (rows of 128 bytes, 16-byte pieces XOR-swizzled by row & 7)
        const int ar = wm * 16 + (lane & 15), ac = lane >> 4;
        const int br = wn * (TN / cfg::WN) + ((lane >> 4) << 3) + (lane & 7), bc = (lane >> 3) & 1;
        const uint32_t a_row = (uint32_t)ar * 128u, b_row = (uint32_t)br * 128u;
        const uint32_t ax = (uint32_t)(ar & 7), bx = (uint32_t)(br & 7);
        uint32_t fa[2][4][4], fb[2][4][cfg::GN][4];
        auto load_k = [&](uint32_t at, uint32_t bt, int p, int k) {
            ldmatrix_x4(at + (((uint32_t)(2 * k + ac) ^ ax) << 4), fa[p][k]);
#pragma unroll
            for (int t = 0; t < cfg::GN; ++t)
                ldmatrix_x4(bt + (uint32_t)t * 2048u + (((uint32_t)(2 * k + bc) ^ bx) << 4), fb[p][k][t]);
        };
        auto a_at = [&](int kb) {
            return ring + ((uint32_t)(kb / KG) % cfg::STAGES) * cfg::STAGE_BYTES + (uint32_t)(kb % KG) * cfg::A_BYTES + a_row;
        };
        auto b_at = [&](int kb) {
            return ring + ((uint32_t)(kb / KG) % cfg::STAGES) * cfg::STAGE_BYTES + KG * cfg::A_BYTES +
                   (uint32_t)(kb % KG) * cfg::W_BYTES + b_row;
        };
        auto ready = [&](int kb) {  // the k-block's stage has landed: one answer for the warp, whose lanes stay together
            if (kb % KG) return true;
            const uint32_t gi = (uint32_t)(kb / KG);
            const uint32_t bar = full0 + 8 * (gi % cfg::STAGES), ph = (gi / cfg::STAGES) & 1u;
            const bool in = g.acc_wait_ns ? mbar_wait_brief(bar, ph, abort_flag, g.acc_wait_ns) : mbar_wait(bar, ph, abort_flag);
            return __all_sync(0xffffffffu, in) != 0;
        };
        bool ok = ready(0);
        if (ok) {
#pragma unroll
            for (int k = 0; k < 4; ++k) load_k(a_at(0), b_at(0), 0, k);
        }
        auto step = [&](int kb, int p) {
            if (kb + 1 < num_kb) {
                ok = ready(kb + 1);
                if (!ok) return;
            }
            const uint32_t at = a_at(kb + 1), bt = b_at(kb + 1);  // (past the last k-block: a stage of the ring, unused)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                load_k(at, bt, p ^ 1, k);
#pragma unroll
                for (int t = 0; t < cfg::GN; ++t) {
                    mma_bf16(acc[t][0], fa[p][k], fb[p][k][t][0], fb[p][k][t][1]);
                    mma_bf16(acc[t][1], fa[p][k], fb[p][k][t][2], fb[p][k][t][3]);
                }
            }
            if (kb % KG == KG - 1) {  // this warp is done with the stage
                __syncwarp();
                if (lane == 0) mbar_arrive(empty0 + 8 * ((uint32_t)(kb / KG) % cfg::STAGES));
            }
        };
        for (int kb = 0; kb < num_kb && ok; kb += 2) {
            step(kb, 0);
            if (ok && kb + 1 < num_kb) step(kb + 1, 1);
        }
        if (!ok && lane == 0) {
            *abort_flag = 1;
            atomicExch(g.error_flag, 8);
        }
        float* at = acc_tile + (wm * 16 + (lane >> 2)) * cfg::PITCH + wn * (TN / cfg::WN) + (lane & 3) * 2;
#pragma unroll
        for (int t = 0; t < cfg::GN; ++t)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float* p0 = at + t * 16 + h * 8;
                *reinterpret_cast<float2*>(p0) = make_float2(acc[t][h][0], acc[t][h][1]);
                *reinterpret_cast<float2*>(p0 + 8 * cfg::PITCH) = make_float2(acc[t][h][2], acc[t][h][3]);
            }
    }
    asm volatile("bar.sync 1, %0;" ::"n"((cfg::NW + cfg::HELP) * 32) : "memory");
    if (*abort_flag || !finisher) return;
    const float rscale = RES ? 1.0f : row_scale[lane];

    uint32_t r[32];
    {
        const float4* src = reinterpret_cast<const float4*>(acc_tile + lane * cfg::PITCH + warp * 32);
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            const float4 t = src[v];
            r[4 * v] = __float_as_uint(t.x);
            r[4 * v + 1] = __float_as_uint(t.y);
            r[4 * v + 2] = __float_as_uint(t.z);
            r[4 * v + 3] = __float_as_uint(t.w);
        }
    }
    if (RES) {
        // new residual = old + acc, its bf16 copy and the chunk's sum of squares
        const float ss = residual_chunk(pre, r);
        uint4* cp = reinterpret_cast<uint4*>(g.C + (size_t)row * N + col);
#pragma unroll
        for (int v = 0; v < 8; ++v) cp[v] = make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
        if (EPI == EPI_ADDNORM) {
            uint4* hp = reinterpret_cast<uint4*>(g.hb + (size_t)row * N + col);
#pragma unroll
            for (int v = 0; v < 4; ++v)
                hp[v] = make_uint4(pack_bf16x2(__uint_as_float(r[8 * v]), __uint_as_float(r[8 * v + 1])),
                                   pack_bf16x2(__uint_as_float(r[8 * v + 2]), __uint_as_float(r[8 * v + 3])),
                                   pack_bf16x2(__uint_as_float(r[8 * v + 4]), __uint_as_float(r[8 * v + 5])),
                                   pack_bf16x2(__uint_as_float(r[8 * v + 6]), __uint_as_float(r[8 * v + 7])));
            g.ssq_out[(size_t)row * (N / 32) + col / 32] = ss;
        }
    } else if (EPI == EPI_STORE) {
        if (g.ssq_in != nullptr) {
#pragma unroll
            for (int v = 0; v < 32; ++v) r[v] = __float_as_uint(__uint_as_float(r[v]) * rscale);
        }
        uint4* cp = reinterpret_cast<uint4*>(g.C + (size_t)row * N + col);
#pragma unroll
        for (int v = 0; v < 8; ++v) cp[v] = make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
    } else if (EPI == EPI_SWIGLU) {
        uint32_t o[8];
        swiglu_chunk(r, rscale, o);
        uint4* dst = reinterpret_cast<uint4*>(g.out + (size_t)row * (N / 2) + col / 2);
        dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
        dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
    } else {  // EPI_QKV
        const size_t kvoff = row_off[lane];
        if (kvoff == ~(size_t)0) return;  // no input in this row
        const int D = g.st.D;
        const int sec = col / D, cs = col % D;  // 0 q, 1 k, 2 v; a chunk never straddles sections
        uint32_t o[16];
        if (sec < 2) {
            const float4* src = reinterpret_cast<const float4*>(rope_tile + (warp * TM + lane) * cfg::ROPE_PITCH);
#pragma unroll
            for (int v = 0; v < 8; ++v) pre[v] = src[v];
            rope_chunk(r, rscale, pre, o);
        } else {
            plain_chunk(r, rscale, o);
        }
        bf16* base = sec == 0 ? g.out + (size_t)row * D + cs : (bf16*)(sec == 1 ? g.kv.k : g.kv.v) + kvoff + cs;
        uint4* dst = reinterpret_cast<uint4*>(base);
#pragma unroll
        for (int v = 0; v < 4; ++v) dst[v] = make_uint4(o[4 * v], o[4 * v + 1], o[4 * v + 2], o[4 * v + 3]);
    }
}

template <int TM, int TN, int EPI>
cudaError_t launch(const CUtensorMap& ma, const CUtensorMap& mw, GemmArgs g, Stream& s) {
    using cfg = SkinnyCfg<TM, TN, EPI>;
    static int configured[64] = {0};
    cudaError_t e = ensure_dynamic_smem(k_gemm_skinny<TM, TN, EPI>, cfg::SMEM, configured);
    if (e != cudaSuccess) return e;
    const int tiles = (g.N / TN) * ((g.M + TM - 1) / TM);
    g.early = s.late;
    return launch_k(k_gemm_skinny<TM, TN, EPI>, dim3(tiles), dim3(cfg::THREADS), (size_t)cfg::SMEM, s, ma, mw, g);
}

template <int TM, int TN>
cudaError_t launch_epi(int epi, const CUtensorMap& ma, const CUtensorMap& mw, const GemmArgs& g, Stream& s) {
    switch (epi) {
        case EPI_STORE: return launch<TM, TN, EPI_STORE>(ma, mw, g, s);
        case EPI_ADD: return launch<TM, TN, EPI_ADD>(ma, mw, g, s);
        case EPI_SWIGLU: return launch<TM, TN, EPI_SWIGLU>(ma, mw, g, s);
        case EPI_ADDNORM: return launch<TM, TN, EPI_ADDNORM>(ma, mw, g, s);
        default: return launch<TM, TN, EPI_QKV>(ma, mw, g, s);
    }
}

}  // namespace

bool skinny_tile_exists(int code) { return code == 16032 || code == 16064 || code == 32032 || code == 32064; }

// The narrowest tile whose CTAs are all resident at once (two per SM): with more CTAs the second round costs more
// than the tcgen05 kernel's longer chain (back to back, best tile of each kernel: M = 64, N 5632: 8.6 against 7.8 us; M = 128,
// N 3072: 9.1 against 7.5), with fewer the chain is what is left (N 1024: K 2816 at M = 64, 128, 208, 288: 7.3, 8.9, 10.5, 10.5
// against 12.7 to 13.1 us, K 1024 at M = 288, the last that fits: 6.3 against 7.5; N 768 up to M = 384: 6.0 against 6.8; N 1280 up
// to M = 224: 7.1 against 8.1).  The LM head has so many columns that only the widest tile gets close, up to 32 rows
// (M = 32, N 16384: 8.7 against 12.2 us).  Three row tiles of 16 x 64 fit where two of 32 x 32 do not (M = 48, N 5632, 264
// CTAs: 6.6 against 8.7 us).  Of the B, L and XL decoders' products of 16 to 512 rows the rule takes 96, at 0.73 times the
// best tcgen05 tile's time on average and 0.90 at most, and leaves 114, where this kernel takes at least 1.07 times.
int skinny_tile_code(int M, int N, int sms) {
    const long m16 = (M + 15) / 16, m32 = (M + 31) / 32, most = 2L * sms;
    if (N % 64 != 0) return 0;
    if (m16 * (N / 32) <= most) return 16032;
    if (m32 * (N / 32) <= most) return 32032;
    if (m16 * (N / 64) <= most) return 16064;
    if (M <= 32 && N / 64 <= most) return 32064;
    return 0;
}

int gemm_skinny_launch(int epi, int code, const bf16* A, const bf16* W, const GemmArgs& g, int m_rows, Stream& s,
                       char* err, size_t errlen) {
    CUtensorMap ma, mw;
    const int tm = code / 1000, tn = code % 1000, kg = tn == 32 ? 4 : 2;
    if (!make_tensor_map_kblocks(&ma, A, m_rows, g.K, tm, kg) || !make_tensor_map_kblocks(&mw, W, g.N, g.K, tn, kg)) {
        snprintf(err, errlen, "gemm: cuTensorMapEncodeTiled failed (M=%d N=%d K=%d)", g.M, g.N, g.K);
        return -3;
    }
    cudaError_t e;
    switch (code) {
        case 16032: e = launch_epi<16, 32>(epi, ma, mw, g, s); break;
        case 16064: e = launch_epi<16, 64>(epi, ma, mw, g, s); break;
        case 32032: e = launch_epi<32, 32>(epi, ma, mw, g, s); break;
        default: e = launch_epi<32, 64>(epi, ma, mw, g, s); break;
    }
    if (e != cudaSuccess) {
        snprintf(err, errlen, "gemm launch: %s", cudaGetErrorString(e));
        return -3;
    }
    return 0;
}

}  // namespace hbsjd
