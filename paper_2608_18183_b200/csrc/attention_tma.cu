// Ragged attention over paged per-image KV caches (Sec. 4.2 "Batched verification"), bf16, head size 64:
// persistent, warp-specialised, K/V blocks moved by TMA.
//
// Work item = one (branch, slot) x HPC heads.  The items of a forward are dealt to the CTAs from a
// list sorted by context length (longest first, alternate stripes reversed), so every CTA streams about the
// same number of key blocks.  Inside a CTA
//   warp 0 (one lane)   producer: for every item, its keys in stages of one or two blocks of 32, K and V of a block and
//                       all heads of the item one cp.async.bulk.tensor copy each (128-byte swizzle), completion on
//                       mbarriers; an item's last stage brings only the blocks that it needs.  The producer runs ahead
//                       across item boundaries: the next item's first keys are in flight while the current item's
//                       last ones are used.
//   warps 1..QB*HPC     consumers: warp (head, q-block) owns 16 consecutive window inputs of one head (its query
//                       fragments come straight from global memory, once per item); online
//                       softmax in fp32, products on mma.sync m16n8k16 (the work is about W FLOP per byte of K, V:
//                       far below the tensor ridge, the tensor cores only keep the math off the critical path).
// Query i of the row sits at sequence index s = c + i and attends keys 0..s: the cached prefix 0..c-1 plus the
// window's own keys c..c+i written just before by the QKV epilogue (intra-window causal mask).  Keys are
// streamed in ABSOLUTE blocks (block j = keys 32 j .. 32 j + 31), so a query's arithmetic depends on its
// sequence index only -- not on the cursor, the window or the batch: prefill chunks, Full and Compact execution
// agree bit for bit.  Rows of a block past the row's last key hold whatever the page holds (finite values of
// older rounds, zeros at first); they are masked before the softmax.
//
// Every mbarrier wait is bounded (about a second); after the limit the kernel raises the error flag, all roles
// leave their loops, the producer waits (bounded again) for its copies in flight, and the CTA returns.
// No multicast anywhere; all tensor maps cover this GPU's own memory.
#include <cuda.h>

#include <cstdio>

#include "internal.h"

namespace hbsjd {

namespace {

constexpr int DH = 64;   // head size
constexpr int KB = 32;   // keys per block
constexpr int TILE_BYTES = KB * DH * 2;  // one K or V tile of one head: 4 KB

// Split by the window's 16-query blocks QB.  A consumer warp takes 16 queries of one head; windows above 32 inputs have
// three or four consumer warps with one head, smaller ones two heads.  What bounds an item is the latency of its chain
// of key blocks, so windows above 16 take two blocks at a time (see attend), at the price of registers for two CTAs per
// SM instead of three: 6 images of 36 layers, contexts up to 576: 16.6 -> 12.9 us per launch, the rollout 0.95 times the
// time; scoring of 128 images (windows of 64) 0.985.  Up to 16 inputs three CTAs with one block at a time stay
// ahead (two at a time: 24 images one token at a time 1.01 to 1.05 times the time, 64 images of 16 inputs 1.02).
template <int QB>
struct AttnCfg {
    static constexpr int HPC = QB >= 3 ? 1 : 2;
    static constexpr int NCW = QB * HPC;                      // consumer warps
    static constexpr int NBLK = QB == 1 ? 1 : 2;              // key blocks per stage
    static constexpr int BLOCK_BYTES = HPC * 2 * TILE_BYTES;  // K and V of 32 keys, all heads of the item
    static constexpr int STAGE_BYTES = NBLK * BLOCK_BYTES;
    static constexpr int STAGES = QB == 1 ? 3 : 98304 / STAGE_BYTES;
    static constexpr int CTAS = QB == 1 ? 3 : 2;              // per SM
};
// A CTA's work list in shared memory: as many entries as leave the CTAs per SM alone; later items (beyond 148 x CTAS x 512)
// are looked up in global memory.
constexpr int LIST_MAX = 512;

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
// Bounded wait (about one second).  Returns false when it gave up or another role raised `abort`.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort) {
    if (mbar_try(bar, parity)) return true;
    unsigned long long t0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (;;) {
        for (int it = 0; it < 64; ++it)
            if (mbar_try(bar, parity)) return true;
        if (*abort) return false;
        unsigned long long t1;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
        if (t1 - t0 > 1000000000ull) return false;
    }
}
// Keys and values are read once per layer and round, a stream larger than L2 at full batch: marked to be evicted first,
// so that the layer's activations and residual stream, which the next kernels read, stay in L2 (rollout of 200 L images with
// long prefixes 0.987 times the time, 128 images 0.994).
__device__ __forceinline__ uint64_t evict_first_policy() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar,
                                            uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(dst),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                                  uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// A tile is rows of 128 bytes (64 bf16) with the 16-byte chunk index XOR-swizzled by (row & 7): the layout a TMA
// copy with 128-byte swizzle leaves in a 1024-byte aligned buffer.
__device__ __forceinline__ uint32_t tile_off(int row, int chunk) { return row * 128 + ((chunk ^ (row & 7)) << 4); }

struct AttnArgs {
    State st;
    int S, layer, G, hpc;  // slots, layer, head groups (heads / hpc), heads per group
    KvView kv;
    const bf16* q;
    bf16* out;
    int32_t* error_flag;
    bool few;    // a small grid of one-block windows: trigger early
    bool early;  // the kernel before triggers late (see pdl_wait)
};

struct Item {
    int row0, crow, c, n, head0;
};
// (first row, n + 128 x first head, c, cache row) of the item at position `pos`, from the slot with that rank of context length
__device__ __forceinline__ int4 item_entry(const AttnArgs& a, int pos) {
    const State& st = a.st;
    const int per_slot = st.nb * a.G;
    const int r = pos / per_slot, rem = pos % per_slot;
    const int br = rem / a.G, g = rem % a.G;
    const int4 e = __ldcg(st.slot_sorted + r);  // first row, n, c, image
    return make_int4(br * st.R + e.x, e.y | (g * a.hpc) << 7, e.z, br * st.Bmax + e.w);
}
// Stripe s of the sorted list: CTA j takes position s * grid + j, in reversed order on odd stripes.
__device__ __forceinline__ int position(int stripe) {
    const int grid = (int)gridDim.x, cta = (int)blockIdx.x;
    return stripe * grid + ((stripe & 1) ? grid - 1 - cta : cta);
}
// The CTA's item of a stripe.  Returns false for an inactive slot.
__device__ __forceinline__ bool item_at(const AttnArgs& a, uint32_t list, int stripe, Item& it) {
    int4 e;
    if (stripe < LIST_MAX)
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(e.x), "=r"(e.y), "=r"(e.z), "=r"(e.w)
                     : "r"(list + 16u * stripe));
    else
        e = item_entry(a, position(stripe));
    it.n = e.y & 127;
    it.c = e.z;
    it.row0 = e.x;
    it.crow = e.w;
    it.head0 = e.y >> 7;
    return it.n != 0;
}

// 2^x for the softmax weights and corrections, by the one instruction.  exp2f also returns results below 2^-126; here they
// meet a normaliser of at least 1 and outputs of the values' size, whose last bits they cannot reach, and the range
// handling was a sixth of this kernel's instructions (rollouts of six XL images and of 24 L images one token at a time
// 0.988 times the time).
__device__ __forceinline__ float ex2(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// One or two consecutive blocks of 32 keys of one head for the 16 queries of a warp: S = Q K^T, causal mask, online
// softmax in fp32, O += P V.  The blocks' score products, maxima, exponentials and row sums do not depend on one
// another (the running maximum is the only link, and a maximum is exact in any order), so two blocks at a time hide
// each other's latencies; the accumulation into the normaliser and into O stays block after block, so the result is
// the same bits as one block at a time.  An all-masked block is an exact no-op.
// kt / vt: shared addresses of the first block's K and V tile; the second block's lie block_bytes further.
template <int NB>
__device__ __forceinline__ void attend(uint32_t kt, uint32_t vt, uint32_t block_bytes, int key0, int s0, int s1,
                                       int q_first, int lane, const uint32_t (&qa)[4][4], float (&o)[8][4], float& m0,
                                       float& m1, float& l0, float& l1) {
    const float sl2 = 0.125f * 1.4426950408889634f;  // 1/sqrt(64) * log2(e)
    float sc[NB][4][4], bx0[NB], bx1[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        // 32 keys: 4 n-tiles of 8 keys
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            sc[b][nt][0] = sc[b][nt][1] = sc[b][nt][2] = sc[b][nt][3] = 0.f;
            const int krow = nt * 8 + (lane & 7);
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t b0, b1, b2, b3;  // k-chunks 2*half (b0,b1) and 2*half+1 (b2,b3)
                ldmatrix_x4(kt + b * block_bytes + tile_off(krow, half * 4 + (lane >> 3)), b0, b1, b2, b3);
                mma_bf16(sc[b][nt], qa[half * 2], b0, b1);
                mma_bf16(sc[b][nt], qa[half * 2 + 1], b2, b3);
            }
        }
    }
    // causal mask and block maxima (rows r0 = lane/4 and r0+8; columns (lane%4)*2 + {0,1} per n-tile).  A block wholly
    // at or before the warp's first query needs no mask; scaling a visible score is the same multiplication either
    // way, so the two paths agree bit for bit.
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const int kb0 = key0 + b * KB;
        float mx0 = -INFINITY, mx1 = -INFINITY;
        if (kb0 + KB - 1 <= q_first) {
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                sc[b][nt][0] *= sl2;
                sc[b][nt][1] *= sl2;
                sc[b][nt][2] *= sl2;
                sc[b][nt][3] *= sl2;
                mx0 = fmaxf(mx0, fmaxf(sc[b][nt][0], sc[b][nt][1]));
                mx1 = fmaxf(mx1, fmaxf(sc[b][nt][2], sc[b][nt][3]));
            }
        } else {
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                const int key = kb0 + nt * 8 + (lane & 3) * 2;
                sc[b][nt][0] = key <= s0 ? sc[b][nt][0] * sl2 : -INFINITY;
                sc[b][nt][1] = key + 1 <= s0 ? sc[b][nt][1] * sl2 : -INFINITY;
                sc[b][nt][2] = key <= s1 ? sc[b][nt][2] * sl2 : -INFINITY;
                sc[b][nt][3] = key + 1 <= s1 ? sc[b][nt][3] * sl2 : -INFINITY;
                mx0 = fmaxf(mx0, fmaxf(sc[b][nt][0], sc[b][nt][1]));
                mx1 = fmaxf(mx1, fmaxf(sc[b][nt][2], sc[b][nt][3]));
            }
        }
        bx0[b] = mx0;
        bx1[b] = mx1;
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        bx0[b] = fmaxf(bx0[b], __shfl_xor_sync(0xffffffffu, bx0[b], 1));
        bx1[b] = fmaxf(bx1[b], __shfl_xor_sync(0xffffffffu, bx1[b], 1));
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        bx0[b] = fmaxf(bx0[b], __shfl_xor_sync(0xffffffffu, bx0[b], 2));
        bx1[b] = fmaxf(bx1[b], __shfl_xor_sync(0xffffffffu, bx1[b], 2));
    }
    float corr0[NB], corr1[NB], rs0[NB], rs1[NB];
    uint32_t pa[NB][2][4];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        // key 0 is visible to every query, so the running maximum is finite from the first block on
        const float mx0 = fmaxf(m0, bx0[b]), mx1 = fmaxf(m1, bx1[b]);
        corr0[b] = ex2(m0 - mx0);
        corr1[b] = ex2(m1 - mx1);
        m0 = mx0;
        m1 = mx1;
        rs0[b] = rs1[b] = 0.f;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const float p0 = ex2(sc[b][nt][0] - mx0), p1 = ex2(sc[b][nt][1] - mx0);
            const float p2 = ex2(sc[b][nt][2] - mx1), p3 = ex2(sc[b][nt][3] - mx1);
            rs0[b] += p0 + p1;
            rs1[b] += p2 + p3;
            // the softmax weights enter the P.V product as bf16 (the normaliser keeps the fp32 values)
            pa[b][nt >> 1][(nt & 1) * 2] = pack_bf16(p0, p1);
            pa[b][nt >> 1][(nt & 1) * 2 + 1] = pack_bf16(p2, p3);
        }
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            o[t][0] *= corr0[b];
            o[t][1] *= corr0[b];
            o[t][2] *= corr1[b];
            o[t][3] *= corr1[b];
        }
        // O += P V: two k-chunks of 16 keys, 8 n-tiles of 8 dims
#pragma unroll
        for (int kc = 0; kc < 2; ++kc) {
            const int vrow = kc * 16 + ((lane >> 3) & 1) * 8 + (lane & 7);
#pragma unroll
            for (int dp = 0; dp < 4; ++dp) {  // pairs of n-tiles: dims dp*16 .. dp*16+15
                uint32_t b0, b1, b2, b3;
                ldmatrix_x4_trans(vt + b * block_bytes + tile_off(vrow, dp * 2 + (lane >> 4)), b0, b1, b2, b3);
                mma_bf16(o[dp * 2], pa[b][kc], b0, b1);
                mma_bf16(o[dp * 2 + 1], pa[b][kc], b2, b3);
            }
        }
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        rs0[b] += __shfl_xor_sync(0xffffffffu, rs0[b], 1);
        rs1[b] += __shfl_xor_sync(0xffffffffu, rs1[b], 1);
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        rs0[b] += __shfl_xor_sync(0xffffffffu, rs0[b], 2);
        rs1[b] += __shfl_xor_sync(0xffffffffu, rs1[b], 2);
        l0 = l0 * corr0[b] + rs0[b];
        l1 = l1 * corr1[b] + rs1[b];
    }
}

template <int QB>
__global__ void __launch_bounds__((AttnCfg<QB>::NCW + 1) * 32, AttnCfg<QB>::CTAS)
    k_attention_tma(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                    const AttnArgs a) {
    // Before or after the wait: a grid that leaves three quarters of the SMs free lets the next kernel's CTAs fetch their
    // weights there early (rollouts of one and two L images, 16 and 32 CTAs, take 0.97 and 0.99 times the time); a larger
    // one is better off without them (three L images, 48 CTAs: 1.007 times with them; six XL images 1.005), and so are
    // windows of two blocks and more, whose attention lasts longer (one to three XL images of window 32, 20 to 60
    // CTAs: 1.016, 1.004, 1.009).
    if (a.few) pdl_trigger();
    using cfg = AttnCfg<QB>;
    constexpr int NCW = cfg::NCW, HPC = cfg::HPC, STAGES = cfg::STAGES;
    constexpr int SK = cfg::NBLK * KB;  // keys per stage
    extern __shared__ unsigned char smem_raw[];
    const State& st = a.st;
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;               // [STAGES][block][K tiles | V tiles]
    const uint32_t bars = ring + STAGES * cfg::STAGE_BYTES;          // full[STAGES], empty[STAGES]
    const uint32_t full0 = bars, empty0 = bars + 8 * STAGES;
    unsigned char* tail = smem_raw + (bars - raw) + 16 * STAGES;
    volatile uint32_t* abort_flag = (volatile uint32_t*)tail;
    const uint32_t list = bars + 16 * STAGES + 16;  // [min(stripes, LIST_MAX)] int4: this CTA's items

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, NCW);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_k) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_v) : "memory");
    }
    if (!a.early) pdl_wait();
    // The kernel before this one is the QKV projection, which lets this grid start only once its own wait is over: all
    // that precedes the projection is complete here, the slot tables and the keys and values of earlier rounds among it
    // (read through L2).  Queries and the window's own keys come after the wait.  The chain of look-ups and the first
    // stages' copies, two microseconds, so lie beside the projection's tail: rollouts of 24 L images token by token
    // 0.97 times the time, one L image 0.96, 64 B images 0.97, six XL images 0.98, 128 L images 0.99.
    const int n_items = a.S * st.nb * a.G;
    int stripes = n_items / (int)gridDim.x;  // stripes with an item of this CTA: the whole ones, and perhaps the last
    if (position(stripes) < n_items) ++stripes;
    // (warp 0 has the barriers to set up)
    for (int s = threadIdx.x - 32; warp > 0 && s < LIST_MAX && s < stripes; s += NCW * 32)
        ((int4*)(tail + 16))[s] = item_entry(a, position(s));
    __syncthreads();

    if (warp == 0) {
        // ---------------------------------------------------------------- producer
        if (lane == 0) {
            const uint64_t policy = evict_first_policy();
            uint32_t gc = 0;  // K/V stages issued so far
            bool ok = true, waited = false;
            for (int stripe = 0; ok && stripe < stripes; ++stripe) {
                Item it;
                if (!item_at(a, list, stripe, it)) continue;
                const int keys = it.c + it.n, nstages = (keys + SK - 1) / SK;
                const int32_t* pages = a.kv.table + (size_t)it.crow * a.kv.pages_per_row;
                const int layer_row0 = a.layer * a.kv.n_pages * a.kv.page;
                int page = pages[0];  // one page holds whole stages (the page size is a multiple of 64)
                for (int sg = 0; sg < nstages; ++sg, ++gc) {
                    const int key0 = sg * SK;
                    // the next stage's page is looked up while this one's turn is waited for
                    const int page_next = sg + 1 < nstages ? pages[(key0 + SK) / a.kv.page] : 0;
                    const uint32_t gs = gc % STAGES, ph = (gc / STAGES) & 1u;
                    if (!mbar_wait(empty0 + 8 * gs, ph ^ 1u, abort_flag)) {
                        ok = false;
                        break;
                    }
                    // the first stage with keys of this forward (an earlier slot of the image may have written any of them)
                    if (!waited && (st.multi || key0 + SK > it.c)) {
                        pdl_wait();
                        waited = true;
                    }
                    const int y = layer_row0 + page * a.kv.page + key0 % a.kv.page;
                    const int blocks = min(cfg::NBLK, (keys - key0 + KB - 1) / KB);
                    mbar_expect_tx(full0 + 8 * gs, blocks * cfg::BLOCK_BYTES);
                    for (int b = 0; b < blocks; ++b) {
                        const uint32_t dst = ring + gs * cfg::STAGE_BYTES + b * cfg::BLOCK_BYTES;
                        tma_load_3d(dst, &map_k, 0, y + b * KB, it.head0, full0 + 8 * gs, policy);
                        tma_load_3d(dst + HPC * TILE_BYTES, &map_v, 0, y + b * KB, it.head0, full0 + 8 * gs, policy);
                    }
                    page = page_next;
                }
            }
            if (!ok) {
                *abort_flag = 1;
                atomicExch(a.error_flag, 5);
            }
            // copies must land before shared memory is released (they have, unless somebody gave up): the stages armed last
            unsigned long long t0, t1;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
            for (uint32_t g2 = gc > (uint32_t)STAGES ? gc - STAGES : 0u; g2 < gc; ++g2)
                while (!mbar_try(full0 + 8 * (g2 % STAGES), (g2 / STAGES) & 1u)) {
                    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
                    if (t1 - t0 > 1000000000ull) break;
                }
        }
    } else {
        // ---------------------------------------------------------------- consumers
        pdl_wait();
        if (!a.few) pdl_trigger();
        const int cw = warp - 1;
        const int wh = cw / QB, wq = cw % QB;  // head within the item, q-block
        uint32_t gc = 0;
        bool ok = true;
        for (int stripe = 0; ok && stripe < stripes; ++stripe) {
            Item it;
            if (!item_at(a, list, stripe, it)) continue;
            const int c = it.c, n = it.n;
            const int keys = c + n, nstages = (keys + SK - 1) / SK;
            // ---- this warp's queries: 16 rows x 64 dims as A fragments.  Fragment rows at or past n repeat the last input:
            // their results are never written back.
            const int i0 = wq * 16 + (lane >> 2), i1 = i0 + 8;
            uint32_t qa[4][4];
            {
                const bf16* qrow0 = a.q + (size_t)(it.row0 + min(i0, n - 1)) * st.D + (it.head0 + wh) * DH;
                const bf16* qrow1 = a.q + (size_t)(it.row0 + min(i1, n - 1)) * st.D + (it.head0 + wh) * DH;
#pragma unroll
                for (int kc = 0; kc < 4; ++kc) {
                    const int d = kc * 16 + (lane & 3) * 2;
                    qa[kc][0] = *reinterpret_cast<const uint32_t*>(qrow0 + d);
                    qa[kc][1] = *reinterpret_cast<const uint32_t*>(qrow1 + d);
                    qa[kc][2] = *reinterpret_cast<const uint32_t*>(qrow0 + d + 8);
                    qa[kc][3] = *reinterpret_cast<const uint32_t*>(qrow1 + d + 8);
                }
            }
            {   // the next item's query rows towards L1 while this item's keys stream (one 128-byte line per row)
                Item nx;
                if (lane < 16 && stripe + 1 < stripes && item_at(a, list, stripe + 1, nx)) {
                    const bf16* nq = a.q + (size_t)(nx.row0 + min(wq * 16 + lane, nx.n - 1)) * st.D + (nx.head0 + wh) * DH;
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(nq));
                }
            }
            const int s0 = c + i0, s1 = c + i1;    // sequence index of this thread's two query rows
            // Keys behind the last one visible to this warp contribute nothing: skip the math (an all-masked
            // block is an exact no-op of the online softmax, so skipping changes no bits).  q-blocks wholly past the
            // window only keep the ring moving.
            const int smax_warp = wq * 16 < n ? c + min(wq * 16 + 15, n - 1) : -1;
            float o[8][4];
#pragma unroll
            for (int t = 0; t < 8; ++t) o[t][0] = o[t][1] = o[t][2] = o[t][3] = 0.f;
            float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;

            for (int sg = 0; sg < nstages; ++sg, ++gc) {
                const uint32_t gs = gc % STAGES, ph = (gc / STAGES) & 1u;
                // The products take all lanes of the warp, so a lane that gave up goes through them too, on whatever the
                // stage holds; the lanes leave together behind them (six XL images 0.2 % faster than with a vote in front).
                const bool in = mbar_wait(full0 + 8 * gs, ph, abort_flag);
                __syncwarp();
                const int key0 = sg * SK;
                const uint32_t kt = ring + gs * cfg::STAGE_BYTES + wh * TILE_BYTES, vt = kt + HPC * TILE_BYTES;
                if (cfg::NBLK == 2 && key0 + KB <= smax_warp)
                    attend<cfg::NBLK>(kt, vt, cfg::BLOCK_BYTES, key0, s0, s1, c + wq * 16, lane, qa, o, m0, m1, l0, l1);
                else if (key0 <= smax_warp)
                    attend<1>(kt, vt, cfg::BLOCK_BYTES, key0, s0, s1, c + wq * 16, lane, qa, o, m0, m1, l0, l1);
                if (!__all_sync(0xffffffffu, in)) {
                    ok = false;
                    break;
                }
                if (lane == 0) mbar_arrive(empty0 + 8 * gs);  // this warp is done with the stage
            }
            if (!ok) break;
            if (smax_warp >= 0) {
                const float inv0 = 1.0f / l0, inv1 = 1.0f / l1;
                item_at(a, list, stripe, it);  // (again: its fields kept over the loop cost spills)
                bf16* orow0 = a.out + (size_t)(it.row0 + i0) * st.D + (it.head0 + wh) * DH;
                bf16* orow1 = a.out + (size_t)(it.row0 + i1) * st.D + (it.head0 + wh) * DH;
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int d = t * 8 + (lane & 3) * 2;
                    if (i0 < it.n) *reinterpret_cast<uint32_t*>(orow0 + d) = pack_bf16(o[t][0] * inv0, o[t][1] * inv0);
                    if (i1 < it.n) *reinterpret_cast<uint32_t*>(orow1 + d) = pack_bf16(o[t][2] * inv1, o[t][3] * inv1);
                }
            }
        }
        if (!ok && lane == 0) {
            *abort_flag = 1;
            atomicExch(a.error_flag, 6);
        }
    }
    __syncthreads();  // no role leaves while another may still touch the ring or the barriers
}

template <int QB>
cudaError_t launch_qb(const CUtensorMap& mk, const CUtensorMap& mv, AttnArgs a, Stream& s) {
    using cfg = AttnCfg<QB>;
    constexpr int threads = (cfg::NCW + 1) * 32;
    constexpr int fixed = 1024 + cfg::STAGES * cfg::STAGE_BYTES + 16 * cfg::STAGES + 16, most = fixed + 16 * LIST_MAX;
    static int configured[64] = {0};
    cudaError_t e = ensure_dynamic_smem(k_attention_tma<QB>, most, configured);
    if (e != cudaSuccess) return e;
    // resident CTAs per SM (registers and shared memory): the grid is exactly what is resident at once
    static int resident[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    dev &= 63;
    if (resident[dev] == 0) {
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_attention_tma<QB>, threads, (size_t)most);
        if (e != cudaSuccess) return e;
        resident[dev] = n < 1 ? 1 : (n > cfg::CTAS ? cfg::CTAS : n);
    }
    const int per_sm = resident[dev];
    const long items = (long)a.S * a.st.nb * a.G;
    long grid = (long)device_sm_count() * per_sm;
    if (grid > items) grid = items;
    a.few = QB == 1 && 4 * grid <= device_sm_count();
    const long stripes = (items + grid - 1) / grid;
    const int smem = fixed + 16 * (int)(stripes < LIST_MAX ? stripes : LIST_MAX);
    a.early = s.late;
    return launch_kc(!a.few, k_attention_tma<QB>, dim3((unsigned)grid), dim3(threads), (size_t)smem, s, 1, mk, mv, a);
}

}  // namespace

bool attention_tma_supported(const State& st, const KvView& kv) {
    return st.dh == DH && st.W <= 64 && kv.page % (2 * KB) == 0 && st.Hh % 2 == 0 && st.slot_sorted != nullptr;
}

int launch_attention_tma(const State& st, int S, int layer, const bf16* q, int q_rows_cap, KvView kv, bf16* out,
                         int32_t* error_flag, Stream& s, char* err, size_t errlen) {
    CUtensorMap mk, mv;
    const int qb = (st.W + 15) / 16;
    const long kv_rows = (long)st.L * kv.n_pages * kv.page;
    (void)q_rows_cap;
    const int hpc = qb == 1 ? AttnCfg<1>::HPC : qb == 2 ? AttnCfg<2>::HPC : AttnCfg<3>::HPC;
    // the pool as (64 columns of a head, rows, heads): the same form as a GEMM operand's k-blocks
    if (kv_rows > 0x7fffffffL || !make_tensor_map_kblocks(&mk, kv.k, (int)kv_rows, st.D, KB, hpc) ||
        !make_tensor_map_kblocks(&mv, kv.v, (int)kv_rows, st.D, KB, hpc)) {
        snprintf(err, errlen, "attention: cuTensorMapEncodeTiled failed");
        return -3;
    }
    AttnArgs a;
    a.st = st;
    a.S = S;
    a.layer = layer;
    a.hpc = hpc;
    a.G = st.Hh / hpc;
    a.kv = kv;
    a.out = out;
    a.q = q;
    a.error_flag = error_flag;
    cudaError_t e;
    switch (qb) {
        case 1: e = launch_qb<1>(mk, mv, a, s); break;
        case 2: e = launch_qb<2>(mk, mv, a, s); break;
        case 3: e = launch_qb<3>(mk, mv, a, s); break;
        default: e = launch_qb<4>(mk, mv, a, s); break;
    }
    if (e != cudaSuccess) {
        snprintf(err, errlen, "attention launch: %s", cudaGetErrorString(e));
        return -3;
    }
    return 0;
}

}  // namespace hbsjd
