// Prefix build on the tensor cores (Algorithm 1, the prefix build; Eq. 1): for every packed (hidden state, token) pair
//     u = W_fc [h ; E[id]] + rho_0,   a = gamma_1 * u / rms(u),   K = RoPE(W_k a + b_k, position),   V = W_v a + b_v
// and K, V go to the pair's cache row.  Unlike a draft step this is a dense contraction - thousands of pairs share
// every weight tile - so it runs as two tcgen05 GEMMs with the pairs as the M operand and the weight rows as N:
//   GEMM 1 (fusion FC):  pairs x [2d] x [d rows].  The k-blocks of the hidden half come from the caller's hidden
//                        states, those of the embedding half from a buffer of gathered embedding rows.  Output
//                        stage: + rho_0, per-pair partial sums of squares of the tile's columns, gamma_1 * u as bf16
//                        (pair-major, the operand of GEMM 2).  The RMSNorm scale is applied after GEMM 2.
//   GEMM 2 (K and V):    pairs x [d] x [2 * Hkv * dh rows].  Output stage: scale by 1/rms, bias, rotate K at the
//                        pair's position, store to the cache rows; pending pairs (row -1) are skipped.
//
// What bounds it is the path from L2 to shared memory: a 128 x 128 tile computed by one CTA needs 128 bytes per SM and
// clock of tensor time, twice what an SM can fetch.  So two CTAs (a cluster of two: the SMs of one TPC) work on one
// tile of 256 pairs x 256 weight rows with cta_group::2 MMAs: each CTA stages its own 128 pairs and HALF of the weight
// rows, which the tensor cores of both read - 64 bytes per SM and clock.  With the pairs as M every thread of the
// output stage owns one pair: sums of squares, the rotation and 16-byte stores need no exchange between threads.
// The kernel is persistent (one cluster per TPC) with two accumulators in tensor memory, so that a tile's output stage
// runs under the next tile's MMAs; consecutive tiles go through the weight rows first (the weights stay in L2, the pairs
// are read from memory once).
//
// 34 800 pairs of the LLaVA shape (16 sequences of 2176): 3.5 ms, 1.35 PFLOP/s (of 1.4 to 1.7 for a library GEMM; the SM
// clock drops to 1.3-1.5 GHz under the power cap); with 128 x 128 tiles, one per CTA and launch slot, and the tile turned in
// shared memory for the output stage 7.9 ms.  17 to 256 pairs: 65 to 70 us (87 to 91 before the
// MMAs were issued by an elected thread), a serial chain of 128 k-blocks in GEMM 1.
//
// Warp 0 (one thread, both CTAs) issues the copies, warp 1 (one thread of the leader, rank 0) the MMAs for both, warps
// 2-5 run the output stage.  A stage's full barrier lives in the leader and counts the bytes of both CTAs; tcgen05.commit
// hands stages and accumulators back to both CTAs.  Every wait is bounded; a wait that runs out raises the error word,
// both CTAs let their copies land and leave together.
#include <cuda.h>

#include "attn_body.cuh"

#define PF_THREADS 192
#define PF_MAX_STAGES 9
#define PF_BK 64
#define PF_TM 256                    // pairs of a tile: 128 per CTA
#define PF_A_BYTES (128 * PF_BK * 2)

namespace {

struct PfCtl {
    u64 full[PF_MAX_STAGES], empty[PF_MAX_STAGES], tfull[2], tempty[2];
    uint32_t tmem_base;
    int abort_flag;
};

__device__ __forceinline__ uint32_t pf_saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void pf_mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void pf_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool pf_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait; false: gave up (error word raised, the CTA's other roles stop as well)
__device__ __forceinline__ bool pf_wait(uint32_t bar, uint32_t parity, PfCtl* ctl, long long limit, int* error_flag) {
    if (pf_try(bar, parity)) return true;
    const long long t0 = clock64();
    unsigned it = 0;
    while (!pf_try(bar, parity)) {
        if ((++it & 63u) == 0u) {
            if (*(volatile int*)&ctl->abort_flag) return false;
            if (*(volatile int*)error_flag != 0) { *(volatile int*)&ctl->abort_flag = 1; return false; }
            if (clock64() - t0 > limit) {
                atomicCAS(error_flag, 0, 30);
                *(volatile int*)&ctl->abort_flag = 1;
                return false;
            }
        }
    }
    return true;
}
// after a give-up: time for copies and MMAs in flight
__device__ __forceinline__ void pf_drain() {
    const long long t1 = clock64();
    while (clock64() - t1 < 4000000ll) {}
}
// The address of `bar` (own shared memory) in the CTA of the cluster with rank `rank`.
__device__ __forceinline__ uint32_t pf_mapa(uint32_t bar, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(bar), "r"(rank));
    return r;
}
__device__ __forceinline__ void pf_arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void pf_cluster_sync() {
    __syncwarp();               // (aligned instructions)
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// One thread of a converged warp, known to the compiler to be one: MMAs are issued at the tensor core's pace (under a test of
// the lane number one every 53 to 64 clocks, however small).  117 pairs at d 4096 and a draft of five: 826 -> 808 us.
__device__ __forceinline__ bool pf_elect() {
    uint32_t p;
    __syncwarp();
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// copy into this CTA's shared memory that completes on a barrier of the leader
__device__ __forceinline__ void pf_tma_2d(uint32_t dst, const void* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void pf_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void pf_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// arrives on the barrier at this offset in both CTAs once the MMAs issued before are complete
__device__ __forceinline__ void pf_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
                 "h"((unsigned short)3)
                 : "memory");
}
template <int BN>
__device__ __forceinline__ void pf_mma(uint32_t d_tmem, u64 adesc, u64 bdesc, uint32_t accumulate) {
    constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((BN >> 3) << 17) | ((PF_TM >> 4) << 24);
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(IDESC), "r"(accumulate)
        : "memory");
}
// K-major tile with 128-byte rows, 128-byte swizzle, 8-row groups 1024 bytes apart
__device__ __forceinline__ u64 pf_smem_desc(uint32_t addr) {
    const uint32_t lo = ((addr >> 4) & 0x3FFFu) | (1u << 16);
    const uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    return ((u64)hi << 32) | lo;
}
__device__ __forceinline__ void pf_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    __syncwarp();               // the load is one instruction of the whole warp; lanes without a pair come here early
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,"
        "%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

struct PfParams {
    alignas(64) unsigned char map_w[128];      // weights [rows][K], box 64 x BN / 2
    alignas(64) unsigned char map_x0[128];     // operand of k-blocks [0, kb_split): [pairs][.], box 64 x 128
    alignas(64) unsigned char map_x1[128];     // operand of k-blocks [kb_split, nkb)
    int rows, K, kb_split, n_pairs, m_tiles, n_tiles;
    long long wait_cycles;
    int* error_flag;
    // GEMM 1 output stage
    const float* rho;          // [rows] nullable
    const bf16* rho_h;         // [rows] nullable, read where rho is null
    const bf16* gamma;         // [rows]
    bf16* xq;                  // [pairs][rows]
    float* ssq;                // [column blocks of 128][pair capacity]
    int pair_cap;
    // GEMM 2 output stage
    const float* ssq_in;       // [ssq_tiles][pair capacity]
    int ssq_tiles, d;
    float eps;
    const bf16* bias;          // [rows] nullable
    int kvw, Hkv, dh, max_len;
    const int *slot_of, *row_of;
    const float2* rope;        // [pairs][dh / 2] (cos, sin) at the pair's position
    bf16 *Kc, *Vc;
};

__device__ __forceinline__ unsigned pf_pack(float x0, float x1) {
    return (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(x0)) | ((unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(x1)) << 16);
}
__device__ __forceinline__ void pf_store32(bf16* dst, const float (&x)[32]) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *(uint4*)(dst + 8 * q) = make_uint4(pf_pack(x[8 * q], x[8 * q + 1]), pf_pack(x[8 * q + 2], x[8 * q + 3]),
                                            pf_pack(x[8 * q + 4], x[8 * q + 5]), pf_pack(x[8 * q + 6], x[8 * q + 7]));
}
// 32 bf16 values that are the same for all threads of a warp (16-byte aligned), widened
__device__ __forceinline__ void pf_load32(const bf16* src, float (&x)[32]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint4 w = __ldg((const uint4*)src + q);
        x[8 * q] = bf16_lo(w.x); x[8 * q + 1] = bf16_hi(w.x); x[8 * q + 2] = bf16_lo(w.y); x[8 * q + 3] = bf16_hi(w.y);
        x[8 * q + 4] = bf16_lo(w.z); x[8 * q + 5] = bf16_hi(w.z); x[8 * q + 6] = bf16_lo(w.w); x[8 * q + 7] = bf16_hi(w.w);
    }
}

// Stages of the ring: as many as shared memory holds.
template <int BN> struct PfRing { static constexpr unsigned STAGES = BN == 256 ? 7 : 9; };

// GEMM 1 output stage of one pair: 128 columns of u from column c0 of the tile (fewer at the end of the rows), their
// squares added one after the other.
__device__ __forceinline__ void pf_out_fc(const PfParams& P, uint32_t tacc, int c0, int n0, int pair, bool live) {
    float ss = 0.f;
#pragma unroll 1
    for (int c = c0; c < c0 + 128 && n0 + c < P.rows; c += 32) {
        const int n = n0 + c;
        float v[32], g[32];
        pf_ld32(tacc + c, v);
        if (!live) continue;
        pf_load32(P.gamma + n, g);
        if (P.rho) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 r = __ldg((const float4*)(P.rho + n) + q);
                v[4 * q] += r.x; v[4 * q + 1] += r.y; v[4 * q + 2] += r.z; v[4 * q + 3] += r.w;
            }
        } else if (P.rho_h) {
            float r[32];
            pf_load32(P.rho_h + n, r);
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] += r[i];
        }
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            ss = fmaf(v[i], v[i], ss);
            g[i] *= v[i];
        }
        pf_store32(P.xq + (long long)pair * P.rows + n, g);
    }
    if (live) P.ssq[(long long)((n0 + c0) >> 7) * P.pair_cap + pair] = ss;
}

// GEMM 2 output stage of one pair: 32 elements of a head from c and their partners half a head on.
struct PfPair {
    float sc;
    long long slot_base;
    int crow;
};
__device__ __forceinline__ PfPair pf_pair(const PfParams& P, int pair, bool live) {
    PfPair p;
    p.crow = live ? P.row_of[pair] : -1;
    p.sc = 0.f;
    p.slot_base = 0;
    if (p.crow >= 0) {
        float tot = 0.f;
        for (int t = 0; t < P.ssq_tiles; ++t) tot += P.ssq_in[(long long)t * P.pair_cap + pair];
        p.sc = rsqrtf(tot / (float)P.d + P.eps);
        p.slot_base = (long long)P.slot_of[pair] * P.Hkv;
    }
    return p;
}
__device__ __forceinline__ void pf_out_kv(const PfParams& P, uint32_t tacc, const PfPair& pp, int c, int n0, int pair) {
    const int half = P.dh >> 1, g = n0 + c;                 // row of the stacked [K ; V] projection
    const bool isK = g < P.kvw;
    const int head = (isK ? g : g - P.kvw) / P.dh, e0 = g % P.dh;
    float lo[32], hi[32], x[32];
    pf_ld32(tacc + c, lo);
    pf_ld32(tacc + c + half, hi);
    if (pp.crow < 0) return;
    bf16* dst = (isK ? P.Kc : P.Vc) + ((pp.slot_base + head) * P.max_len + pp.crow) * P.dh + e0;
    // (one rounding for scale and bias, as in the builds of 16 pairs per pass)
    if (P.bias) {
        pf_load32(P.bias + g, x);
#pragma unroll
        for (int i = 0; i < 32; ++i) lo[i] = fmaf(lo[i], pp.sc, x[i]);
        pf_load32(P.bias + g + half, x);
#pragma unroll
        for (int i = 0; i < 32; ++i) hi[i] = fmaf(hi[i], pp.sc, x[i]);
    } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) { lo[i] *= pp.sc; hi[i] *= pp.sc; }
    }
    if (isK) {
        const float4* tab = (const float4*)(P.rope + (long long)pair * half + e0);
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const float4 t = __ldg(tab + q);
            const float l0 = lo[2 * q], l1 = lo[2 * q + 1], u0 = hi[2 * q], u1 = hi[2 * q + 1];
            // (written out, so that every build of the code rounds the same product)
            lo[2 * q] = fmaf(l0, t.x, -__fmul_rn(u0, t.y));
            hi[2 * q] = fmaf(u0, t.x, __fmul_rn(l0, t.y));
            lo[2 * q + 1] = fmaf(l1, t.z, -__fmul_rn(u1, t.w));
            hi[2 * q + 1] = fmaf(u1, t.z, __fmul_rn(l1, t.w));
        }
    }
    pf_store32(dst, lo);
    pf_store32(dst + half, hi);
}
template <int EPI, int BN>   // EPI 0: fusion FC, 1: K and V
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PF_THREADS, 1) prefill_tc_kernel(const __grid_constant__ PfParams P) {
    constexpr int B_BYTES = (BN / 2) * PF_BK * 2;
    constexpr unsigned PF_STAGES = PfRing<BN>::STAGES;
    extern __shared__ __align__(1024) unsigned char pf_smem_raw[];
    // (the stages must lie at the same offset in both CTAs: the window's start is the same for all CTAs of a launch)
    unsigned char* smem = (unsigned char*)(((uintptr_t)pf_smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t smemA = pf_saddr(smem), smemB = smemA + PF_STAGES * PF_A_BYTES;
    PfCtl* ctl = (PfCtl*)(smem + PF_STAGES * (PF_A_BYTES + B_BYTES));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint32_t rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int cluster = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
    const int nkb = P.K / PF_BK, units = P.m_tiles * P.n_tiles;
    if (tid == 0) {
        for (int i = 0; i < (int)PF_STAGES; ++i) {
            pf_mbar_init(pf_saddr(&ctl->full[i]), 1);
            pf_mbar_init(pf_saddr(&ctl->empty[i]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            pf_mbar_init(pf_saddr(&ctl->tfull[i]), 1);
            pf_mbar_init(pf_saddr(&ctl->tempty[i]), 8);          // the four output warps of both CTAs
        }
        ctl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(pf_saddr(&ctl->tmem_base)),
                     "r"((uint32_t)(2 * BN))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    pf_fence_before();
    __syncthreads();
    pf_cluster_sync();
    pf_fence_after();
    pdl_wait();                 // (set up while the launch before ended)
    pdl_trigger();

    if (warp == 0) {
        if (pf_elect()) {
            unsigned it = 0;
            bool ok = true;
            for (int w = cluster; w < units && ok; w += n_clusters) {
                const int pair0 = (w / P.n_tiles) * PF_TM + (int)rank * 128, row0 = (w % P.n_tiles) * BN + (int)rank * (BN / 2);
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const unsigned slot = it % PF_STAGES, round = it / PF_STAGES;
                    ok = round == 0 || pf_wait(pf_saddr(&ctl->empty[slot]), (round - 1) & 1u, ctl, P.wait_cycles, P.error_flag);
                    if (!ok) break;
                    if (rank == 0) pf_expect_tx(pf_saddr(&ctl->full[slot]), 2 * (PF_A_BYTES + B_BYTES));
                    const uint32_t bar = pf_mapa(pf_saddr(&ctl->full[slot]), 0);
                    if (kb < P.kb_split) pf_tma_2d(smemA + slot * PF_A_BYTES, P.map_x0, kb * PF_BK, pair0, bar);
                    else pf_tma_2d(smemA + slot * PF_A_BYTES, P.map_x1, (kb - P.kb_split) * PF_BK, pair0, bar);
                    pf_tma_2d(smemB + slot * B_BYTES, P.map_w, kb * PF_BK, row0, bar);
                }
            }
            if (!ok) pf_drain();          // copies already issued still land in this CTA's shared memory
        }
        __syncwarp();
    } else if (warp == 1) {
        if (rank == 0 && pf_elect()) {
            const uint32_t tmem = ctl->tmem_base;
            unsigned it = 0, seg = 0;
            bool ok = true;
            for (int w = cluster; w < units && ok; w += n_clusters, ++seg) {
                const unsigned acc = seg & 1u, use = seg >> 1;
                ok = use == 0 || pf_wait(pf_saddr(&ctl->tempty[acc]), (use - 1) & 1u, ctl, P.wait_cycles, P.error_flag);
                pf_fence_after();
                for (int kb = 0; kb < nkb && ok; ++kb, ++it) {
                    const unsigned slot = it % PF_STAGES, round = it / PF_STAGES;
                    ok = pf_wait(pf_saddr(&ctl->full[slot]), round & 1u, ctl, P.wait_cycles, P.error_flag);
                    if (!ok) break;
                    pf_fence_after();
                    const u64 ad = pf_smem_desc(smemA + slot * PF_A_BYTES), bd = pf_smem_desc(smemB + slot * B_BYTES);
#pragma unroll
                    for (int kk = 0; kk < PF_BK / 16; ++kk)
                        pf_mma<BN>(tmem + acc * BN, ad + (u64)(kk * 2), bd + (u64)(kk * 2), (kb > 0 || kk > 0) ? 1u : 0u);
                    pf_commit(pf_saddr(&ctl->empty[slot]));
                }
                if (ok) pf_commit(pf_saddr(&ctl->tfull[acc]));
            }
            if (!ok) pf_drain();          // MMAs issued are over before tensor memory is freed
        }
        __syncwarp();
    } else {
        // ---- output stage: warps 2..5 read the tensor-memory lanes their number modulo 4 selects; a lane is a pair
        const int quarter = warp & 3;
        unsigned seg = 0;
        for (int w = cluster; w < units; w += n_clusters, ++seg) {
            const unsigned acc = seg & 1u, use = seg >> 1;
            const int pair = (w / P.n_tiles) * PF_TM + (int)rank * 128 + quarter * 32 + lane, n0 = (w % P.n_tiles) * BN;
            const bool live = pair < P.n_pairs;
            PfPair pp;
            if (EPI == 1) pp = pf_pair(P, pair, live);
            bool ok = true;
            if (lane == 0) ok = pf_wait(pf_saddr(&ctl->tfull[acc]), use & 1u, ctl, P.wait_cycles, P.error_flag);
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            if (!ok) break;
            pf_fence_after();
            const uint32_t tacc = ctl->tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN;
            if (EPI == 0) {
#pragma unroll 1
                for (int c = 0; c < BN && n0 + c < P.rows; c += 128) pf_out_fc(P, tacc, c, n0, pair, live);
            } else {
                // 32 elements of a head and their partners, half a head on
#pragma unroll 1
                for (int q = 0; q < BN / 64; ++q) {
                    const int c = P.dh == 64 ? 64 * q : 128 * (q >> 1) + 32 * (q & 1);
                    if (n0 + c >= P.rows) break;                    // (uniform)
                    pf_out_kv(P, tacc, pp, c, n0, pair);
                }
            }
            pf_fence_before();
            __syncwarp();
            if (lane == 0) pf_arrive_cluster(pf_mapa(pf_saddr(&ctl->tempty[acc]), 0));
        }
    }
    pf_fence_before();
    __syncthreads();
    pf_cluster_sync();          // nobody leaves while its shared memory or its barriers may still be used by the other CTA
    if (warp == 1) {
        pf_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(ctl->tmem_base), "r"((uint32_t)(2 * BN)) : "memory");
    }
}

// (cos, sin) of every pair's position, once per call: every K tile of GEMM 2 rotates with the same angles
__global__ void prefill_rope_kernel(const int* row_of, int n_pairs, int half, const double* inv_freq, float2* rope) {
    pdl_wait();
    pdl_trigger();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)n_pairs * half; i += (long long)gridDim.x * blockDim.x) {
        const int n = (int)(i / half), f = (int)(i % half);
        const int pos = row_of[n];
        float cs = 1.f, sn = 0.f;
        if (pos >= 0) rope_cs(pos, inv_freq[f], cs, sn);
        rope[i] = make_float2(cs, sn);
    }
}

typedef CUresult (*PfEncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                               const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                               CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
cudaError_t pf_encode(unsigned char* out, const void* base, long long rows, long long cols, int box_rows) {
    static PfEncodeFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return cudaErrorNotSupported;
        }
        fn = (PfEncodeFn)p;
    }
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {PF_BK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn((CUtensorMap*)out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int EPI, int BN>
cudaError_t pf_launch_t(PfParams& P, int clusters, cudaStream_t st) {
    static bool attr_set[HIVIS_MAX_DEVICES] = {false};
    const size_t smem = 1024 + (size_t)PfRing<BN>::STAGES * (PF_A_BYTES + (BN / 2) * PF_BK * 2) + 512;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= HIVIS_MAX_DEVICES || !attr_set[dev]) {
        e = cudaFuncSetAttribute(prefill_tc_kernel<EPI, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < HIVIS_MAX_DEVICES) attr_set[dev] = true;
    }
    P.n_tiles = (P.rows + BN - 1) / BN;
    const int units = P.m_tiles * P.n_tiles;
    return launch_pdl(prefill_tc_kernel<EPI, BN>, dim3(2u * (unsigned)(units < clusters ? units : clusters)), dim3(PF_THREADS), smem, st, P);
}

// Tile width, by the time of the busiest cluster in units of 10 ns a k-block (0.36 us at 256 weight rows, 0.24 at 128; the line
// between them was drawn at 0.45 to 0.33, and both give the same choices but where the waves are as 7 to 5).  128 / 256 wide: 17 pairs
// 65 / 87 us (d 4096), 72 / 103 (d 3584), 58 / 69 (d 2560); 512 pairs 85 / 98, 84 / 99, 60 / 74; 600 pairs 123 / 114, 113 / 101,
// 59 / 76; 2048 pairs 260 / 226, 144 / 130, 96 / 102.
// A tile is never split over clusters, and no call goes through the chain kernel, whose phases are split over CTAs (64 pairs:
// 45 us there, 61 here): u and the cached rows are rounded to bf16, and parts of their long sums added in fp32 instead of
// in the tensor core's accumulator move one element in forty to the other side of a rounding.  Two to eleven of a hundred
// cached elements then differ, enough to exchange nodes of a draft tree and to move a token drawn by inverse CDF.
template <int EPI>
cudaError_t pf_launch(PfParams& P, const void* W, int num_sms, cudaStream_t st) {
    const int clusters = num_sms / 2 > 0 ? num_sms / 2 : 1;
    P.m_tiles = (P.n_pairs + PF_TM - 1) / PF_TM;
    int bn = 256;
    long long best = -1;
    for (int b = 256; b >= 128; b -= 128) {
        const int tiles = P.m_tiles * ((P.rows + b - 1) / b);
        const long long cost = (long long)((tiles + clusters - 1) / clusters) * (b == 256 ? 45 : 33);
        if (best < 0 || cost < best) { best = cost; bn = b; }
    }
    cudaError_t e = pf_encode(P.map_w, W, P.rows, P.K, bn / 2);
    if (e != cudaSuccess) return e;
    return bn == 256 ? pf_launch_t<EPI, 256>(P, clusters, st) : pf_launch_t<EPI, 128>(P, clusters, st);
}

}  // namespace

bool prefill_tc_supported(int d, int kvw) {
    static_assert(sizeof(CUtensorMap) == 128, "tensor map size");
    return d % PF_BK == 0 && (2 * kvw) % 8 == 0;
}

cudaError_t launch_prefill_tc(const PrefillTcArgs& a, cudaStream_t st) {
    const int d = a.d;
    cudaError_t e;
    if ((e = launch_pdl(prefill_rope_kernel, dim3(296), dim3(256), 0, st, a.row_of, a.n_pairs, a.dh / 2, a.inv_freq, a.rope)) != cudaSuccess) return e;
    PfParams P;
    memset(&P, 0, sizeof(P));
    // ---- GEMM 1: u = W_fc [h ; E[id]] + rho_0
    if ((e = pf_encode(P.map_x0, a.hidden, a.n_pairs, d, 128)) != cudaSuccess) return e;
    if ((e = pf_encode(P.map_x1, a.xe, a.n_pairs, d, 128)) != cudaSuccess) return e;
    P.rows = d; P.K = 2 * d; P.kb_split = d / PF_BK; P.n_pairs = a.n_pairs;
    P.wait_cycles = a.wait_cycles; P.error_flag = a.error_flag;
    P.rho = a.rho0; P.rho_h = a.rho0_h; P.gamma = a.norm1; P.xq = a.xq; P.ssq = a.ssq; P.pair_cap = a.pair_cap;
    if ((e = pf_launch<0>(P, a.fc, a.num_sms, st)) != cudaSuccess) return e;
    // ---- GEMM 2: K, V
    PfParams Q;
    memset(&Q, 0, sizeof(Q));
    if ((e = pf_encode(Q.map_x0, a.xq, a.n_pairs, d, 128)) != cudaSuccess) return e;
    memcpy(Q.map_x1, Q.map_x0, 128);
    Q.rows = 2 * a.kvw; Q.K = d; Q.kb_split = d / PF_BK; Q.n_pairs = a.n_pairs;
    Q.wait_cycles = a.wait_cycles; Q.error_flag = a.error_flag;
    Q.ssq_in = a.ssq; Q.ssq_tiles = (d + 127) / 128; Q.pair_cap = a.pair_cap; Q.d = d; Q.eps = a.eps;
    Q.bias = a.bkv; Q.kvw = a.kvw; Q.Hkv = a.Hkv; Q.dh = a.dh; Q.max_len = a.max_len;
    Q.slot_of = a.slot_of; Q.row_of = a.row_of; Q.rope = a.rope; Q.Kc = a.Kc; Q.Vc = a.Vc;
    return pf_launch<1>(Q, a.wkv, a.num_sms, st);
}
