// Persistent draft-chain kernel for one sequence: all k chained draft steps in ONE cooperative launch.
//
// One CTA per SM, 16 warps.  Every weight matrix of the step (fusion FC, QKV, O, gate/up, down, LM
// head) is split by rows across the CTAs; inside a CTA the rows are cut into chunks of at most 4 KB of
// contiguous weights ("units") which the warps take round-robin.  Each warp owns a private ring of
// shared-memory stages and keeps it full with bulk-async copies (cp.async.bulk + mbarrier
// complete_tx): after it has consumed a stage it refills that stage itself with the unit that lies
// STAGES units ahead in ITS OWN unit sequence, and that sequence runs on across phase and step
// boundaries.  Weights do not depend on activations, so while a CTA finishes a phase, waits at the grid
// barrier and stages the next activation vector, the first units of the next phase are already
// landing in its rings: HBM keeps streaming through every dependency of the chain.
//
// The fusion FC is streamed in two parts: the hidden half needs nothing that the LM head before it decides and is used while that
// one's grid barrier is awaited.  All parts of all steps run through ONE copy of the code (staging, weight loop, output stage).
//
// Phases of a step (grid barrier after each):
//   FC (+rho) -> QKV (RMSNorm in the input stage) -> attention (RoPE, KV append, split-KV, arrival-
//   counter merge) -> O (+u) -> gate/up (RMSNorm in, SiLU*up out) -> down (+y) -> LM head + argmax.
// Partial dot products of a row's chunks go to shared-memory slots and are added in chunk order, the
// argmax is an integer max over packed (value, index) keys: results do not depend on timing.
//
// Every wait is bounded (grid barrier, mbarrier): when a bound is hit the kernel raises an error
// flag, waits (bounded) for its own copies in flight and returns.
#include "attn_body.cuh"

#ifndef CHAIN_WARPS
#define CHAIN_WARPS 16
#endif
#define CHAIN_THREADS (CHAIN_WARPS * 32)
#ifndef CHAIN_STAGES
#define CHAIN_STAGES 2
#endif
#ifndef CHAIN_CHUNK_BYTES
#define CHAIN_CHUNK_BYTES 4096
#endif

// ------------------------------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ u64 make_evict_first_policy() {
    u64 pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
// contiguous global -> shared copy by the bulk-copy engine; completion is counted in bytes on `bar`
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar, u64 pol) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
        ::"r"(dst), "l"(src), "r"(bytes), "r"(bar), "l"(pol)
        : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ u64 ld_acquire_u64(const u64* p) {
    u64 v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_add_u64(u64* p, u64 v) {
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ int ld_relaxed_int(const int* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

#define CHAIN_BARRIERS 7         // grid barriers of a step

// Matrices as the warps see them: those of the phases, the fusion FC in two parts - whole chunks of its hidden half, which
// the step before has left in place, and the rest, which needs the step's token.  The hidden part lies under the grid barrier
// of the LM head before it.
enum { CW_FCH = 0, CW_FCE, CW_QKV, CW_O, CW_GU, CW_DOWN, CW_LM, CW_COUNT };
struct ChainSeg {
    const char* base;          // this CTA's first row, first column of the part
    long long ld;              // bytes from row to row
    int rows;                  // rows of this CTA
    int K;                     // columns of the part
};
__device__ __forceinline__ int chain_phase(int w) { return w == CW_FCH ? PH_FC : w - 1; }

// A warp's place in its units of a part.  A warp keeps to one chunk of the columns where the number of chunks divides the
// number of warps, else it has a run of the units taken chunk by chunk.
struct ChainCursor {
    int row, ch, left, step;
    __device__ void begin(int rows, int cpr, int warp) {
        if (CHAIN_WARPS % cpr == 0) {
            step = CHAIN_WARPS / cpr;
            ch = warp % cpr;
            row = warp / cpr;
            left = row < rows ? (rows - 1 - row) / step + 1 : 0;
        } else {
            const int U = rows * cpr, u0 = U * warp / CHAIN_WARPS;
            step = 1;
            ch = rows > 0 ? u0 / rows : 0;
            row = u0 - ch * rows;
            left = U * (warp + 1) / CHAIN_WARPS - u0;
        }
    }
    __device__ __forceinline__ void next(int rows) {
        --left;
        row += step;
        if (row >= rows) { row = 0; ++ch; }          // (not reached by warps that keep to a chunk: none is left)
    }
};
// Every warp's place at the start of every part, worked out once per launch: lane w of the warp keeps that of part w, in 16 bits
// a number (a CTA's units of a part have a partial sum each in shared memory, so there are fewer than 65536).  It is in registers
// because shared memory is full: a table of it, and of the parts, took 2 KB from x, and drafters with the widest feed-forward
// layers that had fitted did not fit any more.  A round of four steps at d 256: 116 us with the table, 112 with this; d 4096 level.
struct ChainFirst {
    uint32_t a, b;
    __device__ __forceinline__ void set(const ChainCursor& c) {
        a = (uint32_t)c.row | (uint32_t)c.ch << 16;
        b = (uint32_t)c.left | (uint32_t)c.step << 16;
    }
    // (all lanes of the warp)
    __device__ __forceinline__ ChainCursor get(int w) const {
        const uint32_t x = __shfl_sync(0xffffffffu, a, w), y = __shfl_sync(0xffffffffu, b, w);
        ChainCursor c;
        c.row = (int)(x & 0xffffu);
        c.ch = (int)(x >> 16);
        c.left = (int)(y & 0xffffu);
        c.step = (int)(y >> 16);
        return c;
    }
};
// A warp's stream of units: how many it has asked for and used, and the next one to ask for.
struct ChainStream {
    unsigned fi, ci;
    int step, w;
    ChainCursor at;
};
struct ChainMisc {
    float red[CHAIN_WARPS];
    u64 kred[CHAIN_WARPS];
    int abort_flag;
    int row0[PH_COUNT], rows[PH_COUNT];            // this CTA's rows of every phase
    u64 bar_base;              // value of the barrier counter when the launch began
};
// What the plan sets aside for it, beside x: it decides how wide a feed-forward layer fits, and with it which drafters run here.
#define CHAIN_MISC_BYTES 280
static_assert(sizeof(ChainMisc) <= CHAIN_MISC_BYTES, "");
// The rows of a part that are this CTA's (kh: columns of the fusion FC in its first part).
template <typename WT>
__device__ __forceinline__ ChainSeg chain_seg(const ChainArgs& a, const ChainMisc* misc, int w, int kh) {
    const int p = chain_phase(w), K = a.ph[p].K;
    ChainSeg g;
    g.ld = (long long)K * (int)sizeof(WT);
    g.base = (const char*)a.ph[p].W + misc->row0[p] * g.ld + (w == CW_FCE ? (long long)kh * (int)sizeof(WT) : 0ll);
    g.rows = misc->rows[p];
    g.K = w == CW_FCH ? kh : w == CW_FCE ? K - kh : K;
    return g;
}

// CTA barrier; true, for all threads alike, while no wait of the CTA has run out.
__device__ __forceinline__ bool cta_alive(const ChainMisc* misc) {
    return __syncthreads_or(*(volatile const int*)&misc->abort_flag) == 0;
}
// Grid-wide barrier on a monotonically increasing counter, in two halves: what does not need the others' results goes between.
__device__ __forceinline__ void grid_arrive(const ChainArgs& a) {
    __syncthreads();
    if (threadIdx.x == 0) red_release_add_u64(a.bar_counter, 1ull);
}
// false = gave up (error flag raised)
__device__ __forceinline__ bool grid_wait(const ChainArgs& a, ChainMisc* misc, u64 target) {
    if (threadIdx.x == 0 && *(volatile int*)&misc->abort_flag == 0) {
        const long long t0 = clock64();
        unsigned it = 0;
        while (ld_acquire_u64(a.bar_counter) < target) {
            if ((++it & 255u) == 0u && (ld_relaxed_int(a.error_flag) != 0 || clock64() - t0 > a.wait_cycles)) {
                atomicExch(a.error_flag, 1);
                *(volatile int*)&misc->abort_flag = 1;
                break;
            }
        }
    }
    return cta_alive(misc);
}

template <typename WT>
__device__ __forceinline__ int x_index(int k, int K) {
    if (sizeof(WT) == 2) return ((k >> 3) << 2) + (k & 3) + ((k >> 2) & 1) * (K >> 1);
    return k;
}

// dot product of one staged chunk with the matching slice of x
template <typename WT>
__device__ __forceinline__ float dot_chunk(const uint4* wsm, const float* xs, int K, int k0, int nvec, int lane) {
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
    if (sizeof(WT) == 2) {
        const float4* xlo = (const float4*)xs + (k0 >> 3);
        const float4* xhi = (const float4*)(xs + (K >> 1)) + (k0 >> 3);
#pragma unroll 4
        for (int j = lane; j < nvec; j += 32) {
            const uint4 w = wsm[j];
            const float4 xa = xlo[j], xb = xhi[j];
            a0 = fmaf(bf16_lo(w.x), xa.x, a0); a1 = fmaf(bf16_hi(w.x), xa.y, a1);
            a2 = fmaf(bf16_lo(w.y), xa.z, a2); a3 = fmaf(bf16_hi(w.y), xa.w, a3);
            a0 = fmaf(bf16_lo(w.z), xb.x, a0); a1 = fmaf(bf16_hi(w.z), xb.y, a1);
            a2 = fmaf(bf16_lo(w.w), xb.z, a2); a3 = fmaf(bf16_hi(w.w), xb.w, a3);
        }
    } else {
        const float4* x4 = (const float4*)xs + (k0 >> 2);
#pragma unroll 4
        for (int j = lane; j < nvec; j += 32) {
            const uint4 w = wsm[j];
            const float4 xa = x4[j];
            a0 = fmaf(__uint_as_float(w.x), xa.x, a0); a1 = fmaf(__uint_as_float(w.y), xa.y, a1);
            a2 = fmaf(__uint_as_float(w.z), xa.z, a2); a3 = fmaf(__uint_as_float(w.w), xa.w, a3);
        }
    }
    float acc = (a0 + a1) + (a2 + a3);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}

// Asks for the warp's next unit (lane 0 issues; every lane tracks the cursor).
template <typename WT>
__device__ __forceinline__ void chain_fetch(ChainStream& t, const ChainArgs& a, const ChainMisc* misc, const ChainFirst& first, int kh,
                                            uint32_t ring0, uint32_t bar0, u64 pol, int lane) {
    while (t.at.left == 0) {
        if (++t.w == CW_COUNT) {
            t.w = 0;
            ++t.step;
        }
        if (t.step >= a.k) return;
        t.at = first.get(t.w);
    }
    if (t.step >= a.k) return;
    const ChainSeg g = chain_seg<WT>(a, misc, t.w, kh);
    if (lane == 0) {
        const unsigned st = t.fi % CHAIN_STAGES;
        const uint32_t bar = bar0 + st * 8;
        const uint32_t bytes = (uint32_t)min(CHAIN_CHUNK_BYTES, g.K * (int)sizeof(WT) - t.at.ch * CHAIN_CHUNK_BYTES);
        mbar_expect_tx(bar, bytes);
        bulk_g2s(ring0 + st * CHAIN_CHUNK_BYTES, g.base + t.at.row * g.ld + t.at.ch * CHAIN_CHUNK_BYTES, bytes, bar, pol);
    }
    ++t.fi;
    t.at.next(g.rows);
}

// ---- attention -----------------------------------------------------------------------------------
// A unit = (split of the cache rows, query head), a CTA each; the arithmetic and its order are attn_unit's (attn_body.cuh, one
// head per unit), so the results are the same bits.  What bounds it is a chain of latencies: with attn_unit, one or two warps of a
// CTA working from global memory, the phase took 29 000 clocks of a step's 286 000 (d 4096, 128 rows), 15 000 of 52 000 at d 256.
// So the unit's rows of K and V, which earlier steps have written, are copied to shared memory by all warps before the grid
// barrier is awaited, and the angles worked out there; q, k and v are rotated side by side, the new row being one more row of
// the copies; warps without rows are left out of the merge; the splits' partial results come in one round trip.  Units whose
// rows shared memory does not hold take attn_unit.
// Five steps and the refresh: 803 -> 749 us (d 4096, 128 rows), 131 -> 119 (d 256).
// (No more registers than the projections need: the acquire of a grid barrier empties L1, so a spilled register comes back from
// L2.  A variant with rows in registers spilled 100 words and made a step 24 us slower.)
template <typename WT, int DH>
struct ChainAttnSmem {
    static constexpr int KROW = DH * (int)sizeof(WT) + 16;       // bytes from K row to K row: lanes read rows side by side
    static constexpr int VROW = DH * (int)sizeof(WT);
    alignas(16) float q[DH];
    float2 cs[DH / 2];
    float m[CHAIN_WARPS], l[CHAIN_WARPS];
    alignas(16) float acc[CHAIN_WARPS][DH];
    int last;
    alignas(16) unsigned char rows[16];                          // K rows [attn_rows][KROW], V rows [attn_rows][VROW]
};
template <typename WT, int DH>
__device__ __forceinline__ void chain_attn_prepare(const ChainArgs& a, ChainAttnSmem<WT, DH>& sm, int unit, int p, int slot) {
    typedef ChainAttnSmem<WT, DH> S;
    constexpr int NCH = S::VROW / 16;
    const int split = unit % a.attn_nsplit, kvh = unit / a.attn_nsplit / (a.Hq / a.Hkv);
    const int r0 = split * a.attn_chunk, n = min(p, r0 + a.attn_chunk) - r0;     // rows without the new one
    const int tid = threadIdx.x;
    const long long row0 = (((long long)slot * a.Hkv + kvh) * a.max_len + r0) * (long long)DH;
    const char* K = (const char*)((const WT*)a.Kc + row0);
    const char* V = (const char*)((const WT*)a.Vc + row0);
    const uint32_t ks = smem_addr(sm.rows), vs = ks + a.attn_rows * S::KROW;
#pragma unroll 2
    for (int i = tid; i < n * NCH; i += CHAIN_THREADS) {
        const int r = i / NCH, c = i - r * NCH;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ks + r * S::KROW + c * 16), "l"(K + (long long)i * 16) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(vs + i * 16), "l"(V + (long long)i * 16) : "memory");
    }
    if (tid < DH / 2) {
        float c, s;
        rope_cs(p, a.inv_freq[tid], c, s);
        sm.cs[tid] = make_float2(c, s);
    }
}
template <typename WT, int DH>
__device__ __forceinline__ void chain_attn_run(const ChainArgs& a, ChainAttnSmem<WT, DH>& sm, int unit, int p, int slot) {
    typedef ChainAttnSmem<WT, DH> S;
    constexpr int EPL = DH / 32;                 // head-dim elements per lane in the PV phase
    constexpr int NCH = S::VROW / 16;            // 16-byte vectors of a row
    constexpr int half = DH / 2;
    asm volatile("cp.async.wait_all;" ::: "memory");
    const int nsplits = (p + a.attn_chunk) / a.attn_chunk, split = unit % a.attn_nsplit, h = unit / a.attn_nsplit;
    if (split >= nsplits) return;
    const int r0 = split * a.attn_chunk, n = min(p + 1, r0 + a.attn_chunk) - r0, kvh = h / (a.Hq / a.Hkv);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char* const ks = sm.rows;
    unsigned char* const vs = sm.rows + a.attn_rows * S::KROW;
    __syncthreads();                             // the angles and the copies
    {
        // q of the head, and the new row of the unit that has it; one unit per KV head appends the row to the cache
        const int pn = p - r0;
        const bool owns_new = pn < n, writer = owns_new && h % (a.Hq / a.Hkv) == 0;
        const long long row = (((long long)slot * a.Hkv + kvh) * a.max_len + p) * (long long)DH;
        if (tid < DH) {
            const bool is_q = tid < half;
            const int j = is_q ? tid : tid - half;
            if (is_q || owns_new) {
                const float* x = a.qkv + (is_q ? h * DH : a.qw + kvh * DH);
                const float x0 = __ldcg(x + j), x1 = __ldcg(x + j + half);
                const float2 cs = sm.cs[j];
                // (written out, so that every build of the code rounds the same product)
                const float y0 = fmaf(x0, cs.x, -__fmul_rn(x1, cs.y)), y1 = fmaf(x1, cs.x, __fmul_rn(x0, cs.y));
                if (is_q) {
                    sm.q[j] = y0 * a.scale;
                    sm.q[j + half] = y1 * a.scale;
                } else {
                    store_from_float<WT>(ks + pn * S::KROW, j, y0);
                    store_from_float<WT>(ks + pn * S::KROW, j + half, y1);
                    if (writer) {
                        store_from_float<WT>(a.Kc, row + j, y0);
                        store_from_float<WT>(a.Kc, row + j + half, y1);
                    }
                }
            }
        } else if (tid < 2 * DH && owns_new) {
            const int j = tid - DH;
            const float v = __ldcg(a.qkv + a.qw + a.kvw + kvh * DH + j);
            store_from_float<WT>(vs + pn * S::VROW, j, v);
            if (writer) store_from_float<WT>(a.Vc, row + j, v);
        }
    }
    __syncthreads();

    float m_run = -INFINITY, l_run = 0.f, acc[EPL];
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
#pragma unroll 1
    for (int base = warp * 32; base < n; base += CHAIN_THREADS) {
        const int r = base + lane;
        const bool ok = r < n;
        float s = 0.f;
        const uint4* k4 = (const uint4*)(ks + (ok ? r : base) * S::KROW);
        const float4* q4 = (const float4*)sm.q;
#pragma unroll 4
        for (int c = 0; c < NCH; ++c) {
            const uint4 w = k4[c];
            if constexpr (sizeof(WT) == 2) {
                const float4 qa = q4[2 * c], qb = q4[2 * c + 1];
                s = fmaf(qa.x, bf16_lo(w.x), s); s = fmaf(qa.y, bf16_hi(w.x), s);
                s = fmaf(qa.z, bf16_lo(w.y), s); s = fmaf(qa.w, bf16_hi(w.y), s);
                s = fmaf(qb.x, bf16_lo(w.z), s); s = fmaf(qb.y, bf16_hi(w.z), s);
                s = fmaf(qb.z, bf16_lo(w.w), s); s = fmaf(qb.w, bf16_hi(w.w), s);
            } else {
                const float4 qa = q4[c];
                s = fmaf(qa.x, __uint_as_float(w.x), s); s = fmaf(qa.y, __uint_as_float(w.y), s);
                s = fmaf(qa.z, __uint_as_float(w.z), s); s = fmaf(qa.w, __uint_as_float(w.w), s);
            }
        }
        // online softmax over this block of 32 rows
        const float sv = ok ? s : -INFINITY;
        float mb = sv;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
        const float mn = fmaxf(m_run, mb);       // finite: the block has at least one valid row
        const float corr = expf(m_run - mn);
        const float pr = ok ? expf(sv - mn) : 0.f;
        float ps = pr;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, o);
        l_run = l_run * corr + ps;
        m_run = mn;
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[e] *= corr;
        // PV: lane owns head-dim elements [lane * EPL, + EPL)
        const int nrows = min(32, n - base);
        const unsigned char* v0 = vs + base * S::VROW + lane * EPL * (int)sizeof(WT);
#pragma unroll 8
        for (int j = 0; j < nrows; ++j) {
            const float pj = __shfl_sync(0xffffffffu, pr, j);
            constexpr int VW = EPL * (int)sizeof(WT) / 4;            // words of the slice: one load
            struct alignas(4 * VW) Slice { unsigned w[VW]; };
            const Slice v = *(const Slice*)(v0 + j * S::VROW);
#pragma unroll
            for (int e = 0; e < EPL; ++e) {
                const float x = sizeof(WT) == 4 ? __uint_as_float(v.w[e % VW]) : (e & 1) ? bf16_hi(v.w[e / 2]) : bf16_lo(v.w[e / 2]);
                acc[e] = fmaf(pj, x, acc[e]);
            }
        }
    }
    // merge the warps that had rows
    if (lane == 0) {
        sm.m[warp] = m_run;
        sm.l[warp] = l_run;
    }
#pragma unroll
    for (int e = 0; e < EPL; ++e) sm.acc[warp][lane * EPL + e] = acc[e];
    __syncthreads();
    const int nw = min(CHAIN_WARPS, (n + 31) / 32);
    float M = -INFINITY, L = 0.f, A = 0.f;
    auto merge = [&](int count) {                // of what lies in sm.m, sm.l and sm.acc, in order
        M = -INFINITY;
        L = A = 0.f;
        for (int w = 0; w < count; ++w) M = fmaxf(M, sm.m[w]);
        for (int w = 0; w < count; ++w) {
            const float f = expf(sm.m[w] - M);
            L += sm.l[w] * f;
            A += sm.acc[w][tid] * f;
        }
    };
    if (tid < DH) merge(nw);
    if (nsplits == 1) {
        if (tid < DH) a.attn[h * DH + tid] = A / L;
        return;
    }
    const long long p0 = (long long)h * a.attn_nsplit;
    if (tid < DH) {
        a.part_acc[(p0 + split) * DH + tid] = A;
        if (tid == 0) {
            a.part_ml[(p0 + split) * 2] = M;
            a.part_ml[(p0 + split) * 2 + 1] = L;
        }
    }
    // arrival counter: the last unit of the head merges the splits; nobody waits
    __syncthreads();
    if (tid == 0) {
        int* ctr = a.counters + h;
        const int old = atom_add_acq_rel(ctr, 1);
        sm.last = (old == nsplits - 1);
        if (sm.last) *ctr = 0;
    }
    __syncthreads();
    if (!sm.last) return;
    if (nsplits <= CHAIN_WARPS) {
        if (tid < nsplits) {
            sm.m[tid] = __ldcg(a.part_ml + (p0 + tid) * 2);
            sm.l[tid] = __ldcg(a.part_ml + (p0 + tid) * 2 + 1);
        }
#pragma unroll 4
        for (int i = tid; i < nsplits * DH; i += CHAIN_THREADS) sm.acc[i / DH][i % DH] = __ldcg(a.part_acc + p0 * DH + i);
        __syncthreads();
        if (tid < DH) merge(nsplits);
    } else if (tid < DH) {
        M = -INFINITY;
        L = A = 0.f;
        for (int q = 0; q < nsplits; ++q) M = fmaxf(M, __ldcg(a.part_ml + (p0 + q) * 2));
        for (int q = 0; q < nsplits; ++q) {
            const float f = expf(__ldcg(a.part_ml + (p0 + q) * 2) - M);
            L += __ldcg(a.part_ml + (p0 + q) * 2 + 1) * f;
            A += __ldcg(a.part_acc + (p0 + q) * DH + tid) * f;
        }
    }
    if (tid < DH) a.attn[h * DH + tid] = A / L;
}

template <typename WT, int DH>
__global__ void __launch_bounds__(CHAIN_THREADS, 1) draft_chain_kernel(const ChainArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int ES = (int)sizeof(WT);
    constexpr int CE = CHAIN_CHUNK_BYTES / ES;              // elements per full chunk
    float* xs = (float*)(smem + a.off_x);
    float* part = (float*)(smem + a.off_part);
    u64* bars = (u64*)(smem + a.off_bar);
    ChainMisc* misc = (ChainMisc*)(smem + a.off_misc);
    AttnSmem<CHAIN_WARPS, 1, DH>* asm_ = (AttnSmem<CHAIN_WARPS, 1, DH>*)(smem + a.off_x);   // x is idle during attention
    ChainAttnSmem<WT, DH>* cs = (ChainAttnSmem<WT, DH>*)(smem + a.off_x);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cta = blockIdx.x, G = gridDim.x;
    const int d = a.d;
    const int kh = d / CE * CE;                             // columns of the fusion FC that the first part covers

    if (tid < PH_COUNT) {
        const int p = tid;
        const long long N = a.ph[p].N;
        long long r0, r1;
        if (p == PH_GU) {                                // keep (gate_i, up_i) row pairs together
            r0 = 2 * ((N / 2) * cta / G);
            r1 = 2 * ((N / 2) * (cta + 1) / G);
        } else {
            r0 = N * cta / G;
            r1 = N * (cta + 1) / G;
        }
        misc->row0[p] = (int)r0;
        misc->rows[p] = (int)(r1 - r0);
    } else if (tid == 32) {
        misc->abort_flag = 0;
        misc->bar_base = barrier_base(a.bar_counter, (unsigned)G) + a.bar_off;
    } else if (tid >= 64 && tid < 64 + CHAIN_WARPS * CHAIN_STAGES) {
        mbar_init(smem_addr(bars + tid - 64), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    __syncthreads();
    // chunks of a row of part w: those that the hidden part of the fusion FC leaves are the other part's
    auto chunks = [&](int w) {
        const int all = (a.ph[chain_phase(w)].K * ES + CHAIN_CHUNK_BYTES - 1) / CHAIN_CHUNK_BYTES;
        return w == CW_FCH ? max(kh / CE, 1) : w == CW_FCE ? all - kh / CE : all;
    };
    ChainFirst first;
    {
        const int w = min(lane, CW_COUNT - 1);
        ChainCursor c;
        c.begin(w == CW_FCH && kh == 0 ? 0 : misc->rows[chain_phase(w)], chunks(w), warp);
        first.set(c);
    }
    __syncwarp();

    pdl_trigger();                                          // (the launch after this one is set up as CTAs leave)
    const int slot = a.slot;
    const int pos0 = a.kv_len[slot];
    if (cta == 0 && tid < a.k) a.keys[tid] = 0ull;       // consumed after several grid barriers

    // ---------------------------------------------------------------- per-warp weight stream
    const u64 pol = make_evict_first_policy();
    unsigned char* const stages = smem + warp * (CHAIN_STAGES * CHAIN_CHUNK_BYTES);
    const uint32_t ring0 = smem_addr(stages), bar0 = smem_addr(bars + warp * CHAIN_STAGES);
    ChainStream t;
    t.fi = t.ci = 0;
    t.step = t.w = 0;
    t.at = first.get(0);
    for (int i = 0; i < CHAIN_STAGES; ++i) chain_fetch<WT>(t, a, misc, first, kh, ring0, bar0, pol, lane);

    u64 bar_target = misc->bar_base;                        // of the newest barrier that this CTA has arrived on
    bool alive = true;
    auto arrive = [&]() {
        bar_target += (u64)G;
        grid_arrive(a);
    };
    auto wait = [&]() { return alive = grid_wait(a, misc, bar_target); };
    constexpr int XB = 8;                                   // words of x per thread and turn

    AttnArgs aa;
    aa.qkv = a.qkv; aa.ld = a.qw + 2 * a.kvw; aa.Kc = a.Kc; aa.Vc = a.Vc; aa.slots = nullptr; aa.pos0 = nullptr;
    aa.step = 0; aa.inv_freq = a.inv_freq; aa.Hq = a.Hq; aa.Hkv = a.Hkv; aa.dh = a.dh; aa.max_len = a.max_len;
    aa.B = 1; aa.scale = a.scale; aa.chunk = a.attn_chunk; aa.nsplit = a.attn_nsplit; aa.part_acc = a.part_acc;
    aa.part_ml = a.part_ml; aa.counters = a.counters; aa.attn = a.attn; aa.attn_h = nullptr; aa.lo_rows = 0;

    // One loop over the parts of all steps, so that every piece of code is there once: a step runs through all of it, and what the
    // instruction caches do not hold comes from L2 again, in the middle of the phase boundaries.  (A copy of the weight loop and of
    // the barriers for every phase made 175 KB, now 135.)  With the hidden half of the fusion FC under the LM head's barrier, gains and
    // addends asked for before the barriers and x staged four words at a time: d 4096, five steps and the refresh 750 -> 731 us, an
    // opening 765 -> 739; d 256 118 -> 121, where there is next to nothing to stream (135 at first).
    int s = 0, w = CW_FCH;
#pragma unroll 1
    for (; s < a.k; s += w == CW_LM ? 1 : 0, w = w == CW_LM ? CW_FCH : w + 1) {
        const int ph = chain_phase(w), rows = misc->rows[ph], r0 = misc->row0[ph];
        const int K = w == CW_FCH ? kh : w == CW_FCE ? 2 * d - kh : a.ph[ph].K;
        // ------------------------------------------------------------ x of the part
        if (w == CW_FCH) {
            // the hidden half of the fusion FC: behind the LM head x is still the layer output
            if (K == 0) continue;
            if (s == 0 || K != d) {
                const float* f = s == 0 ? a.pend_feat + (long long)slot * d : a.feat;
                for (int kk = tid; kk < K; kk += CHAIN_THREADS) xs[x_index<WT>(kk, K)] = __ldcg(f + kk);
                __syncthreads();
            }
        } else if (w == CW_FCE) {
            if (!(alive = cta_alive(misc))) break;           // (x of the other half has been used)
            const float* f = (s == 0 ? a.pend_feat + (long long)slot * d : a.feat) + kh;
            const int fk = d - kh;
            for (int kk = tid; kk < fk; kk += CHAIN_THREADS) xs[x_index<WT>(kk, K)] = __ldcg(f + kk);
            if (s > 0 && !wait()) break;                     // the keys of the last step are complete
            int tok;
            if (s == 0) tok = a.pend_id[slot];
            else if (a.forced) tok = a.forced[s - 1];
            else tok = key_index(__ldcg(a.keys + (s - 1)));
            tok = checked_token(tok, a.V, a.id_flag);
            const long long e0 = (long long)tok * d;
            for (int kk = tid; kk < d; kk += CHAIN_THREADS) xs[x_index<WT>(fk + kk, K)] = load_as_float<WT>(a.embed, e0 + kk);
            __syncthreads();
        } else {
            const bool norm = w == CW_QKV || w == CW_GU;
            const float* src = w == CW_QKV ? a.u : w == CW_O ? a.attn : w == CW_GU ? a.y : w == CW_DOWN ? a.act : a.feat;
            const void* gain = w == CW_QKV ? a.norm1 : a.norm2;
            float gn[XB];
            if (norm) {                                     // (asked for before the barrier)
#pragma unroll
                for (int i = 0; i < XB; ++i) {
                    const int kk = tid + i * CHAIN_THREADS;
                    gn[i] = kk < K ? load_as_float<WT>(gain, kk) : 0.f;
                }
            }
            if (w == CW_O) {
                // attention over the text-only cache
                const int nunits = a.Hq * a.attn_nsplit;
                const bool staged = a.attn_chunk <= a.attn_rows;
                if (staged && cta < nunits) chain_attn_prepare<WT, DH>(a, *cs, cta, pos0 + s, slot);
                if (!wait()) break;
#pragma unroll 1
                for (int unit = cta; unit < nunits; unit += G) {
                    if (staged) {
                        if (unit != cta) {
                            __syncthreads();                // the unit before has been read
                            chain_attn_prepare<WT, DH>(a, *cs, unit, pos0 + s, slot);
                        }
                        chain_attn_run<WT, DH>(a, *cs, unit, pos0 + s, slot);
                    } else {
                        attn_unit<WT, DH, 1, CHAIN_WARPS>(aa, unit % a.attn_nsplit, unit / a.attn_nsplit, 0, pos0 + s, slot, *asm_);
                    }
                }
                arrive();
            }
            if (!wait()) break;
            if (norm) {
                // a thread's first words stay in registers until the scale is known
                float v[XB], ss = 0.f;
#pragma unroll
                for (int i = 0; i < XB; ++i) {
                    const int kk = tid + i * CHAIN_THREADS;
                    v[i] = kk < K ? __ldcg(src + kk) : 0.f;
                }
#pragma unroll
                for (int i = 0; i < XB; ++i) ss += v[i] * v[i];
#pragma unroll 1
                for (int kk = tid + XB * CHAIN_THREADS; kk < K; kk += CHAIN_THREADS) {
                    const float y = __ldcg(src + kk);
                    ss += y * y;
                    xs[x_index<WT>(kk, K)] = y;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
                if (lane == 0) misc->red[warp] = ss;
                __syncthreads();
                float tot = 0.f;
#pragma unroll
                for (int q = 0; q < CHAIN_WARPS; ++q) tot += misc->red[q];
                const float inv = rsqrtf(tot / (float)K + a.eps);
#pragma unroll
                for (int i = 0; i < XB; ++i) {
                    const int kk = tid + i * CHAIN_THREADS;
                    if (kk < K) xs[x_index<WT>(kk, K)] = v[i] * gn[i] * inv;
                }
#pragma unroll 1
                for (int kk = tid + XB * CHAIN_THREADS; kk < K; kk += CHAIN_THREADS) {
                    const int j = x_index<WT>(kk, K);
                    xs[j] = xs[j] * load_as_float<WT>(gain, kk) * inv;
                }
            } else {
                // four words at a time (the layout keeps four together), all of a thread's loads in flight up to K = 12288
                constexpr int XV = 6;
#pragma unroll 1
                for (int k0 = 4 * tid; k0 < K; k0 += 4 * XV * CHAIN_THREADS) {
                    float4 v[XV];
#pragma unroll
                    for (int i = 0; i < XV; ++i) {
                        const int kk = k0 + 4 * i * CHAIN_THREADS;
                        if (kk < K) v[i] = __ldcg((const float4*)(src + kk));
                    }
#pragma unroll
                    for (int i = 0; i < XV; ++i) {
                        const int kk = k0 + 4 * i * CHAIN_THREADS;
                        if (kk < K) *(float4*)(xs + x_index<WT>(kk, K)) = v[i];
                    }
                }
            }
            __syncthreads();
        }
        const int slots = (a.ph[ph].K * ES + CHAIN_CHUNK_BYTES - 1) / CHAIN_CHUNK_BYTES;   // partial sums of a row
        // what the output of this thread's row is added to
        const float* const add = w == CW_O ? a.u : a.y;
        const long long rho_row = (long long)(s < a.n_resid - 1 ? s : a.n_resid - 1) * d;
        auto addend = [&](int r) {
            if (w == CW_FCE) return a.rho ? a.rho[rho_row + r] : a.rho_w ? load_as_float<WT>(a.rho_w, rho_row + r) : 0.f;
            if (w == CW_QKV) return a.bqkv ? load_as_float<WT>(a.bqkv, r) : 0.f;
            return __ldcg(add + r);
        };
        float first_add = 0.f;
        if (w != CW_FCH && w != CW_GU && w != CW_LM && tid < rows) first_add = addend(r0 + tid);
        // ------------------------------------------------------------ this warp's units: partial dot products into part[row][slot]
        {
            ChainCursor c = first.get(w);
            float* const part_w = part + (w == CW_FCE ? kh / CE : 0);
            int have = -1, nvec = 0;
            bool gave_up = false;
#pragma unroll 1
            while (c.left > 0) {
                if (c.ch != have) {
                    have = c.ch;
                    nvec = (min(CE, K - have * CE) * ES) >> 4;
                }
                const unsigned st = t.ci % CHAIN_STAGES;
                const uint32_t parity = (t.ci / CHAIN_STAGES) & 1u;
                const uint32_t bar = bar0 + st * 8;
                if (!mbar_try_wait(bar, parity)) {
                    const long long t0 = clock64();
                    while (!mbar_try_wait(bar, parity)) {
                        if (clock64() - t0 > a.wait_cycles) {
                            atomicExch(a.error_flag, 2);
                            *(volatile int*)&misc->abort_flag = 1;
                            gave_up = true;
                            break;
                        }
                    }
                }
                if (__any_sync(0xffffffffu, gave_up)) break;        // one answer for the warp
                const float acc = dot_chunk<WT>((const uint4*)(stages + st * CHAIN_CHUNK_BYTES), xs, K, have * CE, nvec, lane);
                if (lane == 0) part_w[c.row * slots + c.ch] = acc;
                ++t.ci;
                __syncwarp();
                fence_proxy_async();                        // our reads of the stage precede its refill
                chain_fetch<WT>(t, a, misc, first, kh, ring0, bar0, pol, lane);
                c.next(rows);
            }
        }
        if (w == CW_FCH) continue;                          // (its partial sums wait for those of the other half)
        if (!(alive = cta_alive(misc))) break;
        // ------------------------------------------------------------ output stage
        auto row_sum = [&](int rl) {                        // add a row's chunk partials in chunk order
            float v = 0.f;
            for (int q = 0; q < slots; ++q) v += part[rl * slots + q];
            return v;
        };
        if (w == CW_GU) {
            for (int pl = tid; pl < rows / 2; pl += CHAIN_THREADS) {
                const float gate = row_sum(2 * pl), up = row_sum(2 * pl + 1);
                a.act[r0 / 2 + pl] = gate / (1.f + expf(-gate)) * up;
            }
        } else if (w == CW_LM) {
            u64 best = 0;
            for (int rl = tid; rl < rows; rl += CHAIN_THREADS) {
                const float v = row_sum(rl);
                if (a.logits_out) a.logits_out[(long long)s * a.V + r0 + rl] = v;
                const u64 key = a.gumbel_u ? pack_key(gumbel_perturbed(v, a.inv_t, __ldg(a.gumbel_u + (long long)s * a.V + r0 + rl)), r0 + rl)
                                           : pack_key(v, r0 + rl);
                best = key > best ? key : best;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const u64 other = __shfl_xor_sync(0xffffffffu, best, o);
                best = other > best ? other : best;
            }
            if (lane == 0) misc->kred[warp] = best;
            __syncthreads();
            if (tid == 0) {
                u64 m = misc->kred[0];
#pragma unroll
                for (int q = 1; q < CHAIN_WARPS; ++q) m = misc->kred[q] > m ? misc->kred[q] : m;
                if (m) atomicMax(a.keys + s, m);
            }
        } else {
            float* const out = w == CW_FCE ? a.u : w == CW_QKV ? a.qkv : w == CW_O ? a.y : a.feat;
            for (int rl = tid; rl < rows; rl += CHAIN_THREADS) out[r0 + rl] = row_sum(rl) + (rl == tid ? first_add : addend(r0 + rl));
        }
        arrive();
    }
    if (alive && (cta != 0 || wait())) {                    // (only the CTA that reads the last keys waits for them)
        if (cta == 0) {
            if (tid < a.k) a.out_ids[tid] = key_index(__ldcg(a.keys + tid));
            if (tid == 0) a.kv_len[slot] = pos0 + a.k;
        }
        return;                                             // every fetched unit has been consumed
    }
    // gave up: make the arrivals that are left (the next launch counts on whole barriers), wait (bounded) for this warp's
    // copies that are still in flight, then leave
    if (tid == 0) red_release_add_u64(a.bar_counter, (u64)(CHAIN_BARRIERS * a.k) - (bar_target - misc->bar_base) / (u64)G);
    for (unsigned ci = t.ci; ci < t.fi; ++ci) {
        const uint32_t bar = bar0 + (ci % CHAIN_STAGES) * 8;
        const uint32_t parity = (ci / CHAIN_STAGES) & 1u;
        const long long t0 = clock64();
        while (!mbar_try_wait(bar, parity))
            if (clock64() - t0 > a.wait_cycles) break;
    }
}

// ------------------------------------------------------------------------------------------ host side
// Cache rows of a unit that are staged, at most.  With 32 heads a head has four units, of a quarter of the rows in whole blocks of 32:
// all of up to 512 rows in bf16, and at d 4096 in fp32, where x leaves room for 84, of up to 256.  Longer ones are attn_unit's: five
// steps at d 4096 take 661 us at 128 to 512 rows, 709 from 513 on, 725 at 1024.
#define CHAIN_ATTN_ROWS 128
struct ChainPlan {
    int off_x, off_part, off_bar, off_misc;
    int attn_rows;             // rows of K and V that the room of x holds
    size_t smem_bytes;
};

static ChainPlan chain_plan(const ChainArgs& a, int es, int dh, int grid) {
    ChainPlan p;
    int kmax = 0;
    long long slots = 0;
    for (int i = 0; i < PH_COUNT; ++i) {
        if (a.ph[i].K > kmax) kmax = a.ph[i].K;
        const long long rows = (a.ph[i].N + grid - 1) / grid + 2;
        const long long cpr = ((long long)a.ph[i].K * es + CHAIN_CHUNK_BYTES - 1) / CHAIN_CHUNK_BYTES;
        if (rows * cpr > slots) slots = rows * cpr;
    }
    size_t x_bytes = (size_t)kmax * 4;
    const size_t attn_bytes = dh == 128 ? sizeof(AttnSmem<CHAIN_WARPS, 1, 128>) : sizeof(AttnSmem<CHAIN_WARPS, 1, 64>);
    if (attn_bytes > x_bytes) x_bytes = attn_bytes;
    // the attention stages up to CHAIN_ATTN_ROWS rows of K and V, as many as fit beside the rest
    const size_t fixed = dh == 128 ? sizeof(ChainAttnSmem<float, 128>) : sizeof(ChainAttnSmem<float, 64>);
    const size_t row = (size_t)(2 * dh * es + 16);
    const size_t other = (size_t)CHAIN_WARPS * CHAIN_STAGES * (CHAIN_CHUNK_BYTES + 8) + (size_t)slots * 4 + CHAIN_MISC_BYTES + 512;
    const size_t room = (size_t)227 * 1024 > other ? (size_t)227 * 1024 - other : 0;
    size_t want = fixed + CHAIN_ATTN_ROWS * row;
    if (want > room) want = room;
    if (want > x_bytes) x_bytes = want;
    p.attn_rows = x_bytes > fixed ? (int)((x_bytes - fixed) / row) : 0;
    size_t off = (size_t)CHAIN_WARPS * CHAIN_STAGES * CHAIN_CHUNK_BYTES;
    p.off_x = (int)off;
    off += (x_bytes + 127) & ~(size_t)127;
    p.off_part = (int)off;
    off += ((size_t)slots * 4 + 127) & ~(size_t)127;
    p.off_bar = (int)off;
    off += CHAIN_WARPS * CHAIN_STAGES * 8;
    off = (off + 15) & ~(size_t)15;
    p.off_misc = (int)off;
    off += CHAIN_MISC_BYTES;
    p.smem_bytes = off;
    return p;
}

template <typename WT, int DH>
static cudaError_t chain_launch_t(ChainArgs& a, int grid, size_t smem, cudaStream_t st) {
    // the shared-memory opt-in is a per-device attribute of the function: remember it per device ordinal
    static size_t attr_smem[HIVIS_MAX_DEVICES] = {0};
    int dev = 0;
    cudaError_t e0 = cudaGetDevice(&dev);
    if (e0 != cudaSuccess) return e0;
    if (dev < 0 || dev >= HIVIS_MAX_DEVICES || smem > attr_smem[dev]) {
        cudaError_t e = cudaFuncSetAttribute(draft_chain_kernel<WT, DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < HIVIS_MAX_DEVICES) attr_smem[dev] = smem;
    }
    void* params[] = {(void*)&a};
    return cudaLaunchCooperativeKernel((const void*)draft_chain_kernel<WT, DH>, dim3(grid), dim3(CHAIN_THREADS), params, smem, st);
}

// Shared-memory bytes the chain kernel needs for these dimensions (0 = does not fit).
size_t chain_smem_bytes(const ChainArgs& a, int dtype, int grid) {
    const ChainPlan p = chain_plan(a, dtype == HIVIS_BF16 ? 2 : 4, a.dh, grid);
    return p.smem_bytes <= 227 * 1024 ? p.smem_bytes : 0;
}

cudaError_t launch_draft_chain(ChainArgs& a, int dtype, int grid, cudaStream_t st) {
    const ChainPlan p = chain_plan(a, dtype == HIVIS_BF16 ? 2 : 4, a.dh, grid);
    if (p.smem_bytes > 227 * 1024) return cudaErrorInvalidValue;
    a.attn_rows = p.attn_rows;
    a.off_x = p.off_x; a.off_part = p.off_part; a.off_bar = p.off_bar; a.off_misc = p.off_misc;
    if (dtype == HIVIS_BF16)
        return a.dh == 128 ? chain_launch_t<bf16, 128>(a, grid, p.smem_bytes, st) : chain_launch_t<bf16, 64>(a, grid, p.smem_bytes, st);
    return a.dh == 128 ? chain_launch_t<float, 128>(a, grid, p.smem_bytes, st) : chain_launch_t<float, 64>(a, grid, p.smem_bytes, st);
}
