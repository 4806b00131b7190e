// Host side of the tensor-core draft-chain kernel (tc_chain.cuh): tensor maps, the set-up kernel, the choice of the
// kernel variant.  The variants are instantiated one or two per file (kernels_tc_*.cu): each takes tens of seconds to
// compile.
#include <cuda.h>

#include "hivis_internal.cuh"

#define TC_BK 64
#define TC_TM 128

template <int DH, int GQ, bool SMP, int NG>
cudaError_t tc_launch_t(const TcMaps& maps, const TcArgs& a, int grid, cudaStream_t st);

// ------------------------------------------------------------------------------------------ set-up kernel
// One CTA per operand row, eight elements per thread and turn (d is a multiple of 64): a chain of two loads, 11.5 us with
// an element per thread and turn.
__global__ void __launch_bounds__(512) tc_setup_kernel(SlotList sl, int k, int d, int lo, int* d_slots, int* d_pos0, int* kv_len,
                                const float* pend_feat, const int* pend_id, float* feat, bf16* feat_h, int* cur_id,
                                u64* keys, int key_stride, const bf16* embed, int vocab, bf16* xe_h, int* id_flag) {
    pdl_wait();
    pdl_trigger();
    const int b = blockIdx.x, upr = d >> 3;
    uint4* xe = (uint4*)(xe_h + (long long)b * d);
    if (b >= sl.n) {
        // Rows of the embedding operand beyond the batch: the tiled copy always brings all rows, and the accumulator
        // columns of the remainder rows are added to those of the batch rows (an embedding row is exact in bf16, so
        // its remainder is zero).  An earlier, larger batch may have left rows here.
        for (int i = threadIdx.x; i < upr; i += blockDim.x) xe[i] = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    const int slot = sl.slot[b];
    const int tok = pend_id[slot];
    if (threadIdx.x == 0) {
        d_slots[b] = slot;
        const int rows = kv_len[slot];
        d_pos0[b] = rows;
        kv_len[slot] = rows + k;            // every draft step appends one K/V row
        cur_id[b] = tok;
    }
    if (threadIdx.x < k) keys[(long long)b * key_stride + threadIdx.x] = 0ull;
    // embedding row of the pending token: the fusion FC's embedding operand of step 0
    const uint4* er = (const uint4*)(embed + (long long)checked_token(tok, vocab, id_flag) * d);
    const float4* pf = (const float4*)(pend_feat + (long long)slot * d);
    float4* ff = (float4*)(feat + (long long)b * d);
    for (int i = threadIdx.x; i < upr; i += blockDim.x) {
        const float4 x = pf[2 * i], y = pf[2 * i + 1];
        xe[i] = er[i];
        ff[2 * i] = x;
        ff[2 * i + 1] = y;
        const float v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
        unsigned hi[4], rem[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bf16 h0 = __float2bfloat16_rn(v[2 * q]), h1 = __float2bfloat16_rn(v[2 * q + 1]);
            hi[q] = (unsigned)__bfloat16_as_ushort(h0) | ((unsigned)__bfloat16_as_ushort(h1) << 16);
            rem[q] = (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(v[2 * q] - __bfloat162float(h0))) |
                     ((unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(v[2 * q + 1] - __bfloat162float(h1))) << 16);
        }
        ((uint4*)(feat_h + (long long)b * d))[i] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        if (lo) ((uint4*)(feat_h + (long long)(b + lo) * d))[i] = make_uint4(rem[0], rem[1], rem[2], rem[3]);
    }
}
cudaError_t launch_tc_setup(const SlotList& sl, int k, int d, int lo, int* d_slots, int* d_pos0, int* kv_len,
                            const float* pend_feat, const int* pend_id, float* feat, bf16* feat_h, int* cur_id,
                            u64* keys, int key_stride, const bf16* embed, int vocab, bf16* xe_h, int* id_flag,
                            cudaStream_t st) {
    return launch_pdl(tc_setup_kernel, dim3(sl.n <= TC_OP_ROWS ? TC_OP_ROWS : HIVIS_MAX_BATCH), dim3(512), 0, st, sl, k, d, lo, d_slots, d_pos0, kv_len, pend_feat, pend_id, feat, feat_h,
                      cur_id, keys, key_stride, embed, vocab, xe_h, id_flag);
}

// ------------------------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        fn = (EncodeTiledFn)p;
    }
    return fn;
}

// bf16 row-major [rows][cols] matrix, box = box_rows x 64 columns, 128-byte swizzle, zero fill outside
static cudaError_t encode_map(unsigned char* out, const void* base, long long rows, long long cols, int box_rows,
                              CUtensorMapL2promotion promo) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {TC_BK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn((CUtensorMap*)out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                          box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, promo,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

bool tc_supported(int d, int dh, int Hq, int Hkv, int F) {
    return d % TC_BK == 0 && (dh == 64 || dh == 128) && Hkv > 0 && Hq % Hkv == 0 && F % 8 == 0;
}

int tc_max_tiles(const ChainPhase* ph) {
    int m = 0;
    for (int p = 0; p < PH_COUNT; ++p) {
        const int t = (ph[p].N + TC_TM - 1) / TC_TM;
        if (t > m) m = t;
    }
    return m;
}

// column groups of 16 sequences of a launch: the kernel is built for 1, 2 and 4
int tc_groups(int B) { return B <= 16 ? 1 : B <= 32 ? 2 : 4; }
// Row offset of the rounding remainders in the operand buffers for a batch of B (0: none are kept).
int tc_lo_offset(int B) { return B <= 16 ? 16 : 0; }

cudaError_t tc_build_maps(TcMaps* maps, const ChainPhase* ph, int d, int qw, int F,
                          const bf16* feat_h, const bf16* xq_h, const bf16* attn_h, const bf16* xm_h,
                          const bf16* act_h, const bf16* xe_h, const void* Kc, const void* Vc, long long cache_rows, int dh,
                          int op_rows) {
    static_assert(sizeof(CUtensorMap) == 128, "tensor map size");
    cudaError_t e;
    for (int p = 0; p < PH_COUNT; ++p) {
        e = encode_map(maps->m[TCM_W + p], ph[p].W, ph[p].N, ph[p].K, TC_TM, CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
        if (e != cudaSuccess) return e;
    }
    const struct { int idx; const bf16* base; int cols; } ops[5] = {
        {TCM_X_FEAT, feat_h, d}, {TCM_X_XQ, xq_h, d}, {TCM_X_ATTN, attn_h, qw}, {TCM_X_XM, xm_h, d}, {TCM_X_ACT, act_h, F}};
    for (int i = 0; i < 5; ++i) {
        e = encode_map(maps->m[ops[i].idx], ops[i].base, op_rows, ops[i].cols, op_rows, CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
        if (e != cudaSuccess) return e;
    }
    e = encode_map(maps->m[TCM_X_EMB], xe_h, op_rows, d, op_rows, CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
    if (e != cudaSuccess) return e;
    // the caches as matrices of [slot x KV head x position] rows: boxes of 32 rows x 64 elements
    e = encode_map(maps->m[TCM_K], Kc, cache_rows, dh, 32, CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
    if (e != cudaSuccess) return e;
    return encode_map(maps->m[TCM_V], Vc, cache_rows, dh, 32, CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
}

template <int DH, int GQ>
static cudaError_t tc_launch_greedy(const TcMaps& maps, const TcArgs& a, int grid, cudaStream_t st) {
    switch (tc_groups(a.B)) {
        case 1: return tc_launch_t<DH, GQ, false, 1>(maps, a, grid, st);
        case 2: return tc_launch_t<DH, GQ, false, 2>(maps, a, grid, st);
        default: return tc_launch_t<DH, GQ, false, 4>(maps, a, grid, st);
    }
}
cudaError_t launch_tc_chain(const TcMaps& maps, const TcArgs& a, int grid, cudaStream_t st) {
    const int G = a.Hq / a.Hkv;
    const int gq = (G % 7 == 0) ? 7 : 1;
    if (a.gumbel_u) {
        if (a.B > 16) return cudaErrorInvalidValue;
        if (a.dh == 128) return gq == 7 ? tc_launch_t<128, 7, true, 1>(maps, a, grid, st) : tc_launch_t<128, 1, true, 1>(maps, a, grid, st);
        return gq == 7 ? tc_launch_t<64, 7, true, 1>(maps, a, grid, st) : tc_launch_t<64, 1, true, 1>(maps, a, grid, st);
    }
    if (a.dh == 128) return gq == 7 ? tc_launch_greedy<128, 7>(maps, a, grid, st) : tc_launch_greedy<128, 1>(maps, a, grid, st);
    return gq == 7 ? tc_launch_greedy<64, 7>(maps, a, grid, st) : tc_launch_greedy<64, 1>(maps, a, grid, st);
}
