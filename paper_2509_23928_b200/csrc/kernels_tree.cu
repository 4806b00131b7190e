// Tree drafting and greedy tree verification: the kernels around the layer.
//
// A draft tree is built level by level.  Level 0 runs the pending pair (one row); level l >= 1 runs the `topk`
// frontier nodes of depth l as a batch of rows through the same fused linear kernels as a chained step.  What is
// specific to the tree lives here: the gather of every node's input (the layer output of the forward that proposed
// it, its token), tree attention (a node sees the prefix, its ancestors and itself), log-softmax + top-k of every
// node's logits, the choice of the next frontier by cumulative log-probability, the final ranking of all
// candidates, and - after the target has scored the kept nodes - the walk along the accepted path with the
// compaction of its K/V rows.  All bookkeeping stays on the device; the host only sequences launches.
//
// Where the rows of the tree live: the node that is the j-th of the level-l frontier keeps its K/V row in cache row
// P + 1 + (l - 1) * topk + j of its slot (P = rows of the slot before the draft, row P = the root position).
#include "attn_body.cuh"

// ------------------------------------------------------------------------------------------ begin / gather
__global__ void tree_begin_kernel(int slot, int d, const int* kv_len, const float* pend_feat, const int* pend_id,
                                  float* feat, bf16* feat_h, int* cur_id, int* d_slots, TreeBufs T) {
    pdl_wait();
    pdl_trigger();
    if (threadIdx.x == 0) {
        *T.P = kv_len[slot];
        *T.cand_n = 0;
        cur_id[0] = pend_id[slot];
        T.fr_cand[0] = -1;
        T.fr_store[0] = 0;
        T.fr_score[0] = 0.f;
    }
    if (threadIdx.x < TREE_MAX_TOPK) d_slots[threadIdx.x] = slot;
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
        const float v = pend_feat[(long long)slot * d + i];
        feat[i] = v;
        feat_h[i] = __float2bfloat16_rn(v);
    }
}
cudaError_t launch_tree_begin(int slot, int d, const int* kv_len, const float* pend_feat, const int* pend_id, float* feat,
                              bf16* feat_h, int* cur_id, int* d_slots, const TreeBufs& T, cudaStream_t st) {
    return launch_pdl(tree_begin_kernel, dim3(1), dim3(256), 0, st, slot, d, kv_len, pend_feat, pend_id, feat, feat_h, cur_id, d_slots, T);
}

// row j of the level's input: the layer output of the forward that proposed node j, and node j's token
__global__ void tree_gather_kernel(int d, const float* g_prev, TreeBufs T, float* feat, bf16* feat_h, int* cur_id) {
    pdl_wait();
    pdl_trigger();
    const int j = blockIdx.x;
    const float* src = g_prev + (long long)T.fr_pslot[j] * d;
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
        const float v = src[i];
        feat[(long long)j * d + i] = v;
        feat_h[(long long)j * d + i] = __float2bfloat16_rn(v);
    }
    if (threadIdx.x == 0) cur_id[j] = T.fr_tok[j];
}
cudaError_t launch_tree_gather(int nb, int d, const float* g_prev, const TreeBufs& T, float* feat, bf16* feat_h, int* cur_id,
                               cudaStream_t st) {
    return launch_pdl(tree_gather_kernel, dim3((unsigned)nb), dim3(256), 0, st, d, g_prev, T, feat, feat_h, cur_id);
}

// The level's rows in the form the tensor-core chain kernel reads them: the features as bf16 rows with their rounding
// remainders `lo_rows` rows further down, the embedding rows of the nodes' tokens (zero rows beyond the level: the
// tiled copy always brings all rows).  Level 0 (g_prev null): the slot's pending pair, and the bookkeeping of a new tree;
// later levels: row j = the layer output of the forward that proposed node j, and node j's token.  Eight elements per
// thread: 11 us with one (and 10 us more for a level-0 launch of its own).
__global__ void __launch_bounds__(512) tree_operands_tc_kernel(int nb, int d, int lo_rows, int slot, const int* kv_len,
                                        const float* pend_feat, const int* pend_id, const float* g_prev,
                                        TreeBufs T, const bf16* embed, int vocab, bf16* feat_h, bf16* xe_h, int* id_flag) {
    pdl_wait();
    pdl_trigger();
    const int j = blockIdx.x, upr = d >> 3;
    uint4* xe = (uint4*)(xe_h + (long long)j * d);
    if (j >= nb) {
        for (int i = threadIdx.x; i < upr; i += blockDim.x) xe[i] = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    const int tok = g_prev ? T.fr_tok[j] : pend_id[slot];
    const float4* src = (const float4*)(g_prev ? g_prev + (long long)T.fr_pslot[j] * d : pend_feat + (long long)slot * d);
    if (!g_prev && threadIdx.x == 0) {
        *T.P = kv_len[slot];
        *T.cand_n = 0;
        T.fr_cand[0] = -1;
        T.fr_store[0] = 0;
        T.fr_score[0] = 0.f;
    }
    const uint4* er = (const uint4*)(embed + (long long)checked_token(tok, vocab, id_flag) * d);
    for (int i = threadIdx.x; i < upr; i += blockDim.x) {
        const float4 x = src[2 * i], y = src[2 * i + 1];
        xe[i] = er[i];
        const float v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
        unsigned hi[4], rem[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bf16 h0 = __float2bfloat16_rn(v[2 * q]), h1 = __float2bfloat16_rn(v[2 * q + 1]);
            hi[q] = (unsigned)__bfloat16_as_ushort(h0) | ((unsigned)__bfloat16_as_ushort(h1) << 16);
            rem[q] = (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(v[2 * q] - __bfloat162float(h0))) |
                     ((unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(v[2 * q + 1] - __bfloat162float(h1))) << 16);
        }
        ((uint4*)(feat_h + (long long)j * d))[i] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        ((uint4*)(feat_h + (long long)(j + lo_rows) * d))[i] = make_uint4(rem[0], rem[1], rem[2], rem[3]);
    }
}
cudaError_t launch_tree_operands_tc(int nb, int rows, int d, int lo_rows, int slot, const int* kv_len, const float* pend_feat,
                                    const int* pend_id, const float* g_prev, const TreeBufs& T, const bf16* embed, int vocab,
                                    bf16* feat_h, bf16* xe_h, int* id_flag, cudaStream_t st) {
    return launch_pdl(tree_operands_tc_kernel, dim3((unsigned)rows), dim3(512), 0, st, nb, d, lo_rows, slot, kv_len, pend_feat, pend_id, g_prev, T, embed, vocab, feat_h, xe_h, id_flag);
}

// ------------------------------------------------------------------------------------------ tree attention
// One CTA of four warps per (query head, node).  The node attends to the prefix rows [0, P), to the rows of its ancestors
// (the root position first) and to its own row: `level` + 1 tree rows.  Its own K (rotated) and V are made here, in the form
// the cache holds, and read from shared memory in their place at the end of the rows; the first head of a KV group writes them
// to the cache: nobody else reads that row in this level (a launch of its own for the rows took 15 us).  Blocks of 32 rows are
// dealt to the warps in turn.  Scores: a lane takes one row of the block and the whole dot product with the query (in shared
// memory), so no shuffle is needed; the block's probabilities then go through an online softmax, and for the weighted sum
// of the V rows a lane owns DH/32 output elements and every row's probability is broadcast from its lane, eight rows' loads
// in flight.  The four warps' (max, sum, accumulator) are merged at the end.  The order of all sums belongs to the result:
// a tree's list of nodes is decided by differences that another order would move.
#define TREE_ATT_WARPS 4
template <typename WT, int DH>
__device__ __forceinline__ float tree_row_dot(const WT* k, const float* q) {
    float sc = 0.f;
    if constexpr (sizeof(WT) == 2) {
        const uint4* kp = (const uint4*)k;
#pragma unroll
        for (int c = 0; c < DH / 8; ++c) {
            const uint4 w = kp[c];
            sc = fmaf(q[8 * c + 0], bf16_lo(w.x), sc); sc = fmaf(q[8 * c + 1], bf16_hi(w.x), sc);
            sc = fmaf(q[8 * c + 2], bf16_lo(w.y), sc); sc = fmaf(q[8 * c + 3], bf16_hi(w.y), sc);
            sc = fmaf(q[8 * c + 4], bf16_lo(w.z), sc); sc = fmaf(q[8 * c + 5], bf16_hi(w.z), sc);
            sc = fmaf(q[8 * c + 6], bf16_lo(w.w), sc); sc = fmaf(q[8 * c + 7], bf16_hi(w.w), sc);
        }
    } else {
        const float4* kp = (const float4*)k;
#pragma unroll
        for (int c = 0; c < DH / 4; ++c) {
            const float4 w = kp[c];
            sc = fmaf(q[4 * c + 0], w.x, sc); sc = fmaf(q[4 * c + 1], w.y, sc);
            sc = fmaf(q[4 * c + 2], w.z, sc); sc = fmaf(q[4 * c + 3], w.w, sc);
        }
    }
    return sc;
}
template <typename WT, int DH>
__global__ void __launch_bounds__(TREE_ATT_WARPS * 32) tree_attn_kernel(const float* qkv, int ld, int Hq, int Hkv, int max_len, int slot,
                                                        int level, TreeBufs T, const double* inv_freq, float scale,
                                                        void* Kc, void* Vc, float* attn, bf16* attn_h, int lo_rows) {
    pdl_wait();
    pdl_trigger();
    constexpr int EPL = DH / 32, NT = TREE_ATT_WARPS * 32;
    __shared__ float s_m[TREE_ATT_WARPS], s_l[TREE_ATT_WARPS], s_acc[TREE_ATT_WARPS][DH];
    __shared__ __align__(16) float s_q[DH];
    __shared__ __align__(16) WT s_k[DH], s_v[DH];
    __shared__ float2 s_cs[DH / 2];
    const int h = blockIdx.x, j = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int P = *T.P, pos = P + level, G = Hq / Hkv, kvh = h / G, half = DH / 2;
    const long long base = ((long long)slot * Hkv + kvh) * max_len;
    const float* qh = qkv + (long long)j * ld + h * DH;
    const float* kh = qkv + (long long)j * ld + (Hq + kvh) * DH;
    const float* vh = kh + Hkv * DH;
    if (threadIdx.x < half) {
        float c, s;
        rope_cs(pos, inv_freq[threadIdx.x], c, s);
        s_cs[threadIdx.x] = make_float2(c, s);
    }
    __syncthreads();
    // the rotated, scaled query; the node's own row
    const long long own = (base + P + T.fr_store[j]) * DH;
    const bool writer = h % G == 0;
    for (int t = threadIdx.x; t < 3 * DH; t += NT) {
        const int what = t / DH, i = t % DH, f = i % half;
        const float* src = what == 0 ? qh : what == 1 ? kh : vh;
        const float x = src[i];
        if (what == 2) {
            store_from_float<WT>(s_v, i, x);
            if (writer) store_from_float<WT>(Vc, own + i, x);
            continue;
        }
        const float c = s_cs[f].x, s = s_cs[f].y;
        const float y = src[i < half ? i + half : i - half];
        // (written out, so that every build of the code rounds the same product)
        const float r = i < half ? fmaf(x, c, -__fmul_rn(y, s)) : what == 0 ? fmaf(x, c, __fmul_rn(y, s)) : fmaf(y, s, __fmul_rn(x, c));
        if (what == 0) {
            s_q[i] = r * scale;
        } else {
            store_from_float<WT>(s_k, i, r);
            if (writer) store_from_float<WT>(Kc, own + i, r);
        }
    }
    __syncthreads();
    const int nrows = P + level + 1;                                 // the prefix, the ancestors, the node itself
    float m = -INFINITY, l = 0.f, acc[EPL];
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
    for (int r0 = warp * 32; r0 < nrows; r0 += NT) {
        const int r = r0 + lane;
        const bool ok = r < nrows;
        int row = ok ? r : r0;
        if (ok && r >= P) row = r - P < level ? P + T.fr_anc[j * TREE_MAX_DEPTH + (r - P)] : -1;     // -1: the node's own row
        row = __shfl_sync(0xffffffffu, row, ok ? lane : 0);          // lanes beyond the rows read the block's first
        const float sc = ok ? tree_row_dot<WT, DH>(row < 0 ? s_k : (const WT*)Kc + (base + row) * DH, s_q) : -INFINITY;
        float bm = sc;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, off));
        const float mn = fmaxf(m, bm);                               // finite: the block has at least one row
        const float corr = expf(m - mn), p = ok ? expf(sc - mn) : 0.f;
        float ps = p;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, off);
        l = l * corr + ps;
        m = mn;
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[e] *= corr;
        const int nr = min(32, nrows - r0);
#pragma unroll 1
        for (int t0 = 0; t0 < nr; t0 += 8) {
            float vf[8][EPL];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int rowj = __shfl_sync(0xffffffffu, row, t0 + t);
                const WT* vp = (rowj < 0 ? s_v : (const WT*)Vc + (base + rowj) * DH) + lane * EPL;
                if constexpr (sizeof(WT) == 2 && EPL == 4) {
                    const uint2 w = *(const uint2*)vp;
                    vf[t][0] = bf16_lo(w.x); vf[t][1] = bf16_hi(w.x); vf[t][2] = bf16_lo(w.y); vf[t][3] = bf16_hi(w.y);
                } else if constexpr (sizeof(WT) == 2 && EPL == 2) {
                    const unsigned w = *(const unsigned*)vp;
                    vf[t][0] = bf16_lo(w); vf[t][1] = bf16_hi(w);
                } else {
#pragma unroll
                    for (int e = 0; e < EPL; ++e) vf[t][e] = load_as_float<WT>(vp, e);
                }
            }
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const float pj = __shfl_sync(0xffffffffu, p, t0 + t);        // 0 beyond the rows
                if (t0 + t < nr) {
#pragma unroll
                    for (int e = 0; e < EPL; ++e) acc[e] = fmaf(pj, vf[t][e], acc[e]);
                }
            }
        }
    }
    if (lane == 0) { s_m[warp] = m; s_l[warp] = l; }
#pragma unroll
    for (int e = 0; e < EPL; ++e) s_acc[warp][lane * EPL + e] = acc[e];
    __syncthreads();
    if (warp == 0) {
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < TREE_ATT_WARPS; ++w) M = fmaxf(M, s_m[w]);
        float L = 0.f, A[EPL];
#pragma unroll
        for (int e = 0; e < EPL; ++e) A[e] = 0.f;
#pragma unroll
        for (int w = 0; w < TREE_ATT_WARPS; ++w) {
            const float f = s_l[w] > 0.f ? expf(s_m[w] - M) : 0.f;   // a warp without rows contributes nothing
            L += s_l[w] * f;
#pragma unroll
            for (int e = 0; e < EPL; ++e) A[e] += s_acc[w][lane * EPL + e] * f;
        }
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            const float o = A[e] / L;
            const long long oi = (long long)j * Hq * DH + h * DH + lane * EPL + e;
            attn[oi] = o;
            const bf16 hi = __float2bfloat16_rn(o);
            attn_h[oi] = hi;
            if (lo_rows > 0) attn_h[oi + (long long)lo_rows * Hq * DH] = __float2bfloat16_rn(o - __bfloat162float(hi));
        }
    }
}

cudaError_t launch_tree_attention(int dtype, int nb, const float* qkv, int ld, int Hq, int Hkv, int dh, int max_len,
                                  int slot, int level, const TreeBufs& T, const double* inv_freq, void* Kc, void* Vc,
                                  float* attn, bf16* attn_h, int lo_rows, cudaStream_t st) {
    const float scale = 1.0f / sqrtf((float)dh);
    const dim3 grid((unsigned)Hq, (unsigned)nb);
    const int nt = TREE_ATT_WARPS * 32;
    auto kernel = dtype == HIVIS_BF16 ? (dh == 128 ? tree_attn_kernel<bf16, 128> : tree_attn_kernel<bf16, 64>)
                                      : (dh == 128 ? tree_attn_kernel<float, 128> : tree_attn_kernel<float, 64>);
    return launch_pdl(kernel, grid, dim3(nt), 0, st, qkv, ld, Hq, Hkv, max_len, slot, level, T, inv_freq, scale, Kc, Vc, attn, attn_h, lo_rows);
}

// ------------------------------------------------------------------------------------------ log-softmax + top-k
// One CTA per node: maximum, log-sum-exp, then the `topk` largest logits one after the other.  The packed key
// orders by value, then by lower token id, and every round takes the largest key below the previous one, so
// equal logits come out in token order.
__device__ __forceinline__ float block_reduce_max(float v, float* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float r = red[0];
    for (int w = 1; w < 8; ++w) r = fmaxf(r, red[w]);
    return r;
}
__device__ __forceinline__ float block_reduce_sum(float v, float* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float r = 0.f;
    for (int w = 0; w < 8; ++w) r += red[w];
    return r;
}
#define TREE_PIECE 4096          // logits of a node that one CTA covers (16 per thread, kept in registers)
int tree_topk_pieces(int V) { return (V + TREE_PIECE - 1) / TREE_PIECE; }

// One launch per level: log-softmax and top-k of every node, then the next frontier.
//   One CTA per (piece of the row, node): the piece's maximum and sum of exp(x - max), and its `topk` largest keys, largest
//   first.  A thread keeps its 16 logits in registers and its current best key; a round takes the block's best, and only
//   the thread that owned it looks for its next one.
//   The CTA that completes a node's count merges the node: log-sum-exp from the pieces, and the pieces' keys ranked by
//   counting the larger ones (keys are unique; the order is by value, then by lower token id).
//   The CTA that completes the level's count chooses the frontier.  Nobody waits for anybody.  As three launches the level
//   spent 27 us here, most of it in a single warp that walked the sorted lists.
#define TREE_MERGE_CAP 1024      // keys of a node ranked from shared memory (more: from global memory)

// What a score ranks as.  A score that is not a number (weights or states that are not) ranks last: compared as it is it
// would be beaten by nobody, and more nodes would be chosen than the lists hold.
__device__ __forceinline__ float tree_rank_of(float score) { return score == score ? score : -INFINITY; }

// The nb * topk children of this level become candidates (creation order: frontier order, then rank); unless this was
// the last level, the `topk` of them with the highest cumulative log-probability (earlier candidate first among
// equals) form the next frontier, kept in creation order.
__device__ void tree_select(int level, int depth, int nb, int topk, const TreeBufs& T) {
    __shared__ float s_score[256];
    __shared__ int s_sel[256];
    __shared__ int s_anc[TREE_MAX_TOPK][TREE_MAX_DEPTH], s_store[TREE_MAX_TOPK], s_cand[TREE_MAX_TOPK];
    const int i = threadIdx.x, n = nb * topk;
    const int base = *T.cand_n;
    const int j = i / topk, r = i % topk;
    if (i < TREE_MAX_TOPK * TREE_MAX_DEPTH) s_anc[i / TREE_MAX_DEPTH][i % TREE_MAX_DEPTH] = T.fr_anc[i];
    if (i < TREE_MAX_TOPK) { s_store[i] = T.fr_store[i]; s_cand[i] = T.fr_cand[i]; }
    float score = -INFINITY;
    int tok = 0;
    if (i < n) {
        tok = __ldcg(T.top_tok + j * TREE_MAX_TOPK + r);
        score = T.fr_score[j] + __ldcg(T.top_lp + j * TREE_MAX_TOPK + r);
        T.cand_tok[base + i] = tok;
        T.cand_par[base + i] = T.fr_cand[j];
        T.cand_depth[base + i] = level + 1;
        T.cand_score[base + i] = score;
        T.cand_store[base + i] = -1;
    }
    const float mine = tree_rank_of(score);
    s_score[i] = mine;
    __syncthreads();
    int sel = 0;
    if (i < n && level + 1 < depth) {
        int rank = 0;
        for (int o = 0; o < n; ++o) rank += (s_score[o] > mine || (s_score[o] == mine && o < i)) ? 1 : 0;
        sel = rank < topk ? 1 : 0;
    }
    s_sel[i] = sel;
    __syncthreads();
    if (sel) {
        int pos = 0;
        for (int o = 0; o < i; ++o) pos += s_sel[o];
        const int store = 1 + level * topk + pos;              // the node joins the frontier of level + 1
        T.fr_cand[pos] = base + i;
        T.fr_tok[pos] = tok;
        T.fr_score[pos] = score;
        T.fr_pslot[pos] = j;
        T.fr_store[pos] = store;
        for (int a = 0; a < level; ++a) T.fr_anc[pos * TREE_MAX_DEPTH + a] = s_anc[j][a];
        T.fr_anc[pos * TREE_MAX_DEPTH + level] = s_store[j];   // the parent's row (the root's when level == 0)
        T.cand_store[base + i] = store;
    }
    if (i == 0) *T.cand_n = base + n;
}

// the CTA arrives on *counter; true for all its threads if it completed the count (the counter is zero again then)
__device__ __forceinline__ bool tree_arrive(int* counter, int count) {
    __shared__ int s_last;
    __syncthreads();                          // every thread's stores are before the arrival
    if (threadIdx.x == 0) {
        __threadfence();
        const int last = atomicAdd(counter, 1) == count - 1;
        if (last) *counter = 0;
        __threadfence();
        s_last = last;
    }
    __syncthreads();
    return s_last != 0;
}

__global__ void __launch_bounds__(256) tree_topk_select_kernel(const float* logits, int V, int topk, int level, int depth,
                                                               float2* piece_stats, u64* piece_keys, TreeBufs T) {
    pdl_wait();
    pdl_trigger();
    __shared__ float red[8];
    __shared__ u64 kred[8];
    __shared__ u64 s_keys[TREE_MERGE_CAP];
    const int piece = blockIdx.x, j = blockIdx.y, pieces = gridDim.x, nb = gridDim.y;
    const float* x = logits + (long long)j * V;
    const int c0 = piece * TREE_PIECE;
    u64 key[TREE_PIECE / 256];
    float v[TREE_PIECE / 256];
    float mx = -INFINITY;
#pragma unroll
    for (int t = 0; t < TREE_PIECE / 256; ++t) {
        const int i = c0 + t * 256 + threadIdx.x;
        v[t] = i < V ? x[i] : -INFINITY;
        key[t] = i < V ? pack_key(v[t], i) : 0ull;
        mx = fmaxf(mx, v[t]);
    }
    mx = block_reduce_max(mx, red);
    float se = 0.f;
#pragma unroll
    for (int t = 0; t < TREE_PIECE / 256; ++t) se += expf(v[t] - mx);          // exp(-inf) = 0 beyond the row
    se = block_reduce_sum(se, red);
    if (threadIdx.x == 0) piece_stats[(long long)j * pieces + piece] = make_float2(mx, se);
    u64 mine = 0;
#pragma unroll
    for (int t = 0; t < TREE_PIECE / 256; ++t) mine = key[t] > mine ? key[t] : mine;
    u64* out = piece_keys + ((long long)j * pieces + piece) * TREE_MAX_TOPK;
    for (int r = 0; r < topk; ++r) {
        u64 best = mine;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const u64 other = __shfl_xor_sync(0xffffffffu, best, o);
            best = other > best ? other : best;
        }
        __syncthreads();
        if ((threadIdx.x & 31) == 0) kred[threadIdx.x >> 5] = best;
        __syncthreads();
        best = kred[0];
#pragma unroll
        for (int w = 1; w < 8; ++w) best = kred[w] > best ? kred[w] : best;
        if (threadIdx.x == 0) out[r] = best;
        if (best != 0ull && mine == best) {         // keys are unique (they carry the token id): one owner
            mine = 0;
#pragma unroll
            for (int t = 0; t < TREE_PIECE / 256; ++t) {
                if (key[t] == best) key[t] = 0ull;
                mine = key[t] > mine ? key[t] : mine;
            }
        }
    }
    if (!tree_arrive(T.arrive + j, pieces)) return;
    // ---- merge of the node
    const float2* ps = piece_stats + (long long)j * pieces;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        float mx2 = -INFINITY;
        for (int c = lane; c < pieces; c += 32) mx2 = fmaxf(mx2, __ldcg(ps + c).x);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx2 = fmaxf(mx2, __shfl_xor_sync(0xffffffffu, mx2, o));
        float se2 = 0.f;
        for (int c = lane; c < pieces; c += 32) {
            const float2 w = __ldcg(ps + c);
            se2 += w.y * expf(w.x - mx2);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) se2 += __shfl_xor_sync(0xffffffffu, se2, o);
        if (lane == 0) red[0] = mx2 + logf(se2);
    }
    const u64* pk = piece_keys + (long long)j * pieces * TREE_MAX_TOPK;
    const int nk = pieces * topk;
    const bool in_smem = nk <= TREE_MERGE_CAP;
    if (in_smem)
        for (int i = threadIdx.x; i < nk; i += 256) s_keys[i] = __ldcg(pk + (i / topk) * TREE_MAX_TOPK + i % topk);
    __syncthreads();
    const float lse = red[0];
    for (int i = threadIdx.x; i < nk; i += 256) {
        const u64 mine2 = in_smem ? s_keys[i] : __ldcg(pk + (i / topk) * TREE_MAX_TOPK + i % topk);
        if (mine2 == 0ull) continue;                 // the piece had fewer entries
        int rank = i % topk;                         // its own list is sorted
        for (int c = 0; c < pieces && rank < topk; ++c) {
            if (c == i / topk) continue;
            for (int t = 0; t < topk; ++t) {
                const u64 o = in_smem ? s_keys[c * topk + t] : __ldcg(pk + c * TREE_MAX_TOPK + t);
                if (o < mine2) break;
                ++rank;
            }
        }
        if (rank < topk) {
            const int tok = key_index(mine2);
            __stcg(T.top_tok + j * TREE_MAX_TOPK + rank, tok);
            __stcg(T.top_lp + j * TREE_MAX_TOPK + rank, x[tok] - lse);
        }
    }
    if (!tree_arrive(T.arrive + TREE_MAX_TOPK, nb)) return;
    tree_select(level, depth, nb, topk, T);
}
cudaError_t launch_tree_topk_select(int nb, const float* logits, int V, int topk, int level, int depth, const TreeBufs& T,
                                    cudaStream_t st) {
    return launch_pdl(tree_topk_select_kernel, dim3((unsigned)tree_topk_pieces(V), (unsigned)nb), dim3(256), 0, st, logits, V, topk, level, depth, T.piece_stats, T.piece_keys, T);
}

// ------------------------------------------------------------------------------------------ final ranking
// Of all candidates the `keep` with the highest score (earlier candidate first among equals) are the draft tree,
// listed in creation order, parents re-numbered within the list.
__global__ void __launch_bounds__(1024) tree_finalize_kernel(int keep, TreeBufs T, int32_t* out_tokens, int32_t* out_parents,
                                                             float* out_scores, int32_t* out_count) {
    pdl_wait();
    pdl_trigger();
    __shared__ float s_score[TREE_MAX_CAND];
    __shared__ unsigned short s_pos[TREE_MAX_CAND];          // 1 + position among the kept, 0 = not kept
    __shared__ int s_sum[32];
    const int n = *T.cand_n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < n; i += 1024) s_score[i] = tree_rank_of(T.cand_score[i]);
    __syncthreads();
    int before = 0;                                          // kept candidates of the earlier turns
    for (int i0 = 0; i0 < n; i0 += 1024) {
        const int i = i0 + tid;
        bool kept = false;
        if (i < n) {
            const float sc = s_score[i];
            int rank = 0;
#pragma unroll 4
            for (int o = 0; o < n; ++o) rank += (s_score[o] > sc || (s_score[o] == sc && o < i)) ? 1 : 0;
            kept = rank < keep;
        }
        const unsigned mask = __ballot_sync(0xffffffffu, kept);
        if (lane == 0) s_sum[warp] = __popc(mask);
        __syncthreads();
        int pos = before + __popc(mask & ((1u << lane) - 1u));
        for (int w = 0; w < 32; ++w) {
            if (w < warp) pos += s_sum[w];
            before += s_sum[w];
        }
        if (i < n) s_pos[i] = kept ? (unsigned short)(pos + 1) : 0;
        __syncthreads();
    }
    for (int i = tid; i < n; i += 1024) {
        const int pos = (int)s_pos[i] - 1;
        if (pos < 0) continue;
        const int par = T.cand_par[i];
        const int pp = par < 0 ? -1 : (int)s_pos[par] - 1;
        const int tok = T.cand_tok[i];
        T.kept_tok[pos] = tok;
        T.kept_par[pos] = pp;
        T.kept_store[pos] = T.cand_store[i];
        out_tokens[pos] = tok;
        out_parents[pos] = pp;
        out_scores[pos] = T.cand_score[i];
    }
    if (tid == 0) {
        const int cnt = n < keep ? n : keep;
        *T.kept_n = cnt;
        if (out_count) *out_count = cnt;
    }
}
cudaError_t launch_tree_finalize(int keep, const TreeBufs& T, int32_t* out_tokens, int32_t* out_parents, float* out_scores,
                                 int32_t* out_count, cudaStream_t st) {
    return launch_pdl(tree_finalize_kernel, dim3(1), dim3(1024), 0, st, keep, T, out_tokens, out_parents, out_scores, out_count);
}

// ------------------------------------------------------------------------------------------ verification
template <typename LT>
__global__ void __launch_bounds__(256) tree_row_argmax_kernel(const void* logits, int V, u64* keys) {
    pdl_wait();
    pdl_trigger();
    __shared__ u64 kred[8];
    const LT* row = (const LT*)logits + (long long)blockIdx.y * V;
    const int c0 = blockIdx.x * 2048, c1 = min(V, c0 + 2048);
    u64 best = 0;
    for (int i = c0 + threadIdx.x; i < c1; i += 256) {
        const u64 kk = pack_key(load_as_float<LT>(row, i), i);
        best = kk > best ? kk : best;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const u64 other = __shfl_xor_sync(0xffffffffu, best, o);
        best = other > best ? other : best;
    }
    if ((threadIdx.x & 31) == 0) kred[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        u64 m = kred[0];
        for (int w = 1; w < 8; ++w) m = kred[w] > m ? kred[w] : m;
        atomicMax(keys + blockIdx.y, m);
    }
}

// The walk: from the root, follow the child that carries the target's argmax for as long as there is one (the kept nodes
// in shared memory, one per lane and turn).  Then the K/V rows of the accepted nodes that have one are moved right behind
// the root's row, in path order, and the slot gets its new row count.  Every CTA walks, and moves a slice of the rows: a
// thread reads its 16 bytes of all rows before it writes the first, and nobody else touches them.
#define TREE_WALK_CTAS 8
template <typename WT>
__global__ void __launch_bounds__(256) tree_walk_kernel(int slot, int depth, int Hkv, int dh, int max_len, TreeBufs T,
                                                        const u64* keys, void* Kc, void* Vc, int* kv_len, int32_t* out_accept,
                                                        int32_t* out_path, int32_t* out_next, int32_t* out_kv_len) {
    pdl_wait();
    pdl_trigger();
    __shared__ int s_path[TREE_MAX_DEPTH], s_src[TREE_MAX_DEPTH], s_rows;
    __shared__ int s_tok[HIVIS_TREE_MAX_KEEP], s_par[HIVIS_TREE_MAX_KEEP], s_store[HIVIS_TREE_MAX_KEEP], s_arg[HIVIS_TREE_MAX_KEEP + 1];
    const int n = *T.kept_n, P = *T.P, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < n; i += 256) {
        s_tok[i] = T.kept_tok[i];
        s_par[i] = T.kept_par[i];
        s_store[i] = T.kept_store[i];
    }
    for (int i = threadIdx.x; i <= n; i += 256) s_arg[i] = key_index(keys[i]);
    __syncthreads();
    if (threadIdx.x < 32) {
        int cur = -1, acc = 0, t = 0;
        for (;;) {
            t = s_arg[cur + 1];
            unsigned nxt = 0xffffffffu;
            for (int i = lane; i < n; i += 32)
                if (s_par[i] == cur && s_tok[i] == t) { nxt = (unsigned)i; break; }
            nxt = __reduce_min_sync(0xffffffffu, nxt);
            if (nxt == 0xffffffffu || acc >= depth) break;
            cur = (int)nxt;
            if (lane == 0) s_path[acc] = cur;
            ++acc;
        }
        __syncwarp();
        int rows = 0;
        while (rows < acc && s_store[s_path[rows]] >= 0) ++rows;
        if (lane < rows) s_src[lane] = P + s_store[s_path[lane]];
        if (lane == 0) s_rows = rows;
        if (blockIdx.x == 0) {
            if (lane < depth) out_path[lane] = lane < acc ? s_path[lane] : -1;
            if (lane == 0) {
                *out_accept = acc;
                *out_next = t;
                kv_len[slot] = P + 1 + rows;
                if (out_kv_len) *out_kv_len = P + 1 + rows;
            }
        }
    }
    __syncthreads();
    const int rows = s_rows, vpr = dh * (int)sizeof(WT) / 16;        // 16-byte units of a head's row
    for (int i = blockIdx.x * 256 + threadIdx.x; i < 2 * Hkv * vpr; i += TREE_WALK_CTAS * 256) {
        const int h = (i / vpr) % Hkv, e = i % vpr;
        uint4* base = (uint4*)(i < Hkv * vpr ? Kc : Vc) + ((long long)slot * Hkv + h) * max_len * vpr + e;
        uint4 w[TREE_MAX_DEPTH];
#pragma unroll
        for (int m = 0; m < TREE_MAX_DEPTH; ++m)
            if (m < rows) w[m] = base[(long long)s_src[m] * vpr];
#pragma unroll
        for (int m = 0; m < TREE_MAX_DEPTH; ++m)
            if (m < rows) base[(long long)(P + 1 + m) * vpr] = w[m];
    }
}

cudaError_t launch_tree_verify(int dtype, int logits_dtype, int slot, int depth, int rows, int V, int Hkv, int dh, int max_len,
                               const TreeBufs& T, const void* logits, void* Kc, void* Vc, int* kv_len, int32_t* out_accept,
                               int32_t* out_path, int32_t* out_next, int32_t* out_kv_len, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(T.row_keys, 0, sizeof(u64) * rows, st);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((V + 2047) / 2048), (unsigned)rows);
    e = launch_pdl(logits_dtype == HIVIS_BF16 ? tree_row_argmax_kernel<bf16> : tree_row_argmax_kernel<float>, grid, dim3(256), 0, st, logits, V, T.row_keys);
    if (e != cudaSuccess) return e;
    return launch_pdl(dtype == HIVIS_BF16 ? tree_walk_kernel<bf16> : tree_walk_kernel<float>, dim3(TREE_WALK_CTAS), dim3(256), 0, st, slot, depth, Hkv, dh, max_len, T, T.row_keys, Kc, Vc, kv_len,
                      out_accept, out_path, out_next, out_kv_len);
}
