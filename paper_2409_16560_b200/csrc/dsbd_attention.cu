// dsbd_forest_attention: forest-masked attention for sm_100a.
//
// Every draft node attends to the KV prefix of its own beam plus its ancestors-or-self inside
// its own tree (the topology-aware tree mask, one KV cache per input beam).  A work unit is
// one (beam, KV head): its prefix is a contiguous [L_b, d] matrix for K and for V, and all
// query rows of the tree that map to this KV head (n_tree * Hq/Hkv of them) share it, so the
// prefix is streamed once per unit.
//
// k_forest_attn_simt  fp32-accumulating CUDA-core kernel for any dtype: K/V tiles are staged
//                     in shared memory with 128-bit loads, one to four thread pairs per query row.
#include <cuda_bf16.h>
#include <math.h>


#include "dsbd_attention.cuh"

using namespace dsbd;

namespace {

constexpr int kThreads = 128;
constexpr int kRowsPerBlock = 64;     // query rows per CTA at two threads a row
constexpr int kTok = 32;              // tokens per staged tile
constexpr int kChunk = 8;             // tokens a thread takes between two updates of its running maximum

template <class T> struct Elem;
template <> struct Elem<float> {
    static constexpr int kPerVec = 4;
    __device__ static void widen(const uint4 &v, float *dst) {
        dst[0] = __uint_as_float(v.x); dst[1] = __uint_as_float(v.y);
        dst[2] = __uint_as_float(v.z); dst[3] = __uint_as_float(v.w);
    }
    __device__ static float to_float(float v) { return v; }
    __device__ static float from_float(float v) { return v; }
};
template <> struct Elem<__nv_bfloat16> {
    static constexpr int kPerVec = 8;
    __device__ static void widen(const uint4 &v, float *dst) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            dst[2 * i] = __uint_as_float(w[i] << 16);
            dst[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
    __device__ static float to_float(__nv_bfloat16 v) { return __bfloat162float(v); }
    __device__ static __nv_bfloat16 from_float(float v) { return __float2bfloat16_rn(v); }
};

struct AttnArgs {
    int B, N, Hq, Hkv, group;
    float scale_log2;              // scale * log2(e)
    const int32_t *beam_node_off, *parent;
    const int64_t *prefix_off;
    const void *q, *k_new, *v_new, *k_prefix, *v_prefix;
    void *out;
    int32_t *status;
    int row_blocks;
    int splits;                    // thread pairs per query row
};

// A row belongs to `splits` pairs of neighbouring threads; a pair takes every splits-th token, its two threads
// every other four elements of it.  This kernel serves small calls, whose time is latency: few CTAs, each a
// chain of tiles.  So the next tile's K and V are on their way in registers while one is worked on, small trees use
// the threads that have no row of their own for tokens (4 pairs up to 16 rows, 2 up to 32: a tile's work is the
// chain's step), and the parents are read at once.  Smem rows are padded by 32 bytes: the 16-byte words that
// the pairs of a row and the threads of a pair read together lie in different banks.
// fp32, one thread pair a row, tiles loaded when needed, parents read one by one against this: 2 beams x 15 nodes x
// 4 heads of 64 after 64 tokens 22.7 and 13.7 us a call (10.4 since the binding takes less of it); 8 requests, 6 nodes, 8 heads of 64 after 200-600 tokens
// 174 and 47; 40 requests, 24 rows a unit 507 and 143; heads of 128 in groups of 4 334 and 158 (fp32 at d = 128 spills
// 84 bytes at 255 registers).
template <class T, int D>
__global__ void __launch_bounds__(kThreads)
k_forest_attn_simt(AttnArgs a) {
    constexpr int H = D / 2;              // elements per thread of a pair
    constexpr int RS = D + 8;             // floats from one staged row to the next
    constexpr int PV = Elem<T>::kPerVec, VPR = D / PV, NV = kTok * VPR / kThreads;
    extern __shared__ __align__(16) float smem[];
    float *ks = smem;                     // [kTok][RS]
    float *vs = smem + kTok * RS;         // [kTok][RS]
    __shared__ int par_s[DSBD_MAX_TREE_NODES];
    __shared__ unsigned long long anc[DSBD_MAX_TREE_NODES];

    int unit = blockIdx.x;
    const int rb = unit % a.row_blocks; unit /= a.row_blocks;
    const int g = unit % a.Hkv;
    const int b = unit / a.Hkv;
    const int n_lo = a.beam_node_off[b];
    const int n_tree = a.beam_node_off[b + 1] - n_lo;
    const int M = n_tree * a.group;
    const int rows = kRowsPerBlock / a.splits;
    if (rb * rows >= M) return;
    const int tid = threadIdx.x;

    const int64_t L = a.prefix_off[b + 1] - a.prefix_off[b];
    const T *kp = static_cast<const T *>(a.k_prefix) + (a.prefix_off[b] * a.Hkv + (int64_t)g * L) * D;
    const T *vp = static_cast<const T *>(a.v_prefix) + (a.prefix_off[b] * a.Hkv + (int64_t)g * L) * D;
    const T *kn = static_cast<const T *>(a.k_new) + ((int64_t)n_lo * a.Hkv + g) * D;
    const T *vn = static_cast<const T *>(a.v_new) + ((int64_t)n_lo * a.Hkv + g) * D;

    // a tile never straddles the prefix / tree boundary
    const int64_t p_tiles = (L + kTok - 1) / kTok, n_tiles = p_tiles + (n_tree + kTok - 1) / kTok;
    uint4 kr[NV], vr[NV];
    auto tile_tokens = [&](int64_t t) -> int {
        return (int)(t < p_tiles ? min((int64_t)kTok, L - t * kTok) : min((int64_t)kTok, n_tree - (t - p_tiles) * kTok));
    };
    auto load = [&](int64_t t) {
        const int cnt = tile_tokens(t);
        const bool in_tree = t >= p_tiles;
        const int64_t stride = in_tree ? (int64_t)a.Hkv * D : D;
        const int64_t first = in_tree ? (t - p_tiles) * kTok * stride : t * kTok * stride;
        const T *kt = (in_tree ? kn : kp) + first, *vt = (in_tree ? vn : vp) + first;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int at = i * kThreads + tid, row = at / VPR, c = (at - row * VPR) * PV;
            kr[i] = row < cnt ? *reinterpret_cast<const uint4 *>(kt + row * stride + c) : make_uint4(0, 0, 0, 0);
            vr[i] = row < cnt ? *reinterpret_cast<const uint4 *>(vt + row * stride + c) : make_uint4(0, 0, 0, 0);
        }
    };
    auto store = [&] {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int at = i * kThreads + tid, row = at / VPR, c = (at - row * VPR) * PV;
            float k[PV], v[PV];
            Elem<T>::widen(kr[i], k);
            Elem<T>::widen(vr[i], v);
#pragma unroll
            for (int e = 0; e < PV; e += 4) {
                *reinterpret_cast<float4 *>(ks + row * RS + c + e) = make_float4(k[e], k[e + 1], k[e + 2], k[e + 3]);
                *reinterpret_cast<float4 *>(vs + row * RS + c + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
            }
        }
    };
    load(0);

    const int pair = tid >> 1, half = tid & 1;
    const int split = pair % a.splits, row = rb * rows + pair / a.splits;   // query row inside the unit
    const bool active = row < M;
    const int node = active ? row / a.group : 0;          // tree-local node
    const int hq = g * a.group + (active ? row % a.group : 0);
    const T *Q = static_cast<const T *>(a.q) + ((int64_t)(n_lo + node) * a.Hq + hq) * D;
    // element e of the thread's H: 4 (2 (e / 4) + half) + e % 4 of the row
    float qv[H], o[H];
#pragma unroll
    for (int e = 0; e < H; ++e) {
        qv[e] = active ? Elem<T>::to_float(Q[4 * (2 * (e / 4) + half) + e % 4]) * a.scale_log2 : 0.f;
        o[e] = 0.f;
    }
    float mrun = -INFINITY, lrun = 0.f;
    if (tid < n_tree) par_s[tid] = a.parent[n_lo + tid];
    __syncthreads();
    // ancestor-or-self bitmasks of the tree
    if (tid < n_tree) {
        unsigned long long m = 0ull;
        for (int i = tid; ;) {
            m |= 1ull << i;
            const int par = par_s[i];
            if (par < n_lo || par >= n_lo + i) {
                if (i == tid && (par != -1 || i != 0)) report(a.status, DSBD_DEV_BAD_FOREST);
                break;
            }
            i = par - n_lo;
        }
        anc[tid] = m;
    }
    __syncthreads();
    const unsigned long long my_anc = anc[node];

    for (int64_t t = 0; t < n_tiles; ++t) {
        store();
        __syncthreads();
        if (t + 1 < n_tiles) load(t + 1);
        const int cnt = tile_tokens(t);
        const unsigned visible = t < p_tiles ? kFull : (unsigned)(my_anc >> ((t - p_tiles) * kTok));
#pragma unroll 1
        for (int j0 = split; j0 < cnt; j0 += kChunk * a.splits) {
            float s[kChunk];
            float tmax = -INFINITY;
            bool any = false;                                    // some token counts (a NaN does, and is no maximum)
#pragma unroll
            for (int i = 0; i < kChunk; ++i) {
                const int j = j0 + i * a.splits;
                const float4 *row4 = reinterpret_cast<const float4 *>(ks + j * RS) + half;
                float acc = 0.f;
#pragma unroll
                for (int c = 0; c < H / 4; ++c) {
                    const float4 kv = row4[2 * c];
                    acc = fmaf(qv[4 * c], kv.x, acc);
                    acc = fmaf(qv[4 * c + 1], kv.y, acc);
                    acc = fmaf(qv[4 * c + 2], kv.z, acc);
                    acc = fmaf(qv[4 * c + 3], kv.w, acc);
                }
                s[i] = acc;
            }
            // (the pairs of a warp differ in their number of chunks: a pair's two threads do not)
#pragma unroll
            for (int i = 0; i < kChunk; ++i) {
                const int j = j0 + i * a.splits;
                s[i] += __shfl_xor_sync(3u << (tid & 30), s[i], 1);
                if (j >= cnt || !(visible >> j & 1u)) s[i] = -INFINITY;
                tmax = fmaxf(tmax, s[i]);
                any = any || s[i] != -INFINITY;
            }
            if (any) {
                const float mnew = fmaxf(mrun, tmax);
                const float corr = exp2f(mrun - mnew);      // 0 when mrun == -inf
                lrun *= corr;
#pragma unroll
                for (int e = 0; e < H; ++e) o[e] *= corr;
#pragma unroll
                for (int i = 0; i < kChunk; ++i) {
                    const int j = j0 + i * a.splits;
                    const float p = exp2f(s[i] - mnew);      // 0 for masked entries
                    lrun += p;
                    const float4 *row4 = reinterpret_cast<const float4 *>(vs + j * RS) + half;
#pragma unroll
                    for (int c = 0; c < H / 4; ++c) {
                        const float4 vv = row4[2 * c];
                        o[4 * c] = fmaf(p, vv.x, o[4 * c]);
                        o[4 * c + 1] = fmaf(p, vv.y, o[4 * c + 1]);
                        o[4 * c + 2] = fmaf(p, vv.z, o[4 * c + 2]);
                        o[4 * c + 3] = fmaf(p, vv.w, o[4 * c + 3]);
                    }
                }
                mrun = mnew;
            }
        }
        __syncthreads();
    }
    // the pairs of a row
    for (int off = 2; off < 2 * a.splits; off *= 2) {
        const float m2 = __shfl_xor_sync(kFull, mrun, off), l2 = __shfl_xor_sync(kFull, lrun, off);
        const float mnew = fmaxf(mrun, m2);
        const float c1 = mrun > -INFINITY ? exp2f(mrun - mnew) : 0.f, c2 = m2 > -INFINITY ? exp2f(m2 - mnew) : 0.f;
        lrun = lrun * c1 + l2 * c2;
#pragma unroll
        for (int e = 0; e < H; ++e) o[e] = o[e] * c1 + __shfl_xor_sync(kFull, o[e], off) * c2;
        mrun = mnew;
    }
    if (active && split == 0) {
        T *O = static_cast<T *>(a.out) + ((int64_t)(n_lo + node) * a.Hq + hq) * D;
        const float inv = 1.f / lrun;
#pragma unroll
        for (int e = 0; e < H; ++e) O[4 * (2 * (e / 4) + half) + e % 4] = Elem<T>::from_float(o[e] * inv);
    }
}

template <class T, int D>
int launch_simt(const AttnArgs &a, int units, cudaStream_t stream) {
    const size_t smem = sizeof(float) * 2 * kTok * (D + 8);
    k_forest_attn_simt<T, D><<<units, kThreads, smem, stream>>>(a);
    return cudaGetLastError() == cudaSuccess ? DSBD_OK : DSBD_ERR_CUDA;
}

int check(const dsbd_forest_t *f, const dsbd_attn_desc_t *d) {
    if (!f || !d || f->B <= 0 || f->N <= 0 || !f->beam_node_off || !f->parent) return DSBD_ERR_INVALID_ARG;
    if (d->Hq <= 0 || d->Hkv <= 0 || d->Hq % d->Hkv) return DSBD_ERR_INVALID_ARG;
    if (d->d != 64 && d->d != 128) return DSBD_ERR_UNSUPPORTED;
    if (d->dtype != DSBD_DTYPE_BF16 && d->dtype != DSBD_DTYPE_F32) return DSBD_ERR_UNSUPPORTED;
    if (f->max_tree_nodes <= 0) return DSBD_ERR_INVALID_ARG;
    if (f->max_tree_nodes > DSBD_MAX_TREE_NODES_TC) return DSBD_ERR_UNSUPPORTED;
    return DSBD_OK;
}

}  // namespace

extern "C" size_t dsbd_forest_attention_workspace(const dsbd_forest_t *f, const dsbd_attn_desc_t *d) {
    if (check(f, d) != DSBD_OK) return 0;
    if (attention_tr_supported(f, d)) return attention_tr_workspace(f, d);
    return attention_tc_supported(f, d) ? attention_tc_workspace(f, d) : 256;
}

extern "C" int dsbd_forest_attention_launches(const dsbd_forest_t *f, const dsbd_attn_desc_t *d) {
    if (check(f, d) != DSBD_OK) return 0;
    if (attention_tr_supported(f, d)) return attention_tr_launches(f, d);
    return attention_tc_supported(f, d) ? attention_tc_launches(f, d) : 1;
}

extern "C" int dsbd_forest_attention(const dsbd_forest_t *f, const dsbd_attn_desc_t *d, const void *q,
                                     const void *k_new, const void *v_new, const void *k_prefix,
                                     const void *v_prefix, const int64_t *prefix_off, void *out,
                                     void *workspace, size_t workspace_bytes, int32_t *status,
                                     dsbd_stream_t stream_) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    const int rc = check(f, d);
    if (rc) return rc;
    if (!q || !k_new || !v_new || !prefix_off || !out || !status) return DSBD_ERR_INVALID_ARG;
    if (d->total_prefix > 0 && (!k_prefix || !v_prefix)) return DSBD_ERR_INVALID_ARG;
    if (workspace_bytes < dsbd_forest_attention_workspace(f, d) || !workspace) return DSBD_ERR_WORKSPACE_TOO_SMALL;
    const uintptr_t bits = reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(k_new) |
                           reinterpret_cast<uintptr_t>(v_new) | reinterpret_cast<uintptr_t>(k_prefix) |
                           reinterpret_cast<uintptr_t>(v_prefix) | reinterpret_cast<uintptr_t>(out);
    if (bits & 15) return DSBD_ERR_UNSUPPORTED;

    if (attention_tr_supported(f, d))
        return launch_attention_tr(f, d, q, k_new, v_new, k_prefix, v_prefix, prefix_off, out, workspace,
                                   workspace_bytes, status, stream);
    if (attention_tc_supported(f, d))
        return launch_attention_tc(f, d, q, k_new, v_new, k_prefix, v_prefix, prefix_off, out, workspace,
                                   workspace_bytes, status, stream);

    if (f->max_tree_nodes > DSBD_MAX_TREE_NODES) return DSBD_ERR_UNSUPPORTED;      // CUDA-core kernel: 64-bit masks
    AttnArgs a = {};
    a.B = f->B; a.N = f->N; a.Hq = d->Hq; a.Hkv = d->Hkv; a.group = d->Hq / d->Hkv;
    a.scale_log2 = d->scale * 1.4426950408889634f;
    a.beam_node_off = f->beam_node_off; a.parent = f->parent; a.prefix_off = prefix_off;
    a.q = q; a.k_new = k_new; a.v_new = v_new; a.k_prefix = k_prefix; a.v_prefix = v_prefix;
    a.out = out; a.status = status;
    const int max_rows = f->max_tree_nodes * a.group;
    a.splits = max_rows <= kRowsPerBlock / 4 ? 4 : max_rows <= kRowsPerBlock / 2 ? 2 : 1;
    a.row_blocks = (max_rows * a.splits + kRowsPerBlock - 1) / kRowsPerBlock;
    const int units = f->B * d->Hkv * a.row_blocks;
    if (d->dtype == DSBD_DTYPE_F32)
        return d->d == 64 ? launch_simt<float, 64>(a, units, stream) : launch_simt<float, 128>(a, units, stream);
    return d->d == 64 ? launch_simt<__nv_bfloat16, 64>(a, units, stream)
                      : launch_simt<__nv_bfloat16, 128>(a, units, stream);
}

extern "C" size_t dsbd_forest_attention_paged_workspace(const dsbd_forest_t *f, const dsbd_attn_desc_t *d,
                                                        const dsbd_kv_pages_t *pages) {
    if (check(f, d) != DSBD_OK || !pages || pages->n_pages <= 0 || pages->n_layers < 0) return 0;
    if (!attention_tc_supported(f, d, pages->n_pages) || !attention_tc_layers_ok(f, d, pages)) return 0;
    return attention_tr_supported(f, d, pages->n_pages) ? attention_tr_workspace(f, d, pages->n_layers)
                                                        : attention_tc_workspace(f, d, pages->n_layers);
}

extern "C" int dsbd_forest_attention_paged(const dsbd_forest_t *f, const dsbd_attn_desc_t *d, const void *q,
                                           const void *k_new, const void *v_new, const void *k_pool,
                                           const void *v_pool, const dsbd_kv_pages_t *pages,
                                           const int64_t *prefix_off, void *out, void *workspace,
                                           size_t workspace_bytes, int32_t *status, dsbd_stream_t stream_) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    const int rc = check(f, d);
    if (rc) return rc;
    if (!q || !k_new || !v_new || !k_pool || !v_pool || !pages || !pages->page_table || !pages->page_off ||
        pages->n_pages <= 0 || !prefix_off || !out || !status)
        return DSBD_ERR_INVALID_ARG;
    if (!attention_tc_supported(f, d, pages->n_pages)) return DSBD_ERR_UNSUPPORTED;
    if (pages->n_layers < 0 || !attention_tc_layers_ok(f, d, pages)) return DSBD_ERR_INVALID_ARG;
    const bool tr = attention_tr_supported(f, d, pages->n_pages);
    if (!workspace || workspace_bytes < (tr ? attention_tr_workspace(f, d, pages->n_layers)
                                            : attention_tc_workspace(f, d, pages->n_layers)))
        return DSBD_ERR_WORKSPACE_TOO_SMALL;
    const uintptr_t bits = reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(k_new) |
                           reinterpret_cast<uintptr_t>(v_new) | reinterpret_cast<uintptr_t>(k_pool) |
                           reinterpret_cast<uintptr_t>(v_pool) | reinterpret_cast<uintptr_t>(out);
    if (bits & 15) return DSBD_ERR_UNSUPPORTED;
    return (tr ? launch_attention_tr : launch_attention_tc)(f, d, q, k_new, v_new, k_pool, v_pool, prefix_off, out,
                                                            workspace, workspace_bytes, status, stream, pages);
}
