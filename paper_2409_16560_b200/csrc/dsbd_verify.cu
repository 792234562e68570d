// dsbd_verify_step / dsbd_select_width: the verification step of speculative beam decoding
// (Algorithm 1 with the dynamic layer width) for sm_100a.
//
// Kernels
//   k_tile_stats   one dense streaming pass over every logits row of both models: per
//                  1024-token tile the row maximum and sum of exponentials (warp-autonomous,
//                  128-bit loads, warp-shuffle reductions).  HBM-bound; this is the pass the
//                  algorithmic bytes 8*N*V belong to.
//   k_row_finish   per row: log-sum-exp from the tile statistics (dsbd_node_stats and
//                  dsbd_select_width; dsbd_verify_step does this inside k_verify).
//   k_verify       one thread-block cluster per request.  Prologue: log-sum-exp of the request's
//                  rows, log-prob of every draft token, cumulative beam scores.  Then layer by
//                  layer: live set and beam weights; ONE pass over the live rows that builds a
//                  fixed-point histogram of the cells' ratios p_beam/q_beam, from which all the
//                  residual masses c_{j+1} = F(s_j) of the layer follow without touching the
//                  rows again; the acceptance-count recursion; the accept loop; the
//                  inverse-CDF completion draws.  A layer whose width does not depend on the residual
//                  masses tests its drafts at once and, unless many are left behind the first
//                  rejection, makes a plain pass for each rejection in place of the histogram.
//
// The residual chain uses the closed form of the paper's recursion p_{k+1} = norm(max(p_k -
// q_beam, 0)):  with F(s) = sum max(p_beam - s q_beam, 0), c_1 = 1, s_0 = 0, s_j = s_{j-1} + c_j
// and c_{j+1} = F(s_j) one has p_j = max(p_beam - s_{j-1} q_beam, 0) / c_j, hence
// alpha_j = 1 - c_{j+1}/c_j and the accept ratio of a draft x at run position j is
// max(rho(x) - s_{j-1}, 0) / c_j with rho = p_beam(x)/q_beam(x).  F(s) = P(rho > s) - s Q(rho > s)
// only needs the p and q mass above a ratio threshold, which is what the histogram holds; the
// one bin that s falls into is bracketed from its two sums and its edges, and when half the
// bracket plus the bound on the histogram's fixed-point error exceeds 2.5e-7 that F(s_j) is
// recomputed exactly by a pass over the rows.
//
// Building with -DDSBD_PHASE_TIMING makes k_verify record %globaltimer stamps of its phases at
// the end of the workspace (a tuning aid; off in normal builds).
#include <cooperative_groups.h>
#include <math.h>

#include "dsbd_common.cuh"

namespace cg = cooperative_groups;
using namespace dsbd;

namespace {

constexpr int kTile = 1024;          // tokens per tile: 32 lanes x 8 x float4
constexpr int kThreads = 256;        // streaming kernels
constexpr int kWarps = kThreads / 32;
constexpr int kVThreads = 512;       // the per-request kernel: two CTAs of 16 warps per SM
constexpr int kVWarps = kVThreads / 32;
constexpr int kMaxLive = DSBD_MAX_LIVE;
constexpr float kLog2e = 1.4426950408889634f;
constexpr double kLn2 = 0.6931471805599453;

// A load before griddepcontrol.wait: from L2.
template <class V>
__device__ __forceinline__ V ld_early(const V *p) { return __ldcg(p); }

struct TileStat { float mx; float sum; };   // max of the raw logits, sum exp((z-mx)/tau)

// kWritten: the row may have been written while the kernel was resident already (it has waited since).  Its single words by
// predicated loads: as plain conditional ones they took 6 registers more, and five draft layers of 16 x 8 rows 180 us instead of 173.
template <bool kWritten>
__device__ __forceinline__ void load_tile(const float *row, int e0, int V, bool aligned, int lane, float4 (&v)[8]) {
    auto four = [&](int e) {
        const float4 *p = reinterpret_cast<const float4 *>(row + e);
        return kWritten ? ld_stream(p) : ldg_stream(p);
    };
    auto one = [&](int e) {
        if (!kWritten) return e < V ? __ldg(row + e) : -INFINITY;
        float x;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "setp.lt.s32 p, %2, %3;\n\t"
                     "mov.f32 %0, 0fFF800000;\n\t"
                     "@p ld.global.f32 %0, [%1];\n\t}"
                     : "=&f"(x) : "l"(row + e), "r"(e), "r"(V));
        return x;
    };
    if (aligned && e0 + kTile <= V) {
#pragma unroll
        for (int it = 0; it < 8; ++it) v[it] = four(e0 + it * 128 + lane * 4);
        return;
    }
#pragma unroll
    for (int it = 0; it < 8; ++it) {
        const int e = e0 + it * 128 + lane * 4;
        if (aligned && e + 3 < V) v[it] = four(e);
        else v[it] = make_float4(one(e), one(e + 1), one(e + 2), one(e + 3));
    }
}

// Half a tile of a row that is not aligned, or ends in it (whole aligned ones are loaded where they are used).
__device__ __forceinline__ void load_half_tile(const float *__restrict__ row, int e0, int V, int lane, float4 (&v)[4]) {
    const float ninf = -INFINITY;
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int e = e0 + it * 128 + lane * 4;
        v[it].x = e < V ? __ldg(row + e) : ninf;
        v[it].y = e + 1 < V ? __ldg(row + e + 1) : ninf;
        v[it].z = e + 2 < V ? __ldg(row + e + 2) : ninf;
        v[it].w = e + 3 < V ? __ldg(row + e + 3) : ninf;
    }
}

// ---------------------------------------------------------------------------------------
// Dense pass: tile statistics of every (model, row).  Item = (model, row, tile), tile fastest,
// one warp per item.  rows == nullptr: all n_rows rows; else the listed rows (n_rows read
// from *n_rows_dev when it is given, never more than the n_rows the launch was sized for; a
// listed row outside [0, N) is skipped -- the kernel that consumes the list reports it).
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads)
k_tile_stats(const float *zp, const float *zq, int64_t stride, int V, int T, int N, int n_rows, const int32_t *rows,
             const int32_t *n_rows_dev, float k2, TileStat *__restrict__ stats, int one_model = 0) {
    // Launched with programmatic stream serialization: its blocks are in place when the work ahead in the stream ends, and
    // read nothing before (five draft layers of 16 x 8 rows of 128256: 183 -> 175 us); what they read then may have been
    // written while they were in place, so not through .nc.  In this order: the kernel behind it, which may be set up while
    // the last blocks run, must not start (and read what the caller gave) before all earlier work is done.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    if (n_rows_dev) n_rows = min(max(*n_rows_dev, 0), n_rows);
    const int64_t total = (int64_t)(one_model ? 1 : 2) * n_rows * T;
    for (int64_t item = warp; item < total; item += nwarps) {
        const int t = (int)(item % T);
        const int64_t rm = item / T;
        const int model = (int)(rm / n_rows);
        const int ri = (int)(rm % n_rows);
        const int row = rows ? rows[ri] : ri;
        if (row < 0 || row >= N) continue;
        const float *z = (model ? zq : zp) + (int64_t)row * stride;
        const bool aligned = (reinterpret_cast<uintptr_t>(z) & 15) == 0;
        float4 v[8];
        load_tile<true>(z, t * kTile, V, aligned, lane, v);
        float mx = -INFINITY;
#pragma unroll
        for (int it = 0; it < 8; ++it)
            mx = fmaxf(mx, fmaxf(fmaxf(v[it].x, v[it].y), fmaxf(v[it].z, v[it].w)));
        mx = warp_max(mx);
        float sum = 0.f;
        if (fabsf(mx) * k2 > 65536.f) {
            // a tile masked with a huge value: the rounding of its product with k2 is no longer small against one, and
            // the product may overflow (2^x of either would be infinite, and the row's sum with it).  -inf: no mass
            if (mx > -INFINITY)
#pragma unroll
                for (int it = 0; it < 8; ++it)
                    sum += exp2f((v[it].x - mx) * k2) + exp2f((v[it].y - mx) * k2) +
                           exp2f((v[it].z - mx) * k2) + exp2f((v[it].w - mx) * k2);
        } else {
            const float b = -mx * k2;
#pragma unroll
            for (int it = 0; it < 8; ++it) {
                sum += exp2f(fmaf(v[it].x, k2, b)) + exp2f(fmaf(v[it].y, k2, b)) +
                       exp2f(fmaf(v[it].z, k2, b)) + exp2f(fmaf(v[it].w, k2, b));
            }
        }
        sum = warp_sum(sum);
        if (lane == 0) {
            TileStat s; s.mx = mx; s.sum = sum;
            stats[((int64_t)model * N + row) * T + t] = s;
        }
    }
}

// log-sum-exp of a tempered row from its tile statistics, by one warp (same value on every lane;
// the order of the sums depends on T only).
__device__ __forceinline__ double row_lse(const TileStat *s, int T, double inv_tau, int lane) {
    double mx = -INFINITY;
    for (int t = lane; t < T; t += 32) mx = fmax(mx, (double)s[t].mx);
    mx = warp_max(mx);
    double acc = 0.0;
    if (mx > -INFINITY)
        for (int t = lane; t < T; t += 32)
            if (s[t].sum > 0.f) acc += (double)s[t].sum * exp(((double)s[t].mx - mx) * inv_tau);
    acc = warp_sum(acc);
    return (mx > -INFINITY) ? mx * inv_tau + log(acc) : -INFINITY;
}

// log-sum-exp of the tempered row from its tile statistics; one warp per (model, row).
__global__ void k_row_finish(const TileStat *__restrict__ stats, int T, int N, int n_rows,
                             const int32_t *__restrict__ rows, const int32_t *__restrict__ n_rows_dev,
                             double inv_tau, double *__restrict__ lse /*[2][N]*/,
                             float *__restrict__ lse_p_out, float *__restrict__ lse_q_out) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (n_rows_dev) n_rows = min(max(*n_rows_dev, 0), n_rows);
    if (warp >= (int64_t)2 * n_rows) return;
    const int model = (int)(warp / n_rows);
    const int ri = (int)(warp % n_rows);
    const int row = rows ? rows[ri] : ri;
    if (row < 0 || row >= N) return;
    const double v = row_lse(stats + ((int64_t)model * N + row) * T, T, inv_tau, lane);
    if (lane == 0) {
        lse[(int64_t)model * N + row] = v;
        if (model == 0 && lse_p_out) lse_p_out[row] = (float)v;
        if (model == 1 && lse_q_out) lse_q_out[row] = (float)v;
    }
}

// ---------------------------------------------------------------------------------------
// The per-request kernel.
// ---------------------------------------------------------------------------------------
struct VerifyArgs {
    // forest
    int R, N, gamma;
    const int32_t *req_beam_off, *beam_node_off, *parent, *token, *draft_rank;
    // parameters
    int V, T;
    float k2;                 // log2(e)/tau
    double inv_tau, thresh;
    int W_min, W_max, W_nom;
    const int32_t *W_min_r, *W_max_r, *W_nom_r;
    uint64_t seed, step;
    int top_k;                // 0: unwarped joints
    double top_p;             // outside (0,1): off
    // inputs
    const float *zp, *zq;
    int64_t stride;
    // workspace
    const TileStat *stats;    // [2][N][T]
    const double *lse;        // [2][N]
    const double *score;      // [2][N]
    const int32_t *depth;     // [N]
    double *tile_sums;        // [R][2][max_m+1][max_live*T]: per bank the histogram pass's sums (half tiles may take
                              // two slots), then those of the exact pass at j >= 2 in slot j
    unsigned long long *dbg;  // phase time stamps (DSBD_PHASE_TIMING builds only)
    // verify mode computes the row and tree statistics of its own request first
    double *lse_w, *score_w;
    int32_t *depth_w;
    const float *root_logp, *root_logq;
    int max_m, max_live;
    int check_widths;            // verification / width selection: per-request widths are validated
    // outputs
    dsbd_verify_out_t out;
    int32_t *status;
    // select-width mode
    int select_mode;
    const float *sel_logp, *sel_logq;
    const int32_t *live_off, *live_nodes, *m_in;
    int sel_rows;             // list entries the dense pass was sized for
    int32_t *width_out;
    float *alpha_out, *tail_out;
    int out_stride;
};

struct Shared {
    int nA, m, W, count, done, chain_len, err;
    int A[kMaxLive];
    int S[kMaxLive];
    int S_parent_idx[kMaxLive];
    int acc[kMaxLive];
    // log2 of (beam weight / sum of the row's exponentials), split so that the cell masses do not
    // inherit the rounding of one large float: bp/bq hold the nearest integer (exact in fp32), cp/cq
    // the factor 2^(remainder) in [2^-0.5, 2^0.5], rp/rq the remainders
    float bp[kMaxLive], bq[kMaxLive], cp[kMaxLive], cq[kMaxLive];
    double rp[kMaxLive], rq[kMaxLive];
    double lwp[kMaxLive], lwq[kMaxLive];    // natural log of the beam weights
    double wp[kMaxLive];
    double s_arr[kMaxLive + 2];             // s_0 .. s_m
    double c_arr[kMaxLive + 2];             // c_1 .. c_{m+1} (index j)
    double alpha[kMaxLive + 1];
    double first[kMaxLive + 1];             // alpha_i prod_{j<i}(1-alpha_j)
    double col_a[kMaxLive + 1], col_b[kMaxLive + 1];
    double tail[kMaxLive + 2];
    int bank, halves, need_exact, res_j, run_j, chain_pos;
    int on_demand, next_i;                  // a layer of known width: its passes are made when the accept loop asks
    // sums of an exact pass, in units of 2^-60, 2^-120 (what the first leaves) and 2^-44 (q): of this CTA's warps; of every
    // CTA, two passes in turn
    long long warp_part[3][kVWarps], part[2][3][16];
    int n_out, n_fill;                      // output beams so far; p_beam fills left to the whole CTA
    int n_layers, n_tests, n_exact, n_respass;
    int n_near, n_rows;                     // accept tests inside the 1e-5 tie band; live rows of layers that looked into them
    unsigned long long wtot_p[kVWarps], wtot_q[kVWarps];
    unsigned long long slice_p[16], slice_q[16];   // mass of the bins of every CTA's slice
    unsigned long long above_p[16], above_q[16];   // mass of the bins above every CTA's slice
    unsigned long long w_tot[2][10];        // per bank, sums of one histogram pass: see histogram_pass / hist_fold_over
    int n_wrapped;                          // layers where a w word of the histogram wrapped
    double rho[kMaxLive], uu[kMaxLive];     // per live draft: p_beam/q_beam and its uniform
};

// mass of one cell of the residual max(p_beam - s q_beam, 0); s == 0 gives p_beam
struct RowOff { float bp, bq, cp, cq, dc; };
__device__ __forceinline__ float cell_mass(float zp, float zq, float k2, const RowOff &o, float s, float *q) {
    const float a = exp2f(fmaf(zp, k2, o.bp)) * o.cp;
    const float b = exp2f(fmaf(zq, k2, o.bq)) * o.cq;
    *q = b;
    return fmaxf(fmaf(-s, b, a), 0.f);
}
// Splits b = log2(weight) - lse*log2(e) (double) into its nearest integer and the factor 2^(rest).
__device__ __forceinline__ void split_offset(double b, float *bi, float *c, double *rest) {
    if (b == b && fabs(b) < 1e30) {
        const double r = rint(b);
        *bi = (float)r; *c = (float)exp2(b - r); *rest = b - r;
    } else {
        *bi = (float)b; *c = 1.f; *rest = 0.0;
    }
}

__device__ __forceinline__ RowOff row_off(const Shared &sh, int i) {
    return RowOff{sh.bp[i], sh.bq[i], sh.cp[i], sh.cq[i], (float)(sh.rp[i] - sh.rq[i])};
}

// Inverse-CDF search over tile masses (canonical order).  mass(i) must be the same on every
// lane.  Returns the tile holding the first cell whose running sum reaches the target, and the
// target minus the mass before that tile; if rounding leaves the target beyond the total, the last
// tile with mass.  -1 if there is no mass at all.  The target is u * total when of_total, else u.
// Every round cuts the range by 32: a lane sums its share (its loads are independent, one memory
// latency a round instead of one per 32 tiles), the lanes' sums are scanned, one lane is chosen.
template <class F>
__device__ int locate_tile(F mass, int n, double u, bool of_total, int lane, double *rest) {
    int lo = 0, len = n;
    double target = u;
    while (true) {
        const int per = (len + 31) >> 5, i0 = lo + lane * per, i1 = min(i0 + per, lo + len);
        double v = 0.0;
#pragma unroll 4
        for (int i = i0; i < i1; ++i) v += mass(i);
        const double incl = warp_scan(v, lane);
        if (of_total) { target = u * __shfl_sync(kFull, incl, 31); of_total = false; }
        const unsigned pos = __ballot_sync(kFull, v > 0.0);
        if (!pos) return -1;
        const unsigned hits = __ballot_sync(kFull, v > 0.0 && incl >= target);
        const int l = hits ? __ffs(hits) - 1 : 31 - __clz(pos);
        target -= __shfl_sync(kFull, incl - v, l);
        lo += l * per;
        len = min(per, len - l * per);
        if (per == 1) { *rest = target; return lo; }
    }
}

// Inverse-CDF search inside one tile of row `row` (and its q row when s > 0): the first
// token whose running mass reaches `target`, else the last token with mass.  -1: no mass.
// A lane sums 32 consecutive tokens (two batches of independent loads), then the lanes take the 32 tokens
// of the lane that was hit.
__device__ __noinline__ int locate_token(const float *__restrict__ rp, const float *__restrict__ rq, int V, float k2,
                                         int t, const RowOff ro, float s, double target, int lane) {
    const bool al = ((reinterpret_cast<uintptr_t>(rp) | reinterpret_cast<uintptr_t>(rq)) & 15) == 0;
    const int e0 = t * kTile + lane * 32;
    float q;
    auto mass = [&](float zp, float zq) { return s > 0.f ? cell_mass(zp, zq, k2, ro, s, &q) : exp2f(fmaf(zp, k2, ro.bp)) * ro.cp; };
    double v = 0.0;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        float4 zp[4], zq[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = e0 + half * 16 + i * 4;
            zq[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (al && e + 3 < V) {
                zp[i] = __ldg(reinterpret_cast<const float4 *>(rp + e));
                if (s > 0.f) zq[i] = __ldg(reinterpret_cast<const float4 *>(rq + e));
            } else {
                const float ninf = -INFINITY;
                zp[i].x = e < V ? __ldg(rp + e) : ninf;         zp[i].y = e + 1 < V ? __ldg(rp + e + 1) : ninf;
                zp[i].z = e + 2 < V ? __ldg(rp + e + 2) : ninf; zp[i].w = e + 3 < V ? __ldg(rp + e + 3) : ninf;
                if (s > 0.f) {
                    zq[i].x = e < V ? __ldg(rq + e) : ninf;         zq[i].y = e + 1 < V ? __ldg(rq + e + 1) : ninf;
                    zq[i].z = e + 2 < V ? __ldg(rq + e + 2) : ninf; zq[i].w = e + 3 < V ? __ldg(rq + e + 3) : ninf;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v += (double)mass(zp[i].x, zq[i].x); v += (double)mass(zp[i].y, zq[i].y);
            v += (double)mass(zp[i].z, zq[i].z); v += (double)mass(zp[i].w, zq[i].w);
        }
    }
    int first = 0;                                               // the hit lane's first token
    for (int level = 0; ; ++level) {
        const double incl = warp_scan(v, lane);
        const unsigned pos = __ballot_sync(kFull, v > 0.0);
        if (!pos) return -1;
        const unsigned hits = __ballot_sync(kFull, v > 0.0 && incl >= target);
        const int l = hits ? __ffs(hits) - 1 : 31 - __clz(pos);
        if (level) return first + l;
        target -= __shfl_sync(kFull, incl - v, l);
        first = t * kTile + l * 32;
        const int e = first + lane;
        v = e < V ? (double)mass(__ldg(rp + e), s > 0.f ? __ldg(rq + e) : 0.f) : 0.0;
    }
}

// Per-node data of the request that every layer's set-up reads, kept in shared memory when the
// request is small enough (otherwise the set-up reads the global arrays).
constexpr int kCacheNodes = 256;
struct NodeCache {
    double score_p[kCacheNodes], score_q[kCacheNodes], lse_p[kCacheNodes], lse_q[kCacheNodes];
    int16_t parent[kCacheNodes];          // local index of the parent, -1 for a root, -2: none inside the request
    uint8_t depth[kCacheNodes];
    uint8_t tree[kCacheNodes];            // tree of the node, inside the request
    int root[kMaxLive];                   // first node of every tree
};

// Writes output beam number `index` of request r (the caller has checked the slot range).  nc: the
// request's node cache or nullptr; n_lo: first node of the request.
__device__ void emit_at(const VerifyArgs &a, int r, int index, int parent, int node, int tok, int source,
                        const NodeCache *nc, int n_lo) {
    const int s = a.out.out_off[r] + index;
    const float zp = a.zp[(int64_t)parent * a.stride + tok], zq = a.zq[(int64_t)parent * a.stride + tok];
    const int lo = a.req_beam_off[r];
    int beam = lo;
    double lse_p, lse_q, score_p, score_q;
    if (nc) {
        const int i = parent - n_lo;
        beam += nc->tree[i];
        lse_p = nc->lse_p[i]; lse_q = nc->lse_q[i]; score_p = nc->score_p[i]; score_q = nc->score_q[i];
    } else {
        // the tree of a node: walk to the root, then find which beam starts there
        int root = parent;
        while (a.parent[root] >= 0) root = a.parent[root];
        const int hi = a.req_beam_off[r + 1];
        for (int b = lo; b < hi; ++b) if (a.beam_node_off[b] == root) beam = b;
        lse_p = a.lse[parent]; lse_q = a.lse[a.N + parent]; score_p = a.score[parent]; score_q = a.score[a.N + parent];
    }
    a.out.out_parent[s] = parent;
    a.out.out_node[s] = node;
    a.out.out_root_beam[s] = beam;
    a.out.out_token[s] = tok;
    a.out.out_source[s] = source;
    a.out.out_logp[s] = (float)(score_p + ((double)zp * a.inv_tau - lse_p));
    a.out.out_logq[s] = (float)(score_q + ((double)zq * a.inv_tau - lse_q));
}


// Natural log of the softmax of n scores, by one warp (lanes over the scores).
__device__ __forceinline__ void log_softmax_warp(const double *s, int n, int lane, double *out) {
    double mx = -INFINITY;
    for (int i = lane; i < n; i += 32) mx = fmax(mx, s[i]);
    mx = warp_max(mx);
    double t = 0.0;
    for (int i = lane; i < n; i += 32) t += exp(s[i] - mx);
    t = warp_sum(t);
    const double lt = log(t);
    for (int i = lane; i < n; i += 32) out[i] = (s[i] - mx) - lt;
    __syncwarp();
}

// The weights of one model (0: p, 1: q) over the live set: softmax of the cumulative scores over A (Eq. 1 factorised),
// by one warp; the two models' warps work side by side.
// nc: the request's node cache or nullptr; n_lo: first node of the request.
__device__ void live_weights(const VerifyArgs &a, Shared &sh, int model, const double *scores, int lane,
                             const NodeCache *nc, int n_lo) {
    double *lw = model ? sh.lwq : sh.lwp;
    log_softmax_warp(scores, sh.nA, lane, lw);
    const double *lse = nc ? (model ? nc->lse_q : nc->lse_p) - n_lo : a.lse + (int64_t)model * a.N;
    for (int i = lane; i < sh.nA; i += 32) {
        if (!model) sh.wp[i] = exp(lw[i]);
        split_offset((lw[i] - lse[sh.A[i]]) * (1.0 / kLn2), model ? &sh.bq[i] : &sh.bp[i],
                     model ? &sh.cq[i] : &sh.cp[i], model ? &sh.rq[i] : &sh.rp[i]);
    }
    __syncwarp();
}

// Acceptance-count recursion by one warp (lanes over n): tail[K] = P(at least K accepts),
// returns W~ = max{K : tail[K] >= thresh}.
// k_stop >= 0: stop once W = min(W_max = k_stop, max(W_min, W~)) is decided; -1: the whole tail
__device__ int width_rule(Shared &sh, int m, double thresh, int lane, int k_stop) {
    if (lane == 0) {
        double none = 1.0;
        for (int i = 1; i <= m; ++i) {
            sh.first[i] = sh.alpha[i] * none;
            none *= (1.0 - sh.alpha[i]);
            sh.col_a[i] = none;                    // P(n, 0) = prod_{j<=n}(1 - alpha_j)
        }
        sh.col_a[0] = 1.0;
        sh.tail[0] = 1.0;
    }
    __syncwarp();
    double *prev = sh.col_a, *cur = sh.col_b;
    double below = 0.0;
    for (int k = 0; k <= m; ++k) {
        // prev = P(., k); record tail
        below += prev[m];
        if (lane == 0) sh.tail[k + 1] = 1.0 - below;
        if (k == m) break;
        // tails only fall: past the first one below the threshold, or past the cap, nothing changes W
        if (k_stop >= 0 && (1.0 - below < thresh || k + 1 >= k_stop)) {
            for (int K = k + 2 + lane; K <= m + 1; K += 32) sh.tail[K] = 0.0;
            break;
        }
        for (int n = lane; n <= m; n += 32) {
            double acc = 0.0;
            if (n >= k + 1)
                for (int i = 1; i <= n; ++i) acc += sh.first[i] * prev[n - i];
            cur[n] = acc;                          // P(n, k+1), zero for n < k+1
        }
        __syncwarp();
        double *tmp = prev; prev = cur; cur = tmp;
    }
    __syncwarp();
    int wt = 0;
    for (int K = 0; K <= m; ++K) if (sh.tail[K] >= thresh) wt = K;
    if (lane == 0) sh.tail[m + 1] = 0.0;
    return wt;
}

// ---------------------------------------------------------------------------------------
// Ratio histogram of one layer.  Every cell with rho = p_beam/q_beam > 1 adds its p and q mass to
// the bin of log2(rho); bin kBins collects rho beyond the last edge.  F(s) for any s in [1, top]
// is then (sum of the bins above s) plus the straddled bin, whose contribution is bracketed from
// its two sums and its edges.
//
// Masses are summed as integers in units of 2^-44, so the sums do not depend on the order in which
// warps and CTAs add, and a cell of mass >= 2^-20 enters without any rounding (its 24-bit
// mantissa is a whole number of units); a smaller cell is rounded by at most 2^-45.  With n cells
// the fixed-point error of any partial sum is therefore at most n 2^-45 (2.8e-8 for a million
// cells), which the chain adds to its bracket.
// In shared memory a bin has two 32-bit words per model, fed by plain (non-returning) atomic adds:
//   w: units of 2^-44.  A cell below 2^-16 adds all of itself here (less than 2^28 units); a larger
//      cell only its remainder below 2^-28 (less than 2^16 units).
//   b: units of 2^-28, the whole multiples of 2^-28 of the cells of at least 2^-16; it cannot
//      overflow because a joint distribution sums to one.
// A w word wraps once the small cells of ONE bin that ONE CTA added reach 2^-12 of the mass.  Two models sigma nats
// apart have up to 0.4 / sigma of their mass per nat, shared out over the cluster's CTAs, and a bin of a layer of m drafts is
// ln(max(m, 2)) / 4096 nats wide: with 4 CTAs, 8 drafts and sigma = 1 that is a fifth of 2^-12, with 2 CTAs, 2 drafts and
// sigma = 0.4 a third; the fullest bin holds about twice that.  The copies of the last bin take 256 times 2^-12, a sixteenth of
// the mass.  Closer models or a flat vocabulary with one CTA (more requests than SMs), and rows that are proportional, where every cell
// lands in the same bin, can reach it.  A wrap is always detected: every thread
// keeps a total of the mass that it added, and the sum of those totals is compared with the sum of
// all words; a difference marks the layer, whose residual masses are
// then all computed by exact passes over the rows.
// ---------------------------------------------------------------------------------------
constexpr int kBins = 4096;
constexpr int kOverSlots = 256;                   // copies of the last bin (rho beyond the last edge): one per
                                                  // warp and half-warp lane, so that none collects enough to wrap
constexpr int kHistWords = kBins + kOverSlots + 16;  // bins 0..kBins-1, the copies of bin kBins, spare words
static_assert(kHistWords % 4 == 0, "the arrays that share this memory need 16-byte alignment");
constexpr float kFix = 17592186044416.f;          // 2^44
constexpr double kUnfix = 1.0 / 17592186044416.0;
constexpr double kErrTol = 2.5e-7;                // error bound of F(s) above which it is recomputed exactly
constexpr int kHistArrays = 4;
struct HistSmem { uint32_t *wp, *wq, *bp, *bq; };

__device__ __forceinline__ HistSmem hist_arrays(uint32_t *base) {
    return HistSmem{base, base + kHistWords, base + 2 * kHistWords, base + 3 * kHistWords};
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Two fp32 values in one 64-bit register: an instruction does both (rounding as the plain ones).
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
    return v;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Items of a pass over n_tiles tiles by n_warps warps: 1, whole tiles; 2, half tiles, where whole ones would leave a part
// of the last round's warps idle (a warp's own work is the pass's length: V = 32000, 16 CTAs, 3 rows: 4.5 us instead of 7).
__device__ __forceinline__ int item_halves(int n_tiles, int n_warps) {
    return (2 * n_tiles + n_warps - 1) / n_warps < 2 * ((n_tiles + n_warps - 1) / n_warps) ? 2 : 1;
}

// The cells of one half tile (4 x float4 per lane and model) into the histogram; adds p - q and q of its cells with
// p_beam > q_beam, in units of 2^-44, to sd and sq.  (p - q cell by cell: the difference of two sums loses what lies
// next to a heavy cell, and a completion draw looks for its tile by these sums.)
// The work per cell decides the speed of this pass (it is bound by instruction issue, not by
// memory), so the common case is straight-line code, two cells to a packed instruction up to the exponentials:
// masses are computed directly in units (the row's factor 2^rest carries the 2^44), the bin comes from an fma
// onto 1.5 * 2^23 whose low mantissa bits are then the integer (no conversion instruction), the two atomic adds
// and the two sums are predicated on p_beam > q_beam inside one asm block, and only cells
// of at least 2^-16 take a branch, one for four cells.  (64 requests x 8 rows of 128256: 236 us to 210 for the
// kernel against one cell to an instruction and a sum of integers to detect wraps.  Slower: eight cells at a time
// or the loads of the next quarter tile in flight (spills at 64 registers), the split of big cells without a branch,
// the next item prefetched into L2: 32 warps hide the loads already.)
// wbase: shared-memory byte address of wp[0] minus 4 * (the bits of the fma's constant), so that
// the address of a bin's word is wbase + 4 * (bits of the fma's result); the q array follows the p
// array at kHistWords words, the b arrays at twice that.
// (ex2.approx flushes results below 2^-126 to zero; a cell enters the sums from 2^-45 on.)
// kBinned = false: the sums alone, by the same instructions, so that a draw finds the same tile whether the layer took
// the histogram or a pass on demand; and in *units the total of p - q in units of 2^-60, by a compensated sum, so that the
// residual mass is as exact as that of the histogram's whole units.  (Whole units, two conversions a cell: a pass 1.5 us longer, the
// compensated sum 0.3.)
constexpr float kBinMagic = 12582912.f;                         // 1.5 * 2^23
constexpr float kBigUnits = 268435456.f;                        // 2^28 units = a cell of 2^-16
template <bool kBinned>
__device__ __forceinline__ void hist_half_tile(const float4 (&vp)[4], const float4 (&vq)[4], float k2,
                                               const RowOff &o, float binscale, float half_bin, float top, uint32_t wbase,
                                               uint32_t over_bits, float &sd, float &sq, long long *units) {
    // dl = log2(rho) - half: the half bin (in log2 units) that turns the fma's round-to-nearest into
    // the bin's floor is part of the row offset, so p_beam > q_beam reads dl > -half
    const float bd = ((o.bp - o.bq) + o.dc) - half_bin;
    const float pass_thr = -half_bin;
    const float cpu = o.cp * kFix, cqu = o.cq * kFix;           // exact: powers of two
    const unsigned long long k22 = pack2(k2, k2), bd2 = pack2(bd, bd), bp2 = pack2(o.bp, o.bp), bq2 = pack2(o.bq, o.bq);
    const unsigned long long cp2 = pack2(cpu, cpu), cq2 = pack2(cqu, cqu), neg2 = pack2(-1.f, -1.f);
    const unsigned long long bs2 = pack2(binscale, binscale), mg2 = pack2(kBinMagic, kBinMagic);
    unsigned long long sum = 0ull, rest = 0ull;
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        float dl[4], pm[4], qm[4], df[4];
        uint32_t addr[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 &zp = vp[it], &zq = vq[it];
            const unsigned long long p2 = h & 1 ? pack2(zp.z, zp.w) : pack2(zp.x, zp.y);
            const unsigned long long q2 = h & 1 ? pack2(zq.z, zq.w) : pack2(zq.x, zq.y);
            const unsigned long long dl2 = fma2(fma2(q2, neg2, p2), k22, bd2);     // NaN compares false
            const float2 d = unpack2(dl2), t = unpack2(fma2(dl2, bs2, mg2));
            const float2 pe = unpack2(fma2(p2, k22, bp2)), qe = unpack2(fma2(q2, k22, bq2));
            const unsigned long long pu2 = mul2(pack2(ex2_approx(pe.x), ex2_approx(pe.y)), cp2);
            const unsigned long long qu2 = mul2(pack2(ex2_approx(qe.x), ex2_approx(qe.y)), cq2);
            const float2 pu = unpack2(pu2), qu = unpack2(qu2), du = unpack2(fma2(qu2, neg2, pu2));
            // floor(log2(rho) * binscale) in the low bits (round to nearest of x - 0.5; an x that is a
            // whole number may fall to either side, both within the bins' edge tolerance)
            // (all cells beyond the last edge in one word would wrap it: every warp and half-warp
            // lane has its own copy of that bin)
            addr[2 * h] = wbase + ((d.x < top ? __float_as_uint(t.x) : over_bits) << 2);
            addr[2 * h + 1] = wbase + ((d.y < top ? __float_as_uint(t.y) : over_bits) << 2);
            dl[2 * h] = d.x; pm[2 * h] = pu.x; qm[2 * h] = qu.x; df[2 * h] = fmaxf(du.x, 0.f);
            dl[2 * h + 1] = d.y; pm[2 * h + 1] = pu.y; qm[2 * h + 1] = qu.y; df[2 * h + 1] = fmaxf(du.y, 0.f);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (kBinned)
                asm("{\n\t.reg .pred p;\n\t"
                    "setp.gt.f32 p, %2, %5;\n\t"
                    "@p add.f32 %0, %0, %3;\n\t"
                    "@p add.f32 %1, %1, %4;\n\t}"
                    : "+f"(sd), "+f"(sq) : "f"(dl[c]), "f"(df[c]), "f"(qm[c]), "f"(pass_thr));
            else {
                df[c] = dl[c] > pass_thr ? df[c] : 0.f;
                sd += df[c];
            }
        if (!kBinned) {
            // compensated (Kahan), two cells to an instruction
#pragma unroll
            for (int c = 0; c < 4; c += 2) {
                const unsigned long long y = fma2(rest, neg2, pack2(df[c], df[c + 1])), t = add2(sum, y);
                rest = fma2(y, neg2, fma2(sum, neg2, t));
                sum = t;
            }
            continue;
        }
        const float big = fmaxf(fmaxf(pm[0], pm[1]), fmaxf(pm[2], pm[3]));
        if (big >= kBigUnits) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (pm[c] >= kBigUnits && dl[c] > pass_thr) {
                    // whole multiples of 2^-28 of a big cell go to the b word (units of 2^-28), the
                    // remainder (below 2^16 units) stays for the w word
                    const float hp = floorf(pm[c] * (1.f / 65536.f));
                    pm[c] = fmaf(-hp, 65536.f, pm[c]);
                    asm volatile("red.shared.add.u32 [%0+%1], %2;" ::"r"(addr[c]), "n"(2 * kHistWords * 4), "r"((uint32_t)hp) : "memory");
                    if (qm[c] >= kBigUnits) {
                        const float hq = floorf(qm[c] * (1.f / 65536.f));
                        qm[c] = fmaf(-hq, 65536.f, qm[c]);
                        asm volatile("red.shared.add.u32 [%0+%1], %2;" ::"r"(addr[c]), "n"(3 * kHistWords * 4), "r"((uint32_t)hq) : "memory");
                    }
                }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
            asm volatile(
                "{\n\t.reg .pred p;\n\t"
                "setp.gt.f32 p, %0, %5;\n\t"
                "@p red.shared.add.u32 [%1], %2;\n\t"
                "@p red.shared.add.u32 [%1+%4], %3;\n\t}"
                :: "f"(dl[c]), "r"(addr[c]), "r"(__float2uint_rn(pm[c])), "r"(__float2uint_rn(qm[c])), "n"(kHistWords * 4), "f"(pass_thr)
                : "memory");
    }
    if (!kBinned) {
        const float2 t = unpack2(sum), e = unpack2(rest);
        *units += __double2ll_rn((((double)t.x - (double)e.x) + ((double)t.y - (double)e.y)) * 65536.0);
    }
}

// One cluster-wide pass without a histogram: item sums of max(p_beam - s q_beam, 0) over the live rows.
// kFirst: s = 1, in the arithmetic (and the half-tile items) of the histogram pass; half_bin is that of the layer's histogram.
// Else: any s, in the arithmetic of the search inside a tile (cell_mass), so that a tile with a sum has a cell that the search
// finds; whole tiles.  sh.warp_part gets the total of each warp's items as whole numbers, so the order in which warps and CTAs add
// up changes nothing.  Unless kFirst, in two words, so that a small F keeps its digits, and the q mass of the cells with
// p_beam > s q_beam.  kTotal = false: the item sums alone.
// Bound by latency where a cluster is alone with its pass (a warp takes about 1.8 us a half tile), by issue where many are at it:
// 54 requests x 7 rows of 90496, 18 of which make a pass for a draw, 198 us the call with totals that nobody reads, 194 without.
// Straight-line loads for whole aligned halves.  (The next item prefetched into L2: no difference.  Totals in registers: spills,
// a call 1 per cent slower.)
// Functions of their own: the callers would each carry the unrolled loop.
constexpr double kSumUnit = 1152921504606846976.0;               // 2^60
template <bool kFirst, bool kTotal>
__device__ __noinline__ void residual_pass(const float *__restrict__ zp, const float *__restrict__ zq, int64_t stride,
                                                int V, int T, float k2, Shared &sh, float s, float half_bin, double *sums,
                                                int warp, int nwarps, int halves) {
    const int lane = threadIdx.x & 31;
    const int row_items = T * halves, items = sh.nA * row_items;
    if (lane < 3) sh.warp_part[lane][threadIdx.x >> 5] = 0ll;
    __syncwarp();
    long long units = 0ll;
    for (int item = warp; item < items; item += nwarps) {
        const int i = item / row_items, t = item - i * row_items;
        const int row = sh.A[i];
        const float *rp = zp + (int64_t)row * stride;
        const float *rq = zq + (int64_t)row * stride;
        const bool al = ((reinterpret_cast<uintptr_t>(rp) | reinterpret_cast<uintptr_t>(rq)) & 15) == 0;
        const RowOff ro = row_off(sh, i);
        double res1 = 0.0;
        float acc = 0.f, q_acc = 0.f;
        int e0 = t * (kTile / halves);
#pragma unroll 1
        for (int half = halves; half < 3; ++half, e0 += kTile / 2) {
            float4 vp[4], vq[4];
            if (al && e0 + kTile / 2 <= V) {
#pragma unroll
                for (int it = 0; it < 4; ++it) vp[it] = ldg_stream(reinterpret_cast<const float4 *>(rp + e0 + it * 128) + lane);
#pragma unroll
                for (int it = 0; it < 4; ++it) vq[it] = ldg_stream(reinterpret_cast<const float4 *>(rq + e0 + it * 128) + lane);
            } else {
                load_half_tile(rp, e0, V, lane, vp);
                load_half_tile(rq, e0, V, lane, vq);
            }
            if (kFirst) {
                float sd = 0.f, sq = 0.f;
                hist_half_tile<false>(vp, vq, k2, ro, 0.f, half_bin, 0.f, 0u, 0u, sd, sq, &units);
                res1 += (double)sd;
            } else {
                // cell_mass, two cells to an instruction around the exponentials
                const unsigned long long k22 = pack2(k2, k2), bp2 = pack2(ro.bp, ro.bp), bq2 = pack2(ro.bq, ro.bq);
                const unsigned long long cp2 = pack2(ro.cp, ro.cp), cq2 = pack2(ro.cq, ro.cq), s2 = pack2(-s, -s);
#pragma unroll
                for (int it = 0; it < 4; ++it)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float2 pe = unpack2(fma2(h ? pack2(vp[it].z, vp[it].w) : pack2(vp[it].x, vp[it].y), k22, bp2));
                        const float2 qe = unpack2(fma2(h ? pack2(vq[it].z, vq[it].w) : pack2(vq[it].x, vq[it].y), k22, bq2));
                        const unsigned long long p2 = mul2(pack2(exp2f(pe.x), exp2f(pe.y)), cp2);
                        const unsigned long long q2 = mul2(pack2(exp2f(qe.x), exp2f(qe.y)), cq2);
                        const float2 d = unpack2(fma2(s2, q2, p2)), q = unpack2(q2);
                        acc += fmaxf(d.x, 0.f);
                        acc += fmaxf(d.y, 0.f);
                        if (kTotal) {
                            q_acc += d.x > 0.f ? q.x : 0.f;
                            q_acc += d.y > 0.f ? q.y : 0.f;
                        }
                    }
            }
        }
        const double tot = kFirst ? warp_sum(res1) * kUnfix : warp_sum((double)acc);
        const double q = kFirst || !kTotal ? 0.0 : warp_sum((double)q_acc) * (double)kFix;
        if (lane == 0) {
            sums[item] = tot;
            if (!kFirst && kTotal) {
                const long long hi = __double2ll_rn(tot * kSumUnit);
                sh.warp_part[0][threadIdx.x >> 5] += hi;
                sh.warp_part[1][threadIdx.x >> 5] += __double2ll_rn((tot * kSumUnit - (double)hi) * kSumUnit);
                sh.warp_part[2][threadIdx.x >> 5] += __double2ll_rn(q);
            }
        }
    }
    if (kFirst) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) units += __shfl_xor_sync(kFull, units, o);
        if (lane == 0) sh.warp_part[0][threadIdx.x >> 5] = units;
    }
}

// F(s) by a pass of the whole cluster over the live rows, whose item sums go to `sums`.  first: s = 1, with the sums that the
// histogram pass would have left.  Else the cells meet s as one float, as in the search of a draw; what that leaves out of
// F, the remainder of s times the q mass above, is taken off the total.  n_pass: passes of the kernel before this one.
// want_total = false: the item sums alone, for a draw.
__device__ __forceinline__ double exact_pass(const VerifyArgs &a, Shared &sh, double s, double *sums, bool first, float half_bin,
                                          int halves, bool want_total, int n_pass) {
    cg::cluster_group cluster = cg::this_cluster();
    const int n_cta = (int)cluster.num_blocks(), cta_rank = (int)cluster.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float s_hi = (float)s;
    const int w = cta_rank * kVWarps + warp, nw = n_cta * kVWarps;
    if (first) residual_pass<true, true>(a.zp, a.zq, a.stride, a.V, a.T, a.k2, sh, s_hi, half_bin, sums, w, nw, halves);
    else if (want_total) residual_pass<false, true>(a.zp, a.zq, a.stride, a.V, a.T, a.k2, sh, s_hi, 0.f, sums, w, nw, halves);
    else residual_pass<false, false>(a.zp, a.zq, a.stride, a.V, a.T, a.k2, sh, s_hi, 0.f, sums, w, nw, halves);
    if (!want_total) {
        cluster.sync();
        return 0.0;
    }
    __syncthreads();
    if (warp < 3) {
        long long v = lane < kVWarps ? sh.warp_part[warp][lane] : 0ll;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        if (lane < n_cta) cluster.map_shared_rank(&sh, lane)->part[n_pass & 1][warp][cta_rank] = v;
    }
    cluster.sync();                                    // (two buffers: who is here has read those of the pass before)
    long long hi = 0ll, lo = 0ll, q = 0ll;
    for (int c = 0; c < n_cta; ++c) {
        hi += sh.part[n_pass & 1][0][c];
        lo += sh.part[n_pass & 1][1][c];
        q += sh.part[n_pass & 1][2][c];
    }
    if (first) return (double)hi * (1.0 / kSumUnit);
    const double total = ((double)lo * (1.0 / kSumUnit) + (double)hi) * (1.0 / kSumUnit);
    const double rest = (s - (double)s_hi) * ((double)q * kUnfix);
    return rest < total ? total - rest : total;
}

// One cluster-wide pass over the live rows; every CTA fills its own shared-memory histogram.
// tot (shared memory, zero before the call): [0] the mass that the CTA added (p and q), from floating-point sums.
__device__ void histogram_pass(const VerifyArgs &a, const Shared &sh, float binscale, const HistSmem &h,
                               double *sums1, int cta_rank, int n_cta, int halves, unsigned long long *tot) {
    // halves = 2: an item is a half tile (when the cluster has a warp for each), with a sum of its own
    const int lane = threadIdx.x & 31;
    const int warp = cta_rank * kVWarps + (threadIdx.x >> 5);
    const int nwarps = n_cta * kVWarps;
    const int items = sh.nA * a.T * halves;
    unsigned long long added = 0ull;
    const uint32_t magic_bits = __float_as_uint(kBinMagic);
    const uint32_t wbase = (uint32_t)__cvta_generic_to_shared(h.wp) - (magic_bits << 2);
    const uint32_t over_bits = magic_bits + (uint32_t)(kBins + ((threadIdx.x >> 5) & 15) * 16 + (threadIdx.x & 15));
    const float half_bin = 0.5f / binscale;                      // half a bin in log2 units
    const float top = (float)kBins / binscale - half_bin;       // log2 of the last edge (minus the half), as the bins see it
    const int row_items = a.T * halves;
    for (int item = warp; item < items; item += nwarps) {
        const int i = item / row_items, t = item - i * row_items;
        const int row = sh.A[i];
        const float *rp = a.zp + (int64_t)row * a.stride;
        const float *rq = a.zq + (int64_t)row * a.stride;
        const bool al = ((reinterpret_cast<uintptr_t>(rp) | reinterpret_cast<uintptr_t>(rq)) & 15) == 0;
        const RowOff ro = row_off(sh, i);
        double res1 = 0.0;                               // sum of (p - q)+ over the item in units: residual mass at s = 1
        int e0 = t * (kTile / halves);
#pragma unroll 1
        for (int half = halves; half < 3; ++half, e0 += kTile / 2) {
            float4 vp[4], vq[4];
            if (al && e0 + kTile / 2 <= a.V) {
#pragma unroll
                for (int it = 0; it < 4; ++it) vp[it] = ldg_stream(reinterpret_cast<const float4 *>(rp + e0 + it * 128) + lane);
#pragma unroll
                for (int it = 0; it < 4; ++it) vq[it] = ldg_stream(reinterpret_cast<const float4 *>(rq + e0 + it * 128) + lane);
            } else {
                load_half_tile(rp, e0, a.V, lane, vp);
                load_half_tile(rq, e0, a.V, lane, vq);
            }
            float sd = 0.f, sq = 0.f;
            hist_half_tile<true>(vp, vq, a.k2, ro, binscale, half_bin, top, wbase, over_bits, sd, sq, nullptr);
            added += __float2ull_rn(fmaf(2.f, sq, sd));
            res1 += (double)sd;
        }
        // the items' sums of the residual after ONE rejection (s_1 = 1): what a completion draw at run
        // position 2 searches, so that this common case needs no second pass over the rows
        const double tot1 = warp_sum(res1) * kUnfix;
        if (lane == 0) sums1[item] = tot1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) added += __shfl_xor_sync(kFull, added, o);
    if (lane == 0 && added) atomicAdd(tot, added);
}

// The copies of the last bin (rho beyond the last edge), folded by each CTA and added to every CTA's total
// (tot[7], tot[8]); before the cluster barrier that follows the pass.  Also tot[6] += what the CTA's threads
// added minus what these copies hold of it.
__device__ void hist_fold_over(cg::cluster_group &cluster, const HistSmem &h, unsigned long long *tot, int n_cta) {
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < kOverSlots) {
        const int i = kBins + (int)threadIdx.x;
        unsigned long long P = ((unsigned long long)h.bp[i] << 16) + h.wp[i], Q = ((unsigned long long)h.bq[i] << 16) + h.wq[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            P += __shfl_xor_sync(kFull, P, o);
            Q += __shfl_xor_sync(kFull, Q, o);
        }
        unsigned long long w = P + Q;
        if (threadIdx.x < 32) w -= tot[0];
        if (lane < n_cta) {
            unsigned long long *to = cluster.map_shared_rank(tot, lane);
            if (w) atomicAdd(to + 6, 0ull - w);
            if (P) atomicAdd(to + 7, P);
            if (Q) atomicAdd(to + 8, Q);
        }
    }
}

// Merge of the cluster's histograms, after a cluster barrier that follows the pass: every CTA sums one slice of
// the bins over all CTAs' shared memory.  A lane takes four bins of two CTAs (eight bins when there is one CTA), so
// that all its loads are in flight together; the lanes that share bins add up by shuffles, and with 16 CTAs two
// warps share bins.  The CTA's suffix sums (p and q mass of the slice's bins >= k, units of 2^-44) replace the words of
// its own slice, which no other CTA reads here: w words the low, b words the high halves.  Every CTA
// gets the slice's totals.  The caller puts a cluster barrier behind this before anyone looks at another's slice.
// Bound by distributed shared memory (64 KB a CTA, 4.5 us), as long as an instruction takes at least 128 bytes from
// each CTA it reads: with 64 bytes from each of 8, one warp to the bins, 16 CTAs took 7 to 10 us.  (512 bytes
// an instruction and the sums of 2 to 8 warps through a stage of 16 KB were no faster with 8 CTAs, and the shared
// memory came off the L1 cache: 64 requests x 8 rows of 128256 30 us slower.  Half the words to fetch, by b words
// that are added at once in the CTA that will merge them: merge 4.4 -> 3.3 us, but the pass 110 -> 115 and, for one request
// of V = 32000, 7.5 -> 9.5: an atomic add to another CTA's shared memory costs its warp more than a local one.  Half the
// bins for layers of few drafts: merge 4.4 -> 3.1, but their w words wrap on ordinary data when one CTA has the whole layer.)
__device__ void hist_merge(cg::cluster_group &cluster, const HistSmem &h, Shared &sh, int cta_rank, int n_cta) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int share = n_cta > 1 ? min(n_cta / 2, 4) : 1;     // lanes that share four bins
    const int parts = n_cta > 8 ? 2 : 1;                     // warps that share them
    const int per_warp = 32 / share, place = lane % per_warp, segs = kVWarps / parts;
    const int seg = warp % segs, part = warp / segs;
    const int n_bins = n_cta > 1 ? 4 : 8;                    // of a lane
    const int i0 = cta_rank * (kBins / n_cta) + (seg * per_warp + place) * n_bins;
    unsigned long long P[8] = {}, Q[8] = {};
    auto add4 = [&](int c, int i, unsigned long long *p, unsigned long long *q) {
        const uint4 wp = *reinterpret_cast<const uint4 *>(cluster.map_shared_rank(h.wp, c) + i);
        const uint4 wq = *reinterpret_cast<const uint4 *>(cluster.map_shared_rank(h.wq, c) + i);
        const uint4 bp = *reinterpret_cast<const uint4 *>(cluster.map_shared_rank(h.bp, c) + i);
        const uint4 bq = *reinterpret_cast<const uint4 *>(cluster.map_shared_rank(h.bq, c) + i);
        p[0] += ((unsigned long long)bp.x << 16) + wp.x; p[1] += ((unsigned long long)bp.y << 16) + wp.y;
        p[2] += ((unsigned long long)bp.z << 16) + wp.z; p[3] += ((unsigned long long)bp.w << 16) + wp.w;
        q[0] += ((unsigned long long)bq.x << 16) + wq.x; q[1] += ((unsigned long long)bq.y << 16) + wq.y;
        q[2] += ((unsigned long long)bq.z << 16) + wq.z; q[3] += ((unsigned long long)bq.w << 16) + wq.w;
    };
    const int c0 = part * 8 + lane / per_warp;
    if (n_cta > 1) {
        add4(c0, i0, P, Q);
        add4(c0 + share, i0, P, Q);
    } else {
        add4(0, i0, P, Q);
        add4(0, i0 + 4, P + 4, Q + 4);
    }
    for (int o = per_warp; o < 32; o <<= 1) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            P[k] += __shfl_xor_sync(kFull, P[k], o);
            Q[k] += __shfl_xor_sync(kFull, Q[k], o);
        }
    }
    auto store4 = [&](int i, const unsigned long long *p, const unsigned long long *q, unsigned long long rp, unsigned long long rq) {
        auto words = [&](uint32_t *low, uint32_t *high, const unsigned long long *v, unsigned long long r) {
            *reinterpret_cast<uint4 *>(low + i) = make_uint4((uint32_t)(v[0] + r), (uint32_t)(v[1] + r), (uint32_t)(v[2] + r), (uint32_t)(v[3] + r));
            *reinterpret_cast<uint4 *>(high + i) = make_uint4((uint32_t)((v[0] + r) >> 32), (uint32_t)((v[1] + r) >> 32),
                                                             (uint32_t)((v[2] + r) >> 32), (uint32_t)((v[3] + r) >> 32));
        };
        words(h.wp, h.bp, p, rp);
        words(h.wq, h.bq, q, rq);
    };
    if (parts == 2) {
        // the second warp's sums through the slice itself, once the whole CTA has read its own words there
        __syncthreads();
        if (part == 1 && lane < per_warp) store4(i0, P, Q, 0ull, 0ull);
        __syncthreads();
        if (part == 0) {
            const uint4 lp = *reinterpret_cast<const uint4 *>(h.wp + i0), up = *reinterpret_cast<const uint4 *>(h.bp + i0);
            const uint4 lq = *reinterpret_cast<const uint4 *>(h.wq + i0), uq = *reinterpret_cast<const uint4 *>(h.bq + i0);
            auto whole = [](uint32_t low, uint32_t high) { return ((unsigned long long)high << 32) | low; };
            P[0] += whole(lp.x, up.x); P[1] += whole(lp.y, up.y); P[2] += whole(lp.z, up.z); P[3] += whole(lp.w, up.w);
            Q[0] += whole(lq.x, uq.x); Q[1] += whole(lq.y, uq.y); Q[2] += whole(lq.z, uq.z); Q[3] += whole(lq.w, uq.w);
        }
    }
    // suffix sums: in the lane, over the lanes' places, over the warps of part 0
#pragma unroll
    for (int k = 6; k >= 0; --k) { P[k] += P[k + 1]; Q[k] += Q[k + 1]; }
    unsigned long long ap = P[0], aq = Q[0];
    for (int o = 1; o < per_warp; o <<= 1) {
        const unsigned long long tp = __shfl_down_sync(kFull, ap, o), tq = __shfl_down_sync(kFull, aq, o);
        if (place + o < per_warp) { ap += tp; aq += tq; }
    }
    if (part == 0 && lane == 0) { sh.wtot_p[seg] = ap; sh.wtot_q[seg] = aq; }
    __syncthreads();
    if (part > 0) return;
    unsigned long long rp = ap - P[0], rq = aq - Q[0];
    for (int w = seg + 1; w < segs; ++w) { rp += sh.wtot_p[w]; rq += sh.wtot_q[w]; }
    if (lane < per_warp) {
        store4(i0, P, Q, rp, rq);
        if (n_cta == 1) store4(i0 + 4, P + 4, Q + 4, rp, rq);
    }
    if (seg == 0) {
        // place 0: the whole slice
        const unsigned long long tp = __shfl_sync(kFull, P[0] + rp, 0), tq = __shfl_sync(kFull, Q[0] + rq, 0);
        if (lane < n_cta) {
            Shared *to = cluster.map_shared_rank(&sh, lane);
            to->slice_p[cta_rank] = tp;
            to->slice_q[cta_rank] = tq;
        }
    }
}

// One completion draw (residual if s_res > 0 else p_beam) by one warp; returns the token or -1
// and the index of the live parent.
__device__ int draw_cell(const VerifyArgs &a, const Shared &sh, double u, bool use_res, float s_res,
                         const double *res_sums, int halves, int lane, int *ia_out) {
    int ia, t;
    double target;
    if (use_res) {
        // (res_sums: one per tile, or two when the pass that wrote them worked on half tiles)
        auto sum = [&](int i) { return halves == 1 ? __ldcg(res_sums + i) : __ldcg(res_sums + 2 * i) + __ldcg(res_sums + 2 * i + 1); };
        const int tile = locate_tile(sum, sh.nA * a.T, u, true, lane, &target);
        if (tile < 0) return -1;
        ia = tile / a.T; t = tile - ia * a.T;
    } else {
        // p_beam: first the live parent (its row holds exactly its beam weight), then the tile
        ia = locate_tile([&](int i) { return sh.wp[i]; }, sh.nA, u, true, lane, &target);
        if (ia < 0) return -1;
        const int row = sh.A[ia];
        const double wpa = sh.wp[ia], lse_row = a.lse[row];
        const TileStat *st = a.stats + (int64_t)row * a.T;
        t = locate_tile([&](int i) {
            const TileStat ts = st[i];
            if (!(ts.sum > 0.f)) return 0.0;
            return wpa * (double)ts.sum * exp((double)ts.mx * a.inv_tau - lse_row);
        }, a.T, target, false, lane, &target);
        if (t < 0) return -1;
    }
    *ia_out = ia;
    const RowOff ro = row_off(sh, ia);
    const int64_t row = (int64_t)sh.A[ia] * a.stride;
    return locate_token(a.zp + row, a.zq + row, a.V, a.k2, t, ro, use_res ? s_res : 0.f, target, lane);
}

// ---------------------------------------------------------------------------------------
// Warped joints (top-k / top-p).  The support of T o p_beam has at most top_k <= 64 cells, so
// once it is known everything else of the layer is scalar work.  Finding it needs no pass over
// the rows: the maximum of every 1024-token tile is known from the dense pass, the k largest
// tile maxima are k distinct cells, hence the k-th largest cell of the joint is at least the
// k-th largest tile bound and every cell of the top k lies in a tile whose bound reaches it.
// Only those (about k) tiles are read.
// ---------------------------------------------------------------------------------------
constexpr int kMaxTopK = 64;
constexpr int kMaxCand = 680;      // candidate cells per model (two lists overlay one histogram array)
constexpr int kHalf = kVThreads / 2;   // threads that build one model's support when the two models run side by side
// scratch of one build_support instance
struct SupportTmp {
    float off[kMaxLive];          // log(beam weight) - lse of each live row
    int sel[256];                 // tiles whose bound reaches the threshold
    unsigned lo[kVWarps], hi[kVWarps];   // per warp, images of the smallest finite and of the largest bound
    int finite[kVWarps];          // per warp, finite bounds
    int count[3];                 // of the bisection's rounds, in turn
    unsigned low;                 // image of the smallest bound from the cut on
    int n_sel, n_cand, err;
};
struct WarpScratch {
    double prob[2][kMaxTopK];     // warped probabilities, most probable first (0: p, 1: q)
    double qat[kMaxTopK];         // q~ at the cells of the p support
    int cell[2][kMaxTopK];        // live parent index * V + token
    int order[kMaxTopK];          // the p support in canonical (cell-ascending) order
    int n[2];
    SupportTmp tmp[2];
};
constexpr int kBoundCache = kHistWords;   // tile bounds kept in shared memory: the third (p) or fourth (q) histogram array
static_assert(sizeof(WarpScratch) <= kHistWords * sizeof(uint32_t), "the support scratch overlays the second histogram array");
static_assert(2 * kMaxCand * (sizeof(double) + sizeof(int)) <= (kBins + 2) * sizeof(uint32_t),
              "the two candidate lists overlay the other histogram array");

// barrier of the NT threads that work on one model (ids 1 and 2; 0 is __syncthreads)
template <int NT>
__device__ __forceinline__ void part_sync(int model) {
    asm volatile("bar.sync %0, %1;" ::"r"(model + 1), "n"(NT) : "memory");
}

// Support of the warped joint of one model by NT threads: a half of the CTA for each model (warps 0-7: p, warps
// 8-15: q) side by side on their own scratch, or the whole CTA where only p is wanted.  hist_p / hist_q: the first two
// of the idle histogram arrays.  Returns 0 or a DSBD_DEV_* code (the same on every thread of the part).
// Latency decides (a chain of short steps between barriers): the threshold is a bisection whose rounds have one
// barrier each and that stops at the first cut with k to k + 2 tiles above it, about 8 rounds.  Exact radix
// selection (4 rounds of three barriers with colliding atomics), one warp that lists the tiles, one thread that cuts
// at top-p and half the CTA for a draft layer's only model took, for a draft of 5 layers of 16 x 8 rows of 128256 with
// top-k 10, 419 us instead of 337; 20 requests with top-k 50 took 169 instead of 144.  (As a function that is
// not inlined, with generic loads: 363 and 165.)
template <int NT>
__device__ int build_support(const VerifyArgs &a, const Shared &sh, int model, uint32_t *hist_p, uint32_t *hist_q) {
    WarpScratch &ws = *reinterpret_cast<WarpScratch *>(hist_q);
    SupportTmp &tp = ws.tmp[model];
    double *cand_key = reinterpret_cast<double *>(hist_p) + model * kMaxCand;
    int *cand_cell = reinterpret_cast<int *>(reinterpret_cast<double *>(hist_p) + 2 * kMaxCand) + model * kMaxCand;
    const int tl = threadIdx.x & (NT - 1);                    // thread and warp inside the part
    const int lane = threadIdx.x & 31, warp = tl >> 5;
    constexpr int kPartWarps = NT / 32;
    const int T = a.T, nt = sh.nA * T, k = a.top_k;
    const TileStat *stats = a.stats + (int64_t)model * a.N * T;
    const double *lw = model ? sh.lwq : sh.lwp;
    const double *lse = a.lse + (int64_t)model * a.N;
    const float *z = model ? a.zq : a.zp;
    const float inv_tau_f = (float)a.inv_tau;
    for (int i = tl; i < sh.nA; i += NT) tp.off[i] = (float)(lw[i] - lse[sh.A[i]]);
    if (tl < 3) tp.count[tl] = 0;
    if (tl == 0) { tp.low = 0xffffffffu; tp.n_sel = 0; tp.n_cand = 0; tp.err = 0; ws.n[model] = 0; }
    part_sync<NT>(model);
    // float upper bound of log(joint probability) over tile i
    auto bound = [&](int i) -> float {
        const int ia = i / T;
        return fmaf(stats[(int64_t)sh.A[ia] * T + (i - ia * T)].mx, inv_tau_f, tp.off[ia]);
    };
    // order-preserving integer image of a float and back
    auto image = [](float v) -> unsigned {
        const unsigned b = __float_as_uint(v);
        return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
    };
    auto value = [](unsigned u) -> float { return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u); };
    // A cut not above the k-th largest tile bound (with multiplicity: k tiles each hold a cell at least that
    // large) with few tiles below it; with fewer than k finite bounds every tile counts.  Bounds that do not fit
    // the cache are computed again in every round.
    unsigned *bcache = hist_p + (2 + model) * kHistWords;
    const bool cached = nt <= kBoundCache;
    {
        unsigned lo = 0xffffffffu, hi = 0u;
        int finite = 0;
#pragma unroll 4
        for (int i = tl; i < nt; i += NT) {
            const float v = bound(i);
            const unsigned u = image(v);
            if (cached) bcache[i] = u;
            if (v > -INFINITY) { ++finite; lo = min(lo, u); hi = max(hi, u); }
        }
        lo = __reduce_min_sync(kFull, lo); hi = __reduce_max_sync(kFull, hi); finite = __reduce_add_sync(kFull, finite);
        if (lane == 0) { tp.lo[warp] = lo; tp.hi[warp] = hi; tp.finite[warp] = finite; }
    }
    part_sync<NT>(model);
    unsigned lo = 0xffffffffu, hi = 0u;
    int finite = 0;
#pragma unroll
    for (int w = 0; w < kPartWarps; ++w) { lo = min(lo, tp.lo[w]); hi = max(hi, tp.hi[w]); finite += tp.finite[w]; }
    if (finite >= k) {
        // count(>= lo) >= k always holds; hi is above the k-th largest.  One or two too many are fine where they are close
        // (cells 30 below the largest have no mass to speak of)
        const float near = value(hi) - 30.f;
        ++hi;
        for (int round = 0; hi - lo > 1; ++round) {
            const unsigned mid = lo + (hi - lo) / 2;
            int n = 0;
            for (int i = tl; i < nt; i += NT) n += (cached ? bcache[i] : image(bound(i))) >= mid;
            n = __reduce_add_sync(kFull, n);
            if (lane == 0 && n) atomicAdd(&tp.count[round % 3], n);
            if (tl == 0) tp.count[(round + 1) % 3] = 0;           // (last read two rounds ago)
            part_sync<NT>(model);
            n = tp.count[round % 3];
            if (n < k) { hi = mid; continue; }
            lo = mid;
            if (n == k || (n <= k + 2 && value(lo) > near)) break;
        }
    }
    // The tiles from the cut on, and the smallest bound among them, which is the threshold: a cut may lie far down in
    // the gap above masked tiles, where it would pass every cell of the tiles above.
    // (the float keys carry an error of about 1e-5; the slack keeps the selection conservative)
    auto slack = [](float t) -> float { return t - 5e-5f - 4e-6f * fabsf(t); };
    float theta = -INFINITY, cut = finite >= k ? slack(value(lo)) : -INFINITY;
    for (int again = 0; ; ++again) {
        unsigned low = 0xffffffffu;
        for (int i = tl; i < nt; i += NT) {
            const float bv = cached ? value(bcache[i]) : bound(i);
            if (bv >= cut && bv > -INFINITY) {
                const int pos = atomicAdd(&tp.n_sel, 1);
                if (pos < 256) tp.sel[pos] = i;
                if (image(bv) >= lo) low = min(low, image(bv));
            }
        }
        low = __reduce_min_sync(kFull, low);
        if (lane == 0 && low != 0xffffffffu) atomicMin(&tp.low, low);
        part_sync<NT>(model);
        if (finite >= k) theta = slack(value(tp.low));
        if (tp.n_sel <= 256) break;
        if (again) return DSBD_DEV_CAPACITY;                      // hundreds of tiles tie at the threshold
        // (or closely below the cut)
        part_sync<NT>(model);
        if (tl == 0) tp.n_sel = 0;
        cut = theta;
        part_sync<NT>(model);
    }
    const int n_sel = tp.n_sel;
    // One sweep over the selected tiles by all warps: counts the cells whose key reaches th and,
    // when asked, appends them to the candidate list (order is irrelevant: the final choice is
    // by (key, cell)).
    auto sweep = [&](float th, bool collect) {
        part_sync<NT>(model);                      // every thread has taken the previous sweep's count
        if (tl == 0) tp.n_cand = 0;
        part_sync<NT>(model);
        // this warp's tiles into L2 first (a tile is 32 lines of 128 bytes: one per lane), so that
        // the dependent tile loads below do not each pay a trip to HBM
        for (int sidx = warp; sidx < n_sel; sidx += kPartWarps) {
            const int ti = tp.sel[sidx], ia = ti / T, t = ti - ia * T;
            const int e = t * kTile + lane * 32;
            if (e < a.V) asm volatile("prefetch.global.L2 [%0];" ::"l"(z + (int64_t)sh.A[ia] * a.stride + e));
        }
        for (int sidx = warp; sidx < n_sel; sidx += kPartWarps) {
            const int ti = tp.sel[sidx], ia = ti / T, t = ti - ia * T, row = sh.A[ia];
            const float *rowp = z + (int64_t)row * a.stride;
            const bool al = (reinterpret_cast<uintptr_t>(rowp) & 15) == 0;
            float4 v[8];
            load_tile<false>(rowp, t * kTile, a.V, al, lane, v);
            const float off_f = tp.off[ia];
            const double off_d = lw[ia] - lse[row];
            unsigned hits = 0;                               // bit (it*4+c) of this lane's 32 cells
#pragma unroll
            for (int it = 0; it < 8; ++it) {
                const float zz[4] = {v[it].x, v[it].y, v[it].z, v[it].w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float kf = fmaf(zz[c], inv_tau_f, off_f);
                    if (kf >= th && kf > -INFINITY) hits |= 1u << (it * 4 + c);
                }
            }
            const int mine = __popc(hits);
            int incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int tmp = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += tmp;
            }
            const int total = __shfl_sync(kFull, incl, 31);
            int base_pos = 0;
            if (lane == 0 && total) base_pos = atomicAdd(&tp.n_cand, total);
            base_pos = __shfl_sync(kFull, base_pos, 0);
            if (collect && mine) {
                int pos = base_pos + incl - mine;
#pragma unroll
                for (int it = 0; it < 8; ++it) {
                    const float zz[4] = {v[it].x, v[it].y, v[it].z, v[it].w};
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (hits & (1u << (it * 4 + c))) {
                            if (pos < kMaxCand) {
                                cand_key[pos] = off_d + (double)zz[c] * a.inv_tau;
                                cand_cell[pos] = ia * a.V + t * kTile + it * 128 + lane * 4 + c;
                            }
                            ++pos;
                        }
                }
            }
        }
        part_sync<NT>(model);
        return tp.n_cand;
    };
    int n_cand = sweep(theta, true);
    if (n_cand > kMaxCand) {
        // too many cells reach the conservative threshold (few tiles, large k, or near ties):
        // bisect for a threshold with between k and kMaxCand cells above it
        float lo_t = theta, hi_t = -INFINITY;
        for (int sidx = 0; sidx < n_sel; ++sidx) hi_t = fmaxf(hi_t, bound(tp.sel[sidx]));
        if (!(lo_t > -INFINITY)) lo_t = hi_t - 400.f;
        bool found = false;
        for (int itn = 0; itn < 60 && hi_t > lo_t; ++itn) {
            // (first out of the gap above a mask of finite values: halving does not come back from -1e30)
            const float half = 0.5f * (lo_t + hi_t), mid = itn ? half : fmaxf(half, hi_t - 400.f);
            const int c = sweep(mid, false);
            if (c > kMaxCand) lo_t = mid;
            else if (c < k) hi_t = mid;
            else { theta = mid; found = true; break; }
        }
        if (!found) return DSBD_DEV_CAPACITY;              // a huge tie at the cut
        n_cand = sweep(theta, true);
    }
    // exact top k of the candidates: every candidate counts those that beat it (key descending,
    // cell ascending -- a total order, cells are unique) and, if fewer than k do, that count is its
    // place in the support
    if (n_cand > kMaxCand) n_cand = kMaxCand;
    for (int jc = tl; jc < n_cand; jc += NT) {
        const double key = cand_key[jc];
        const int cell = cand_cell[jc];
        int rank = 0;
#pragma unroll 4
        for (int i = 0; i < n_cand; ++i) {
            const double ki = cand_key[i];
            rank += (ki > key) || (ki == key && cand_cell[i] < cell);
        }
        if (rank < k) {
            ws.prob[model][rank] = exp(key);
            ws.cell[model][rank] = cell;
        }
    }
    part_sync<NT>(model);
    if (warp == 0) {
        // renormalise over the top k, then the top-p cut and its renormalisation: a lane has the places 2 lane, 2 lane + 1
        const int n_sup = n_cand < k ? n_cand : k;
        const double p0 = 2 * lane < n_sup ? ws.prob[model][2 * lane] : 0.0;
        const double p1 = 2 * lane + 1 < n_sup ? ws.prob[model][2 * lane + 1] : 0.0;
        const double incl = warp_scan(p0 + p1, lane), cum0 = incl - p1;
        double zsum = __shfl_sync(kFull, incl, 31);
        int keep = n_sup;
        if (a.top_p > 0.0 && a.top_p < 1.0 && zsum > 0.0) {
            // the first place whose running sum reaches top_p is the last one kept
            const unsigned b0 = __ballot_sync(kFull, cum0 < a.top_p * zsum), b1 = __ballot_sync(kFull, incl < a.top_p * zsum);
            keep = min(n_sup, __popc(b0) + __popc(b1) + 1);
            const double c0 = __shfl_sync(kFull, cum0, (keep - 1) / 2), c1 = __shfl_sync(kFull, incl, (keep - 1) / 2);
            zsum = (keep & 1) ? c0 : c1;
        }
        const double inv = zsum > 0.0 ? 1.0 / zsum : 0.0;
        if (2 * lane < keep) ws.prob[model][2 * lane] = p0 * inv;
        if (2 * lane + 1 < keep) ws.prob[model][2 * lane + 1] = p1 * inv;
        if (lane == 0) ws.n[model] = keep;
    }
    part_sync<NT>(model);
    return 0;
}

__device__ __forceinline__ double support_lookup(const WarpScratch &ws, int model, int cell) {
    int at = -1;
    for (int j = 0, n = ws.n[model]; j < n; ++j) at = ws.cell[model][j] == cell ? j : at;      // (cells are unique)
    return at >= 0 ? ws.prob[model][at] : 0.0;
}

// Inverse-CDF draws over the p support in canonical order; mass max(p~ - s q~, 0) (s = 0: p~).  By one warp, one
// draw for each lane that wants one (u per lane).  Returns the index into the p support or -1.
__device__ int draw_support(const WarpScratch &ws, double u, double s, int lane) {
    const int n = ws.n[0];
    double w0 = 0.0, w1 = 0.0;                                // places 2 lane and 2 lane + 1
    if (2 * lane < n) { const int i = ws.order[2 * lane]; w0 = fmax(ws.prob[0][i] - s * ws.qat[i], 0.0); }
    if (2 * lane + 1 < n) { const int i = ws.order[2 * lane + 1]; w1 = fmax(ws.prob[0][i] - s * ws.qat[i], 0.0); }
    const double incl = warp_scan(w0 + w1, lane), cum0 = incl - w1;
    const double zsum = __shfl_sync(kFull, incl, 31);
    const unsigned m0 = __ballot_sync(kFull, w0 > 0.0), m1 = __ballot_sync(kFull, w1 > 0.0);
    const double target = u * zsum;
    int pick = -1;
    bool found = false;
    for (int l = 0; 2 * l < n; ++l) {
        const double c0 = __shfl_sync(kFull, cum0, l), c1 = __shfl_sync(kFull, incl, l);
        if (!found && (m0 >> l & 1)) { pick = 2 * l; found = c0 >= target; }
        if (!found && (m1 >> l & 1)) { pick = 2 * l + 1; found = c1 >= target; }
    }
    return pick < 0 || !(zsum > 0.0) ? -1 : ws.order[pick];
}

// After build_support(p) [and q]: q~ at the p cells and the canonical order of the p support.
__device__ void finish_supports(WarpScratch &ws, bool have_q, int lane) {
    for (int i = lane; i < ws.n[0]; i += 32) ws.qat[i] = have_q ? support_lookup(ws, 1, ws.cell[0][i]) : 0.0;
    // canonical order: the place of a cell is the number of support cells below it (cells are unique)
    const int n = ws.n[0];
    for (int i = lane; i < n; i += 32) {
        const int c = ws.cell[0][i];
        int place = 0;
        for (int j = 0; j < n; ++j) place += ws.cell[0][j] < c;
        ws.order[place] = i;
    }
    __syncwarp();
}

#ifdef DSBD_PHASE_TIMING
#define TS(slot) do { if (threadIdx.x == 0 && writer) { unsigned long long t_; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_)); a.dbg[(int64_t)r * 256 + ts_n] = ((unsigned long long)(slot) << 48) | (t_ & 0xFFFFFFFFFFFFull); if (ts_n < 255) ++ts_n; } } while (0)
#else
#define TS(slot) do {} while (0)
#endif

// Drafts behind the first rejection of a layer of known width up to which its residual masses are computed on demand: a pass
// for that rejection and at most one for each of them, against one histogram, and a pass more where the layer ends in a residual
// draw behind a second rejection.  A histogram costs about 1.9 passes where a warp has eight tiles of a pass and 2.8 where it
// has one or two, its merge and chain being as long for few tiles.  Layers of three and four drafts, mean of the benchmark's
// distributions with as many accepts and with fewer, against a histogram for every rejection: 64 requests of 128256
// tokens up to 2 drafts 1.03 and 1.01 times as fast, up to 3 0.97 and 0.93; 160 of 32000 1.05 and 1.03, 1.00 and 0.95; 16
// of 128256 1.16 and 1.11, 1.20 and 1.14; one of 32000 1.12 and 1.07, 1.14 and 1.09.
__device__ __forceinline__ int on_demand_left(int n_tiles, int n_warps) { return n_tiles <= 2 * n_warps ? 3 : 2; }

// dynamic shared memory of k_verify: the histogram of a layer as four 32-bit arrays while it is
// being built, then (over the same bytes) this CTA's slice of the suffix sums of its p and q mass
constexpr size_t kVerifyDynSmem = kHistArrays * sizeof(uint32_t) * kHistWords;

// Two instances, with warped joints and without: neither carries the other's code, whose registers it would spill around
// (64 requests x 8 rows of 128256 with top-k 10: a call 781 us as one kernel, 772 as two; unwarped calls alike).
template <bool kWarped>
__global__ void __launch_bounds__(kVThreads, 2)
k_verify(const __grid_constant__ VerifyArgs a) {
    cg::cluster_group cluster = cg::this_cluster();
    const int n_cta = (int)cluster.num_blocks();
    const int cta_rank = (int)cluster.block_rank();
    const int r = blockIdx.x / n_cta;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const bool writer = (cta_rank == 0);
    __shared__ Shared sh;
    __shared__ double sp_live[kMaxLive], sq_live[kMaxLive];
    __shared__ int8_t st[kMaxLive * kMaxLive];     // status of the request's nodes, local index
    __shared__ NodeCache nc;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    uint32_t *hp = reinterpret_cast<uint32_t *>(dyn_smem), *hq = hp + kHistWords;     // first two digit arrays
    const HistSmem hs = hist_arrays(hp);

    // Launched with programmatic stream serialization: everything before griddepcontrol.wait overlaps the tail of the dense
    // pass ahead in the stream.  That pass lets this kernel start only when each of its blocks has waited for all earlier work,
    // so what earlier kernels and the caller left lies in L2 and may be read here, from there (ld_early: the pass's wait says
    // nothing about this SM's L1); the tile statistics only after the wait.
    const int b_lo = ld_early(a.req_beam_off + r), b_hi = ld_early(a.req_beam_off + r + 1);
    const int n_lo = ld_early(a.beam_node_off + b_lo), n_hi = ld_early(a.beam_node_off + b_hi);
    int W_min = a.W_min_r ? ld_early(a.W_min_r + r) : a.W_min;
    int W_max = a.W_max_r ? ld_early(a.W_max_r + r) : a.W_max;
    int W_nom = a.W_nom_r ? ld_early(a.W_nom_r + r) : a.W_nom;
    // per-request widths come from device memory: a width below 1 or a cap below the minimum is
    // reported (after the set-up below) and the request is not verified
    const bool bad_widths = a.check_widths && (W_min < 1 || W_max < W_min || W_nom < 1);
    if (bad_widths) { W_min = W_max = W_nom = 1; }
    double *sums_base = a.tile_sums + (int64_t)r * 2 * (a.max_m + 1) * ((int64_t)a.max_live * a.T);
    const int64_t slot_stride = (int64_t)a.max_live * a.T;
    int n_out = 0, n_pass = 0, n_hist = 0;
#ifdef DSBD_PHASE_TIMING
    int ts_n = 0;
#endif

    TS(1);
    // (a CTA may store into another's shared memory once that CTA runs: arrived here, waited for below)
    if (threadIdx.x < 20) sh.w_tot[threadIdx.x / 10][threadIdx.x % 10] = 0ull;
    cluster.barrier_arrive();
    const int n_req_nodes = n_hi - n_lo, n_trees = min(b_hi - b_lo, kMaxLive);
    const bool cached = !a.select_mode && n_req_nodes <= kCacheNodes && a.gamma < 256;
    if (!a.select_mode) {
        const int n_req = n_req_nodes;
        const int cw = cta_rank * kVWarps + warp, ncw = n_cta * kVWarps;
        // Small requests (as many nodes as the cache holds): every CTA of the cluster keeps the request's nodes in shared memory and computes all of
        // their scores itself; the log-sum-exps, shared out over the cluster's warps, are stored into every
        // CTA's copy.  One cluster barrier instead of three and no pass through global memory between them, and what
        // the caller gave is read while the dense pass drains: 5.6 us instead of 8.5 (4 beams of 4 nodes, V = 32000),
        // 9 instead of 15 with 84 nodes.  Node i is thread i's.
        int par = -1, tok = -1;
        float zp_tok = 0.f, zq_tok = 0.f;
        if (cached) {
            if ((int)threadIdx.x < n_trees) nc.root[threadIdx.x] = ld_early(a.beam_node_off + b_lo + threadIdx.x);
            const int i = threadIdx.x, n = n_lo + i;
            if (i < n_req) {
                par = ld_early(a.parent + n);
                if (par >= 0) {
                    tok = ld_early(a.token + n);
                    if (par < n_lo || par >= n) { if (writer) report(a.status, DSBD_DEV_BAD_FOREST); tok = -2; }
                    else if (tok < 0 || tok >= a.V) { if (writer) report(a.status, DSBD_DEV_BAD_TOKEN); tok = -2; }
                    else {
                        zp_tok = ld_early(a.zp + (int64_t)par * a.stride + tok);
                        zq_tok = ld_early(a.zq + (int64_t)par * a.stride + tok);
                    }
                }
                nc.parent[i] = (int16_t)((par >= n_lo && par < n) ? par - n_lo : par < 0 ? -1 : -2);
            }
        }
        cluster.barrier_wait();
        asm volatile("griddepcontrol.wait;" ::: "memory");
        TS(13);
        // ---- log-sum-exp of every row of the request from the dense pass's tile statistics ----
        for (int task = cw; task < 2 * n_req; task += ncw) {
            const int model = task / n_req, row = n_lo + (task - model * n_req);
            const double v = row_lse(a.stats + ((int64_t)model * a.N + row) * a.T, a.T, a.inv_tau, lane);
            if (cached && lane < n_cta)
                cluster.map_shared_rank(model ? nc.lse_q : nc.lse_p, lane)[row - n_lo] = v;
            if (lane == 0) {
                a.lse_w[(int64_t)model * a.N + row] = v;
                float *o = model ? a.out.lse_q : a.out.lse_p;
                if (o) o[row] = (float)v;
            }
        }
        TS(14);
        if (cached) {
            cluster.sync();
            // ---- log-prob of every draft token given its parent, then every node sums its path to the root ----
            double *slp = reinterpret_cast<double *>(hp), *slq = slp + kCacheNodes;     // (the histogram arrays are idle)
            const int i = threadIdx.x;
            if (i < n_req) {
                double lp = 0.0, lq = 0.0;
                if (tok == -2) lp = lq = -INFINITY;
                else if (tok >= 0) {
                    lp = (double)zp_tok * a.inv_tau - nc.lse_p[par - n_lo];
                    lq = (double)zq_tok * a.inv_tau - nc.lse_q[par - n_lo];
                }
                slp[i] = lp; slq[i] = lq;
            }
            __syncthreads();
            if (i < b_hi - b_lo && a.beam_node_off[b_lo + i] < n_hi) {
                const int root = a.beam_node_off[b_lo + i];
                if (writer && a.parent[root] != -1) report(a.status, DSBD_DEV_BAD_FOREST);
                slp[root - n_lo] = (double)a.root_logp[b_lo + i];
                slq[root - n_lo] = (double)a.root_logq[b_lo + i];
            }
            __syncthreads();
            if (i < n_req) {
                double sp = 0.0, sq = 0.0;
                int dep = 0, cur = i;
                while (true) {
                    sp += slp[cur];
                    sq += slq[cur];
                    const int up = nc.parent[cur];
                    if (up < 0) break;                                       // root or malformed
                    cur = up;
                    if (++dep > a.gamma) { if (writer) report(a.status, DSBD_DEV_BAD_FOREST); break; }
                }
                nc.score_p[i] = sp; nc.score_q[i] = sq;
                nc.depth[i] = (uint8_t)min(dep, 255);
                int tree = 0;
                while (tree + 1 < n_trees && nc.root[tree + 1] <= n_lo + i) ++tree;
                nc.tree[i] = (uint8_t)tree;
                if (writer) {
                    a.score_w[n_lo + i] = sp;
                    a.score_w[a.N + n_lo + i] = sq;
                    a.depth_w[n_lo + i] = dep;
                    if (a.out.node_logp) a.out.node_logp[n_lo + i] = (float)sp;
                    if (a.out.node_logq) a.out.node_logq[n_lo + i] = (float)sq;
                }
            }
            __syncthreads();
        } else {
        __threadfence();
        cluster.sync();
        // ---- log-prob of every draft token given its parent (all nodes at once) ----
        for (int i = cta_rank * kVThreads + threadIdx.x; i < n_req; i += n_cta * kVThreads) {
            const int n = n_lo + i, par = a.parent[n];
            double lp = 0.0, lq = 0.0;
            if (par >= 0) {
                const int tok = a.token[n];
                if (par < n_lo || par >= n) {
                    report(a.status, DSBD_DEV_BAD_FOREST);
                    lp = lq = -INFINITY;
                } else if (tok < 0 || tok >= a.V) {
                    report(a.status, DSBD_DEV_BAD_TOKEN);
                    lp = lq = -INFINITY;
                } else {
                    lp = (double)a.zp[(int64_t)par * a.stride + tok] * a.inv_tau - a.lse_w[par];
                    lq = (double)a.zq[(int64_t)par * a.stride + tok] * a.inv_tau - a.lse_w[a.N + par];
                }
            }
            a.score_w[n] = lp;
            a.score_w[a.N + n] = lq;
        }
        __threadfence();
        cluster.sync();
        // ---- cumulative beam scores and depths (rank 0 of the cluster) ----
        if (writer) {
            if (n_req <= 1024) {
                // stage the per-node log-probs in shared memory (the histogram arrays are idle
                // here), then every node sums its own path to the root
                double *slp = reinterpret_cast<double *>(hp), *slq = reinterpret_cast<double *>(hq);
                for (int i = threadIdx.x; i < n_req; i += kVThreads) {
                    slp[i] = a.score_w[n_lo + i];
                    slq[i] = a.score_w[a.N + n_lo + i];
                }
                __syncthreads();
                for (int b = b_lo + (int)threadIdx.x; b < b_hi; b += kVThreads) {
                    const int root = a.beam_node_off[b];
                    if (a.parent[root] != -1) report(a.status, DSBD_DEV_BAD_FOREST);
                    slp[root - n_lo] = (double)a.root_logp[b];
                    slq[root - n_lo] = (double)a.root_logq[b];
                }
                __syncthreads();
                for (int i = threadIdx.x; i < n_req; i += kVThreads) {
                    double sp = 0.0, sq = 0.0;
                    int dep = 0, cur = i;
                    while (true) {
                        sp += slp[cur];
                        sq += slq[cur];
                        const int par = a.parent[n_lo + cur];
                        if (par < n_lo || par >= n_lo + cur) break;      // root (-1) or malformed
                        cur = par - n_lo;
                        if (++dep > a.gamma) { report(a.status, DSBD_DEV_BAD_FOREST); break; }
                    }
                    a.score_w[n_lo + i] = sp;
                    a.score_w[a.N + n_lo + i] = sq;
                    a.depth_w[n_lo + i] = dep;
                    if (a.out.node_logp) a.out.node_logp[n_lo + i] = (float)sp;
                    if (a.out.node_logq) a.out.node_logq[n_lo + i] = (float)sq;
                }
                __syncthreads();
            } else {
                for (int b = b_lo + (int)threadIdx.x; b < b_hi; b += kVThreads) {
                    const int lo = a.beam_node_off[b], hi = a.beam_node_off[b + 1];
                    for (int n = lo; n < hi; ++n) {
                        const int par = a.parent[n];
                        double sp, sq;
                        int dep = 0;
                        if (n == lo) {
                            sp = (double)a.root_logp[b];
                            sq = (double)a.root_logq[b];
                            if (par != -1) report(a.status, DSBD_DEV_BAD_FOREST);
                        } else if (par < lo || par >= n) {
                            sp = sq = -INFINITY;
                            dep = a.gamma + 1;
                        } else {
                            sp = a.score_w[par] + a.score_w[n];
                            sq = a.score_w[a.N + par] + a.score_w[a.N + n];
                            dep = a.depth_w[par] + 1;
                            if (dep > a.gamma) report(a.status, DSBD_DEV_BAD_FOREST);
                        }
                        a.score_w[n] = sp;
                        a.score_w[a.N + n] = sq;
                        a.depth_w[n] = dep;
                        if (a.out.node_logp) a.out.node_logp[n] = (float)sp;
                        if (a.out.node_logq) a.out.node_logq[n] = (float)sq;
                    }
                }
            }
        }
        __threadfence();
        cluster.sync();
        }
    } else {
        cluster.barrier_wait();
        asm volatile("griddepcontrol.wait;" ::: "memory");
    }

    // Warped layers have no step in which the cluster works together, and only rank 0 writes: the others would
    // build the same supports beside it.  (Nobody stores into their shared memory any more.)
    if (kWarped && !writer) return;

    // ---- set-up ----
    auto is_root = [&](int i) { return cached ? nc.parent[i] == -1 : a.parent[n_lo + i] < 0; };
    if (warp == 0) {
        if (lane == 0) {
            sh.err = 0; sh.done = 0; sh.n_out = 0; sh.n_fill = 0;
            sh.n_layers = sh.n_tests = sh.n_exact = sh.n_respass = 0;
            sh.n_wrapped = 0; sh.n_near = 0; sh.n_rows = 0;
            if (a.select_mode) {
                const int lo = a.live_off[r], hi = a.live_off[r + 1];
                sh.nA = hi - lo;
                // the dense pass before this kernel covered the first sel_rows list entries only
                if (sh.nA > kMaxLive || sh.nA < 0 || lo < 0 || hi > a.sel_rows) {
                    sh.err = DSBD_DEV_BAD_FOREST;
                    sh.nA = 0;
                }
                for (int i = 0; i < sh.nA; ++i)
                    if (a.live_nodes[lo + i] < 0 || a.live_nodes[lo + i] >= a.N) sh.err = DSBD_DEV_BAD_FOREST;
                if (sh.err) sh.nA = 0;
                for (int i = 0; i < sh.nA; ++i) {
                    sh.A[i] = a.live_nodes[lo + i];
                    sp_live[i] = (double)a.sel_logp[sh.A[i]];
                    sq_live[i] = (double)a.sel_logq[sh.A[i]];
                }
            } else {
                sh.nA = b_hi - b_lo;
                if (sh.nA > kMaxLive) { sh.err = DSBD_DEV_BAD_FOREST; sh.nA = 0; }
            }
        }
        __syncwarp();
        if (!a.select_mode) {
            for (int i = lane; i < sh.nA; i += 32) {
                const int root = a.beam_node_off[b_lo + i];
                sh.A[i] = root;
                sp_live[i] = cached ? nc.score_p[root - n_lo] : a.score[root];
                sq_live[i] = cached ? nc.score_q[root - n_lo] : a.score[a.N + root];
            }
            if (writer) {
                for (int l = lane; l <= a.gamma; l += 32) a.out.layer_width[(int64_t)r * (a.gamma + 1) + l] = -1;
                if (lane == 0) { a.out.l_last[r] = a.gamma + 1; a.out.out_width[r] = 0; }
            }
        }
        __syncwarp();
        if (!a.select_mode && writer)
            for (int n = n_lo + lane; n < n_hi; n += 32)
                a.out.node_status[n] = is_root(n - n_lo) ? DSBD_NODE_ACCEPTED : DSBD_NODE_UNREACHED;
    }
    // Every CTA of the cluster takes identical decisions from identical data, so each keeps its
    // own copy of the node statuses and only rank 0 writes results.
    const int n_layers = a.select_mode ? 1 : a.gamma;
    const bool st_ok = n_req_nodes <= kMaxLive * kMaxLive;
    if (!a.select_mode)
        for (int n = threadIdx.x; n < n_req_nodes && st_ok; n += blockDim.x)
            st[n] = is_root(n) ? DSBD_NODE_ACCEPTED : DSBD_NODE_UNREACHED;
    __syncthreads();
    if (!a.select_mode && !st_ok && threadIdx.x == 0) sh.err = DSBD_DEV_BAD_FOREST;
    if (bad_widths && threadIdx.x == 0) sh.err = DSBD_DEV_BAD_PARAM;
    __syncthreads();
    // node data by local index, from the cache when there is one
    auto nd_depth = [&](int i) -> int { return cached ? (int)nc.depth[i] : a.depth[n_lo + i]; };
    auto nd_parent = [&](int i) -> int { return cached ? (int)nc.parent[i] : a.parent[n_lo + i] - n_lo; };
    auto nd_score = [&](int model, int i) -> double {
        return cached ? (model ? nc.score_q[i] : nc.score_p[i]) : a.score[(int64_t)model * a.N + n_lo + i];
    };

    // per live draft of layer l: index of its parent in A, rho = p_beam/q_beam of its cell, its uniform (one warp)
    auto draft_tests = [&](int l, int m) {
        for (int i = lane; i < m; i += 32) {
            const int n = sh.S[i];
            const int pl = nd_parent(n - n_lo), par = n_lo + pl;
            int ai = 0;
            while (ai < sh.nA && sh.A[ai] != par) ++ai;
            sh.S_parent_idx[i] = ai;
            const double lp = nd_score(0, n - n_lo) - nd_score(0, pl);
            const double lq = nd_score(1, n - n_lo) - nd_score(1, pl);
            double rho;
            if (lq == -INFINITY || sh.lwq[ai] == -INFINITY)
                rho = (lp > -INFINITY && sh.lwp[ai] > -INFINITY) ? INFINITY : 0.0;
            else
                rho = exp((sh.lwp[ai] - sh.lwq[ai]) + (lp - lq));
            sh.rho[i] = rho;
            sh.uu[i] = decision_uniform(a.seed, a.step, (uint32_t)r, (uint32_t)l, 0u, (uint32_t)i);
        }
        __syncwarp();
    };

    for (int l = 1; l <= n_layers && !sh.done && !sh.err; ++l) {
        // ---- live drafts of layer l, in draw order; beam weights ----
        TS(2);
        if (warp == 0) {
            int m = 0;
            if (a.select_mode) {
                m = a.m_in[r];
                if (m < 0 || m > kMaxLive) { if (lane == 0) sh.err = DSBD_DEV_BAD_FOREST; m = 0; }
            } else {
                for (int base = 0; base < n_req_nodes; base += 32) {
                    const int n = base + lane;
                    bool live = false;
                    if (n < n_req_nodes && nd_depth(n) == l) {
                        const int pl = nd_parent(n);
                        live = pl >= 0 && st[pl] == DSBD_NODE_ACCEPTED;
                        if (!live) {
                            st[n] = DSBD_NODE_PRUNED;
                            if (writer) a.out.node_status[n_lo + n] = DSBD_NODE_PRUNED;
                        }
                    }
                    const unsigned mask = __ballot_sync(kFull, live);
                    const int pos = m + __popc(mask & ((1u << lane) - 1));
                    if (live && pos < kMaxLive) sh.S[pos] = n_lo + n;
                    m += __popc(mask);
                }
                if (m > kMaxLive) { if (lane == 0) sh.err = DSBD_DEV_BAD_FOREST; m = 0; }
                __syncwarp();
                if (a.draft_rank) {
                    // order of (draft_rank, node id), ids being ascending: a draft's place is the number before it
                    for (int i = lane; i < m; i += 32) sh.S_parent_idx[i] = a.draft_rank[sh.S[i]];
                    __syncwarp();
                    for (int i = lane; i < m; i += 32) {
                        const int key = sh.S_parent_idx[i];
                        int place = 0;
                        for (int j = 0; j < m; ++j) place += sh.S_parent_idx[j] < key || (j < i && sh.S_parent_idx[j] == key);
                        sh.acc[place] = sh.S[i];
                    }
                    __syncwarp();
                    for (int i = lane; i < m; i += 32) sh.S[i] = sh.acc[i];
                }
            }
            __syncwarp();
            if (lane == 0) {
                sh.m = m;
                sh.s_arr[0] = 0.0;
                sh.c_arr[1] = 1.0;
                sh.chain_len = 0;          // c_{j+1} is known for j = 1..chain_len
                sh.next_i = sh.count = 0;
                sh.run_j = 1;
                sh.bank = l & 1;
            }
        } else if (warp <= 2) {
            live_weights(a, sh, warp - 1, warp == 1 ? sp_live : sq_live, lane, cached ? &nc : nullptr, n_lo);
        } else {
            uint4 *words = reinterpret_cast<uint4 *>(hp);
            for (int i = threadIdx.x - 96; i < kHistArrays * kHistWords / 4; i += kVThreads - 96) words[i] = make_uint4(0, 0, 0, 0);
        }
        __syncthreads();
        const int m = sh.m;
        bool looked_up = false, on_demand = false;
        TS(3);

        // The accept loop (lane 0 of warp 0), from draft sh.next_i on.  on_demand: ends with sh.need_exact = 1 after a
        // rejection whose residual mass c_{j+1} is not known yet.
        auto accept_loop = [&](int W, bool on_demand) {
            int i = sh.next_i, count = sh.count, j = sh.run_j, tests = 0, near = 0, need = 0;
            for (; i < m && count < W && !need; ++i) {
                const int n = sh.S[i];
                const double rho = sh.rho[i];
                double ratio;
                if (j == 1) ratio = rho;
                else ratio = fmax(rho - sh.s_arr[j - 1], 0.0) / sh.c_arr[j];
                if (ratio > 1.0) ratio = 1.0;
                const double u = sh.uu[i];
                ++tests;
                near += fabs(u - ratio) < 1e-5;
                if (u <= ratio) {
                    st[n - n_lo] = DSBD_NODE_ACCEPTED;
                    if (writer) a.out.node_status[n] = DSBD_NODE_ACCEPTED;
                    sh.acc[count++] = n;
                    j = 1;
                } else {
                    st[n - n_lo] = DSBD_NODE_REJECTED;
                    if (writer) a.out.node_status[n] = DSBD_NODE_REJECTED;
                    // an empty residual means p' == q_beam: the rejected draft lay outside the
                    // support of q_beam, there is nothing to subtract and p' stays
                    if (on_demand && j > sh.chain_len) { sh.s_arr[j] = sh.s_arr[j - 1] + sh.c_arr[j]; need = 1; }
                    else if (j <= sh.chain_len && sh.c_arr[j + 1] > 0.0) ++j;
                }
            }
            sh.next_i = i;
            sh.count = count;
            sh.run_j = j;
            sh.n_tests += tests;
            sh.n_near += near;
            sh.need_exact = need;
        };
        constexpr bool warped = kWarped;
        WarpScratch &wsup = *reinterpret_cast<WarpScratch *>(hq);       // the histogram arrays are idle when warped
        if (warped) {
            // ---- supports of T o p_beam and T o q_beam, then the whole chain on <= 64 cells ----
            if (!sh.err) {
                // the first half of the warps builds the support of p, the second that of q, side by side
                const int half = warp / (kHalf / 32);
                const int e_half = build_support<kHalf>(a, sh, half, hp, hq);
                if (e_half && (threadIdx.x & (kHalf - 1)) == 0) wsup.tmp[half].err = e_half;
                __syncthreads();
                const int e = wsup.tmp[0].err ? wsup.tmp[0].err : wsup.tmp[1].err;
                if (e) { if (threadIdx.x == 0) sh.err = e; }
                else if (warp == 0) {
                    finish_supports(wsup, true, lane);
                    // rho of every live draft from the warped joints
                    if (!a.select_mode) {
                        draft_tests(l, m);
                        for (int i = lane; i < m; i += 32) {
                            const int cell = sh.S_parent_idx[i] * a.V + a.token[sh.S[i]];
                            const double pw = support_lookup(wsup, 0, cell), qw = support_lookup(wsup, 1, cell);
                            sh.rho[i] = qw > 0.0 ? pw / qw : (pw > 0.0 ? INFINITY : 0.0);
                        }
                    }
                    // c_{j+1} = F(s_j) over the p support, lanes over cells
                    // (every lane keeps its at most two cells and the running s, c in registers)
                    const int ns = wsup.n[0];
                    const double p0 = lane < ns ? wsup.prob[0][lane] : 0.0, q0 = lane < ns ? wsup.qat[lane] : 0.0;
                    const double p1 = lane + 32 < ns ? wsup.prob[0][lane + 32] : 0.0;
                    const double q1 = lane + 32 < ns ? wsup.qat[lane + 32] : 0.0;
                    double s_prev = 0.0, c_cur = 1.0;
                    for (int j = 1; j <= m; ++j) {
                        const double s_j = s_prev + c_cur;
                        double acc = fmax(p0 - s_j * q0, 0.0);
                        if (lane + 32 < ns) acc += fmax(p1 - s_j * q1, 0.0);
                        acc = warp_sum(acc);
                        if (lane == 0) { sh.s_arr[j] = s_j; sh.c_arr[j + 1] = acc; sh.chain_len = j; }
                        s_prev = s_j;
                        c_cur = acc;
                        if (!(acc > 0.0)) break;
                    }
                    __syncwarp();
                }
            }
            __syncthreads();
        } else if (m >= 1 && !sh.err && !a.select_mode && (m <= W_min || W_max <= W_min)) {
            // ---- the width is W_min whatever the residual masses are (W~ <= m): the drafts are tested at once.  Up to
            // the first rejection that takes no pass over the rows at all, and every rejection one pass, without a histogram,
            // whose sums also serve the completion draw.  With more drafts behind the first rejection (on_demand_left) the
            // histogram is the better way.  (Two live rows of 128256, 4 CTAs: a layer of accepted drafts 5 us instead of 38; a
            // rejection 16 instead of 37.  Calls, W_min = 2: 64 requests x 8 rows 978 -> 907 us, 16 ragged requests 222 -> 164,
            // one request of V = 32000 61 -> 53.) ----
            if (warp == 0) {
                draft_tests(l, m);
                const int W = W_min < W_max ? W_min : W_max;
                int first = m;                         // the first rejection
                for (int base = 0; base < m && first == m; base += 32) {
                    const int i = base + lane;
                    const unsigned rejects = __ballot_sync(kFull, i < m && sh.uu[i] > fmin(sh.rho[i], 1.0));
                    if (rejects) first = base + __ffs(rejects) - 1;
                }
                if (lane == 0) {
                    sh.on_demand = first >= W || m - 1 - first <= on_demand_left(sh.nA * a.T, n_cta * kVWarps);
                    sh.need_exact = 0;
                    if (sh.on_demand) accept_loop(W, true);
                }
            }
            __syncthreads();
            on_demand = sh.on_demand;
            while (on_demand && sh.need_exact) {
                const int j = sh.run_j;
                const int halves = j == 1 ? item_halves(sh.nA * a.T, n_cta * kVWarps) : 1;   // (slot 0 has room for half tiles)
                const float half_bin = 0.5f / (float)((double)kBins / log2((double)(m > 2 ? m : 2)));
                const double c_next = exact_pass(a, sh, sh.s_arr[j], sums_base + ((int64_t)sh.bank * (a.max_m + 1) + (j == 1 ? 0 : j)) * slot_stride,
                                                 j == 1, half_bin, halves, true, n_pass++);
                if (threadIdx.x == 0) {
                    if (j == 1) sh.halves = halves;
                    sh.c_arr[j + 1] = c_next;
                    sh.chain_len = j;
                    if (c_next > 0.0) sh.run_j = j + 1;
                    accept_loop(W_min < W_max ? W_min : W_max, true);
                }
                __syncthreads();
            }
        }
        if (m >= 1 && !sh.err && !warped && !on_demand) {
            // ---- one pass: ratio histogram of the layer over the live rows ----
            const double top = log2((double)(m > 2 ? m : 2));          // s_j <= j <= m
            const float binscale = (float)((double)kBins / top);
            // (counted by histograms, not by layers: the other bank is cleared between the barriers of this one)
            const int bank = n_hist++ & 1;
            unsigned long long *tot = sh.w_tot[bank];
            const int halves = item_halves(sh.nA * a.T, n_cta * kVWarps);
            histogram_pass(a, sh, binscale, hs, sums_base + ((int64_t)sh.bank * (a.max_m + 1)) * slot_stride, cta_rank,
                           n_cta, halves, tot);
            __syncthreads();
            hist_fold_over(cluster, hs, tot, n_cta);
            TS(4);
            cluster.sync();                            // every CTA's histogram is complete
            TS(6);
            if (threadIdx.x < 10) sh.w_tot[bank ^ 1][threadIdx.x] = 0ull;     // the next layer's; nobody adds to it before
                                                       // the barrier below
            hist_merge(cluster, hs, sh, cta_rank, n_cta);
            TS(7);
            cluster.sync();                            // every slice of the suffix sums is complete
            TS(5);
            if (threadIdx.x == 32) sh.halves = halves;
            if (warp == 1 && !a.select_mode) draft_tests(l, m);
            // lane c of warp 0: mass of the bins above CTA c's slice
            unsigned long long above_p = 0ull, above_q = 0ull;
            double n_cells = 0.0;
            bool wrapped = false;
            const int slice = kBins / n_cta;
            if (warp == 0) {
                const unsigned long long own_p = lane < n_cta ? sh.slice_p[lane] : 0ull, own_q = lane < n_cta ? sh.slice_q[lane] : 0ull;
                above_p = own_p; above_q = own_q;
#pragma unroll
                for (int o = 1; o < 16; o <<= 1) {
                    const unsigned long long tp = __shfl_down_sync(kFull, above_p, o), tq = __shfl_down_sync(kFull, above_q, o);
                    if (lane + o < 32) { above_p += tp; above_q += tq; }
                }
                // what all threads added, by their floating-point sums, minus what the words hold.  Without a wrap
                // that is rounding: half a unit for each cell and 2^-20 of the mass (16 cells in a float sum), less
                // than 2^26 units; a wrap lowers the words by 2^32
                wrapped = (long long)(tot[6] - __shfl_sync(kFull, above_p + above_q, 0)) > (1ll << 31);
                above_p += tot[7] - own_p; above_q += tot[8] - own_q;
                n_cells = (double)sh.nA * (double)a.V;      // every cell of the live rows, at most
                if (lane == 0 && wrapped) ++sh.n_wrapped;
            }
            if (warp == 0) {
                if (lane < n_cta) { sh.above_p[lane] = above_p; sh.above_q[lane] = above_q; }
                __syncwarp();
            }
            // suffix sums of bin k (warp 0; the same on every lane): one word of each kind from the CTA that has it
            const int shift = 31 - __clz(slice);
            auto suffix = [&](int k, unsigned long long &P, unsigned long long &Q) {
                if (k >= kBins) { P = tot[7]; Q = tot[8]; return; }
                const int c = k >> shift;
                const uint32_t lp = cluster.map_shared_rank(hs.wp, c)[k], hi_p = cluster.map_shared_rank(hs.bp, c)[k];
                const uint32_t lq = cluster.map_shared_rank(hs.wq, c)[k], hi_q = cluster.map_shared_rank(hs.bq, c)[k];
                P = (((unsigned long long)hi_p << 32) | lp) + sh.above_p[c];
                Q = (((unsigned long long)hi_q << 32) | lq) + sh.above_q[c];
            };

            int j0 = 1;
            while (j0 <= m) {
                if (warp == 0) {
                    int j = j0;
                    int need = 0;
                    double s_j = sh.s_arr[j - 1], c_j = sh.c_arr[j];
                    for (; j <= m; ++j) {
                        s_j += c_j;
                        if (lane == 0) { sh.s_arr[j] = s_j; sh.chain_len = j; }
                        double c_next;
                        // every partial sum of the histogram is off by at most half a unit per cell
                        const double fix_err = n_cells * (0.5 * kUnfix) * (1.0 + s_j);
                        if (wrapped) { need = 1; break; }                // a wrapped word: exact passes only
                        unsigned long long P[2], Q[2];
                        if (j == 1) {
                            P[0] = __shfl_sync(kFull, above_p, 0) + sh.slice_p[0];
                            Q[0] = __shfl_sync(kFull, above_q, 0) + sh.slice_q[0];
                            c_next = ((double)P[0] - (double)Q[0]) * kUnfix;
                            if (fix_err > kErrTol) { need = 1; break; }
                        } else {
                            // (up to s = 64 the bin found is off by at most 9e-7 of an edge: the logarithm's last place 3.3e-7, s as a
                            // float 0.6e-7, the product with binscale 5e-7; an edge by 6e-7.  The bracket below takes the edges
                            // 2e-6 wider.  Approximate logarithm and exponential, reciprocals for the division: 1 us less, 1.6e-6)
                            int k = (int)(log2f((float)s_j) * binscale);
                            if (k < 0) k = 0;
                            if (k >= kBins) { need = 1; break; }     // cannot happen for s_j <= m
                            suffix(k, P[0], Q[0]);
                            suffix(k + 1, P[1], Q[1]);
                            const double Pa = (double)P[1] * kUnfix, Qa = (double)Q[1] * kUnfix;
                            const double Pk = (double)(P[0] - P[1]) * kUnfix;
                            const double Qk = (double)(Q[0] - Q[1]) * kUnfix;
                            const double r_lo = (double)exp2f((float)k / binscale) * (1.0 - 2e-6);
                            const double r_hi = (double)exp2f((float)(k + 1) / binscale) * (1.0 + 2e-6);
                            const double lo_b = fmax(Pk - s_j * Qk, 0.0);
                            double q_hi = (Pk - r_lo * Qk) / (r_hi - r_lo);
                            q_hi = fmin(fmax(q_hi, 0.0), Qk);
                            const double hi_b = fmax(q_hi * (r_hi - s_j), lo_b);
                            // the midpoint of the bracket is used: half its width plus the fixed-point term
                            if (0.5 * (hi_b - lo_b) + fix_err > kErrTol) { need = 1; break; }
                            c_next = fmax(Pa - s_j * Qa, 0.0) + 0.5 * (lo_b + hi_b);
                        }
                        if (lane == 0) sh.c_arr[j + 1] = c_next;
                        c_j = c_next;
                        if (!(c_next > 0.0)) { j = m; }               // chain exhausted: stop walking
                    }
                    if (lane == 0) {
                        sh.need_exact = need;
                        sh.chain_pos = need ? j : m + 1;
                    }
                }
                __syncthreads();
                if (!sh.need_exact) break;
                const int j = sh.chain_pos;
                if (threadIdx.x == 0) ++sh.n_exact;
                // (at j = 1 these are the sums that the histogram pass left in slot 0)
                double *sums = sums_base + ((int64_t)sh.bank * (a.max_m + 1) + (j == 1 ? 0 : j)) * slot_stride;
                if (j == 1 && threadIdx.x == 0) sh.halves = 1;
                const double c_next = exact_pass(a, sh, sh.s_arr[j], sums, false, 0.f, 1, true, n_pass++);
                if (threadIdx.x == 0) sh.c_arr[j + 1] = c_next;
                __syncthreads();
                if (!(sh.c_arr[j + 1] > 0.0)) break;
                j0 = j + 1;
            }
            cluster.barrier_arrive();                  // this CTA has done with the others' slices
            looked_up = true;
        }
        __syncthreads();

        TS(8);
        // ---- width and accept loop (warp 0) ----
        if (warp == 0 && !sh.err) {
            int W = W_min < W_max ? W_min : W_max;
            if (!on_demand) {
                // alpha_j = 1 - c_{j+1}/c_j; once a residual has no mass every later alpha is 1
                for (int j = 1 + lane; j <= m; j += 32) {
                    double al = 1.0;
                    if (j <= sh.chain_len && sh.c_arr[j] > 0.0 && sh.c_arr[j + 1] > 0.0)
                        al = fmin(fmax(1.0 - sh.c_arr[j + 1] / sh.c_arr[j], 0.0), 1.0);
                    sh.alpha[j] = al;
                }
                __syncwarp();
                // (the verification only needs W~ up to W_max and can stop at the first tail below the
                // threshold; dsbd_select_width returns the whole tail)
                const int wt = width_rule(sh, m, a.thresh, lane, a.select_mode ? -1 : W_max);
                W = wt > W_min ? wt : W_min;
                if (W > W_max) W = W_max;
            }
            if (a.select_mode) {
                if (writer && lane == 0) {
                    a.width_out[r] = W;
                    if (a.alpha_out)
                        for (int j = 0; j < m && j < a.out_stride; ++j)
                            a.alpha_out[(int64_t)r * a.out_stride + j] = (float)sh.alpha[j + 1];
                    if (a.tail_out)
                        for (int K = 0; K <= m && K < a.out_stride; ++K)
                            a.tail_out[(int64_t)r * a.out_stride + K] = (float)sh.tail[K];
                }
                if (lane == 0) sh.done = 1;
            } else if (lane == 0) {
                if (writer) a.out.layer_width[(int64_t)r * (a.gamma + 1) + (l - 1)] = W;
                if (!on_demand) accept_loop(W, false);
                const int count = sh.count, j = sh.run_j;
                for (int i = 0; i < m; ++i)
                    if (st[sh.S[i] - n_lo] == DSBD_NODE_UNREACHED) {
                        st[sh.S[i] - n_lo] = DSBD_NODE_CUT;
                        if (writer) a.out.node_status[sh.S[i]] = DSBD_NODE_CUT;
                    }
                sh.W = W;
                if (m >= 1 && (!on_demand || sh.chain_len > 0)) sh.n_rows += sh.nA;
                ++sh.n_layers;
                // a residual draw at run position j needs tile sums (a layer of known width has them)
                sh.res_j = (count < W && j > 1 && !on_demand) ? j : 0;
            }
        }
        __syncthreads();

        if (looked_up) cluster.barrier_wait();         // the others have done with this CTA's slice
        TS(9);
        // ---- a residual draw locates its tile through tile sums of max(p_beam - s_{j-1} q_beam, 0) ----
        // slot 0 of the bank; in a layer of known width that of the rejection before the draw
        const int res_slot = on_demand && sh.run_j > 2 ? sh.run_j - 1 : 0;
        double *res_sums = sums_base + ((int64_t)sh.bank * (a.max_m + 1) + res_slot) * slot_stride;
        if (!a.select_mode && !sh.err && !warped && sh.res_j > 2) {   // run position 2 is served by the histogram pass
            if (threadIdx.x == 0) { ++sh.n_respass; sh.halves = 1; }
            exact_pass(a, sh, sh.s_arr[sh.res_j - 1], res_sums, false, 0.f, 1, false, n_pass++);
        }

        TS(10);
        // ---- completion of a short layer, or the next layer's input beams (warp 0) ----
        if (warp == 0 && !a.select_mode && !sh.err) {
            const int W = sh.W, count = sh.count, j = sh.run_j;
            int err = 0;
            if (count < W) {
                // accepted drafts, then the residual draw, then fills from p_beam, all independent of one another:
                // spread over lanes when the joint is warped, else over the warps of the CTA (below)
                const int cap = a.out.out_off[r + 1] - a.out.out_off[r];
                const NodeCache *cache = cached ? &nc : nullptr;
                const int n_acc = min(count, max(cap - n_out, 0));
                if (writer)
                    for (int i = lane; i < n_acc; i += 32)
                        emit_at(a, r, n_out + i, a.parent[sh.acc[i]], sh.acc[i], a.token[sh.acc[i]], DSBD_SRC_DRAFT, cache,
                                n_lo);
                n_out += n_acc;
                if (n_acc < count) err = DSBD_DEV_CAPACITY;
                const bool use_res = j > 1;
                if (warped && !err) {
                    const int want = W - count, n_draw = min(want, max(cap - n_out, 0));
                    for (int k0 = 0; k0 < n_draw; k0 += 32) {
                        const int kk = k0 + lane;
                        const double u = decision_uniform(a.seed, a.step, (uint32_t)r, (uint32_t)l, kk ? 2u : 1u,
                                                          kk ? (uint32_t)(kk - 1) : 0u);
                        int pick = draw_support(wsup, u, 0.0, lane);
                        if (k0 == 0 && use_res) {
                            const int of_res = draw_support(wsup, u, sh.s_arr[j - 1], lane);
                            if (kk == 0) pick = of_res;
                        }
                        if (kk >= n_draw) continue;
                        if (pick < 0) { err = DSBD_DEV_EXHAUSTED; continue; }
                        const int ia = wsup.cell[0][pick] / a.V, tok = wsup.cell[0][pick] - ia * a.V;
                        if (writer)
                            emit_at(a, r, n_out + kk, sh.A[ia], -1, tok, kk ? DSBD_SRC_FILL : DSBD_SRC_RESIDUAL, cache, n_lo);
                    }
                    if (__any_sync(kFull, err)) err = DSBD_DEV_EXHAUSTED;
                    else {
                        n_out += n_draw;
                        if (n_draw < want) err = DSBD_DEV_CAPACITY;
                    }
                }
                if (lane == 0) {
                    sh.done = 1;
                    if (writer) a.out.l_last[r] = l;
                    sh.n_out = n_out;
                    sh.n_fill = (!warped && !err) ? W - count : 0;
                }
            } else {
                // the accepted drafts, ascending node id, are the next layer's input beams
                int nA = 0;
                for (int base = 0; base < n_req_nodes; base += 32) {
                    const int n = base + lane;
                    const bool in = n < n_req_nodes && nd_depth(n) == l && st[n] == DSBD_NODE_ACCEPTED;
                    const unsigned mask = __ballot_sync(kFull, in);
                    const int pos = nA + __popc(mask & ((1u << lane) - 1));
                    if (in && pos < kMaxLive) {
                        sh.A[pos] = n_lo + n;
                        sp_live[pos] = nd_score(0, n);
                        sq_live[pos] = nd_score(1, n);
                    }
                    nA += __popc(mask);
                }
                if (lane == 0) sh.nA = nA;
            }
            if (lane == 0 && err) sh.err = err;
        }
        __syncthreads();
        if (writer && !a.select_mode && sh.done && sh.n_fill > 0 && !sh.err) {
            // draw f is output beam n_out + f: the residual draw at the run position where the layer ended, then the
            // fills from p_beam, each with its own uniform
            const int cap = a.out.out_off[r + 1] - a.out.out_off[r];
            const int base = sh.n_out, want = sh.n_fill, j = sh.run_j;
            const int n_draw = min(want, max(cap - base, 0));
            __syncthreads();
            for (int f = warp; f < n_draw; f += kVWarps) {
                const double u = decision_uniform(a.seed, a.step, (uint32_t)r, (uint32_t)l, f ? 2u : 1u, f ? (uint32_t)(f - 1) : 0u);
                const bool use_res = f == 0 && j > 1;
                int ia = 0;
                const int tok = draw_cell(a, sh, u, use_res, use_res ? (float)sh.s_arr[j - 1] : 0.f, res_sums, res_slot ? 1 : sh.halves, lane, &ia);
                if (tok < 0) { if (lane == 0) sh.err = DSBD_DEV_EXHAUSTED; }
                else if (lane == 0)
                    emit_at(a, r, base + f, sh.A[ia], -1, tok, f ? DSBD_SRC_FILL : DSBD_SRC_RESIDUAL, cached ? &nc : nullptr, n_lo);
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                if (!sh.err) { sh.n_out = base + n_draw; if (want > n_draw) sh.err = DSBD_DEV_CAPACITY; }
                sh.n_fill = 0;
            }
            __syncthreads();
            n_out = sh.n_out;
        }
    }

    TS(11);
    // ---- every layer passed: W_nom beams from p_beam^(gamma+1) ----
    const bool extra = writer && !a.select_mode && !sh.done && !sh.err;
    WarpScratch &wsx = *reinterpret_cast<WarpScratch *>(hq);
    int extra_err = 0;
    if (extra) {
        if (warp < 2) live_weights(a, sh, warp, warp == 0 ? sp_live : sq_live, lane, cached ? &nc : nullptr, n_lo);
        __syncthreads();
        if (kWarped) {
            extra_err = build_support<kVThreads>(a, sh, 0, hp, hq);       // one model only: by the whole CTA
            if (!extra_err && warp == 0) finish_supports(wsx, false, lane);
        }
    }
    if (extra && !kWarped) {
        // W_nom independent draws from p_beam, one warp each
        const int cap = a.out.out_off[r + 1] - a.out.out_off[r];
        const int n_draw = min(W_nom, max(cap - n_out, 0));
        if (threadIdx.x == 0) a.out.layer_width[(int64_t)r * (a.gamma + 1) + a.gamma] = W_nom;
        for (int kk = warp; kk < n_draw; kk += kVWarps) {
            const double u = decision_uniform(a.seed, a.step, (uint32_t)r, (uint32_t)(a.gamma + 1), 3u,
                                              (uint32_t)kk);
            int ia = 0;
            const int tok = draw_cell(a, sh, u, false, 0.f, nullptr, 1, lane, &ia);
            if (tok < 0) { if (lane == 0) sh.err = DSBD_DEV_EXHAUSTED; }
            else if (lane == 0)
                emit_at(a, r, n_out + kk, sh.A[ia], -1, tok, DSBD_SRC_EXTRA, cached ? &nc : nullptr, n_lo);
        }
        __syncthreads();
        if (!sh.err) {
            n_out += n_draw;
            if (W_nom > n_draw && threadIdx.x == 0) sh.err = DSBD_DEV_CAPACITY;
        }
    } else if (extra && warp == 0) {
        // independent draws from the support, one lane each
        int err = extra_err;
        if (lane == 0) a.out.layer_width[(int64_t)r * (a.gamma + 1) + a.gamma] = W_nom;
        const int cap = a.out.out_off[r + 1] - a.out.out_off[r];
        const int n_draw = err ? 0 : min(W_nom, max(cap - n_out, 0));
        for (int k0 = 0; k0 < n_draw; k0 += 32) {
            const int kk = k0 + lane;
            const double u = decision_uniform(a.seed, a.step, (uint32_t)r, (uint32_t)(a.gamma + 1), 3u,
                                              (uint32_t)kk);
            const int pick = draw_support(wsx, u, 0.0, lane);
            if (kk >= n_draw) continue;
            if (pick < 0) { err = DSBD_DEV_EXHAUSTED; continue; }
            const int ia = wsx.cell[0][pick] / a.V, tok = wsx.cell[0][pick] - ia * a.V;
            emit_at(a, r, n_out + kk, sh.A[ia], -1, tok, DSBD_SRC_EXTRA, cached ? &nc : nullptr, n_lo);
        }
        if (!extra_err) {
            if (__any_sync(kFull, err)) err = DSBD_DEV_EXHAUSTED;
            else {
                n_out += n_draw;
                if (n_draw < W_nom) err = DSBD_DEV_CAPACITY;
            }
        }
        if (lane == 0 && err) sh.err = err;
    }
    __syncthreads();
    TS(12);
    if (threadIdx.x == 0 && writer) {
        if (!a.select_mode) {
            a.out.out_width[r] = n_out;
            if (a.out.req_error) a.out.req_error[r] = sh.err;
            if (a.out.req_stats) {
                int32_t *rs = a.out.req_stats + (int64_t)DSBD_REQ_STATS * r;
                rs[0] = sh.n_layers; rs[1] = sh.n_tests; rs[2] = sh.n_exact; rs[3] = sh.n_respass;
                rs[4] = sh.n_near; rs[5] = sh.n_rows; rs[6] = sh.n_wrapped; rs[7] = n_pass - sh.n_exact - sh.n_respass;
            }
        }
        if (sh.err) report(a.status, sh.err);
    }
}

// ------------------------------------------------------------------------------ host side
struct Layout {
    size_t stats, lse, score, depth, sums, total;
    int T, max_m, max_live;
};

Layout make_layout(const dsbd_forest_t *f, int V) {
    Layout L;
    L.T = (V + kTile - 1) / kTile;
    L.max_live = f->max_req_beams > f->max_layer_nodes ? f->max_req_beams : f->max_layer_nodes;
    if (L.max_live < 1) L.max_live = 1;
    L.max_m = f->max_layer_nodes > 1 ? f->max_layer_nodes : 1;
    size_t off = 0;
    L.stats = off; off = align_up(off + sizeof(TileStat) * 2 * (size_t)f->N * L.T, 256);
    L.lse = off;   off = align_up(off + sizeof(double) * 2 * (size_t)f->N, 256);
    L.score = off; off = align_up(off + sizeof(double) * 2 * (size_t)f->N, 256);
    L.depth = off; off = align_up(off + sizeof(int32_t) * (size_t)f->N, 256);
    L.sums = off;
    off = align_up(off + sizeof(double) * (size_t)f->R * 2 * (L.max_m + 1) * (size_t)L.max_live * L.T, 256);
#ifdef DSBD_PHASE_TIMING
    off = align_up(off + sizeof(unsigned long long) * (size_t)f->R * 256, 256);
#endif
    L.total = off;
    return L;
}

int check_forest(const dsbd_forest_t *f) {
    if (!f || f->R <= 0 || f->B <= 0 || f->N <= 0 || f->max_depth < 0) return DSBD_ERR_INVALID_ARG;
    if (!f->req_beam_off || !f->beam_node_off || !f->parent || !f->token) return DSBD_ERR_INVALID_ARG;
    if (f->max_req_beams <= 0 || f->max_layer_nodes < 0) return DSBD_ERR_INVALID_ARG;
    if (f->max_req_beams > DSBD_MAX_LIVE || f->max_layer_nodes > DSBD_MAX_LIVE) return DSBD_ERR_UNSUPPORTED;
    return DSBD_OK;
}

// The widths of the width rule W_L^(l) = min(W_max, max(W_min, W~)): without per-request
// overrides a zero width or a cap below the minimum is a caller's mistake (a zero-initialised
// struct), not a setting.
int check_widths(const dsbd_verify_params_t *p) {
    if (!p->W_min_r && p->W_min < 1) return DSBD_ERR_INVALID_ARG;
    if (!p->W_max_r && p->W_max < 1) return DSBD_ERR_INVALID_ARG;
    if (!p->W_nom_r && p->W_nom < 1) return DSBD_ERR_INVALID_ARG;
    if (!p->W_min_r && !p->W_max_r && p->W_max < p->W_min) return DSBD_ERR_INVALID_ARG;
    return DSBD_OK;
}

int check_params(const dsbd_verify_params_t *p) {
    if (!p || p->V <= 0 || !(p->temperature > 0.f)) return DSBD_ERR_INVALID_ARG;
    if (p->W_min < 1 && !p->W_min_r) return DSBD_ERR_INVALID_ARG;
    if (p->top_k < 0) return DSBD_ERR_INVALID_ARG;
    if (p->top_k > 64) return DSBD_ERR_UNSUPPORTED;
    if (p->top_k == 0 && p->top_p > 0.f && p->top_p < 1.f) return DSBD_ERR_UNSUPPORTED;   // top-p needs a top-k bound
    return DSBD_OK;
}

// Cluster size: as many CTAs per request as its tile count can use, but few enough that all
// requests are resident at once (two CTAs per SM fit).
int cluster_size_for(int tiles, int R) {
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int cs = 1;
    if (tiles >= 256) cs = 16;
    else if (tiles >= 64) cs = 8;
    else if (tiles >= 32) cs = 4;
    else if (tiles >= 16) cs = 2;
    while (cs > 1 && (long long)R * cs > 2ll * sms) cs >>= 1;
    return cs;
}

int launch_verify(const VerifyArgs &args, int R, int tiles, cudaStream_t stream) {
    const auto kernel = args.top_k > 0 ? k_verify<true> : k_verify<false>;
    const int cs = cluster_size_for(tiles, R);
    if (cs > 8 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        return DSBD_ERR_CUDA;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVerifyDynSmem) != cudaSuccess)
        return DSBD_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(R * cs));
    cfg.blockDim = dim3(kVThreads);
    cfg.dynamicSmemBytes = kVerifyDynSmem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // the clusters may be set up while the dense pass before them drains.  Before griddepcontrol.wait the kernel
    // reads what the caller gave (forest, widths, logits) from L2, after it the statistics: the dense pass lets it start only
    // when all earlier work in the stream is done
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, args) == cudaSuccess ? DSBD_OK : DSBD_ERR_CUDA;
}

int stats_grid(int64_t items) {
    // enough warps to cover the items, capped at a few waves of a 148-SM part
    int64_t blocks = (items + kWarps - 1) / kWarps;
    const int64_t cap = 148 * 8 * 4;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return (int)blocks;
}

int launch_tile_stats(int64_t items, cudaStream_t stream, const float *zp, const float *zq, int64_t stride, int V, int T, int N,
                      int n_rows, const int32_t *rows, const int32_t *n_rows_dev, float k2, TileStat *stats, int one_model) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)stats_grid(items));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_tile_stats, zp, zq, stride, V, T, N, n_rows, rows, n_rows_dev, k2, stats, one_model) == cudaSuccess
               ? DSBD_OK : DSBD_ERR_CUDA;
}

}  // namespace

extern "C" size_t dsbd_verify_workspace(const dsbd_forest_t *forest, const dsbd_verify_params_t *params) {
    if (check_forest(forest) != DSBD_OK || check_params(params) != DSBD_OK) return 0;
    return make_layout(forest, params->V).total;
}

extern "C" int dsbd_verify_step(const dsbd_forest_t *f, const dsbd_verify_params_t *p,
                                const float *logits_p, const float *logits_q, int64_t row_stride,
                                const float *root_logp, const float *root_logq,
                                const dsbd_verify_out_t *out, void *workspace, size_t workspace_bytes,
                                int32_t *status, dsbd_stream_t stream_) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    int rc = check_forest(f);
    if (rc) return rc;
    rc = check_params(p);
    if (rc) return rc;
    rc = check_widths(p);
    if (rc) return rc;
    if (!logits_p || !logits_q || !root_logp || !root_logq || !out || !workspace || !status)
        return DSBD_ERR_INVALID_ARG;
    if (row_stride < p->V) return DSBD_ERR_INVALID_ARG;
    if (!out->l_last || !out->out_width || !out->out_off || !out->out_parent || !out->out_node ||
        !out->out_root_beam || !out->out_token || !out->out_logp || !out->out_logq ||
        !out->out_source || !out->node_status || !out->layer_width)
        return DSBD_ERR_INVALID_ARG;
    const Layout L = make_layout(f, p->V);
    if (workspace_bytes < L.total) return DSBD_ERR_WORKSPACE_TOO_SMALL;
    if (reinterpret_cast<uintptr_t>(workspace) & 255) return DSBD_ERR_INVALID_ARG;
    char *ws = static_cast<char *>(workspace);
    TileStat *stats = reinterpret_cast<TileStat *>(ws + L.stats);
    double *lse = reinterpret_cast<double *>(ws + L.lse);
    double *score = reinterpret_cast<double *>(ws + L.score);
    int32_t *depth = reinterpret_cast<int32_t *>(ws + L.depth);
    const double inv_tau = 1.0 / (double)p->temperature;
    const float k2 = (float)((double)kLog2e * inv_tau);

    const int64_t items = (int64_t)2 * f->N * L.T;
    if (launch_tile_stats(items, stream, logits_p, logits_q, row_stride, p->V, L.T, f->N, f->N,
                          nullptr, nullptr, k2, stats, 0) != DSBD_OK) return DSBD_ERR_CUDA;
    if (cudaGetLastError() != cudaSuccess) return DSBD_ERR_CUDA;

    VerifyArgs a = {};
    a.R = f->R; a.N = f->N; a.gamma = f->max_depth;
    a.req_beam_off = f->req_beam_off; a.beam_node_off = f->beam_node_off;
    a.parent = f->parent; a.token = f->token; a.draft_rank = f->draft_rank;
    a.V = p->V; a.T = L.T; a.k2 = k2; a.inv_tau = inv_tau; a.thresh = (double)p->thresh;
    a.W_min = p->W_min; a.W_max = p->W_max; a.W_nom = p->W_nom;
    a.W_min_r = p->W_min_r; a.W_max_r = p->W_max_r; a.W_nom_r = p->W_nom_r;
    a.seed = p->seed; a.step = p->step;
    a.top_k = p->top_k; a.top_p = (double)p->top_p;
    a.zp = logits_p; a.zq = logits_q; a.stride = row_stride;
    a.stats = stats; a.lse = lse; a.score = score; a.depth = depth;
    a.tile_sums = reinterpret_cast<double *>(ws + L.sums);
    a.max_m = L.max_m; a.max_live = L.max_live;
#ifdef DSBD_PHASE_TIMING
    a.dbg = reinterpret_cast<unsigned long long *>(ws + L.total) - (size_t)f->R * 256;
#endif
    a.out = *out; a.status = status; a.select_mode = 0; a.check_widths = 1;
    a.lse_w = lse; a.score_w = score; a.depth_w = depth;
    a.root_logp = root_logp; a.root_logq = root_logq;
    return launch_verify(a, f->R, L.max_live * L.T, stream);
}

extern "C" int dsbd_node_stats(const dsbd_forest_t *f, const dsbd_verify_params_t *p,
                               const float *logits_p, const float *logits_q, int64_t row_stride,
                               float *lse_p, float *lse_q, void *workspace, size_t workspace_bytes,
                               dsbd_stream_t stream_) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    int rc = check_forest(f);
    if (rc) return rc;
    rc = check_params(p);
    if (rc) return rc;
    if (!logits_p || !logits_q || !lse_p || !lse_q || !workspace || row_stride < p->V)
        return DSBD_ERR_INVALID_ARG;
    const Layout L = make_layout(f, p->V);
    if (workspace_bytes < L.total) return DSBD_ERR_WORKSPACE_TOO_SMALL;
    if (reinterpret_cast<uintptr_t>(workspace) & 255) return DSBD_ERR_INVALID_ARG;
    char *ws = static_cast<char *>(workspace);
    TileStat *stats = reinterpret_cast<TileStat *>(ws + L.stats);
    double *lse = reinterpret_cast<double *>(ws + L.lse);
    const double inv_tau = 1.0 / (double)p->temperature;
    const float k2 = (float)((double)kLog2e * inv_tau);
    const int64_t items = (int64_t)2 * f->N * L.T;
    if (launch_tile_stats(items, stream, logits_p, logits_q, row_stride, p->V, L.T, f->N, f->N,
                          nullptr, nullptr, k2, stats, 0) != DSBD_OK) return DSBD_ERR_CUDA;
    const int64_t warps = (int64_t)2 * f->N;
    k_row_finish<<<(unsigned)((warps + kWarps - 1) / kWarps), kThreads, 0, stream>>>(
        stats, L.T, f->N, f->N, nullptr, nullptr, inv_tau, lse, lse_p, lse_q);
    return cudaGetLastError() == cudaSuccess ? DSBD_OK : DSBD_ERR_CUDA;
}

// ---------------------------------------------------------------------------------------
// dsbd_draft_layer: a beam-sampling step of the small model is the extra layer of the
// verification on the current beams, with one model: W_S inverse-CDF draws from T o q_beam.
// One CTA per request after the dense pass over the beams' rows.  What is left is a chain of short steps on a
// few thousand numbers, so a CTA that does them alone beats the verification kernel's cluster, whose CTAs all
// repeat the chain between barriers (and which needed a launch for the root-only forest it walked): with top-k 10
// over 16 x 8 rows of 128256 the kernel takes 16 us instead of 43, unwarped over 8 x 4 rows of 32000 9 instead of 15.5.
// ---------------------------------------------------------------------------------------
namespace {
struct DraftArgs {
    VerifyArgs v;             // what the shared steps read: V, T, k2, inv_tau, seed, step, top_k, top_p, zp, stride, stats, lse
    uint32_t layer;           // layer number in the Philox counter
    const float *beam_logq;
    int W;
    const int32_t *W_r, *out_off;
    int32_t *out_parent, *out_token;
    float *out_logq;
    int32_t *req_error;
};

__global__ void __launch_bounds__(kVThreads)
k_draft(const __grid_constant__ DraftArgs d) {
    const VerifyArgs &a = d.v;
    __shared__ Shared sh;
    __shared__ double score[kMaxLive], lse[kMaxLive];
    __shared__ int s_err;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    uint32_t *hp = reinterpret_cast<uint32_t *>(dyn_smem), *hq = hp + kHistWords;
    const int r = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // (before the wait as in k_verify: what earlier work left, from L2)
    const int b_lo = ld_early(a.req_beam_off + r), o_lo = ld_early(d.out_off + r), cap = ld_early(d.out_off + r + 1) - o_lo;
    const int W = d.W_r ? ld_early(d.W_r + r) : d.W;
    int nA = ld_early(a.req_beam_off + r + 1) - b_lo, err = 0;
    if (nA > kMaxLive) { err = DSBD_DEV_BAD_FOREST; nA = 0; }
    if (threadIdx.x < nA) {
        sh.A[threadIdx.x] = b_lo + threadIdx.x;
        score[threadIdx.x] = (double)ld_early(d.beam_logq + b_lo + threadIdx.x);
    }
    if (threadIdx.x == 0) { sh.nA = nA; s_err = 0; }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int i = warp; i < nA; i += kVWarps) {
        const double v = row_lse(a.stats + (int64_t)(b_lo + i) * a.T, a.T, a.inv_tau, lane);
        if (lane == 0) { lse[i] = v; a.lse_w[b_lo + i] = v; }
    }
    __syncthreads();
    if (warp == 0) live_weights(a, sh, 0, score, lane, nullptr, 0);
    __syncthreads();
    const int n_draw = err ? 0 : min(W, max(cap, 0));
    auto emit = [&](int kk, int ia, int tok) {
        const float z = a.zp[(int64_t)(b_lo + ia) * a.stride + tok];
        d.out_parent[o_lo + kk] = b_lo + ia;
        d.out_token[o_lo + kk] = tok;
        d.out_logq[o_lo + kk] = (float)(score[ia] + ((double)z * a.inv_tau - lse[ia]));
    };
    if (a.top_k > 0) {
        WarpScratch &ws = *reinterpret_cast<WarpScratch *>(hq);
        if (!err) err = build_support<kVThreads>(a, sh, 0, hp, hq);
        if (!err && warp == 0) {
            finish_supports(ws, false, lane);
            for (int k0 = 0; k0 < n_draw; k0 += 32) {
                const int kk = k0 + lane;
                const double u = decision_uniform(a.seed, a.step, (uint32_t)r, d.layer, 3u, (uint32_t)kk);
                const int pick = draw_support(ws, u, 0.0, lane);
                if (kk >= n_draw) continue;
                if (pick < 0) { s_err = DSBD_DEV_EXHAUSTED; continue; }
                const int ia = ws.cell[0][pick] / a.V;
                emit(kk, ia, ws.cell[0][pick] - ia * a.V);
            }
        }
    } else {
        for (int kk = warp; kk < n_draw; kk += kVWarps) {
            const double u = decision_uniform(a.seed, a.step, (uint32_t)r, d.layer, 3u, (uint32_t)kk);
            int ia = 0;
            const int tok = draw_cell(a, sh, u, false, 0.f, nullptr, 1, lane, &ia);
            if (lane == 0) {
                if (tok < 0) s_err = DSBD_DEV_EXHAUSTED;
                else emit(kk, ia, tok);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!err) err = s_err;
        if (!err && n_draw < W) err = DSBD_DEV_CAPACITY;
        if (d.req_error) d.req_error[r] = err;
        if (err) report(a.status, err);
    }
}

struct DraftLayout {
    size_t stats, lse, total;
    int T;
};

bool draft_args_ok(int R, int n_beams, const dsbd_draft_params_t *p) {
    return p && R > 0 && n_beams > 0 && p->V > 0 && p->temperature > 0.f && p->n_slots > 0 &&
           p->max_req_beams > 0 && (p->W_S >= 0 || p->W_S_r) && p->layer >= 0 && p->top_k >= 0;
}

DraftLayout make_draft_layout(int n_beams, const dsbd_draft_params_t *p) {
    DraftLayout D;
    D.T = (p->V + kTile - 1) / kTile;
    D.stats = 0;
    D.lse = align_up(sizeof(TileStat) * (size_t)n_beams * D.T, 256);
    D.total = align_up(D.lse + sizeof(double) * (size_t)n_beams, 256);
    return D;
}
}  // namespace

extern "C" size_t dsbd_draft_workspace(int32_t R, int32_t n_beams, const dsbd_draft_params_t *p) {
    if (!draft_args_ok(R, n_beams, p)) return 0;
    return make_draft_layout(n_beams, p).total;
}

extern "C" int dsbd_draft_layer(int32_t R, int32_t n_beams, const int32_t *req_beam_off,
                                const dsbd_draft_params_t *p, const float *logits_q, int64_t row_stride,
                                const float *beam_logq, const int32_t *out_off, int32_t *out_parent,
                                int32_t *out_token, float *out_logq, int32_t *req_error, void *workspace,
                                size_t workspace_bytes, int32_t *status, dsbd_stream_t stream_) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (!draft_args_ok(R, n_beams, p)) return DSBD_ERR_INVALID_ARG;
    if (!req_beam_off || !logits_q || !beam_logq || !out_off || !out_parent || !out_token || !out_logq ||
        !workspace || !status || row_stride < p->V)
        return DSBD_ERR_INVALID_ARG;
    if (p->max_req_beams > DSBD_MAX_LIVE || p->top_k > 64) return DSBD_ERR_UNSUPPORTED;
    if (p->top_k == 0 && p->top_p > 0.f && p->top_p < 1.f) return DSBD_ERR_UNSUPPORTED;
    const DraftLayout D = make_draft_layout(n_beams, p);
    if (workspace_bytes < D.total) return DSBD_ERR_WORKSPACE_TOO_SMALL;
    if (reinterpret_cast<uintptr_t>(workspace) & 255) return DSBD_ERR_INVALID_ARG;
    char *ws = static_cast<char *>(workspace);
    DraftArgs d = {};
    VerifyArgs &a = d.v;
    a.R = R; a.N = n_beams;
    a.req_beam_off = req_beam_off;
    a.V = p->V; a.T = D.T;
    a.inv_tau = 1.0 / (double)p->temperature;
    a.k2 = (float)((double)kLog2e * a.inv_tau);
    a.seed = p->seed; a.step = p->step;
    a.top_k = p->top_k; a.top_p = (double)p->top_p;
    a.zp = a.zq = logits_q; a.stride = row_stride;
    TileStat *stats = reinterpret_cast<TileStat *>(ws + D.stats);
    a.stats = stats;
    a.lse = a.lse_w = reinterpret_cast<double *>(ws + D.lse);
    a.status = status;
    d.layer = (1u << 29) + (uint32_t)p->layer;
    d.beam_logq = beam_logq;
    d.W = p->W_S; d.W_r = p->W_S_r;
    d.out_off = out_off; d.out_parent = out_parent; d.out_token = out_token; d.out_logq = out_logq;
    d.req_error = req_error;

    const int64_t items = (int64_t)n_beams * D.T;
    if (launch_tile_stats(items, stream, logits_q, logits_q, row_stride, p->V, D.T, n_beams,
                          n_beams, nullptr, nullptr, a.k2, stats, 1) != DSBD_OK) return DSBD_ERR_CUDA;
    if (cudaGetLastError() != cudaSuccess) return DSBD_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)R);
    cfg.blockDim = dim3(kVThreads);
    cfg.dynamicSmemBytes = p->top_k > 0 ? kVerifyDynSmem : 0;           // the support's scratch
    cfg.stream = stream;
    if (p->top_k > 0 && cudaFuncSetAttribute(k_draft, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVerifyDynSmem) != cudaSuccess)
        return DSBD_ERR_CUDA;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;       // see launch_verify
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_draft, d) == cudaSuccess ? DSBD_OK : DSBD_ERR_CUDA;
}

// ---------------------------------------------------------------------------------------
// dsbd_node_stats_static: the same two kernels as dsbd_node_stats, with their scratch (tile
// statistics and double-precision row sums) in a fixed array that is part of the library image
// instead of a caller-supplied workspace.
// ---------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_static_scratch[DSBD_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
unsigned char *g_static_scratch_ptr[kMaxDevices];   // device address of the array, per device

// The array's name is only a host-side handle; the device address a kernel can use has to be
// asked for, once per device, while that device is current.
int static_scratch_address(unsigned char **ptr) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return DSBD_ERR_CUDA;
    unsigned char *p = __atomic_load_n(&g_static_scratch_ptr[dev], __ATOMIC_ACQUIRE);
    if (!p) {
        void *addr = nullptr;
        if (cudaGetSymbolAddress(&addr, g_static_scratch) != cudaSuccess || !addr) return DSBD_ERR_CUDA;
        p = static_cast<unsigned char *>(addr);
        __atomic_store_n(&g_static_scratch_ptr[dev], p, __ATOMIC_RELEASE);
    }
    *ptr = p;
    return DSBD_OK;
}
}  // namespace

extern "C" int dsbd_node_stats_static(const dsbd_forest_t *f, const dsbd_verify_params_t *p,
                                      const float *logits_p, const float *logits_q, int64_t row_stride,
                                      float *lse_p, float *lse_q, dsbd_stream_t stream_) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    int rc = check_forest(f);
    if (rc) return rc;
    rc = check_params(p);
    if (rc) return rc;
    if (!logits_p || !logits_q || !lse_p || !lse_q || row_stride < p->V) return DSBD_ERR_INVALID_ARG;
    // scratch this call needs: tile statistics of both models, then the double row sums
    const int T = (p->V + kTile - 1) / kTile;
    const size_t stats_bytes = align_up(sizeof(TileStat) * 2 * (size_t)f->N * T, 256);
    const size_t need = stats_bytes + sizeof(double) * 2 * (size_t)f->N;
    if (need > (size_t)DSBD_STATIC_SCRATCH_BYTES) return DSBD_ERR_WORKSPACE_TOO_SMALL;
    unsigned char *scratch = nullptr;
    rc = static_scratch_address(&scratch);
    if (rc) return rc;
    // Nothing here has to start from zero: both kernels overwrite every entry they later read.
    TileStat *stats = reinterpret_cast<TileStat *>(scratch);
    double *lse = reinterpret_cast<double *>(scratch + stats_bytes);
    const double inv_tau = 1.0 / (double)p->temperature;
    const float k2 = (float)((double)kLog2e * inv_tau);
    const int64_t items = (int64_t)2 * f->N * T;
    if (launch_tile_stats(items, stream, logits_p, logits_q, row_stride, p->V, T, f->N, f->N,
                          nullptr, nullptr, k2, stats, 0) != DSBD_OK) return DSBD_ERR_CUDA;
    const int64_t warps = (int64_t)2 * f->N;
    k_row_finish<<<(unsigned)((warps + kWarps - 1) / kWarps), kThreads, 0, stream>>>(
        stats, T, f->N, f->N, nullptr, nullptr, inv_tau, lse, lse_p, lse_q);
    return cudaGetLastError() == cudaSuccess ? DSBD_OK : DSBD_ERR_CUDA;
}

extern "C" int dsbd_select_width(const dsbd_forest_t *f, const dsbd_verify_params_t *p,
                                 const float *logits_p, const float *logits_q, int64_t row_stride,
                                 const float *node_logp, const float *node_logq,
                                 const int32_t *live_off, const int32_t *live_nodes, const int32_t *m,
                                 int32_t *width, float *alpha, float *tail, int32_t out_stride,
                                 void *workspace, size_t workspace_bytes, int32_t *status,
                                 dsbd_stream_t stream_) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    int rc = check_forest(f);
    if (rc) return rc;
    rc = check_params(p);
    if (rc) return rc;
    rc = check_widths(p);
    if (rc) return rc;
    if (!logits_p || !logits_q || !node_logp || !node_logq || !live_off || !live_nodes || !m ||
        !width || !workspace || !status)
        return DSBD_ERR_INVALID_ARG;
    if (row_stride < p->V || ((alpha || tail) && out_stride < 1)) return DSBD_ERR_INVALID_ARG;
    const Layout L = make_layout(f, p->V);
    if (workspace_bytes < L.total) return DSBD_ERR_WORKSPACE_TOO_SMALL;
    if (reinterpret_cast<uintptr_t>(workspace) & 255) return DSBD_ERR_INVALID_ARG;
    char *ws = static_cast<char *>(workspace);
    TileStat *stats = reinterpret_cast<TileStat *>(ws + L.stats);
    double *lse = reinterpret_cast<double *>(ws + L.lse);
    const double inv_tau = 1.0 / (double)p->temperature;
    const float k2 = (float)((double)kLog2e * inv_tau);

    // statistics of the live rows only; their number is live_off[R], known on the device
    const int max_rows = f->R * L.max_live < f->N ? f->R * L.max_live : f->N;
    const int64_t items = (int64_t)2 * max_rows * L.T;
    if (launch_tile_stats(items, stream, logits_p, logits_q, row_stride, p->V, L.T, f->N, max_rows,
                          live_nodes, live_off + f->R, k2, stats, 0) != DSBD_OK) return DSBD_ERR_CUDA;
    {
        const int64_t warps = (int64_t)2 * max_rows;
        k_row_finish<<<(unsigned)((warps + kWarps - 1) / kWarps), kThreads, 0, stream>>>(
            stats, L.T, f->N, max_rows, live_nodes, live_off + f->R, inv_tau, lse, nullptr, nullptr);
    }
    if (cudaGetLastError() != cudaSuccess) return DSBD_ERR_CUDA;

    VerifyArgs a = {};
    a.R = f->R; a.N = f->N; a.gamma = f->max_depth;
    a.req_beam_off = f->req_beam_off; a.beam_node_off = f->beam_node_off;
    a.parent = f->parent; a.token = f->token; a.draft_rank = f->draft_rank;
    a.V = p->V; a.T = L.T; a.k2 = k2; a.inv_tau = inv_tau; a.thresh = (double)p->thresh;
    a.W_min = p->W_min; a.W_max = p->W_max; a.W_nom = p->W_nom;
    a.W_min_r = p->W_min_r; a.W_max_r = p->W_max_r; a.W_nom_r = p->W_nom_r;
    a.seed = p->seed; a.step = p->step;
    a.top_k = p->top_k; a.top_p = (double)p->top_p;
    a.zp = logits_p; a.zq = logits_q; a.stride = row_stride;
    a.stats = stats; a.lse = lse; a.score = nullptr; a.depth = nullptr;
    a.tile_sums = reinterpret_cast<double *>(ws + L.sums);
    a.max_m = L.max_m; a.max_live = L.max_live;
#ifdef DSBD_PHASE_TIMING
    a.dbg = reinterpret_cast<unsigned long long *>(ws + L.total) - (size_t)f->R * 256;
#endif
    a.status = status; a.select_mode = 1; a.check_widths = 1;
    a.sel_logp = node_logp; a.sel_logq = node_logq;
    a.live_off = live_off; a.live_nodes = live_nodes; a.m_in = m; a.sel_rows = max_rows;
    a.width_out = width; a.alpha_out = alpha; a.tail_out = tail; a.out_stride = out_stride;
    return launch_verify(a, f->R, L.max_live * L.T, stream);
}
