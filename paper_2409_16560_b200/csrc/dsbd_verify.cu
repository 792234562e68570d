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

#include <atomic>

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

// By a whole warp (never behind a branch on the lane): the value of lane 0, for one that all lanes have.  The compiler then knows that a branch on it leaves the warp together.
// Behind a branch on a thread index, a function's argument or a word of memory it does not, and gathers the lanes anew for every
// shuffle: about 300 cycles each instead of 23, and three times the code (a warp_sum of doubles 1.5 us instead of 0.12).
__device__ __forceinline__ int uniform(int x) { return __shfl_sync(kFull, x, 0); }
__device__ __forceinline__ int warp_index() { return uniform((int)(threadIdx.x >> 5)); }

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
    const int64_t warp = (int64_t)blockIdx.x * kWarps + warp_index();
    const int64_t nwarps = (int64_t)gridDim.x * kWarps;
    if (n_rows_dev) n_rows = uniform(min(max(*n_rows_dev, 0), n_rows));
    const int64_t total = (int64_t)(one_model ? 1 : 2) * n_rows * T;
    for (int64_t item = warp; item < total; item += nwarps) {
        const int t = (int)(item % T);
        const int64_t rm = item / T;
        const int model = (int)(rm / n_rows);
        const int ri = (int)(rm % n_rows);
        const int row = rows ? uniform(rows[ri]) : ri;
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
    float top = -INFINITY;
#pragma unroll 4
    for (int t0 = 0; t0 < T; t0 += 32)
        if (t0 + lane < T) top = fmaxf(top, s[t0 + lane].mx);
    const double mx = (double)warp_max(top);
    double acc = 0.0;
    if (mx > -INFINITY)
#pragma unroll 2
        for (int t0 = 0; t0 < T; t0 += 32) {
            const TileStat x = s[min(t0 + lane, T - 1)];
            const double e = (double)x.sum * exp(((double)x.mx - mx) * inv_tau);
            if (t0 + lane < T && x.sum > 0.f) acc += e;
        }
    acc = warp_sum(acc);
    return (mx > -INFINITY) ? mx * inv_tau + log(acc) : -INFINITY;
}

// log-sum-exp of the tempered row from its tile statistics; one warp per (model, row).
__global__ void k_row_finish(const TileStat *__restrict__ stats, int T, int N, int n_rows,
                             const int32_t *__restrict__ rows, const int32_t *__restrict__ n_rows_dev,
                             double inv_tau, double *__restrict__ lse /*[2][N]*/,
                             float *__restrict__ lse_p_out, float *__restrict__ lse_q_out) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t)blockIdx.x * kWarps + warp_index();
    if (n_rows_dev) n_rows = uniform(min(max(*n_rows_dev, 0), n_rows));
    if (warp >= (int64_t)2 * n_rows) return;
    const int model = (int)(warp / n_rows);
    const int ri = (int)(warp % n_rows);
    const int row = rows ? uniform(rows[ri]) : ri;
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
    int R, B, N, gamma;
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

constexpr int kBins = 4096;
constexpr int kOverSlots = 256;                   // copies of the last bin (rho beyond the last edge): one per
                                                  // warp and half-warp lane, so that none collects enough to wrap

// The bins of a layer of m drafts: scale bins to a power of two; the upper edge of a bin over 2^(k / scale), and one over the width
// of a bin over the same, both with the edges' tolerance (2e-6).
struct BinEdges { float scale; double inv_scale, hi, inv_width; };
constexpr double kEdgeTol = 2e-6;

struct Shared {
    int nA, m, W, count, chain_len, err;         // m: -1 if too many
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
    int n_draw;                             // completion draws of the request
    int empty_tree;                         // some tree of the request has no nodes
    int on_demand, next_i;                  // a layer of known width: its passes are made when the accept loop asks
    // sums of an exact pass, in units of 2^-60, 2^-120 (what the first leaves) and 2^-44 (q): of this CTA's warps; of every
    // CTA, two passes in turn
    long long warp_part[3][kVWarps], part[2][3][16];
    int n_out;                              // output beams
    int n_layers, n_tests, n_exact, n_respass;
    int n_near, n_rows;                     // accept tests inside the 1e-5 tie band; live rows of layers that looked into them
    unsigned long long wtot[2][kVWarps], over[2][kOverSlots / 32];   // mass (p, q) of every warp's bins and copies of the last bin
    unsigned long long added;               // mass that this CTA's histogram pass added (p and q), by floating-point sums
    int n_wrapped;                          // layers where one did
#ifdef DSBD_PHASE_TIMING
    unsigned long long *ts, *ts_end;        // next and last time stamp of the CTA that writes
#endif
    double rho[kMaxLive], lq[kMaxLive];     // per live draft: p_beam/q_beam (before: its log-prob under p); log-prob under q
    double uu[kMaxLive];                    // and its uniform
    BinEdges bins[kMaxLive + 1];            // by m
};

#ifdef DSBD_PHASE_TIMING
#define TS(slot) do { if (threadIdx.x == 0 && sh.ts) { unsigned long long t_; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_)); *sh.ts = ((unsigned long long)(slot) << 48) | (t_ & 0xFFFFFFFFFFFFull); if (sh.ts < sh.ts_end) ++sh.ts; } } while (0)
#else
#define TS(slot) do {} while (0)
#endif

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

// A value that the compiler takes for a new one: keeps it from making copies of a loop for its first round or for a flag.
__device__ __forceinline__ void one_copy(int &x) { asm volatile("" : "+r"(x)); }

// Inverse-CDF search over n weights in shared memory, by one warp.  Returns the first index whose running sum reaches the
// target and leaves in target what that takes off the sum before it; if rounding leaves the target beyond the total, the last
// index with mass (open: n, and the total taken off, where more weights follow).  -1 if there is no mass at all.  The target
// is target * total when of_total.  Every round cuts the range by 32: a lane sums its share, the lanes' sums are
// scanned, one lane is chosen.
// One copy for all searches of a kernel, over weights that its callers have put side by side: text is what a draw waits for
// (a search of its own in global memory for each kind of weight, unrolled: 24 KB, and 17 KB for the search inside a tile).
__device__ __noinline__ int locate(const double *w, int n, double &target, bool of_total, bool open, int lane) {
    int lo = 0, len = uniform(n), scale = uniform(of_total), go_on = uniform(open);
#pragma unroll 1
    while (true) {
        one_copy(scale); one_copy(go_on);
        const int per = (len + 31) >> 5, i0 = lo + lane * per, i1 = min(i0 + per, lo + len);
        double v = 0.0;
#pragma unroll 1
        for (int i = i0; i < i1; ++i) v += w[i];
        const double incl = warp_scan(v, lane);
        const double total = __shfl_sync(kFull, incl, 31);
        if (scale) target *= total;
        scale = 0;
        const unsigned pos = __ballot_sync(kFull, v > 0.0);
        const unsigned hits = __ballot_sync(kFull, v > 0.0 && incl >= target);
        if (!hits && go_on) { target -= total; return n; }
        if (!pos) return -1;
        const int l = hits ? __ffs(hits) - 1 : 31 - __clz(pos);
        target -= __shfl_sync(kFull, incl - v, l);
        lo += l * per;
        len = min(per, len - l * per);
        go_on = 0;
        if (per == 1) return lo;
    }
}

// Inverse-CDF search inside one tile of row `row` (and its q row when s > 0), by one warp: the first
// token whose running mass reaches `target`, else the last token with mass.  -1: no mass.
// mass: 33 x 32 words of shared memory.  All sectors of the tile are asked for at once; then the lanes take the tokens side by side,
// and each sums 32 consecutive ones.
constexpr int kTokWords = 33 * 32;
__device__ __noinline__ int locate_token(const float *__restrict__ rp, const float *__restrict__ rq, int V, float k2,
                                         int t, const RowOff ro, float s, double target, int lane, float *mass) {
    const int e0 = t * kTile, n = min(kTile, V - e0);
    rp += e0; rq += e0;
    const bool res = uniform(s > 0.f);
    float first_of[8];                               // (of a sector; all in flight together)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int e = (i * 32 + lane) * 8;
        first_of[i] = e < n ? __ldg(rp + e) : 0.f;
        first_of[4 + i] = res && e < n ? __ldg(rq + e) : 0.f;
    }
    asm volatile("" :: "f"(first_of[0]), "f"(first_of[1]), "f"(first_of[2]), "f"(first_of[3]), "f"(first_of[4]), "f"(first_of[5]),
                       "f"(first_of[6]), "f"(first_of[7]));
#pragma unroll 1
    for (int i0 = 0; i0 < 32; i0 += 8) {
        float zp[8], zq[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int e = (i0 + i) * 32 + lane;
            zp[i] = e < n ? __ldg(rp + e) : -INFINITY;
            zq[i] = res && e < n ? __ldg(rq + e) : -INFINITY;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float q, m = exp2f(fmaf(zp[i], k2, ro.bp)) * ro.cp;
            if (res) m = cell_mass(zp[i], zq[i], k2, ro, s, &q);
            mass[(i0 + i) * 33 + lane] = m;
        }
    }
    __syncwarp();
    double v = 0.0;
#pragma unroll 8
    for (int i = 0; i < 32; ++i) v += (double)mass[lane * 33 + i];
    int first = 0;                                               // the hit lane's first token
#pragma unroll 1
    for (int level = 0; ; ++level) {
        one_copy(level);
        const double incl = warp_scan(v, lane);
        const unsigned pos = __ballot_sync(kFull, v > 0.0);
        if (!pos) return -1;
        const unsigned hits = __ballot_sync(kFull, v > 0.0 && incl >= target);
        const int l = hits ? __ffs(hits) - 1 : 31 - __clz(pos);
        if (level) return first + l;
        target -= __shfl_sync(kFull, incl - v, l);
        first = e0 + l * 32;
        v = (double)mass[l * 33 + lane];
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
    int rank[kCacheNodes];                // draft_rank, where the caller gave one
    uint8_t live[kCacheNodes];            // index of an accepted node among the live rows
};

// Writes output beam number `index` of request r (the caller has checked the slot range).  nc: the
// request's node cache or nullptr; n_lo: first node of the request.
__device__ __forceinline__ void emit_at(const VerifyArgs &a, int r, int index, int parent, int node, int tok, int source,
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
#pragma unroll 1
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
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 32)
        if (const int i = i0 + lane; i < n) mx = fmax(mx, s[i]);
    mx = warp_max(mx);
    double t = 0.0;
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 32)
        if (const int i = i0 + lane; i < n) t += exp(s[i] - mx);
    t = warp_sum(t);
    const double lt = log(t);
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 32)
        if (const int i = i0 + lane; i < n) out[i] = (s[i] - mx) - lt;
    __syncwarp();
}

// The weights of one model (0: p, 1: q) over the live set: softmax of the cumulative scores over A (Eq. 1 factorised),
// by one warp; the two models' warps work side by side.
// lse: the model's log-sum-exps by node.
__device__ __forceinline__ void live_weights(Shared &sh, int model, const double *scores, const double *lse, int lane) {
    double *lw = model ? sh.lwq : sh.lwp;
    const int nA = uniform(sh.nA);
    log_softmax_warp(scores, nA, lane, lw);
#pragma unroll 1
    for (int i0 = 0; i0 < nA; i0 += 32) {
        const int i = i0 + lane;
        if (i >= nA) continue;
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
    // With 1 - alpha_j = c_{j+1} / c_j and c_1 = 1: P(n, 0) = prod_{j<=n}(1 - alpha_j) = c_{n+1}, and the first accept is the i-th
    // draft's with alpha_i prod_{j<i}(1 - alpha_j) = c_i - c_{i+1}.  No residual mass from some c on: every later alpha is 1
    const int len = uniform(sh.chain_len);
#pragma unroll 1
    for (int i0 = 0; i0 <= m; i0 += 32) {
        const int i = min(i0 + lane, m);                     // (the last one more than once)
        auto mass = [&](int j) { return j <= len + 1 && sh.c_arr[j] > 0.0 ? sh.c_arr[j] : 0.0; };
        const double c = mass(i + 1);
        sh.col_a[i] = c;
        if (i > 0) sh.first[i] = fmax(mass(i) - c, 0.0);
    }
    if (lane == 0) sh.tail[0] = 1.0;
    __syncwarp();
    double *prev = sh.col_a, *cur = sh.col_b;
    double below = 0.0;
#pragma unroll 1
    for (int k = 0; k <= m; ++k) {
        // prev = P(., k); record tail
        below += prev[m];
        if (lane == 0) sh.tail[k + 1] = 1.0 - below;
        if (k == m) break;
        // tails only fall: past the first one below the threshold, or past the cap, nothing changes W
        if (k_stop >= 0 && (uniform(1.0 - below < thresh) || k + 1 >= k_stop)) {
#pragma unroll 1
            for (int K0 = k + 2; K0 <= m + 1; K0 += 32)
                if (K0 + lane <= m + 1) sh.tail[K0 + lane] = 0.0;
            break;
        }
#pragma unroll 1
        for (int n0 = 0; n0 <= m; n0 += 32) {
            const int n = n0 + lane;
            double acc = 0.0;
#pragma unroll 4
            for (int i = 1; i <= m; ++i)
                if (i <= n && n <= m) acc += sh.first[i] * prev[n - i];
            if (n <= m) cur[n] = n > k ? acc : 0.0;         // P(n, k+1), zero for n < k+1
        }
        __syncwarp();
        double *tmp = prev; prev = cur; cur = tmp;
    }
    __syncwarp();
    int wt = 0;
#pragma unroll 1
    for (int K0 = 0; K0 <= m; K0 += 32) {
        const unsigned reach = __ballot_sync(kFull, K0 + lane <= m && sh.tail[min(K0 + lane, m)] >= thresh);
        if (reach) wt = K0 + 31 - __clz(reach);
    }
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
constexpr int kHistWords = kBins + kOverSlots + 16;  // bins 0..kBins-1, the copies of bin kBins, spare words
static_assert(kHistWords % 4 == 0, "the arrays that share this memory need 16-byte alignment");
constexpr float kFix = 17592186044416.f;          // 2^44
constexpr double kUnfix = 1.0 / 17592186044416.0;
constexpr double kErrTol = 2.5e-7;                // error bound of F(s) above which it is recomputed exactly
constexpr int kHistArrays = 4;
constexpr uint32_t kWrapped = 0x80000000u;
struct HistSmem { uint32_t *wp, *wq, *bp, *bq; };

__device__ __forceinline__ HistSmem hist_arrays(uint32_t *base) {
    return HistSmem{base, base + kHistWords, base + 2 * kHistWords, base + 3 * kHistWords};
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Shared memory of CTA c of the cluster: the address of what p is here, and 16 bytes from there.
__device__ __forceinline__ uint32_t cluster_address(const void *p, int c) {
    uint32_t to;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(c));
    return to;
}
__device__ __forceinline__ uint4 ld_cluster(uint32_t at) {
    uint4 v;
    asm volatile("ld.shared::cluster.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at) : "memory");
    return v;
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
    nwarps = uniform(nwarps); halves = uniform(halves);
    const int row_items = T * halves, items = uniform(sh.nA * row_items);
    if (lane < 3) sh.warp_part[lane][threadIdx.x >> 5] = 0ll;
    __syncwarp();
    long long units = 0ll;
    for (int item = uniform(warp); item < items; item += nwarps) {
        const int i = item / row_items, t = item - i * row_items;
        const int row = uniform(sh.A[i]);
        const float *rp = zp + (int64_t)row * stride;
        const float *rq = zq + (int64_t)row * stride;
        const bool al = uniform(((reinterpret_cast<uintptr_t>(rp) | reinterpret_cast<uintptr_t>(rq)) & 15) == 0);
        V = uniform(V);
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
    const int n_cta = uniform((int)cluster.num_blocks()), cta_rank = uniform((int)cluster.block_rank());
    const int lane = threadIdx.x & 31, warp = warp_index();
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
    // (warp 0's lanes: only its first thread goes on with the mass)
    long long sum[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
        sum[x] = lane < n_cta ? sh.part[n_pass & 1][x][lane] : 0ll;
        if (x && first) continue;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) sum[x] += __shfl_xor_sync(kFull, sum[x], o);
    }
    const long long hi = sum[0], lo = sum[1], q = sum[2];
    if (first) return (double)hi * (1.0 / kSumUnit);
    const double total = ((double)lo * (1.0 / kSumUnit) + (double)hi) * (1.0 / kSumUnit);
    const double rest = (s - (double)s_hi) * ((double)q * kUnfix);
    return rest < total ? total - rest : total;
}

// One cluster-wide pass over the live rows; every CTA fills its own shared-memory histogram.
// sh.warp_part[0]: the mass that each warp added (p and q), from floating-point sums.
__device__ __forceinline__ void histogram_pass(const VerifyArgs &a, Shared &sh, float binscale, const HistSmem &h,
                               double *sums1, int cta_rank, int n_cta, int halves) {
    // halves = 2: an item is a half tile (when the cluster has a warp for each), with a sum of its own
    const int lane = threadIdx.x & 31;
    const int warp = cta_rank * kVWarps + warp_index();
    const int nwarps = n_cta * kVWarps;
    const int items = uniform(sh.nA) * a.T * halves;
    unsigned long long added = 0ull;
    const uint32_t magic_bits = __float_as_uint(kBinMagic);
    const uint32_t wbase = (uint32_t)__cvta_generic_to_shared(h.wp) - (magic_bits << 2);
    const uint32_t over_bits = magic_bits + (uint32_t)(kBins + ((threadIdx.x >> 5) & 15) * 16 + (threadIdx.x & 15));
    const float half_bin = 0.5f / binscale;                      // half a bin in log2 units
    const float top = (float)kBins / binscale - half_bin;       // log2 of the last edge (minus the half), as the bins see it
    const int row_items = a.T * halves;
    for (int item = warp; item < items; item += nwarps) {
        const int i = item / row_items, t = item - i * row_items;
        const int row = uniform(sh.A[i]);
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
    // (below 2^46: two parts of 23 bits)
    const unsigned lo = __reduce_add_sync(kFull, (unsigned)added & 0x7fffffu), hi = __reduce_add_sync(kFull, (unsigned)(added >> 23));
    if (lane == 0) sh.warp_part[0][threadIdx.x >> 5] = (long long)hi * 0x800000ll + lo;
}

// This CTA's histogram into suffix sums (p and q mass of its bins >= k, units of 2^-44), over the words: entry k is 16 bytes, p
// low and high half, then q, so that a look-up is one load.  Entry kBins is the last bin, whose copies are folded here.  Entries of
// eight bins are rotated against one another: a thread takes eight bins, and eight threads that store an entry each touch all banks.  Each CTA keeps the sums of its own cells; the chain adds the few that it looks up over the
// CTAs (a merge of the 4096 bins over the cluster before it took 4.5 us a layer and another cluster barrier, for at most 2 m bins that
// anybody looks at).
static_assert(kBins == 8 * kVThreads, "eight bins to a thread");
__device__ __forceinline__ int suffix_entry(int k) { return k ^ ((k >> 3) & 7); }
static_assert((kBins + 8) * 16 <= kHistArrays * kHistWords * 4, "an entry for every bin and the last one");
__device__ __forceinline__ void hist_suffix(const HistSmem &h, Shared &sh) {
    const int lane = threadIdx.x & 31, warp = warp_index(), i0 = threadIdx.x * 8;
    unsigned long long v[2][8];                              // p, q
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const uint32_t *w = x ? h.wq : h.wp, *b = x ? h.bq : h.bp;
#pragma unroll
        for (int k = 0; k < 8; k += 4) {
            const uint4 lo = *reinterpret_cast<const uint4 *>(w + i0 + k), hi = *reinterpret_cast<const uint4 *>(b + i0 + k);
            v[x][k] = ((unsigned long long)hi.x << 16) + lo.x; v[x][k + 1] = ((unsigned long long)hi.y << 16) + lo.y;
            v[x][k + 2] = ((unsigned long long)hi.z << 16) + lo.z; v[x][k + 3] = ((unsigned long long)hi.w << 16) + lo.w;
        }
#pragma unroll
        for (int k = 6; k >= 0; --k) v[x][k] += v[x][k + 1];
    }
    unsigned long long above[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        unsigned long long s = v[x][0];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_down_sync(kFull, s, o);
            if (lane + o < 32) s += t;
        }
        above[x] = s - v[x][0];
        if (lane == 0) sh.wtot[x][warp] = s;
    }
    if (warp < kOverSlots / 32) {
        const int i = kBins + (int)threadIdx.x;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            unsigned long long s = ((unsigned long long)(x ? h.bq : h.bp)[i] << 16) + (x ? h.wq : h.wp)[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
            if (lane == 0) sh.over[x][warp] = s;
        }
    } else if (warp == kOverSlots / 32) {
        long long s = lane < kVWarps ? sh.warp_part[0][lane] : 0ll;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        if (lane == 0) sh.added = (unsigned long long)s;
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        // lanes 0 to 15: the warps behind this one; 16 to 23: the copies of the last bin
        unsigned long long t = lane < kVWarps ? (lane > warp ? sh.wtot[x][lane] : 0ull) : lane < kVWarps + kOverSlots / 32 ? sh.over[x][lane - kVWarps] : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
        above[x] += t;
    }
    // what the threads added, by their floating-point sums, minus what the words hold.  Without a wrap that is rounding: half a
    // unit for each cell and 2^-20 of the mass (16 cells in a float sum), less than 2^26 units; a wrap lowers the words by 2^32.
    // The top bit of the first entry tells (a sum takes 46 bits)
    uint32_t wrapped = 0u;
    if (threadIdx.x == 0 && (long long)(sh.added - (v[0][0] + above[0]) - (v[1][0] + above[1])) > (1ll << 31)) wrapped = kWrapped;
    uint4 *entries = reinterpret_cast<uint4 *>(h.wp);
    auto entry = [](unsigned long long p, unsigned long long q) { return make_uint4((uint32_t)p, (uint32_t)(p >> 32), (uint32_t)q, (uint32_t)(q >> 32)); };
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        uint4 e = entry(v[0][k] + above[0], v[1][k] + above[1]);
        if (k == 0) e.y |= wrapped;
        entries[suffix_entry(i0 + k)] = e;
    }
    if (threadIdx.x == kVThreads - 1) entries[suffix_entry(kBins)] = entry(above[0], above[1]);
}

// Per live draft: rho = p_beam/q_beam of its cell, by one warp.
__device__ __noinline__ void draft_tests(Shared &sh, int m, int lane) {
    m = uniform(m);
#pragma unroll 1
    for (int i0 = 0; i0 < m; i0 += 32) {
        const int i = i0 + lane;
        if (i >= m) continue;
        const int ai = sh.S_parent_idx[i];
        const double lp = sh.rho[i], lq = sh.lq[i];
        double rho;
        if (lq == -INFINITY || sh.lwq[ai] == -INFINITY)
            rho = (lp > -INFINITY && sh.lwp[ai] > -INFINITY) ? INFINITY : 0.0;
        else
            rho = exp((sh.lwp[ai] - sh.lwq[ai]) + (lp - lq));
        sh.rho[i] = rho;
    }
    __syncwarp();
}

// The accept loop from draft sh.next_i on, by one warp.  The run position rises by one with every rejection and falls back to 1
// with an accept, so the drafts behind one another are tested side by side, each at the position that it has if
// all before it are rejected; the first accept among them ends the round.
// on_demand: ends with sh.need_exact = 1 after a rejection whose residual mass c_{j+1} is not known yet.
// node_status: nullptr in a CTA that writes no results.
__device__ __noinline__ void accept_drafts(Shared &sh, int8_t *st, int8_t *node_status, int n_lo, int m, int W, bool on_demand, int lane) {
    int i = uniform(sh.next_i), count = uniform(sh.count), j = uniform(sh.run_j), tests = 0, near = 0, need = 0;
    const int len = uniform(sh.chain_len);
    m = uniform(m); W = uniform(W); on_demand = uniform(on_demand);
#pragma unroll 1
    while (i < m && count < W && !need) {
        const int n = min(m - i, 32);
        // an empty residual means p' == q_beam: the rejected draft lay outside the support of q_beam, there is nothing to
        // subtract and p' stays, and so does the run position
        const unsigned rises = __ballot_sync(kFull, j + lane <= len && sh.c_arr[min(j + lane, kMaxLive) + 1] > 0.0);
        const int stop = ~rises ? __ffs(~rises) - 1 : 32;         // positions j .. j + stop are reached
        const int jt = j + min(lane, stop);
        const bool asks = on_demand && j + stop == len + 1;       // a rejection at the last position asks for its residual mass
        const int lanes = asks ? min(n, stop + 1) : n;
        bool accept = false, close = false;
        if (lane < lanes) {
            // u <= min(max(rho - s, 0) / c, 1), times c
            const double c = sh.c_arr[jt], u = sh.uu[i + lane] * c, top = fmin(fmax(sh.rho[i + lane] - sh.s_arr[jt - 1], 0.0), c);
            accept = u <= top;
            close = fabs(u - top) < 1e-5 * c;
        }
        const unsigned accepts = __ballot_sync(kFull, accept);
        const int done = accepts ? __ffs(accepts) : lanes;        // drafts tested in this round
        near += __popc(__ballot_sync(kFull, close && lane < done));
        if (lane < done) {
            const int node = sh.S[i + lane], status = lane == done - 1 && accepts ? DSBD_NODE_ACCEPTED : DSBD_NODE_REJECTED;
            st[node - n_lo] = (int8_t)status;
            if (node_status) node_status[node] = (int8_t)status;
            if (status == DSBD_NODE_ACCEPTED) sh.acc[count] = node;
        }
        tests += done;
        i += done;
        if (accepts) { ++count; j = 1; }
        else if (asks && done == stop + 1) {
            j += stop;
            if (lane == 0) sh.s_arr[j] = sh.s_arr[j - 1] + sh.c_arr[j];
            need = 1;
        } else j += min(done, stop);
    }
    __syncwarp();
    if (lane == 0) {
        sh.next_i = i;
        sh.count = count;
        sh.run_j = j;
        sh.n_tests += tests;
        sh.n_near += near;
        sh.need_exact = need;
        sh.chain_pos = j;                          // (the position whose residual mass is asked for)
    }
    __syncwarp();
}

// Where the warps of a CTA keep what a draw searches (the histogram arrays are idle then): a warp's token masses or a piece of
// its tile masses, and behind them, for the residual draw, the sums of kParts equal shares of the layer's item sums.
constexpr int kParts = 256, kPiece = 512;
static_assert(kPiece * sizeof(double) <= kTokWords * sizeof(float), "a piece of tile masses fits a warp's words");
static_assert(kVWarps * kTokWords * sizeof(float) + kParts * sizeof(double) <= kHistArrays * kHistWords * sizeof(uint32_t),
              "what the draws search overlays the histogram arrays");

// One completion draw by one warp: from p_beam, or (use_res) from the residual at s_res; returns the token or -1
// and the index of the live parent.  parts: see draw_shares.
__device__ __forceinline__ int draw_cell(const VerifyArgs &a, const Shared &sh, double u, bool use_res, float s_res,
                                         const double *res_sums, int halves, const double *parts, float *words, int lane, int *ia_out) {
    double *piece = reinterpret_cast<double *>(words);
    double target = u;
    // p_beam: first the live parent (its row holds exactly its beam weight), then the tile.  Residual: the share, then the tile
    const int tiles = sh.nA * a.T, per = (tiles + kParts - 1) / kParts;
    int ia = uniform(locate(use_res ? parts : sh.wp, use_res ? kParts : sh.nA, target, true, false, lane));
    if (ia < 0) return -1;
    const int at = use_res ? ia * per : 0, row_a = use_res ? 0 : sh.A[ia];
    int n = use_res ? min(per, tiles - at) : a.T, t = 0;          // tile masses to search, from `at` on
    const double wpa = use_res ? 0.0 : sh.wp[ia], lse_row = use_res ? 0.0 : a.lse[row_a];
    const TileStat *st = a.stats + (int64_t)row_a * a.T;
#pragma unroll 1
    for (int base = 0; ; base += kPiece) {
        const int len = min(kPiece, n - base);
#pragma unroll 1
        for (int i0 = 0; i0 < len; i0 += 32) {
            const int i = i0 + lane;
            double x = 0.0;
            if (use_res) {
                // (one per tile, or two when the pass that wrote them worked on half tiles)
                const double *k = res_sums + (int64_t)(at + base + min(i, len - 1)) * halves;
                x = __ldcg(k);
                if (halves > 1) x += __ldcg(k + 1);
            } else if (i < len) {
                const TileStat ts = st[base + i];
                if (ts.sum > 0.f) x = wpa * (double)ts.sum * exp((double)ts.mx * a.inv_tau - lse_row);
            }
            if (i < len) piece[i] = x;
        }
        __syncwarp();
        const bool more = base + len < n;
        t = uniform(locate(piece, len, target, false, more, lane));
        __syncwarp();
        if (t >= 0 && !(more && t == len)) { t += at + base; break; }
        if (t < 0) {
            if (base == 0) return -1;
            n = base;                                // no mass from here on: the last tile with mass before
            target = INFINITY;
            base -= 2 * kPiece;
        }
    }
    if (use_res) { ia = t / a.T; t -= ia * a.T; }
    *ia_out = ia;
    const RowOff ro = row_off(sh, ia);
    const int64_t row = (int64_t)sh.A[ia] * a.stride;
    return locate_token(a.zp + row, a.zq + row, a.V, a.k2, t, ro, use_res ? s_res : 0.f, target, lane, words);
}

// Sums of kParts equal shares of the layer's item sums, by the CTA's first kParts threads: what a residual draw searches first.
__device__ __forceinline__ void draw_shares(const double *res_sums, int halves, int tiles, double *parts) {
    if (threadIdx.x >= kParts) return;
    const int per = (tiles + kParts - 1) / kParts * halves;
    const int i1 = min(((int)threadIdx.x + 1) * per, tiles * halves);
    double v = 0.0;
#pragma unroll 4
    for (int i = (int)threadIdx.x * per; i < i1; ++i) v += __ldcg(res_sums + i);
    parts[threadIdx.x] = v;
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
    int count[3][3];              // of a round's three cuts, for three rounds in turn
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
// Latency decides (a chain of short steps between barriers): the threshold is a search whose rounds have one
// barrier each, try three cuts and stop at the first with k tiles above it or not many more, about 4 rounds (with one cut a round and at most
// k + 2 tiles 8 rounds, 2.3 us of a draft layer's 11).  Exact radix
// selection (4 rounds of three barriers with colliding atomics), one warp that lists the tiles, one thread that cuts
// at top-p and half the CTA for a draft layer's only model took, for a draft of 5 layers of 16 x 8 rows of 128256 with
// top-k 10, 419 us instead of 337; 20 requests with top-k 50 took 169 instead of 144.  (As a function that is
// not inlined, with generic loads: 363 and 165.)
template <int NT>
__device__ int build_support(const VerifyArgs &a, const Shared &sh, int model, const double *lse, uint32_t *hist_p, uint32_t *hist_q) {
    WarpScratch &ws = *reinterpret_cast<WarpScratch *>(hist_q);
    SupportTmp &tp = ws.tmp[model];
    double *cand_key = reinterpret_cast<double *>(hist_p) + model * kMaxCand;
    int *cand_cell = reinterpret_cast<int *>(reinterpret_cast<double *>(hist_p) + 2 * kMaxCand) + model * kMaxCand;
    const int tl = threadIdx.x & (NT - 1);                    // thread and warp inside the part
    const int lane = threadIdx.x & 31, warp = uniform(tl >> 5);
    constexpr int kPartWarps = NT / 32;
    const int T = a.T, nt = uniform(sh.nA) * T, k = a.top_k;
    const TileStat *stats = a.stats + (int64_t)model * a.N * T;
    const double *lw = model ? sh.lwq : sh.lwp;
    const float *z = model ? a.zq : a.zp;
    const float inv_tau_f = (float)a.inv_tau;
#pragma unroll 1
    for (int i = tl; i < sh.nA; i += NT) tp.off[i] = (float)(lw[i] - lse[sh.A[i]]);
    if (tl < 3) tp.count[0][tl] = 0;
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
#pragma unroll 2
        for (int i0 = 0; i0 < nt; i0 += NT) {
            const int i = i0 + tl;
            if (i >= nt) continue;
            const float v = bound(i);
            const unsigned u = image(v);
            if (cached) bcache[i] = u;
            if (v > -INFINITY) { ++finite; lo = min(lo, u); hi = max(hi, u); }
        }
        lo = __reduce_min_sync(kFull, lo); hi = __reduce_max_sync(kFull, hi); finite = __reduce_add_sync(kFull, finite);
        if (lane == 0) { tp.lo[warp] = lo; tp.hi[warp] = hi; tp.finite[warp] = finite; }
    }
    part_sync<NT>(model);
    unsigned lo = __reduce_min_sync(kFull, tp.lo[lane & (kPartWarps - 1)]), hi = __reduce_max_sync(kFull, tp.hi[lane & (kPartWarps - 1)]);
    const int finite = __reduce_add_sync(kFull, lane < kPartWarps ? tp.finite[lane] : 0);
    if (finite >= k) {
        // count(>= lo) >= k always holds; hi is above the k-th largest.  A tile for every warp costs no more than k of them, and one or
        // two too many are fine, where they are close (cells 30 below the largest have no mass to speak of)
        const float near = value(hi) - 30.f;
        const int enough = max(k + 2, kPartWarps);
        ++hi;
#pragma unroll 1
        for (int round = 0; hi - lo > 1; ++round) {
            const unsigned step = max((hi - lo) >> 2, 1u);           // (a cut at hi or above it counts fewer than k)
            int n[3] = {0, 0, 0};
            auto count = [&](unsigned u) {
#pragma unroll
                for (int c = 0; c < 3; ++c) n[c] += u >= lo + (c + 1) * step;
            };
            if (cached) {
#pragma unroll 2
                for (int i0 = 0; i0 < nt; i0 += NT)
                    if (const int i = i0 + tl; i < nt) count(bcache[i]);
            } else {
#pragma unroll 1
                for (int i0 = 0; i0 < nt; i0 += NT)
                    if (const int i = i0 + tl; i < nt) count(image(bound(i)));
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) n[c] = __reduce_add_sync(kFull, n[c]);
            int *counts = tp.count[round % 3], *next = tp.count[(round + 1) % 3];
            if (lane < 3) {
                atomicAdd(&counts[lane], lane == 0 ? n[0] : lane == 1 ? n[1] : n[2]);
                if (warp == 0) next[lane] = 0;                       // (last read two rounds ago)
            }
            part_sync<NT>(model);
            // the cuts with at least k tiles (below hi: bounds that are not numbers count above every cut)
            const int mine = counts[min(lane, 2)], at = __popc(__ballot_sync(kFull, lane < 3 && mine >= k && (lane + 1) * step < hi - lo));
            if (at < 3) hi = min(hi, lo + (at + 1) * step);
            lo += at * step;
            if (at == 0) continue;
            const int reached = __shfl_sync(kFull, mine, at - 1);
            if (reached == k || (reached <= enough && value(lo) > near)) break;
        }
    }
    // The tiles from the cut on, and the smallest bound among them, which is the threshold: a cut may lie far down in
    // the gap above masked tiles, where it would pass every cell of the tiles above.
    // (the float keys carry an error of about 1e-5; the slack keeps the selection conservative)
    auto slack = [](float t) -> float { return t - 5e-5f - 4e-6f * fabsf(t); };
    float theta = -INFINITY, cut = finite >= k ? slack(value(lo)) : -INFINITY;
    for (int again = 0; ; ++again) {
        unsigned low = 0xffffffffu;
#pragma unroll 1
        for (int i0 = 0; i0 < nt; i0 += NT) {
            const int i = i0 + tl;
            if (i >= nt) continue;
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
        if (uniform(tp.n_sel) <= 256) break;
        if (again) return DSBD_DEV_CAPACITY;                      // hundreds of tiles tie at the threshold
        // (or closely below the cut)
        part_sync<NT>(model);
        if (tl == 0) tp.n_sel = 0;
        cut = theta;
        part_sync<NT>(model);
    }
    const int n_sel = uniform(tp.n_sel);
    // Sweeps over the selected tiles by all warps: each counts the cells whose key reaches th and, when collect is set, lists
    // them (order is irrelevant: the final choice is by (key, cell)).  The first one nearly always fits the list.  Too many
    // cells reach the conservative threshold where there are few tiles, a large k or near ties: then a bisection, by sweeps that
    // only count, finds a threshold with between k and kMaxCand cells above it, and one more sweep lists those.
    // (One copy of the sweep, and lanes that walk their hits: the three copies with an unrolled list each were 60 KB of code.)
    float th = theta, lo_t = 0.f, hi_t = 0.f;
    bool collect = true;
    int n_cand;
#pragma unroll 1
    for (int itn = -1; ; ++itn) {
        const float th_f = fmaxf(th, -3.402823466e38f);      // (a key of -infinity has no mass)
#pragma unroll 1
        for (int sidx = warp; sidx < n_sel; sidx += kPartWarps) {
            const int ti = tp.sel[sidx], ia = ti / T, t = ti - ia * T, row = sh.A[ia];
            const float *rowp = z + (int64_t)row * a.stride;
            const bool al = (reinterpret_cast<uintptr_t>(rowp) & 15) == 0;
            float4 v[8];
            load_tile<false>(rowp, t * kTile, a.V, al, lane, v);
            // the warp's next tile on its way to L2 (a tile is 32 lines of 128 bytes: one per lane)
            if (sidx + kPartWarps < n_sel) {
                const int tn = tp.sel[sidx + kPartWarps], in = tn / T, e = (tn - in * T) * kTile + lane * 32;
                if (e < a.V) asm volatile("prefetch.global.L2 [%0];" ::"l"(z + (int64_t)sh.A[in] * a.stride + e));
            }
            const float off_f = tp.off[ia];
            unsigned hits = 0;                               // bit (it*4+c) of this lane's 32 cells
#pragma unroll
            for (int it = 0; it < 8; ++it) {
                const float zz[4] = {v[it].x, v[it].y, v[it].z, v[it].w};
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (fmaf(zz[c], inv_tau_f, off_f) >= th_f) hits |= 1u << (it * 4 + c);
            }
            if (hits) {
                int pos = atomicAdd(&tp.n_cand, __popc(hits));
                if (collect) {
                    const double off_d = lw[ia] - lse[row];
#pragma unroll 1
                    for (; hits && pos < kMaxCand; hits &= hits - 1, ++pos) {
                        const int bit = __ffs(hits) - 1, tok = t * kTile + (bit >> 2) * 128 + lane * 4 + (bit & 3);
                        cand_key[pos] = off_d + (double)__ldg(rowp + tok) * a.inv_tau;
                        cand_cell[pos] = ia * a.V + tok;
                    }
                }
            }
        }
        part_sync<NT>(model);
        n_cand = uniform(tp.n_cand);
        if (collect) {
            if (n_cand <= kMaxCand || itn >= 0) break;
            lo_t = theta; hi_t = -INFINITY;
#pragma unroll 1
            for (int sidx = 0; sidx < n_sel; ++sidx) hi_t = fmaxf(hi_t, bound(tp.sel[sidx]));
            if (!(lo_t > -INFINITY)) lo_t = hi_t - 400.f;
            collect = false;
        } else if (n_cand > kMaxCand) lo_t = th;
        else if (n_cand < k) hi_t = th;
        else collect = true;
        if (!collect) {
            if (itn + 1 >= 60 || !(hi_t > lo_t)) return DSBD_DEV_CAPACITY;              // a huge tie at the cut
            // (first out of the gap above a mask of finite values: halving does not come back from -1e30)
            const float half = 0.5f * (lo_t + hi_t);
            th = itn < 0 ? fmaxf(half, hi_t - 400.f) : half;
        }
        part_sync<NT>(model);                      // every thread has taken the count
        if (tl == 0) tp.n_cand = 0;
        part_sync<NT>(model);
    }
    // exact top k of the candidates: every candidate counts those that beat it (key descending,
    // cell ascending -- a total order, cells are unique) and, if fewer than k do, that count is its
    // place in the support.  Eight lanes to a candidate: a few dozen candidates take one round.
    if (n_cand > kMaxCand) n_cand = kMaxCand;
#pragma unroll 1
    for (int j0 = 0; j0 < n_cand; j0 += NT / 8) {
        const int jc = j0 + (tl >> 3);
        double key = 0.0;
        int cell = 0, rank = 0;
        if (jc < n_cand) {
            key = cand_key[jc];
            cell = cand_cell[jc];
#pragma unroll 2
            for (int i = tl & 7; i < n_cand; i += 8) {
                const double ki = cand_key[i];
                rank += (ki > key) || (ki == key && cand_cell[i] < cell);
            }
        }
        rank += __shfl_xor_sync(kFull, rank, 1);
        rank += __shfl_xor_sync(kFull, rank, 2);
        rank += __shfl_xor_sync(kFull, rank, 4);
        if (jc < n_cand && (tl & 7) == 0 && rank < k) {
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
#pragma unroll 2
    for (int j = 0, n = ws.n[model]; j < n; ++j) at = ws.cell[model][j] == cell ? j : at;      // (cells are unique)
    return at >= 0 ? ws.prob[model][at] : 0.0;
}

// Inverse-CDF draws over the p support in canonical order; mass max(p~ - s q~, 0) (s = 0: p~).  By one warp, one
// draw for each lane that wants one (u per lane).  Returns the index into the p support or -1.
__device__ int draw_support(const WarpScratch &ws, double u, double s, int lane) {
    const int n = uniform(ws.n[0]);
    double w0 = 0.0, w1 = 0.0;                                // places 2 lane and 2 lane + 1
    if (2 * lane < n) { const int i = ws.order[2 * lane]; w0 = fmax(ws.prob[0][i] - s * ws.qat[i], 0.0); }
    if (2 * lane + 1 < n) { const int i = ws.order[2 * lane + 1]; w1 = fmax(ws.prob[0][i] - s * ws.qat[i], 0.0); }
    const double incl = warp_scan(w0 + w1, lane), cum0 = incl - w1;
    const double zsum = __shfl_sync(kFull, incl, 31);
    const unsigned m0 = __ballot_sync(kFull, w0 > 0.0), m1 = __ballot_sync(kFull, w1 > 0.0);
    const double target = u * zsum;
    int pick = -1;
    bool found = false;
#pragma unroll 1
    for (int l = 0; 2 * l < n; ++l) {
        const double c0 = __shfl_sync(kFull, cum0, l), c1 = __shfl_sync(kFull, incl, l);
        if (!found && (m0 >> l & 1)) { pick = 2 * l; found = c0 >= target; }
        if (!found && (m1 >> l & 1)) { pick = 2 * l + 1; found = c1 >= target; }
    }
    return pick < 0 || !(zsum > 0.0) ? -1 : ws.order[pick];
}

// After build_support(p) [and q]: q~ at the p cells and the canonical order of the p support.
__device__ void finish_supports(WarpScratch &ws, bool have_q, int lane) {
    // canonical order: the place of a cell is the number of support cells below it (cells are unique)
    const int n = uniform(ws.n[0]);
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        if (i >= n) continue;
        const int c = ws.cell[0][i];
        int place = 0;
#pragma unroll 2
        for (int j = 0; j < n; ++j) place += ws.cell[0][j] < c;
        ws.order[place] = i;
        ws.qat[i] = have_q ? support_lookup(ws, 1, c) : 0.0;
    }
    __syncwarp();
}

// Drafts behind the first rejection of a layer of known width up to which its residual masses are computed on demand: a pass
// for that rejection and at most one for each of them, against one histogram, and a pass more where the layer ends in a residual
// draw behind a second rejection.  Us a call with limits of none to four, every layer of known width, mean of three to six inputs of
// the benchmark's distributions (without passes on demand: 31.4, 43.7, 55.3, 130, 460, 925):
//                                             0      1      2      3      4
//    one request, 4 beams, V = 32000       31.4   31.4   29.4   29.0   29.1      a warp has at most two tiles of a pass
//    one request, 4 beams, V = 128256      42.1   40.8   40.5   39.8   39.8      likewise
//    16 requests, 4 beams, V = 32000       54.9   53.2   52.9   56.0   56.0      likewise: the slowest of 16 counts
//    16 requests, 4 beams, V = 128256       130    129    131    139    139
//    64 requests, 4 beams, V = 128256       460    457    463    492    490
//    64 requests, 8 beams, V = 128256       925    922    920    935    977
// 2 is within 1.5 per cent of the best wherever there are many tiles.  Where there are few, 3 gains 1 to 2 per cent for a single request
// and loses 6 for 16 of them.
__device__ __forceinline__ int on_demand_left(int n_tiles, int n_warps) { return n_tiles <= 2 * n_warps ? 3 : 2; }

// dynamic shared memory of k_verify: the histogram of a layer as four 32-bit arrays while it is
// being built, then (over the same bytes) the suffix sums of this CTA's p and q mass
constexpr size_t kVerifyDynSmem = kHistArrays * sizeof(uint32_t) * kHistWords;

// Two instances, with warped joints and without: neither carries the other's code, whose registers it would spill around
// (64 requests x 8 rows of 128256 with top-k 10: a call 781 us as one kernel, 772 as two; unwarped calls alike).
template <bool kWarped>
__global__ void __launch_bounds__(kVThreads, 2)
k_verify(const __grid_constant__ VerifyArgs a) {
    cg::cluster_group cluster = cg::this_cluster();
    const int n_cta = uniform((int)cluster.num_blocks());
    const int cta_rank = uniform((int)cluster.block_rank());
    const int r = blockIdx.x / n_cta;
    const int lane = threadIdx.x & 31;
    const int warp = warp_index();
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
    int b_lo = uniform(ld_early(a.req_beam_off + r)), b_hi = uniform(ld_early(a.req_beam_off + r + 1));
    // (what is below uses the offsets as indexes: a request whose own contradict the forest is reported and taken as empty.  Those of its
    // trees are looked at further down, by a thread each: all warps together here cost 16 requests 0.9 us, warp 0 alone in the
    // set-up one request 0.3)
    bool bad_off = b_lo < 0 || b_hi > a.B || b_lo > b_hi;
    if (bad_off) b_lo = b_hi = 0;
    int n_lo = uniform(ld_early(a.beam_node_off + b_lo)), n_hi = uniform(ld_early(a.beam_node_off + b_hi));
    bad_off = bad_off || n_lo < 0 || n_hi > a.N || n_lo > n_hi;
    if (bad_off) b_lo = b_hi = n_lo = n_hi = 0;
    int W_min = a.W_min_r ? ld_early(a.W_min_r + r) : a.W_min;
    int W_max = a.W_max_r ? ld_early(a.W_max_r + r) : a.W_max;
    int W_nom = a.W_nom_r ? ld_early(a.W_nom_r + r) : a.W_nom;
    // per-request widths come from device memory: a width below 1 or a cap below the minimum is
    // reported (after the set-up below) and the request is not verified
    W_min = uniform(W_min); W_max = uniform(W_max); W_nom = uniform(W_nom);
    const bool bad_widths = a.check_widths && (W_min < 1 || W_max < W_min || W_nom < 1);
    if (bad_widths) { W_min = W_max = W_nom = 1; }
    double *sums_base = a.tile_sums + (int64_t)r * 2 * (a.max_m + 1) * ((int64_t)a.max_live * a.T);
    const int64_t slot_stride = (int64_t)a.max_live * a.T;
    int n_pass = 0;
#ifdef DSBD_PHASE_TIMING
    if (threadIdx.x == 0) { sh.ts = writer ? a.dbg + (int64_t)r * 256 : nullptr; sh.ts_end = sh.ts + 255; }
#endif

    TS(1);
    if (threadIdx.x == 0) sh.empty_tree = 0;
    // (a CTA may store into another's shared memory once that CTA runs: arrived here, waited for below)
    cluster.barrier_arrive();
    if (!kWarped && threadIdx.x >= kVThreads - 1 - kMaxLive) {               // (the last warps: the first ones read the nodes)
        const int m = threadIdx.x - (kVThreads - 1 - kMaxLive);
        BinEdges e;
        e.scale = (float)((double)kBins / log2((double)max(m, 2)));          // s_j <= j <= m
        e.inv_scale = 1.0 / (double)e.scale;
        e.hi = exp2(e.inv_scale) * (1.0 + kEdgeTol);
        e.inv_width = 1.0 / (e.hi - (1.0 - kEdgeTol));
        sh.bins[m] = e;
    }
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
        float zp_tok = 0.f, zq_tok = 0.f, root_p = 0.f, root_q = 0.f;          // (the last two: of tree threadIdx.x)
        if (cached) {
            if ((int)threadIdx.x < n_trees) {
                nc.root[threadIdx.x] = ld_early(a.beam_node_off + b_lo + threadIdx.x);
                root_p = ld_early(a.root_logp + b_lo + threadIdx.x);
                root_q = ld_early(a.root_logq + b_lo + threadIdx.x);
            }
            const int i = threadIdx.x, n = n_lo + i;
            if (i < n_req) {
                par = ld_early(a.parent + n);
                if (a.draft_rank) nc.rank[i] = ld_early(a.draft_rank + n);
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
#pragma unroll 1
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
            // Every tree has nodes: then every root lies in the request and is one tree's only (else it would have either's score, another one in
            // every CTA).
            if (i < n_trees && nc.root[i] >= (i + 1 < n_trees ? nc.root[i + 1] : n_hi)) sh.empty_tree = 1;
            if (i < n_trees && nc.root[i] >= n_lo && nc.root[i] < n_hi) {
                const int root = nc.root[i] - n_lo;
                if (writer && nc.parent[root] != -1) report(a.status, DSBD_DEV_BAD_FOREST);
                slp[root] = (double)root_p;
                slq[root] = (double)root_q;
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
#pragma unroll 1
                while (tree + 1 < n_trees && nc.root[tree + 1] <= n_lo + i) ++tree;
                nc.tree[i] = (uint8_t)tree;
                if (nc.parent[i] == -1 && nc.root[tree] != n_lo + i) {
                    // a second root inside a tree (paths end there whichever negative value they see)
                    nc.parent[i] = -2;
                    if (writer) report(a.status, DSBD_DEV_BAD_FOREST);
                }
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
#pragma unroll 1
        for (int b = b_lo + (int)threadIdx.x; b < b_hi; b += kVThreads)
            if (a.beam_node_off[b] >= a.beam_node_off[b + 1]) sh.empty_tree = 1;
        __threadfence();
        cluster.sync();
        // ---- log-prob of every draft token given its parent (all nodes at once) ----
#pragma unroll 1
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
#pragma unroll 1
                for (int i = threadIdx.x; i < n_req; i += kVThreads) {
                    slp[i] = a.score_w[n_lo + i];
                    slq[i] = a.score_w[a.N + n_lo + i];
                }
                __syncthreads();
#pragma unroll 1
                for (int b = b_lo + (int)threadIdx.x; b < b_hi; b += kVThreads) {
                    const int root = a.beam_node_off[b];
                    if (root < n_lo || root >= n_hi) continue;                // (an empty tree's)
                    if (a.parent[root] != -1) report(a.status, DSBD_DEV_BAD_FOREST);
                    slp[root - n_lo] = (double)a.root_logp[b];
                    slq[root - n_lo] = (double)a.root_logq[b];
                }
                __syncthreads();
#pragma unroll 1
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
                    if (lo < n_lo || hi > n_hi) continue;
#pragma unroll 1
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
    // The roots are accepted: the first node of each tree.  Another node without a parent would be a live parent that has no place among the
    // input beams; it is reported and stays unreached.
    auto is_root = [&](int i) {
        if (cached) return nc.parent[i] == -1;
        if (a.parent[n_lo + i] >= 0) return false;
        int lo = b_lo, hi = b_hi;                            // first tree that starts at the node or behind it
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (a.beam_node_off[mid] < n_lo + i) lo = mid + 1; else hi = mid;
        }
        return a.beam_node_off[lo] == n_lo + i;
    };
    if (warp == 0) {
        if (lane == 0) {
            sh.err = 0; sh.n_out = 0; sh.n_draw = 0;
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
#pragma unroll 1
                for (int i = 0; i < sh.nA; ++i)
                    if (a.live_nodes[lo + i] < 0 || a.live_nodes[lo + i] >= a.N) sh.err = DSBD_DEV_BAD_FOREST;
                if (sh.err) sh.nA = 0;
#pragma unroll 1
                for (int i = 0; i < sh.nA; ++i) {
                    sh.A[i] = a.live_nodes[lo + i];
                    sp_live[i] = (double)a.sel_logp[sh.A[i]];
                    sq_live[i] = (double)a.sel_logq[sh.A[i]];
                }
            } else {
                sh.nA = b_hi - b_lo;
                if (sh.nA > kMaxLive || sh.empty_tree || bad_off) { sh.err = DSBD_DEV_BAD_FOREST; sh.nA = 0; }
            }
        }
        __syncwarp();
        if (!a.select_mode) {
            const int nA = uniform(sh.nA);
#pragma unroll 1
            for (int i0 = 0; i0 < nA; i0 += 32) {
                const int i = i0 + lane;
                if (i >= nA) continue;
                const int root = cached ? nc.root[i] : a.beam_node_off[b_lo + i];
                sh.A[i] = root;
                if (cached) nc.live[root - n_lo] = (uint8_t)i;
                sp_live[i] = cached ? nc.score_p[root - n_lo] : a.score[root];
                sq_live[i] = cached ? nc.score_q[root - n_lo] : a.score[a.N + root];
            }
            if (writer) {
#pragma unroll 1
                for (int l0 = 0; l0 <= a.gamma; l0 += 32)
                    if (const int l = l0 + lane; l <= a.gamma) a.out.layer_width[(int64_t)r * (a.gamma + 1) + l] = -1;
                if (lane == 0) { a.out.l_last[r] = a.gamma + 1; a.out.out_width[r] = 0; }
            }
        }
        __syncwarp();
        if (!a.select_mode && writer)
#pragma unroll 1
            for (int n0 = n_lo; n0 < n_hi; n0 += 32)
                if (const int n = n0 + lane; n < n_hi) {
                    const bool root = is_root(n - n_lo);
                    a.out.node_status[n] = root ? DSBD_NODE_ACCEPTED : DSBD_NODE_UNREACHED;
                    if (!cached && !root && a.parent[n] < 0) report(a.status, DSBD_DEV_BAD_FOREST);
                }
    }
    // Every CTA of the cluster takes identical decisions from identical data, so each keeps its
    // own copy of the node statuses and only rank 0 writes results.
    const bool st_ok = n_req_nodes <= kMaxLive * kMaxLive;
    if (!a.select_mode)
#pragma unroll 1
        for (int n0 = 0; n0 < n_req_nodes && st_ok; n0 += kVThreads)
            if (const int n = n0 + threadIdx.x; n < n_req_nodes) st[n] = is_root(n) ? DSBD_NODE_ACCEPTED : DSBD_NODE_UNREACHED;
    __syncthreads();
    if (!a.select_mode && !st_ok && threadIdx.x == 0) sh.err = DSBD_DEV_BAD_FOREST;
    if (bad_widths && threadIdx.x == 0) sh.err = DSBD_DEV_BAD_PARAM;
    __syncthreads();
    // node data by local index, from the cache when there is one
    auto nd_depth = [&](int i) -> int { return cached ? (int)nc.depth[i] : a.depth[n_lo + i]; };
    auto nd_parent = [&](int i) -> int { return cached ? (int)nc.parent[i] : a.parent[n_lo + i] - n_lo; };
    auto node_lse = [&](int model) -> const double * {
        return cached ? (model ? nc.lse_q : nc.lse_p) - n_lo : a.lse + (int64_t)model * a.N;
    };
    auto nd_score = [&](int model, int i) -> double {
        return cached ? (model ? nc.score_q[i] : nc.score_p[i]) : a.score[(int64_t)model * a.N + n_lo + i];
    };

    const bool failed = uniform(sh.err);
    // Layers 1 .. gamma; then, in the CTA that writes, the extra layer: no drafts, W_nom beams from p_beam^(gamma+1).
    const int n_layers = a.select_mode ? 1 : a.gamma + (writer ? 1 : 0);
#pragma unroll 1
    for (int l = 1; l <= n_layers && !failed; ++l) {
        const bool extra = !a.select_mode && l > a.gamma;
        // ---- live drafts of layer l, in draw order; beam weights ----
        TS(2);
        if (warp == 0) {
            int m = 0;
            if (a.select_mode) {
                m = uniform(a.m_in[r]);
                if (m < 0 || m > kMaxLive) m = -1;
            } else if (!extra) {
#pragma unroll 1
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
                if (m > kMaxLive) m = -1;
                __syncwarp();
                if (a.draft_rank) {
                    // order of (draft_rank, node id), ids being ascending: a draft's place is the number before it
#pragma unroll 1
                    for (int i0 = 0; i0 < m; i0 += 32)
                        if (const int i = i0 + lane; i < m) sh.S_parent_idx[i] = cached ? nc.rank[sh.S[i] - n_lo] : a.draft_rank[sh.S[i]];
                    __syncwarp();
#pragma unroll 1
                    for (int i0 = 0; i0 < m; i0 += 32) {
                        const int i = i0 + lane;
                        if (i >= m) continue;
                        const int key = sh.S_parent_idx[i];
                        int place = 0;
#pragma unroll 2
                        for (int j = 0; j < m; ++j) place += sh.S_parent_idx[j] < key || (j < i && sh.S_parent_idx[j] == key);
                        sh.acc[place] = sh.S[i];
                    }
                    __syncwarp();
#pragma unroll 1
                    for (int i0 = 0; i0 < m; i0 += 32)
                        if (const int i = i0 + lane; i < m) sh.S[i] = sh.acc[i];
                    __syncwarp();
                }
                // index of a draft's parent in A, and its log-prob under either model given that parent
                const int nA = uniform(sh.nA);
#pragma unroll 1
                for (int i0 = 0; i0 < m; i0 += 32) {
                    const int i = i0 + lane;
                    if (i >= m) continue;
                    const int n = sh.S[i] - n_lo, pl = nd_parent(n);
                    int ai = nA;
                    if (cached) ai = nc.live[pl];
                    else
#pragma unroll 1
                        for (int k = 0; k < nA; ++k) ai = sh.A[k] == n_lo + pl ? k : ai;      // (nodes are unique)
                    sh.S_parent_idx[i] = ai;
                    sh.rho[i] = nd_score(0, n) - nd_score(0, pl);
                    sh.lq[i] = nd_score(1, n) - nd_score(1, pl);
                }
            }
            __syncwarp();
            if (lane == 0) {
                sh.m = m;
                sh.s_arr[0] = 0.0;
                sh.c_arr[1] = 1.0;
                sh.chain_len = 0;          // c_{j+1} is known for j = 1..chain_len
                sh.next_i = sh.count = 0;
                sh.run_j = sh.chain_pos = 1;
                sh.bank = l & 1;
            }
        } else if (warp <= 2) {
            live_weights(sh, warp - 1, warp == 1 ? sp_live : sq_live, node_lse(warp - 1), lane);
        } else if (warp == 3) {
            // the drafts' uniforms, as many as there can be
            if (!extra)
#pragma unroll 1
                for (int i = lane; i < kMaxLive; i += 32) sh.uu[i] = decision_uniform(a.seed, a.step, (uint32_t)r, (uint32_t)l, 0u, (uint32_t)i);
        } else if (!kWarped) {
            uint4 *words = reinterpret_cast<uint4 *>(hp);
#pragma unroll 4
            for (int i0 = 0; i0 < kHistArrays * kHistWords / 4; i0 += kVThreads - 128)
                if (const int i = i0 + threadIdx.x - 128; i < kHistArrays * kHistWords / 4) words[i] = make_uint4(0, 0, 0, 0);
        }
        __syncthreads();
        const int m = uniform(sh.m);
        if (m < 0) {
            if (threadIdx.x == 0) sh.err = DSBD_DEV_BAD_FOREST;
            break;
        }
        bool looked_up = false, on_demand = false;
        const int W_known = extra ? W_nom : W_min < W_max ? W_min : W_max;
        TS(3);

        constexpr bool warped = kWarped;
        WarpScratch &wsup = *reinterpret_cast<WarpScratch *>(hq);       // the histogram arrays are idle when warped
        if (warped) {
            // ---- supports of T o p_beam and T o q_beam, then the whole chain on <= 64 cells ----
            {
                // the first half of the warps builds the support of p, the second that of q, side by side; the extra layer's only one the
                // whole CTA (calls without drafts: 8 x 8 rows of 128256 with top-k 50 35.8 us instead of 38.2, 1 x 4 of 32000 with top-k 10
                // 14.8 instead of 15.6)
                const int half = extra ? 0 : warp / (kHalf / 32);
                const int e_part = extra ? build_support<kVThreads>(a, sh, 0, node_lse(0), hp, hq) : build_support<kHalf>(a, sh, half, node_lse(half), hp, hq);
                if (e_part && (threadIdx.x & (kHalf - 1)) == 0) wsup.tmp[half].err = e_part;
                __syncthreads();
                const int e = uniform(wsup.tmp[0].err ? wsup.tmp[0].err : extra ? 0 : wsup.tmp[1].err);
                if (e) {
                    if (threadIdx.x == 0) {
                        sh.err = e;
                        if (extra) a.out.layer_width[(int64_t)r * (a.gamma + 1) + a.gamma] = W_nom;      // (reached, and its width known)
                    }
                } else if (warp == 0) {
                    finish_supports(wsup, !extra, lane);
                    // rho of every live draft from the warped joints
                    if (!a.select_mode) {
#pragma unroll 1
                        for (int i0 = 0; i0 < m; i0 += 32) {
                            const int i = i0 + lane;
                            if (i >= m) continue;
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
#pragma unroll 1
                    for (int j = 1; j <= m; ++j) {
                        const double s_j = s_prev + c_cur;
                        double acc = fmax(p0 - s_j * q0, 0.0);
                        if (lane + 32 < ns) acc += fmax(p1 - s_j * q1, 0.0);
                        acc = warp_sum(acc);
                        if (lane == 0) { sh.s_arr[j] = s_j; sh.c_arr[j + 1] = acc; sh.chain_len = j; }
                        s_prev = s_j;
                        c_cur = acc;
                        if (!uniform(acc > 0.0)) break;
                    }
                    __syncwarp();
                }
            }
            __syncthreads();
        } else if (m >= 1) {
            const bool known = !a.select_mode && (m <= W_min || W_max <= W_min);
            if (known) {
                // ---- the width is W_min whatever the residual masses are (W~ <= m): the drafts are tested at once.  Up to
                // the first rejection that takes no pass over the rows at all, and every rejection one pass, without a histogram,
                // whose sums also serve the completion draw.  With more drafts behind the first rejection (on_demand_left) the
                // histogram is the better way.  (Two live rows of 128256, 4 CTAs: a layer of accepted drafts 5 us instead of 38; a
                // rejection 16 instead of 37.  Calls, W_min = 2: 64 requests x 8 rows 978 -> 907 us, 16 ragged requests 222 -> 164,
                // one request of V = 32000 61 -> 53.) ----
                if (warp == 0) {
                    draft_tests(sh, m, lane);
                    int first = m;                         // the first rejection
#pragma unroll 1
                    for (int base = 0; base < m && first == m; base += 32) {
                        const int i = base + lane;
                        const unsigned rejects = __ballot_sync(kFull, i < m && sh.uu[i] > fmin(sh.rho[i], 1.0));
                        if (rejects) first = base + __ffs(rejects) - 1;
                    }
                    if (lane == 0) sh.on_demand = first >= W_known || m - 1 - first <= on_demand_left(sh.nA * a.T, n_cta * kVWarps);
                }
                __syncthreads();
                on_demand = uniform(sh.on_demand);
            }
            const BinEdges bins = sh.bins[m];
            const float binscale = bins.scale;
            if (!on_demand) {
                // ---- one pass: ratio histogram of the layer over the live rows ----
                const int halves = item_halves(sh.nA * a.T, n_cta * kVWarps);
                histogram_pass(a, sh, binscale, hs, sums_base + ((int64_t)sh.bank * (a.max_m + 1)) * slot_stride, cta_rank,
                               n_cta, halves);
                __syncthreads();
                TS(4);
                hist_suffix(hs, sh);
                TS(7);
                cluster.sync();                            // every CTA's suffix sums are complete
                TS(5);
                if (threadIdx.x == 32) sh.halves = halves;
                if (warp == 1 && !a.select_mode && !known) draft_tests(sh, m, lane);
            }
            bool wrapped = false;
            // The chain c_{j+1} = F(s_j) from sh.chain_pos on (warp 0).  sh.need_exact = 1 where the histogram leaves one open.
            auto walk_chain = [&]() {
                int j = uniform(sh.chain_pos), need = 0;
                // lane c looks up bins k and k + 1 in CTA c
                const uint32_t mine = lane < n_cta ? 0xffffffffu : 0u;
                const uint32_t entries = cluster_address(hs.wp, min(lane, n_cta - 1));
                const double n_cells = (double)sh.nA * (double)a.V;      // every cell of the live rows, at most
                double s_j = sh.s_arr[j - 1], c_j = sh.c_arr[j];
#pragma unroll 1
                for (; j <= m; ++j) {
                    s_j += c_j;
                    if (lane == 0) { sh.s_arr[j] = s_j; sh.chain_len = j; }
                    // (up to s = 64 the bin found is off by at most 9e-7 of an edge: the logarithm's last place 3.3e-7, s as a
                    // float 0.6e-7, the product with binscale 5e-7; an edge by 6e-7.  The bracket below takes the edges
                    // 2e-6 wider.)
                    const int found = j == 1 ? 0 : (int)(log2f((float)s_j) * binscale), k = min(max(found, 0), kBins - 1);   // (s_1 = 1, the first edge)
                    uint4 e0 = ld_cluster(entries + suffix_entry(k) * 16);
                    const uint4 e1 = ld_cluster(entries + suffix_entry(k + 1) * 16);
                    // the bin's edges while the words are on their way; k / scale, rounded to a float (a division of floats: 0.6 us of
                    // 36.9, one request of V = 32000)
                    const float t = (float)((double)k * bins.inv_scale);
                    const double edge = (double)exp2f(t), inv = (double)exp2f(-t) * bins.inv_width;
                    const double r_lo = edge * (1.0 - kEdgeTol), r_hi = edge * bins.hi;
                    // every partial sum of the histogram is off by at most half a unit per cell
                    const double fix_err = n_cells * (0.5 * kUnfix) * (1.0 + s_j);
                    if (j == 1 && __any_sync(kFull, e0.y & mine & kWrapped)) wrapped = true;
                    e0.y &= ~kWrapped;
                    // the sums over the CTAs in two parts of 24 and 22 bits, so that a part's sum is one word; [0] above the bin, [1] in it
                    double P[2], Q[2];
                    auto add = [&](uint32_t low0, uint32_t high0, uint32_t low1, uint32_t high1, double (&sum)[2]) {
                        const unsigned lo0 = __reduce_add_sync(kFull, low0 & mine & 0xffffffu), hi0 = __reduce_add_sync(kFull, __funnelshift_l(low0, high0, 8) & mine);
                        const unsigned lo1 = __reduce_add_sync(kFull, low1 & mine & 0xffffffu), hi1 = __reduce_add_sync(kFull, __funnelshift_l(low1, high1, 8) & mine);
                        sum[0] = fma((double)hi1, 16777216.0, (double)lo1);
                        sum[1] = fma((double)(int)(hi0 - hi1), 16777216.0, (double)(int)(lo0 - lo1));
                    };
                    add(e0.x, e0.y, e1.x, e1.y, P);
                    add(e0.z, e0.w, e1.z, e1.w, Q);
                    // (in units of 2^-44)
                    double lo_b = 0.0, hi_b = 0.0, c_next = (P[0] + P[1]) - (Q[0] + Q[1]);
                    if (j > 1) {
                        auto larger = [](double x, double y) { return x > y ? x : y; };
                        lo_b = larger(P[1] - s_j * Q[1], 0.0);
                        double q_hi = larger((P[1] - r_lo * Q[1]) * inv, 0.0);
                        q_hi = q_hi < Q[1] ? q_hi : Q[1];
                        hi_b = larger(q_hi * (r_hi - s_j), lo_b);
                        c_next = larger(P[0] - s_j * Q[0], 0.0) + 0.5 * (lo_b + hi_b);
                    }
                    c_next *= kUnfix;
                    // the midpoint of the bracket is used: half its width plus the fixed-point term
                    // (a wrapped word: exact passes only)
                    need = __any_sync(kFull, 0.5 * kUnfix * (hi_b - lo_b) + fix_err > kErrTol || found >= kBins || wrapped);
                    if (need) break;
                    if (lane == 0) sh.c_arr[j + 1] = c_next;
                    c_j = c_next;
                    if (!__any_sync(kFull, c_next > 0.0)) j = m;     // chain exhausted: stop walking
                }
                if (lane == 0) {
                    sh.need_exact = need;
                    if (need && wrapped && j == 1) ++sh.n_wrapped;
                    sh.chain_pos = need ? j : m + 1;
                }
            };
            // ---- the residual masses, and (on demand) the accept loop between them ----
#pragma unroll 1
            while (true) {
                if (warp == 0) {
                    if (on_demand) accept_drafts(sh, st, writer ? a.out.node_status : nullptr, n_lo, m, W_known, true, lane);
                    else walk_chain();
                }
                __syncthreads();
                if (!uniform(sh.need_exact)) break;
                const int j = uniform(sh.chain_pos);
                const bool first = on_demand && j == 1;
                // (in a layer with a histogram that pass left the sums at j = 1 in slot 0; half tiles have room there only)
                const int halves = first ? item_halves(sh.nA * a.T, n_cta * kVWarps) : 1;
                const double c_next = exact_pass(a, sh, sh.s_arr[j], sums_base + ((int64_t)sh.bank * (a.max_m + 1) + (j == 1 ? 0 : j)) * slot_stride,
                                                 first, 0.5f / binscale, halves, true, n_pass++);
                if (threadIdx.x == 0) {
                    if (j == 1) sh.halves = halves;
                    sh.c_arr[j + 1] = c_next;
                    sh.chain_len = j;
                    if (!on_demand) { ++sh.n_exact; sh.chain_pos = c_next > 0.0 ? j + 1 : m + 1; }
                    else if (c_next > 0.0) sh.run_j = j + 1;
                }
                __syncthreads();
            }
            if (!on_demand) {
                cluster.barrier_arrive();                  // this CTA has done with the others' sums
                looked_up = true;
            }
        }

        TS(8);
        // ---- width and accept loop (warp 0) ----
        if (warp == 0 && !uniform(sh.err)) {
            int W = W_known;
            if (!on_demand && !extra) {
                // (the verification only needs W~ up to W_max and can stop at the first tail below the
                // threshold; dsbd_select_width returns the whole tail)
                const int wt = width_rule(sh, m, a.thresh, lane, a.select_mode ? -1 : W_max);
                W = wt > W_min ? wt : W_min;
                if (W > W_max) W = W_max;
            }
            if (a.select_mode) {
                if (writer && lane == 0) {
                    a.width_out[r] = W;
                    // alpha_j = 1 - c_{j+1}/c_j; once a residual has no mass every later alpha is 1
#pragma unroll 1
                    for (int j = 1; j <= m; ++j) {
                        double al = 1.0;
                        if (j <= sh.chain_len && sh.c_arr[j] > 0.0 && sh.c_arr[j + 1] > 0.0)
                            al = fmin(fmax(1.0 - sh.c_arr[j + 1] / sh.c_arr[j], 0.0), 1.0);
                        sh.alpha[j] = al;
                    }
                    if (a.alpha_out)
#pragma unroll 1
                        for (int j = 0; j < m && j < a.out_stride; ++j)
                            a.alpha_out[(int64_t)r * a.out_stride + j] = (float)sh.alpha[j + 1];
                    if (a.tail_out)
#pragma unroll 1
                        for (int K = 0; K <= m && K < a.out_stride; ++K)
                            a.tail_out[(int64_t)r * a.out_stride + K] = (float)sh.tail[K];
                }
            } else {
                if (!on_demand) accept_drafts(sh, st, writer ? a.out.node_status : nullptr, n_lo, m, W, false, lane);
#pragma unroll 1
                for (int i0 = uniform(sh.next_i); i0 < m; i0 += 32) {
                    const int i = i0 + lane;
                    if (i >= m) continue;
                    st[sh.S[i] - n_lo] = DSBD_NODE_CUT;
                    if (writer) a.out.node_status[sh.S[i]] = DSBD_NODE_CUT;
                }
                if (lane == 0) {
                    if (writer) a.out.layer_width[(int64_t)r * (a.gamma + 1) + (l - 1)] = W;
                    sh.W = W;
                    if (m >= 1 && (!on_demand || sh.chain_len > 0)) sh.n_rows += sh.nA;
                    if (!extra) ++sh.n_layers;
                    // a residual draw at run position j needs tile sums (a layer of known width has them)
                    sh.res_j = (sh.count < W && sh.run_j > 1 && !on_demand) ? sh.run_j : 0;
                }
            }
        }
        __syncthreads();

        if (looked_up) cluster.barrier_wait();         // the others have done with this CTA's sums
        TS(9);
        // ---- a residual draw locates its tile through tile sums of max(p_beam - s_{j-1} q_beam, 0) ----
        // slot 0 of the bank; in a layer of known width that of the rejection before the draw
        const int err = uniform(sh.err), j = uniform(sh.run_j), res_j = uniform(sh.res_j);
        const int res_slot = on_demand && j > 2 ? j - 1 : 0;
        double *res_sums = sums_base + ((int64_t)sh.bank * (a.max_m + 1) + res_slot) * slot_stride;
        if (!a.select_mode && !err && !warped && res_j > 2) {   // run position 2 is served by the histogram pass
            if (threadIdx.x == 0) { ++sh.n_respass; sh.halves = 1; }
            exact_pass(a, sh, sh.s_arr[res_j - 1], res_sums, false, 0.f, 1, false, n_pass++);
        }

        TS(10);
        if (a.select_mode || err) break;
        const int count = uniform(sh.count), want = uniform(sh.W) - count;
        if (want <= 0) {
            // ---- the accepted drafts, ascending node id, are the next layer's input beams (warp 0) ----
            if (warp == 0) {
                int nA = 0;
#pragma unroll 1
                for (int base = 0; base < n_req_nodes; base += 32) {
                    const int n = base + lane;
                    const bool in = n < n_req_nodes && nd_depth(n) == l && st[n] == DSBD_NODE_ACCEPTED;
                    const unsigned mask = __ballot_sync(kFull, in);
                    const int pos = nA + __popc(mask & ((1u << lane) - 1));
                    if (in && pos < kMaxLive) {
                        sh.A[pos] = n_lo + n;
                        if (cached) nc.live[n] = (uint8_t)pos;
                        sp_live[pos] = nd_score(0, n);
                        sq_live[pos] = nd_score(1, n);
                    }
                    nA += __popc(mask);
                }
                if (lane == 0) sh.nA = nA;
            }
            __syncthreads();
            continue;
        }
        // ---- a short layer ends the request: accepted drafts, then the residual draw, then fills from p_beam (in the extra layer
        // draws from p_beam alone), all independent of one another: a warp for each ----
        if (!writer) break;
        const int cap = uniform(a.out.out_off[r + 1] - a.out.out_off[r]);
        const int n_acc = min(count, max(cap, 0)), n_draw = n_acc < count ? 0 : min(want, max(cap - n_acc, 0));
        const bool use_res = j > 1;
        const int halves = res_slot ? 1 : uniform(sh.halves);
        float *words = reinterpret_cast<float *>(hp) + warp * kTokWords;
        double *parts = reinterpret_cast<double *>(reinterpret_cast<float *>(hp) + kVWarps * kTokWords);
        if (!warped && use_res) {
            draw_shares(res_sums, halves, sh.nA * a.T, parts);
            __syncthreads();
        }
#pragma unroll 1
        for (int b = warp; b < n_acc + n_draw; b += kVWarps) {
            int parent, node = -1, tok, source = DSBD_SRC_DRAFT;
            if (b < n_acc) {
                node = sh.acc[b];
                parent = a.parent[node];
                tok = a.token[node];
            } else {
                // draw f: the residual draw at the run position where the layer ended, then the fills, each with its own uniform
                const int f = b - n_acc;
                const double u = decision_uniform(a.seed, a.step, (uint32_t)r, (uint32_t)l, extra ? 3u : f ? 2u : 1u,
                                                  extra || !f ? (uint32_t)f : (uint32_t)(f - 1));
                const bool res = uniform(f == 0 && use_res);
                source = extra ? DSBD_SRC_EXTRA : f ? DSBD_SRC_FILL : DSBD_SRC_RESIDUAL;
                int ia = 0;
                if (warped) {
                    const int pick = draw_support(wsup, u, res ? sh.s_arr[j - 1] : 0.0, lane);
                    tok = -1;
                    if (pick >= 0) { ia = wsup.cell[0][pick] / a.V; tok = wsup.cell[0][pick] - ia * a.V; }
                } else {
                    tok = draw_cell(a, sh, u, res, res ? (float)sh.s_arr[j - 1] : 0.f, res_sums, halves, parts, words, lane, &ia);
                }
                parent = sh.A[ia];
            }
            if (lane == 0) {
                if (tok < 0) sh.n_draw = -1;
                else emit_at(a, r, b, parent, node, tok, source, cached ? &nc : nullptr, n_lo);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            a.out.l_last[r] = l;
            if (sh.n_draw < 0) { sh.err = DSBD_DEV_EXHAUSTED; sh.n_out = n_acc; }
            else {
                sh.n_out = n_acc + n_draw;
                if (n_acc < count || n_draw < want) sh.err = DSBD_DEV_CAPACITY;
            }
        }
        break;
    }
    __syncthreads();
    TS(11);
    if (threadIdx.x == 0 && writer) {
        if (!a.select_mode) {
            a.out.out_width[r] = sh.n_out;
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

// Clusters of 1 << log2 CTAs of k_verify that the current device holds at once.  Clusters stay inside a GPC, and GPCs have different numbers
// of SMs, so this is less than the CTAs that fit over the cluster's size; asked once per device (it takes some 10 us).  Where the
// device has no answer: the CTAs that fit (two per SM) over the cluster's size, none of the 16 that not every device takes, and asked
// again by the next call.
constexpr int kMaxDevices = 64;
int resident_clusters(void (*kernel)(VerifyArgs), bool warped, int log2) {
    static std::atomic<int> known[kMaxDevices][2][5];       // the answer plus one; 0: not asked yet
    int dev = -1, sms = 148;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
    std::atomic<int> *slot = dev >= 0 && dev < kMaxDevices ? &known[dev][warped][log2] : nullptr;
    int n = slot ? slot->load(std::memory_order_relaxed) - 1 : -1;
    if (n >= 0) return n;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1u << log2);
    cfg.blockDim = dim3(kVThreads);
    cfg.dynamicSmemBytes = kVerifyDynSmem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1u << log2;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (dev >= 0 && cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n >= 0) {
        if (slot) slot->store(n + 1, std::memory_order_relaxed);
        return n;
    }
    if (dev >= 0) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaGetLastError();
    return log2 > 3 ? 0 : 2 * sms >> log2;
}

// Cluster size (its logarithm): as many CTAs per request as its tile count can use, but few enough that all requests are resident at
// once.  16 from six tiles a CTA on (half a tile a warp instead of one): requests of four
// live rows, 128 tiles 41.9 us instead of 44.3 with 8 CTAs (one request), 252 tiles 43.5 for 47.9; eight requests 56.7 for 59.6 and
// 66.4 for 74.2.  64 tiles: 41.3 for 40.5, so 8 stay.  Clusters that do not fit wait for a whole request: 18 requests of 128
// tiles 80 us with 16 CTAs, of which 14 clusters fit, 67 with 8; 12 requests 65 and 68.
// Where the kernel may not have 16, 8.
int cluster_log2_for(void (*kernel)(VerifyArgs), bool warped, int tiles, int R) {
    int log2 = tiles >= 96 ? 4 : tiles >= 64 ? 3 : tiles >= 32 ? 2 : tiles >= 16 ? 1 : 0;
    if (log2 == 4 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        log2 = 3;
    }
    while (log2 > 0 && R > resident_clusters(kernel, warped, log2)) --log2;
    return log2;
}

int launch_verify(const VerifyArgs &args, int R, int tiles, cudaStream_t stream) {
    const bool warped = args.top_k > 0;
    const auto kernel = warped ? k_verify<true> : k_verify<false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVerifyDynSmem) != cudaSuccess)
        return DSBD_ERR_CUDA;
    const int cs = 1 << cluster_log2_for(kernel, warped, tiles, R);
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

extern "C" int dsbd_verify_cluster_ctas(const dsbd_forest_t *forest, const dsbd_verify_params_t *params, int32_t *resident) {
    if (check_forest(forest) != DSBD_OK || check_params(params) != DSBD_OK) return 0;
    const Layout L = make_layout(forest, params->V);
    const bool warped = params->top_k > 0;
    const auto kernel = warped ? k_verify<true> : k_verify<false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVerifyDynSmem) != cudaSuccess) cudaGetLastError();
    const int log2 = cluster_log2_for(kernel, warped, L.max_live * L.T, forest->R);
    if (resident) *resident = resident_clusters(kernel, warped, log2);
    return 1 << log2;
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
    a.R = f->R; a.B = f->B; a.N = f->N; a.gamma = f->max_depth;
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
    const int r = blockIdx.x, lane = threadIdx.x & 31, warp = warp_index();
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
#pragma unroll 1
    for (int i = warp; i < nA; i += kVWarps) {
        const double v = row_lse(a.stats + (int64_t)(b_lo + i) * a.T, a.T, a.inv_tau, lane);
        if (lane == 0) { lse[i] = v; a.lse_w[b_lo + i] = v; }
    }
    __syncthreads();
    if (warp == 0) live_weights(sh, 0, score, lse - b_lo, lane);
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
        if (!err) err = build_support<kVThreads>(a, sh, 0, lse - b_lo, hp, hq);
        if (!err && warp == 0) {
            finish_supports(ws, false, lane);
#pragma unroll 1
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
#pragma unroll 1
        for (int kk = warp; kk < n_draw; kk += kVWarps) {
            const double u = decision_uniform(a.seed, a.step, (uint32_t)r, d.layer, 3u, (uint32_t)kk);
            int ia = 0;
            const int tok = draw_cell(a, sh, u, false, 0.f, nullptr, 1, nullptr, reinterpret_cast<float *>(hp) + warp * kTokWords, lane, &ia);
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
    cfg.dynamicSmemBytes = kVerifyDynSmem;                             // the support's scratch, or what the draws search
    cfg.stream = stream;
    if (cudaFuncSetAttribute(k_draft, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVerifyDynSmem) != cudaSuccess)
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
    a.R = f->R; a.B = f->B; a.N = f->N; a.gamma = f->max_depth;
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
