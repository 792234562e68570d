// Forest attention on the 5th-generation tensor cores (tcgen05 + TMEM + TMA), bf16, d = 64 or 128.
//
// Work unit = (beam, KV head, row block): the query rows of the beam's draft tree that map to this KV
// head (row = node * group + head; blocks of at most NMAX = 32 or 64 rows) against the beam's KV
// prefix and then the tree's own keys and values under the ancestor-or-self mask.
//
// A draft tree has few query rows (36 for nine nodes and four heads per KV head), so the products are
// taken transposed: the TOKENS and the head dimension fill the 128 rows of an MMA and the query rows
// are its N columns, as many as there are (a multiple of 16):
//   S^T = K Q^T    (M = 128 tokens, N = rows, K = d)         both operands K-major in shared memory
//   O^T += V^T P^T (M = d, N = rows, K = 128 tokens)         both operands MN-major in shared memory
//
// One CTA per SM, groups of four warps:
//   softmax   NMAX / 16 groups, each with a share of the rows (at most 16 columns of S^T).  A thread owns
//             one token (its TMEM lane) and walks its group's rows, so a tile's exponentials are spread over
//             all 128 lanes however few rows there are.
//   output    O^T / row sum -> global, or the partial result of a cut unit.  The accumulators are double
//             buffered over the units, so the softmax goes straight on to the next unit.
//   then one warp each: TMA producer (K and V tiles of 128 tokens, boxes of 64 tokens x 64 columns with
//             128-byte swizzle, through two rings of shared-memory slots, and the unit's query rows), the
//             issuer of S^T (as many tiles ahead as there are S^T buffers), the issuer of O^T, and the one that
//             walks the work list and hands its segments to all others.
// Producer and issuers run converged and only predicate the copy / MMA instructions on one lane: issued from
// a branch of a single thread an MMA takes 95 cycles (the operands go to uniform registers lane by lane),
// issued like this 41 to 50 at N = 16 to 64 (M = 128, K = 16), which is the operand traffic of A.  One
// warp for both products took 2050 cycles a tile at d = 128, about as long as the tile's bytes take.
//
// A row's reference is its largest logit in the unit's first tile, moved to a later tile's largest when that exceeds
// it by more than 2^8.  The heaviest weight of a row is then mostly a power of two, which bf16 holds exactly: with the
// first token's logit as the reference (one barrier less a unit) the error against 64 bits was up to 7.5 % larger,
// at prefixes of about 70 tokens.  Weights in two terms (kSplit) do not need that: there the first token's logit is the
// reference, moved when exceeded by more than 2^40 (0.4 us of 31.3 for 8 x 4 beams after 512 to 2047 tokens).
//
// Work split: the tiles of a layer's units form one sequence (beam, KV head, row block), cut into equal
// runs, one per CTA; a unit that straddles a cut leaves partial results that k_attn_merge merges.
// Where whole units fill the CTAs about as evenly nothing is cut (make_plan).  Every CTA finds its own
// start with one scan over the beams; there is no plan kernel.
//
// Every mbarrier wait is bounded; on a time-out the kernel records DSBD_DEV_TIMEOUT, lets its copies
// and products land, frees its TMEM and returns.
#include <math.h>

#include <algorithm>

#include "dsbd_tc.cuh"

using namespace dsbd;

namespace {

constexpr int kTile = 128;              // tokens per tile = the M rows of the S^T product
constexpr int kMaxTree = DSBD_MAX_TREE_NODES;
static_assert(kMaxTree <= kBN, "a tree is one box: a part never starts behind the tree's root");
constexpr uint32_t kHalfStride = kTile * 128;        // bytes of one 64-column half of a tile (or of 64 rows of P)

// Shape of one kernel instance.  kSplit: the probabilities enter the second product as the sum of two
// bf16 terms (2^-17 relative); used at d = 64, where they were kept in fp32 by the kernel this one replaced.
template <int D, int NMAX>
struct Shape {
    static constexpr int kGroups = NMAX / 16;                 // softmax groups of 128 threads
    static constexpr int kCols = NMAX / kGroups, kCh = kCols / 8;               // rows of a group, in chunks of 8
    static constexpr int kThreads = kGroups * 128 + 256;
    static constexpr bool kSplit = D == 64;
    // The results depend on the unit's own values only, whatever lies behind them, as on the CUDA cores, which served
    // d = 64 before (d = 128 asks for finite values there).
    static constexpr bool kExactRanges = D == 64;
    static constexpr float kMoveRef = kSplit ? 40.f : 8.f;    // log2 of the factor by which a logit may exceed its row's reference
    static constexpr int kHalves = D / 64;                    // 64-column halves of a row of Q, K or V
    static constexpr uint32_t kSlot = kTile * D * 2;          // one K or V tile
    static constexpr uint32_t kPTerm = kHalfStride;                                     // [token][128 B]
    // Up to 32 rows: both terms in one operand (a token's 128 bytes: 32 rows of the first term, 32 of the second) and in columns of their
    // own of the accumulators, which the output adds.  A product of 48 or 64 columns takes as long as one of 32 (the
    // traffic of A), so a tile's O^T is issued in 500 cycles instead of 975; and four P buffers fit instead of two, so that S^T
    // no longer waits for the O^T two tiles back.  (8 x 4 beams after 512 to 2047 tokens: 31.5 us a call -> 30.5.)
    static constexpr bool kJoint = kSplit && NMAX == 32;
    static constexpr uint32_t kPBuf = (kSplit && !kJoint ? 2 : 1) * kPTerm;
    static constexpr int kPBufs = kJoint ? 4 : 2;
    static constexpr uint32_t kOCols = kJoint ? 2 * NMAX : NMAX;                        // of one unit's accumulators
    static constexpr bool kSWaits = D == 64 || NMAX == 64;                  // S^T waits until the tile's P buffer is free
    // query rows of one unit, or of two when they fit (a unit's copy then runs a whole unit ahead; with one
    // buffer its latency, 2800 cycles while HBM is saturated, shows at every unit's start)
    static constexpr uint32_t kQBytes = (D == 64 ? 17 : 21) * 1024;
    // K and V have rings of their own: each is consumed in order by one issuer, so that a wait for a slot's
    // next filling can never be satisfied by the one before it
    static constexpr int kKSlots = D == 64 ? 4 : 2, kVSlots = D == 64 ? 4 : 3;
    // order: K ring, V ring, P, Q (at d = 64 the upper 64 rows of the V^T operand alias the 16 KB after a slot,
    // which therefore must exist; rows of an MMA are independent and those rows are never read back)
    static constexpr uint32_t kOffV = kKSlots * kSlot, kOffP = kOffV + kVSlots * kSlot, kOffQ = kOffP + kPBufs * kPBuf;
    static constexpr uint32_t kSmem = kOffQ + kQBytes;
    // TMEM: four S^T buffers, then O^T of two units
    static constexpr uint32_t kSBufs = 4, kColO = kSBufs * NMAX, kTmemCols = NMAX == 32 ? 256 : 512;
};

// Tries of a wait before it gives up.  A try is suspended for 4 us here before it returns without success (4000 tries
// that failed took 16 ms), so this is about two seconds; 20e6 were 80.  A limit in clock cycles costs the waits
// 0.3 us of 31.2 (8 x 4 beams, heads of 64).
#ifdef DSBD_TEST_WAIT_TIMEOUT
// Test build only (a second library that no product path loads): waits give up after about a
// millisecond and the producer leaves out one tile, so that a wait runs out without anything
// faulting or hanging.  The test checks the status, and that the next launch of the normal
// library on the same context is correct.
constexpr uint32_t kWaitTries = 250;
#else
constexpr uint32_t kWaitTries = 500000;
#endif

// What a run left for the merge.  tail: its last unit (of the tree n_lo .. n_lo + n_tree) starts here and goes on in the next run;
// head_ends: the part of a unit that the run began with is the last one of that unit.
struct CutRec { int tail, head_ends, g, rb, n_lo, n_tree, pad0, pad1; };
// Whether a record names a unit of the forest.  One that nobody wrote (a CTA that left before) may hold anything, so no sum is made of it.
__host__ __device__ inline bool names_unit(const CutRec &rec, int N, int Hkv) {
    return (unsigned)rec.n_tree <= (unsigned)kMaxTree && rec.n_lo >= 0 && rec.n_lo <= N - rec.n_tree && (unsigned)rec.g < (unsigned)Hkv &&
           (unsigned)rec.rb <= (unsigned)kMaxTree;
}

struct TcArgs {
    int B, N, Hq, Hkv, group;
    int block_rows;                   // query rows per row block: whole nodes, at most NMAX
    int nodes_per_block;              // block_rows / group
    int q_nodes, q_rows, q_bufs;      // nodes of a query box, rows (a multiple of 8) and number of the Q buffers
    int n_layers;                     // >= 1: transformer layers in one launch (paged caches)
    int runs;                         // runs per layer; CTA c takes run c % runs of the layers c / runs + k * layer_step
    int layer_step;
    int unit_cost;                    // tiles that a unit's start and end are worth
    int uni_nt;                       // > 0: every unit has one row block and this many tiles
    int whole;                        // runs are whole units: nothing is cut
    int reread;                       // some tree has several row blocks: its prefix is read more than once
    float scale_log2;                 // scale * log2(e)
    const int32_t *beam_node_off, *parent;
    const int64_t *prefix_off;
    const int32_t *page_table;        // paged caches: page ids of beam b at page_off[b] ..; nullptr: packed
    const int64_t *page_off;
    __nv_bfloat16 *out;
    int32_t *status;
    // layer l uses the same page tables and forest; its pools, new keys/values, queries and outputs lie
    // l strides further
    int pool_layer_rows;              // rows of the pool map between consecutive layers
    int new_layer_rows;               // rows of the k_new / v_new maps between consecutive layers
    int64_t q_layer_stride;           // elements between consecutive layers' q (and out)
    int q_layer_nodes;                // the same in nodes (rows of the query map between consecutive layers)
    CutRec *recs;                     // [n_layers * runs]
    float *partial;                   // [2 * n_layers * runs][NMAX][D + 2]: reference, row sum, O; run i's first
                                      // unit in slot 2 i, its last one in slot 2 i + 1
};

// The part of one unit that a run holds: tiles [t0, t1).  layer = -1: the run is over.
struct __align__(16) Seg {
    int layer, b, g, rb, t0, t1;
    int whole;                             // the part is the whole unit
    int last;                              // it holds the unit's last tile
    int nhp, nh, L;                        // boxes of 64 tokens (the prefix's; with the tree's), prefix tokens
    int n_lo, n_tree, rows;                // the tree, the query rows of the row block
    int pad[2];
};

constexpr int kMaxSlots = 4, kSegs = 8;
struct Barriers {
    unsigned long long k_full[kMaxSlots], k_empty[kMaxSlots], v_full[kMaxSlots], v_empty[kMaxSlots];
    unsigned long long s_full[4], p_full[4], pv_done[4], q_full[2], q_empty[2];
    unsigned long long sum_full[2], o_full[2], o_empty[2];     // by unit parity
    unsigned long long drain[2];
    unsigned long long seg_full[kSegs], seg_empty[kSegs];
    Seg seg[kSegs];
    uint32_t tmem_base;
    int abort;
    int scan[32];                          // warp sums of the start-up scan
    int start[3];                          // beam, unit inside the beam, cost offset inside the unit
    int run;                               // cost of the run
};
// (The groups are not in step: what a group changes on its own is its own, since the share of the rows that a
// column belongs to differs from unit to unit.)
struct SoftmaxShared {
    float negref[4][16];                   // [group] minus the row references (log2 units)
    float ref[2][64];                      // [unit parity] the references a unit ended with
    float red[2][4][64];                   // [unit parity] row sums per warp quarter
    float colmax[4][4][16];                // [group] column maxima per warp quarter
    float move[4][16];                     // [group] rescale factors when references move
    float fac[64];                         // 1 / row sum
    int rowoff[64];                        // output offset of a row inside its block
    int16_t par[4][kMaxTree];              // [group] the tree's parents, local
    uint32_t see[4][kMaxTree];             // [group] tree token j: the group's rows that see it
};

// Bounded wait: false if it gave up (time-out here, or another role already aborted; the kernel's end reports it).
__device__ __forceinline__ bool mbar_wait(void *bar, uint32_t parity, Barriers *sb) {
#pragma unroll 1
    for (uint32_t i = 0; !mbar_try(bar, parity); ++i)
        if (i == kWaitTries || *reinterpret_cast<volatile int *>(&sb->abort)) {
            *reinterpret_cast<volatile int *>(&sb->abort) = 1;
            return false;
        }
    return true;
}

// Barrier of the 128 threads of group g (softmax groups, then the output warps; id 0 is __syncthreads),
// plain and with an OR.  The warps arrive, and leave, converged: the TMEM accesses between the barriers
// need whole warps.
__device__ __forceinline__ void group_sync(int g) {
    __syncwarp();
    asm volatile("barrier.cta.sync.aligned %0, 128;" ::"r"(g + 1) : "memory");
}
__device__ __forceinline__ bool group_any(int g, bool v) {
    uint32_t r;
    __syncwarp();
    asm volatile(
        "{\n\t.reg .pred a, b;\n\tsetp.ne.u32 a, %1, 0;\n\t"
        "barrier.cta.red.or.pred.aligned b, %2, 128, a;\n\tselp.u32 %0, 1, 0, b;\n\t}"
        : "=r"(r) : "r"((uint32_t)v), "r"(g + 1) : "memory");
    return r != 0;
}
// A bounded wait by a converged warp: the same answer on every lane.
__device__ __forceinline__ bool warp_wait(void *bar, uint32_t parity, Barriers *sb) {
    return __all_sync(kFull, mbar_wait(bar, parity, sb));
}
// After a time-out: waits (again with a limit) until the products this warp has issued are done, so that TMEM
// and shared memory can be given back.
__device__ __forceinline__ bool land(void *bar, uint32_t parity) {
    uint32_t i = 0;
#pragma unroll 1
    while (!__all_sync(kFull, mbar_try(bar, parity)) && i < kWaitTries) ++i;
    return i < kWaitTries;
}
__device__ __forceinline__ void drain(bool on, void *bar) {
    tc_commit(on, bar);
    land(bar, 0);
}

// Two fp32 operations an instruction (sm_100), and a maximum of three.
struct F2 { float x, y; };
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 d;
    asm("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 d;
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "add.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Combines 8 columns over the 32 lanes with 9 shuffles; lane i ends up with column i & 7 in v[0].
template <class F>
__device__ __forceinline__ void fold8(float *v, int lane, F op) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float send = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
            v[i] = op(keep, __shfl_xor_sync(kFull, send, o));
        }
    }
    v[0] = op(v[0], __shfl_xor_sync(kFull, v[0], 8));
    v[0] = op(v[0], __shfl_xor_sync(kFull, v[0], 16));
}

// Facts of a beam: prefix length, tree, boxes of 64 tokens (the prefix's, then the tree's), tiles of a
// unit (two boxes each), row blocks.
struct BeamFacts { int L, n_lo, n_tree, nhp, nh, nt, nrb; };
__device__ __forceinline__ BeamFacts beam_facts(const TcArgs &a, int b) {
    BeamFacts f;
    f.L = (int)(a.prefix_off[b + 1] - a.prefix_off[b]);
    f.n_lo = a.beam_node_off[b];
    f.n_tree = min(max(a.beam_node_off[b + 1] - f.n_lo, 0), kMaxTree);
    f.nhp = (f.L + kBN - 1) / kBN;
    f.nh = f.nhp + (f.n_tree + kBN - 1) / kBN;
    f.nt = (f.nh + 1) / 2;
    f.nrb = max(1, (f.n_tree * a.group + a.block_rows - 1) / a.block_rows);
    return f;
}

// Walks the runs of this CTA.  One warp does and hands the segments to the others, so that the beams' data
// is fetched ahead and the walk's code exists once (with a copy in every role the kernel outgrew the
// instruction cache: a fifth of all stalls at three tiles a unit).
// Ragged runs are equal in cost: a unit costs its tiles plus unit_cost for its start and end (without it the
// CTAs that met the short prefixes of a batch of 99 to 4911 tokens ended at 172 us, the median at 128).
struct Cursor {
    int left, layer, b, k, at, loaded;       // at: cost offset inside the unit
    BeamFacts f;
    __device__ __forceinline__ Cursor(const TcArgs &a, const Barriers &sb) {
        layer = a.whole && a.uni_nt ? 0 : (int)blockIdx.x / a.runs;
        loaded = -1;
        rewind(sb);
        if (a.whole && a.uni_nt) { layer = b / a.B; b -= layer * a.B; }      // the layers' units are one sequence
    }
    __device__ __forceinline__ void rewind(const Barriers &sb) {
        left = sb.run; b = sb.start[0]; k = sb.start[1]; at = sb.start[2];
    }
    __device__ __forceinline__ bool next(const TcArgs &a, const Barriers &sb, Seg &s) {
        while (layer < a.n_layers) {
            if (left <= 0 || b >= a.B) {
                if (a.whole && a.uni_nt) {
                    if (left <= 0) return false;
                    b = 0; ++layer;
                    continue;
                }
                layer += a.layer_step;
                rewind(sb);
                if (left <= 0) return false;
                continue;
            }
            if (loaded != b) { f = beam_facts(a, b); loaded = b; }
            s.layer = layer; s.b = b; s.g = f.nrb == 1 ? k : k / f.nrb; s.rb = k - s.g * f.nrb;
            const int extra = a.uni_nt ? 0 : a.unit_cost, stop = min(f.nt + extra, at + left);
            s.t0 = max(at - extra, 0); s.t1 = max(stop - extra, 0);
            s.whole = s.t0 == 0 && s.t1 == f.nt; s.last = s.t1 == f.nt;
            s.nhp = f.nhp; s.nh = f.nh; s.L = f.L; s.n_lo = f.n_lo; s.n_tree = f.n_tree;
            s.rows = min(a.block_rows, f.n_tree * a.group - s.rb * a.block_rows);
            left -= stop - at;
            at = 0;
            if (++k == f.nrb * a.Hkv) { k = 0; ++b; }
            if (s.t1 > s.t0) return true;
        }
        return false;
    }
};

// The unit-th segment, for a converged warp; false after the last one or a time-out.
__device__ __forceinline__ bool get_seg(Barriers &sb, uint32_t unit, Seg &s) {
    const uint32_t i = unit % kSegs;
    if (!warp_wait(&sb.seg_full[i], (unit / kSegs) & 1, &sb)) return false;
    s = sb.seg[i];
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&sb.seg_empty[i]);
    return s.layer >= 0;
}

// Start of the r-th of G nearly equal shares of n.
__device__ __forceinline__ int share(int n, int r, int G) { return n / G * r + min(r, n % G); }

// Finds the run of this CTA: first unit and tile, number of tiles (all threads).
template <int kThreads>
__device__ void find_run(const TcArgs &a, Barriers &sb) {
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(kFull, tid >> 5, 0);
    const bool joint = a.whole && a.uni_nt;                   // the units of all layers in one sequence
    const int r = joint ? (int)blockIdx.x : (int)blockIdx.x % a.runs, G = joint ? (int)gridDim.x : a.runs;
    const int units = a.B * a.Hkv * (joint ? a.n_layers : 1);     // (where row blocks are one per tree)
    if (a.uni_nt > 0 || a.whole) {
        if (tid == 0) {
            const int nt = a.uni_nt;
            int lo, hi, unit;
            if (a.whole) {
                unit = share(units, r, G);
                lo = 0; hi = (share(units, r + 1, G) - unit) * nt;
                if (nt == 0) { hi = beam_facts(a, unit / a.Hkv).nt + a.unit_cost; }      // ragged: one unit per run
            } else {
                lo = share(units * nt, r, G); hi = share(units * nt, r + 1, G);
                unit = lo / nt;
            }
            sb.start[0] = unit / a.Hkv; sb.start[1] = unit % a.Hkv; sb.start[2] = a.whole ? 0 : lo - unit * nt;
            sb.run = hi - lo;
        }
        __syncthreads();
        return;
    }
    // cost before every thread's share of the beams
    const int per = (a.B + kThreads - 1) / kThreads;
    const int b0 = min(tid * per, a.B), b1 = min(b0 + per, a.B);
    int sum = 0;
    BeamFacts f = {};                                        // of the last beam of the share (nearly always its only one)
#pragma unroll 1
    for (int b = b0; b < b1; ++b) {
        f = beam_facts(a, b);
        sum += (f.nt + a.unit_cost) * f.nrb * a.Hkv;
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) sb.scan[warp] = incl;
    if (tid == 0) { sb.start[0] = 0; sb.start[1] = 0; sb.start[2] = 0; sb.run = 0; }
    __syncthreads();
    static_assert(kThreads <= 1024, "the warps' sums fit the lanes");
    const int scan = lane < kThreads / 32 ? sb.scan[lane] : 0;
    const int before = incl - sum + __reduce_add_sync(kFull, lane < warp ? scan : 0), total = __reduce_add_sync(kFull, scan);
    const int lo = share(total, r, G), hi = share(total, r + 1, G);
    if (lo < hi && lo >= before && lo < before + sum) {
        int at = before;
#pragma unroll 1
        for (int b = b0; b < b1; ++b) {
            if (per > 1) f = beam_facts(a, b);
            const int cost = f.nt + a.unit_cost, w = cost * f.nrb * a.Hkv;
            if (lo < at + w) {
                sb.start[0] = b; sb.start[1] = (lo - at) / cost; sb.start[2] = (lo - at) % cost;
                sb.run = hi - lo;
                break;
            }
            at += w;
        }
    }
    __syncthreads();
}

template <int D, int NMAX>
__global__ void __launch_bounds__(Shape<D, NMAX>::kThreads, 1)
k_forest_attn_tr(const __grid_constant__ CUtensorMap map_kp, const __grid_constant__ CUtensorMap map_vp,
                 const __grid_constant__ CUtensorMap map_kn, const __grid_constant__ CUtensorMap map_vn,
                 const __grid_constant__ CUtensorMap map_q, TcArgs a) {
    using S = Shape<D, NMAX>;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *p_s = smem + S::kOffP, *q_s = smem + S::kOffQ;
    __shared__ Barriers sb;
    __shared__ __align__(16) SoftmaxShared sx;
    const int warp = __shfl_sync(kFull, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    constexpr int kGroups = S::kGroups, kWarpOut = kGroups * 4, kWarpTma = kWarpOut + 4, kWarpS = kWarpTma + 1,
                  kWarpO = kWarpTma + 2, kWarpSeg = kWarpTma + 3;
    if ((smem_u32(smem) & 1023u) != 0u) {                    // the swizzled operands need 1024-byte alignment
        if (threadIdx.x == 0) report(a.status, DSBD_DEV_BAD_FOREST);
        return;
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxSlots; ++s) {
            mbar_init(&sb.k_full[s], 1); mbar_init(&sb.k_empty[s], 1);
            mbar_init(&sb.v_full[s], 1); mbar_init(&sb.v_empty[s], 1);
        }
        for (int b = 0; b < 4; ++b) { mbar_init(&sb.s_full[b], 1); mbar_init(&sb.p_full[b], kGroups * 4); mbar_init(&sb.pv_done[b], 1); }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sb.q_full[b], 1); mbar_init(&sb.q_empty[b], 1);
            mbar_init(&sb.sum_full[b], kGroups * 4); mbar_init(&sb.o_full[b], 1); mbar_init(&sb.o_empty[b], 4);
            mbar_init(&sb.drain[b], 1);
        }
        for (int i = 0; i < kSegs; ++i) { mbar_init(&sb.seg_full[i], 1); mbar_init(&sb.seg_empty[i], kGroups * 4 + 7); }
        sb.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kWarpS) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sb.tmem_base)),
                     "r"(S::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // query rows past a block's last one are never copied in: keep them finite
    for (uint32_t i = threadIdx.x * 16; i < S::kQBytes; i += S::kThreads * 16)
        *reinterpret_cast<uint4 *>(q_s + i) = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (threadIdx.x < 64) {
        const int node = (int)threadIdx.x / a.group;
        sx.rowoff[threadIdx.x] = (node * a.Hq + (int)threadIdx.x - node * a.group) * D;
    }
    // launched with programmatic stream serialization: what is above overlaps the kernel before
    asm volatile("griddepcontrol.wait;" ::: "memory");
    tc_fence_before();
    find_run<S::kThreads>(a, sb);                            // (has the block barriers)
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(kFull, *reinterpret_cast<volatile uint32_t *>(&sb.tmem_base), 0);
    Seg sg;
    // four softmax groups: 4 x 96 + 2 x 48 = the 6 x 80 registers per lane of the launch
    if (kGroups == 4 && warp >= kWarpOut) asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");

    if (warp == kWarpTma) {
        // ------------------------------------------------------------ TMA producer
        const bool on = lane == 0;
        uint32_t n_k = 0, n_v = 0, unit = 0;                 // K and V tiles so far
        bool ok = true;
        // keys and values are read once: their lines are the first to leave L2 again, so that the queries and the
        // metadata the units keep coming back to stay there (the row blocks of a big tree read the same prefix:
        // ordinary policy)
        uint64_t pol;
        if (!a.reread) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
        else asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
        const uint32_t ring = smem_u32(smem);
        while (ok && get_seg(sb, unit, sg)) {
            const int row0 = a.page_table ? 0 : (int)(a.prefix_off[sg.b] * a.Hkv + (int64_t)sg.g * sg.L);
            const int32_t *pages = a.page_table ? a.page_table + a.page_off[sg.b] : nullptr;
            int pg[2] = {0, 0};                              // pages of the next tile's two boxes
            auto fetch_pages = [&](int h) {
                if (!pages) return;
                if (h < sg.nhp) pg[0] = pages[h];
                if (h + 1 < sg.nhp) pg[1] = pages[h + 1];
            };
            fetch_pages(2 * sg.t0);
            auto load_tile = [&](int j, int kv) -> bool {    // K or V of tile j into the next slot
                const uint32_t slots = kv ? S::kVSlots : S::kKSlots, n = kv ? n_v : n_k, s = n % slots;
                void *full = kv ? &sb.v_full[s] : &sb.k_full[s], *empty = kv ? &sb.v_empty[s] : &sb.k_empty[s];
                if (!warp_wait(empty, ((n / slots) & 1) ^ 1, &sb)) return false;
                if (kv) ++n_v; else ++n_k;
                const int boxes = min(2, sg.nh - 2 * j);
                const uint32_t dst = ring + (kv ? S::kOffV : 0) + s * S::kSlot;
                mbar_expect_tx_if(on, full, (uint32_t)boxes * kBN * D * 2);
#ifdef DSBD_TEST_WAIT_TIMEOUT
                if (n == 1 && !kv && blockIdx.x == 0) return true;   // the bytes this barrier expects never come
#endif
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    if (i >= boxes) break;
                    const int h = 2 * j + i;
                    const bool tree = h >= sg.nhp;
                    const CUtensorMap *map = tree ? (kv ? &map_vn : &map_kn) : (kv ? &map_vp : &map_kp);
                    const int x = tree ? sg.g * D : 0;
                    const int y = tree ? sg.n_lo + (h - sg.nhp) * kBN + sg.layer * a.new_layer_rows
                                  : pages ? (pg[i] * a.Hkv + sg.g) * kBN + sg.layer * a.pool_layer_rows : row0 + h * kBN;
#pragma unroll
                    for (int hc = 0; hc < S::kHalves; ++hc)
                        tma_load_2d_hint(on, dst + hc * kHalfStride + i * (kHalfStride / 2), map, x + hc * 64, y, full, pol);
                }
                return true;
            };
            // K and V of the tiles in turn.  The first K tile does not have to wait for the query rows, whose
            // buffer is free once the last S^T product of the unit that had it has completed.
            const uint32_t qb = unit & (a.q_bufs - 1), q_use = unit >> (a.q_bufs - 1);      // (one or two buffers)
#pragma unroll 1
            for (int i = 0; i < 2 * (sg.t1 - sg.t0) && ok; ++i) {
                if (i >= 2 && !(i & 1)) fetch_pages(2 * (sg.t0 + i / 2));
                ok = load_tile(sg.t0 + i / 2, i & 1);
                if (i == 0 && ok) {
                    ok = warp_wait(&sb.q_empty[qb], (q_use & 1) ^ 1, &sb);
                    if (!ok) break;
                    const int z = sg.n_lo + sg.rb * a.nodes_per_block + sg.layer * a.q_layer_nodes;
                    mbar_expect_tx_if(on, &sb.q_full[qb], (uint32_t)(a.q_nodes * a.group) * D * 2);
#pragma unroll
                    for (int hc = 0; hc < S::kHalves; ++hc)
                        tma_load_3d(on, smem_u32(q_s) + (qb * S::kHalves + hc) * a.q_rows * 128, &map_q, hc * 64,
                                    sg.g * a.group, z, &sb.q_full[qb]);
                    ++unit;
                }
            }
        }
        if (!ok) {
            // let the copies already issued land before the CTA goes away
            auto land_all = [&](unsigned long long *full, uint32_t n, uint32_t slots) {
#pragma unroll 1
                for (uint32_t k = 1; k <= slots && k <= n; ++k) land(&full[(n - k) % slots], ((n - k) / slots) & 1);
            };
            land_all(sb.k_full, n_k, S::kKSlots);
            land_all(sb.v_full, n_v, S::kVSlots);
            land_all(sb.q_full, unit, (uint32_t)a.q_bufs);
        }
    } else if (warp == kWarpS) {
        // ------------------------------------------------------------ S^T issuer
        const bool on = lane == 0;
        uint32_t tile = 0, unit = 0;
        bool ok = true;
        while (ok && get_seg(sb, unit, sg)) {
            const uint32_t idesc = instr_desc(kTile, max(16, (sg.rows + 15) & ~15), 0, 0);
            const uint32_t qb = unit & (a.q_bufs - 1), q_half = (uint32_t)a.q_rows * 128;
            const uint64_t qd = desc_k_major(smem_u32(q_s) + qb * S::kHalves * q_half);
            ok = warp_wait(&sb.q_full[qb], (unit >> (a.q_bufs - 1)) & 1, &sb);
#pragma unroll 1
            for (int j = sg.t0; j < sg.t1 && ok; ++j, ++tile) {
                const uint32_t s = tile % S::kKSlots, sbuf = tile % S::kSBufs;
                ok = warp_wait(&sb.k_full[s], (tile / S::kKSlots) & 1, &sb);
                // The softmax has read what the buffer held.  Where the softmax sets the pace (d = 64, more than 32
                // rows): wait for the O^T product that last read the tile's P buffer, which came after; S^T then also says
                // that the buffer is free.  Where HBM does: no longer than needed, so that the K slot is free early.
                if (S::kSWaits) {
                    if (ok && tile >= S::kPBufs) ok = warp_wait(&sb.pv_done[tile % S::kPBufs], (tile / S::kPBufs - 1) & 1, &sb);
                } else if (ok && tile >= S::kSBufs) {
                    ok = warp_wait(&sb.p_full[sbuf], (tile / S::kSBufs - 1) & 1, &sb);
                }
                if (!ok) break;
                tc_fence_after();
                const uint64_t kd = desc_k_major(smem_u32(smem + s * S::kSlot));
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks)
                    mma_ss(on, tmem + sbuf * NMAX, kd + (uint64_t)((ks / 4) * (kHalfStride >> 4) + (ks % 4) * 2),
                           qd + (uint64_t)((ks / 4) * (q_half >> 4) + (ks % 4) * 2), idesc, ks > 0);
                tc_commit(on, &sb.k_empty[s]);
                tc_commit(on, &sb.s_full[sbuf]);
                if (j + 1 == sg.t1) tc_commit(on, &sb.q_empty[qb]);          // the unit's last S^T product
            }
            ++unit;
        }
        if (!ok) drain(on, &sb.drain[0]);
    } else if (warp == kWarpO) {
        // ------------------------------------------------------------ O^T issuer
        const bool on = lane == 0;
        uint32_t tile = 0, unit = 0;
        bool ok = true;
        while (ok && get_seg(sb, unit, sg)) {
            const uint32_t idesc = instr_desc(128, (S::kJoint ? NMAX : 0) + max(16, (sg.rows + 15) & ~15), 1, 1);
            const uint32_t col = tmem + S::kColO + (unit & 1) * S::kOCols;
            // the accumulators were last used two units ago
            ok = warp_wait(&sb.o_empty[unit & 1], ((unit >> 1) & 1) ^ 1, &sb);
#pragma unroll 1
            for (int j = sg.t0; j < sg.t1 && ok; ++j, ++tile) {
                const uint32_t s = tile % S::kVSlots;
                ok = warp_wait(&sb.v_full[s], (tile / S::kVSlots) & 1, &sb);
                if (S::kExactRanges && ok && (2 * j + 2) * kBN > sg.L) {      // (while the weights are worked out)
                    // rows that a box holds past the end of the prefix or of the tree: the weights there are zero, but
                    // zero times a NaN or an infinity of someone else's values is not
#pragma unroll 1
                    for (int i = 0; i < 2; ++i) {
                        const int h = 2 * j + i, end = h < sg.nhp ? sg.L - h * kBN : sg.n_tree - (h - sg.nhp) * kBN;
                        uint4 *box = reinterpret_cast<uint4 *>(smem + S::kOffV + s * S::kSlot + i * (kHalfStride / 2));
                        if (h < sg.nh)
#pragma unroll 1
                            for (int e = end * 8 + lane; e < kBN * 8; e += 32) box[e] = make_uint4(0u, 0u, 0u, 0u);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                }
                if (ok) ok = warp_wait(&sb.p_full[tile % S::kSBufs], (tile / S::kSBufs) & 1, &sb);
                if (!ok) break;
                tc_fence_after();
                const uint64_t vd = desc_mn_major(smem_u32(smem + S::kOffV + s * S::kSlot), kHalfStride);
                const bool both = sg.nh - 2 * j >= 2;        // a lone box: 64 tokens
                const uint32_t acc = j > sg.t0 ? 1u : 0u;
#pragma unroll
                for (int term = 0; term < (S::kSplit && !S::kJoint ? 2 : 1); ++term) {
                    const uint64_t pd = desc_mn_major(
                        smem_u32(p_s + (tile % S::kPBufs) * S::kPBuf + term * S::kPTerm), kHalfStride);
#pragma unroll
                    for (int ks = 0; ks < kTile / 16; ++ks)
                        mma_ss(on && (ks < 4 || both), col, vd + (uint64_t)(ks * ((16 * 128) >> 4)),
                               pd + (uint64_t)(ks * ((16 * 128) >> 4)), idesc, (term + ks > 0) ? 1u : acc);
                }
                tc_commit(on, &sb.v_empty[s]);
                tc_commit(on, &sb.pv_done[tile % S::kPBufs]);
            }
            if (ok) tc_commit(on, &sb.o_full[unit & 1]);
            ++unit;
        }
        if (!ok) drain(on, &sb.drain[1]);
    } else if (warp == kWarpSeg) {
        // ------------------------------------------------------------ segments
        Cursor cur(a, sb);
        for (uint32_t unit = 0; ; ++unit) {
            const bool more = cur.next(a, sb, sg);
            if (!more) sg.layer = -1;
            const uint32_t i = unit % kSegs;
            if (!warp_wait(&sb.seg_empty[i], ((unit / kSegs) & 1) ^ 1, &sb)) break;
            if (lane == 0) {
                sb.seg[i] = sg;
                mbar_arrive(&sb.seg_full[i]);
            }
            if (!more) break;
        }
    } else if (warp >= kWarpOut && warp < kWarpTma) {
        // ------------------------------------------------------------ output
        const int q = warp & 3, tid = threadIdx.x & 127;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        uint32_t unit = 0;
        CutRec rec = {};
        int rec_layer = a.whole ? 0 : (int)blockIdx.x / a.runs;
        auto put_rec = [&](int layer) {
            if (!a.whole && tid == 0) a.recs[layer * a.runs + (int)blockIdx.x % a.runs] = rec;
        };
        // (the merge reads the records of all layers, also of those a CTA does not reach after a time-out)
        if (!a.whole)
            for (int l = rec_layer; l < a.n_layers; l += a.layer_step) put_rec(l);
        while (get_seg(sb, unit, sg)) {
            if (sg.layer != rec_layer) { put_rec(rec_layer); rec = CutRec{}; rec_layer = sg.layer; }
            const int rows = sg.rows;
            const uint32_t ub = unit & 1;
            const uint32_t o_addr = tmem + lane_base + S::kColO + ub * S::kOCols;
            bool ok = warp_wait(&sb.sum_full[ub], (unit >> 1) & 1, &sb);
            if (ok) ok = warp_wait(&sb.o_full[ub], (unit >> 1) & 1, &sb);
            if (group_any(kGroups, !ok)) break;
            tc_fence_after();
            const bool whole = sg.whole;
            float *part = a.partial;
            if (!whole) {
                part += (2 * ((int64_t)sg.layer * a.runs + (int)blockIdx.x % a.runs) + (sg.t0 == 0 ? 1 : 0)) *
                        NMAX * (D + 2);
                if (sg.t0 > 0) rec.head_ends = sg.last;
                else { rec.tail = 1; rec.g = sg.g; rec.rb = sg.rb; rec.n_lo = sg.n_lo; rec.n_tree = sg.n_tree; }
            }
            if (tid < rows) {
                const float sum = (sx.red[ub][0][tid] + sx.red[ub][1][tid]) + (sx.red[ub][2][tid] + sx.red[ub][3][tid]);
                if (whole) {
                    sx.fac[tid] = 1.f / sum;
                } else {
                    sx.fac[tid] = 1.f;
                    part[tid * (D + 2)] = sum > 0.f ? sx.ref[ub][tid] : -INFINITY;
                    part[tid * (D + 2) + 1] = sum;
                }
            }
            group_sync(kGroups);
            if (tid < D) {                                   // (d = 64: lanes 64.. hold aliased rows; whole warps)
                __nv_bfloat16 *dst = a.out + (int64_t)sg.layer * a.q_layer_stride +
                                     ((int64_t)(sg.n_lo + sg.rb * a.nodes_per_block) * a.Hq + sg.g * a.group) * D +
                                     (tid & ~1);
#pragma unroll 1
                for (int r0 = 0; r0 < rows; r0 += 8) {
                    uint32_t ov[8], ow[8];
                    tmem_ld8(o_addr + r0, ov);
                    if (S::kJoint) tmem_ld8(o_addr + NMAX + r0, ow);
                    tmem_wait_ld();
                    if (S::kJoint) {
#pragma unroll
                        for (int c = 0; c < 8; ++c) ov[c] = __float_as_uint(__uint_as_float(ov[c]) + __uint_as_float(ow[c]));
                    }
                    float v[8];
#pragma unroll
                    for (int c = 0; c < 8; c += 4) {
                        const float4 f = *reinterpret_cast<const float4 *>(&sx.fac[r0 + c]);
                        v[c] = __uint_as_float(ov[c]) * f.x; v[c + 1] = __uint_as_float(ov[c + 1]) * f.y;
                        v[c + 2] = __uint_as_float(ov[c + 2]) * f.z; v[c + 3] = __uint_as_float(ov[c + 3]) * f.w;
                    }
                    if (whole) {
                        // two lanes swap halves of two rows, so that each stores a pair of columns of one row
#pragma unroll
                        for (int c = 0; c < 8; c += 2) {
                            const int row = r0 + c + (lane & 1);
                            const float swap = __shfl_xor_sync(kFull, (lane & 1) ? v[c] : v[c + 1], 1);
                            const uint32_t w = (lane & 1) ? pack_bf16(swap, v[c + 1]) : pack_bf16(v[c], swap);
                            if (row < rows) *reinterpret_cast<uint32_t *>(dst + sx.rowoff[row]) = w;
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            if (r0 + c < rows) part[(r0 + c) * (D + 2) + 2 + tid] = v[c];
                    }
                    __syncwarp();
                }
            }
            tc_fence_before();
            group_sync(kGroups);                             // (the factors are read before they are written again)
            if (lane == 0) mbar_arrive(&sb.o_empty[ub]);
            ++unit;
        }
        put_rec(rec_layer);
    } else if (warp < kWarpOut) {
        if (kGroups == 4) asm volatile("setmaxnreg.inc.sync.aligned.u32 96;");
        // ------------------------------------------------------------ softmax groups
        const int grp = warp >> 2, q = warp & 3, tok = threadIdx.x & 127;     // token inside the tile = TMEM lane
        const int box = tok >> 6, in_box = tok & 63;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        uint32_t tile = 0, unit = 0;
        int mask_b = -1, mask_rb = -1;                       // the tree whose mask this group holds
        bool ok = true;
        while (get_seg(sb, unit, sg)) {
            // the group's columns: chunks of 8 rows, shared out evenly
            const int rows = sg.rows;
            const int n8 = (rows + 7) / 8, per = (n8 + kGroups - 1) / kGroups;
            const int cbase = grp * per * 8, nch = min(max(n8 - grp * per, 0), per);
            const uint32_t o_addr = tmem + lane_base + S::kColO + (unit & 1) * S::kOCols + cbase;
            float l[S::kCols];
#pragma unroll
            for (int c = 0; c < S::kCols; ++c) l[c] = 0.f;
#pragma unroll 1
            for (int j = sg.t0; j < sg.t1; ++j, ++tile) {
                // what this thread's token is: a prefix token every row sees, a tree token some rows see,
                // or nothing
                const int h = 2 * j + box;
                const bool plain = (2 * j + 2) * kBN <= sg.L;
                uint32_t see = ~0u;
                if (!plain) {
                    if (2 * j + 2 > sg.nhp && (mask_b != sg.b || mask_rb != sg.rb)) {
                        // which rows of the group see tree token j: the rows whose node has j on its path to
                        // the root (kept over the KV heads of a beam)
                        mask_b = sg.b; mask_rb = sg.rb;
                        if (tok < sg.n_tree) {
                            const int par = a.parent[sg.n_lo + tok];
                            int p = par - sg.n_lo;
                            // (the entry point's rules differ: d = 64 reports every parent outside the tree)
                            const bool bad = D == 64 ? (p < 0 || p >= tok) && (tok > 0 || par != -1) : par >= 0 && p >= tok;
                            if (bad) report(a.status, DSBD_DEV_BAD_FOREST);
                            if (par < 0 || p < 0 || p >= tok) p = -1;
                            sx.par[grp][tok] = (int16_t)p;
                        }
                        if (tok < kMaxTree) sx.see[grp][tok] = 0u;
                        group_sync(grp);
                        if (tok < nch * 8 && cbase + tok < rows)
#pragma unroll 1
                            for (int n = (sg.rb * a.block_rows + cbase + tok) / a.group; n >= 0; n = sx.par[grp][n])
                                atomicOr(&sx.see[grp][n], 1u << tok);
                        group_sync(grp);
                    }
                    const int jt = (h - sg.nhp) * kBN + in_box;
                    if (h < sg.nhp) {
                        if (h * kBN + in_box >= sg.L) see = 0u;
                    } else if (h < sg.nh && jt < sg.n_tree) {
                        see = sx.see[grp][jt];
                    } else {
                        see = 0u;
                    }
                }
                ok = warp_wait(&sb.s_full[tile % S::kSBufs], (tile / S::kSBufs) & 1, &sb);
                tc_fence_after();
                const bool work = ok && nch > 0 && h < sg.nh;   // (a lone box leaves the upper two warps idle)
                const uint32_t s_addr = tmem + lane_base + (tile % S::kSBufs) * NMAX + cbase;
                // the columns' maxima over the tile's tokens that their rows see, times the scale (> 0, checked by the
                // host): thread tok has column tok of the group's
                auto column_max = [&] {
#pragma unroll 1
                    for (int ch = 0; ch < nch; ++ch) {
                        uint32_t v[8];
                        if (work) tmem_ld8(s_addr + ch * 8, v);
                        tmem_wait_ld();
                        float f[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            f[i] = work && ((see >> (ch * 8 + i)) & 1u) ? __uint_as_float(v[i]) : -INFINITY;
                        fold8(f, lane, [](float x, float y) { return fmaxf(x, y); });
                        if (lane < 8) sx.colmax[grp][q][ch * 8 + lane] = f[0];
                        __syncwarp();
                    }
                    group_sync(grp);
                    return tok < nch * 8 ? fmaxf(fmaxf(sx.colmax[grp][0][tok], sx.colmax[grp][1][tok]),
                                                 fmaxf(sx.colmax[grp][2][tok], sx.colmax[grp][3][tok])) * a.scale_log2
                                         : 0.f;
                };
                if (j == sg.t0) {                            // the first tile sets the references
                    if (!S::kSplit) {
                        const float m = column_max();
                        if (tok < nch * 8) sx.negref[grp][tok] = m > -INFINITY ? -m : 0.f;
                    } else if (q == 0 && work) {             // (its first token is a prefix token or the root)
                        uint32_t v[S::kCols];
#pragma unroll
                        for (int ch = 0; ch < S::kCh; ++ch)
                            if (ch < nch) tmem_ld8(s_addr + ch * 8, v + ch * 8);
                        tmem_wait_ld();
                        if (tok == 0) {
#pragma unroll
                            for (int c = 0; c < S::kCols; c += 4)
                                if (c / 8 < nch)
                                    *reinterpret_cast<float4 *>(&sx.negref[grp][c]) =
                                        make_float4(-__uint_as_float(v[c]) * a.scale_log2, -__uint_as_float(v[c + 1]) * a.scale_log2,
                                                    -__uint_as_float(v[c + 2]) * a.scale_log2, -__uint_as_float(v[c + 3]) * a.scale_log2);
                        }
                    }
                    group_sync(grp);
                }
                // the P buffer is free once the product that last read it has landed
                if (!S::kSWaits && ok && tile >= S::kPBufs)
                    ok = warp_wait(&sb.pv_done[tile % S::kPBufs], (tile / S::kPBufs - 1) & 1, &sb);
                // the weights: bf16 pairs (SPLIT: the sums of their two terms) of the group's rows
                constexpr int kW = S::kSplit ? S::kCols : S::kCols / 2;
                uint32_t w[kW];
                float over = 0.f;                            // how far logits exceed the references
                for (int attempt = 0; ; ++attempt) {
                    if (work && ok) {
                        over = 0.f;
                        uint32_t sv[S::kCols];
#pragma unroll
                        for (int ch = 0; ch < S::kCh; ++ch)
                            if (ch < nch) tmem_ld8(s_addr + ch * 8, sv + ch * 8);
                        tmem_wait_ld();
                        if (!plain) {
#pragma unroll
                            for (int c = 0; c < S::kCols; ++c)
                                if (!((see >> c) & 1u)) sv[c] = 0xff800000u;           // -inf: weight 0
                        }
#pragma unroll
                        for (int ch = 0; ch < S::kCh; ++ch) {
                            if (ch >= nch) break;
                            uint32_t pk[4], lo[4];
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                const int c = ch * 8 + 4 * i;
                                const float4 nr = *reinterpret_cast<const float4 *>(&sx.negref[grp][c]);
                                const F2 sc = {a.scale_log2, a.scale_log2};
                                const F2 da = fma2(F2{__uint_as_float(sv[c]), __uint_as_float(sv[c + 1])}, sc, F2{nr.x, nr.y});
                                const F2 db = fma2(F2{__uint_as_float(sv[c + 2]), __uint_as_float(sv[c + 3])}, sc, F2{nr.z, nr.w});
                                over = max3(over, da.x, da.y);
                                over = max3(over, db.x, db.y);
                                const float p0 = ex2_ftz(da.x), p1 = ex2_ftz(da.y), p2 = ex2_ftz(db.x), p3 = ex2_ftz(db.y);
                                pk[2 * i] = pack_bf16(p0, p1);
                                pk[2 * i + 1] = pack_bf16(p2, p3);
                                if (S::kSplit) {
                                    lo[2 * i] = pack_bf16(p0 - bf16_lo(pk[2 * i]), p1 - bf16_hi(pk[2 * i]));
                                    lo[2 * i + 1] = pack_bf16(p2 - bf16_lo(pk[2 * i + 1]), p3 - bf16_hi(pk[2 * i + 1]));
                                }
                            }
                            const int r8 = cbase / 8 + ch;   // eight rows are one 16-byte piece of the token's line
                            unsigned char *line = p_s + (tile % S::kPBufs) * S::kPBuf + tok * 128;
                            const int at = (r8 ^ (tok & 7)) << 4;
                            *reinterpret_cast<uint4 *>(line + at) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                            if (S::kSplit)             // (joint: rows + 32, four pieces on)
                                *reinterpret_cast<uint4 *>(line + (S::kJoint ? at ^ 64 : at + (int)S::kPTerm)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                if (S::kSplit) {
                                    w[(ch * 8 + 2 * i) % kW] = __float_as_uint(bf16_lo(pk[i]) + bf16_lo(lo[i]));
                                    w[(ch * 8 + 2 * i + 1) % kW] = __float_as_uint(bf16_hi(pk[i]) + bf16_hi(lo[i]));
                                } else {
                                    w[(ch * 4 + i) % kW] = pk[i];
                                }
                            }
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    }
                    if (!group_any(grp, !ok || over > S::kMoveRef) || attempt == 2) break;
                    // rare: some reference has to move (or a wait ran out): O^T is rescaled, so the previous
                    // product must have landed
                    if (ok && j > sg.t0) ok = warp_wait(&sb.pv_done[(tile - 1) % S::kPBufs], ((tile - 1) / S::kPBufs) & 1, &sb);
                    if (group_any(grp, !ok)) { ok = false; break; }
                    tc_fence_after();
const float m = column_max();
                    if (tok < nch * 8) {
                        const float nr = sx.negref[grp][tok];
                        const bool move = m + nr > 0.f;
                        sx.move[grp][tok] = move ? exp2f(-(m + nr)) : 1.f;
                        if (move) sx.negref[grp][tok] = -m;
                    }
                    group_sync(grp);
                    if (j > sg.t0) {
#pragma unroll 1
                        for (int i = 0; i < (S::kJoint ? 2 : 1) * nch; ++i) {
                            const int ch = i < nch ? i : i - nch;                      // (the second term's columns)
                            const uint32_t at = o_addr + ch * 8 + (i < nch ? 0 : NMAX);
                            uint32_t ov[8];
                            tmem_ld8(at, ov);
                            tmem_wait_ld();
#pragma unroll
                            for (int c = 0; c < 8; ++c)
                                ov[c] = __float_as_uint(__uint_as_float(ov[c]) * sx.move[grp][ch * 8 + c]);
                            tmem_st8(at, ov);
                        }
                        tmem_wait_st();
#pragma unroll
                        for (int c = 0; c < S::kCols; ++c)
                            if (c < nch * 8) l[c] *= sx.move[grp][c];
                    }
                }
                if (!ok) break;
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sb.p_full[tile % S::kSBufs]);
                if (work) {
                    // (the row sum must match what the tensor core sees: the rounded values)
#pragma unroll
                    for (int ch = 0; ch < S::kCh; ++ch) {
                        if (ch >= nch) break;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int c = ch * 8 + 2 * i;
                            const F2 wt = S::kSplit ? F2{__uint_as_float(w[c % kW]), __uint_as_float(w[(c + 1) % kW])}
                                                    : F2{bf16_lo(w[(ch * 4 + i) % kW]), bf16_hi(w[(ch * 4 + i) % kW])};
                            const F2 t = add2(F2{l[c], l[c + 1]}, wt);
                            l[c] = t.x; l[c + 1] = t.y;
                        }
                    }
                }
            }
            if (!ok) break;
            // ---- the unit's (or the part's) end: references and row sums over the tokens for the output warps,
            // which have read those of the unit before the previous one
            const uint32_t ub = unit & 1;
            ok = warp_wait(&sb.o_empty[ub], ((unit >> 1) & 1) ^ 1, &sb);
#pragma unroll
            for (int ch = 0; ch < S::kCh; ++ch) {
                if (ch >= nch) break;
                fold8(l + ch * 8, lane, [](float x, float y) { return x + y; });
                if (lane < 8) sx.red[ub][q][cbase + ch * 8 + lane] = l[ch * 8];
            }
            if (tok < nch * 8) sx.ref[ub][cbase + tok] = -sx.negref[grp][tok];
            // (read before the next unit sets new references)
            if (group_any(grp, !ok)) { ok = false; break; }
            if (lane == 0) mbar_arrive(&sb.sum_full[ub]);
            ++unit;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *reinterpret_cast<volatile int *>(&sb.abort)) report(a.status, DSBD_DEV_TIMEOUT);
    if (warp == kWarpS) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S::kTmemCols) : "memory");
    }
}

// Merge of the units that were cut: block (i, y, layer) takes the unit that starts as the last one of run i,
// a warp to a row (a chain of four loads from L2 each; with 32 rows to a block of 8 warps the kernel took 5.6 us, 3.5 now);
// out = sum_p O_p 2^(m_p - m) / sum_p l_p 2^(m_p - m).
constexpr int kMergeThreads = 256;
template <int D, int NMAX>
__global__ void __launch_bounds__(kMergeThreads)
k_attn_merge(TcArgs a) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int layer = blockIdx.z, i0 = layer * a.runs + (int)blockIdx.x, end = (layer + 1) * a.runs - 1;
    const CutRec rec = a.recs[i0];
    int last = min(i0 + 1, end);                             // the runs that hold the other parts
    int ends = a.recs[last].head_ends;
    if (!rec.tail) return;
    if (!names_unit(rec, a.N, a.Hkv)) return;
    while (last < end && !ends) ends = a.recs[++last].head_ends;
    const int n_lo = rec.n_lo;
    const int rows = min(a.block_rows, rec.n_tree * a.group - rec.rb * a.block_rows);
    const int lane = threadIdx.x & 31;
    constexpr int kPer = D / 32;                             // values per lane: 2 (d = 64) or 4
    for (int row = (blockIdx.y * kMergeThreads + threadIdx.x) >> 5; row < rows; row += gridDim.y * kMergeThreads / 32) {
        auto part = [&](int i) { return a.partial + ((2 * (int64_t)i + (i == i0 ? 1 : 0)) * NMAX + row) * (D + 2); };
        float m = -INFINITY;
        for (int i = i0; i <= last; ++i) m = fmaxf(m, part(i)[0]);
        float l = 0.f, o[kPer] = {};
        for (int i = i0; i <= last; ++i) {
            const float *src = part(i);
            if (src[0] == -INFINITY) continue;
            const float w = exp2f(src[0] - m);
            l += src[1] * w;
#pragma unroll
            for (int e = 0; e < kPer; e += 2) {
                const float2 x = *reinterpret_cast<const float2 *>(src + 2 + lane * kPer + e);
                o[e] += x.x * w; o[e + 1] += x.y * w;
            }
        }
        const float inv = 1.f / l;
        const int r = rec.rb * a.block_rows + row, node = r / a.group, hq = rec.g * a.group + (r - node * a.group);
        uint32_t *dst = reinterpret_cast<uint32_t *>(a.out + (int64_t)layer * a.q_layer_stride +
                                                     ((int64_t)(n_lo + node) * a.Hq + hq) * D + lane * kPer);
#pragma unroll
        for (int e = 0; e < kPer; e += 2) dst[e / 2] = pack_bf16(o[e] * inv, o[e + 1] * inv);
    }
}

// Launch shape shared by the workspace query and the launch.  It does not depend on the number of layers
// of a call (nor do the results).
struct TcPlan {
    int nmax;                 // query rows of the kernel instance: 32 or 64
    int block_rows;           // rows of a row block: whole nodes (the copy engine fetches them as a box of
                              // nodes x heads), the largest tree's nodes shared out evenly
    int row_blocks;           // of the largest tree
    int q_nodes, q_rows;      // nodes and rows (a multiple of 8) of a block's query box
    int runs, uni_nt;
    int sms;
    bool whole;               // no unit is cut: no partial results, no merge
};

// Cutting units into equal runs costs partial results and the merge kernel: about as long as kCutTiles
// tiles of one CTA.  A run of fewer than kMinTiles tiles is not worth another CTA.
constexpr int64_t kCutTiles = 6, kMinTiles = 8;
constexpr int kMaxRows = 64;              // rows of a row block, at most

TcPlan make_plan(const dsbd_forest_t *f, const dsbd_attn_desc_t *d) {
    TcPlan p = {};
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int group = d->Hq / d->Hkv, rows = f->max_tree_nodes * group;
    p.sms = sms;
    int nb = (rows + kMaxRows - 1) / kMaxRows;
    while ((f->max_tree_nodes + nb - 1) / nb * group > kMaxRows) ++nb;
    p.block_rows = (f->max_tree_nodes + nb - 1) / nb * group;
    p.row_blocks = nb;
    p.nmax = p.block_rows <= 32 ? 32 : 64;
    p.q_nodes = std::min(p.block_rows / group, f->max_tree_nodes);
    p.q_rows = (p.q_nodes * group + 7) / 8 * 8;
    const int64_t max_nt = ((d->max_prefix + kBN - 1) / kBN + 2) / 2;         // (the tree is one box)
    const int64_t units = (int64_t)f->B * d->Hkv;
    const bool uniform = p.row_blocks == 1 && d->max_prefix * f->B == d->total_prefix;
    // tiles of a layer (ragged: a lower bound)
    const int64_t tiles = uniform ? units * max_nt : std::max<int64_t>(units, d->total_prefix / kTile * d->Hkv);
    const int64_t cut_len = std::max<int64_t>((tiles + sms - 1) / sms, kMinTiles) + kCutTiles;
    int64_t runs = std::min<int64_t>(sms, std::max<int64_t>(tiles / kMinTiles, 1));
    if (uniform) {
        p.uni_nt = (int)max_nt;
        p.whole = (units + sms - 1) / sms * max_nt <= cut_len;
    } else {
        p.whole = p.row_blocks == 1 && units <= sms && max_nt <= cut_len;
    }
    if (p.whole) runs = std::min<int64_t>(units, sms);       // (ragged: one unit each)
    p.runs = (int)runs;
    return p;
}

size_t partial_offset(const TcPlan &p, int n_layers) { return align_up(sizeof(CutRec) * (size_t)p.runs * n_layers, 256); }
// (d = 64 takes a workspace of any alignment, as it always has, and aligns it itself)
size_t workspace_of(const TcPlan &p, int n_layers, int d) {
    if (p.whole) return 256;
    return align_up(partial_offset(p, n_layers) + sizeof(float) * 2 * (size_t)p.runs * n_layers * p.nmax * (d + 2), 256) +
           (d == 64 ? 256 : 0);
}

template <int D, int NMAX>
int launch(const TcPlan &p, const CUtensorMap (&maps)[5], TcArgs a, cudaStream_t stream) {
    using S = Shape<D, NMAX>;
    if (cudaFuncSetAttribute(k_forest_attn_tr<D, NMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)S::kSmem) != cudaSuccess)
        return DSBD_ERR_CUDA;
    // (an S^T product reads up to 8 rows past a buffer's last one: columns that nobody uses)
    a.q_bufs = (uint32_t)(2 * S::kHalves * p.q_rows + 8) * 128 <= S::kQBytes ? 2 : 1;
    // several layers: the units of all layers as one sequence when they are equal and whole; else as many
    // layers side by side as the SMs hold, each CTA with the same run of its layers
    a.layer_step = std::max(1, std::min(a.n_layers, p.sms / p.runs));
    const int grid = p.whole && p.uni_nt ? (int)std::min<int64_t>(p.sms, (int64_t)a.B * a.Hkv * a.n_layers)
                                         : p.runs * a.layer_step;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(S::kThreads);
    cfg.dynamicSmemBytes = S::kSmem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, k_forest_attn_tr<D, NMAX>, maps[0], maps[1], maps[2], maps[3], maps[4], a) !=
        cudaSuccess)
        return DSBD_ERR_CUDA;
    if (p.whole) return DSBD_OK;
    cfg.gridDim = dim3((unsigned)p.runs, (unsigned)((p.block_rows + kMergeThreads / 32 - 1) / (kMergeThreads / 32)), (unsigned)a.n_layers);
    cfg.blockDim = dim3(kMergeThreads);
    cfg.dynamicSmemBytes = 0;
    return cudaLaunchKernelEx(&cfg, k_attn_merge<D, NMAX>, a) == cudaSuccess ? DSBD_OK : DSBD_ERR_CUDA;
}

}  // namespace

namespace dsbd {

// Trees of more than 64 query rows are better off with the rows on the M side at d = 128 (20 nodes x 4 heads,
// 300-900 tokens: 68 us there, 102 us here, where the keys and values pass twice); at d = 64, where that
// kernel does not exist, they run here as several row blocks (4189 us on the CUDA cores, 248 us here).
bool attention_tr_supported(const dsbd_forest_t *f, const dsbd_attn_desc_t *d, int64_t n_pages) {
    const int group = d->Hq / d->Hkv;
    if (d->dtype != DSBD_DTYPE_BF16 || group > kMaxRows) return false;
    if (d->d == 128 && f->max_tree_nodes * group > kMaxRows) return false;
    // heads of 64: packed caches, trees of one tree box (the limits of the entry point for d = 64)
    if (d->d == 64 ? (n_pages > 0 || f->max_tree_nodes > DSBD_MAX_TREE_NODES) : d->d != 128) return false;
    if (!(d->scale > 0.f)) return false;                                     // the row maximum is taken before scaling
    if (d->total_prefix <= 0) return false;
    // row coordinates of the K/V maps are 32-bit
    const int64_t rows = n_pages > 0 ? n_pages * d->Hkv * kBN : (int64_t)d->total_prefix * d->Hkv;
    if (rows >= (int64_t)1 << 31) return false;
    return encode_fn() != nullptr;
}

size_t attention_tr_workspace(const dsbd_forest_t *f, const dsbd_attn_desc_t *d, int n_layers) {
    return workspace_of(make_plan(f, d), n_layers < 1 ? 1 : n_layers, d->d);
}

int attention_tr_launches(const dsbd_forest_t *f, const dsbd_attn_desc_t *d) { return make_plan(f, d).whole ? 1 : 2; }

int launch_attention_tr(const dsbd_forest_t *f, const dsbd_attn_desc_t *d, const void *q, const void *k_new,
                        const void *v_new, const void *k_prefix, const void *v_prefix, const int64_t *prefix_off,
                        void *out, void *workspace, size_t workspace_bytes, int32_t *status, cudaStream_t stream,
                        const dsbd_kv_pages_t *pages) {
    const LayerDims LD = layer_dims(f, d, pages);
    if (!LD.ok) return DSBD_ERR_INVALID_ARG;
    const int nl = LD.n_layers;
    const TcPlan plan = make_plan(f, d);
    if (workspace_bytes < workspace_of(plan, nl, d->d)) return DSBD_ERR_WORKSPACE_TOO_SMALL;
    const uintptr_t ws = d->d == 64 ? align_up(reinterpret_cast<uintptr_t>(workspace), 256) : reinterpret_cast<uintptr_t>(workspace);
    if (!plan.whole && (ws & 255)) return DSBD_ERR_INVALID_ARG;
    // one map per operand over all layers: layer l starts l * (layer stride in rows) further down
    const uint64_t D = (uint64_t)d->d;
    const uint64_t prows = pages ? (uint64_t)pages->n_pages * d->Hkv * kBN + (uint64_t)(nl - 1) * LD.pool_rows
                                 : (uint64_t)d->total_prefix * d->Hkv;
    const uint64_t nrows = (uint64_t)f->N + (uint64_t)(nl - 1) * LD.new_rows;
    const int group = d->Hq / d->Hkv;
    const int64_t q_layer_nodes = nl > 1 ? LD.q_stride / ((int64_t)d->Hq * d->d) : 0;
    if ((uint64_t)f->N + (uint64_t)(nl - 1) * q_layer_nodes >= ((uint64_t)1 << 31)) return DSBD_ERR_UNSUPPORTED;
    CUtensorMap maps[5];
    if (!make_map(&maps[0], k_prefix, D, prows, D * 2) || !make_map(&maps[1], v_prefix, D, prows, D * 2) ||
        !make_map(&maps[2], k_new, (uint64_t)d->Hkv * D, nrows, (uint64_t)d->Hkv * D * 2) ||
        !make_map(&maps[3], v_new, (uint64_t)d->Hkv * D, nrows, (uint64_t)d->Hkv * D * 2) ||
        !make_map_q(&maps[4], q, D, (uint64_t)d->Hq, (uint64_t)f->N + (uint64_t)(nl - 1) * q_layer_nodes,
                    (uint32_t)group, (uint32_t)plan.q_nodes))
        return DSBD_ERR_CUDA;
    TcArgs a = {};
    a.B = f->B; a.N = f->N; a.Hq = d->Hq; a.Hkv = d->Hkv; a.group = group;
    a.block_rows = plan.block_rows;
    a.nodes_per_block = plan.block_rows / group;
    a.q_nodes = plan.q_nodes; a.q_rows = plan.q_rows;
    a.runs = plan.runs; a.uni_nt = plan.uni_nt; a.whole = plan.whole;
    // (tiles of 64-wide heads are half as long: 222 us at 1, 195 at 2 for 33 x 2-5 beams of 92 to 6875 tokens)
    a.unit_cost = d->d == 64 ? 2 : 1;
    a.reread = plan.row_blocks > 1;
    a.scale_log2 = d->scale * 1.4426950408889634f;
    a.beam_node_off = f->beam_node_off; a.parent = f->parent; a.prefix_off = prefix_off;
    if (pages) { a.page_table = pages->page_table; a.page_off = pages->page_off; }
    a.out = static_cast<__nv_bfloat16 *>(out);
    a.status = status;
    a.n_layers = nl; a.pool_layer_rows = LD.pool_rows; a.new_layer_rows = LD.new_rows;
    a.q_layer_stride = LD.q_stride;
    a.q_layer_nodes = (int)q_layer_nodes;
    a.recs = reinterpret_cast<CutRec *>(ws);
    a.partial = reinterpret_cast<float *>(ws + partial_offset(plan, nl));
    if (d->d == 64)
        return plan.nmax == 32 ? launch<64, 32>(plan, maps, a, stream) : launch<64, 64>(plan, maps, a, stream);
    return plan.nmax == 32 ? launch<128, 32>(plan, maps, a, stream) : launch<128, 64>(plan, maps, a, stream);
}

}  // namespace dsbd

#ifdef DSBD_TEST_WAIT_TIMEOUT
// The merge's check of a record, on the host (records are 8 words; see CutRec).
extern "C" int dsbd_test_names_unit(const int32_t *rec, int32_t N, int32_t Hkv) {
    CutRec r;
    static_assert(sizeof(r) == 8 * sizeof(int32_t), "a record is 8 words");
    std::copy(rec, rec + 8, reinterpret_cast<int32_t *>(&r));
    return names_unit(r, N, Hkv);
}
#endif
