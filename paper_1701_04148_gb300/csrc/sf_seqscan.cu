// sf_seqscan.cu -- the paper's one-at-a-time rule (S = 1) by sorts and scans (sm_103a).
//
// Rules (Yang et al., SF-sketch): an insertion (Sec. 3.4, kept by SF_F in Sec. 3.5) adds 1 to the
// item's d Fat counters and then raises its Slim counters to T = min(m + 1, F), where m is the minimum
// of its Slim counters before and F the minimum of its Fat counters after; a deletion (Sec. 3.5)
// takes 1 from the Fat counters and lowers A_i[h_i] to M_i = max_k B_i[h_i][k] (SF_4, Sec. 3.4: to the
// bucket's sum).  The stream is taken in pieces of up to kSeqPiece updates, one cooperative launch
// each.  What makes a piece parallel:
//   - A Fat counter's value right after an update is its value before the piece plus the signed count
//     of the piece's updates on it up to that one: with every row sorted by counter (stable, so stream
//     order within a counter) a segmented sum.  So every F, and with a search in those sorted rows
//     every M_i, is known before any Slim counter moves.
//   - A Slim counter sees, in stream order, x -> max(x, T) at insertions and x -> min(x, M) at
//     deletions.  Such clamps compose, so with every T known its value before each update is a
//     segmented scan over the row sorted by bucket.
//   - Left is T_t = min(m_t + 1, F_t) with m_t depending on earlier T's.  The right side never falls
//     when a T rises, and m_t reads earlier updates only, so exactly one assignment satisfies it for
//     every t.  An assignment that an iteration leaves unchanged is therefore the stream-order result.
//   - From above: T = F everywhere is an upper bound; a scan shows where some row holds less than
//     T - 1 before the insertion, and T falls to that value plus one.  Sketches whose keys mostly have
//     one Fat counter to themselves end here at once, or, with the raises along a bucket bounded by their
//     number (RaiseMap), in a few iterations.
//   - From below, when that does not end soon: every T at first without any other key's raises.  An
//     iteration follows a key's own raises along the whole piece: on the row sorted by key,
//     T_j >= min(F_j, 1 + max(a_j, min(T_{j-1}, G_j))), with a_j the key's Slim minimum of the last
//     iteration and G_j a lower bound of the key's Fat minimum between its updates j - 1 and j (every
//     clamp M_i in between is at least that).  These maps compose as well (a shift and a clamp), so
//     this is one more segmented scan.  Up to four rows, the scan along a bucket also lets each insertion whose
//     least counter lies there raise whatever it finds by one, as far as its other rows' bounds and F allow
//     (ClimbMap): keys that take turns in a bucket climb together, where one iteration a turn was needed.
//     Dense sketches (z = 1, tens of updates per bucket) take 10 to 55 iterations, 11 to 13 us each at d = 2; each
//     settles at least the first insertion that is not settled yet.  100,000 insertions, w = 1,024, z = 1, by
//     the stream: d = 2 740-1,455 us without ClimbMap, 255-710 with it; d = 3 470-1,125, 275-720; d = 4
//     450-1,100, 305-780.
//
// One block of 1,024 threads holds 1,024 consecutive entries of every sorted row, one per thread, in
// registers across the iterations.  The launch is bound by grid barriers and L2 round trips (10 barriers
// when T = F holds and the indices of a row's buckets and counters take two radix passes), not by bandwidth: its
// arrays (tens of megabytes at d = 4) stay in L2.
// Measured on 100,000 Zipf(1) u32 updates (d = 4, w = 4,096, z = 16), a pass, by the stream: insertions 58 to 101 us,
// where a walk of the stream's dependency graph by one block took 378 to 690; a tenth of them deletions
// 76 to 114 us, where the window kernel (sf_seq.cu) takes 27.3 ms.  Sorting takes 30 us of it, the Fat 9, the
// deletions' bounds 12, each scan with its check 8 to 15.
#include "sf_seqscan.h"

#include <type_traits>

namespace sfk {

namespace {

constexpr uint32_t kTile = 1024;                   // entries of a row per block
constexpr uint32_t kBlocks = kSeqPiece / kTile;    // blocks of a full piece
constexpr uint32_t kBins = 256;                    // radix digit of 8 bits
constexpr uint32_t kGroup = 8;                     // rows ranked at a time (shared memory)
constexpr uint32_t kAbove = 32;                    // most iterations from above before those from below
constexpr uint32_t kNear = 16;                     // entries searched back one by one for a key's previous update
constexpr uint32_t kDirectBlocks = 16;             // up to here every block sums the others' digit counts itself
constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr uint32_t kTop = 0xFFFFFFFFu;
constexpr uint32_t kOpIns = 1u, kOpDel = 2u;       // operation codes of a sorted element (0: none)
constexpr uint32_t kSlotShift = 19;                // a bucket row's element carries the update's slot above its position
constexpr uint32_t kHead = 1u << 30, kLast = 1u << 31;
static_assert(kSeqPiece == 1u << (kSlotShift - 2) && kMaxZ <= 64, "position and slot fit their bits");

// Workspace of one piece.  A sorted element is key << 32 | position << 2 | operation code, so elements
// compare by (key, position).  Rows 0..d-1 are sorted by bucket, d..2d-1 by Fat counter (bucket x z +
// slot), 2d by key hash.
struct ScanWs {
    unsigned long long *el0, *el1;  // [2d + 1][N] elements, the two sides of a radix pass
    ulonglong2* kx;                 // [N] key words by position
    uint32_t *V, *W, *a;            // [N][row stride] by position: Fat counters after the update; their minima since
                                    // the key's previous update; Slim counters before the update
    uint32_t* Vs;                   // [d][N] the Fat counter after the update, in counter order
    uint32_t *X, *P;                // [N] the raise target; the previous update of the same key
    uint32_t *hist, *off, *tot;     // digit counts per block (two 16-bit counts a word), first outputs, totals
    uint4* agg;                     // [2d + 1][blocks] block aggregates of the scans (Slim and Fat, keys, raises: a scan
                                    // may follow one of another kind without a barrier between them)
    uint32_t* low;                  // [d][blocks] least Fat counter of a block's entries in counter order
    uint32_t* flag;                 // [8] "not settled" and "changed" words of the iterations
};

__host__ __device__ inline uint32_t rows_of(uint32_t d) { return 2u * d + 1u; }

// Words per position of V, W and a: the rows, so that a thread reads its update's with 16-byte loads.
__host__ __device__ constexpr uint32_t row_stride(uint32_t d) { return d <= 1 ? 1 : d <= 2 ? 2 : d <= 4 ? 4 : 8; }

__host__ __device__ inline ScanWs carve(void* base, uint32_t d) {
    const uint64_t N = kSeqPiece, R = rows_of(d);
    ScanWs w;
    uint8_t* p = static_cast<uint8_t*>(base);
    auto take = [&](uint64_t bytes) {
        uint8_t* q = p;
        p += (bytes + 255) & ~255ull;
        return q;
    };
    w.el0 = (unsigned long long*)take(R * N * 8);
    w.el1 = (unsigned long long*)take(R * N * 8);
    w.kx = (ulonglong2*)take(N * 16);
    w.V = (uint32_t*)take(row_stride(d) * N * 4);
    w.W = (uint32_t*)take(row_stride(d) * N * 4);
    w.a = (uint32_t*)take(row_stride(d) * N * 4);
    w.Vs = (uint32_t*)take(d * N * 4);
    w.X = (uint32_t*)take(N * 4);
    w.P = (uint32_t*)take(N * 4);
    w.hist = (uint32_t*)take(R * kBlocks * (kBins / 2) * 4);
    w.off = (uint32_t*)take(R * kBlocks * kBins * 4);
    w.tot = (uint32_t*)take(R * kBins * 4);
    w.agg = (uint4*)take((2 * d + 1) * kBlocks * 16);
    w.low = (uint32_t*)take(d * kBlocks * 4);
    w.flag = (uint32_t*)take(32);
    return w;
}

uint64_t ws_bytes(uint32_t d) {
    const ScanWs w = carve(nullptr, d);
    return (uint64_t)(uintptr_t)w.flag + 256;
}

struct ScanArgs {
    SketchDesc s;
    const uint8_t* keys;
    const int8_t* ops;  // nullptr: every update is op_const
    int32_t op_const;
    uint32_t n;         // updates of the piece, at most kSeqPiece
    uint32_t bucket_passes, counter_passes, key_passes;
    void* ws;
    uint32_t* ctrl;
    uint64_t timeout_ns;
};

// ---- maps composed by the scans (compose(a, b): first a, then b) -----------------------------

// Segmented sum: y restarts the sum.
struct SumMap {
    using T = uint2;  // {sum, restarted}
    static __device__ __forceinline__ T identity() { return make_uint2(0u, 0u); }
    static __device__ __forceinline__ T compose(const T& a, const T& b) {
        return b.y ? b : make_uint2(a.x + b.x, a.y);
    }
    static __device__ __forceinline__ T shfl_up(const T& v, int o) {
        return make_uint2(__shfl_up_sync(kFull, v.x, o), __shfl_up_sync(kFull, v.y, o));
    }
    static __device__ __forceinline__ T shfl_down(const T& v, int o) {
        return make_uint2(__shfl_down_sync(kFull, v.x, o), __shfl_down_sync(kFull, v.y, o));
    }
    static __device__ __forceinline__ uint4 pack(const T& v) { return make_uint4(v.x, v.y, 0u, 0u); }
    static __device__ __forceinline__ T unpack(const uint4& v) { return make_uint2(v.x, v.y); }
};

// x -> max(lo, min(hi, x)), lo <= hi; a constant when lo = hi.
struct ClampMap {
    using T = uint2;  // {lo, hi}
    static __device__ __forceinline__ T identity() { return make_uint2(0u, kTop); }
    static __device__ __forceinline__ T compose(const T& a, const T& b) {
        return make_uint2(max(b.x, min(b.y, a.x)), max(b.x, min(b.y, a.y)));
    }
    static __device__ __forceinline__ T shfl_up(const T& v, int o) { return SumMap::shfl_up(v, o); }
    static __device__ __forceinline__ T shfl_down(const T& v, int o) { return SumMap::shfl_down(v, o); }
    static __device__ __forceinline__ uint4 pack(const T& v) { return make_uint4(v.x, v.y, 0u, 0u); }
    static __device__ __forceinline__ T unpack(const uint4& v) { return make_uint2(v.x, v.y); }
};

__device__ __forceinline__ uint32_t add_sat(uint32_t a, uint32_t b) {
    const uint32_t s = a + b;
    return s < a ? kTop : s;
}

// x -> max(lo, min(hi, x + k)), sums saturating at 2^32 - 1.
struct ShiftMap {
    using T = uint3;  // {lo, hi, k}
    static __device__ __forceinline__ T identity() { return make_uint3(0u, kTop, 0u); }
    static __device__ __forceinline__ T compose(const T& a, const T& b) {
        return make_uint3(max(b.x, min(b.y, add_sat(a.x, b.z))), max(b.x, min(b.y, add_sat(a.y, b.z))), a.z + b.z);
    }
    static __device__ __forceinline__ T shfl_up(const T& v, int o) {
        return make_uint3(__shfl_up_sync(kFull, v.x, o), __shfl_up_sync(kFull, v.y, o), __shfl_up_sync(kFull, v.z, o));
    }
    static __device__ __forceinline__ T shfl_down(const T& v, int o) {
        return make_uint3(__shfl_down_sync(kFull, v.x, o), __shfl_down_sync(kFull, v.y, o),
                          __shfl_down_sync(kFull, v.z, o));
    }
    static __device__ __forceinline__ uint4 pack(const T& v) { return make_uint4(v.x, v.y, v.z, 0u); }
    static __device__ __forceinline__ T unpack(const uint4& v) { return make_uint3(v.x, v.y, v.z); }
};

// Upper bounds along a bucket when an insertion raises by at most one: x -> min(H, max(x, min(x + k, X))), k
// raises up to the largest of their targets X.  w restarts with the constant H (after a restart z is the
// value itself).
struct RaiseMap {
    using T = uint4;  // {k, X, H, restarted}
    static __device__ __forceinline__ T identity() { return make_uint4(0u, 0u, kTop, 0u); }
    static __device__ __forceinline__ T compose(const T& a, const T& b) {
        if (b.w) return b;
        const uint32_t up = max(a.z, min(add_sat(a.z, b.x), b.y));
        return make_uint4(a.x + b.x, max(a.y, b.y), min(b.z, up), a.w);
    }
    static __device__ __forceinline__ T shfl_up(const T& v, int o) {
        return make_uint4(__shfl_up_sync(kFull, v.x, o), __shfl_up_sync(kFull, v.y, o), __shfl_up_sync(kFull, v.z, o),
                          __shfl_up_sync(kFull, v.w, o));
    }
    static __device__ __forceinline__ T shfl_down(const T& v, int o) {
        return make_uint4(__shfl_down_sync(kFull, v.x, o), __shfl_down_sync(kFull, v.y, o),
                          __shfl_down_sync(kFull, v.z, o), __shfl_down_sync(kFull, v.w, o));
    }
    static __device__ __forceinline__ uint4 pack(const T& v) { return v; }
    static __device__ __forceinline__ T unpack(const uint4& v) { return v; }
};

// Lower bounds along a bucket: x -> max(lo, min(hi, x), min(x + k, X)), a clamp and k raises by one up to X.  Composing
// keeps the clamp exactly (raised by the raises of lo) and one ramp of raises, that of all of them together:
// min(x + k, X) of both, the smaller of the possible caps.  What it drops only lowers the bound, and never
// below the clamps alone.
struct ClimbMap {
    using T = uint4;  // {lo, hi, k, X}; k = 0: no raises
    static __device__ __forceinline__ T identity() { return make_uint4(0u, kTop, 0u, 0u); }
    static __device__ __forceinline__ T compose(const T& a, const T& b) {
        T r;
        r.x = max(b.x, min(b.y, a.x));
        r.y = max(b.x, min(b.y, a.y));
        r.z = a.z + b.z;
        r.w = min(a.w, b.y);
        if (b.z) {
            r.x = max(r.x, min(add_sat(a.x, b.z), b.w));
            r.w = min(add_sat(a.z ? a.w : a.y, b.z), b.w);
        }
        return r;
    }
    static __device__ __forceinline__ T shfl_up(const T& v, int o) { return RaiseMap::shfl_up(v, o); }
    static __device__ __forceinline__ T shfl_down(const T& v, int o) { return RaiseMap::shfl_down(v, o); }
    static __device__ __forceinline__ uint4 pack(const T& v) { return v; }
    static __device__ __forceinline__ T unpack(const uint4& v) { return v; }
};

// Inclusive scan of the 32 lanes of a warp.
template <class Map>
__device__ __forceinline__ typename Map::T warp_scan(typename Map::T v, uint32_t lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const typename Map::T u = Map::shfl_up(v, o);
        if (lane >= (uint32_t)o) v = Map::compose(u, v);
    }
    return v;
}

struct Shared {
    union {
        uint16_t cnt[kGroup][32][kBins];  // digit counts per warp, then first ranks
        uint32_t part[32][64];            // digit counts of a group of blocks
        struct {
            uint32_t V[kMaxD][kTile], pos[kMaxD][kTile], low[kMaxD][32];
        } tile;
        struct {
            uint32_t at[kMaxD][32][kMaxZ];     // a bucket's counters behind / before a warp's entries
            uint32_t has[kMaxD][32][2];        // which of them the warp determines
            uint32_t lanes[32][kMaxZ];         // a warp's lanes by slot
        } bucket;
    } u;
    uint32_t base[2 * kMaxD + 1][kBins], tot[2 * kMaxD + 1][kBins];
    uint4 warp_agg[kMaxD][32];
    uint4 stage[32][32];
};

// A barrier of the launch's blocks; false: it gave up.
__device__ __forceinline__ bool piece_barrier(const ScanArgs& a, unsigned long long& target) {
    if (gridDim.x == 1) {
        __syncthreads();
        return true;
    }
    const bool ok = grid_barrier(a.ctrl, target, a.timeout_ns);
    target += gridDim.x;
    return ok;
}

// Scan over R rows at once of the whole grid's entries (one per thread and row): v[r] in, the composition
// of every entry up to and including this one out; prev[r] (if wanted) without it.  One grid barrier, or none
// when `last` is given: the earlier blocks' part is then what they wrote there at the scan before, with a barrier
// since.  False: the barrier gave up.
template <class Map, int R, bool kPrev>
__device__ __forceinline__ bool grid_scan(typename Map::T (&v)[R], typename Map::T (&prev)[R], Shared& sh, uint4* agg,
                                          const ScanArgs& a, unsigned long long& target, const uint4* last = nullptr) {
    using T = typename Map::T;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        v[r] = warp_scan<Map>(v[r], lane);
        if (lane == 31u) sh.warp_agg[r][warp] = Map::pack(v[r]);
    }
    __syncthreads();
    if (warp < (uint32_t)R) {  // warp r: the warps' prefixes of row r, and the block's aggregate
        const T w = warp_scan<Map>(Map::unpack(sh.warp_agg[warp][lane]), lane);
        if (lane == 31u) agg[warp * kBlocks + blockIdx.x] = Map::pack(w);
        T e = Map::shfl_up(w, 1);
        if (lane == 0u) e = Map::identity();
        sh.warp_agg[warp][lane] = Map::pack(e);
    }
    if (gridDim.x > 1) {
        if (!last) {
            if (!grid_barrier(a.ctrl, target, a.timeout_ns)) return false;
            target += gridDim.x;
            last = agg;
        }
        if (warp < (uint32_t)R && blockIdx.x > 0) {
            T c = Map::identity();
#pragma unroll
            for (uint32_t j = 0; j < kBlocks / 32; ++j) {
                const uint32_t b = lane * (kBlocks / 32) + j;
                if (b < blockIdx.x) c = Map::compose(c, Map::unpack(__ldcg(last + warp * kBlocks + b)));
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) c = Map::compose(c, Map::shfl_down(c, o));
            // lane 0 holds the composition of all earlier blocks
            const uint4 c0 = Map::pack(c);
            const T carry = Map::unpack(
                make_uint4(__shfl_sync(kFull, c0.x, 0), __shfl_sync(kFull, c0.y, 0), __shfl_sync(kFull, c0.z, 0),
                           __shfl_sync(kFull, c0.w, 0)));
            sh.warp_agg[warp][lane] = Map::pack(Map::compose(carry, Map::unpack(sh.warp_agg[warp][lane])));
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const T before = Map::unpack(sh.warp_agg[r][warp]);
        if (kPrev) {
            T e = Map::shfl_up(v[r], 1);
            if (lane == 0u) e = Map::identity();
            prev[r] = Map::compose(before, e);
        }
        v[r] = Map::compose(before, v[r]);
    }
    __syncthreads();  // warp_agg is free again
    return true;
}

__device__ __forceinline__ uint32_t el_pos(unsigned long long e) { return (uint32_t)e >> 2 & (kSeqPiece - 1u); }
__device__ __forceinline__ uint32_t el_op(unsigned long long e) { return (uint32_t)e & 3u; }
__device__ __forceinline__ uint32_t el_key(unsigned long long e) { return (uint32_t)(e >> 32); }

// Stable radix sort, 8 bits a pass, of rows R0..R1-1 (passes(r) passes each; elements start in el0).
template <int R0, int R1, class Passes>
__device__ __forceinline__ bool radix_sort(const ScanArgs& a, const ScanWs& w, Shared& sh, unsigned long long& target,
                                           Passes&& passes_of) {
    constexpr int R = R1 - R0;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, blk = blockIdx.x;
    const uint32_t q = blk * kTile + tid;
    const bool valid = q < a.n;
    uint32_t passes = 0;
#pragma unroll
    for (int r = R0; r < R1; ++r) passes = max(passes, passes_of(r));
    for (uint32_t p = 0; p < passes; ++p) {
        const unsigned long long* src = (p & 1u) ? w.el1 : w.el0;
        unsigned long long* dst = (p & 1u) ? w.el0 : w.el1;
        uint32_t rk[R];  // rank among the block's equal digits << 8 | digit
#pragma unroll
        for (int r = 0; r < R; ++r)
            rk[r] = valid && p < passes_of(R0 + r)
                        ? (reinterpret_cast<const uint32_t*>(src + (uint64_t)(R0 + r) * kSeqPiece + q)[1] >> (8u * p)) &
                              (kBins - 1u)
                        : 0u;
        const unsigned act = __ballot_sync(kFull, valid);
        // ranks: the warp's lanes with the same digit from eight ballots (__match_any_sync, which serves the
        // distinct values one after another, took 2.2 us a row here, the ballots 0.3), then over the
        // warps in order
#pragma unroll
        for (int g = 0; g < R; g += kGroup) {
#pragma unroll
            for (int j = 0; j < (int)kGroup && g + j < R; ++j)
                reinterpret_cast<uint4*>(sh.u.cnt[j][warp])[lane] = make_uint4(0u, 0u, 0u, 0u);
            __syncwarp();
#pragma unroll
            for (int j = 0; j < (int)kGroup && g + j < R; ++j) {
                if (p >= passes_of(R0 + g + j)) continue;
                const uint32_t dig = rk[g + j];
                unsigned peers = act;
#pragma unroll
                for (int b = 0; b < 8; ++b) {
                    const bool one = (dig >> b) & 1u;
                    const unsigned m = __ballot_sync(kFull, one);
                    peers &= one ? m : ~m;
                }
                const uint32_t rank = (uint32_t)__popc(peers & ((1u << lane) - 1u));
                if (valid && rank == 0u) sh.u.cnt[j][warp][dig] = (uint16_t)__popc(peers);
                rk[g + j] = rank << 8 | dig;
            }
            __syncthreads();
            {
                const uint32_t j = tid / (kBins / 2), wd = tid % (kBins / 2);  // kGroup rows of 128 words
                const int r = g + (int)j;
                if (r < R && p < passes_of(R0 + r)) {
                    uint32_t run = 0u;  // two 16-bit counts, at most 1,024 each
#pragma unroll 16
                    for (uint32_t v = 0; v < 32u; ++v) {
                        uint32_t* c = reinterpret_cast<uint32_t*>(sh.u.cnt[j][v]) + wd;
                        const uint32_t x = *c;
                        *c = run;
                        run += x;
                    }
                    w.hist[((uint32_t)(R0 + r) * kBlocks + blk) * (kBins / 2) + wd] = run;
                }
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < (int)kGroup && g + j < R; ++j) {
                if (p >= passes_of(R0 + g + j)) continue;
                rk[g + j] += (uint32_t)sh.u.cnt[j][warp][rk[g + j] & (kBins - 1u)] << 8;
            }
            __syncwarp();
        }
        if (!piece_barrier(a, target)) return false;
        // first output of every digit of this block: the same digit of earlier blocks, after all smaller
        // digits.  A few blocks sum the counts themselves; many share the work, for one more barrier.
        if (gridDim.x <= kDirectBlocks) {
            for (uint32_t x = tid; x < (uint32_t)R * (kBins / 2); x += kTile) {
                const uint32_t r = x / (kBins / 2), wd = x % (kBins / 2);
                if (p >= passes_of(R0 + (int)r)) continue;
                uint32_t lo = 0u, hi = 0u, tlo = 0u, thi = 0u;
                for (uint32_t b = 0; b < gridDim.x; ++b) {
                    const uint32_t c = __ldcg(w.hist + ((R0 + r) * kBlocks + b) * (kBins / 2) + wd);
                    if (b == blk) {
                        lo = tlo;
                        hi = thi;
                    }
                    tlo += c & 0xFFFFu;
                    thi += c >> 16;
                }
                sh.base[r][2 * wd] = lo;
                sh.base[r][2 * wd + 1] = hi;
                sh.tot[r][2 * wd] = tlo;
                sh.tot[r][2 * wd + 1] = thi;
            }
        } else {
            for (uint32_t x = blk; x < (uint32_t)R * 4u; x += gridDim.x) {  // 64 digits of one row
                const uint32_t r = R0 + (x >> 2), part = x & 3u;
                if (p >= passes_of((int)r)) continue;
                constexpr uint32_t kPer = kBlocks / 32;
                uint32_t lo[kPer], hi[kPer], slo = 0u, shi = 0u;
#pragma unroll
                for (uint32_t j = 0; j < kPer; ++j) {
                    const uint32_t b = warp * kPer + j;
                    const uint32_t c = b < gridDim.x ? __ldcg(w.hist + (r * kBlocks + b) * (kBins / 2) + part * 32u + lane) : 0u;
                    lo[j] = slo;
                    hi[j] = shi;
                    slo += c & 0xFFFFu;
                    shi += c >> 16;
                }
                sh.u.part[warp][2 * lane] = slo;
                sh.u.part[warp][2 * lane + 1] = shi;
                __syncthreads();
                if (tid < 64u) {
                    uint32_t run = 0u;
#pragma unroll 16
                    for (uint32_t v = 0; v < 32u; ++v) {
                        const uint32_t y = sh.u.part[v][tid];
                        sh.u.part[v][tid] = run;
                        run += y;
                    }
                    w.tot[r * kBins + part * 64u + tid] = run;
                }
                __syncthreads();
                const uint32_t blo = sh.u.part[warp][2 * lane], bhi = sh.u.part[warp][2 * lane + 1];
#pragma unroll
                for (uint32_t j = 0; j < kPer; ++j) {
                    const uint32_t b = warp * kPer + j;
                    if (b < gridDim.x)
                        *reinterpret_cast<uint2*>(w.off + (r * kBlocks + b) * kBins + part * 64u + 2 * lane) =
                            make_uint2(blo + lo[j], bhi + hi[j]);
                }
                __syncthreads();
            }
            if (!piece_barrier(a, target)) return false;
            for (uint32_t x = tid; x < (uint32_t)R * kBins; x += kTile) {
                const uint32_t r = x / kBins, b = x % kBins;
                if (p >= passes_of(R0 + (int)r)) continue;
                sh.base[r][b] = __ldcg(w.off + ((R0 + r) * kBlocks + blk) * kBins + b);
                sh.tot[r][b] = __ldcg(w.tot + (R0 + r) * kBins + b);
            }
        }
        __syncthreads();
        for (uint32_t r = warp; r < (uint32_t)R; r += 32u) {  // digits of a row: exclusive scan of the totals
            if (p >= passes_of(R0 + (int)r)) continue;
            uint32_t c[8], sum = 0u;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                c[j] = sum;
                sum += sh.tot[r][lane * 8u + j];
            }
            uint32_t incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, incl, o);
                if (lane >= (uint32_t)o) incl += y;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) sh.base[r][lane * 8u + j] += incl - sum + c[j];
        }
        __syncthreads();
        if (valid) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (p < passes_of(R0 + r))
                    dst[(uint64_t)(R0 + r) * kSeqPiece + sh.base[r][rk[r] & (kBins - 1u)] + (rk[r] >> 8)] =
                        src[(uint64_t)(R0 + r) * kSeqPiece + q];
        }
        if (!piece_barrier(a, target)) return false;
    }
    return true;
}

// kIns: the piece holds insertions only; kDel: deletions only.
template <int D, bool kIns, bool kDel>
__global__ void __launch_bounds__(kTile, 1) seq_scan_kernel(const __grid_constant__ ScanArgs a) {
    constexpr uint32_t kStride = row_stride(D);
    // Bounds from below with the raises along a bucket: fewer iterations (d = 2, w = 1,024, z = 1, warm: 155 down to
    // 23), but twice a clamp's registers a row: at d = 8 the spills cost up to 1.35x of the time.
    constexpr bool kClimb = D <= 4;
    using Low = std::conditional_t<kClimb, ClimbMap, ClampMap>;
    extern __shared__ __align__(16) unsigned char s_raw[];
    Shared& sh = *reinterpret_cast<Shared*>(s_raw);
    const SketchDesc& s = a.s;
    const ScanWs w = carve(a.ws, D);
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, blk = blockIdx.x;
    const uint32_t q = blk * kTile + tid;  // this thread's position, and its index in every sorted row
    const bool valid = q < a.n;
    const uint32_t wz = s.w * s.z;
    unsigned long long target = gridDim.x;
    auto barrier = [&]() { return piece_barrier(a, target); };
    // A launch whose wait gave up leaves the barrier's counter and the count of leaving blocks anywhere, and
    // every later launch of the stream, until sf_sync zeroes them, would pass its barriers at once and index
    // with half-written sums.  Such launches do nothing: the error bit stands until sf_sync.  Read ahead of
    // the hash, whose loads cover its latency.
    const uint32_t failed = __ldcg(a.ctrl + kCtrlErr) & kErrTimeout;

    // ---- hash --------------------------------------------------------------------------------
    {
        const uint32_t kb = s.key_bytes;
        const uint32_t first = blk * kTile + warp * 32u;
        const uint32_t nv = first < a.n ? min(32u, a.n - first) : 0u;
        Key k{0ull, 0ull};
        if (kb != 4u && kb != 8u) {
            if (nv) k = load_key_staged(a.keys, (uint64_t)a.n * kb, first, nv, kb, lane, sh.stage[warp]);
        } else if (valid) {
            k = load_key(a.keys, q, kb);
        }
        uint32_t h[D], f[D], op = 0u;
        uint64_t probe = 0;
#pragma unroll
        for (int i = 0; i < D; ++i) h[i] = f[i] = 0u;
        if (valid) {
            const int o = a.ops ? (int)a.ops[q] : a.op_const;
            op = o > 0 ? kOpIns : o < 0 ? kOpDel : 0u;
            if (op && !key_indices<D>(s, k, h, f, &probe)) {
                atomicOr(a.ctrl + kCtrlErr, kErrBadKey);
                op = 0u;
#pragma unroll
                for (int i = 0; i < D; ++i) h[i] = f[i] = 0u;  // does nothing, in bucket 0
            }
        }
        const uint32_t pay = q << 2 | op;
        const uint32_t tag = (uint32_t)(probe >> 32) * 0x9E3779B1u ^ (uint32_t)probe;
        if (valid) {
#pragma unroll
            for (int i = 0; i < D; ++i) {
                w.el0[(uint64_t)i * kSeqPiece + q] = (unsigned long long)h[i] << 32 | f[i] << kSlotShift | pay;
                w.el0[(uint64_t)(D + i) * kSeqPiece + q] = (unsigned long long)(h[i] * s.z + f[i]) << 32 | pay;
            }
            if constexpr (!kDel) {
                w.el0[(uint64_t)(2 * D) * kSeqPiece + q] =
                    (unsigned long long)(tag >> (32u - 8u * a.key_passes)) << 32 | pay;
                w.kx[q] = make_ulonglong2(k.x0, k.x1);
            }
        }
        if (blk == 0 && tid < 8u) w.flag[tid] = 0u;
    }
    if (__syncthreads_or((int)failed)) return;

    // ---- sort by bucket and by Fat counter -----------------------------------------------------------
    if (!radix_sort<0, 2 * D>(a, w, sh, target, [&](int r) { return r < D ? a.bucket_passes : a.counter_passes; })) return;
    auto row = [&](int r) {  // the sorted row
        const uint32_t passes = r < D ? a.bucket_passes : r < 2 * D ? a.counter_passes : a.key_passes;
        return ((passes & 1u) ? w.el1 : w.el0) + (uint64_t)r * kSeqPiece;
    };

    // ---- Fat counters after every update -------------------------------------------------------------
    {
        uint2 v[D], unused[D];
        uint32_t po[D];
#pragma unroll
        for (int i = 0; i < D; ++i) {
            v[i] = SumMap::identity();
            po[i] = 0u;
            if (valid) {
                const unsigned long long* C = row(D + i);
                const unsigned long long e = C[q];
                const uint32_t key = el_key(e), op = el_op(e);
                const bool head = q == 0u || el_key(C[q - 1u]) != key;
                po[i] = (uint32_t)e;
                v[i].x = op == kOpIns ? 1u : op == kOpDel ? kTop : 0u;
                if (head) {
                    v[i].x += __ldcg(s.B + (uint64_t)i * wz + key);
                    v[i].y = 1u;
                }
            }
        }
        if (!grid_scan<SumMap, D, false>(v, unused, sh, w.agg, a, target)) return;
        bool under = false;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            if (!valid) continue;
            w.V[(uint64_t)(po[i] >> 2) * kStride + i] = v[i].x;
            w.Vs[(uint64_t)i * kSeqPiece + q] = v[i].x;
            under |= (po[i] & 3u) == kOpDel && v[i].x == kTop;
        }
        if (under) atomicOr(a.ctrl + kCtrlErr, kErrUnderflow);
    }
    if (!barrier()) return;

    // ---- this thread's entries of the bucket orders; deletions find their bounds ----------------------
    uint32_t bpo[D], M[D];
#pragma unroll
    for (int i = 0; i < D; ++i) {
        bpo[i] = 0u;
        M[i] = 0u;
        const unsigned long long* Bo = row(i);
        if (valid) {
            const unsigned long long e = Bo[q];
            bpo[i] = (uint32_t)e;
            if (q == 0u || el_key(Bo[q - 1u]) != el_key(e)) bpo[i] |= kHead;
            if (q + 1u == a.n || el_key(Bo[q + 1u]) != el_key(e)) bpo[i] |= kLast;
        }
    }
    if constexpr (!kIns) {
        // M_i: the bucket's counters right after the deletion, each the value its last update left.  In the
        // warp that value is a lane's; before the warp it is carried along the block's warps; before the
        // block it is found by a binary search in the row sorted by counter, once a counter and block;
        // before the bucket's first update it is the piece's first.  (A search for every deletion and
        // counter took 50 of 100 us on 100,000 updates with 10,000 deletions.)
        uint32_t val[D];
        // the warp's lanes by slot in row i: lanes[k] for slot k
        auto lanes_by_slot = [&](int i) -> const uint32_t* {
            uint32_t* tab = sh.u.bucket.lanes[warp];
            __syncwarp();
            for (uint32_t k = lane; k < s.z; k += 32u) tab[k] = 0u;
            __syncwarp();
            if (valid) atomicOr(&tab[bpo[i] >> kSlotShift & 63u], 1u << lane);
            __syncwarp();
            return tab;
        };
        auto fat0 = [&](int i, uint32_t key) { return __ldcg(s.B + (uint64_t)i * wz + key); };
#pragma unroll
        for (int i = 0; i < D; ++i) {  // the counters of the warp's last bucket behind the warp
            val[i] = valid ? __ldcg(w.V + (uint64_t)(bpo[i] >> 2 & (kSeqPiece - 1u)) * kStride + i) : 0u;
            const unsigned heads = __ballot_sync(kFull, (bpo[i] & kHead) != 0u);
            const uint32_t* tab = lanes_by_slot(i);
            const int begin = heads ? 31 - __clz(heads) : -1;  // where that bucket begins, if in this warp
            const uint32_t h = __shfl_sync(kFull, valid ? el_key(row(i)[q]) : 0u, begin < 0 ? 0 : begin);
            for (uint32_t k0 = 0; k0 < s.z; k0 += 32u) {
                const uint32_t k = k0 + lane;
                const unsigned m = k < s.z ? tab[k] & (begin < 0 ? kFull : kFull << begin) : 0u;
                uint32_t v = __shfl_sync(kFull, val[i], m ? 31 - __clz(m) : 0);
                if (!m && begin >= 0 && k < s.z) v = fat0(i, h * s.z + k);
                const unsigned has = __ballot_sync(kFull, k < s.z && (m || begin >= 0));
                if (k < s.z) sh.u.bucket.at[i][warp][k] = v;
                if (lane == 0u) sh.u.bucket.has[i][warp][k0 / 32u] = has;
            }
        }
        __syncthreads();
        if (tid / kMaxZ < (uint32_t)D && tid % kMaxZ < s.z) {  // the counters before each warp
            const uint32_t i = tid / kMaxZ, k = tid % kMaxZ;
            const unsigned long long* Bo = row((int)i);
            const unsigned long long* C = row(D + (int)i);
            uint32_t carry = 0u;
            const unsigned long long e = Bo[blk * kTile];
            if (blk > 0u && el_key(Bo[blk * kTile - 1u]) == el_key(e)) {
                const uint32_t key = el_key(e) * s.z + k;
                const unsigned long long want = (unsigned long long)key << 32 | (el_pos(e) << 2);
                uint32_t lo = 0u, hi = a.n;  // entries below lo are < want, from hi on >= want
                while (lo < hi) {
                    const uint32_t mid = (lo + hi) >> 1;
                    if (C[mid] < want) lo = mid + 1u;
                    else hi = mid;
                }
                carry = lo > 0u && el_key(C[lo - 1u]) == key ? w.Vs[(uint64_t)i * kSeqPiece + lo - 1u] : fat0((int)i, key);
            }
#pragma unroll 8
            for (uint32_t v = 0; v < 32u; ++v) {
                const uint32_t x = sh.u.bucket.at[i][v][k];
                sh.u.bucket.at[i][v][k] = carry;
                if (sh.u.bucket.has[i][v][k / 32u] >> (k % 32u) & 1u) carry = x;
            }
        }
        __syncthreads();
        // a group of lanes takes a deletion, a lane its counters
        const uint32_t gl = s.z <= 4u ? 4u : s.z <= 8u ? 8u : s.z <= 16u ? 16u : 32u;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            unsigned todo = __ballot_sync(kFull, (bpo[i] & 3u) == kOpDel);
            if (!todo) continue;
            const unsigned heads = __ballot_sync(kFull, (bpo[i] & kHead) != 0u);
            const uint32_t* tab = lanes_by_slot(i);
            const uint32_t h = valid ? el_key(row(i)[q]) : 0u;
            while (todo) {
                // the group's deletion: the (lane / gl)-th lane of todo that still waits
                unsigned rest = todo;
                for (uint32_t g = 0; g < lane / gl && rest; ++g) rest &= rest - 1u;
                const int from = rest ? __ffs(rest) - 1 : 0;
                const uint32_t hd = __shfl_sync(kFull, h, from);
                const unsigned upto = kFull >> (31 - from), begun = heads & upto;
                const unsigned span = begun ? upto & (kFull << (31 - __clz(begun))) : upto;
                uint32_t mx = 0u;
                uint64_t sum = 0ull;
                for (uint32_t k0 = 0; k0 < s.z; k0 += gl) {
                    const uint32_t k = k0 + lane % gl;
                    const unsigned m = k < s.z ? tab[k] & span : 0u;
                    uint32_t v = __shfl_sync(kFull, val[i], m ? 31 - __clz(m) : 0);
                    if (k < s.z) {
                        if (!m) v = begun ? fat0(i, hd * s.z + k) : sh.u.bucket.at[i][warp][k];
                        mx = max(mx, v);
                        sum += v;
                    }
                }
                for (uint32_t o = gl >> 1; o > 0u; o >>= 1) {
                    mx = max(mx, __shfl_xor_sync(kFull, mx, o));
                    sum += __shfl_xor_sync(kFull, sum, o);
                }
                const uint32_t bound = s.sf4_delete ? (sum < (uint64_t)kTop ? (uint32_t)sum : kTop) : mx;
                // hand the bounds back and strike the deletions taken
                for (uint32_t g = 0; g < 32u / gl && todo; ++g) {
                    const int at = __ffs(todo) - 1;
                    const uint32_t x = __shfl_sync(kFull, bound, g * gl);
                    if ((int)lane == at) M[i] = x;
                    todo &= todo - 1u;
                }
            }
        }
    }
    // the rows' values at a position, and their minimum
    auto read_rows = [&](const uint32_t* by_pos, uint32_t pos, uint32_t (&r)[kStride]) -> uint32_t {
        uint32_t m = kTop;
        if constexpr (kStride >= 4u) {
#pragma unroll
            for (uint32_t j = 0; j < kStride; j += 4u)
                *reinterpret_cast<uint4*>(r + j) = __ldcg(reinterpret_cast<const uint4*>(by_pos + (uint64_t)pos * kStride + j));
        } else {
#pragma unroll
            for (uint32_t j = 0; j < kStride; ++j) r[j] = __ldcg(by_pos + (uint64_t)pos * kStride + j);
        }
#pragma unroll
        for (int i = 0; i < D; ++i) m = min(m, r[i]);
        return m;
    };
    auto least_of = [&](const uint32_t* by_pos, uint32_t pos) {
        uint32_t r[kStride];
        return read_rows(by_pos, pos, r);
    };

    // Slim counters along the bucket orders with raise targets T[i] of this thread's entries: v[i].x after
    // an entry, prev[i].x before it (want_prev).  The read behind the scan's barrier is for callers that meet another
    // barrier before the counters after the piece are stored: the last scan asks for v alone, since by then
    // other blocks store the counters of buckets that begin in this one.
    uint2 v[D], prev[D];
    auto slim_scan = [&](const uint32_t (&T)[D], auto want_prev) -> bool {
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const uint32_t op = bpo[i] & 3u;
            v[i] = op == kOpIns ? make_uint2(T[i], kTop) : op == kOpDel ? make_uint2(0u, M[i]) : ClampMap::identity();
            if (bpo[i] & kHead) {
                const uint32_t A0 = __ldcg(slim_ptr(s, i, el_key(row(i)[q])));
                const uint32_t x = max(v[i].x, min(v[i].y, A0));
                v[i] = make_uint2(x, x);
            }
        }
        constexpr bool kPrev = decltype(want_prev)::value;
        if (!grid_scan<ClampMap, D, kPrev>(v, prev, sh, w.agg, a, target)) return false;
        if constexpr (kPrev) {
#pragma unroll
            for (int i = 0; i < D; ++i)
                if (bpo[i] & kHead) prev[i].x = __ldcg(slim_ptr(s, i, el_key(row(i)[q])));
        }
        return true;
    };
    auto pos_of = [&](int i) { return bpo[i] >> 2 & (kSeqPiece - 1u); };
    // How many threads of the grid say yes: the words of w.flag rotate over four, and each is cleared two
    // calls before its next use.  One grid barrier; kNone: it gave up.
    uint32_t calls = 0;
    auto count_of_grid = [&](bool mine) -> uint32_t {
        const uint32_t word = calls & 3u;
        if (blk == 0u && tid == 0u) w.flag[(calls + 2u) & 3u] = 0u;
        ++calls;
        const uint32_t c = (uint32_t)__syncthreads_count(mine);
        if (c && tid == 0u) atomicAdd(w.flag + word, c);
        if (!barrier()) return kNone;
        return __ldcg(w.flag + word);
    };

    uint32_t T[D];
    bool settled = true;
    if constexpr (kDel) {
#pragma unroll
        for (int i = 0; i < D; ++i) T[i] = 0u;
        if (!slim_scan(T, std::false_type{})) return;
    } else {
        // ---- raise targets from above: T = F, lowered where a row holds less than T - 1 ------------------
        if (valid) w.X[q] = least_of(w.V, q);
        auto lower_where_less = [&](int i, uint32_t before) -> bool {
            if ((bpo[i] & 3u) != kOpIns || before >= T[i] || before + 1u >= T[i]) return false;
            atomicMin(w.X + pos_of(i), before + 1u);
            return true;
        };
#pragma unroll
        for (int i = 0; i < D; ++i) T[i] = (bpo[i] & 3u) == kOpIns ? least_of(w.V, pos_of(i)) : 0u;
        if (!slim_scan(T, std::true_type{})) return;
        bool lower = false;
#pragma unroll
        for (int i = 0; i < D; ++i) lower |= lower_where_less(i, prev[i].x);
        uint32_t more = count_of_grid(lower);
        if (more == kNone) return;
        settled = more == 0u;
        if (!settled && 8u * more <= a.n) {
            // A key whose Fat counters all count other keys too climbs by one an insertion: lowering one T at
            // a time would take an iteration for each.  So the bounds along a bucket are taken as if an
            // insertion raised the row's own value by one (T <= a_i + 1 holds in every row), leaving out
            // the insertions whose T the row holds whatever was raised before (its value under the
            // clamps alone).  When no T has to fall, T <= m + 1 holds with the raises proper as well.
            uint32_t hold[D];
            if constexpr (kIns) {
#pragma unroll
                for (int i = 0; i < D; ++i) hold[i] = valid ? __ldcg(slim_ptr(s, i, el_key(row(i)[q]))) : 0u;
            } else {
                uint32_t none[D];
#pragma unroll
                for (int i = 0; i < D; ++i) none[i] = 0u;
                if (!slim_scan(none, std::true_type{})) return;
#pragma unroll
                for (int i = 0; i < D; ++i) hold[i] = prev[i].x;
            }
            uint32_t last = more;
            for (uint32_t it = 1; it <= kAbove; ++it) {
                uint4 u[D], before[D];
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    const uint32_t op = bpo[i] & 3u;
                    T[i] = op == kOpIns ? __ldcg(w.X + pos_of(i)) : 0u;
                    u[i] = RaiseMap::identity();
                    if (op == kOpIns && T[i] > hold[i]) u[i] = make_uint4(1u, T[i], kTop, 0u);
                    if (op == kOpDel) u[i].z = M[i];
                    if (bpo[i] & kHead) {
                        uint4 start = make_uint4(0u, 0u, __ldcg(slim_ptr(s, i, el_key(row(i)[q]))), 1u);
                        u[i] = RaiseMap::compose(start, u[i]);
                    }
                }
                if (!grid_scan<RaiseMap, D, true>(u, before, sh, w.agg + (uint64_t)(D + 1) * kBlocks, a, target)) return;
                lower = false;
#pragma unroll
                for (int i = 0; i < D; ++i)
                    lower |= lower_where_less(i, (bpo[i] & kHead) ? __ldcg(slim_ptr(s, i, el_key(row(i)[q]))) : before[i].z);
                more = count_of_grid(lower);
                if (more == kNone) return;
                settled = more == 0u;
                // three to five iterations settle most streams; where the count does not fall fast the way
                // from below is shorter (8 us an iteration here; 30 us before the first one there and 15
                // for each, at d = 4)
                if (settled || (it >= 3u && 8u * more > 5u * last)) break;
                last = more;
            }
            if (settled && !slim_scan(T, std::false_type{})) return;
        }
    }
    if constexpr (!kDel) {
        if (!settled) {
            // ---- from below: the rows in key order, and each entry's previous update of its key ----------
            if (!radix_sort<2 * D, 2 * D + 1>(a, w, sh, target, [&](int) { return a.key_passes; })) return;
            uint32_t kpo = 0u;  // this thread's entry: position << 2 | operation, kHead
            if (valid) {
                const unsigned long long* K = row(2 * D);
                const unsigned long long e = K[q];
                const uint32_t pos = el_pos(e);
                uint32_t before = kNone;
                if (q > 0u) {
                    const unsigned long long b = K[q - 1u];
                    if (el_key(b) == el_key(e)) {
                        const ulonglong2 x = w.kx[pos], y = w.kx[el_pos(b)];
                        if (x.x == y.x && x.y == y.y && el_op(e) && el_op(b)) before = el_pos(b);
                    }
                }
                kpo = (uint32_t)e | (before == kNone ? kHead : 0u);
                w.P[pos] = before;
            }
            if constexpr (!kIns) {
                // W: a lower bound of the counter's least value since the key's previous update, from the
                // entries before this one in counter order until the previous update is covered: at least
                // kNear one by one, then whole warps' and whole blocks' least values (which may hold
                // entries of another counter, or of before the previous update: lower at worst)
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    const uint32_t x = valid ? w.Vs[(uint64_t)i * kSeqPiece + q] : kTop;
                    sh.u.tile.V[i][tid] = x;
                    sh.u.tile.pos[i][tid] = valid ? el_pos(row(D + i)[q]) : kNone;
                    const uint32_t l = __reduce_min_sync(kFull, x);
                    if (lane == 0u) sh.u.tile.low[i][warp] = l;
                }
                __syncthreads();
                if (tid < 32u) {
#pragma unroll
                    for (int i = 0; i < D; ++i) {
                        const uint32_t l = __reduce_min_sync(kFull, sh.u.tile.low[i][tid]);
                        if (tid == 0u) w.low[i * kBlocks + blk] = l;
                    }
                }
                if (!barrier()) return;
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    if (!valid) continue;
                    const uint32_t pos = sh.u.tile.pos[i][tid], target_pos = w.P[pos];
                    uint32_t least = kTop;
                    if (target_pos != kNone) {
                        bool found = false;
                        uint32_t j = q;  // the entries from j on have been looked at
                        for (uint32_t c = 0; !found && j > 0u && (c < kNear || (j & 31u) != 0u); ++c) {
                            --j;
                            const bool here = j >= blk * kTile;
                            least = min(least, here ? sh.u.tile.V[i][j - blk * kTile]
                                                    : __ldcg(w.Vs + (uint64_t)i * kSeqPiece + j));
                            found = (here ? sh.u.tile.pos[i][j - blk * kTile] : el_pos(row(D + i)[j])) == target_pos;
                        }
                        // A warp or block is passed whole while its first entry is a later update of this
                        // counter.  Where its first entry is on another counter, the counter's entries
                        // begin inside it, so the previous update lies inside it or was passed.
                        while (!found && j > blk * kTile) {
                            j -= 32u;
                            least = min(least, sh.u.tile.low[i][(j - blk * kTile) / 32u]);
                            found = sh.u.tile.pos[i][j - blk * kTile] <= target_pos;
                        }
                        for (uint32_t b = (j + kTile - 1u) / kTile; !found && b-- > 0u;) {
                            least = min(least, __ldcg(w.low + i * kBlocks + b));
                            found = el_pos(row(D + i)[b * kTile]) <= target_pos;
                        }
                    }
                    w.W[(uint64_t)pos * kStride + i] = least;
                }
            }
            const uint32_t kop = kpo & 3u, kpos = (kpo & ~kHead) >> 2;
            // {target, where it may be raised: distance of the cap above it << 3 | row} by position, in the half of
            // the key row that its sort left
            uint2* rec = reinterpret_cast<uint2*>(((a.key_passes & 1u) ? w.el0 : w.el1) + (uint64_t)(2 * D) * kSeqPiece);
            uint32_t F = kTop, G = kTop, start[D], had[D], word = 0u;
            uint2 mine = make_uint2(0u, 0u);
            if (valid) F = least_of(w.V, kpos);
#pragma unroll
            for (int i = 0; i < D; ++i) {
                start[i] = (bpo[i] & kHead) ? __ldcg(slim_ptr(s, i, el_key(row(i)[q]))) : 0u;
                had[i] = 0u;
            }
            // at most one iteration per update: each settles at least the first unsettled insertion
            for (uint32_t it = 0; it <= a.n + 1u; ++it) {
                // the last iteration's count, targets and caps, in one trip
                const uint32_t more = it > 0u ? __ldcg(w.flag + word) : 1u;
                typename Low::T u[D], before[D];
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    const uint32_t op = bpo[i] & 3u;
                    u[i] = Low::identity();
                    if (op == kOpIns && it > 0u) {
                        const uint2 r = __ldcg(rec + pos_of(i));
                        u[i].x = r.x;
                        if constexpr (kClimb) {
                            if ((r.y & 7u) == (uint32_t)i && r.y > 7u) {
                                u[i].z = 1u;
                                u[i].w = r.x + (r.y >> 3);
                            }
                        }
                    }
                    if (op == kOpDel) u[i].y = M[i];
                    if (bpo[i] & kHead) {
                        typename Low::T c = Low::identity();
                        c.x = c.y = start[i];
                        u[i] = Low::compose(c, u[i]);
                    }
                }
                if (more == 0u) break;  // the targets are as before the last iteration, so v holds the counters after it
                if (!grid_scan<Low, D, true>(u, before, sh, w.agg, a, target)) return;
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    v[i].x = u[i].x;
                    const uint32_t b = (bpo[i] & kHead) ? start[i] : before[i].x;
                    // (kClimb's bounds settle unevenly: most are as the last iteration left them)
                    if ((bpo[i] & 3u) == kOpIns && (!kClimb || it == 0u || b != had[i]))
                        w.a[(uint64_t)pos_of(i) * kStride + i] = b;
                    had[i] = b;
                }
                if (!barrier()) return;
                uint3 f[1], unused[1];
                f[0] = ShiftMap::identity();
                uint32_t av[kStride], m = kTop;
                if (valid) {
                    if (kop == kOpIns) {
                        m = read_rows(w.a, kpos, av);
                        if constexpr (!kIns)
                            if (it == 0u) G = least_of(w.W, kpos);
                        const uint32_t lo = min(F, add_sat(m, 1u));
                        f[0] = (kpo & kHead) ? make_uint3(lo, lo, 0u)
                                             : make_uint3(lo, min(F, add_sat(max(m, G), 1u)), 1u);
                    } else if (kpo & kHead) {
                        f[0] = make_uint3(0u, 0u, 0u);  // nothing known of the key's Slim minimum yet
                    } else {
                        if constexpr (!kIns)
                            if (it == 0u) G = least_of(w.W, kpos);
                        f[0] = make_uint3(0u, min(G, F), 0u);  // a deletion
                    }
                }
                // From the fourth iteration on, a key's run enters the next block an iteration late, for a barrier less: a
                // bound from below all the same.  Streams that settle in three or four would take one more.
                uint4* runs = w.agg + (uint64_t)(D + (it & 1u)) * kBlocks;
                const uint4* last_runs = it >= 3u ? w.agg + (uint64_t)(D + (~it & 1u)) * kBlocks : nullptr;
                if (!grid_scan<ShiftMap, 1, false>(f, unused, sh, runs, a, target, last_runs)) return;
                bool changed = false;
                if (valid && kop == kOpIns) {
                    changed = it == 0u || f[0].x != mine.x;
                    // In the row that alone holds the least of the key's Slim counters the insertion raises whatever
                    // is there by one, as far as the other rows' bounds and F allow.
                    uint2 r = make_uint2(f[0].x, 0u);
                    if constexpr (kClimb) {
                        uint32_t at = 0u, others = kTop;
#pragma unroll
                        for (int i = 0; i < D; ++i) {
                            if (av[i] == m) at = i;
                            uint32_t o = kTop;
#pragma unroll
                            for (int j = 0; j < D; ++j)
                                if (j != i) o = min(o, av[j]);
                            if (av[i] == m) others = o;
                        }
                        const uint32_t cap = min(F, add_sat(others, 1u));
                        if (cap > r.x) r.y = min(cap - r.x, (1u << 29) - 1u) << 3 | at;
                    }
                    if (it == 0u || r.x != mine.x || r.y != mine.y) rec[kpos] = r;
                    mine = r;
                }
                word = calls & 3u;
                if (blk == 0u && tid == 0u) w.flag[(calls + 2u) & 3u] = 0u;
                ++calls;
                const uint32_t c = (uint32_t)__syncthreads_count(changed);
                if (c && tid == 0u) atomicAdd(w.flag + word, c);
                if (!barrier()) return;
            }
        }
    }

    // ---- the counters after the piece ------------------------------------------------------------------
#pragma unroll
    for (int i = 0; i < D; ++i) {
        if (bpo[i] & kLast) *slim_ptr(s, i, el_key(row(i)[q])) = v[i].x;
        if (valid) {
            const unsigned long long* C = row(D + i);
            const uint32_t key = el_key(C[q]);
            if (q + 1u == a.n || el_key(C[q + 1u]) != key)
                s.B[(uint64_t)i * wz + key] = w.Vs[(uint64_t)i * kSeqPiece + q];
        }
    }
    // the last block to leave resets the barrier for the next launch
    if (tid == 0u && gridDim.x > 1u) {
        if (atomicAdd(a.ctrl + kCtrlSeqDone, 1u) == gridDim.x - 1u) {
            *reinterpret_cast<unsigned long long*>(a.ctrl + kCtrlBarrier64) = 0ull;
            a.ctrl[kCtrlSeqDone] = 0u;
        }
    }
}

template <int D, bool kIns, bool kDel>
cudaError_t launch_kind(const ScanArgs& a, uint32_t blocks, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(seq_scan_kernel<D, kIns, kDel>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(Shared));
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kTile);
    cfg.dynamicSmemBytes = sizeof(Shared);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, seq_scan_kernel<D, kIns, kDel>, a);
}

template <int D>
cudaError_t launch_d(const ScanArgs& a, uint32_t blocks, cudaStream_t st) {
    if (a.ops) return launch_kind<D, false, false>(a, blocks, st);
    if (a.op_const > 0) return launch_kind<D, true, false>(a, blocks, st);
    return launch_kind<D, false, true>(a, blocks, st);
}

uint32_t digits_of(uint64_t limit) {  // 8-bit digits of keys below limit
    uint32_t p = 1;
    while (p < 4 && ((limit - 1) >> (8 * p)) != 0) ++p;
    return p;
}

}  // namespace

uint64_t seq_scan_workspace_bytes(uint32_t d) { return ws_bytes(d); }

cudaError_t launch_seq_scan(const SketchDesc& s, const uint8_t* keys, const int8_t* ops, int32_t op_const, uint64_t n,
                            void* ws, uint32_t* ctrl, int num_sms, cudaStream_t st) {
    const uint64_t wz = (uint64_t)s.w * s.z;
    if (wz >= (1ull << 32)) return cudaErrorInvalidValue;
    // every block of a launch must be resident: one per SM
    const uint64_t most = (uint64_t)num_sms * kTile;
    const uint64_t piece = most < kSeqPiece ? most : kSeqPiece;
    for (uint64_t base = 0; base < n; base += piece) {
        ScanArgs a{};
        a.s = s;
        a.keys = keys + base * s.key_bytes;
        a.ops = ops ? ops + base : nullptr;
        a.op_const = op_const;
        a.n = (uint32_t)(n - base < piece ? n - base : piece);
        a.bucket_passes = digits_of(s.w);
        a.counter_passes = digits_of(wz);
        a.key_passes = a.n <= 2048u ? 2u : 3u;
        a.ws = ws;
        a.ctrl = ctrl;
        a.timeout_ns = kBarrierTimeoutNs;
        const uint32_t blocks = (a.n + kTile - 1) / kTile;
        cudaError_t e = cudaErrorInvalidValue;
        switch (s.d) {
            case 1: e = launch_d<1>(a, blocks, st); break;
            case 2: e = launch_d<2>(a, blocks, st); break;
            case 3: e = launch_d<3>(a, blocks, st); break;
            case 4: e = launch_d<4>(a, blocks, st); break;
            case 5: e = launch_d<5>(a, blocks, st); break;
            case 6: e = launch_d<6>(a, blocks, st); break;
            case 7: e = launch_d<7>(a, blocks, st); break;
            case 8: e = launch_d<8>(a, blocks, st); break;
            default: break;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace sfk
