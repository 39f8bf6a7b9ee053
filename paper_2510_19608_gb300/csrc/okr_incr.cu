// okr_incr.cu -- the exhaustive search (Algorithm 1, Sec. IV) with every
// candidate's score carried from one iteration to the next.
//
// Why scores can be carried.  As in okr_persist.cu, candidate c = (s, r) with
// a = lca(s, r) moves voltages only in two preorder ranges (the subtrees of the
// children of a toward s and toward r), and its SMICE is s_cur + D(c) with
//   D(c) = sum over its positions k and scenarios l of
//          (new MICE of k) - MICE_k  [- MICE_r when k = s: the merged cluster],
// the positions being the super-nodes of the two ranges (r excluded) and s.
// One term reads only: k's voltage, extremes and MICE; r's aggregated
// injection; the geometry (s, r, a); and, for k = s, r's extremes and MICE.
// A merge (s*, r*) changes those inputs only for the clusters whose voltage
// moves (the merge's own two ranges), for s* (extremes, MICE, injection) and
// for r* (removed); the quotient edges change only around s* and r*.  So after
// a merge only the terms that read a changed input are evaluated again:
//   - candidates next to s* or r* (slot pairs of s* and of the children of s*
//     and r* in the quotient tree) are rebuilt and every term evaluated;
//   - every other candidate evaluates the terms of its positions inside the
//     changed set, once on the state before the merge (subtracted) and once
//     on the state after it (added), plus its s term when r's MICE changed.
// On a 1,000-bus feeder that is about 0.2 % of the terms a full sweep
// evaluates.
//
// Exactness.  Carried sums are 128-bit fixed-point integers (units of 2^-100
// p.u.).  A term is converted by a fixed function of its bits; integer
// addition is associative, so removing a term's old value and adding its new
// one gives exactly the sum a fresh evaluation of every term gives, in any
// order.  The old value is recomputed from the unchanged inputs by the same
// arithmetic, every operation of which is explicitly rounded (no contraction
// into fused multiply-adds, whose use could differ between inlined copies), so
// it is bit-identical to the value added earlier.  Counts of terms above the
// margin are carried the same way.
// Engine 3 checks the carried values against a fresh evaluation after every
// merge.
//
// Precision 0 carries FP64 terms and selects on them exactly: the minimum m
// over feasible candidates, the tie band D <= m + tau, the smallest (r, s) key
// in it.  Precision 1 (GB300's FP64 rate is a small fraction of its FP32 rate)
// carries FP32 terms of the same quantities with the rigorous per-term bound
// of okr_persist.cu, summed into a bound B(c) >= |D32 - D64|, and counts of
// terms surely / possibly above the margin.  The selection of okr_persist.cu's
// screen then decides the FP64 winner, or names the few candidates whose FP64
// score it needs; those are evaluated in FP64 from scratch.  Merges are always
// applied in FP64.
//
// Execution.  One cluster of eight CTAs (inc_plan; in a batch one CTA, or a
// cluster for the longest searches, inc_batch_clusters) runs a feeder's whole
// search; its steps are separated by block or cluster barriers only (no grid
// barrier, no device-side wait).  The chain of dependent merges bounds it: neither a pipe nor memory is busy, so what counts is the number of
// dependent steps per merge and the latency of each.  A term is evaluated by a
// group of lanes, one per (scenario, phase).  Each merge takes three steps:
//   1. selection over the records (in a cluster two exchanges of minima);
//   2. the merge: its own FP64 evaluation into a scratch on the last warps and,
//      beside it on the others, the previous merge's write-back, the changed
//      candidates, the rebuilt ones (which read the clusters through the merge's
//      view) and the bookkeeping of clusters and super-nodes;
//   3. the terms that change, each before the merge (the state as stored) and
//      after it (the stored state overlaid with the scratch's new values), and
//      the merge's score.
// The write-back waits for the next merge's step 2, whose evaluation reads the
// not yet written values through the overlay, so no barrier is needed for it.
// (Rebuilding in a step of its own, between barriers, with the write-back after
// the terms took 14.0 us a merge on 1,000 buses, a cluster, FP32 terms; 9.8 now.)
#include "okr_internal.cuh"
#include "okr_kernels.cuh"

#include <climits>
#include <type_traits>

namespace okr {

namespace {

typedef unsigned __int128 u128;

constexpr int kFxShift = 100;               // fixed point: value * 2^100
constexpr u128 kSignBit = (u128)1 << 127;
constexpr u128 kNone = ~(u128)0;
constexpr int kMaxCluster = 8;              // CTAs of one search, at most
constexpr float kU32 = 5.9604645e-08f;      // 2^-24

__device__ __forceinline__ unsigned long long gtimer_inc() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// d * 2^100 truncated toward zero, modulo 2^128 (|d| < 2^27 is represented
// exactly up to the truncation; larger values wrap, which subtraction of the
// same value undoes).  Non-finite d counts as 0 (its term is infeasible anyway).
__device__ __forceinline__ u128 to_fx(double d) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    int e = (int)((b >> 52) & 0x7ff);
    if (e == 0x7ff) return 0;
    unsigned long long m = b & 0xfffffffffffffull;
    if (e == 0) e = 1;
    else m |= 1ull << 52;
    // d = m * 2^(e - 1075), so d * 2^100 = m * 2^(e - 975)
    const int sh = e - 1075 + kFxShift;
    u128 v;
    if (sh >= 0) v = sh >= 128 ? (u128)0 : ((u128)m << sh);
    else v = sh <= -64 ? (u128)0 : (u128)(m >> (-sh));
    return (b >> 63) ? (u128)0 - v : v;
}

__device__ __forceinline__ double fx_to_d(u128 v) {
    const bool neg = (v & kSignBit) != 0;
    const u128 a = neg ? (u128)0 - v : v;
    const double r = (double)(unsigned long long)(a >> 64) * 18446744073709551616.0 + (double)(unsigned long long)a;
    const double x = r * 7.8886090522101180541e-31;     // 2^-100
    return neg ? -x : x;
}

__device__ __forceinline__ u128 ld128(const unsigned long long *p) {
    return ((u128)p[1] << 64) | (u128)p[0];
}
__device__ __forceinline__ void st128(unsigned long long *p, u128 v) {
    p[0] = (unsigned long long)v;
    p[1] = (unsigned long long)(v >> 64);
}
// signed order as unsigned order
__device__ __forceinline__ u128 okey(u128 v) { return v ^ kSignBit; }
__device__ __forceinline__ u128 umin(u128 a, u128 b) { return a < b ? a : b; }

__device__ __forceinline__ u128 shfl_xor_u128(u128 v, int o) {
    const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)v, o);
    const unsigned long long hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(v >> 64), o);
    return ((u128)hi << 64) | lo;
}

// Exact 128-bit accumulation into shared memory from many threads: the low
// words add modulo 2^64 and every addition that wraps carries one into the high
// word, so the pair ends as the exact sum modulo 2^128 in any order.
__device__ __forceinline__ void sadd128(unsigned long long *lo, unsigned long long *hi, u128 v) {
    const unsigned long long vl = (unsigned long long)v, vh = (unsigned long long)(v >> 64);
    const unsigned long long old = atomicAdd(lo, vl);
    atomicAdd(hi, vh + ((old + vl < old) ? 1ull : 0ull));
}

// ---------------------------------------------------------------- clusters
// A search runs on one cluster of cs CTAs (1, 2, 4 or 8).  csync: every thread
// of the cluster waits for every other's, and all memory written before it
// (shared, remote shared, device) is seen after it.
__device__ __forceinline__ void csync(int cs) {
    if (cs == 1) {
        __syncthreads();
    } else {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}
__device__ __forceinline__ int cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}
// What is published: written to another CTA's copy of the same shared array.
struct __align__(16) Pub {
    unsigned long long a, b, c, d;
};
__device__ __forceinline__ void publish(void *slot, int rank, const void *v, int chunks) {     // chunks of 16 bytes
    unsigned at;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((unsigned)__cvta_generic_to_shared(slot)), "r"(rank));
#pragma unroll
    for (int i = 0; i < chunks; ++i) {
        const ulonglong2 q = static_cast<const ulonglong2 *>(v)[i];
        asm volatile("st.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(at + 16 * i), "l"(q.x), "l"(q.y) : "memory");
    }
}

// ---------------------------------------------------------------- block primitives
// Every reduction: warps reduce with shuffles, warp 0 reduces the warps'
// partials and publishes the result; two barriers.
struct Red {
    u128 a, b, c;
    int i;
};

__device__ __forceinline__ Red red_op(Red x, Red y) {
    Red r;
    r.a = umin(x.a, y.a);
    r.b = umin(x.b, y.b);
    r.c = umin(x.c, y.c);
    r.i = x.i + y.i;
    return r;
}
__device__ __forceinline__ Red red_shfl(Red x, int o) {
    Red r;
    r.a = shfl_xor_u128(x.a, o);
    r.b = shfl_xor_u128(x.b, o);
    r.c = shfl_xor_u128(x.c, o);
    r.i = __shfl_xor_sync(0xffffffffu, x.i, o);
    return r;
}

// Three 128-bit minima and one int sum over the block.
template <int NT>
__device__ __forceinline__ Red block_red(Red v, Red *sm) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) v = red_op(v, red_shfl(v, o));
    if (lane == 0) sm[wid] = v;
    __syncthreads();
    if (wid == 0) {
        Red x;
        x.a = x.b = x.c = kNone;
        x.i = 0;
        if (lane < NT / 32) x = sm[lane];
        for (int o = 16; o > 0; o >>= 1) x = red_op(x, red_shfl(x, o));
        if (lane == 0) sm[32] = x;
    }
    __syncthreads();
    return sm[32];
}

// A 64-bit minimum over the warp by redux.sync: the minimum of the high words,
// then of the low words among the lanes that hold it.
__device__ __forceinline__ unsigned long long warp_min64(unsigned long long v) {
    const unsigned hi = (unsigned)(v >> 32);
    const unsigned mh = __reduce_min_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_min_sync(0xffffffffu, hi == mh ? (unsigned)v : 0xffffffffu);
    return ((unsigned long long)mh << 32) | ml;
}

// Exclusive prefix sum of one int per thread; *total = the block's sum.
template <int NT>
__device__ __forceinline__ int block_excl_scan(int v, int *total, int *sm) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sm[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int y = lane < NT / 32 ? sm[lane] : 0;
        const int y0 = y;
        for (int o = 1; o < 32; o <<= 1) {
            const int z = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += z;
        }
        if (lane < NT / 32) sm[lane] = y - y0;      // exclusive offsets of the warps
        if (lane == 31) sm[32] = y;                 // total
    }
    __syncthreads();
    *total = sm[32];
    return sm[wid] + x - v;
}

// ---------------------------------------------------------------- geometry
__device__ __forceinline__ int child_toward_inc(const Topo &T, int a, int v) {
    // children of a have increasing preorder ids; v's branch is the last one <= v
    int lo = T.child_off[a], hi = T.child_off[a + 1] - 1;
    if (hi < lo) return v;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (T.child[mid] <= v) lo = mid;
        else hi = mid - 1;
    }
    return T.child[lo];
}

// The clusters as a merge (s*, r*) leaves them, read while that merge is being
// written: r*'s members belong to s*; with dir = 1 s* takes r*'s top; ranks
// past r* drop by one.  Either value of an entry the merge is rewriting reads
// the same through the view, and the ranks are rewritten only after the
// rebuild.  With no merge (s = -1) the state as stored.
struct View {
    int s, r, dir;
    __device__ __forceinline__ int label(const State &S, int b) const {
        const int l = S.label[b];
        return l == r ? s : l;
    }
    __device__ __forceinline__ int top(const State &S, int w) const {
        return (w == s && dir == 1) ? S.top[r] : S.top[w];
    }
    __device__ __forceinline__ int ptop(const State &S, int w) const {
        return (w == s && dir == 1) ? S.ptop[r] : S.ptop[w];
    }
};
__device__ __forceinline__ View no_view() {
    View v;
    v.s = v.r = -1;
    v.dir = 0;
    return v;
}

// The two candidates of the quotient edge above super-node w, from the current
// clusters: x = super-node holding the parent of w's top, a = lca(x, w), cw and
// cx the children of a toward w and x.  Slot 2w: w's cluster joins x (s = x,
// r = w); slot 2w + 1: x's cluster joins w (s = w, r = x; never the slack's
// cluster).  js/ns and jr/nr hold the s-side and r-side subtrees as BUS
// ranges [j, j + size) (preorder ids); fixed = 1 when s is the common ancestor.
// Returns x (-1 for the slack's cluster, which has no edge above it).
__device__ int slot_geometry(const Topo &T, const State &S, const View &V, int n, int w, Cand &c0, Cand &c1) {
    c0.s = -1;
    c1.s = -1;
    const int pb = V.ptop(S, w);
    if (pb < 0 || V.label(S, w) != w) return -1;
    const int tw = V.top(S, w);
    const int x = V.label(S, pb);
    const bool direct = (x == pb);
    const int a = direct ? x : (int)T.lca[(size_t)x * n + w];
    const int cw = direct ? tw : child_toward_inc(T, a, w);
    const int cx = (x != a) ? child_toward_inc(T, a, x) : -1;
    const int szw = T.sz[cw], szx = cx >= 0 ? T.sz[cx] : 0;
    const unsigned pw = T.ph[w], px = T.ph[x];
    const unsigned long long ow = (unsigned)T.orig[w], ox = (unsigned)T.orig[x];
    if ((pw & px) == pw) {
        c0.s = x; c0.r = w; c0.a = a; c0.dir = 0;
        c0.js = cx >= 0 ? cx : 0; c0.ns = szx; c0.jr = cw; c0.nr = szw;
        c0.fixed = (x == a) ? 1 : 0; c0.pad = 0;
        c0.key = (ow << 15) | ox;                   // (caller r, caller s)
    }
    if (x != 0 && (px & pw) == px) {
        c1.s = w; c1.r = x; c1.a = a; c1.dir = 1;
        c1.js = cw; c1.ns = szw; c1.jr = cx >= 0 ? cx : 0; c1.nr = szx;
        c1.fixed = 0; c1.pad = 0;
        c1.key = (ox << 15) | ow;
    }
    return x;
}

// ---------------------------------------------------------------- sums of terms
// The sums of one tile of kTile work entries, as kLimbs signed limbs of
// kLimbBits bits in 32-bit words of shared memory (limb i counts units of
// 2^(kLimbBits i - 100)): a term is added limb by limb by the four lanes of its
// scenario, each with one 32-bit add that returns nothing, and the entry's
// 128-bit sum is put together once, modulo 2^128 -- the same integer as adding
// 128-bit terms, in any order.  An entry takes at most 2 states x kMaxScen scenarios
// x n positions, a limb one add of at most 2^14 + 2 in size each: 31 bits hold
// kLimbMaxBus buses (16,382), and kIncSmemMax admits fewer (asserted there).  (The
// 128-bit adds these replace, a 64-bit shared add that returns the old value,
// then the carry's, cost about 500 cycles of each round's chain, and the
// 128-bit shifts and shuffles before them as much.)
constexpr int kLimbBits = 14, kLimbs = 10, kTile = 192;
constexpr int kLimbMaxBus = (int)(INT_MAX / (2 * kMaxScen * ((1 << kLimbBits) + 2)));
struct EvalSmem {
    int d[kLimbs][kTile + 1], b[kLimbs][kTile + 1];     // (+ 1: the limbs of an entry in different banks)
    int n1[kTile], n2[kTile];
};
__device__ __forceinline__ u128 limb_sum(const int (*x)[kTile + 1], int i) {
    u128 v = 0;
#pragma unroll
    for (int k = 0; k < kLimbs; ++k) v += (u128)(__int128)x[k][i] << (kLimbBits * k);
    return v;
}
__device__ __forceinline__ void limb_add(int (*x)[kTile + 1], int i, int k, int piece) {
    if (piece != 0 && k < kLimbs) atomicAdd(&x[k][i], piece);
}
// Adds sgn * to_fx((double)f) to sum i: lane p of the scenario's four adds piece p
// (a 24-bit mantissa at any shift lies in three limbs); p = 3 adds `extra` to
// the lowest limb.
__device__ __forceinline__ void add_fx32(int (*x)[kTile + 1], int i, float f, int sgn, int p, int extra) {
    const unsigned b = __float_as_uint(f);
    int e = (int)((b >> 23) & 0xff);
    unsigned m = b & 0x7fffffu;
    if (e == 0xff) m = 0;
    else if (e == 0) e = 1;
    else m |= 1u << 23;
    int sh = e - 150 + kFxShift;
    if (sh < 0) {
        m = sh <= -32 ? 0u : m >> (-sh);
        sh = 0;
    }
    const int k = sh / kLimbBits, r = sh - k * kLimbBits;
    int piece = (int)((unsigned)(((unsigned long long)m << r) >> (kLimbBits * p)) & ((1u << kLimbBits) - 1));
    if (b >> 31) piece = -piece;
    if (p == 3) piece = extra;
    limb_add(x, i, p == 3 ? 0 : k + p, sgn < 0 ? -piece : piece);
}
// Adds sgn * to_fx(v) to sum i: lane p adds piece p, lane 0 also piece 4 (a
// 53-bit mantissa lies in five limbs).
__device__ __forceinline__ void add_fx64(int (*x)[kTile + 1], int i, double v, int sgn, int p) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    int e = (int)((b >> 52) & 0x7ff);
    unsigned long long m = b & 0xfffffffffffffull;
    if (e == 0x7ff) m = 0;
    else if (e == 0) e = 1;
    else m |= 1ull << 52;
    int sh = e - 1075 + kFxShift;
    if (sh < 0) {
        m = sh <= -64 ? 0ull : m >> (-sh);
        sh = 0;
    }
    const int k = sh / kLimbBits, r = sh - k * kLimbBits;
    const bool neg = ((b >> 63) != 0) != (sgn < 0);
    const int mask = (1 << kLimbBits) - 1;
    // bits [14 p, 14 p + 14) of m << r: m has 53 bits, r < 14
    const int lo = kLimbBits * p - r;
    const int piece = (int)(lo >= 0 ? m >> lo : m << -lo) & mask;
    limb_add(x, i, k + p, neg ? -piece : piece);
    if (p == 0) {
        const int top = (int)(m >> (4 * kLimbBits - r)) & mask;
        limb_add(x, i, k + 4, neg ? -top : top);
    }
}

// ---------------------------------------------------------------- term groups
// A term (candidate c, position k) is evaluated by a group of G = 4 Lp lanes
// (Lp = scenarios rounded up to a power of two): lane gl takes scenario
// l = gl / 4 and phase p = gl % 4 (p = 3 idles).  Every lane of the warp calls
// the group function (it shuffles); the four lanes of a scenario add its term
// to the sums of the group's work entry.
//
// A group evaluates its term on one or two states (as many in every group of a
// warp): e = 0, the state as stored; e = 1,
// the state after the merge in progress, whose new values (voltage,
// magnitude, extremes, MICE of the merge's positions) are not yet written
// back and are read through the overlay.  With both, the result is the term
// on state 1 minus the term on state 0.  v_old / v_new say whether the group
// has a term on state 0 / 1.  The geometry (the voltage change the candidate
// causes) is the same on both states and is computed once.  The arithmetic of
// a term on one state's inputs (term_arith32, term_arith64) rounds every
// operation explicitly, so equal inputs give bit-equal results in every
// inlined copy.

// A merge whose new values are not in the state yet: map[x] = 1 + the index of
// super-node x among the merge's positions (0: unchanged), whose new values the
// merge's own evaluation left in cbuf (per position: per (l, p) the new voltage
// x, y and magnitude; per l the new MICE).  Positions from nfree on are the
// fixed s (its voltage does not move).  s* takes r*'s extremes.  A merge's
// values are written back while the next merge is evaluated, which reads them
// through the overlay, so there is one overlay (map and scratch) for the odd
// merges and one for the even; the state under an overlay may be read before or
// while it is written (s*'s extremes read the same either way).
struct Ovl {
    const unsigned short *map;
    const double *cbuf;
    int s, r, nfree;
};

// A position's FP32 copies in its scratch (after the 10 L FP64 values): per
// (l, p) the voltage, and the extremes relative to the magnitude; per l the MICE.
__device__ __forceinline__ float4 *cb_f4(const double *cb_pos, int L, int l, int p) {
    return reinterpret_cast<float4 *>(const_cast<double *>(cb_pos) + 10 * L) + (l * 3 + p);
}
__device__ __forceinline__ float *cb_mice32(const double *cb_pos, int L, int l) {
    return reinterpret_cast<float *>(const_cast<double *>(cb_pos) + 10 * L) + 12 * L + l;
}

// The super-node of a scratch position.
__device__ __forceinline__ int *cb_bus(const double *cb_pos, int L) {
    return reinterpret_cast<int *>(const_cast<double *>(cb_pos) + 10 * L) + 13 * L;
}

// FP64 state of super-node x, phase p, scenario l on state e (0 stored, 1 overlay).
__device__ __forceinline__ void at64(const State &S, const Ovl &O, int e, int x, int l, int p, int n, int L,
                                     bool need_v, double2 *v, double *hh, double *ll) {
    const size_t ix = sidx(l, p, x, n);
    const int j = e ? (int)O.map[x] - 1 : -1;
    double h = S.hi[ix], lo = S.lo[ix];
    if (j >= 0 && x == O.s) {
        const size_t irs = sidx(l, p, O.r, n);
        h = fmax(h, S.hi[irs]);
        lo = fmin(lo, S.lo[irs]);
    }
    *hh = h;
    *ll = lo;
    if (need_v) {
        if (j >= 0 && j < O.nfree) {
            const double *cb = O.cbuf + (size_t)j * kIncCbStride * L + (l * 3 + p) * 3;
            *v = make_double2(cb[0], cb[1]);
        } else {
            *v = S.vcur[ix];
        }
    }
}
__device__ __forceinline__ double mice64(const State &S, const Ovl &O, int e, int x, int l, int n, int L) {
    const int j = e ? (int)O.map[x] - 1 : -1;
    return j >= 0 ? O.cbuf[(size_t)j * kIncCbStride * L + 9 * L + l] : S.mice[(size_t)l * n + x];
}

// FP32 copies (voltage, extremes relative to the magnitude) and the FP64
// magnitude of super-node x on state e: the values the write-back stores.
__device__ __forceinline__ void at32(const State &S, const Ovl &O, int e, int x, int l, int p, int n, int L,
                                     bool need_v, bool need_mc, float2 *v, float *hr, float *lr, double *mc) {
    const size_t ix = sidx(l, p, x, n);
    const int j = e ? (int)O.map[x] - 1 : -1;
    if (j < 0) {
        *hr = S.hr32[ix];
        *lr = S.lr32[ix];
        if (need_v) *v = S.v32[ix];
        if (need_mc) *mc = S.mcur[ix];
        return;
    }
    // the FP32 copies the merge's evaluation derived (the write-back stores the same)
    const double *cbp = O.cbuf + (size_t)j * kIncCbStride * L;
    const float4 f = *cb_f4(cbp, L, l, p);
    *hr = f.z;
    *lr = f.w;
    if (need_v) *v = make_float2(f.x, f.y);
    if (need_mc) *mc = j >= O.nfree ? S.mcur[ix] : cbp[(l * 3 + p) * 3 + 2];
}
__device__ __forceinline__ float mice32(const State &S, const Ovl &O, int e, int x, int l, int n, int L) {
    const int j = e ? (int)O.map[x] - 1 : -1;
    return j >= 0 ? *cb_mice32(O.cbuf + (size_t)j * kIncCbStride * L, L, l) : S.mice32[(size_t)l * n + x];
}

// The arithmetic of one FP64 term on one state's inputs (every lane of the
// warp calls it: it shuffles).  Explicitly rounded operations: equal inputs
// give bit-equal results wherever it is inlined.
struct In64 {
    double2 v;
    double h, lo, hr, lr, mo, mr;
};
struct Out64 {
    double dd;
    int tv;
    double2 v;          // the merge's own evaluation: the new voltage, its magnitude, the distances of the
    double mag, up, dn, m;      // cluster's extremes above and below it, its MICE
};
__device__ __forceinline__ Out64 term_arith64(In64 x, double2 dv, bool one, bool moves, bool is_s, bool lv,
                                              double margin) {
    // every operation explicitly rounded (no contraction): each inlined copy
    // gives the same bits for the same inputs
    double em = 0.0;
    Out64 r;
    r.v = make_double2(0.0, 0.0);
    r.mag = r.up = r.dn = 0.0;
    if (one) {
        double2 v = x.v;
        if (moves) v = make_double2(__dadd_rn(v.x, dv.x), __dadd_rn(v.y, dv.y));
        const double mag = cmag(v);
        double h = x.h, lo = x.lo;
        if (is_s) {
            h = fmax(h, x.hr);
            lo = fmin(lo, x.lr);
        }
        r.up = __dsub_rn(h, mag);
        r.dn = __dsub_rn(mag, lo);
        em = fmax(r.up, r.dn);
        r.v = v;
        r.mag = mag;
    }
    double m = fmax(em, __shfl_xor_sync(0xffffffffu, em, 1));
    m = fmax(m, __shfl_xor_sync(0xffffffffu, m, 2));
    r.dd = 0.0;                         // (dd, tv, m: the same in the scenario's four lanes)
    r.tv = 0;
    r.m = m;
    if (lv) {
        r.dd = __dsub_rn(m, x.mo);
        if (is_s) r.dd = __dsub_rn(r.dd, x.mr);
        r.tv = (m > margin) ? 1 : 0;
    }
    return r;
}

// FP64 term, per l fixed(new MICE - MICE_k [- MICE_r]) and whether the new MICE
// exceeds the margin, added to sum ei of E: ne states from e0 on (e0 may differ
// between groups when ne = 1), state 1 with sign +, state 0 with sign sgn0.
// COMMIT (one state): the merge's own evaluation; returns the new values, and
// nothing is added.
template <bool COMMIT>
__device__ __forceinline__ Out64 group_term64(const Topo &T, const State &S, const uint8_t *ph, int n, int L, int G,
                                              const Cand &c, int k, int e0, int ne, int sgn0, bool v_old, bool v_new,
                                              const Ovl &O, int gl, double margin, EvalSmem *E, int ei) {
    const bool valid = v_old || v_new;
    const int l = gl >> 2, p = gl & 3;
    const bool lv = valid && l < L;
    const unsigned phk = valid ? ph[k] : 0u, phr = valid ? ph[c.r] : 0u;
    const bool on = lv && p < 3 && (phk >> p & 1u);
    const bool is_s = (k == c.s);
    const bool fixed = is_s && c.fixed;
    const bool sside = (k >= c.js && k < c.js + c.ns);
    const bool moves = on && !fixed;
    const int li = lv ? l : 0, pi = p < 3 ? p : 0;
    // the inputs of state e, loaded ahead of the arithmetic that uses them
    typedef In64 St;
    auto fetch = [&](int e, St &x) {
        const bool ve = e == 0 ? v_old : v_new;
        x.v = make_double2(0.0, 0.0);
        x.h = x.lo = x.mo = x.mr = 0.0;
        x.hr = -INFINITY;
        x.lr = INFINITY;
        if (on && ve) {
            at64(S, O, e, k, li, pi, n, L, true, &x.v, &x.h, &x.lo);
            if (is_s) at64(S, O, e, c.r, li, pi, n, L, false, nullptr, &x.hr, &x.lr);
        }
        if (lv && ve && !COMMIT) {
            x.mo = mice64(S, O, e, k, l, n, L);
            if (is_s) x.mr = mice64(S, O, e, c.r, l, n, L);
        }
    };
    St cur;
    fetch(e0, cur);
    // the voltage change at k (the same on both states)
    double2 dv = make_double2(0.0, 0.0);
    if (moves) {
        const int y = __ldg(T.lca + (size_t)(sside ? c.s : c.r) * n + k);
        double2 iq[3], za[3];
        for (int q = 0; q < 3; ++q) {
            iq[q] = (phr >> q & 1u) ? S.icur[sidx(li, q, c.r, n)] : make_double2(0.0, 0.0);
            za[q] = __ldg(T.zc + (size_t)c.a * 9 + pi * 3 + q);
        }
        // (every entry is loaded whatever the phases: one trip to L2, not three)
        const double2 *zp = T.zc + (size_t)y * 9 + pi * 3;
        const double2 zy[3] = {__ldg(zp), __ldg(zp + 1), __ldg(zp + 2)};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            if (!(phr >> q & 1u)) continue;
            const double2 g = sside ? csub(zy[q], za[q]) : csub(za[q], zy[q]);
            dv = cadd(dv, cmul(g, iq[q]));
        }
    }
    Out64 r;
#pragma unroll 1
    for (int i = 0; i < ne; ++i) {
        const int e = e0 + i;
        const bool ve = e == 0 ? v_old : v_new;
        const bool one = on && ve;
        St nxt = cur;
        if (i + 1 < ne) fetch(e + 1, nxt);
        r = term_arith64(cur, dv, one, moves, is_s, lv && ve, margin);
        cur = nxt;
        if (!COMMIT && lv && ve) {
            const int sgn = e == 1 ? 1 : sgn0;
            add_fx64(E->d, ei, r.dd, sgn, p);
            if (p == 0 && r.tv) atomicAdd(&E->n1[ei], sgn);
        }
    }
    return r;
}

// The arithmetic of one FP32 term with its bound on one state's inputs (every
// lane of the warp calls it: it shuffles).  Explicitly rounded operations:
// equal inputs give bit-equal results wherever it is inlined.
struct In32 {
    float hr, lr, hrr, lrr, mo, mr;
    float2 v;
    double mck, mcr;
};
struct Out32 {
    float dd, bl;
    int ts, tm;
};
__device__ __forceinline__ Out32 term_arith32(In32 x, float2 dv, float sdv, bool one, bool moves, bool sterm,
                                              bool lv, float margin_lo, float margin_hi) {
    // every operation explicitly rounded (no contraction): each inlined copy
    // gives the same bits for the same inputs
    float em = 0.0f, b = 0.0f;
    if (one) {
        float hr = x.hr, lr = x.lr, hrr = x.hrr, lrr = x.lrr;
        float bx = 0.0f;
        if (sterm) {
            const float dr = (float)__dsub_rn(x.mcr, x.mck);
            hrr = __fadd_rn(hrr, dr);
            lrr = __fadd_rn(lrr, dr);
            hr = fmaxf(hr, hrr);
            lr = fminf(lr, lrr);
            bx = __fmul_rn(2.0f * kU32, __fadd_rn(__fadd_rn(fabsf(hrr), fabsf(lrr)), __fmul_rn(2.0f, fabsf(dr))));
        }
        float delta = 0.0f, bd = 0.0f;
        if (moves) {
            const float2 v = x.v;
            const float s1 = __fadd_rn(__fmul_rn(v.x, dv.x), __fmul_rn(v.y, dv.y));
            const float s2 = __fadd_rn(__fmul_rn(dv.x, dv.x), __fmul_rn(dv.y, dv.y));
            const float num = __fadd_rn(__fmul_rn(2.0f, s1), s2);
            const float wx = __fadd_rn(v.x, dv.x), wy = __fadd_rn(v.y, dv.y);
            const float mv = __fsqrt_rn(__fadd_rn(__fmul_rn(v.x, v.x), __fmul_rn(v.y, v.y)));
            const float den = __fadd_rn(__fsqrt_rn(__fadd_rn(__fmul_rn(wx, wx), __fmul_rn(wy, wy))), mv);
            delta = __fdiv_rn(num, den);
            const float v1 = __fadd_rn(fabsf(v.x), fabsf(v.y));
            bd = __fmul_rn(kU32, __fadd_rn(__fdiv_rn(__fmul_rn(__fmul_rn(40.0f, __fadd_rn(v1, sdv)), sdv), den),
                                           __fmul_rn(8.0f, fabsf(delta))));
        }
        em = fmaxf(__fsub_rn(hr, delta), __fsub_rn(delta, lr));
        const float ab = __fadd_rn(__fadd_rn(fabsf(hr), fabsf(lr)), fabsf(em));
        b = __fadd_rn(__fadd_rn(__fmul_rn(1.5f, __fadd_rn(__fmul_rn(kU32, ab), bd)), bx), 4e-15f);
    }
    float m = fmaxf(em, __shfl_xor_sync(0xffffffffu, em, 1));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
    float bm = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, 1));
    bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 2));
    Out32 r;                            // (the same in the scenario's four lanes)
    r.dd = r.bl = 0.0f;
    r.ts = r.tm = 0;
    if (lv) {
        r.dd = __fsub_rn(__fsub_rn(m, x.mo), x.mr);
        // rounding of MICE_k, MICE_r to FP32 and of the two subtractions; the
        // factor 1.001 covers the rounding of the bound's own arithmetic
        const float am = __fadd_rn(__fadd_rn(fabsf(x.mo), fabsf(x.mr)), fabsf(m));
        r.bl = __fmul_rn(1.001f, __fadd_rn(bm, __fmul_rn(3.0f * kU32, am)));
        r.ts = (__fsub_rd(m, bm) > margin_hi) ? 1 : 0;
        r.tm = (__fadd_ru(m, bm) > margin_lo) ? 1 : 0;
    }
    return r;
}

// FP32 term with a rigorous bound (the screen of okr_persist.cu, per item
// e = max(hr - delta, delta - lr) relative to the cluster's present magnitude).
// Added to sum ei of E, over l: d, fixed(D32 term); b, a fixed-point bound on
// |fixed(D32 term) - fixed(D64 term)|; n1, scenarios whose new MICE is surely
// above the margin; n2, scenarios where it may be.  States and signs as above.
__device__ __forceinline__ void group_term32(const Topo &T, const State &S, const uint8_t *ph, int n, int L, int G,
                                             const Cand &c, int k, int e0, int ne, int sgn0, bool v_old, bool v_new,
                                             const Ovl &O, int gl, float margin_lo, float margin_hi, EvalSmem *E,
                                             int ei) {
    const bool valid = v_old || v_new;
    const int l = gl >> 2, p = gl & 3;
    const bool lv = valid && l < L;
    const unsigned phk = valid ? ph[k] : 0u, phr = valid ? ph[c.r] : 0u;
    const bool on = lv && p < 3 && (phk >> p & 1u);
    const bool is_s = (k == c.s);
    const bool fixed = is_s && c.fixed;
    const bool sside = (k >= c.js && k < c.js + c.ns);
    const bool sterm = on && is_s && (phr >> p & 1u);
    const bool moves = on && !fixed;
    const int li = lv ? l : 0, pi = p < 3 ? p : 0;
    // the inputs of state e, loaded ahead of the arithmetic that uses them
    typedef In32 St;
    auto fetch = [&](int e, St &x) {
        const bool ve = e == 0 ? v_old : v_new;
        x.hr = x.lr = x.hrr = x.lrr = x.mo = x.mr = 0.0f;
        x.v = make_float2(0.0f, 0.0f);
        x.mck = x.mcr = 0.0;
        if (on && ve) at32(S, O, e, k, li, pi, n, L, moves, sterm, &x.v, &x.hr, &x.lr, &x.mck);
        if (on && ve && sterm) {
            float2 vr;
            at32(S, O, e, c.r, li, pi, n, L, false, true, &vr, &x.hrr, &x.lrr, &x.mcr);
        }
        if (lv && ve) {
            x.mo = mice32(S, O, e, k, l, n, L);
            if (is_s) x.mr = mice32(S, O, e, c.r, l, n, L);
        }
    };
    St cur;
    fetch(e0, cur);
    // the voltage change at k (the same on both states)
    float2 dv = make_float2(0.0f, 0.0f);
    float sdv = 0.0f;
    if (moves) {
        const int y = __ldg(T.lca + (size_t)(sside ? c.s : c.r) * n + k);
        float2 iq[3], ha[3], la[3];
        for (int q = 0; q < 3; ++q) {
            iq[q] = (phr >> q & 1u) ? S.icur32[sidx(li, q, c.r, n)] : make_float2(0.0f, 0.0f);
            ha[q] = __ldg(T.zh + (size_t)c.a * 9 + pi * 3 + q);
            la[q] = __ldg(T.zlo + (size_t)c.a * 9 + pi * 3 + q);
        }
        // (every entry is loaded whatever the phases: one trip to L2, not three)
        const float2 *zhp = T.zh + (size_t)y * 9 + pi * 3, *zlp = T.zlo + (size_t)y * 9 + pi * 3;
        const float2 zhy[3] = {__ldg(zhp), __ldg(zhp + 1), __ldg(zhp + 2)};
        const float2 zly[3] = {__ldg(zlp), __ldg(zlp + 1), __ldg(zlp + 2)};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            if (!(phr >> q & 1u)) continue;
            const float2 hy = zhy[q], ly = zly[q];
            float gx = (hy.x - ha[q].x) + (ly.x - la[q].x);
            float gy = (hy.y - ha[q].y) + (ly.y - la[q].y);
            if (!sside) { gx = -gx; gy = -gy; }
            dv.x = fmaf(gx, iq[q].x, fmaf(-gy, iq[q].y, dv.x));
            dv.y = fmaf(gx, iq[q].y, fmaf(gy, iq[q].x, dv.y));
            sdv = fmaf(fabsf(gx) + fabsf(gy), fabsf(iq[q].x) + fabsf(iq[q].y), sdv);
        }
    }
#pragma unroll 1
    for (int i = 0; i < ne; ++i) {
        const int e = e0 + i;
        const bool ve = e == 0 ? v_old : v_new;
        const bool one = on && ve;
        St nxt = cur;
        if (i + 1 < ne) fetch(e + 1, nxt);
        const Out32 r = term_arith32(cur, dv, sdv, one, moves, sterm, lv && ve, margin_lo, margin_hi);
        cur = nxt;
        if (lv && ve) {
            const int sgn = e == 1 ? 1 : sgn0;
            add_fx32(E->d, ei, r.dd, sgn, p, 0);
            add_fx32(E->b, ei, r.bl, sgn, p, 3);        // (3: the truncations of both terms to fixed point)
            if (p == 0 && r.ts) atomicAdd(&E->n1[ei], sgn);
            if (p == 0 && r.tm) atomicAdd(&E->n2[ei], sgn);
        }
    }
}

// ---------------------------------------------------------------- the changed set of a merge
struct Win {
    int slot, s, r, a, dir, fixed;
    int w1lo, w1hi, w2lo, w2hi;     // bus ranges whose voltages move
    int jr;                         // rank of r before the merge
    int npos;                       // positions of the merge (ranks of the two ranges, r excluded, + fixed s)
    int q1lo, q1hi, q2lo, q2hi;     // their rank ranges before the merge
};

__device__ __forceinline__ bool in_range(int b, int lo, int hi) { return b >= lo && b < hi; }

// The winner's record from its candidate (slot ws) and the super-node ranks.
__device__ __forceinline__ Win make_win(const Cand &w, int ws, const unsigned short *rank) {
    Win h;
    h.slot = ws; h.s = w.s; h.r = w.r; h.a = w.a; h.dir = w.dir; h.fixed = w.fixed;
    h.w1lo = w.js; h.w1hi = w.js + w.ns; h.w2lo = w.jr; h.w2hi = w.jr + w.nr;
    h.jr = rank[w.r];
    h.q1lo = w.ns > 0 ? rank[w.js] : 0;
    h.q1hi = w.ns > 0 ? rank[w.js + w.ns] : 0;
    h.q2lo = w.nr > 0 ? rank[w.jr] : 0;
    h.q2hi = w.nr > 0 ? rank[w.jr + w.nr] : 0;
    h.npos = (h.q1hi - h.q1lo) + (h.q2hi - h.q2lo) + w.fixed;
    return h;
}


// Whether candidate c (not next to s* or r*) has a term that reads an input
// the merge h changes: a position in the moved ranges or at s*, r*; its fixed
// s when that cluster changed; its s term when r's MICE changed.
__device__ __forceinline__ bool touched(const Cand &c, const Win &h) {
    auto in_cr = [&](int b) { return in_range(b, c.js, c.js + c.ns) || in_range(b, c.jr, c.jr + c.nr); };
    auto in_w = [&](int b) { return in_range(b, h.w1lo, h.w1hi) || in_range(b, h.w2lo, h.w2hi); };
    const int clo[2] = {c.js, c.jr}, chi[2] = {c.js + c.ns, c.jr + c.nr};
    const int wlo[2] = {h.w1lo, h.w2lo}, whi[2] = {h.w1hi, h.w2hi};
    for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 2; ++j)
            if (max(clo[i], wlo[j]) < min(chi[i], whi[j])) return true;
    if (in_cr(h.s) || in_cr(h.r)) return true;
    if (c.fixed && (in_w(c.s) || c.s == h.s || c.s == h.r)) return true;
    return in_w(c.r) || c.r == h.s || c.r == h.r;
}

// Rank ranges of the terms of candidate c that read an input the merge h
// changes (c is not next to s* or r*).  Returns their number.
__device__ int changed_segments(const Cand &c, const Win &h, const unsigned short *sn_rank, int2 *seg) {
    int k = 0;
    const int clo[2] = {c.js, c.jr}, chi[2] = {c.js + c.ns, c.jr + c.nr};
    const int wlo[2] = {h.w1lo, h.w2lo}, whi[2] = {h.w1hi, h.w2hi};
    for (int i = 0; i < 2; ++i) {
        if (clo[i] >= chi[i]) continue;
        for (int j = 0; j < 2; ++j) {
            if (wlo[j] >= whi[j]) continue;
            const int lo = max(clo[i], wlo[j]), hi = min(chi[i], whi[j]);
            if (lo < hi) {
                const int a = sn_rank[lo], b = sn_rank[hi];
                if (a < b) seg[k++] = make_int2(a, b);
            }
        }
    }
    // points: s* and r* where a range of c holds them outside the moved ranges,
    // and s when its term changes (it is not inside the ranges when fixed)
    auto in_cr = [&](int b) { return in_range(b, c.js, c.js + c.ns) || in_range(b, c.jr, c.jr + c.nr); };
    auto in_w = [&](int b) { return in_range(b, h.w1lo, h.w1hi) || in_range(b, h.w2lo, h.w2hi); };
    auto point = [&](int b) { const int a = sn_rank[b]; seg[k++] = make_int2(a, a + 1); };
    if (h.s != c.r && in_cr(h.s) && !in_w(h.s)) point(h.s);
    if (h.r != c.r && in_cr(h.r) && !in_w(h.r)) point(h.r);
    // the s term also reads r's MICE
    const bool r_changed = in_w(c.r) || c.r == h.s || c.r == h.r;
    if (c.fixed) {
        if (in_w(c.s) || c.s == h.s || c.s == h.r || r_changed) point(c.s);
    } else if (r_changed && !in_w(c.s) && c.s != h.s && c.s != h.r) {
        point(c.s);
    }
    return k;
}

// Every term of candidate c: its two ranges and the fixed s, as ranks.
template <typename RK>
__device__ int full_segments(const Cand &c, const RK *sn_rank, int2 *seg, int rdead = -1) {
    // rdead >= 0: ranks past bus rdead drop by one (the merge of r* = rdead)
    auto rk = [&](int b) { return sn_rank[b] - (rdead >= 0 && b > rdead ? 1 : 0); };
    int k = 0;
    if (c.ns > 0) {
        const int a = rk(c.js), b = rk(c.js + c.ns);
        if (a < b) seg[k++] = make_int2(a, b);
    }
    if (c.nr > 0) {
        const int a = rk(c.jr), b = rk(c.jr + c.nr);
        if (a < b) seg[k++] = make_int2(a, b);
    }
    if (c.fixed) { const int a = rk(c.s); seg[k++] = make_int2(a, a + 1); }
    return k;
}

// The list of work entries: its length (low word) and the items of its entries
// (high word), so that an entry learns its place and its first item at once.
__device__ __forceinline__ unsigned long long append(unsigned long long *list, int nseg, const int2 *seg) {
    int items = 0;
    for (int i = 0; i < nseg; ++i) items += seg[i].y - seg[i].x;
    return atomicAdd(list, ((unsigned long long)items << 32) | 1ull);
}
__device__ __forceinline__ void write_entry(IncWork *w, int slot, int mode, int off, int nseg, const int2 *seg,
                                            const Cand &c) {
    w->slot = slot;
    w->mode = mode;
    w->nseg = nseg;
    w->off = off;
    for (int i = 0; i < nseg; ++i) w->seg[i] = seg[i];
    w->s = c.s; w->r = c.r; w->a = c.a;
    w->js = c.js; w->ns = c.ns; w->jr = c.jr; w->nr = c.nr; w->fixed = c.fixed;
}

__device__ __forceinline__ Cand entry_cand(const IncWork &w) {
    Cand c;
    c.s = w.s; c.r = w.r; c.a = w.a; c.dir = 0;
    c.js = w.js; c.ns = w.ns; c.jr = w.jr; c.nr = w.nr;
    c.fixed = w.fixed; c.pad = 0; c.key = 0;
    return c;
}

// Where one search keeps its per-merge data: the first `se` work entries
// (at most kSEMax), the super-node lists (16-bit, by merge parity) and the
// phase masks in shared memory; further entries in global memory.
constexpr int kSEMax = 256;
struct Loc {
    IncWork *wsm, *wgl;         // (wgl: this CTA's part of the feeder's work buffer)
    int *rlist;                 // this CTA's part of Inc::rlist
    int se;                     // work entries in shared memory
    unsigned short *lst[2];
    const uint8_t *ph;
    unsigned short *rank;       // [n + 1] rank of each bus's super-node among the super-nodes
    // the candidates and their carried sums and counts (as in Search::slot and
    // Inc): in device memory by slot (lg < 0), or the CTA's own slots in shared
    // memory, by record (lg: log2 of the cluster's size)
    int lg;
    Cand *slot;
    unsigned long long *acc, *bnd;
    int *viol, *vmay;
    __device__ __forceinline__ int at(int sl) const { return lg < 0 ? sl : ((sl >> (lg + 1)) << 1) | (sl & 1); }
    __device__ __forceinline__ IncWork *ent(int i) const { return i < se ? wsm + i : wgl + (i - se); }
};

// ---------------------------------------------------------------- evaluation of work entries
enum Pass {
    kMerge = 0,     // after a merge: mode 0 adds (term after - term before), mode 1 sets every term after
    kFresh = 2,     // carried precision, every term after the merge in progress, into vacc / vviol
    kF64 = 3,       // FP64, every term on the stored state, into vacc / vviol
    kInitPart = 4   // the stored state, every term of the entries (parts of candidates): added to the carried
                    // sums with atomics, the records left to the search
};

// Per-slot selection records (shared memory when they fit, else global):
//   r0 (precision 0): okey(D) of a feasible candidate, kNone otherwise;
//   r1 (precision 1): order-preserving keys of the lower and upper end of the
//       interval that holds the FP64 score, in units of 2^-56 p.u. (lower end
//       rounded down, upper end up); the lower key is ~0 when the candidate is
//       surely infeasible, the upper key when it is not surely feasible (or
//       the slot holds no candidate).  Integer keys keep the selection off the
//       FP64 pipe;
//   tkey: the tie key (caller r, caller s), ~0u for an empty slot;
//   maxm: per super-node, its largest MICE over the scenarios (0 when absorbed);
//   span: per slot pair, what the changed-set scan tests first.
// The slot pairs of a search are dealt out to its cluster's CTAs, pair w to
// CTA w % cs; a CTA keeps its own pairs' records, pair w at index w / cs.
struct Rec {
    int lg;             // log2 of the cluster's size
    u128 *r0;
    ulonglong2 *r1;
    unsigned *tkey;
    double *maxm;
    ushort4 *span;      // per slot pair: bus span [x, y) holding both candidates' ranges, s and r;
                        // z: the quotient parent (0xffff: none); w: empty pair when 0
    // Summaries of blocks of 32 slots (shared memory), so that a selection
    // reads the blocks, not every record: the smallest r0 (precision 0) or the
    // smallest lower and upper keys (precision 1), the slots holding a
    // candidate, and the largest maxm over the block's 16 super-nodes (bit
    // patterns: MICE >= 0 orders like its bits).  A block whose records
    // changed since the last selection is marked dirty and summarised again
    // before the next one.
    void *bsum;         // [nb] u128 (precision 0) or ulonglong2 (precision 1)
    int *bcnt;          // [nb]
    unsigned long long *bmx;    // [nb]
    unsigned char *dirty;       // [nb]
    int nb;
    // index of slot sl's record
    __device__ __forceinline__ int at(int sl) const { return ((sl >> (lg + 1)) << 1) | (sl & 1); }
    // (dirty is null where there are no summaries: the first evaluation on many
    // CTAs, and a cluster of several CTAs, whose selection reads every record)
    __device__ __forceinline__ void touch(int sl) const { if (dirty) dirty[sl >> 5] = 1; }
    __device__ __forceinline__ void touch_sn(int k) const { if (dirty) dirty[k >> 4] = 1; }   // maxm of super-node k (slot 2k)
};

constexpr int kKeyShift = 44;                       // 2^-100 -> 2^-56 units
constexpr unsigned long long kKeyNone = ~0ull;

// floor(v / 2^44) of a signed fixed-point value, as an order-preserving key;
// *ok = false when it does not fit 64 bits.
__device__ __forceinline__ unsigned long long key_floor(u128 v, bool *ok) {
    const bool neg = (v & kSignBit) != 0;
    const u128 q = neg ? ~((~v) >> kKeyShift) : (v >> kKeyShift);      // arithmetic shift
    const u128 top = q >> 63;                                          // all sign bits above 63
    *ok = neg ? (top == ((u128)1 << 65) - 1) : (top == 0);
    return (unsigned long long)q ^ 0x8000000000000000ull;
}
__device__ __forceinline__ unsigned long long key_ceil(u128 v, bool *ok) {
    // ceil(v / 2^44) = -floor(-v / 2^44)
    const unsigned long long k = key_floor((u128)0 - v, ok);
    return (unsigned long long)(-(long long)(k ^ 0x8000000000000000ull)) ^ 0x8000000000000000ull;
}
__device__ __forceinline__ long long key_val(unsigned long long k) { return (long long)(k ^ 0x8000000000000000ull); }
__device__ __forceinline__ unsigned long long val_key(long long v) {
    return (unsigned long long)v ^ 0x8000000000000000ull;
}

__device__ __forceinline__ unsigned long long warp_max64(unsigned long long v) { return ~warp_min64(~v); }
__device__ __forceinline__ u128 warp_min128(u128 v) {
    // the smallest high word, then the smallest low word among the lanes that hold it
    const unsigned long long hi = (unsigned long long)(v >> 64), mh = warp_min64(hi);
    const unsigned long long ml = warp_min64(hi == mh ? (unsigned long long)v : ~0ull);
    return ((u128)mh << 64) | ml;
}

// Pass B of the selection reads every record when they are in shared memory
// and the feeder has at most this many buses (at most 8 records a thread of
// a 384-thread CTA; measured faster up to 1,000 buses, slower from 2,200);
// otherwise it reads the blocks that may hold a candidate of the tie band, one
// warp per block (or all warps each, when there are at most kFewBlocks).
constexpr int kFlatSelectMax = 1536;
constexpr int kFewBlocks = 8;

// The summaries of the dirty blocks, one warp per block, then a barrier.
template <int NT, int PREC>
__device__ __forceinline__ void refresh_blocks(const Rec &R, int n) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int j = wid; j < R.nb; j += NT / 32) {
        if (!R.dirty[j]) continue;                      // (the same for the whole warp)
        const int c = 32 * j + lane;
        const bool in = c < 2 * n;
        const unsigned long long mb =
            (in && (c & 1) == 0) ? (unsigned long long)__double_as_longlong(R.maxm[c >> 1]) : 0ull;
        const unsigned cnt = __popc(__ballot_sync(0xffffffffu, in && R.tkey[c] != ~0u));
        const unsigned long long mx = warp_max64(mb);
        if (PREC == 0) {
            const u128 k = warp_min128(in ? R.r0[c] : kNone);
            if (lane == 0) reinterpret_cast<u128 *>(R.bsum)[j] = k;
        } else {
            const ulonglong2 q = in ? R.r1[c] : make_ulonglong2(kKeyNone, kKeyNone);
            const unsigned long long lo = warp_min64(q.x), hi = warp_min64(q.y);
            if (lane == 0) reinterpret_cast<ulonglong2 *>(R.bsum)[j] = make_ulonglong2(lo, hi);
        }
        if (lane == 0) {
            R.bcnt[j] = (int)cnt;
            R.bmx[j] = mx;
            R.dirty[j] = 0;
        }
    }
    __syncthreads();
}

// The span record of a pair with candidates c (x: its quotient parent, -1: none).
__device__ __forceinline__ ushort4 pair_span(int n, const Cand *c, int x) {
    int lo = n, hi = 0;
    for (int d = 0; d < 2; ++d) {
        if (c[d].s < 0) continue;
        lo = min(lo, min(min(c[d].s, c[d].r), c[d].ns > 0 ? c[d].js : n));
        lo = min(lo, c[d].nr > 0 ? c[d].jr : n);
        hi = max(hi, max(max(c[d].s, c[d].r) + 1, max(c[d].js + c[d].ns, c[d].jr + c[d].nr)));
    }
    const bool any = c[0].s >= 0 || c[1].s >= 0;
    return make_ushort4((unsigned short)(any ? lo : 0), (unsigned short)(any ? hi : 0),
                        (unsigned short)(x >= 0 ? x : 0xffff), (unsigned short)(any ? 1 : 0));
}

template <int PREC>
__device__ __forceinline__ void set_rec(const Rec &R, int sl, u128 d, u128 b, int viol, int vmay) {
    R.touch(sl);
    const int at = R.at(sl);
    if (PREC == 0) {
        R.r0[at] = (viol == 0) ? okey(d) : kNone;
    } else {
        unsigned long long lo = kKeyNone, hi = kKeyNone;
        if (viol == 0) {
            bool ok;
            lo = key_floor(d - b, &ok);
            if (!ok) lo = ((d - b) & kSignBit) ? 0ull : kKeyNone - 1;
            if (vmay == 0) {
                hi = key_ceil(d + b, &ok);
                if (!ok) hi = kKeyNone;
            }
        }
        R.r1[at] = make_ulonglong2(lo, hi);
    }
}
template <int PREC>
__device__ __forceinline__ void kill_rec(const Rec &R, int sl) {
    R.touch(sl);
    const int at = R.at(sl);
    if (PREC == 0) R.r0[at] = kNone;
    else R.r1[at] = make_ulonglong2(kKeyNone, kKeyNone);
    R.tkey[at] = ~0u;
}

// The merge's own evaluation (FP64, state before the merge): new voltage,
// magnitude and MICE of each of its positions into the scratch, the positions
// spread over the cluster.
struct Commit {
    const Win *h;
    Cand wc;
    const unsigned short *list;     // super-nodes before the merge
    const uint8_t *ph;
    Ovl O;                          // the merge before, still being written back
    double *cbuf;                   // this merge's scratch
};

// Run by warps [warp0, warp0 + nw) of every CTA of the cluster (CTA cr of cs).
__device__ __forceinline__ long long commit_groups(const Topo &T, const State &S, int n, int L, int G, double margin,
                                                   const Commit &cm, int warp0, int nw, int cr, int cs) {
    long long items = 0;
    // (positions go round the CTAs first, so that few positions meet few warps each;
    // G is a power of two: shifts, not divisions, on every thread's path)
    const int lgG = __ffs(G) - 1, lane = threadIdx.x & 31;
    const int lw = (((int)threadIdx.x >> 5) - warp0) * cs + cr, gpw = 32 >> lgG, gl = lane & (G - 1);
    const int gi = lw * gpw + (lane >> lgG), NG = nw * gpw * cs;
    const Win &h = *cm.h;
    const int n1 = h.q1hi - h.q1lo, n2 = h.q2hi - h.q2lo;
    for (int r0 = 0; r0 < h.npos; r0 += NG) {
        if (r0 + lw * gpw >= h.npos) break;             // this warp's groups are all past the end
        const int q = r0 + gi;
        bool valid = q < h.npos;
        int k = cm.wc.s;
        if (valid) {
            k = q < n1 ? cm.list[h.q1lo + q] : (q < n1 + n2 ? cm.list[h.q2lo + q - n1] : cm.wc.s);
            if (gl == 0) *cb_bus(cm.cbuf + (size_t)q * kIncCbStride * L, L) = k;
            if (k == cm.wc.r) { valid = false; k = cm.wc.s; }
        }
        const Out64 r = group_term64<true>(T, S, cm.ph, n, L, G, cm.wc, k, 1, 1, 1, false, valid, cm.O, gl, margin,
                                           nullptr, 0);
        if (valid) {
            // the new values, and their FP32 copies (what the write-back will store)
            const int l = gl >> 2, p = gl & 3;
            double *cb = cm.cbuf + (size_t)q * kIncCbStride * L;
            if (l < L && p < 3 && (cm.ph[k] >> p & 1u)) {
                double *o = cb + (l * 3 + p) * 3;
                o[0] = r.v.x;
                o[1] = r.v.y;
                o[2] = r.mag;
                *cb_f4(cb, L, l, p) = make_float4((float)r.v.x, (float)r.v.y, (float)r.up, 0.0f - (float)r.dn);
            }
            if (l < L && p == 0) {
                cb[9 * L + l] = r.m;
                *cb_mice32(cb, L, l) = (float)r.m;
            }
            if (gl == 0) items += __popc(cm.ph[k]) * L;
        }
    }
    return items;
}

// Evaluates the terms of work entries [0, ne_all), which hold `items` items (tiles
// of kTile entries), and applies them per the pass; ends without a barrier after
// the last tile's updates.  kMerge: mode-0 entries take positions from list_pre
// and add, per term, its value after the merge (r* has none) minus its value
// before; mode-1 entries take positions from list_post and set every term after
// the merge.  kFresh / kF64 / kInitPart: every term of the entries, positions
// from list_pre, on the state under the overlay (kInitPart: as stored).  The
// sums E are zero before and after.  Returns the number of terms evaluated.
template <int NT, int PREC>
__device__ __forceinline__ long long run_entries(const Topo &T, const State &S, const Inc &I, int n, int L, int G,
                                 double margin, float mlo, float mhi, int ne_all, int items, int pass,
                                 const unsigned short *list_pre, const unsigned short *list_post, int rstar,
                                 const Ovl O, EvalSmem &E, const Rec &R, const Loc &Lc,
                                 unsigned long long *prof = nullptr) {
    static_assert(NT >= kTile, "one thread per entry of a tile");
    const int lgG = __ffs(G) - 1;
    const int tid = threadIdx.x, gl = tid & (G - 1), gi = tid >> lgG, NG = NT >> lgG;
    long long terms = 0;
    unsigned long long tq = (prof && tid == 0) ? gtimer_inc() : 0;
    auto sub = [&](int i) {             // profile mode: time of the pass's steps (thread 0, after barriers)
        if (prof && tid == 0) { const unsigned long long now = gtimer_inc(); prof[i] += now - tq; tq = now; }
    };
    for (int t0 = 0; t0 < ne_all; t0 += kTile) {
        const int ne = min(kTile, ne_all - t0);
        const int q0 = t0 > 0 ? Lc.ent(t0)->off : 0, q1 = t0 + kTile < ne_all ? Lc.ent(t0 + kTile)->off : items;
        // the states: after a merge two, one after the other in a group, or, when
        // the CTA has groups enough for every item twice, one in each of two groups
        const bool both = pass == kMerge, apart = both && 2 * (q1 - q0) <= NG;
        const int tot = apart ? 2 * (q1 - q0) : q1 - q0;
        unsigned long long cq = (prof && tid == 0) ? clock64() : 0;
        // the first items of the tile's entries, two a lane, when 64 hold them all
        const bool near = ne <= 64;
        int of0 = INT_MAX, of1 = INT_MAX;
        if (near && (tid & 31) < ne) of0 = Lc.ent(t0 + (tid & 31))->off;
        if (near && (tid & 31) + 32 < ne) of1 = Lc.ent(t0 + (tid & 31) + 32)->off;
        for (int r0 = 0; r0 < tot; r0 += NG) {
            if (r0 + ((tid >> 5) << (5 - lgG)) >= tot) break;     // this warp's groups are all past the end
            const int u = r0 + gi, q = q0 + (apart ? u >> 1 : u);
            const int st0 = apart ? u & 1 : (both || pass == kInitPart ? 0 : 1), nst = both && !apart ? 2 : 1;
            bool valid = u < tot, v_old = false, v_new = false;
            int ei = 0, k = 0;
            Cand c;
            c.s = c.r = c.a = c.js = c.ns = c.jr = c.nr = c.fixed = 0;
            // the entry holding item q: the last one whose first item is <= q
            if (near) {
                const int g0 = r0 + ((tid >> 5) << (5 - lgG));      // the warp's first group
                for (int g = 0; g < (32 >> lgG); ++g) {
                    const int qg = q0 + (apart ? (g0 + g) >> 1 : g0 + g);
                    const int k2 = __popc(__ballot_sync(0xffffffffu, of0 <= qg)) + __popc(__ballot_sync(0xffffffffu, of1 <= qg));
                    if (g0 + g == u) ei = k2 - 1;
                }
            }
            if (valid) {
                if (!near) {
                    int lo = 0, hi = ne - 1;
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (Lc.ent(t0 + mid)->off <= q) lo = mid;
                        else hi = mid - 1;
                    }
                    ei = lo;
                }
                const IncWork &w = *Lc.ent(t0 + ei);
                int rem = q - w.off, j = 0;
                for (int i = 0; i < w.nseg; ++i) {
                    const int len = w.seg[i].y - w.seg[i].x;
                    if (rem < len) { j = w.seg[i].x + rem; break; }
                    rem -= len;
                }
                k = ((both && w.mode == 1) ? list_post : list_pre)[j];
                c = entry_cand(w);
                if (k == c.r) valid = false;
                if (both) {
                    v_old = valid && w.mode == 0;
                    v_new = valid && !(w.mode == 0 && k == rstar);
                } else {
                    v_old = v_new = valid;
                }
            }
            // (the state a group does not evaluate)
            if (nst == 1 && st0 == 0) v_new = false;
            if (nst == 1 && st0 == 1) v_old = false;
            if (gl == 0 && (v_old || v_new))                          // (phase-node, scenario) items
                terms += ((v_old ? 1 : 0) + (v_new ? 1 : 0)) * __popc(Lc.ph[k]) * L;
            const unsigned long long c0 = (prof && tid == 0) ? clock64() : 0;
            if (prof && tid == 0) { prof[3] += c0 - cq; prof[7] += 1; }     // lookup cycles, rounds
            if (PREC == 0 || pass == kF64)
                group_term64<false>(T, S, Lc.ph, n, L, G, c, k, st0, nst, both ? -1 : 1, v_old, v_new, O, gl, margin, &E, ei);
            else
                group_term32(T, S, Lc.ph, n, L, G, c, k, st0, nst, both ? -1 : 1, v_old, v_new, O, gl, mlo, mhi, &E, ei);
            if (prof && tid == 0) { cq = clock64(); prof[4] += cq - c0; }   // term cycles
        }
        __syncthreads();
        sub(1);
        if (tid < ne) {
            const IncWork &w = *Lc.ent(t0 + tid);
            const int sl = w.slot;
            const u128 d = limb_sum(E.d, tid), b = PREC == 1 ? limb_sum(E.b, tid) : (u128)0;
            const int n1 = E.n1[tid], n2 = E.n2[tid];
#pragma unroll
            for (int i = 0; i < kLimbs; ++i) {
                E.d[i][tid] = 0;
                if (PREC == 1) E.b[i][tid] = 0;
            }
            E.n1[tid] = E.n2[tid] = 0;
            const int at = Lc.at(sl);
            unsigned long long *a = Lc.acc + 2 * (size_t)at, *bp = Lc.bnd + 2 * (size_t)at;
            if (pass == kInitPart) {
                sadd128(a, a + 1, d);
                if (n1) atomicAdd(Lc.viol + at, n1);
                if (PREC == 1) {
                    sadd128(bp, bp + 1, b);
                    if (n2) atomicAdd(Lc.vmay + at, n2);
                }
            } else if (pass == kMerge) {
                u128 na, nb = 0;
                int nv, nm = 0;
                if (w.mode == 1) {
                    na = d;
                    nv = n1;
                    if (PREC == 1) { nb = b; nm = n2; }
                } else {
                    na = ld128(a) + d;
                    nv = Lc.viol[at] + n1;
                    if (PREC == 1) { nb = ld128(bp) + b; nm = Lc.vmay[at] + n2; }
                }
                st128(a, na);
                Lc.viol[at] = nv;
                if (PREC == 1) {
                    st128(bp, nb);
                    Lc.vmay[at] = nm;
                }
                set_rec<PREC>(R, sl, na, nb, nv, nm);
            } else {
                st128(I.vacc + 2 * (size_t)sl, d);
                I.vviol[sl] = n1;
            }
        }
        if (t0 + kTile < ne_all) __syncthreads();       // else the caller synchronises
        sub(2);
    }
    return terms;
}

// Clears the sums of a tile (the caller synchronises).
template <int NT>
__device__ __forceinline__ void clear_sums(EvalSmem &E) {
    for (int i = threadIdx.x; i < kLimbs * (kTile + 1); i += NT) {
        (&E.d[0][0])[i] = 0;
        (&E.b[0][0])[i] = 0;
    }
    for (int i = threadIdx.x; i < kTile; i += NT) E.n1[i] = E.n2[i] = 0;
}

// Rebuilds slot pair w from the clusters as the view shows them and appends
// a full work entry for each valid candidate.
template <int PREC>
__device__ void rebuild_pair(const Topo &T, const State &S, int n, int w, unsigned long long *list, const Rec &R,
                             const Loc &Lc, const View &V) {
    Cand c[2];
    const int x = slot_geometry(T, S, V, n, w, c[0], c[1]);
    R.span[w >> R.lg] = pair_span(n, c, x);
    for (int d = 0; d < 2; ++d) {
        const int sl = 2 * w + d, at = Lc.at(sl);
        Lc.slot[at] = c[d];
        if (c[d].s >= 0) {
            int2 seg[kIncMaxSeg];
            const int ns = full_segments(c[d], Lc.rank, seg, V.r);
            const unsigned long long o = append(list, ns, seg);
            write_entry(Lc.ent((int)(unsigned)o), sl, 1, (int)(o >> 32), ns, seg, c[d]);
            R.tkey[R.at(sl)] = (unsigned)c[d].key;
            R.touch(sl);
        } else {
            Lc.viol[at] = kIncDead;
            st128(Lc.acc + 2 * (size_t)at, 0);
            kill_rec<PREC>(R, sl);
        }
    }
}

}  // namespace

// Writes the new values of the merge O (npos positions) from its scratch into
// the state (the values the overlay gives: FP64 voltage, magnitude, MICE, s*'s
// merged extremes, and their FP32 copies), and zeroes r*'s MICE.  By the first
// nt threads of every CTA, from the last of them down.
__device__ __forceinline__ void write_back(const State &S, const Ovl &O, int npos, const uint8_t *ph, int n, int L,
                                           int G, int nt, int cr, int cs) {
    const int lgG = __ffs(G) - 1;
    const int rt = nt - 1 - (int)threadIdx.x;
    if (rt < 0) return;
    const int gl = rt & (G - 1), gi = rt >> lgG, NG = nt >> lgG, l = gl >> 2, p = gl & 3;
    for (int j = gi * cs + cr; j < npos; j += NG * cs) {
        const double *cb = O.cbuf + (size_t)j * kIncCbStride * L;
        const int k = *cb_bus(cb, L);
        if (k == O.r) continue;
        const bool fx = j >= O.nfree;
        if (l < L && p < 3 && (ph[k] >> p & 1u)) {
            const size_t ik = sidx(l, p, k, n);
            const float4 f = *cb_f4(cb, L, l, p);
            if (!fx) {
                S.vcur[ik] = make_double2(cb[(l * 3 + p) * 3 + 0], cb[(l * 3 + p) * 3 + 1]);
                S.mcur[ik] = cb[(l * 3 + p) * 3 + 2];
                S.v32[ik] = make_float2(f.x, f.y);
            }
            if (k == O.s) {
                const size_t ir = sidx(l, p, O.r, n);
                S.hi[ik] = fmax(S.hi[ik], S.hi[ir]);
                S.lo[ik] = fmin(S.lo[ik], S.lo[ir]);
            }
            S.hr32[ik] = f.z;
            S.lr32[ik] = f.w;
        }
        if (l < L && p == 0) {
            S.mice[(size_t)l * n + k] = cb[9 * L + l];
            S.mice32[(size_t)l * n + k] = *cb_mice32(cb, L, l);
        }
    }
    if (rt < L && cr == 0) {                // r's cluster is gone
        S.mice[(size_t)rt * n + O.r] = 0.0;
        S.mice32[(size_t)rt * n + O.r] = 0.0f;
    }
}

// ---------------------------------------------------------------- the search
// Bytes of the selection records of n slot pairs.
__host__ __device__ constexpr size_t rec_bytes(int n) { return (size_t)48 * n + 64; }
// ... and with the per-super-node largest MICE after them (shared memory only).
__host__ __device__ constexpr size_t rec_maxm_bytes(int n) { return rec_bytes(n) + (size_t)8 * n; }

// What a cluster's CTAs publish to each other: the minima of a pass of the
// selection, and with them the candidate that holds the CTA's own.
struct __align__(16) PubCand {
    Pub v;
    Cand c;
};
struct Pubs {
    Pub a[kMaxCluster], c[kMaxCluster];                 // by CTA: pass A, the rescored candidates' minimum
    PubCand b[kMaxCluster], d[kMaxCluster];             // pass B, the rescored candidates' tie band
};

// Shared memory of one CTA of a search: [work entries][two super-node lists]
// [phase masks][two overlay maps][super-node ranks][a cluster of one: block
// summaries of the selection records; of several: what its CTAs publish],
// then the records of the CTA's slot pairs when they fit, then (a cluster of
// several) their candidates and carried sums when they fit.
__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) / 16 * 16; }
// Blocks of 32 selection slots, and the bytes of their summaries.
__host__ __device__ constexpr int sel_blocks(int n) { return (2 * n + 31) / 32; }
__host__ __device__ constexpr size_t sel_bytes(int n) {
    return align16((size_t)16 * sel_blocks(n)) + align16((size_t)4 * sel_blocks(n)) +
           align16((size_t)8 * sel_blocks(n)) + align16((size_t)sel_blocks(n));
}
// Every region is rounded up to 16 bytes: the block summaries, the published
// values and the selection records are 16-byte keys.
__host__ __device__ constexpr size_t base_bytes(int n, int se, int cs) {
    return align16((size_t)se * sizeof(IncWork)) + align16((size_t)4 * n) + align16((size_t)n) +
           2 * align16((size_t)2 * n) + align16((size_t)2 * (n + 1)) + (cs == 1 ? sel_bytes(n) : sizeof(Pubs));
}
// The candidates (2 x 48 bytes a pair), sums (2 x 2 x 16) and counts (2 x 2 x 4) of n pairs.
__host__ __device__ constexpr size_t sums_bytes(int n) { return (size_t)176 * n; }
// Slot pairs of CTA cr of a cluster of cs, and how many the CTAs before it have.
__host__ __device__ constexpr int own_pairs(int n, int cr, int cs) { return (n - cr + cs - 1) / cs; }
__host__ __device__ constexpr int own_first(int n, int cr, int cs) {
    return cr * (n / cs) + (cr < n % cs ? cr : n % cs);
}

// rec_mode: where the selection records live (k_search_inc); + 4: the
// candidates and carried sums in shared memory too.  CS: CTAs of the search, a
// constant: one kernel for both kinds holds the code of both selections, and
// the instructions of a merge, executed once each, miss the instruction cache
// (16 % of the stalls): a batch's search was 3 to 7 % slower with CS a variable.
template <int NT, int PREC, int CS>
__device__ void inc_run(const Topo &T, const State &S, const Search &X, const Inc &I, Ctrl *C, bool verify,
                        unsigned char *dyn, int rec_mode, int se, int cw) {
    constexpr int cs = CS;
    static_assert(NT >= 128 && NT <= 512 && NT % 32 == 0, "thread count");
    __shared__ __align__(16) EvalSmem E;
    __shared__ __align__(16) Red sred[33];
    __shared__ Pub wpub[NT / 32];               // the warps' minima of a selection pass
    __shared__ int sscan[33];
    __shared__ unsigned long long s_sfx[2];     // SMICE of the committed state, fixed point
    __shared__ unsigned long long s_dsum[2];    // the last merge's change of it
    __shared__ unsigned long long s_app[2];     // work entries (append): the merge's; rescoring and verification
    const int n = T.n, L = T.L, tid = threadIdx.x;
    const int G = 4 * (L <= 1 ? 1 : (L <= 2 ? 2 : 4));
    const double margin = C->margin;
    const float mlo = __double2float_rd(margin), mhi = __double2float_ru(margin);
    const int max_merges = C->max_merges;
    const bool prof = C->profile != 0;
    const u128 tau_fx = to_fx(C->tau);
    long long tau_dn, tau_up;                   // in key units, rounded down and up
    {
        bool ok;
        tau_dn = key_val(key_floor(tau_fx, &ok));
        tau_up = key_val(key_ceil(tau_fx, &ok));
    }
    if (C->done || C->t >= max_merges) return;
    const int cr = cs == 1 ? 0 : cluster_rank(), lg = cs == 1 ? 0 : (cs == 2 ? 1 : (cs == 4 ? 2 : 3));
    const int np = own_pairs(n, cr, cs), pfirst = own_first(n, cr, cs);     // this CTA's slot pairs: w = cr, cr + cs, ...
    const bool own = (rec_mode & 4) != 0;
    rec_mode &= 3;
    // shared memory: entries, lists, phases; selection records: r0 or r1
    // (16 B a slot), tkey (4 B a slot), span (8 B a pair)
    Loc Lc;
    Lc.wsm = reinterpret_cast<IncWork *>(dyn);
    Lc.wgl = I.work + 2 * (size_t)pfirst;
    Lc.rlist = I.rlist + 2 * (size_t)pfirst;
    Lc.se = se;
    Lc.lst[0] = reinterpret_cast<unsigned short *>(dyn + align16((size_t)se * sizeof(IncWork)));
    Lc.lst[1] = Lc.lst[0] + n;
    uint8_t *phs = dyn + align16((size_t)se * sizeof(IncWork)) + align16((size_t)4 * n);
    Lc.ph = phs;
    unsigned short *map0 = reinterpret_cast<unsigned short *>(phs + align16((size_t)n)),
                   *map1 = map0 + align16((size_t)2 * n) / 2;
    // the super-node ranks live in shared memory during the search (copied back at the end)
    unsigned short *rank = map1 + align16((size_t)2 * n) / 2;
    Lc.rank = rank;
    unsigned char *aux = reinterpret_cast<unsigned char *>(rank) + align16((size_t)2 * (n + 1));
    Pubs *pub = reinterpret_cast<Pubs *>(aux);                                      // (a cluster of several)
    unsigned char *recmem = rec_mode ? dyn + base_bytes(n, se, cs) : I.recbuf;      // (rec_mode 0: a cluster of one)
    const int nrec = own_pairs(n, 0, cs);
    Rec R;
    R.lg = lg;
    R.r0 = reinterpret_cast<u128 *>(recmem);
    R.r1 = reinterpret_cast<ulonglong2 *>(recmem);
    R.tkey = reinterpret_cast<unsigned *>(recmem + (size_t)32 * nrec);
    R.span = reinterpret_cast<ushort4 *>(recmem + (size_t)40 * nrec);
    R.maxm = rec_mode == 2 ? reinterpret_cast<double *>(recmem + rec_bytes(nrec)) : I.maxm;
    R.bsum = nullptr;
    R.bcnt = nullptr;
    R.bmx = nullptr;
    R.dirty = nullptr;
    R.nb = 0;
    if (cs == 1) {
        unsigned char *sm = aux;
        R.nb = sel_blocks(n);
        R.bsum = sm;
        sm += align16((size_t)16 * R.nb);
        R.bcnt = reinterpret_cast<int *>(sm);
        sm += align16((size_t)4 * R.nb);
        R.bmx = reinterpret_cast<unsigned long long *>(sm);
        sm += align16((size_t)8 * R.nb);
        R.dirty = sm;
    }
    Lc.lg = -1;
    Lc.slot = X.slot;
    Lc.acc = I.acc;
    Lc.bnd = I.bnd;
    Lc.viol = I.viol;
    Lc.vmay = I.vmay;
    if (own) {
        unsigned char *sm = recmem + align16(rec_maxm_bytes(nrec));
        Lc.lg = lg;
        Lc.slot = reinterpret_cast<Cand *>(sm);
        Lc.acc = reinterpret_cast<unsigned long long *>(sm + (size_t)96 * nrec);
        Lc.bnd = Lc.acc + 4 * (size_t)nrec;
        Lc.viol = reinterpret_cast<int *>(Lc.bnd + 4 * (size_t)nrec);
        Lc.vmay = Lc.viol + 2 * (size_t)nrec;
    }
    Ovl O, P;                                   // the merge in progress; the one before it, until it is written back
    O.s = O.r = -1;
    O.nfree = 0;
    O.map = map0;
    O.cbuf = I.cbuf;
    P = O;
    int pnpos = 0;                              // positions of P
    int t = 0, ns = n;
    if (tid == 0) {
        s_sfx[0] = s_sfx[1] = 0ull;                 // every MICE starts at 0
    }
    unsigned long long tp = 0;
    auto stamp = [&](int i) {
        if (prof && tid == 0 && cr == 0) { const unsigned long long now = gtimer_inc(); C->phase_ns[i] += now - tp; tp = now; }
    };
    long long terms = 0, cands_run = 0;
    int rechecks = 0, recheck_cands = 0;

    // ---- the initial clusters (all singletons); the first evaluation of every
    // candidate ran on many CTAs (k_inc_init), its records in device memory
    for (int w = tid; w < n; w += NT) {
        Lc.lst[0][w] = (unsigned short)w;
        phs[w] = __ldg(T.ph + w);
        map0[w] = map1[w] = 0;
        rank[w] = (unsigned short)S.sn_rank[w];
    }
    if (tid == 0) rank[n] = (unsigned short)S.sn_rank[n];
    clear_sums<NT>(E);
    for (int j = tid; j < R.nb; j += NT) R.dirty[j] = 1;
    {
        const unsigned *tk = reinterpret_cast<const unsigned *>(I.recbuf + (size_t)32 * n);
        const ushort4 *sp = reinterpret_cast<const ushort4 *>(I.recbuf + (size_t)40 * n);
        for (int i = tid; i < np; i += NT) {
            const int w = i * cs + cr;
            R.maxm[i] = 0.0;
            if (rec_mode) R.span[i] = sp[w];
            for (int d = 0; d < 2; ++d) {
                // the live candidates' keys from their carried sums (the first
                // evaluation may have summed a candidate's terms on several CTAs)
                const int sl = 2 * w + d, v = I.viol[sl];
                if (rec_mode) R.tkey[2 * i + d] = tk[sl];
                if (v == kIncDead) {
                    if (rec_mode) kill_rec<PREC>(R, sl);
                    continue;
                }
                set_rec<PREC>(R, sl, ld128(I.acc + 2 * (size_t)sl), PREC == 1 ? ld128(I.bnd + 2 * (size_t)sl) : (u128)0,
                              v, PREC == 1 ? I.vmay[sl] : 0);
            }
            for (int d = 0; own && d < 2; ++d) {
                const int sl = 2 * w + d, at = 2 * i + d;
                Lc.slot[at] = X.slot[sl];
                st128(Lc.acc + 2 * (size_t)at, ld128(I.acc + 2 * (size_t)sl));
                st128(Lc.bnd + 2 * (size_t)at, ld128(I.bnd + 2 * (size_t)sl));
                Lc.viol[at] = I.viol[sl];
                Lc.vmay[at] = I.vmay[sl];
            }
        }
    }
    csync(cs);                              // (every CTA runs before the first one publishes to another)
    if (prof && tid == 0) tp = gtimer_inc();

    for (;;) {
        const unsigned short *list_old = Lc.lst[t & 1];
        unsigned short *list_new = Lc.lst[(t + 1) & 1];
        // ============================================================ selection
        // pass A: precision 0: the minimum over feasible candidates; precision 1:
        // the smallest lower end (m_lo) and the smallest upper end (m_hi); the
        // largest MICE after the last merge; the candidates.
        //   A cluster of one: the blocks whose records changed are summarised
        // again (one warp per block, one barrier), then every warp reduces the
        // summaries on its own.
        //   A cluster of several: every CTA reduces its own records (one or two a
        // thread) and publishes the result to every CTA; one cluster barrier, then
        // every warp of every CTA reduces what was published.
        if (tid == 0) s_app[0] = s_app[1] = 0ull;
        const int lane = tid & 31, wid = tid >> 5;
        constexpr int NW = NT / 32;
        Red ra;
        ra.a = ra.b = ra.c = kNone;
        ra.i = 0;
        {
            unsigned long long mx = 0;
            unsigned cnt = 0;
            u128 mn = kNone;
            unsigned long long lo = ~0ull, hi = ~0ull;
            if (cs == 1) {
                refresh_blocks<NT, PREC>(R, n);
                for (int j = lane; j < R.nb; j += 32) {
                    if (PREC == 0) {
                        mn = umin(mn, reinterpret_cast<const u128 *>(R.bsum)[j]);
                    } else {
                        const ulonglong2 b = reinterpret_cast<const ulonglong2 *>(R.bsum)[j];
                        lo = b.x < lo ? b.x : lo;
                        hi = b.y < hi ? b.y : hi;
                    }
                    cnt += (unsigned)R.bcnt[j];
                    mx = R.bmx[j] > mx ? R.bmx[j] : mx;
                }
            } else {
                for (int c = tid; c < 2 * np; c += NT) {
                    if (PREC == 0) {
                        mn = umin(mn, R.r0[c]);
                    } else {
                        const ulonglong2 q = R.r1[c];
                        lo = q.x < lo ? q.x : lo;
                        hi = q.y < hi ? q.y : hi;
                    }
                    cnt += R.tkey[c] != ~0u ? 1u : 0u;
                    if ((c & 1) == 0) {
                        const unsigned long long mb = (unsigned long long)__double_as_longlong(R.maxm[c >> 1]);
                        mx = mb > mx ? mb : mx;
                    }
                }
                // by warp, then by the first warp, then by every warp over the CTAs
                auto fold = [&]() {
                    Pub v;
                    if (PREC == 0) {
                        mn = warp_min128(mn);
                        v.a = (unsigned long long)mn;
                        v.b = (unsigned long long)(mn >> 64);
                    } else {
                        v.a = warp_min64(lo);
                        v.b = warp_min64(hi);
                    }
                    v.c = warp_max64(mx);
                    v.d = __reduce_add_sync(0xffffffffu, cnt);
                    return v;
                };
                auto take = [&](bool in, const Pub *src) {
                    mn = kNone;
                    lo = hi = ~0ull;
                    mx = 0;
                    cnt = 0;
                    if (in) {
                        const Pub v = *src;
                        mn = ((u128)v.b << 64) | (u128)v.a;
                        lo = v.a;
                        hi = v.b;
                        mx = v.c;
                        cnt = (unsigned)v.d;
                    }
                };
                const Pub v = fold();
                if (lane == 0) wpub[wid] = v;
                __syncthreads();
                if (wid == 0) {
                    take(lane < NW, wpub + lane);
                    const Pub u = fold();
                    if (lane < cs) publish(&pub->a[cr], lane, &u, 2);
                }
                csync(cs);
                take(lane < cs, pub->a + lane);
            }
            if (PREC == 0) {
                ra.a = warp_min128(mn);
            } else {
                lo = warp_min64(lo);
                hi = warp_min64(hi);
                ra.a = lo == kKeyNone ? kNone : (u128)lo;
                ra.b = hi == kKeyNone ? kNone : (u128)hi;
            }
            ra.i = (int)__reduce_add_sync(0xffffffffu, cnt);
            ra.c = ~(u128)warp_max64(mx);               // kNone when every maxm is 0
        }
        const int nvalid = ra.i;
        stamp(11);                                      // profile: block summaries and pass A
        if (tid == 0 && cr == 0 && t > 0)
            X.dec_maxerr[t - 1] = ra.c == kNone ? 0.0 : __longlong_as_double((long long)(unsigned long long)~ra.c);
        if (t >= max_merges) {
            if (tid == 0 && cr == 0) { C->done = 1; C->stop_reason = 0; }
            break;
        }
        Cand wc;                                         // the winner
        if (tid == 0 && cr == 0) {
            cands_run += nvalid;
            X.dec_ncand[t] = nvalid;
        }
        if (t < X.rec_iters) {
            const double s_cur = fx_to_d(ld128(s_sfx));
            // every candidate's SMICE (+inf when (surely) infeasible), compacted in slot order
            int base = 0;
            for (int c0 = 0; c0 < 2 * n; c0 += NT) {
                const int c = c0 + tid;
                const int v = c < 2 * n ? Lc.viol[c] : kIncDead;      // (recording runs one CTA, sums in device memory)
                const int f = v < kIncDead ? 1 : 0;
                int tot = 0;
                const int o = block_excl_scan<NT>(f, &tot, sscan) + base;
                if (f) {
                    const Cand &cc = Lc.slot[c];
                    const size_t at = (size_t)t * 2 * n + o;
                    X.rec_s[at] = T.orig[cc.s];
                    X.rec_r[at] = T.orig[cc.r];
                    X.rec_score[at] = v == 0 ? s_cur + fx_to_d(ld128(I.acc + 2 * (size_t)c)) : INFINITY;
                    X.rec_bound[at] = (PREC == 1 && v == 0) ? fx_to_d(ld128(I.bnd + 2 * (size_t)c)) * (1.0 + 1e-12) : 0.0;
                }
                base += tot;
            }
            if (tid == 0) X.rec_count[t] = nvalid;
        }
        if (ra.a == kNone) {                             // nothing (possibly) feasible
            if (tid == 0 && cr == 0) { C->done = 1; C->stop_reason = 1; }
            break;
        }
        // pass B: the smallest (tie key, slot) in the tie band and the smallest
        // key above it (precision 0); in precision 1, the smallest (tie key,
        // slot) surely in the band, the smallest tie key of a candidate the
        // screen cannot place, and the smallest lower end surely out of it.
        // Records in shared memory, at most kFlatSelectMax buses (or a cluster of
        // several CTAs): every record once, each thread a strided share of the
        // slots, then one block reduction (the cluster: published by warp, as in
        // pass A).  Otherwise only the blocks that may hold a candidate of the band are
        // read record by record (a block whose smallest key lies above the
        // band counts whole); with few such blocks every warp reads them all
        // and needs no barrier, with more they are spread over the warps.
        int ws = -1;
        double gap = INFINITY;
        const bool flat_b = cs > 1 || (rec_mode != 0 && n <= kFlatSelectMax);
        auto slot_of = [&](int c) { return ((((c >> 1) << lg) + cr) << 1) | (c & 1); };   // of the CTA's record c
        if (PREC == 0) {
            const u128 edge = (ra.a ^ kSignBit) + tau_fx, ek = okey(edge);
            u128 pa = kNone, pb = kNone;        // smallest (key, slot) in the band; smallest score above it
            if (flat_b) {
                for (int c = tid; c < 2 * np; c += NT) {
                    const u128 k = R.r0[c];
                    if (k == kNone) continue;
                    if (k <= ek) pa = umin(pa, ((u128)R.tkey[c] << 32) | (u128)(unsigned)slot_of(c));
                    else pb = umin(pb, k);
                }
                {
                    // (a tie key with its slot fits 64 bits)
                    unsigned long long qa = (unsigned long long)pa;
                    auto fold = [&]() {
                        Pub v;
                        v.a = qa = warp_min64(qa);
                        pb = warp_min128(pb);
                        v.b = 0;
                        v.c = (unsigned long long)pb;
                        v.d = (unsigned long long)(pb >> 64);
                        return v;
                    };
                    auto take = [&](bool in, const Pub *src) {
                        qa = ~0ull;
                        pb = kNone;
                        if (in) {
                            const Pub u = *src;
                            qa = u.a;
                            pb = ((u128)u.d << 64) | (u128)u.c;
                        }
                    };
                    const Pub v = fold();
                    if (lane == 0) wpub[wid] = v;
                    __syncthreads();
                    if (cs > 1) {
                        if (wid == 0) {
                            take(lane < NW, wpub + lane);
                            PubCand u;
                            u.v = fold();
                            u.c = Lc.slot[Lc.at(qa != ~0ull ? (int)(unsigned)qa : 2 * cr)];
                            if (lane < cs) publish(&pub->b[cr], lane, &u, 5);
                        }
                        csync(cs);
                        take(lane < cs, &pub->b[lane < cs ? lane : 0].v);
                        const unsigned long long q0 = qa;
                        fold();
                        wc = pub->b[__ffs(__ballot_sync(0xffffffffu, q0 == qa && lane < cs)) - 1].c;
                    } else {
                        take(lane < NW, wpub + lane);
                        fold();
                    }
                    pa = qa == ~0ull ? kNone : (u128)qa;
                }
            } else {
                const u128 *bs = reinterpret_cast<const u128 *>(R.bsum);
                auto relevant = [&](int j) {
                    const u128 bk = j < R.nb ? bs[j] : kNone;
                    return bk != kNone && bk <= ek;
                };
                int nrel = 0;
                for (int j0 = 0; j0 < R.nb; j0 += 32) {
                    const int j = j0 + lane;
                    const bool rel = relevant(j);
                    if (!rel && j < R.nb) pb = umin(pb, bs[j]);          // the whole block above the band
                    nrel += __popc(__ballot_sync(0xffffffffu, rel));
                }
                const bool few = nrel <= kFewBlocks;
                int kq = 0;
                for (int j0 = 0; j0 < R.nb; j0 += 32) {
                    unsigned mask = __ballot_sync(0xffffffffu, relevant(j0 + lane));
                    while (mask) {
                        const int b = __ffs(mask) - 1;
                        mask &= mask - 1;
                        if (few || kq % (NT / 32) == wid) {
                            const int c = 32 * (j0 + b) + lane;
                            if (c < 2 * n) {
                                const u128 k = R.r0[c];
                                if (k <= ek) pa = umin(pa, ((u128)R.tkey[c] << 32) | (u128)(unsigned)c);
                                else pb = umin(pb, k);
                            }
                        }
                        ++kq;
                    }
                }
                if (few) {
                    pa = warp_min128(pa);
                    pb = warp_min128(pb);
                } else {
                    Red rb;
                    rb.a = pa;
                    rb.b = pb;
                    rb.c = kNone;
                    rb.i = 0;
                    rb = block_red<NT>(rb, sred);
                    pa = rb.a;
                    pb = rb.b;
                }
            }
            ws = (int)(unsigned)(pa & 0xffffffffu);
            if (tid == 0 && pb != kNone) gap = fx_to_d((pb ^ kSignBit) - edge);
        } else {
            const bool has_hi = ra.b != kNone;
            const long long m_lo = key_val((unsigned long long)ra.a);
            const long long m_hi = has_hi ? key_val((unsigned long long)ra.b) : 0;
            const unsigned long long ein = val_key(m_lo + tau_dn);
            const unsigned long long eout = has_hi ? val_key(m_hi + tau_up) : kKeyNone;
            unsigned long long pa = ~0ull, pb = ~0ull, pc = ~0ull;
            if (flat_b) {
                for (int c = tid; c < 2 * np; c += NT) {
                    const ulonglong2 q = R.r1[c];
                    if (q.x == kKeyNone) continue;
                    const bool in_sure = q.y <= ein;
                    const bool out_sure = has_hi && q.x > eout;     // (never both: lo <= hi, m_lo <= m_hi)
                    if (in_sure) {
                        const unsigned long long kc = ((unsigned long long)R.tkey[c] << 32) | (unsigned)slot_of(c);
                        pa = kc < pa ? kc : pa;
                    } else if (!out_sure) {
                        const unsigned long long key = R.tkey[c];
                        pb = key < pb ? key : pb;
                    } else {
                        pc = q.x < pc ? q.x : pc;
                    }
                }
                {
                    auto fold = [&]() {
                        Pub v;
                        v.a = pa = warp_min64(pa);
                        v.b = pb = warp_min64(pb);
                        v.c = pc = warp_min64(pc);
                        v.d = 0;
                        return v;
                    };
                    auto take = [&](bool in, const Pub *src) {
                        pa = pb = pc = ~0ull;
                        if (in) {
                            const Pub u = *src;
                            pa = u.a;
                            pb = u.b;
                            pc = u.c;
                        }
                    };
                    const Pub v = fold();
                    if (lane == 0) wpub[wid] = v;
                    __syncthreads();
                    if (cs > 1) {
                        if (wid == 0) {
                            take(lane < NW, wpub + lane);
                            PubCand u;
                            u.v = fold();
                            u.c = Lc.slot[Lc.at(pa != ~0ull ? (int)(unsigned)pa : 2 * cr)];
                            if (lane < cs) publish(&pub->b[cr], lane, &u, 5);
                        }
                        csync(cs);
                        take(lane < cs, &pub->b[lane < cs ? lane : 0].v);
                        const unsigned long long p0 = pa;
                        fold();
                        wc = pub->b[__ffs(__ballot_sync(0xffffffffu, p0 == pa && lane < cs)) - 1].c;
                    } else {
                        take(lane < NW, wpub + lane);
                        fold();
                    }
                }
            } else {
                const ulonglong2 *bs = reinterpret_cast<const ulonglong2 *>(R.bsum);
                // a block is read record by record unless every candidate in it is
                // surely out of the band (its smallest lower end above eout)
                auto relevant = [&](int j) {
                    const unsigned long long bl = j < R.nb ? bs[j].x : kKeyNone;
                    return bl != kKeyNone && !(has_hi && bl > eout);
                };
                int nrel = 0;
                for (int j0 = 0; j0 < R.nb; j0 += 32) {
                    const int j = j0 + lane;
                    const bool rel = relevant(j);
                    const unsigned long long bl = j < R.nb ? bs[j].x : kKeyNone;
                    if (bl != kKeyNone && !rel) pc = bl < pc ? bl : pc;        // the whole block surely out
                    nrel += __popc(__ballot_sync(0xffffffffu, rel));
                }
                const bool few = nrel <= kFewBlocks;
                int kq = 0;
                for (int j0 = 0; j0 < R.nb; j0 += 32) {
                    unsigned mask = __ballot_sync(0xffffffffu, relevant(j0 + lane));
                    while (mask) {
                        const int b = __ffs(mask) - 1;
                        mask &= mask - 1;
                        if (few || kq % (NT / 32) == wid) {
                            const int c = 32 * (j0 + b) + lane;
                            if (c < 2 * n) {
                                const ulonglong2 q = R.r1[c];
                                if (q.x != kKeyNone) {
                                    const bool in_sure = q.y <= ein;
                                    const bool out_sure = has_hi && q.x > eout;
                                    const unsigned key = R.tkey[c];
                                    if (in_sure) {
                                        const unsigned long long kc = ((unsigned long long)key << 32) | (unsigned)c;
                                        pa = kc < pa ? kc : pa;
                                    } else if (!out_sure) {
                                        pb = key < pb ? key : pb;
                                    }
                                    if (out_sure) pc = q.x < pc ? q.x : pc;
                                }
                            }
                        }
                        ++kq;
                    }
                }
                pa = warp_min64(pa);
                pb = warp_min64(pb);
                pc = warp_min64(pc);
                if (!few) {
                    if (lane == 0) {
                        Pub v;
                        v.a = pa;
                        v.b = pb;
                        v.c = pc;
                        v.d = 0;
                        wpub[wid] = v;
                    }
                    __syncthreads();
                    const Pub u = wpub[lane < NW ? lane : 0];
                    pa = warp_min64(u.a);
                    pb = warp_min64(u.b);
                    pc = warp_min64(u.c);
                }
            }
            Red rb;
            rb.a = pa == ~0ull ? kNone : (u128)pa;
            rb.b = pb == ~0ull ? kNone : (u128)pb;
            rb.c = pc == ~0ull ? kNone : (u128)pc;
            rb.i = 0;
            const u128 ks = rb.a == kNone ? kNone : (rb.a >> 32);
            if (!(rb.b < ks)) {                          // no uncertain candidate can take the band's smallest key
                ws = (int)(unsigned)(rb.a & 0xffffffffu);
                if (tid == 0 && rb.c != kNone) gap = (double)(key_val((unsigned long long)rb.c) - key_val(eout)) * 0x1p-56;
            } else {
                // FP64 rescoring of R: the possible minimizers and the uncertain
                // candidates with a key below the smallest surely-in key
                const unsigned long long mh = has_hi ? (unsigned long long)ra.b : kKeyNone;
                for (int c = tid; c < 2 * np; c += NT) {
                    const ulonglong2 q = R.r1[c];
                    if (q.x == kKeyNone) continue;
                    const bool in_sure = q.y <= ein;
                    const bool out_sure = has_hi && q.x > eout;
                    const bool unc = !in_sure && !out_sure && (u128)R.tkey[c] < ks;
                    if (unc || q.x <= mh) {
                        const int sl = slot_of(c);
                        const Cand cc = Lc.slot[Lc.at(sl)];
                        int2 seg[kIncMaxSeg];
                        const int k = full_segments(cc, rank, seg);
                        const unsigned long long o = append(&s_app[1], k, seg);
                        Lc.rlist[(int)(unsigned)o] = sl;
                        write_entry(Lc.ent((int)(unsigned)o), sl, 1, (int)(o >> 32), k, seg, cc);
                    }
                }
                __syncthreads();
                const int nR = (int)(unsigned)s_app[1];
                terms += run_entries<NT, PREC>(T, S, I, n, L, G, margin, mlo, mhi, nR, (int)(s_app[1] >> 32), kF64,
                                               list_old, list_old, -1, P, E, R, Lc);
                __syncthreads();
                // exact selection over every CTA's R, with the surely-in candidate of key ks
                Red rc;
                rc.a = rc.b = rc.c = kNone;
                rc.i = 0;
                for (int i = tid; i < nR; i += NT) {
                    const int c = Lc.rlist[i];
                    if (I.vviol[c] == 0) rc.a = umin(rc.a, okey(ld128(I.vacc + 2 * (size_t)c)));
                }
                rc = block_red<NT>(rc, sred);
                int nR_all = nR;
                if (cs > 1) {
                    Pub v;
                    v.a = (unsigned long long)rc.a;
                    v.b = (unsigned long long)(rc.a >> 64);
                    v.c = (unsigned long long)nR;
                    v.d = 0;
                    if (tid < cs) publish(&pub->c[cr], tid, &v, 2);
                    csync(cs);
                    rc.a = kNone;
                    nR_all = 0;
                    for (int j = 0; j < cs; ++j) {
                        rc.a = umin(rc.a, ((u128)pub->c[j].b << 64) | (u128)pub->c[j].a);
                        nR_all += (int)pub->c[j].c;
                    }
                }
                Red rd;
                rd.a = rd.b = rd.c = kNone;
                rd.i = 0;
                if (rc.a != kNone) {
                    const u128 edge = (rc.a ^ kSignBit) + tau_fx, ek = okey(edge);
                    for (int i = tid; i < nR; i += NT) {
                        const int c = Lc.rlist[i];
                        if (I.vviol[c] != 0) continue;
                        const u128 k = okey(ld128(I.vacc + 2 * (size_t)c));
                        if (k <= ek) rd.a = umin(rd.a, ((u128)R.tkey[R.at(c)] << 32) | (u128)(unsigned)c);
                        else rd.b = umin(rd.b, k);
                    }
                    rd = block_red<NT>(rd, sred);
                    if (cs > 1) {
                        PubCand v;                  // (a tie key with its slot fits 64 bits; none: ~0)
                        v.v.a = (unsigned long long)rd.a;
                        v.v.b = (unsigned long long)rd.b;
                        v.v.c = (unsigned long long)(rd.b >> 64);
                        v.v.d = 0;
                        v.c = Lc.slot[Lc.at(rd.a != kNone ? (int)(unsigned)rd.a : 2 * cr)];
                        if (tid < cs) publish(&pub->d[cr], tid, &v, 5);
                        csync(cs);
                        rd.a = rd.b = kNone;
                        for (int j = 0; j < cs; ++j) {
                            const Pub u = pub->d[j].v;
                            if (u.a != ~0ull && (u128)u.a < rd.a) {
                                rd.a = (u128)u.a;
                                if (rd.a < rb.a) wc = pub->d[j].c;
                            }
                            rd.b = umin(rd.b, ((u128)u.c << 64) | (u128)u.b);
                        }
                    }
                    if (tid == 0 && rd.b != kNone) gap = fx_to_d((rd.b ^ kSignBit) - edge);
                }
                const u128 best = umin(rd.a, rb.a);
                ws = best == kNone ? -1 : (int)(unsigned)(best & 0xffffffffu);
                ++rechecks;
                recheck_cands += nR_all;
            }
        }
        if (ws < 0) {                                    // FP64 rescoring found nothing feasible
            if (tid == 0 && cr == 0) { C->done = 1; C->stop_reason = 1; }
            break;
        }
        stamp(0);
        // ============================================================ the merge
        // The winner's record: every thread builds its own at once, so no warp
        // waits for another's copy.
        const int CW = cw;                  // warps that evaluate the merge (1 .. NW - 1)
        const bool commit_warp = wid >= NW - CW;
        if (cs == 1) {
            wc = Lc.slot[Lc.at(ws)];
            __syncthreads();                // (the rebuilt pairs below may write the winner's slot)
        }
        const Win hw = make_win(wc, ws, rank);
        if (tid == 0) {
            if (cr == 0) X.dec_gap[t] = gap;
            s_dsum[0] = 0ull;
            s_dsum[1] = 0ull;
        }
        stamp(12);                                      // profile: the winner's record
        const int n1 = hw.q1hi - hw.q1lo, n2 = hw.q2hi - hw.q2lo;
        O.map = t & 1 ? map1 : map0;
        O.cbuf = I.cbuf + (t & 1 ? (size_t)n * kIncCbStride * L : 0);
        O.s = hw.s;
        O.r = hw.r;
        O.nfree = n1 + n2;
        // One step, nothing in it waiting for anything else in it:
        //   - the last warps of every CTA evaluate the merge's own FP64 values
        // into its scratch (the state under the overlay of the merge before, P);
        //   - the others write P back, map the merge's positions, find the
        // candidates that change among the CTA's own (their terms are listed in
        // any order: the sums are exact), rebuild the pairs next to s* and r*
        // through the merge's view of the clusters, and do the merge's
        // bookkeeping (clusters, super-node list, s*'s injection).
        if (commit_warp) {
            Commit cm;
            cm.h = &hw;
            cm.wc = wc;
            cm.list = list_old;
            cm.ph = Lc.ph;
            cm.O = P;
            cm.cbuf = const_cast<double *>(O.cbuf);
            terms += commit_groups(T, S, n, L, G, margin, cm, NW - CW, CW, cr, cs);
        } else {
            const int nsc = (NW - CW) * 32;
            View V;
            V.s = hw.s;
            V.r = hw.r;
            V.dir = hw.dir;
            // the changed buses lie in [hl, hh): a candidate whose span misses it is unchanged
            int hl = min(hw.s, hw.r), hh = max(hw.s, hw.r) + 1;
            if (hw.w1lo < hw.w1hi) { hl = min(hl, hw.w1lo); hh = max(hh, hw.w1hi); }
            if (hw.w2lo < hw.w2hi) { hl = min(hl, hw.w2lo); hh = max(hh, hw.w2hi); }
            for (int i = tid; i < np; i += nsc) {
                const ushort4 sp = R.span[i];
                const int w = (i << lg) + cr;
                if (w == hw.r) {                        // r's cluster is gone
                    R.maxm[i] = 0.0;
                    R.touch_sn(w);
                    R.span[i] = make_ushort4(0, 0, 0xffff, 0);
                    for (int d = 0; d < 2; ++d) {
                        Lc.slot[Lc.at(2 * w + d)].s = -1;
                        Lc.viol[Lc.at(2 * w + d)] = kIncDead;
                        kill_rec<PREC>(R, 2 * w + d);
                    }
                    continue;
                }
                if (sp.w == 0) continue;
                const int qp = sp.z == 0xffff ? -1 : (int)sp.z;
                if (w == hw.s || qp == hw.r || qp == hw.s) {
                    rebuild_pair<PREC>(T, S, n, w, &s_app[0], R, Lc, V);
                    continue;
                }
                if ((int)sp.y <= hl || (int)sp.x >= hh) continue;
                for (int d = 0; d < 2; ++d) {
                    const Cand c = Lc.slot[Lc.at(2 * w + d)];
                    if (c.s < 0 || !touched(c, hw)) continue;
                    int2 seg[kIncMaxSeg];
                    const int k = changed_segments(c, hw, rank, seg);
                    const unsigned long long o = append(&s_app[0], k, seg);
                    write_entry(Lc.ent((int)(unsigned)o), 2 * w + d, 0, (int)(o >> 32), k, seg, c);
                }
            }
            if (pnpos > 0) write_back(S, P, pnpos, Lc.ph, n, L, G, nsc, cr, cs);
            unsigned short *map = t & 1 ? map1 : map0;
            for (int q = tid; q < hw.npos; q += nsc) {      // the terms after the merge read k's new values here
                const int k = q < n1 ? list_old[hw.q1lo + q] : (q < O.nfree ? list_old[hw.q2lo + q - n1] : hw.s);
                if (k != hw.r) map[k] = (unsigned short)(q + 1);
            }
            // r's members join s (they lie in the subtree of r's top; a rebuilt pair
            // reads either value the same); the new super-node list
            const int rtop = S.top[hw.r], rtop_end = rtop + T.sz[rtop];
            for (int b = rtop + tid * cs + cr; b < rtop_end; b += nsc * cs)
                if (S.label[b] == hw.r) S.label[b] = hw.s;
            for (int j = tid; j < ns - 1; j += nsc) list_new[j] = list_old[j + (j >= hw.jr ? 1 : 0)];
            // s takes r's injection (no term before the merge reads s's injection:
            // every candidate with r = s* is rebuilt; the merge's own evaluation
            // reads r's)
            if (tid < 3 * L && cr == 0 && (Lc.ph[hw.r] >> (tid % 3) & 1u)) {
                const size_t is = sidx(tid / 3, tid % 3, hw.s, n), ir = sidx(tid / 3, tid % 3, hw.r, n);
                const double2 ni = cadd(S.icur[is], S.icur[ir]);
                S.icur[is] = ni;
                S.icur32[is] = make_float2((float)ni.x, (float)ni.y);
            }
            if (tid == 0 && cr == 0) {
                if (hw.dir == 1) {                      // (read through the view: r's)
                    S.top[hw.s] = S.top[hw.r];
                    S.ptop[hw.s] = S.ptop[hw.r];
                }
                X.dec_s[t] = T.orig[hw.s];
                X.dec_r[t] = T.orig[hw.r];
            }
        }
        csync(cs);
        ns -= 1;
        const int ne = (int)(unsigned)s_app[0], items = (int)(s_app[0] >> 32);
        stamp(1);
        // ============================================================ the terms that change, and the score
        {
            // the merge's exact score change (its FP64 terms in fixed point) and
            // each position's largest MICE, one lane per (position, scenario), from
            // the last thread down; P's map is cleared (its values are in the state)
            const int lgG = __ffs(G) - 1, rt = NT - 1 - tid;
            const int gl = rt & (G - 1), gi = rt >> lgG, NG = NT >> lgG, l = gl >> 2, p = gl & 3;
            u128 dsum = 0;
            for (int r0 = 0; r0 < hw.npos; r0 += NG) {
                if (r0 + ((rt >> 5) << (5 - lgG)) >= hw.npos) break;
                const int j = r0 + gi;
                bool valid = j < hw.npos;
                int k = hw.s;
                if (valid) {
                    k = j < n1 ? list_old[hw.q1lo + j] : (j < n1 + n2 ? list_old[hw.q2lo + j - n1] : hw.s);
                    valid = k != hw.r;
                }
                const bool mine = valid && (k & (cs - 1)) == cr;
                unsigned long long mb = 0;                  // MICE >= 0: bit patterns order like values
                if (valid && l < L && p == 0 && (mine || cr == 0)) {
                    const double m = O.cbuf[(size_t)j * kIncCbStride * L + 9 * L + l];
                    mb = (unsigned long long)__double_as_longlong(m);
                    if (cr == 0) {
                        double dd = m - S.mice[(size_t)l * n + k];
                        if (k == hw.s) dd -= S.mice[(size_t)l * n + hw.r];
                        dsum += to_fx(dd);
                    }
                }
                for (int o = 4; o < G; o <<= 1) {
                    const unsigned long long y = __shfl_xor_sync(0xffffffffu, mb, o);
                    mb = y > mb ? y : mb;
                }
                if (mine && gl == 0) {
                    R.maxm[k >> lg] = __longlong_as_double((long long)mb);
                    R.touch_sn(k);
                }
            }
            if (dsum != 0) sadd128(&s_dsum[0], &s_dsum[1], dsum);
            unsigned short *pmap = t & 1 ? map0 : map1;
            for (int j = rt; j < pnpos; j += NT) pmap[*cb_bus(P.cbuf + (size_t)j * kIncCbStride * L, L)] = 0;
        }
        terms += run_entries<NT, PREC>(T, S, I, n, L, G, margin, mlo, mhi, ne, items, kMerge, list_old, list_new, hw.r,
                                       O, E, R, Lc, prof && cr == 0 ? C->phase_ns + 6 : nullptr);
        for (int b = hw.r + 1 + tid; b <= n; b += NT) rank[b] -= 1;     // ranks past r* drop by one
        __syncthreads();
        stamp(3);
        if (tid == 0 && cr == 0) {
            const u128 sfx = ld128(s_sfx) + ld128(s_dsum);
            st128(s_sfx, sfx);
            X.dec_score[t] = fx_to_d(sfx);
        }
        P = O;
        pnpos = hw.npos;
        t += 1;
        if (verify) {
            // every candidate again from scratch, on the state with the merge
            // written back; the carried values must match bit for bit
            if (tid == 0) s_app[1] = 0ull;
            csync(cs);
            write_back(S, P, pnpos, Lc.ph, n, L, G, NT, cr, cs);
            unsigned short *pmap = t & 1 ? map0 : map1;
            for (int j = tid; j < pnpos; j += NT) pmap[*cb_bus(P.cbuf + (size_t)j * kIncCbStride * L, L)] = 0;
            pnpos = 0;
            csync(cs);
            for (int i = tid; i < 2 * np; i += NT) {
                const int c = slot_of(i);
                const Cand cc = Lc.slot[Lc.at(c)];
                if (cc.s < 0) continue;
                int2 seg[kIncMaxSeg];
                const int k = full_segments(cc, rank, seg);
                const unsigned long long o = append(&s_app[1], k, seg);
                write_entry(Lc.ent((int)(unsigned)o), c, 1, (int)(o >> 32), k, seg, cc);
            }
            __syncthreads();
            run_entries<NT, PREC>(T, S, I, n, L, G, margin, mlo, mhi, (int)(unsigned)s_app[1], (int)(s_app[1] >> 32),
                                  kFresh, list_new, list_new, -1, P, E, R, Lc);
            __syncthreads();
            int bad = 0;
            for (int i = tid; i < 2 * np; i += NT) {
                const int c = slot_of(i), at = Lc.at(c);
                if (Lc.slot[at].s < 0) continue;
                if (Lc.viol[at] != I.vviol[c] || ld128(Lc.acc + 2 * (size_t)at) != ld128(I.vacc + 2 * (size_t)c)) ++bad;
            }
            Red rv;
            rv.a = rv.b = rv.c = kNone;
            rv.i = bad;
            rv = block_red<NT>(rv, sred);
            if (tid == 0 && rv.i) atomicAdd(&C->inc_mismatch, rv.i);
        }
    }
    // the last merge into the state (every CTA is past its terms: the selection's barrier)
    if (pnpos > 0) write_back(S, P, pnpos, Lc.ph, n, L, G, NT, cr, cs);
    if (prof) {                                     // (phase-node, scenario) items evaluated over the run
        unsigned long long tt = (unsigned long long)terms;
        for (int o = 16; o > 0; o >>= 1) tt += __shfl_xor_sync(0xffffffffu, tt, o);
        if ((tid & 31) == 0) atomicAdd(reinterpret_cast<unsigned long long *>(&C->sweep_ns), tt);
    }
    if (cr != 0) return;
    for (int b = tid; b <= n; b += NT) S.sn_rank[b] = rank[b];
    if (tid == 0) {
        C->t = t;
        C->n_super = ns;
        C->candidates += cands_run;
        C->iters += t + (C->stop_reason == 1 ? 1 : 0);
        C->s_cur = fx_to_d(ld128(s_sfx));
        C->rechecks = rechecks;
        C->recheck_cands = recheck_cands;
    }
}

namespace {

// Per-merge data in dynamic shared memory; rec_mode 0: the selection records
// in I.recbuf; 1: in shared memory; 2: in shared memory, with the largest MICE
// per super-node.  se: work entries in shared memory; cw: warps that evaluate
// the merge beside the changed-set scan.
template <int NT, int PREC, int CS>
__global__ void __launch_bounds__(NT, 1) k_search_inc(Topo T, State S, Search X, Inc I, Ctrl *C, int verify,
                                                      int rec_mode, int se, int cw) {
    extern __shared__ __align__(16) unsigned char inc_dyn[];
    if (X.setup_err && *X.setup_err != 0) return;           // the setup failed: no result (C->done stays 0)
    inc_run<NT, PREC, CS>(T, S, X, I, C, verify != 0, inc_dyn, rec_mode, se, cw);
}

// The first evaluation of every candidate (every slot pair from the initial
// clusters, all singletons, every term), which needs no merge before it: its
// work is spread over many CTAs instead of the search's one to eight.  The
// CTAs write the candidates, carried sums and tie keys to device memory, in
// the layout the search reads (it copies its records into shared memory and
// derives the selection keys from the sums).  The
// terms are evaluated by the same code as in the search, so the carried sums
// are the ones the search's own first evaluation gives.
constexpr int kInitPairs = kIncInitPairs;
constexpr int kInitCtasMax = kIncInitCtasMax;
// The first evaluation of one feeder with its work spread evenly over the
// grid.  A pair's candidates can hold up to n positions each (the pairs next
// to the root), so splitting by pairs leaves one CTA with most of the work.
// Instead every CTA derives the position count of every initial candidate
// (the geometry of a pair of singletons is a few loads), lays the candidates'
// positions end to end in slot order, and takes an equal share of them; a
// candidate cut by a share's ends is summed in parts, added to the carried
// sums with 128-bit atomics (integer sums: exact in any order; the sums start
// at zero).  Each pair's own outputs (the slots, its span, the tie keys and
// the dead slots' records) are written by one CTA, and the search derives
// the live candidates' selection keys from the finished sums.
// Dynamic shared memory: the identity super-node list (2n bytes) and the
// position count of every slot (8n bytes).
// CTA b of the B CTAs that evaluate one feeder (dyn: dynamic shared memory of
// 2n + 8n bytes, 16-byte aligned parts).
template <int NT, int PREC>
__device__ void inc_init_share(const Topo &T, const State &S, const Search &X, const Inc &I, Ctrl *C, int b, int B,
                               unsigned char *dyn, EvalSmem &E, int *sscan, int &s_first, unsigned long long &s_app) {
    const int n = T.n, L = T.L, tid = threadIdx.x;
    const int G = 4 * (L <= 1 ? 1 : (L <= 2 ? 2 : 4));
    const double margin = C->margin;
    const float mlo = __double2float_rd(margin), mhi = __double2float_ru(margin);
    unsigned short *list = reinterpret_cast<unsigned short *>(dyn);
    int *pcnt = reinterpret_cast<int *>(dyn + align16((size_t)2 * n));
    for (int w = tid; w < n; w += NT) list[w] = (unsigned short)w;
    Loc Lc;
    Lc.wsm = nullptr;
    Lc.wgl = I.work;
    Lc.rlist = nullptr;
    Lc.se = 0;
    Lc.lst[0] = Lc.lst[1] = list;
    Lc.ph = T.ph;
    Lc.rank = nullptr;                          // (the ranks are read from S.sn_rank)
    Lc.lg = -1;
    Lc.slot = X.slot;
    Lc.acc = I.acc;
    Lc.bnd = I.bnd;
    Lc.viol = I.viol;
    Lc.vmay = I.vmay;
    Rec R;
    R.lg = 0;
    R.r0 = reinterpret_cast<u128 *>(I.recbuf);
    R.r1 = reinterpret_cast<ulonglong2 *>(I.recbuf);
    R.tkey = reinterpret_cast<unsigned *>(I.recbuf + (size_t)32 * n);
    R.maxm = I.maxm;
    R.span = reinterpret_cast<ushort4 *>(I.recbuf + (size_t)40 * n);
    R.bsum = nullptr;
    R.bcnt = nullptr;
    R.bmx = nullptr;
    R.dirty = nullptr;
    R.nb = 0;
    Ovl O;
    O.map = nullptr;                            // (the first evaluation reads the stored state only)
    O.cbuf = I.cbuf;
    O.s = O.r = -1;
    O.nfree = 0;
    const View V = no_view();
    // this CTA's pairs: the slots, the span, the tie keys, the dead slots
    for (int w = b + B * tid; w < n; w += B * NT) {
        Cand c[2];
        const int x = slot_geometry(T, S, V, n, w, c[0], c[1]);
        R.span[w] = pair_span(n, c, x);
        for (int d = 0; d < 2; ++d) {
            const int sl = 2 * w + d;
            X.slot[sl] = c[d];
            if (c[d].s >= 0) {
                R.tkey[sl] = (unsigned)c[d].key;
            } else {
                I.viol[sl] = kIncDead;
                kill_rec<PREC>(R, sl);
            }
        }
    }
    // every slot's position count; thread tid takes the pairs [p0, p1)
    const int per = (n + NT - 1) / NT, p0 = min(n, tid * per), p1 = min(n, p0 + per);
    int mine = 0;
    for (int w = p0; w < p1; ++w) {
        Cand c[2];
        slot_geometry(T, S, V, n, w, c[0], c[1]);
        for (int d = 0; d < 2; ++d) {
            int k = 0;
            if (c[d].s >= 0) {
                int2 seg[kIncMaxSeg];
                const int ns = full_segments(c[d], S.sn_rank, seg);
                for (int i = 0; i < ns; ++i) k += seg[i].y - seg[i].x;
            }
            pcnt[2 * w + d] = k;
            mine += k;
        }
    }
    if (tid == 0) { s_first = 2 * n; s_app = 0ull; }
    clear_sums<NT>(E);
    int tot = 0;
    const int base = block_excl_scan<NT>(mine, &tot, sscan);
    // this CTA's share of the positions: [q0, q1)
    const int share = max(1, (tot + B - 1) / B);
    const int q0 = min(tot, b * share), q1 = min(tot, q0 + share);
    {
        int off = base;
        for (int sl = 2 * p0; sl < 2 * p1; ++sl) {
            const int k = pcnt[sl];
            if (k > 0 && off < q1 && off + k > q0) atomicMin(&s_first, sl);
            off += k;
        }
    }
    __syncthreads();
    // the entries: one per candidate that meets the share, its segments cut to
    // the share, at [first slot + b, ...) (the CTAs' ranges do not overlap)
    {
        Lc.wgl = I.work + (s_first + b);
        int off = base;
        for (int sl = 2 * p0; sl < 2 * p1; ++sl) {
            const int k = pcnt[sl];
            if (k > 0 && off < q1 && off + k > q0) {
                Cand c[2];
                slot_geometry(T, S, V, n, sl >> 1, c[0], c[1]);
                const Cand &cc = c[sl & 1];
                int2 seg[kIncMaxSeg], cut[kIncMaxSeg];
                const int ns = full_segments(cc, S.sn_rank, seg);
                const int lo = max(q0 - off, 0), hi = min(q1 - off, k);    // the share, in the candidate's positions
                int nc = 0, at = 0;
                for (int i = 0; i < ns; ++i) {
                    const int len = seg[i].y - seg[i].x;
                    const int a = max(lo, at), z = min(hi, at + len);
                    if (a < z) cut[nc++] = make_int2(seg[i].x + (a - at), seg[i].x + (z - at));
                    at += len;
                }
                const unsigned long long o = append(&s_app, nc, cut);
                write_entry(Lc.ent((int)(unsigned)o), sl, 1, (int)(o >> 32), nc, cut, cc);
            }
            off += k;
        }
    }
    __syncthreads();
    if (s_app == 0ull) return;
    const long long terms = run_entries<NT, PREC>(T, S, I, n, L, G, margin, mlo, mhi, (int)(unsigned)s_app,
                                                  (int)(s_app >> 32), kInitPart, list, list, -1, O, E, R, Lc);
    if (C->profile) {                           // (phase-node, scenario) items
        unsigned long long tt = (unsigned long long)terms;
        for (int o = 16; o > 0; o >>= 1) tt += __shfl_xor_sync(0xffffffffu, tt, o);
        if ((tid & 31) == 0 && tt) atomicAdd(reinterpret_cast<unsigned long long *>(&C->sweep_ns), tt);
    }
}

template <int NT, int PREC>
__global__ void __launch_bounds__(NT) k_inc_init(Topo T, State S, Search X, Inc I, Ctrl *C) {
    extern __shared__ __align__(16) unsigned char init_dyn[];
    __shared__ __align__(16) EvalSmem E;
    __shared__ int sscan[33];
    __shared__ int s_first;
    __shared__ unsigned long long s_app;
    if (X.setup_err && *X.setup_err != 0) return;
    inc_init_share<NT, PREC>(T, S, X, I, C, blockIdx.x, gridDim.x, init_dyn, E, sscan, s_first, s_app);
}

// The same for many feeders: cta_off[i] = the first CTA of the i-th feeder of
// the order (the feeder's CTAs end where the next feeder's begin, the last
// feeder's at the end of the grid); each feeder's CTAs split its positions
// as above.  Feeders whose setup failed are skipped.  The carried sums of
// every feeder start at zero (k_inc_zero_batch).
template <int NT, int PREC>
__global__ void __launch_bounds__(NT) k_inc_init_batch(const BatchFeeder *fd, const int *order, const int *cta_off,
                                                       int nf, int cta0) {
    extern __shared__ __align__(16) unsigned char init_dyn[];
    __shared__ __align__(16) EvalSmem E;
    __shared__ int sscan[33];
    __shared__ int s_first;
    __shared__ unsigned long long s_app;
    __shared__ Topo sT;
    __shared__ State sS;
    __shared__ Search sX;
    __shared__ Inc sI;
    __shared__ int s_f, s_b, s_B;
    const int b = blockIdx.x + cta0;             // (cta0: the first CTA of the launch's first feeder)
    if (threadIdx.x == 0) {
        int lo = 0, hi = nf - 1;                 // the last feeder whose first CTA is <= b
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (cta_off[mid] <= b) lo = mid;
            else hi = mid - 1;
        }
        const int f = order[lo];
        s_f = f;
        s_b = b - cta_off[lo];
        s_B = (lo + 1 < nf ? cta_off[lo + 1] : (int)gridDim.x + cta0) - cta_off[lo];
        sT = fd[f].T;
        sS = fd[f].S;
        sX = fd[f].X;
        sI = fd[f].I;
    }
    __syncthreads();
    const int f = s_f;
    if (*fd[f].setup_err != 0 || s_b >= s_B) return;
    inc_init_share<NT, PREC>(sT, sS, sX, sI, fd[f].C, s_b, s_B, init_dyn, E, sscan, s_first, s_app);
}

// The carried sums, violation counts and their bounds of every feeder of the
// order set to zero before its first evaluation adds to them (one CTA per
// feeder).
static __global__ void k_inc_zero_batch(const BatchFeeder *fd, const int *order, int nf) {
    const int q = blockIdx.x;
    if (q >= nf) return;
    const Inc &I = fd[order[q]].I;
    const int n = fd[order[q]].T.n;
    unsigned char *p0 = reinterpret_cast<unsigned char *>(I.acc);
    const size_t bytes = reinterpret_cast<const unsigned char *>(I.vmay + 2 * (size_t)n) - p0;
    for (size_t i = threadIdx.x; i < bytes / 4; i += blockDim.x) reinterpret_cast<unsigned *>(p0)[i] = 0u;
}

// One CTA or cluster (of CS CTAs) per feeder, feeders in the order given (largest first).
template <int NT, int PREC, int CS>
__global__ void __launch_bounds__(NT) k_search_inc_batch(const BatchFeeder *fd, const int *order, int nf,
                                                         int rec_mode, int se, int cw) {
    constexpr int cs = CS;
    extern __shared__ __align__(16) unsigned char inc_dyn[];
    __shared__ Topo sT;
    __shared__ State sS;
    __shared__ Search sX;
    __shared__ Inc sI;
    const int q = blockIdx.x / cs;
    if (q >= nf) return;
    const int f = order[q];
    if (threadIdx.x == 0) {
        sT = fd[f].T;
        sS = fd[f].S;
        sX = fd[f].X;
        sI = fd[f].I;
    }
    __syncthreads();
    Ctrl *C = fd[f].C;
    const bool ok = *fd[f].setup_err == 0;
    if (ok) inc_run<NT, PREC, CS>(sT, sS, sX, sI, C, false, inc_dyn, rec_mode, se, cw);
    csync(cs);                              // (every CTA's labels)
    if (cs > 1 && cluster_rank() != 0) return;
    for (int i = threadIdx.x; i < sT.n; i += NT) fd[f].super_out[i] = ok ? sT.orig[sS.label[sT.pre[i]]] : -1;
    if (threadIdx.x == 0) {
        const int t = ok ? C->t : 0;
        *fd[f].max_err = t > 0 ? sX.dec_maxerr[t - 1] : 0.0;
    }
}

constexpr size_t kIncSmemMax = 200 * 1024;  // largest dynamic shared memory of one search
// no feeder that fits (fewest entries in shared memory, one CTA or a cluster) overflows the sums' limbs
constexpr size_t least_bytes(int n, int cs) {
    return base_bytes(n, 1, cs) + (cs > 1 ? align16(rec_maxm_bytes(own_pairs(n, 0, cs))) : 0);
}
static_assert(least_bytes(kLimbMaxBus + 1, 1) > kIncSmemMax && least_bytes(kLimbMaxBus + 1, 2) > kIncSmemMax &&
              least_bytes(kLimbMaxBus + 1, kMaxCluster) > kIncSmemMax, "limb_sum: more buses than 31 bits hold");
constexpr int kInitThreads = 384;           // CTAs of the first evaluation
constexpr int kClusterThreads = 256;        // threads a CTA of a cluster of kMaxCluster, unless the caller says
constexpr int kClusterMin = 32;             // buses from which a cluster searches (inc_plan)
constexpr int kBatchCluster = 500;          // ... one of a batch's feeders (inc_batch_clusters; below it eight CTAs
                                            // were slower in the one batch tried, two have not been measured)

// Before every launch, whatever its size: without asking a launch gets 48 KB less
// the kernel's 17 to 21 KB of static arrays.  Always the same limit: it is the
// process's, and one set for a smaller feeder would hold for a larger one's launch
// on another thread (fifteen threads with feeders of 4 to 1,200 buses: 8 of 30,000
// calls refused).
template <typename K>
cudaError_t set_smem(K kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kIncSmemMax);
}

}  // namespace

// The launches of one precision: its kernels are compiled in a translation unit
// of their own (okr_incr64.cu includes this file for the FP64 terms), so that
// the two compile side by side.
template <int PREC> cudaError_t launch_one_prec(Topo T, State S, Search X, Inc I, Ctrl *C, int verify, const IncPlan &pl, cudaStream_t st);
template <int PREC> cudaError_t prepare_batch_prec(const IncPlan &pl);
template <int PREC> cudaError_t launch_batch_prec(const BatchFeeder *fd, const int *order, int nf, const IncPlan &pl, cudaStream_t st);
template <int PREC> int batch_clusters_prec(const IncPlan &pl);          // clusters of the plan resident at once
template <int PREC> cudaError_t prepare_init_prec();
template <int PREC> void launch_init_prec(const BatchFeeder *fd, const int *order, const int *cta_off, int nf, int cta0, int ctas,
                                          size_t ismem, cudaStream_t st);

#ifndef OKR_INCR_FP64

IncShape inc_shape_resolve(IncShape sh) {
    if (sh.threads != 256 && sh.threads != 384 && sh.threads != 512) sh.threads = kIncDefaultThreads;
    const int nw = sh.threads / 32;
    if (sh.cw < 1 || sh.cw > nw - 1) sh.cw = sh.threads == 512 ? 4 : 2;
    if (sh.se < 1 || sh.se > kSEMax) sh.se = kSEMax;
    if (sh.rec < -1 || sh.rec > 2) sh.rec = -1;
    return sh;
}

// Dynamic shared memory for an n-bus feeder: the per-merge data always, the
// selection records (and, when `maxm`, the largest MICE per super-node) when
// the total stays within kIncSmemMax, or where sh.rec places them.  Returns
// false when a forced placement does not fit (or asks for the per-super-node
// maximum where `maxm` is false).
bool inc_smem(int n, bool maxm, const IncShape &sh, int *rec_mode, size_t *bytes) {
    const size_t base = base_bytes(n, sh.se, 1);
    const bool fit2 = maxm && base + rec_maxm_bytes(n) <= kIncSmemMax;
    const bool fit1 = base + rec_bytes(n) <= kIncSmemMax;
    int m = sh.rec;
    if (m < 0) m = fit2 ? 2 : (fit1 ? 1 : 0);
    if ((m == 2 && !fit2) || (m == 1 && !fit1) || base > kIncSmemMax) return false;
    *rec_mode = m;
    *bytes = m == 2 ? base + rec_maxm_bytes(n) : (m == 1 ? base + rec_bytes(n) : base);
    return true;
}

// One CTA or a cluster of kMaxCluster.  A cluster shares out the scan over the
// slot pairs, the FP64 evaluation of the merge, the changed terms and the
// records (in shared memory up to 9,792 buses, above which one CTA searches; the
// carried sums and candidates too up to 4,404), and pays three cluster barriers a
// merge and L2 in place of L1 latency.  us a merge, one CTA of 384 threads / eight of 256 (one
// scenario; 400 buses two):
//   FP64 terms:  60 buses 13.4 / 12.3, 100 12.5 / 11.6, 400 16.3 / 11.7, 600 15.3 / 11.2, 1,500 17.7 / 11.5
//   FP32 terms:  60 buses 12.0 / 11.5, 100 11.1 / 10.6, 400 13.2 / 10.9, 600 12.2 / 9.8, 1,500 13.8 / 9.8
// A forced record placement asks for one CTA's memory, and recorded iterations
// are compacted by one CTA.
bool inc_plan(int n, const IncShape &raw, bool records_iters, IncPlan *out) {
    out->sh = inc_shape_resolve(raw);
    out->cs = 1;
    if (!inc_smem(n, true, out->sh, &out->rec, &out->bytes)) return false;
    out->mode = out->rec;
    if (out->sh.rec >= 0 || records_iters || n < kClusterMin) return true;
    const int np = own_pairs(n, 0, kMaxCluster);
    const size_t b = base_bytes(n, out->sh.se, kMaxCluster) + align16(rec_maxm_bytes(np));
    if (b > kIncSmemMax) return true;
    out->cs = kMaxCluster;
    const bool own = b + sums_bytes(np) <= kIncSmemMax;
    out->mode = own ? 2 + 4 : 2;
    out->bytes = own ? b + sums_bytes(np) : b;
    // fewer warps meet at the cluster's barriers (384 threads, FP32 terms: 100 buses 11.3 us, 1,500
    // 10.2); a caller's eval_warps that 256 threads cannot give keeps 384
    if (raw.threads == 0 && raw.cw < kClusterThreads / 32) {
        IncShape sh = raw;
        sh.threads = kClusterThreads;
        out->sh = inc_shape_resolve(sh);
    }
    return true;
}

#endif

namespace {

cudaLaunchConfig_t search_config(int ctas, int threads, int cs, size_t bytes, cudaStream_t st, cudaLaunchAttribute *at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = st;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)cs;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cs > 1 ? 1 : 0;
    return cfg;
}

template <int NT, int PREC, int CS>
cudaError_t launch_cs(Topo T, State S, Search X, Inc I, Ctrl *C, int verify, const IncPlan &pl, cudaStream_t st) {
    const cudaError_t e = set_smem(k_search_inc<NT, PREC, CS>);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = search_config(CS, NT, CS, pl.bytes, st, at);
    return cudaLaunchKernelEx(&cfg, k_search_inc<NT, PREC, CS>, T, S, X, I, C, verify, pl.mode, pl.sh.se, pl.sh.cw);
}

template <int NT, int PREC>
cudaError_t launch_one(Topo T, State S, Search X, Inc I, Ctrl *C, int verify, const IncPlan &pl, cudaStream_t st) {
    // the first evaluation spread over the SMs (its sums start at zero), then
    // the search on one cluster
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                      cudaSuccess || sms < 1)
            sms = 1;
    }
    const int ginit = std::min(std::min(sms, kInitCtasMax), std::max(1, (T.n + kInitPairs - 1) / kInitPairs));
    const size_t ismem = align16((size_t)2 * T.n) + align16((size_t)8 * T.n);
    cudaError_t e = cudaMemsetAsync(I.acc, 0, reinterpret_cast<const char *>(I.vmay + 2 * (size_t)T.n) -
                                                  reinterpret_cast<const char *>(I.acc), st);
    if (e == cudaSuccess) e = set_smem(k_inc_init<kInitThreads, PREC>);
    if (e == cudaSuccess) k_inc_init<kInitThreads, PREC><<<ginit, kInitThreads, ismem, st>>>(T, S, X, I, C);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (pl.cs == 1) return launch_cs<NT, PREC, 1>(T, S, X, I, C, verify, pl, st);
    return launch_cs<NT, PREC, kMaxCluster>(T, S, X, I, C, verify, pl, st);
}

template <int NT, int PREC, int CS>
cudaError_t launch_batch(const BatchFeeder *fd, const int *order, int nf, const IncPlan &pl, cudaStream_t st) {
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = search_config(nf * CS, NT, CS, pl.bytes, st, at);
    return cudaLaunchKernelEx(&cfg, k_search_inc_batch<NT, PREC, CS>, fd, order, nf, pl.mode, pl.sh.se, pl.sh.cw);
}

// The batch kernels: one CTA of 256, 384 or 512 threads, clusters of two of 384
// and of eight of 256 (inc_batch_plan).
template <int PREC, typename F>
cudaError_t batch_kernels(int cs, int threads, F f) {
    if (cs == kMaxCluster) return f(std::integral_constant<int, 256>(), std::integral_constant<int, kMaxCluster>());
    if (cs == 2) return f(std::integral_constant<int, 384>(), std::integral_constant<int, 2>());
    if (threads == 256) return f(std::integral_constant<int, 256>(), std::integral_constant<int, 1>());
    if (threads == 384) return f(std::integral_constant<int, 384>(), std::integral_constant<int, 1>());
    return f(std::integral_constant<int, 512>(), std::integral_constant<int, 1>());
}
}  // namespace

template <int PREC>
cudaError_t launch_one_prec(Topo T, State S, Search X, Inc I, Ctrl *C, int verify, const IncPlan &pl, cudaStream_t st) {
    if (pl.sh.threads == 256) return launch_one<256, PREC>(T, S, X, I, C, verify, pl, st);
    if (pl.sh.threads == 384) return launch_one<384, PREC>(T, S, X, I, C, verify, pl, st);
    return launch_one<512, PREC>(T, S, X, I, C, verify, pl, st);
}
template <int PREC>
cudaError_t prepare_batch_prec(const IncPlan &pl) {
    return batch_kernels<PREC>(pl.cs, pl.sh.threads, [&](auto nt, auto c) {
        return set_smem(k_search_inc_batch<decltype(nt)::value, PREC, decltype(c)::value>);
    });
}
template <int PREC>
cudaError_t launch_batch_prec(const BatchFeeder *fd, const int *order, int nf, const IncPlan &pl, cudaStream_t st) {
    return batch_kernels<PREC>(pl.cs, pl.sh.threads, [&](auto nt, auto c) {
        return launch_batch<decltype(nt)::value, PREC, decltype(c)::value>(fd, order, nf, pl, st);
    });
}
template <int PREC>
int batch_clusters_prec(const IncPlan &pl) {
    int count = 0;
    const cudaError_t e = batch_kernels<PREC>(pl.cs, pl.sh.threads, [&](auto nt, auto c) {
        constexpr int cs = decltype(c)::value;
        const auto kern = k_search_inc_batch<decltype(nt)::value, PREC, cs>;
        cudaLaunchAttribute at[1];
        const cudaLaunchConfig_t cfg = search_config(cs, decltype(nt)::value, cs, pl.bytes, nullptr, at);
        const cudaError_t e1 = set_smem(kern);
        return e1 != cudaSuccess ? e1 : cudaOccupancyMaxActiveClusters(&count, kern, &cfg);
    });
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? count : 0;
}
template <int PREC>
cudaError_t prepare_init_prec() {
    return set_smem(k_inc_init_batch<kInitThreads, PREC>);
}
template <int PREC>
void launch_init_prec(const BatchFeeder *fd, const int *order, const int *cta_off, int nf, int cta0, int ctas, size_t ismem,
                      cudaStream_t st) {
    k_inc_init_batch<kInitThreads, PREC><<<ctas, kInitThreads, ismem, st>>>(fd, order, cta_off, nf, cta0);
}

#ifdef OKR_INCR_FP64

template cudaError_t launch_one_prec<0>(Topo, State, Search, Inc, Ctrl *, int, const IncPlan &, cudaStream_t);
template cudaError_t prepare_batch_prec<0>(const IncPlan &);
template cudaError_t launch_batch_prec<0>(const BatchFeeder *, const int *, int, const IncPlan &, cudaStream_t);
template int batch_clusters_prec<0>(const IncPlan &);
template cudaError_t prepare_init_prec<0>();
template void launch_init_prec<0>(const BatchFeeder *, const int *, const int *, int, int, int, size_t, cudaStream_t);

#else

extern template cudaError_t launch_one_prec<0>(Topo, State, Search, Inc, Ctrl *, int, const IncPlan &, cudaStream_t);
extern template cudaError_t prepare_batch_prec<0>(const IncPlan &);
extern template cudaError_t launch_batch_prec<0>(const BatchFeeder *, const int *, int, const IncPlan &, cudaStream_t);
extern template int batch_clusters_prec<0>(const IncPlan &);
extern template cudaError_t prepare_init_prec<0>();
extern template void launch_init_prec<0>(const BatchFeeder *, const int *, const int *, int, int, int, size_t, cudaStream_t);

cudaError_t launch_search_inc(int precision, Topo T, State S, Search X, Inc I, Ctrl *C, int verify, const IncPlan &pl,
                              cudaStream_t st) {
    return precision == 1 ? launch_one_prec<1>(T, S, X, I, C, verify, pl, st) : launch_one_prec<0>(T, S, X, I, C, verify, pl, st);
}

bool inc_batch_plan(int max_n, int cs, const IncShape &raw, IncPlan *out) {
    IncShape sh = raw;
    if (sh.threads == 0 && cs == kMaxCluster) sh.threads = kClusterThreads;
    out->sh = inc_shape_resolve(sh);
    out->cs = cs;
    if (cs == 1) {
        if (!inc_smem(max_n, false, out->sh, &out->rec, &out->bytes)) return false;
        out->mode = out->rec;
        return true;
    }
    const int np = own_pairs(max_n, 0, cs);
    const size_t b = base_bytes(max_n, out->sh.se, cs) + align16(rec_maxm_bytes(np));
    if (b > kIncSmemMax) return false;
    const bool own = b + sums_bytes(np) <= kIncSmemMax;
    out->rec = 2;
    out->mode = own ? 2 + 4 : 2;
    out->bytes = own ? b + sums_bytes(np) : b;
    return true;
}

// How many of the first feeders (largest first) are searched by clusters, and of
// how many CTAs (none under a forced record placement or another thread count).
// With SMs for eight CTAs a feeder, all that gain take eight, as far as those
// clusters are resident at once (a merge on one CTA / eight, FP32 terms, one
// scenario: 600 buses 12.2 / 9.8 us, 1,500 13.8 / 9.8).  Otherwise the feeders
// whose chain alone outlasts an even share of the work by a quarter take two (a
// merge on two CTAs costs 1.7 of the SM time of one, on four 2.7: more would take
// from the others what the longest chains gain).  256 feeders of 200 .. 2,000
// buses, FP32: 30.1 ms of search, 32.8 with one CTA each; 48 feeders of 60 .. 400
// with eight for the 14 largest 4.8 ms, with one CTA each 4.6.
void inc_batch_clusters(int precision, int nf, const int *n, const int *merges, int num_sms, const IncShape &raw, int *count,
                        int *cs) {
    *count = 0;
    *cs = 1;
    // (clusters of eight have 256 threads a CTA: not for a caller's eval_warps above 7)
    const bool spare = (long long)nf * kMaxCluster <= num_sms && (raw.threads != 0 || raw.cw < kClusterThreads / 32);
    if (raw.rec >= 0 || (raw.threads != 0 && raw.threads != (spare ? kClusterThreads : 384)) || nf < 1) return;
    // us on one CTA, FP32 terms (compared with the other feeders of the launch, which
    // have the same precision: FP64 terms cost a tenth to a quarter more on each)
    auto chain = [&](int i) { return merges[i] * (11.0 + 0.002 * n[i]); };
    double sum = 0.0;
    for (int i = 0; i < nf; ++i) sum += chain(i);
    int k = 0, max_n = 2;
    while (k < nf && n[k] >= kBatchCluster && (spare || (chain(k) > 1.25 * sum / num_sms && 4 * (k + 1) <= num_sms)))
        max_n = std::max(max_n, n[k++]);
    IncPlan pl;
    if (k == 0 || !inc_batch_plan(max_n, spare ? kMaxCluster : 2, raw, &pl)) return;
    k = std::min(k, precision == 1 ? batch_clusters_prec<1>(pl) : batch_clusters_prec<0>(pl));
    if (k < 1) return;
    *count = k;
    *cs = pl.cs;
}

cudaError_t prepare_search_inc_batch(int precision, const IncPlan &pl) {
    return precision == 1 ? prepare_batch_prec<1>(pl) : prepare_batch_prec<0>(pl);
}

cudaError_t launch_search_inc_batch(int precision, const BatchFeeder *fd, const int *order, int nf, const IncPlan &pl,
                                    cudaStream_t st) {
    if (nf <= 0) return cudaSuccess;
    return precision == 1 ? launch_batch_prec<1>(fd, order, nf, pl, st) : launch_batch_prec<0>(fd, order, nf, pl, st);
}

cudaError_t prepare_inc_init_batch(int precision) {
    return precision == 1 ? prepare_init_prec<1>() : prepare_init_prec<0>();
}

cudaError_t launch_inc_init_batch(int precision, int max_n, const BatchFeeder *fd, const int *order,
                                  const int *cta_off, int nf, int cta0, int ctas, cudaStream_t st) {
    if (nf <= 0 || ctas <= 0) return cudaSuccess;
    const size_t ismem = align16((size_t)2 * max_n) + align16((size_t)8 * max_n);
    k_inc_zero_batch<<<nf, 256, 0, st>>>(fd, order, nf);
    if (precision == 1) launch_init_prec<1>(fd, order, cta_off, nf, cta0, ctas, ismem, st);
    else launch_init_prec<0>(fd, order, cta_off, nf, cta0, ctas, ismem, st);
    return cudaGetLastError();
}

#endif

}  // namespace okr
