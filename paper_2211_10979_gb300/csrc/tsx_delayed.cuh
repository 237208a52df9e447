// Delayed updates: the pivots of the condensed tableau (arXiv 2211.10979,
// Section III, Steps 1-3) with the rank-1 updates of up to K pivots applied in
// one pass over the tableau.
//
// A pivot needs only four parts of the tableau up to date: the objective row
// (Step 1), column q and the right-hand side (Step 2), and row p (Step 3).  So
// the G blocks that work on an LP keep the objective row and the right-hand
// side current and hold the updates of the other entries back: pivot u of a
// round leaves its multipliers F_u (column q before the update) and its scaled
// row R_u.  Column q and row p of the next pivot are read from the tableau and
// brought up to date by the pending updates in their order,
//   t = fma(-F_u[i], R_u[j], t)   for u = 0, 1, ...,
// and after K pivots (or at the end) one pass applies the same chain to every
// entry.  Each entry so takes the fused multiply-adds of the undelayed update,
// in the same order on the same operands: every stored value, pivot and result
// is the same, bit for bit (up to the sign of zeros, which no step can see).
//
// Entries that a pivot replaces start their chain anew: row p becomes R_u at
// once and its pending multipliers are set to zero; column q starts from zero
// and the pending rows' entries of that column are set to zero.  A zeroed step
// is the identity, fma(-0, r, t) = t, as long as the other factor is finite; a
// pivot with a non-finite multiplier or row entry therefore ends its round at
// once, and row p is stored again after that pass.
//
// What bounds it: the undelayed update moves the whole tableau through HBM per
// pivot (8192^2 FP64: 151 of 166 us a pivot; 12288^2 FP32: 172 of 178 us).
// Delayed, that traffic is divided by K and the pass is bound by its fused
// multiply-adds (FP64 pipe: 626 G fma/s), plus a latency chain per pivot of
// two exchanges between the blocks (6.5-8.5 us).  Measured, undelayed -> delayed,
// us a pivot: FP64 1024^2 15.3 -> 9.6, 4096^2 51 -> 36.6 (pass 26.8, its fmas
// alone 26.8), 8192^2 166 -> 118.1 (pass 108.8, its fmas 107.2); FP32 4096^2
// 33 -> 8.0, 12288^2 178 -> 16.3.
#pragma once

#include "tsx_device.cuh"

namespace tsx {

// Pivots per round: the pass costs 1/K of an HBM sweep per pivot and the
// chains of column q and row p K/2 dependent steps on average.  Measured (us a
// pivot): FP64 K = 8 / 16 / 32 at 1024^2 12.3 / 11.5 / 12.2, at 8192^2 122.9 /
// 120.5 / 119.8; FP32 K = 32 / 64 at 4096^2 9.1 / 9.5, at 12288^2 18.4 / 18.2.
template <typename V> struct DelayK;
template <> struct DelayK<double> { static constexpr int K = 16; };
template <> struct DelayK<float> { static constexpr int K = 32; };

// One exchange record: the candidate of one block.
struct __align__(16) DelayRec {
    unsigned long long hi;  // the value's integer key (delay_key)
    int key;                // tie-break key, INT_MAX: no candidate
    unsigned low;           // index within the block << 1 | the block met a non-finite entry
};

template <typename V>
struct Delayed {            // one LP and the blocks that work on it
    V* T;                   // condensed tableau, (m+1) x ld
    int ld, m, n;
    int* basis;
    int* var;
    V* Fh;                  // (m+1) x K: multipliers of the round's pivots
    V* Rh;                  // K x ld: scaled rows of the round's pivots (columns >= n stay zero)
    V* RhT;                 // ld x K: the same, transposed
    V* rhs;                 // m+1: right-hand side, up to date (blocks that keep theirs in shared memory: unused)
    DelayRec* rat;          // G: leaving candidates
    DelayRec* arg;          // G: entering candidates
    unsigned* bar_count;    // counted barrier of the G blocks
    int* fail;              // nonzero: a wait ran out
    int* status;            // state word to mark on a timeout (may be null)
    int bt, G;              // this block, blocks
    unsigned smem;          // dynamic shared memory of a block, bytes
    V eps_d, eps_p;         // delay_eps of the tolerances
    long long max_iters;
    int k_cyc, rule;
    long long timeout_ns;
    int* qlog;
    int* plog;
    long long log_cap;
};

struct DelayPart {          // one warp's part of a block reduction
    unsigned long long hi;
    int key, idx, nonfinite, pad;
};
// Words of one exchange: the send's are written before its block barrier and
// read by warp 0 before it arrives at the gather's, and the other way round,
// so that each half needs one block barrier only.
struct DelayScratch {
    DelayPart send[kMaxWarps];
    DelayPart got;
    int fail;
    unsigned passed;        // counted barriers this block has passed (thread 0)
    unsigned tile;          // tiles handed out in a pass
};

// State of a solve between its rounds (shared memory; thread 0 writes it).
struct DelayState {
    int status;             // kRunning, the final status, or kDelayFailed
    int bland, degen;
    int k;                  // pending pivots
    int last;               // row of the last of them
    int flag;               // it met a non-finite entry
    unsigned passes;        // update passes over the tableau
    long long it;
    unsigned long long ehi; // the entering candidate of the next pivot
    int ekey, eidx;
};
constexpr int kDelayFailed = INT_MIN;

// ------------------------------------------------------------ exchange
struct DelayCand {          // smallest (hi, key); idx: its row or column slot
    unsigned long long hi;
    int key, idx;
};
__device__ __forceinline__ DelayCand delay_none() { return DelayCand{~0ull, INT_MAX, INT_MAX}; }
// bland: the lowest key decides and hi only carries the value.
__device__ __forceinline__ void delay_merge(DelayCand& a, const DelayCand& b, int bland = 0) {
    if (bland ? b.key < a.key : (b.hi < a.hi || (b.hi == a.hi && b.key < a.key))) a = b;
}
// The warp's smallest candidate, in every lane: minimum reductions of the
// value's halves, then of the keys among the lanes that hold them (five
// shuffle rounds of four words took 0.1 us more).
__device__ __forceinline__ DelayCand delay_warp(DelayCand a, int bland = 0) {
    constexpr unsigned all = 0xffffffffu;
    bool in = true;
    if (!bland) {
        const unsigned h = (unsigned)(a.hi >> 32), l = (unsigned)a.hi;
        in = h == __reduce_min_sync(all, h);
        const unsigned x = in ? l : ~0u, y = __reduce_min_sync(all, x);
        in = in && l == y;
    }
    const unsigned k = in ? (unsigned)a.key : ~0u;
    const unsigned m = __reduce_min_sync(all, k);
    const int from = __ffs(__ballot_sync(all, in && (unsigned)a.key == m)) - 1;
    DelayCand b;
    b.hi = __shfl_sync(all, a.hi, from);
    b.key = (int)m;
    b.idx = __shfl_sync(all, a.idx, from);
    return b;
}
// Values as unsigned keys in their order (dkey; -0 counts as +0): 64 bits of a
// double, or 32 bits of a float in the upper half, so that the float pivots
// need no FP64 instruction.
__device__ __forceinline__ unsigned long long delay_key(double x) {
    return (unsigned long long)dkey(x) ^ 0x8000000000000000ull;
}
__device__ __forceinline__ unsigned long long delay_key(float x) {
    int b = __float_as_int(x);
    if (b == INT_MIN) b = 0;
    b ^= (b >> 31) & 0x7fffffff;
    return (unsigned long long)((unsigned)b ^ 0x80000000u) << 32;
}
template <typename V> __device__ __forceinline__ V delay_value(unsigned long long k);
template <> __device__ __forceinline__ double delay_value<double>(unsigned long long k) {
    return dkey_value((long long)(k ^ 0x8000000000000000ull));
}
template <> __device__ __forceinline__ float delay_value<float>(unsigned long long k) {
    const int b = (int)((unsigned)(k >> 32) ^ 0x80000000u);
    return __int_as_float(b ^ ((b >> 31) & 0x7fffffff));
}
// The tolerances as values of V: x > eps exactly if x > the largest V not
// above eps.
__device__ __forceinline__ void delay_eps(double eps, double& v) { v = eps; }
__device__ __forceinline__ void delay_eps(double eps, float& v) { v = __double2float_rd(eps); }
__device__ __forceinline__ bool delay_finite(double x) { return dbits_finite(x); }
__device__ __forceinline__ bool delay_finite(float x) {
    return (__float_as_uint(x) & 0x7f800000u) != 0x7f800000u;
}
__device__ __forceinline__ bool delay_nan(double x) { return dbits_nan(x); }
__device__ __forceinline__ bool delay_nan(float x) { return (__float_as_uint(x) & 0x7fffffffu) > 0x7f800000u; }

template <typename V>
__device__ __forceinline__ void delay_give_up(const Delayed<V>& D) {
    atomicExch(D.fail, 1);
    if (D.status) atomicCAS(D.status, kRunning, kTimeout);
}

// Barrier of the block's NT threads (BAR = 0), or of the NT threads that use the
// named barrier BAR.
template <int BAR, int NT>
__device__ __forceinline__ void delay_sync() {
    if (BAR == 0)
        __syncthreads();
    else
        asm volatile("bar.sync %0, %1;" ::"n"(BAR), "n"(NT) : "memory");
}

// An exchange between the D.G blocks: every block sends a candidate, every
// block gets the smallest.  It is a counted barrier (as grid_barrier_counted)
// whose arrival also publishes the block's record, so that what a block has
// written before its send is visible to the others after their gather.
// Measured over 152 blocks: 1.9 us; with every block polling all the records
// for a tag instead of one counter 3.2 us (23k polls at a time hold up the
// records' own stores).
// cnt: the threads that may hold a candidate; idx0: the block's first row or
// column.
template <int NT, int BAR = 0, typename V>
__device__ __forceinline__ void delay_send(const Delayed<V>& D, DelayRec* recs, DelayCand a, int nonfinite, int idx0,
                                           int cnt, int bland, DelayScratch& s) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w == 0 || w * 32 < cnt) {
        a = delay_warp(a, bland);
        nonfinite = __any_sync(0xffffffffu, nonfinite);
        if (lane == 0) s.send[w] = DelayPart{a.hi, a.key, a.idx, nonfinite, 0};
    }
    delay_sync<BAR, NT>();
    if (threadIdx.x == 0) {
        for (int k = 1; k < NT / 32 && k * 32 < cnt; ++k) {
            const DelayPart x = s.send[k];
            delay_merge(a, DelayCand{x.hi, x.key, x.idx}, bland);
            nonfinite |= x.nonfinite;
        }
        const unsigned low = (a.key == INT_MAX ? 0u : (unsigned)(a.idx - idx0) << 1) | (nonfinite ? 1u : 0u);
        __stcg(reinterpret_cast<uint4*>(recs + D.bt),
               make_uint4((unsigned)a.hi, (unsigned)(a.hi >> 32), (unsigned)a.key, low));
        red_add_release(D.bar_count, 1u);
    }
}

// Thread 0: waits until all blocks have arrived `passed` + 1 times on the
// counter.  Bounded in time like the grid barrier: false if the wait ran out
// here or in another block.
template <typename V>
__device__ __forceinline__ bool delay_wait(const Delayed<V>& D, unsigned& passed) {
    const unsigned target = (passed + 1u) * (unsigned)D.G;
    passed += 1u;
    if ((int)(ld_acquire(D.bar_count) - target) >= 0) return true;
    const long long t0 = global_ns();
    const unsigned long long max_spins = (unsigned long long)(D.timeout_ns > 0 ? D.timeout_ns : 0) + 4096ull;
    for (unsigned long long spins = 0; (int)(ld_acquire(D.bar_count) - target) < 0; ++spins) {
        if ((spins & 31ull) == 0) {
            if (global_ns() - t0 >= D.timeout_ns || spins > max_spins) {
                delay_give_up(D);
                return false;
            }
            if (spins && ld_relaxed(D.fail) != 0) return false;
        }
    }
    return true;
}

// The smallest candidate of all blocks (every thread returns it); per: rows or
// columns per block.  False if a wait ran out.  Warp 0 waits, reads the records
// and reduces them; the others wait at the block barrier.
template <int NT, int BAR = 0, typename V>
__device__ __forceinline__ bool delay_gather(const Delayed<V>& D, const DelayRec* recs, int per, int bland,
                                             DelayCand& out, int& nonfinite, DelayScratch& s) {
    if (threadIdx.x < 32) {
        int ok = 1;
        if (threadIdx.x == 0) ok = delay_wait(D, s.passed);
        ok = __shfl_sync(0xffffffffu, ok, 0);
        __syncwarp();   // orders the records' loads after thread 0's acquire
        DelayCand a = delay_none();
        int nf = 0;
        constexpr int U = 5;   // records in flight per lane: 160 blocks at once
#pragma unroll 1
        for (int k0 = threadIdx.x; k0 < D.G; k0 += 32 * U) {
            uint4 x[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (k0 + 32 * u < D.G) x[u] = __ldcg(reinterpret_cast<const uint4*>(recs + k0 + 32 * u));
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (k0 + 32 * u < D.G) {
                    nf |= (int)(x[u].w & 1u);
                    delay_merge(a, DelayCand{((unsigned long long)x[u].y << 32) | x[u].x, (int)x[u].z,
                                             (k0 + 32 * u) * per + (int)(x[u].w >> 1)}, bland);
                }
        }
        a = delay_warp(a, bland);
        nf = __any_sync(0xffffffffu, nf);
        if (threadIdx.x == 0) {
            s.got = DelayPart{a.hi, a.key, a.idx, nf, 0};
            s.fail = !ok;
        }
    }
    delay_sync<BAR, NT>();
    out = DelayCand{s.got.hi, s.got.key, s.got.idx};
    nonfinite = s.got.nonfinite;
    return s.fail == 0;
}

// A plain barrier of the D.G blocks on the same counter.
template <int NT, int BAR = 0, typename V>
__device__ __forceinline__ bool delay_barrier(const Delayed<V>& D, DelayScratch& s) {
    delay_sync<BAR, NT>();
    if (threadIdx.x == 0) {
        red_add_release(D.bar_count, 1u);
        s.fail = !delay_wait(D, s.passed);
    }
    delay_sync<BAR, NT>();
    return s.fail == 0;
}

// ---------------------------------------------------------- pending chains
// t through the k pending updates: the entry's own factors at own[u * step]
// (the multipliers of its row, or the row entries of its column, kept by the
// block) and the other factors at other[u] (shared memory); both arrays hold K
// entries.  In float a step costs less than a branch: eight at a time, the steps
// beyond k computed and dropped; a dropped FP64 step would hold the pipe (~80
// cycles).
template <int K>
__device__ __forceinline__ double delay_chain(const double* own, int step, const double* other, int k, double t) {
#pragma unroll 4
    for (int u = 0; u < k; ++u) t = fma_rn(-own[u * step], other[u], t);
    return t;
}
template <int K>
__device__ __forceinline__ float delay_chain(const float* own, int step, const float* other, int k, float t) {
    static_assert(K % 8 == 0, "eight steps at a time");
#pragma unroll 1
    for (int u = 0; u < k; u += 8) {
        float f[8], r[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            f[x] = own[(u + x) * step];
            r[x] = other[u + x];
        }
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            const float y = fma_rn(-f[x], r[x], t);
            t = u + x < k ? y : t;
        }
    }
    return t;
}
// All K pending updates: every load ahead of the chain.
template <int K, typename V>
__device__ __forceinline__ V delay_chain_all(const V* own, int step, const V* other, V t) {
    V f[K];
#pragma unroll
    for (int u = 0; u < K; ++u) f[u] = own[u * step];
#pragma unroll
    for (int u = 0; u < K; ++u) t = fma_rn(-f[u], other[u], t);
    return t;
}

// -------------------------------------------------------------- the pass
// The update tile of a warp: `RS` rows x 1 KB of columns, held in registers as
// four 64-bit words per row and lane (a double, or two floats run by the packed
// fma.rn.f32x2: one rounding per float, as fmaf): 16 bytes of each half of the
// 1 KB, so that a last strip of half the width or less takes half the fused
// multiply-adds.  Per pending pivot a lane takes its 32 bytes of R (shared memory, staged once per column
// strip for the whole block) and the rows' multipliers (shared memory, staged
// per tile, already negated; broadcast reads of two rows at a time).  With one
// block of 8 warps per SM the next tile's loads are in flight while a tile is
// updated: 64 KB per SM at any time with 8-row tiles, which is what the HBM
// stream needs.  Four pending pivots per turn of the loop, so that their reads
// of shared memory overlap (FP32 12288^2: the pass 10.5 -> 8.6 us a pivot; HBM
// alone 5.6, the fused multiply-adds alone 3.8).
template <typename V> struct Word;
template <> struct Word<double> {
    static __device__ __forceinline__ unsigned long long neg(double f) { return __double_as_longlong(-f); }
    static __device__ __forceinline__ unsigned long long fma(unsigned long long f, unsigned long long r,
                                                             unsigned long long t) {
        return __double_as_longlong(__fma_rn(__longlong_as_double(f), __longlong_as_double(r),
                                             __longlong_as_double(t)));
    }
};
template <> struct Word<float> {
    static __device__ __forceinline__ unsigned long long neg(float f) {
        const unsigned long long u = __float_as_uint(-f);
        return u | (u << 32);
    }
    static __device__ __forceinline__ unsigned long long fma(unsigned long long f, unsigned long long r,
                                                             unsigned long long t) {
        unsigned long long d;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(f), "l"(r), "l"(t));
        return d;
    }
};

constexpr int kDelayStrips = 2;   // column strips staged at a time
template <int RS>
__host__ __device__ constexpr int delay_fstride() { return RS * 8 + 16; }   // bytes per pending pivot (padded: banks)
template <typename V>
__host__ __device__ constexpr size_t delay_smem_bytes(int nt, int rs) {
    return (size_t)kDelayStrips * DelayK<V>::K * 1024 + (size_t)(nt / 32) * DelayK<V>::K * (size_t)(rs * 8 + 16);
}

// 16-byte accesses, each of a warp's 512 contiguous bytes.  (With 256-bit ones of
// four 64-bit words the team kernels' build, 128 registers a thread, gave wrong
// tableaux: the last three words not updated, also with every word of the tile
// set before its loads; k_pivot_delayed and k_pivot_overlap were right, and no
// faster.  The cause is not known; nvcc 13.0.88.)
__device__ __forceinline__ void ld_words(const void* p, unsigned long long* w) {
    asm volatile("ld.global.L1::no_allocate.v2.b64 {%0,%1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_words(void* p, const unsigned long long* w) {
    asm volatile("st.global.v2.b64 [%0], {%1,%2};" ::"l"(p), "l"(w[0]), "l"(w[1]) : "memory");
}

template <typename V, int RS, int K>
struct DelayTile {
    static constexpr int FS = delay_fstride<RS>(), NF = RS * K / 32, HALF = 512 / (int)sizeof(V);
    unsigned long long t[RS][4];
    V f[NF];                    // the rows' multipliers, entry lane + 32 x of the RS x K block
    const V* at;                // the lane's first entry; the other 16 bytes lie HALF entries on
    int na, nb;                 // rows to load and store in each half (0: beyond the tableau)
    int strip;                  // staged strip
    bool wide;                  // the strip has a second half

    // left: columns of the tableau from the strip's first on
    __device__ __forceinline__ void load(const Delayed<V>& D, const V* from, const V* Fh, int k, int i0, int col,
                                         int left, int staged) {
        constexpr int N = 16 / (int)sizeof(V);
        const int lane = threadIdx.x & 31, rows = min(RS, D.m + 1 - i0);
        at = from + (size_t)i0 * (size_t)D.ld + col + lane * N;
        na = lane * N < left ? rows : 0;
        nb = HALF + lane * N < left ? rows : 0;
        wide = left > HALF;
        strip = staged;
#pragma unroll
        for (int r = 0; r < RS; ++r) {
            if (r < na) ld_words(at + (size_t)r * (size_t)D.ld, t[r]);
            if (r < nb) ld_words(at + (size_t)r * (size_t)D.ld + HALF, t[r] + 2);
        }
        const V* fh = Fh + (size_t)i0 * K;
#pragma unroll
        for (int x = 0; x < NF; ++x) {
            const int e = lane + 32 * x;
            f[x] = e / K < rows && e % K < k ? __ldcg(fh + e) : V(0);
        }
    }
    // the first W of the four words of every row
    template <int W>
    __device__ __forceinline__ void chain(int k, const unsigned char* rs, const unsigned char* fs) {
#pragma unroll 4
        for (int u = 0; u < k; ++u) {
            const ulonglong2 ra = *reinterpret_cast<const ulonglong2*>(rs + u * 1024);
            ulonglong2 rb = make_ulonglong2(0, 0);
            if (W > 2) rb = *reinterpret_cast<const ulonglong2*>(rs + u * 1024 + 512);
#pragma unroll
            for (int r = 0; r < RS; r += 2) {
                const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(fs + u * FS + r * 8);
                t[r][0] = Word<V>::fma(g.x, ra.x, t[r][0]);
                t[r][1] = Word<V>::fma(g.x, ra.y, t[r][1]);
                t[r + 1][0] = Word<V>::fma(g.y, ra.x, t[r + 1][0]);
                t[r + 1][1] = Word<V>::fma(g.y, ra.y, t[r + 1][1]);
                if (W > 2) {
                    t[r][2] = Word<V>::fma(g.x, rb.x, t[r][2]);
                    t[r][3] = Word<V>::fma(g.x, rb.y, t[r][3]);
                    t[r + 1][2] = Word<V>::fma(g.y, rb.x, t[r + 1][2]);
                    t[r + 1][3] = Word<V>::fma(g.y, rb.y, t[r + 1][3]);
                }
            }
        }
    }
    // shift: from the tableau read to the one written, in entries
    __device__ __forceinline__ void update(const Delayed<V>& D, ptrdiff_t shift, int k, const unsigned char* rs,
                                           unsigned char* fs) {
        const int lane = threadIdx.x & 31;
        rs += strip * (K * 1024) + lane * 16;
        __syncwarp();   // the warp has read its previous tile's multipliers
#pragma unroll
        for (int x = 0; x < NF; ++x) {
            const int e = lane + 32 * x;
            *reinterpret_cast<unsigned long long*>(fs + (e % K) * FS + (e / K) * 8) = Word<V>::neg(f[x]);
        }
        __syncwarp();
        if (wide)
            chain<4>(k, rs, fs);
        else
            chain<2>(k, rs, fs);
        V* to = const_cast<V*>(at) + shift;
#pragma unroll
        for (int r = 0; r < RS; ++r) {
            if (r < na) st_words(to + (size_t)r * (size_t)D.ld, t[r]);
            if (r < nb) st_words(to + (size_t)r * (size_t)D.ld + HALF, t[r] + 2);
        }
    }
};

// Rows 1..m, columns 0..n-1: k pending updates applied to every entry.  Tiles
// are numbered strip by strip (a strip: 1 KB of columns); block b takes a
// contiguous range of them, so that it stages the pending rows of few strips,
// and its warps take the range's tiles from a counter.  Two strips are staged
// at a time: most ranges touch at most two, and a block barrier between strips
// would leave its last tiles without company (measured at 8192^2 FP64 against
// one strip and tiles in turn: the wait after the pass 4.5 -> 2.5 us a pivot).
// from, to: the tableau read and the one written (the same, or two).
// `rev`: the range backwards (alternate passes start on the tiles the previous
// one left in L2).
// AHEAD: the next tile's loads in flight while a tile is updated (needs the
// registers of one block of 256 threads per SM); without, the other warps of
// the SM cover a tile's loads.
// Not inlined: the tile takes most of a thread's registers.
template <int NT, int RS, bool AHEAD, int K, int BAR = 0, int T0 = 0, typename V>
__device__ __noinline__ void delay_pass(const Delayed<V>& D, const V* from, V* to, const V* Fh, const V* Rh, int k,
                                        int rev, unsigned char* smem, DelayScratch& s) {
    constexpr int CS = 1024 / (int)sizeof(V), NS = kDelayStrips;
    const int tid = threadIdx.x - T0, lane = tid & 31, w = tid >> 5;
    const ptrdiff_t shift = to - from;
    unsigned char* rs = smem;
    unsigned char* fs = smem + (size_t)NS * K * 1024 + (size_t)w * K * delay_fstride<RS>();
    const int nstrips = (D.n + CS - 1) / CS;
    const int ntiles = (D.m + RS - 1) / RS;
    const long long units = (long long)nstrips * ntiles;
    const long long u0 = units * D.bt / D.G, u1 = units * (D.bt + 1) / D.G;
    if (u0 >= u1) return;
    const int s0 = (int)(u0 / ntiles), s1 = (int)((u1 - 1) / ntiles);
    const int nchunks = (s1 - s0 + NS) / NS;
    for (int x = 0; x < nchunks; ++x) {
        const int f = s0 + (rev ? nchunks - 1 - x : x) * NS, l = min(s1, f + NS - 1);   // strips f..l
        const long long a = max(u0, (long long)f * ntiles), b = min(u1, (long long)(l + 1) * ntiles);
        delay_sync<BAR, NT>();   // the warps are done with the previous strips
        if (tid == 0) s.tile = 0;
        for (int e = tid; e < (l - f + 1) * k * 64; e += NT) {
            const int c = e & 63, v = e >> 6, y = v / k, u = v - y * k;   // 16-byte piece c of pivot u, strip f + y
            const int j = (f + y) * CS + c * (CS / 64);
            if (j < D.ld)
                *reinterpret_cast<ulonglong2*>(rs + (y * K + u) * 1024 + c * 16) =
                    __ldcg(reinterpret_cast<const ulonglong2*>(Rh + (size_t)u * (size_t)D.ld + j));
        }
        delay_sync<BAR, NT>();
        const unsigned count = (unsigned)(b - a);
        auto next = [&]() {
            unsigned z = 0;
            if (lane == 0) z = atomicAdd(&s.tile, 1u);
            return __shfl_sync(0xffffffffu, z, 0);
        };
        auto load = [&](DelayTile<V, RS, K>& tile, unsigned z) {
            const long long unit = rev ? b - 1 - (long long)z : a + (long long)z;
            const int strip = (int)(unit / ntiles), row = (int)(unit - (long long)strip * ntiles);
            tile.load(D, from, Fh, k, 1 + row * RS, strip * CS, D.n - strip * CS, strip - f);
        };
        unsigned z = next();
        if constexpr (AHEAD) {
            DelayTile<V, RS, K> cur, ahead;
            if (z < count) load(cur, z);
#pragma unroll 1
            while (z < count) {
                z = next();
                if (z < count) load(ahead, z);
                cur.update(D, shift, k, rs, fs);
                cur = ahead;
            }
        } else {
#pragma unroll 1
            for (; z < count; z = next()) {
                DelayTile<V, RS, K> tile;
                load(tile, z);
                tile.update(D, shift, k, rs, fs);
            }
        }
    }
}

// ------------------------------------------------------------- the pivots
// Shared memory of a block that keeps its own parts there: its rows' pending
// multipliers and its columns' pending row entries (dead during a pass, whose
// staging takes the same bytes), then the right-hand sides of its rows and the
// objective-row entries and variables of its columns.
__host__ __device__ constexpr int delay_per(int count, int blocks) { return (count + blocks - 1) / blocks; }
template <typename V>
__host__ __device__ constexpr size_t delay_own_offset(int m, int n, int blocks, size_t pass_bytes) {
    const size_t own = (size_t)(delay_per(m + 1, blocks) + delay_per(n, blocks)) * DelayK<V>::K * sizeof(V);
    return ((own > pass_bytes ? own : pass_bytes) + 15) / 16 * 16;
}
template <typename V>
__host__ __device__ constexpr size_t delay_own_bytes(int m, int n, int blocks, size_t pass_bytes) {
    return delay_own_offset<V>(m, n, blocks, pass_bytes) + (size_t)delay_per(m + 1, blocks) * sizeof(V) +
           (size_t)delay_per(n, blocks) * (sizeof(V) + sizeof(int));
}

// Where a block finds its own parts: in shared memory, or in place in the
// global buffers where they do not fit (pending entries: [u * fu + row * fr]
// and [u * ru + column * rr]).
template <typename V>
struct DelayOwn {
    int rper, cper, rb, nr, cb, nc;
    bool own;
    V *fo, *ro, *rhs, *obj;
    int* var;
    int fu, fr, ru, rr;
    V *sf, *sr;   // the pending entries' place in shared memory
    __device__ __forceinline__ DelayOwn(const Delayed<V>& D, unsigned char* smem, size_t pass_bytes) {
        constexpr int K = DelayK<V>::K;
        rper = delay_per(D.m + 1, D.G);
        cper = delay_per(D.n, D.G);
        rb = min(D.m + 1, D.bt * rper);
        nr = min(D.m + 1, rb + rper) - rb;
        cb = min(D.n, D.bt * cper);
        nc = min(D.n, cb + cper) - cb;
        own = delay_own_bytes<V>(D.m, D.n, D.G, pass_bytes) <= D.smem;
        V* keep = reinterpret_cast<V*>(smem + delay_own_offset<V>(D.m, D.n, D.G, pass_bytes));
        fo = own ? reinterpret_cast<V*>(smem) : D.Fh + (size_t)rb * K;
        ro = own ? reinterpret_cast<V*>(smem) + (size_t)rper * K : D.RhT + (size_t)cb * K;
        rhs = own ? keep : D.rhs + rb;
        obj = own ? keep + rper : D.T + cb;
        var = own ? reinterpret_cast<int*>(keep + rper + cper) : D.var + cb;
        sf = reinterpret_cast<V*>(smem);
        sr = sf + (size_t)rper * K;
        fu = own ? rper : 1;
        fr = own ? 1 : K;
        ru = own ? cper : 1;
        rr = own ? 1 : K;
    }
    // the chains of row i (the block's) and of column j; the shared-memory
    // case apart, so that its loads are shared-memory loads
    __device__ __forceinline__ V row_chain(int i, const V* other, int k, V t) const {
        constexpr int K = DelayK<V>::K;
        return own ? delay_chain<K>(sf + i, rper, other, k, t) : delay_chain<K>(fo + (size_t)i * K, 1, other, k, t);
    }
    __device__ __forceinline__ V column_chain(int j, const V* other, int k, V t) const {
        constexpr int K = DelayK<V>::K;
        return own ? delay_chain<K>(sr + j, cper, other, k, t) : delay_chain<K>(ro + (size_t)j * K, 1, other, k, t);
    }
};

// The block's own parts, the padding of the pending rows, and the first Step 1.
template <int NT, typename V>
__device__ __forceinline__ void delay_begin(const Delayed<V>& D, unsigned char* smem, size_t pass_bytes, DelayScratch& s,
                                         DelayState& S) {
    constexpr int K = DelayK<V>::K;
    const int t = threadIdx.x, n = D.n, bland = D.rule == 1 ? 1 : 0;
    const size_t ld = (size_t)D.ld;
    const DelayOwn<V> B(D, smem, pass_bytes);
    if (D.bt == 0)
        for (int e = t; e < K * (D.ld - n); e += NT)
            __stcg(D.Rh + (size_t)(e / (D.ld - n)) * ld + n + e % (D.ld - n), V(0));
    for (int i = t; i < B.nr; i += NT) B.rhs[i] = __ldcg(D.T + (size_t)(B.rb + i) * ld + n);
    DelayCand c = delay_none(), e;
    for (int j = t; j < B.nc; j += NT) {
        const V x = __ldcg(D.T + B.cb + j);
        const int v = __ldcg(D.var + B.cb + j);
        B.obj[j] = x;
        B.var[j] = v;
        if (x < -D.eps_d) delay_merge(c, DelayCand{delay_key(x), v, B.cb + j}, bland);
    }
    int nf = 0;
    delay_send<NT>(D, D.arg, c, 0, B.cb, B.nc, bland, s);
    const bool ok = delay_gather<NT>(D, D.arg, B.cper, bland, e, nf, s);
    if (t == 0) {
        S.status = !ok ? kDelayFailed : e.key == INT_MAX ? kOptimal : D.max_iters <= 0 ? kIterLimit : kRunning;
        S.bland = bland;
        S.degen = 0;
        S.k = 0;
        S.last = 0;
        S.flag = 0;
        S.passes = 0;
        S.it = 0;
        S.ehi = e.hi;
        S.ekey = e.key;
        S.eidx = e.idx;
    }
    __syncthreads();
}

// A round: pivots from S's entering candidate on until K are pending, one has
// met a non-finite entry, or the solve ends.
template <int NT, typename V, typename Clock>
__device__ __forceinline__ void delay_round(const Delayed<V>& D, unsigned char* smem, size_t pass_bytes, DelayScratch& s,
                                         DelayState& S, Clock& clk) {
    constexpr int K = DelayK<V>::K;
    static_assert(K <= NT && K % 4 == 0, "one thread per pending pivot, chains by four");
    __shared__ __align__(16) V other[K];   // the broadcast factors of a chain
    const int t = threadIdx.x;
    const size_t ld = (size_t)D.ld;
    const DelayOwn<V> B(D, smem, pass_bytes);
    const int rb = B.rb, nr = B.nr, cb = B.cb, nc = B.nc;
    int status = kRunning, bland = S.bland, degen = S.degen, k = 0, last = 0, flag = 0;
    long long it = S.it;
    DelayCand e{S.ehi, S.ekey, S.eidx};
    while (status == kRunning) {
        // Step 2: the block's rows of column q, up to date; ratios.  The loads
        // that need q are issued together.
        const int q = e.idx, qv = e.key;
        const V f0 = delay_value<V>(e.hi);   // the objective-row entry of column q
        V a = V(0);
        if (t < nr) a = __ldcg(D.T + (size_t)(rb + t) * ld + q);
        if (t < k) other[t] = __ldcg(D.RhT + (size_t)q * K + t);
        __syncthreads();
        DelayCand c = delay_none();
        int nf = 0;
#pragma unroll 1
        for (int i = t; i < nr; i += NT) {
            const int row = rb + i;
            if (i != t) a = __ldcg(D.T + (size_t)row * ld + q);
            a = row == 0 ? f0 : B.row_chain(i, other, k, a);
            __stcg(D.Fh + (size_t)row * K + k, a);
            if (B.own) B.fo[(size_t)k * B.fu + i] = a;
            nf |= !delay_finite(a);
            if (row > 0 && a > D.eps_p) {
                const V r = div_rn(B.rhs[i], a);
                const int key = bland ? __ldcg(D.basis + (row - 1)) : row;
                if (!delay_nan(r)) delay_merge(c, DelayCand{delay_key(r), key, row});
            }
        }
        delay_send<NT>(D, D.rat, c, nf, rb, nr, 0, s);
        clk.lap(0);
        DelayCand l;
        if (!delay_gather<NT>(D, D.rat, B.rper, 0, l, nf, s)) { status = kDelayFailed; break; }
        clk.lap(3);
        flag |= nf;
        const int p = l.idx;
        const V theta = delay_value<V>(l.hi);
        if (l.key == INT_MAX) { status = kUnbounded; break; }
        if (!delay_finite(theta)) { status = kNumeric; break; }
        // Step 3, row p: the block's columns up to date, scaled; the objective row
        V* rowp = D.T + (size_t)p * ld + cb;
        V x = V(0);
        if (t < nc) x = __ldcg(rowp + t);
        if (t < k) other[t] = __ldcg(D.Fh + (size_t)p * K + t);
        const V piv = __ldcg(D.Fh + (size_t)p * K + k);
        const int jq = q - cb;   // column q among the block's
        int leaving = 0;
        if (jq >= 0 && jq < nc && t == jq % NT) leaving = __ldcg(D.basis + (p - 1));
        __syncthreads();
        if (!delay_finite(piv)) { status = kNumeric; break; }
        if (jq >= 0 && jq < nc && t < k) {   // the pending entries of column q, which starts from zero
            __stcg(D.Rh + (size_t)t * ld + q, V(0));
            __stcg(D.RhT + (size_t)q * K + t, V(0));
            if (B.own) B.ro[(size_t)t * B.ru + jq] = V(0);
        }
        // the cycling guard decides the rule of the next Step 1
        if (D.rule == 0) {
            if (theta <= V(0)) {
                ++degen;
                if (D.k_cyc > 0 && degen >= D.k_cyc) bland = 1;
            } else {
                degen = 0;
                bland = 0;
            }
        }
        c = delay_none();
        nf = 0;
#pragma unroll 1
        for (int j = t; j < nc; j += NT) {
            if (j != t) x = __ldcg(rowp + j);
            V ob = B.obj[j];
            if (j == jq) {   // the leaving variable's unit column
                x = V(1);
                ob = V(0);
                B.var[j] = leaving;
                D.var[q] = leaving;
            } else {
                x = B.column_chain(j, other, k, x);
            }
            const V rj = div_rn(x, piv);
            nf |= !delay_finite(rj);
            __stcg(rowp + j, rj);
            __stcg(D.RhT + (size_t)(cb + j) * K + k, rj);
            __stcg(D.Rh + (size_t)k * ld + cb + j, rj);
            if (B.own) B.ro[(size_t)k * B.ru + j] = rj;
            ob = fma_rn(-f0, rj, ob);
            B.obj[j] = ob;
            if (ob < -D.eps_d) delay_merge(c, DelayCand{delay_key(ob), B.var[j], cb + j}, bland);
        }
        delay_send<NT>(D, D.arg, c, nf, cb, nc, bland, s);
        clk.lap(1);
        // The block's rows, while the candidates travel (visible to the others
        // with the next send): right-hand side; column q starts from zero.
#pragma unroll 1
        for (int i = t; i < nr; i += NT) {
            const int row = rb + i;
            if (row == p) {
                B.rhs[i] = theta;
            } else {
                const V f = B.own ? B.fo[(size_t)k * B.fu + i] : __ldcg(D.Fh + (size_t)row * K + k);
                B.rhs[i] = fma_rn(-f, theta, B.rhs[i]);
                if (row > 0) __stcg(D.T + (size_t)row * ld + q, V(0));
            }
        }
        if (D.bt == 0 && t == 0 && it < D.log_cap) {
            D.qlog[it] = qv;
            D.plog[it] = p;
        }
        last = p;
        ++k;
        ++it;
        if (!delay_gather<NT>(D, D.arg, B.cper, bland, e, nf, s)) { status = kDelayFailed; break; }   // Step 1
        clk.lap(4);
        flag |= nf;
        if (p >= rb && p < rb + nr) {
            // row p, whose multipliers no block reads any more: its chain starts from R
            if (t < k) {
                __stcg(D.Fh + (size_t)p * K + t, V(0));
                if (B.own) B.fo[(size_t)t * B.fu + (p - rb)] = V(0);
            }
            if (t == 0) __stcg(D.basis + (p - 1), qv);
        }
        if (e.key == INT_MAX)
            status = kOptimal;
        else if (it >= D.max_iters)
            status = kIterLimit;
        else if (k == K || flag)
            break;
    }
    if (t == 0) {
        S.status = status;
        S.bland = bland;
        S.degen = degen;
        S.k = k;
        S.last = last;
        S.flag = flag;
        S.it = it;
        S.ehi = e.hi;
        S.ekey = e.key;
        S.eidx = e.idx;
    }
    __syncthreads();
}

// Steps 1-3 from a built tableau until termination, by D.G blocks.  The
// tableau, basis and var[] are complete when the blocks have returned (the
// caller orders later reads after a barrier or the launch).  D, s, S and clk
// are in shared memory; s.passed is set by the caller.
// clk: work of {Steps 1-2, row p and the objective row, the passes}, then the
// wait after each.
template <int NT, int RS, bool AHEAD = false, typename V, typename Clock>
__device__ __forceinline__ void delayed_solve(const Delayed<V>& D, unsigned char* smem, DelayScratch& s, DelayState& S,
                                              Clock& clk) {
    const size_t pass_bytes = delay_smem_bytes<V>(NT, RS);
    delay_begin<NT>(D, smem, pass_bytes, s, S);
    clk.lap(0);
    while (S.status == kRunning) {
        delay_round<NT>(D, smem, pass_bytes, s, S, clk);
        if (S.status == kDelayFailed) return;
        const int k = S.k;
        if (k > 0) {   // the pending updates applied to the whole tableau, between two barriers
            if (!delay_barrier<NT>(D, s)) break;
            const int rev = (int)(S.passes & 1u);
            delay_pass<NT, RS, AHEAD, DelayK<V>::K>(D, D.T, D.T, D.Fh, D.Rh, k, rev, smem, s);
            clk.lap(2);
            if (!delay_barrier<NT>(D, s)) break;
            if (S.flag) {   // 0 x inf in row p: the row again
                const int cper = delay_per(D.n, D.G), c1 = min(D.n, D.bt * cper + cper);
                for (int j = D.bt * cper + threadIdx.x; j < c1; j += NT)
                    __stcg(D.T + (size_t)S.last * (size_t)D.ld + j, __ldcg(D.Rh + (size_t)(k - 1) * (size_t)D.ld + j));
                if (!delay_barrier<NT>(D, s)) break;
            }
            if (threadIdx.x == 0) ++S.passes;
            __syncthreads();
            clk.lap(5);
        }
    }
    if (s.fail) {
        __syncthreads();
        if (threadIdx.x == 0) S.status = kDelayFailed;
        __syncthreads();
        return;
    }
    // the stored right-hand side and objective row
    const DelayOwn<V> B(D, smem, pass_bytes);
    for (int i = threadIdx.x; i < B.nr; i += NT) __stcg(D.T + (size_t)(B.rb + i) * (size_t)D.ld + D.n, B.rhs[i]);
    if (B.own)
        for (int j = threadIdx.x; j < B.nc; j += NT) __stcg(D.T + B.cb + j, B.obj[j]);
}

}  // namespace tsx
