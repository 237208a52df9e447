// Delayed updates with the pass behind the pivots: while the pass of one round
// runs, the next round's pivots go on.
//
// In tsx_delayed.cuh a round's pivots and its pass take turns; a pivot is a chain
// of latencies (6.5-8.5 us, the pipes idle), the pass is bound by them.  Here a
// block has two groups of warps: kOverFg threads run the pivots, the others the
// pass of the previous round, which reads one copy of the tableau and writes
// another, so that the pivots can read the first one meanwhile.  An entry that a
// pivot needs takes the previous round's chain and then the current one's, the
// same fused multiply-adds in the same order.  What a pivot replaces (row p by R,
// column q from zero) is not stored at once, as the copies change: the round
// remembers it (chains of such rows and columns start there) and the copy the
// next pass reads gets it at the end of the round, between two grid barriers.
//
// Measured, in turn -> overlapped, us a pivot: FP64 2049x1531 13.8 -> 11.3,
// 4096^2 36.1 -> 29.3, 8192^2 117.9 -> 111.3 (the fused multiply-adds alone
// 107.2; the FP64 pipe is busy with the pass, so a pivot's own chains take twice
// as long), FP32 12288^2 16.4 -> 12.2.
#pragma once

#include "tsx_delayed.cuh"
#include "tsx_kernels.cuh"

namespace tsx {

// Pivots per round: the chains take up to two rounds (FP64 steps are ~80
// cycles, so fewer), the pass one read and write of the tableau per round.
template <typename V> struct OverK;
template <> struct OverK<double> { static constexpr int K = 8; };
template <> struct OverK<float> { static constexpr int K = 32; };

constexpr int kOverFg = 128;               // threads of the pivots
constexpr int kOverNt = 512;               // threads of a block (128 registers each)
constexpr int kOverBg = kOverNt - kOverFg; // threads of the pass
constexpr int kOverRows = 4;               // rows of its tiles (the next tile's loads in flight)
constexpr int kBarFg = 1, kBarBg = 2, kBarStart = 3, kBarDone = 4;   // named barriers

template <typename V>
struct Overlap {             // one LP; D.T is the copy the pivots read
    Delayed<V> D;            // D.Fh, D.Rh, D.RhT: two rounds' buffers each
    V* other;                // the other copy
};

// Work for the pass, from the pivots' threads of the same block.
template <typename V>
struct OverCmd {
    int k;                   // pending pivots; 0: leave
    int rev;
    const V* from;
    V* to;
    const V *Fh, *Rh;
};

// Shared memory of a block: the pass's staging, then the pending entries of its
// rows and columns for two rounds, then its right-hand sides, objective-row
// entries, variables, and the pivot of this round that replaced each of its
// rows and columns (-1: none).
template <typename V>
__host__ __device__ constexpr size_t over_pass_bytes() {
    return (size_t)kDelayStrips * OverK<V>::K * 1024 + (size_t)(kOverBg / 32) * OverK<V>::K * (kOverRows * 8 + 16);
}
template <typename V>
__host__ __device__ constexpr size_t over_bytes(int m, int n, int blocks) {
    const size_t rper = delay_per(m + 1, blocks), cper = delay_per(n, blocks);
    return over_pass_bytes<V>() + 2 * (rper + cper) * OverK<V>::K * sizeof(V) + rper * (sizeof(V) + 4) +
           cper * (sizeof(V) + 8) + 16;
}

template <typename V>
struct OverOwn {
    int rper, cper, rb, nr, cb, nc;
    V *f, *r;                // pending entries of round parity 0; the other K x rper (cper) on
    V *rhs, *obj;
    int *var, *rlast, *clast;
    __device__ __forceinline__ OverOwn(const Delayed<V>& D, unsigned char* smem) {
        constexpr int K = OverK<V>::K;
        rper = delay_per(D.m + 1, D.G);
        cper = delay_per(D.n, D.G);
        rb = min(D.m + 1, D.bt * rper);
        nr = min(D.m + 1, rb + rper) - rb;
        cb = min(D.n, D.bt * cper);
        nc = min(D.n, cb + cper) - cb;
        f = reinterpret_cast<V*>(smem + over_pass_bytes<V>());
        r = f + 2 * (size_t)K * rper;
        rhs = r + 2 * (size_t)K * cper;
        obj = rhs + rper;
        var = reinterpret_cast<int*>(obj + cper);
        rlast = var + cper;
        clast = rlast + rper;
    }
};

template <typename V>
struct OverShared {
    DelayScratch ds;
    Delayed<V> D;
    V* other;
    OverCmd<V> cmd;
    __align__(16) V cur[OverK<V>::K], prev[OverK<V>::K];   // broadcast factors of a chain
    int plist[OverK<V>::K], qlist[OverK<V>::K];            // rows and columns of this round's pivots
    unsigned hit;                                          // which of them are the chain's row or column
};

// t through the pending pivots u0 .. k - 1.
template <int K, typename V>
__device__ __forceinline__ V over_chain(const V* own, int step, const V* other, int u0, int k, V t) {
    if (u0 == 0) return delay_chain<K>(own, step, other, k, t);
#pragma unroll 1
    for (int u = u0; u < k; ++u) t = fma_rn(-own[u * step], other[u], t);
    return t;
}

// The pass starts: the block's pivots' threads hand over and go on.
template <typename V>
__device__ __forceinline__ void over_start(OverShared<V>& s, int k, int rev, const V* from, V* to, const V* Fh,
                                           const V* Rh) {
    if (threadIdx.x == 0) s.cmd = OverCmd<V>{k, rev, from, to, Fh, Rh};
    __threadfence_block();
    asm volatile("bar.arrive %0, %1;" ::"n"(kBarStart), "n"(kOverNt) : "memory");
}
__device__ __forceinline__ void over_wait_pass() {
    asm volatile("bar.sync %0, %1;" ::"n"(kBarDone), "n"(kOverNt) : "memory");
}

// The pivots, by threads 0 .. kOverFg - 1 of each block.  Returns the copy that
// holds the final tableau (0: D.T as given, 1: the other), -1 if a wait ran out.
template <typename V, typename Clock>
__device__ int over_pivots(OverShared<V>& s, unsigned char* smem, DelayState& S, Clock& clk) {
    constexpr int K = OverK<V>::K, NT = kOverFg;
    static_assert(K <= 32 && K % 4 == 0, "one lane of warp 0 per pending pivot, chains by four");
    const Delayed<V>& D = s.D;
    const int t = threadIdx.x, m = D.m, n = D.n;
    const size_t ld = (size_t)D.ld;
    const OverOwn<V> B(D, smem);
    const int rb = B.rb, nr = B.nr, cb = B.cb, nc = B.nc;
    const V* T = D.T;          // read by the pivots (and by the running pass)
    int which = 0, par = 0;    // the copy T is; parity of the round
    int kprev = 0;             // pivots of the previous round, 0 or K (its pass is running)
    int bland = D.rule == 1 ? 1 : 0, degen = 0, status = kRunning;
    unsigned passes = 0;
    long long it = 0;
    // the block's own parts, the padding of the pending rows, the first Step 1
    if (D.bt == 0)
        for (int e = t; e < 2 * K * (D.ld - n); e += NT)
            __stcg(D.Rh + (size_t)(e / (D.ld - n)) * ld + n + e % (D.ld - n), V(0));
    for (int i = t; i < nr; i += NT) {
        B.rhs[i] = __ldcg(T + (size_t)(rb + i) * ld + n);
        B.rlast[i] = -1;
    }
    DelayCand c = delay_none(), e;
    int nf = 0;
    for (int j = t; j < nc; j += NT) {
        const V x = __ldcg(T + cb + j);
        const int v = __ldcg(D.var + cb + j);
        B.obj[j] = x;
        B.var[j] = v;
        B.clast[j] = -1;
        if (x < -D.eps_d) delay_merge(c, DelayCand{delay_key(x), v, cb + j}, bland);
    }
    delay_send<NT, kBarFg>(D, D.arg, c, 0, cb, nc, bland, s.ds);
    if (!delay_gather<NT, kBarFg>(D, D.arg, B.cper, bland, e, nf, s.ds)) return -1;
    if (e.key == INT_MAX)
        status = kOptimal;
    else if (D.max_iters <= 0)
        status = kIterLimit;
    clk.lap(0);
    while (status == kRunning) {
        // ---- a round, as in delay_round
        V* Fh = D.Fh + (size_t)par * (size_t)(m + 1) * K;
        V* Rh = D.Rh + (size_t)par * K * ld;
        V* RhT = D.RhT + (size_t)par * K * ld;
        const V* Fp = D.Fh + (size_t)(1 - par) * (size_t)(m + 1) * K;
        const V* RpT = D.RhT + (size_t)(1 - par) * K * ld;
        V *fc = B.f + (size_t)par * K * B.rper, *rc = B.r + (size_t)par * K * B.cper;
        const V *fp = B.f + (size_t)(1 - par) * K * B.rper, *rp = B.r + (size_t)(1 - par) * K * B.cper;
        int k = 0, flag = 0;
        while (status == kRunning) {
            // Step 2
            const int q = e.idx, qv = e.key;
            const V f0 = delay_value<V>(e.hi);
            V a = V(0);
            if (t < nr) a = __ldcg(T + (size_t)(rb + t) * ld + q);
            if (t < 32) {
                if (t < k) s.cur[t] = __ldcg(RhT + (size_t)q * K + t);
                const unsigned hit = __ballot_sync(0xffffffffu, t < k && s.qlist[t] == q);
                if (t == 0) s.hit = hit;
            } else if (t < 64 && t - 32 < kprev) {
                s.prev[t - 32] = __ldcg(RpT + (size_t)q * K + t - 32);
            }
            delay_sync<kBarFg, NT>();
            const unsigned qhit = s.hit;
            c = delay_none();
            nf = 0;
#pragma unroll 1
            for (int i = t; i < nr; i += NT) {
                const int row = rb + i, u = B.rlast[i];
                if (i != t) a = __ldcg(T + (size_t)row * ld + q);
                if (row == 0) {
                    a = f0;
                } else if (u >= 0) {   // replaced by the row of pivot u
                    a = over_chain<K>(fc + i, B.rper, s.cur, u + 1, k, s.cur[u]);
                } else if (qhit) {     // column q started from zero at that pivot
                    a = over_chain<K>(fc + i, B.rper, s.cur, 31 - __clz((int)qhit), k, V(0));
                } else {
                    if (kprev) a = delay_chain_all<K>(fp + i, B.rper, s.prev, a);
                    a = delay_chain<K>(fc + i, B.rper, s.cur, k, a);
                }
                __stcg(Fh + (size_t)row * K + k, a);
                fc[k * B.rper + i] = a;
                nf |= !delay_finite(a);
                if (row > 0 && a > D.eps_p) {
                    const V r = div_rn(B.rhs[i], a);
                    const int key = bland ? __ldcg(D.basis + (row - 1)) : row;
                    if (!delay_nan(r)) delay_merge(c, DelayCand{delay_key(r), key, row});
                }
            }
            delay_send<NT, kBarFg>(D, D.rat, c, nf, rb, nr, 0, s.ds);
            clk.lap(0);
            DelayCand l;
            if (!delay_gather<NT, kBarFg>(D, D.rat, B.rper, 0, l, nf, s.ds)) { status = kDelayFailed; break; }
            clk.lap(3);
            flag |= nf;
            const int p = l.idx;
            const V theta = delay_value<V>(l.hi);
            if (l.key == INT_MAX) { status = kUnbounded; break; }
            if (!delay_finite(theta)) { status = kNumeric; break; }
            // Step 3, row p and the objective row
            const V* rowp = T + (size_t)p * ld + cb;
            V x = V(0);
            if (t < nc) x = __ldcg(rowp + t);
            const V piv = __ldcg(Fh + (size_t)p * K + k);
            if (t < 32) {
                if (t < k) s.cur[t] = __ldcg(Fh + (size_t)p * K + t);
                const unsigned hit = __ballot_sync(0xffffffffu, t < k && s.plist[t] == p);
                if (t == 0) s.hit = hit;
            } else if (t < 64 && t - 32 < kprev) {
                s.prev[t - 32] = __ldcg(Fp + (size_t)p * K + t - 32);
            }
            const int jq = q - cb;   // column q among the block's
            int leaving = 0;
            if (jq >= 0 && jq < nc && t == jq % NT) leaving = __ldcg(D.basis + (p - 1));
            delay_sync<kBarFg, NT>();
            if (!delay_finite(piv)) { status = kNumeric; break; }
            const unsigned phit = s.hit;
            if (jq >= 0 && jq < nc && t < k) {   // the pending entries of column q, which starts from zero
                __stcg(Rh + (size_t)t * ld + q, V(0));
                __stcg(RhT + (size_t)q * K + t, V(0));
                rc[t * B.cper + jq] = V(0);
            }
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
                    B.clast[j] = k;
                } else if (phit) {   // row p is the row of that pivot
                    const int u = 31 - __clz((int)phit);
                    x = over_chain<K>(rc + j, B.cper, s.cur, u + 1, k, rc[u * B.cper + j]);
                } else if (B.clast[j] >= 0) {
                    x = over_chain<K>(rc + j, B.cper, s.cur, B.clast[j], k, V(0));
                } else {
                    if (kprev) x = delay_chain_all<K>(rp + j, B.cper, s.prev, x);
                    x = delay_chain<K>(rc + j, B.cper, s.cur, k, x);
                }
                const V rj = div_rn(x, piv);
                nf |= !delay_finite(rj);
                __stcg(RhT + (size_t)(cb + j) * K + k, rj);
                __stcg(Rh + (size_t)k * ld + cb + j, rj);
                rc[k * B.cper + j] = rj;
                ob = fma_rn(-f0, rj, ob);
                B.obj[j] = ob;
                if (ob < -D.eps_d) delay_merge(c, DelayCand{delay_key(ob), B.var[j], cb + j}, bland);
            }
            if (t == 0) {
                s.plist[k] = p;
                s.qlist[k] = q;
            }
            delay_send<NT, kBarFg>(D, D.arg, c, nf, cb, nc, bland, s.ds);
            clk.lap(1);
#pragma unroll 1
            for (int i = t; i < nr; i += NT) {
                if (rb + i == p) {
                    B.rhs[i] = theta;
                    B.rlast[i] = k;
                } else {
                    B.rhs[i] = fma_rn(-fc[k * B.rper + i], theta, B.rhs[i]);
                }
            }
            if (D.bt == 0 && t == 0 && it < D.log_cap) {
                D.qlog[it] = qv;
                D.plog[it] = p;
            }
            ++k;
            ++it;
            if (!delay_gather<NT, kBarFg>(D, D.arg, B.cper, bland, e, nf, s.ds)) { status = kDelayFailed; break; }
            clk.lap(4);
            flag |= nf;
            if (p >= rb && p < rb + nr) {   // row p's multipliers, which no block reads any more
                if (t < k) {
                    __stcg(Fh + (size_t)p * K + t, V(0));
                    fc[t * B.rper + (p - rb)] = V(0);
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
        // ---- the end of the round: the previous pass is done everywhere, its
        // copy takes this round's rows and columns, this round's pass starts
        if (kprev) {
            over_wait_pass();
            if (status == kDelayFailed) return -1;
            clk.lap(2);
            if (!delay_barrier<NT, kBarFg>(D, s.ds)) return -1;
            which ^= 1;
            T = which ? s.other : D.T;
            kprev = 0;
        } else {
            if (status == kDelayFailed) return -1;
            if (k > 0 && !delay_barrier<NT, kBarFg>(D, s.ds)) return -1;   // no block reads T any more
        }
        if (k == 0) break;
        V* Tw = which ? s.other : D.T;
        for (int z = t; z < nr * k; z += NT) {
            const int i = z / k, u = z - i * k;
            if (rb + i > 0 && B.rlast[i] < 0) __stcg(Tw + (size_t)(rb + i) * ld + s.qlist[u], V(0));
        }
        for (int u = 0; u < k; ++u) {
            bool last = true;
            for (int v = u + 1; v < k; ++v) last = last && s.plist[v] != s.plist[u];
            if (!last) continue;
            for (int j = t; j < nc; j += NT) __stcg(Tw + (size_t)s.plist[u] * ld + cb + j, rc[u * B.cper + j]);
        }
        if (!delay_barrier<NT, kBarFg>(D, s.ds)) return -1;
        const int prow = s.plist[k - 1];
        for (int i = t; i < nr; i += NT) B.rlast[i] = -1;
        for (int j = t; j < nc; j += NT) B.clast[j] = -1;
        over_start<V>(s, k, (int)(passes & 1u), Tw, which ? D.T : s.other, Fh, Rh);
        ++passes;
        kprev = k;
        par ^= 1;
        if (status != kRunning || flag) {   // the last pass, or one whose row p needs another store
            over_wait_pass();
            if (!delay_barrier<NT, kBarFg>(D, s.ds)) return -1;
            which ^= 1;
            T = which ? s.other : D.T;
            kprev = 0;
            if (flag) {
                V* to = which ? s.other : D.T;
                for (int j = t; j < nc; j += NT) __stcg(to + (size_t)prow * ld + cb + j, rc[(k - 1) * B.cper + j]);
                if (!delay_barrier<NT, kBarFg>(D, s.ds)) return -1;
            }
        }
        clk.lap(5);
    }
    // the stored right-hand side and objective row
    V* Tf = which ? s.other : D.T;
    for (int i = t; i < nr; i += NT) __stcg(Tf + (size_t)(rb + i) * ld + n, B.rhs[i]);
    for (int j = t; j < nc; j += NT) __stcg(Tf + cb + j, B.obj[j]);
    if (t == 0) {
        S.status = status;
        S.bland = bland;
        S.degen = degen;
        S.it = it;
        S.passes = passes;
    }
    return which;
}

// One cooperative launch per solve; *copy receives the copy (0 or 1) that holds
// the final tableau.
template <typename V>
__global__ void __launch_bounds__(kOverNt, 1) k_pivot_overlap(Overlap<V> P, double eps_d, double eps_p,
                                                              DevState* st) {
    extern __shared__ __align__(128) unsigned char tsx_dyn[];
    __shared__ OverShared<V> s;
    __shared__ DelayState S;
    __shared__ PhaseClock clk;
    if (threadIdx.x == 0) {
        s.D = P.D;
        s.D.bt = blockIdx.x;
        s.D.G = gridDim.x;
        delay_eps(eps_d, s.D.eps_d);
        delay_eps(eps_p, s.D.eps_p);
        s.other = P.other;
        s.ds.passed = 0;
    }
    __syncthreads();
    if (threadIdx.x < kOverFg) {
        clk.start();
        const int which = over_pivots<V>(s, tsx_dyn, S, clk);
        // the pass's threads leave (none is running: every start has been waited for,
        // or the pivots gave up after its end)
        over_start<V>(s, 0, 0, nullptr, nullptr, nullptr, nullptr);
        if (blockIdx.x == 0 && threadIdx.x == 0 && which >= 0) {
            atomicCAS(&st->status, kRunning, S.status);
            st->iters = S.it;
            st->bland = S.bland;
            st->degen_run = S.degen;
            st->passes = S.passes;
            st->copy = which;
            for (int k = 0; k < 6; ++k) st->phase_ns[k] = clk.acc[k];
        }
    } else {
        for (;;) {
            asm volatile("bar.sync %0, %1;" ::"n"(kBarStart), "n"(kOverNt) : "memory");
            const OverCmd<V> c = s.cmd;
            if (c.k == 0) break;
            delay_pass<kOverBg, kOverRows, true, OverK<V>::K, kBarBg, kOverFg>(s.D, c.from, c.to, c.Fh, c.Rh, c.k, c.rev,
                                                                              tsx_dyn, s.ds);
            asm volatile("bar.arrive %0, %1;" ::"n"(kBarDone), "n"(kOverNt) : "memory");
        }
    }
}

}  // namespace tsx
