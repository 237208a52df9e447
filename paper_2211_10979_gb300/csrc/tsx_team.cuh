// Team solve: many LPs at once, each by a team of C thread blocks (the
// full-tableau simplex of arXiv 2211.10979, Section III, Steps 1-3), for LPs
// too large for one block's shared memory and too small to fill the GPU.
//
// One cooperative launch holds every team; a team takes the next LP from a
// list (largest first), builds its condensed tableau in global memory, a range
// of rows per block, and solves it with delayed updates (tsx_delayed.cuh): its
// blocks are the blocks of one delayed solve, so that the updates of up to 16
// (FP32: 32) pivots share one pass over the tableau.  The arithmetic and the
// tie rules are those of the single-LP kernels, so every pivot and value equals
// lp_solve's.  Measured against one update per pivot (bound by HBM, 0.86 of
// it): 96 FP64 LPs with m, n log-uniform in [180, 3000] 114 -> 85 ms a call (67-79
// with the largest solved on the whole grid), a burst of 200
// FP32 requests with m, n in [32, 4096] 201 -> 71 ms.
#pragma once

#include "tsx_delayed.cuh"
#include "tsx_device.cuh"

namespace tsx {

constexpr int kTeamMax = 160;  // blocks per team, upper bound
#ifndef TSX_TEAM_SM_THREADS
#define TSX_TEAM_SM_THREADS 512   // threads per SM the team kernel is compiled for
#endif
// Threads per SM of the team kernel with blocks of nt threads, and the rows of
// a warp's update tile.
__host__ __device__ constexpr int team_sm_threads(int nt) { return nt > TSX_TEAM_SM_THREADS ? nt : TSX_TEAM_SM_THREADS; }
constexpr int kTeamRows = 8;

template <typename V>
struct TeamJob {
    const double* A;           // inputs (device), m x n row-major, m, n
    const double* b;
    const double* c;
    V* T;                      // condensed tableau (m+1) x ld
    int* basis;                // m
    int* var;                  // n
    DevState* st;              // the LP's state words: status, iters, bland, degen_run, passes
    V* Fh;                     // buffers of the delayed updates
    V* Rh;
    V* RhT;
    V* rhs;
    int m, n, ld;
    int pad;
};

struct __align__(256) TeamState {   // one per team
    unsigned bar_count;
    unsigned bar_gen;
    int job;
    int fail;                  // set when a team barrier wait ran out
    int bad;                   // the current LP's inputs are not finite or b < 0
    unsigned seq;              // continuous launch: sequence number of the job
    unsigned delay_count;      // arrivals of the delayed solve's exchanges and barriers
    DelayRec arg[kTeamMax];    // entering candidate of each block
    DelayRec rat[kTeamMax];    // leaving candidate of each block
};

template <typename V>
struct TeamParams {
    const TeamJob<V>* jobs;
    const int* order[2];       // job indices of the two lists, largest first
    int count[2];              // their lengths
    unsigned* next;            // list position counters (2); [1] starts behind the wide teams' first LPs
    TeamState* teams;
    const int* team_of;        // grid: the team of each block
    const int* first;          // teams: first block, size, own list (0 or 1)
    const int* size;
    const int* list;
    double eps_d, eps_p;
    long long max_iters;       // < 0: 50 (m + n)
    int k_cyc, rule;
    long long timeout_ns;
};

// Barrier of the C blocks of one team; bounded like grid_barrier.  Returns
// false (in every thread) if the wait ran out or another block of the team
// gave up.
// With TSX_BARRIER_COUNT the arrival counter only grows within a launch (the
// team states are zeroed before it): a block adds 1 (release, no returned
// value) and waits for (barriers passed + 1) x C, `passed` counting its own
// barriers; otherwise the last arrival resets the counter and bumps a
// generation word.
__device__ inline bool team_barrier(TeamState* ts, unsigned C, long long timeout_ns, int& sok, unsigned& passed) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        bool done = false;
        unsigned gen = 0, target = 0;
        if (TSX_BARRIER_COUNT) {
            target = (passed + 1u) * C;
            red_add_release(&ts->bar_count, 1u);
        } else {
            gen = ld_acquire(&ts->bar_gen);
            const unsigned arrived = atom_add_acq_rel(&ts->bar_count, 1u);
            if (arrived == C - 1) {
                ts->bar_count = 0;
                st_release(&ts->bar_gen, gen + 1);
                done = true;
            }
        }
        if (!done) {
            const long long t0 = global_ns();
            const unsigned long long max_spins = (unsigned long long)(timeout_ns > 0 ? timeout_ns : 0) + 4096ull;
            unsigned long long spins = 0;
            while (TSX_BARRIER_COUNT ? (int)(ld_acquire(&ts->bar_count) - target) < 0
                                     : ld_acquire(&ts->bar_gen) == gen) {
                ++spins;
                if ((spins & 31ull) == 1) {
                    if (ld_relaxed(&ts->fail) != 0) { ok = 0; break; }
                    if (global_ns() - t0 >= timeout_ns || spins > max_spins) {
                        atomicExch(&ts->fail, 1);
                        ok = 0;
                        break;
                    }
                }
            }
        }
        passed += 1u;
        __threadfence();
        sok = ok;
    }
    __syncthreads();
    return sok != 0;
}

// Rows of block bt among C: [r0, r1) of 0..m.
__device__ __forceinline__ void team_rows(int m, int C, int bt, int& r0, int& r1) {
    const int per = (m + 1 + C - 1) / C;
    r0 = min(m + 1, bt * per);
    r1 = min(m + 1, r0 + per);
}

// Condensed Table I rows [r0, r1) (slack basis): row 0 = [-c | 0], row i =
// [A_i | b_i], padding zero; the LP's basis words of those rows; var[] by block
// 0.  Inputs that are not finite, or b_i < 0, mark the LP bad in the team state
// (the input check of lp_create, done while the data pass by).
template <typename V>
__device__ void team_build(const TeamJob<V>& J, int r0, int r1, int bt, TeamState* ts) {
    constexpr int E = Lanes<V>::E;
    const int n = J.n, ld = J.ld;
    const long long per_row = ld / E;
    const long long total = (long long)(r1 - r0) * per_row;
    int bad = 0;
    for (long long g = threadIdx.x; g < total; g += blockDim.x) {
        const int i = r0 + (int)(g / per_row);
        const int j0 = (int)(g - (long long)(i - r0) * per_row) * E;
        Sector<V> out;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int j = j0 + e;
            double v = 0.0;
            if (i == 0) {
                if (j < n) v = -J.c[j];
            } else if (j < n) {
                v = J.A[(size_t)(i - 1) * (size_t)n + j];
            } else if (j == n) {
                v = J.b[i - 1];
                bad |= !(v >= 0.0);
            }
            bad |= !isfinite(v);
            out.v[e] = (V)v;
        }
        st_sector(J.T + (size_t)i * (size_t)ld + j0, out);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&ts->bad, 1);
    for (int i = max(r0, 1) + threadIdx.x; i < r1; i += blockDim.x) J.basis[i - 1] = n + i - 1;
    if (bt == 0)
        for (int j = threadIdx.x; j < n; j += blockDim.x) J.var[j] = j;
}

struct NoClock {
    __device__ void lap(int) {}
};

// Shared memory of a team's block.
template <typename V>
struct TeamScratch {
    DelayScratch ds;
    DelayState state;
    Delayed<V> lp;
    TeamJob<V> job;
    int ok;
    unsigned passed;   // team barriers this block has passed (thread 0)
};

// A job entry from global memory (written before the team's last barrier) into
// shared memory.
template <typename V>
__device__ __forceinline__ void team_copy_job(TeamJob<V>& to, const TeamJob<V>* from) {
    static_assert(sizeof(TeamJob<V>) % 8 == 0, "copied in 8-byte words");
    const unsigned w = threadIdx.x;
    if (w < sizeof(TeamJob<V>) / 8) {
        const unsigned long long x = __ldcg(reinterpret_cast<const unsigned long long*>(from) + w);
        memcpy(reinterpret_cast<char*>(&to) + 8 * w, &x, 8);
    }
    __syncthreads();
}

// Solves one LP with the team of C blocks; false if a team barrier failed.
template <int NT, typename V>
__device__ bool team_solve_one(const TeamParams<V>& P, const TeamJob<V>& J, TeamState* ts, int bt, unsigned C,
                               unsigned char* smem, unsigned smem_bytes, TeamScratch<V>& s) {
    const int m = J.m, n = J.n;
    int r0, r1;
    team_rows(m, (int)C, bt, r0, r1);
    team_build(J, r0, r1, bt, ts);
    if (threadIdx.x == 0) {
        Delayed<V>& D = s.lp;
        D.T = J.T;
        D.ld = J.ld;
        D.m = m;
        D.n = n;
        D.basis = J.basis;
        D.var = J.var;
        D.Fh = J.Fh;
        D.Rh = J.Rh;
        D.RhT = J.RhT;
        D.rhs = J.rhs;
        D.rat = ts->rat;
        D.arg = ts->arg;
        D.bar_count = &ts->delay_count;
        D.fail = &ts->fail;
        D.status = nullptr;
        D.bt = bt;
        D.G = (int)C;
        D.smem = smem_bytes;
        delay_eps(P.eps_d, D.eps_d);
        delay_eps(P.eps_p, D.eps_p);
        D.max_iters = P.max_iters < 0 ? 50LL * ((long long)m + n) : P.max_iters;
        D.k_cyc = P.k_cyc;
        D.rule = P.rule;
        D.timeout_ns = P.timeout_ns;
        D.qlog = nullptr;
        D.plog = nullptr;
        D.log_cap = 0;
    }
    if (!team_barrier(ts, C, P.timeout_ns, s.ok, s.passed)) return false;
    int status = kInvalid;
    if (!ld_relaxed(&ts->bad)) {
        NoClock clk;
        delayed_solve<NT, kTeamRows>(s.lp, smem, s.ds, s.state, clk);
        status = s.state.status;
        if (status == kDelayFailed) return false;
    }
    // commit: the status is written only once every block of the team has
    // finished its part (a block that gave up at a barrier never gets here,
    // and the LP stays unfinished)
    if (!team_barrier(ts, C, P.timeout_ns, s.ok, s.passed)) return false;
    if (bt == 0 && threadIdx.x == 0) {
        J.st->status = status;
        if (status != kInvalid) {
            J.st->iters = s.state.it;
            J.st->bland = s.state.bland;
            J.st->degen_run = s.state.degen;
            J.st->passes = s.state.passes;
        } else {
            J.st->iters = 0;
            J.st->bland = P.rule == 1;
            J.st->degen_run = 0;
            J.st->passes = 0;
        }
    }
    return true;
}

// One cooperative launch: team t (blocks first[t] .. first[t] + size[t] - 1)
// takes entries of its own list, then of the other one, until both are empty.
// The wide teams, 0 .. their count - 1, start with that entry of their list: with
// a counter alone a narrow team without work of its own could take an LP from a
// wide team that began a moment later (5 FP64 LPs of 1000 x 900, blocks = 1: 55 ms
// a call, 17 with every LP on a wide team).
// Dynamic shared memory per block: smem_bytes, for the delayed solves.
template <int NT, typename V>
__global__ void __launch_bounds__(NT, team_sm_threads(NT) / NT) k_team_solve(TeamParams<V> P, unsigned smem_bytes) {
    extern __shared__ __align__(128) unsigned char tsx_dyn[];
    __shared__ TeamScratch<V> s;
    if (threadIdx.x == 0) s.passed = s.ds.passed = 0;
    const int t = P.team_of[blockIdx.x];
    const int bt = blockIdx.x - P.first[t];
    const unsigned C = (unsigned)P.size[t];
    TeamState* ts = P.teams + t;
    int li = P.list[t];
    for (bool start = true;; start = false) {
        if (bt == 0 && threadIdx.x == 0) {
            ts->bad = 0;   // read after the next barrier; set during the build
            int k = start && li == 1 ? P.order[1][t] : -1;
            for (int pass = 0; pass < 2 && k < 0; ++pass) {
                const int l = pass == 0 ? li : 1 - li;
                const int pos = (int)atomicAdd(P.next + l, 1u);
                if (pos < P.count[l]) k = P.order[l][pos];
            }
            ts->job = k;
        }
        if (!team_barrier(ts, C, P.timeout_ns, s.ok, s.passed)) return;
        const int k = *(volatile const int*)&ts->job;
        if (k < 0) return;
        team_copy_job(s.job, P.jobs + k);
        if (!team_solve_one<NT>(P, s.job, ts, bt, C, tsx_dyn, smem_bytes, s)) return;
    }
}

// ---------------------------------------------------------------------------
// Continuous team launch (the request server's lane for large LPs): the same
// teams and the same team_solve_one, but the jobs come from rings that the
// host appends to while the launch runs, so an LP admitted at any moment is
// taken by the next team that finishes one, and each LP reports its end on
// its own instead of at the end of a launch.
//   - rings in mapped host memory, one per list (light / heavy LPs): the host
//     writes a job entry, then publishes it by a release store of the list's
//     tail; a team's leader claims the next entry with a compare-and-swap on
//     the list's head (device memory) after an acquire load of the tail, and
//     copies the entry into device memory for the team;
//   - when an LP is solved (after the team's commit barrier) the leader
//     stores the job's sequence number + 1 into its done word (release,
//     system scope), which the host polls;
//   - a team that finds nothing to claim keeps polling while another team
//     still works (a job published meanwhile is taken at once); once no team
//     has had work for idle_ns (or at once, when the host asks for it) one of
//     them closes the launch, every team exits, and the host starts a new launch
//     when jobs are waiting and none runs.
//     Closing is a bit of the busy word, set by a compare-and-swap from zero,
//     and a team marks itself busy before it claims: a launch never goes on
//     with some of its teams gone.  (When each team left on its own clock, one
//     that claimed a job just then kept the launch alive alone, and the stream
//     behind it waited for that team: 7 s at 2000 LPs/s.)  Every wait is
//     bounded: the claim loop by idle_cap_ns and a spin cap, after which the
//     launch closes as well, the other blocks' wait for their leader by more
//     than that, the team barriers of a solve as in k_team_solve.  A team that
//     gives up clears its busy mark, closes the launch and claims nothing more;
//     an LP it has claimed is reported as timed out.
// ---------------------------------------------------------------------------
template <typename V>
struct ServeRing {
    TeamJob<V>* jobs;          // host memory: 2 lists x cap entries
    unsigned* tail;            // host memory: jobs published per list [2]
    unsigned* done;            // host memory: per entry, its sequence number + 1 once solved
    unsigned* stop;            // host memory: kServeStop, kServeYield or 0
};

template <typename V>
struct TeamServeParams {
    TeamParams<V> tp;          // tolerances, rules and team tables (jobs, order, count, next unused)
    ServeRing<V> ring;
    unsigned cap;              // entries per list, a power of two
    unsigned* head;            // device memory: jobs claimed per list [2]
    unsigned* busy;            // device memory: teams solving a job (zero at launch) and kServeClosed
    TeamJob<V>* jcopy;         // device memory: per team, the job it solves
    long long idle_ns;         // every team leaves once none has had work for this long
    long long idle_cap_ns;     // bound on a team's wait while others still work
};

constexpr unsigned kServeClosed = 0x80000000u;   // no further job is claimed in this launch
constexpr unsigned kServeStop = 1;    // teams with nothing to claim exit now
constexpr unsigned kServeYield = 2;   // the launch closes as soon as no team works, without waiting for idle_ns

__device__ __forceinline__ unsigned ld_acquire_sys(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_sys(unsigned* p, unsigned v) {
    asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

template <int NT, typename V>
__global__ void __launch_bounds__(NT, team_sm_threads(NT) / NT) k_team_serve(TeamServeParams<V> P, unsigned smem_bytes) {
    extern __shared__ __align__(128) unsigned char tsx_dyn[];
    __shared__ TeamScratch<V> s;
    if (threadIdx.x == 0) s.passed = s.ds.passed = 0;
    const int t = P.tp.team_of[blockIdx.x];
    const int bt = blockIdx.x - P.tp.first[t];
    const unsigned C = (unsigned)P.tp.size[t];
    TeamState* ts = P.tp.teams + t;
    const int li = P.tp.list[t];
    TeamJob<V>* jc = P.jcopy + t;
    // the blocks of a team without work wait for their leader, which polls for
    // up to idle_cap_ns, at a barrier (with timeout_ns alone, 2 s, they left a
    // leader behind that then claimed an LP it could not solve)
    const long long work_ns = P.idle_cap_ns + P.tp.timeout_ns;
    for (;;) {
        int got = -1;   // the leader's: list of the LP it has claimed
        if (bt == 0 && threadIdx.x == 0) {
            ts->bad = 0;   // read after the next barrier; set during the build
            unsigned gseq = 0;
            const long long t0 = global_ns();
            const unsigned long long max_spins =
                (unsigned long long)(P.idle_cap_ns > 0 ? P.idle_cap_ns : 0) / 500ull + 64ull;
            long long t_idle = t0;   // since when no team has been seen working
            for (unsigned long long spins = 0;; ++spins) {
                bool marked = false, closed = false;
                if (ld_relaxed(&ts->fail) != 0) {   // a block of this team has left
                    atomicOr(P.busy, kServeClosed);
                    break;
                }
                for (int pass = 0; pass < 2 && got < 0 && !closed; ++pass) {
                    const int l = pass == 0 ? li : 1 - li;
                    const unsigned tl = ld_acquire_sys(P.ring.tail + l);
                    unsigned h = *(volatile unsigned*)(P.head + l);
                    if ((int)(tl - h) > 0 && !marked) {
                        marked = true;
                        closed = (atomicAdd(P.busy, 1u) & kServeClosed) != 0u;
                    }
                    while (!closed && (int)(tl - h) > 0) {
                        const unsigned prev = atomicCAS(P.head + l, h, h + 1u);
                        if (prev == h) {
                            got = l;
                            gseq = h;
                            break;
                        }
                        h = prev;
                    }
                }
                if (got >= 0) break;
                if (marked) atomicSub(P.busy, 1u);
                const long long now = global_ns();
                const unsigned busy = *(volatile unsigned*)P.busy;
                if (closed || (busy & kServeClosed)) break;
                if (busy != 0u) t_idle = now;
                const unsigned stop = ld_acquire_sys(P.ring.stop);
                if (stop == kServeStop) break;
                if ((stop == kServeYield || now - t_idle >= P.idle_ns) && atomicCAS(P.busy, 0u, kServeClosed) == 0u)
                    break;
                if (now - t0 >= P.idle_cap_ns || spins >= max_spins) {
                    atomicOr(P.busy, kServeClosed);
                    break;
                }
                __nanosleep(500);
            }
            if (got >= 0) {
                const unsigned slot = (unsigned)got * P.cap + (gseq & (P.cap - 1u));
                const volatile unsigned long long* src =
                    reinterpret_cast<const volatile unsigned long long*>(P.ring.jobs + slot);
                unsigned long long* dst = reinterpret_cast<unsigned long long*>(jc);
                for (int w = 0; w < (int)(sizeof(TeamJob<V>) / 8); ++w) dst[w] = src[w];
                ts->job = (int)slot;
                ts->seq = gseq;
                // the LP's state words start from zero here (no reset launch per job)
                DevState* st = jc->st;
                st->status = kRunning;
                st->q = -1;
                st->p = -1;
                st->bland = 0;
                st->degen_run = 0;
                st->bad = 0;
                st->iters = 0;
                st->active_sectors = 0;
                st->theta = 0.0;
                st->bar_count = 0;
                st->bar_gen = 0;
                st->nact = 0;
                st->next_slot = 0;
                st->fail = 0;
                st->passes = 0;
                for (int q = 2; q < 6; ++q) st->phase_ns[q] = 0;
                st->phase_ns[1] = 0;
                st->phase_ns[0] = global_ns();
            } else {
                ts->job = -1;
            }
        }
        if (!team_barrier(ts, C, work_ns, s.ok, s.passed)) {
            if (bt == 0 && threadIdx.x == 0) {
                atomicOr(P.busy, kServeClosed);
                if (got >= 0) atomicSub(P.busy, 1u);
            }
            return;
        }
        const int slot = *(volatile const int*)&ts->job;
        if (slot < 0) return;
        team_copy_job(s.job, jc);
        if (!team_solve_one<NT>(P.tp, s.job, ts, bt, C, tsx_dyn, smem_bytes, s)) {
            if (bt == 0 && threadIdx.x == 0) {
                atomicOr(P.busy, kServeClosed);
                atomicSub(P.busy, 1u);
            }
            return;
        }
        if (bt == 0 && threadIdx.x == 0) {
            s.job.st->phase_ns[1] = global_ns();
            __threadfence_system();
            st_release_sys(P.ring.done + slot, *(volatile unsigned*)&ts->seq + 1u);
            atomicSub(P.busy, 1u);
        }
    }
}

}  // namespace tsx
