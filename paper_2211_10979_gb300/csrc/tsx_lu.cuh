// LU solves of the FP64 recovery: x_S of A_RS x_S = b_R and y_R of A_RS^T y_R =
// c_S (tsx_recover.cuh) without the explicit inverse, for the usual case that
// the checks pass and no cleanup pivot needs rows or columns of the inverse.
// Partial pivoting (largest entry, lowest row on ties), rows not swapped:
// piv[c] is the row of step c.  Both systems take one step of iterative
// refinement with residuals from A, summed to twice the precision.
//
//   k_rec_lu_small   k up to ~165: one block, the matrix in shared memory.  The
//                    elimination by a cooperative grid took a grid barrier and
//                    more (8 us) per column and ~11 launches around it; here
//                    everything is one launch and no cooperative one, so that
//                    recoveries of several LPs also run side by side.
//   k_lu_panel,      larger k: panels of 32 columns by one thread-block cluster
//   k_lu_update,     (rows in its shared memory, one cluster barrier a column),
//   k_lu_solve       the rest of the matrix by the whole GPU with 32 steps per
//                    pass (k^3 / 3 fused multiply-adds instead of the inverse's
//                    k^3), then blocked triangular solves in one launch.
// Whole recovery, inverse -> LU: k = 44 0.49 -> 0.38 ms, 128 1.04 -> 0.70, 512
// 4.5 -> 3.1, 2048 37.2 -> 16.5, 4096 253 -> 64.  Errors of x_S and y_R against
// quad precision over k = 9 .. 600: 3e-17 .. 6e-17 (inverse 1e-16 .. 7e-15).
#pragma once

#include <cooperative_groups.h>

#include "tsx_device.cuh"

namespace tsx {

// Largest |x| of the warp's lanes and the lowest row that holds it, on the
// bits (rows with none: key 0, row INT_MAX); every lane gets both.
__device__ __forceinline__ void lu_warp_max(unsigned long long& key, int& row) {
    constexpr unsigned all = 0xffffffffu;
    const unsigned h = __reduce_max_sync(all, (unsigned)(key >> 32));
    bool in = (unsigned)(key >> 32) == h;
    const unsigned l = __reduce_max_sync(all, in ? (unsigned)key : 0u);
    in = in && (unsigned)key == l;
    row = __reduce_min_sync(all, in ? row : INT_MAX);
    key = ((unsigned long long)h << 32) | l;
}
__device__ __forceinline__ unsigned long long lu_abs_key(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

// x / d from r = 1 / d: the rounded product and one correction by its remainder
// (Markstein, IBM J. Res. Dev. 34, 1990; a third of a division's latency).
__device__ __forceinline__ double lu_quotient(double x, double d, double r) {
    const double q = x * r;
    return __fma_rn(__fma_rn(-q, d, x), r, q);
}

// A sum of products kept as value + error (exact products by fma, two-sums:
// Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26, 2005): the residual that the
// refinement step solves for, which a plain sum would lose most digits of.
struct LuSum {
    double v, e;
    __device__ __forceinline__ void add(double x) {
        const double t = v + x, z = t - v;
        e += (v - (t - z)) + (x - z);
        v = t;
    }
    __device__ __forceinline__ void sub_product(double a, double b, bool plain) {
        if (plain) {   // the last residual is only reported
            v = __fma_rn(-a, b, v);
            return;
        }
        const double p = a * b;
        e -= __fma_rn(a, b, -p);
        add(-p);
    }
    __device__ __forceinline__ double warp_total() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ov = __shfl_xor_sync(0xffffffffu, v, o), oe = __shfl_xor_sync(0xffffffffu, e, o);
            add(ov);
            e += oe;
        }
        return v + e;
    }
};

// ------------------------------------------------------------- small k
__host__ __device__ constexpr size_t lu_small_smem(int k) {
    return ((size_t)k * (k | 1) + 5 * (size_t)k) * 8 + 4 * (size_t)k * 4;
}
constexpr int kLuSmallMax = 192;   // k of the small kernel, upper bound (vectors in six registers a lane)

// One triangular sweep by one warp: v (k entries, v[i] of lane i % 32) with the
// factors coef(a, c) of entry c in entry a; entries in the order first, first +
// step, ...; scale: the finished entry divided by coef(c, c) = 1 / scale[c].
template <int NV, typename Coef>
__device__ __forceinline__ void lu_sweep(double (&v)[NV], int k, bool down, const double* scale, Coef coef) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int y = 0; y < NV; ++y) {
        const int i = down ? y : NV - 1 - y;
        for (int x = 0; x < 32; ++x) {
            const int l = down ? x : 31 - x, c = i * 32 + l;
            if (c >= k) continue;
            double vc = __shfl_sync(0xffffffffu, v[i], l);
            if (scale) {
                vc = lu_quotient(vc, coef(c, c), scale[c]);
                if (lane == l) v[i] = vc;
            }
#pragma unroll
            for (int z = 0; z < NV; ++z) {
                const int a = z * 32 + lane;
                if (a < k && (down ? a > c : a < c)) v[z] = __fma_rn(-coef(a, c), vc, v[z]);
            }
        }
    }
}

template <int NT>
__global__ void __launch_bounds__(NT) k_rec_lu_small(int n, const double* __restrict__ A, const double* __restrict__ b,
                                                    const double* __restrict__ c, const int* __restrict__ S,
                                                    const int* __restrict__ Rr, int k, double* __restrict__ xS,
                                                    double* __restrict__ yR, double* __restrict__ rp,
                                                    double* __restrict__ rd, int* singular) {
    extern __shared__ __align__(16) double lu_dyn[];
    __shared__ double s_ip;
    __shared__ int s_pr;
    const int ld = k | 1;
    double* M = lu_dyn;
    double *ip = M + (size_t)k * ld, *x = ip + k, *y = x + k, *u = y + k, *v = u + k;   // u, v: right-hand sides
    int *sS = reinterpret_cast<int*>(v + k), *sR = sS + k, *piv = sR + k, *pos = piv + k;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    constexpr int NW = NT / 32, NV = kLuSmallMax / 32;
    for (int i = t; i < k; i += NT) {
        sS[i] = S[i];
        sR[i] = Rr[i];
        pos[i] = -1;
        u[i] = b[Rr[i]];
        v[i] = c[S[i]];
        x[i] = 0.0;
        y[i] = 0.0;
    }
    __syncthreads();
    for (int r = w; r < k; r += NW) {
        const double* row = A + (size_t)sR[r] * n;
        for (int j = lane; j < k; j += 32) M[r * ld + j] = row[sS[j]];
    }
    __syncthreads();
    for (int j = 0; j < k; ++j) {
        if (w == 0) {
            unsigned long long key = 0;
            int row = INT_MAX;
            for (int r = lane; r < k; r += 32)
                if (pos[r] < 0) {
                    const unsigned long long q = lu_abs_key(M[r * ld + j]);
                    if (q > key) { key = q; row = r; }
                }
            lu_warp_max(key, row);
            if (lane == 0) {
                s_pr = row;
                if (row != INT_MAX) {
                    piv[j] = row;
                    pos[row] = j;
                    s_ip = ip[j] = 1.0 / M[row * ld + j];
                }
            }
        }
        __syncthreads();
        const int pr = s_pr;
        if (pr == INT_MAX) {   // no nonzero candidate
            if (t == 0) *singular = 1;
            return;
        }
        for (int r = t; r < k; r += NT)
            if (pos[r] < 0) M[r * ld + j] = lu_quotient(M[r * ld + j], M[pr * ld + j], s_ip);
        __syncthreads();
        // two rows a warp at a time, all of their entries in flight
        for (int r = w; r < k; r += 2 * NW) {
            const int r2 = r + NW;
            const bool in = pos[r] < 0, in2 = r2 < k && pos[r2] < 0;
            if (!in && !in2) continue;
            double *row = M + r * ld, *row2 = M + (in2 ? r2 : r) * ld;
            const double l = row[j], l2 = row2[j];
            double e[NV], e2[NV], g[NV];
#pragma unroll
            for (int z = 0; z < NV; ++z) {
                const int q = j + 1 + lane + 32 * z;
                if (q < k) {
                    g[z] = M[pr * ld + q];
                    e[z] = row[q];
                    e2[z] = row2[q];
                }
            }
#pragma unroll
            for (int z = 0; z < NV; ++z) {
                const int q = j + 1 + lane + 32 * z;
                if (j + 1 + 32 * z >= k) break;
                if (in) e[z] = __fma_rn(-l, g[z], e[z]);
                if (in2) e2[z] = __fma_rn(-l2, g[z], e2[z]);
                if (in && q < k) row[q] = e[z];
                if (in2 && q < k) row2[q] = e2[z];
            }
        }
        __syncthreads();
    }
    // x += (LU)^-1 u, y += (LU)^-T v, then u, v = the residuals; twice
    for (int pass = 0; pass < 2; ++pass) {
        if (w < 2) {
            double z[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const int a = i * 32 + lane;
                z[i] = a < k ? (w == 0 ? u[piv[a]] : v[a]) : 0.0;
            }
            if (w == 0) {
                lu_sweep<NV>(z, k, true, nullptr, [&](int a, int q) { return M[piv[a] * ld + q]; });
                lu_sweep<NV>(z, k, false, ip, [&](int a, int q) { return M[piv[a] * ld + q]; });
            } else {
                lu_sweep<NV>(z, k, true, ip, [&](int a, int q) { return M[piv[q] * ld + a]; });
                lu_sweep<NV>(z, k, false, nullptr, [&](int a, int q) { return M[piv[q] * ld + a]; });
            }
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const int a = i * 32 + lane;
                if (a < k) {
                    if (w == 0) x[a] += z[i];
                    else y[piv[a]] += z[i];
                }
            }
        }
        __syncthreads();
        for (int r = w; r < 2 * k; r += NW) {
            LuSum sum{lane == 0 ? (r < k ? b[sR[r]] : c[sS[r - k]]) : 0.0, 0.0};
            if (r < k) {
                const double* row = A + (size_t)sR[r] * n;
                for (int j = lane; j < k; j += 32) sum.sub_product(row[sS[j]], x[j], pass > 0);
            } else {
                const double* col = A + sS[r - k];
                for (int a = lane; a < k; a += 32) sum.sub_product(col[(size_t)sR[a] * n], y[a], pass > 0);
            }
            const double total = sum.warp_total();
            if (lane == 0) (r < k ? u[r] : v[r - k]) = total;
        }
        __syncthreads();
    }
    for (int i = t; i < k; i += NT) {
        xS[i] = x[i];
        yR[i] = y[i];
        rp[i] = u[i];
        rd[i] = v[i];
    }
}

// ------------------------------------------------------------- large k
constexpr int kLuNb = 32;        // columns of a panel
constexpr int kLuCluster = 16;   // blocks of the panel cluster

struct LuCand {
    unsigned long long key;
    int row, pos;      // row, and its place in the owner's rows
};

constexpr int kLuMax = kLuCluster * 256;   // k of the panels, upper bound: a row a thread

__global__ void k_lu_init(int k, int* __restrict__ act) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < k; t += gridDim.x * blockDim.x) act[t] = t;
}

// What the blocks of a panel's cluster share in their shared memory.
template <int NT>
struct LuPanel {
    LuCand offers[2][kLuCluster], sw[NT / 32], won;
    double crow[2][kLuNb + 1];   // the offered row from the column on, its reciprocal
    double prow[kLuNb + 1];
    int hole[kLuNb];
};

// Columns j0 .. j0 + 7 of a panel: p[0 .. W) are a thread's row from column j
// on, shifted by one every column (a loop: 32 unrolled columns would fetch 4 KB
// of instructions each).  False: no pivot left.
template <int NT, int W>
__device__ __forceinline__ bool lu_panel_columns(double (&p)[kLuNb], int j0, int row, int& used, double* M, double* U,
                                                 int k, int c0, int nb, int per, int* piv, double* ip,
                                                 LuPanel<NT>& s) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int rank = (int)cl.block_rank(), C = (int)cl.num_blocks();
#pragma unroll 1
    for (int j = j0; j < min(j0 + 8, nb); ++j) {
        unsigned long long key = used < 0 ? lu_abs_key(p[0]) : 0;
        int r = key ? row : INT_MAX;
        lu_warp_max(key, r);
        const int at = __ffs(__ballot_sync(0xffffffffu, used < 0 && row == r)) - 1 + w * 32;
        if (lane == 0) s.sw[w] = LuCand{key, key ? r : INT_MAX, at};
        __syncthreads();
        LuCand best = s.sw[0];
#pragma unroll
        for (int q = 1; q < NT / 32; ++q) {
            const LuCand o = s.sw[q];
            if (o.key > best.key || (o.key == best.key && o.row < best.row)) best = o;
        }
        // the offer goes to every block of the cluster, the row stays here
        if (t < C) *cl.map_shared_rank(&s.offers[j & 1][rank], t) = best;
        if (best.key != 0 && row == best.row) {
#pragma unroll
            for (int q = 0; q < W; ++q) s.crow[j & 1][q] = p[q];
            s.crow[j & 1][kLuNb] = 1.0 / p[0];
        }
        cl.sync();
        // every block takes the same winner; its row comes from the owner
        if (w == 0) {
            LuCand o{0, INT_MAX, 0};
            if (lane < C) o = s.offers[j & 1][lane];
            unsigned long long bk = o.key;
            int br = o.row;
            lu_warp_max(bk, br);
            const int owner = __ffs(__ballot_sync(0xffffffffu, o.row == br && o.key == bk)) - 1;
            const int place = __shfl_sync(0xffffffffu, o.pos, owner);
            const double* from = cl.map_shared_rank(&s.crow[j & 1][0], owner);
            if (lane < W) s.prow[lane] = from[lane];
            if (lane == 0) {
                s.prow[kLuNb] = from[kLuNb];
                s.won = LuCand{bk, br, owner * per + place};
            }
        }
        __syncthreads();
        if (s.won.key == 0) return false;
        const double inv = s.prow[kLuNb];
        if (rank == 0) {
            if (t == 0) {
                piv[c0 + j] = s.won.row;
                ip[c0 + j] = inv;
                s.hole[j] = s.won.pos;
            }
            if (w == 1 && j + lane < nb) U[(size_t)(c0 + j) * k + c0 + j + lane] = s.prow[lane];
        }
        if (row == s.won.row) used = j;
        if (used < 0) {
            const double l = p[0] * inv;
            M[(size_t)row * k + c0 + j] = l;
#pragma unroll
            for (int q = 1; q < W; ++q) p[q - 1] = __fma_rn(-l, s.prow[q], p[q]);
        }
    }
    return true;
}

// Panel c0: columns c0 .. c0 + nb - 1 of the rows in act[0 .. na), na = k - c0,
// by one cluster, a row per thread, its 32 entries in registers (those beyond a
// last, narrower panel are zero).  Per column every block offers its largest
// entry, one cluster barrier, and every block takes the same winner, whose row
// and reciprocal come from its owner's shared memory.  Writes the multipliers
// into M, the pivot rows' entries into U (row c of U: pivot row of step c), piv,
// ip = 1 / pivot, and takes the panel's pivot rows out of act.
template <int NT>
__global__ void __launch_bounds__(NT) k_lu_panel(double* __restrict__ M, double* __restrict__ U, int k, int c0,
                                                int* __restrict__ act, int* __restrict__ piv,
                                                double* __restrict__ ip, int* singular) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ LuPanel<NT> s;
    if (*(volatile int*)singular) return;   // set by an earlier panel: the same for every block
    const int t = threadIdx.x;
    const int rank = (int)cl.block_rank(), C = (int)cl.num_blocks();
    const int na = k - c0, nb = min(kLuNb, na), per = (na + C - 1) / C;
    const int a0 = rank * per;
    const bool mine = t < per && a0 + t < na;
    const int row = mine ? act[a0 + t] : INT_MAX;
    int used = mine ? -1 : 0;
    double p[kLuNb];
    const double* src = M + (size_t)(mine ? row : 0) * k + c0;
#pragma unroll
    for (int q = 0; q < kLuNb; ++q) p[q] = mine && q < nb ? src[q] : 0.0;
    cl.sync();   // every block of the cluster runs before its shared memory is written
    const bool ok = lu_panel_columns<NT, 32>(p, 0, row, used, M, U, k, c0, nb, per, piv, ip, s) &&
                    lu_panel_columns<NT, 24>(p, 8, row, used, M, U, k, c0, nb, per, piv, ip, s) &&
                    lu_panel_columns<NT, 16>(p, 16, row, used, M, U, k, c0, nb, per, piv, ip, s) &&
                    lu_panel_columns<NT, 8>(p, 24, row, used, M, U, k, c0, nb, per, piv, ip, s);
    cl.sync();   // no block reads act, or another's shared memory, any more
    if (!ok) {   // the same for every block
        if (rank == 0 && t == 0) *singular = 1;
        return;
    }
    if (rank == 0 && t == 0) {
        // the last entries of the list fill the pivot rows' places
        int tail = na;
        for (int j = 0; j < nb; ++j) {
            if (s.hole[j] >= na - nb) continue;   // lies in the part cut off
            for (;;) {
                --tail;
                bool is = false;
                for (int q = 0; q < nb; ++q) is |= s.hole[q] == tail;
                if (!is) break;
            }
            act[s.hole[j]] = act[tail];
        }
    }
}

// U's rows of panel c0 right of it: forward substitution with the panel's unit
// lower triangle, a column per thread, one warp per block (the FP64 pipe of an
// SM takes 3.8 us for 32 columns).
__global__ void __launch_bounds__(32) k_lu_rows(const double* __restrict__ M, double* __restrict__ U, int k, int c0,
                                               const int* __restrict__ piv, const int* singular) {
    __shared__ double L[kLuNb][kLuNb + 1];
    if (*singular) return;
    const int lane = threadIdx.x, j = c0 + kLuNb + blockIdx.x * 32 + lane;
    const int pl = piv[c0 + lane];
    double z[kLuNb];
#pragma unroll
    for (int a = 0; a < kLuNb; ++a) {
        const size_t row = (size_t)__shfl_sync(0xffffffffu, pl, a) * k;
        L[a][lane] = M[row + c0 + lane];
        z[a] = j < k ? M[row + j] : 0.0;
    }
    __syncwarp();
#pragma unroll
    for (int a = 0; a < kLuNb; ++a)
#pragma unroll
        for (int q = a + 1; q < kLuNb; ++q) z[q] = __fma_rn(-L[q][a], z[a], z[q]);
    if (j < k)
#pragma unroll
        for (int a = 0; a < kLuNb; ++a) U[(size_t)(c0 + a) * k + j] = z[a];
}

// The other rows right of panel c0: its 32 steps in one pass.  Block (x, y):
// strip x of 128 columns, the row tiles y, y + gridDim.y, ... a warp each.
constexpr size_t lu_update_smem(int nt) { return (size_t)(kLuNb * 128 + (nt / 32) * kLuNb * 10) * 8; }
template <int NT>
__global__ void __launch_bounds__(NT) k_lu_update(double* __restrict__ M, const double* __restrict__ U, int k, int c0,
                                                 const int* __restrict__ act, const int* singular) {
    constexpr int RS = 8, FS = RS + 2;
    extern __shared__ __align__(16) double lu_dyn[];   // lu_update_smem
    double (*R)[128] = reinterpret_cast<double (*)[128]>(lu_dyn);
    double* F = lu_dyn + kLuNb * 128;
    if (*singular) return;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int j0 = c0 + kLuNb + blockIdx.x * 128, width = min(128, k - j0), na = k - c0 - kLuNb;
    for (int e = t; e < kLuNb * 128; e += NT) {
        const int a = e >> 7, q = e & 127;
        R[a][q] = q < width ? U[(size_t)(c0 + a) * k + j0 + q] : 0.0;
    }
    __syncthreads();
    double* f = F + w * (kLuNb * FS);
    const int ntiles = (na + RS - 1) / RS;
    // consecutive tiles on different SMs first: eight warps of one share its FP64 pipe
    for (int tile = w * gridDim.y + blockIdx.y; tile < ntiles; tile += gridDim.y * (NT / 32)) {
        int row[RS];
        double v[RS][4];
        const int nr = min(RS, na - tile * RS);
#pragma unroll
        for (int r = 0; r < RS; ++r) {
            row[r] = r < nr ? act[tile * RS + r] : 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int col = q * 32 + lane;
                v[r][q] = r < nr && col < width ? M[(size_t)row[r] * k + j0 + col] : 0.0;
            }
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < RS; ++r) f[lane * FS + r] = r < nr ? -M[(size_t)row[r] * k + c0 + lane] : 0.0;
        __syncwarp();
#pragma unroll 2
        for (int u = 0; u < kLuNb; ++u) {
            double x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = R[u][q * 32 + lane];
#pragma unroll
            for (int r = 0; r < RS; ++r) {
                const double g = f[u * FS + r];
#pragma unroll
                for (int q = 0; q < 4; ++q) v[r][q] = __fma_rn(g, x[q], v[r][q]);
            }
        }
#pragma unroll
        for (int r = 0; r < RS; ++r)
            if (r < nr)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int col = q * 32 + lane;
                    if (col < width) M[(size_t)row[r] * k + j0 + col] = v[r][q];
                }
    }
}

// The solves: x += (LU)^-1 u and y += (LU)^-T v in blocks of 32 steps, both
// systems side by side, one grid barrier per block; then the residuals u, v;
// twice.  z, q: k doubles of work each.  Every block solves the 32 x 32
// triangles itself (one warp each) and takes a share of the other entries.
template <int NT>
__global__ void __launch_bounds__(NT) k_lu_solve(int n, const double* __restrict__ A, const double* __restrict__ b,
                                                const double* __restrict__ c, const int* __restrict__ S,
                                                const int* __restrict__ Rr, int k, const double* __restrict__ M,
                                                const double* __restrict__ U, const int* __restrict__ piv,
                                                const double* __restrict__ ip, double* z, double* q, double* x,
                                                double* y, double* u, double* v, const int* singular, DevState* st,
                                                long long timeout_ns) {
    __shared__ BlockScratch s;
    __shared__ double zx[32], zy[32];
    if (*singular) return;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int gt = blockIdx.x * NT + t, nth = gridDim.x * NT, gw = gt >> 5, nw = nth >> 5;
    const int nblk = (k + 31) / 32;
    for (int i = gt; i < k; i += nth) {
        z[i] = b[Rr[piv[i]]];
        q[i] = c[S[i]];
        x[i] = 0.0;
        y[i] = 0.0;
    }
    if (!grid_barrier(st, timeout_ns, s)) return;
    for (int pass = 0; pass < 2; ++pass) {
        for (int half = 0; half < 2; ++half) {
            const bool down = half == 0;
            for (int bi = 0; bi < nblk; ++bi) {
                const int blk = down ? bi : nblk - 1 - bi, o = blk * 32, nb = min(32, k - o);
                // the triangle of this block, in every thread block: lane's
                // factors of all its steps first (L or U for x, their
                // transposes for y), then the chain
                if (w < 2) {
                    double e = lane < nb ? (w == 0 ? __ldcg(z + o + lane) : __ldcg(q + o + lane)) : 0.0;
                    const int pl = lane < nb ? piv[o + lane] : 0;
                    const double rl = lane < nb ? ip[o + lane] : 0.0;
                    double g[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        const int pi = __shfl_sync(0xffffffffu, pl, i);
                        const bool in = i < nb && lane < nb && (down ? lane > i : lane < i);
                        g[i] = !in ? 0.0
                               : w == 0 ? (down ? M[(size_t)pl * k + o + i] : U[(size_t)(o + lane) * k + o + i])
                                        : (down ? U[(size_t)(o + i) * k + o + lane] : M[(size_t)pi * k + o + lane]);
                    }
                    const bool scaled = (w == 0) != down;   // U's diagonal: x going up, y going down
#pragma unroll
                    for (int i0 = 0; i0 < 32; ++i0) {
                        // g is 0 outside the triangle, so the steps beyond nb change nothing
                        const int iu = 31 - i0;
                        double ei = __shfl_sync(0xffffffffu, e, down ? i0 : iu);
                        const double ri = __shfl_sync(0xffffffffu, rl, down ? i0 : iu);
                        if (scaled) {
                            ei *= ri;
                            if (lane == (down ? i0 : iu)) e = ei;
                        }
                        e = __fma_rn(-(down ? g[i0] : g[iu]), ei, e);
                    }
                    if (w == 0) zx[lane] = lane < nb ? e : 0.0;
                    else zy[lane] = lane < nb ? e : 0.0;
                }
                __syncthreads();
                if (blockIdx.x == 0 && w < 2 && lane < nb) {
                    if (w == 0) {   // finished entries, kept apart from the ones others still read
                        if (!down) x[o + lane] += zx[lane];
                    } else if (!down) {
                        y[piv[o + lane]] += zy[lane];
                    }
                }
                // the entries beyond the block (down) or before it (up)
                const int e0 = down ? o + nb : 0, e1 = down ? k : o;
                for (int a = e0 + gw; a < e1; a += nw) {   // x: a warp per row of L or U
                    const double* row = down ? M + (size_t)piv[a] * k : U + (size_t)a * k;
                    double sum = lane < nb ? row[o + lane] * zx[lane] : 0.0;
#pragma unroll
                    for (int h = 16; h > 0; h >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, h);
                    if (lane == 0) __stcg(z + a, __ldcg(z + a) - sum);
                }
                for (int a = e0 + gt; a < e1; a += nth) {   // y: a thread per column
                    double e = __ldcg(q + a);
#pragma unroll 8
                    for (int i = 0; i < nb; ++i)
                        e = __fma_rn(-(down ? U[(size_t)(o + i) * k + a] : M[(size_t)piv[o + i] * k + a]), zy[i], e);
                    __stcg(q + a, e);
                }
                // the solved block, for the sweep up
                if (down) {
                    __syncthreads();
                    if (!grid_barrier(st, timeout_ns, s)) return;   // every block has read z, q of this block
                    if (blockIdx.x == 0 && w < 2 && lane < nb) {
                        if (w == 0) __stcg(z + o + lane, zx[lane]);
                        else __stcg(q + o + lane, zy[lane]);
                    }
                    __syncthreads();
                } else {
                    if (!grid_barrier(st, timeout_ns, s)) return;
                }
            }
            if (down && !grid_barrier(st, timeout_ns, s)) return;   // block 0's last stores
        }
        // residuals, one warp per entry
        for (int r = gw; r < 2 * k; r += nw) {
            LuSum sum{lane == 0 ? (r < k ? b[Rr[r]] : c[S[r - k]]) : 0.0, 0.0};
            if (r < k) {
                const double* row = A + (size_t)Rr[r] * n;
                for (int j = lane; j < k; j += 32) sum.sub_product(row[S[j]], __ldcg(x + j), pass > 0);
            } else {
                const double* col = A + S[r - k];
                for (int a = lane; a < k; a += 32) sum.sub_product(col[(size_t)Rr[a] * n], __ldcg(y + a), pass > 0);
            }
            const double total = sum.warp_total();
            if (lane == 0) __stcg(r < k ? u + r : v + (r - k), total);
        }
        if (!grid_barrier(st, timeout_ns, s)) return;
        if (pass == 0) {
            for (int i = gt; i < k; i += nth) {
                __stcg(z + i, __ldcg(u + piv[i]));
                __stcg(q + i, __ldcg(v + i));
            }
            if (!grid_barrier(st, timeout_ns, s)) return;
        }
    }
}

}  // namespace tsx
