// multilevel.cu -- an aggregation multilevel preconditioner for the inner solve.
//
// The paper preconditions the trimmed systems with combinatorial multigrid (Sec. 3.2; Remark 3.2,
// with the deflated form of Eq. 3.6).  This file builds a multilevel preconditioner of the same
// kind for M ~ Lh, the trimmed Laplacian (Theorem 2.3: an SPD M-matrix):
//  * level 0 is the graph without the trimmed vertex, with the full degrees on the diagonal (the
//    trimmed vertex acts as a Dirichlet node for its neighbours);
//  * the vertices of a level are grouped into small connected clusters by greedy aggregation
//    (a vertex whose neighbours are all free starts a cluster with them; leftover vertices join
//    the neighbouring cluster they are most strongly tied to);
//  * each cluster becomes one vertex of the next level, whose matrix is the Galerkin product
//    P^T A P with the piecewise-constant P: again a weighted Laplacian, with edge weights summed
//    between clusters and the clusters' Dirichlet mass kept on the diagonal;
//  * levels stop at <= kMlCoarse vertices, whose matrix is inverted densely on the host.
// M^{-1} b is one V-cycle: on each level x0 = w D^{-1} b, the residual restricted to the next level,
// x1 = x0 + a P x_c, and one more damped Jacobi step x1 + w D^{-1} (b - A x1).  With the same
// smoother before and after the coarse correction the cycle is a symmetric operator, positive
// definite for w < 1 (the levels are diagonally dominant, so rho(D^{-1} A) <= 2) and any a > 0.
//
// Storage per level l >= 1: CSR (int32 row pointers) of the off-diagonal weights W (positive; the
// matrix is diag(d) - W), 1/d, the cluster map of level l-1 (fine vertex -> cluster) and the member
// lists of the clusters (CSR over the clusters).  Level 0 uses the solver's own gather for W x.
//
// Launches of one V-cycle: level 0 takes the gather twice (W x0 with the residual, W x1) with a restriction
// and a prolongation / post-smoothing around them (x0, and the last gather with the post-smoothing, usually come
// with the caller's own kernels); each level l >= 1 takes one kernel down and one up, and the
// coarsest level one product with its dense inverse.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>
#include <vector>

#include "internal.h"

namespace isira {

constexpr int kMlCoarse = 512;       // the coarsest level is solved with a dense inverse
constexpr int kMlMaxLevels = 12;

struct HostLevel {
    int64_t n = 0;
    std::vector<int64_t> rp;
    std::vector<int32_t> ci;
    std::vector<double> w;       // off-diagonal weights (positive)
    std::vector<double> d;       // diagonal
};

// Greedy aggregation.  skip: a vertex excluded from every cluster (-1: none).  Returns the
// cluster id of every vertex (-1 for skip) and the cluster count.
static std::vector<int32_t> aggregate(const HostLevel& A, int64_t skip, int64_t* n_agg) {
    const int64_t n = A.n;
    std::vector<int32_t> agg(n, -1);
    std::vector<char> p1(n, 0);
    int32_t next = 0;
    // phase 1: a vertex whose neighbours are all free starts a cluster with all of them
    for (int64_t i = 0; i < n; ++i) {
        if (i == skip || agg[i] >= 0) continue;
        bool free_nb = true;
        for (int64_t e = A.rp[i]; e < A.rp[i + 1] && free_nb; ++e) {
            const int64_t j = A.ci[e];
            if (j != skip && agg[j] >= 0) free_nb = false;
        }
        if (!free_nb) continue;
        agg[i] = next;
        p1[i] = 1;
        for (int64_t e = A.rp[i]; e < A.rp[i + 1]; ++e) {
            const int64_t j = A.ci[e];
            if (j != skip) {
                agg[j] = next;
                p1[j] = 1;
            }
        }
        ++next;
    }
    // phase 2: every free vertex joins the phase-1 cluster it is most strongly tied to
    std::vector<int32_t> join(n, -1);
    for (int64_t i = 0; i < n; ++i) {
        if (i == skip || agg[i] >= 0) continue;
        double best = 0.0;
        int32_t bid = -1;
        for (int64_t e = A.rp[i]; e < A.rp[i + 1]; ++e) {
            const int64_t j = A.ci[e];
            if (j == skip || !p1[j]) continue;
            if (A.w[e] > best || (A.w[e] == best && agg[j] < bid)) {
                best = A.w[e];
                bid = agg[j];
            }
        }
        join[i] = bid;
    }
    for (int64_t i = 0; i < n; ++i)
        if (join[i] >= 0) agg[i] = join[i];
    // phase 3: what is still free forms clusters with its free neighbours
    for (int64_t i = 0; i < n; ++i) {
        if (i == skip || agg[i] >= 0) continue;
        agg[i] = next;
        for (int64_t e = A.rp[i]; e < A.rp[i + 1]; ++e) {
            const int64_t j = A.ci[e];
            if (j != skip && agg[j] < 0) agg[j] = next;
        }
        ++next;
    }
    *n_agg = next;
    return agg;
}

// Galerkin coarse matrix P^T A P for the piecewise-constant P of `agg`.
static HostLevel coarsen(const HostLevel& A, const std::vector<int32_t>& agg, int64_t nc) {
    HostLevel C;
    C.n = nc;
    C.d.assign(nc, 0.0);
    // members of each cluster, in fine order
    std::vector<int64_t> mrp(nc + 1, 0);
    for (int64_t i = 0; i < A.n; ++i)
        if (agg[i] >= 0) mrp[agg[i] + 1]++;
    for (int64_t I = 0; I < nc; ++I) mrp[I + 1] += mrp[I];
    std::vector<int64_t> mem(mrp[nc]);
    {
        std::vector<int64_t> pos(mrp.begin(), mrp.end() - 1);
        for (int64_t i = 0; i < A.n; ++i)
            if (agg[i] >= 0) mem[pos[agg[i]]++] = i;
    }
    std::vector<double> acc(nc, 0.0);
    std::vector<int32_t> mark(nc, -1);
    std::vector<int32_t> cols;
    C.rp.assign(nc + 1, 0);
    for (int64_t I = 0; I < nc; ++I) {
        cols.clear();
        double dI = 0.0;
        for (int64_t q = mrp[I]; q < mrp[I + 1]; ++q) {
            const int64_t i = mem[q];
            dI += A.d[i];
            for (int64_t e = A.rp[i]; e < A.rp[i + 1]; ++e) {
                const int32_t J = agg[A.ci[e]];
                if (J < 0) continue;                         // an edge to the excluded vertex
                if (J == I) {
                    dI -= A.w[e];                            // internal edge: P^T A P adds -w twice
                    continue;
                }
                if (mark[J] != I) {
                    mark[J] = (int32_t)I;
                    acc[J] = 0.0;
                    cols.push_back(J);
                }
                acc[J] += A.w[e];
            }
        }
        std::sort(cols.begin(), cols.end());
        for (int32_t J : cols) {
            C.ci.push_back(J);
            C.w.push_back(acc[J]);
        }
        C.d[I] = dI;
        C.rp[I + 1] = (int64_t)C.ci.size();
    }
    return C;
}

// Dense inverse of the SPD matrix of a (small) level by Cholesky; column-major n x n.  The row
// and column of `skip` (the trimmed vertex, when level 0 itself is the coarsest) become identity.
static bool dense_inverse(const HostLevel& A, int64_t skip, std::vector<double>& inv) {
    const int64_t n = A.n;
    std::vector<double> M(n * n, 0.0);
    for (int64_t i = 0; i < n; ++i) {
        M[i + i * n] = A.d[i];
        for (int64_t e = A.rp[i]; e < A.rp[i + 1]; ++e) M[i + (int64_t)A.ci[e] * n] -= A.w[e];
    }
    if (skip >= 0 && skip < n) {
        for (int64_t i = 0; i < n; ++i) {
            M[i + skip * n] = 0.0;
            M[skip + i * n] = 0.0;
        }
        M[skip + skip * n] = 1.0;
    }
    // Cholesky M = L L^T in place (lower triangle)
    for (int64_t j = 0; j < n; ++j) {
        double s = M[j + j * n];
        for (int64_t k = 0; k < j; ++k) s -= M[j + k * n] * M[j + k * n];
        if (!(s > 0.0)) return false;
        const double ljj = std::sqrt(s);
        M[j + j * n] = ljj;
        for (int64_t i = j + 1; i < n; ++i) {
            double t = M[i + j * n];
            for (int64_t k = 0; k < j; ++k) t -= M[i + k * n] * M[j + k * n];
            M[i + j * n] = t / ljj;
        }
    }
    inv.assign(n * n, 0.0);
    std::vector<double> y(n);
    for (int64_t c = 0; c < n; ++c) {
        for (int64_t i = 0; i < n; ++i) {
            double t = (i == c) ? 1.0 : 0.0;
            for (int64_t k = 0; k < i; ++k) t -= M[i + k * n] * y[k];
            y[i] = t / M[i + i * n];
        }
        for (int64_t i = n - 1; i >= 0; --i) {
            double t = y[i];
            for (int64_t k = i + 1; k < n; ++k) t -= M[k + i * n] * y[k];
            y[i] = t / M[i + i * n];
        }
        for (int64_t i = 0; i < n; ++i) inv[i + c * n] = y[i];
    }
    return true;
}

// ------------------------------------------------------------------ device kernels of the V-cycle

template <typename T>
__global__ void __launch_bounds__(kThreads) k_ml_stage(const T* __restrict__ x, const int32_t* __restrict__ perm,
                                                       const T* __restrict__ dinv, T om, int64_t n, int64_t skip,
                                                       T* __restrict__ b, T* __restrict__ x0) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const T v = x[perm ? perm[i] : i];
        b[i] = v;
        x0[i] = i == skip ? T(0) : om * v * dinv[i];
    }
}

// Level 0 -> 1: bc[I] = sum over the members i of cluster I of the residual res_i = (1 - w) b_i + (W x0)_i that the
// gather stored, and qc = bc / dc for level 1's first smoothing step (null: level 1 is the coarsest).
// One thread per cluster, four member indices and then four residuals in flight, added in member order:
// the sums on the way down cancel (the trimmed Laplacian is nearly singular), so their order shows in FP32.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_ml_restrict(const T* __restrict__ res, const int64_t* __restrict__ mrp,
                                                          const int32_t* __restrict__ mem, int64_t nc,
                                                          T* __restrict__ bc, const T* __restrict__ dinvc,
                                                          T* __restrict__ qc, const int* __restrict__ done) {
    if (done && *done) return;
    for (int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; I < nc; I += (int64_t)gridDim.x * blockDim.x) {
        T s = T(0);
        const int64_t end = mrp[I + 1];
        for (int64_t q = mrp[I]; q < end; q += 4) {
            int32_t i[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) i[u] = q + u < end ? mem[q + u] : -1;
            T v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = i[u] >= 0 ? res[i[u]] : T(0);
#pragma unroll
            for (int u = 0; u < 4; ++u) s += v[u];
        }
        bc[I] = s;
        if (qc) qc[I] = s * dinvc[I];
    }
}

// level 0: x1 = x0 + a xc[agg(i)]; the excluded vertex stays 0
template <typename T>
__global__ void __launch_bounds__(kThreads) k_ml_prolong(const T* __restrict__ x0, const int32_t* __restrict__ agg,
                                                         const T* __restrict__ xc, T alpha, int64_t n,
                                                         T* __restrict__ x1, const int* __restrict__ done) {
    if (done && *done) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t I = agg[i];
        x1[i] = I < 0 ? T(0) : x0[i] + alpha * xc[I];
    }
}

// level 0's post-smoothing: out = x1 + w D^{-1} (b - d x1 + W x1), (W x1) from the gather; out in the caller's
// numbering if perm is given
template <typename T>
__global__ void __launch_bounds__(kThreads) k_ml_post(const T* __restrict__ b, const T* __restrict__ dinv,
                                                      const T* __restrict__ x1, const T* __restrict__ wx1, T om,
                                                      int64_t n, int64_t skip, T* __restrict__ out,
                                                      const int32_t* __restrict__ perm,
                                                      const int* __restrict__ done) {
    if (done && *done) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const T xi = x1[i], di = dinv[i];
        const T x = xi + om * (b[i] * di - xi + wx1[i] * di);
        out[perm ? perm[i] : i] = i == skip ? T(0) : x;
    }
}

// Levels l >= 1 (no excluded vertex there).  The rows are ordered by cluster (ml_build), so the members of
// cluster I are the rows mrp[I] .. mrp[I+1]-1 and their entries one contiguous CSR range.  Every level's
// q = D^{-1} b (x0 = w q) is written by the kernel that forms its b, and its x1 = x0 + a P xc by the kernel that
// forms xc (a coarse row writes its members), so a sweep gathers one vector and a level takes two launches:
//   down  bc[I] = sum_{i in I} ((1 - w) b_i + w sum_{c in N(i)} w_ic q_c)     (restricted residual)
//   up    out_i = x1_i + w (b_i - d_i x1_i + sum_c w_ic x1_c) / d_i
// Both are bound by the latency of their index -> value chains, so a lane keeps four in flight.
// (Forming x0 and x1 of the neighbours per entry instead cost two and three gathers: 12.1 and 14.3 us a
// sweep on the 118 x 109 x 101 grid's level 1.)

// stores x1 of the level below for the members of row I: x1_i = w q_i + alpha xI; G lanes (j of G)
template <typename T>
__device__ __forceinline__ void ml_store_members(const int64_t* __restrict__ mrp, const T* __restrict__ q, T om, T alpha,
                                                 T xI, int64_t I, int j, int G, T* __restrict__ x1) {
    for (int64_t i = mrp[I] + j; i < mrp[I + 1]; i += G) x1[i] = om * q[i] + alpha * xI;
}

// coarsest level: x = A^{-1} b with the dense inverse, one warp per row (the inverse is symmetric,
// so row i is column i: coalesced)
template <typename T>
__global__ void __launch_bounds__(kThreads) k_ml_dense(const T* __restrict__ inv, const T* __restrict__ b, int64_t n,
                                                       T* __restrict__ x, const int64_t* __restrict__ mrp,
                                                       const T* __restrict__ q, T om, T alpha, T* __restrict__ x1,
                                                       const int* __restrict__ done) {
    if (done && *done) return;
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = w0; i < n; i += nw) {
        T s = T(0);
#pragma unroll 4
        for (int64_t j = lane; j < n; j += 32) s += inv[j + i * n] * b[j];
        s = warp_sum(s);
        if (lane == 0) x[i] = s;
        if (x1) ml_store_members(mrp, q, om, alpha, s, i, lane, 32, x1);
    }
}

// one warp per cluster, lanes striding over its rows and its entries (coalesced)
template <typename T>
__global__ void __launch_bounds__(kThreads) k_ml_down(const T* __restrict__ b, const int32_t* __restrict__ rp,
                                                      const int32_t* __restrict__ ci, const T* __restrict__ w,
                                                      const int64_t* __restrict__ mrp, const T* __restrict__ qv, T om,
                                                      int64_t nc, T* __restrict__ bc, const T* __restrict__ dinvc,
                                                      T* __restrict__ qc, const int* __restrict__ done) {
    if (done && *done) return;
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t I = w0; I < nc; I += nw) {
        const int64_t r_beg = mrp[I], r_end = mrp[I + 1];
        const int32_t e_end = rp[r_end];
        T own = T(0), s = T(0);
        for (int64_t i = r_beg + lane; i < r_end; i += 32) own += b[i];
        for (int32_t e = rp[r_beg] + lane; e < e_end; e += 128) {
            int32_t c[4];
            T v[4], q[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool ok = e + 32 * u < e_end;
                c[u] = ok ? ci[e + 32 * u] : -1;
                q[u] = ok ? w[e + 32 * u] : T(0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = c[u] >= 0 ? qv[c[u]] : T(0);
            s += q[0] * v[0];
            s += q[1] * v[1];
            if (e - lane + 64 < e_end) {
                s += q[2] * v[2];
                s += q[3] * v[3];
            }
        }
        s *= om;
        const T acc = warp_sum((T(1) - om) * own + s);
        if (lane == 0) {
            bc[I] = acc;
            if (qc) qc[I] = acc * dinvc[I];
        }
    }
}

// The same for a small level above the coarsest (at most kMlRowsMax rows): one warp per cluster, a lane per
// member row, its entries in order.  Few clusters leave the entry-strided form short of warps, and the
// row's own residual is what the sums on the way down are made of.
constexpr int kMlRowsMax = 4096;

template <typename T>
__global__ void __launch_bounds__(kThreads) k_ml_down_rows(const T* __restrict__ b, const int32_t* __restrict__ rp,
                                                           const int32_t* __restrict__ ci, const T* __restrict__ w,
                                                           const int64_t* __restrict__ mrp, const T* __restrict__ qv,
                                                           T om, int64_t nc, T* __restrict__ bc,
                                                           const int* __restrict__ done) {
    if (done && *done) return;
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t I = w0; I < nc; I += nw) {
        T acc = T(0);
        for (int64_t i = mrp[I] + lane; i < mrp[I + 1]; i += 32) {
            T s = T(0);
            const int32_t e_end = rp[i + 1];
            for (int32_t e = rp[i]; e < e_end; e += 4) {
                int32_t c[4];
                T v[4], q[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    c[u] = e + u < e_end ? ci[e + u] : -1;
                    q[u] = e + u < e_end ? w[e + u] : T(0);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = c[u] >= 0 ? qv[c[u]] : T(0);
#pragma unroll
                for (int u = 0; u < 4; ++u) s += q[u] * v[u];
            }
            acc += (T(1) - om) * b[i] + om * s;
        }
        acc = warp_sum(acc);
        if (lane == 0) bc[I] = acc;
    }
}

// G lanes per row; out (level 1: the prolongation to level 0 reads it) or the members' x1 one level below
template <typename T, int G>
__global__ void __launch_bounds__(kThreads) k_ml_up(const T* __restrict__ b, const T* __restrict__ dinv,
                                                    const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                                    const T* __restrict__ w, const T* __restrict__ x1, T om, T alpha,
                                                    int64_t n, T* __restrict__ out, const int64_t* __restrict__ mrp,
                                                    const T* __restrict__ qf, T* __restrict__ x1f,
                                                    const int* __restrict__ done) {
    if (done && *done) return;
    const int64_t groups = ((int64_t)gridDim.x * blockDim.x) / G;
    const int64_t g0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int64_t passes = (n + groups - 1) / groups;
    const int j = threadIdx.x & (G - 1);
    for (int64_t p = 0; p < passes; ++p) {
        const int64_t row = g0 + p * groups;
        const bool valid = row < n;
        T s0 = T(0), s1 = T(0);
        if (valid) {
            const int32_t e_end = rp[row + 1];
            for (int32_t e = rp[row] + j; e < e_end; e += 4 * G) {
                int32_t c[4];
                T v[4], q[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool ok = e + G * u < e_end;
                    c[u] = ok ? ci[e + G * u] : -1;
                    q[u] = ok ? w[e + G * u] : T(0);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = c[u] >= 0 ? x1[c[u]] : T(0);
                s0 += q[0] * v[0] + q[1] * v[1];
                s1 += q[2] * v[2] + q[3] * v[3];
            }
        }
        T s = s0 + s1;
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        if (valid) {
            const T di = dinv[row], xi = x1[row];
            const T x = xi + om * (b[row] * di - xi + s * di);
            if (x1f) ml_store_members(mrp, qf, om, alpha, x, row, j, G, x1f);
            else if (j == 0) out[row] = x;
        }
    }
}

// ------------------------------------------------------------------ hierarchy

template <typename T>
static void upload(T** dst, const std::vector<double>& src) {
    std::vector<T> tmp(src.begin(), src.end());
    CUDA_OK(cudaMalloc(dst, sizeof(T) * std::max<size_t>(1, tmp.size())));
    if (!tmp.empty()) CUDA_OK(cudaMemcpy(*dst, tmp.data(), sizeof(T) * tmp.size(), cudaMemcpyHostToDevice));
}

template <typename I>
static void upload_i(I** dst, const std::vector<I>& src) {
    CUDA_OK(cudaMalloc(dst, sizeof(I) * std::max<size_t>(1, src.size())));
    if (!src.empty()) CUDA_OK(cudaMemcpy(*dst, src.data(), sizeof(I) * src.size(), cudaMemcpyHostToDevice));
}

// Sampled cost of level 0's gathers in a numbering (order: new -> old; null: as it is): the 128-byte lines that
// the warp-wide loads of x touch, counting a column of a slice, also a padded one, as at least one; *cols
// receives the number of columns.
static int64_t gather_lines(const HostLevel& A, const std::vector<int32_t>* order, const std::vector<int32_t>& pos,
                            int64_t* cols) {
    const int64_t ns = A.n / 32, step = std::max<int64_t>(1, ns / 256);
    int64_t lines = 0;
    int32_t ln[32];
    *cols = 0;
    for (int64_t s = 0; s < ns; s += step) {
        int64_t wid = 0;
        for (int64_t r = 32 * s; r < 32 * s + 32; ++r) {
            const int64_t i = order ? (*order)[r] : r;
            wid = std::max(wid, A.rp[i + 1] - A.rp[i]);
        }
        *cols += wid;
        for (int64_t q = 0; q < wid; ++q) {
            int m = 0;
            for (int64_t r = 32 * s; r < 32 * s + 32; ++r) {
                const int64_t i = order ? (*order)[r] : r;
                if (A.rp[i] + q < A.rp[i + 1]) {
                    const int32_t c = A.ci[A.rp[i] + q];
                    ln[m++] = (order ? pos[c] : c) >> 5;
                }
            }
            std::sort(ln, ln + m);
            lines += std::max<int64_t>(1, std::unique(ln, ln + m) - ln);
        }
    }
    return lines;
}

// A numbering of level 0 that keeps clusters, and clusters of clusters, together (level 1's numbers are
// hierarchical), with the rows of every kMlWindow consecutive ones by descending degree, so that the slices of
// 32 rows stay nearly unpadded.
constexpr int64_t kMlWindow = 128;

static std::vector<int32_t> cluster_order(const HostLevel& A, const std::vector<int32_t>& agg, int64_t nc) {
    std::vector<int64_t> start(nc + 2, 0);                 // the excluded vertex (-1) goes last
    for (int64_t i = 0; i < A.n; ++i) start[(agg[i] < 0 ? nc : agg[i]) + 1]++;
    for (int64_t I = 0; I <= nc; ++I) start[I + 1] += start[I];
    std::vector<int32_t> order(A.n);
    for (int64_t i = 0; i < A.n; ++i) order[start[agg[i] < 0 ? nc : agg[i]]++] = (int32_t)i;
    // counting sort of each window (all rows are sliced: degrees up to 64)
    constexpr int kDeg = 65;
    int32_t deg[kMlWindow], row[kMlWindow];
    for (int64_t w = 0; w < A.n; w += kMlWindow) {
        const int m = (int)std::min(kMlWindow, A.n - w);
        int cnt[kDeg + 1] = {};
        for (int t = 0; t < m; ++t) {
            row[t] = order[w + t];
            deg[t] = kDeg - 1 - (int32_t)std::min<int64_t>(kDeg - 1, A.rp[row[t] + 1] - A.rp[row[t]]);
            ++cnt[deg[t] + 1];
        }
        for (int d = 0; d < kDeg; ++d) cnt[d + 1] += cnt[d];
        for (int t = 0; t < m; ++t) order[w + cnt[deg[t]]++] = row[t];
    }
    return order;
}

template <typename T>
cudaError_t ml_build(MlHierarchy<T>& H, const int64_t* d_rp, const int32_t* d_ci, const double* d_w, int64_t n,
                     int64_t ld, int64_t skip, const std::vector<int32_t>& visit, std::vector<int32_t>* place,
                     cudaStream_t s) {
    try {
        HostLevel A0;
        A0.n = n;
        A0.rp.resize(n + 1);
        CUDA_OK(cudaMemcpyAsync(A0.rp.data(), d_rp, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToHost, s));
        CUDA_OK(cudaStreamSynchronize(s));
        A0.ci.resize(A0.rp[n]);
        CUDA_OK(cudaMemcpyAsync(A0.ci.data(), d_ci, sizeof(int32_t) * A0.rp[n], cudaMemcpyDeviceToHost, s));
        CUDA_OK(cudaStreamSynchronize(s));
        A0.w.assign(A0.rp[n], 1.0);
        if (d_w) {
            CUDA_OK(cudaMemcpyAsync(A0.w.data(), d_w, sizeof(double) * A0.rp[n], cudaMemcpyDeviceToHost, s));
            CUDA_OK(cudaStreamSynchronize(s));
        }
        // the rows in their degree-descending order (old); pos: old -> the numbering in use
        std::vector<int32_t> order = visit, pos;
        if (!order.empty()) {
            pos.resize(n);
            for (int64_t r = 0; r < n; ++r) pos[order[r]] = (int32_t)r;
            HostLevel B;
            B.n = n;
            B.rp.assign(n + 1, 0);
            B.ci.resize(A0.ci.size());
            B.w.resize(A0.w.size());
            for (int64_t i = 0; i < n; ++i) {
                int64_t e2 = B.rp[i];
                for (int64_t e = A0.rp[pos[i]]; e < A0.rp[pos[i] + 1]; ++e, ++e2) {
                    B.ci[e2] = order[A0.ci[e]];
                    B.w[e2] = A0.w[e];
                }
                B.rp[i + 1] = e2;
            }
            A0 = std::move(B);
        }
        const int64_t skip_old = order.empty() || skip < 0 ? skip : order[skip];
        A0.d.assign(n, 0.0);
        for (int64_t i = 0; i < n; ++i)
            for (int64_t e = A0.rp[i]; e < A0.rp[i + 1]; ++e) A0.d[i] += A0.w[e];
        H.n0 = n;
        std::vector<HostLevel> levels;
        levels.push_back(std::move(A0));
        std::vector<std::vector<int32_t>> aggs;
        while ((int)levels.size() < kMlMaxLevels && levels.back().n > kMlCoarse) {
            int64_t nc = 0;
            const int64_t sk = levels.size() == 1 ? skip_old : -1;
            std::vector<int32_t> agg = aggregate(levels.back(), sk, &nc);
            if (nc >= levels.back().n * 9 / 10 || nc < 1) break;    // no useful coarsening left
            HostLevel C = coarsen(levels.back(), agg, nc);
            aggs.push_back(std::move(agg));
            levels.push_back(std::move(C));
        }
        // Order the rows of every level l >= 1 that has a next level by cluster (stable), from the
        // coarse end down, so that cluster ids are final when their members are sorted: the members
        // of a cluster become consecutive rows in increasing cluster order, and the down sweep reads
        // one contiguous range per cluster.
        for (int l = (int)levels.size() - 2; l >= 1; --l) {
            const HostLevel& A = levels[l];
            std::vector<int32_t>& ag = aggs[l];
            std::vector<int64_t> order(A.n), pos(A.n);
            std::iota(order.begin(), order.end(), (int64_t)0);
            std::stable_sort(order.begin(), order.end(), [&](int64_t x, int64_t y) { return ag[x] < ag[y]; });
            for (int64_t p = 0; p < A.n; ++p) pos[order[p]] = p;
            HostLevel B;
            B.n = A.n;
            B.rp.assign(A.n + 1, 0);
            B.d.resize(A.n);
            B.ci.reserve(A.ci.size());
            B.w.reserve(A.w.size());
            std::vector<int32_t> ag2(A.n);
            for (int64_t p = 0; p < A.n; ++p) {
                const int64_t i = order[p];
                B.d[p] = A.d[i];
                for (int64_t e = A.rp[i]; e < A.rp[i + 1]; ++e) {
                    B.ci.push_back((int32_t)pos[A.ci[e]]);
                    B.w.push_back(A.w[e]);
                }
                B.rp[p + 1] = (int64_t)B.ci.size();
                ag2[p] = ag[i];
            }
            levels[l] = std::move(B);
            ag = std::move(ag2);
            for (int32_t& x : aggs[l - 1])
                if (x >= 0) x = (int32_t)pos[x];
        }
        const int L = (int)levels.size();
        if (place) {
            place->clear();
            // Worth the second relabelling where it halves the lines.  A random geometric graph numbered at random
            // touches a line per entry (45 us a gather of 1M vertices, 41 us of them lines at one per cycle and
            // SM; 20 us relabelled); a grid in its own order touches two or three per column of a slice, which
            // no numbering halves: below six the order is not even formed.
            int64_t cols = 0, cols_new = 0;
            const int64_t lines = L > 1 && order.empty() ? gather_lines(levels[0], nullptr, pos, &cols) : 0;
            if (lines >= 6 * std::max<int64_t>(1, cols)) {
                std::vector<int32_t> o = cluster_order(levels[0], aggs[0], levels[1].n), p(n);
                for (int64_t r = 0; r < n; ++r) p[o[r]] = (int32_t)r;
                if (2 * gather_lines(levels[0], &o, p, &cols_new) < lines) {
                    *place = o;
                    order = std::move(o);
                    pos = std::move(p);
                }
            }
        }
        H.skip = order.empty() || skip_old < 0 ? skip_old : pos[skip_old];
        H.nlev = L;
        H.lev.assign(L, MlLevel<T>{});
        for (int l = 0; l < L; ++l) {
            MlLevel<T>& D = H.lev[l];
            const HostLevel& A = levels[l];
            D.n = A.n;
            D.nnz = (int64_t)A.ci.size();
            std::vector<double> dinv(l == 0 ? ld : A.n, 0.0);
            auto place_of = [&](int64_t i) { return l == 0 && !pos.empty() ? (int64_t)pos[i] : i; };
            for (int64_t i = 0; i < A.n; ++i) dinv[place_of(i)] = (l == 0 && i == skip_old) ? 0.0 : 1.0 / A.d[i];
            upload<T>(&D.dinv, dinv);
            if (l > 0) {
                std::vector<int32_t> rp32(A.n + 1);
                for (int64_t i = 0; i <= A.n; ++i) rp32[i] = (int32_t)A.rp[i];
                upload_i<int32_t>(&D.rp, rp32);
                upload_i<int32_t>(&D.ci, A.ci);
                upload<T>(&D.w, A.w);
            }
            const size_t nv = (size_t)(l == 0 ? ld : A.n);
            CUDA_OK(cudaMalloc(&D.b, sizeof(T) * nv));
            CUDA_OK(cudaMalloc(&D.x0, sizeof(T) * nv));
            CUDA_OK(cudaMalloc(&D.x1, sizeof(T) * nv));
            CUDA_OK(cudaMalloc(&D.x, sizeof(T) * nv));
            CUDA_OK(cudaMemsetAsync(D.x0, 0, sizeof(T) * nv, s));
            CUDA_OK(cudaMemsetAsync(D.x1, 0, sizeof(T) * nv, s));
            if (l + 1 < L) {
                // cluster boundaries; the coarse rows are ordered by cluster, level 0's are not: it also takes
                // the cluster of every row and the members of every cluster
                const std::vector<int32_t>& agg = aggs[l];
                const int64_t nc = levels[l + 1].n;
                std::vector<int64_t> mrp(nc + 1, 0);
                for (int32_t I : agg)
                    if (I >= 0) mrp[I + 1]++;
                for (int64_t I = 0; I < nc; ++I) mrp[I + 1] += mrp[I];
                upload_i<int64_t>(&D.mrp, mrp);
                if (l == 0) {
                    std::vector<int32_t> agg_pad(nv, -1), mem(mrp[nc]);
                    std::vector<int64_t> fill(mrp.begin(), mrp.end() - 1);
                    for (int64_t i = 0; i < (int64_t)agg.size(); ++i) {
                        agg_pad[place_of(i)] = agg[i];
                        if (agg[i] >= 0) mem[fill[agg[i]]++] = (int32_t)place_of(i);   // members in the old order
                    }
                    upload_i<int32_t>(&D.agg, agg_pad);
                    upload_i<int32_t>(&D.mem, mem);
                }
            }
        }
        std::vector<double> inv;
        if (!dense_inverse(levels[L - 1], L == 1 ? skip_old : -1, inv)) throw CudaFailure{cudaErrorInvalidValue};
        upload<T>(&H.inv, inv);
        H.n_coarse = levels[L - 1].n;
        CUDA_OK(cudaStreamSynchronize(s));
    } catch (CudaFailure& f) {
        ml_free<T>(H);                       // nothing half built stays: the next call builds again
        return f.e;
    } catch (std::bad_alloc&) {
        ml_free<T>(H);
        return cudaErrorMemoryAllocation;
    }
    return cudaSuccess;
}

template <typename T>
void ml_free(MlHierarchy<T>& H) {
    for (MlLevel<T>& D : H.lev) {
        void* ptrs[] = {D.dinv, D.rp, D.ci, D.w, D.agg, D.mrp, D.mem, D.b, D.x0, D.x1, D.x};
        for (void* p : ptrs)
            if (p) cudaFree(p);
    }
    if (H.inv) cudaFree(H.inv);
    H.lev.clear();
    H.inv = nullptr;
    H.nlev = 0;
}

static int ml_grid(int64_t n) {
    const int64_t g = (n + kThreads - 1) / kThreads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, 1216));
}

static int ml_warp_grid(int64_t n) {
    const int64_t g = (n * 32 + kThreads - 1) / kThreads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, 2432));
}

static int ml_group_grid(int64_t n, int G) {
    const int64_t g = (n * G + kThreads - 1) / kThreads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, 2432));
}

constexpr int kMlLanes = 4;          // lanes per coarse CSR row

// out = M^{-1} b (b on level 0, n-space, the trimmed entry ignored; out may alias nothing else).
// gather(x, res, g) must compute g = W x (+ (1 - omega) res, if res is not null) for level 0.
// Level 0's x0 = w D^{-1} b is in H.lev[0].x0 already (nlev >= 2; written by the caller's kernel).
// skip_post0 (nlev >= 2): stop before the gather of x1 (H.lev[0].x1) that the caller's next kernels make, with
// level 0's post-smoothing (out is then not written).
template <typename T>
void ml_vcycle(MlHierarchy<T>& H, const T* b, T* out, const GatherFn<T>& gather, T omega, T alpha, const int* done,
               bool skip_post0, const int32_t* perm, cudaStream_t s) {
    const int L = H.nlev;
    MlLevel<T>& F = H.lev[0];
    if (L == 1) {
        k_ml_dense<T><<<ml_warp_grid(F.n), kThreads, 0, s>>>(H.inv, b, F.n, out, nullptr, nullptr, omega, alpha,
                                                             nullptr, done);
        return;
    }
    // level 0 down: the residual (1 - w) b + W x0 in the solver's gather, restricted
    gather(F.x0, b, F.x, s);
    {
        MlLevel<T>& C = H.lev[1];
        k_ml_restrict<T><<<ml_grid(C.n), kThreads, 0, s>>>(F.x, F.mrp, F.mem, C.n, C.b, C.dinv,
                                                          L > 2 ? C.x0 : nullptr, done);
    }
    for (int l = 1; l + 1 < L; ++l) {
        MlLevel<T>& D = H.lev[l];
        MlLevel<T>& C = H.lev[l + 1];
        if (l + 2 == L && D.n <= kMlRowsMax)
            k_ml_down_rows<T><<<ml_warp_grid(C.n), kThreads, 0, s>>>(D.b, D.rp, D.ci, D.w, D.mrp, D.x0, omega, C.n, C.b,
                                                                     done);
        else
            k_ml_down<T><<<ml_warp_grid(C.n), kThreads, 0, s>>>(D.b, D.rp, D.ci, D.w, D.mrp, D.x0, omega, C.n, C.b,
                                                                C.dinv, l + 2 < L ? C.x0 : nullptr, done);
    }
    {
        MlLevel<T>& C = H.lev[L - 1];
        MlLevel<T>& D = H.lev[L - 2];
        const bool below = L > 2;                                    // level L - 2 is not level 0
        k_ml_dense<T><<<ml_warp_grid(C.n), kThreads, 0, s>>>(H.inv, C.b, C.n, C.x, D.mrp, D.x0, omega, alpha,
                                                             below ? D.x1 : nullptr, done);
    }
    for (int l = L - 2; l >= 1; --l) {
        MlLevel<T>& D = H.lev[l];
        MlLevel<T>& B = H.lev[l - 1];
        k_ml_up<T, kMlLanes><<<ml_group_grid(D.n, kMlLanes), kThreads, 0, s>>>(
            D.b, D.dinv, D.rp, D.ci, D.w, D.x1, omega, alpha, D.n, D.x, B.mrp, B.x0, l > 1 ? B.x1 : nullptr, done);
    }
    // level 0 up: prolong, neighbour sums of x1, post-smooth
    k_ml_prolong<T><<<ml_grid(F.n), kThreads, 0, s>>>(F.x0, F.agg, H.lev[1].x, alpha, F.n, F.x1, done);
    if (skip_post0) return;
    gather(F.x1, nullptr, F.x0, s);                                  // F.x0 <- W x1 (x0 is free now)
    k_ml_post<T><<<ml_grid(F.n), kThreads, 0, s>>>(b, F.dinv, F.x1, F.x0, omega, F.n, H.skip, out, perm, done);
}

// launches of one call (without the caller's gather of x1 when skip_post0)
template <typename T>
int ml_launches(const MlHierarchy<T>& H, bool skip_post0) {
    if (H.nlev <= 1) return 1;
    return 2 + 2 * (H.nlev - 2) + 1 + 1 + (skip_post0 ? 0 : 2);
}

// b = x (the caller's vector and numbering) and level 0's x0 = w D^{-1} b
template <typename T>
void ml_stage(MlHierarchy<T>& H, const T* x, const int32_t* perm, T omega, T* b, cudaStream_t s) {
    MlLevel<T>& F = H.lev[0];
    k_ml_stage<T><<<ml_grid(F.n), kThreads, 0, s>>>(x, perm, F.dinv, omega, F.n, H.skip, b, F.x0);
}

#define ISIRA_INSTANTIATE_ML(T)                                                                              \
    template cudaError_t ml_build<T>(MlHierarchy<T>&, const int64_t*, const int32_t*, const double*, int64_t,  \
                                     int64_t, int64_t, const std::vector<int32_t>&, std::vector<int32_t>*,   \
                                     cudaStream_t);                                                          \
    template void ml_free<T>(MlHierarchy<T>&);                                                               \
    template void ml_vcycle<T>(MlHierarchy<T>&, const T*, T*, const GatherFn<T>&, T, T, const int*, bool,     \
                               const int32_t*, cudaStream_t);                                                \
    template void ml_stage<T>(MlHierarchy<T>&, const T*, const int32_t*, T, T*, cudaStream_t);               \
    template int ml_launches<T>(const MlHierarchy<T>&, bool);
ISIRA_INSTANTIATE_ML(float)
ISIRA_INSTANTIATE_ML(double)

}  // namespace isira
