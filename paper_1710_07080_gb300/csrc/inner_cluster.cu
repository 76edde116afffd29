// inner_cluster.cu -- the whole diagonally preconditioned inner solve of a small graph in one launch.
//
// On a small graph an iteration of the three-launch solve (inner_impl.cuh) is launch and latency
// bound: three kernels of a few microseconds each around a few hundred nanoseconds of work, plus the
// turn of the WHILE node.  Here one thread-block cluster runs the solve from the right-hand side to
// the FP64 result: the CTAs own the rows, every Krylov vector but z_k lives in shared memory, z_k is
// exchanged through L2 (written by its owner, gathered by everybody), and the two reductions of an
// iteration travel through distributed shared memory.  Two cluster barriers an iteration are all the
// synchronisation: the first ends phase 1 (its sums, and the last gather of z_k), the second ends
// phase 2 (its sums, and z_{k+1}).  Every CTA forms the scalars from the same values in the same
// order, so all of them stop at the same iteration.
//
// Arithmetic as in k_phase1 / k_phase2 / minres_step; sums are taken per thread, per warp, per CTA
// and over the CTAs in a fixed order that depends on the graph and on c only.
//
// What bounds an iteration: in FP32 the chain of two reductions and two cluster barriers (2.3 us on 20
// vertices, 3.5 us on a grid of 9,856) and, on random graphs, the lines that the gathers touch; in FP64
// the FP64 pipe, which issues a warp instruction every 16 to 19 cycles on an SM: hence few warps (a warp
// reduction costs as much as a row), D z kept instead of D, folded w coefficients, additions only
// where a slice has entries, and the w / x update placed under the first barrier (9.3 us on the grid of
// 9,856; 13.3 us before those).
#include <algorithm>

#include "internal.h"

namespace isira {

namespace {

constexpr int kClMaxCtas = 16;
// most threads of a CTA: a lane per row for FP32; the FP64 rows are bound by the FP64 pipe, not by
// latency, and want the registers
template <typename T> struct ClThreads { static constexpr int value = sizeof(T) == 4 ? 1024 : 256; };
constexpr int kClMaxWarps = 32;
constexpr int kClMaxC = kCMax - 1;
constexpr int kClVecs = 10;                // shared vectors per row: z (2), D z (2), Y, w (2), x, deg - sigma, 1/D

__device__ __forceinline__ unsigned cl_addr(const void* p, unsigned rank) {
    unsigned a = smem_u32(p), r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cl_store(unsigned a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" :: "r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_store(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" :: "r"(a), "d"(v) : "memory");
}
// release / acquire at cluster scope: orders the shared and global writes of all CTAs of the cluster
__device__ __forceinline__ void cl_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_barrier() {
    cl_arrive();
    cl_wait();
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

template <typename T> struct ClVec;
template <> struct ClVec<float> { static constexpr int N = 4; using V = float4; };
template <> struct ClVec<double> { static constexpr int N = 2; using V = double2; };

template <typename T>
struct ClShared {
    T in1[1 + 2 * kClMaxC][kClMaxCtas + 1];     // phase 1 sums of every CTA (padded rows: no bank conflicts)
    T in2[2][kClMaxCtas];                       // phase 2 sums of every CTA
    T red[2][kClMaxWarps];
    T col[2][kClMaxWarps];                      // partial column sums (one warp each)
    T tv[kClMaxC], as[kClMaxC];
    double gc[kClMaxC], uc[kClMaxC];
    double Ci[kClMaxC * kClMaxC];               // C^{-1}
    double CG[kClMaxC * kClMaxC];               // C^{-1} G
    // scalars of the current iteration
    T inv_beta, cprev, s_term, wz, w2c, w1c, phi, coef;
    double inv_beta_d;
    int done, itn, pending;
};

// pairwise sum of the CTAs' contributions (slots beyond the cluster are zero)
template <typename T>
__device__ __forceinline__ T cl_total(const T* v) {
    T s[kClMaxCtas];
#pragma unroll
    for (int i = 0; i < kClMaxCtas; ++i) s[i] = v[i];
#pragma unroll
    for (int o = kClMaxCtas / 2; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < o; ++i) s[i] += s[i + o];
    return s[0];
}

// Sum of the r gathered values of a pass (r uniform over the warp).  FP64: only the additions that
// the width needs, since one SM issues an FP64 warp instruction every 16 to 19 cycles; FP32: all eight.
template <typename T>
__device__ __forceinline__ T cl_pass_sum(const T (&v)[8], int r) {
    if constexpr (sizeof(T) == 4) return ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    return pass_sum(v, r);
}

}  // namespace

// Rows are dealt to the CTAs by slices of 32 (slice s to CTA s mod P): the numbering is by
// descending degree, so contiguous ranges would give the first CTA the longest rows.  Warp w of a
// CTA takes its local slices w, w + W, ..., a lane one row, the same lane in every phase.
template <typename T>
__global__ void __launch_bounds__(ClThreads<T>::value, 1) k_minres_cluster(InnerArgs<T> a, const double* R,
                                                                     const double* rnorm_dev, double* Z, int cap,
                                                                     int staged, int prof) {
    extern __shared__ __align__(16) unsigned char cl_dyn[];
    __shared__ ClShared<T> sh;
    T* zc = reinterpret_cast<T*>(cl_dyn);
    T* zp = zc + cap;
    T* Qc = zp + cap;                          // D z_k, D z_{k-1}: phase 2 has them before it divides by D
    T* Qp = Qc + cap;
    T* Y = Qp + cap;
    T* w1 = Y + cap;
    T* w2 = w1 + cap;
    T* x = w2 + cap;
    T* Ad = x + cap;
    T* di = Ad + cap;
    T* zs = di + cap;                          // staged: the whole of z_k, ld entries
    const RowSched& S = a.rs;
    const int P = gridDim.x, rank = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = blockDim.x >> 5;
    const int c = a.c;
    const int64_t n = S.n, trim = a.trim;
    const int nsl = rank < S.n_slices ? (S.n_slices - rank + P - 1) / P : 0;
    const T* __restrict__ sw = S.swts<T>();
    const double delta = (double)a.delta;
    T* zg = a.z0;

    // sums over the warps' slots of red[0] (lanes 0-15) and red[1] (lanes 16-31)
    auto sum_red = [&]() -> T {
        const int v = lane >> 4, i = lane & 15;
        T s = i < W ? sh.red[v][i] : T(0);
        if (W > 16) s += i + 16 < W ? sh.red[v][i + 16] : T(0);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
            if (o < W) s += __shfl_xor_sync(kFull, s, o);
        return __shfl_sync(kFull, s, lane & 16);
    };
    // sum of the two per-lane values over the CTA, sent to slot `rank` of in2[0], in2[1] in every CTA
    auto send2 = [&](T v0, T v1) {
        const T v[2] = {v0, v1};
        T o[1];
        warp_reduce_multi<T, 2>(v, o);
        if ((lane & 15) == 0) sh.red[lane >> 4][warp] = o[0];
        __syncthreads();
        if (warp == 0) {
            const T s = sum_red();
            if ((lane & 15) < P) cl_store(cl_addr(&sh.in2[lane >> 4][rank], lane & 15), s);
        }
    };
    // column sums (Vh^T D^{-1} Y)_t and (Vh^T z)_t: the warps are dealt to the columns, several to a column
    // while there are more warps than columns
    const int parts = c > 0 && W > c ? W / c : 1;
    auto send_columns = [&]() {
        for (int t0 = 0; t0 < c; t0 += W) {
            const int t = t0 + (parts > 1 ? warp % c : warp), part = parts > 1 ? warp / c : 0;
            T sa = T(0), sg = T(0);
            if (t < c && part < parts) {
                const T* __restrict__ col = a.Vt + (int64_t)t * a.ldv;
#pragma unroll 4
                for (int j = part; j < nsl; j += parts) {
                    const int64_t row = ((int64_t)j * P + rank) * 32 + lane;
                    const int l = j * 32 + lane;
                    const T v = row < n ? __ldg(col + row) : T(0);
                    sa += v * (Y[l] * di[l]);
                    sg += v * zc[l];
                }
            }
            const T v[2] = {sa, sg};
            T o[1];
            warp_reduce_multi<T, 2>(v, o);                  // lanes 0-15: sa, lanes 16-31: sg
            if (parts > 1) {
                if ((lane & 15) == 0) sh.col[lane >> 4][warp] = o[0];
                __syncthreads();
                if (warp < c) {
                    const int i = lane & 15;
                    o[0] = i < parts ? sh.col[lane >> 4][warp + i * c] : T(0);
                    if (parts > 16) o[0] += i + 16 < parts ? sh.col[lane >> 4][warp + (i + 16) * c] : T(0);
#pragma unroll
                    for (int s = 8; s > 0; s >>= 1)
                        if (s < parts) o[0] += __shfl_xor_sync(kFull, o[0], s);
                    o[0] = __shfl_sync(kFull, o[0], lane & 16);
                }
            }
            if (t < c && part == 0 && (lane & 15) < P)
                cl_store(cl_addr(&sh.in1[1 + (lane >> 4) * c + t][rank], lane & 15), o[0]);
        }
    };
    // phase 2: y = Y + Vh as - coef D z, z' = (y - Vh tv) / D; sums y^T z', 1^T z'.  On the trimmed and the
    // padding rows Y, D z and 1/D are zero, and so is everything formed from them.
    auto phase2 = [&]() {
        const T coef = sh.coef;
        T a0 = T(0), a1 = T(0);
        for (int j = warp; j < nsl; j += W) {
            const int64_t row = ((int64_t)j * P + rank) * 32 + lane;
            const int l = j * 32 + lane;
            const bool ok = row < n && row != trim;
            T ya = T(0), zt = T(0);
            if (ok)
                for (int t = 0; t < c; ++t) {
                    const T v = __ldg(a.Vt + (int64_t)t * a.ldv + row);
                    ya += v * sh.as[t];
                    zt += v * sh.tv[t];
                }
            T y = Y[l] - coef * Qc[l];
            if (c > 0) y += ya;
            const T q = c > 0 ? y - zt : y;
            const T z = q * di[l];
            Qp[l] = q;
            zp[l] = z;
            if (row < n) __stcg(zg + row, z);
            a0 += y * z;
            a1 += z;
        }
        send2(a0, a1);
        T* t = zc;                        // z_{k+1} becomes the current vector, z_k the previous one
        zc = zp;
        zp = t;
        t = Qc;
        Qc = Qp;
        Qp = t;
    };

    // ---------------------------------------------------------------- set-up
    {
        const double rn = *rnorm_dev;
        const double inv = rn > 0.0 ? 1.0 / rn : 0.0;
        for (int i = tid; i < (1 + 2 * kClMaxC) * (kClMaxCtas + 1); i += blockDim.x) (&sh.in1[0][0])[i] = T(0);
        for (int i = tid; i < 2 * kClMaxCtas; i += blockDim.x) (&sh.in2[0][0])[i] = T(0);
        for (int i = tid; i < c * c; i += blockDim.x) {
            sh.Ci[i] = a.Cinv[i];
            const int p = i % c, q = i / c;
            double s = 0.0;
            for (int t = 0; t < c; ++t) s += a.Cinv[p + t * c] * a.Gm[t + q * c];
            sh.CG[i] = s;
        }
        for (int j = warp; j < nsl; j += W) {
            const int64_t row = ((int64_t)j * P + rank) * 32 + lane;
            const int l = j * 32 + lane;
            const bool ok = row < n && row != trim;
            const T deg = row < n ? row_degree<T>(S, row) : T(1);
            const T m = deg - a.sigma, hf = deg * T(0.5);
            const T d = m < hf ? hf : m;
            Ad[l] = m;
            di[l] = ok ? T(1) / d : T(0);
            Y[l] = ok ? (T)(R[row] * inv) : T(0);
            zc[l] = zp[l] = Qc[l] = Qp[l] = w1[l] = w2[l] = x[l] = T(0);
        }
    }
    // the first send must not reach a CTA that has not zeroed its inbox (nor started at all)
    cl_barrier();
    double g_cur = 0.0;                       // warp 0, lane t < c: (Vh^T z_k)_t
    if (c > 0) {                              // tv = C^{-1} Vh^T D^{-1} b
        send_columns();
        cl_barrier();
        if (warp == 0) {
            if (lane < c) sh.gc[lane] = (double)cl_total(sh.in1[1 + lane]);
            __syncwarp();
            if (lane < c) {
                double tv = 0.0;
                for (int q = 0; q < c; ++q) tv += sh.Ci[lane + q * c] * sh.gc[q];
                sh.tv[lane] = (T)tv;
                sh.as[lane] = T(0);
            }
        }
    }
    if (tid == 0) { sh.coef = T(0); sh.pending = 0; sh.itn = 0; }
    __syncthreads();
    phase2();
    // the whole of z_k into shared memory (warps 1 and up, while warp 0 forms the scalars)
    auto stage = [&]() {
        if (!staged || warp == 0) return;
        using V = typename ClVec<T>::V;
        const int nv = (int)((n + ClVec<T>::N - 1) / ClVec<T>::N);
        const V* __restrict__ src = reinterpret_cast<const V*>(zg);
        V* dst = reinterpret_cast<V*>(zs);
#pragma unroll 4
        for (int i = tid - 32; i < nv; i += blockDim.x - 32) dst[i] = __ldcg(src + i);
    };
    // MINRES scalars (warp 0): beta_k, and the state of the Givens recurrence
    T beta1 = T(0), cs = T(-1), sn = T(0), dbar = T(0), epsln = T(0), phibar = T(0), alpha = T(0);
    int itn = 0;
    T d2 = T(0), gbar = T(0), gbar2 = T(0);
    // phase 2 ends: what needs only alpha_k of the Givens step is formed while the barrier completes
    auto scalars = [&](bool init) {
        cl_arrive();
        if (warp == 0 && !init) {
            d2 = cs * dbar + sn * alpha;
            gbar = sn * dbar - cs * alpha;
            gbar2 = gbar * gbar;
        }
        cl_wait();
        stage();
        if (warp == 0) {
            T s = sh.in2[lane >> 4][lane & 15];
#pragma unroll
            for (int o = kClMaxCtas / 2; o > 0; o >>= 1)
                if (o < P) s += __shfl_xor_sync(kFull, s, o);
            const T bb = __shfl_sync(kFull, s, 0), ss = __shfl_sync(kFull, s, 16);
            T bnew, ib, ig;
            if constexpr (sizeof(T) == 8) {
                // FP64 operations are slow one after the other: both reciprocal square roots in one call
                const T r = rsqrt((lane & 1) ? gbar2 + bb : bb);
                ib = __shfl_sync(kFull, r, 0);
                ig = __shfl_sync(kFull, r, 1);
                bnew = bb > T(0) ? bb * ib : T(0);
                ib = bb > T(0) ? ib : T(0);
                if (!(gbar2 + bb > T(0))) ig = T(1e30);
            } else {
                bnew = bb > T(0) ? sqrt(bb) : T(0);
                ib = bnew > T(0) ? T(1) / bnew : T(0);
                const T gamma = sqrt(gbar2 + bnew * bnew);
                ig = T(1) / (gamma > T(0) ? gamma : T(1e-30));
            }
            const T inv_old = sh.inv_beta;
            int done;
            if (init) {
                beta1 = bnew;
                phibar = bnew;
                done = !(bnew > T(0));
            } else {
                const T oldeps = epsln;
                epsln = sn * bnew;
                dbar = -cs * bnew;
                cs = gbar * ig;
                sn = bnew * ig;
                const T ph = cs * phibar;
                phibar = sn * phibar;
                ++itn;
                done = (phibar <= a.tau * beta1) || (itn >= a.max_it) || !(bnew > T(0));
                if (lane == 0) {
                    sh.wz = inv_old * ig;       // w_k = wz z_k - w2c w_{k-2} - w1c w_{k-1}
                    sh.w2c = oldeps * ig;
                    sh.w1c = d2 * ig;
                    sh.phi = ph;
                    sh.cprev = bnew * inv_old;
                    sh.itn = itn;
                    sh.pending = 1;
                }
            }
            __syncwarp();
            if (lane == 0) {
                sh.inv_beta = ib;
                if (c > 0) sh.inv_beta_d = sizeof(T) == 8 ? (double)ib : (bnew > T(0) ? 1.0 / (double)bnew : 0.0);
                sh.s_term = a.sig_n * ss;
                sh.done = done;
            }
        }
        __syncthreads();
    };
    scalars(true);

    unsigned long long t_gather = 0, t_rows = 0, t_p2 = 0, t0 = 0, t1 = 0;
    const bool timer = prof && rank == 0 && tid == 0;
    // ---------------------------------------------------------------- iterations
    while (!sh.done) {
        const bool has_prev = sh.pending != 0;
        const T inv_beta = sh.inv_beta, cprev = has_prev ? sh.cprev : T(0), s_term = sh.s_term;
        const T wz = sh.wz, w2c = sh.w2c, w1c = sh.w1c, phi = sh.phi;
        if (timer) t0 = globaltimer_ns();
        T acc = T(0);
        for (int j = warp; j < nsl; j += W) {
            const int s = j * P + rank;
            const int64_t row = (int64_t)s * 32 + lane;
            const int l = j * 32 + lane;
            const bool ok = row < n && row != trim;
            const int64_t o0 = __ldg(S.sell_off + s);
            const int wa = (int)((__ldg(S.sell_off + s + 1) - o0) >> 5);
            T g0 = T(0);
            for (int q = 0; q < wa; q += 8) {
                int32_t ia[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) ia[u] = q + u < wa ? __ldg(S.sell_ci + o0 + (int64_t)(q + u) * 32 + lane) : -1;
                T va[8];
                if (staged) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) va[u] = ia[u] >= 0 ? zs[ia[u]] : T(0);
                } else {
#pragma unroll
                    for (int u = 0; u < 8; ++u) va[u] = ia[u] >= 0 ? __ldcg(zg + ia[u]) : T(0);
                }
                T t;
                if (sw) {
                    if constexpr (sizeof(T) == 4) {
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            va[u] *= ia[u] >= 0 ? __ldg(sw + o0 + (int64_t)(q + u) * 32 + lane) : T(0);
                        t = cl_pass_sum(va, wa - q);
                    } else {
                        T wt[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            wt[u] = ia[u] >= 0 ? __ldg(sw + o0 + (int64_t)(q + u) * 32 + lane) : T(0);
                        t = pass_dot(va, wt, wa - q);
                    }
                } else {
                    t = cl_pass_sum(va, wa - q);
                }
                g0 = q == 0 ? t : g0 + t;
            }
            const T z = zc[l];
            T y = Ad[l] * z - g0;
            if (a.sig_n != T(0)) y += s_term;
            y *= inv_beta;
            if (has_prev) y -= cprev * Qp[l];
            y = ok ? y : T(0);
            Y[l] = y;
            acc += z * y;
        }
        acc *= inv_beta;
        if (timer) { t1 = globaltimer_ns(); t_gather += t1 - t0; }
        acc = warp_sum(acc);
        if (lane == 0) sh.red[0][warp] = acc;
        __syncthreads();
        if (warp == W - 1) {
            const T s = sum_red();
            if (lane < P) cl_store(cl_addr(&sh.in1[0][rank], lane), s);
        }
        send_columns();
        cl_arrive();
        double ib = 0.0, dib = 0.0, gprev = 0.0;
        if (warp == 0 && c > 0) {
            ib = sh.inv_beta_d;
            dib = delta * ib;
            gprev = has_prev ? delta * (double)cprev * g_cur : 0.0;
        }
        if (has_prev) {                       // the deferred w / x update, while the barrier completes
            for (int j = warp; j < nsl; j += W) {
                const int l = j * 32 + lane;  // the trimmed and the padding rows have z = 0: w and x stay 0
                const T w = wz * zp[l] - w2c * w2[l] - w1c * w1[l];
                w2[l] = w;
                x[l] += phi * w;
            }
            T* t = w1;                        // w_j took the place of w_{j-2}
            w1 = w2;
            w2 = t;
        }
        cl_wait();
        if (warp == 0) {
            // u1 = delta (g_k / beta_k - (beta_k / beta_{k-1}) g_{k-1}), alpha_k = alpha' + (g_k / beta_k)^T u1,
            // tv = C^{-1} (a - coef g) + C^{-1} G (u1 - coef delta g), coef = alpha_k / beta_k
            double al = (double)cl_total(sh.in1[0]);
            if (c > 0) {
                const double av = lane < c ? (double)cl_total(sh.in1[1 + lane]) : 0.0;
                const double gn = lane < c ? (double)cl_total(sh.in1[1 + c + lane]) : 0.0;
                const double u1 = dib * gn - gprev;
                g_cur = gn;
                double gu = (gn * ib) * u1;
                for (int o = c > 16 ? 16 : c > 8 ? 8 : c > 4 ? 4 : 2; o > 0; o >>= 1) gu += __shfl_xor_sync(kFull, gu, o);
                al += gu;
                const double cf = al * ib;
                if (lane < c) {
                    sh.gc[lane] = av - cf * gn;
                    sh.uc[lane] = u1 - cf * delta * gn;
                }
                __syncwarp();
                if (lane < c) {
                    double tv = 0.0, tu = 0.0;
                    for (int q = 0; q < c; ++q) {
                        tv += sh.Ci[lane + q * c] * sh.gc[q];
                        tu += sh.CG[lane + q * c] * sh.uc[q];
                    }
                    sh.tv[lane] = (T)(tv + tu);
                    sh.as[lane] = (T)u1 - (T)(cf * delta * gn);
                }
            }
            alpha = (T)al;
            if (lane == 0) sh.coef = alpha * sh.inv_beta;
        }
        __syncthreads();
        if (timer) { t0 = globaltimer_ns(); t_rows += t0 - t1; }
        phase2();
        scalars(false);
        if (timer) t_p2 += globaltimer_ns() - t0;
    }

    // ---------------------------------------------------------------- last deferred update, result
    {
        const bool pend = sh.pending != 0;
        const T wz = sh.wz, w2c = sh.w2c, w1c = sh.w1c, phi = sh.phi;
        for (int j = warp; j < nsl; j += W) {
            const int64_t row = ((int64_t)j * P + rank) * 32 + lane;
            const int l = j * 32 + lane;
            if (row >= n) continue;
            T xv = x[l];
            if (pend) xv += phi * (wz * zp[l] - w2c * w2[l] - w1c * w1[l]);
            Z[row] = row == trim ? 0.0 : (double)xv;
        }
        if (rank == 0 && tid == 0) {
            a.hs->inner_done = 1;
            a.hs->inner_iters = itn;
            a.hs->inner_relres = beta1 > T(0) ? (double)(phibar / beta1) : 0.0;
            if (prof) {
                a.hs->prof_ns[0] = t_gather;
                a.hs->prof_ns[1] = t_rows;
                a.hs->prof_ns[2] = t_p2;
            }
        }
    }
}

template <typename T>
static cudaLaunchConfig_t cl_config(const ClusterPlan& p, cudaLaunchAttribute* at, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(p.ctas);
    cfg.blockDim = dim3(p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = p.ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

// Cache lines that the warp-wide gathers of the sliced copy touch, summed over its 32-entry columns
// (line = idx >> shift): the cost of gathering z_k from L2, one line per cycle and SM.
__global__ void __launch_bounds__(kThreads) k_sell_lines(const int32_t* __restrict__ ci, int64_t total, int shift,
                                                         unsigned long long* out) {
    const int lane = threadIdx.x & 31;
    unsigned long long cnt = 0;
    for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31ll; g < total;
         g += (int64_t)gridDim.x * blockDim.x) {           // total is a multiple of 32
        const int32_t idx = ci[g + lane];
        const unsigned same = __match_any_sync(kFull, idx < 0 ? -1 : idx >> shift);
        cnt += __popc(__ballot_sync(kFull, idx >= 0 && lane == __ffs(same) - 1));
    }
    if (lane == 0 && cnt) atomicAdd(out, cnt);
}

// Microseconds that an FP64 iteration takes in one launch and in three, fitted to the measurements below: 16 SMs
// issue in one launch what 152 issue in three, so rows, columns (rounds of eight, one warp each) and entries
// cost more there, and the launches cost a constant.
static bool fp64_one_launch_pays(int64_t n, int64_t entries, bool weighted, int c) {
    const double kn = 1e-3 * (double)n, ke = 1e-3 * (double)entries;
    const double rounds = c <= 8 ? c / 8.0 : (double)((c + 7) / 8);
    const double one = 4.0 + (c > 0 ? 3.0 : 0.0) + 0.17 * c + 0.15 * rounds + kn * (0.36 + 0.055 * c + 0.21 * rounds) +
                       ke * (weighted ? 0.041 : 0.032);
    const double three = 26.5 + 0.007 * ke + (c > 0 ? 9.2 + 0.55 * std::min(c, 8) + 1.28 * std::max(c - 8, 0) : 0.0);
    return one <= three;
}

// Which solves take this path, and how.  The choice depends on the graph, the precision and the deflation rank
// alone, so a graph gives the same bits alone and in a batch.  Times are us per iteration on GB300, one launch
// against three.
//  * All rows sliced (no row above 64 neighbours): a long row would need its own split over the warps.
//  * FP32 up to 80,000 rows, where the ten vectors fill the shared memory of 16 CTAs.  2-D grids of 19,881 /
//    40,000 / 77,841 vertices at rank 0: 5.0 / 6.3 / 8.7 against 18.5 / 19.4 / 20.5; rank 31: 19 / 28 / 44 against
//    48 / 51 / 53.  A random graph is bound by the lines its gathers touch, one per cycle and SM (ER of 39,984:
//    14.8 against 21.7, of 55,986: 19.2 against 22.1), so beyond kClusterLines lines a CTA the whole GPU is the
//    better place.
//  * FP32 with more than 196 KB of shared memory a CTA (above 71,168 rows): the L1 that is left no longer holds
//    what the gathers of a line-heavy graph reuse (Watts-Strogatz of 68,000 / 72,000 / 79,900 at rank 0: 14.3 /
//    20.6 / 22.1 against 22.5; rank 8: 24.3 / 30.9 / 33.0 against 31.7; rank 24: 38.7 / 45.8 / 49.1 against 45.1).
//    Above kClusterLinesTight lines it is taken up to rank 8 only; a grid of 77,841 (1,263 lines) at all.
//  * FP64 up to 30,720 rows, at the ranks where fp64_one_launch_pays: rank 0 / 8 / 16 / 31, grid of 7,921: 8.2 /
//    17.0 / 23.9 / 36.8 against 26.6 / 39.0 / 49.2 / 67.6; of 19,881: 13.8 / 30.6 / 45.2 / 71.9 against 26.7 / 40.9 /
//    49.8 / 69.7; of 29,929: 19.0 / 43.0 / 64.2 / 103.8 against 26.7 / 41.0 / 50.2 / 70.6.  Entries count too: of
//    20,000 rows, 800,000 entries at rank 0: 33.0 against 31.1.  The fit's choice is at most 4 % from the
//    better path over the 29 graphs that were measured (4,000 to 30,000 rows, 4 to 40 entries a row, with
//    and without weights, ranks 0 to 31).
//  * CTAs: enough for 256 rows each in FP32 (latency) and 64 in FP64 (its narrow pipe), 16 at most.
//  * Staging copies z_k whole into every CTA's shared memory each iteration and gathers from there: it pays
//    in FP32 when the gathers touch more lines than the copy moves (ER of 12,339: 4.7 us against 6.6 us; grid of
//    9,856: 3.5 us staged, 3.3 us not); in FP64 the gather hides behind the FP64 pipe (ER of 12,339: 15.5 staged, 14.1 not).
constexpr int64_t kClusterLinesTight = 8000;
constexpr int kL1Step = 196 * 1024;         // shared memory beyond which the L1 falls to its smallest size

template <typename T>
void cluster_plan(const RowSched& rs, int64_t sell_total, unsigned long long* scratch, cudaStream_t s, ClusterPlan* out) {
    *out = ClusterPlan{};
    constexpr bool f32 = sizeof(T) == 4;
    if (!slices_only(rs) || rs.light0 != 0 || rs.n > (f32 ? kClusterRows32 : kClusterRows64)) return;
    int ctas = 1;
    while (ctas < kClMaxCtas && (int64_t)ctas * (f32 ? kClusterRowsPerCta32 : kClusterRowsPerCta64) < rs.n) ctas *= 2;
    const int nsl = (rs.n_slices + ctas - 1) / ctas;
    ClusterPlan p;
    p.ctas = ctas;
    p.cap = nsl * 32;
    p.threads = std::min(ClThreads<T>::value, std::max(128, nsl * 32));
    p.smem = (int)sizeof(T) * kClVecs * p.cap;
    p.staged = 0;
    p.ranks = ~0u;
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return;
    const int room = optin - (int)sizeof(ClShared<T>) - 1024;
    if (p.smem > room) return;
    if (f32) {
        unsigned long long lines = 0;
        if (cudaMemsetAsync(scratch, 0, sizeof(lines), s) != cudaSuccess) return;
        k_sell_lines<<<152, kThreads, 0, s>>>(rs.sell_ci, sell_total, 5, scratch);
        if (cudaMemcpyAsync(&lines, scratch, sizeof(lines), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return;
        const int64_t per_cta = (int64_t)lines / p.ctas, zbytes = (int64_t)sizeof(T) * ((rs.n + 31) / 32 * 32);
        if (per_cta > kClusterLines) return;
        if (p.smem + zbytes <= room && per_cta > zbytes / 32 + sell_total / (8 * p.ctas)) {
            p.staged = 1;
            p.smem += (int)zbytes;
        }
        if (!p.staged && p.smem + (int)sizeof(ClShared<T>) + 1024 > kL1Step && per_cta > kClusterLinesTight)
            p.ranks = (1u << 9) - 1;
    } else {
        p.ranks = 0;
        for (int c = 0; c < kCMax; ++c)
            if (fp64_one_launch_pays(rs.n, sell_total, rs.swd != nullptr, c)) p.ranks |= 1u << c;
    }
    if (cudaFuncSetAttribute(k_minres_cluster<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, room) != cudaSuccess ||
        cudaFuncSetAttribute(k_minres_cluster<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        (void)cudaGetLastError();
        return;
    }
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = cl_config<T>(p, at, nullptr);
    int num = 0;
    if (cudaOccupancyMaxActiveClusters(&num, k_minres_cluster<T>, &cfg) != cudaSuccess || num < 1) {
        (void)cudaGetLastError();
        return;
    }
    *out = p;
}

template <typename T>
cudaError_t cluster_minres(const InnerArgs<T>& a, const ClusterPlan& p, const double* R, const double* rnorm_dev,
                           double* Z, bool prof, cudaStream_t s) {
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = cl_config<T>(p, at, s);
    return cudaLaunchKernelEx(&cfg, k_minres_cluster<T>, a, R, rnorm_dev, Z, p.cap, p.staged, prof ? 1 : 0);
}

#define ISIRA_INSTANTIATE_CLUSTER(T)                                                                          \
    template void cluster_plan<T>(const RowSched&, int64_t, unsigned long long*, cudaStream_t, ClusterPlan*);                                             \
    template cudaError_t cluster_minres<T>(const InnerArgs<T>&, const ClusterPlan&, const double*, const double*, \
                                           double*, bool, cudaStream_t);
ISIRA_INSTANTIATE_CLUSTER(float)
ISIRA_INSTANTIATE_CLUSTER(double)

}  // namespace isira
