// Least-squares DM fitting over fitting directions (Sec. 4.1: with more reconstructed
// layers than DMs the fitting step becomes a least-squares problem of its own).
//
// The commands a minimise sum_k w_k ||Pi (A_k a - L_k phi)||^2 + eps ||a||^2: along
// fitting direction k the pupil nodes see the layers phi (L_k, linear stencils on the
// layer grids) and the DMs (A_k, bilinear actuator hats), and Pi removes the mean over
// the pupil nodes.  The normal equations N a = sum_k w_k A_k^T Pi L_k phi,
// N = sum_k w_k A_k^T Pi A_k + eps I, are solved by CG.  One CG step is two kernels:
//   k_lsf_sample<DM>  a grid of (slices, directions): beta from the r.r shares, p = r + beta
//                     p_old on the fly at the actuators under each node, u_k = A_k p (zero off
//                     the pupil), and the slice's sums of u_k, of w_k u_k^2 and, over a chunk
//                     of the actuators (whose p it stores), of eps p^2;
//   k_lsf_adj         an actuator per lane, a direction per warp: the means of the u_k, and
//                     p.q = eps p.p + sum_k w_k (sum u_k^2 - (sum u_k)^2 / n) from the shares
//                     in a fixed order, q = sum_k w_k A_k^T Pi u_k + eps p gathered over the
//                     pupil rows and columns whose stencils touch the actuator (host-built
//                     ranges, no atomics), a += alpha p, r -= alpha q, the shares of r.r.
// p.q is known before q, so no kernel waits for a total over its own grid.  The right-hand
// side is k_lsf_sample<LAYER> on phi followed by k_lsf_adj<RHS>.  Once the CG has stopped
// (state[0] != 0) the kernels of the remaining steps of a chunk return at once.
//
// Bound: latency of the dependent loads of two small kernels (450 KB a step at nine directions
// of 75 x 75 nodes and 9094 actuators).  Three kernels, one of them a single CTA over all
// actuators and one an actuator per thread over all directions, took 65 us a step; a fit of 128 steps went
// from 8.24 to 1.71 ms, phi included.
//
// Single precision: a CTA's sums are double-float (DotAcc), its shares' totals and the scalars
// double.  Plain double sums give the same commands bit for bit (the 37 m fit of ten seeds, twenty
// drawn systems) at 2.11 ms: the FP64 pipe takes 16 cycles for a warp's addition.  Against the 64-bit
// solution these forms and the three kernels before them, which took p.q from q, are equally far:
// 3.79e-6 and 3.74e-6 for the 37 m fit, 0.98 times over the drawn ones (geometric means).
#pragma once

#include "fewha_internal.h"
#ifdef __CUDACC__
#include "fewha_tile.cuh"
#endif

namespace fewha {

constexpr int LSF_SBLK = 256;    // k_lsf_sample: threads per slice of a direction's pupil grid
constexpr int LSF_MAXSL = 304;   // most (direction, slice) CTAs of k_lsf_sample (2 per SM)
constexpr int LSF_ABLK = 32;     // k_lsf_adj: actuators per CTA
constexpr int LSF_AW = 9;        // k_lsf_adj: most warps with directions (one more has the totals)
constexpr int LSF_KW = 6;        // rows and columns of an actuator's range held in registers
constexpr int LSF_SM = 3;        // sources of a node with their loads in flight together
constexpr int LSF_CHUNK = 32;    // CG steps between two looks at the state
constexpr int LSF_MAXK = FEWHA_MAX_FIT_DIRS;

template <class T>
struct LsDesc {
    int n_dirs, nf1, n_pup, n_layers, n_dms, n_a;
    int n_slices;                        // k_lsf_sample CTAs per direction
    int lay_n[MAXL], lay_off[MAXL];
    int dm_n[MAXM], dm_off[MAXM];
    T w[LSF_MAXK];
    T eps;
    const unsigned char* mask;           // nf1 * nf1 pupil nodes
    const int *ly0, *lx0, *my0, *mx0;    // see LsfitHost
    const T *lfy, *lfx, *mfy, *mfx;
    const int *ylo, *yhi, *xlo, *xhi;
};

// Value at pupil node (i, j) along direction k of the layers (LAYER) or the DMs: the sum
// over the sources of the separable two-point stencils.  Taps outside a DM lattice are
// zero; layer stencils never leave their grid (checked at set-up).
template <class T, bool LAYER>
__host__ __device__ inline T lsf_sample(const LsDesc<T>& d, const T* src, int k, int i, int j) {
    T val = T(0);
    const int ns = LAYER ? d.n_layers : d.n_dms;
    for (int s = 0; s < ns; ++s) {
        const int n = LAYER ? d.lay_n[s] : d.dm_n[s];
        const T* g = src + (LAYER ? d.lay_off[s] : d.dm_off[s]);
        const int e = (k * (LAYER ? MAXL : MAXM) + s) * d.nf1;
        const int y0 = (LAYER ? d.ly0 : d.my0)[e + i];
        const int x0 = (LAYER ? d.lx0 : d.mx0)[e + j];
        const T fy = (LAYER ? d.lfy : d.mfy)[e + i];
        const T fx = (LAYER ? d.lfx : d.mfx)[e + j];
        const T wy[2] = {T(1) - fy, fy};
        const T wx[2] = {T(1) - fx, fx};
        for (int t = 0; t < 2; ++t) {
            const int r = y0 + t;
            if (r < 0 || r >= n) continue;
            T row = T(0);
            for (int u = 0; u < 2; ++u) {
                const int c = x0 + u;
                if (c < 0 || c >= n) continue;
                row += wx[u] * g[r * n + c];
            }
            val += wy[t] * row;
        }
    }
    return val;
}

// (A_k^T Pi u_k) at actuator (p, q) of DM m, u_k zero off the pupil and mk its mean over the
// pupil nodes: the pupil rows [ylo, yhi) and columns [xlo, xhi) are those whose stencils
// include the actuator; its hat weight in each is the stencil weight on that actuator.
template <class T>
__host__ __device__ inline T lsf_adjoint_dir(const LsDesc<T>& d, const T* vk, T mk, int k, int m, int p, int q) {
    const int nf1 = d.nf1, e = k * MAXM + m;
    const int ylo = d.ylo[e * MAXNACT + p], yhi = d.yhi[e * MAXNACT + p];
    const int xlo = d.xlo[e * MAXNACT + q], xhi = d.xhi[e * MAXNACT + q];
    T sk = T(0);
    for (int i = ylo; i < yhi; ++i) {
        const int y0 = d.my0[e * nf1 + i];
        const T fy = d.mfy[e * nf1 + i];
        const T wy = y0 == p ? T(1) - fy : fy;   // y0 is p or p - 1 inside the range
        T row = T(0);
        for (int j = xlo; j < xhi; ++j) {
            const int x0 = d.mx0[e * nf1 + j];
            const T fx = d.mfx[e * nf1 + j];
            const int g = i * nf1 + j;
            row += (x0 == q ? T(1) - fx : fx) * (vk[g] - mk * static_cast<T>(d.mask[g]));
        }
        sk += wy * row;
    }
    return sk;
}

// The weighted sum of it over the directions, mean[k] the mean of u_k.
template <class T>
__host__ __device__ inline T lsf_adjoint(const LsDesc<T>& d, const T* v, const T* mean, int m, int p, int q) {
    T acc = T(0);
    for (int k = 0; k < d.n_dirs; ++k)
        acc += d.w[k] * lsf_adjoint_dir<T>(d, v + static_cast<size_t>(k) * d.nf1 * d.nf1, mean[k], k, m, p, q);
    return acc;
}

#ifdef __CUDACC__

template <class T>
struct LsCg {
    int n, nparts, max_iters;
    double tol2;          // stop once r.r <= tol2 * (r.r at the start)
    T *a, *r, *p[2];      // the direction buffers, in turn
    T *v;                 // u_k
    double *us;           // shares of the sums of u_k: [direction][slice]
    double *s2;           // of sum_k w_k u_k^2 + eps p^2, as us
    double *rs;           // of r.r, per CTA of k_lsf_adj
    double *sc;           // r.r of even and odd steps, [2] at the start, [3] the latest
    int* state;           // [0] 0 running, 1 stopped, 2 p.q <= 0 or not a number; [1] steps run
};

// The step's r.r from its shares, by one warp, and whether the CG has stopped; the CTA with
// `own` keeps both.  Every CTA comes to the same result.  Lane 0 returns beta, or a negative
// value if it has stopped.
template <class T>
__device__ __forceinline__ double lsf_beta(const LsCg<T>& g, int step, bool own) {
    using A = typename AccOf<T>::type;
    const int lane = threadIdx.x & 31;
    const double old = step > 0 ? __ldcg(g.sc + ((step - 1) & 1)) : 0.0;
    const double start = step > 0 ? __ldcg(g.sc + 2) : 0.0;
    const int st = __ldcg(g.state);
    const A x = shares_total<T, 10>(g.rs, g.nparts);
    if (lane != 0) return 0.0;
    const double rn = warp_value(x);
    const bool stop = st != 0 || step >= g.max_iters || (step > 0 ? !(rn > g.tol2 * start) : rn == 0.0);
    if (own && st == 0) {
        if (step == 0) g.sc[2] = rn;
        g.sc[step & 1] = rn;
        g.sc[3] = rn;
        if (stop) {
            g.state[0] = 1;
            g.state[1] = step;
        }
    }
    return stop ? -1.0 : step > 0 ? rn / old : 0.0;
}

// u_k = A_k p (DMs) or L_k src (LAYER) on slice blockIdx.x of the nf1 x nf1 pupil grid of
// direction k = blockIdx.y, zero off the pupil, and the sums above.
template <class T, bool LAYER>
__global__ void __launch_bounds__(LSF_SBLK) k_lsf_sample(__grid_constant__ const LsDesc<T> d,
                                                         __grid_constant__ const LsCg<T> g, const T* src, int step) {
    using A = typename AccOf<T>::type;
    constexpr int NW = LSF_SBLK / 32;
    __shared__ A red[3][NW];
    __shared__ double s_beta;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31, k = blockIdx.y;
    const int nf1 = d.nf1, npix = nf1 * nf1;
    const int chunk = (npix + d.n_slices - 1) / d.n_slices;
    const int n0 = blockIdx.x * chunk, n1 = min(npix, n0 + chunk);
    const int ns = LAYER ? d.n_layers : d.n_dms;
    const bool first = step == 0;
    const T* po = LAYER ? nullptr : g.p[(step + 1) & 1];
    T* pn = LAYER ? nullptr : g.p[step & 1];
    DotAcc<T> su, s2, pp;
    T beta = T(0);
    bool waited = false;
    for (int base = n0; base < n1 || !waited; base += LSF_SBLK) {
        const int node = base + t;
        const bool on = node < n1 && d.mask[node];
        const int i = node / nf1, j = node - i * nf1;
        T val = T(0);
        for (int s0 = 0; s0 < ns; s0 += LSF_SM) {
            int at[LSF_SM][4];
            T w[LSF_SM][4], x[LSF_SM][4], y[LSF_SM][4];
#pragma unroll
            for (int m = 0; m < LSF_SM; ++m) {
                const int s = s0 + m;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    w[m][c] = x[m][c] = y[m][c] = T(0);
                    at[m][c] = -1;
                }
                if (!on || s >= ns) continue;
                const int n = LAYER ? d.lay_n[s] : d.dm_n[s], off = LAYER ? d.lay_off[s] : d.dm_off[s];
                const int e = (k * (LAYER ? MAXL : MAXM) + s) * nf1;
                const int y0 = (LAYER ? d.ly0 : d.my0)[e + i], x0 = (LAYER ? d.lx0 : d.mx0)[e + j];
                const T fy = (LAYER ? d.lfy : d.mfy)[e + i], fx = (LAYER ? d.lfx : d.mfx)[e + j];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int yr = y0 + (c >> 1), xc = x0 + (c & 1);
                    if (yr >= 0 && yr < n && xc >= 0 && xc < n) at[m][c] = off + yr * n + xc;
                    w[m][c] = (c & 1 ? fx : T(1) - fx);
                }
                w[m][2] = fy;                                   // (the rows' weights)
                w[m][3] = T(1) - fy;
                if (!LAYER && !first)
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (at[m][c] >= 0) y[m][c] = po[at[m][c]];      // written two kernels back
            }
            if (!waited) {
                pdl_wait();
                pdl_trigger();
            }
#pragma unroll
            for (int m = 0; m < LSF_SM; ++m)
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (at[m][c] >= 0) x[m][c] = LAYER ? src[at[m][c]] : g.r[at[m][c]];
            if (!waited) {
                waited = true;
                if (!LAYER) {
                    if (warp == NW - 1) {
                        const double b = lsf_beta<T>(g, step, blockIdx.x == 0 && blockIdx.y == 0);
                        if (lane == 0) s_beta = b;
                    }
                    __syncthreads();
                    if (s_beta < 0.0) return;
                    beta = static_cast<T>(s_beta);
                }
            }
#pragma unroll
            for (int m = 0; m < LSF_SM; ++m) {
                if (!LAYER && !first)
#pragma unroll
                    for (int c = 0; c < 4; ++c) x[m][c] += beta * y[m][c];
                const T r0 = w[m][0] * x[m][0] + w[m][1] * x[m][1], r1 = w[m][0] * x[m][2] + w[m][1] * x[m][3];
                val += w[m][3] * r0 + w[m][2] * r1;
            }
        }
        if (node < n1) g.v[static_cast<size_t>(k) * npix + node] = val;
        su.add(val, T(1));
        s2.add(val, val);
    }
    if (!LAYER) {
        // this CTA's chunk of the direction itself
        const int cta = blockIdx.y * gridDim.x + blockIdx.x, all = gridDim.x * gridDim.y * LSF_SBLK;
        for (int a = cta * LSF_SBLK + t; a < g.n; a += all) {
            T p = g.r[a];
            if (!first) p += beta * po[a];
            pn[a] = p;
            pp.add(p, p);
        }
    }
    const A x0 = acc_warp(AccOf<T>::of(su)), x1 = acc_warp(AccOf<T>::of(s2)), x2 = acc_warp(AccOf<T>::of(pp));
    if (lane == 0) {
        red[0][warp] = x0;
        red[1][warp] = x1;
        red[2][warp] = x2;
    }
    __syncthreads();
    const int slot = k * d.n_slices + blockIdx.x;
    if (warp == 0) {
        const A x = acc_warp(lane < NW ? red[0][lane] : AccOf<T>::zero());
        if (lane == 0) g.us[slot] = warp_value(x);
    } else if (warp == 1 && !LAYER) {
        double x = 0.0;
        if (lane < 2 * NW) x = lane < NW ? double(d.w[k]) * warp_value(red[1][lane]) : double(d.eps) * warp_value(red[2][lane - NW]);
        x = warp_sum(x);
        if (lane == 0) g.s2[slot] = x;
    }
}

// An actuator's range in one direction: the weights of its rows and columns and the pupil mask,
// or `small` false if it exceeds LSF_KW either way.
template <class T>
struct LsRange {
    T wy[LSF_KW], wx[LSF_KW];
    unsigned long long in;
    int at;
    bool small;
};

template <class T>
__device__ __forceinline__ void lsf_range(const LsDesc<T>& d, int k, int m, int p, int q, LsRange<T>& R) {
    const int e = k * MAXM + m, nf1 = d.nf1;
    const int ylo = d.ylo[e * MAXNACT + p], yhi = d.yhi[e * MAXNACT + p];
    const int xlo = d.xlo[e * MAXNACT + q], xhi = d.xhi[e * MAXNACT + q];
    R.small = yhi - ylo <= LSF_KW && xhi - xlo <= LSF_KW;
    R.at = ylo * nf1 + xlo;
    R.in = 0;
#pragma unroll
    for (int c = 0; c < LSF_KW; ++c) {
        R.wy[c] = R.wx[c] = T(0);
        if (R.small && ylo + c < yhi) {
            const T f = d.mfy[e * nf1 + ylo + c];
            R.wy[c] = d.my0[e * nf1 + ylo + c] == p ? T(1) - f : f;
        }
        if (R.small && xlo + c < xhi) {
            const T f = d.mfx[e * nf1 + xlo + c];
            R.wx[c] = d.mx0[e * nf1 + xlo + c] == q ? T(1) - f : f;
        }
    }
    if (R.small)
#pragma unroll
        for (int i = 0; i < LSF_KW; ++i)
#pragma unroll
            for (int j = 0; j < LSF_KW; ++j)
                if (ylo + i < yhi && xlo + j < xhi && d.mask[R.at + i * nf1 + j]) R.in |= 1ull << (i * LSF_KW + j);
}

// RHS: r = sum_k w_k A_k^T Pi u_k, a = 0, the CG's start.  Otherwise the second half of CG step
// `step`.
template <class T, bool RHS>
__global__ void __launch_bounds__((LSF_AW + 1) * 32, 2) k_lsf_adj(__grid_constant__ const LsDesc<T> d,
                                                                  __grid_constant__ const LsCg<T> g, int step) {
    using A = typename AccOf<T>::type;
    __shared__ T part[LSF_AW][LSF_ABLK];
    __shared__ double s_sum[LSF_MAXK], s_sq;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31, W = (blockDim.x >> 5) - 1;
    const int a = blockIdx.x * LSF_ABLK + lane;
    const bool on = a < d.n_a;
    int m = 0;
    while (m + 1 < d.n_dms && a >= d.dm_off[m + 1]) ++m;
    const int n = d.dm_n[m], p = (a - d.dm_off[m]) / n, q = a - d.dm_off[m] - p * n;
    const int nf1 = d.nf1, npix = nf1 * nf1;
    LsRange<T> R;
    R.small = true;
    if (on && warp < W) lsf_range<T>(d, warp, m, p, q, R);
    T ra = T(0), aa = T(0);                              // written two kernels back
    if (!RHS && on && warp == 0) {
        ra = g.r[a];
        aa = g.a[a];
    }
    pdl_wait();
    pdl_trigger();
    const int st = RHS ? 0 : __ldcg(g.state);
    const double rr = RHS ? 0.0 : __ldcg(g.sc + (step & 1));
    T pa = T(0);
    if (!RHS && on && warp == 0) pa = g.p[step & 1][a];
    if (warp < W) {
        T acc = T(0);
        for (int k = warp; k < d.n_dirs; k += W) {
            if (k != warp && on) lsf_range<T>(d, k, m, p, q, R);
            const T* vk = g.v + static_cast<size_t>(k) * npix;
            T x[LSF_KW][LSF_KW];
#pragma unroll
            for (int i = 0; i < LSF_KW; ++i)
#pragma unroll
                for (int j = 0; j < LSF_KW; ++j) {
                    x[i][j] = T(0);
                    if (on && R.small && (R.in >> (i * LSF_KW + j) & 1)) x[i][j] = vk[R.at + i * nf1 + j];
                }
            double sum = 0.0;
            for (int i = lane; i < d.n_slices; i += 32) sum += __ldcg(g.us + k * d.n_slices + i);
            sum = __shfl_sync(0xffffffffu, warp_sum(sum), 0);
            if (lane == 0) s_sum[k] = sum;
            const T mk = static_cast<T>(sum / d.n_pup);
            T sk = T(0);
            if (on && R.small) {
#pragma unroll
                for (int i = 0; i < LSF_KW; ++i) {
                    T row = T(0);
#pragma unroll
                    for (int j = 0; j < LSF_KW; ++j)
                        row += R.wx[j] * (x[i][j] - (R.in >> (i * LSF_KW + j) & 1 ? mk : T(0)));
                    sk += R.wy[i] * row;
                }
            } else if (on) {
                sk = lsf_adjoint_dir<T>(d, vk, mk, k, m, p, q);
            }
            acc += d.w[k] * sk;
        }
        part[warp][lane] = acc;
    } else if (!RHS) {
        double x = 0.0;
        const int cnt = d.n_dirs * d.n_slices;
        for (int k0 = 0; k0 < cnt; k0 += 320) {
            double v[10];
#pragma unroll
            for (int c = 0; c < 10; ++c) {
                const int i = k0 + 32 * c + lane;
                v[c] = i < cnt ? __ldcg(g.s2 + i) : 0.0;
            }
            x += (((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]))) + (v[8] + v[9]);
        }
        x = warp_sum(x);
        if (lane == 0) s_sq = x;
    }
    __syncthreads();
    if (warp != 0 || st != 0) return;
    T val = T(0);
    for (int w = 0; w < W; ++w) val += part[w][lane];
    DotAcc<T> dot;
    if (RHS) {
        if (on) {
            g.r[a] = val;
            g.a[a] = T(0);
            dot.add(val, val);
        }
        if (blockIdx.x == 0 && lane < 2) g.state[lane] = 0;
    } else {
        double x = 0.0;
        for (int k = lane; k < d.n_dirs; k += 32) x += double(d.w[k]) * s_sum[k] * (s_sum[k] / d.n_pup);
        const double pq = s_sq - __shfl_sync(0xffffffffu, warp_sum(x), 0);
        if (!(pq > 0.0)) {
            if (blockIdx.x == 0 && lane == 0) {
                g.state[0] = 2;
                g.state[1] = step;
            }
            return;
        }
        const T al = static_cast<T>(rr / pq);
        if (on) {
            val += d.eps * pa;
            ra -= al * val;
            g.r[a] = ra;
            g.a[a] = aa + al * pa;
            dot.add(ra, ra);
        }
    }
    const A x = acc_warp(AccOf<T>::of(dot));
    if (lane == 0) *reinterpret_cast<A*>(g.rs + blockIdx.x) = x;
}

// The state after `step` steps, for the host to read.
template <class T>
__global__ void __launch_bounds__(32) k_lsf_check(__grid_constant__ const LsCg<T> g, int step) {
    pdl_wait();
    pdl_trigger();
    lsf_beta<T>(g, step, true);
}

#endif  // __CUDACC__

}  // namespace fewha
