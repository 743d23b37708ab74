// Tile kernels of the wavelet transforms: one CTA per square tile of a layer, no exchange
// between CTAs.  The periodic db3 synthesis of a tile of ts x ts nodes needs, level by
// level, only a window of w_(j+1) = w_j / 2 + 2 coefficients a side of every sub-band, so a
// CTA forms its tile of phi = W^T c from all levels by itself.
//
// Bound: latency.  A layer moves 4 n^2 values through L2 and does ~100 operations a value;
// what a frame waits for is the chain launch -> loads -> levels -> store.  A cluster of 8
// CTAs per layer (bands exchanged through distributed shared memory, the coarse levels on
// one leader CTA, three cluster barriers) took 8.0 us a launch on the 9 layers of the MAORY
// geometry and filled 72 of the 152 SMs; the tiles redo the halos (2.2 times the arithmetic
// at ts = 32) but wait for nobody: 120 CTAs, 5.7 us with the sums over the sensors in it.
#pragma once

#include "fewha_cluster.cuh"

namespace fewha {

constexpr int TINV_NT = 512;     // threads of the inverse tile kernel
constexpr int TINV_SL = 4;       // coefficient slots per thread and round
// Entries of a functional on a tile that 8 lanes take; one of more has a weight per node, for
// all threads.  Boundary sums have at most some 150 entries a tile and take 1 us beside one
// another; the elongation's have up to 1024, and as lists they took 6 us a launch, as weights
// reduced together 1.2 (37 m frame 86.7 against 75.8 us).
constexpr int TINV_FEW = 160;
constexpr int TINV_DN = 16;      // functionals of more entries taken together

// ---------------------------------------------------------------------------
// Sums in a fixed order, in the arithmetic of DotAcc.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double acc_merge(double a, double b) { return a + b; }
__device__ __forceinline__ DFloat acc_merge(DFloat a, DFloat b) { return df_merge(a, b); }
__device__ __forceinline__ double acc_warp(double a) { return warp_sum(a); }
__device__ __forceinline__ DFloat acc_warp(DFloat a) { return warp_df_sum(a); }
__device__ __forceinline__ double acc_shfl_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ DFloat acc_shfl_xor(DFloat a, int o) {
    return DFloat{__shfl_xor_sync(0xffffffffu, a.s, o), __shfl_xor_sync(0xffffffffu, a.c, o)};
}
__device__ __forceinline__ double acc_from(double x) { return x; }
__device__ __forceinline__ DFloat acc_from(float x) { return DFloat{x, 0.f}; }
__device__ __forceinline__ double acc_neg(double a) { return -a; }
__device__ __forceinline__ DFloat acc_neg(DFloat a) { return DFloat{-a.s, -a.c}; }
template <class T> struct AccOf;
template <> struct AccOf<float> {
    using type = DFloat;
    static __device__ __forceinline__ DFloat zero() { return DFloat{0.f, 0.f}; }
    static __device__ __forceinline__ DFloat of(const DotAcc<float>& d) { return DFloat{d.s, d.c}; }
};
template <> struct AccOf<double> {
    using type = double;
    static __device__ __forceinline__ double zero() { return 0.0; }
    static __device__ __forceinline__ double of(const DotAcc<double>& d) { return d.v; }
};
static_assert(sizeof(DFloat) == sizeof(double), "a share is 8 bytes in both precisions");

__device__ __forceinline__ double warp_value(double x) { return x; }
__device__ __forceinline__ double warp_value(DFloat x) { return double(x.s) + double(x.c); }

// Total of `cnt` shares by one warp (lane 0): rounds of up to 32 U loads in flight, merged as
// a tree.
template <class T, int U = 4>
__device__ __forceinline__ typename AccOf<T>::type shares_total(const double* p, int cnt) {
    using A = typename AccOf<T>::type;
    A s = AccOf<T>::zero();
    for (int k0 = 0; k0 < cnt; k0 += 32 * U) {
        A v[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int i = k0 + 32 * k + (threadIdx.x & 31);
            v[k] = AccOf<T>::zero();
            if (i < cnt) {
                const double x = __ldcg(p + i);
                v[k] = *reinterpret_cast<const A*>(&x);
            }
        }
#pragma unroll
        for (int w = 1; w < U; w *= 2)
#pragma unroll
            for (int k = 0; k + w < U; k += 2 * w)
                if (k0 + 32 * (k + w) < cnt) v[k] = acc_merge(v[k], v[k + w]);
        s = k0 ? acc_merge(s, v[0]) : v[0];
    }
    return acc_warp(s);
}

// The CTA's share of an inner product (plus `extra`, if any) into its slot, fixed order;
// `sh` holds one share per warp.
template <class T>
__device__ __forceinline__ void cta_share(const DotAcc<T>& d, double* sh, const double* extra, double* slot) {
    using A = typename AccOf<T>::type;
    A* s = reinterpret_cast<A*>(sh);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const A v = acc_warp(AccOf<T>::of(d));
    if (lane == 0) s[warp] = v;
    __syncthreads();
    if (warp == 0) {
        A x = acc_warp(lane < nw ? s[lane] : AccOf<T>::zero());
        if (lane == 0) {
            if (extra) x = acc_merge(x, *reinterpret_cast<const A*>(extra));
            *reinterpret_cast<A*>(slot) = x;
        }
    }
}

template <class T> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };
__device__ __forceinline__ void cp_async_pair(float2* smem, const float2* gmem) { cp_async8(smem, gmem); }
__device__ __forceinline__ void cp_async_pair(double2* smem, const double2* gmem) { cp_async16(smem, gmem); }

// Quotient of t < 2048 by n <= 64 through the host's reciprocal ceil(65536 / n).
__device__ __forceinline__ int tdiv(int t, int magic) { return (t * magic) >> 16; }

// One output pair of a synthesis step (Sec. 3.1) from the coefficients k, k - 1, k - 2 of the
// scaling (a) and wavelet (d) half.
template <class T>
__device__ __forceinline__ void synth_pair(T a0, T a1, T a2, T d0, T d1, T d2, T& e, T& o) {
    e = fmadd(tap_g<T>(4), d2, fmadd(tap_g<T>(2), d1, fmadd(tap_g<T>(0), d0, fmadd(tap_h<T>(4), a2, dot2(tap_h<T>(0), a0, tap_h<T>(2), a1)))));
    o = fmadd(tap_g<T>(5), d2, fmadd(tap_g<T>(3), d1, fmadd(tap_g<T>(1), d0, fmadd(tap_h<T>(5), a2, dot2(tap_h<T>(1), a0, tap_h<T>(3), a1)))));
}

// Sums over one sensor's measured slopes, as its functionals sum the modelled ones: tip and
// tilt of a laser star and, with spot elongation (Eq. 3), gamma beta (beta . s).  Compensated: the
// residual's sums are the difference of these and the modelled ones.
template <class T, int NT>
__device__ __forceinline__ void measured_sums(const Desc<T>& d, const T* s, double* out, int g) {
    using A = typename AccOf<T>::type;
    __shared__ A ws[4][CWMAX + 2];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const WfsInfo& W = d.G[g];
    const int N = W.N, K = W.n_active, el = W.el;
    DotAcc<T> sum[4];
    pdl_wait();
    pdl_trigger();
    if (!W.lgs) return;
    for (int k = t; k < N * N; k += NT) {
        const int id = d.sidx[W.mask_off + k];
        if (id >= 0) {
            const T sx = s[W.soff + id], sy = s[W.soff + K + id];
            sum[0].add(sx, T(1));
            sum[1].add(sy, T(1));
            if (el) {
                T b1, b2, gam;
                elong(W, k / N, k % N, b1, b2, gam);
                const T bs = dot2(b1, sx, b2, sy);
                sum[2].add(gam * b1, bs);
                sum[3].add(gam * b2, bs);
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const A x = acc_warp(AccOf<T>::of(sum[e]));
        if (lane == 0) ws[e][warp] = x;
    }
    __syncthreads();
    if (warp < (el ? 4 : 2)) {
        const A x = acc_warp(lane < NT / 32 ? ws[warp][lane] : AccOf<T>::zero());
        if (lane == 0) *reinterpret_cast<A*>(out + d.f0[g] + warp) = x;
    }
}

template <class T>
__global__ void __launch_bounds__(TINV_NT) k_msum(__grid_constant__ const Desc<T> d, const T* s, double* out) {
    measured_sums<T, TINV_NT>(d, s, out, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Inverse tile kernel: phi = W^T c on tile `unit` (d.tunit), optionally advancing the CG
// direction first (Sec. 3.3): PUPD = 0, phi = W^T a.in.  PUPD = 1, p = z + beta p_old into
// a.pout (another buffer than a.pupd: neighbouring tiles read p_old in their halos), beta =
// rz_k / rz_(k-1), then phi = W^T p.  PUPD = 2, the augmented PCG of Sec. 3.4:
// p_new = z + beta p_old - sum_j mu_j P_j.  Every coefficient belongs to one tile, whose CTA
// writes it; the halos are advanced redundantly.
// ---------------------------------------------------------------------------
template <class T, int PUPD>
__device__ __forceinline__ void tinv_body(const Desc<T>& d, const ClArgs<T>& a, const int unit) {
    constexpr int NT = TINV_NT, SL = TINV_SL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sop = reinterpret_cast<T*>(smem_raw);             // the tail operator (TAIL_N), if any
    __shared__ TileLayer tl;
    __shared__ int ss[2][8];                              // window starts per dimension and level
    __shared__ T sbeta;
    __shared__ typename AccOf<T>::type fden_w[TINV_DN][NT / 32];
    __shared__ T smu[AUG_MAX];
    using A = typename AccOf<T>::type;
    const int t = threadIdx.x;
    if (unit >= d.n_tu) {
        measured_sums<T, NT>(d, a.ms, a.msum, unit - d.n_tu);
        return;
    }
    int l = 0;
    while (unit >= d.tu0[l + 1]) ++l;
    const LayerInfo L = d.L[l];
    const int n = L.n;
    // the tile's functionals (see Desc::fidx): offsets and, as far as they fit, the entries
    int* foff = reinterpret_cast<int*>(sop + (d.tailop ? TAIL_N : 0));
    using V2 = typename Vec2<T>::type;
    V2* fent = reinterpret_cast<V2*>(foff + d.fpad);
    const V2* gent = reinterpret_cast<const V2*>(d.fent);
    if (a.fsh) {
        for (int k = t; k < d.fpad; k += NT) cp_async(foff + k, d.foff + unit * d.fpad + k);
    }
    if (t < static_cast<int>(sizeof(TileLayer) / sizeof(int)))
        reinterpret_cast<int*>(&tl)[t] = reinterpret_cast<const int*>(d.tl + l)[t];
    T* sc = reinterpret_cast<T*>(fent + d.fcap);          // the levels' quadrants
    if (d.tailop) stage16(sop, d.tailop, TAIL_N, t, NT);
    __syncthreads();
    cp_async_wait();
    __syncthreads();
    if (a.fsh) {
        const int f0 = foff[2 * d.n_fun];
        const int cnt = min(foff[2 * d.n_fun + 1] + foff[2 * d.n_fun + 2] * ((tl.w[0] * tl.w[0]) >> 1), d.fcap);
        for (int k = t; k < cnt; k += NT) cp_async_pair(fent + k, gent + f0 + k);
    }
    if (t < 2) {
        const int side = tl.side, u = unit - d.tu0[l];
        int w0 = (t ? u & (side - 1) : u / side) << tl.lts;
        ss[t][0] = w0;
        for (int j = 1; j <= tl.J; ++j) {
            w0 = (w0 >> 1) - 2;
            if (tl.whole[j]) w0 = 0;
            ss[t][j] = w0;
        }
    }
    const bool has_old = PUPD == 1 || (PUPD == 2 && a.pupd != nullptr);
    bool waited = false;
    // the unit's slots: place in the coefficient vector (its sign bit: this tile owns it) and
    // in shared memory
    const int cnt = d.tcnt[l];
    double rz_old = 0.0;                                  // rz of the iteration before: long written
    if (PUPD && has_old && t == 0) rz_old = a.pcg.rztot[a.iter - 1];
    const int2* slots = reinterpret_cast<const int2*>(d.tslot + static_cast<size_t>(unit) * d.tslot_ld);
    for (int r0 = 0; r0 < cnt; r0 += NT * SL) {
        int dst[SL], pos[SL];
        T po[SL], zv[SL];
        bool own[SL];
#pragma unroll
        for (int s = 0; s < SL; ++s) {
            const int k = r0 + s * NT + t;
            int2 e = make_int2(-1, 0);
            if (k < cnt) e = __ldg(slots + k);
            own[s] = k < cnt && e.x < 0;
            pos[s] = k < cnt ? (e.x & 0x7fffffff) : -1;
            dst[s] = e.y;
        }
#pragma unroll
        for (int s = 0; s < SL; ++s)
            if (pos[s] >= 0) {
                // p_old was last written two kernels back or earlier
                if (PUPD && has_old) po[s] = a.pupd[pos[s]];
            }
        if (!waited) {
            pdl_wait();
            pdl_trigger();
        }
#pragma unroll
        for (int s = 0; s < SL; ++s)
            if (pos[s] >= 0) zv[s] = PUPD ? a.zupd[pos[s]] : a.in[pos[s]];
        if (!waited) {
            waited = true;
            // beta and the mu_j while the loads are in flight; a deferred r.z total first
            // (warp 0, fixed order: the same value in every CTA)
            if (t < 32 && (PUPD || a.rz_cnt > 0)) {
                double rz_new = 0.0;
                if (a.rz_cnt > 0) {
                    rz_new = warp_value(shares_total<T>(a.rz_parts, a.rz_cnt));
                    if (t == 0 && unit == 0) a.pcg.rztot[a.rz_slot] = rz_new;
                } else if (has_old && t == 0) {
                    rz_new = a.pcg.rztot[a.iter];
                }
                if (PUPD && t == 0) sbeta = T(has_old && rz_old != 0.0 ? rz_new / rz_old : 0.0);
            }
            if (PUPD == 2) {
                if (a.aug_pcnt > 0) {
                    const int warp1 = t >> 5, nw1 = NT >> 5;
                    for (int j = warp1 - 1; warp1 > 0 && j < a.aug_m; j += nw1 - 1) {
                        const double num = warp_total(a.aug_parts + static_cast<long long>(j) * a.aug_pcnt, a.aug_pcnt,
                                                      static_cast<const DotAcc<T>*>(nullptr));
                        if ((t & 31) == 0) {
                            const double den = a.aug_pq[j];
                            smu[j] = T(den > 0.0 ? num / den : 0.0);
                        }
                    }
                } else if (t >= 32 && t < 32 + a.aug_m) {
                    const int j = t - 32;
                    const double num = a.aug_tot[AUG_MAX + j], den = a.aug_pq[j];
                    smu[j] = T(den > 0.0 ? num / den : 0.0);
                }
            }
            if (PUPD) __syncthreads();
        }
        if (PUPD) {
            const T beta = sbeta;
            T cor[SL];
            if (PUPD == 2) {
#pragma unroll
                for (int s = 0; s < SL; ++s) cor[s] = T(0);
                for (int j = 0; j < a.aug_m; ++j) {
                    const T mu = smu[j];
                    const T* Pj = a.augP + static_cast<long long>(j) * a.aug_ld;
#pragma unroll
                    for (int s = 0; s < SL; ++s)
                        if (pos[s] >= 0) cor[s] = fmadd(mu, __ldg(Pj + pos[s]), cor[s]);
                }
            }
#pragma unroll
            for (int s = 0; s < SL; ++s)
                if (pos[s] >= 0) {
                    if (has_old) zv[s] = fmadd(beta, po[s], zv[s]);
                    if (PUPD == 2) zv[s] -= cor[s];
                    if (own[s]) a.pout[pos[s]] = zv[s];
                }
        }
#pragma unroll
        for (int s = 0; s < SL; ++s)
            if (pos[s] >= 0) {
                // Input of the data path of M (a.zero_piston): Gamma annihilates constants and
                // bilinear weights sum to one, so a full-depth layer's piston coefficient (its
                // constant function) contributes nothing to P, Gamma and back, and is left out.
                // Exact; without it a large piston component (the adjoint vectors of the
                // gradient passes carry one, J^-1 of that coefficient being ~1e5) rounds into
                // phi and leaks through the differences of Gamma.  p itself is stored unchanged.
                sc[dst[s]] = (a.zero_piston && L.full && pos[s] == L.off) ? T(0) : zv[s];
            }
    }
    cp_async_wait();
    __syncthreads();
    const T* tailb = sc + tl.tailb;
    T* vb = sc + tl.vbuf;                                 // a level's column pass
    // ---- the last three levels of a full decomposition, one 64 x 64 map: eight threads an
    // output, each 8 terms
    if (tl.tail) {
        const int o = t >> 3, part = t & 7;
        T acc[2] = {T(0), T(0)};
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i & 1] = fmadd(sop[o * TAIL_LD + part * 8 + i], tailb[part * 8 + i], acc[i & 1]);
        T y = acc[0] + acc[1];
        y += __shfl_down_sync(0xffffffffu, y, 4);
        y += __shfl_down_sync(0xffffffffu, y, 2);
        y += __shfl_down_sync(0xffffffffu, y, 1);
        if (part == 0) sc[tl.base[tl.J] + (o >> 3) * tl.stride[tl.J] + (o & 7)] = y;
        __syncthreads();
    }
    // ---- the levels, coarse to fine; level j's quadrants give level j - 1's window, columns
    // first, then rows
    for (int j = tl.J; j >= 1; --j) {
        const int np = tl.np[j - 1], w = tl.w[j], st = tl.stride[j], m = n >> j, w0 = tl.w[j - 1];
        const int w2 = 2 * w, vst = w2 + 1;
        const bool whole = tl.whole[j] != 0;
        const int s0y = ss[0][j - 1], s0x = ss[1][j - 1], ky0 = s0y >> 1, kx0 = s0x >> 1;
        for (int b = t, mg = tl.magicw[j]; b < np * w2; b += NT) {
            const int by = tdiv(b, mg), c = b - by * w2, xh = c >= w;
            const T* Al = sc + tl.base[j] + xh * w * st + c - xh * w;       // y-low, then y-high rows
            const T* Dl = Al + 2 * w * st;
            int iy[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) iy[q] = (whole ? ((ky0 + by - q) & (m - 1)) : by + 2 - q) * st;
            T e, o;
            synth_pair(Al[iy[0]], Al[iy[1]], Al[iy[2]], Dl[iy[0]], Dl[iy[1]], Dl[iy[2]], e, o);
            const int ry = 2 * (ky0 + by) - s0y;
            if (ry >= 0 && ry < w0) vb[ry * vst + c] = e;
            if (ry + 1 < w0) vb[(ry + 1) * vst + c] = o;
        }
        __syncthreads();
        for (int b = t, mg = tl.magic[j - 1]; b < np * w0; b += NT) {
            const int row = tdiv(b, mg), bx = b - row * np;
            const T* Al = vb + row * vst;
            int ix[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) ix[q] = whole ? ((kx0 + bx - q) & (m - 1)) : bx + 2 - q;
            T e, o;
            synth_pair(Al[ix[0]], Al[ix[1]], Al[ix[2]], Al[w + ix[0]], Al[w + ix[1]], Al[w + ix[2]], e, o);
            const int x = 2 * (kx0 + bx);
            if (j == 1) {
                T* dst = a.out + L.off + (s0y + row) * n + x;
                dst[0] = e;
                dst[1] = o;
                // the tile in shared memory too (this level's quadrants have been read)
                T* keep = sc + row * w0 + 2 * bx;
                keep[0] = e;
                keep[1] = o;
            } else {
                T* dst = sc + tl.base[j - 1] + row * tl.stride[j - 1];
                const int rx = x - s0x;
                if (rx >= 0 && rx < w0) dst[rx] = e;
                if (rx + 1 < w0) dst[rx + 1] = o;
            }
        }
        if (j > 1) __syncthreads();
    }
    if (!a.fsh) return;
    // ---- the tile's share of every functional: a warp each, fixed order
    __syncthreads();
    // (8 lanes each for the few boundary nodes of a sum; the dense ones of the elongation by
    // the whole CTA)
    const int f0 = foff[2 * d.n_fun], lg = t & 7;
    for (int f = t >> 3; f < ((d.n_fun + NT / 8 - 1) & ~(NT / 8 - 1)); f += NT / 8) {
        DotAcc<T> s;
        const int k0 = f < d.n_fun ? foff[2 * f] : 0, k1 = f < d.n_fun ? foff[2 * f + 1] : 0;
        for (int k = k0 + lg; k < k1; k += 32) {
            V2 e[4];
            T x = T(0);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (k + 8 * q < k1) e[q] = k + 8 * q < d.fcap ? fent[k + 8 * q] : gent[f0 + k + 8 * q];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (k + 8 * q < k1) x = fmadd(e[q].y, sc[static_cast<int>(e[q].x)], x);
            s.add(x, T(1));
        }
        A x = AccOf<T>::of(s);
#pragma unroll
        for (int o = 4; o; o >>= 1) x = acc_merge(x, acc_shfl_xor(x, o));
        if (f < d.n_fun && lg == 0 && k1 >= k0) *reinterpret_cast<A*>(a.fsh + f * d.n_tu + unit) = x;
    }
    // those of many entries (elongation): a weight per node, two nodes a thread for TINV_DN of
    // them at a time; their sums go through the warp together, halving the set at each step
    const int nd = foff[2 * d.n_fun + 2], w0 = tl.w[0], np2 = (w0 * w0) >> 1, lane = t & 31;
    const int* fden = foff + 2 * d.n_fun + 3;
    for (int i0 = 0; i0 < nd; i0 += TINV_DN) {
        T x[TINV_DN];
        V2 v{T(0), T(0)};
        if (t < np2) v = reinterpret_cast<const V2*>(sc)[t];
#pragma unroll
        for (int i = 0; i < TINV_DN; ++i) {
            x[i] = T(0);
            if (t < np2 && i0 + i < nd) {
                const int k = foff[2 * d.n_fun + 1] + (i0 + i) * np2 + t;
                const V2 e = k < d.fcap ? fent[k] : gent[f0 + k];
                x[i] = dot2(e.x, v.x, e.y, v.y);
            }
        }
        // after the step at width w a lane holds w of the sums, over 32 w / TINV_DN lanes; the
        // first two, up to eight products, in T
        A y[TINV_DN / 4];
#pragma unroll
        for (int w = TINV_DN / 2; w >= 1; w >>= 1) {
            const int o = w * (32 / TINV_DN);
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < w; ++i) {
                if (w >= TINV_DN / 4) {
                    const T send = up ? x[i] : x[i + w], mine = up ? x[i + w] : x[i];
                    x[i] = mine + __shfl_xor_sync(0xffffffffu, send, o);
                    if (w == TINV_DN / 4) y[i] = acc_from(x[i]);
                } else {
                    const A send = up ? y[i] : y[i + w], mine = up ? y[i + w] : y[i];
                    y[i] = acc_merge(mine, acc_shfl_xor(send, o));
                }
            }
        }
#pragma unroll
        for (int o = 16 / TINV_DN; o; o >>= 1) y[0] = acc_merge(y[0], acc_shfl_xor(y[0], o));
        if ((lane & (32 / TINV_DN - 1)) == 0) fden_w[lane / (32 / TINV_DN)][t >> 5] = y[0];
        __syncthreads();
        if (t < TINV_DN * (NT / 32)) {
            // TINV_DN x NT / 32 partial sums: NT / 32 neighbouring lanes a sum
            A z = (&fden_w[0][0])[t];
#pragma unroll
            for (int o = NT / 64; o; o >>= 1) z = acc_merge(z, acc_shfl_xor(z, o));
            const int i = i0 + t / (NT / 32);
            if (t % (NT / 32) == 0 && i < nd) *reinterpret_cast<A*>(a.fsh + fden[i] * d.n_tu + unit) = z;
        }
        if (i0 + TINV_DN < nd) __syncthreads();
    }
}

template <class T, int PUPD>
__global__ void __launch_bounds__(TINV_NT, sizeof(T) == 4 ? 2 : 1) k_tinv(__grid_constant__ const Desc<T> d, __grid_constant__ const ClArgs<T> a) {
    tinv_body<T, PUPD>(d, a, blockIdx.x);
}

// Analysis levels lev0 .. levels - 1 of the h x h block at buf (row stride ld), `tmp` of the
// same size beside it: rows into tmp, columns back, one barrier a pass.  `tail`: the tail
// operator in shared memory, or null.
template <class T>
__device__ __forceinline__ void analyse(T* buf, T* tmp, const T* tail, int n, int lev0, int levels, int ld) {
    constexpr int NT = cblk<T>();
    const int t = threadIdx.x;
    const int lev_end = (tail && tail_applies(n, lev0, levels)) ? levels - 3 : levels;
    for (int lev = lev0; lev < lev_end; ++lev) {
        const int m = n >> lev, hm = m >> 1, lhm = __ffs(hm) - 1, lm = lhm + 1;
        for (int b = t; b < m << lhm; b += NT) {
            const int row = b >> lhm, k = b & (hm - 1);
            const T* x = buf + row * ld;
            T a = T(0), dd = T(0);
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const T v = x[(2 * k + q) & (m - 1)];
                a = fmadd(tap_h<T>(q), v, a);
                dd = fmadd(tap_g<T>(q), v, dd);
            }
            tmp[row * ld + k] = a;
            tmp[row * ld + hm + k] = dd;
        }
        __syncthreads();
        for (int b = t; b < m << lhm; b += NT) {
            const int k = b >> lm, c = b & (m - 1);
            T a = T(0), dd = T(0);
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const T v = tmp[((2 * k + q) & (m - 1)) * ld + c];
                a = fmadd(tap_h<T>(q), v, a);
                dd = fmadd(tap_g<T>(q), v, dd);
            }
            buf[k * ld + c] = a;
            buf[(hm + k) * ld + c] = dd;
        }
        __syncthreads();
    }
    if (lev_end < levels) {
        // the last three levels, one 64 x 64 map: four threads an output, each 16 terms
        T y = T(0);
        const int o = t >> 2, part = t & 3;
        if (t < 256) {
            T acc[2] = {T(0), T(0)};
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int k = 16 * part + i;
                acc[i & 1] = fmadd(tail[k * TAIL_LD + o], buf[(k >> 3) * ld + (k & 7)], acc[i & 1]);
            }
            y = acc[0] + acc[1];
            y += __shfl_down_sync(0xffffffffu, y, 2);
            y += __shfl_down_sync(0xffffffffu, y, 1);
        }
        __syncthreads();
        if (t < 256 && part == 0) buf[(o >> 3) * ld + (o & 7)] = y;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Forward band kernels: c = W sum_g P_g^T u_g (Sec. 2 adjoint, Sec. 3.1) with the epilogue of
// the apply or of the initial residual.  The sensor kernel has applied the column half of
// P_g^T (R_x, per sensor and layer, in pb.Y).  k_tfwd, a CTA per band of rows of a layer and
// its halo of 4: the row half summed over the sensors, the finest analysis level, the
// epilogue of the three detail bands; its LL block goes to a.ll.  k_tcoarse, the other levels
// of a layer of several bands and their epilogue.  A layer of one band (side
// at most 32) is finished by k_tfwd.
//
// Bound: latency again (launch, one block of staged reads, two passes).  Before, a kernel of
// (sensor, layer) pairs made the whole adjoint projection (4.9 us on the MAORY geometry), a
// cluster per layer summed the pairs, transformed and finished on one leader CTA (11 us) and the
// CG update was a kernel (4.3 us); stamps inside a frame now: 6.5 us for the bands and 5 for the
// coarse levels.  Bands of 8 whole rows keep every global read a contiguous block and need a halo
// in one direction only; square tiles with a halo on four sides read the aperture vectors 1.9
// times over and were slower.
// ---------------------------------------------------------------------------
constexpr int TF_BAND = 8;       // rows of a band
constexpr int TF_ONE = 32;       // a layer of this side or less is one band

// Shared-memory offsets of k_tfwd in T units (after the reduction scratch).
struct TfLayout {
    int ye, yo, w, src, lbuf, tail, st, total;
    int gb;             // sensors per pass
};
constexpr int TF_K = 4;          // 16-byte groups per thread, at most

template <class T> struct Quad;
template <> struct Quad<float> {
    float4 v;
    __device__ __forceinline__ void zero() { v = make_float4(0.f, 0.f, 0.f, 0.f); }
    __device__ __forceinline__ void fma(float w, const Quad& q) {
        v = make_float4(fmadd(w, q.v.x, v.x), fmadd(w, q.v.y, v.y), fmadd(w, q.v.z, v.z), fmadd(w, q.v.w, v.w));
    }
    // even and odd columns
    __device__ __forceinline__ void split(float* e, float* o) const {
        *reinterpret_cast<float2*>(e) = make_float2(v.x, v.z);
        *reinterpret_cast<float2*>(o) = make_float2(v.y, v.w);
    }
};
template <> struct Quad<double> {
    double2 v;
    __device__ __forceinline__ void zero() { v = make_double2(0.0, 0.0); }
    __device__ __forceinline__ void fma(double w, const Quad& q) { v = make_double2(fmadd(w, q.v.x, v.x), fmadd(w, q.v.y, v.y)); }
    __device__ __forceinline__ void split(double* e, double* o) const {
        *e = v.x;
        *o = v.y;
    }
};

// Operands of the epilogue at one coefficient.
template <class T>
struct EpiOp {
    T p, b, j, r;
};

// The epilogue at one coefficient: v = (W y)(pos), dl its D.
//   APPLY: q = v + alpha D p, written, p.q;  COEF: v written (PHI has none: the layer itself
//   is written, before the transform);
//   RESID_INIT: r0 = v - alpha D c0 (v is the residual's data term), z = J^-1 r, p = z, r.z;
//   APPLY_INIT: r0 = b - q, the same, and b_prev = b;
//   UPDATE: r -= a q (q written to a.out too, if given), z = J^-1 r, r.z and, with upc,
//   c += a p (step a).
template <class T, int DST>
__device__ __forceinline__ void epi_load(const ClArgs<T>& a, int pos, EpiOp<T>& o) {
    if (DST != LDST_COEF && DST != LDST_PHI) o.p = a.pin[pos];
    if (DST == LDST_APPLY_INIT) o.b = a.vb[pos];
    if (DST == LDST_APPLY_INIT || DST == LDST_RESID_INIT || DST == LDST_UPDATE) o.j = a.vj[pos];
    if (DST == LDST_UPDATE) {
        o.r = a.rin[pos];
    }
}
template <class T, int DST>
__device__ __forceinline__ void epi_apply(const ClArgs<T>& a, T alpha, T dl, int pos, T v, const EpiOp<T>& o,
                                          DotAcc<T>& dot, T step = T(0), bool upc = false) {
    if (DST == LDST_COEF) {
        a.out[pos] = v;
    } else if (DST == LDST_APPLY) {
        const T q = fmadd(alpha * dl, o.p, v);
        a.out[pos] = q;
        dot.add(o.p, q);
    } else if (DST == LDST_UPDATE) {
        const T q = fmadd(alpha * dl, o.p, v);
        if (a.out) a.out[pos] = q;
        const T rr = fmadd(-step, q, o.r);
        const T z = o.j * rr;
        if (upc) a.vc[pos] = fmadd(step, o.p, a.vc[pos]);
        a.vr[pos] = rr;
        a.vz[pos] = z;
        dot.add(rr, z);
    } else {
        const T rr = DST == LDST_RESID_INIT ? fmadd(-(alpha * dl), o.p, v) : o.b - fmadd(alpha * dl, o.p, v);
        const T z = o.j * rr;
        a.vr[pos] = rr;
        a.vz[pos] = z;
        a.vp[pos] = z;
        if (DST == LDST_APPLY_INIT) a.vbprev[pos] = o.b;
        dot.add(rr, z);
    }
}

// Shares of the epilogue's inner product: TC_SH slots a layer (the bands' and the coarse
// levels', then one per quadrant CTA of k_tcoarse), in the instance's slot row.  Unless the
// total is left to the next kernel, the last of the `writers` CTAs forms it (fixed order).
constexpr int TC_SH = 5;
template <class T, int DST>
__device__ __forceinline__ double* layer_slot(const ClArgs<T>& a, int l) {
    return a.lsh + l * TC_SH;
}
template <class T, int DST>
__device__ __forceinline__ void layer_total(const ClArgs<T>& a, int n_layers, int writers) {
    if (DST == LDST_COEF || a.defer_total) return;
    __shared__ bool last;
    unsigned* count = a.pcg.count + (DST == LDST_APPLY ? 1 : 0);
    if (last_arrival(count, static_cast<unsigned>(writers), &last) && threadIdx.x < 32) {
        const typename AccOf<T>::type x = shares_total<T>(layer_slot<T, DST>(a, 0), n_layers * TC_SH);
        const double tot = warp_value(x);
        if (threadIdx.x == 0) {
            if (DST == LDST_APPLY)
                a.pcg.pqtot[a.iter] = tot;
            else
                a.pcg.rztot[a.rzslot] = tot;
            *count = 0;
        }
    }
}

// The row half of P^T at one band row and 16 bytes of columns: acc += sum over nb sensors (in
// order) of at most KT aperture rows each, staged at st.  w: per sensor KT weights (0: no
// such row), then the stage offset of its first row (box column 0); box: per sensor first
// column and columns of its box.
template <class T, int KT>
__device__ __forceinline__ void tf_rows(Quad<T>& acc, const T* st, const T* w, const int2* box, int nb, int j0) {
#pragma unroll 3
    for (int g = 0; g < nb; ++g) {
        const int2 x = box[g];
        const int c = j0 - x.x;
        T f[KT + 1];
        if (KT == 3 && sizeof(T) == 4) {
            const float4 v = *reinterpret_cast<const float4*>(w + g * 4);
            f[0] = v.x; f[1] = v.y; f[2] = v.z; f[KT] = v.w;
        } else {
#pragma unroll
            for (int q = 0; q <= KT; ++q) f[q] = w[g * (KT + 1) + q];
        }
        if (c >= 0 && c < x.y) {
            const T* row = st + static_cast<int>(f[KT]) + c;
#pragma unroll
            for (int q = 0; q < KT; ++q)
                if (f[q] != T(0)) acc.fma(f[q], *reinterpret_cast<const Quad<T>*>(row + q * x.y));
        }
    }
}

template <class T, int DST>
__device__ __forceinline__ void tfwd_body(const Desc<T>& d, const ClArgs<T>& a, const TfLayout& lay,
                                          const PairBufs<T>& pb, const int unit) {
    constexpr int NT = cblk<T>(), V = vec16<T>(), LV = V == 4 ? 2 : 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* red = reinterpret_cast<double*>(smem_raw);
    T* sm = reinterpret_cast<T*>(red + CWMAX);
    const int t = threadIdx.x;
    int l = 0;
    while (unit >= d.bu0[l + 1]) ++l;
    const int band = unit - d.bu0[l], bands = d.bu0[l + 1] - d.bu0[l];
    const LayerInfo L = d.L[l];
    const int n = L.n, h = n >> 1, lh = L.log2n - 1;
    const int bh = bands > 1 ? TF_BAND : n, ry = bands > 1 ? TF_BAND + 4 : n, Y0 = band * bh;
    T* ye = sm + lay.ye;                       // even and odd columns of y, row stride ysd
    T* yo = sm + lay.yo;
    T* sw = sm + lay.w;                        // row weights: [band row][sensor][kt + 1]
    T* lbuf = sm + lay.lbuf;
    const int ysd = (h + 1) & ~1, lsd = h + 1;
    const int kt = d.bkt[l] & 15, tail = d.bkt[l] >> 4;
    __shared__ T sD[MAXLEV + 1];
    __shared__ T salpha;
    if (t <= MAXLEV) sD[t] = d.Dlev[l][t];
    if (t == 0) salpha = d.alpha;
    {
        const int cnt = ry * d.n_wfs * (kt + 1);
        const T* src = d.brow + d.broff[l] + band * cnt;
        for (int k = t; k < cnt; k += NT) cp_async(sw + k, src + k);
    }
    // the staged blocks, and the boxes' columns, per sensor
    int4* src = reinterpret_cast<int4*>(sm + lay.src);
    int2* box = reinterpret_cast<int2*>(src + d.n_wfs);
    for (int k = t; k < d.n_wfs; k += NT) {
        src[k] = reinterpret_cast<const int4*>(d.bsrc)[unit * d.n_wfs + k];
        box[k] = make_int2(d.box[k][l][2], d.box[k][l][3]);
    }
    const bool tail_on = bands == 1 && tail;
    if (tail_on) stage16(sm + lay.tail, d.tailop, TAIL_N, t, NT);
    // the epilogue's operands at this thread's detail coefficients (written two kernels back
    // or earlier)
    const int nblk = (bh >> 1) << lh;
    const int ck = (Y0 >> 1) + (t >> lh), cl = t & (h - 1);
    int pos[3];
    pos[0] = L.off + ck * n + h + cl;
    pos[1] = L.off + (h + ck) * n + cl;
    pos[2] = pos[1] + h;
    EpiOp<T> op[3];
    if (t < nblk) {
#pragma unroll
        for (int e = 0; e < 3; ++e) epi_load<T, DST>(a, pos[e], op[e]);
    }
    constexpr bool UPD = DST == LDST_UPDATE;
    using A = typename AccOf<T>::type;
    __shared__ A spq[2];
    __shared__ T sstep;
    // a layer of one band: its LL quadrant's operands, one per thread, and its layers of c
    const bool one = bands == 1, cll = one && t < h * h;
    const int pll = L.off + (t >> lh) * n + (t & (h - 1));
    EpiOp<T> oll;
    if (cll) epi_load<T, DST>(a, pll, oll);
    constexpr int CPT = TF_ONE * TF_ONE / NT;             // the layers of c and of p, n <= TF_ONE
    T cph[CPT], pph[CPT];
    const bool carry = UPD && one && a.phic;
#pragma unroll
    for (int k = 0; k < CPT; ++k)
        if (carry && t + k * NT < n * n) {
            cph[k] = a.phic[L.off + t + k * NT];
            pph[k] = a.phip[L.off + t + k * NT];
        }
    double rz = 0.0;
    if (UPD && t == NT - 1) rz = a.pcg.rztot[a.iter];
    cp_async_wait();
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    // ---- the row half of the adjoint projection: the aperture rows under the band are one
    // contiguous block per sensor; every copy of a pass in flight together -------------------
    T* st = sm + lay.st;
    const bool quads = n >= V;                            // else a layer narrower than 16 bytes
    const int lq = quads ? L.log2n - LV : L.log2n;        // log2 of the groups per row
    Quad<T> acc[TF_K];
#pragma unroll
    for (int k = 0; k < TF_K; ++k) acc[k].zero();
    const bool layers = DST == LDST_COEF && a.in;         // W of given layers (16-byte aligned)
    if (layers)
#pragma unroll
        for (int k = 0; k < TF_K; ++k) {
            const int task = t + k * NT;
            if (task < (ry << lq)) {
                const T* src = a.in + L.off + ((Y0 + (task >> lq)) & (n - 1)) * n + (task & ((1 << lq) - 1)) * (quads ? V : 1);
                if (quads)
                    acc[k] = *reinterpret_cast<const Quad<T>*>(src);
                else
                    acc[k].v.x = *src;
            }
        }
    for (int g0 = 0; g0 < d.n_wfs && !layers; g0 += lay.gb) {
        const int nb = min(lay.gb, d.n_wfs - g0);
        if (g0 > 0) __syncthreads();
        for (int g = g0; g < g0 + nb; ++g) {
            const int4 e = src[g];
            for (int k = t * V; k < e.y; k += NT * V) cp_async16(st + e.z + k, pb.Y + e.x + k);
        }
        if (UPD && g0 == 0 && t >= NT - 64) {
            // beside the copies, p.q from its shares: two warps, fixed order
            const int w = (t - (NT - 64)) >> 5, half = (a.n_pqs + 1) >> 1;
            const A x = shares_total<T>(a.pqs + w * half, w ? a.n_pqs - half : half);
            if ((t & 31) == 0) spq[w] = x;
        }
        cp_async_wait();
        __syncthreads();
        if (UPD && g0 == 0 && t == NT - 1) {
            // alpha = rz_k / (p . q)_k; zero if rz vanished (the iterate is final)
            const double pq = warp_value(acc_merge(spq[0], spq[1]));
            sstep = T(pq > 0.0 && rz != 0.0 ? rz / pq : 0.0);
            if (unit == 0) {
                a.alphas[a.iter] = sstep;
                a.pcg.pqtot[a.iter] = pq;
            }
        }
#pragma unroll
        for (int k = 0; k < TF_K; ++k) {
            const int task = t + k * NT;
            if (task < (ry << lq)) {
                const int i = task >> lq, j0 = (task & ((1 << lq) - 1)) * (quads ? V : 1);
                const T* w = sw + (i * d.n_wfs + g0) * (kt + 1);
                if (!quads) {
                    T x = T(0);
                    for (int g = 0; g < nb; ++g) {
                        const int2 b = box[g0 + g];
                        const int c = j0 - b.x;
                        if (c < 0 || c >= b.y) continue;
                        const T* row = st + static_cast<int>(w[g * (kt + 1) + kt]) + c;
                        for (int q = 0; q < kt; ++q)
                            if (w[g * (kt + 1) + q] != T(0)) x = fmadd(w[g * (kt + 1) + q], row[q * b.y], x);
                    }
                    acc[k].v.x += x;
                } else if (kt == 3) {
                    tf_rows<T, 3>(acc[k], st, w, box + g0, nb, j0);
                } else if (kt == 5) {
                    tf_rows<T, 5>(acc[k], st, w, box + g0, nb, j0);
                } else {
                    tf_rows<T, KMAX>(acc[k], st, w, box + g0, nb, j0);
                }
            }
        }
    }
    if (DST == LDST_PHI) {
#pragma unroll
        for (int k = 0; k < TF_K; ++k) {
            const int task = t + k * NT;
            if (task < (bh << lq)) {
                T* o = a.out + L.off + (Y0 + (task >> lq)) * n + (task & ((1 << lq) - 1)) * (quads ? V : 1);
                const T* x = reinterpret_cast<const T*>(&acc[k].v);
#pragma unroll
                for (int e = 0; e < V; ++e)
                    if (quads || e == 0) o[e] = x[e];
            }
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < TF_K; ++k) {
        const int task = t + k * NT;
        if (task < (ry << lq)) {
            const int i = task >> lq, j0 = (task & ((1 << lq) - 1)) * (quads ? V : 1);
            if (quads)
                acc[k].split(ye + i * ysd + (j0 >> 1), yo + i * ysd + (j0 >> 1));
            else
                (j0 & 1 ? yo : ye)[i * ysd + (j0 >> 1)] = acc[k].v.x;
        }
    }
    __syncthreads();
    const T step = UPD ? sstep : T(0);
#pragma unroll
    for (int k = 0; k < CPT; ++k)
        if (carry && t + k * NT < n * n) a.phic[L.off + t + k * NT] = fmadd(step, pph[k], cph[k]);
    // ---- the finest analysis level: rows, then columns ---------------------------------------
    // In double the row half once per row, through shared memory (the staging buffer, read
    // by now): about 50 multiply-adds a block of four where the fused form has 96, on a pipe of
    // two a cycle; the MAORY frame takes 550 us, 563 with the fused form, an 8 m iteration 43, 48.
    // Single precision is bound by latency and keeps the form with one barrier less.
    constexpr bool SPLIT = sizeof(T) == 8;
    const int msd = n + 1;
    T* mid = st;
    if (SPLIT) {
        for (int b = t; b < ry << lh; b += NT) {
            const int i = b >> lh, kx = b & (h - 1);
            T av = T(0), dv = T(0);
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const T x = (q & 1 ? yo : ye)[i * ysd + ((kx + (q >> 1)) & (h - 1))];
                av = fmadd(tap_h<T>(q), x, av);
                dv = fmadd(tap_g<T>(q), x, dv);
            }
            mid[i * msd + kx] = av;
            mid[i * msd + h + kx] = dv;
        }
        __syncthreads();
    }
    DotAcc<T> dot;
    // A block per thread: pos and op are those of block t.  Written as a loop, which runs once, the
    // MAORY frame takes 135.2 us, as a condition 137.4 (the same commands).
    static_assert((TF_BAND / 2) * (MAXN / 2) <= NT && (TF_ONE / 2) * (TF_ONE / 2) <= NT, "a block per thread");
    for (int b = t; b < nblk; b += NT) {
        const int msk = bands > 1 ? 15 : n - 1;           // a band holds its halo
        const int ky = 2 * (b >> lh), kx = b & (h - 1);
        T ra[6], rd[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            if (SPLIT) {
                const T* m = mid + ((ky + r) & msk) * msd + kx;
                ra[r] = m[0];
                rd[r] = m[h];
                continue;
            }
            const T* re = ye + ((ky + r) & msk) * ysd;
            const T* ro = yo + ((ky + r) & msk) * ysd;
            T av = T(0), dv = T(0);
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const T x = (q & 1 ? ro : re)[(kx + (q >> 1)) & (h - 1)];
                av = fmadd(tap_h<T>(q), x, av);
                dv = fmadd(tap_g<T>(q), x, dv);
            }
            ra[r] = av;
            rd[r] = dv;
        }
        T ll = T(0), v[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            ll = fmadd(tap_h<T>(r), ra[r], ll);
            v[0] = fmadd(tap_h<T>(r), rd[r], v[0]);
            v[1] = fmadd(tap_g<T>(r), ra[r], v[1]);
            v[2] = fmadd(tap_g<T>(r), rd[r], v[2]);
        }
        const int rk = (Y0 >> 1) + (b >> lh);
        if (bands > 1)
            a.ll[(L.off >> 2) + rk * h + kx] = ll;
        else
            lbuf[rk * lsd + kx] = ll;
#pragma unroll
        for (int e = 0; e < 3; ++e) epi_apply<T, DST>(a, salpha, sD[1], pos[e], v[e], op[e], dot, step, one);
    }
    if (bands == 1) {
        // ---- the other levels of a layer of one band ------------------------------------------
        __syncthreads();
        if (L.levels >= 2) analyse<T>(lbuf, lbuf + h * lsd, tail_on ? sm + lay.tail : nullptr, n, 1, L.levels, lsd);
        // The data term has no piston component: Gamma annihilates constants and bilinear
        // weights sum to one, so its full-depth LL coefficient is exactly 0.  Write that zero
        // rather than the rounding residue of a cancelling sum, which the solve would amplify
        // by 1 / (alpha D_LL).
        if (a.zero_piston && L.full && t == 0) lbuf[0] = T(0);
        __syncthreads();
        if (cll) {
            const int i = t >> lh, j = t & (h - 1);
            epi_apply<T, DST>(a, salpha, sD[level_of(i, j, L)], pll, lbuf[i * lsd + j], oll, dot, step, true);
        }
    }
    if (DST != LDST_COEF) {
        cta_share<T>(dot, red, nullptr, bands > 1 ? a.tshare + unit : layer_slot<T, DST>(a, l));
        if (bands == 1) layer_total<T, DST>(a, d.n_layers, d.n_writers);
    }
}

template <class T, int DST>
__global__ void __launch_bounds__(cblk<T>(), sizeof(T) == 4 ? 2 : 1)
    k_tfwd(__grid_constant__ const Desc<T> d, __grid_constant__ const ClArgs<T> a,
           __grid_constant__ const TfLayout lay, __grid_constant__ const PairBufs<T> pb) {
    tfwd_body<T, DST>(d, a, lay, pb, blockIdx.x);
}

// The levels below the finest of a layer of several bands and their epilogue, CTA `unit` of
// d.tcl = {layer, part}: part 0, the leader, the level below the finest (its scaling half only)
// and all coarser ones; parts 1 .. 4 the detail bands of the level below the finest, a
// quadrant of 16 x 16 coefficients each; parts above, c += alpha p and the layers of c, a
// chunk of TC_VEC each (they hide behind the leader).  The LL block (a.ll) comes from k_tfwd;
// operands are read before the wait.
//
// Bound: the leader's chain of passes, latency of one CTA: 5.0 us of a MAORY iteration in
// single precision, with the updates of c, of its layers, of r and z hidden beside it on CTAs of
// their own.
constexpr int TC_VEC = 2048;
struct TcLayout {
    int lbuf, tmp, tail, st, total;  // T units after the reduction scratch; st: staged operands
};

template <class T, int DST>
__device__ __forceinline__ void tcoarse_body(const Desc<T>& d, const ClArgs<T>& a, const TcLayout& lay, const int unit) {
    constexpr int NT = cblk<T>();
    constexpr bool QP = DST != LDST_COEF, UPD = DST == LDST_UPDATE;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* red = reinterpret_cast<double*>(smem_raw);
    T* sm = reinterpret_cast<T*>(red + CWMAX);
    const int t = threadIdx.x;
    const int code = d.tcl[unit], l = code & 255, part = code >> 8;
    const LayerInfo L = d.L[l];
    const int n = L.n, h = n >> 1, lh = L.log2n - 1, hh = h >> 1, lhh = lh - 1;
    __shared__ T sD[MAXLEV + 1];
    __shared__ T salpha, sstep;
    __shared__ double bands;             // the bands' share of the inner product
    if (part > TC_SH - 1) {
        // ---- c += alpha p, phi_c += alpha phi_p --------------------------------------------
        pdl_wait();
        pdl_trigger();
        if (!UPD) return;
        const T step = a.alphas[a.iter];
        const int k0 = (part - TC_SH) * TC_VEC, k1 = min(k0 + TC_VEC, n * n);
        for (int k = k0 + t; k < k1; k += NT) {
            a.vc[L.off + k] = fmadd(step, a.pin[L.off + k], a.vc[L.off + k]);
            if (a.phic) a.phic[L.off + k] = fmadd(step, a.phip[L.off + k], a.phic[L.off + k]);
        }
        return;
    }
    if (t <= MAXLEV) sD[t] = d.Dlev[l][t];
    if (t == 0) salpha = d.alpha;
    const T* src = a.ll + (L.off >> 2);
    DotAcc<T> dot;
    if (part > 0) {
        // ---- detail bands of the level below the finest: 16 x 16 coefficients each ------------
        constexpr int R = 36, RS = 37;   // region of the LL block, its row stride
        T* buf = sm + lay.lbuf;
        const bool has = L.levels >= 2;
        const int ky0 = hh > 16 ? ((part - 1) >> 1) * 16 : 0, kx0 = hh > 16 ? ((part - 1) & 1) * 16 : 0;
        const int ck = ky0 + ((t >> 4) & 15), cl = kx0 + (t & 15);
        const int pos[3] = {L.off + ck * n + hh + cl, L.off + (hh + ck) * n + cl, L.off + (hh + ck) * n + hh + cl};
        EpiOp<T> op[3];
        if (t < 256 && has) {
#pragma unroll
            for (int e = 0; e < 3; ++e) epi_load<T, DST>(a, pos[e], op[e]);
        }
        __syncthreads();
        pdl_wait();
        pdl_trigger();
        if (!has) return;
        if (UPD && t == 0) sstep = a.alphas[a.iter];
        for (int k = t; k < R * R; k += NT) {
            const int i = k / R, j = k - i * R;
            buf[i * RS + j] = src[((2 * ky0 + i) & (h - 1)) * h + ((2 * kx0 + j) & (h - 1))];
        }
        __syncthreads();
        if (t < 256) {
            const int ky = 2 * (t >> 4), kx = 2 * (t & 15);
            T v[3] = {T(0), T(0), T(0)};
#pragma unroll
            for (int r = 0; r < 6; ++r) {
                const T* x = buf + (ky + r) * RS + kx;
                T av = T(0), dv = T(0);
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    av = fmadd(tap_h<T>(q), x[q], av);
                    dv = fmadd(tap_g<T>(q), x[q], dv);
                }
                v[0] = fmadd(tap_h<T>(r), dv, v[0]);
                v[1] = fmadd(tap_g<T>(r), av, v[1]);
                v[2] = fmadd(tap_g<T>(r), dv, v[2]);
            }
#pragma unroll
            for (int e = 0; e < 3; ++e) epi_apply<T, DST>(a, salpha, sD[2], pos[e], v[e], op[e], dot, sstep);
        }
        if (QP) {
            cta_share<T>(dot, red, nullptr, layer_slot<T, DST>(a, l) + part);
            layer_total<T, DST>(a, d.n_layers, d.n_writers);
        }
        return;
    }
    // ---- the leader: LL of the level below the finest, the coarser levels -----------------------
    T* lbuf = sm + lay.lbuf;
    T* tmp = sm + lay.tmp;
    const bool two = L.levels >= 2;      // else the LL block is the layer's LL band
    const int m = two ? hh : h, lm = two ? lhh : lh, ld = m + 1, hs = h + 1;
    const bool tail_on = lay.tail > 0 && (d.bkt[l] >> 4);
    const int unit0 = d.bu0[l], units = d.bu0[l + 1] - d.bu0[l];
    if (tail_on) stage16(sm + lay.tail, d.tailop, TAIL_N, t, NT);
    // operands of the epilogue at this thread's coefficients (two a thread at h = 64)
    constexpr int TK = 4;
    EpiOp<T> op[TK];
#pragma unroll
    for (int k = 0; k < TK; ++k) {
        const int b = t + k * NT;
        if (b < m << lm) epi_load<T, DST>(a, L.off + (b >> lm) * n + (b & (m - 1)), op[k]);
    }
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    if (UPD && t == 0) sstep = a.alphas[a.iter];
    if (QP && t >= NT - 32) {
        const typename AccOf<T>::type x = shares_total<T>(a.tshare + unit0, units);
        if (t == NT - 32) *reinterpret_cast<typename AccOf<T>::type*>(&bands) = x;
    }
    if (two) {
        // the scaling half of the level below the finest, rows then columns
        T* raw = tmp;                                     // h x h, row stride h + 1
        T* mid = sm + lay.st;                             // h x hh, row stride hh + 1
        for (int k = t; k < h << lh; k += NT) raw[(k >> lh) * hs + (k & (h - 1))] = src[k];
        cp_async_wait();
        __syncthreads();
        for (int b = t; b < h << lhh; b += NT) {
            const int row = b >> lhh, k = b & (hh - 1);
            const T* x = raw + row * hs;
            T av = T(0);
#pragma unroll
            for (int q = 0; q < 6; ++q) av = fmadd(tap_h<T>(q), x[(2 * k + q) & (h - 1)], av);
            mid[row * ld + k] = av;
        }
        __syncthreads();
        for (int b = t; b < hh << lhh; b += NT) {
            const int k = b >> lhh, c = b & (hh - 1);
            T av = T(0);
#pragma unroll
            for (int q = 0; q < 6; ++q) av = fmadd(tap_h<T>(q), mid[((2 * k + q) & (h - 1)) * ld + c], av);
            lbuf[k * ld + c] = av;
        }
        __syncthreads();
        if (L.levels >= 3) analyse<T>(lbuf, tmp, tail_on ? sm + lay.tail : nullptr, n, 2, L.levels, ld);
    } else {
        cp_async_wait();
        for (int k = t; k < h << lh; k += NT) lbuf[(k >> lh) * ld + (k & (h - 1))] = src[k];
        __syncthreads();
    }
    if (a.zero_piston && L.full && t == 0) lbuf[0] = T(0);   // no piston in the data term (see tfwd_body)
    __syncthreads();
#pragma unroll
    for (int k = 0; k < TK; ++k) {
        const int b = t + k * NT, i = b >> lm, j = b & (m - 1);
        if (b < m << lm)
            epi_apply<T, DST>(a, salpha, sD[level_of(i, j, L)], L.off + i * n + j, lbuf[i * ld + j], op[k], dot,
                              UPD ? sstep : T(0));
    }
    for (int b = t + TK * NT; b < m << lm; b += NT) {        // an LL band that is not transformed further
        const int i = b >> lm, j = b & (m - 1), p = L.off + i * n + j;
        EpiOp<T> o;
        epi_load<T, DST>(a, p, o);
        epi_apply<T, DST>(a, salpha, sD[level_of(i, j, L)], p, lbuf[i * ld + j], o, dot, UPD ? sstep : T(0));
    }
    if (QP) {
        cta_share<T>(dot, red, &bands, layer_slot<T, DST>(a, l));
        layer_total<T, DST>(a, d.n_layers, d.n_writers);
    }
}

template <class T, int DST>
__global__ void __launch_bounds__(cblk<T>(), sizeof(T) == 4 ? 2 : 1)
    k_tcoarse(__grid_constant__ const Desc<T> d, __grid_constant__ const ClArgs<T> a, __grid_constant__ const TcLayout lay) {
    tcoarse_body<T, DST>(d, a, lay, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Sensor kernel, a CTA per band of TS_ROWS subaperture rows of a sensor: P_g (Sec. 2),
// Gamma_g, C_hat_g^-1 (Eq. 2, Sec. 3.2), Gamma_g^T and the column half of P_g^T.  SRC_PHI:
// slopes of the projected layers (the M-apply); SRC_RESID: measured minus modelled slopes
// (the initial residual); SRC_SLOPES: measured slopes (the right-hand side); SRC_RAW: the same
// without C_hat_g^-1 (the model's adjoint).  The layers are read by direct bilinear gathers; the
// result goes out per layer as the aperture rows' values on the layer's columns (pb.Y, slot g * n_layers + l, rows of box[3] columns), whose
// row half the band kernel applies.
//
// No CTA waits for another.  What the weighting of one subaperture needs of all the others
// (the tip/tilt means of a laser star, the block sums of a coarse sensor, the elongation's
// sums) are linear functionals of the layers, whose shares the inverse kernel's tiles have
// formed; the slopes of the row below the band are formed here once more.
//
// Bound: latency (launch, the gather's L2 reads, two barriers): 6 us a launch on the MAORY
// geometry, 180 CTAs; with the sums inside clusters of 16 CTAs 8.5 us, 3 of them before the
// clusters started: a cluster waits for a group of SMs to be free, so nothing of
// its prologue hides behind the kernel before.  Bands of 4 rows instead of 5 keep a CTA at
// 512 threads of 64 registers, which fit beside the neighbours'; 576 of 56 did not.
// ---------------------------------------------------------------------------
constexpr int TS_ROWS = 4;       // 6 node rows of 81 nodes are one pass of 512 threads
constexpr int TS_LG = 5;         // layers with their loads in flight together
constexpr int TS_FUN = 2 * MAXCOARSE;            // functionals of a sensor, at most

// 512 threads of at most 64 registers fit beside the CTAs of the kernels before and after
// (each scheduler's registers hold four warps of each), so the prologue is hidden.
template <class T>
__host__ __device__ constexpr int tsnt() {
    return sizeof(T) == 4 ? 512 : 256;
}
struct TsLayout {       // shared-memory offsets in T units
    int V, SX, SY, msk, xi, xf, yi, yf, ci, dot, total;
};

template <class T, int SRC>
__device__ __forceinline__ void tsen_body(const Desc<T>& d, const SensorArgs<T>& a, const TsLayout& lay,
                                          const PairBufs<T>& pb, const int unit) {
    constexpr int NT = tsnt<T>(), SR = TS_ROWS;
    constexpr bool FROM_PHI = SRC == SSRC_PHI || SRC == SSRC_RESID;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31, nwarp = NT >> 5;
    // the sensor's constants in shared memory: the kernel-parameter bank is cold, and its
    // first reads would stand behind the dependency wait (a copy in device memory is read:
    // indexed reads of the parameters are slow)
    __shared__ WfsInfo sW;
    __shared__ int sco[MAXL + 1];                        // first column of each layer
    __shared__ int4 ybox[MAXL];                          // each layer: box columns, offset in Y, place of box column 0
    __shared__ T tot[TS_FUN];                            // the sensor's functionals
    __shared__ T cw[TS_FUN];                             // weighted coarse slopes / nb
    int g = 0;
    while (unit >= d.su0[g + 1]) ++g;
    const int nl = d.n_layers, NPs = d.tnp, n_tu = d.n_tu;
    const int N = d.G[g].N, NP = N + 1, f0 = d.f0[g], nf = d.f0[g + 1] - f0;
    const int s0 = (unit - d.su0[g]) * SR, s1 = min(s0 + SR, N), rows = s1 - s0;
    const int h0 = s0 > 0 ? 1 : 0;                       // the row below the band, if any
    const int q0 = s0 - h0, nrow = rows + h0;            // slope rows [q0, s1), node rows [q0, s1]
    T* Vb = sm + lay.V;         // (nrow + 1) x NP: node values, later the adjoint's
    T* SX = sm + lay.SX;        // nrow x N
    T* SY = sm + lay.SY;
    int* msk = reinterpret_cast<int*>(sm + lay.msk);
    int* xi = reinterpret_cast<int*>(sm + lay.xi);       // [layer][node column]: place of its layer column
    T* xf = sm + lay.xf;
    int2* yi = reinterpret_cast<int2*>(sm + lay.yi);     // [layer][node row]: offset of its layer row, row pitch
    T* yf = sm + lay.yf;
    int* cin = reinterpret_cast<int*>(sm + lay.ci);      // per layer column: first aperture column | count << 16
    using A = typename AccOf<T>::type;
    A* dots = reinterpret_cast<A*>(sm + lay.dot);        // the threads' shares of p.q
    // ---- set-up tables, copied before the dependency wait ---------------------------------
    for (int k = t; k < static_cast<int>(sizeof(WfsInfo) / sizeof(int)); k += NT)
        reinterpret_cast<int*>(&sW)[k] = reinterpret_cast<const int*>(d.gdev + g)[k];
    {
        const int* src = d.sidx + d.G[g].mask_off + q0 * N;
        for (int k = t; k < nrow * N; k += NT) cp_async(msk + k, src + k);
    }
    const int nx = nl * NPs;
    stage16(xi, d.txi + g * nx, nx, t, NT);
    stage16(xf, d.txf + g * nx, nx, t, NT);
    if (FROM_PHI) {
        for (int k = t; k < nl * 8; k += NT) {
            const int l = k >> 3, i = k & 7;
            if (i <= nrow) {
                yi[l * (SR + 2) + i] = reinterpret_cast<const int2*>(d.tyi)[g * nx + l * NPs + q0 + i];
                yf[l * (SR + 2) + i] = d.tyf[g * nx + l * NPs + q0 + i];
            }
        }
    }
    if (t < 32) {
        for (int k = t; k <= nl; k += 32) sco[k] = d.tsco[g * (MAXL + 1) + k];
        for (int k = t; k < nl; k += 32) ybox[k] = reinterpret_cast<const int4*>(d.tybox)[g * MAXL + k];
    }
    stage16(cin, d.tcin + g * d.tcols, d.tcols, t, NT);
    cp_async_wait();
    __syncthreads();
    const WfsInfo& W = sW;
    const T inv = SRC == SSRC_RAW ? T(1) : T(W.sig2inv);
    const T nbinv = T(1) / T(W.nb);
    const int nu = d.su0[d.n_wfs], np = (d.n_c + nu - 1) / nu;           // this CTA's part of p.D p
    const T alpha = d.alpha;
    pdl_wait();
    pdl_trigger();
    bool bad = false;                          // a non-finite measured slope (SLOPES, RESID)
    DotAcc<T> dot;
    // ---- the sensor's functionals: the tiles' shares, a warp each, in flight beside the gather
    for (int f = warp; f < (SRC == SSRC_RAW ? 0 : nf); f += nwarp) {
        A x = AccOf<T>::zero();
        if (FROM_PHI) x = shares_total<T, 6>(a.fsh + (f0 + f) * n_tu, n_tu);
        if (lane == 0) {
            // the residual of a laser star: measured minus modelled
            if (SRC != SSRC_PHI && W.lgs)
                x = acc_merge(*reinterpret_cast<const A*>(a.msum + f0 + f), acc_neg(x));
            tot[f] = T(warp_value(x));
        }
    }
    if (FROM_PHI) {
        // ---- V = P_g phi on node rows [q0, s1]: a thread per node, the layers in order ----
        for (int k = t; k < (nrow + 1) * NP; k += NT) {
            const int ia = k / NP, b = k - ia * NP;
            T v = T(0);
            for (int l0 = 0; l0 < nl; l0 += TS_LG) {
                T q[TS_LG][4];
#pragma unroll
                for (int e = 0; e < TS_LG; ++e)
                    if (l0 + e < nl) {
                        const int2 y = yi[(l0 + e) * (SR + 2) + ia];
                        const T* p = a.phi + xi[(l0 + e) * NPs + b] + y.x;
                        q[e][0] = p[0];
                        q[e][1] = p[1];
                        q[e][2] = p[y.y];
                        q[e][3] = p[y.y + 1];
                    }
#pragma unroll
                for (int e = 0; e < TS_LG; ++e)
                    if (l0 + e < nl) {
                        const T fx = xf[(l0 + e) * NPs + b], fy = yf[(l0 + e) * (SR + 2) + ia];
                        const T h0 = dot2(T(1) - fx, q[e][0], fx, q[e][1]), h1 = dot2(T(1) - fx, q[e][2], fx, q[e][3]);
                        v += dot2(T(1) - fy, h0, fy, h1);
                    }
            }
            Vb[k] = v;
        }
    }
    if (SRC == SSRC_PHI && a.pqs) {
        // this CTA's part of alpha p.D p
        for (int k = t; k < np; k += NT) {
            const int i = unit * np + k;
            if (i < d.n_c) {
                const T p = a.p[i];
                dot.add(alpha * d.D[i] * p, p);
            }
        }
    }
    __syncthreads();
    const bool coarse = FROM_PHI && W.nb > 1;
    if (coarse) {
        // coarse slope = block sum / nb; Gamma_coarse^T spreads sigma^-2 slope / nb.  The
        // residual form subtracts it from the block's measured slope.
        const int ns = W.n_sub;
        if (t < 2 * ns * ns) {
            T x = tot[t] * nbinv;
            if (SRC == SSRC_RESID) {
                const int K = d.cidx[W.cmask_off + (t >> 1)];
                T m = T(0);
                if (K >= 0) {
                    m = a.in[W.soff + (t & 1) * W.n_active + K];
                    bad |= !isfinite(m);
                }
                x = m - x;
            } else if (unit == d.su0[g] && a.pqs) {
                dot.add(x, inv * x);                         // s . sigma^-2 s, once a sensor
            }
            cw[t] = x * inv * nbinv;
        }
        __syncthreads();
    }
    // ---- the weighted slopes of rows [q0, s1) ------------------------------------------------
    T mx = T(0), my = T(0), g1 = T(0), g2 = T(0);
    if (W.lgs && SRC != SSRC_RAW) {
        mx = tot[0] / T(W.n_active);
        my = tot[1] / T(W.n_active);
        if (W.el) {
            g1 = (tot[2] - dot2(el_K(W, 0, T()), mx, el_K(W, 1, T()), my)) / T(W.n_active);
            g2 = (tot[3] - dot2(el_K(W, 1, T()), mx, el_K(W, 2, T()), my)) / T(W.n_active);
        }
    }
    for (int k = t; k < nrow * N; k += NT) {
        const int ii = k / N, j = k - ii * N, id = msk[k];
        T wx = T(0), wy = T(0);
        if (id >= 0) {
            if (coarse) {
                const int blk = ((q0 + ii) / W.nb) * W.n_sub + j / W.nb;
                wx = cw[2 * blk];
                wy = cw[2 * blk + 1];
            } else {
                T sx = T(0), sy = T(0);
                if (FROM_PHI) {
                    // Gamma_g on the modelled nodes
                    const T v00 = Vb[ii * NP + j], v01 = Vb[ii * NP + j + 1];
                    const T v10 = Vb[(ii + 1) * NP + j], v11 = Vb[(ii + 1) * NP + j + 1];
                    sx = T(0.5) * ((v01 - v00) + (v11 - v10));
                    sy = T(0.5) * ((v10 - v00) + (v11 - v01));
                }
                if (SRC != SSRC_PHI) {
                    const T ax = a.in[W.soff + id], ay = a.in[W.soff + W.n_active + id];
                    bad |= !(isfinite(ax) && isfinite(ay));
                    sx = ax - sx;
                    sy = ay - sy;
                }
                if (W.lgs && SRC != SSRC_RAW) {
                    // C_hat^-1 = (I - T) C^-1 (I - T): sigma^-2 (s - m) or, elongated,
                    // sigma^-2 (u - gamma beta (beta . u) + g), u = s - m, g = (e - K m) / |M|
                    // the mean of gamma beta (beta . u)
                    T ux = sx - mx, uy = sy - my;
                    if (W.el) {
                        T b1, b2, gam;
                        elong(W, q0 + ii, j, b1, b2, gam);
                        const T bu = dot2(b1, ux, b2, uy);
                        ux = fmadd(-(gam * b1), bu, ux) + g1;
                        uy = fmadd(-(gam * b2), bu, uy) + g2;
                    }
                    wx = inv * ux;
                    wy = inv * uy;
                } else if (W.nb > 1) {
                    wx = sx * (nbinv * inv);                 // SLOPES of a coarse sensor
                    wy = sy * (nbinv * inv);
                } else {
                    wx = inv * sx;                           // NGS: C^-1 = sigma^-2 I
                    wy = inv * sy;
                }
                if (SRC == SSRC_PHI && a.pqs && ii >= h0) {
                    dot.add(sx, wx);
                    dot.add(sy, wy);
                }
            }
        }
        SX[k] = wx;
        SY[k] = wy;
    }
    if (SRC == SSRC_PHI && a.pqs) dots[t] = AccOf<T>::of(dot);
    if (bad && a.status) atomicOr(a.status, 1u);
    __syncthreads();
    // ---- Gamma_g^T on node rows [s0, s1) (and row N on the last band) ------------------------
    const int nout = (s1 == N) ? rows + 1 : rows;
    for (int k = t; k < nout * NP; k += NT) {
        const int ia = k / NP, b = k - ia * NP;
        // subaperture row s0 + ia (below the node) and the one before (above)
        const bool has0 = s0 + ia < N, has1 = s0 + ia > 0, c0 = b < N, c1 = b > 0;
        const T* x0 = SX + (ia + h0) * N;
        const T* y0 = SY + (ia + h0) * N;
        const T* x1 = x0 - N;
        const T* y1 = y0 - N;
        const T x_ab = (has0 && c0) ? x0[b] : T(0);
        const T x_ab1 = (has0 && c1) ? x0[b - 1] : T(0);
        const T x_a1b = (has1 && c0) ? x1[b] : T(0);
        const T x_a1b1 = (has1 && c1) ? x1[b - 1] : T(0);
        const T y_ab = (has0 && c0) ? y0[b] : T(0);
        const T y_ab1 = (has0 && c1) ? y0[b - 1] : T(0);
        const T y_a1b = (has1 && c0) ? y1[b] : T(0);
        const T y_a1b1 = (has1 && c1) ? y1[b - 1] : T(0);
        Vb[k] = T(0.5) * ((x_ab1 - x_ab) + (x_a1b1 - x_a1b)) + T(0.5) * ((y_a1b - y_ab) + (y_a1b1 - y_ab1));
    }
    __syncthreads();
    if (SRC == SSRC_PHI && a.pqs && warp == nwarp - 1) {
        // the CTA's share of p.q, by the warp with the fewest columns below
        A x = dots[lane];
        for (int k = lane + 32; k < NT; k += 32) x = acc_merge(x, dots[k]);
        x = acc_warp(x);
        if (lane == 0) *reinterpret_cast<A*>(a.pqs + unit) = x;
    }
    // ---- the column half of P_g^T: a thread owns a layer column and takes every row -----------
    for (int k = t; k < sco[nl]; k += NT) {
        int l = 0;
        while (k >= sco[l + 1]) ++l;
        const int4 yb = ybox[l];
        const int j = k - sco[l], cols = yb.x, at = yb.z + j;    // at: the column's place, as in xi
        if (j >= cols) continue;
        const int2 c = make_int2(cin[k] & 0xffff, cin[k] >> 16);
        T* dst = pb.Y + yb.y + s0 * cols + j;
        const T* src = Vb + c.x;
        // node column b has the weight 1 - f on its layer column and f on the next one
        const int* bi = xi + l * NPs + c.x;
        const T* bf = xf + l * NPs + c.x;
        if (c.y <= 3) {
            T w[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) w[q] = q < c.y ? (bi[q] == at ? T(1) - bf[q] : bf[q]) : T(0);
#pragma unroll
            for (int ia = 0; ia < SR + 1; ++ia)
                if (ia < nout) {
                    T x = T(0);
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        if (q < c.y) x = fmadd(w[q], src[ia * NP + q], x);
                    dst[ia * cols] = x;
                }
        } else {
            T w[KMAX];
#pragma unroll
            for (int q = 0; q < KMAX; ++q) w[q] = q < c.y ? (bi[q] == at ? T(1) - bf[q] : bf[q]) : T(0);
            for (int ia = 0; ia < nout; ++ia) {
                T x = T(0);
#pragma unroll
                for (int q = 0; q < KMAX; ++q)
                    if (q < c.y) x = fmadd(w[q], src[ia * NP + q], x);
                dst[ia * cols] = x;
            }
        }
    }
}

template <class T, int SRC>
__global__ void __launch_bounds__(tsnt<T>(), sizeof(T) == 4 ? 2 : 1)
    k_tsen(__grid_constant__ const Desc<T> d, __grid_constant__ const SensorArgs<T> a,
           __grid_constant__ const TsLayout lay, __grid_constant__ const PairBufs<T> pb) {
    tsen_body<T, SRC>(d, a, lay, pb, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Operators beside the frame.  One CTA per sensor or layer took 34 us for the slopes of a
// MAORY-size system's layers, 133 us for the adjoint and 41 us for the adjoint of the fit;
// these spread each over the chip: 19 us, 11 us (k_tsen, k_tfwd) and about 8 us.
// ---------------------------------------------------------------------------

// Slopes of layers, s = Gamma P phi: a CTA per band of TS_ROWS subaperture rows of a fine sensor
// or per subaperture of a coarse one (the mean over its block, summed in double).  Bound by
// the latency of the tables' and the layers' loads.
constexpr int OP_NT = 256;

template <class T>
__global__ void __launch_bounds__(OP_NT) k_model_slopes(__grid_constant__ const Desc<T> d, const T* phi, T* out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* V = reinterpret_cast<T*>(smem_raw);
    __shared__ double ws[2][OP_NT / 32];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    int g = 0, u = blockIdx.x;
    for (;; ++g) {
        const int cnt = d.G[g].nb > 1 ? d.G[g].n_sub * d.G[g].n_sub : (d.G[g].N + TS_ROWS - 1) / TS_ROWS;
        if (u < cnt) break;
        u -= cnt;
    }
    const WfsInfo& W = d.G[g];
    const int N = W.N, nb = W.nb, K = nb > 1 ? d.cidx[W.cmask_off + u] : 0;
    if (K < 0) return;                                   // an inactive coarse subaperture
    const int i0 = nb > 1 ? u / W.n_sub * nb : u * TS_ROWS, j0 = nb > 1 ? u % W.n_sub * nb : 0;
    const int rows = nb > 1 ? nb : min(TS_ROWS, N - i0), cols = nb > 1 ? nb : N, vw = cols + 1;
    pdl_wait();
    pdl_trigger();
    for (int k = t; k < (rows + 1) * vw; k += OP_NT) {
        const int ia = k / vw, aa = i0 + ia, bb = j0 + k - ia * vw;
        T v = T(0);
#pragma unroll 3
        for (int l = 0; l < d.n_layers; ++l) {
            const int tp = (g * MAXL + l) * TAB, n = d.L[l].n;
            const T fy = d.pfy[tp + aa], fx = d.pfx[tp + bb];
            const T* P = phi + d.L[l].off + d.pi0y[tp + aa] * n + d.pi0x[tp + bb];
            v += (T(1) - fy) * ((T(1) - fx) * P[0] + fx * P[1]) + fy * ((T(1) - fx) * P[n] + fx * P[n + 1]);
        }
        V[k] = v;
    }
    __syncthreads();
    double tx = 0.0, ty = 0.0;
    for (int k = t; k < rows * cols; k += OP_NT) {
        const int i = k / cols, j = k - i * cols, id = d.sidx[W.mask_off + (i0 + i) * N + j0 + j];
        if (id < 0) continue;
        const T* p = V + i * vw + j;
        const T sx = T(0.5) * ((p[1] - p[0]) + (p[vw + 1] - p[vw])), sy = T(0.5) * ((p[vw] - p[0]) + (p[vw + 1] - p[1]));
        if (nb > 1) {
            tx += double(sx);
            ty += double(sy);
        } else {
            out[W.soff + id] = sx;
            out[W.soff + W.n_active + id] = sy;
        }
    }
    if (nb <= 1) return;
    tx = warp_sum(tx);
    ty = warp_sum(ty);
    if (lane == 0) {
        ws[0][warp] = tx;
        ws[1][warp] = ty;
    }
    __syncthreads();
    if (t < 2) {
        double x = 0.0;
        for (int w = 0; w < OP_NT / 32; ++w) x += ws[t][w];
        out[W.soff + t * W.n_active + K] = T(x / nb);
    }
}

// C_hat^-1 s of every sensor (blockIdx.y) from the sums of k_msum (Sec. 3.2, Eq. 3), as in
// tsen_body, but the means and e - K m, which cancels for an elongated star, in double.
template <class T>
__global__ void __launch_bounds__(OP_NT) k_weigh(__grid_constant__ const Desc<T> d, const T* s, const double* msum,
                                                 T* out, unsigned* status) {
    using A = typename AccOf<T>::type;
    const int g = blockIdx.y, k = blockIdx.x * OP_NT + threadIdx.x;
    const WfsInfo& W = d.G[g];
    const int cells = W.nb > 1 ? W.n_active : W.N * W.N;
    const int id = k >= cells ? -1 : W.nb > 1 ? k : d.sidx[W.mask_off + k];
    pdl_wait();
    pdl_trigger();
    if (id < 0) return;
    const T inv = T(W.sig2inv);
    T ux = s[W.soff + id], uy = s[W.soff + W.n_active + id];
    if (!(isfinite(ux) && isfinite(uy)) && status) atomicOr(status, 1u);
    if (W.lgs && W.nb == 1) {
        const A* m = reinterpret_cast<const A*>(msum + d.f0[g]);
        const T mx = T(warp_value(m[0]) / W.n_active), my = T(warp_value(m[1]) / W.n_active);
        ux -= mx;
        uy -= my;
        if (W.el) {
            const T g1 = T((warp_value(m[2]) - (W.el_K11 * double(mx) + W.el_K12 * double(my))) / W.n_active);
            const T g2 = T((warp_value(m[3]) - (W.el_K12 * double(mx) + W.el_K22 * double(my))) / W.n_active);
            T b1, b2, gam;
            elong(W, k / W.N, k % W.N, b1, b2, gam);
            const T bu = b1 * ux + b2 * uy;
            ux = fmadd(-(gam * b1), bu, ux) + g1;
            uy = fmadd(-(gam * b2), bu, uy) + g2;
        }
    }
    out[W.soff + id] = inv * ux;
    out[W.soff + W.n_active + id] = inv * uy;
}

// The layers F^T a of the DM fit's adjoint: y_l(i, j) = sum_m w_lm sum_p sum_q wy(p, i)
// wx(q, j) a_m(p, q), a thread per layer node.
template <class T>
__global__ void __launch_bounds__(OP_NT) k_fit_adj(__grid_constant__ const Desc<T> d, const T* act, T* out) {
    const int e = blockIdx.x * OP_NT + threadIdx.x;
    pdl_wait();
    pdl_trigger();
    if (e >= d.n_c) return;
    int l = 0;
    while (l + 1 < d.n_layers && e >= d.L[l + 1].off) ++l;
    const int n = d.L[l].n, i = (e - d.L[l].off) / n, j = (e - d.L[l].off) & (n - 1);
    T acc = T(0);
    for (int m = 0; m < d.n_dms; ++m) {
        const T w = d.fitw[m][l];
        if (w == T(0)) continue;
        const int rb = (m * MAXL + l) * MAXN, tb = (m * MAXL + l) * MAXNACT, na = d.Mi[m].n_act;
        const int p0 = d.dr_lo[rb + i], p1 = d.dr_hi[rb + i], q0 = d.dr_lo[rb + j], q1 = d.dr_hi[rb + j];
        const T* am = act + d.Mi[m].off;
        T sm = T(0);
        for (int p = p0; p < p1; ++p) {
            const T wy = d.di0[tb + p] == i ? T(1) - d.dfw[tb + p] : d.dfw[tb + p];
            T row = T(0);
            for (int q = q0; q < q1; ++q)
                row += (d.di0[tb + q] == j ? T(1) - d.dfw[tb + q] : d.dfw[tb + q]) * am[p * na + q];
            sm += wy * row;
        }
        acc += w * sm;
    }
    out[e] = acc;
}

}  // namespace fewha
