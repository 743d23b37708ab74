// Tile kernels of the wavelet transforms: one CTA per square tile of a layer, no exchange
// between CTAs.  The periodic db3 synthesis of a tile of ts x ts nodes needs, level by
// level, only a window of w_(j+1) = w_j / 2 + 2 coefficients a side of every sub-band, so a
// CTA forms its tile of phi = W^T c from all levels by itself.
//
// Bound: latency.  A layer moves 4 n^2 values through L2 and does ~100 operations a value;
// what a frame waits for is the chain launch -> loads -> levels -> store.  A cluster of 8
// CTAs per layer (bands exchanged through distributed shared memory, the coarse levels on
// one leader CTA, three cluster barriers) took 8.0 us a launch on the 9 layers of the MAORY
// geometry and filled 72 of the 152 SMs; the tiles redo the halos (1.4 times the level-0
// arithmetic at ts = 32) but wait for nobody: 144 CTAs, 4.8 us, and the MAORY frame went
// from 192.6 to 176.4 us (FP64 842 to 827), a batch of 16 instances from 686 to 577 us.
#pragma once

#include "fewha_cluster.cuh"

namespace fewha {

constexpr int TINV_NT = 512;     // threads of the inverse tile kernel
constexpr int TINV_SL = 4;       // coefficient slots per thread and round

// ---------------------------------------------------------------------------
// Sums in a fixed order, in the arithmetic of DotAcc.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double acc_merge(double a, double b) { return a + b; }
__device__ __forceinline__ DFloat acc_merge(DFloat a, DFloat b) { return df_merge(a, b); }
__device__ __forceinline__ double acc_warp(double a) { return warp_sum(a); }
__device__ __forceinline__ DFloat acc_warp(DFloat a) { return warp_df_sum(a); }
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

// Total of `cnt` shares by one warp (lane 0), L2 loads first.
template <class T>
__device__ __forceinline__ typename AccOf<T>::type shares_total(const double* p, int cnt) {
    using A = typename AccOf<T>::type;
    A s = AccOf<T>::zero();
    for (int k0 = 0; k0 < cnt; k0 += 128) {
        A v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = k0 + 32 * k + (threadIdx.x & 31);
            v[k] = AccOf<T>::zero();
            if (i < cnt) {
                const double x = __ldcg(p + i);
                v[k] = *reinterpret_cast<const A*>(&x);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k0 + 32 * k < cnt) s = acc_merge(s, v[k]);
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

// Quotient of t < 2048 by n <= 64 through the host's reciprocal ceil(65536 / n).
__device__ __forceinline__ int tdiv(int t, int magic) { return (t * magic) >> 16; }

// One output pair of a synthesis step (Sec. 3.1) from the coefficients k, k - 1, k - 2 of the
// scaling (a) and wavelet (d) half.
template <class T>
__device__ __forceinline__ void synth_pair(T a0, T a1, T a2, T d0, T d1, T d2, T& e, T& o) {
    e = tap_h<T>(0) * a0 + tap_h<T>(2) * a1 + tap_h<T>(4) * a2 + tap_g<T>(0) * d0 + tap_g<T>(2) * d1 + tap_g<T>(4) * d2;
    o = tap_h<T>(1) * a0 + tap_h<T>(3) * a1 + tap_h<T>(5) * a2 + tap_g<T>(1) * d0 + tap_g<T>(3) * d1 + tap_g<T>(5) * d2;
}

// Quotient of two inner products as an operand of the vector updates, rounded to T: double
// totals, or double-float ones divided on the FP32 pipes (a double division is a chain of
// ~10 instructions of ~64 cycles).  Zero if the divisor is zero.
__device__ __forceinline__ double acc_ratio(double a, double b) { return b != 0.0 ? a / b : 0.0; }
__device__ __forceinline__ float acc_ratio(DFloat a, DFloat b) {
    if (b.s == 0.f) return 0.f;
    const float q = __fdiv_rn(a.s, b.s);
    const float rem = __fadd_rn(__fmaf_rn(-q, b.s, a.s), __fmaf_rn(-q, b.c, a.c));
    return __fadd_rn(q, __fdiv_rn(rem, b.s));
}
__device__ __forceinline__ void acc_of(double x, double& a) { a = x; }
__device__ __forceinline__ void acc_of(double x, DFloat& a) {
    a.s = static_cast<float>(x);
    a.c = static_cast<float>(x - static_cast<double>(a.s));
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
    __shared__ T smu[AUG_MAX];
    using A = typename AccOf<T>::type;
    const int t = threadIdx.x;
    int l = 0;
    while (unit >= d.tu0[l + 1]) ++l;
    const LayerInfo L = d.L[l];
    const int n = L.n;
    if (t < static_cast<int>(sizeof(TileLayer) / sizeof(int)))
        reinterpret_cast<int*>(&tl)[t] = reinterpret_cast<const int*>(d.tl + l)[t];
    T* sc = sop + (d.tailop ? TAIL_N : 0);                // the levels' quadrants
    if (d.tailop) stage16(sop, d.tailop, TAIL_N, t, NT);
    __syncthreads();
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
    A rz_old = AccOf<T>::zero();                          // rz of the iteration before: long written
    if (PUPD && has_old && t == 0) acc_of(a.pcg.rztot[a.iter - 1], rz_old);
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
                A rz_new = AccOf<T>::zero();
                if (a.rz_cnt > 0) {
                    rz_new = shares_total<T>(a.rz_parts, a.rz_cnt);
                    if (t == 0 && unit == 0) a.pcg.rztot[a.rz_slot] = warp_value(rz_new);
                } else if (has_old && t == 0) {
                    acc_of(a.pcg.rztot[a.iter], rz_new);
                }
                if (PUPD && t == 0) sbeta = has_old ? acc_ratio(rz_new, rz_old) : T(0);
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
                        if (pos[s] >= 0) cor[s] += mu * __ldg(Pj + pos[s]);
                }
            }
#pragma unroll
            for (int s = 0; s < SL; ++s)
                if (pos[s] >= 0) {
                    if (has_old) zv[s] = zv[s] + beta * po[s];
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
        for (int i = 0; i < 8; ++i) acc[i & 1] += sop[o * TAIL_LD + part * 8 + i] * tailb[part * 8 + i];
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
            } else {
                T* dst = sc + tl.base[j - 1] + row * tl.stride[j - 1];
                const int rx = x - s0x;
                if (rx >= 0 && rx < w0) dst[rx] = e;
                if (rx + 1 < w0) dst[rx + 1] = o;
            }
        }
        if (j > 1) __syncthreads();
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
                a += tap_h<T>(q) * v;
                dd += tap_g<T>(q) * v;
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
                a += tap_h<T>(q) * v;
                dd += tap_g<T>(q) * v;
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
                acc[i & 1] += tail[k * TAIL_LD + o] * buf[(k >> 3) * ld + (k & 7)];
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
// epilogue of the three detail bands; its LL block goes to a.ll.  k_tcoarse, a CTA per
// epilogue of the three detail bands; its LL block goes to a.ll.  k_tcoarse, a CTA per
// layer of several bands: the other levels and their epilogue.  A layer of one band (side
// at most 32) is finished by k_tfwd.
//
// Bound: latency again (launch, one block of staged reads, two passes).  Before, a kernel of
// (sensor, layer) pairs made the whole adjoint projection (4.9 us on the MAORY geometry) and
// a cluster per layer summed the pairs, transformed and finished on one leader CTA (11 us).
// Bands of 8 whole rows keep every global read a contiguous block and need a halo in one
// direction only; square tiles with a halo on four sides read the aperture vectors 1.9 times
// over and were slower (the frame 212 us).  Stamps inside a frame: 5.3 us for the bands, 4.8
// for the coarse levels.
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
        v.x += w * q.v.x; v.y += w * q.v.y; v.z += w * q.v.z; v.w += w * q.v.w;
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
    __device__ __forceinline__ void fma(double w, const Quad& q) { v.x += w * q.v.x; v.y += w * q.v.y; }
    __device__ __forceinline__ void split(double* e, double* o) const {
        *e = v.x;
        *o = v.y;
    }
};

// Operands of the epilogue at one coefficient.
template <class T>
struct EpiOp {
    T p, b, j;
};

// The epilogue at one coefficient: v = (W y)(pos), dl its D.
//   APPLY: q = v + alpha D p, written, p.q;  COEF: v written;
//   RESID_INIT: r0 = v - alpha D c0 (v is the residual's data term), z = J^-1 r, p = z, r.z;
//   APPLY_INIT: r0 = b - q, the same, and b_prev = b.
template <class T, int DST>
__device__ __forceinline__ void epi_load(const ClArgs<T>& a, int pos, EpiOp<T>& o) {
    if (DST != LDST_COEF) o.p = a.pin[pos];
    if (DST == LDST_APPLY_INIT) o.b = a.vb[pos];
    if (DST == LDST_APPLY_INIT || DST == LDST_RESID_INIT) o.j = a.vj[pos];
}
template <class T, int DST>
__device__ __forceinline__ void epi_apply(const ClArgs<T>& a, T alpha, T dl, int pos, T v, const EpiOp<T>& o,
                                          DotAcc<T>& dot) {
    if (DST == LDST_COEF) {
        a.out[pos] = v;
    } else if (DST == LDST_APPLY) {
        const T q = v + alpha * dl * o.p;
        a.out[pos] = q;
        dot.add(o.p, q);
    } else {
        const T rr = DST == LDST_RESID_INIT ? v - alpha * dl * o.p : o.b - (v + alpha * dl * o.p);
        const T z = o.j * rr;
        a.vr[pos] = rr;
        a.vz[pos] = z;
        a.vp[pos] = z;
        if (DST == LDST_APPLY_INIT) a.vbprev[pos] = o.b;
        dot.add(rr, z);
    }
}

// Where a layer's share of the epilogue's inner product goes, and, unless it is left to the
// next kernel, the total by the last of the instance's layers (fixed order).
template <class T, int DST>
__device__ __forceinline__ double* layer_slot(const ClArgs<T>& a, int l) {
    return DST == LDST_APPLY ? a.pcg.pqpart + a.iter * PQ_SLOTS + l : a.rzp + l;
}
template <class T, int DST>
__device__ __forceinline__ void layer_total(const ClArgs<T>& a, int n_layers) {
    if (DST == LDST_COEF || a.defer_total) return;
    __shared__ bool last;
    unsigned* count = a.pcg.count + (DST == LDST_APPLY ? 1 : 0);
    if (last_arrival(count, static_cast<unsigned>(n_layers), &last) && threadIdx.x < 32) {
        const typename AccOf<T>::type x = shares_total<T>(layer_slot<T, DST>(a, 0), n_layers);
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
    for (int g0 = 0; g0 < d.n_wfs; g0 += lay.gb) {
        const int nb = min(lay.gb, d.n_wfs - g0);
        if (g0 > 0) __syncthreads();
        for (int g = g0; g < g0 + nb; ++g) {
            const int4 e = src[g];
            for (int k = t * V; k < e.y; k += NT * V) cp_async16(st + e.z + k, pb.Y + e.x + k);
        }
        cp_async_wait();
        __syncthreads();
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
                            if (w[g * (kt + 1) + q] != T(0)) x += w[g * (kt + 1) + q] * row[q * b.y];
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
    // ---- the finest analysis level: rows, then columns ---------------------------------------
    DotAcc<T> dot;
    for (int b = t; b < nblk; b += NT) {                  // one block per thread, but for wide layers in double
        const int msk = bands > 1 ? 15 : n - 1;           // a band holds its halo
        const int ky = 2 * (b >> lh), kx = b & (h - 1);
        T ra[6], rd[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            const T* re = ye + ((ky + r) & msk) * ysd;
            const T* ro = yo + ((ky + r) & msk) * ysd;
            T av = T(0), dv = T(0);
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const T x = (q & 1 ? ro : re)[(kx + (q >> 1)) & (h - 1)];
                av += tap_h<T>(q) * x;
                dv += tap_g<T>(q) * x;
            }
            ra[r] = av;
            rd[r] = dv;
        }
        T ll = T(0), v[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            ll += tap_h<T>(r) * ra[r];
            v[0] += tap_h<T>(r) * rd[r];
            v[1] += tap_g<T>(r) * ra[r];
            v[2] += tap_g<T>(r) * rd[r];
        }
        const int rk = (Y0 >> 1) + (b >> lh);
        if (bands > 1)
            a.ll[(L.off >> 2) + rk * h + kx] = ll;
        else
            lbuf[rk * lsd + kx] = ll;
#pragma unroll
        for (int e = 0; e < 3; ++e) epi_apply<T, DST>(a, salpha, sD[1], pos[e], v[e], op[e], dot);
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
        for (int k = t; k < h * h; k += NT) {
            const int i = k >> lh, j = k & (h - 1), p = L.off + i * n + j;
            EpiOp<T> o;
            epi_load<T, DST>(a, p, o);
            epi_apply<T, DST>(a, salpha, sD[level_of(i, j, L)], p, lbuf[i * lsd + j], o, dot);
        }
    }
    if (DST != LDST_COEF) {
        cta_share<T>(dot, red, nullptr, bands > 1 ? a.tshare + unit : layer_slot<T, DST>(a, l));
        if (bands == 1) layer_total<T, DST>(a, d.n_layers);
    }
}

template <class T, int DST>
__global__ void __launch_bounds__(cblk<T>(), sizeof(T) == 4 ? 2 : 1)
    k_tfwd(__grid_constant__ const Desc<T> d, __grid_constant__ const ClArgs<T> a,
           __grid_constant__ const TfLayout lay, __grid_constant__ const PairBufs<T> pb) {
    tfwd_body<T, DST>(d, a, lay, pb, blockIdx.x);
}

// The levels below the finest of layer l (of several bands) and their epilogue.  The LL
// block (a.ll) comes from k_tfwd; the epilogue's operands are staged before the wait.
struct TcLayout {
    int lbuf, tmp, tail, st, total;  // T units after RED_DBL doubles; st: staged operands
};

template <class T, int DST>
__device__ __forceinline__ void tcoarse_body(const Desc<T>& d, const ClArgs<T>& a, const TcLayout& lay, const int l) {
    constexpr int NT = cblk<T>(), V = vec16<T>();
    constexpr bool QP = DST != LDST_COEF, QB = DST == LDST_APPLY_INIT;
    constexpr bool QJ = DST == LDST_APPLY_INIT || DST == LDST_RESID_INIT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* red = reinterpret_cast<double*>(smem_raw);
    T* sm = reinterpret_cast<T*>(red + CWMAX);
    const int t = threadIdx.x;
    const LayerInfo L = d.L[l];
    const int n = L.n, h = n >> 1, lh = L.log2n - 1, lsd = h + 1;
    T* lbuf = sm + lay.lbuf;
    T* sp = sm + lay.st;
    T* sb = sp + (MAXN / 2) * (MAXN / 2);
    T* sj = sb + (QB ? (MAXN / 2) * (MAXN / 2) : 0);
    __shared__ T sD[MAXLEV + 1];
    __shared__ T salpha;
    __shared__ double tiles;             // the bands' share of the inner product
    if (t <= MAXLEV) sD[t] = d.Dlev[l][t];
    if (t == 0) salpha = d.alpha;
    const bool tail_on = lay.tail > 0 && (d.bkt[l] >> 4);
    const int unit0 = d.bu0[l], units = d.bu0[l + 1] - d.bu0[l];
    if (tail_on) stage16(sm + lay.tail, d.tailop, TAIL_N, t, NT);
    if (QP) {
        // a caller's vector (the apply's input) may start off a 16-byte boundary
        const bool wide = ((reinterpret_cast<size_t>(a.pin) | reinterpret_cast<size_t>(QB ? a.vb : a.pin)) & 15) == 0;
        const int lc = wide ? lh - (V == 4 ? 2 : 1) : lh;    // log2 of the copies per row
        for (int k = t; k < (h << lc); k += NT) {
            const int i = k >> lc, c = (k & ((1 << lc) - 1)) * (wide ? V : 1), pos = L.off + i * n + c;
            if (wide) {
                cp_async16(sp + i * h + c, a.pin + pos);
                if (QB) cp_async16(sb + i * h + c, a.vb + pos);
                if (QJ) cp_async16(sj + i * h + c, a.vj + pos);
            } else {
                cp_async(sp + i * h + c, a.pin + pos);
                if (QB) cp_async(sb + i * h + c, a.vb + pos);
                if (QJ) cp_async(sj + i * h + c, a.vj + pos);
            }
        }
    }
    pdl_wait();
    pdl_trigger();
    const T* src = a.ll + (L.off >> 2);
    for (int k = t * V; k < h * h; k += NT * V) {
        const Quad<T> v = *reinterpret_cast<const Quad<T>*>(src + k);
        T* dst = lbuf + (k >> lh) * lsd + (k & (h - 1));
#pragma unroll
        for (int e = 0; e < V; ++e) dst[e] = reinterpret_cast<const T*>(&v)[e];
    }
    if (QP && t >= NT - 32) {
        const typename AccOf<T>::type x = shares_total<T>(a.tshare + unit0, units);
        if (t == NT - 32) *reinterpret_cast<typename AccOf<T>::type*>(&tiles) = x;
    }
    cp_async_wait();
    __syncthreads();
    if (L.levels >= 2) analyse<T>(lbuf, sm + lay.tmp, tail_on ? sm + lay.tail : nullptr, n, 1, L.levels, lsd);
    if (a.zero_piston && L.full && t == 0) lbuf[0] = T(0);   // no piston in the data term (see tfwd_body)
    __syncthreads();
    DotAcc<T> dot;
    for (int k = t; k < h * h; k += NT) {
        const int i = k >> lh, j = k & (h - 1);
        EpiOp<T> o;
        if (QP) o.p = sp[k];
        if (QB) o.b = sb[k];
        if (QJ) o.j = sj[k];
        epi_apply<T, DST>(a, salpha, sD[level_of(i, j, L)], L.off + i * n + j, lbuf[i * lsd + j], o, dot);
    }
    if (QP) {
        cta_share<T>(dot, red, &tiles, layer_slot<T, DST>(a, l));
        layer_total<T, DST>(a, d.n_layers);
    }
}

template <class T, int DST>
__global__ void __launch_bounds__(cblk<T>(), sizeof(T) == 4 ? 2 : 1)
    k_tcoarse(__grid_constant__ const Desc<T> d, __grid_constant__ const ClArgs<T> a, __grid_constant__ const TcLayout lay) {
    tcoarse_body<T, DST>(d, a, lay, d.tcl[blockIdx.x]);
}

// ---------------------------------------------------------------------------
// Sensor kernel (cluster of SCL CTAs per sensor, a band of subaperture rows per CTA): P_g
// (Sec. 2), Gamma_g, C_hat_g^-1 (Eq. 2, Sec. 3.2), Gamma_g^T and the column half of P_g^T.
// SRC_PHI: slopes of the projected layers (the M-apply); SRC_RESID: measured minus modelled
// slopes (the initial residual); SRC_SLOPES: measured slopes (the right-hand side).  The
// layers are read by direct bilinear gathers; the result goes out per layer as the aperture
// rows' values on the layer's columns (pb.Y, slot g * n_layers + l, rows of box[3]
// columns), whose row half the band kernel applies.
//
// Every CTA also forms the slopes of the row below its band, so that nothing but the
// tip/tilt and coarse-block sums crosses the cluster: one barrier.  The sums are formed per
// subaperture row and then over the rows, in an order that does not depend on SCL.
//
// Bound: latency (tables, one gather, one cluster barrier).  With the slopes of the row below
// formed here too, two cluster barriers and a distributed-shared-memory read are gone; with
// the projection and the column half of its adjoint in this kernel, so are the two kernels of
// (sensor, layer) pairs.  Clusters of 16 CTAs halve the bands where the device holds all of
// an instance's clusters at once (14 of them: the MAORY frame 156 us, with clusters of 8
// 173); a batch fills the device with clusters of 8 (391 us a batch of 16 instances, with
// clusters of 16 535).  Staging the layers' rows in shared memory first took 3 to 5 us more
// than gathering from L2.  From the cluster kernels: frame of the 8 m system 91.3 -> 65.8 us,
// paper's geometry 111 -> 77.7, MAORY 173.5 -> 156.4, in double 817 -> 664, closed loop
// 200 -> 163, a batch of 16 uneven instances 566 -> 391.
// ---------------------------------------------------------------------------
constexpr int TS_LG = 5;         // layers with their loads in flight together
constexpr int TS_NV = 2 * FEWHA_MAX_COARSE;      // sums per subaperture row, at most

// Threads: in single precision 7 node rows of 81 nodes in one pass.
template <class T>
__host__ __device__ constexpr int tsnt() {
    return sizeof(T) == 4 ? 576 : 288;
}
struct TsLayout {       // shared-memory offsets in T units, for clusters of 16 and 8
    int V, SX, SY, msk, xi, xf, yi, yf, cw, ci, total;
};

template <class T, int SRC, int SCL>
__device__ __forceinline__ void tsen_body(const Desc<T>& d, const SensorArgs<T>& a, const TsLayout& lay,
                                          const PairBufs<T>& pb, const int g) {
    constexpr int NT = tsnt<T>();
    constexpr bool FROM_PHI = SRC == SSRC_PHI || SRC == SSRC_RESID;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int r = static_cast<int>(cluster.block_rank());
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31, nwarp = NT >> 5;
    // peers' shared memory is written before the first full cluster barrier (the pushes
    // below): arrive now, wait before the first push, so that every CTA has started
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");
    // the sensor's constants in shared memory: the kernel-parameter bank is cold, and its
    // first reads would stand behind the dependency wait (a copy in device memory is read:
    // indexed reads of the parameters are slow)
    __shared__ WfsInfo sW;
    __shared__ int sco[MAXL + 1];                        // first column of each layer
    __shared__ int2 ybox[MAXL];                          // each layer: box columns, offset in Y
    __shared__ T rsum[MAXNF][TS_NV];                     // every subaperture row's sums (pushed)
    __shared__ T tot[4];
    __shared__ T cw[2 * MAXCOARSE];                      // weighted coarse slopes / nb
    const int nl = d.n_layers, ks = d.tks;
    const int N = d.G[g].N, NP = N + 1, NPs = d.tnp;
    const int sr = (N + SCL - 1) / SCL;
    const int s0 = min(r * sr, N), s1 = min((r + 1) * sr, N), rows = s1 - s0;
    const int h0 = s0 > 0 && rows > 0 ? 1 : 0;           // the row below the band, if any
    const int q0 = s0 - h0, nrow = rows + h0;            // slope rows [q0, s1), node rows [q0, s1]
    T* Vb = sm + lay.V;         // (nrow + 1) x NP: node values, later the adjoint's
    T* SX = sm + lay.SX;        // nrow x N
    T* SY = sm + lay.SY;
    int* msk = reinterpret_cast<int*>(sm + lay.msk);
    int* xi = reinterpret_cast<int*>(sm + lay.xi);       // [layer][node column]: place of its layer column
    T* xf = sm + lay.xf;
    int2* yi = reinterpret_cast<int2*>(sm + lay.yi);     // [layer][node row]: offset of its layer row, row pitch
    T* yf = sm + lay.yf;
    T* cwt = sm + lay.cw;                                // column weights of P^T: [column][ks]
    int2* cin = reinterpret_cast<int2*>(sm + lay.ci);    // first aperture column, count
    // ---- set-up tables, copied before the dependency wait; those of the column half of P^T
    // in a group of their own, waited for where they are used ------------------------------
    for (int k = t; k < static_cast<int>(sizeof(WfsInfo) / sizeof(int)); k += NT)
        reinterpret_cast<int*>(&sW)[k] = reinterpret_cast<const int*>(d.gdev + g)[k];
    {
        const int* src = d.sidx + d.G[g].mask_off + q0 * N;
        for (int k = t; k < nrow * N; k += NT) cp_async(msk + k, src + k);
    }
    if (FROM_PHI) {
        const int nx = nl * NPs;
        stage16(xi, d.txi + g * nx, nx, t, NT);
        stage16(xf, d.txf + g * nx, nx, t, NT);
        for (int k = t; k < nl * 16; k += NT) {
            const int l = k >> 4;
            for (int i = k & 15; i <= nrow; i += 16) {
                yi[l * (sr + 2) + i] = reinterpret_cast<const int2*>(d.tyi)[g * nx + l * NPs + q0 + i];
                yf[l * (sr + 2) + i] = d.tyf[g * nx + l * NPs + q0 + i];
            }
        }
    }
    if (t < 32) {
        for (int k = t; k <= nl; k += 32) sco[k] = d.tsco[g * (MAXL + 1) + k];
        for (int k = t; k < nl; k += 32) ybox[k] = reinterpret_cast<const int2*>(d.tybox)[g * MAXL + k];
    }
    cp_async_commit();
    stage16(cwt, d.tcw + static_cast<size_t>(g) * d.tcols * ks, d.tcols * ks, t, NT);
    stage16(reinterpret_cast<int*>(cin), d.tcin + g * d.tcols * 2, 2 * d.tcols, t, NT);
    cp_async_commit();
    cp_async_wait_group<1>();
    __syncthreads();
    const WfsInfo& W = sW;
    const T inv = T(W.sig2inv);
    const T nbinv = T(1) / T(W.nb);
    pdl_wait();
    pdl_trigger();
    bool bad = false;                          // a non-finite measured slope (SLOPES, RESID)
    if (FROM_PHI && rows > 0) {
        // ---- V = P_g phi on node rows [q0, s1]: a thread per node, the layers in order ----
        for (int k = t; k < (nrow + 1) * NP; k += NT) {
            const int ia = k / NP, b = k - ia * NP;
            T v = T(0);
            for (int l0 = 0; l0 < nl; l0 += TS_LG) {
                T q[TS_LG][4];
#pragma unroll
                for (int e = 0; e < TS_LG; ++e)
                    if (l0 + e < nl) {
                        const int2 y = yi[(l0 + e) * (sr + 2) + ia];
                        const T* p = a.phi + xi[(l0 + e) * NPs + b] + y.x;
                        q[e][0] = p[0];
                        q[e][1] = p[1];
                        q[e][2] = p[y.y];
                        q[e][3] = p[y.y + 1];
                    }
#pragma unroll
                for (int e = 0; e < TS_LG; ++e)
                    if (l0 + e < nl) {
                        const T fx = xf[(l0 + e) * NPs + b], fy = yf[(l0 + e) * (sr + 2) + ia];
                        const T h0 = (T(1) - fx) * q[e][0] + fx * q[e][1], h1 = (T(1) - fx) * q[e][2] + fx * q[e][3];
                        v += (T(1) - fy) * h0 + fy * h1;
                    }
            }
            Vb[k] = v;
        }
        __syncthreads();
    }
    // ---- the slopes of rows [q0, s1) and each band row's sums: a warp per row ---------------
    const bool need_tt = W.lgs;
    const bool need_coarse = FROM_PHI && W.nb > 1;
    asm volatile("barrier.cluster.wait.aligned;\n" ::: "memory");
    for (int ii = warp; ii < nrow; ii += nwarp) {
        T sum[4] = {T(0), T(0), T(0), T(0)};
        for (int j = lane; j < N; j += 32) {
            const int k = ii * N + j;
            T sx = T(0), sy = T(0);
            const int id = msk[k];
            if (id >= 0) {
                if (FROM_PHI) {
                    // Gamma_g on the modelled nodes
                    const T v00 = Vb[ii * NP + j], v01 = Vb[ii * NP + j + 1];
                    const T v10 = Vb[(ii + 1) * NP + j], v11 = Vb[(ii + 1) * NP + j + 1];
                    sx = T(0.5) * ((v01 - v00) + (v11 - v10));
                    sy = T(0.5) * ((v10 - v00) + (v11 - v01));
                }
                if ((SRC == SSRC_RESID && W.nb == 1) || SRC == SSRC_SLOPES) {
                    // measured slopes; the residual of an ordinary sensor is measured minus
                    // modelled (a coarse sensor's measurement enters after its block sums)
                    const T mx = a.in[W.soff + id], my = a.in[W.soff + W.n_active + id];
                    bad |= !(isfinite(mx) && isfinite(my));
                    sx = SRC == SSRC_RESID ? mx - sx : mx;
                    sy = SRC == SSRC_RESID ? my - sy : my;
                    if (SRC == SSRC_SLOPES && W.nb > 1) {    // (1/nb) sigma^-2 s_K on each active fine one
                        sx *= nbinv * inv;
                        sy *= nbinv * inv;
                    }
                }
                if (W.nb == 1 && !W.lgs) {                   // NGS: C^-1 = sigma^-2 I
                    sx *= inv;
                    sy *= inv;
                }
                if (need_tt) {
                    sum[0] += sx;
                    sum[1] += sy;
                    if (W.el) {
                        // spot elongation (Eq. 3): the sums of gamma beta (beta . s) as well
                        T b1, b2, gam;
                        elong(W, q0 + ii, j, b1, b2, gam);
                        const T bs = b1 * sx + b2 * sy;
                        sum[2] += gam * b1 * bs;
                        sum[3] += gam * b2 * bs;
                    }
                }
            }
            SX[k] = sx;
            SY[k] = sy;
        }
        // a row's sums go to every rank; the row below the band is its owner's
        if (need_tt && ii >= h0) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (e < 2 || W.el) {
                    sum[e] = warp_sum_t(sum[e]);
                    sum[e] = __shfl_sync(0xffffffffu, sum[e], 0);
                    if (lane < SCL) cluster.map_shared_rank(&rsum[0][0], static_cast<unsigned>(lane))[(q0 + ii) * TS_NV + e] = sum[e];
                }
        }
        if (need_coarse && ii >= h0) {
            // per block column: the row's fine-slope sums
            __syncwarp();
            for (int J = 0; J < W.n_sub; ++J) {
                T sx = T(0), sy = T(0);
                for (int j = J * W.nb + lane; j < (J + 1) * W.nb; j += 32) {
                    sx += SX[ii * N + j];
                    sy += SY[ii * N + j];
                }
                sx = __shfl_sync(0xffffffffu, warp_sum_t(sx), 0);
                sy = __shfl_sync(0xffffffffu, warp_sum_t(sy), 0);
                if (lane < SCL) {
                    T* dst = cluster.map_shared_rank(&rsum[0][0], static_cast<unsigned>(lane)) + (q0 + ii) * TS_NV + 2 * J;
                    dst[0] = sx;
                    dst[1] = sy;
                }
            }
        }
    }
    if (bad && a.status) atomicOr(a.status, 1u);
    if (need_tt || need_coarse)
        cluster.sync();                        // every row's sums are here; no remote access after this
    else
        __syncthreads();
    if (need_tt) {
        // the sums over the rows (fixed order), then the weighting
        if (warp < (W.el ? 4 : 2)) {
            T x = T(0);
            for (int i = lane; i < N; i += 32) x += rsum[i][warp];
            x = warp_sum_t(x);
            if (lane == 0) tot[warp] = x;
        }
        __syncthreads();
        const T mx = tot[0] / T(W.n_active), my = tot[1] / T(W.n_active);
        if (!W.el) {
            // C_hat^-1 = (I - T) sigma^-2 (I - T) = sigma^-2 (I - T) for an LGS
            for (int k = t; k < nrow * N; k += NT) {
                if (msk[k] >= 0) {
                    SX[k] = inv * (SX[k] - mx);
                    SY[k] = inv * (SY[k] - my);
                }
            }
        } else {
            // elongated: C_hat^-1 s = sigma^-2 (u - gamma beta (beta . u) + g), u = s
            // minus its means m, g = (e - K m) / |M| the mean of gamma beta (beta . u)
            const T ex = tot[2], ey = tot[3];
            const T g1 = (ex - (el_K(W, 0, T()) * mx + el_K(W, 1, T()) * my)) / T(W.n_active);
            const T g2 = (ey - (el_K(W, 1, T()) * mx + el_K(W, 2, T()) * my)) / T(W.n_active);
            for (int ii = warp; ii < nrow; ii += nwarp)
            for (int j = lane; j < N; j += 32) {
                const int k = ii * N + j;
                if (msk[k] >= 0) {
                    T b1, b2, gam;
                    elong(W, q0 + ii, j, b1, b2, gam);
                    const T ux = SX[k] - mx, uy = SY[k] - my;
                    const T bu = b1 * ux + b2 * uy;
                    SX[k] = inv * ((ux - gam * b1 * bu) + g1);
                    SY[k] = inv * ((uy - gam * b2 * bu) + g2);
                }
            }
        }
        __syncthreads();
    }
    if (need_coarse) {
        // coarse slope = sum / nb; Gamma_coarse^T spreads sigma^-2 slope / nb.  The residual
        // form subtracts it from the block's measured slope.
        const int ns = W.n_sub, nb = W.nb;
        for (int e = warp; e < 2 * ns * ns; e += nwarp) {
            const int blk = e >> 1, xy = e & 1, I = blk / ns, J = blk - I * ns;
            T x = T(0);
            for (int i = I * nb + lane; i < (I + 1) * nb; i += 32) x += rsum[i][2 * J + xy];
            x = warp_sum_t(x);
            if (lane == 0) {
                x *= nbinv;
                if (SRC == SSRC_RESID) {
                    const int K = d.cidx[W.cmask_off + blk];
                    T m = T(0);
                    if (K >= 0) {
                        m = a.in[W.soff + xy * W.n_active + K];
                        if (!isfinite(m) && a.status) atomicOr(a.status, 1u);
                    }
                    x = m - x;
                }
                cw[e] = x * inv * nbinv;
            }
        }
        __syncthreads();
        for (int ii = warp; ii < nrow; ii += nwarp)
        for (int j = lane; j < N; j += 32) {
            const int k = ii * N + j;
            T sx = T(0), sy = T(0);
            if (msk[k] >= 0) {
                const int blk = ((q0 + ii) / nb) * ns + j / nb;
                sx = cw[2 * blk];
                sy = cw[2 * blk + 1];
            }
            SX[k] = sx;
            SY[k] = sy;
        }
        __syncthreads();
    }
    cp_async_wait();
    if (rows > 0) {
        // ---- Gamma_g^T on node rows [s0, s1) (and row N on the last band) ------------------
        const int nout = (s1 == N) ? rows + 1 : rows;
        for (int ia = warp; ia < nout; ia += nwarp)
        for (int b = lane; b < NP; b += 32) {
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
            Vb[ia * NP + b] =
                T(0.5) * ((x_ab1 - x_ab) + (x_a1b1 - x_a1b)) + T(0.5) * ((y_a1b - y_ab) + (y_a1b1 - y_ab1));
        }
        __syncthreads();
        // ---- the column half of P_g^T: a thread owns a layer column and takes every row -----
        for (int k = t; k < sco[nl]; k += NT) {
            int l = 0;
            while (k >= sco[l + 1]) ++l;
            const int2 yb = ybox[l], c = cin[k];
            const int j = k - sco[l], cols = yb.x;
            if (j >= cols) continue;
            T* dst = pb.Y + yb.y + s0 * cols + j;
            const T* src = Vb + c.x;
            const T* wk = cwt + k * ks;
            if (c.y <= 3) {
                T w[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) w[q] = q < c.y ? wk[q] : T(0);
#pragma unroll 3
                for (int ia = 0; ia < nout; ++ia) {
                    T x = T(0);
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        if (q < c.y) x += w[q] * src[ia * NP + q];
                    dst[ia * cols] = x;
                }
            } else {
                T w[KMAX];
#pragma unroll
                for (int q = 0; q < KMAX; ++q) w[q] = q < c.y ? wk[q] : T(0);
                for (int ia = 0; ia < nout; ++ia) {
                    T x = T(0);
#pragma unroll
                    for (int q = 0; q < KMAX; ++q)
                        if (q < c.y) x += w[q] * src[ia * NP + q];
                    dst[ia * cols] = x;
                }
            }
        }
    }
}

template <class T, int SRC, int SCL>
__global__ void __cluster_dims__(SCL, 1, 1) __launch_bounds__(tsnt<T>(), sizeof(T) == 4 ? 2 : 1)
    k_tsen(__grid_constant__ const Desc<T> d, __grid_constant__ const SensorArgs<T> a,
           __grid_constant__ const TsLayout lay, __grid_constant__ const PairBufs<T> pb) {
    tsen_body<T, SRC, SCL>(d, a, lay, pb, blockIdx.y);
}

}  // namespace fewha
