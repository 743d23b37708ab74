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

constexpr int TINV_NT = 256;     // threads of the inverse tile kernel
constexpr int TINV_SL = 7;       // coefficient slots per thread and round

// Quotient of t < 2048 by n <= 64 through the host's reciprocal ceil(65536 / n).
__device__ __forceinline__ int tdiv(int t, int magic) { return (t * magic) >> 16; }

// One 2 x 2 output block of a synthesis step: rows iy[t], columns ix[t] of the quadrants are
// the coefficients k - t of the block's pair (Sec. 3.1; columns first, then rows).
template <class T>
__device__ __forceinline__ void synth_block(const T* LL, int qsz, const int iy[3], const int ix[3], T out[2][2]) {
    T e[2][3], o[2][3];          // [x half][tap]: even and odd output row
#pragma unroll
    for (int xh = 0; xh < 2; ++xh) {
        const T* A = LL + xh * qsz;          // y-low rows
        const T* D = A + 2 * qsz;            // y-high rows
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            const T a0 = A[iy[0] + ix[t]], a1 = A[iy[1] + ix[t]], a2 = A[iy[2] + ix[t]];
            const T d0 = D[iy[0] + ix[t]], d1 = D[iy[1] + ix[t]], d2 = D[iy[2] + ix[t]];
            e[xh][t] = tap_h<T>(0) * a0 + tap_h<T>(2) * a1 + tap_h<T>(4) * a2 + tap_g<T>(0) * d0 +
                       tap_g<T>(2) * d1 + tap_g<T>(4) * d2;
            o[xh][t] = tap_h<T>(1) * a0 + tap_h<T>(3) * a1 + tap_h<T>(5) * a2 + tap_g<T>(1) * d0 +
                       tap_g<T>(3) * d1 + tap_g<T>(5) * d2;
        }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const T* l = r ? o[0] : e[0];
        const T* g = r ? o[1] : e[1];
        out[r][0] = tap_h<T>(0) * l[0] + tap_h<T>(2) * l[1] + tap_h<T>(4) * l[2] + tap_g<T>(0) * g[0] +
                    tap_g<T>(2) * g[1] + tap_g<T>(4) * g[2];
        out[r][1] = tap_h<T>(1) * l[0] + tap_h<T>(3) * l[1] + tap_h<T>(5) * l[2] + tap_g<T>(1) * g[0] +
                    tap_g<T>(3) * g[1] + tap_g<T>(5) * g[2];
    }
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
    const int t = threadIdx.x;
    const int pk = d.tunit[unit];
    const int l = pk & 255, ty = (pk >> 8) & 255, tx = pk >> 16;
    const LayerInfo L = d.L[l];
    const int n = L.n;
    {
        const int* src = reinterpret_cast<const int*>(d.tl + l);
        int* dst = reinterpret_cast<int*>(&tl);
        if (t < static_cast<int>(sizeof(TileLayer) / sizeof(int))) dst[t] = src[t];
    }
    __syncthreads();
    T* sc = sop + (tl.tail ? TAIL_N : 0);                // the levels' quadrants
    if (tl.tail) stage16(sop, d.tailop, TAIL_N, t, NT);
    if (t < 2) {
        int s = (t ? tx : ty) << tl.lts;
        ss[t][0] = s;
        for (int j = 1; j <= tl.J; ++j) {
            s = (s >> 1) - 2;
            if (tl.whole[j]) s = 0;
            ss[t][j] = s;
        }
    }
    __syncthreads();
    const bool has_old = PUPD == 1 || (PUPD == 2 && a.pupd != nullptr);
    const int lts = tl.lts;
    bool waited = false;
    T* tailb = sc + tl.tailb;
    for (int r0 = 0; r0 < tl.slot_cnt; r0 += NT * SL) {
        unsigned dst[SL];
        int pos[SL];
        T po[SL], zv[SL];
        bool own[SL];
#pragma unroll
        for (int s = 0; s < SL; ++s) {
            const int k = r0 + s * NT + t;
            pos[s] = -1;
            own[s] = false;
            dst[s] = 0;
            if (k < tl.slot_cnt) {
                // packed slot: level (0: the tail block), quadrant, row, column
                const unsigned c = d.tslot[tl.slot_off + k];
                const int j = c & 15, q = (c >> 4) & 3, row = (c >> 6) & 63, col = (c >> 12) & 63;
                if (j == 0) {
                    pos[s] = L.off + row * n + col;
                    own[s] = ty == 0 && tx == 0;
                    dst[s] = tl.tailb + row * 8 + col;
                } else {
                    const int h = n >> j;
                    const int y = (ss[0][j] + row) & (h - 1), x = (ss[1][j] + col) & (h - 1);
                    own[s] = ((y << j) >> lts) == ty && ((x << j) >> lts) == tx;
                    pos[s] = L.off + (y + (q >> 1) * h) * n + x + (q & 1) * h;
                    dst[s] = tl.base[j] + (q * tl.w[j] + row) * tl.stride[j] + col;
                }
                // p_old was last written two kernels back or earlier
                if (PUPD && has_old) po[s] = a.pupd[pos[s]];
            }
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
                    rz_new = warp_total(a.rz_parts, a.rz_cnt, static_cast<const DotAcc<T>*>(nullptr));
                    if (t == 0 && unit == 0) a.pcg.rztot[a.rz_slot] = rz_new;
                }
                if (PUPD && t == 0) {
                    double b = 0.0;
                    if (has_old) {
                        if (a.rz_cnt == 0) rz_new = a.pcg.rztot[a.iter];
                        const double rz_old = a.pcg.rztot[a.iter - 1];
                        b = rz_old != 0.0 ? rz_new / rz_old : 0.0;
                    }
                    sbeta = T(b);
                }
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
    if (tl.tail) cp_async_wait();
    __syncthreads();
    // ---- the last three levels of a full decomposition, one 64 x 64 map: four threads an
    // output, each 16 terms
    if (tl.tail) {
        const int o = t >> 2, part = t & 3;
        T acc[2] = {T(0), T(0)};
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int k = part * 8 + (i & 7) + 32 * (i >> 3);
            acc[i & 1] += sop[o * TAIL_LD + k] * tailb[k];
        }
        T y = acc[0] + acc[1];
        y += __shfl_down_sync(0xffffffffu, y, 2);
        y += __shfl_down_sync(0xffffffffu, y, 1);
        if (part == 0) sc[tl.base[tl.J] + (o >> 3) * tl.stride[tl.J] + (o & 7)] = y;
        __syncthreads();
    }
    // ---- the levels, coarse to fine; level j's quadrants give level j - 1's window
    for (int j = tl.J; j >= 1; --j) {
        const int np = tl.np[j - 1], mg = tl.magic[j - 1], w = tl.w[j], st = tl.stride[j], m = n >> j;
        const bool whole = tl.whole[j] != 0;
        const T* Q = sc + tl.base[j];
        const int qsz = w * st;
        const int s0y = ss[0][j - 1], s0x = ss[1][j - 1], w0 = tl.w[j - 1];
        const int ky0 = s0y >> 1, kx0 = s0x >> 1;
        for (int b = t; b < np * np; b += NT) {
            const int by = tdiv(b, mg), bx = b - by * np;
            int iy[3], ix[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int uy = whole ? ((ky0 + by - q) & (m - 1)) : by + 2 - q;
                const int ux = whole ? ((kx0 + bx - q) & (m - 1)) : bx + 2 - q;
                iy[q] = uy * st;
                ix[q] = ux;
            }
            T o[2][2];
            synth_block<T>(Q, qsz, iy, ix, o);
            const int y = 2 * (ky0 + by), x = 2 * (kx0 + bx);
            if (j == 1) {
                T* dst = a.out + L.off + y * n + x;
                dst[0] = o[0][0];
                dst[1] = o[0][1];
                dst[n] = o[1][0];
                dst[n + 1] = o[1][1];
            } else {
                T* dst = sc + tl.base[j - 1];
                const int st0 = tl.stride[j - 1], ry = y - s0y, rx = x - s0x;
#pragma unroll
                for (int e = 0; e < 2; ++e)
#pragma unroll
                    for (int f = 0; f < 2; ++f)
                        if (ry + e >= 0 && ry + e < w0 && rx + f >= 0 && rx + f < w0) dst[(ry + e) * st0 + rx + f] = o[e][f];
            }
        }
        if (j > 1) __syncthreads();
    }
}

template <class T, int PUPD>
__global__ void __launch_bounds__(TINV_NT) k_tinv(__grid_constant__ const Desc<T> d, __grid_constant__ const ClArgs<T> a) {
    tinv_body<T, PUPD>(d, a, blockIdx.x);
}

}  // namespace fewha
