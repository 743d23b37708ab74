// Batched kernels: thin wrappers that run the single-instance kernel bodies on work items
// of many instances in one launch.  A CTA first copies its instance's descriptor into
// shared memory (the bodies then read it from there, as the single-instance kernels read
// theirs from the constant bank), then runs the body on its unit.
#include <algorithm>
#include <utility>

#include "fewha_batch.h"

namespace fewha {

namespace {

// Copy the leading desc_bytes of the instance's descriptor into shared memory.
template <class T>
__device__ __forceinline__ void load_desc(Desc<T>& sd, const BInst<T>* __restrict__ I) {
    const int4* src = reinterpret_cast<const int4*>(&I->d);
    int4* dst = reinterpret_cast<int4*>(&sd);
    const int nb = (I->desc_bytes + 15) >> 4;
    for (int k = threadIdx.x; k < nb; k += blockDim.x) dst[k] = src[k];
    __syncthreads();
}

// The transform and sensor kernels copy the descriptor and read their tables before their
// body's wait: none of it is written inside the graph.
template <class T, int PUPD>
__global__ void __launch_bounds__(TINV_NT)
    kb_tinv(const BInst<T>* __restrict__ inst, const ClArgs<T>* __restrict__ args, const BItem* __restrict__ items) {
    __shared__ __align__(16) Desc<T> sd;
    const BItem it = items[blockIdx.x];
    const BInst<T>* I = inst + it.inst;
    load_desc<T>(sd, I);
    const ClArgs<T> a = args[it.inst];
    tinv_body<T, PUPD>(sd, a, it.unit);
}

template <class T, int DST>
__global__ void __launch_bounds__(cblk<T>(), sizeof(T) == 4 ? 2 : 1)
    kb_tfwd(const BInst<T>* __restrict__ inst, const ClArgs<T>* __restrict__ args, const BItem* __restrict__ items) {
    __shared__ __align__(16) Desc<T> sd;
    const BItem it = items[blockIdx.x];
    const BInst<T>* I = inst + it.inst;
    load_desc<T>(sd, I);
    const ClArgs<T> a = args[it.inst];
    const TfLayout lay = I->lay_tf;
    const PairBufs<T> pb = I->pb;
    tfwd_body<T, DST>(sd, a, lay, pb, it.unit);
}

template <class T, int DST>
__global__ void __launch_bounds__(cblk<T>(), sizeof(T) == 4 ? 2 : 1)
    kb_tcoarse(const BInst<T>* __restrict__ inst, const ClArgs<T>* __restrict__ args, const BItem* __restrict__ items) {
    __shared__ __align__(16) Desc<T> sd;
    const BItem it = items[blockIdx.x];
    const BInst<T>* I = inst + it.inst;
    load_desc<T>(sd, I);
    const ClArgs<T> a = args[it.inst];
    const TcLayout lay = I->lay_tc;
    tcoarse_body<T, DST>(sd, a, lay, it.unit);
}

template <class T, int SRC>
__global__ void __launch_bounds__(tsnt<T>(), sizeof(T) == 4 ? 2 : 1)
    kb_tsen(const BInst<T>* __restrict__ inst, const SensorArgs<T>* __restrict__ args, const BItem* __restrict__ items) {
    __shared__ __align__(16) Desc<T> sd;
    const BItem it = items[blockIdx.x];
    const BInst<T>* I = inst + it.inst;
    load_desc<T>(sd, I);
    const SensorArgs<T> a = args[it.inst];
    const TsLayout lay = I->lay_ts;
    const PairBufs<T> pb = I->pb;
    tsen_body<T, SRC>(sd, a, lay, pb, it.unit);
}

template <class T, int PHASE, int NTV>
__global__ void __launch_bounds__(NTV)
    kb_vec(const BInst<T>* __restrict__ inst, const VecArgs<T>* __restrict__ args,
           const BItem* __restrict__ items) {
    pdl_enter();
    const BItem it = items[blockIdx.x];
    const BInst<T>* I = inst + it.inst;
    const VecArgs<T> v = args[it.inst];
    vec_body<T, PHASE, NTV>(I->d.n_c, v, it.unit, I->nparts);
}

template <class T>
__global__ void __launch_bounds__(PBLK)
    kb_fit(const BInst<T>* __restrict__ inst, const FitArgs<T>* __restrict__ args,
           const BItem* __restrict__ items) {
    __shared__ __align__(16) Desc<T> sd;
    pdl_enter();
    const BItem it = items[blockIdx.x];
    const BInst<T>* I = inst + it.inst;
    load_desc<T>(sd, I);
    const FitArgs<T> f = args[it.inst];
    fit_body<T>(sd, f.phi, f.a_prev, f.out, f.apply_gain, it.unit, nullptr, f.cpist);
}

// The kernel of a step kind in one launch shape (variant v: 1 = the vector kernels with 512
// threads).
template <class T>
const void* kernel_of(int kind, int v) {
    const bool half = (v & 1) != 0;
    switch (kind) {
        case BK_INV: case BK_INV_MS: case BK_MSUM: return reinterpret_cast<const void*>(kb_tinv<T, 0>);
        case BK_INV_UPD: return reinterpret_cast<const void*>(kb_tinv<T, 1>);
        case BK_SEN_PHI: return reinterpret_cast<const void*>(kb_tsen<T, SSRC_PHI>);
        case BK_SEN_SLOPES: return reinterpret_cast<const void*>(kb_tsen<T, SSRC_SLOPES>);
        case BK_SEN_RESID: return reinterpret_cast<const void*>(kb_tsen<T, SSRC_RESID>);
        case BK_FWD_UPD: return reinterpret_cast<const void*>(kb_tfwd<T, LDST_UPDATE>);
        case BK_TC_UPD: return reinterpret_cast<const void*>(kb_tcoarse<T, LDST_UPDATE>);
        case BK_FWD_COEF: return reinterpret_cast<const void*>(kb_tfwd<T, LDST_COEF>);
        case BK_TC_COEF: return reinterpret_cast<const void*>(kb_tcoarse<T, LDST_COEF>);
        case BK_FWD_RINIT: return reinterpret_cast<const void*>(kb_tfwd<T, LDST_RESID_INIT>);
        case BK_FWD_AINIT: return reinterpret_cast<const void*>(kb_tfwd<T, LDST_APPLY_INIT>);
        case BK_TC_AINIT: return reinterpret_cast<const void*>(kb_tcoarse<T, LDST_APPLY_INIT>);
        case BK_TC_RINIT: return reinterpret_cast<const void*>(kb_tcoarse<T, LDST_RESID_INIT>);
        case BK_VEC_WARM:
            return half ? reinterpret_cast<const void*>(kb_vec<T, V_INIT_WARM, 2 * PBLK>)
                        : reinterpret_cast<const void*>(kb_vec<T, V_INIT_WARM, PBLK>);
        case BK_FIT: return reinterpret_cast<const void*>(kb_fit<T>);
        default: return nullptr;
    }
}

}  // namespace

template <class T>
cudaError_t batch_smem_limit(int kind, size_t* bytes) {
    if (bkind_list(kind) == BL_VEC) {
        *bytes = 0;
        return cudaSuccess;
    }
    int lim = 227 * 1024;
    for (int v = 0; v < 2; ++v) {
        const void* k = kernel_of<T>(kind, v);
        if (!k) return cudaErrorInvalidValue;
        cudaFuncAttributes fa;
        cudaError_t e = cudaFuncGetAttributes(&fa, k);
        if (e != cudaSuccess) return e;
        const int avail = 227 * 1024 - static_cast<int>(fa.sharedSizeBytes);
        if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, avail)) != cudaSuccess) return e;
        lim = std::min(lim, avail);
    }
    *bytes = static_cast<size_t>(lim);
    return cudaSuccess;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_b(bool pdl, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                     Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <class T>
cudaError_t batch_launch(const BLaunch& L, cudaStream_t st) {
    if (L.n_items <= 0) return cudaSuccess;
    const BInst<T>* I = static_cast<const BInst<T>*>(L.inst);
    const int n = L.n_items;
    const dim3 sn(tsnt<T>()), pg(n), nt(cblk<T>()), vt(L.vec_nt);
    const bool v2 = L.vec_nt != PBLK;
    const ClArgs<T>* ca = static_cast<const ClArgs<T>*>(L.args);
    const SensorArgs<T>* sa = static_cast<const SensorArgs<T>*>(L.args);
    const VecArgs<T>* va = static_cast<const VecArgs<T>*>(L.args);
    const FitArgs<T>* fa = static_cast<const FitArgs<T>*>(L.args);
    switch (L.kind) {
        case BK_INV: case BK_INV_MS: case BK_MSUM: return launch_b(L.pdl, kb_tinv<T, 0>, pg, dim3(TINV_NT), L.smem, st, I, ca, L.items);
        case BK_INV_UPD: return launch_b(L.pdl, kb_tinv<T, 1>, pg, dim3(TINV_NT), L.smem, st, I, ca, L.items);
        case BK_FWD_UPD: return launch_b(L.pdl, kb_tfwd<T, LDST_UPDATE>, pg, nt, L.smem, st, I, ca, L.items);
        case BK_TC_UPD: return launch_b(L.pdl, kb_tcoarse<T, LDST_UPDATE>, pg, nt, L.smem, st, I, ca, L.items);
        case BK_FWD_COEF: return launch_b(L.pdl, kb_tfwd<T, LDST_COEF>, pg, nt, L.smem, st, I, ca, L.items);
        case BK_TC_COEF: return launch_b(L.pdl, kb_tcoarse<T, LDST_COEF>, pg, nt, L.smem, st, I, ca, L.items);
        case BK_FWD_RINIT: return launch_b(L.pdl, kb_tfwd<T, LDST_RESID_INIT>, pg, nt, L.smem, st, I, ca, L.items);
        case BK_FWD_AINIT: return launch_b(L.pdl, kb_tfwd<T, LDST_APPLY_INIT>, pg, nt, L.smem, st, I, ca, L.items);
        case BK_TC_AINIT: return launch_b(L.pdl, kb_tcoarse<T, LDST_APPLY_INIT>, pg, nt, L.smem, st, I, ca, L.items);
        case BK_TC_RINIT: return launch_b(L.pdl, kb_tcoarse<T, LDST_RESID_INIT>, pg, nt, L.smem, st, I, ca, L.items);
        case BK_SEN_PHI: return launch_b(L.pdl, kb_tsen<T, SSRC_PHI>, pg, sn, L.smem, st, I, sa, L.items);
        case BK_SEN_SLOPES: return launch_b(L.pdl, kb_tsen<T, SSRC_SLOPES>, pg, sn, L.smem, st, I, sa, L.items);
        case BK_SEN_RESID: return launch_b(L.pdl, kb_tsen<T, SSRC_RESID>, pg, sn, L.smem, st, I, sa, L.items);
        case BK_VEC_WARM:
            return v2 ? launch_b(L.pdl, kb_vec<T, V_INIT_WARM, 2 * PBLK>, pg, vt, 0, st, I, va, L.items)
                      : launch_b(L.pdl, kb_vec<T, V_INIT_WARM, PBLK>, pg, vt, 0, st, I, va, L.items);
        case BK_FIT: return launch_b(L.pdl, kb_fit<T>, pg, dim3(PBLK), L.smem, st, I, fa, L.items);
        default: return cudaErrorInvalidValue;
    }
}

template cudaError_t batch_launch<float>(const BLaunch&, cudaStream_t);
template cudaError_t batch_launch<double>(const BLaunch&, cudaStream_t);
template cudaError_t batch_smem_limit<float>(int, size_t*);
template cudaError_t batch_smem_limit<double>(int, size_t*);

}  // namespace fewha
