// Host-side launchers of the device kernels, one table per (D, K, rain,
// storage type).  Instantiated in dg_inst_*.cu so that the configurations
// compile in parallel.
#pragma once

#include <type_traits>

#include "dg_column.cuh"
#include "dg_device.cuh"
#include "dg_once.h"
#include "dg_stage64.cuh"

namespace dgm {

template <typename Real>
struct Launchers {
    int nf, np, nfp1, nd, ntr, epb, nt;
    int trace_face;   // values of one face of one element in the trace buffer (TraceLayout)
    // diff: with the artificial diffusion of Eq. (3.7) (face pass only)
    cudaError_t (*prepare)(const KArgs<Real> &, bool diff, cudaStream_t);
    // pf: the stage kernel takes its face fluxes from the face pass
    cudaError_t (*stage)(const KArgs<Real> &, int mode, bool pf, bool diff, cudaStream_t);
    cudaError_t (*face)(const KArgs<Real> &, bool diff, cudaStream_t);
    cudaError_t (*alpha_vertex)(const KArgs<Real> &, cudaStream_t);
    cudaError_t (*split)(const KArgs<Real> &, double *, double *, double *, double *, cudaStream_t);
    cudaError_t (*init_bubble)(const KArgs<Real> &, const BubbleArgs &, cudaStream_t);
    cudaError_t (*reduce)(const KArgs<Real> &, double *partials, int nblocks, cudaStream_t);
    // column march (float32 forms only; null for float64): a stage or the
    // right-hand side with the face fluxes evaluated on chip
    cudaError_t (*column)(const KArgs<Real> &, int mode, cudaStream_t);
};

constexpr int kGridStrideBlocks = 152 * 8;

inline int grid_for(size_t n, int threads) {
    size_t b = (n + threads - 1) / threads;
    if (b > (size_t)kGridStrideBlocks) b = kGridStrideBlocks;
    return (int)(b > 0 ? b : 1);
}

// Launch, with programmatic dependent launch (dependents_go / dependents_wait,
// dg_device.cuh) where it pays: the launch and the kernel's set-up overlap the
// end of the kernel before it.  Blocks that start early sit where there is
// room, not where they would be spread, so a grid of about one to six blocks
// per SM ends up unbalanced (64x32 order 3 float64: 116 -> 178 us per step, the
// same for a small grid behind a larger one).  It pays for a full chip of
// threads and more (128x64 order 4 FP32-bulk: 99 -> 87 us per step) and in a
// chain of kernels of at most one block per SM (`chain`; 20x10 order 3: 58 ->
// 54 us).
constexpr int kSMs = 152;

template <class K, class... P>
inline cudaError_t launch(K kern, int grid, int block, size_t smem, cudaStream_t st, bool chain,
                          const P &...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = ((chain && grid <= kSMs) || (long long)grid * block >= kSMs * 768) ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Opt-in of a kernel to its dynamic shared memory on the current device (the
// attribute is the device's own: several tiles need more than the default
// 48 KB, and a context may be on any device)
template <class K>
inline cudaError_t allow_smem(OncePerDevice &once, K kern, size_t smem) {
    int dev = 0;
    const cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    return (cudaError_t)once(dev, [&] {
        return (int)cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
}

template <class S, typename Real>
struct Impl {
    static constexpr bool F64 = std::is_same<Real, double>::value;

    // shared memory of the prepare and stage tiles
    template <bool DIFF>
    static constexpr size_t prep_smem() {
        if constexpr (F64) return prepare64_smem_bytes<S, DIFF>();
        else return sizeof(Real) * (size_t)(S::NTR + (DIFF ? 2 : 0)) * S::EPB * S::NP;
    }
    template <bool PF, bool DIFF>
    static constexpr size_t stage_smem() {
        if constexpr (F64) return stage64_smem_bytes<S, DIFF>();
        else return stage_smem_bytes<S, Real, PF, DIFF>();
    }

    static int blocks(const KArgs<Real> &A) { return (A.M.ne + S::EPB - 1) / S::EPB; }

    template <bool DIFF>
    static constexpr auto prepare_kernel() {
        if constexpr (F64) return &k_prepare64<S, DIFF>;
        else return &k_prepare<S, Real, DIFF>;
    }

    template <bool DIFF>
    static cudaError_t launch_prepare(const KArgs<Real> &A, cudaStream_t st) {
        constexpr size_t smem = prep_smem<DIFF>();
        const auto kern = prepare_kernel<DIFF>();
        static OncePerDevice once;
        const cudaError_t err = allow_smem(once, kern, smem);
        if (err != cudaSuccess) return err;
        return launch(kern, A.ntiles > 0 ? A.ntiles : blocks(A), S::NT, smem, st, true, A);
    }

    static cudaError_t prepare(const KArgs<Real> &A, bool diff, cudaStream_t st) {
        return diff ? launch_prepare<true>(A, st) : launch_prepare<false>(A, st);
    }

    // the stage kernel of one schedule: float32 face-pass tiles of 64, 128
    // or 256 threads take the variant with the 48-register budget
    template <int MODE, bool PF, bool DIFF>
    static constexpr auto stage_kernel() {
        if constexpr (F64)
            return &k_stage64<S, MODE, PF, DIFF>;
        else if constexpr (PF && !DIFF && (S::NT == 64 || S::NT == 128 || S::NT == 256))
            return &k_stage_f32pf<S, MODE>;
        else
            return &k_stage<S, Real, MODE, PF, DIFF>;
    }

    template <int MODE, bool PF, bool DIFF>
    static cudaError_t launch_stage(const KArgs<Real> &A, cudaStream_t st) {
        constexpr size_t smem = stage_smem<PF, DIFF>();
        const auto kern = stage_kernel<MODE, PF, DIFF>();
        static OncePerDevice once;
        const cudaError_t err = allow_smem(once, kern, smem);
        if (err != cudaSuccess) return err;
        return launch(kern, A.ntiles > 0 ? A.ntiles : blocks(A), S::NT, smem, st, !PF, A);
    }

    static cudaError_t stage(const KArgs<Real> &A, int mode, bool pf, bool diff, cudaStream_t st) {
        if (diff) {
            if (!pf) return cudaErrorInvalidValue;
            return mode == MODE_RHS ? launch_stage<MODE_RHS, true, true>(A, st)
                                    : launch_stage<MODE_STAGE, true, true>(A, st);
        }
        if (mode == MODE_RHS)
            return pf ? launch_stage<MODE_RHS, true, false>(A, st)
                      : launch_stage<MODE_RHS, false, false>(A, st);
        return pf ? launch_stage<MODE_STAGE, true, false>(A, st)
                  : launch_stage<MODE_STAGE, false, false>(A, st);
    }

    static cudaError_t face(const KArgs<Real> &A, bool diff, cudaStream_t st) {
        const int nb = A.M.fblk[0] + A.M.fblk[1] + A.M.fblk[2];
        return launch(diff ? &k_face<S, Real, true> : &k_face<S, Real, false>, nb, kFaceThreads, 0, st,
                      false, A);
    }

    static cudaError_t alpha_vertex(const KArgs<Real> &A, cudaStream_t st) {
        const size_t nvt = (size_t)A.M.nv[0] * A.M.nv[1] * (S::D == 3 ? A.M.nv[2] : 1);
        return launch(&k_alpha_vertex<S::D, Real>, grid_for(nvt, 256), 256, 0, st, false, A.M,
                      (const Real *)A.alphaK, const_cast<Real *>(A.alphaV));
    }

    static cudaError_t split(const KArgs<Real> &A, double *T, double *rv, double *rc, double *pp,
                             cudaStream_t st) {
        const size_t nodes = (size_t)A.M.ne * S::NP;
        k_split<S, Real><<<grid_for(nodes, 256), 256, 0, st>>>(A, T, rv, rc, pp);
        return cudaGetLastError();
    }

    static cudaError_t init_bubble(const KArgs<Real> &A, const BubbleArgs &B, cudaStream_t st) {
        const size_t nodes = (size_t)A.M.ne * S::NP;
        k_init_bubble<S, Real><<<grid_for(nodes, 256), 256, 0, st>>>(A, B);
        return cudaGetLastError();
    }

    static cudaError_t reduce(const KArgs<Real> &A, double *partials, int nblocks, cudaStream_t st) {
        k_reduce_partial<S, Real><<<nblocks, kRedThreads, 0, st>>>(A, partials);
        return cudaGetLastError();
    }

    template <int MODE>
    static cudaError_t launch_column(const KArgs<Real> &A, cudaStream_t st) {
        using C = ColShape<S>;
        constexpr size_t smem = column_smem_bytes<S, Real>();
        static OncePerDevice once;
        const cudaError_t err = allow_smem(once, &k_column<S, Real, MODE>, smem);
        if (err != cudaSuccess) return err;
        const int nxb = (A.M.n[0] + C::BX - 1) / C::BX;
        const int nyb = S::D == 3 ? (A.M.n[1] + C::BY - 1) / C::BY : 1;
        k_column<S, Real, MODE><<<nxb * nyb, C::NT, smem, st>>>(A);
        return cudaGetLastError();
    }

    static cudaError_t column(const KArgs<Real> &A, int mode, cudaStream_t st) {
        return mode == MODE_RHS ? launch_column<MODE_RHS>(A, st) : launch_column<MODE_STAGE>(A, st);
    }

    static Launchers<Real> table() {
        Launchers<Real> L;
        L.nf = S::NF;
        L.np = S::NP;
        L.nfp1 = S::NFP1;
        L.nd = S::ND;
        L.ntr = S::NTR;
        L.trace_face = TraceLayout<S, Real>::FACE;
        L.epb = S::EPB;
        L.nt = S::NT;
        L.prepare = &prepare;
        L.stage = &stage;
        L.face = &face;
        L.alpha_vertex = &alpha_vertex;
        L.split = &split;
        L.init_bubble = &init_bubble;
        L.reduce = &reduce;
        if constexpr (!F64)
            L.column = &column;
        else
            L.column = nullptr;
        return L;
    }
};

// Tables defined in the instantiation units; NULL for an unsupported order.
const Launchers<double> *launchers_d2_f64(int K, int rain);
const Launchers<double> *launchers_d3_f64(int K, int rain);
const Launchers<float> *launchers_d2_f32(int K, int rain);
const Launchers<float> *launchers_d3_f32(int K, int rain);
// float64 reference tables with the coefficients scaled by 2/h_j (dg_api.cu)
RefData<double> scaled_ref64(int dim, int order, const double two_over_h[3]);

}  // namespace dgm

namespace dgm {
// Tile of the kernels of one storage type: 128 threads, but 256 for float32 in
// 2-D (128 threads cost the 256-member ensemble 3 %).  Float64 in 2-D: 128
// threads spread small meshes over more SMs (20x10 order 3: 75 us per step
// against 84) and waste fewer lanes (order 4: 125 of 128; 128x64 with rain,
// four steps: 1.52 ms against 1.62 at 256 and 1.75 at 64).
template <int D, int K, bool RAIN, typename Real>
using TileShape = Shape<D, K, RAIN, (D == 2 && sizeof(Real) == sizeof(float)) ? 256 : 128>;
}  // namespace dgm

#define DGM_DEFINE_LAUNCHERS(NAME, DIM, REAL)                                          \
    namespace dgm {                                                                    \
    const Launchers<REAL> *NAME(int K, int rain) {                                     \
        static const Launchers<REAL> t[5][2] = {                                       \
            {Impl<TileShape<DIM, 1, false, REAL>, REAL>::table(), Impl<TileShape<DIM, 1, true, REAL>, REAL>::table()}, \
            {Impl<TileShape<DIM, 2, false, REAL>, REAL>::table(), Impl<TileShape<DIM, 2, true, REAL>, REAL>::table()}, \
            {Impl<TileShape<DIM, 3, false, REAL>, REAL>::table(), Impl<TileShape<DIM, 3, true, REAL>, REAL>::table()}, \
            {Impl<TileShape<DIM, 4, false, REAL>, REAL>::table(), Impl<TileShape<DIM, 4, true, REAL>, REAL>::table()}, \
            {Impl<TileShape<DIM, 5, false, REAL>, REAL>::table(), Impl<TileShape<DIM, 5, true, REAL>, REAL>::table()}, \
        };                                                                             \
        if (K < 1 || K > 5) return nullptr;                                            \
        return &t[K - 1][rain ? 1 : 0];                                                \
    }                                                                                  \
    }

// ---------------------------------------------------------------------------
// Adjoint launchers (float64 only), instantiated in dg_adj_*.cu
// ---------------------------------------------------------------------------
#include "dg_adjoint.cuh"

namespace dgm {

struct AdjLaunchers {
    int ntr;
    cudaError_t (*local)(const AdjArgs &, cudaStream_t);
    cudaError_t (*gather)(const AdjArgs &, cudaStream_t);
    cudaError_t (*cloud)(const AdjArgs &, double *partials, int nblocks, cudaStream_t);
};

template <class S>
struct AdjImpl {
    static constexpr size_t smem = adj_smem_bytes<S>();
    static cudaError_t local(const AdjArgs &A, cudaStream_t st) {
        static OncePerDevice once;
        const cudaError_t err = allow_smem(once, &k_adj_local<S>, smem);
        if (err != cudaSuccess) return err;
        k_adj_local<S><<<(A.M.ne + S::EPB - 1) / S::EPB, S::NT, smem, st>>>(A);
        return cudaGetLastError();
    }
    static cudaError_t gather(const AdjArgs &A, cudaStream_t st) {
        const size_t nodes = (size_t)A.M.ne * S::NP;
        k_adj_gather<S><<<grid_for(nodes, 256), 256, 0, st>>>(A);
        return cudaGetLastError();
    }
    static cudaError_t cloud(const AdjArgs &A, double *partials, int nblocks, cudaStream_t st) {
        k_cloud<S><<<nblocks, kRedThreads, 0, st>>>(A, partials);
        return cudaGetLastError();
    }
    static AdjLaunchers table() {
        AdjLaunchers L;
        L.ntr = S::NTR;
        L.local = &local;
        L.gather = &gather;
        L.cloud = &cloud;
        return L;
    }
};

const AdjLaunchers *adj_launchers_d2(int K, int rain);
const AdjLaunchers *adj_launchers_d3(int K, int rain);

}  // namespace dgm

#define DGM_DEFINE_ADJ_LAUNCHERS(NAME, DIM)                                             \
    namespace dgm {                                                                    \
    const AdjLaunchers *NAME(int K, int rain) {                                        \
        static const AdjLaunchers t[5][2] = {                                          \
            {AdjImpl<Shape<DIM, 1, false>>::table(), AdjImpl<Shape<DIM, 1, true>>::table()}, \
            {AdjImpl<Shape<DIM, 2, false>>::table(), AdjImpl<Shape<DIM, 2, true>>::table()}, \
            {AdjImpl<Shape<DIM, 3, false>>::table(), AdjImpl<Shape<DIM, 3, true>>::table()}, \
            {AdjImpl<Shape<DIM, 4, false>>::table(), AdjImpl<Shape<DIM, 4, true>>::table()}, \
            {AdjImpl<Shape<DIM, 5, false>>::table(), AdjImpl<Shape<DIM, 5, true>>::table()}, \
        };                                                                             \
        if (K < 1 || K > 5) return nullptr;                                            \
        return &t[K - 1][rain ? 1 : 0];                                                \
    }                                                                                  \
    }
