// Float64 tiles: the stage kernel's and k_prepare's work on EPB consecutive
// elements with the linear contractions (volume term, lift of the face
// fluxes, face traces, and with diffusion the derivatives) on the integer
// pipe (dg_fixed.cuh).
//
// The float64 tile is bound by the FP64 pipe (2 fmas per SM and clock); the
// contractions are 203 of the ~370 float64 operations per node and stage of
// 3-D order 4 with rain.  As fixed point they are 609 integer multiply-adds
// and ~1000 integer operations of conversion per node, on a pipe that is
// otherwise 4 % busy.  A group of the fixed point is one field of one tile.
//
// The rain density does not share the tile's scale: v_r ~ rho_r^(1/8) and the
// adjoint's rain powers see the sign and the relative size of rain many orders
// below the tile's largest (1e-22 kg/m^3 still falls at 0.1 m/s; a shared scale
// cost 2e-9 of the state after two steps at the edge of a rain shaft, against
// 2e-14).  Its volume and lift sums take a scale per line of each node
// (rain_sum), which keeps 57 bits against the line's largest term as a float64
// chain keeps 53; its short trace sums stay float64.
#pragma once

#include "dg_device.cuh"
#include "dg_fixed.cuh"

namespace dgm {

// A CTA's fixed-point coefficients, per direction j: the volume rows
// dhat_s[j][a][0 .. P1), liftm_s[j], liftp_s[j], with diffusion also
// dliftm_s[j], dliftp_s[j], (2/h_j) dmat[a][0 .. P1) and (2/h_j) dlm, dlp;
// then lm, lp of the traces.  In shared memory: a thread indexes them by its
// own a_j, where the parameter bank serves one address of a warp at a time.
template <class S, bool DIFF>
struct FxCoef {
    static constexpr int P1 = S::P1, ROWS = P1 * P1;
    static constexpr int LM = ROWS, LP = LM + P1;
    static constexpr int DLM = LP + P1, DLP = DLM + P1, DM = DLP + P1, DTM = DM + ROWS, DTP = DTM + P1;
    static constexpr int BLK = DIFF ? DTP + P1 : LP + P1;
    static constexpr int TM = S::D * BLK, TP = TM + P1;
    static constexpr int N = TP + P1;
};

// fields whose contractions are fixed point (the rain density's are float64)
template <class S>
__host__ __device__ constexpr bool fx_field(int f) {
    return !(S::RAIN && f == 2);
}

template <class S, bool DIFF>
__device__ __forceinline__ void fx_coef_fill(const KArgs<double> &A, int2 *s_cf) {
    using C = FxCoef<S, DIFF>;
    const RefData<double> &r = A.ref;
    for (int i = threadIdx.x; i < C::N; i += blockDim.x) {
        double v;
        int q;
        if (i >= C::TM) {
            v = i < C::TP ? r.lm[i - C::TM] : r.lp[i - C::TP];
            q = r.q_trace;
        } else {
            const int j = i / C::BLK, k = i - j * C::BLK;
            if (k < C::LM) {
                v = r.dhat_s[j][k / S::P1][k % S::P1];
                q = r.q_vol[j];
            } else if (k < C::LP + S::P1) {
                v = k < C::LP ? r.liftm_s[j][k - C::LM] : r.liftp_s[j][k - C::LP];
                q = r.q_lift[j];
            } else if (k < C::DM) {
                v = k < C::DLP ? r.dliftm_s[j][k - C::DLM] : r.dliftp_s[j][k - C::DLP];
                q = r.q_dlift[j];
            } else if (k < C::DTM) {
                v = A.M.two_over_h[j] * r.dmat[(k - C::DM) / S::P1][(k - C::DM) % S::P1];
                q = r.q_dmat[j];
            } else {
                v = A.M.two_over_h[j] * (k < C::DTP ? r.dlm[k - C::DTM] : r.dlp[k - C::DTP]);
                q = r.q_dtrace[j];
            }
        }
        s_cf[i] = fx_from(v, 1022 + q);
    }
}

// a per-direction exponent of the coefficient tables by a run-time direction
__device__ __forceinline__ int pick3(const int *q, int j) { return j == 0 ? q[0] : (j == 1 ? q[1] : q[2]); }

// Bits of the values of a group that are taken as fixed point, |x| < 2^bits:
// densities, mass fluxes and temperatures (kg/m^3, kg/m^2/s, K) 2^14, momenta
// with their fluxes and p' (Pa) 2^22, energies and energy fluxes (J/m^3, W/m^2)
// 2^34 -- 30 to 60 times what air at 1 bar and the speed of sound has.  A tile
// with a larger value in it takes float64 sums: the elements of a tile share
// the scale, and one that blows up must not cost the others their bits.  Below
// the line it costs them at most 2^-57 of it: 1e-13 kg/m^2/s, 3e-11 Pa,
// 1e-7 W/m^2, the rounding of the base state's own p, E and rho.
// Returns the largest exponent of group k (a field, or S::NF, + 1, + 2 for T,
// rho_v, p') with coefficients below 2^q in it.  Evaluated by one lane per group
// (fx_reduce_max): by every thread for every group it cost a small mesh 2 %.
template <class S>
__device__ __forceinline__ int fx_limit(int k, int q) {
    const int bits = k < S::IM || k == S::NF || k == S::NF + 1 ? 14 : (k == S::IE ? 34 : 22);
    return min(kFxMaxE, 1022 + bits + q);
}

// group exponents of N groups from the CTA's maxima (clamped below); true if
// any group leaves the fixed-point range (then every thread takes float64)
template <int N>
__device__ __forceinline__ bool fx_group(const int *s_e, int *E) {
    bool bad = false;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        E[k] = max(s_e[k], kFxMinE);
        bad = bad || E[k] > kFxMaxE;
    }
    return bad;
}

// Shared memory of a float64 stage tile: nodal fluxes s_fl [D][NF][STR] (then
// the node values of the traces [NTR][STR] in the same place; with diffusion
// those have their own, as the derivatives read them first), face fluxes s_fh
// [EPB][2D] (FaceLayout), element indices, with diffusion the vertex
// coefficients and alpha terms, coefficients s_cf, group exponents s_e.
template <class S, bool DIFF>
__host__ __device__ constexpr size_t stage64_fh_offset() {
    constexpr size_t FL = (size_t)S::D * S::NF;
    return (sizeof(double) * (DIFF ? FL + S::NTR : (FL > (size_t)S::NTR ? FL : (size_t)S::NTR)) * S::EPB *
            S::NP + 15) / 16 * 16;
}

template <class S, bool DIFF>
__host__ __device__ constexpr size_t stage64_cf_offset() {
    constexpr size_t fh = (size_t)S::EPB * S::NFACE * FaceLayout<S, double, DIFF ? 2 * S::NF : S::NF>::FACE;
    return (stage64_fh_offset<S, DIFF>() + sizeof(double) * fh + sizeof(int) * 8 * (size_t)S::EPB +
            (DIFF ? sizeof(double) * (size_t)S::EPB * (2 * S::NCORNER + 2 * S::NP) : 0) + 15) / 16 * 16;
}

template <class S, bool DIFF>
struct FxExp {   // s_e: nodal fluxes, traced values, with diffusion the differentiated fields
    static constexpr int FLUX = 0, TRACE = S::NF, NODE = S::NF + S::NTR, N = NODE + (DIFF ? S::NF : 0);
};

template <class S, bool DIFF>
constexpr size_t stage64_smem_bytes() {
    return stage64_cf_offset<S, DIFF>() + sizeof(int2) * FxCoef<S, DIFF>::N +
           sizeof(int) * FxExp<S, DIFF>::N;
}

// k_prepare: [NTR][STR] node values, alpha terms, coefficients, exponents
template <class S, bool DIFF>
constexpr size_t prepare64_smem_bytes() {
    return sizeof(double) * (size_t)(S::NTR + (DIFF ? 2 : 0)) * S::EPB * S::NP + sizeof(int2) * FxCoef<S, DIFF>::N +
           sizeof(int) * FxExp<S, DIFF>::N;
}

// Traces of the tile's node values v (U, T, rho_v, p' of this thread's node)
// on all 2D faces, one thread per face point in direction-major order; DIFF:
// also the traces of d/dx_j U.  s_tr [NTR][STR]; s_e (FxExp) starts at zero.
// Has barriers; the first also ends every earlier read of s_tr's memory.
template <class S, bool DIFF>
__device__ __forceinline__ void write_traces64(const KArgs<double> &A, const double *v, bool valid, int bidx,
                                               double *s_tr, const int2 *s_cf, int *s_e) {
    using C = FxCoef<S, DIFF>;
    constexpr int STR = S::EPB * S::NP;
    const int ne = A.M.ne, t = threadIdx.x;
    int E[S::NTR];
#pragma unroll
    for (int f = 0; f < S::NTR; ++f) E[f] = valid && fx_field<S>(f) ? fx_expo(v[f]) : 0;
    fx_reduce_max<S::NTR>(E, fx_limit<S>(t & 31, 0), s_e + FxExp<S, DIFF>::TRACE);
    __syncthreads();
    if (fx_group<S::NTR>(s_e + FxExp<S, DIFF>::TRACE, E)) {
        if (valid) {
#pragma unroll
            for (int f = 0; f < S::NTR; ++f) s_tr[f * STR + t] = v[f];
        }
        __syncthreads();
        write_traces_points<S, double, DIFF>(A, A.ref, s_tr, A.trace_out, bidx);
        return;
    }
    int2 *s_x = reinterpret_cast<int2 *>(s_tr);
    if (valid) {
#pragma unroll
        for (int f = 0; f < S::NTR; ++f) {
            if (fx_field<S>(f))
                s_x[f * STR + t] = fx_from(v[f], E[f]);
            else
                s_tr[f * STR + t] = v[f];
        }
    }
    __syncthreads();
    auto dot = [](const double *c, const double *x, int st) {   // float64 sum along a line (rain)
        double acc = 0.0;
#pragma unroll
        for (int i = 0; i < S::P1; ++i) acc = fma(c[i], x[i * st], acc);
        return acc;
    };
    constexpr int PER_J = S::EPB * 2 * S::NFP1;
    for (int item = t; item < S::EPB * S::NFACE * S::NFP1; item += S::NT) {
        const int j = item / PER_J;
        const int r = item - j * PER_J;
        const int el = r / (2 * S::NFP1);
        const int r2 = r - el * (2 * S::NFP1);
        const int side = r2 / S::NFP1;
        const int q = r2 - side * S::NFP1;
        const int e = bidx * S::EPB + el;
        if (e >= ne) continue;
        const int x0 = el * S::NP + line_node<S::D, S::P1>(j, q, 0);
        const int2 *x = s_x + x0;
        const double *xd = s_tr + x0;
        const int st = stride_of<S::P1>(j);
        double *out = A.trace_out + TraceLayout<S, double>::face(e, 2 * j + side) + q;
        int2 c[S::P1];
#pragma unroll
        for (int i = 0; i < S::P1; ++i) c[i] = s_cf[(side ? C::TP : C::TM) + i];
#pragma unroll
        for (int f = 0; f < S::NTR; ++f) {
            if (!has_trace<S>(f, j)) continue;
            if (!fx_field<S>(f)) {
                out[f * S::NFP1] = dot(side ? A.ref.lp : A.ref.lm, xd + f * STR, st);
                continue;
            }
            long long a2 = 0, a1 = 0;
#pragma unroll
            for (int i = 0; i < S::P1; ++i) fx_mac(c[i], x[f * STR + i * st], a2, a1);
            out[f * S::NFP1] = fx_value(a2, a1, E[f] + A.ref.q_trace);
        }
        if constexpr (DIFF) {
            double *dout = A.dtrace_out + ((size_t)e * S::NFACE + 2 * j + side) * S::NF * S::NFP1 + q;
            const int qd = pick3(A.ref.q_dtrace, j);
#pragma unroll
            for (int i = 0; i < S::P1; ++i) c[i] = s_cf[j * C::BLK + (side ? C::DTP : C::DTM) + i];
#pragma unroll
            for (int f = 0; f < S::NF; ++f) {
                if (!fx_field<S>(f)) {
                    dout[f * S::NFP1] = A.M.two_over_h[j] * dot(side ? A.ref.dlp : A.ref.dlm, xd + f * STR, st);
                    continue;
                }
                long long a2 = 0, a1 = 0;
#pragma unroll
                for (int i = 0; i < S::P1; ++i) fx_mac(c[i], x[f * STR + i * st], a2, a1);
                dout[f * S::NFP1] = fx_value(a2, a1, E[f] + qd);
            }
        }
    }
}

// Split and traces of a state (first stage, dg_rhs, uploads)
template <class S, bool DIFF>
__device__ __forceinline__ void prepare_block64(const KArgs<double> &A, int bidx, unsigned char *smem_raw) {
    constexpr int STR = S::EPB * S::NP;
    double *s_tr = reinterpret_cast<double *>(smem_raw);      // [NTR][STR]
    double *s_red = s_tr + S::NTR * STR;                      // DIFF: [2][STR]
    int2 *s_cf = reinterpret_cast<int2 *>(s_red + (DIFF ? 2 * STR : 0));
    int *s_e = reinterpret_cast<int *>(s_cf + FxCoef<S, DIFF>::N);
    const int t = threadIdx.x;
    const int el = t / S::NP, a = t - el * S::NP;
    const int e = bidx * S::EPB + el;
    const bool valid = t < STR && e < A.M.ne;
    double v[S::NTR];
    fx_coef_fill<S, DIFF>(A, s_cf);
    if (t < FxExp<S, DIFF>::N) s_e[t] = 0;
    dependents_wait();
    __syncthreads();
    if (valid) {
        const size_t nodes = (size_t)A.M.ne * S::NP, gi = (size_t)e * S::NP + a;
#pragma unroll
        for (int f = 0; f < S::NF; ++f) v[f] = A.Uin[f * nodes + gi];
        double vr;
        derive_and_store<S, double>(A, v, e, a, vert_index<S::D>(A.M, e), -1.0, v[S::NF], v[S::NF + 1],
                                    v[S::NF + 2], vr);
        if (DIFF)
            alpha_accumulate<S, double>(A, A.ref, v, vr, a,
                                        vert_index<S::D>(A.M, e) * S::P1 + digit<S::D, S::P1>(a, S::VERT),
                                        s_red, t);
    }
    write_traces64<S, DIFF>(A, v, valid, bidx, s_tr, s_cf, s_e);
    if (DIFF) alpha_store<S, double>(A, s_red, bidx);
}

// F_j of flux_dir (dg_device.cuh) for every direction at a node; m_i u_j is
// formed once for both orders of its indices.
template <class S>
__device__ __forceinline__ void flux_all(const Prim<S::D, S::RAIN, double> &P, double (*F)[S::NF]) {
    double q = 0.0, e = P.E + P.p;
    if (S::RAIN) q = P.rr * P.vr;
#pragma unroll
    for (int j = 0; j < S::D; ++j) {
        F[j][0] = P.rd * P.u[j];
        F[j][1] = P.rm * P.u[j];
        if (S::RAIN) F[j][2] = j == S::VERT ? fma(P.rr, P.u[j], -q) : P.rr * P.u[j];
        F[j][S::IM + j] = fma(P.m[j], P.u[j], P.pp);
#pragma unroll
        for (int i = 0; i < j; ++i) F[j][S::IM + i] = F[i][S::IM + j] = P.m[i] * P.u[j];
        F[j][S::IE] = e * P.u[j];
    }
    if (S::RAIN) {
        double ke = 0.0;
#pragma unroll
        for (int i = 0; i < S::D; ++i) {
            ke = fma(P.u[i], P.u[i], ke);
            F[S::VERT][S::IM + i] = fma(-q, P.u[i], F[S::VERT][S::IM + i]);
        }
        F[S::VERT][S::IE] = fma(-q, fma(kCl, P.T - kTref, 0.5 * ke), F[S::VERT][S::IE]);
    }
}

// Volume and lift terms of field f at a node as float64 sums
template <class S, bool PF, bool DIFF, int FACE>
__device__ __noinline__ double line_sums(const KArgs<double> &A, const double *s_fl, const double *s_fh,
                                         int el, int a, int f) {
    constexpr int STR = S::EPB * S::NP;
    double r = 0.0;
#pragma unroll 1
    for (int j = 0; j < S::D; ++j) {
        const int aj = digit<S::D, S::P1>(a, j), st = stride_of<S::P1>(j);
        const double *fl = s_fl + (j * S::NF + f) * STR + el * S::NP + a - aj * st;
        const double *fm = s_fh + (el * S::NFACE + 2 * j) * FACE + f * S::NFP1 + face_q<S::D, S::P1>(a, j);
        const double *fp = fm + FACE;
        const double cm = PF ? A.ref.liftm_s[j][aj] : -A.ref.liftm_s[j][aj], cp = A.ref.liftp_s[j][aj];
        for (int i = 0; i < S::P1; ++i) r = fma(A.ref.dhat_s[j][aj][i], fl[i * st], r);
        r = fma(cm, *fm, fma(-cp, *fp, r));
        if (DIFF)
            r = fma(A.ref.dliftm_s[j][aj], fm[S::NF * S::NFP1],
                    fma(A.ref.dliftp_s[j][aj], fp[S::NF * S::NFP1], r));
    }
    return r;
}

// Volume and lift terms of the rain density at a node: per direction the P1
// flux values (fl0, stride st) and the two face values (fm0, face block FACE)
// as fixed point with the line's own exponent, the three sums aligned to the
// largest.  About 500 integer operations for 21 float64 fmas: at the 32 : 1
// rate of the pipes half the time, on the one that has room.  ok is cleared
// where a value leaves the fixed-point range.
template <class S, bool PF, bool DIFF, int FACE>
__device__ __forceinline__ double rain_sum(const KArgs<double> &A, const double *s_fl, const double *s_fh,
                                           const int2 *s_cf, int el, int a, bool &ok) {
    using C = FxCoef<S, DIFF>;
    constexpr int STR = S::EPB * S::NP;
    constexpr int NL = S::P1 + (DIFF ? 4 : 2);
    long long v = 0;
    int E = kFxMinE;
#pragma unroll 1
    for (int j = 0; j < S::D; ++j) {
        const int aj = digit<S::D, S::P1>(a, j), st = stride_of<S::P1>(j);
        const double *fl = s_fl + (j * S::NF + 2) * STR + el * S::NP + a - aj * st;
        const double *gm = s_fh + (el * S::NFACE + 2 * j) * FACE + 2 * S::NFP1 + face_q<S::D, S::P1>(a, j);
        const double *gp = gm + FACE;
        const int2 *cf = s_cf + j * C::BLK;
        const int qv = A.ref.q_vol[j], ql = A.ref.q_lift[j], qd = DIFF ? A.ref.q_dlift[j] : 0;
        double x[NL];
        int Ej = kFxMinE;
#pragma unroll
        for (int i = 0; i < S::P1; ++i) {
            x[i] = fl[i * st];
            Ej = max(Ej, fx_expo(x[i]) + qv);
        }
        x[S::P1] = *gp;
        x[S::P1 + 1] = *gm;
        Ej = max(Ej, max(fx_expo(*gp), fx_expo(*gm)) + ql);
        if constexpr (DIFF) {
            x[S::P1 + 2] = gp[S::NF * S::NFP1];
            x[S::P1 + 3] = gm[S::NF * S::NFP1];
            Ej = max(Ej, max(fx_expo(x[S::P1 + 2]), fx_expo(x[S::P1 + 3])) + qd);
        }
        ok = ok && Ej <= kFxMaxE;
        long long a2 = 0, a1 = 0;
#pragma unroll
        for (int i = 0; i < S::P1; ++i) fx_mac(cf[aj * S::P1 + i], fx_from(x[i], Ej - qv), a2, a1);
        // -(high face), +(low face along +e_j) or -(outward flux)
        const int2 cp = cf[C::LP + aj], cm = cf[C::LM + aj];
        fx_mac(make_int2(-cp.x, -cp.y), fx_from(x[S::P1], Ej - ql), a2, a1);
        fx_mac(PF ? cm : make_int2(-cm.x, -cm.y), fx_from(x[S::P1 + 1], Ej - ql), a2, a1);
        if constexpr (DIFF) {
            fx_mac(cf[C::DLP + aj], fx_from(x[S::P1 + 2], Ej - qd), a2, a1);
            fx_mac(cf[C::DLM + aj], fx_from(x[S::P1 + 3], Ej - qd), a2, a1);
        }
        const int En = max(E, Ej);
        v = fx_shift(v, En - E) + fx_shift(a2 + (a1 >> 28), En - Ej);
        E = En;
    }
    return fx_round(v, E);
}

// One tile of EPB consecutive elements (tile index bidx) of the stage kernel:
// stage_block's phases (dg_device.cuh) with fixed-point contractions.  Every
// thread of the CTA takes part.
template <class S, int MODE, bool PF, bool DIFF>
__device__ __forceinline__ void stage_block64(const KArgs<double> &A, int bidx, unsigned char *smem_raw) {
    static_assert(!DIFF || PF, "artificial diffusion runs with the face pass");
    using C = FxCoef<S, DIFF>;
    using X = FxExp<S, DIFF>;
    constexpr int STR = S::EPB * S::NP;
    constexpr int NFP = DIFF ? 2 * S::NF : S::NF;             // per face: fluxes [, symmetry terms]
    constexpr int FACE = FaceLayout<S, double, NFP>::FACE;
    constexpr int EB = S::NFACE * FACE;                       // face values of one element
    double *s_fl = reinterpret_cast<double *>(smem_raw);
    double *s_tr = DIFF ? s_fl + S::D * S::NF * STR : s_fl;
    double *s_fh = reinterpret_cast<double *>(smem_raw + stage64_fh_offset<S, DIFF>());
    int *s_info = reinterpret_cast<int *>(s_fh + S::EPB * EB);             // inline: [EPB][8] neighbours
    double *s_al = reinterpret_cast<double *>(s_info + 8 * S::EPB);        // DIFF: [EPB][2][NCORNER]
    double *s_red = s_al + S::EPB * 2 * S::NCORNER;                        // DIFF: [2][STR]
    int2 *s_cf = reinterpret_cast<int2 *>(smem_raw + stage64_cf_offset<S, DIFF>());
    int *s_e = reinterpret_cast<int *>(s_cf + C::N);
    int2 *x_fl = reinterpret_cast<int2 *>(s_fl), *x_fh = reinterpret_cast<int2 *>(s_fh);
    int2 *x_tr = reinterpret_cast<int2 *>(s_tr);
    const MeshData &M = A.M;
    const int ne = M.ne;
    const size_t nodes = (size_t)ne * S::NP;
    const int t = threadIdx.x;
    const int el = t / S::NP, a = t - el * S::NP;
    const int e = bidx * S::EPB + el;
    const bool valid = (t < STR) && (e < ne);
    const size_t gi = (size_t)e * S::NP + a;

    fx_coef_fill<S, DIFF>(A, s_cf);
    if (t < X::N) s_e[t] = 0;
    dependents_wait();
    // the node's state and derived fields: loads issued first, so that their
    // latency overlaps the set-up below
    double u[S::NF], dT = 0.0, dir = 1.0, dpp = 0.0, dgm = 0.0, dvr = 0.0;
    if (valid) {
#pragma unroll
        for (int f = 0; f < S::NF; ++f) u[f] = A.Uin[f * nodes + gi];
        dT = A.derived[gi];
        dir = A.derived[nodes + gi];
        dpp = A.derived[2 * nodes + gi];
        if (S::RAIN) {
            dgm = A.derived[3 * nodes + gi];
            dvr = A.derived[4 * nodes + gi];
        }
    }
    // face pass: copy the tile's face values to shared memory while the
    // nodal phase runs (one contiguous block per face)
    if (PF) cp_async_faces<S, double, NFP>(A.fbuf, A.ftab, s_fh, bidx, min(S::EPB, ne - bidx * S::EPB));
    if (DIFF || !PF) {
        if (t < S::EPB && bidx * S::EPB + t < ne) {
            int im[3];
            elem_multi(M, bidx * S::EPB + t, im[0], im[1], im[2]);
#pragma unroll
            for (int j = 0; j < (PF ? 0 : S::D); ++j) {
                s_info[t * 8 + 2 * j] = neighbour_of<S::D>(M, im, j, -1);
                s_info[t * 8 + 2 * j + 1] = neighbour_of<S::D>(M, im, j, 1);
            }
            if (DIFF) alpha_corners<S, double>(A, im, s_al + t * 2 * S::NCORNER);
        }
    }
    const int iz = e / (S::D == 3 ? M.n[0] * M.n[1] : M.n[0]);

    // ---- phase 1: nodal fluxes (Eq. (2.11))
    int ex[S::NF];
#pragma unroll
    for (int f = 0; f < S::NF; ++f) ex[f] = 0;
    if (valid) {
        const int lev = iz * S::P1 + digit<S::D, S::P1>(a, S::VERT);
        double brd, brm, bE, bp;
        load_base<S, double>(A.bnode, M.nzlev_node, lev, brd, brm, bE, bp);
        Prim<S::D, S::RAIN, double> P;
        make_prim_inv<S, double>(P, u, brd, brm, bE, bp, dT, 0.0, dpp, dir);
        if (S::RAIN) P.vr = dvr;
        double F[S::D][S::NF];
        flux_all<S>(P, F);
#pragma unroll
        for (int j = 0; j < S::D; ++j)
#pragma unroll
            for (int f = 0; f < S::NF; ++f) {
                s_fl[(j * S::NF + f) * STR + t] = F[j][f];
                if (!DIFF && fx_field<S>(f)) ex[f] = max(ex[f], fx_expo(F[j][f]) + A.ref.q_vol[j]);
            }
    }

    // ---- phase 1b (diffusion): F_j -= alpha du/dx_j at the node, so that the
    // volume term below also carries (alpha grad u, grad phi_a) of Eq. (3.7)
    if constexpr (DIFF) {
        int E[S::NF];
#pragma unroll
        for (int f = 0; f < S::NF; ++f) E[f] = valid && fx_field<S>(f) ? fx_expo(u[f]) : 0;
        __syncthreads();
        fx_reduce_max<S::NF>(E, fx_limit<S>(t & 31, 0), s_e + X::NODE);
        __syncthreads();
        const bool bad = fx_group<S::NF>(s_e + X::NODE, E);
        if (valid) {
#pragma unroll
            for (int f = 0; f < S::NF; ++f) {
                if (bad || !fx_field<S>(f))
                    s_tr[f * STR + t] = u[f];
                else
                    x_tr[f * STR + t] = fx_from(u[f], E[f]);
            }
        }
        __syncthreads();
        if (valid) {
            double xi[3];
#pragma unroll
            for (int j = 0; j < S::D; ++j) xi[j] = A.ref.xi[digit<S::D, S::P1>(a, j)];
            const double *cv = s_al + el * 2 * S::NCORNER;
            const double au = q1_interp<S, double>(cv, xi), ar = q1_interp<S, double>(cv + S::NCORNER, xi);
#pragma unroll
            for (int j = 0; j < S::D; ++j) {
                const int aj = digit<S::D, S::P1>(a, j);
                const int st = stride_of<S::P1>(j);
                const int b0 = el * S::NP + a - aj * st;
#pragma unroll
                for (int f = 0; f < S::NF; ++f) {
                    double du;
                    if (bad || !fx_field<S>(f)) {
                        du = 0.0;
#pragma unroll
                        for (int i = 0; i < S::P1; ++i)
                            du = fma(A.ref.dmat[aj][i], s_tr[f * STR + b0 + i * st], du);
                        du *= M.two_over_h[j];
                    } else {
                        long long a2 = 0, a1 = 0;
#pragma unroll
                        for (int i = 0; i < S::P1; ++i)
                            fx_mac(s_cf[j * C::BLK + C::DM + aj * S::P1 + i], x_tr[f * STR + b0 + i * st], a2, a1);
                        du = fx_value(a2, a1, E[f] + A.ref.q_dmat[j]);
                    }
                    const double al = (S::RAIN && f == 2) ? ar : au;
                    double &F = s_fl[(j * S::NF + f) * STR + t];
                    F = fma(-al, du, F);
                    if (fx_field<S>(f)) ex[f] = max(ex[f], fx_expo(F) + A.ref.q_vol[j]);
                }
            }
        }
    }

    // ---- phase 2: face fluxes: from the face pass (copied asynchronously
    // since the start), or the Lax-Friedrichs flux at every face point of the
    // CTA's elements.  Face points go in direction-major order (direction,
    // element, side, point), so that the lanes of a warp mostly share the
    // direction.  Then the group exponents over fluxes and face fluxes.
    if (PF) cp_async_wait_all();
    __syncthreads();
    constexpr int PER_J = S::EPB * 2 * S::NFP1, FACE_ITEMS = S::EPB * S::NFACE * S::NFP1;
    auto face_item = [&](int item, int &jd, int &el2, int &face, int &q) {
        jd = item / PER_J;
        const int r = item - jd * PER_J;
        el2 = r / (2 * S::NFP1);
        const int r2 = r - el2 * (2 * S::NFP1);
        face = 2 * jd + r2 / S::NFP1;
        q = r2 - (face & 1) * S::NFP1;
        return bidx * S::EPB + el2 < ne;
    };
    for (int item = t; item < FACE_ITEMS; item += S::NT) {
        int jd, el2, face, q;
        if (!face_item(item, jd, el2, face, q)) continue;
        if constexpr (!PF) {
            const int e2 = bidx * S::EPB + el2, nb = s_info[el2 * 8 + face];
            const int iz2 = e2 / (S::D == 3 ? M.n[0] * M.n[1] : M.n[0]);
            switch (jd) {
                case 0: face_point<S, double, 0>(A, A.ref, s_tr, s_fh, el2, face, q, e2, nb, iz2); break;
                case 1: face_point<S, double, 1>(A, A.ref, s_tr, s_fh, el2, face, q, e2, nb, iz2); break;
                default:
                    face_point<S, double, (S::D == 3 ? 2 : 1)>(A, A.ref, s_tr, s_fh, el2, face, q, e2, nb, iz2);
                    break;
            }
        }
        const double *g = s_fh + (el2 * S::NFACE + face) * FACE + q;
        const int ql = pick3(A.ref.q_lift, jd);
#pragma unroll
        for (int f = 0; f < S::NF; ++f)
            if (fx_field<S>(f)) ex[f] = max(ex[f], fx_expo(g[f * S::NFP1]) + ql);
        if constexpr (DIFF) {
            const int qd = pick3(A.ref.q_dlift, jd);
#pragma unroll
            for (int f = 0; f < S::NF; ++f)
                if (fx_field<S>(f)) ex[f] = max(ex[f], fx_expo(g[(S::NF + f) * S::NFP1]) + qd);
        }
    }
    fx_reduce_max<S::NF>(ex, fx_limit<S>(t & 31, A.ref.q_max), s_e + X::FLUX);
    __syncthreads();

    // ---- phase 3: volume term of Eq. (3.2), sum factorised,
    //   R_a = (2/h_j) sum_i dhat[a_j][i] F_j(i),
    // and the lift of the face fluxes, R_a -= (2/h_j) l_a(s)/w_a Fhat(j, s).
    // The low face holds the outward flux (inline) or G along +e_j, minus
    // this element's outward flux (face pass), hence the sign.
    const bool bad = fx_group<S::NF>(s_e + X::FLUX, ex);
    double R[S::NF];
    if (!bad) {
        // in place: each thread converts the words that it wrote or scanned
        if (valid) {
#pragma unroll 1
            for (int j = 0; j < S::D; ++j)
#pragma unroll
                for (int f = 0; f < S::NF; ++f) {
                    if (!fx_field<S>(f)) continue;
                    const int k = (j * S::NF + f) * STR + t;
                    x_fl[k] = fx_from(s_fl[k], ex[f] - A.ref.q_vol[j]);
                }
        }
        for (int item = t; item < FACE_ITEMS; item += S::NT) {
            int jd, el2, face, q;
            if (!face_item(item, jd, el2, face, q)) continue;
            const int k = (el2 * S::NFACE + face) * FACE + q;
            const int ql = pick3(A.ref.q_lift, jd), qd = DIFF ? pick3(A.ref.q_dlift, jd) : 0;
#pragma unroll
            for (int f = 0; f < NFP; ++f) {
                if (!fx_field<S>(f % S::NF)) continue;
                x_fh[k + f * S::NFP1] =
                    fx_from(s_fh[k + f * S::NFP1], f < S::NF ? ex[f] - ql : ex[f - S::NF] - qd);
            }
        }
        __syncthreads();
        if (valid) {
            long long a2[S::NF], a1[S::NF];
#pragma unroll
            for (int f = 0; f < S::NF; ++f) a2[f] = a1[f] = 0;
#pragma unroll 1
            for (int j = 0; j < S::D; ++j) {
                const int aj = digit<S::D, S::P1>(a, j);
                const int st = stride_of<S::P1>(j);
                const int q = face_q<S::D, S::P1>(a, j);
                const int fl0 = j * S::NF * STR + el * S::NP + a - aj * st;
                const int fm0 = (el * S::NFACE + 2 * j) * FACE + q;
                const int2 *fl = x_fl + fl0, *fm = x_fh + fm0, *fp = fm + FACE;
                const int2 *cf = s_cf + j * C::BLK;
                int2 c[S::P1], cm = cf[C::LM + aj], cp = cf[C::LP + aj];
#pragma unroll
                for (int i = 0; i < S::P1; ++i) c[i] = cf[aj * S::P1 + i];
                cp = make_int2(-cp.x, -cp.y);
                if (!PF) cm = make_int2(-cm.x, -cm.y);
#pragma unroll
                for (int f = 0; f < S::NF; ++f) {
                    if (!fx_field<S>(f)) continue;
#pragma unroll
                    for (int i = 0; i < S::P1; ++i) fx_mac(c[i], fl[f * STR + i * st], a2[f], a1[f]);
                    fx_mac(cp, fp[f * S::NFP1], a2[f], a1[f]);
                    fx_mac(cm, fm[f * S::NFP1], a2[f], a1[f]);
                }
                if constexpr (DIFF) {
                    // symmetry term of Eq. (3.7): + (2/h_j)^2 l_a'(s)/w_a S on both faces
                    const int2 dm = cf[C::DLM + aj], dp = cf[C::DLP + aj];
#pragma unroll
                    for (int f = 0; f < S::NF; ++f) {
                        if (!fx_field<S>(f)) continue;
                        fx_mac(dp, fp[(S::NF + f) * S::NFP1], a2[f], a1[f]);
                        fx_mac(dm, fm[(S::NF + f) * S::NFP1], a2[f], a1[f]);
                    }
                }
            }
#pragma unroll
            for (int f = 0; f < S::NF; ++f) R[f] = fx_field<S>(f) ? fx_value(a2[f], a1[f], ex[f]) : 0.0;
            if constexpr (S::RAIN) {
                bool ok = true;
                R[2] = rain_sum<S, PF, DIFF, FACE>(A, s_fl, s_fh, s_cf, el, a, ok);
                if (!ok) R[2] = line_sums<S, PF, DIFF, FACE>(A, s_fl, s_fh, el, a, 2);
            }
        }
    } else if (valid) {
        // values outside the fixed-point range (blown up, infinite, NaN): float64 sums
#pragma unroll
        for (int f = 0; f < S::NF; ++f) R[f] = line_sums<S, PF, DIFF, FACE>(A, s_fl, s_fh, el, a, f);
    }

    // ---- phase 4: sources G (Eq. (2.11): microphysics and gravity), then
    // dU/dt or the stage update, the next stage's split and its traces
    double v[S::NTR];
    if (valid) {
        if (S::RAIN) {
            R[1] += dgm;
            R[2] -= dgm;
        }
        R[S::IM + S::VERT] = fma(-M.g, u[0] + u[1] + (S::RAIN ? u[2] : 0.0), R[S::IM + S::VERT]);
        R[S::IE] = fma(-M.g, u[S::IM + S::VERT], R[S::IE]);
        if (MODE == MODE_RHS) {
#pragma unroll
            for (int f = 0; f < S::NF; ++f) A.Uout[f * nodes + gi] = R[f];
        } else {
#pragma unroll
            for (int f = 0; f < S::NF; ++f) {
                double w = fma(A.gdt, R[f], is_one(A.beta) ? u[f] : A.beta * u[f]);
                if (nonzero(A.alpha)) w = fma(A.alpha, A.Un[f * nodes + gi], w);
                v[f] = w;
            }
            if (A.sponge) apply_sponge<S, double>(A.sponge[iz * S::P1 + digit<S::D, S::P1>(a, S::VERT)], v);
#pragma unroll
            for (int f = 0; f < S::NF; ++f) A.Uout[f * nodes + gi] = v[f];
            double vr;
            derive_and_store<S, double>(A, v, e, a, iz, dT, v[S::NF], v[S::NF + 1], v[S::NF + 2], vr);
            if (DIFF)
                alpha_accumulate<S, double>(A, A.ref, v, vr, a, iz * S::P1 + digit<S::D, S::P1>(a, S::VERT),
                                            s_red, t);
        }
    }
    if (MODE == MODE_STAGE) {
        write_traces64<S, DIFF>(A, v, valid, bidx, s_tr, s_cf, s_e);
        if (DIFF) alpha_store<S, double>(A, s_red, bidx);
    }
}

template <class S, bool DIFF>
__global__ void __launch_bounds__(S::NT) k_prepare64(KArgs<double> A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    dependents_go();
    prepare_block64<S, DIFF>(A, blockIdx.x + A.tile0, smem_raw);
}

// Register budget for 768 threads per SM (80 registers): one tile alternates
// float64 and integer phases, so more tiles in flight keep the FP64 pipe
// busier (64x64x32 order 4 with rain, two steps: 74.0 ms at the natural 114
// registers, 72.6 for 640 threads, 71.4 for 768).  With diffusion the tile's
// shared memory is the limit and a budget only cost (12.2 against 12.5 ms).
template <class S, bool DIFF>
constexpr int stage64_min_blocks() {
    return DIFF ? 0 : 768 / S::NT;
}

template <class S, int MODE, bool PF, bool DIFF>
__global__ void __launch_bounds__(S::NT, (stage64_min_blocks<S, DIFF>())) k_stage64(KArgs<double> A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    dependents_go();
    stage_block64<S, MODE, PF, DIFF>(A, blockIdx.x + A.tile0, smem_raw);
}

}  // namespace dgm
