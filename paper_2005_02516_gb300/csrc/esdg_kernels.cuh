// CUDA kernels of the ESDG shallow-water right-hand side and LSRK45 stage
// (Wu, Kubatko, Chan, arXiv 2005.02516).  Written for sm_103a.
//
// Per RK stage one fused kernel does, per element (a warp per element):
//   volume flux differencing with the entropy-conservative SWE flux
//   (eqs. (SWE_flux1/2)) and its well-balanced bathymetry term, on the skew
//   hybridized operator of Sec. 5.2 (Q_skew = Q_h - Q_h^T, whose lower-right
//   block is zero and skipped), with the curved metric average of Sec. 2.7;
//   the interface flux f_S(u~+, u~) with Lax-Friedrichs (Sec. 2.8);
//   the lift V_h^T and the stored inverse curved mass matrix (Sec. 2.7, 5.1);
//   the LSRK45 stage update in FP64 (Sec. 4);
//   and the entropy projection (Sec. 2.6) of the updated state, written for
//   the next stage (its face values are what neighbours read).
//
// Algebra used by the volume loop.  With sums over the pair (l, m)
//   HU = hu_l + hu_m, HV = hv_l + hv_m, U = u_l + u_m, V = v_l + v_m,
// and the metric average folded into the operator entries
//   Qx = 1/4 Qskew^x[l,m] = qr (rx_l + rx_m) + qs (sx_l + sx_m), (metrics / 8)
// the row-l contribution of Qskew^x o F^x + Qskew^y o F^y is
//   h  : 2 (Qx HU + Qy HV)
//   hu : U (Qx HU + Qy HV) + Qx * 2 g h_l H_m
//   hv : V (Qx HU + Qy HV) + Qy * 2 g h_l H_m
// where the pressure g{h}^2 - g{h^2}/2 = g h_l h_m / 2 and the source
// -g h~ (1/2 Qskew b) combine into g/2 h_l (h_m + b_m) = g/2 h_l H_m.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "esdg_async.cuh"
#include "esdg_fixed.cuh"

namespace esdg {

// Points of the fully symmetric volume rule exact to degree 2N.
constexpr int symmetric_points(int N) { return N == 1 ? 3 : N == 2 ? 6 : N == 3 ? 12 : N == 4 ? 16 : 25; }

// Template parameter NR = N + 8 * rule + 16 * wadg: the degree N (1..5), the
// volume rule (0: collapsed (N+1)^2 points, 1: symmetric, exact to 2N) and the
// inverse mass matrix (0: the stored (M_h^k)^{-1} of Sec. 2.7; 1: the
// weight-adjusted inverse M^{-1} M_{1/J} M^{-1} = Vq^T W diag(1/J) Vq applied
// on the fly, the alternative Sec. 2.8 names; M = I for these rules), plus
// 32 * tc for the FP32 kernel whose dense contractions run on the tensor cores and
// 64 * compact for the FP64 kernel that stores no operators per element (25-point
// rules: the metrics are averaged and the inverse applied in each stage).
template <int NR>
struct Dims {
    static constexpr int N = NR & 7;
    static constexpr int rule = (NR >> 3) & 1;
    static constexpr int wadg = (NR >> 4) & 1;
    static constexpr int tc = (NR >> 5) & 1;    // dense contractions on the tensor cores (FP32 kernel)
    static constexpr int compact = (NR >> 6) & 1;
    static constexpr int Np = (N + 1) * (N + 2) / 2;
    static constexpr int Nq = rule ? symmetric_points(N) : (N + 1) * (N + 1);
    static constexpr int Nfp = N + 1;
    static constexpr int Nfq = 3 * (N + 1);
    static constexpr int Nh = Nq + Nfq;
    static constexpr int NpP = Np * (Np + 1) / 2;
};

// The FP64 kernel's unique-pair schedule (rules of up to 32 volume points):
// lane j of a group stands for volume row j, volume-volume pairs run along the
// diagonals (j, j + d mod V), d = 1..SVV, and volume-face pairs along
// (j, V + (j + t) mod L), t < L.  With L <= 16 the two half-warps are two groups
// that split the diagonals (half 0: d <= SVV0 and t < SVF0); larger rules run
// one group over the warp.  NSTEP steps in all.
template <int NR>
struct PairSched {
    typedef Dims<NR> D;
    static constexpr int V = D::Nq, F = D::Nfq, L = V > F ? V : F;
    static constexpr bool DIAG = L <= 32 && !D::compact;
    static constexpr int HALVES = L <= 16 ? 2 : 1;
    static constexpr int SVV = V / 2, SVV0 = (SVV + HALVES - 1) / HALVES, SVF0 = (L + HALVES - 1) / HALVES;
    static constexpr int NSTEP = SVV0 + SVF0;
};

// The FP64 path keeps the stored inverse's products with the shared operators
// per element (StageParams lk, gk, pk) where the lane mapping covers them: up to
// 16 modes and 32 hybrid nodes (two half-warps of modes), and the 25-point rule
// of N = 5 (a lane per mode, two passes over the hybrid nodes).
template <int NR>
constexpr bool composed_inverse() {
    typedef Dims<NR> D;
    return !D::wadg && !D::compact && ((D::Np <= 16 && D::Nh <= 32) || (D::N == 5 && D::rule == 1));
}
template <int NR>
struct Composed {
    typedef Dims<NR> D;
    static constexpr bool SPLIT = D::Np <= 16;              // modes n = lane & 15, else n = lane
    static constexpr int LT = SPLIT ? (D::Nh + 1) / 2 : D::Nh;  // terms a lane takes of M^-1 Vh^T
    static constexpr int GT = SPLIT ? (D::Nq + 1) / 2 : D::Nq;  // ... of M^-1 Vq^T
    static constexpr int PP = (D::Nh + 31) / 32;            // passes over the hybrid nodes
};

// status bits written by the device
constexpr int STATUS_NONPOSITIVE = 1;
constexpr int STATUS_NONFINITE = 2;

template <typename real>
struct StageParams {
    int K;
    real g;
    real ig2;          // 1 / (2 g)
    int lf;
    // reference operators (global, staged into shared memory)
    const real* QsT;   // [Nh(m)][Nh(l)][2]: (Qskew^r[l][m], Qskew^s[l][m])
    const real* Vq;    // [Nq][Np]
    const real* VqT;   // [Np][Nq]
    const real* Vh;    // [Nh][Np]
    const real* VhT;   // [Np][Nh]
    const real* wf;    // [Nfq]
    const real* nrs;   // [Nfq][2] scaled reference normals
    const real* wq;    // [Nq]     volume weights (weight-adjusted inverse: w_q / J_q = w_q^2 / (w_q J_q))
    const real* iwJ;   // [K][Nq]  DG-SBP FP64: 1 / (w_q J_q), the inverse of the diagonal mass (else null)
    const int* fmap;   // [Nfq]    DG-SBP: the volume node of each face node (the selection I_f)
    // per element
    const real* geo;   // [K][Nh][4] rxJ sxJ ryJ syJ (FP64: only where the pair loop reads them, Smem::PIECES)
    const real* face;  // FP64 where geo is not read [K][Nfq][4]: w/2 (nxJ, nyJ, sJ sqrt(g)) at the face nodes, 0
    const real* wJq;   // [K][Nq]   w_q J_q
    const real* minv;  // [K][mstride] packed (M_h^k)^{-1} (stored inverse only)
    int mstride;       // element stride of minv (NpP rounded up to a multiple of 4)
    const real* bh;    // [K][Nh]   bathymetry at hybrid nodes
    const int* nbr;    // [K][3]    4 * neighbour element + neighbour face (4 e + 3: wall)
    int walls;         // reflective walls present (Sec. 2.9)
    const real* xq;    // [K][Nq]   (forcing only, FP32)
    const real* yq;
    // forcing in FP64: [K][Nq] (sin pi (x + y), cos pi (x + y), b_x, b_y) at the
    // volume nodes, and (sin, cos) pi t of the stage
    const double4* frc;
    double sin_t, cos_t;
    // FP64 unique-pair schedule: the metric-averaged skew operator entries
    // (Qskew^x, Qskew^y)[j][m] of the pair each lane takes in each step, as
    // fixed-point limbs (esdg_fixed.cuh), [K][NSTEP][32][2] (zero where the lane
    // has no pair); stage-independent, formed once on the host
    const real* qxy;
    // FP64 fixed-point scales of element e's operators, [K][4]: qxy (fx_pack of Qx's
    // and Qy's), lk, gk, pk (each: the largest absolute row sum is below 2^X), and of Vq;
    // DG-SBP: [K] int, qxy's
    const int4* fexp;
    int xvq;
    // FP64 path with the stored inverse (composed_inverse): per-element
    // products of the inverse mass with the shared operators, formed once on
    // the host, as fixed-point limbs in the order the lanes read them
    // (zero-padded):
    //   lk [K][LT][32]      M^-1 Vh^T   (lift + inverse mass), lane = n + 16 hf,
    //                        column l = hf LT + t at step t (lane = n, l = t where
    //                        Np > 16)
    //   gk [K][GT][32]      M^-1 Vq^T W J   (forcing), the same with columns q
    //   pk [K][Nq][PP][32]  Vh M^-1 Vq^T W J (projection to the hybrid nodes), l = lane + 32 pass
    // (composed_inverse; elsewhere the inverse is applied to the shared
    // operators' results in turn)
    const real* lk;
    const real* gk;
    const real* pk;
    // state
    const double* u_in;  // [3][K][Np]  (projection input)
    double* u;           // [3][K][Np]  RK state (updated in place)
    double* res;         // [3][K][Np]  RK residual
    double* rhs_out;     // [3][K][Np]  RHS mode output
    double* u_out;       // [3][K][Np]  if set: the stage's new state also written here (host-state calls)
    int copy_in;         // projection of u_in: also store u_in into u and zero res
    const real* ut_in;   // [K][Nh][4]  entropy-projected (h, u, v, H) of this stage (the FP32 batched
                         //             kernel k_stage2 stores H - H_0, H_0 the element's H at node 0)
    real* ut_out;        // [K][Nh][4]  ... of the next stage
    double rkA, rkB, dt, t;
    int forcing;
    real mms_amp, mms_bamp, mms_u0, mms_v0;
    int* status;
};

// Programmatic dependent launch: a stage kernel is launched while the kernel
// before it on the stream drains.  Its prologue (the shared operators into
// shared memory, barrier set-up) reads constants only; pdl_wait returns once
// the kernels before it have completed and their writes are visible, so
// everything a stage reads or writes comes after it.  pdl_trigger lets the next
// kernel's blocks take the places that this one's leave; every block calls it
// after its own pdl_wait, at its last round.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Element of a warp of the warp-per-element kernels in the round of the
// gridDim.x * wpb elements from e0: neighbouring warps take neighbouring
// elements, but in a last round of fewer elements neighbouring blocks do, so
// that its elements are spread over the blocks and with them over the SMs
// (which block lands on which SM is not fixed: a dependent launch's blocks take
// the places that come free).
__device__ __forceinline__ int element_of(int K, int e0, int warp, int wpb) {
    return e0 + (K - e0 < (int)gridDim.x * wpb ? (int)(blockIdx.x + gridDim.x * warp)
                                               : (int)(blockIdx.x * wpb + warp));
}

template <typename real>
struct V2;
template <>
struct V2<float> { typedef float2 t; };
template <>
struct V2<double> { typedef double2 t; };

template <typename real>
__device__ __forceinline__ real r_sqrt(real x);
template <>
__device__ __forceinline__ float r_sqrt<float>(float x) { return sqrtf(x); }
template <>
__device__ __forceinline__ double r_sqrt<double>(double x) { return sqrt(x); }

// The manufactured-solution forcing of Sec. 4.1 (sine solution) in FP64 at
// volume node i = e Nq + q.  sin and cos of pi (x + y - t) by the addition
// theorem from the stored values of the node and the stage's (three sincospi a
// node were more than half of this path's FP64 instructions).
template <typename P>
__device__ __forceinline__ void mms_forcing64(const P& p, size_t i, double& f0, double& f1, double& f2) {
    const double2* q = reinterpret_cast<const double2*>(p.frc + i);
    const double2 a = q[0], b = q[1];
    const double sth = a.x * p.cos_t - a.y * p.sin_t, cth = a.y * p.cos_t + a.x * p.sin_t;
    const double h = fma((double)p.mms_amp, sth, 2.0), gh = (double)p.g * h;
    const double c = (double)p.mms_amp * 3.14159265358979323846 * cth;  // h_x = h_y = -h_t
    const double u0 = p.mms_u0, v0 = p.mms_v0, w0 = u0 + v0 - 1.0;
    f0 = w0 * c;
    f1 = u0 * f0 + gh * (c + b.x);
    f2 = v0 * f0 + gh * (c + b.y);
}

// Finite, and positive (infinity included): on the integer pipes, where a
// floating-point comparison of doubles would hold the FP64 pipe.
__device__ __forceinline__ bool r_finite(double x) { return fx_exp(x) != FX_NONFINITE; }
__device__ __forceinline__ bool r_positive(double x) {
    return (unsigned long long)__double_as_longlong(x) - 1u < 0x7ff0000000000000ull;
}
// Row r of a three-field contraction with T terms, for R <= 16 rows: the two
// half-warps take half of the terms each and the sums meet by a shuffle, so
// all 32 lanes work (rows r = lane & 15).  acc(r, t, a0, a1, a2) adds term t.
// Every lane of the warp calls it; it returns true on lanes 0..R-1, which hold
// the sums of row r = lane.
template <int R, int T, typename real, typename Acc>
__device__ __forceinline__ bool split_rows(int lane, Acc acc, real& a0, real& a1, real& a2) {
    static_assert(R <= 16, "two half-warps of rows");
    constexpr int TH = (T + 1) / 2;
    const int r = lane & 15, hf = lane >> 4;
    a0 = a1 = a2 = real(0);
    if (r < R) {
#pragma unroll
        for (int tt = 0; tt < TH; ++tt) {
            const int t = hf * TH + tt;
            if (t < T) acc(r, t, a0, a1, a2);
        }
    }
    a0 += __shfl_down_sync(0xffffffffu, a0, 16);
    a1 += __shfl_down_sync(0xffffffffu, a1, 16);
    a2 += __shfl_down_sync(0xffffffffu, a2, 16);
    return lane < R;
}

// The same in block fixed point: sum of op(t) x[f][t] over the terms t of this
// lane's half (SPLIT: rows r = lane & 15, the halves' sums meet by a shuffle;
// else all T terms), x[f] the limbs of field f at x + f F.  s[f]: the three
// sums in units of 2^56.
template <int T, int F, bool SPLIT, typename Op>
__device__ __forceinline__ void fx_rows(int lane, const int2* x, Op op, long long (&s)[3]) {
    constexpr int TH = SPLIT ? (T + 1) / 2 : T;
    const int t0 = SPLIT ? (lane >> 4) * TH : 0;
    FxSum a0 = {0, 0}, a1 = {0, 0}, a2 = {0, 0};
    constexpr int U = TH <= 16 ? TH : 13;  // (N = 5: 6% slower with 5, spills unrolled in full)
#pragma unroll (U)
    for (int tt = 0; tt < TH; ++tt) {
        if (T % 2 == 0 || !SPLIT || tt < TH - 1 || t0 + tt < T) {
            const int2 v = op(tt);
            const int2* xt = x + t0 + tt;
            fx_mac(a0, v, xt[0]);
            fx_mac(a1, v, xt[F]);
            fx_mac(a2, v, xt[2 * F]);
        }
    }
    s[0] = fx_value(a0);
    s[1] = fx_value(a1);
    s[2] = fx_value(a2);
    if (SPLIT)
#pragma unroll
        for (int f = 0; f < 3; ++f) s[f] += __shfl_down_sync(0xffffffffu, s[f], 16);
}

// Limbs of three fields' values of this lane, M sets x[i] (in[i]: it has them),
// with a scale per field over the warp, written to o[at[i]], F apart; X the
// scales.  False if one of the values is not finite.
template <int F, int M>
__device__ __forceinline__ bool fx_store(const bool (&in)[M], const double (&x)[M][3], int2* o, const int (&at)[M],
                                         int (&X)[3]) {
    int most = 0;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        int e = 0;
#pragma unroll
        for (int i = 0; i < M; ++i) e = max(e, in[i] ? fx_exp(x[i][f]) : 0);
        e = fx_max(e);
        most = max(most, e);
        X[f] = fx_scale(e);
    }
#pragma unroll
    for (int i = 0; i < M; ++i)
        if (in[i])
#pragma unroll
            for (int f = 0; f < 3; ++f) o[at[i] + f * F] = fx_limbs(fx_from<FX_VAL>(x[i][f], X[f]));
    return most != FX_NONFINITE;
}
template <int F>
__device__ __forceinline__ bool fx_store(bool in, double x0, double x1, double x2, int2* o, int at, int (&X)[3]) {
    const bool in1[1] = {in};
    const double x[1][3] = {{x0, x1, x2}};
    const int at1[1] = {at};
    return fx_store<F, 1>(in1, x, o, at1, X);
}
// The row sums of fx_rows as doubles: field f's values of scale X[f], operator of scale Xo.
__device__ __forceinline__ void fx_row_values(const long long (&s)[3], const int (&X)[3], int Xo, bool finite,
                                              double (&y)[3]) {
    fx_to<3>(s, [&](int f) { return X[f] + Xo - (FX_VAL + FX_ROW - 2 * FX_LO); }, y);
    if (!finite) y[0] = y[1] = y[2] = __longlong_as_double(0x7ff8000000000000ll);
}

// Volume flux differencing of one element along the diagonals of PS, in block
// fixed point.  rec: the node records, six 8-byte words a node, the first five the
// limbs of hu, hv (scales of fx_align), u (Xu), v (Xv) and H (XH); qe: this lane's operator
// entries, (Qx, Qy) of step k at qe[32 k].  a: the sums of T, u_m T, v_m T, Qx H_m
// and Qy H_m over the pairs of volume row j that this lane (its half-warp) took,
// b: the same of face row V + j (fx_pair_sums).
//
// Every non-zero pair (l, m) of Q_skew is evaluated once (the face-face block is
// zero) by the lane of volume row l: T = Qx (hu_l + hu_m) + Qy (hv_l + hv_m) is
// antisymmetric in (l, m), and so are Qx and Qy.  In every step each row also
// receives exactly one pair's T and (Qx, Qy), from the lane d (or t) places
// before it, by shuffles, and adds that pair's terms of its own side from the
// sender's node record.  Steps without a pair carry stored entries of zero.  In
// fixed point: 30 IMAD.WIDE a pair for both rows, against 14 instructions on the
// FP64 pipe (and 17 when the sender formed the receiver's terms).
template <class PS>
__device__ __forceinline__ void fx_diagonals(const double* rec, const int4* qe, int lane, long long (&a)[5],
                                             long long (&b)[5]) {
    constexpr int V = PS::V, F = PS::F, L = PS::L, HV = PS::HALVES, REC = 6;
    const int j = HV == 2 ? lane & 15 : lane, hf = HV == 2 ? lane >> 4 : 0;
    const int4 m_l = *reinterpret_cast<const int4*>(rec + (j < V ? j : 0) * REC);  // hu, hv
    long long A0 = 0, B0 = 0;
    FxSum A1 = {0, 0}, A2 = {0, 0}, A3 = {0, 0}, A4 = {0, 0};
    FxSum B1 = {0, 0}, B2 = {0, 0}, B3 = {0, 0}, B4 = {0, 0};  // received terms only: the opposite sign
    int2 Tr, Qxr, Qyr;
    auto pair = [&](int m, int4 q, int src) {
        const int4* rm = reinterpret_cast<const int4*>(rec + m * REC);
        const int4 x = rm[0], y = rm[1];
        const int2 H = *reinterpret_cast<const int2*>(rm + 2);
        const int2 qx = make_int2(q.x, q.y), qy = make_int2(q.z, q.w);
        const long long t =
            fx_pair_t(qx, qy, make_int2(m_l.x + x.x, m_l.y + x.y), make_int2(m_l.z + x.z, m_l.w + x.w));
        const int2 T = fx_limbs(t);
        A0 += t;
        fx_mac(A1, make_int2(y.x, y.y), T);
        fx_mac(A2, make_int2(y.z, y.w), T);
        fx_mac(A3, H, qx);
        fx_mac(A4, H, qy);
        const int sl = HV == 2 ? 16 * hf + (src & 15) : src & 31;
        Tr = fx_shfl(T, sl);
        Qxr = fx_shfl(qx, sl);
        Qyr = fx_shfl(qy, sl);
    };
    auto receive = [&](int src, long long& a0, FxSum& a1, FxSum& a2, FxSum& p1, FxSum& p2) {
        const int4* rs = reinterpret_cast<const int4*>(rec + src * REC);
        const int4 y = rs[1];
        const int2 H = *reinterpret_cast<const int2*>(rs + 2);
        a0 += (long long)Tr.y * (1 << FX_LO) + Tr.x;
        fx_mac(a1, make_int2(y.x, y.y), Tr);
        fx_mac(a2, make_int2(y.z, y.w), Tr);
        fx_mac(p1, H, Qxr);
        fx_mac(p2, H, Qyr);
    };
    constexpr int UVV = 4, UVF = V == 16 ? 1 : HV == 2 ? 4 : 5;
    // (unrolled steps, swept: with more, the 16-point rules spill at 80 registers; the
    // operator entries of the 25-point rules come from memory, several at a time)
#pragma unroll (UVV)
    for (int k = 0; k < PS::SVV0; ++k) {
        const int d = 1 + k + (HV == 2 ? PS::SVV0 * hf : 0);
        int m = j + d, src = j - d;
        m -= m >= V ? V : 0;
        src += src < 0 ? V : 0;
        pair(j < V ? m : 0, qe[32 * k], src);
        Tr = fx_neg(Tr);
        Qxr = fx_neg(Qxr);
        Qyr = fx_neg(Qyr);
        receive(j < V ? src : 0, A0, A1, A2, A3, A4);
    }
#pragma unroll (UVF)
    for (int k = 0; k < PS::SVF0; ++k) {
        const int t = k + (HV == 2 ? PS::SVF0 * hf : 0);
        int f = j + t, src = j - t;
        f -= f >= L ? L : 0;
        src += src < 0 ? L : 0;
        pair(V + (f < F ? f : 0), qe[32 * (PS::SVV0 + k)], src);
        receive(src < V ? src : 0, B0, B1, B2, B3, B4);
    }
    a[0] = A0;
    a[1] = fx_value(A1);
    a[2] = fx_value(A2);
    a[3] = fx_value(A3);
    a[4] = fx_value(A4);
    b[0] = -B0;
    b[1] = -fx_value(B1);
    b[2] = -fx_value(B2);
    b[3] = -fx_value(B3);
    b[4] = -fx_value(B4);
}
// The scales of the sums of fx_diagonals: T's, and in pairs those of u_m T and v_m T and
// of Qx H_m and Qy H_m.
struct FxScales {
    int T, uT, QH;
};
__device__ __forceinline__ FxScales fx_scales(int XQx, int XQy, int XT, int Xu, int Xv, int XH) {
    return {XT, fx_pack(XT + Xu, XT + Xv), fx_pack(XQx + XH, XQy + XH)};
}
// The sums of fx_diagonals as doubles.
__device__ __forceinline__ void fx_pair_sums(const long long (&s)[5], FxScales X, bool finite, double (&x)[5]) {
    constexpr int T = FX_T, UT = FX_VAL + FX_T - 2 * FX_LO, QH = FX_PAIR + FX_VAL - 2 * FX_LO;
    fx_to<5>(s, [&](int i) {
        return i == 0 ? X.T - T : i == 1 ? fx_pack_x(X.uT) - UT : i == 2 ? fx_pack_y(X.uT) - UT
               : i == 3 ? fx_pack_x(X.QH) - QH : fx_pack_y(X.QH) - QH;
    }, x);
    if (!finite) x[0] = x[1] = x[2] = x[3] = x[4] = __longlong_as_double(0x7ff8000000000000ll);
}

// Shared-memory layout of one CTA: reference operators, then one slab per warp.
template <int N, typename real>
struct Smem {
    typedef Dims<N> D;
    // pair loop of the rules too large for the diagonals (see k_stage): the
    // NPAIR non-zero pairs, row-major, cut into 32 pieces of PL, each piece
    // touching at most PR rows; partial row sums in w_part [32][PR][4]
    static constexpr bool PIECES = !PairSched<N>::DIAG;
    static constexpr bool COMP = composed_inverse<N>();
    // node record: diagonals the limbs of hu hv u v H (48 bytes: the 128-bit
    // reads of consecutive rows fall in distinct banks); pieces h hu hv u v H rx sx ry sy 2gh
    static constexpr int REC = PIECES ? 12 : 6;
    // operators, as far as the kernel applies them (the diagonals read the
    // stored metric-averaged operator, the composed inverse its products)
    static constexpr int ops_QsT = 0;
    static constexpr int ops_Vq = ops_QsT + (PIECES ? D::Nh * D::Nh * 2 : 0);
    static constexpr int ops_VqT = ops_Vq + D::Nq * D::Np;
    static constexpr int ops_Vh = ops_VqT + (COMP ? 0 : D::Np * D::Nq);
    static constexpr int ops_VhT = ops_Vh + (COMP ? 0 : D::Nh * D::Np);
    static constexpr int ops_wf = ops_VhT + (COMP ? 0 : D::Np * D::Nh);
    static constexpr int ops_nrs = ops_wf + D::Nfq;
    static constexpr int ops_wq = ops_nrs + 2 * D::Nfq;
    static constexpr int ops_end = ((ops_wq + D::Nq) + 3) & ~3;
    // per-warp slab
    // (the row sums and the later phases take the node records' place once the
    // pair loop of the diagonals is done with them)
    static constexpr int w_rec = 0;                              // [Nh][REC]
    static constexpr int w_rt = w_rec + (PIECES ? D::Nh * REC : 0);  // [3][Nh]
    static constexpr int w_a = w_rt + 3 * D::Nh;                 // [3][Nq]
    static constexpr int w_b = w_a + 3 * D::Nq;                  // [3][Np]
    static constexpr int w_c = w_b + 3 * D::Np;                  // [3][Np]
    static constexpr int w_c_end = w_c + 3 * D::Np;
    static constexpr int w_minv = PIECES || w_c_end > D::Nh * REC ? w_c_end : D::Nh * REC;  // [NpP] (not composed)
    // Staged operators (two half-warps of rows): the element's stored pair
    // operator, then M^-1 Vh^T, then Vh M^-1 Vq^T come by bulk copies into one
    // region, each issued when the one before it has been read, so that the
    // phase in between hides the copy.
    static constexpr bool STAGED = PairSched<N>::HALVES == 2;
    static constexpr int ST_PAIR = PairSched<N>::NSTEP * 512;              // bytes
    static constexpr int ST_L = COMP ? Composed<N>::LT * 256 : 0;
    static constexpr int ST_P = COMP ? D::Nq * Composed<N>::PP * 256 : 0;
    static constexpr int ST_MAX = ST_PAIR > ST_L ? (ST_PAIR > ST_P ? ST_PAIR : ST_P) : (ST_L > ST_P ? ST_L : ST_P);
    static constexpr int w_st = ((w_minv + (D::wadg || COMP ? 0 : D::NpP)) + 3) & ~3;
    static constexpr int NPAIR = D::Nq * D::Nh + D::Nfq * D::Nq;
    static constexpr int PL = (NPAIR + 31) / 32;
    static constexpr int PR = (PL + D::Nq - 2) / D::Nq + 1;
    static constexpr int w_part = w_st + (STAGED ? ST_MAX / 8 : 0);
    static constexpr int w_end = ((w_part + (PIECES ? 32 * PR * 4 : 0)) + 3) & ~3;
    // operators, the warps' slabs, a copy barrier per warp
    static constexpr size_t bytes(int warps) {
        return sizeof(real) * (size_t(ops_end) + size_t(warps) * w_end) + 8 * size_t(warps);
    }
};

template <int N, typename real>
__device__ __forceinline__ void stage_ops_to_smem(const StageParams<real>& p, real* sm) {
    typedef Dims<N> D;
    typedef Smem<N, real> S;
    if constexpr (S::PIECES)
        for (int i = threadIdx.x; i < D::Nh * D::Nh * 2; i += blockDim.x) sm[S::ops_QsT + i] = p.QsT[i];
    for (int i = threadIdx.x; i < D::Nq * D::Np; i += blockDim.x) {
        sm[S::ops_Vq + i] = p.Vq[i];
        if constexpr (!S::COMP) sm[S::ops_VqT + i] = p.VqT[i];
    }
    if constexpr (!S::COMP)
        for (int i = threadIdx.x; i < D::Nh * D::Np; i += blockDim.x) {
            sm[S::ops_Vh + i] = p.Vh[i];
            sm[S::ops_VhT + i] = p.VhT[i];
        }
    for (int i = threadIdx.x; i < D::Nfq; i += blockDim.x) {
        sm[S::ops_wf + i] = p.wf[i];
        sm[S::ops_nrs + 2 * i] = p.nrs[2 * i];
        sm[S::ops_nrs + 2 * i + 1] = p.nrs[2 * i + 1];
    }
    for (int i = threadIdx.x; i < D::Nq; i += blockDim.x) sm[S::ops_wq + i] = p.wq[i];
}

// Weight-adjusted inverse mass (Sec. 2.8's alternative to storing the
// inverses): out = Vq^T diag(w / J) Vq y for the three fields of one element,
// y and out [3][Np] (may alias), t [3][Nq] scratch.
template <int N, typename real>
__device__ __forceinline__ void wadg_apply(const StageParams<real>& p, const real* ops, const real* y, real* t,
                                           real* out, int e, int lane, real sign) {
    typedef Dims<N> D;
    typedef Smem<N, real> S;
    const real* Vq = ops + S::ops_Vq;
    const real* VqT = ops + S::ops_VqT;
    for (int q = lane; q < D::Nq; q += 32) {
        real a0 = 0, a1 = 0, a2 = 0;
#pragma unroll
        for (int n = 0; n < D::Np; ++n) {
            const real v = Vq[q * D::Np + n];
            a0 += v * y[n];
            a1 += v * y[D::Np + n];
            a2 += v * y[2 * D::Np + n];
        }
        const real w = ops[S::ops_wq + q];
        const real sc = w * w / p.wJq[(size_t)e * D::Nq + q];
        t[q] = a0 * sc;
        t[D::Nq + q] = a1 * sc;
        t[2 * D::Nq + q] = a2 * sc;
    }
    __syncwarp();
    for (int n = lane; n < D::Np; n += 32) {
        real a0 = 0, a1 = 0, a2 = 0;
#pragma unroll 4
        for (int q = 0; q < D::Nq; ++q) {
            const real v = VqT[n * D::Nq + q];
            a0 += v * t[q];
            a1 += v * t[D::Nq + q];
            a2 += v * t[2 * D::Nq + q];
        }
        out[n] = sign * a0;
        out[D::Np + n] = sign * a1;
        out[2 * D::Np + n] = sign * a2;
    }
}

// Entropy projection of one element's modal state (in w_b, FP `real`) into
// u~ at the hybrid nodes, written to ut_out[e] (Sec. 2.6, J-weighted, Sec. 2.7).
// Pk: this lane's entries of the composed operator (global or staged), valid
// once wait() returns true; false if it gave up.
template <int N, typename real, typename Wait>
__device__ __forceinline__ bool project_element(const StageParams<real>& p, const real* ops, real* ws, int e,
                                                int lane, const int2* Pk, Wait wait) {
    typedef Dims<N> D;
    typedef Smem<N, real> S;
    typedef typename V2<real>::t real2;
    const real* Vq = ops + S::ops_Vq;
    const real* VqT = ops + S::ops_VqT;
    const real* Vh = ops + S::ops_Vh;
    real* us = ws + S::w_b;     // [3][Np] modal state
    real* ta = ws + S::w_a;     // [3][Nq]
    real* tc = ws + S::w_c;     // [3][Np]
    real* mi = ws + S::w_minv;  // [NpP]
    int bad = 0;
    // v(u_q) at volume node q with u_q = (h, a1, a2), its first entry over g:
    // (h + b) - (u^2 + v^2) / (2 g), so that v~ gives H without products by g
    auto entropy_var = [&](int q, real h, real a1, real a2, real& t0, real& t1, real& t2) {
        if (!r_positive(h)) bad |= STATUS_NONPOSITIVE;
        const real ih = real(1) / h;
        t1 = a1 * ih;
        t2 = a2 * ih;
        t0 = fma(-p.ig2, fma(t1, t1, t2 * t2), h + p.bh[(size_t)e * D::Nh + q]);
    };
    // u~ = u(v~) at hybrid node l from v~ = (a0 g, a1, a2):
    // H = a0 + (v2^2 + v3^2) / (2 g), h = H - b
    auto emit = [&](int l, real a0, real a1, real a2) {
        const real H = fma(p.ig2, fma(a1, a1, a2 * a2), a0);
        const real h = H - p.bh[(size_t)e * D::Nh + l];
        if (!r_positive(h)) bad |= STATUS_NONPOSITIVE;
        if (!r_finite(H) || !r_finite(a1) || !r_finite(a2)) bad |= STATUS_NONFINITE;
        real2* o = reinterpret_cast<real2*>(p.ut_out + ((size_t)e * D::Nh + l) * 4);
        o[0] = real2{h, a1};
        o[1] = real2{a2, H};
    };
    if constexpr (S::COMP) {
        // in block fixed point: u_q = Vq u (rows q = lane & 15 over the modes of
        // half-warp lane >> 4, or q = lane), then v~ = (Vh M^-1 Vq^T) (W J v_q), the
        // product stored per element; rows l = lane + 32 pass
        static_assert(D::Np <= 32 && D::Nq <= 32, "one lane per mode and volume node");
        const bool im = lane < D::Np, iq = lane < D::Nq;
        int X[3];
        const real u0 = im ? us[lane] : 0, u1 = im ? us[D::Np + lane] : 0, u2 = im ? us[2 * D::Np + lane] : 0;
        bool finite = fx_store<D::Np>(im, u0, u1, u2, reinterpret_cast<int2*>(tc), lane, X);
        __syncwarp();
        long long s[3];
        constexpr bool QS = D::Nq <= 16;
        const int r = QS ? lane & 15 : lane;
        const int2* V2 = reinterpret_cast<const int2*>(Vq) + (r < D::Nq ? r : 0) * D::Np +
                         (QS ? (lane >> 4) * ((D::Np + 1) / 2) : 0);
        fx_rows<D::Np, D::Np, QS>(lane, reinterpret_cast<const int2*>(tc), [&](int t) { return V2[t]; }, s);
        real t0 = 0, t1 = 0, t2 = 0, y[3];
        if (iq) {
            fx_row_values(s, X, p.xvq, finite, y);
            entropy_var(lane, y[0], y[1], y[2], t0, t1, t2);
        }
        finite = fx_store<D::Nq>(iq, t0, t1, t2, reinterpret_cast<int2*>(ta), lane, X);
        __syncwarp();
        constexpr int PP = Composed<N>::PP;
        const int XP = p.fexp[e].w;
        if (!wait()) return false;
#pragma unroll
        for (int i = 0; i < PP; ++i) {
            fx_rows<D::Nq, D::Nq, false>(lane, reinterpret_cast<const int2*>(ta),
                                         [&](int t) { return Pk[32 * (t * PP + i)]; }, s);
            if (lane + 32 * i < D::Nh) {
                fx_row_values(s, X, XP, finite, y);
                emit(lane + 32 * i, y[0], y[1], y[2]);
            }
        }
        if (bad) atomicOr(p.status, bad);
        return true;
    }
    // u_q = Vq u_h, v_q = v(u_q), scaled by w_q J_q
    auto vq_term = [&](int q, int n, real& a0, real& a1, real& a2) {
        const real v = Vq[q * D::Np + n];
        a0 += v * us[n];
        a1 += v * us[D::Np + n];
        a2 += v * us[2 * D::Np + n];
    };
    for (int q0 = 0; q0 < D::Nq; q0 += 32) {
        real a0 = 0, a1 = 0, a2 = 0;
        const int q = q0 + lane;
        if constexpr (D::Nq <= 16) {
            if (!split_rows<D::Nq, D::Np>(lane, vq_term, a0, a1, a2)) continue;
        } else {
            if (q >= D::Nq) continue;
#pragma unroll
            for (int n = 0; n < D::Np; ++n) vq_term(q, n, a0, a1, a2);
        }
        const real w = p.wJq[(size_t)e * D::Nq + q];
        real t0, t1, t2;
        entropy_var(q, a0, a1, a2, t0, t1, t2);
        ta[q] = w * t0;
        ta[D::Nq + q] = w * t1;
        ta[2 * D::Nq + q] = w * t2;
    }
    __syncwarp();
    // y = Vq^T W J v_q
    auto vqt_term = [&](int n, int q, real& a0, real& a1, real& a2) {
        const real v = VqT[n * D::Nq + q];
        a0 += v * ta[q];
        a1 += v * ta[D::Nq + q];
        a2 += v * ta[2 * D::Nq + q];
    };
    for (int n0 = 0; n0 < D::Np; n0 += 32) {
        real a0 = 0, a1 = 0, a2 = 0;
        const int n = n0 + lane;
        if constexpr (D::Np <= 16) {
            if (!split_rows<D::Np, D::Nq>(lane, vqt_term, a0, a1, a2)) continue;
        } else {
            if (n >= D::Np) continue;
#pragma unroll 5
            for (int q = 0; q < D::Nq; ++q) vqt_term(n, q, a0, a1, a2);
        }
        tc[n] = a0;
        tc[D::Np + n] = a1;
        tc[2 * D::Np + n] = a2;
    }
    __syncwarp();
    if constexpr (D::wadg) {
        // v_h = Vq^T diag(w / J) Vq y  (weight-adjusted inverse; ta is free again)
        wadg_apply<N, real>(p, ops, tc, ta, us, e, lane, real(1));
    } else {
        // v_h = (M_h^k)^{-1} y   (packed symmetric)
        auto mi_term = [&](int n, int j, real& a0, real& a1, real& a2) {
            const int ij = n >= j ? n * (n + 1) / 2 + j : j * (j + 1) / 2 + n;
            const real m = mi[ij];
            a0 += m * tc[j];
            a1 += m * tc[D::Np + j];
            a2 += m * tc[2 * D::Np + j];
        };
        for (int n0 = 0; n0 < D::Np; n0 += 32) {
            real a0 = 0, a1 = 0, a2 = 0;
            const int n = n0 + lane;
            if constexpr (D::Np <= 16) {
                if (!split_rows<D::Np, D::Np>(lane, mi_term, a0, a1, a2)) continue;
            } else {
                if (n >= D::Np) continue;
#pragma unroll
                for (int j = 0; j < D::Np; ++j) mi_term(n, j, a0, a1, a2);
            }
            us[n] = a0;   // us is free again: reuse for v_h
            us[D::Np + n] = a1;
            us[2 * D::Np + n] = a2;
        }
    }
    __syncwarp();
    // v~ = Vh v_h, then u~ = u(v~)
    for (int l = lane; l < D::Nh; l += 32) {
        real a0 = 0, a1 = 0, a2 = 0;
#pragma unroll
        for (int n = 0; n < D::Np; ++n) {
            real v = Vh[l * D::Np + n];
            a0 += v * us[n];
            a1 += v * us[D::Np + n];
            a2 += v * us[2 * D::Np + n];
        }
        emit(l, a0, a1, a2);
    }
    if (bad) atomicOr(p.status, bad);
    return true;
}

// This lane's entries of the composed projection in global memory.
template <int N, typename real>
__device__ __forceinline__ const int2* composed_pk(const StageParams<real>& p, int e, int lane) {
    return reinterpret_cast<const int2*>(p.pk) + (size_t)e * Dims<N>::Nq * Composed<N>::PP * 32 + lane;
}

template <int N, typename real>
__device__ __forceinline__ void load_minv(const StageParams<real>& p, real* ws, int e, int lane) {
    typedef Dims<N> D;
    typedef Smem<N, real> S;
    // (not read where the products with the inverse are stored)
    if constexpr (!D::wadg && !S::COMP)
        for (int i = lane; i < D::NpP; i += 32) ws[S::w_minv + i] = p.minv[(size_t)e * p.mstride + i];
}

// Standalone projection: u_in (FP64 modal) -> ut_out.
template <int N, typename real>
__global__ void __launch_bounds__(256) k_project(StageParams<real> p) {
    typedef Dims<N> D;
    typedef Smem<N, real> S;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    real* ops = reinterpret_cast<real*>(smem_raw);
    stage_ops_to_smem<N, real>(p, ops);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    real* ws = ops + S::ops_end + warp * S::w_end;
    pdl_wait();
    const int round = gridDim.x * wpb;
    for (int e0 = 0; e0 < p.K; e0 += round) {
        if (warp == 0 && e0 + round >= p.K) pdl_trigger();
        const int e = element_of(p.K, e0, warp, wpb);
        if (e >= p.K) break;
        load_minv<N, real>(p, ws, e, lane);
        for (int i = lane; i < 3 * D::Np; i += 32) {
            int c = i / D::Np, n = i - c * D::Np;
            const size_t gi = ((size_t)c * p.K + e) * D::Np + n;
            const double un = p.u_in[gi];
            ws[S::w_b + i] = (real)un;
            if (p.copy_in) {
                p.u[gi] = un;
                p.res[gi] = 0.0;
            }
        }
        __syncwarp();
        project_element<N, real>(p, ops, ws, e, lane, composed_pk<N>(p, e, lane), [] { return true; });
        __syncwarp();
    }
}

// MODE 0: write du/dt to rhs_out.  MODE 1: LSRK45 stage update of (u, res)
// followed by the entropy projection of the new state into ut_out.
template <int N, typename real, int MODE>
__device__ __forceinline__ void k_stage_body(const StageParams<real>& p) {
    typedef Dims<N> D;
    typedef Smem<N, real> S;
    typedef typename V2<real>::t real2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    real* ops = reinterpret_cast<real*>(smem_raw);
    stage_ops_to_smem<N, real>(p, ops);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    real* ws = ops + S::ops_end + warp * S::w_end;
    real* rec = ws + S::w_rec;
    real* rt = ws + S::w_rt;
    const real2* QsT = reinterpret_cast<const real2*>(ops + S::ops_QsT);
    const real g = p.g;
    const real g2 = real(2) * g;
    const real eighth = real(0.125);
    const int round = gridDim.x * wpb;
    // staged operators: the copy of this warp's region that is under way
    uint64_t* bar = reinterpret_cast<uint64_t*>(ops + S::ops_end + wpb * S::w_end) + warp;
    real* stg = ws + S::w_st;
    uint32_t parity = 0;
    auto stage_copy = [&](const real* src, int bytes) {
        fence_proxy_async_smem();  // this lane's reads of the region come before the copy's writes
        __syncwarp();
        if (lane == 0) {
            mbar_arrive_expect_tx(bar, bytes);
            tma_bulk_g2s(stg, src, bytes, bar);
        }
    };
    auto stage_wait = [&]() -> bool {
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, p.status))) return false;
        parity ^= 1;
        return true;
    };
    auto stage_pairs = [&](int e0) {  // of this warp's element in the round from e0, if it has one
        const int e = e0 < p.K ? element_of(p.K, e0, warp, wpb) : p.K;
        if (e < p.K) stage_copy(p.qxy + (size_t)e * PairSched<N>::NSTEP * 64, S::ST_PAIR);
    };
    if constexpr (S::STAGED) {
        if (lane == 0) mbar_init(bar, 1);
        fence_mbar_init();
        __syncwarp();
        stage_pairs(0);  // (constants of the problem: before the wait for the kernels before this one)
    }
    pdl_wait();
    for (int e0 = 0; e0 < p.K; e0 += round) {
        if (warp == 0 && e0 + round >= p.K) pdl_trigger();
        const int e = element_of(p.K, e0, warp, wpb);
        if (e >= p.K) break;
        // ---- the element's node records -------------------------------------------
        auto trace = [&](int l, real& h, real& u, real& v, real& H) {
            const real2* ut = reinterpret_cast<const real2*>(p.ut_in + ((size_t)e * D::Nh + l) * 4);
            const real2 a = ut[0], b = ut[1];
            h = a.x;
            u = a.y;
            v = b.x;
            H = b.y;
        };
        if constexpr (S::PIECES) {
            for (int l = lane; l < D::Nh; l += 32) {
                const real* gg = p.geo + ((size_t)e * D::Nh + l) * 4;
                real* r = rec + l * S::REC;
                real h, u, v, H;
                trace(l, h, u, v, H);
                r[0] = h;
                r[1] = h * u;
                r[2] = h * v;
                r[3] = u;
                r[4] = v;
                r[5] = H;
                r[6] = gg[0] * eighth;
                r[7] = gg[1] * eighth;
                r[8] = gg[2] * eighth;
                r[9] = gg[3] * eighth;
                r[10] = g2 * h;
            }
        } else {
            constexpr int NL = (D::Nh + 31) / 32;
            const int XQ = p.fexp[e].x;
            real hu[NL], hv[NL], u[NL], v[NL], H[NL];
            int ehu = 0, ehv = 0, eu = 0, ev = 0, eH = 0;
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int l = lane + 32 * i;
                if (l < D::Nh) {
                    real h;
                    trace(l, h, u[i], v[i], H[i]);
                    hu[i] = h * u[i];
                    hv[i] = h * v[i];
                    ehu = max(ehu, fx_exp(hu[i]));
                    ehv = max(ehv, fx_exp(hv[i]));
                    eu = max(eu, fx_exp(u[i]));
                    ev = max(ev, fx_exp(v[i]));
                    eH = max(eH, fx_exp(H[i]));
                }
            }
            ehu = fx_max(ehu);
            ehv = fx_max(ehv);
            eu = fx_max(eu);
            ev = fx_max(ev);
            eH = fx_max(eH);
            const bool finite = max(max(ehu, ehv), max(max(eu, ev), eH)) != FX_NONFINITE;
            // (a scale of its own for each velocity: the momentum equations take them apart)
            const int XQx = fx_pack_x(XQ), XQy = fx_pack_y(XQ);
            const int Xu = fx_scale(eu), Xv = fx_scale(ev), XH = fx_scale(eH);
            int Xhu = fx_scale(ehu), Xhv = fx_scale(ehv);
            const int XT = fx_align(XQx, XQy, Xhu, Xhv);
            const FxScales X = fx_scales(XQx, XQy, XT, Xu, Xv, XH);
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int l = lane + 32 * i;
                if (l < D::Nh) {
                    int2* r = reinterpret_cast<int2*>(rec + l * S::REC);
                    r[0] = fx_limbs(fx_from<FX_MOM>(hu[i], Xhu));
                    r[1] = fx_limbs(fx_from<FX_MOM>(hv[i], Xhv));
                    r[2] = fx_limbs(fx_from<FX_VAL>(u[i], Xu));
                    r[3] = fx_limbs(fx_from<FX_VAL>(v[i], Xv));
                    r[4] = fx_limbs(fx_from<FX_VAL>(H[i], XH));
                }
            }
            // (kept in the records' spare words over the pair loop, which needs the
            // registers: N = 4, K = 32768 1% faster than with them held, N = 2 and 3 collapsed 1 to 3%)
            if (lane < 2)
                reinterpret_cast<int2*>(rec + lane * S::REC)[5] = lane ? make_int2(X.QH, finite) : make_int2(X.T, X.uT);
        }
        load_minv<N, real>(p, ws, e, lane);
        __syncwarp();
        // Row sums of the flux differencing: a0 = sum T, a1 = sum u_m T and a2 =
        // sum v_m T, (p1, p2) = sum (Qx, Qy) H_m.  (u_l + u_m) T summed over m is
        // u_l (sum of T) + sum of u_m T, and the pressure 2 g h_l sum (Qx, Qy) H_m:
        // the row's own factors enter once, here.
        auto finish_row = [&](real h_l, real u_l, real v_l, real a0, real a1, real a2, real p1, real p2, real& r0,
                              real& r1, real& r2) {
            const real gh2 = g2 * h_l;
            r0 = a0 + a0;
            r1 = fma(u_l, a0, fma(gh2, p1, a1));
            r2 = fma(v_l, a0, fma(gh2, p2, a2));
        };
        // w/2 times the scaled normal of face node f, and w/2 sJ sqrt(g) (pieces: its
        // square, from the node's metrics; no array of the normals is stored)
        auto face_normal = [&](int f, real& ax, real& ay, real& as) {
            if constexpr (S::PIECES) {
                const real* r = rec + (D::Nq + f) * S::REC;
                const real w4 = real(4) * ops[S::ops_wf + f];
                const real nr = ops[S::ops_nrs + 2 * f], ns = ops[S::ops_nrs + 2 * f + 1];
                ax = w4 * (r[6] * nr + r[7] * ns);
                ay = w4 * (r[8] * nr + r[9] * ns);
                as = g * (ax * ax + ay * ay);
                return;
            }
            const real2* ff = reinterpret_cast<const real2*>(p.face + ((size_t)e * D::Nfq + f) * 4);
            const real2 a = ff[0];
            ax = a.x;
            ay = a.y;
            as = ff[1].x;
        };
        // the neighbour's trace at face node f; false at a wall
        auto neighbour = [&](int f, real& hP, real& uP, real& vP) -> bool {
            const int face = f / D::Nfp, i = f - face * D::Nfp;
            const int nb = p.nbr[(size_t)e * 3 + face];
            if ((nb & 3) == 3) return false;
            const real2* up = reinterpret_cast<const real2*>(
                p.ut_in + ((size_t)(nb >> 2) * D::Nh + D::Nq + (nb & 3) * D::Nfp + (D::Nfp - 1 - i)) * 4);
            const real2 a = up[0], b = up[1];
            hP = a.x;
            uP = a.y;
            vP = b.x;
            return true;
        };
        // Lax-Friedrichs speed sJ (|u.n| + sqrt(g h)) times w/2
        auto wave_speed = [&](real h, real u, real v, real ax, real ay, real as) {
            if constexpr (S::PIECES) return r_sqrt(as * h) + fabs(u * ax + v * ay);
            return fma(as, r_sqrt(h), fabs(u * ax + v * ay));
        };
        // interface at face node f of an element with trace (h_l, u_l, v_l): f_S(u~+, u~) with
        // the well-balanced pressure g/2 h (h+ + b), and Lax-Friedrichs with speed c (times w/2)
        // on the jump of u~
        auto add_interface = [&](int f, real h_l, real u_l, real v_l, real ax, real ay, bool wall, real hP, real uP,
                                 real vP, real c, real& r0, real& r1, real& r2) {
            if (wall) {
                // reflective wall (Sec. 2.9): h+ = h, u_n+ = -u_n, tangential kept
                const real sJw = r_sqrt(ax * ax + ay * ay);
                const real wnx = ax / sJw, wny = ay / sJw;
                const real un = u_l * wnx + v_l * wny;
                hP = h_l;
                uP = u_l - real(2) * un * wnx;
                vP = v_l - real(2) * un * wny;
            }
            const real b_l = p.bh[(size_t)e * D::Nh + D::Nq + f];
            const real hu_l = h_l * u_l, hv_l = h_l * v_l, huP = hP * uP, hvP = hP * vP;
            const real Fn = ax * (hu_l + huP) + ay * (hv_l + hvP);
            const real Fh = real(0.5) * Fn;
            const real pw = g * h_l * (hP + b_l);
            r0 += Fn;
            r1 = fma(u_l + uP, Fh, fma(ax, pw, r1));
            r2 = fma(v_l + vP, Fh, fma(ay, pw, r2));
            if (p.lf) {
                r0 -= c * (hP - h_l);
                r1 -= c * (huP - hu_l);
                r2 -= c * (hvP - hv_l);
            }
        };
        // ---- volume flux differencing and interface flux ---------------------------
        // With the pair terms and the contractions in fixed point the FP64 pipe keeps
        // 68 warp instructions per element-stage of the 439 it had at N = 4 and is 47%
        // busy; the stage waits on latencies and the serial chain of an element, with the
        // warps that the registers allow.  N = 4, K = 32768: 866 -> 261 us per stage; N = 5,
        // K = 8192: 836 -> 165 (778 in the compact form); N = 3 with forcing, K = 8192:
        // 283 -> 82.
        int Xr[3] = {0, 0, 0};  // composed inverse: rt holds limbs, scale and state of each field
        bool rfinite = true;
        if constexpr (!S::PIECES) {
            typedef PairSched<N> PS;
            constexpr int V = PS::V, F = PS::F, HV = PS::HALVES;
            const int j = HV == 2 ? lane & 15 : lane, hf = HV == 2 ? lane >> 4 : 0;
            // this lane's stored operator entries, one (Qx, Qy) per step
            const int4* qe = S::STAGED ? reinterpret_cast<const int4*>(stg) + lane
                                       : reinterpret_cast<const int4*>(p.qxy) + (size_t)e * PS::NSTEP * 32 + lane;
            if constexpr (S::STAGED)
                if (!stage_wait()) return;
            long long a[5], b[5];
            fx_diagonals<PS>(rec, qe, lane, a, b);
            const int2 x0 = reinterpret_cast<const int2*>(rec)[5], x1 = reinterpret_cast<const int2*>(rec + S::REC)[5];
            const FxScales X = {x0.x, x0.y, x1.x};
            const bool finite = x1.y != 0;
            if constexpr (S::STAGED && S::COMP)
                stage_copy(p.lk + (size_t)e * Composed<N>::LT * 32, S::ST_L);
            else if constexpr (S::STAGED)
                stage_pairs(e0 + round);
            __syncwarp();  // every lane is done with the node records
            real r0, r1, r2;
            if constexpr (HV == 2) {
                // half 0 keeps the volume rows and half 1 the face rows: lane j
                // holds row j, lane 16 + f face row V + f
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    const long long send = hf ? a[k] : b[k];
                    a[k] = (hf ? b[k] : a[k]) + __shfl_xor_sync(0xffffffffu, send, 16);
                }
                const int row = hf ? V + j : j;
                const bool valid = hf ? j < F : j < V;
                real h_l, u_l, v_l, H_l, x[5];
                trace(valid ? row : 0, h_l, u_l, v_l, H_l);
                fx_pair_sums(a, X, finite, x);
                finish_row(h_l, u_l, v_l, x[0], x[1], x[2], x[3], x[4], r0, r1, r2);
                // the wave speeds of both sides of every face node in one pass:
                // lane 16 + f its own trace, lane f the neighbour's (a wall
                // mirrors the normal velocity and keeps h: its speed is the own one)
                real ax = 0, ay = 0, as = 0, hN = 0, uN = 0, vN = 0, lam = 0;
                bool wall = false;
                if (j < F) {
                    face_normal(j, ax, ay, as);
                    real HN;
                    trace(V + j, hN, uN, vN, HN);
                    if (lane < 16) wall = !neighbour(j, hN, uN, vN);
                    if (p.lf) lam = wave_speed(hN, uN, vN, ax, ay, as);
                }
                const real hP = __shfl_sync(0xffffffffu, hN, lane & 15), uP = __shfl_sync(0xffffffffu, uN, lane & 15);
                const real vP = __shfl_sync(0xffffffffu, vN, lane & 15), lamP = __shfl_sync(0xffffffffu, lam, lane & 15);
                wall = __shfl_sync(0xffffffffu, (int)wall, lane & 15) != 0;
                if (hf && j < F)
                    add_interface(j, h_l, u_l, v_l, ax, ay, wall, hP, uP, vP, r_max_nonneg(lam, lamP), r0, r1, r2);
                if constexpr (S::COMP) {
                    rfinite = fx_store<D::Nh>(valid, r0, r1, r2, reinterpret_cast<int2*>(rt), row, Xr);
                } else if (valid) {
                    rt[row] = r0;
                    rt[D::Nh + row] = r1;
                    rt[2 * D::Nh + row] = r2;
                }
            } else {
                real h_l, u_l, v_l, H_l, x[5];
                real row[2][3] = {};  // this lane's volume row and face row
                if (lane < V) {
                    trace(lane, h_l, u_l, v_l, H_l);
                    fx_pair_sums(a, X, finite, x);
                    finish_row(h_l, u_l, v_l, x[0], x[1], x[2], x[3], x[4], row[0][0], row[0][1], row[0][2]);
                }
                if (lane < F) {
                    trace(V + lane, h_l, u_l, v_l, H_l);
                    fx_pair_sums(b, X, finite, x);
                    finish_row(h_l, u_l, v_l, x[0], x[1], x[2], x[3], x[4], r0, r1, r2);
                    real ax, ay, as, hP = h_l, uP = u_l, vP = v_l, lam = 0;
                    face_normal(lane, ax, ay, as);
                    const bool wall = !neighbour(lane, hP, uP, vP);
                    if (p.lf)
                        lam = r_max_nonneg(wave_speed(h_l, u_l, v_l, ax, ay, as), wave_speed(hP, uP, vP, ax, ay, as));
                    add_interface(lane, h_l, u_l, v_l, ax, ay, wall, hP, uP, vP, lam, r0, r1, r2);
                    row[1][0] = r0;
                    row[1][1] = r1;
                    row[1][2] = r2;
                }
                const bool in[2] = {lane < V, lane < F};
                const int at[2] = {lane, V + lane};
                if constexpr (S::COMP) {
                    rfinite = fx_store<D::Nh, 2>(in, row, reinterpret_cast<int2*>(rt), at, Xr);
                } else {
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        if (in[i])
#pragma unroll
                            for (int f = 0; f < 3; ++f) rt[f * D::Nh + at[i]] = row[i][f];
                }
            }
        } else {
            // Larger rules: the non-zero pairs (volume rows x Nh columns, then face
            // rows x Nq columns), row-major, in 32 equal pieces, one per lane; a
            // piece files its partial row sums when a row ends, and each row's
            // owner adds up the pieces of its row below.
            real* part = ws + S::w_part;
            const int p0 = lane * S::PL;
            const int p1 = p0 + S::PL < S::NPAIR ? p0 + S::PL : S::NPAIR;
            const int pp = p0 < p1 ? p0 : 0;
            int r, m, len, slot = 0;
            if (pp < D::Nq * D::Nh) {
                r = pp / D::Nh;
                m = pp - r * D::Nh;
                len = D::Nh;
            } else {
                const int q = pp - D::Nq * D::Nh;
                r = D::Nq + q / D::Nq;
                m = q - (r - D::Nq) * D::Nq;
                len = D::Nq;
            }
            const real* rl = rec + r * S::REC;
            real hu_l = rl[1], hv_l = rl[2], rx_l = rl[6], sx_l = rl[7], ry_l = rl[8], sy_l = rl[9], gh2_l = rl[10];
            real c0 = 0, c1 = 0, c2 = 0;
            for (int k = 0; k < S::PR * 4; ++k) part[lane * S::PR * 4 + k] = real(-1);
#pragma unroll 1
            for (int it = 0; it < S::PL; ++it) {
                if (p0 + it < p1) {
                    const real2 q = QsT[m * D::Nh + r];
                    const real* rm = rec + m * S::REC;
                    const real Qx = q.x * (rx_l + rm[6]) + q.y * (sx_l + rm[7]);
                    const real Qy = q.x * (ry_l + rm[8]) + q.y * (sy_l + rm[9]);
                    const real HU = hu_l + rm[1], HV = hv_l + rm[2];
                    const real T = Qx * HU + Qy * HV;
                    const real P = gh2_l * rm[5];
                    c0 += T;
                    c1 = fma(rm[3], T, fma(Qx, P, c1));
                    c2 = fma(rm[4], T, fma(Qy, P, c2));
                    if (++m == len || p0 + it + 1 == p1) {
                        real* o = part + (lane * S::PR + slot) * 4;
                        o[0] = c0;
                        o[1] = c1;
                        o[2] = c2;
                        o[3] = real(r);
                        ++slot;
                        c0 = c1 = c2 = 0;
                        if (m == len && r + 1 < D::Nh) {
                            ++r;
                            m = 0;
                            len = r < D::Nq ? D::Nh : D::Nq;
                            rl = rec + r * S::REC;
                            hu_l = rl[1]; hv_l = rl[2]; rx_l = rl[6]; sx_l = rl[7]; ry_l = rl[8]; sy_l = rl[9];
                            gh2_l = rl[10];
                        }
                    }
                }
            }
            __syncwarp();
            for (int l = lane; l < D::Nh; l += 32) {
                const real* ro = rec + l * S::REC;
                const real h_l = ro[0], u_l = ro[3], v_l = ro[4];
                real a0 = 0, a1 = 0, a2 = 0;
                // the pieces of row l, in lane order
                const int start = l < D::Nq ? l * D::Nh : D::Nq * D::Nh + (l - D::Nq) * D::Nq;
                const int rlen = l < D::Nq ? D::Nh : D::Nq;
                const int k0 = start / S::PL, k1 = (start + rlen - 1) / S::PL;
                for (int k = k0; k <= k1; ++k)
#pragma unroll
                    for (int sl = 0; sl < S::PR; ++sl) {
                        const real* o = part + (k * S::PR + sl) * 4;
                        if (o[3] == real(l)) {
                            a0 += o[0];
                            a1 += o[1];
                            a2 += o[2];
                        }
                    }
                real r0, r1, r2;
                finish_row(h_l, u_l, v_l, a0, a1, a2, real(0), real(0), r0, r1, r2);
                if (l >= D::Nq) {
                    const int f = l - D::Nq;
                    real ax, ay, as, hP = h_l, uP = u_l, vP = v_l, lam = 0;
                    face_normal(f, ax, ay, as);
                    const bool wall = !neighbour(f, hP, uP, vP);
                    if (p.lf)
                        lam = r_max_nonneg(wave_speed(h_l, u_l, v_l, ax, ay, as), wave_speed(hP, uP, vP, ax, ay, as));
                    add_interface(f, h_l, u_l, v_l, ax, ay, wall, hP, uP, vP, lam, r0, r1, r2);
                }
                rt[l] = r0;
                rt[D::Nh + l] = r1;
                rt[2 * D::Nh + l] = r2;
            }
        }
        // forcing at the volume nodes, J-weighted: added as + Vq^T W J f
        real* fa = ws + S::w_a;
        if (p.forcing) {
            for (int q = lane; q < D::Nq; q += 32) {
                // (the composed M^-1 Vq^T W J carries the weights)
                const real w = S::COMP ? real(1) : p.wJq[(size_t)e * D::Nq + q];
                real f0, f1, f2;
                mms_forcing64(p, (size_t)e * D::Nq + q, f0, f1, f2);
                fa[q] = w * f0;
                fa[D::Nq + q] = w * f1;
                fa[2 * D::Nq + q] = w * f2;
            }
        }
        __syncwarp();
        real* sc = ws + S::w_c;
        if constexpr (S::COMP) {
            // ---- M^-1 s = (M^-1 Vh^T) r - (M^-1 Vq^T) (W J f), the products stored
            // per element: rows n = lane & 15 over the columns of half-warp
            // lane >> 4, or rows n = lane
            constexpr int LT = Composed<N>::LT, GT = Composed<N>::GT;
            constexpr bool SP = Composed<N>::SPLIT;
            const int4 fe = p.fexp[e];
            long long s[3];
            const int2* Lk = S::STAGED ? reinterpret_cast<const int2*>(stg) + lane
                                       : reinterpret_cast<const int2*>(p.lk) + (size_t)e * LT * 32 + lane;
            if constexpr (S::STAGED)
                if (!stage_wait()) return;
            fx_rows<D::Nh, D::Nh, SP>(lane, reinterpret_cast<const int2*>(rt), [&](int t) { return Lk[32 * t]; }, s);
            if constexpr (S::STAGED && MODE == 1)
                stage_copy(p.pk + (size_t)e * D::Nq * Composed<N>::PP * 32, S::ST_P);
            else if constexpr (S::STAGED)
                stage_pairs(e0 + round);
            real y[3];
            fx_row_values(s, Xr, fe.y, rfinite, y);
            if (p.forcing) {
                int Xf[3];
                const bool in = lane < D::Nq;
                const real f0 = in ? fa[lane] : 0, f1 = in ? fa[D::Nq + lane] : 0, f2 = in ? fa[2 * D::Nq + lane] : 0;
                __syncwarp();  // every lane has read its values: the limbs take their place
                const bool ff = fx_store<D::Nq>(in, f0, f1, f2, reinterpret_cast<int2*>(fa), lane, Xf);
                __syncwarp();
                const int2* Gk = reinterpret_cast<const int2*>(p.gk) + (size_t)e * GT * 32 + lane;
                fx_rows<D::Nq, D::Nq, SP>(lane, reinterpret_cast<const int2*>(fa), [&](int t) { return Gk[32 * t]; }, s);
                real yf[3];
                fx_row_values(s, Xf, fe.z, ff, yf);
#pragma unroll
                for (int c = 0; c < 3; ++c) y[c] -= yf[c];
            }
            if (lane < D::Np) {
                sc[lane] = y[0];
                sc[D::Np + lane] = y[1];
                sc[2 * D::Np + lane] = y[2];
            }
        } else {
        // ---- lift: s = Vh^T r - Vq^T W J f --------------------------------------
        const real* VhT = ops + S::ops_VhT;
        const real* VqT = ops + S::ops_VqT;
        real* sb = ws + S::w_b;
        auto vht_term = [&](int n, int l, real& a0, real& a1, real& a2) {
            const real v = VhT[n * D::Nh + l];
            a0 += v * rt[l];
            a1 += v * rt[D::Nh + l];
            a2 += v * rt[2 * D::Nh + l];
        };
        auto frc_term = [&](int n, int q, real& a0, real& a1, real& a2) {
            const real v = VqT[n * D::Nq + q];
            a0 -= v * fa[q];
            a1 -= v * fa[D::Nq + q];
            a2 -= v * fa[2 * D::Nq + q];
        };
        for (int n0 = 0; n0 < D::Np; n0 += 32) {
            real a0 = 0, a1 = 0, a2 = 0;
            const int n = n0 + lane;
            if constexpr (D::Np <= 16) {
                const bool own = split_rows<D::Np, D::Nh>(lane, vht_term, a0, a1, a2);
                if (p.forcing) {
                    real f0, f1, f2;
                    split_rows<D::Np, D::Nq>(lane, frc_term, f0, f1, f2);
                    a0 += f0;
                    a1 += f1;
                    a2 += f2;
                }
                if (!own) continue;
            } else {
                if (n >= D::Np) continue;
#pragma unroll 8
                for (int l = 0; l < D::Nh; ++l) vht_term(n, l, a0, a1, a2);
                if (p.forcing)
                    for (int q = 0; q < D::Nq; ++q) frc_term(n, q, a0, a1, a2);
            }
            sb[n] = a0;
            sb[D::Np + n] = a1;
            sb[2 * D::Np + n] = a2;
        }
        __syncwarp();
        // ---- du/dt = -(M_h^k)^{-1} s; then output or RK update --------------------
        if constexpr (D::wadg) {
            wadg_apply<N, real>(p, ops, sb, fa, sc, e, lane, real(1));  // fa (forcing) is consumed
        } else {
            const real* mi = ws + S::w_minv;
            auto mi_term = [&](int n, int j, real& a0, real& a1, real& a2) {
                const int ij = n >= j ? n * (n + 1) / 2 + j : j * (j + 1) / 2 + n;
                const real m = mi[ij];
                a0 += m * sb[j];
                a1 += m * sb[D::Np + j];
                a2 += m * sb[2 * D::Np + j];
            };
            for (int n0 = 0; n0 < D::Np; n0 += 32) {
                real a0 = 0, a1 = 0, a2 = 0;
                const int n = n0 + lane;
                if constexpr (D::Np <= 16) {
                    if (!split_rows<D::Np, D::Np>(lane, mi_term, a0, a1, a2)) continue;
                } else {
                    if (n >= D::Np) continue;
#pragma unroll
                    for (int j = 0; j < D::Np; ++j) mi_term(n, j, a0, a1, a2);
                }
                sc[n] = a0;
                sc[D::Np + n] = a1;
                sc[2 * D::Np + n] = a2;
            }
        }
        }
        __syncwarp();
        for (int i = lane; i < 3 * D::Np; i += 32) {
            const int c = i / D::Np, n = i - c * D::Np;
            const size_t gi = ((size_t)c * p.K + e) * D::Np + n;
            const double r = (double)sc[i];  // du/dt = -r
            if (MODE == 0) {
                p.rhs_out[gi] = -r;
            } else {
                const double rs = p.rkA * p.res[gi] - p.dt * r;
                p.res[gi] = rs;
                const double un = p.u[gi] + p.rkB * rs;
                p.u[gi] = un;
                if (p.u_out) p.u_out[gi] = un;
                ws[S::w_b + i] = (real)un;  // the projection's input
            }
        }
        __syncwarp();
        if constexpr (MODE == 1) {
            if constexpr (S::STAGED && S::COMP) {
                if (!project_element<N, real>(p, ops, ws, e, lane, reinterpret_cast<const int2*>(stg) + lane, stage_wait))
                    return;
                stage_pairs(e0 + round);
            } else {
                project_element<N, real>(p, ops, ws, e, lane, composed_pk<N>(p, e, lane), [] { return true; });
            }
            __syncwarp();
        }
    }
}

// Blocks of WARPS warps, with a floor of MINB of them per SM for the register
// allocator (stage_min_blocks): the 16-point rules run three blocks of 8 warps at 80
// registers and small spills, in both modes; without the floor MODE 0 takes 148 and one
// block fits an SM for which the grid counts three.  A right-hand side (projection and
// stage) at N = 4, K = 2048, 8192, 32768: 52 -> 49, 137 -> 103, 353 -> 285 us; N = 3
// collapsed 49 -> 47, 129 -> 99, 335 -> 270.  Three blocks of up to FEW_WARPS warps fit at
// 148 registers too, and right-hand sides of that size keep them (K = 1152: 40 us,
// 48 at 80 registers).  The other rules: two blocks at 128 (N = 2
// 30 us of 600 faster per 10 steps at K = 128 than with three).
constexpr int FEW_WARPS = 4;
template <int N, typename real, int MODE, int MINB, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, MINB) k_stage(StageParams<real> p) {
    k_stage_body<N, real, MODE>(p);
}
template <int N>
constexpr int stage_min_blocks() {
    return Dims<N>::Nq == 16 && !Dims<N>::wadg ? 3 : 2;
}

// Warps of the blocks that problems of more than one round of 16 warps per SM
// take instead, two blocks per SM: 24 warps at 80 registers, small spills.  K =
// 2592, 5408, 12800, 32768, per stage: N = 5 75.9 -> 58.9, 123 -> 117, 253 -> 236,
// 648 -> 596 us; N = 2 collapsed 28.3 -> 23.9, 44.7 -> 42.7, 92.0 -> 88.1, 213 -> 204.
// Smaller problems do not fill 16 warps and keep the 128 registers (N = 5, K =
// 2048: 48 us, 52 at 80 registers).  0: none (the 16-point rules have 24 warps
// already; with contractions that stay in FP64 the gain was -4 to 3%; N = 1 keeps 16
// warps, 24 measure 24.5 -> 21.1 us per stage at K = 3200, 50.2 -> 49.3 at 8192, 172 -> 167
// at 32768).
template <int N>
constexpr int stage_wide_warps() {
    return Dims<N>::Nq != 16 && Dims<N>::N >= 2 && composed_inverse<N>() ? 12 : 0;
}

// FP64 diagnostics: per-CTA partial sums of (entropy, mass, entropy rate).
template <int N>
__global__ void __launch_bounds__(256) k_entropy(int K, double g, const double* __restrict__ u,
                                                 const double* __restrict__ rhs, const double* __restrict__ Vq,
                                                 const double* __restrict__ wJq, const double* __restrict__ bq,
                                                 int bq_stride, double* __restrict__ partial) {
    typedef Dims<N> D;
    double s_ent = 0, s_mass = 0, s_rate = 0;
    const size_t total = (size_t)K * D::Nq;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
        const int e = (int)(idx / D::Nq), q = (int)(idx - (size_t)e * D::Nq);
        double a[3] = {0, 0, 0}, d[3] = {0, 0, 0};
        for (int n = 0; n < D::Np; ++n) {
            const double v = Vq[q * D::Np + n];
            for (int c = 0; c < 3; ++c) {
                a[c] += v * u[((size_t)c * K + e) * D::Np + n];
                if (rhs) d[c] += v * rhs[((size_t)c * K + e) * D::Np + n];
            }
        }
        const double w = wJq[idx], b = bq[(size_t)e * bq_stride + q];
        const double h = a[0], uu = a[1] / h, vv = a[2] / h;  // (divided: one rounding, exact where u = 1)
        s_ent += w * (0.5 * (a[1] * uu + a[2] * vv) + 0.5 * g * h * h + g * h * b);
        s_mass += w * h;
        if (rhs) s_rate += w * ((g * (h + b) - 0.5 * (uu * uu + vv * vv)) * d[0] + uu * d[1] + vv * d[2]);
    }
    __shared__ double red[3][256];
    red[0][threadIdx.x] = s_ent;
    red[1][threadIdx.x] = s_mass;
    red[2][threadIdx.x] = s_rate;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s)
            for (int c = 0; c < 3; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int c = 0; c < 3; ++c) partial[blockIdx.x * 3 + c] = red[c][0];
}

// Sum the per-CTA partials in a fixed order (deterministic).
constexpr int FINALIZE_THREADS = 256;
__global__ void k_entropy_finalize(int nparts, const double* __restrict__ partial, double* __restrict__ out);

}  // namespace esdg
