// Expected-emission operator and its adjoint (see pcc.h).
//
// Per cell c with plasma parameters theta = (n_i, T_e, Z*, s_TF, s_D) and
// electron samples (gamma_s, w_s), for ions at rest:
//   R_gamma = n_i sum_s w_s v_s sigma_B(gamma_s)          (rate form of Eq. N_br_theo1)
//   R_pair  = n_i sum_s w_s v_s sigma_T(gamma_s)          (Sec. II.D fit)
//   P_rad   = n_i sum_s w_s v_s int k dsigma_B/dk dk      (radiative stopping power, Sec. III.B)
// where the k-integrals run over x = k/(gamma-1) in [1e-7, 1] by one n-point
// Gauss-Legendre panel in ln x.  dsigma/dk is Eq. (cs_br_nr) with the Elwert
// factor for gamma <= 2, Eq. (csre) for 2 < gamma <= 100 and Eq. (csur)
// above, with the screening of Sec. II.A.
//
// Work.  A block takes a cell.  Its samples are sorted into relativistic and
// non-relativistic ones, 32 to a warp, and the (chunk of samples, node) pairs are
// dealt out evenly to the warps: a lane keeps its sample's factors in registers
// and walks the nodes, whose x = exp(l), 1 - x, 1/x and weight come from the
// host (in double) through the constant bank.  With a warp per sample and the
// lanes over the nodes, the per-sample factors, the compensated sums and the
// pair rate cost as much as the nodes, and a lane evaluated exp and expm1 of the
// same few numbers for every sample.  4096 cells x 512 samples x 64 nodes:
// forward 2.05 -> 0.53 ms, adjoint 2.91 -> 0.85 ms, bound by FP32 issue.
//
// Precision.  Nodes run in FP32.  The printed closed form of I2 (Eq. deriv_I2)
// cancels terms of size (L delta)^2 ln L down to O(1), which destroys FP32 once
// L delta >> 1 (L_R is 45 to 10^4 here).  For u = L delta > 1 it is evaluated in a
// rearranged form with no such cancellation: with rho = L^2/(1+L^2),
// z = L(1-delta)/(1+L u), g(z) = z - atan z,
//   2 I2 = -2 ln d - 6 u^2 ln d/(1+L^2) + (1+3u^2)(log1p(L^-2) - log1p(u^-2))
//          + 4 u^3 g(z) + 4 u^2 (1-d)/(1+u L) - 4 u^2 (1-d)/(1+L^2) + rho (d^2-1)
// (the same function), and atan L - atan u is atan(z) in both forms.  The arc
// tangent takes the smaller of z and 1/z, the logarithm the smaller of u^2 and
// 1/u^2, through polynomials fitted on [0, 1] (Chebyshev fits of degree 8 and 9,
// 8e-8 and 9e-8 relative including the rounding; the first gives g(z) without
// cancellation); divisions are a reciprocal and one Newton step.  Non-
// relativistic nodes (gamma <= 2) use q_+^2 - q_-^2 = 4 p1 p2, so that the
// logarithms of the Yukawa terms are those of the cross term, or FP64 in cells
// where L_D is within 5 % of L_TF, where the cross term's divided difference
// cancels (or where a length is beyond 1e15).  Sums over a lane's nodes and samples are compensated FP32, over
// lanes and warps FP64.
//
// Adjoint.  The parameters enter only through the screening quantities
// (L_R for gamma > 2; L_TF, L_D and eta_D = Z*/Z = 1 - eta_TF for gamma <= 2)
// and the n_i prefactor.  The adjoint kernel carries the derivatives of the node
// integrands with respect to those four quantities, written out by hand (dual
// numbers in the FP64 branch), reduces them per cell, and contracts them with grad_out through the
// analytic Jacobian of the screening quantities:
//   L_TF = s_TF Z^(-1/3)/alpha,  L_D = s_D max(lambda_D, r_i)/r_C,
//   a = I_TFD, h(x) = ln(1+x) - x/(1+x), h(L_R^2) = 2a  =>  dL_R/da = (1+L_R^2)^2/L_R^3.
#include <algorithm>
#include <cmath>
#include <vector>

#include "pcc_internal.h"
#include "pcc_physics.cuh"

namespace {

using namespace pcc;

constexpr int kMaxQuad = 128;
constexpr int kEmThreads = 256;
constexpr int kEmWarps = kEmThreads / 32;

// ---------------------------------------------------------------- duals ---
template <typename T, int N>
struct Dual {
    T v;
    T d[N];
};

template <typename T> __device__ __forceinline__ T val(T x) { return x; }
template <typename T, int N> __device__ __forceinline__ T val(const Dual<T, N>& x) { return x.v; }

template <typename T, int N>
__device__ __forceinline__ Dual<T, N> mk(T v)
{
    Dual<T, N> r;
    r.v = v;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = T(0);
    return r;
}

#define DUAL_BIN(OP, DV)                                                                                  \
    template <typename T, int N>                                                                          \
    __device__ __forceinline__ Dual<T, N> operator OP(const Dual<T, N>& a, const Dual<T, N>& b)           \
    {                                                                                                     \
        Dual<T, N> r;                                                                                     \
        r.v = a.v OP b.v;                                                                                 \
        _Pragma("unroll") for (int i = 0; i < N; ++i) r.d[i] = DV;                                        \
        return r;                                                                                         \
    }
DUAL_BIN(+, a.d[i] + b.d[i])
DUAL_BIN(-, a.d[i] - b.d[i])
DUAL_BIN(*, a.d[i] * b.v + a.v * b.d[i])
#undef DUAL_BIN

template <typename T, int N>
__device__ __forceinline__ Dual<T, N> operator/(const Dual<T, N>& a, const Dual<T, N>& b)
{
    Dual<T, N> r;
    const T ib = T(1) / b.v;
    r.v = a.v * ib;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = (a.d[i] - r.v * b.d[i]) * ib;
    return r;
}

template <typename T, int N>
__device__ __forceinline__ Dual<T, N> operator-(const Dual<T, N>& a)
{
    Dual<T, N> r;
    r.v = -a.v;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = -a.d[i];
    return r;
}

// mixed with a plain scalar
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> operator+(const Dual<T, N>& a, T b) { Dual<T, N> r = a; r.v += b; return r; }
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> operator+(T b, const Dual<T, N>& a) { return a + b; }
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> operator-(const Dual<T, N>& a, T b) { Dual<T, N> r = a; r.v -= b; return r; }
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> operator-(T b, const Dual<T, N>& a) { return -a + b; }
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> operator*(const Dual<T, N>& a, T b)
{
    Dual<T, N> r;
    r.v = a.v * b;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * b;
    return r;
}
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> operator*(T b, const Dual<T, N>& a) { return a * b; }
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> operator/(T a, const Dual<T, N>& b)
{
    Dual<T, N> r;
    const T ib = T(1) / b.v;
    r.v = a * ib;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = -r.v * b.d[i] * ib;
    return r;
}
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> operator/(const Dual<T, N>& a, T b) { return a * (T(1) / b); }

// chain rule for a scalar function with value f and derivative df at a.v
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> chain(const Dual<T, N>& a, T f, T df)
{
    Dual<T, N> r;
    r.v = f;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * df;
    return r;
}

__device__ __forceinline__ double f_log1p(double x) { return log1p(x); }
__device__ __forceinline__ double f_log(double x) { return log(x); }

template <typename T, int N>
__device__ __forceinline__ Dual<T, N> f_log1p(const Dual<T, N>& a) { return chain(a, f_log1p(a.v), T(1) / (T(1) + a.v)); }
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> f_log(const Dual<T, N>& a) { return chain(a, f_log(a.v), T(1) / a.v); }

// -------------------------------------------- non-relativistic (FP64) ----
// g of Eq. (cs_br_nr).
template <typename R>
__device__ __forceinline__ R nr_g_t(double qp, double qm, R eta, R L)
{
    const R L2 = L * L;
    const R Dp = 1.0 + (qp * qp) * L2, Dm = 1.0 + (qm * qm) * L2;
    return 0.5 * (eta * eta) * (f_log1p(((qp * qp - qm * qm) * L2) / Dm) + 1.0 / Dp - 1.0 / Dm);
}

// Gamma_c of Eq. (cs_br_nr), midpoint limit when L_D ~ L_TF.
template <typename R>
__device__ __forceinline__ R nr_cross_t(double qp, double qm, R eTF, R LTF, R eD, R LD)
{
    const R A = LTF * LTF, B = LD * LD;
    const R d = B - A;
    if (fabs(val(d)) <= 1e-6 * fmax(val(A), val(B))) {
        const R M = 0.5 * (A + B);
        const R Mp = 1.0 + (qp * qp) * M, Mm = 1.0 + (qm * qm) * M;
        return eTF * eD * (f_log(Mp / Mm) + 1.0 / Mp - 1.0 / Mm);
    }
    const R Tp = 1.0 + (qp * qp) * A, Tm = 1.0 + (qm * qm) * A;
    const R Dp = 1.0 + (qp * qp) * B, Dm = 1.0 + (qm * qm) * B;
    return eTF * eD / d * (A * f_log(Dm / Dp) + B * f_log(Tp / Tm));
}

// ---------------------------------------------------------------- cells ---
// What the relativistic nodes need of L_R alone, rounded from FP64: in FP32
// these shared factors put the same error on every node of the cell (they were
// the larger part of the gradient's).
struct RelCell {
    // 1/L, 1/(1+L^2), L^2/(1+L^2) and its derivative, ln(1+L^2) in two parts, ln(1+L^-2)
    float L, iL, i1L2, rho, rhop, ln1L2, ln1L2_lo, l1pi;
};

constexpr double kNrMax = 1e30;   // largest L^2 of the FP32 non-relativistic nodes (12 L^2 is a normal float)

struct CellScreen {
    double LTF, LD, etaTF, etaD, a, LR;
    double n_i, T_e, Zs, sTF, sD;
    RelCell rel;
    // derivatives of L_R through a = I_TFD (adjoint only)
    double LR_eD, LR_LTF, LR_LD;
    bool debye;   // lambda_D > r_i (the Debye branch of L_D is active)
    bool nr32;    // L_D and L_TF far enough apart, and small enough, for the FP32 non-relativistic branch
    bool ok;
};

__device__ CellScreen cell_screen(const float* p, int Z)
{
    CellScreen c;
    c.n_i = p[0]; c.T_e = p[1]; c.Zs = p[2]; c.sTF = p[3]; c.sD = p[4];
    c.ok = c.n_i > 0.0 && c.T_e >= 0.0 && c.Zs >= 0.0 && c.Zs <= Z && c.sTF > 0.0 && c.sD > 0.0 &&
           isfinite(c.n_i) && isfinite(c.T_e);
    if (!c.ok) return c;
    c.LTF = c.sTF * exp(-log((double)Z) / 3.0) / kAlpha;
    const double ri = cbrt(3.0 / (4.0 * kPi * c.n_i));
    if (c.Zs > 0.0) {
        const double lam = sqrt(kEps0 * c.T_e / (kQe * c.n_i * c.Zs * (c.Zs + 1.0)));
        c.debye = lam > ri;
        c.LD = c.sD * fmax(lam, ri) / kRc;
    } else {
        // Z* = 0: Eq. LDH gives lambda_D = infinity.  Nothing depends on L_D
        // then (eta_D = 0), and the derivative with respect to Z* is the limit
        // from Z* > 0, in which the cross terms take their L_D -> infinity
        // values.  A finite stand-in 1e5 L_TF gives those limits to ~1e-9
        // and keeps every FP32 product of the non-relativistic duals finite.
        c.debye = false;
        c.LD = 1e5 * c.LTF;
    }
    c.etaD = c.Zs / Z;
    c.etaTF = 1.0 - c.etaD;
    c.a = i_tfd(c.etaTF, c.LTF, c.etaD, c.LD);
    const double w = lambert_w0_neg(-exp(-1.0 - 2.0 * c.a));
    c.LR = sqrt(expm1(w + 1.0 + 2.0 * c.a));
    const double A = c.LTF * c.LTF, B = c.LD * c.LD;
    c.nr32 = fabs(B - A) > 0.05 * fmax(A, B) && fmax(A, B) < kNrMax;
    const double x = c.LR * c.LR, ix = 1.0 / (1.0 + x);
    const double ln = log1p(x);
    c.rel = RelCell{(float)c.LR, (float)(1.0 / c.LR), (float)ix, (float)(x * ix), (float)(2.0 * c.LR * ix * ix),
                    (float)ln, (float)(ln - (float)ln), (float)log1p(1.0 / x)};
    return c;
}

// dL_R/d(eta_D, L_TF, L_D) through a = I_TFD(eta_TF, L_TF, eta_D, L_D).
__device__ void screen_jacobian(CellScreen& c)
{
    const double A = c.LTF * c.LTF, B = c.LD * c.LD;
    const double lA = log1p(A), lB = log1p(B);
    const double hA = lA - A / (1.0 + A), hB = lB - B / (1.0 + B);
    const double hpA = A / ((1.0 + A) * (1.0 + A)), hpB = B / ((1.0 + B) * (1.0 + B));
    double X, XA, XB;
    const double D = B - A;
    if (fabs(D) <= 1e-4 * fmax(A, B)) {
        const double M = 0.5 * (A + B);
        X = log1p(M) - M / (1.0 + M);
        XA = XB = 0.5 * M / ((1.0 + M) * (1.0 + M));
    } else {
        const double N = B * lA - A * lB;
        X = N / D;
        XA = ((B / (1.0 + A) - lB) * D + N) / (D * D);
        XB = ((lA - A / (1.0 + B)) * D - N) / (D * D);
    }
    const double eT = c.etaTF, eDv = c.etaD;
    const double x = c.LR * c.LR, dLR_da = (1.0 + x) * (1.0 + x) / (x * c.LR);
    c.LR_eD = dLR_da * (-eT * hA + eDv * hB + (eT - eDv) * X);
    c.LR_LTF = dLR_da * (0.5 * eT * eT * hpA + eT * eDv * XA) * 2.0 * c.LTF;
    c.LR_LD = dLR_da * (0.5 * eDv * eDv * hpB + eT * eDv * XB) * 2.0 * c.LD;
}

// Screening quantities of every cell, one thread per cell (FP64).
template <bool GRAD>
__global__ void screen_kernel(const float* __restrict__ params, int n_cells, int Z, CellScreen* __restrict__ out)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n_cells) return;
    CellScreen s = cell_screen(params + 5 * (size_t)c, Z);
    if (GRAD && s.ok) screen_jacobian(s);
    out[c] = s;
}

struct EmArgs {
    int n_cells, n_samples, Z, n_quad;
    double fC;          // Coulomb correction f_C(Z)
    const float* params;
    const float* gamma;
    const float* w;
    const float* grad_out;
    float* out;
    DevStats* st;
    const CellScreen* screen;   // per-cell screening, computed by screen_kernel
    // nodes: x, 1 - x, half-width times weight h, ln x; h x and 1/x
    float4 node[kMaxQuad];
    float2 node2[kMaxQuad];
};

// Per-lane accumulators: value sums of sigma and k sigma, and their
// tangents with respect to L_R (relativistic) and (L_TF, L_D, eta_D) (NR).
struct Acc {
    Kahan r, p;
    Kahan r_LR, p_LR;
    double r_nr[3], p_nr[3];
};

// 1/x for normal x: the hardware reciprocal and one Newton step.
__device__ __forceinline__ float rcp_nr(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(r, fmaf(-x, r, 1.0f), r);
}

// t^3 P(t^2) = atan t - t on [0, 1].
__device__ __forceinline__ float atan_tail(float t, float t2)
{
    float p = -2.4470311891e-03f;
    p = fmaf(p, t2, 1.3750284160e-02f);
    p = fmaf(p, t2, -3.6270174200e-02f);
    p = fmaf(p, t2, 6.2843609111e-02f);
    p = fmaf(p, t2, -8.6731708692e-02f);
    p = fmaf(p, t2, 1.1037994282e-01f);
    p = fmaf(p, t2, -1.4279110916e-01f);
    p = fmaf(p, t2, 1.9999765999e-01f);
    p = fmaf(p, t2, -3.3333331951e-01f);
    return p * t2 * t;
}

// ln(1 + s) on [0, 1].
__device__ __forceinline__ float log1p_unit(float s)
{
    float p = 2.8738837408e-03f;
    p = fmaf(p, s, -1.7512242810e-02f);
    p = fmaf(p, s, 4.9931181021e-02f);
    p = fmaf(p, s, -9.2029632547e-02f);
    p = fmaf(p, s, 1.3071328270e-01f);
    p = fmaf(p, s, -1.6378508865e-01f);
    p = fmaf(p, s, 1.9959356165e-01f);
    p = fmaf(p, s, -2.4997024128e-01f);
    p = fmaf(p, s, 3.3333247560e-01f);
    p = fmaf(p, s, -4.9999999588e-01f);
    return fmaf(p * s, s, s);
}

// Compensated sum of products a b.
struct KahanProd {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float a, float b)
    {
        const float y = fmaf(a, b, -c), t = s + y;
        c = (t - s) - y;
        s = t;
    }
};

// Nodes [q0, q1) of one relativistic sample (per lane).
template <bool GRAD>
__device__ __forceinline__ void rel_nodes(const EmArgs& a, const RelCell& L, float g, float w3, float fC, int q0, int q1,
                                          Acc& acc)
{
    const float T = g - 1.0f, ig = rcp_nr(g), cd = 0.5f * T * ig, icd = 2.0f * g * rcp_nr(T), lc = logf(cd);
    // three times the bracket, so that no factor 2/3 is rounded the same way for every node
    const float fc = g > 100.0f ? fC : 0.0f, fc1 = 1.0f - fc, fc2 = 5.0f / 3.0f - 2.0f * fc;
    const float bw = w3 / 3.0f;
    KahanProd sr, sp, dr, dp;
#pragma unroll 1
    for (int q = q0; q < q1; ++q) {
        const float4 nd = a.node[q];
        const float2 ne = a.node2[q];
        const float gk = fmaf(T, nd.y, 1.0f);                      // gamma - k
        const float d = nd.x * cd * rcp_nr(gk);                    // k / (2 gamma (gamma - k))
        const float eps = gk * ig, omd = 1.0f - d;
        const float u = L.L * d, u2 = u * u;
        const float num = L.L * omd, den = fmaf(L.L, u, 1.0f);
        const bool swap = num > den;
        const float h = rcp_nr(swap ? num : den), t = (swap ? den : num) * h, t2 = t * t;
        const float tail = atan_tail(t, t2), at = t + tail;
        const float A = swap ? 1.57079632679f - at : at;           // atan L - atan u
        const float lnd = (nd.w + lc) - __logf(gk);
        const float qd = L.rho * omd;
        float lnr, tI2, lnrp = 0.f, Ap = 0.f, tI2p = 0.f;
        const float iu1 = GRAD ? rcp_nr(1.0f + u2) : 0.f;
        if (u <= 1.0f) {
            const float v = fmaf(4.0f, u2, -1.0f - d);
            lnr = (L.ln1L2 - log1p_unit(u2)) + L.ln1L2_lo;
            tI2 = -4.0f * u2 * u * A + fmaf(3.0f, u2, 1.0f) * lnr + 6.0f * lnd * u2 * L.rho + qd * v;
            if (GRAD) {
                Ap = L.i1L2 - d * iu1;
                lnrp = 2.0f * (L.L * L.i1L2 - u * d * iu1);
                tI2p = -4.0f * u2 * (3.0f * d * A + u * Ap) + 6.0f * u * d * lnr + fmaf(3.0f, u2, 1.0f) * lnrp +
                       6.0f * lnd * u * (2.0f * d * L.rho + u * L.rhop) + omd * (v * L.rhop + 8.0f * L.rho * u * d);
            }
        } else {   // here z = t < 1 and h = 1/(1 + L u)
            const float iu = ne.y * icd * gk * L.iL;
            const float l = L.l1pi - log1p_unit(iu * iu), gz = -tail, hd = h - L.i1L2;
            lnr = l - 2.0f * lnd;
            tI2 = -2.0f * lnd - 6.0f * lnd * u2 * L.i1L2 + fmaf(3.0f, u2, 1.0f) * l + 4.0f * u2 * u * gz +
                  4.0f * omd * u2 * hd - qd * (1.0f + d);
            if (GRAD) {
                lnrp = 2.0f * L.iL * (iu1 - L.i1L2);
                const float zp = h * (omd - 2.0f * u * t);
                Ap = zp * rcp_nr(1.0f + t2);
                tI2p = -12.0f * lnd * u * d * L.i1L2 * L.i1L2 + 6.0f * u * d * l + fmaf(3.0f, u2, 1.0f) * lnrp +
                       4.0f * u2 * (3.0f * d * gz + u * Ap * t2) + 8.0f * omd * u * d * hd +
                       4.0f * omd * u2 * (L.rhop - 2.0f * u * h * h) - omd * (1.0f + d) * L.rhop;
            }
        }
        const float I1 = -u * A - 0.5f * qd * omd + 0.5f * lnr;
        const float c1 = fmaf(3.0f * eps, eps, 3.0f);
        float f = c1 * (I1 + fc1) - eps * (tI2 + fc2), df = 0.f;
        if (GRAD) {
            const float I1p = -d * A - u * Ap - 0.5f * omd * omd * L.rhop + 0.5f * lnrp;
            df = c1 * I1p - eps * tI2p;
        }
        if (!(f > 0.0f)) { f = 0.0f; df = 0.0f; }
        const float hk = ne.x * T;
        sr.add(nd.z, f);
        sp.add(hk, f);
        if (GRAD) { dr.add(nd.z, df); dp.add(hk, df); }
    }
    acc.r.add(bw * (sr.s - sr.c));
    acc.p.add(bw * (sp.s - sp.c));
    if (GRAD) {
        acc.r_LR.add(bw * (dr.s - dr.c));
        acc.p_LR.add(bw * (dp.s - dp.c));
    }
}

// What the non-relativistic nodes need of the screening.
struct NrCell {
    float A, B, iBA, eT, eD, LTF2, LD2;   // L_TF^2, L_D^2, 1/(B - A), eta_TF, eta_D, 2 L_TF, 2 L_D
    float kA, kB;                         // B/(B - A) 2 L_TF, A/(B - A) 2 L_D
};

// Nodes [q0, q1) of one sample with gamma <= 2 (per lane), Eq. (cs_br_nr) with the
// Elwert factor, where L_D and L_TF differ by more than 5 %.  With
// P = q+^2 - q-^2 = 4 p1 p2 exactly, T-+ = 1 + q-+^2 A, D-+ = 1 + q-+^2 B,
// la = ln(T+/T-) = log1p(P A / T-), lb likewise, the bracket is
//   eta_TF^2/2 (la - P A/(T+ T-)) + eta_D^2/2 (lb - P B/(D+ D-)) + eta_TF eta_D X,
//   X = (B la - A lb)/(B - A),
//   dX/dA = B (P/(T+ T-) - (lb - la)/(B - A))/(B - A), dX/dB = A ((lb - la)/(B - A) - P/(D+ D-))/(B - A):
// no difference of nearly equal numbers is formed.  Every factor has a reciprocal
// of its own: B reaches 1e22 in thin plasmas (and kNrMax), and the product D+ D-
// passes the FP32 range from L_D = 1e9 on.
template <bool GRAD>
__device__ __forceinline__ void nr_nodes(const EmArgs& a, const NrCell& C, float g, float bw, int q0, int q1, Acc& acc)
{
    const float T1 = g - 1.0f, p1 = sqrtf(T1 * (T1 + 2.0f)), b1 = p1 / g;
    const float az = 2.0f * (float)kPi * (float)a.Z * (float)kAlpha;
    const float pre1 = 4.0f / (3.0f * p1 * p1) * b1 * -expm1f(-az / b1);
    KahanProd sr, sp, dr[3], dp[3];
#pragma unroll 1
    for (int q = q0; q < q1; ++q) {
        const float4 nd = a.node[q];
        const float hx = a.node2[q].x;
        const float k = nd.x * T1, T2 = T1 * nd.y;
        if (!(k > 0.f && T2 > 0.f)) continue;
        const float p2 = sqrtf(T2 * (T2 + 2.0f));
        const float qm = k * (T1 + T2 + 2.0f) * rcp_nr(p1 + p2), qm2 = qm * qm, P = 4.0f * p1 * p2, qp2 = qm2 + P;
        const float ib2 = (1.0f + T2) * rcp_nr(p2);
        const float pre = pre1 * ib2 * rcp_nr(-expm1f(-az * ib2));
        const float Tm = fmaf(qm2, C.A, 1.0f), Tp = fmaf(qp2, C.A, 1.0f), Dm = fmaf(qm2, C.B, 1.0f), Dp = fmaf(qp2, C.B, 1.0f);
        const float iTm = rcp_nr(Tm), iTp = rcp_nr(Tp), iDm = rcp_nr(Dm), iDp = rcp_nr(Dp);
        const float ya = P * C.A * iTm, yb = P * C.B * iDm;   // T+/T- - 1, D+/D- - 1
        const float la = log1pf(ya), lb = log1pf(yb);
        const float gT = la - ya * iTp, gD = lb - yb * iDp, X = (C.B * la - C.A * lb) * C.iBA;
        float f = pre * (0.5f * C.eT * C.eT * gT + 0.5f * C.eD * C.eD * gD + C.eT * C.eD * X);
        float df[3];
        if (GRAD) {
            const float dl = (lb - la) * C.iBA;
            const float dgT = C.LTF2 * iTp * ya * (qm2 * iTm + qp2 * iTp), dgD = C.LD2 * iDp * yb * (qm2 * iDm + qp2 * iDp);
            df[0] = pre * (0.5f * C.eT * C.eT * dgT + C.eT * C.eD * (C.kA * (P * iTm * iTp - dl)));
            df[1] = pre * (0.5f * C.eD * C.eD * dgD + C.eT * C.eD * (C.kB * (dl - P * iDm * iDp)));
            df[2] = pre * (-C.eT * gT + C.eD * gD + (C.eT - C.eD) * X);
        }
        if (f <= 0.f) {
            f = 0.f;
            if (GRAD) df[0] = df[1] = df[2] = 0.f;
        }
        const float hk = hx * T1;
        sr.add(nd.z, f);
        sp.add(hk, f);
        if (GRAD)
#pragma unroll
            for (int i = 0; i < 3; ++i) { dr[i].add(nd.z, df[i]); dp[i].add(hk, df[i]); }
    }
    acc.r.add(bw * (sr.s - sr.c));
    acc.p.add(bw * (sp.s - sp.c));
    if (GRAD)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            acc.r_nr[i] += (double)(bw * (dr[i].s - dr[i].c));
            acc.p_nr[i] += (double)(bw * (dp[i].s - dp[i].c));
        }
}

// One sample with gamma <= 2 in a cell where L_D is near L_TF, in FP64, a warp per
// sample and the lanes over the nodes.  Out of line: it would take the registers
// of the common paths.  Returns the lane's sums times bw.
struct NrSums { double r, p, dr[3], dp[3]; };
template <bool GRAD>
__device__ __noinline__ NrSums nr_sample(const EmArgs* ap, double g, double bw, const CellScreen* csp, int lane)
{
    const EmArgs& a = *ap;
    const CellScreen cs = *csp;
    const double T1 = g - 1.0, p1 = sqrt(T1 * (T1 + 2.0)), b1 = p1 / g;
    const double Z = a.Z, az = 2.0 * kPi * Z * kAlpha;
    double sr = 0.0, sp = 0.0, dr[3] = {0, 0, 0}, dp[3] = {0, 0, 0};
    for (int q = lane; q < a.n_quad; q += 32) {
        const double l = a.node[q].w;
        const double x = exp(l), k = x * T1;
        const double T2 = T1 * (-expm1(l));
        if (!(k > 0.0 && T2 > 0.0)) continue;
        const double p2 = sqrt(T2 * (T2 + 2.0));
        const double qp = p1 + p2, qm = k * (T1 + T2 + 2.0) / (p1 + p2);
        const double b2 = p2 / (1.0 + T2);
        const double fE = (b1 / b2) * (-expm1(-az / b1)) / (-expm1(-az / b2));
        // f / (4 Z^2 r_e^2 alpha) = 4/(3 p1^2) * bracket * f_E
        const double pre = 4.0 / (3.0 * p1 * p1) * fE;
        double fv;
        double fd[3] = {0, 0, 0};
        if (GRAD) {
            Dual<double, 3> LTF = mk<double, 3>(cs.LTF), LD = mk<double, 3>(cs.LD);
            Dual<double, 3> eD = mk<double, 3>(cs.etaD), eTF = mk<double, 3>(cs.etaTF);
            LTF.d[0] = 1.0; LD.d[1] = 1.0; eD.d[2] = 1.0; eTF.d[2] = -1.0;
            const Dual<double, 3> br = nr_g_t(qp, qm, eTF, LTF) + nr_g_t(qp, qm, eD, LD) +
                                       nr_cross_t(qp, qm, eTF, LTF, eD, LD);
            fv = pre * br.v;
            for (int i = 0; i < 3; ++i) fd[i] = pre * br.d[i];
        } else {
            const double br = nr_g_t(qp, qm, cs.etaTF, cs.LTF) + nr_g_t(qp, qm, cs.etaD, cs.LD) +
                              nr_cross_t(qp, qm, cs.etaTF, cs.LTF, cs.etaD, cs.LD);
            fv = pre * br;
        }
        if (!(fv > 0.0)) { fv = 0.0; fd[0] = fd[1] = fd[2] = 0.0; }
        const double h = a.node[q].z;
        sr += h * fv;
        sp += h * fv * k;
        if (GRAD)
            for (int i = 0; i < 3; ++i) { dr[i] += h * fd[i]; dp[i] += h * fd[i] * k; }
    }
    NrSums o;
    o.r = bw * sr;
    o.p = bw * sp;
    for (int i = 0; i < 3; ++i) { o.dr[i] = bw * dr[i]; o.dp[i] = bw * dp[i]; }
    return o;
}

// Sums per cell, in units of 4 Z^2 r_e^2 alpha c (rates) and m_e c^2 (power):
// [0] sum w beta sigma, [1] sum w beta k-sigma, [2] sum w v sigma_T (SI),
// [3] d[0]/dL_R, [4] d[1]/dL_R, [5..7] d[0]/d(L_TF, L_D, eta_D), [8..10] d[1]/d(...)
constexpr int kSums = 11;

// The pairs (chunk of 32 listed samples, node) of a list, dealt out evenly to the
// block's warps as runs of nodes: work(sample, q0, q1) per lane.
template <typename F>
__device__ __forceinline__ void deal_nodes(int n, int n_quad, F work)
{
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int total = ((n + 31) >> 5) * n_quad;
    int e = total * wid / kEmWarps;
    const int end = total * (wid + 1) / kEmWarps;
    while (e < end) {   // warp-uniform
        const int chunk = e / n_quad, q0 = e - chunk * n_quad, q1 = min(n_quad, q0 + end - e);
        const int i = 32 * chunk + lane;
        if (i < n) work(i, q0, q1);
        e += q1 - q0;
    }
}

template <bool GRAD>
__global__ void __launch_bounds__(kEmThreads, GRAD ? 3 : 4) emission_kernel(const __grid_constant__ EmArgs a)
{
    constexpr int kOut = GRAD ? kSums : 3;
    __shared__ double part[kOut][kEmThreads];
    __shared__ float2 list[2][kEmThreads];       // (gamma, w beta) of the batch: relativistic, non-relativistic
    __shared__ int count[2][kEmWarps];
    const int c = blockIdx.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const CellScreen& cs = a.screen[c];
    if (!cs.ok) {
        if (threadIdx.x == 0) {
            raise_status(a.st, PCC_ST_NONFINITE);
            const float nan = __int_as_float(0x7fc00000);
            if (GRAD) for (int k = 0; k < 5; ++k) a.out[5 * (size_t)c + k] = nan;
            else for (int k = 0; k < 3; ++k) a.out[3 * (size_t)c + k] = nan;
        }
        return;
    }
    Acc acc;
    for (int i = 0; i < 3; ++i) acc.r_nr[i] = acc.p_nr[i] = 0.0;
    Kahan pair;
    const RelCell L = cs.rel;
    const bool nr32 = cs.nr32;
    const float* gs = a.gamma + (size_t)c * a.n_samples;
    const float* ws = a.w + (size_t)c * a.n_samples;
    for (int s0 = 0; s0 < a.n_samples; s0 += kEmThreads) {
        const int s = s0 + threadIdx.x;
        const float g = s < a.n_samples ? gs[s] : 0.f, wt = s < a.n_samples ? ws[s] : 0.f;
        const bool on = g > 1.0f && wt != 0.0f;                   // at rest or no weight: no emission
        const int nr = on && g <= 2.0f ? 1 : 0;
        float bw = 0.f;
        if (on) {
            const float T = g - 1.0f;
            bw = wt * (sqrtf(T * (T + 2.0f)) / g);                // w beta, FP32 (the FP64 units are scarce)
            if (g >= 3.0f) pair.add(bw * sigma_trident<float>((float)a.Z, g));
        }
        // the lists in sample order, so that a result does not depend on the run
        unsigned m[2];
        for (int k = 0; k < 2; ++k) {
            m[k] = __ballot_sync(0xffffffffu, on && nr == k);
            if (lane == 0) count[k][wid] = __popc(m[k]);
        }
        __syncthreads();
        int n[2] = {0, 0}, at = __popc(m[nr] & ((1u << lane) - 1u));
#pragma unroll
        for (int w = 0; w < kEmWarps; ++w) {
            const int c0 = count[0][w], c1 = count[1][w];
            n[0] += c0;
            n[1] += c1;
            if (w < wid) at += nr ? c1 : c0;
        }
        if (on) list[nr][at] = make_float2(g, bw);
        __syncthreads();
        const int n_rel = n[0], n_nr = n[1];
        const float fC = (float)a.fC;
        deal_nodes(n_rel, a.n_quad, [&](int i, int q0, int q1) {
            rel_nodes<GRAD>(a, L, list[0][i].x, list[0][i].y, fC, q0, q1, acc);
        });
        if (n_nr && nr32) {
            NrCell C;
            C.A = (float)(cs.LTF * cs.LTF);
            C.B = (float)(cs.LD * cs.LD);
            C.iBA = (float)(1.0 / (cs.LD * cs.LD - cs.LTF * cs.LTF));
            C.eT = (float)cs.etaTF;
            C.eD = (float)cs.etaD;
            C.LTF2 = 2.0f * (float)cs.LTF;
            C.LD2 = 2.0f * (float)cs.LD;
            const double A = cs.LTF * cs.LTF, B = cs.LD * cs.LD;
            C.kA = (float)(2.0 * cs.LTF * B / (B - A));
            C.kB = (float)(2.0 * cs.LD * A / (B - A));
            deal_nodes(n_nr, a.n_quad, [&](int i, int q0, int q1) {
                nr_nodes<GRAD>(a, C, list[1][i].x, list[1][i].y, q0, q1, acc);
            });
        } else if (n_nr) {
            for (int i = wid; i < n_nr; i += kEmWarps) {
                const NrSums v = nr_sample<GRAD>(&a, (double)list[1][i].x, (double)list[1][i].y, &cs, lane);
                acc.r.add((float)v.r);
                acc.p.add((float)v.p);
                if (GRAD)
                    for (int k = 0; k < 3; ++k) { acc.r_nr[k] += v.dr[k]; acc.p_nr[k] += v.dp[k]; }
            }
        }
        __syncthreads();   // the lists are read before the next batch fills them
    }
    part[0][threadIdx.x] = (double)acc.r.s - acc.r.c;
    part[1][threadIdx.x] = (double)acc.p.s - acc.p.c;
    part[2][threadIdx.x] = (double)pair.s - pair.c;
    if (GRAD) {
        part[3][threadIdx.x] = (double)acc.r_LR.s - acc.r_LR.c;
        part[4][threadIdx.x] = (double)acc.p_LR.s - acc.p_LR.c;
        for (int i = 0; i < 3; ++i) { part[5 + i][threadIdx.x] = acc.r_nr[i]; part[8 + i][threadIdx.x] = acc.p_nr[i]; }
    }
    __syncthreads();
    // a warp per sum: eight values a lane, then across the lanes
    for (int i = wid; i < kOut; i += kEmWarps) {
        double v = 0.0;
        for (int k = lane; k < kEmThreads; k += 32) v += part[i][k];
        v = warp_sum(v);
        if (lane == 0) part[i][0] = v;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    double S[kOut];
    for (int i = 0; i < kOut; ++i) S[i] = part[i][0];
    const double C0 = 4.0 * a.Z * a.Z * kRe * kRe * kAlpha * kC;   // rate unit
    const double R = cs.n_i * C0 * S[0], P = cs.n_i * C0 * S[1], Rp = cs.n_i * kC * S[2];
    if constexpr (!GRAD) {
        a.out[3 * (size_t)c + 0] = (float)R;
        a.out[3 * (size_t)c + 1] = (float)Rp;
        a.out[3 * (size_t)c + 2] = (float)P;
    } else {
    // ---- adjoint: d out / d theta through the screening quantities
    const double g0 = a.grad_out[3 * (size_t)c + 0], g1 = a.grad_out[3 * (size_t)c + 1],
                 g2 = a.grad_out[3 * (size_t)c + 2];
    // d(g0 R + g2 P)/dS for S = L_R, L_TF, L_D, eta_D (without the n_i C0 factor)
    const double dLR = g0 * S[3] + g2 * S[4];
    const double dLTF = g0 * S[5] + g2 * S[8];
    const double dLD = g0 * S[6] + g2 * S[9];
    const double deD = g0 * S[7] + g2 * S[10];
    // totals with respect to L_TF, L_D, eta_D (direct NR part + through L_R)
    const double tLTF = dLTF + dLR * cs.LR_LTF;
    const double tLD = dLD + dLR * cs.LR_LD;
    const double teD = deD + dLR * cs.LR_eD;
    // d(L_TF, L_D, eta_D)/d theta
    double dLD_dth[5] = {0, 0, 0, 0, 0};
    if (cs.Zs == 0.0) {
        // no path through L_D (see cell_screen)
    } else if (cs.debye) {
        dLD_dth[0] = -0.5 * cs.LD / cs.n_i;
        dLD_dth[1] = 0.5 * cs.LD / cs.T_e;
        dLD_dth[2] = -0.5 * cs.LD * (2.0 * cs.Zs + 1.0) / (cs.Zs * (cs.Zs + 1.0));
    } else {
        dLD_dth[0] = -cs.LD / (3.0 * cs.n_i);
    }
    if (cs.Zs != 0.0) dLD_dth[4] = cs.LD / cs.sD;
    const double dLTF_dsTF = cs.LTF / cs.sTF;
    const double deD_dZs = 1.0 / a.Z;
    const double scale = cs.n_i * C0;
    double gp[5];
    gp[0] = scale * tLD * dLD_dth[0] + (g0 * R + g1 * Rp + g2 * P) / cs.n_i;
    gp[1] = scale * tLD * dLD_dth[1];
    gp[2] = scale * (tLD * dLD_dth[2] + teD * deD_dZs);
    gp[3] = scale * tLTF * dLTF_dsTF;
    gp[4] = scale * tLD * dLD_dth[4];
    for (int k = 0; k < 5; ++k) a.out[5 * (size_t)c + k] = (float)gp[k];
    }
}

// Gauss-Legendre nodes and weights on [-1, 1] (Newton iteration on P_n).
void gauss_legendre(int n, std::vector<double>& x, std::vector<double>& w)
{
    x.assign(n, 0.0);
    w.assign(n, 0.0);
    for (int i = 0; i < n; ++i) {
        double z = std::cos(kPi * (i + 0.75) / (n + 0.5)), dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int l = 2; l <= n; ++l) {
                const double p2 = ((2.0 * l - 1.0) * z * p1 - (l - 1.0) * p0) / l;
                p0 = p1;
                p1 = p2;
            }
            dp = n * (z * p1 - p0) / (z * z - 1.0);
            const double dz = p1 / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

int launch(pcc_ctx* ctx, bool grad, int n_cells, int n_samples, int Z, int n_quad, const float* params,
           const float* gamma, const float* w, const float* grad_out, float* out, void* stream, const char* name)
{
    if (!ctx || n_cells < 1 || n_samples < 0 || Z < 1 || Z > 100 || n_quad < 2 || n_quad > kMaxQuad || !params ||
        !out || (n_samples > 0 && (!gamma || !w)) || (grad && !grad_out)) {
        set_error(std::string(name) + ": invalid argument");
        return PCC_E_INVALID;
    }
    EmArgs a{};
    a.n_cells = n_cells;
    a.n_samples = n_samples;
    a.Z = Z;
    a.n_quad = n_quad;
    a.fC = coulomb_fc(Z);
    a.params = params;
    a.gamma = gamma;
    a.w = w;
    a.grad_out = grad_out;
    a.out = out;
    a.st = ctx->stats;
    // the rule is found once per node count and kept by the context (64 nodes took 0.2 ms of each call)
    if (ctx->em_quad != n_quad) {
        std::vector<double> gx, gw;
        gauss_legendre(n_quad, gx, gw);
        const double lo = std::log(1e-7), hi = 0.0, mid = 0.5 * (lo + hi), half = 0.5 * (hi - lo);
        ctx->em_node.resize(n_quad);
        ctx->em_node2.resize(n_quad);
        for (int q = 0; q < n_quad; ++q) {
            const double l = mid + half * gx[q];
            ctx->em_node[q] = make_float4((float)std::exp(l), (float)-std::expm1(l), (float)(half * gw[q]), (float)l);
            ctx->em_node2[q] = make_float2((float)(half * gw[q] * std::exp(l)), (float)std::exp(-l));
        }
        ctx->em_quad = n_quad;
    }
    std::copy(ctx->em_node.begin(), ctx->em_node.end(), a.node);
    std::copy(ctx->em_node2.begin(), ctx->em_node2.end(), a.node2);
    const int rc = ensure_scratch(ctx, (size_t)n_cells * sizeof(CellScreen));
    if (rc) return rc;
    CellScreen* screen = static_cast<CellScreen*>(ctx->scratch);
    a.screen = screen;
    cudaStream_t st = (cudaStream_t)stream;
    const int sb = (n_cells + 31) / 32;   // one warp a block: the cells spread over the SMs
    if (grad) screen_kernel<true><<<sb, 32, 0, st>>>(params, n_cells, Z, screen);
    else screen_kernel<false><<<sb, 32, 0, st>>>(params, n_cells, Z, screen);
    if (grad) emission_kernel<true><<<n_cells, kEmThreads, 0, st>>>(a);
    else emission_kernel<false><<<n_cells, kEmThreads, 0, st>>>(a);
    note_launches(2);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PCC_OK : cuda_fail(e, name);
}

}  // namespace

extern "C" int pcc_expected_emission_fwd(pcc_ctx* ctx, int n_cells, int n_samples, int Z, int n_quad,
                                         const float* params, const float* gamma, const float* w, float* out,
                                         void* stream)
{
    return launch(ctx, false, n_cells, n_samples, Z, n_quad, params, gamma, w, nullptr, out, stream,
                  "pcc_expected_emission_fwd");
}

extern "C" int pcc_expected_emission_bwd(pcc_ctx* ctx, int n_cells, int n_samples, int Z, int n_quad,
                                         const float* params, const float* gamma, const float* w,
                                         const float* grad_out, float* grad_params, void* stream)
{
    return launch(ctx, true, n_cells, n_samples, Z, n_quad, params, gamma, w, grad_out, grad_params, stream,
                  "pcc_expected_emission_bwd");
}
