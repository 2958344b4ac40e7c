// Material preparation and table build (Sec. II, Sec. III.A) in FP64, plus
// the FP32 copies used by the batched collision kernel.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "pcc_internal.h"
#include "pcc_physics.cuh"

namespace pcc {

TableGeom make_geom(const pcc_table_spec& s)
{
    TableGeom g;
    g.n_rows = s.n_rows;
    g.n_cols = s.n_cols;
    g.T_min = s.gamma_min - 1.0;
    g.T_max = s.gamma_max - 1.0;
    g.ln_T_min = std::log(g.T_min);
    g.inv_dln_row = (s.n_rows - 1) / std::log(g.T_max / g.T_min);
    g.ln_x_min = -s.cutoff_exp * std::log(10.0);
    g.ln_tri_min = std::log(s.tri_y_min);
    g.f_ln_T_min = (float)g.ln_T_min;
    g.f_inv_dln_row = (float)g.inv_dln_row;
    g.f_ln_x_min = (float)g.ln_x_min;
    g.f_ln_tri_min = (float)g.ln_tri_min;
    return g;
}

enum TableKind { kBrems = 0, kBH = 1, kTriPair = 2, kTriSplit = 3 };
constexpr int kEdgePanels = 12;   // graded sub-panels (ratio 1/4) on the outer column intervals
constexpr int kMaxQuad = 32;

__global__ void material_prep_kernel(const pcc_material* mats, int n, double* screen)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Screen s = screen_from_material(mats[i]);
    double* o = screen + (size_t)i * kScreenFields;
    o[0] = s.LTF; o[1] = s.LD; o[2] = s.etaTF; o[3] = s.etaD;
    o[4] = s.ITFD; o[5] = s.LR; o[6] = s.fC; o[7] = s.Z;
}

// Gauss-Legendre nodes and weights on [-1, 1] (Newton on the Legendre
// recurrence), found once on the host: one thread of every block spent up to 0.4
// ms on them.
constexpr int kTfdNodes = 12;
struct QuadRule {
    double x[kMaxQuad], w[kMaxQuad], tx[kTfdNodes], tw[kTfdNodes];
};
static void legendre_nodes(int n, double* x, double* w)
{
    for (int i = 0; i < n; ++i) {
        double z = std::cos(kPi * (i + 0.75) / (n + 0.5)), dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double a = 1.0, b = z;
            for (int l = 2; l <= n; ++l) {
                const double c = ((2.0 * l - 1.0) * z * b - (l - 1.0) * a) / l;
                a = b;
                b = c;
            }
            dp = n == 1 ? 1.0 : n * (z * b - a) / (z * z - 1.0);
            const double dz = b / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-15) break;
        }
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

// Flags of the table kernels: the printed non-relativistic momentum-transfer
// bounds, and the TFD-quadrature screening mode.
constexpr int kFlagPrinted = 1, kFlagTfdQuad = 2;

// ---- full Thomas-Fermi-Debye potential ----------------------------------------
// Eqs. (defphi1) and (defphi2) for the form factor (Eq. defF, Eq. V_TFD)
//   1 - F(u) = eta_TF a^2 / (1 + a^2) + eta_D b^2 / (1 + b^2),  a = L_TF u, b = L_D u,
// by quadrature in t = ln u on unit panels from t = 0 down to ln delta (the last
// one shorter), kTfdNodes-point Gauss-Legendre each.  With r = u/delta the
// integrands in t are (1 - 1/r)^2 (1 - F)^2 and (1 + (3 - 6 ln r)/r^2 - 4/r^3) (1 - F)^2:
// polynomials in delta and ln delta over moments of (1 - F)^2 that do not depend
// on delta.  The moments of the whole panels are summed once per material, so
// that an integral takes one lookup and the nodes of its last panel instead of
// those of up to thirty panels.
constexpr int kTfdPanels = 128, kTfdMoments = 5;   // f2, f2/u, f2/u^2, f2 ln u/u^2, f2/u^3

__device__ __forceinline__ double tfd_form2(const Screen& s, double u2)
{
    const double a2 = s.LTF * s.LTF * u2, b2 = s.LD * s.LD * u2;
    const double f = (s.etaTF * a2 * (1.0 + b2) + s.etaD * b2 * (1.0 + a2)) / ((1.0 + a2) * (1.0 + b2));
    return f * f;
}

// Sums of the moments over panels 0 .. n - 1 at [mat][n][moment].
__global__ void tfd_moments_kernel(const double* screen, const __grid_constant__ QuadRule rule, double* out)
{
    __shared__ double part[kTfdPanels][kTfdMoments];
    const Screen s = load_screen(screen + (size_t)blockIdx.x * kScreenFields);
    for (int j = threadIdx.x; j < kTfdPanels; j += blockDim.x) {
        double m[kTfdMoments] = {0, 0, 0, 0, 0};
        for (int q = 0; q < kTfdNodes; ++q) {
            const double t = -(j + 0.5) + 0.5 * rule.tx[q], iu = exp(-t);
            const double f = 0.5 * rule.tw[q] * tfd_form2(s, 1.0 / (iu * iu));
            m[0] += f;
            m[1] += f * iu;
            m[2] += f * iu * iu;
            m[3] += f * iu * iu * t;
            m[4] += f * iu * iu * iu;
        }
        for (int k = 0; k < kTfdMoments; ++k) part[j][k] = m[k];
    }
    __syncthreads();
    if (threadIdx.x < kTfdMoments) {
        double acc = 0.0;
        double* o = out + (size_t)blockIdx.x * (kTfdPanels + 1) * kTfdMoments + threadIdx.x;
        o[0] = 0.0;
        for (int j = 0; j < kTfdPanels; ++j) o[(j + 1) * kTfdMoments] = acc += part[j][threadIdx.x];
    }
}

// One panel of the quadrature, [lo, hi] in ln u, added to I1, I2.
__device__ __forceinline__ void tfd_panel(const Screen& s, double lnd, double lo, double hi, const QuadRule& rule,
                                          double& I1, double& I2)
{
    const double h = 0.5 * (hi - lo), m = 0.5 * (hi + lo);
    double p1 = 0.0, p2 = 0.0;
    for (int q = 0; q < kTfdNodes; ++q) {
        const double t = m + h * rule.tx[q], lr = t - lnd;
        const double ir = exp(-lr), u = exp(t), om = -expm1(-lr);
        const double f2 = tfd_form2(s, u * u);
        p1 += rule.tw[q] * om * om * f2;
        p2 += rule.tw[q] * (1.0 + (3.0 - 6.0 * lr) * ir * ir - 4.0 * ir * ir * ir) * f2;
    }
    I1 += h * p1;
    I2 += h * p2;
}

__device__ __forceinline__ void tfd_I12(const Screen& s, const double* moments, const YukawaD& g, const QuadRule& rule,
                                        double& I1, double& I2)
{
    I1 = I2 = 0.0;
    if (!(g.d > 0.0 && g.d < 1.0)) return;
    const int n = min((int)floor(-g.ln), kTfdPanels);
    const double* M = moments + n * kTfdMoments;
    const double d2 = g.d * g.d;
    I1 = M[0] - 2.0 * g.d * M[1] + d2 * M[2];
    I2 = M[0] + d2 * ((3.0 + 6.0 * g.ln) * M[2] - 6.0 * M[3]) - 4.0 * d2 * g.d * M[4];
    for (double hi = -(double)n; hi > g.ln; hi -= 1.0) tfd_panel(s, g.ln, fmax(hi - 1.0, g.ln), hi, rule, I1, I2);
}

// ---- integrands -----------------------------------------------------------------
// A material of a block: its screening and what the integrands need of it alone.
struct BlockMat {
    Screen s;
    YukawaL y;
    double unit;            // 4 Z^2 r_e^2 alpha
    double A, B, iBA;       // L_TF^2, L_D^2, eta_TF eta_D / (B - A)
    double ex1;             // expm1(-2 pi alpha Z / beta_1) of the row
    int near;               // L_TF ~ L_D: the cross term takes its limit
    const double* moments;
};

__device__ __forceinline__ BlockMat block_mat(const double* screen, const double* tfd, int mat, double rowv)
{
    BlockMat m;
    m.s = load_screen(screen + (size_t)mat * kScreenFields);
    m.y = yukawa_length(m.s.LR);
    m.unit = 4.0 * m.s.Z * m.s.Z * kRe * kRe * kAlpha;
    m.A = m.s.LTF * m.s.LTF;
    m.B = m.s.LD * m.s.LD;
    m.near = fabs(m.B - m.A) <= 1e-6 * fmax(m.A, m.B);
    m.iBA = m.near ? 0.0 : m.s.etaTF * m.s.etaD / (m.B - m.A);
    m.ex1 = expm1(-2.0 * kPi * kAlpha * m.s.Z * (1.0 + rowv) / sqrt(rowv * (rowv + 2.0)));
    m.moments = tfd ? tfd + (size_t)mat * (kTfdPanels + 1) * kTfdMoments : nullptr;
    return m;
}

// A node's geometry, shared by the materials of the block.
struct NodeGeom {
    YukawaD g;
    double c1, c2;          // factors of I1 and I2 in the relativistic bracket, or gp^2 + gm^2 and 2/3 gp gm
    double scale;           // what multiplies the bracket
    double k, T2, p2, qm2, P, ib2;   // non-relativistic: photon energy, T_2, p_2, q_-^2, q_+^2 - q_-^2, 1/beta_2
};

// ln(1 + x), x >= 0, to 1e-14 relative: cheaper than log1p, which holds the last bit.
__device__ __forceinline__ double log1p_any(double x) { return x < 0.015625 ? log1p_small(x) : log(1.0 + x); }

// At column variable v (ln x for Brems, else y).
template <int KIND>
__device__ __forceinline__ NodeGeom node_geom(double rowv, double v, bool rel)
{
    NodeGeom n;
    if (KIND == kBrems) {
        const double x = exp(v), omx = -expm1(v), g1 = 1.0 + rowv;
        n.k = x * rowv;
        n.T2 = rowv * omx;
        if (rel) {
            const double gk = 1.0 + n.T2, eps = gk / g1;     // gamma - k
            n.g.d = n.k / (2.0 * g1 * gk);
            n.g.omd = 1.0 - n.g.d;
            n.g.inv = 1.0 / n.g.d;
            n.g.ln = log(n.g.d);
            n.c1 = 1.0 + eps * eps;
            n.c2 = (2.0 / 3.0) * eps;
            n.scale = 1.0;
        } else {
            const double p1 = sqrt(rowv * (rowv + 2.0));
            n.p2 = sqrt(n.T2 * (n.T2 + 2.0));
            const double qm = n.k * (rowv + n.T2 + 2.0) / (p1 + n.p2);
            n.qm2 = qm * qm;
            n.P = 4.0 * p1 * n.p2;
            n.ib2 = (1.0 + n.T2) / n.p2;
            n.scale = 4.0 / (3.0 * p1 * p1) * (p1 / g1) * n.ib2;   // 4/(3 p1^2) beta_1/beta_2
        }
    } else {
        const double k = 2.0 + rowv, gp = 1.0 + v * rowv, gm = 1.0 + (1.0 - v) * rowv, pp = 2.0 * gp * gm;
        const double ipp = 1.0 / pp;
        n.g.d = k * ipp;
        n.g.omd = (rowv + 2.0 * v * (1.0 - v) * rowv * rowv) * ipp;   // 1 - d, without the cancellation near 1
        n.g.inv = pp / k;
        n.g.ln = log(n.g.d);
        n.c1 = gp * gp + gm * gm;
        n.c2 = pp * (1.0 / 3.0);
        n.scale = rowv / (k * k * k);
    }
    return n;
}

// The integrand at the node: dsigma/dk k per d ln k (Brems), or dsigma/dgamma_+
// times the row variable.  exZ, ex2: the node's Elwert factor for the charge exZ.
template <int KIND>
__device__ __forceinline__ double node_value(const BlockMat& m, const NodeGeom& n, double rowv, bool rel, int flags,
                                             const QuadRule& rule, double& exZ, double& ex2)
{
    if (KIND == kBrems && !rel) {
        if (!(n.k > 0.0 && n.T2 > 0.0)) return 0.0;
        if ((flags & kFlagPrinted) || m.near) return dsdk_nonrel(m.s, 1.0 + rowv, n.k, flags & kFlagPrinted) * n.k;
        // Eq. (cs_br_nr): with P = q_+^2 - q_-^2 the logarithms of the two Yukawa
        // terms are those of the cross term, and no difference of nearly equal
        // numbers is formed
        const double Tm = 1.0 + n.qm2 * m.A, Dm = 1.0 + n.qm2 * m.B, PA = n.P * m.A, PB = n.P * m.B;
        const double Tp = Tm + PA, Dp = Dm + PB;
        const double tt = Tm * Tp, dd = Dm * Dp, inv = 1.0 / (tt * dd);
        const double it = dd * inv, id = tt * inv;           // 1/(Tm Tp), 1/(Dm Dp)
        const double la = log1p_any(PA * Tp * it), lb = log1p_any(PB * Dp * id);
        const double br = 0.5 * m.s.etaTF * m.s.etaTF * (la - PA * it) + 0.5 * m.s.etaD * m.s.etaD * (lb - PB * id) +
                          m.iBA * (m.B * la - m.A * lb);
        if (m.s.Z != exZ) {   // uniform: the materials of a run are mostly states of one element
            exZ = m.s.Z;
            ex2 = n.scale / expm1(-2.0 * kPi * kAlpha * m.s.Z * n.ib2);
        }
        return m.unit * br * m.ex1 * ex2;
    }
    double I1, I2;
    if (flags & kFlagTfdQuad) tfd_I12(m.s, m.moments, n.g, rule, I1, I2);
    else yukawa_I12(m.y, n.g, I1, I2);
    if (KIND == kBrems) {
        // Eq. (csre), or Eq. (csur) with f_C; dsigma/dk k
        const double fc = 1.0 + rowv <= 100.0 ? 0.0 : m.s.fC;
        return m.unit * fmax(n.c1 * (I1 + 1.0 - fc) - n.c2 * (I2 + 5.0 / 6.0 - fc), 0.0);
    }
    return m.unit * n.scale * fmax(n.c1 * (I1 + 1.0) + n.c2 * (I2 + 5.0 / 6.0), 0.0);   // Eq. (dsdkbh)
}

// ---- rows --------------------------------------------------------------------------
// Panel p of a row's quadrature: its ends [a, b] and column.  One panel per
// column interval, kEdgePanels + 1 graded ones on the last interval and, on a
// linear grid, on the first.
struct Panel { double a, b; int col, grade; };
__device__ __forceinline__ double col_edge(int c, int nc, bool logcol, double ly)
{
    return logcol ? ly * (1.0 - (double)c / (nc - 1)) : (double)c / (nc - 1);
}
__device__ __forceinline__ Panel panel_of(int p, int nc, bool logcol, double ly)
{
    constexpr int G = kEdgePanels + 1;
    Panel r;
    const int left = logcol ? 0 : G;                       // panels of the graded first column
    if (p < left) {
        r.col = 0;
        r.grade = p;
    } else {
        const int c = p - left + (logcol ? 0 : 1);
        r.col = min(c, nc - 2);
        r.grade = c - (nc - 2);                            // < 0: an ordinary column
    }
    r.a = col_edge(r.col, nc, logcol, ly);
    r.b = col_edge(r.col + 1, nc, logcol, ly);
    if (p < left) {                                        // cut towards a
        const double w = r.b - r.a, lo = r.a;
        r.b = p == 0 ? r.b : lo + w * ldexp(1.0, -2 * p);
        r.a = p == kEdgePanels ? lo : lo + w * ldexp(1.0, -2 * (p + 1));
    } else if (r.grade >= 0) {                             // cut towards b
        const double w = r.b - r.a, hi = r.b;
        r.a = r.grade == 0 ? r.a : hi - w * ldexp(1.0, -2 * r.grade);
        r.b = r.grade == kEdgePanels ? hi : hi - w * ldexp(1.0, -2 * (r.grade + 1));
    }
    return r;
}

// One block per row and up to kBlockMats materials: integrals over every column
// interval, then the cumulative sum in column order, normalisation and the
// total.  A group of lanes takes a panel, a lane a node, so that the graded
// panels do not fall to one thread; the node's geometry (its exponential,
// logarithm, divisions) is shared by the materials; the Bethe-Heitler and split
// shapes are symmetric in the energy share, so that half of their columns are
// mirrored.  Bound by the FP64 units (two instructions per clock and SM):
// 31 materials x 256 x 256, 8 nodes: Brems 28.7 -> 4.1 ms, Bethe-Heitler 34.2 -> 2.2 ms;
// one material in the full potential: 24.3 -> 1.5 and 11.8 -> 0.8 ms.
constexpr int kBlockMats = 8, kRowThreads = 256;
constexpr int kRowSmem = 96 * 1024;   // dynamic shared memory of a block at most

template <int KIND>
__global__ void __launch_bounds__(kRowThreads) table_rows_kernel(const double* screen, const double* tfd, int n_mats,
                                                                 int per_block, TableGeom g,
                                                                 const __grid_constant__ QuadRule rule, int Q, int group,
                                                                 int flags, double* sigma_out, double* cdf_out)
{
    constexpr bool kMat = KIND == kBrems || KIND == kBH, kLog = KIND == kBrems || KIND == kTriPair;
    constexpr int kEdge = 2 * (kEdgePanels + 1);
    extern __shared__ double sm[];
    __shared__ BlockMat mats[kBlockMats];
    __shared__ double total[kBlockMats];
    const int r = blockIdx.x, mat0 = blockIdx.y * per_block, nm = kMat ? min(per_block, n_mats - mat0) : 1;
    const int nc = g.n_cols, stride = nc + kEdge;          // part[nc], then the graded panels
    const double rowv = g.T_min * pow(g.T_max / g.T_min, (double)r / (g.n_rows - 1));
    const double ly = (KIND == kBrems) ? g.ln_x_min : g.ln_tri_min;
    const bool rel = 1.0 + rowv > 2.0;
    if (kMat && threadIdx.x < nm) mats[threadIdx.x] = block_mat(screen, tfd, mat0 + threadIdx.x, rowv);
    __syncthreads();
    const int N = nc - 1, half = kLog ? N : (N + 1) / 2;   // columns computed
    const int panels = kLog ? nc - 2 + kEdgePanels + 1 : kEdgePanels + 1 + half - 1;
    const int gi = threadIdx.x / group, q = threadIdx.x % group, groups = blockDim.x / group;
    for (int p0 = 0; p0 < panels; p0 += groups) {          // uniform
        const int p = p0 + gi;
        const bool on = p < panels && q < Q;
        const Panel P = panel_of(min(p, panels - 1), nc, kLog, ly);
        const double h = 0.5 * (P.b - P.a), mid = 0.5 * (P.a + P.b), v = mid + h * rule.x[on ? q : 0];
        const double w = on ? h * rule.w[q] : 0.0;
        NodeGeom n;
        if (kMat) n = node_geom<KIND>(rowv, v, rel);
        double exZ = 0.0, ex2 = 0.0;
        for (int m = 0; m < nm; ++m) {
            double f;
            if (kMat) f = node_value<KIND>(mats[m], n, rowv, rel, flags, rule, exZ, ex2);
            else if (KIND == kTriPair) { const double y = exp(v); f = trident_pair_shape(3.0 + rowv, 2.0 + y * rowv) * rowv * y; }
            else f = trident_split_shape(2.0 + rowv, 1.0 + v * rowv) * rowv;
            f = on ? w * f : 0.0;
            for (int o = group >> 1; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
            if (q == 0 && p < panels) {
                double* part = sm + (size_t)m * stride;
                if (P.grade < 0) part[P.col + 1] = f;
                else part[nc + (P.col == 0 && !kLog ? 0 : kEdgePanels + 1) + P.grade] = f;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x % 32 == 0 && threadIdx.x / 32 < nm) {  // a warp's first lane per material
        const int m = threadIdx.x / 32;
        double* part = sm + (size_t)m * stride;
        for (int e = kLog ? 1 : 0; e < (kLog ? 2 : 1); ++e) {   // the graded columns, panels in order
            double s = 0.0;
            for (int i = 0; i <= kEdgePanels; ++i) s += part[nc + e * (kEdgePanels + 1) + i];
            part[e ? N : 1] = s;
        }
        if (!kLog)
            for (int c = 0; c < half; ++c) part[N - c] = part[c + 1];
        double cum = 0.0;
        part[0] = 0.0;
        for (int c = 1; c < nc; ++c) {
            cum += part[c];
            part[c] = cum;
        }
        total[m] = cum;
    }
    __syncthreads();
    for (int m = 0; m < nm; ++m) {
        const double* part = sm + (size_t)m * stride;
        double* row = cdf_out + ((size_t)(mat0 + m) * g.n_rows + r) * nc;
        const double tot = total[m], inv = 1.0 / tot;
        for (int c = threadIdx.x; c < nc; c += blockDim.x) {
            double v;
            if (tot > 0.0) v = (c == nc - 1) ? 1.0 : fmin(part[c] * inv, 1.0);
            else v = (double)c / (nc - 1);   // zero shape: uniform in the column variable
            row[c] = v;
        }
        if (threadIdx.x == 0 && sigma_out) sigma_out[(size_t)(mat0 + m) * g.n_rows + r] = tot;
    }
}

__global__ void to_float_kernel(const double* in, float* out, size_t n, int take_log)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = take_log ? (float)log(in[i]) : (float)in[i];
}

__global__ void z_to_float_kernel(const double* screen, float* out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (float)screen[(size_t)i * kScreenFields + 7];
}

// Per-material upper bounds B with x <= coef * B for every pair (coef =
// (n_p n_t / n_pt) c dt), used to reject a pair from its uniform alone:
//   Brems:   x = coef sigma(T') p'/(g_e g_i) <= coef sigma(T') beta' (1 + |beta_i|),
//            and the log-log interpolated sigma between rows j, j+1 is at most
//            max(sigma_j, sigma_j+1) while beta' <= beta(T_j+1); the last row
//            covers energies above the table.
//   Trident: sigma_T is increasing in gamma; the bound holds for gamma' <= 1e7.
//   BH:      x = coef sigma(k') k'/(k g_i) <= coef sigma(k') (1 + |beta_i|).
// The factor 2 covers 1 + |beta_i|; 1e-3 more covers float rounding of x.
// One warp per material, lanes over the rows (one thread took 1.1 ms for 256 powers).
__global__ void bounds_kernel(const double* screen, const double* brems_sigma, const double* bh_sigma, TableGeom g,
                              int n_mat, float* bound)
{
    const int m = blockIdx.x, lane = threadIdx.x;
    const double* sb = brems_sigma + (size_t)m * g.n_rows;
    const double* sh = bh_sigma + (size_t)m * g.n_rows;
    double bb = sb[g.n_rows - 1], bh = 0.0;
    for (int j = lane; j + 1 < g.n_rows; j += 32) {
        const double T = g.T_min * pow(g.T_max / g.T_min, (double)(j + 1) / (g.n_rows - 1));
        const double beta = sqrt(T * (T + 2.0)) / (1.0 + T);
        bb = fmax(bb, fmax(sb[j], sb[j + 1]) * beta);
    }
    for (int j = lane; j < g.n_rows; j += 32) bh = fmax(bh, sh[j]);
    for (int o = 16; o > 0; o >>= 1) {
        bb = fmax(bb, __shfl_xor_sync(0xffffffffu, bb, o));
        bh = fmax(bh, __shfl_xor_sync(0xffffffffu, bh, o));
    }
    if (lane) return;
    const double Z = screen[(size_t)m * kScreenFields + 7];
    const double l = log((1e7 + 4.5) / 6.89);
    const double bt = 5.22e-34 * Z * Z * l * l * l;
    const double margin = 2.0 * 1.001;
    bound[3 * m + 0] = (float)(margin * bb);
    bound[3 * m + 1] = (float)(margin * bt);
    bound[3 * m + 2] = (float)(margin * bh);
}

}  // namespace pcc

using namespace pcc;

static void free_tables(pcc_ctx* ctx)
{
    void* ptrs[] = {ctx->screen, ctx->brems_sigma, ctx->brems_cdf, ctx->bh_sigma, ctx->bh_cdf, ctx->tri_gp_cdf,
                    ctx->tri_split_cdf, ctx->f_brems_lnsig, ctx->f_brems_cdf, ctx->f_bh_lnsig, ctx->f_bh_cdf,
                    ctx->f_tri_gp_cdf, ctx->f_tri_split_cdf, ctx->f_Z, ctx->f_bound};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    ctx->screen = ctx->brems_sigma = ctx->brems_cdf = ctx->bh_sigma = ctx->bh_cdf = nullptr;
    ctx->tri_gp_cdf = ctx->tri_split_cdf = nullptr;
    ctx->f_brems_lnsig = ctx->f_brems_cdf = ctx->f_bh_lnsig = ctx->f_bh_cdf = nullptr;
    ctx->f_tri_gp_cdf = ctx->f_tri_split_cdf = ctx->f_Z = ctx->f_bound = nullptr;
    ctx->n_mat = 0;
}

void pcc_free_tables(pcc_ctx* ctx) { free_tables(ctx); }

extern "C" int pcc_tables_build(pcc_ctx* ctx, const pcc_material* mats, int n_mats, const pcc_table_spec* spec,
                                void* stream)
{
    if (!ctx || !mats || !spec) { set_error("pcc_tables_build: null argument"); return PCC_E_INVALID; }
    const pcc_table_spec& s = *spec;
    if (n_mats < 1 || n_mats > 4096 || s.n_rows < 2 || s.n_rows > 4096 || s.n_cols < 3 || s.n_cols > 4096 ||
        s.quad_nodes < 1 || s.quad_nodes > kMaxQuad || !(s.gamma_min > 1.0) || !(s.gamma_max > s.gamma_min) ||
        s.cutoff_exp < 1 || s.cutoff_exp > 30 || !(s.tri_y_min > 0.0 && s.tri_y_min < 1.0) ||
        (s.nr_qbounds != 0 && s.nr_qbounds != 1) ||
        (s.screening != PCC_SCREEN_REDUCED && s.screening != PCC_SCREEN_TFD_QUAD)) {
        set_error("pcc_tables_build: invalid table spec");
        return PCC_E_INVALID;
    }
    for (int i = 0; i < n_mats; ++i) {
        const pcc_material& m = mats[i];
        if (m.Z < 1 || m.Z > 120 || !(m.Zstar >= 0.0 && m.Zstar <= m.Z) || !(m.n_i > 0.0) || !(m.T_e >= 0.0) ||
            !(m.s_TF > 0.0) || !(m.s_D > 0.0) || (m.Zstar > 0.0 && !(m.T_e > 0.0))) {
            set_error("pcc_tables_build: invalid material " + std::to_string(i));
            return PCC_E_INVALID;
        }
    }
    cudaStream_t st = (cudaStream_t)stream;
    free_tables(ctx);
    const size_t R = s.n_rows, C = s.n_cols, M = n_mats;
    cudaError_t e = cudaSuccess;
    auto A = [&](void** p, size_t bytes) { if (e == cudaSuccess) e = cudaMalloc(p, bytes); };
    A((void**)&ctx->screen, M * kScreenFields * sizeof(double));
    A((void**)&ctx->brems_sigma, M * R * sizeof(double));
    A((void**)&ctx->brems_cdf, M * R * C * sizeof(double));
    A((void**)&ctx->bh_sigma, M * R * sizeof(double));
    A((void**)&ctx->bh_cdf, M * R * C * sizeof(double));
    A((void**)&ctx->tri_gp_cdf, R * C * sizeof(double));
    A((void**)&ctx->tri_split_cdf, R * C * sizeof(double));
    A((void**)&ctx->f_brems_lnsig, M * R * sizeof(float));
    A((void**)&ctx->f_brems_cdf, M * R * C * sizeof(float));
    A((void**)&ctx->f_bh_lnsig, M * R * sizeof(float));
    A((void**)&ctx->f_bh_cdf, M * R * C * sizeof(float));
    A((void**)&ctx->f_tri_gp_cdf, R * C * sizeof(float));
    A((void**)&ctx->f_tri_split_cdf, R * C * sizeof(float));
    A((void**)&ctx->f_Z, M * sizeof(float));
    A((void**)&ctx->f_bound, 3 * M * sizeof(float));
    if (e != cudaSuccess) { free_tables(ctx); return cuda_fail(e, "pcc_tables_build: cudaMalloc"); }

    pcc_material* dmats = nullptr;
    e = cudaMalloc(&dmats, M * sizeof(pcc_material));
    if (e == cudaSuccess) e = cudaMemcpyAsync(dmats, mats, M * sizeof(pcc_material), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) { free_tables(ctx); if (dmats) cudaFree(dmats); return cuda_fail(e, "pcc_tables_build: upload"); }
    material_prep_kernel<<<(n_mats + 63) / 64, 64, 0, st>>>(dmats, n_mats, ctx->screen);

    const TableGeom g = make_geom(s);
    const int flags = (s.nr_qbounds ? kFlagPrinted : 0) | (s.screening == PCC_SCREEN_TFD_QUAD ? kFlagTfdQuad : 0);
    QuadRule rule;
    legendre_nodes(s.quad_nodes, rule.x, rule.w);
    legendre_nodes(kTfdNodes, rule.tx, rule.tw);
    int group = 1;                          // lanes per panel: a power of two, at least the nodes
    while (group < s.quad_nodes) group <<= 1;
    const size_t row_bytes = (C + 2 * (kEdgePanels + 1)) * sizeof(double);
    const int per = std::max(1, std::min({kBlockMats, n_mats, (int)(kRowSmem / row_bytes)}));
    const int chunks = (n_mats + per - 1) / per, per_block = (n_mats + chunks - 1) / chunks;
    const size_t smem = per_block * row_bytes;
    // Always the same limit: without it a block's static and dynamic shared memory
    // together may not pass 48 KB, and a limit set per call would be another
    // thread's too.
    e = cudaFuncSetAttribute(table_rows_kernel<kBrems>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(table_rows_kernel<kBH>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmem);
    if (e != cudaSuccess) { free_tables(ctx); cudaFree(dmats); return cuda_fail(e, "pcc_tables_build: shared memory"); }
    double* tfd = nullptr;
    if (flags & kFlagTfdQuad) {
        e = cudaMalloc(&tfd, M * (kTfdPanels + 1) * kTfdMoments * sizeof(double));
        if (e != cudaSuccess) { free_tables(ctx); cudaFree(dmats); return cuda_fail(e, "pcc_tables_build: cudaMalloc"); }
        tfd_moments_kernel<<<n_mats, 128, 0, st>>>(ctx->screen, rule, tfd);
        note_launches(1);
    }
    table_rows_kernel<kBrems><<<dim3(s.n_rows, chunks), kRowThreads, smem, st>>>(
        ctx->screen, tfd, n_mats, per_block, g, rule, s.quad_nodes, group, flags, ctx->brems_sigma, ctx->brems_cdf);
    table_rows_kernel<kBH><<<dim3(s.n_rows, chunks), kRowThreads, smem, st>>>(
        ctx->screen, tfd, n_mats, per_block, g, rule, s.quad_nodes, group, flags, ctx->bh_sigma, ctx->bh_cdf);
    table_rows_kernel<kTriPair><<<dim3(s.n_rows, 1), kRowThreads, row_bytes, st>>>(
        ctx->screen, nullptr, 1, 1, g, rule, s.quad_nodes, group, flags, nullptr, ctx->tri_gp_cdf);
    table_rows_kernel<kTriSplit><<<dim3(s.n_rows, 1), kRowThreads, row_bytes, st>>>(
        ctx->screen, nullptr, 1, 1, g, rule, s.quad_nodes, group, flags, nullptr, ctx->tri_split_cdf);
    auto conv = [&](const double* in, float* out, size_t n, int lg) {
        to_float_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(in, out, n, lg);
    };
    conv(ctx->brems_sigma, ctx->f_brems_lnsig, M * R, 1);
    conv(ctx->brems_cdf, ctx->f_brems_cdf, M * R * C, 0);
    conv(ctx->bh_sigma, ctx->f_bh_lnsig, M * R, 1);
    conv(ctx->bh_cdf, ctx->f_bh_cdf, M * R * C, 0);
    conv(ctx->tri_gp_cdf, ctx->f_tri_gp_cdf, R * C, 0);
    conv(ctx->tri_split_cdf, ctx->f_tri_split_cdf, R * C, 0);
    z_to_float_kernel<<<(n_mats + 63) / 64, 64, 0, st>>>(ctx->screen, ctx->f_Z, n_mats);
    bounds_kernel<<<n_mats, 32, 0, st>>>(ctx->screen, ctx->brems_sigma, ctx->bh_sigma, g, n_mats,
                                                     ctx->f_bound);
    note_launches(13);
    std::vector<float> bound(3 * M);
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(bound.data(), ctx->f_bound, bound.size() * sizeof(float), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(dmats);
    cudaFree(tfd);
    if (e != cudaSuccess) { free_tables(ctx); return cuda_fail(e, "pcc_tables_build: kernels"); }
    ctx->pair_rate = 0.0;
    for (size_t m = 0; m < M; ++m)   // the bounds hold twice the cross section, for ions that meet the projectile
        ctx->pair_rate = std::max(ctx->pair_rate, 0.5 * kC * mats[m].n_i * std::max(bound[3 * m], bound[3 * m + 2]));
    ctx->n_mat = n_mats;
    ctx->spec = s;
    return PCC_OK;
}

extern "C" int pcc_tables_read(pcc_ctx* ctx, double* brems_sigma, double* brems_cdf, double* bh_sigma,
                               double* bh_cdf, double* tri_gp_cdf, double* tri_split_cdf, double* screening)
{
    if (!ctx) { set_error("pcc_tables_read: null context"); return PCC_E_INVALID; }
    if (ctx->n_mat == 0) { set_error("pcc_tables_read: no tables"); return PCC_E_NO_TABLES; }
    const size_t R = ctx->spec.n_rows, C = ctx->spec.n_cols, M = ctx->n_mat;
    cudaError_t e = cudaSuccess;
    // A copy into memory that the host has never touched has the device fault its
    // pages in one by one (33 MB: 27 ms); touched first, it takes 1 ms.
    auto cp = [&](double* dst, const double* src, size_t n) {
        if (dst)
            for (size_t i = 0; i < n; i += 512) reinterpret_cast<volatile double*>(dst)[i] = 0.0;
        if (dst && e == cudaSuccess) e = cudaMemcpy(dst, src, n * sizeof(double), cudaMemcpyDeviceToHost);
    };
    cp(brems_sigma, ctx->brems_sigma, M * R);
    cp(brems_cdf, ctx->brems_cdf, M * R * C);
    cp(bh_sigma, ctx->bh_sigma, M * R);
    cp(bh_cdf, ctx->bh_cdf, M * R * C);
    cp(tri_gp_cdf, ctx->tri_gp_cdf, R * C);
    cp(tri_split_cdf, ctx->tri_split_cdf, R * C);
    cp(screening, ctx->screen, M * kScreenFields);
    return e == cudaSuccess ? PCC_OK : cuda_fail(e, "pcc_tables_read");
}
