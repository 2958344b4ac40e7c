// Per-particle sums of the FP64 totals (sum W, sum W E, sum W |u|), shared by
// pcc_totals and pcc_totals_noalloc.
//
// Two FP64 square roots and the sums take about 50 FP64 instructions per
// particle, and this chip issues about two of those per clock and SM: summing
// 5.1e7 electrons that way took 4.1 ms for 0.8 GB of records.  The same values
// are therefore formed in FP32 as unevaluated sums of three floats by
// error-free transformations (Dekker/Knuth two-sums, FMA products): u^2 exactly
// to 2^-70, the square roots by one Newton step and two exactly represented
// remainders, the products with the weight and the running sums with their
// rounding errors carried along.  The parts dropped are below 2^-60 of a term,
// so that a lane's sum is at least as close as the FP64 loop's; it is added to
// FP64 every kFlushAdds particles.  Some 200 FP32 instructions per particle bound
// the kernel: 5.1e7 electrons in 262144 log-normal cells 3.86 -> 0.48 ms (0.12 ms
// for the loads alone), off 64-bit sums by 1.3e-16 (5.4e-16 before).  Particles outside the range in which every
// error term stays a normal float (and non-finite ones) take the FP64 formula.
#pragma once

#include "pcc_device.cuh"

namespace pcc {

constexpr int kFlushAdds = 128;   // products below 1e35 each: a sum of 128 stays finite

// a + b = s + e exactly.
__device__ __forceinline__ float two_sum(float a, float b, float& e)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

// Running sum hi + lo + c.
struct Sum3 {
    float hi = 0.f, lo = 0.f, c = 0.f;
    // adds p + q1 + q2 + t with |q1|, |q2| of the order of p's last bit and t below both
    __device__ __forceinline__ void add(float p, float q1, float q2, float t)
    {
        float e1, e2, e3, e4;
        hi = two_sum(hi, p, e1);
        const float y = two_sum(q1, q2, e2);
        lo = two_sum(lo, y, e3);
        lo = two_sum(lo, e1, e4);
        c += (e2 + e3) + (e4 + t);
    }
    __device__ __forceinline__ void add(float p)
    {
        float e1, e2;
        hi = two_sum(hi, p, e1);
        lo = two_sum(lo, e1, e2);
        c += e2;
    }
    __device__ __forceinline__ double take()
    {
        const double v = (double)hi + ((double)lo + (double)c);
        hi = lo = c = 0.f;
        return v;
    }
};

// sqrt(g + c + d) = s0 + s1 + s2 for g > 0 and |c| up to g's last bit, |d| below it.
__device__ __forceinline__ void sqrt3(float g, float c, float d, float& s0, float& s1, float& s2)
{
    const float r = rsqrtf(g), h = 0.5f * r;
    float s = __fmul_rn(g, r);
    s = fmaf(fmaf(-s, s, g), h, s);       // within an ulp: the remainder below is exact
    float re;
    const float rem = two_sum(fmaf(-s, s, g), c, re);
    s0 = s;
    s1 = __fmul_rn(rem, h);
    const float rem2 = fmaf(-s1, s1, fmaf(-2.f * s, s1, rem) + (re + d));
    s2 = rem2 * h;
}

struct TotalsAcc {
    Sum3 w, we, wu;
    double d[3] = {0.0, 0.0, 0.0};

    __device__ __forceinline__ void flush()
    {
        d[0] += w.take();
        d[1] += we.take();
        d[2] += wu.take();
    }

    template <bool PHOTON>
    __device__ __forceinline__ void add(float ux, float uy, float uz, float wt)
    {
        // u^2 = h + l + m
        const float p1 = __fmul_rn(ux, ux), p2 = __fmul_rn(uy, uy), p3 = __fmul_rn(uz, uz);
        float t1, t2, r1, r2, r3, r4;
        const float h = two_sum(two_sum(p1, p2, t1), p3, t2);
        const float q1 = two_sum(fmaf(ux, ux, -p1), fmaf(uy, uy, -p2), r1);
        const float q2 = two_sum(t1, t2, r2);
        const float l = two_sum(two_sum(q1, q2, r3), fmaf(uz, uz, -p3), r4);
        const float m = (r1 + r2) + (r3 + r4);
        const bool rest = (ux == 0.f) & (uy == 0.f) & (uz == 0.f);
        const float aw = fabsf(wt);
        // E <= 1.5 max(1, |u|): the products with the weight stay below 1e35
        const bool fast = (rest || (h >= 1e-18f && h <= 1e28f)) &&
                          (wt == 0.f || (aw >= 1e-10f && aw <= 1e30f && aw * rsqrtf(fmaxf(1.f, h)) * fmaxf(1.f, h) <= 5e34f));
        if (!fast) {
            const double x = ux, y = uy, z = uz, W = wt;
            const double u = sqrt(x * x + y * y + z * z);
            d[0] += W;
            d[1] += W * (PHOTON ? u : sqrt(1.0 + u * u));
            d[2] += W * u;
            return;
        }
        w.add(wt);
        float s0, s1, s2;
        sqrt3(rest ? 1.f : h, l, m, s0, s1, s2);
        if (rest) s0 = s1 = s2 = 0.f;
        float P = __fmul_rn(wt, s0), Q = __fmul_rn(wt, s1);
        wu.add(P, fmaf(wt, s0, -P), Q, fmaf(wt, s1, -Q) + wt * s2);
        if (!PHOTON) {
            float g1, c1, e;
            const float g = two_sum(1.f, h, g1);
            const float cc = two_sum(g1, l, c1);
            const float gn = two_sum(g, cc, e);
            sqrt3(gn, e, c1 + m, s0, s1, s2);
            P = __fmul_rn(wt, s0);
            Q = __fmul_rn(wt, s1);
            we.add(P, fmaf(wt, s0, -P), Q, fmaf(wt, s1, -Q) + wt * s2);
        }
    }
};

// First cell of [0, n_cells) whose region ends after slot (a 33-way search by the warp).
__device__ __forceinline__ int cell_of_slot(const int* start, int n_cells, int slot, int lane)
{
    int lo = 0, n = n_cells;   // the answer is in [lo, lo + n), or n_cells
    while (n > 0) {
        const int step = (n + 32) / 33;
        const int i = lo + (lane + 1) * step;              // lane's boundary
        const bool after = i >= lo + n || start[i] > slot; // the answer lies before i
        const int k = __ffs(__ballot_sync(0xffffffffu, after)) - 1;
        const int k0 = k < 0 ? 32 : k;
        const int hi = min(lo + n, lo + (k0 + 1) * step);
        lo += k0 * step;
        if (step == 1) break;
        n = hi - lo;
    }
    return lo;
}

// One warp's share of the live particles: the slots [S g/W, S (g+1)/W) of all
// S region slots (warp g of W), lanes over the particles of a cell with four
// loads of each array in flight.  Shares by slots and not by cells, because
// occupancies differ by a factor of a hundred: with whole cells dealt to the
// warps the heaviest warp had more than twice the mean.  Extents are read for
// 32 cells at a time.  The lane's sums end in acc.d.
template <bool PHOTON>
__device__ __forceinline__ void totals_share(const pcc_species& sp, int n_cells, int g, int W, int lane, TotalsAcc& acc)
{
    const int base = sp.cell_start[0];
    const long long S = (long long)sp.cell_start[n_cells] - base;
    const int s0 = base + (int)(S * g / W), s1 = base + (int)(S * (g + 1) / W);
    int adds = 0;
    bool more = s0 < s1;
    for (int c = more ? cell_of_slot(sp.cell_start, n_cells, s0, lane) : 0; more; c += 32) {
        const int ci = c + lane;
        int b = s1, e = s1;
        if (ci < n_cells) {
            b = sp.cell_start[ci];
            e = min(b + sp.cell_count[ci], s1);
        }
        more = __all_sync(0xffffffffu, b < s1);   // else the share ends within these cells
        b = max(b, s0);
        unsigned live = __ballot_sync(0xffffffffu, b < e);
        while (live) {
            const int src = __ffs(live) - 1;
            live &= live - 1u;
            const int cb = __shfl_sync(0xffffffffu, b, src), nc = __shfl_sync(0xffffffffu, e, src) - cb;
            for (int k0 = 0; k0 < nc; k0 += 128) {
                float x[4], y[4], z[4], w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int k = k0 + 32 * j + lane;
                    const bool in = k < nc;
                    x[j] = in ? sp.ux[cb + k] : 0.f;
                    y[j] = in ? sp.uy[cb + k] : 0.f;
                    z[j] = in ? sp.uz[cb + k] : 0.f;
                    w[j] = in ? sp.w[cb + k] : 0.f;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (k0 + 32 * j < nc) acc.add<PHOTON>(x[j], y[j], z[j], w[j]);   // warp-uniform
                adds += 4;
                if (adds >= kFlushAdds) { acc.flush(); adds = 0; }
            }
        }
    }
    acc.flush();
    if (PHOTON) acc.d[1] = acc.d[2];
}

// The block's three sums to partial[3 blockIdx.x ..], in a fixed order.
__device__ __forceinline__ void totals_block_out(const TotalsAcc& acc, double (*sh)[32], double* partial)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = 0; i < 3; ++i) {
        const double s = warp_sum(acc.d[i]);
        if (lane == 0) sh[i][wid] = s;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double t = 0.0;
        for (int k = 0; k < nw; ++k) t += sh[threadIdx.x][k];
        partial[3 * blockIdx.x + threadIdx.x] = t;
    }
}

// Partial sums of nb blocks to out[0..2]: one warp per sum, lanes over the
// blocks in a fixed order (a single thread took 51 us for 304 blocks).
__device__ __forceinline__ void totals_reduce(const double* partial, int nb, double* out)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid >= 3) return;
    double t = 0.0;
    for (int b = lane; b < nb; b += 32) t += partial[3 * b + wid];
    t = warp_sum(t);
    if (lane == 0) out[wid] = t;
}

}  // namespace pcc
