// Device view of a species and the commit of a cell's secondaries.
#pragma once

#include "pcc_device.cuh"

namespace pcc {

struct SpeciesView {
    float *ux, *uy, *uz, *w, *x;
    uint64_t* pid;
    const int* start;
    int* count;
    int* added;
};

__host__ __device__ inline SpeciesView view_of(const pcc_species& s)
{
    return SpeciesView{s.ux, s.uy, s.uz, s.w, s.x, s.pid, s.cell_start, s.cell_count, s.cell_added};
}

// Orders the records appended to cell c by pid (they arrive in the order of
// atomics) and makes them live.
__device__ __forceinline__ void commit_cell(const SpeciesView& sp, int c)
{
    const int a = sp.added[c];
    if (a == 0) return;
    const int b = sp.start[c] + sp.count[c];
    for (int i = 1; i < a; ++i) {   // insertion sort of the (few) appended records
        const uint64_t kp = sp.pid[b + i];
        const float vx = sp.ux[b + i], vy = sp.uy[b + i], vz = sp.uz[b + i], vw = sp.w[b + i];
        const float vxx = sp.x ? sp.x[b + i] : 0.f;
        int j = i - 1;
        while (j >= 0 && sp.pid[b + j] > kp) {
            sp.pid[b + j + 1] = sp.pid[b + j];
            sp.ux[b + j + 1] = sp.ux[b + j];
            sp.uy[b + j + 1] = sp.uy[b + j];
            sp.uz[b + j + 1] = sp.uz[b + j];
            sp.w[b + j + 1] = sp.w[b + j];
            if (sp.x) sp.x[b + j + 1] = sp.x[b + j];
            --j;
        }
        sp.pid[b + j + 1] = kp;
        sp.ux[b + j + 1] = vx; sp.uy[b + j + 1] = vy; sp.uz[b + j + 1] = vz; sp.w[b + j + 1] = vw;
        if (sp.x) sp.x[b + j + 1] = vxx;
    }
    sp.count[c] += a;
    sp.added[c] = 0;
}

}  // namespace pcc
