// vt_grid.cuh -- shared parts of the volume-averaged grid's kernels: arguments, a cell's voxels, a voxel's box.
#pragma once
#include "vt_kernels.cuh"

namespace vt {

struct GridArgs {
    const void* spos;
    int64_t N;
    Geometry geo;
    const Face* faces;
    const uint32_t* face_start;
    const uint16_t* face_count;
    const double* dens;  // sorted order
    const float* rad;    // bound of each cell's radius
    const CellOut* cell;
    uint32_t* big;       // cells whose ball meets more than GV_BIG voxels, and the first unit of work of each
    uint64_t* big_unit;
    GridCounters* ctr;
    int G;
    double h[3];         // voxel side L / G
    double* acc;         // [G^3] sum of rho |cell & voxel|
    int4* retry;         // (cell, voxel x, y, z unwrapped) for the larger polytope
    unsigned retry_cap;
};

// a part that cannot be computed
__device__ __forceinline__ void grid_fail(const GridArgs& A) { atomicAdd(&A.ctr->n_fail, 1u); }

__device__ __forceinline__ void push_retry(const GridArgs& A, int64_t k, int ax, int ay, int az) {
    const unsigned slot = atomicAdd(&A.ctr->n_retry, 1u);
    if (slot < A.retry_cap) A.retry[slot] = make_int4((int)k, ax, ay, az);
    else grid_fail(A);
}

// the voxels that the ball of sorted particle k meets: first index and count per axis; returns their number
__device__ __forceinline__ int64_t ball_voxels(const GridArgs& A, const double* xi, float r, int* a0, int* n) {
    int64_t m = 1;
    for (int c = 0; c < 3; c++) {
        int64_t lo = (int64_t)floor((xi[c] - (double)r - A.geo.lo[c]) / A.h[c]);
        int64_t hi = (int64_t)floor((xi[c] + (double)r - A.geo.lo[c]) / A.h[c]);
        if (!A.geo.periodic) {
            lo = lo < 0 ? 0 : lo;
            hi = hi > A.G - 1 ? A.G - 1 : hi;
        }
        a0[c] = (int)lo;
        n[c] = (int)(hi - lo + 1);
        m *= hi - lo + 1;
    }
    return m;
}

// linear index of voxel (ax, ay, az) (unwrapped), and its box relative to xi, cut down to the ball's
__device__ __forceinline__ int64_t voxel_box(const GridArgs& A, const double* xi, float r, const int* ia, float* lo, float* hi) {
    int64_t v[3];
    for (int c = 0; c < 3; c++) {
        int q = ia[c] % A.G;
        if (q < 0) q += A.G;
        v[c] = q;
        const double sl = (double)((ia[c] - q) / A.G) * A.geo.L[c];
        lo[c] = fmaxf((float)(A.geo.lo[c] + (double)q * A.h[c] + sl - xi[c]), -r);
        hi[c] = fminf((float)(A.geo.lo[c] + (double)(q + 1) * A.h[c] + sl - xi[c]), r);
    }
    return (v[2] * A.G + v[1]) * A.G + v[0];
}

// -1: the box lies outside a facet plane; else the number of facet planes that cross it (0: it lies inside all)
__device__ __forceinline__ int side_of_box(const GridArgs& A, uint32_t st, int cnt, const float* lo, const float* hi) {
    if (!(lo[0] < hi[0] && lo[1] < hi[1] && lo[2] < hi[2])) return -1;
    int n = 0;
    for (int q = 0; q < cnt; q++) {
        const float4 f = *reinterpret_cast<const float4*>(&A.faces[st + q]);
        const float h = 0.5f * __fmaf_rn(f.z, f.z, __fmaf_rn(f.y, f.y, f.x * f.x));
        const float x0 = f.x * lo[0], x1 = f.x * hi[0], y0 = f.y * lo[1], y1 = f.y * hi[1], z0 = f.z * lo[2], z1 = f.z * hi[2];
        if (fminf(x0, x1) + fminf(y0, y1) + fminf(z0, z1) > h) return -1;
        n += fmaxf(x0, x1) + fmaxf(y0, y1) + fmaxf(z0, z1) > h;
    }
    return n;
}

int launch_grid_pairs(const GridArgs& a, int dtype, int sm_count, cudaStream_t s);

}  // namespace vt
