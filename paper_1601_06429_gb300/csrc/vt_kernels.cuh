// vt_kernels.cuh -- host-side launch wrappers shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "vt_internal.cuh"

namespace vt {

// sorted FP64 particle record (x, y, z, mass)
struct __align__(32) dpt4 {
    double x, y, z, w;
};

// A float as a double by integer arithmetic (the conversion instruction runs at the FP64 rate, 1/64 of the FP32 one);
// zeros and denormals, which the shift would misplace, and the rest take the same bits as a cast.
__device__ __forceinline__ double f2d(float v) {
    const uint32_t b = __float_as_uint(v), m = b & 0x7fffffffu;
    if (m < 0x00800000u || m >= 0x7f800000u) return (double)v;
    return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
}

size_t scan_tmp_bytes(int64_t n);
size_t radix_tmp_bytes(int64_t N);
int scan_u32_u32(const uint32_t* in, uint32_t* out, int64_t n, void* tmp, cudaStream_t s);
int scan_u16_i64(const uint16_t* in, int64_t* out, int64_t n, void* tmp, cudaStream_t s);
int radix_sort(uint64_t* key, uint32_t* val, uint64_t* key_alt, uint32_t* val_alt, int64_t N, int bits, void* tmp,
                cudaStream_t s);
int launch_key(const void* pos, int dtype, int64_t N, const Geometry& g, uint64_t* key, uint32_t* idx, DevStatus* st,
                cudaStream_t s);
int launch_gather(const void* pos, const void* mass, int dtype, const uint32_t* perm, int64_t N, void* spos,
                   float4* spos4, uint32_t* inv, cudaStream_t s);
int launch_key_batched(const void* pos, int dtype, int64_t N, const Geometry* sgeo, const uint32_t* setid,
                       uint64_t* key, uint32_t* idx, DevStatus* st, cudaStream_t s);
int launch_set_ids(const int64_t* soff, int n_sets, int64_t N, uint32_t* setid, cudaStream_t s);
int launch_gather_u32(const uint32_t* src, const uint32_t* perm, int64_t N, uint32_t* dst, cudaStream_t s);
int launch_owned_list(const uint32_t* inv, int64_t n_owned, uint32_t* list, DevStatus* st, cudaStream_t s);
void tree_layout(int64_t N, Tree& t);
int launch_tree(const void* spos, int dtype, int64_t N, Tree& t, cudaStream_t s);

// clipping (vt_clip.cu)
struct ClipArgs {
    const void* spos;
    int64_t N;
    Geometry geo;
    Tree tree;
    int k_target;
    int max_passes;
    int radius_policy;  // 0: radius doubling; 1: next pass also limited by the density seen so far
    CellOut* cell;
    uint32_t* face_start;
    uint16_t* face_count;
    uint8_t* cstat;
    uint32_t* exact_list;
    Face* faces;
    uint64_t face_cap;
    DevStatus* st;
    double* xws;   // exact workspace, per warp
    int xws_warps;
    // batched independent sets (NULL for one set): set of each sorted particle, geometry of each set, and the
    // sorted index range [soff[s], soff[s+1]) of each set
    const uint32_t* sset;
    const Geometry* sgeo;
    const int64_t* soff;
    // FP32 filter: the thread-per-cell and lane-group kernels run first and list here (N entries) the cells the
    // warp kernel must take; NULL: the warp kernel takes every cell
    uint32_t* warp_list;
    // batched sets: per-set clipping configuration (k_target in the low 16 bits, bits 16-17: the threads-per-cell
    // mode below), or NULL for the handle's parameters
    const int32_t* set_cfg;
    // threads per cell as a mode: 0 one warp, 1 one thread, 2 four lanes, 3 eight lanes (the handle's; cells of
    // sets with a configuration take that set's), and the modes present among the cells (bit m: mode m)
    int tpc_mode;
    int modes;
    // list_given: warp_list already holds the cells to compute (st->n_warp_cells of them; the other particles
    // are candidates only) and no thread-per-cell kernel runs
    int list_given;
    // the lane-group kernels compute the cells of input rows [0, n_own) only (N: all), told by perm (sorted -> input)
    int64_t n_own;
    const uint32_t* perm;
    // the sorted positions in FP32 for its search (spos itself for FP32 positions)
    const float4* spos4;
    // per-cell radius (sorted order): an upper bound of the largest vertex distance of the final cell, or NULL
    float* rad;
};
// The lane-group kernels' memory (vt_clip_group.cu): per cell of a chunk its status, header, candidate list and the
// state kept between radius passes (with the lists of cells 2.6 KB a cell; chunks of at most GROUP_CHUNK cells), and the
// queue counters of every launch.
constexpr int GROUP_CAND = 96;
constexpr int GROUP_NT = 64, GROUP_NP = 40;  // vertex slots and planes of a cell
constexpr int GROUP_STATE = (GROUP_NT * 20 + GROUP_NP * 21 + 15) / 16 * 16;
constexpr int GROUP_PASSES = 12;
constexpr uint32_t GROUP_CHUNK = 1u << 21;
struct __align__(16) GHdr {
    float rlo2, rhi2, B, cap2;                // range of |d|^2 of the pass, start box, widest search
    float bx0, by0, bz0, bx1, by1, bz1;       // box around the vertices
    uint32_t vlo, vhi, n, meta;               // slots in use; candidates | cuts so far << 16; planes | start walls << 8 | FP64 << 16 | passes << 24
    float first2;                             // squared first radius
};
struct GroupBuf {
    uint8_t* stat;         // wants a pass
    GHdr* hdr;
    uint32_t* list;        // [GROUP_CAND] a cell, in order of distance
    unsigned char* state;  // [GROUP_STATE] a cell
    uint32_t* act;         // [2 * chunk] cells listed for a pass
    uint32_t* ctr;         // [group_counters(N)], zero before the launches
    uint32_t chunk;        // cells of a chunk (a multiple of 32)
};
inline uint32_t group_chunk(int64_t N) {
    const int64_t n = (N + 31) / 32 * 32;
    return n < (int64_t)GROUP_CHUNK ? (uint32_t)n : GROUP_CHUNK;
}
inline size_t group_counters(int64_t N) {
    return 2 * 4 * (size_t)GROUP_PASSES * (size_t)((N + group_chunk(N) - 1) / group_chunk(N));
}
int launch_clip(const ClipArgs& a, const GroupBuf* gb, int dtype, int precision, int sm_count, cudaStream_t s);
int launch_clip_exact(const ClipArgs& a, int dtype, int sm_count, cudaStream_t s);
int launch_clip_thread(const ClipArgs& a, int dtype, int sm_count, cudaStream_t s);
int launch_clip_group(const ClipArgs& a, const GroupBuf& b, int dtype, int lanes, int sm_count, cudaStream_t s);
// Counters of the volume-averaged grid and of the weighted gradient, zero before their launches
struct GridCounters {
    unsigned n_retry, n_fail;  // listed pairs (cells), parts that could not be computed
    unsigned queue;            // next cells to look at
    unsigned pad;
    unsigned long long n_big;      // listed cells over many voxels above bit BIG_BITS, their units of GV_BIG pairs below
    unsigned long long big_queue;  // next unit
};
int launch_fma_probe(int blocks, int iters, float* sink, cudaStream_t s);
int launch_fma_probe64(int blocks, int iters, double* sink, cudaStream_t s);
int launch_cvt_weighted(const void* spos, int dtype, int64_t N, const Geometry& g, const Face* faces,
                        const uint32_t* face_start, const uint16_t* face_count, const CellOut* cell, const float* rad,
                        const uint32_t* perm, const void* w, void* out, int4* retry, unsigned retry_cap,
                        GridCounters* counters, int sm_count, cudaStream_t s);
int launch_grid_volume(const void* spos, int dtype, int64_t N, const Geometry& g, const Face* faces,
                       const uint32_t* face_start, const uint16_t* face_count, const double* dens_sorted, const float* rad,
                       const CellOut* cell, uint32_t* big, uint64_t* big_unit, int G, double* acc, int4* retry, unsigned retry_cap,
                       GridCounters* counters, void* out, int sm_count,
                       cudaStream_t s);
int launch_gradient_gg(const Face* faces, const uint32_t* face_start, const uint16_t* face_count, const CellOut* cell,
                       const double* dens_sorted, const uint32_t* perm, int64_t N, void* grad, int dtype,
                       cudaStream_t s);
size_t exact_ws_doubles_per_warp();

// post-processing (vt_post.cu)
int launch_out_vol(const CellOut* cell, const uint32_t* perm, int64_t N, void* vol, int dtype, cudaStream_t s);
int launch_out_rad(const float* rad, const uint32_t* perm, int64_t N, void* out, int dtype, cudaStream_t s);
int launch_cell_flags(const uint8_t* cstat, const uint32_t* perm, int64_t N, uint8_t* out, cudaStream_t s);
int launch_density(const CellOut* cell, const void* spos, int dtype, const uint32_t* perm, int64_t N,
                    double* dens_sorted, void* dens, cudaStream_t s);
int launch_nbr_count(const uint16_t* face_count, const uint32_t* inv, int64_t N, uint16_t* cnt_in, cudaStream_t s);
int launch_nbr_emit(const Face* faces, const uint32_t* face_start, const uint16_t* face_count, const uint32_t* perm,
                     const uint32_t* inv, const int64_t* nbr_off, int64_t N, int32_t* nbr_id, cudaStream_t s);
int launch_gradient(const Face* faces, const uint32_t* face_start, const uint16_t* face_count, const double* dens_sorted,
                     const uint32_t* perm, int64_t N, void* grad, int dtype, cudaStream_t s);
int launch_grid(const void* spos, int dtype, int64_t N, const Geometry& g, const Face* faces,
                const uint32_t* face_start, const uint16_t* face_count, const uint64_t* keys,
                const double* dens_sorted, const uint32_t* perm, int G, int S, void* grid, cudaStream_t s);
int launch_moments(const CellOut* cell, const void* spos, int dtype, const uint32_t* perm, int64_t N,
                   const Geometry& g, void* cen, void* energy, cudaStream_t s);
int launch_backward(const Face* faces, const uint32_t* face_start, const uint16_t* face_count, const CellOut* cell,
                     const void* spos, int dtype, const uint32_t* perm, const uint32_t* inv, int64_t N,
                     const void* dLdV, double dLdE, void* out, cudaStream_t s);

}  // namespace vt
