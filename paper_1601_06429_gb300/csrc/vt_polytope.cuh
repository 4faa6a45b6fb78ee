// vt_polytope.cuh -- a convex polytope that stays one under cuts whose side tests carry rounding errors.
//
// A simple polytope (three planes at a vertex) is held as its vertices, the three neighbours of each and the planes.  A
// plane removes the vertices on its outer side, and every edge between a removed and a kept vertex gets a new vertex on
// it.  Where planes meet within rounding of one point the signs of the tests may contradict each other: the vertices
// removed, or those kept, fall apart into several groups, and the new face would be several loops.  Exact signs never do
// that, so groups apart from the vertex farthest out (or farthest in) are there by rounding alone and change sides.  With
// both sides connected the boundary is one loop that meets a face at most once, which keeps the polytope simple and any
// two faces on at most one common edge; a cut never fails but for room.
// New vertices are taken on the edge, by the distances of its ends, and not as the intersection of three planes: they lie
// between the ends however small the angle of the planes, within a rounding of the extent a cut.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace vt {

// distance of (x, y, z) beyond the plane n.y <= h (times |n|), and the part of the edge from the removed to the kept end
// (distances so, si) that lies before the plane
__host__ __device__ __forceinline__ float beyond(const float4& pl, float x, float y, float z) {
    return fmaf(pl.x, x, fmaf(pl.y, y, fmaf(pl.z, z, -pl.w)));
}
__host__ __device__ __forceinline__ float edge_part(float so, float si) {
    return !(so > 0.f) ? 0.f : !(si < 0.f) ? 1.f : so / (so - si);
}

// One thread's polytope of up to NV vertices and NP planes (indices of one byte).
template <int NV, int NP>
struct Poly {
    static_assert(NV % 32 == 0 && NV <= 256 && NP <= 255, "indices of one byte");
    float x[NV], y[NV], z[NV];
    uint8_t ad[NV][3], id[NV][3];  // neighbour across edge k (id k -> id k+1), and the plane ids, counter-clockwise
    float4 pl[NP];
    unsigned live[NV / 32];
    int np;

    __host__ __device__ static bool has(const unsigned* m, int s) { return (m[s >> 5] >> (s & 31)) & 1u; }
    __host__ __device__ static void put(unsigned* m, int s) { m[s >> 5] |= 1u << (s & 31); }
    __host__ __device__ static int lowest(unsigned m) {
#ifdef __CUDA_ARCH__
        return __ffs((int)m) - 1;
#else
        return __builtin_ctz(m);
#endif
    }

    // the box [lo, hi]: corner k takes the upper wall of axis c unless bit c of k is set; walls x upper 0 / lower 1, ...
    __host__ __device__ void box(const float* lo, const float* hi) {
        for (int w = 0; w < 6; w++) {
            const float sg = (w & 1) ? -1.f : 1.f;
            pl[w].x = w < 2 ? sg : 0.f;
            pl[w].y = (w >> 1) == 1 ? sg : 0.f;
            pl[w].z = w > 3 ? sg : 0.f;
            pl[w].w = (w & 1) ? -lo[w >> 1] : hi[w >> 1];
        }
        np = 6;
        for (int w = 0; w < NV / 32; w++) live[w] = 0u;
        live[0] = 0xffu;
        for (int k = 0; k < 8; k++) {
            const bool even = (((k >> 2) ^ (k >> 1) ^ k) & 1) == 0;
            const uint8_t X = (k & 1) ? 1 : 0, Y = (k & 2) ? 3 : 2, Z = (k & 4) ? 5 : 4;
            const uint8_t fx = (uint8_t)(k ^ 1), fy = (uint8_t)(k ^ 2), fz = (uint8_t)(k ^ 4);
            x[k] = (k & 1) ? lo[0] : hi[0];
            y[k] = (k & 2) ? lo[1] : hi[1];
            z[k] = (k & 4) ? lo[2] : hi[2];
            id[k][0] = X; id[k][1] = even ? Y : Z; id[k][2] = even ? Z : Y;
            ad[k][0] = even ? fz : fy; ad[k][1] = fx; ad[k][2] = even ? fy : fz;
        }
    }

    // the vertices of `in` reached from `seed` over edges within it
    __host__ __device__ void reach(int seed, const unsigned* in, unsigned* out) const {
        for (int w = 0; w < NV / 32; w++) out[w] = 0u;
        uint8_t todo[NV];
        int n = 0;
        put(out, seed);
        todo[n++] = (uint8_t)seed;
        while (n > 0) {
            const int s = todo[--n];
            for (int k = 0; k < 3; k++) {
                const int t = ad[s][k];
                if (has(in, t) && !has(out, t)) {
                    put(out, t);
                    todo[n++] = (uint8_t)t;
                }
            }
        }
    }

    // Cut by n.y <= h.  0: done (perhaps nothing to cut), 1: nothing is left, -1: no room.
    __host__ __device__ int cut(const float4& f) {
        unsigned rem[NV / 32], keep[NV / 32];
        int far_out = -1, far_in = -1;
        float so = 0.f, si = 0.f;
        for (int w = 0; w < NV / 32; w++) {
            unsigned r = 0u;
            for (unsigned m = live[w]; m; m &= m - 1u) {
                const int b = lowest(m), s = 32 * w + b;
                const float d = beyond(f, x[s], y[s], z[s]);
                if (d > 0.f) {
                    r |= 1u << b;
                    if (far_out < 0 || d > so) { so = d; far_out = s; }
                } else if (far_in < 0 || d < si) {
                    si = d;
                    far_in = s;
                }
            }
            rem[w] = r;
            keep[w] = live[w] & ~r;
        }
        if (far_out < 0) return 0;
        if (far_in < 0) return 1;
        if (np == NP) {  // planes that no vertex lies on are dropped
            uint8_t map[NP];
            for (int p = 0; p < NP; p++) map[p] = p < 6;
            for (int w = 0; w < NV / 32; w++)
                for (unsigned m = live[w]; m; m &= m - 1u)
                    for (int k = 0; k < 3; k++) map[id[32 * w + lowest(m)][k]] = 1;
            np = 0;
            for (int p = 0; p < NP; p++)
                if (map[p]) {
                    pl[np] = pl[p];
                    map[p] = (uint8_t)np++;
                }
            for (int w = 0; w < NV / 32; w++)
                for (unsigned m = live[w]; m; m &= m - 1u)
                    for (int k = 0; k < 3; k++) id[32 * w + lowest(m)][k] = map[id[32 * w + lowest(m)][k]];
            if (np == NP) return -1;
        }
        // the new vertices, one on each edge of the boundary (from plane bx to by, cut off vertex bs, kept neighbour bn);
        // first / last: those whose edge leaves / enters a plane
        uint8_t bx[NP], by[NP], bs[NP], bn[NP], bk[NP], bt[NP], first[NP], last[NP], next[NP];
        float vx[NP], vy[NP], vz[NP];
        int nb = 0;
        for (int tries = 0;; tries++) {
            bool full = false;
            nb = 0;
            for (int w = 0; w < NV / 32; w++)
                for (unsigned m = rem[w]; m; m &= m - 1u) {
                    const int s = 32 * w + lowest(m);
                    for (int k = 0; k < 3; k++) {
                        const int t = ad[s][k];
                        if (has(rem, t)) continue;
                        if (nb == NP) {
                            full = true;
                            continue;
                        }
                        bs[nb] = (uint8_t)s;
                        bn[nb] = (uint8_t)t;
                        bx[nb] = id[s][k];
                        by[nb] = id[s][k == 2 ? 0 : k + 1];
                        next[bx[nb]] = by[nb];
                        nb++;
                    }
                }
            // one loop: back at the first plane after all edges and not before (else an entry may never have been written)
            int steps = 0, p = bx[0];
            if (!full) do {
                p = next[p];
                steps++;
            } while (p != bx[0] && p < NP && steps < nb);
            if (!full && p == bx[0] && steps == nb) break;
            if (tries) return -1;
            unsigned m[NV / 32];
            reach(far_out, rem, m);
            for (int w = 0; w < NV / 32; w++) rem[w] = live[w] & ~m[w];
            reach(far_in, rem, keep);
            for (int w = 0; w < NV / 32; w++) rem[w] = live[w] & ~keep[w];
        }
        int word = 0;
        unsigned room = ~keep[0];
        for (int i = 0; i < nb; i++) {
            const int s = bs[i], t = bn[i];
            while (!room) {
                if (++word == NV / 32) return -1;
                room = ~keep[word];
            }
            const int slot = 32 * word + lowest(room);
            room &= room - 1u;
            const float e = edge_part(beyond(f, x[s], y[s], z[s]), beyond(f, x[t], y[t], z[t]));
            vx[i] = fmaf(e, x[t] - x[s], x[s]);
            vy[i] = fmaf(e, y[t] - y[s], y[s]);
            vz[i] = fmaf(e, z[t] - z[s], z[s]);
            bk[i] = (uint8_t)(ad[t][0] == s ? 0 : ad[t][1] == s ? 1 : 2);
            bt[i] = (uint8_t)slot;
            first[bx[i]] = last[by[i]] = (uint8_t)slot;
        }
        for (int w = 0; w < NV / 32; w++) live[w] = keep[w];
        for (int i = 0; i < nb; i++) {
            const int t = bt[i];
            put(live, t);
            x[t] = vx[i]; y[t] = vy[i]; z[t] = vz[i];
            id[t][0] = bx[i]; id[t][1] = by[i]; id[t][2] = (uint8_t)np;
            ad[t][0] = bn[i]; ad[t][1] = first[by[i]]; ad[t][2] = last[bx[i]];
            ad[bn[i]][bk[i]] = (uint8_t)t;
        }
        pl[np++] = f;
        return 0;
    }

    // The volume from the edges: the edge a -> b of a vertex bounds the face of plane b, so a face's area is the sum of
    // n.(w x w') / 2 over its edges, w relative to the mean vertex, and the volume a third of offset times area.
    __host__ __device__ float volume() const {
        float mx = 0.f, my = 0.f, mz = 0.f;
        int n = 0;
        for (int w = 0; w < NV / 32; w++)
            for (unsigned m = live[w]; m; m &= m - 1u) {
                const int s = 32 * w + lowest(m);
                mx += x[s]; my += y[s]; mz += z[s];
                n++;
            }
        const float im = 1.f / (float)(n > 0 ? n : 1);
        mx *= im; my *= im; mz *= im;
        float vol = 0.f;
        for (int w = 0; w < NV / 32; w++)
            for (unsigned m = live[w]; m; m &= m - 1u) {
                const int s = 32 * w + lowest(m);
                const float ax = x[s] - mx, ay = y[s] - my, az = z[s] - mz;
                for (int k = 0; k < 3; k++) {
                    const int t = ad[s][k];
                    const float4 p = pl[id[s][k == 2 ? 0 : k + 1]];
                    const float bx = x[t] - mx, by = y[t] - my, bz = z[t] - mz;
                    const float off = p.w - (p.x * mx + p.y * my + p.z * mz);
                    const float cr = p.x * (ay * bz - az * by) + p.y * (az * bx - ax * bz) + p.z * (ax * by - ay * bx);
                    vol += off * cr / (p.x * p.x + p.y * p.y + p.z * p.z);
                }
            }
        return vol / 6.f;
    }
};

}  // namespace vt
