// Initial sampling of a closed triangle mesh's volume (Sec. 4): cells of side
// 2 r / sqrt(3) over the mesh's bounding box, random candidates (given),
// those inside the mesh (generalized winding number > 1/2) assigned to their
// cells in input order, then per cell the first candidate at least 2 r from
// every sample taken so far.  The cells are taken in 27 phases
// (cx mod 3, cy mod 3, cz mod 3; phase index (cx mod 3) + 3 (cy mod 3) +
// 9 (cz mod 3) ascending): two cells of a phase are three cells apart along
// some axis, more than 2 r, so one launch takes a whole phase, one warp per
// cell, with the result of taking its cells one by one.  The decisions are
// those of a plain sequential evaluation in double precision: taken in single
// precision where a bound on its error allows, and in double with the
// multiplications and additions rounded one by one where it does not.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <vector>

#include "gs.h"
#include "gs_internal.cuh"

namespace {

__device__ __forceinline__ double dot3_rn(const double* a, const double* b)
{
    return __dadd_rn(__dadd_rn(__dmul_rn(a[0], b[0]), __dmul_rn(a[1], b[1])), __dmul_rn(a[2], b[2]));
}

// Solid angle of the triangle seen from p over 4 pi (Van Oosterom and
// Strackee 1983: tan(Omega / 2) = det[a b c] / (|a||b||c| + (a.b)|c| +
// (b.c)|a| + (c.a)|b|), a, b, c the corners relative to p).
__device__ double tri_winding(const double* A, const double* B, const double* C, const double* p)
{
    double a[3], b[3], c[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a[k] = __dsub_rn(A[k], p[k]);
        b[k] = __dsub_rn(B[k], p[k]);
        c[k] = __dsub_rn(C[k], p[k]);
    }
    const double la = sqrt(dot3_rn(a, a)), lb = sqrt(dot3_rn(b, b)), lc = sqrt(dot3_rn(c, c));
    const double m0 = __dsub_rn(__dmul_rn(b[1], c[2]), __dmul_rn(b[2], c[1]));
    const double m1 = __dsub_rn(__dmul_rn(b[0], c[2]), __dmul_rn(b[2], c[0]));
    const double m2 = __dsub_rn(__dmul_rn(b[0], c[1]), __dmul_rn(b[1], c[0]));
    const double det = __dadd_rn(__dsub_rn(__dmul_rn(a[0], m0), __dmul_rn(a[1], m1)), __dmul_rn(a[2], m2));
    const double den = __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(__dmul_rn(la, lb), lc), __dmul_rn(dot3_rn(a, b), lc)),
                                           __dmul_rn(dot3_rn(b, c), la)),
                                 __dmul_rn(dot3_rn(c, a), lb));
    return atan2(det, den) / (2.0 * 3.14159265358979323846);
}

struct SampleGrid {
    double lo[3];
    double h;
    int64_t dims[3];
    int64_t n_cell;
};

// The winding number decides only a comparison with 1/2, so it is first
// evaluated in single precision with a bound on its error, and in double
// precision only for the candidates that the bound leaves open (those within
// about 1e-5 of the mesh's size from an edge, or exactly in a triangle's
// plane inside it).  FP64 runs at 1/64 of the FP32 rate on sm_103a: a million
// candidates against 344 triangles took 92 ms in double precision and take
// 1.2 ms this way (1.1 here, 0.08 in k_sample_winding), with the same
// decisions (a bound as below, and every case that it does not cover left open).  Issue of FP32 instructions (about 65 per candidate and
// triangle) bounds it.
//
// Coordinates are scaled to the mesh's box, q' = (q - lo) / extent, and
// rounded to single precision (the winding number does not change with
// scale).  With u = 2^-24, P = max_k |p'_k| and a, b, c the corners minus p'
// (each component off by less than 2 u (1 + P), each vector by less than
// d = 4 u (1 + P)), l_a, l_b, l_c their lengths, S = l_a l_b + l_b l_c +
// l_c l_a and L = l_a l_b l_c, the numerator det and the denominator den of
// tan(Omega / 2) are multilinear in the corners: inputs move det by at most
// d S and den by at most 4 d S, the roundings of their evaluation move both
// together by at most 128 u L.  The bound D = 10 d S + 256 u L is twice that.
// The angle of (den, det) is then off by at most 1.5 D / h, h = |(det,
// den)|, as long as D < h / 4 and the pair cannot lie on the other side of
// the cut (den < 0 and |det| <= D): otherwise the candidate is left open.
// NaN and infinity (a corner at p, coordinates out of range) leave it open
// too: every comparison is written to fail with them, and 1 / h = 0 says that
// the sum of squares left the range (from about 2e6 box sizes away).
// The angles are summed without an arctangent per triangle: the unit numbers
// (den + i det) / h are multiplied up and the turns counted where the product
// passes the negative real axis (each angle is below a half turn, so it
// passes upwards only from Im > 0 by det > 0 to Im < 0, downwards the other
// way); one atan2f at the end gives the rest.  Each product rounds by less
// than 8 u.  A product exactly on the negative real axis (Im = 0, as round
// angles make it at the centre of a symmetric mesh) is on neither side of the
// cut, and the next angle would pass it uncounted: such a candidate is left
// open.

// A position relative to its cell's centre in units of r, or NaN where single
// precision would not do: more than 64 r away, or a mesh farther from the
// origin than kMaxUnits r (the host then passes a NaN as 1 / r), whose cell
// centres round by more than 2^-52 kMaxUnits = 7e-6 r.
constexpr double kMaxUnits = 3.0e10;

__device__ __forceinline__ float cell_units(double x, double mid, double inv_r)
{
    const float f = (float)(__dsub_rn(x, mid) * inv_r);
    return fabsf(f) <= 64.0f ? f : __int_as_float(0x7fffffff);
}

constexpr int kTriChunk = 128;      // triangles staged per round (6 KB)
constexpr int kTriFloats = 12;      // nine coordinates, padded to three float4

__global__ void k_sample_triangles(const double* __restrict__ V, const int32_t* __restrict__ T, int64_t nt,
                                   const SampleGrid g, double inv_extent, float* __restrict__ tri)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    for (int v = 0; v < 3; ++v)
        for (int k = 0; k < 3; ++k)
            tri[kTriFloats * t + 3 * v + k] = (float)((V[3 * (int64_t)T[3 * t + v] + k] - g.lo[k]) * inv_extent);
    for (int k = 9; k < kTriFloats; ++k) tri[kTriFloats * t + k] = 0.0f;
}

// Inside flag and cell of every candidate; the cell's counter gives the
// candidate its arrival rank (the counting sort puts each cell in index
// order afterwards).  Candidates the single-precision bound leaves open go
// to `open` (*n_open of them, zero on entry).
// surface: every candidate counts (points on the surface), no winding number.
__global__ void __launch_bounds__(128) k_sample_classify(const float4* __restrict__ tri, int64_t nt,
                                                         const double* __restrict__ cand, int64_t nc,
                                                         const SampleGrid g, double inv_extent,
                                                         uint8_t* __restrict__ inside, uint32_t* __restrict__ keys,
                                                         uint32_t* __restrict__ rank,
                                                         uint32_t* __restrict__ cell_count,
                                                         uint32_t* __restrict__ open, uint32_t* __restrict__ n_open,
                                                         float4* __restrict__ rel, double inv_r, int surface)
{
    __shared__ float4 s_tri[kTriChunk * kTriFloats / 4];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = i < nc;   // every thread stays for the staging barriers
    const double p[3] = {live ? cand[3 * i] : 0.0, live ? cand[3 * i + 1] : 0.0, live ? cand[3 * i + 2] : 0.0};
    if (surface) {
        if (live) inside[i] = 1;
    } else {
        constexpr float u = 5.9604645e-8f;   // 2^-24
        const float px = (float)((p[0] - g.lo[0]) * inv_extent), py = (float)((p[1] - g.lo[1]) * inv_extent),
                    pz = (float)((p[2] - g.lo[2]) * inv_extent);
        const float d10 = 40.0f * u * (1.0f + fmaxf(fabsf(px), fmaxf(fabsf(py), fabsf(pz))));
        float zr = 1.0f, zi = 0.0f, E = 0.0f;   // the product, and the sum of D / h
        int turns = 0;
        bool unsure = false;
        for (int64_t t0 = 0; t0 < nt; t0 += kTriChunk) {
            const int n = (int)(nt - t0 < kTriChunk ? nt - t0 : kTriChunk);
            __syncthreads();
            for (int k = threadIdx.x; k < n * (kTriFloats / 4); k += blockDim.x)
                s_tri[k] = __ldg(tri + t0 * (kTriFloats / 4) + k);
            __syncthreads();
            for (int t = 0; t < n; ++t) {
                const float4 q0 = s_tri[3 * t], q1 = s_tri[3 * t + 1], q2 = s_tri[3 * t + 2];
                const float ax = q0.x - px, ay = q0.y - py, az = q0.z - pz;
                const float bx = q0.w - px, by = q1.x - py, bz = q1.y - pz;
                const float cx = q1.z - px, cy = q1.w - py, cz = q2.x - pz;
                const float aa = ax * ax + ay * ay + az * az, bb = bx * bx + by * by + bz * bz,
                            cc = cx * cx + cy * cy + cz * cz;
                const float la = aa * rsqrtf(aa), lb = bb * rsqrtf(bb), lc = cc * rsqrtf(cc);
                const float det = ax * (by * cz - bz * cy) - ay * (bx * cz - bz * cx) + az * (bx * cy - by * cx);
                const float lab = la * lb, L = lab * lc;
                const float den = L + (ax * bx + ay * by + az * bz) * lc + (bx * cx + by * cy + bz * cz) * la +
                                  (cx * ax + cy * ay + cz * az) * lb;
                const float D = d10 * (lab + lc * (la + lb)) + 256.0f * u * L;
                const float rh = rsqrtf(det * det + den * den);
                const float rel = D * rh;
                unsure |= !(rel < 0.25f && rh > 0.0f && (den > 0.0f || fabsf(det) > D));
                E += rel;
                const float c = den * rh, s = det * rh;
                const float nr = zr * c - zi * s, ni = zr * s + zi * c;
                if (zi > 0.0f && s > 0.0f && ni < 0.0f) ++turns;
                if (zi < 0.0f && s < 0.0f && ni > 0.0f) --turns;
                unsure |= ni == 0.0f && !(nr > 0.0f);
                zr = nr;
                zi = ni;
            }
        }
        const float W = fmaf(6.2831853f, (float)turns, atan2f(zi, zr));   // the sum of Omega / 2
        E = unsure ? 1.0e30f : 1.5f * E + 8.0f * u * ((float)nt + fabsf(W));
        if (live) {
            const float away = W - 3.14159265f;   // w = W / (2 pi), compared with 1/2
            if (fabsf(away) > 1.1f * E + 1.0e-5f) inside[i] = away > 0.0f ? 1 : 0;
            else open[atomicAdd(n_open, 1u)] = (uint32_t)i;
        }
    }
    if (!live) return;
    int64_t c[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double f = floor(__ddiv_rn(__dsub_rn(p[k], g.lo[k]), g.h));
        c[k] = f < 0.0 ? 0 : (f >= (double)(g.dims[k] - 1) ? g.dims[k] - 1 : (int64_t)f);
    }
    const uint32_t key = (uint32_t)(c[0] + g.dims[0] * (c[1] + g.dims[1] * c[2]));
    keys[i] = key;
    rank[i] = atomicAdd(cell_count + key, 1u);
    // the position relative to its cell's centre in units of r (k_sample_phase)
    float f[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) f[k] = cell_units(p[k], g.lo[k] + ((double)c[k] + 0.5) * g.h, inv_r);
    rel[i] = make_float4(f[0], f[1], f[2], 0.0f);
}

// The candidates left open, one warp each: the lanes evaluate 32 triangles at
// a time in double precision and the terms are added one by one in triangle
// order, as a sequential evaluation adds them.
__global__ void __launch_bounds__(128) k_sample_winding(const double* __restrict__ V, const int32_t* __restrict__ T,
                                                        int64_t nt, const double* __restrict__ cand,
                                                        const uint32_t* __restrict__ open,
                                                        const uint32_t* __restrict__ n_open,
                                                        uint8_t* __restrict__ inside)
{
    const int lane = (int)(threadIdx.x & 31u);
    const uint32_t n = *n_open, n_warps = gridDim.x * (blockDim.x >> 5);
    for (uint32_t q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < n; q += n_warps) {   // whole warps
        const int64_t i = open[q];
        const double p[3] = {cand[3 * i], cand[3 * i + 1], cand[3 * i + 2]};
        double w = 0.0;
        for (int64_t t0 = 0; t0 < nt; t0 += 32) {
            const int64_t t = t0 + lane;
            double x = 0.0;
            if (t < nt)
                x = tri_winding(V + 3 * (int64_t)T[3 * t], V + 3 * (int64_t)T[3 * t + 1], V + 3 * (int64_t)T[3 * t + 2],
                                p);
            const int m = (int)(nt - t0 < 32 ? nt - t0 : 32);
            for (int k = 0; k < m; ++k) w = __dadd_rn(w, __shfl_sync(0xffffffffu, x, k));
        }
        if (lane == 0) inside[i] = w > 0.5 ? 1 : 0;
    }
}

// One phase: a warp per cell (cx, cy, cz) = (px + 3 i, py + 3 j, pz + 3 k).
// The samples taken so far around a cell (at most one in each of the 5^3
// cells within reach) do not depend on the candidate, so the lanes load them
// once, up to four each, and every candidate of the cell (in order, 32 loaded
// at a time) is tested against all of them at once: in single precision on
// positions relative to the cell, in units of r, and in double precision only
// when a squared distance comes within 1e-3 of the threshold 4, since FP64
// issues at 1/64 of the FP32 rate.  (Coordinates of at most 64 units round by
// 4e-6 each, and kMaxUnits bounds the rounding of a cell's centre, so a
// squared distance near 4 is off by less than 3e-4; farther candidates, beyond
// the mesh's box, become NaN and are tested in double.)
// With one thread per cell and every test in double a phase was a serial
// chain of up to 125 lookups per candidate: 168 us per phase for a million
// candidates in 265,000 cells (52 us with this layout but all tests in
// double), against 13 us.
constexpr int kReach = 125;
constexpr int kPicksPerLane = (kReach + 31) / 32;

__global__ void __launch_bounds__(128) k_sample_phase(const double* __restrict__ cand,
                                                      const uint8_t* __restrict__ inside,
                                                      const uint32_t* __restrict__ order,
                                                      const uint32_t* __restrict__ cell_start,
                                                      const float4* __restrict__ rel, int32_t* __restrict__ pick,
                                                      const SampleGrid g, int px, int py, int pz, int64_t nx,
                                                      int64_t ny, int64_t n_phase, double d2min)
{
    const int lane = (int)(threadIdx.x & 31u);
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= n_phase) return;   // whole warps
    const int64_t cx = px + 3 * (t % nx), cy = py + 3 * ((t / nx) % ny), cz = pz + 3 * (t / (nx * ny));
    const int64_t c = cx + g.dims[0] * (cy + g.dims[1] * cz);
    const uint32_t b = cell_start[c], e = cell_start[c + 1];
    if (b == e) return;
    float sf[kPicksPerLane][3];
    int32_t has[kPicksPerLane];   // the sample, or -1
#pragma unroll
    for (int k = 0; k < kPicksPerLane; ++k) {
        const int n = lane + 32 * k;
        const int64_t x = cx - 2 + n % 5, y = cy - 2 + (n / 5) % 5, z = cz - 2 + n / 25;
        has[k] = -1;
        if (n < kReach && x >= 0 && y >= 0 && z >= 0 && x < g.dims[0] && y < g.dims[1] && z < g.dims[2])
            has[k] = pick[x + g.dims[0] * (y + g.dims[1] * z)];
        sf[k][0] = sf[k][1] = sf[k][2] = 1.0e10f;
        if (has[k] >= 0) {   // a cell's side is 2 / sqrt(3) units
            const float4 f = rel[has[k]];
            sf[k][0] = fmaf((float)(n % 5 - 2), 1.1547005f, f.x);
            sf[k][1] = fmaf((float)((n / 5) % 5 - 2), 1.1547005f, f.y);
            sf[k][2] = fmaf((float)(n / 25 - 2), 1.1547005f, f.z);
        }
    }
    for (uint32_t q0 = b; q0 < e; q0 += 32) {
        const uint32_t q = q0 + (uint32_t)lane;
        uint32_t i = 0;
        bool in = false;
        if (q < e) {
            i = order[q];
            in = inside[i] != 0;
        }
        float4 pf = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in) pf = rel[i];
        unsigned todo = __ballot_sync(0xffffffffu, in);
        while (todo) {   // warp-uniform
            const int j = __ffs(todo) - 1;
            todo &= todo - 1u;
            const float fx = __shfl_sync(0xffffffffu, pf.x, j), fy = __shfl_sync(0xffffffffu, pf.y, j),
                        fz = __shfl_sync(0xffffffffu, pf.z, j);
            bool close = false;
            unsigned near = 0u;   // bit k: pick k is too near the threshold for single precision
#pragma unroll
            for (int k = 0; k < kPicksPerLane; ++k) {
                const float dx = fx - sf[k][0], dy = fy - sf[k][1], dz = fz - sf[k][2];
                const float d2 = dx * dx + dy * dy + dz * dz;
                if (d2 < 3.999f) close = true;
                else if (!(d2 > 4.001f) && has[k] >= 0) near |= 1u << k;   // NaN included
            }
            if (__any_sync(0xffffffffu, near != 0u)) {
                const double* pj = cand + 3 * (int64_t)__shfl_sync(0xffffffffu, i, j);
#pragma unroll
                for (int k = 0; k < kPicksPerLane; ++k) {
                    if (!((near >> k) & 1u)) continue;
                    const double* s = cand + 3 * (int64_t)has[k];
                    const double d[3] = {__dsub_rn(pj[0], s[0]), __dsub_rn(pj[1], s[1]), __dsub_rn(pj[2], s[2])};
                    close |= dot3_rn(d, d) < d2min;
                }
            }
            if (__any_sync(0xffffffffu, close)) continue;
            if (lane == j) pick[c] = (int32_t)i;
            return;
        }
    }
}

struct DevBufs {
    std::vector<void*> p;
    ~DevBufs()
    {
        for (void* q : p) cudaFree(q);
    }
    template <class T>
    bool get(T** out, size_t count)
    {
        void* q = nullptr;
        if (gs_dalloc_bytes(&q, (count ? count : 1) * sizeof(T)) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        p.push_back(q);
        *out = (T*)q;
        return true;
    }
};

struct StreamGuard {
    cudaStream_t s = nullptr;
    ~StreamGuard()
    {
        if (s) {
            cudaStreamSynchronize(s);
            cudaStreamDestroy(s);
        }
    }
};

}  // namespace

static int sample_impl(const double* vertices, int64_t n_vertices, const int32_t* triangles, int64_t n_triangles,
                       const double* candidates, int64_t n_candidates, double r, int64_t* selected, int64_t capacity,
                       int64_t* n_selected, uint8_t* inside, int surface)
{
    if (!n_selected || n_vertices < 0 || n_triangles < 0 || n_candidates < 0 || capacity < 0) return GS_ERR_ARG;
    *n_selected = 0;
    if (!(r > 0.0) || !std::isfinite(r) || (n_vertices > 0 && !vertices) || (n_triangles > 0 && !triangles) ||
        (n_candidates > 0 && !candidates) || (capacity > 0 && !selected) || n_candidates > 0x7fffffffLL ||
        (n_triangles > 0 && n_vertices == 0))
        return GS_ERR_ARG;
    for (int64_t k = 0; k < 3 * n_triangles; ++k)
        if (triangles[k] < 0 || triangles[k] >= n_vertices) return GS_ERR_ARG;
    for (int64_t k = 0; k < 3 * n_vertices; ++k)
        if (!std::isfinite(vertices[k])) return GS_ERR_DOMAIN;
    for (int64_t k = 0; k < 3 * n_candidates; ++k)
        if (!std::isfinite(candidates[k])) return GS_ERR_DOMAIN;
    // the grid, on the host in double precision
    SampleGrid g;
    double hi[3];
    for (int k = 0; k < 3; ++k) g.lo[k] = hi[k] = n_vertices ? vertices[k] : 0.0;
    for (int64_t i = 0; i < n_vertices; ++i)
        for (int k = 0; k < 3; ++k) {
            g.lo[k] = std::fmin(g.lo[k], vertices[3 * i + k]);
            hi[k] = std::fmax(hi[k], vertices[3 * i + k]);
        }
    g.h = 2.0 * r / std::sqrt(3.0);
    // Surface candidates lie on the triangles, so inside the box up to
    // rounding.  One farther out would be clamped into an edge cell, and the
    // phases keep two picks at least 2 r apart only while every candidate is
    // within (2 h - 2 r) / 2 = 0.154 r of its cell: refuse those beyond 0.15 r.
    if (surface) {
        const double m = 0.15 * r;
        for (int64_t i = 0; i < n_candidates; ++i)
            for (int k = 0; k < 3; ++k)
                if (candidates[3 * i + k] < g.lo[k] - m || candidates[3 * i + k] > hi[k] + m) return GS_ERR_ARG;
    }
    double cells = 1.0;
    for (int k = 0; k < 3; ++k) {
        g.dims[k] = (int64_t)std::floor((hi[k] - g.lo[k]) / g.h) + 1;
        cells *= (double)g.dims[k];
    }
    if (cells > 2147483646.0) return GS_ERR_ARG;   // cell ids and picks are 32-bit
    g.n_cell = g.dims[0] * g.dims[1] * g.dims[2];
    const double d2min = 4.0 * r * r;
    const int64_t nc = n_candidates, ncell = g.n_cell;

    StreamGuard sg;
    if (cudaStreamCreateWithFlags(&sg.s, cudaStreamNonBlocking) != cudaSuccess) return GS_ERR_CUDA;
    cudaStream_t s = sg.s;
    DevBufs B;
    double *dV = nullptr, *dC = nullptr;
    int32_t *dT = nullptr, *dpick = nullptr;
    uint8_t* din = nullptr;
    uint32_t *keys = nullptr, *rank = nullptr, *okeys = nullptr, *oidx = nullptr, *start = nullptr, *aux = nullptr;
    float* dtri = nullptr;
    float4* drel = nullptr;
    uint32_t* dopen = nullptr;   // candidates left open, their count in the last word
    if (!B.get(&dV, 3 * (size_t)n_vertices) || !B.get(&dT, 3 * (size_t)n_triangles) || !B.get(&dC, 3 * (size_t)nc) ||
        !B.get(&din, (size_t)nc) || !B.get(&keys, (size_t)nc) || !B.get(&rank, (size_t)nc) ||
        !B.get(&okeys, (size_t)nc) || !B.get(&oidx, (size_t)nc) || !B.get(&start, (size_t)ncell + 1) ||
        !B.get(&aux, gs_scan_aux_words(ncell + 1)) || !B.get(&dpick, (size_t)ncell) ||
        !B.get(&dtri, (size_t)kTriFloats * n_triangles) || !B.get(&dopen, (surface ? 0 : (size_t)nc) + 1) ||
        !B.get(&drel, (size_t)nc))
        return GS_ERR_OOM;
#define SK(call)                                  \
    do {                                          \
        if ((call) != cudaSuccess) {              \
            cudaGetLastError();                   \
            return GS_ERR_CUDA;                   \
        }                                         \
    } while (0)
    int64_t launches = 0;
    if (n_vertices) SK(cudaMemcpyAsync(dV, vertices, 24 * (size_t)n_vertices, cudaMemcpyHostToDevice, s));
    if (n_triangles) SK(cudaMemcpyAsync(dT, triangles, 12 * (size_t)n_triangles, cudaMemcpyHostToDevice, s));
    if (nc) SK(cudaMemcpyAsync(dC, candidates, 24 * (size_t)nc, cudaMemcpyHostToDevice, s));
    SK(gs_cs_clear(s, start, ncell));
    SK(cudaMemsetAsync(dpick, 0xff, sizeof(int32_t) * (size_t)ncell, s));
    if (nc) {
        const double extent = std::fmax(hi[0] - g.lo[0], std::fmax(hi[1] - g.lo[1], hi[2] - g.lo[2]));
        const double inv_extent = extent > 0.0 ? 1.0 / extent : 1.0;
        double reach = 0.0;
        for (int k = 0; k < 3; ++k) reach = std::fmax(reach, std::fmax(std::fabs(g.lo[k]), std::fabs(hi[k])));
        const double inv_r = reach <= kMaxUnits * r ? 1.0 / r : std::nan("");
        uint32_t* n_open = dopen + (surface ? 0 : nc);
        SK(cudaMemsetAsync(n_open, 0, sizeof(uint32_t), s));
        if (n_triangles) {
            k_sample_triangles<<<gs_blocks(n_triangles, 128), 128, 0, s>>>(dV, dT, n_triangles, g, inv_extent, dtri);
            SK(cudaGetLastError());
        }
        k_sample_classify<<<gs_blocks(nc, 128), 128, 0, s>>>((const float4*)dtri, n_triangles, dC, nc, g, inv_extent,
                                                             din, keys, rank, start, dopen, n_open, drel, inv_r,
                                                             surface);
        SK(cudaGetLastError());
        if (!surface) {
            k_sample_winding<<<304, 128, 0, s>>>(dV, dT, n_triangles, dC, dopen, n_open, din);
            SK(cudaGetLastError());
        }
        // stable counting sort by cell: each cell's candidates in input order
        SK(gs_cs_finish(s, nc, ncell, keys, rank, okeys, oidx, start, aux, nullptr, nullptr, nullptr, nullptr,
                        &launches));
        for (int phase = 0; phase < 27; ++phase) {
            const int px = phase % 3, py = (phase / 3) % 3, pz = phase / 9;
            const int64_t nx = (g.dims[0] - px + 2) / 3, ny = (g.dims[1] - py + 2) / 3, nz = (g.dims[2] - pz + 2) / 3;
            const int64_t n_phase = nx * ny * nz;
            if (n_phase <= 0) continue;
            k_sample_phase<<<gs_blocks(n_phase * 32, 128), 128, 0, s>>>(dC, din, oidx, start, drel, dpick, g, px, py, pz,
                                                                        nx, ny, n_phase, d2min);
            SK(cudaGetLastError());
        }
    }
    // the picks, in ascending cell order, compacted on the host
    std::vector<int32_t> pick((size_t)ncell);
    SK(cudaMemcpyAsync(pick.data(), dpick, sizeof(int32_t) * (size_t)ncell, cudaMemcpyDeviceToHost, s));
    if (inside && nc) SK(cudaMemcpyAsync(inside, din, (size_t)nc, cudaMemcpyDeviceToHost, s));
    SK(cudaStreamSynchronize(s));
#undef SK
    int64_t n = 0;
    for (int64_t c = 0; c < ncell; ++c) {
        if (pick[(size_t)c] < 0) continue;
        if (n < capacity) selected[n] = pick[(size_t)c];
        ++n;
    }
    *n_selected = n;
    return n > capacity ? GS_ERR_CAPACITY : GS_OK;
}

extern "C" int gs_sample_volume(const double* vertices, int64_t n_vertices, const int32_t* triangles,
                                int64_t n_triangles, const double* candidates, int64_t n_candidates, double r,
                                int64_t* selected, int64_t capacity, int64_t* n_selected, uint8_t* inside)
{
    return sample_impl(vertices, n_vertices, triangles, n_triangles, candidates, n_candidates, r, selected, capacity,
                       n_selected, inside, 0);
}

extern "C" int gs_sample_surface(const double* vertices, int64_t n_vertices, const double* candidates,
                                 int64_t n_candidates, double r, int64_t* selected, int64_t capacity,
                                 int64_t* n_selected)
{
    return sample_impl(vertices, n_vertices, nullptr, 0, candidates, n_candidates, r, selected, capacity, n_selected,
                       nullptr, 1);
}
