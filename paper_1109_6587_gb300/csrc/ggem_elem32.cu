// FP32 element rule (mixed plans): the local single- and double-layer sums of
// Sec. 3.4.1 / 3.5.2 over quadrature points grouped by triangle.
//
// The triangles are binned by centroid into cells of r_cut/3 and, within each
// cell, ordered by 4 x 4 x 4 sub-cells.  Every cell carries the points of its
// triangles once per quadrature rule:
//   list 0  the 16 collapsed Gauss points of Eq. (int_l),
//   list 1  the 7-point rule of degree 5 (Radon 1948),
//   list 2  the 3-point rule of degree 2 (Strang and Fix 1973),
// and each (target, cell) pair uses one of the lists: list 1 where the whole
// cell is at least kFarEdges = 4 longest edges from the target, list 2 where it
// also is at least kDimRadius / alpha away, list 0 elsewhere.  The rules
// integrate the same product of the linear density and the kernel; over one
// triangle of edge h at distance d they differ by the kernel's Taylor terms beyond degree 4, of order (0.6 h / d)^5, and the kernel
// falls off as exp(-alpha^2 d^2) besides.  Measured in FP64 with N(0,1)
// densities on suspensions of 642- and 162-node spheres and biconcave cells, h / r_cut
// from 0.02 to 0.16, the whole double-layer sums differ by (rms, over the rms
// sum) 0.3e-8 to 1.1e-8 at 5 edges, 1.0e-8 to 5.5e-8 at 4 and 2.7e-8 to 1.3e-7 at
// 3.5, while two orders of summation differ by 2e-7 to 7e-7.  List 2 lives on the kernel's
// decay: beyond kDimRadius = 3 the terms carry exp(-9), and with alpha h <= 0.33
// the sums differ by 6e-10 to 2.3e-8 (2.8: up to 5.2e-8; alpha h = 0.5: 2.2e-7,
// where the list is not used).  Both as dispatched, by cells: 2e-8 to 8e-8 (rms),
// single targets up to 2e-7 of the largest sum.  In candidates per target the lists halve the work of
// dense suspensions and take a third off dilute ones.
// Triangles large against r_cut keep list 0 only, each point in the cell that holds it
// (kBinRadius).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "ggem_internal.cuh"
#include "ggem_erfcx.cuh"

namespace ggem {

namespace {

// ------------------------------------------------------------- the rules
constexpr int kPts[kElemLists] = {16, 7, 3};
constexpr double kFarEdges = 4.0, kDimRadius = 3.0, kDimEdge = 0.33;

// A point can lie two thirds of a triangle's longest edge h nearer to a target than
// the centroid it is binned by, so a cell dropped for lying beyond r_cut holds
// points within it, down to r_cut - 2 h / 3, whose terms carry up to
// exp(-alpha^2 (r_cut - 2 h / 3)^2); and whole steps are summed unmasked, with points
// beyond r_cut, whose terms carry up to exp(-alpha^2 r_cut^2).  Where
// alpha (r_cut - 2 h / 3) < kBinRadius or alpha r_cut < kBinCut every point is
// therefore binned by itself, its terms masked at r_cut, and list 0 is the only one.
// On these lines (FP64, spheres r_cut apart and less) the terms left out and added are
// up to 8e-7 of the largest double-layer sum, nearly all of it added ones (1.2e-6 at
// r_cut = 3.95 / alpha, 3e-6 at 3.75); by centroid, h = 1.2 r_cut was off by
// 3.7e-4 of the whole double layer and r_cut = 2 / alpha by 2.0e-3.  With r_cut =
// 4 / alpha the line is at h = 0.225 r_cut, beyond the last edge with a list 1
// (0.2125).  The price, double layer of 100 spheres: .55 -> .58 ms at h = 0.62 r_cut,
// .73 -> .75 at 0.33; 2.87 -> 4.23 at r_cut = 3.9 / alpha, h = 0.07, which loses lists
// 1 and 2.
constexpr double kBinRadius = 3.4, kBinCut = 3.999;

// search reach in cells and its neighbour offsets
constexpr int R32 = kElemReach, kSide = 2 * R32 + 1, kOffsets = kSide * kSide * kSide;

// phi_v w of point a of a rule on the unit triangle of area 1/2 (FP64)
struct RuleTab {
    double phi[16][3], w[16];
};

struct ListTab {
    double phi[16][3];
};

RuleTab rule_tab(int list, const QuadRule& g) {
    RuleTab r{};
    if (list == 0) {
        for (int a = 0; a < 16; ++a) {
            const double eta = g.t[a >> 2], xi = (1.0 - eta) * g.t[a & 3];
            r.phi[a][0] = 1.0 - xi - eta;
            r.phi[a][1] = xi;
            r.phi[a][2] = eta;
            r.w[a] = g.w[a & 3] * g.w[a >> 2] * (1.0 - eta);
        }
        return r;
    }
    if (list == 2) {
        for (int a = 0; a < 3; ++a) {
            for (int v = 0; v < 3; ++v) r.phi[a][v] = v == a ? 2.0 / 3.0 : 1.0 / 6.0;
            r.w[a] = 1.0 / 6.0;
        }
        return r;
    }
    const double s = std::sqrt(15.0);
    const double b[2] = {(6.0 + s) / 21.0, (6.0 - s) / 21.0};
    const double w[2] = {(155.0 + s) / 2400.0, (155.0 - s) / 2400.0};
    for (int v = 0; v < 3; ++v) r.phi[0][v] = 1.0 / 3.0;
    r.w[0] = 9.0 / 80.0;
    for (int o = 0; o < 2; ++o)
        for (int k = 0; k < 3; ++k) {
            const int a = 1 + 3 * o + k;
            for (int v = 0; v < 3; ++v) r.phi[a][v] = v == k ? 1.0 - 2.0 * b[o] : b[o];
            r.w[a] = w[o];
        }
    return r;
}

// ------------------------------------------------------- layout of a mesh
// Centroids of the triangles (the points the cells are built from).
__global__ void k_centroids(int m, const double* __restrict__ x, const int* __restrict__ tri,
                            double* __restrict__ c) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= m) return;
    const int a = tri[3 * k], b = tri[3 * k + 1], d = tri[3 * k + 2];
    for (int i = 0; i < 3; ++i)
        c[3 * (size_t)k + i] =
            (x[3 * (size_t)a + i] + x[3 * (size_t)b + i] + x[3 * (size_t)d + i]) * (1.0 / 3.0);
}

// Order of the triangles within each cell: 4 x 4 x 4 sub-cells in Morton
// order, so that consecutive points (the 64-point steps) lie close together.
// One block per cell; a counting sort by the 6-bit key into perm_out.
__device__ __forceinline__ int subcell_key(float4 p, float ihx, float ihy, float ihz) {
    const int ix = min(3, max(0, (int)(p.x * ihx))), iy = min(3, max(0, (int)(p.y * ihy))),
              iz = min(3, max(0, (int)(p.z * ihz)));
    return (ix & 1) | ((iy & 1) << 1) | ((iz & 1) << 2) | ((ix & 2) << 2) | ((iy & 2) << 3) |
           ((iz & 2) << 4);
}

__global__ void k_cell_subsort(const int* __restrict__ start, const float4* __restrict__ pos,
                               const int* __restrict__ perm, float ihx, float ihy, float ihz,
                               int* __restrict__ perm_out) {
    __shared__ int cnt[64];
    const int c = blockIdx.x;
    const int st = start[c], n = start[c + 1] - st;
    if (n == 0) return;                          // block-uniform
    cnt[threadIdx.x] = 0;                        // 64 threads
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        atomicAdd(&cnt[subcell_key(pos[st + i], ihx, ihy, ihz)], 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0;
        for (int k = 0; k < 64; ++k) {
            const int v = cnt[k];
            cnt[k] = run;
            run += v;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        perm_out[st + atomicAdd(&cnt[subcell_key(pos[st + i], ihx, ihy, ihz)], 1)] = perm[st + i];
}

// Sorted triangle s: vertex ids with twice its area (as float bits), and the
// shift that takes a point of the triangle into the frame of its cell's corner
// (the centroid's offset from the corner less the centroid).
__global__ void k_tri_sorted(GridGeom geo, CellGrid cg, int m, const int* __restrict__ perm,
                             const double* __restrict__ cen, const int* __restrict__ tri,
                             const double* __restrict__ tri_area, int4* __restrict__ tv,
                             double* __restrict__ shift) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= m) return;
    const int k = perm[s];
    tv[s] = make_int4(tri[3 * k], tri[3 * k + 1], tri[3 * k + 2],
                      __float_as_int((float)(2.0 * tri_area[k])));
    const double* c = cen + 3 * (size_t)k;
    int cx, cy, cz;
    double o[3];
    locate(geo, cg, c[0], c[1], c[2], cx, cy, cz, o[0], o[1], o[2]);
    for (int i = 0; i < 3; ++i) shift[3 * (size_t)s + i] = o[i] - c[i];
}

// The 16 points of every triangle, for binning them one by one.
__global__ void k_points(int m, const double* __restrict__ x, const int* __restrict__ tri,
                         ListTab tab, double* __restrict__ xq) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= 16 * m) return;
    const int k = e >> 4, a = e & 15;
    const double* xa = x + 3 * (size_t)tri[3 * (size_t)k];
    const double* xb = x + 3 * (size_t)tri[3 * (size_t)k + 1];
    const double* xc = x + 3 * (size_t)tri[3 * (size_t)k + 2];
    for (int i = 0; i < 3; ++i)
        xq[3 * (size_t)e + i] = tab.phi[a][0] * xa[i] + tab.phi[a][1] * xb[i] + tab.phi[a][2] * xc[i];
}

// 64-point steps of list `pts` points per triangle in each cell
__global__ void k_step_counts(int ncell, int pts, const int* __restrict__ start,
                              int* __restrict__ cnt) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < ncell) cnt[c] = ((start[c + 1] - start[c]) * pts + 63) >> 6;
}

// map of the steps: first and last sorted triangle of the step's cell and the
// step's first point within the cell
__global__ void k_step_map(int ncell, const int* __restrict__ start,
                           const int* __restrict__ sstart, int4* __restrict__ map) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncell) return;
    const int a = start[c], b = start[c + 1];
    for (int s = sstart[c], k = 0; s < sstart[c + 1]; ++s, ++k) map[s] = make_int4(a, b, 64 * k, 0);
}

// Neighbour lists of the cells that hold targets: the non-empty cells at
// offsets -R..R whose box comes within r_cut of the cell's box, as entries (first
// step of each list, triangles; or, over points alone, first point and points)
// with their offset index apart.  Dilute suspensions leave most of the (2R + 1)^3
// neighbours empty (30 to 90 of 343 are kept), and a list serves all targets of
// its cell, so the sum's culling per target reads two or three rounds of 32
// entries instead of testing every offset.  A warp per cell; FILL writes the
// entries at start[c], otherwise their number goes to cnt[c].
struct NbrSource {
    const int* count_start;              // [ncell + 1] triangles (or points) of each cell
    const int* sstart[kElemLists];       // first step of each cell (points: all null)
    int base[kElemLists];
};

template <bool FILL>
__global__ void k_neighbours(CellGrid cg, float hx, float hy, float hz, float reach2,
                             const int* __restrict__ tgt_start, NbrSource src,
                             const int* __restrict__ start, int* __restrict__ cnt,
                             int4* __restrict__ out, unsigned short* __restrict__ off) {
    const int ncell = cg.ncx * cg.ncy * cg.ncz;
    const int c0 = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c0 >= ncell) return;                     // warp-uniform
    int n = 0;
    if (tgt_start[c0 + 1] > tgt_start[c0]) {     // warp-uniform
        const int cx = c0 % cg.ncx, cy = (c0 / cg.ncx) % cg.ncy, cz = c0 / (cg.ncx * cg.ncy);
        const unsigned lt = (1u << lane) - 1u;
        for (int r = 0; r < (kOffsets + 31) / 32; ++r) {
            const int oi = r * 32 + lane;
            bool keep = false;
            int4 e = make_int4(0, 0, 0, 0);
            if (oi < kOffsets) {
                const int ix = oi % kSide - R32, iy = (oi / kSide) % kSide - R32,
                          iz = oi / (kSide * kSide) - R32;
                const int cyy = cy + iy;
                const float gx = (float)max(abs(ix) - 1, 0) * hx,
                            gy = (float)max(abs(iy) - 1, 0) * hy,
                            gz = (float)max(abs(iz) - 1, 0) * hz;
                if (cyy >= 0 && cyy < cg.ncy && gx * gx + gy * gy + gz * gz <= reach2) {
                    // ncx, ncz >= 2 R (L > 2 r_cut): one wrap suffices for |i| <= R
                    int cxx = cx + ix, czz = cz + iz;
                    cxx += (cxx < 0) ? cg.ncx : 0;
                    cxx -= (cxx >= cg.ncx) ? cg.ncx : 0;
                    czz += (czz < 0) ? cg.ncz : 0;
                    czz -= (czz >= cg.ncz) ? cg.ncz : 0;
                    const int c = (czz * cg.ncy + cyy) * cg.ncx + cxx;
                    const int st = src.count_start[c], k = src.count_start[c + 1] - st;
                    keep = k > 0;
                    if (FILL && keep) {
                        if (src.sstart[0])
                            e = make_int4(src.sstart[0][c], src.base[1] + src.sstart[1][c],
                                          src.base[2] + src.sstart[2][c], k);
                        else
                            e = make_int4(st, 0, 0, k);
                    }
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (FILL && keep) {
                const int slot = start[c0] + n + __popc(m & lt);
                out[slot] = e;
                off[slot] = (unsigned short)oi;
            }
            n += __popc(m);
        }
    }
    if (!FILL && lane == 0) cnt[c0] = n;
}

// positions of one list, a warp per step, a lane per slot pair: offsets from
// the cell corner in units of 1/(alpha sqrt(log2 e)); slots past the cell's
// last point get the dummy offset 1e4 (terms exactly zero) and zero strength
template <int PTS>
__global__ void k_list_positions(int nsteps, const int4* __restrict__ map,
                                 const int4* __restrict__ tv, const double* __restrict__ shift,
                                 const double* __restrict__ x, ListTab tab, double sc,
                                 float4* __restrict__ pack, int4* __restrict__ vert) {
    __shared__ double phi[PTS][3];
    for (int e = threadIdx.x; e < PTS * 3; e += blockDim.x) phi[e / 3][e % 3] = tab.phi[e / 3][e % 3];
    __syncthreads();
    const int step = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (step >= nsteps) return;                  // warp-uniform
    const int4 mp = map[step];
    float p[2][3];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int e = mp.z + 2 * lane + k;
        const int s = mp.x + e / PTS, a = e % PTS;
        const bool in = s < mp.y;
        if (in) {
            const int4 v = tv[s];
            const double* xa = x + 3 * (size_t)v.x;
            const double* xb = x + 3 * (size_t)v.y;
            const double* xc = x + 3 * (size_t)v.z;
            const double* sh = shift + 3 * (size_t)s;
            for (int i = 0; i < 3; ++i)
                p[k][i] = (float)((phi[a][0] * xa[i] + phi[a][1] * xb[i] + phi[a][2] * xc[i] +
                                   sh[i]) * sc);
        } else {
            p[k][0] = p[k][1] = p[k][2] = 1e4f;
        }
        // vertices of every 16-slot group (list 0: one triangle each)
        if (PTS == 16 && k == 0 && (lane & 7) == 0)
            vert[(size_t)step * 4 + (lane >> 3)] = in ? tv[s] : make_int4(-1, -1, -1, 0);
    }
    float4* o = pack + (size_t)step * 96 + lane;
    o[0] = make_float4(p[0][0], p[1][0], p[0][1], p[1][1]);
    o[32] = make_float4(p[0][2], p[1][2], 0.f, 0.f);
    o[64] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// The same for points binned one by one: a slot's point from the cell order perm
// (point = 16 triangle + rule index), with its triangle's vertices and twice the
// area (float bits) and its rule index.
__global__ void k_point_positions(GridGeom geo, CellGrid cg, int nsteps,
                                  const int4* __restrict__ map, const int* __restrict__ perm,
                                  const double* __restrict__ xq, const int* __restrict__ tri,
                                  const double* __restrict__ tri_area, double sc,
                                  float4* __restrict__ pack, int4* __restrict__ vert,
                                  unsigned char* __restrict__ rule) {
    const int step = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (step >= nsteps) return;                  // warp-uniform
    const int4 mp = map[step];
    float p[2][3];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int s = mp.x + mp.z + 2 * lane + k;
        const size_t slot = (size_t)step * 64 + 2 * lane + k;
        p[k][0] = p[k][1] = p[k][2] = 1e4f;
        int4 v = make_int4(-1, -1, -1, 0);
        int a = 0;
        if (s < mp.y) {
            const int id = perm[s], t = id >> 4;
            const double* c = xq + 3 * (size_t)id;
            int cx, cy, cz;
            double o[3];
            locate(geo, cg, c[0], c[1], c[2], cx, cy, cz, o[0], o[1], o[2]);
            for (int i = 0; i < 3; ++i) p[k][i] = (float)(o[i] * sc);
            v = make_int4(tri[3 * (size_t)t], tri[3 * (size_t)t + 1], tri[3 * (size_t)t + 2],
                          __float_as_int((float)(2.0 * tri_area[t])));
            a = id & 15;
        }
        vert[slot] = v;
        rule[slot] = (unsigned char)a;
    }
    float4* o = pack + (size_t)step * 96 + lane;
    o[0] = make_float4(p[0][0], p[1][0], p[0][1], p[1][1]);
    o[32] = make_float4(p[0][2], p[1][2], 0.f, 0.f);
    o[64] = make_float4(0.f, 0.f, 0.f, 0.f);
}

__global__ void k_density_f32(long n, const double* __restrict__ q, float* __restrict__ out) {
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) out[e] = (float)q[e];
}

struct StrengthTab {
    float c[kElemLists][16][3];      // phi_v w
};

// strengths of the lists: a warp per step (list 0's steps first), a lane per
// slot pair, g = scale 2A sum_v (phi_v w) q_v.  The vertices come from the
// sorted triangles (16 bytes per triangle, shared by its points), so the pass
// moves little more than the strengths it writes: 1.05 ms per evaluation with
// per-point vertex ids and weights for 82 M points (4000 cells), 0.69 ms here
// for those and 36 M of list 1
template <int PTS>
__device__ __forceinline__ void step_strengths(int lane, int4 mp, const int4* __restrict__ tv,
                                               const float* __restrict__ q, float scale,
                                               const float (*c)[3], float4* __restrict__ o) {
    float g[2][3];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int e = mp.z + 2 * lane + k;
        const int s = mp.x + e / PTS, a = e % PTS;
        g[k][0] = g[k][1] = g[k][2] = 0.f;
        if (s < mp.y) {
            const int4 v = tv[s];
            const float f = scale * __int_as_float(v.w);
            const float ca = f * c[a][0], cb = f * c[a][1], cc = f * c[a][2];
#pragma unroll
            for (int i = 0; i < 3; ++i)
                g[k][i] = ca * q[3 * (size_t)v.x + i] + cb * q[3 * (size_t)v.y + i] +
                          cc * q[3 * (size_t)v.z + i];
        }
    }
    *reinterpret_cast<float2*>(&o[32].z) = make_float2(g[0][0], g[1][0]);
    o[64] = make_float4(g[0][1], g[1][1], g[0][2], g[1][2]);
}

__global__ void k_list_strengths(int n0, int n1, int n2, const int4* __restrict__ map0,
                                 const int4* __restrict__ map1, const int4* __restrict__ map2,
                                 const int4* __restrict__ tv,
                                 const float* __restrict__ q, float scale, StrengthTab tab,
                                 float4* __restrict__ pack) {
    __shared__ float c[kElemLists][16][3];
    for (int e = threadIdx.x; e < kElemLists * 48; e += blockDim.x)
        (&c[0][0][0])[e] = (&tab.c[0][0][0])[e];
    __syncthreads();
    const int step = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (step >= n0 + n1 + n2) return;            // warp-uniform
    float4* o = pack + (size_t)step * 96 + lane;
    if (step < n0) step_strengths<kPts[0]>(lane, map0[step], tv, q, scale, c[0], o);
    else if (step < n0 + n1) step_strengths<kPts[1]>(lane, map1[step - n0], tv, q, scale, c[1], o);
    else step_strengths<kPts[2]>(lane, map2[step - n0 - n1], tv, q, scale, c[2], o);
}

// strengths of points binned one by one
__global__ void k_point_strengths(int nsteps, const int4* __restrict__ vert,
                                  const unsigned char* __restrict__ rule,
                                  const float* __restrict__ q, float scale, StrengthTab tab,
                                  float4* __restrict__ pack) {
    __shared__ float c[16][3];
    for (int e = threadIdx.x; e < 48; e += blockDim.x) (&c[0][0])[e] = (&tab.c[0][0][0])[e];
    __syncthreads();
    const int step = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (step >= nsteps) return;                  // warp-uniform
    float g[2][3];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const size_t slot = (size_t)step * 64 + 2 * lane + k;
        const int4 v = vert[slot];
        const int a = rule[slot];
        g[k][0] = g[k][1] = g[k][2] = 0.f;
        if (v.x >= 0) {
            const float f = scale * __int_as_float(v.w);
            const float ca = f * c[a][0], cb = f * c[a][1], cc = f * c[a][2];
#pragma unroll
            for (int i = 0; i < 3; ++i)
                g[k][i] = ca * q[3 * (size_t)v.x + i] + cb * q[3 * (size_t)v.y + i] +
                          cc * q[3 * (size_t)v.z + i];
        }
    }
    float4* o = pack + (size_t)step * 96 + lane;
    *reinterpret_cast<float2*>(&o[32].z) = make_float2(g[0][0], g[1][0]);
    o[64] = make_float4(g[0][1], g[1][1], g[0][2], g[1][2]);
}

// --------------------------------------------------------------- the sum
// Two candidate pairs at once (add/mul/fma .f32x2: one issued instruction
// serves two pairs); rsqrt, exp2 and the reciprocal stay scalar.  Every
// multiply-add is an explicit FMA.
struct PairAcc2 {
    f2 ux = {0ull}, uy = {0ull}, uz = {0ull};
    f2 sn = {0ull};     // double layer: sum of E x.g (times the target normal at the end)
};

__device__ __forceinline__ float rcp_ftz(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// the hardware approximations (about 2 ulp); r is at most r_cut, a cell's diagonal
// (up to 0.9 r_cut where one cell spans the slit) and two thirds of an edge, but for
// the dummies: far from denormal inputs and results
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_ftz(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Constants of the sum.  Coordinates are scaled by s = alpha sqrt(log2 e), so
// exp(-alpha^2 r^2) = 2^(-r_s^2) takes no multiply; the displacements, r and
// 1/r are in scaled units and the constants absorb the scale.  The double
// layer's common factor c4 = 4 alpha^3 / sqrt(pi) is taken out of its
// coefficients into the output factor.
struct Elem32Const {
    float sc, pt, c1, c2, c3, c6, fU, rc2, near2, hx, hy, hz;
};

template <int LAYER>
__device__ __forceinline__ void pair_terms2(const Elem32Const& k, f2 dx, f2 dy, f2 dz, f2 r2,
                                            f2 gx, f2 gy, f2 gz, f2 nx, f2 ny, f2 nz,
                                            PairAcc2& a) {
    float lo, hi;
    f2_split(r2, lo, hi);
    const f2 ir = f2_make(rsqrt_ftz(lo), rsqrt_ftz(hi));
    const f2 ex = f2_make(ex2_ftz(-lo), ex2_ftz(-hi));               // exp(-alpha^2 r^2)
    const f2 r = r2 * ir;
    f2_split(fma2(r, f2_splat(k.pt), f2_splat(1.0f)), lo, hi);
    const f2 t = f2_make(rcp_ftz(lo), rcp_ftz(hi));                 // 1/(1 + P alpha r)
    const f2 xg = fma2(dz, gz, fma2(dy, gy, dx * gx));
    if (LAYER == 0) {
        // A = ec/r - c1 ex,  B = (ec/r^3 + c1 ex/r^2) xg, ec = ex erfcx(alpha r)
        const f2 eir = ex * erfcx_t2(t) * ir;
        const f2 A = fma2(f2_splat(-k.c1), ex, eir);
        const f2 B = (ir * ir) * fma2(f2_splat(k.c1), ex, eir) * xg;
        a.ux = fma2(B, dx, fma2(A, gx, a.ux));
        a.uy = fma2(B, dy, fma2(A, gy, a.uy));
        a.uz = fma2(B, dz, fma2(A, gz, a.uz));
    } else {
        // D = -6 ec/r^5 - c2 ex/r^4 - c3 ex/r^2 and E = c4 ex, both over c4 ex:
        // D' = ir2 (ir2 (c6 erfcx ir - c2) - c3); the update
        // D xg xn d + E (d gn + g xn + n xg) regrouped as
        // ex [d (D' xg xn + gn) + g xn + n xg], the last term's scalar ex xg
        // summed over the pairs and multiplied by the (fixed) target normal
        // once: 40 paired operations per two pairs (44 with E formed apart:
        // 3.41 -> 3.27 ms per launch on 100 capsules)
        const f2 ir2 = ir * ir;
        const f2 D = ir2 * fma2(ir2, fma2(f2_splat(k.c6), erfcx_t2(t) * ir, f2_splat(-k.c2)),
                                f2_splat(-k.c3));
        const f2 xn = fma2(dz, nz, fma2(dy, ny, dx * nx));
        const f2 gn = fma2(gz, nz, fma2(gy, ny, gx * nx));
        const f2 cd = ex * fma2(D * xg, xn, gn), cg = ex * xn;
        a.sn = fma2(ex, xg, a.sn);
        a.ux = fma2(dx, cd, fma2(gx, cg, a.ux));
        a.uy = fma2(dy, cd, fma2(gy, cg, a.uy));
        a.uz = fma2(dz, cd, fma2(gz, cg, a.uz));
    }
}

// Targets, lists and outputs of one launch.
struct Elem32Args {
    Elem32Const k;
    int n_tgt;
    const float4* tpos;              // sorted targets: offsets from the cell corner,
    const int* tcell;                //   cell,
    const int* tperm;                //   caller index
    const int* nstart;               // [ncell + 1] neighbour list of each target cell
    const int4* nbr;
    const unsigned short* noff;
    float lim1, lim2;                // squared distances from which a cell uses lists 1, 2
    const int4* vert;                // list 0: vertices of each 16-slot group (POINTS: slot)
    const double* nrm;               // [n][3] target normals (caller order)
    float* out;
    int out_stride;
};

constexpr int LWE = 4;        // warps (targets) per block, 12 blocks per SM (40 registers; 10 of
                              //   48: 138.5 against 136.0 ms for two launches on 4000 cells)
constexpr int kCap = 128;     // culled cells per batch (a target may need several batches)

// Cull the neighbour list [i, end) of the target's cell in rounds of 32 entries,
// stopping before a round could overflow kCap; i is left at the first entry not
// culled.  Kept are the cells whose nearest point lies within r_cut of the
// target (slightly widened, so that rounding can only keep more).  Entries:
// first step, step count and offset index; bit 15 marks the cells that can
// hold triangles around the target.
template <bool POINTS>
__device__ __forceinline__ int cull_cells_batch(const Elem32Args& a, int lane, float ox, float oy,
                                                float oz, int& i, int end, int* s_st, int* s_cnt,
                                                unsigned short* s_off) {
    const unsigned lt = (1u << lane) - 1u;
    const float reach2 = a.k.rc2 * 1.0001f, near2 = a.k.near2 * 1.0001f;
    int nc = 0;
    for (; i < end && nc + 32 <= kCap; i += 32) {
        bool keep = false, nearc = false;
        int st = 0, cnt = 0, oi = 0;
        if (i + lane < end) {
            const int4 e = a.nbr[i + lane];
            oi = a.noff[i + lane];
            const int ix = oi % kSide - R32, iy = (oi / kSide) % kSide - R32,
                      iz = oi / (kSide * kSide) - R32;
            const float gx = ix > 0 ? (float)ix * a.k.hx - ox
                                    : (ix < 0 ? ox - (float)(ix + 1) * a.k.hx : 0.f);
            const float gy = iy > 0 ? (float)iy * a.k.hy - oy
                                    : (iy < 0 ? oy - (float)(iy + 1) * a.k.hy : 0.f);
            const float gz = iz > 0 ? (float)iz * a.k.hz - oz
                                    : (iz < 0 ? oz - (float)(iz + 1) * a.k.hz : 0.f);
            const float d2 = gx * gx + gy * gy + gz * gz;
            nearc = d2 <= near2;
            keep = d2 <= reach2;
            // steps: the cell's points of the list, 64 at a time
            const int l = d2 >= a.lim2 ? 2 : (d2 >= a.lim1 ? 1 : 0);
            st = l == 2 ? e.z : (l == 1 ? e.y : e.x);
            constexpr int p0 = kPts[0], p1 = kPts[1], p2 = kPts[2];
            cnt = (e.w * (POINTS ? 1 : (l == 2 ? p2 : (l == 1 ? p1 : p0))) + 63) >> 6;
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (keep) {
            const int slot = nc + __popc(m & lt);
            s_st[slot] = st;
            s_cnt[slot] = cnt;
            s_off[slot] = (unsigned short)(oi | (nearc ? 0x8000 : 0));
        }
        nc += __popc(m);
    }
    __syncwarp();
    return nc;
}

// S = 1: one warp per target (neighbouring targets in cell order); S = LWE: a
// block per target, its warps taking the cells in turn.  The warp lists the
// cells within r_cut and walks them in 64-point steps, every lane taking
// two adjacent candidates and evaluating both with paired FP32 arithmetic: no
// hit queue, as about 80 % of the candidates lie within r_cut.  A step is
// 1,536 bytes in three rows of 32 lanes x 16 bytes (x0 x1 y0 y1 | z0 z1 gx0 gx1
// | gy0 gy1 gz0 gz1): a lane's two candidates arrive with three 16-byte loads,
// every coordinate already paired, each load of a warp covering 512 contiguous
// bytes.  Each cell fills whole steps with dummies, so a step needs no bounds
// test.
// Candidates beyond r_cut are evaluated unmasked, and a step with no candidate within
// r_cut is skipped; in the same way a triangle counts with the cell of its
// centroid.  POINTS: the points were binned one by one, and each counts within r_cut only
// (kBinRadius says when).
// Points of the triangles around the target (left to the singular correction)
// can only lie in the cells the culling marks near; only there is each
// candidate within near2 checked and, if excluded, given zero strength.
//
// What bounds it: the FMA pipe (31 / 40 paired operations of two cycles per
// two pairs) and the instructions around it; loads hit L1 / L2 (blocks of 2 to
// 20 warps share more or fewer candidates and run within 5 %).  So the lever
// is the number of candidates and the work per cell.  One launch, single and
// double layer averaged, 4000 biconcave cells: 107.5 ms with every point of list
// 0 and all 343 neighbour offsets tested per target; 76 ms with list 1 from 5
// edges; 72.7 ms with the neighbour lists; 68.0 ms with list 1 from 4 edges;
// 66.4 ms with list 2.  382 spheres at volume fraction 0.1, double layer: 23.6 ->
// 12.4 ms without list 2, 11.3 ms with it.  Cells of
// r_cut / 4 or / 5 have fewer candidates and more cells: 145.7 and 148.1 against
// 145.5 ms per two launches (list 1 from 5 edges).
template <int LAYER, int S, bool POINTS>
__global__ void __launch_bounds__(LWE * 32, POINTS ? 10 : 12) k_local_elem32(Elem32Args a,
                                                          const float4* __restrict__ pk) {
    __shared__ int s_st[LWE][kCap];
    __shared__ int s_cnt[LWE][kCap];
    __shared__ unsigned short s_off[LWE][kCap];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    static_assert(S == 1 || S == LWE, "a target has one warp or a block");
    const int t = S > 1 ? blockIdx.x : blockIdx.x * LWE + wid;
    if (t >= a.n_tgt) return;                     // warp-uniform (S > 1: block-uniform)
    const float4 p = a.tpos[t];
    const int c = a.tcell[t], oidx = a.tperm[t];
    const int nend = a.nstart[c + 1];
    const float ox = p.x * a.k.sc, oy = p.y * a.k.sc, oz = p.z * a.k.sc;
    float nx = 0.f, ny = 0.f, nz = 0.f;
    if (LAYER == 1) {
        nx = (float)a.nrm[3 * (size_t)oidx];
        ny = (float)a.nrm[3 * (size_t)oidx + 1];
        nz = (float)a.nrm[3 * (size_t)oidx + 2];
    }
    const f2 nx2 = f2_splat(nx), ny2 = f2_splat(ny), nz2 = f2_splat(nz);
    const float rc2 = a.k.rc2;
    PairAcc2 acc;
    for (int i = a.nstart[c]; i < nend;) {
        const int nc = cull_cells_batch<POINTS>(a, lane, ox, oy, oz, i, nend, s_st[wid],
                                                s_cnt[wid], s_off[wid]);
        for (int ci = S > 1 ? wid : 0; ci < nc; ci += S) {
            const int st = s_st[wid][ci], end = st + s_cnt[wid][ci];
            const int oi = s_off[wid][ci] & 0x7fff;
            const bool nearc = s_off[wid][ci] >> 15;
            // target position in the frame of this source cell's corner
            const f2 tx = f2_splat(ox - (float)(oi % kSide - R32) * a.k.hx);
            const f2 ty = f2_splat(oy - (float)((oi / kSide) % kSide - R32) * a.k.hy);
            const f2 tz = f2_splat(oz - (float)(oi / (kSide * kSide) - R32) * a.k.hz);
            // one 64-point step; NEAR: check for points of the target's own triangles
            auto step = [&](int s, auto near_tag) {
                constexpr bool NEAR = decltype(near_tag)::value;
                // positions and strengths in one go (the strengths before the
                // test, so their latency overlaps the distance arithmetic)
                const float4* ps = pk + (size_t)s * 96 + lane;
                const float4 pa = ps[0], pb = ps[32], pc = ps[64];
                const f2 dx = tx - f2_make(pa.x, pa.y), dy = ty - f2_make(pa.z, pa.w),
                         dz = tz - f2_make(pb.x, pb.y);
                const f2 r2 = fma2(dz, dz, fma2(dy, dy, dx * dx));
                float r0, r1;
                float2 wx = make_float2(pb.z, pb.w), wy = make_float2(pc.x, pc.y),
                       wz = make_float2(pc.z, pc.w);
                f2_split(r2, r0, r1);
                if (!__any_sync(0xffffffffu, r0 < rc2 || r1 < rc2)) return;
                if (POINTS) {
                    if (NEAR) {
                        const int4* v = a.vert + (size_t)s * 64 + 2 * lane;
                        const int4 v0 = v[0], v1 = v[1];
                        if (v0.x == oidx || v0.y == oidx || v0.z == oidx) r0 = rc2;
                        if (v1.x == oidx || v1.y == oidx || v1.z == oidx) r1 = rc2;
                    }
                    if (!(r0 < rc2)) wx.x = wy.x = wz.x = 0.f;
                    if (!(r1 < rc2)) wx.y = wy.y = wz.y = 0.f;
                } else if (NEAR) {
                    if (r0 < a.k.near2 || r1 < a.k.near2) {
                        // both candidates are points of one triangle (list 0)
                        const int4 v = a.vert[(size_t)s * 4 + (lane >> 3)];
                        if (v.x == oidx || v.y == oidx || v.z == oidx)
                            wx = wy = wz = make_float2(0.f, 0.f);
                    }
                }
                pair_terms2<LAYER>(a.k, dx, dy, dz, r2, f2_make(wx.x, wx.y), f2_make(wy.x, wy.y),
                                   f2_make(wz.x, wz.y), nx2, ny2, nz2, acc);
            };
            if (nearc) {
                for (int s = st; s < end; ++s) step(s, std::true_type{});
            } else {
                for (int s = st; s < end; ++s) step(s, std::false_type{});
            }
        }
        __syncwarp();
    }
    float ux = f2_sum(acc.ux), uy = f2_sum(acc.uy), uz = f2_sum(acc.uz);
    if (LAYER == 1) {
        const float sn = f2_sum(acc.sn);
        ux = fmaf(nx, sn, ux);
        uy = fmaf(ny, sn, uy);
        uz = fmaf(nz, sn, uz);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ux += __shfl_xor_sync(0xffffffffu, ux, o);
        uy += __shfl_xor_sync(0xffffffffu, uy, o);
        uz += __shfl_xor_sync(0xffffffffu, uz, o);
    }
    if (S > 1) {
        // the parts of the target's warps, added in order
        __shared__ float s_part[LWE][3];
        if (lane == 0) {
            s_part[wid][0] = ux;
            s_part[wid][1] = uy;
            s_part[wid][2] = uz;
        }
        __syncthreads();
        if (wid != 0) return;
        for (int w = 1; w < S; ++w) {
            ux += s_part[w][0];
            uy += s_part[w][1];
            uz += s_part[w][2];
        }
    }
    if (lane == 0) {
        float* o = a.out + (size_t)oidx * a.out_stride;
        o[0] = a.k.fU * ux;
        o[1] = a.k.fU * uy;
        o[2] = a.k.fU * uz;
    }
}

float coord_scale(double alpha) { return (float)(alpha * 1.2011224087864498); }

}  // namespace

bool elem32_by_point(double near_edge, double alpha, double rcut) {
    return alpha * (rcut - near_edge * (2.0 / 3.0)) < kBinRadius || alpha * rcut < kBinCut;
}

// A point of a triangle around the target can be farther from it than the
// triangle's longest edge only by rounding; `near` carries that margin.  A far
// cell never is a near one (kFarEdges > 1).
void elem32_far_distances(double near_edge, double alpha, double rcut, double* far) {
    far[0] = 0.0;
    far[1] = kFarEdges * near_edge;
    far[2] = alpha * near_edge <= kDimEdge ? std::max(far[1], kDimRadius / alpha) : rcut;
    for (int l = 1; l < kElemLists; ++l)
        if (!(far[l] < 0.85 * rcut)) far[l] = INFINITY;
}

cudaError_t elem32_steps(const ElemLists32& L, int ncell, int* scratch, cudaStream_t st) {
    for (int l = 0; l < kElemLists; ++l) {
        const int pts = L.points ? (l == 0 ? 1 : 0) : kPts[l];
        k_step_counts<<<(ncell + 255) / 256, 256, 0, st>>>(ncell, pts, L.tri_start, scratch);
        cudaError_t e = scan_counts(ncell, scratch, L.sstart[l], st);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

cudaError_t elem32_neighbours(const GridGeom& geo, const CellGrid& cg, const ElemLists32& L,
                              const int* tgt_start, const int* src_start, int* scratch,
                              bool fill, cudaStream_t st) {
    const int ncell = cg.ncx * cg.ncy * cg.ncz;
    const float reach2 = (float)(geo.rcut * geo.rcut * 1.0002);
    NbrSource src{};
    src.count_start = src_start ? src_start : L.tri_start;
    for (int l = 0, base = 0; l < kElemLists && !src_start; ++l) {
        src.sstart[l] = L.sstart[l];
        src.base[l] = base;
        base += L.nsteps[l];
    }
    const float hx = (float)cg.hx, hy = (float)cg.hy, hz = (float)cg.hz;
    const unsigned nb = (unsigned)((ncell + 7) / 8);
    if (fill) {
        k_neighbours<true><<<nb, 256, 0, st>>>(cg, hx, hy, hz, reach2, tgt_start, src, L.nstart,
                                              nullptr, L.nbr, L.noff);
        return cudaGetLastError();
    }
    k_neighbours<false><<<nb, 256, 0, st>>>(cg, hx, hy, hz, reach2, tgt_start, src, nullptr,
                                           scratch, nullptr, nullptr);
    return scan_counts(ncell, scratch, L.nstart, st);
}

cudaError_t elem32_centroids(int m, const double* x, const int* tri, double* cen,
                             cudaStream_t st) {
    if (m > 0) k_centroids<<<(m + 255) / 256, 256, 0, st>>>(m, x, tri, cen);
    return cudaGetLastError();
}

cudaError_t elem32_points(int m, const double* x, const int* tri, const QuadRule& rule, double* xq,
                          cudaStream_t st) {
    const RuleTab r = rule_tab(0, rule);
    ListTab tab;
    for (int a = 0; a < 16; ++a)
        for (int v = 0; v < 3; ++v) tab.phi[a][v] = r.phi[a][v];
    if (m > 0) k_points<<<(m * 16 + 255) / 256, 256, 0, st>>>(m, x, tri, tab, xq);
    return cudaGetLastError();
}

cudaError_t elem32_point_order(const CellGrid& cg, const ElemLists32& L, const float4* pos,
                               const int* perm, int* perm_out, cudaStream_t st) {
    k_cell_subsort<<<cg.ncx * cg.ncy * cg.ncz, 64, 0, st>>>(
        L.tri_start, pos, perm, (float)(4.0 / cg.hx), (float)(4.0 / cg.hy), (float)(4.0 / cg.hz),
        perm_out);
    return cudaGetLastError();
}

cudaError_t elem32_point_fill(const GridGeom& geo, const CellGrid& cg, const ElemLists32& L,
                              const int* perm, const double* xq, const int* tri,
                              const double* tri_area, cudaStream_t st) {
    const int ncell = cg.ncx * cg.ncy * cg.ncz, ns = L.nsteps[0];
    if (ns == 0) return cudaSuccess;
    k_step_map<<<(ncell + 255) / 256, 256, 0, st>>>(ncell, L.tri_start, L.sstart[0], L.map[0]);
    k_point_positions<<<(ns + 7) / 8, 256, 0, st>>>(geo, cg, ns, L.map[0], perm, xq, tri, tri_area,
                                                    (double)coord_scale(geo.alpha), L.pack, L.vert,
                                                    L.prule);
    return cudaGetLastError();
}

cudaError_t elem32_order(const GridGeom& geo, const CellGrid& cg, int m, const ElemLists32& L,
                         const float4* pos, const int* perm, int* perm_out, const double* cen,
                         const int* tri, const double* tri_area, cudaStream_t st) {
    const int ncell = cg.ncx * cg.ncy * cg.ncz;
    if (m <= 0) return cudaSuccess;
    k_cell_subsort<<<ncell, 64, 0, st>>>(L.tri_start, pos, perm, (float)(4.0 / cg.hx),
                                         (float)(4.0 / cg.hy), (float)(4.0 / cg.hz), perm_out);
    k_tri_sorted<<<(m + 255) / 256, 256, 0, st>>>(geo, cg, m, perm_out, cen, tri, tri_area, L.tv,
                                                  L.shift);
    return cudaGetLastError();
}

cudaError_t elem32_fill(const GridGeom& geo, const CellGrid& cg, const ElemLists32& L,
                        const QuadRule& rule, const double* x, cudaStream_t st) {
    const int ncell = cg.ncx * cg.ncy * cg.ncz;
    const double sc = (double)coord_scale(geo.alpha);
    int base = 0;
    for (int l = 0; l < kElemLists; ++l) {
        const int ns = L.nsteps[l];
        if (ns == 0) continue;
        const RuleTab r = rule_tab(l, rule);
        ListTab tab;
        for (int a = 0; a < 16; ++a)
            for (int v = 0; v < 3; ++v) tab.phi[a][v] = r.phi[a][v];
        k_step_map<<<(ncell + 255) / 256, 256, 0, st>>>(ncell, L.tri_start, L.sstart[l], L.map[l]);
        float4* pk = L.pack + (size_t)base * 96;
        if (l == 0)
            k_list_positions<kPts[0]><<<(ns + 7) / 8, 256, 0, st>>>(ns, L.map[0], L.tv, L.shift, x,
                                                                  tab, sc, pk, L.vert);
        else if (l == 1)
            k_list_positions<kPts[1]><<<(ns + 7) / 8, 256, 0, st>>>(ns, L.map[1], L.tv, L.shift, x,
                                                                  tab, sc, pk, nullptr);
        else
            k_list_positions<kPts[2]><<<(ns + 7) / 8, 256, 0, st>>>(ns, L.map[2], L.tv, L.shift, x,
                                                                  tab, sc, pk, nullptr);
        base += ns;
    }
    return cudaGetLastError();
}

cudaError_t elem32_strengths(const ElemLists32& L, const QuadRule& rule, int nnodes,
                             const double* q, float* q32, double scale, cudaStream_t st) {
    const long ne = 3L * nnodes;
    if (ne > 0) k_density_f32<<<(unsigned)((ne + 255) / 256), 256, 0, st>>>(ne, q, q32);
    StrengthTab tab{};
    for (int l = 0; l < kElemLists; ++l) {
        const RuleTab r = rule_tab(l, rule);
        for (int a = 0; a < kPts[l]; ++a)
            for (int v = 0; v < 3; ++v) tab.c[l][a][v] = (float)(r.phi[a][v] * r.w[a]);
    }
    const int ns = L.nsteps[0] + L.nsteps[1] + L.nsteps[2];
    if (ns > 0 && L.points)
        k_point_strengths<<<(ns + 7) / 8, 256, 0, st>>>(ns, L.vert, L.prule, q32, (float)scale, tab,
                                                        L.pack);
    else if (ns > 0)
        k_list_strengths<<<(ns + 7) / 8, 256, 0, st>>>(L.nsteps[0], L.nsteps[1], L.nsteps[2],
                                                       L.map[0], L.map[1], L.map[2], L.tv, q32,
                                                       (float)scale, tab, L.pack);
    return cudaGetLastError();
}

cudaError_t elem32_sum(const GridGeom& geo, const CellGrid& cg, const ElemLists32& L,
                       double near, const SortedSources<float>& tgt, const double* nrm, int layer,
                       float* out, int out_stride, int nsm, cudaStream_t st) {
    if (tgt.n <= 0) return cudaSuccess;
    const double sp = 1.7724538509055160273, pi = 3.14159265358979323846, al = geo.alpha;
    const double sc = (double)coord_scale(al), c4 = 4.0 * al * al * al / sp;
    Elem32Args a;
    a.n_tgt = tgt.n;
    a.tpos = tgt.pos;
    a.tcell = tgt.cell;
    a.tperm = tgt.perm;
    a.nstart = L.nstart;
    a.nbr = L.nbr;
    a.noff = L.noff;
    float lim[kElemLists];
    for (int l = 1; l < kElemLists; ++l)
        lim[l] = L.nsteps[l] > 0 ? (float)(L.far[l] * L.far[l] * sc * sc) : 3e38f;
    a.lim1 = lim[1];
    a.lim2 = lim[2];
    a.vert = L.vert;
    a.nrm = nrm;
    a.out = out;
    a.out_stride = out_stride;
    Elem32Const& k = a.k;
    k.sc = (float)sc;
    k.hx = (float)(cg.hx * sc);
    k.hy = (float)(cg.hy * sc);
    k.hz = (float)(cg.hz * sc);
    k.rc2 = (float)(geo.rcut * geo.rcut * sc * sc);
    k.near2 = (float)(near * near * sc * sc);
    k.pt = (float)(GGEM_ERFCX_P * al / sc);
    k.c1 = (float)(2.0 * al / sp / sc);
    k.c2 = (float)(12.0 * al / sp * sc * sc / c4);
    k.c3 = (float)(8.0 * al * al * al / sp / c4);
    k.c6 = (float)(-6.0 * sc * sc * sc / c4);
    k.fU = (float)((layer == 0 ? sc : c4 / sc) / (8.0 * pi * geo.mu));
    // about 5 KB of shared memory per block, 12 blocks per SM: ask for a small
    // shared-memory carveout (25 %: the 64 KB configuration) so that the rest
    // of the SM's 256 KB serves as L1 for the candidates the warps of a block
    // re-read (a preference; cheap per launch)
    // A block per target where there are few: four warps share its latencies and the
    // SMs' shares even out.  One against four warps, double / single layer (us): 1,296
    // targets 88 -> 43 / 90 -> 45, 5,184 133 -> 111 / 113 -> 107, 16,200 289 -> 262 / 246
    // -> 246, 24,300 466 -> 436 / 397 -> 410, 64,200 on finer spheres 2.63 -> 2.66 / 2.18
    // -> 2.57 ms: every warp culls the whole neighbour list, which a full chip feels.
    const bool split = tgt.n <= 96 * nsm;
    void (*const kfs[2][2][2])(Elem32Args, const float4*) = {
        {{k_local_elem32<0, 1, false>, k_local_elem32<0, 1, true>},
         {k_local_elem32<0, LWE, false>, k_local_elem32<0, LWE, true>}},
        {{k_local_elem32<1, 1, false>, k_local_elem32<1, 1, true>},
         {k_local_elem32<1, LWE, false>, k_local_elem32<1, LWE, true>}}};
    const auto kf = kfs[layer == 0 ? 0 : 1][split][L.points];
    cudaFuncSetAttribute((const void*)kf, cudaFuncAttributePreferredSharedMemoryCarveout, 25);
    kf<<<split ? tgt.n : (tgt.n + LWE - 1) / LWE, LWE * 32, 0, st>>>(a, L.pack);
    return cudaGetLastError();
}

}  // namespace ggem
