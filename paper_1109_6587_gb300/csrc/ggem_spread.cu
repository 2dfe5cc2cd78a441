// Spreading of the global density onto the grid (paper Eqs. (stokes_gg),
// (rho_int), (rhog_sum)):
//   f(node) = - sum_s g_s rho_g(node - x_s*),   |node - x_s*| < r_cut,
//   rho_g(r) = alpha^3 pi^{-3/2} exp(-alpha^2 r^2) (5/2 - alpha^2 r^2).
//
// Source-parallel: a warp takes two neighbouring sorted sources (the union of
// their stencils, both weights per node, one reduction with their sum), lists
// the columns, rows and planes of its stencil, and adds the weights into an
// interleaved [Ny][Nz][Nx][4] accumulation grid with float4 / double reductions
// in L2; k_deinterleave then writes the planar [Ny][3][Nz][Nx] forcing.  The
// Gaussian factor is separable, exp(-a^2 r^2) = exp(-a^2 dx^2)
// exp(-a^2 dy^2) exp(-a^2 dz^2), so each source costs one exponential per
// column, row and plane (the fast Gaussian gridding idea), the remaining
// work per node being a few multiplies.  Displacements come from per-source
// descriptors (integer grid offsets plus small remainders, built once per
// source set), so the kernel runs in T only: no FP64 instruction, accurate in
// large boxes.
#include "ggem_internal.cuh"

namespace ggem {

namespace {

// Per-source descriptor for spreading, computed once per source set (one
// thread per sorted source, FP64): ixb = floor(x/dx) of the wrapped x,
// rx = x - ixb dx; the same for z; jn = nearest Chebyshev node, ry = y - y_jn;
// [jlo, jhi] = a superset of the nodes with |y_j - y| < r_cut.
template <typename T>
__global__ void k_src_desc(GridGeom geo, const double* __restrict__ yj, int n,
                           const int* __restrict__ perm, const double* __restrict__ x,
                           int4* __restrict__ di, v4_t<T>* __restrict__ df) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    int src = perm[s];
    double xs = x[3 * src], ys = x[3 * src + 1], zs = x[3 * src + 2];
    xs -= geo.Lx * floor(xs / geo.Lx);
    zs -= geo.Lz * floor(zs / geo.Lz);
    int ixb = min((int)floor(xs / geo.dx), geo.Nx - 1);
    int izb = min((int)floor(zs / geo.dz), geo.Nz - 1);
    const int N = geo.Ny - 1;
    const double pi = 3.14159265358979323846, rc = geo.rcut;
    double yb = fmin(1.0, fmax(-1.0, 2.0 * (ys - geo.y0) / geo.W - 1.0));
    int jn = min(max((int)rint(acos(yb) * N / pi), 0), N);
    double yh = fmin(1.0, yb + 2.0 * rc / geo.W), yl = fmax(-1.0, yb - 2.0 * rc / geo.W);
    int jlo = max(0, (int)floor(acos(yh) * N / pi) - 1);
    int jhi = min(N, (int)ceil(acos(yl) * N / pi) + 1);
    di[s] = make_int4(ixb, izb, jn, jlo | (jhi << 16));
    v4_t<T> f;
    f.x = (T)(xs - ixb * geo.dx);
    f.y = (T)(zs - izb * geo.dz);
    f.z = (T)(ys - yj[jn]);
    f.w = (T)0;
    df[s] = f;
}

template <typename T> __device__ __forceinline__ T sexp(T x);
template <> __device__ __forceinline__ float sexp<float>(float x) { return expf(x); }
template <> __device__ __forceinline__ double sexp<double>(double x) { return exp(x); }

// per-kernel constants in T (computed on the host); lo, hi: r_cut^2 less and
// more than the rounding of a single-precision r^2
template <typename T> struct SpreadConst {
    T dx, dz, rc2, al2, cn;
    float lo, hi;
};

constexpr int MAXJ = 272;     // max y nodes of one source stencil (checked on the host)
constexpr int MAXR = 32;      // max columns / rows of one source's stencil

// vector reduction into an interleaved (x, y, z, pad) node
__device__ __forceinline__ void red4(float* p, float a, float b, float c) {
    atomicAdd(reinterpret_cast<float4*>(p), make_float4(a, b, c, 0.f));
}
__device__ __forceinline__ void red4(double* p, double a, double b, double c) {
    atomicAdd(p, a);
    atomicAdd(p + 1, b);
    atomicAdd(p + 2, c);
}

// e + y < r_cut^2 in T; FP64 decides in single precision except within its
// rounding of the cutoff
__device__ __forceinline__ bool inside(const SpreadConst<float>& k, float e, float y, float, float) {
    return e + y < k.rc2;
}
__device__ __forceinline__ bool inside(const SpreadConst<double>& k, double e, double y, float ef,
                                       float yf) {
    const float s = ef + yf;
    return s < k.lo || (s <= k.hi && e + y < k.rc2);
}

// Two consecutive sorted sources per warp.  Neighbouring sources share most of
// their stencils (the nodes within r_cut: columns with dx^2 < rc^2, rows with
// dz^2 < rc^2, planes of the y-range), so the warp walks the union of the two
// stencils, evaluates both weights at every node and issues one reduction with
// their sum: fewer reductions, which bound this kernel.  A pair whose union does
// not fit 32 columns or 32 rows (sources far apart in the sorted order), and an
// odd last source, run one after the other with an empty partner.
// Lanes build the separable factors of the columns, rows and planes in shared
// memory, then walk the (column, row) pairs; each lane runs its pair's planes.
// With -c g e_xz and a^2 d_xz^2 e formed once per column and e_y (5/2 - a^2 dy^2)
// once per plane, a node takes per source one FMA for
//   e_y (5/2 - a^2 r^2) = [e_y (5/2 - a^2 dy^2)] - a^2 d_xz^2 e_y
// and three for the components (FP64, where the pipe counts: 4 operations per node
// and source instead of 8, and one reduction per two sources; with the column list
// 64,200 sources 6.25 -> 4.5 ms per call).
// gridDim.y parts share the planes of every pair: calls with few sources are
// bound by one warp's walk through a stencil, not by the reductions (1,296 sources
// in FP32 96 -> 40 us, without the launch that took handed-back pairs; 162 in FP64
// 136 -> 77).
template <typename T>
__host__ __device__ constexpr size_t pair_smem(int Ny) {
    return ((256 + 6 * (size_t)Ny) * sizeof(T) + 64 * 4 +
            (sizeof(T) == 8 ? 2048 + 8 * (size_t)Ny : 0) + 15) & ~(size_t)15;
}

template <typename T, int WPB>
__global__ void __launch_bounds__(WPB * 32) k_spread_pair(
    GridGeom geo, SpreadConst<T> kc, const T* __restrict__ ydiff, int n, int R,
    const int4* __restrict__ sdi, const v4_t<T>* __restrict__ sdf,
    const v4_t<T>* __restrict__ gsrc, T* __restrict__ f4) {
    // per warp: column and row tables, then three plane tables of Ny per source
    // (sized by Ny: a table for the largest Ny would halve the resident warps)
    extern __shared__ __align__(16) unsigned char smraw[];
    const int Nyp = geo.Ny;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sa = 2 * (blockIdx.x * WPB + wid);
    if (sa >= n) return;                                    // warp-uniform
    unsigned char* wb = smraw + (size_t)wid * pair_smem<T>(Nyp);
    T* s_t = reinterpret_cast<T*>(wb);                       // x d^2, x e, z d^2, z e: [4][2][32]
    T* s_y = s_t + 256;                                      // y d^2, y e, y e q: [3][2][Ny]
    int* s_i = reinterpret_cast<int*>(s_y + 6 * Nyp);        // column, row: [2][32]
    unsigned short* s_c = reinterpret_cast<unsigned short*>(s_i + 64);   // FP64: columns [1024]
    float* s_yf = reinterpret_cast<float*>(s_c + 1024);      // FP64: y d^2 in single: [2][Ny]
    auto XZ = [&](int k, int s, int i) -> T& { return s_t[(k * 2 + s) * 32 + i]; };
    auto YT = [&](int k, int s, int q) -> T& { return s_y[(k * 2 + s) * Nyp + q]; };
    const T rc2 = kc.rc2, al2 = kc.al2;
    const int Nx = geo.Nx, Nz = geo.Nz;
    const int nr = 2 * R + 2;
    const size_t rowst = (size_t)Nx * 4, planest = (size_t)Nz * Nx * 4;
    for (int pass = 0; pass < 2; ++pass) {
        // this pass's sources: the pair, or one of them with an empty partner
        int s0 = sa, s1 = sa + 1 < n ? sa + 1 : sa;
        int4 d0 = sdi[s0], d1 = sdi[s1];
        // signed periodic offsets of source 1's base column/row from source 0's
        int ox = d1.x - d0.x, oz = d1.y - d0.y;
        ox -= (ox > Nx / 2) ? Nx : 0;
        ox += (ox < -Nx / 2) ? Nx : 0;
        oz -= (oz > Nz / 2) ? Nz : 0;
        oz += (oz < -Nz / 2) ? Nz : 0;
        const bool fit = s1 != s0 && abs(ox) + nr <= 32 && abs(oz) + nr <= 32;
        if (pass == 1 && (fit || s1 == s0)) return;          // warp-uniform
        if (!fit) {
            s0 = pass == 0 ? s0 : s1;
            d0 = d1 = sdi[s0];
            ox = oz = 0;
        }
        // the union of offsets [-R, R+1] (source 0) and [o - R, o + R + 1] (source 1),
        // relative to source 0's base column / row
        const int bx = min(0, ox) - R, bz = min(0, oz) - R;
        const int spx = abs(ox) + nr, spz = abs(oz) + nr;
        const v4_t<T> f0 = sdf[s0], f1 = fit ? sdf[s1] : f0;
        __syncwarp();
        // columns and rows of the union: lane = union offset
        {
            const int c = bx + lane;                          // column offset from s0's base
            T v0x = (T)1e30, v1x = (T)1e30;
            if (lane < spx) {
                const int o0 = c + R, o1 = c - ox + R;        // offsets into each stencil
                if (o0 >= 0 && o0 < nr) { T v = fma((T)(o0 - R), kc.dx, -f0.x); v0x = v * v; }
                if (fit && o1 >= 0 && o1 < nr) { T v = fma((T)(o1 - R), kc.dx, -f1.x); v1x = v * v; }
            }
            XZ(0, 0, lane) = v0x;
            XZ(0, 1, lane) = v1x;
            XZ(1, 0, lane) = v0x < rc2 ? sexp<T>(-al2 * v0x) : (T)0;
            XZ(1, 1, lane) = v1x < rc2 ? sexp<T>(-al2 * v1x) : (T)0;
            s_i[lane] = (d0.x + c) & (Nx - 1);
            const int r = bz + lane;
            T v0z = (T)1e30, v1z = (T)1e30;
            if (lane < spz) {
                const int o0 = r + R, o1 = r - oz + R;
                if (o0 >= 0 && o0 < nr) { T v = fma((T)(o0 - R), kc.dz, -f0.y); v0z = v * v; }
                if (fit && o1 >= 0 && o1 < nr) { T v = fma((T)(o1 - R), kc.dz, -f1.y); v1z = v * v; }
            }
            XZ(2, 0, lane) = v0z;
            XZ(2, 1, lane) = v1z;
            XZ(3, 0, lane) = v0z < rc2 ? sexp<T>(-al2 * v0z) : (T)0;
            XZ(3, 1, lane) = v1z < rc2 ? sexp<T>(-al2 * v1z) : (T)0;
            s_i[32 + lane] = (d0.y + r) & (Nz - 1);
        }
        // planes: this part's share of the union of the two y-ranges
        int jlo = min(d0.w & 0xffff, d1.w & 0xffff), jhi = max(d0.w >> 16, d1.w >> 16);
        {
            const int len = jhi - jlo + 1, np = gridDim.y, per = (len + np - 1) / np;
            jlo += per * blockIdx.y;
            jhi = min(jhi, jlo + per - 1);
        }
        const int ny = jhi - jlo + 1;
        for (int q = lane; q < ny; q += 32) {
            const T a0 = ydiff[(size_t)(jlo + q) * geo.Ny + d0.z] - f0.z;
            const T a1 = ydiff[(size_t)(jlo + q) * geo.Ny + d1.z] - f1.z;
            const T q0 = a0 * a0, q1 = a1 * a1;
            const T e0 = sexp<T>(-al2 * q0), e1 = sexp<T>(-al2 * q1);
            YT(0, 0, q) = q0;
            YT(0, 1, q) = q1;
            YT(1, 0, q) = e0;
            YT(1, 1, q) = e1;
            YT(2, 0, q) = e0 * ((T)2.5 - al2 * q0);
            YT(2, 1, q) = e1 * ((T)2.5 - al2 * q1);
            if (sizeof(T) == 8) {
                s_yf[q] = (float)q0;
                s_yf[Nyp + q] = (float)q1;
            }
        }
        __syncwarp();
        const v4_t<T> g0 = gsrc[s0], g1 = gsrc[s1];
        const T h = fit ? -kc.cn : (T)0;
        const T ax = -kc.cn * g0.x, ay = -kc.cn * g0.y, az = -kc.cn * g0.z;
        const T cx = h * g1.x, cy = h * g1.y, cz = h * g1.z;
        const int npair = spx * spz;
        const float inx = 1.0f / (float)spx;
        // FP64: a list of the columns within r_cut of either source, the long chords
        // first, so that the lanes of a warp walk alike (a warp's FP64 instruction
        // takes 16 cycles whatever its active lanes: 6.7 -> 4.5 ms on 100 capsules);
        // FP32 takes the whole box row by row, which its reductions coalesce along
        const unsigned lt = (1u << lane) - 1u;
        constexpr bool listed = sizeof(T) == 8;
        int ncol = listed ? 0 : npair;
        for (int shell = 0; listed && shell < 2; ++shell)
            for (int p0 = 0; p0 < npair; p0 += 32) {
                const int pi = p0 + lane;
                const int b = (int)(((float)pi + 0.5f) * inx);
                const int a = pi - b * spx;
                bool in = false;
                if (pi < npair) {
                    const T e = fmin(XZ(0, 0, a) + XZ(2, 0, b), XZ(0, 1, a) + XZ(2, 1, b));
                    in = shell == 0 ? e < (T)0.5 * rc2 : e >= (T)0.5 * rc2 && e < rc2;
                }
                const unsigned m = __ballot_sync(0xffffffffu, in);
                if (in) s_c[ncol + __popc(m & lt)] = (unsigned short)(a | (b << 8));
                ncol += __popc(m);
            }
        __syncwarp();
        for (int pi = lane; pi < ncol; pi += 32) {
            int b = (int)(((float)pi + 0.5f) * inx), a = pi - b * spx;
            if (listed) {
                a = s_c[pi] & 255;
                b = s_c[pi] >> 8;
            }
            const T e0 = XZ(0, 0, a) + XZ(2, 0, b);
            const T e1 = XZ(0, 1, a) + XZ(2, 1, b);
            if (!(e0 < rc2) && !(e1 < rc2)) continue;
            const T x0 = XZ(1, 0, a) * XZ(3, 0, b);
            const T x1 = XZ(1, 1, a) * XZ(3, 1, b);
            const T m0 = -al2 * e0, m1 = -al2 * e1;
            const T ux = ax * x0, uy = ay * x0, uz = az * x0;
            const T vx = cx * x1, vy = cy * x1, vz = cz * x1;
            const float e0f = (float)e0, e1f = (float)e1;
            T* col = f4 + (size_t)s_i[32 + b] * rowst + (size_t)s_i[a] * 4;
            for (int q = 0; q < ny; ++q) {
                const T y0 = YT(0, 0, q), y1 = YT(0, 1, q);
                const bool wide = sizeof(T) == 8;
                const bool in0 = inside(kc, e0, y0, e0f, wide ? s_yf[q] : 0.f),
                           in1 = inside(kc, e1, y1, e1f, wide ? s_yf[Nyp + q] : 0.f);
                if (!in0 && !in1) continue;
                const T w0 = in0 ? fma(m0, YT(1, 0, q), YT(2, 0, q)) : (T)0;
                const T w1 = in1 ? fma(m1, YT(1, 1, q), YT(2, 1, q)) : (T)0;
                red4(col + (size_t)(jlo + q) * planest, fma(ux, w0, vx * w1), fma(uy, w0, vy * w1),
                     fma(uz, w0, vz * w1));
            }
        }
    }
}

// interleaved [Ny][Nz][Nx][4] -> planar [Ny][3][Nz][Nx]
template <typename T>
__global__ void k_deinterleave(int Ny, int Nz, int Nx, const T* __restrict__ f4,
                               T* __restrict__ grid) {
    size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t plane = (size_t)Nz * Nx;
    if (e >= (size_t)Ny * plane) return;
    size_t j = e / plane, r = e - j * plane;
    const T* p = f4 + e * 4;
    T* o = grid + j * 3 * plane + r;
    o[0] = p[0];
    o[plane] = p[1];
    o[2 * plane] = p[2];
}
}  // namespace

template <typename T>
cudaError_t spread_prepare(const GridGeom& geo, const double* yj, int n, const int* perm,
                           const double* x, int4* di, v4_t<T>* df, cudaStream_t st) {
    // small blocks: three FP64 arc cosines per source, bound by each SM's FP64 pipe
    // (8,000 sources in 32 blocks of 256 threads: 18 us, all of it on 32 SMs)
    if (n > 0) k_src_desc<T><<<(n + 31) / 32, 32, 0, st>>>(geo, yj, n, perm, x, di, df);
    return cudaGetLastError();
}

template <typename T>
cudaError_t spread(const GridGeom& geo, const CellGrid& cg, const double* yj, const T* ydiff,
                   const SortedSources<T>& src, const int4* di, const v4_t<T>* df, T* grid,
                   T* work, int nsm, cudaStream_t st) {
    (void)cg; (void)yj;
    int R = (int)std::ceil(std::max(geo.rcut / geo.dx, geo.rcut / geo.dz)) + 1;
    if (2 * R + 2 > MAXR || geo.Ny > MAXJ) return cudaErrorInvalidConfiguration;
    const double pi = 3.14159265358979323846;
    SpreadConst<T> kc;
    kc.dx = (T)geo.dx; kc.dz = (T)geo.dz;
    kc.rc2 = (T)(geo.rcut * geo.rcut);
    kc.al2 = (T)(geo.alpha * geo.alpha);
    kc.cn = (T)(geo.alpha * geo.alpha * geo.alpha / (pi * std::sqrt(pi)));
    kc.lo = (float)(geo.rcut * geo.rcut * (1.0 - 1e-6));
    kc.hi = (float)(geo.rcut * geo.rcut * (1.0 + 1e-6));
    size_t nodes = (size_t)geo.Ny * geo.Nz * geo.Nx;
    cudaMemsetAsync(work, 0, nodes * 4 * sizeof(T), st);
    if (src.n > 0) {
        constexpr int WPB = 4;
        const int npairs = (src.n + 1) / 2;
        // few pairs: share their planes between up to 4 warps, to 16 warps per SM.  The
        // stage with at most 1, 2, 4, 8, 16 parts (us): 162 sources in FP64 177, 111, 76, 64,
        // 75, in FP32 46, 31, 26, 22, 19; 648 sources 261, 169, 138, 142, 139 and 66, 44,
        // 34, 28, 29; from 1,296 sources on the second bound decides
        const int parts = std::max(1, std::min(4, 16 * nsm / npairs));
        const dim3 g((unsigned)((npairs + WPB - 1) / WPB), (unsigned)parts);
        const size_t smem = WPB * pair_smem<T>(geo.Ny);
        grant_max_smem((const void*)k_spread_pair<T, WPB>);
        k_spread_pair<T, WPB><<<g, WPB * 32, smem, st>>>(geo, kc, ydiff, src.n, R, di, df, src.g,
                                                        work);
    }
    k_deinterleave<T><<<(unsigned)((nodes + 255) / 256), 256, 0, st>>>(geo.Ny, geo.Nz, geo.Nx,
                                                                       work, grid);
    return cudaGetLastError();
}

#define GGEM_INST_SPREAD(T)                                                                  \
    template cudaError_t spread_prepare<T>(const GridGeom&, const double*, int, const int*,    \
                                           const double*, int4*, v4_t<T>*, cudaStream_t);       \
    template cudaError_t spread<T>(const GridGeom&, const CellGrid&, const double*, const T*,   \
                                   const SortedSources<T>&, const int4*, const v4_t<T>*, T*,    \
                                   T*, int, cudaStream_t);
GGEM_INST_SPREAD(float)
GGEM_INST_SPREAD(double)

// ------------------------------------------------------------------ probe
// Throughput of float4 vector reductions into an L2-resident buffer, the
// operation the spreading is bound by: every warp adds into 32 consecutive
// 16-byte vectors (one per lane, as lanes on consecutive grid columns do) at a
// pseudo-random position of the buffer, `iters` times.  The roof the
// spreading's reduction rate is measured against.
namespace {
__global__ void k_red_probe(float4* __restrict__ buf, unsigned nvec, int iters, unsigned seed) {
    const unsigned w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    unsigned h = (w + 1u) * 2654435761u ^ seed;
    for (int it = 0; it < iters; ++it) {
        h = h * 1664525u + 1013904223u;
        const unsigned base = (h % (nvec >> 5)) << 5;
        atomicAdd(buf + base + lane, make_float4(1.f, 1.f, 1.f, 0.f));
    }
}

// Throughput of FP32 atomic adds into shared memory, the operation a spreading
// staged in shared memory would be bound by: a block holds a tile of 4096
// nodes x 3 components (48 KB, as a 16 x 16 x 16 tile of the grid), and every
// warp adds into 32 consecutive nodes (one per lane: no bank conflict within
// the warp) of each component at a pseudo-random place of the tile, `iters`
// times; the warps of a block collide as the sources of a tile would.  The
// tile is added into `out` at the end so that the adds are kept.
constexpr int kProbeNodes = 4096;
__global__ void k_smem_probe(float* __restrict__ out, int iters, unsigned seed) {
    __shared__ float acc[3 * kProbeNodes];
    for (int e = threadIdx.x; e < 3 * kProbeNodes; e += blockDim.x) acc[e] = 0.f;
    __syncthreads();
    const unsigned w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    unsigned h = (w + 1u) * 2654435761u ^ seed;
    for (int it = 0; it < iters; ++it) {
        h = h * 1664525u + 1013904223u;
        const unsigned base = ((h >> 8) % (kProbeNodes >> 5)) << 5;
        atomicAdd(&acc[base + lane], 1.f);
        atomicAdd(&acc[kProbeNodes + base + lane], 1.f);
        atomicAdd(&acc[2 * kProbeNodes + base + lane], 1.f);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 3 * kProbeNodes; e += blockDim.x) atomicAdd(out + e, acc[e]);
}
}  // namespace

}  // namespace ggem

extern "C" ggem_status ggem_probe_smem_reduction(int iters, void* stream, double* ms,
                                                 double* adds_per_s) {
    if (iters < 1 || iters > (1 << 20) || !ms || !adds_per_s) return GGEM_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return GGEM_ERR_CUDA;
    const size_t nout = (size_t)3 * ggem::kProbeNodes;
    float* out = nullptr;
    cudaEvent_t a = nullptr, b = nullptr;
    ggem_status s = GGEM_OK;
    if (cudaMalloc((void**)&out, nout * sizeof(float)) != cudaSuccess) return GGEM_ERR_CUDA;
    const int blocks = 4 * nsm, threads = 256;     // 48 KB per block: 4 blocks per SM
    if (cudaMemsetAsync(out, 0, nout * sizeof(float), st) != cudaSuccess ||
        cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) {
        s = GGEM_ERR_CUDA;
    } else {
        ggem::k_smem_probe<<<blocks, threads, 0, st>>>(out, iters, 7u);  // warm
        cudaEventRecord(a, st);
        ggem::k_smem_probe<<<blocks, threads, 0, st>>>(out, iters, 11u);
        cudaEventRecord(b, st);
        float t = 0.f;
        if (cudaEventSynchronize(b) != cudaSuccess || cudaEventElapsedTime(&t, a, b) != cudaSuccess ||
            cudaGetLastError() != cudaSuccess) {
            s = GGEM_ERR_CUDA;
        } else {
            *ms = t;
            *adds_per_s = 3.0 * blocks * threads * iters / (t * 1e-3);
        }
    }
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
    cudaFree(out);
    return s;
}

extern "C" ggem_status ggem_probe_l2_reduction(long nvec, int iters, void* stream, double* ms,
                                               double* vec_per_s) {
    if (nvec < 32 || (nvec & 31) || nvec > (1L << 28) || iters < 1 || !ms || !vec_per_s)
        return GGEM_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return GGEM_ERR_CUDA;
    float4* buf = nullptr;
    cudaEvent_t a = nullptr, b = nullptr;
    ggem_status s = GGEM_OK;
    if (cudaMalloc((void**)&buf, (size_t)nvec * sizeof(float4)) != cudaSuccess)
        return GGEM_ERR_CUDA;
    const int blocks = 8 * nsm, threads = 256;
    if (cudaMemsetAsync(buf, 0, (size_t)nvec * sizeof(float4), st) != cudaSuccess ||
        cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) {
        s = GGEM_ERR_CUDA;
    } else {
        ggem::k_red_probe<<<blocks, threads, 0, st>>>(buf, (unsigned)nvec, iters, 7u);  // warm
        cudaEventRecord(a, st);
        ggem::k_red_probe<<<blocks, threads, 0, st>>>(buf, (unsigned)nvec, iters, 11u);
        cudaEventRecord(b, st);
        float t = 0.f;
        if (cudaEventSynchronize(b) != cudaSuccess || cudaEventElapsedTime(&t, a, b) != cudaSuccess ||
            cudaGetLastError() != cudaSuccess) {
            s = GGEM_ERR_CUDA;
        } else {
            *ms = t;
            *vec_per_s = (double)blocks * threads * iters / (t * 1e-3);
        }
    }
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
    cudaFree(buf);
    return s;
}
