// Cell list and GGEM local sums (paper Sec. 3.2.1, Eqs. (local), (u_loc)).
//
// Sources are binned into cells no smaller than r_cut/R (R = 2 or 3, the
// grid's search reach) and stored as offsets
// from their cell's corner, so every displacement is formed from small
// numbers (integer cell shift + offset difference) and stays accurate in FP32
// whatever the box size.  x and z are periodic: the neighbour shift of up to
// +-R cells carries the image; as r_cut < L/2 (Sec. 3.2.2, alpha L > 8), at
// most one image of a source lies within r_cut even where a small grid
// visits a cell twice.
#include "ggem_internal.cuh"
#include <algorithm>

#include "ggem_erfcx.cuh"
#include "ggem_smooth64.cuh"

namespace ggem {

template <typename T> __device__ __forceinline__ T d_rsqrt(T x);
// FP32: the hardware approximations (about 2 ulp); r^2 lies in (0, r_cut^2) and
// the exponent in (-23, 0], far from denormal inputs and results
template <> __device__ __forceinline__ float d_rsqrt<float>(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
template <> __device__ __forceinline__ double d_rsqrt<double>(double x) { return rsqrt(x); }

// Threads per block of the per-point kernels below: their FP64 divisions and floors run
// at 2 lanes per cycle and SM, so 8,000 points go to 125 blocks, not 32.
constexpr int kPtBlock = 64;

__global__ void k_cell_count(GridGeom geo, CellGrid cg, int n, const double* __restrict__ x,
                             int* __restrict__ count, int* __restrict__ cell_of) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int cx, cy, cz;
    double ox, oy, oz;
    locate(geo, cg, x[3 * i], x[3 * i + 1], x[3 * i + 2], cx, cy, cz, ox, oy, oz);
    int c = (cz * cg.ncy + cy) * cg.ncx + cx;
    cell_of[i] = c;
    atomicAdd(&count[c], 1);
}

// exclusive scan of count[0..n) into start[0..n], one block
__global__ void k_scan(int n, const int* __restrict__ count, int* __restrict__ start) {
    __shared__ int part[1024];
    int tid = threadIdx.x, nt = blockDim.x;
    int chunk = (n + nt - 1) / nt;
    int b = tid * chunk, e = min(n, b + chunk);
    int s = 0;
    for (int i = b; i < e; ++i) s += count[i];
    part[tid] = s;
    __syncthreads();
    for (int off = 1; off < nt; off <<= 1) {
        int v = (tid >= off) ? part[tid - off] : 0;
        __syncthreads();
        part[tid] += v;
        __syncthreads();
    }
    int run = (tid == 0) ? 0 : part[tid - 1];
    for (int i = b; i < e; ++i) {
        start[i] = run;
        run += count[i];
    }
    if (tid == nt - 1) start[n] = part[nt - 1];
}

template <typename T>
__global__ void k_cell_scatter(GridGeom geo, CellGrid cg, int n, const double* __restrict__ x,
                               const int* __restrict__ cell_of, const int* __restrict__ start,
                               int* __restrict__ cursor, int* __restrict__ src_cell,
                               int* __restrict__ perm, v4_t<T>* __restrict__ pos) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int cx, cy, cz;
    double ox, oy, oz;
    locate(geo, cg, x[3 * i], x[3 * i + 1], x[3 * i + 2], cx, cy, cz, ox, oy, oz);
    int c = cell_of[i];
    int slot = start[c] + atomicAdd(&cursor[c], 1);
    perm[slot] = i;
    src_cell[slot] = c;
    v4_t<T> p;
    p.x = (T)ox; p.y = (T)oy; p.z = (T)oz; p.w = (T)0;
    pos[slot] = p;
}

__global__ void k_gather_int4(int n, const int* __restrict__ perm, const int4* __restrict__ in,
                              int4* __restrict__ out) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < n) out[s] = in[perm[s]];
}

cudaError_t gather_int4(int n, const int* perm, const int4* in, int4* out, cudaStream_t st) {
    if (n > 0) k_gather_int4<<<(n + 255) / 256, 256, 0, st>>>(n, perm, in, out);
    return cudaGetLastError();
}

cudaError_t scan_counts(int n, const int* count, int* start, cudaStream_t st) {
    if (n > 0) k_scan<<<1, 1024, 0, st>>>(n, count, start);
    return cudaGetLastError();
}

template <typename T>
cudaError_t build_cells(const GridGeom& geo, const CellGrid& cg, int n, const double* x,
                        int* cell_count, int* cell_start, int* cursor, int* src_cell,
                        int* perm, v4_t<T>* pos, cudaStream_t st) {
    int ncell = cg.ncx * cg.ncy * cg.ncz;
    cudaMemsetAsync(cell_count, 0, ncell * sizeof(int), st);
    cudaMemsetAsync(cursor, 0, ncell * sizeof(int), st);
    if (n > 0) {
        // src_cell doubles as the per-source cell scratch before the scatter
        int* cell_of = cursor + ncell;   // caller provides cursor[ncell + n]
        const int nb = (n + kPtBlock - 1) / kPtBlock;
        k_cell_count<<<nb, kPtBlock, 0, st>>>(geo, cg, n, x, cell_count, cell_of);
        k_scan<<<1, 1024, 0, st>>>(ncell, cell_count, cell_start);
        k_cell_scatter<T><<<nb, kPtBlock, 0, st>>>(geo, cg, n, x, cell_of, cell_start, cursor,
                                                   src_cell, perm, pos);
    } else {
        cudaMemsetAsync(cell_start, 0, (ncell + 1) * sizeof(int), st);
    }
    return cudaGetLastError();
}

template <typename T>
__global__ void k_gather(int n, const int* __restrict__ perm, const double* __restrict__ q,
                         const double* __restrict__ w, double scale, v4_t<T>* __restrict__ g) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    int i = perm[s];
    double f = scale * (w ? w[i] : 1.0);
    v4_t<T> v;
    v.x = (T)(f * q[3 * i]); v.y = (T)(f * q[3 * i + 1]); v.z = (T)(f * q[3 * i + 2]);
    v.w = (T)0;
    g[s] = v;
}

template <typename T>
cudaError_t gather_strengths(int n, const int* perm, const double* q, const double* w,
                             double scale, v4_t<T>* g, cudaStream_t st) {
    if (n > 0) k_gather<T><<<(n + 255) / 256, 256, 0, st>>>(n, perm, q, w, scale, g);
    return cudaGetLastError();
}

// ------------------------------------------------------------- local sum
// Kernel constants in T, computed on the host so that the kernels execute no
// FP64 instruction (GB300 issues FP64 at a small fraction of the FP32 rate).
template <typename T> struct LocalConst {
    T al, al2, rc2, c1, c2, c3, c4, fU, fS, hx, hy, hz;
    T ke;   // -alpha^2 log2(e): exp(-alpha^2 r^2) = 2^(ke r^2)
    T s2, lam, lam3, lam5;   // FP64 tables: 2 alpha^2, powers of sqrt(2) alpha
    bool beyond;             // r_cut reaches beyond the tables
};

template <typename T> LocalConst<T> local_const(const GridGeom& geo, const CellGrid& cg) {
    const double sp = 1.7724538509055160273, pi = 3.14159265358979323846;
    double a = geo.alpha;
    LocalConst<T> k;
    k.al = (T)a; k.al2 = (T)(a * a); k.rc2 = (T)(geo.rcut * geo.rcut);
    k.c1 = (T)(2.0 * a / sp); k.c2 = (T)(12.0 * a / sp);
    k.c3 = (T)(8.0 * a * a * a / sp); k.c4 = (T)(4.0 * a * a * a / sp);
    k.fU = (T)(1.0 / (8.0 * pi * geo.mu)); k.fS = (T)(1.0 / (8.0 * pi));
    k.hx = (T)cg.hx; k.hy = (T)cg.hy; k.hz = (T)cg.hz;
    k.ke = (T)(-a * a * 1.4426950408889634074);
    const double s2 = 2.0 * a * a, lam = a * 1.4142135623730950488;
    k.s2 = (T)s2; k.lam = (T)lam; k.lam3 = (T)(s2 * lam); k.lam5 = (T)(s2 * s2 * lam);
    k.beyond = s2 * geo.rcut * geo.rcut > GGEM_SMOOTH64_NINT - 0.6;
    return k;
}

template <typename T> struct LocalArgs {
    GridGeom geo;
    CellGrid cg;
    LocalConst<T> k;
    SortedSources<T> src;
    const int4* qvs;         // element rule: vertices of each sorted point's triangle
    T near2;                 // element rule: points closer than this may share a triangle
    int n_tgt;
    const int* tcell;        // TK_POINTS / TK_WALL: located targets (cell, offsets)
    const v4_t<T>* tpos;
    const int* tperm;        // TK_POINTS: caller index of target t (nullptr: t itself)
    const double* nrm;       // OUT_DBL: [n][3] target normals (caller order)
    T* out;
    int out_stride;
};

// Locate targets once (one thread each, FP64): cell index and offsets from
// the cell corner in T.  kind TK_POINTS reads x[n][3]; TK_WALL generates the
// wall grid nodes (x_i, y0 or y0+W, z_k), index = (wall * Nz + k) * Nx + i.
template <typename T>
__global__ void k_locate(GridGeom geo, CellGrid cg, int n, int kind, const double* __restrict__ x,
                         int* __restrict__ cell, v4_t<T>* __restrict__ pos) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    double xx, yy, zz;
    if (kind == TK_POINTS) {
        xx = x[3 * t]; yy = x[3 * t + 1]; zz = x[3 * t + 2];
    } else {
        int nxz = geo.Nz * geo.Nx;
        int w = t / nxz, rem = t - w * nxz;
        int k = rem / geo.Nx, i = rem - k * geo.Nx;
        xx = i * geo.dx; zz = k * geo.dz; yy = geo.y0 + w * geo.W;
    }
    int cx, cy, cz;
    double ox, oy, oz;
    locate(geo, cg, xx, yy, zz, cx, cy, cz, ox, oy, oz);
    cell[t] = (cz * cg.ncy + cy) * cg.ncx + cx;
    v4_t<T> p;
    p.x = (T)ox; p.y = (T)oy; p.z = (T)oz; p.w = (T)0;
    pos[t] = p;
}

template <typename T>
cudaError_t locate_targets(const GridGeom& geo, const CellGrid& cg, int n, int kind,
                           const double* x, int* cell, v4_t<T>* pos, cudaStream_t st) {
    if (n > 0)
        k_locate<T><<<(n + kPtBlock - 1) / kPtBlock, kPtBlock, 0, st>>>(geo, cg, n, kind, x, cell,
                                                                       pos);
    return cudaGetLastError();
}

// Pair arithmetic of Eq. (local), shared by the local-sum kernels.
// exp(-alpha^2 r^2) and erfc(alpha r) = exp(-x^2) erfcx(x) with the
// approximations of ggem_erfcx.cuh (FP32: t Q(t), t = 1/(1 + P x), Q of degree
// 7; FP64: 8 polynomial pieces of degree 12, coefficients in shared memory),
// so the pair needs one exponential and no erfc call; the FP32 exponential is
// 2^(ke r^2), the FP32 reciprocal the hardware's.
template <typename T> struct PairAcc {
    T ux = 0, uy = 0, uz = 0;
    T sxx = 0, sxy = 0, sxz = 0, syy = 0, syz = 0, szz = 0;
};

__device__ __forceinline__ float rcp_ftz(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ void exp_erfc(const LocalConst<float>& k, float r2, float x, float& ex,
                                         float& ec, const double*) {
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ex) : "f"(k.ke * r2));
    ec = ex * erfcx_t(rcp_ftz(fmaf(x, GGEM_ERFCX_P, 1.0f)));
}
__device__ __forceinline__ void exp_erfc(const LocalConst<double>& k, double r2, double x,
                                         double& ex, double& ec, const double* tab) {
    ex = exp(-k.al2 * r2);
    ec = ex * erfcx_poly(x, tab);
}

// adds G^l g (OUT_U), T^l g (OUT_S) or n . T^l g (OUT_DBL) for displacement
// (dx, dy, dz) = target - source, 0 < r2 < rc2
template <typename T, int MODE>
__device__ __forceinline__ void pair_terms(const LocalConst<T>& k, T dx, T dy, T dz, T r2,
                                           const v4_t<T>& g, T nx, T ny, T nz, PairAcc<T>& a,
                                           const double* tab) {
    const T ir = d_rsqrt<T>(r2);
    const T r = r2 * ir;
    T ex, ec;
    exp_erfc(k, r2, k.al * r, ex, ec, tab);
    const T xg = dx * g.x + dy * g.y + dz * g.z;
    if (MODE & OUT_U) {
        const T A = ec * ir - k.c1 * ex;
        const T B = (ec * ir * ir * ir + k.c1 * ex * ir * ir) * xg;
        a.ux += A * g.x + B * dx;
        a.uy += A * g.y + B * dy;
        a.uz += A * g.z + B * dz;
    }
    if (MODE & (OUT_S | OUT_DBL)) {
        const T ir2 = ir * ir;
        const T D = -(T)6 * ec * ir2 * ir2 * ir - k.c2 * ex * ir2 * ir2 - k.c3 * ex * ir2;
        const T E = k.c4 * ex;
        if (MODE & OUT_S) {
            const T Dx = D * xg;
            a.sxx += Dx * dx * dx + E * ((T)2 * g.x * dx + xg);
            a.syy += Dx * dy * dy + E * ((T)2 * g.y * dy + xg);
            a.szz += Dx * dz * dz + E * ((T)2 * g.z * dz + xg);
            a.sxy += Dx * dx * dy + E * (g.y * dx + g.x * dy);
            a.sxz += Dx * dx * dz + E * (g.z * dx + g.x * dz);
            a.syz += Dx * dy * dz + E * (g.z * dy + g.y * dz);
        } else {
            const T xn = dx * nx + dy * ny + dz * nz;
            const T gn = g.x * nx + g.y * ny + g.z * nz;
            const T Dxn = D * xg * xn;
            a.ux += Dxn * dx + E * (dx * gn + g.x * xn + nx * xg);
            a.uy += Dxn * dy + E * (dy * gn + g.y * xn + ny * xg);
            a.uz += Dxn * dz + E * (dz * gn + g.z * xn + nz * xg);
        }
    }
}

// Interval of s = 2 alpha^2 r^2 and the remainder in it.
__device__ __forceinline__ int interval64(const LocalConst<double>& k, double r2, double& u) {
    const double m = fma(r2, k.s2, 6755399441055744.0);   // nearest integer in the low bits
    u = fma(r2, k.s2, -(m - 6755399441055744.0));
    return __double2loint(m);
}

// Two polynomials of the tables.  The coefficients come through L1 (12 KB for the
// two; 20 loads of at most five lines per 32 pairs, against some 900 cycles of FP64
// arithmetic).
__device__ __forceinline__ void poly64(const double* a, const double* b, double u, double& p,
                                       double& q) {
    constexpr int N = GGEM_SMOOTH64_NINT;
    p = __ldg(a + GGEM_SMOOTH64_DEG * N);
    q = __ldg(b + GGEM_SMOOTH64_DEG * N);
#pragma unroll
    for (int d = GGEM_SMOOTH64_DEG - 1; d >= 0; --d) {
        p = fma(p, u, __ldg(a + d * N));
        q = fma(q, u, __ldg(b + d * N));
    }
}

// The same beyond the tables (s > 72.5, exp(-36) of the near field): 1 - rho A_g and
// 1 - rho^3 B_g (F = 0), or 1 - rho^5 D_g and E_g, at x = alpha r.
template <int F> __device__ __noinline__ double2 beyond64(double x) {
    const double ec = erfc(x), ex = exp(-x * x), w = 1.1283791670955125739 * x * ex;
    if (F == 0) return make_double2(ec - w, ec + w);
    return make_double2(fma(w, fma(x * x, 2.0 / 3.0, 1.0), ec), 0.13298076013381091 * ex);
}

// The same terms in FP64, one output kind at a time.  Near the target the singular
// parts 1/r, 1/r^3, 1/r^5 less the smooth ones from tables, no exponential and no
// erfc.  That difference loses digits as the kernels decay (3e-15 of them at s = 5,
// 1e-14 at 8, 2e-10 at 32, r_cut = 4 / alpha), so A and B from interval 6 and D from
// interval 4 on come from tables of the scaled kernels, times 1/r, 1/r^3, 1/r^5: below
// 3e-15 everywhere but near the zero of A.  The two differ by selects only: the whole
// double layer of the case below 1.831 -> 1.838 ms.  The double layer is summed over 6 (the caller
// multiplies), its last term's scalar E x.g in a.sxx.  About 55 FP64 instructions
// per pair where exp and erfcx took about 95: element rule, 1,296 targets,
// 40,960 points 3.2 -> 2.0 ms.
template <int MODE>
__device__ __forceinline__ void pair_terms64(const LocalConst<double>& k, double dx, double dy,
                                             double dz, double r2, const double4_32a& g,
                                             double nx, double ny, double nz, PairAcc<double>& a) {
    constexpr int F = MODE == OUT_U ? 0 : 2, N = GGEM_SMOOTH64_NINT;
    const double ir = rsqrt(r2), ir2 = ir * ir;
    const double xg = fma(dz, g.z, fma(dy, g.y, dx * g.x));
    double u, p, q;
    const int i = interval64(k, r2, u);
    const bool far = i >= (F == 0 ? 6 : 4);
    if (k.beyond && i >= N) {
        const double2 e = beyond64<F>(k.al * (r2 * ir));
        p = e.x;
        q = e.y;
    } else {
        const double* ta = (far ? &kFar64[F][0][0] : &kSmooth64[F][0][0]) + i;
        const double* tb = (F == 0 && far ? &kFar64[1][0][0] : &kSmooth64[F + 1][0][0]) + i;
        poly64(ta, tb, u, p, q);
    }
    if (MODE == OUT_U) {
        const double ir3 = ir2 * ir;
        const double A = fma(far ? ir : -k.lam, p, far ? 0.0 : ir);
        const double B = fma(far ? ir3 : -k.lam3, q, far ? 0.0 : ir3) * xg;
        a.ux = fma(B, dx, fma(A, g.x, a.ux));
        a.uy = fma(B, dy, fma(A, g.y, a.uy));
        a.uz = fma(B, dz, fma(A, g.z, a.uz));
    } else {
        const double ir5 = -(ir2 * ir2 * ir);
        const double D = fma(far ? ir5 : k.lam5, p, far ? 0.0 : ir5), E = k.lam3 * q;   // over 6
        if (MODE == OUT_S) {
            // d_i (D xg d_k + E g_k) + E g_i d_k, and E xg on the diagonal
            const double Dx = D * xg, Ex = E * xg;
            const double ex = E * g.x, ey = E * g.y, ez = E * g.z;
            const double tx = fma(Dx, dx, ex), ty = fma(Dx, dy, ey), tz = fma(Dx, dz, ez);
            a.sxx += fma(tx, dx, fma(ex, dx, Ex));
            a.syy += fma(ty, dy, fma(ey, dy, Ex));
            a.szz += fma(tz, dz, fma(ez, dz, Ex));
            a.sxy += fma(ty, dx, ex * dy);
            a.sxz += fma(tz, dx, ex * dz);
            a.syz += fma(tz, dy, ey * dz);
        } else {
            const double xn = fma(dz, nz, fma(dy, ny, dx * nx));
            const double gn = fma(g.z, nz, fma(g.y, ny, g.x * nx));
            const double cd = fma(D * xg, xn, E * gn), cg = E * xn;
            a.sxx = fma(E, xg, a.sxx);
            a.ux = fma(cd, dx, fma(cg, g.x, a.ux));
            a.uy = fma(cd, dy, fma(cg, g.y, a.uy));
            a.uz = fma(cd, dz, fma(cg, g.z, a.uz));
        }
    }
}

// scaled output of one target in caller order
template <typename T, int MODE>
__device__ __forceinline__ void store_target(const LocalConst<T>& k, const PairAcc<T>& a, T* o) {
    int c = 0;
    if (MODE & (OUT_U | OUT_DBL)) {
        o[0] = k.fU * a.ux; o[1] = k.fU * a.uy; o[2] = k.fU * a.uz;
        c = 3;
    }
    if (MODE & OUT_S) {
        o[c] = k.fS * a.sxx; o[c + 1] = k.fS * a.sxy; o[c + 2] = k.fS * a.sxz;
        o[c + 3] = k.fS * a.syy; o[c + 4] = k.fS * a.syz; o[c + 5] = k.fS * a.szz;
    }
}

// Target t: position in its cell's frame, cell coordinates and caller index.
template <typename T, int KIND>
__device__ __forceinline__ void load_target(const LocalArgs<T>& a, int t, T& ox, T& oy, T& oz,
                                            int& cx, int& cy, int& cz, int& oidx) {
    const CellGrid& cg = a.cg;
    v4_t<T> p;
    int c;
    oidx = t;
    if (KIND == TK_SORTED) {
        p = a.src.pos[t];
        c = a.src.cell[t];
        oidx = a.src.perm[t];
    } else {
        p = a.tpos[t];
        c = a.tcell[t];
        if (a.tperm) oidx = a.tperm[t];
    }
    ox = p.x; oy = p.y; oz = p.z;
    cx = c % cg.ncx;
    cy = (c / cg.ncx) % cg.ncy;
    cz = c / (cg.ncx * cg.ncy);
}

// The warp's list of neighbour cells at offsets -R..R (cells are at least
// r_cut/R wide): the non-empty ones whose nearest point lies within r_cut of
// the target (a slightly widened r_cut, so FP32 rounding can only keep more).
// Of S warps with the same target, warp w takes every S-th offset: neighbouring
// cells go to different warps.  Writes first source, count and offset index of each into the warp's
// shared-memory lists; returns their number (warp-uniform).
template <typename T, int R, int S>
__device__ __forceinline__ int cull_cells(const LocalArgs<T>& a, int w, int lane, float ox,
                                          float oy, float oz, int cx, int cy, int cz,
                                          int* s_cst, int* s_cnt, unsigned short* s_off) {
    const CellGrid& cg = a.cg;
    const unsigned lt = (1u << lane) - 1u;
    const float reach2 = (float)a.k.rc2 * 1.0001f;
    const float hx = (float)a.k.hx, hy = (float)a.k.hy, hz = (float)a.k.hz;
    constexpr int side = 2 * R + 1, nb = side * side * side;
    int nc = 0;
    for (int r = 0; r < (nb + 32 * S - 1) / (32 * S); ++r) {
        const int oi = (r * 32 + lane) * S + w;
        bool keep = false;
        int st = 0, cnt = 0;
        if (oi < nb) {
            const int ix = oi % side - R, iy = (oi / side) % side - R, iz = oi / (side * side) - R;
            const int cyy = cy + iy;
            if (cyy >= 0 && cyy < cg.ncy) {
                const float gx = ix > 0 ? (float)ix * hx - ox
                                        : (ix < 0 ? ox - (float)(ix + 1) * hx : 0.f);
                const float gy = iy > 0 ? (float)iy * hy - oy
                                        : (iy < 0 ? oy - (float)(iy + 1) * hy : 0.f);
                const float gz = iz > 0 ? (float)iz * hz - oz
                                        : (iz < 0 ? oz - (float)(iz + 1) * hz : 0.f);
                if (gx * gx + gy * gy + gz * gz <= reach2) {
                    // ncx, ncz >= 2 R (L > 2 r_cut): one wrap suffices for |i| <= R
                    int cxx = cx + ix, czz = cz + iz;
                    cxx += (cxx < 0) ? cg.ncx : 0;
                    cxx -= (cxx >= cg.ncx) ? cg.ncx : 0;
                    czz += (czz < 0) ? cg.ncz : 0;
                    czz -= (czz >= cg.ncz) ? cg.ncz : 0;
                    const int c = (czz * cg.ncy + cyy) * cg.ncx + cxx;
                    st = a.src.cell_start[c];
                    cnt = a.src.cell_start[c + 1] - st;
                    keep = cnt > 0;
                }
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (keep) {
            const int slot = nc + __popc(m & lt);
            s_cst[slot] = st;
            s_cnt[slot] = cnt;
            s_off[slot] = (unsigned short)oi;
        }
        nc += __popc(m);
    }
    __syncwarp();
    return nc;
}

// 0 < r2 < rc2 and r2 < lim, r2 a sum of squares or NaN.  In FP64 on the bit
// patterns (non-negative doubles order like integers; NaN orders above all): an FP64
// comparison costs as much as an addition.
__device__ __forceinline__ bool in_range(float r2, float rc2) { return r2 < rc2 && r2 > 0.f; }
__device__ __forceinline__ bool below(float r2, float lim) { return r2 < lim; }
__device__ __forceinline__ bool in_range(double r2, double rc2) {
    return (unsigned long long)__double_as_longlong(r2) - 1ull <
           (unsigned long long)__double_as_longlong(rc2) - 1ull;
}
__device__ __forceinline__ bool below(double r2, double lim) {
    return (unsigned long long)__double_as_longlong(r2) <
           (unsigned long long)__double_as_longlong(lim);
}

// u_i = sum G^l_ij g_j ; sigma_ik = sum T^l_ijk g_j ; v_i = n_k sigma_ik
// (unscaled in the loop; the caller-facing factors are applied at the end).
//
// One or four warps per target.  Each warp lists its neighbour cells (offsets
// -R..R) that come within r_cut of the target, then walks them one at a time with
// consecutive lanes on consecutive sorted sources (coalesced float4 loads).
// The hits are compacted into a per-warp queue and evaluated 32 at a time.
// Partial sums are reduced with warp shuffles, and over the warps of a target
// in a fixed order.
template <typename T> constexpr int kLW = sizeof(T) == 8 ? 1 : 8;   // warps per block, S = 1
constexpr int kSplit = 4;   // warps per target, and per block, where targets are split
constexpr int kQueue = 64;  // hit queue per warp: < 32 left + <= 32 new always fit
constexpr int kNb = 7 * 7 * 7;   // neighbour cell offsets for the largest reach (3)

// ELEM: sources are element quadrature points and targets are mesh nodes
// (caller index t); points of triangles having the target as a vertex are
// skipped (their integral is done by the polar rule, Sec. 3.4.1).  Used in
// FP64; the FP32 element rule has a kernel of its own (k_local_elem32).
template <typename T, int KIND, int MODE, bool ELEM, int REACH, int S>
__global__ void __launch_bounds__((S > 1 ? S : kLW<T>) * 32) k_local(LocalArgs<T> a) {
    constexpr int LW = S > 1 ? S : kLW<T>, NB = (kNb + 32 * S - 1) / (32 * S) * 32;
    constexpr bool TAB = sizeof(T) == 8 && MODE != (OUT_U | OUT_S);   // FP64 tables
    constexpr bool ERF = sizeof(T) == 8 && !TAB;
    __shared__ int s_cst[LW][NB];             // this warp's cells: first source,
    __shared__ int s_cnt[LW][NB];             //   source count,
    __shared__ unsigned short s_off[LW][NB];  //   neighbour offset index
    __shared__ v4_t<T> s_qd[LW][kQueue];     // queued hits: displacement, r^2
    __shared__ int s_qs[LW][kQueue];         // queued hits: sorted source index
    __shared__ double s_tab[ERF ? (GGEM_ERFCX64_DEG + 1) * GGEM_ERFCX64_NINT : 1];
    if (ERF) {
        for (int e = threadIdx.x; e < (GGEM_ERFCX64_DEG + 1) * GGEM_ERFCX64_NINT; e += blockDim.x)
            s_tab[e] = kErfcxTab64[e];
        __syncthreads();
    }
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = S > 1 ? blockIdx.x : blockIdx.x * LW + wid;
    if (t >= a.n_tgt) return;                     // warp-uniform (S > 1: block-uniform)
    int cx, cy, cz, oidx;
    T ox, oy, oz;
    load_target<T, KIND>(a, t, ox, oy, oz, cx, cy, cz, oidx);
    constexpr int R = REACH, side = 2 * R + 1;
    const unsigned lt = (1u << lane) - 1u;
    const int nc = cull_cells<T, R, S>(a, S > 1 ? wid : 0, lane, (float)ox, (float)oy, (float)oz,
                                       cx, cy, cz, s_cst[wid], s_cnt[wid], s_off[wid]);
    T nx = 0, ny = 0, nz = 0;
    if (MODE & OUT_DBL) {
        nx = (T)a.nrm[3 * oidx]; ny = (T)a.nrm[3 * oidx + 1]; nz = (T)a.nrm[3 * oidx + 2];
    }
    const T rc2 = a.k.rc2;
    PairAcc<T> acc;
    auto eval = [&](const v4_t<T>& d, const v4_t<T>& g) {
        if constexpr (TAB)
            pair_terms64<MODE>(a.k, d.x, d.y, d.z, d.w, g, nx, ny, nz, acc);
        else
            pair_terms<T, MODE>(a.k, d.x, d.y, d.z, d.w, g, nx, ny, nz, acc, s_tab);
    };
    // Lanes test consecutive sources of one cell at a time; hits go to a
    // per-warp ring queue (ballot + popc ranks) and the pair arithmetic runs on
    // 32 queued hits at a time, so no lane idles through it on a miss.
    int head = 0, qn = 0;                         // warp-uniform
    for (int ci = 0; ci < nc; ++ci) {
        const int st = s_cst[wid][ci], cnt = s_cnt[wid][ci], oi = s_off[wid][ci];
        // target position in the frame of this source cell's corner
        const T tx = ox - (T)(oi % side - R) * a.k.hx;
        const T ty = oy - (T)((oi / side) % side - R) * a.k.hy;
        const T tz = oz - (T)(oi / (side * side) - R) * a.k.hz;
        for (int i0 = 0; i0 < cnt; i0 += 32) {
            const int i = i0 + lane;
            bool hit = false;
            T dx = 0, dy = 0, dz = 0, r2 = 0;
            int s = 0;
            if (i < cnt) {
                s = st + i;
                const v4_t<T> p = a.src.pos[s];
                dx = tx - p.x;
                dy = ty - p.y;
                dz = tz - p.z;
                r2 = dx * dx + dy * dy + dz * dz;
                hit = in_range(r2, rc2);
                if (ELEM && hit && below(r2, a.near2)) {
                    const int4 v = a.qvs[s];
                    hit = !(v.x == oidx || v.y == oidx || v.z == oidx);
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (hit) {
                const int slot = (head + qn + __popc(m & lt)) & (kQueue - 1);
                v4_t<T> d;
                d.x = dx; d.y = dy; d.z = dz; d.w = r2;
                s_qd[wid][slot] = d;
                s_qs[wid][slot] = s;
            }
            qn += __popc(m);
            if (qn >= 32) {
                __syncwarp();
                const int slot = (head + lane) & (kQueue - 1);
                const v4_t<T> d = s_qd[wid][slot];
                eval(d, a.src.g[s_qs[wid][slot]]);
                head = (head + 32) & (kQueue - 1);
                qn -= 32;
                __syncwarp();
            }
        }
    }
    __syncwarp();
    if (lane < qn) {
        const int slot = (head + lane) & (kQueue - 1);
        const v4_t<T> d = s_qd[wid][slot];
        eval(d, a.src.g[s_qs[wid][slot]]);
    }
    if (TAB && MODE == OUT_DBL) {
        const T sn = acc.sxx;
        acc.ux = (T)6 * (acc.ux + nx * sn);
        acc.uy = (T)6 * (acc.uy + ny * sn);
        acc.uz = (T)6 * (acc.uz + nz * sn);
    }
    if (TAB && MODE == OUT_S) {
        acc.sxx *= (T)6; acc.sxy *= (T)6; acc.sxz *= (T)6;
        acc.syy *= (T)6; acc.syz *= (T)6; acc.szz *= (T)6;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (MODE & (OUT_U | OUT_DBL)) {
            acc.ux += __shfl_xor_sync(0xffffffffu, acc.ux, o);
            acc.uy += __shfl_xor_sync(0xffffffffu, acc.uy, o);
            acc.uz += __shfl_xor_sync(0xffffffffu, acc.uz, o);
        }
        if (MODE & OUT_S) {
            acc.sxx += __shfl_xor_sync(0xffffffffu, acc.sxx, o);
            acc.sxy += __shfl_xor_sync(0xffffffffu, acc.sxy, o);
            acc.sxz += __shfl_xor_sync(0xffffffffu, acc.sxz, o);
            acc.syy += __shfl_xor_sync(0xffffffffu, acc.syy, o);
            acc.syz += __shfl_xor_sync(0xffffffffu, acc.syz, o);
            acc.szz += __shfl_xor_sync(0xffffffffu, acc.szz, o);
        }
    }
    if (S > 1) {
        // lane 0 of every warp holds its part; the first warp's adds them in order
        __shared__ T s_part[LW][9];
        T* p = s_part[wid];
        if (lane == 0) {
            if (MODE & (OUT_U | OUT_DBL)) {
                p[0] = acc.ux; p[1] = acc.uy; p[2] = acc.uz;
            }
            if (MODE & OUT_S) {
                p[3] = acc.sxx; p[4] = acc.sxy; p[5] = acc.sxz;
                p[6] = acc.syy; p[7] = acc.syz; p[8] = acc.szz;
            }
        }
        __syncthreads();
        if (threadIdx.x != 0) return;
        for (int w = 1; w < LW; ++w) {
            const T* o = s_part[w];
            if (MODE & (OUT_U | OUT_DBL)) {
                acc.ux += o[0]; acc.uy += o[1]; acc.uz += o[2];
            }
            if (MODE & OUT_S) {
                acc.sxx += o[3]; acc.sxy += o[4]; acc.sxz += o[5];
                acc.syy += o[6]; acc.syz += o[7]; acc.szz += o[8];
            }
        }
    }
    if (lane != 0) return;
    if (KIND == TK_WALL) {
        // global wall data u^g = -u^l (Sec. 3.2.2), layout [wall][c][Nz][Nx]
        const T f = -a.k.fU;
        const int nxz = a.geo.Nz * a.geo.Nx;
        const int wall = t / nxz, rem = t - wall * nxz;
        T* o = a.out + (size_t)wall * 3 * nxz + rem;
        o[0] = f * acc.ux;
        o[nxz] = f * acc.uy;
        o[2 * nxz] = f * acc.uz;
        return;
    }
    store_target<T, MODE>(a.k, acc, a.out + (size_t)oidx * a.out_stride);
}

// Whether a target's cells are split over the kSplit warps of a block.  A call with few
// targets is a chain of latencies, which four warps share; with many targets the
// chip is full and four partly filled last batches cost more than one.
// FP32, one against four warps: 1,296 nodal targets 21.2 -> 14.9 us, 2,592 20.9 ->
// 18.9, 5,184 33.3 -> 35.2, 10,368 39.9 -> 45.9; free targets 2,000 33.9 -> 30.0,
// 100,000 1.87 -> 1.83 ms (20,000 sources) and .60 -> .73 (1,000).  FP64 sums fill
// the FP64 pipe with a few warps per SM: 162 targets 35 -> 18 us, 648 40 -> 42,
// 1,296 80 -> 88.
template <typename T> static bool split_targets(int n_tgt, int nsm) {
    return n_tgt <= (sizeof(T) == 8 ? 2 : 24) * nsm;
}

template <typename T, int KIND, int MODE, int REACH>
static void launch_split(const LocalArgs<T>& a, bool split, cudaStream_t st) {
    constexpr int LW = kLW<T>;
    if (split)
        k_local<T, KIND, MODE, false, REACH, kSplit><<<a.n_tgt, kSplit * 32, 0, st>>>(a);
    else
        k_local<T, KIND, MODE, false, REACH, 1><<<(a.n_tgt + LW - 1) / LW, LW * 32, 0, st>>>(a);
}

template <typename T, int KIND, int REACH>
static void launch_kind(const LocalArgs<T>& a, int mode, int nsm, cudaStream_t st) {
    const bool sp = split_targets<T>(a.n_tgt, nsm);
    if (KIND == TK_WALL) {
        launch_split<T, KIND, OUT_U, REACH>(a, sp, st);
        return;
    }
    switch (mode) {
        case OUT_U: launch_split<T, KIND, OUT_U, REACH>(a, sp, st); break;
        case OUT_S: launch_split<T, KIND, OUT_S, REACH>(a, sp, st); break;
        case OUT_U | OUT_S: launch_split<T, KIND, OUT_U | OUT_S, REACH>(a, sp, st); break;
        case OUT_DBL: launch_split<T, KIND, OUT_DBL, REACH>(a, sp, st); break;
        default: break;
    }
}

// the grid's search reach as a compile-time constant: 2 (cells >= r_cut/2, nodal
// plans) or 3 (cells >= r_cut/3, element plans)
template <typename T, int KIND>
static void launch_kind(const LocalArgs<T>& a, int mode, int nsm, cudaStream_t st) {
    if (a.cg.reach == 3) launch_kind<T, KIND, 3>(a, mode, nsm, st);
    else launch_kind<T, KIND, 2>(a, mode, nsm, st);
}

// Always four warps per target: the 16 points per triangle give each plenty of pairs, and
// the SMs' shares of the targets even out (1,296 targets 2.04 -> 1.88 ms, 648
// .66 -> .50, 16,200 18.4 -> 16.4).
cudaError_t local_sum_elem(const GridGeom& geo, const CellGrid& cg,
                           const SortedSources<double>& src, const int4* qvs, double near,
                           const SortedSources<double>& tgt, const double* nrm_tgt, int layer,
                           double* out, int out_stride, cudaStream_t st) {
    if (tgt.n <= 0) return cudaSuccess;
    // targets: the mesh nodes in cell order, so neighbouring blocks mostly scan
    // the same candidate cells (L1 / L2 reuse); output in caller order
    LocalArgs<double> a{geo, cg, local_const<double>(geo, cg), src, qvs, near * near, tgt.n,
                        tgt.cell, tgt.pos, tgt.perm, nrm_tgt, out, out_stride};
    auto* kf = layer == 0 ? k_local<double, TK_POINTS, OUT_U, true, kElemReach, kSplit>
                          : k_local<double, TK_POINTS, OUT_DBL, true, kElemReach, kSplit>;
    kf<<<tgt.n, kSplit * 32, 0, st>>>(a);
    return cudaGetLastError();
}

template <typename T>
cudaError_t local_sum(const GridGeom& geo, const CellGrid& cg, const SortedSources<T>& src,
                      int kind, int n_tgt, const int* tcell, const v4_t<T>* tpos,
                      const double* nrm_tgt, int out_mode, T* out, int out_stride, int nsm,
                      cudaStream_t st) {
    if (n_tgt <= 0) return cudaSuccess;
    LocalArgs<T> a{geo, cg, local_const<T>(geo, cg), src, nullptr, (T)0, n_tgt, tcell, tpos,
                   nullptr, nrm_tgt, out, out_stride};
    if (kind == TK_SORTED) launch_kind<T, TK_SORTED>(a, out_mode, nsm, st);
    else if (kind == TK_POINTS) launch_kind<T, TK_POINTS>(a, out_mode, nsm, st);
    else launch_kind<T, TK_WALL>(a, OUT_U, nsm, st);
    return cudaGetLastError();
}

#define GGEM_INST_LOCAL(T)                                                                   \
    template cudaError_t build_cells<T>(const GridGeom&, const CellGrid&, int, const double*, \
                                        int*, int*, int*, int*, int*, v4_t<T>*, cudaStream_t); \
    template cudaError_t gather_strengths<T>(int, const int*, const double*, const double*,   \
                                             double, v4_t<T>*, cudaStream_t);                  \
    template cudaError_t local_sum<T>(const GridGeom&, const CellGrid&,                       \
                                      const SortedSources<T>&, int, int, const int*,          \
                                      const v4_t<T>*, const double*, int, T*, int, int,        \
                                      cudaStream_t);                                           \
    template cudaError_t locate_targets<T>(const GridGeom&, const CellGrid&, int, int,        \
                                           const double*, int*, v4_t<T>*, cudaStream_t);
GGEM_INST_LOCAL(float)
GGEM_INST_LOCAL(double)

}  // namespace ggem
