// FP64-accurate element rule in double-float arithmetic (FP64-emulated plans,
// the twins that give mixed solves their true residuals): the local single-
// and double-layer sums of Sec. 3.4.1 / 3.5.2 over the quadrature points.
//
// Lengths are scaled by sqrt(2) alpha.  Offsets from the cell centres are split
// on a common grid Q = 2^-24 of the cell size (rounded up to a power of two): hi
// a multiple of Q (of its own ulp where that is larger), lo the remainder.  The
// difference of two hi parts is then exact when the target's is the smaller,
// as both lie within half a cell, and otherwise its error takes two operations
// (Dekker's fast two-sum); positions are good to 2^-49 of a cell.  The kernels' smooth parts are piecewise
// polynomials in s = r^2 (ggem_fftab.cuh): per pair one reciprocal square root
// and two polynomials, no exponential and no erfc.
#include <algorithm>
#include <cmath>

#include "ggem_internal.cuh"
#include "ggem_ff.cuh"
#include "ggem_fftab.cuh"

namespace ggem {

namespace {

constexpr int FW = 4;         // warps (targets) per block, 6 blocks per SM (80 registers): 27.8 ms per
                              //   launch against 28.0 (3 blocks of 8), 29.3 (64 registers, 8 blocks of 4)
constexpr int kQueueF = 64;   // hit queue per warp: < 32 left + <= 32 new always fit
constexpr int kCapF = 64;     // culled cells per batch
constexpr int RF = kElemReach, kSideF = 2 * RF + 1;

// x = hi + lo, hi a multiple of Q (mag = 1.5 2^52 Q: adding it rounds to one)
__device__ __forceinline__ ff split_on_grid(double x, double mag) {
    const float h = (float)((x + mag) - mag);
    return {h, (float)(x - (double)h)};
}
// t - p, normalised: lo is of the size of Q whatever the difference, and its
// square is dropped further on
__device__ __forceinline__ ff grid_diff(float2 t, float ph, float pl) {
    const float s = t.x - ph;
    return fast_two_sum(s, (t.y - pl) + ((t.x - s) - ph));
}

// positions of the sorted points: hi[s] = (x, y, z hi, -), lo[s] = (x, y, z lo, -)
__global__ void k_ff_positions(int n, const double4_32a* __restrict__ pos, double lam, double mag,
                               double cx, double cy, double cz, float4* __restrict__ hi,
                               float4* __restrict__ lo) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const double4_32a p = pos[s];
    const ff x = split_on_grid((p.x - cx) * lam, mag), y = split_on_grid((p.y - cy) * lam, mag),
             z = split_on_grid((p.z - cz) * lam, mag);
    hi[s] = make_float4(x.hi, y.hi, z.hi, 0.f);
    lo[s] = make_float4(x.lo, y.lo, z.lo, 0.f);
}

// strengths g = scale sum_v (phi_v w) q_v of the sorted points in pairs: gx
// into the free words of hi and lo, gy and gz into g
__global__ void k_ff_strengths(int n, const int4* __restrict__ qv,
                               const double4_32a* __restrict__ qw, const double* __restrict__ q,
                               double scale, float4* __restrict__ hi, float4* __restrict__ lo,
                               float4* __restrict__ g) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const int4 v = qv[s];
    const double4_32a w = qw[s];
    const double a = scale * w.x, b = scale * w.y, c = scale * w.z;
    ff r[3];
    for (int i = 0; i < 3; ++i)
        r[i] = ff_from_double(a * q[3 * (size_t)v.x + i] + b * q[3 * (size_t)v.y + i] +
                              c * q[3 * (size_t)v.z + i]);
    hi[s].w = r[0].hi;
    lo[s].w = r[0].lo;
    g[s] = make_float4(r[1].hi, r[1].lo, r[2].hi, r[2].lo);
}

struct FFArgs {
    int n_tgt;
    const double4_32a* tpos;         // sorted targets: offsets from the cell corner,
    const int* tcell;                //   cell,
    const int* tperm;                //   caller index
    const int* nstart;               // neighbour lists of the target cells
    const int4* nbr;
    const unsigned short* noff;
    const float4* hi;                // sorted points
    const float4* lo;
    const float4* g;
    const int4* qvs;                 // their triangles' vertices
    const double* nrm;               // [n][3] target normals (caller order)
    double* out;
    int out_stride;
    double lam, mag, hx, hy, hz;     // scale, grid, scaled cell size
    ff rc2;                          // scaled r_cut^2
    float rc2_up, near2_up;          // widened for the single-precision test
    double fac;                      // output factor
};

// The block's tables in shared memory, interval fastest.
struct FFTab {
    float2 pair[2][GGEM_FF_PAIRS][GGEM_FF_NINT];
    float4 tail[2][GGEM_FF_NINT];
};

// f(s) on interval i, u = s - i.  The coefficients fall by at least 1/(2 (k +
// 1)) per degree and |u| <= 1/2, so each Horner step's sum has its larger term
// first.
__device__ __forceinline__ ff ff_poly(const FFTab& t, int f, int i, ff u) {
    const float4 c = t.tail[f][i];
    const float q = fmaf(fmaf(c.z, u.hi, c.y), u.hi, c.x);
    float2 k = t.pair[f][GGEM_FF_PAIRS - 1][i];
    const float ph = __fmul_rn(q, u.hi);
    ff p = fast_two_sum(k.x, ph);
    p.lo += fmaf(q, u.lo, fmaf(q, u.hi, -ph)) + k.y;
#pragma unroll
    for (int d = GGEM_FF_PAIRS - 2; d >= 0; --d) {
        k = t.pair[f][d][i];
        const ff m = ff_mul(p, u);
        p = fast_two_sum(k.x, m.hi);
        p.lo += m.lo + k.y;
    }
    return p;
}

struct FFSum {
    ff u[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    ff sn = {0.f, 0.f};              // double layer: sum of E x.g
};

// One target per warp.  The warp culls its cell's neighbour list, walks the
// kept cells with consecutive lanes on consecutive points, testing each in
// single precision (hi parts, widened cutoff), compacts the hits into a queue
// and evaluates 32 at a time: the strict cutoff is tested there, in pairs, and
// the points that fail it count with zero strength.
// What bounds it: FP32 issue (about 430 FP32 operations per pair, of which the
// two polynomials 126).  100 capsules, double layer: 59.1 ms with exp by a
// 2^(j/16) reduction, erfcx from the FP64 table, every operation normalised and
// the update not regrouped (about 1,230 instructions per pair); 27.8 ms here.
// Error of the double layer against FP64 torch 1.11e-14 before, 1.07e-14 now.
template <int LAYER>
__global__ void __launch_bounds__(FW * 32, 6) k_local_elem_ff(FFArgs a) {
    __shared__ FFTab tab;
    __shared__ int s_st[FW][kCapF];
    __shared__ int s_cnt[FW][kCapF];             // bit 31: may hold the target's own triangles
    __shared__ float2 s_t[FW][kCapF][3];         // target in the frame of the cell's centre
    __shared__ int2 s_q[FW][kQueueF];            // queued hits: sorted point, cell slot
    for (int e = threadIdx.x; e < 2 * GGEM_FF_PAIRS * GGEM_FF_NINT; e += blockDim.x)
        (&tab.pair[0][0][0])[e] = (&kFFPair[2 * LAYER][0][0])[e];
    for (int e = threadIdx.x; e < 2 * GGEM_FF_NINT; e += blockDim.x)
        (&tab.tail[0][0])[e] = (&kFFTail[2 * LAYER][0])[e];
    __syncthreads();
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = blockIdx.x * FW + wid;
    if (t >= a.n_tgt) return;                     // warp-uniform
    const double4_32a tp = a.tpos[t];
    const int c = a.tcell[t], oidx = a.tperm[t];
    const double ox = tp.x * a.lam, oy = tp.y * a.lam, oz = tp.z * a.lam;
    const float fx = (float)ox, fy = (float)oy, fz = (float)oz;
    const float hx = (float)a.hx, hy = (float)a.hy, hz = (float)a.hz;
    ff n[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    if (LAYER == 1)
        for (int i = 0; i < 3; ++i) n[i] = ff_from_double(a.nrm[3 * (size_t)oidx + i]);
    const unsigned lt = (1u << lane) - 1u;
    const float rc2u = a.rc2_up, near2u = a.near2_up;
    FFSum acc;

    auto eval = [&](int s, int ci) {
        const float4 ph = a.hi[s], pl = a.lo[s], pg = a.g[s];
        const float2 tx = s_t[wid][ci][0], ty = s_t[wid][ci][1], tz = s_t[wid][ci][2];
        const ff d[3] = {grid_diff(tx, ph.x, pl.x), grid_diff(ty, ph.y, pl.y),
                         grid_diff(tz, ph.z, pl.z)};
        ff r2 = ff_norm(ff_sum3(ff_sqr(d[0]), ff_sqr(d[1]), ff_sqr(d[2])));
        ff g[3] = {{ph.w, pl.w}, {pg.x, pg.y}, {pg.z, pg.w}};
        // (the tables end at s = 72.5, r = 6.02 / alpha: a longer r_cut is cut there,
        // where the terms are exp(-36) of the near field that every sum holds too)
        const bool ok = (r2.hi < a.rc2.hi || (r2.hi == a.rc2.hi && r2.lo < a.rc2.lo)) &&
                        r2.hi > 0.f && r2.hi < (float)GGEM_FF_NINT - 0.5f;
        if (!ok) {
            r2 = {1.f, 0.f};
            for (int i = 0; i < 3; ++i) g[i] = {0.f, 0.f};
        }
        // nearest interval centre and the exact remainder
        const float m = r2.hi + 12582912.f;
        const int iv = __float_as_int(m) & 127;
        const ff u = {r2.hi - (m - 12582912.f), r2.lo};
        const ff ir = ff_rsqrt(r2), ir2 = ff_sqr(ir);
        const ff xg = ff_dot(d, g);
        if (LAYER == 0) {
            const ff A = ff_sub(ir, ff_poly(tab, 0, iv, u));
            const ff B = ff_mul(ff_sub(ff_mul(ir2, ir), ff_poly(tab, 1, iv, u)), xg);
            for (int i = 0; i < 3; ++i) ff_acc(acc.u[i], ff_add(ff_mul(A, g[i]), ff_mul(B, d[i])));
        } else {
            const ff D = ff_sub(ff_poly(tab, 0, iv, u), ff_mul(ff_norm(ff_sqr(ir2)), ir));
            const ff E = ff_poly(tab, 1, iv, u);
            const ff xn = ff_dot(d, n), gn = ff_dot(g, n);
            // D xg xn d + E (d gn + g xn + n xg), the last term's scalar summed
            const ff cd = ff_add(ff_mul(ff_mul(D, xg), xn), ff_mul(E, gn)), cg = ff_mul(E, xn);
            ff_acc(acc.sn, ff_mul(E, xg));
            for (int i = 0; i < 3; ++i)
                ff_acc(acc.u[i], ff_add(ff_mul(cd, d[i]), ff_mul(cg, g[i])));
        }
    };

    const int nend = a.nstart[c + 1];
    for (int i = a.nstart[c]; i < nend;) {
        // a batch of culled cells
        int nc = 0;
        for (; i < nend && nc + 32 <= kCapF; i += 32) {
            bool keep = false, nearc = false;
            int4 e = make_int4(0, 0, 0, 0);
            int ix = 0, iy = 0, iz = 0;
            if (i + lane < nend) {
                e = a.nbr[i + lane];
                const int oi = a.noff[i + lane];
                ix = oi % kSideF - RF;
                iy = (oi / kSideF) % kSideF - RF;
                iz = oi / (kSideF * kSideF) - RF;
                const float gx = ix > 0 ? (float)ix * hx - fx
                                        : (ix < 0 ? fx - (float)(ix + 1) * hx : 0.f);
                const float gy = iy > 0 ? (float)iy * hy - fy
                                        : (iy < 0 ? fy - (float)(iy + 1) * hy : 0.f);
                const float gz = iz > 0 ? (float)iz * hz - fz
                                        : (iz < 0 ? fz - (float)(iz + 1) * hz : 0.f);
                const float d2 = gx * gx + gy * gy + gz * gz;
                keep = d2 <= rc2u * 1.0001f;
                nearc = d2 <= near2u * 1.0001f;
            }
            const unsigned mk = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const int slot = nc + __popc(mk & lt);
                s_st[wid][slot] = e.x;
                s_cnt[wid][slot] = e.w | (nearc ? (int)0x80000000 : 0);
                const ff tx = split_on_grid(ox - (ix + 0.5) * a.hx, a.mag),
                         ty = split_on_grid(oy - (iy + 0.5) * a.hy, a.mag),
                         tz = split_on_grid(oz - (iz + 0.5) * a.hz, a.mag);
                s_t[wid][slot][0] = make_float2(tx.hi, tx.lo);
                s_t[wid][slot][1] = make_float2(ty.hi, ty.lo);
                s_t[wid][slot][2] = make_float2(tz.hi, tz.lo);
            }
            nc += __popc(mk);
        }
        __syncwarp();
        int head = 0, qn = 0;                     // warp-uniform
        for (int ci = 0; ci < nc; ++ci) {
            const int st = s_st[wid][ci], cw = s_cnt[wid][ci], cnt = cw & 0x7fffffff;
            const float tx = s_t[wid][ci][0].x, ty = s_t[wid][ci][1].x, tz = s_t[wid][ci][2].x;
            for (int i0 = 0; i0 < cnt; i0 += 32) {
                const int s = st + i0 + lane;
                bool hit = false;
                if (i0 + lane < cnt) {
                    const float4 p = a.hi[s];
                    const float dx = tx - p.x, dy = ty - p.y, dz = tz - p.z;
                    const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                    hit = r2 < rc2u;
                    if (cw < 0 && r2 < near2u) {
                        const int4 v = a.qvs[s];
                        hit = hit && !(v.x == oidx || v.y == oidx || v.z == oidx);
                    }
                }
                const unsigned m = __ballot_sync(0xffffffffu, hit);
                if (hit) s_q[wid][(head + qn + __popc(m & lt)) & (kQueueF - 1)] = make_int2(s, ci);
                qn += __popc(m);
                if (qn >= 32) {
                    __syncwarp();
                    const int2 e = s_q[wid][(head + lane) & (kQueueF - 1)];
                    eval(e.x, e.y);
                    head = (head + 32) & (kQueueF - 1);
                    qn -= 32;
                    __syncwarp();
                }
            }
        }
        __syncwarp();
        if (lane < qn) {
            const int2 e = s_q[wid][(head + lane) & (kQueueF - 1)];
            eval(e.x, e.y);
        }
        __syncwarp();
    }
    double u[3];
    for (int i = 0; i < 3; ++i) u[i] = ff_to_double(acc.u[i]);
    if (LAYER == 1) {
        const double sn = ff_to_double(acc.sn);
        for (int i = 0; i < 3; ++i) u[i] = fma(ff_to_double(n[i]), sn, u[i]);
    }
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) u[i] += __shfl_xor_sync(0xffffffffu, u[i], o);
    }
    if (lane == 0) {
        double* o = a.out + (size_t)oidx * a.out_stride;
        for (int i = 0; i < 3; ++i) o[i] = a.fac * u[i];
    }
}

double ff_scale(double alpha) { return alpha * 1.4142135623730950488; }

// 1.5 2^52 Q, 2^24 Q the scaled cell size rounded up to a power of two (one more:
// an offset may exceed half a cell by rounding)
double ff_mag(const CellGrid& cg, double lam) {
    const double h = std::max(cg.hx, std::max(cg.hy, cg.hz)) * lam * 1.0001;
    return std::ldexp(6755399441055744.0, (int)std::ceil(std::log2(h)) - 24);
}

}  // namespace

cudaError_t elemff_positions(const GridGeom& geo, const CellGrid& cg, int n,
                             const double4_32a* pos, float4* hi, float4* lo, cudaStream_t st) {
    const double lam = ff_scale(geo.alpha);
    if (n > 0)
        k_ff_positions<<<(n + 255) / 256, 256, 0, st>>>(n, pos, lam, ff_mag(cg, lam), 0.5 * cg.hx,
                                                       0.5 * cg.hy, 0.5 * cg.hz, hi, lo);
    return cudaGetLastError();
}

cudaError_t elemff_strengths(int n, const int4* qv, const double4_32a* qw, const double* q,
                             double scale, float4* hi, float4* lo, float4* g, cudaStream_t st) {
    if (n > 0) k_ff_strengths<<<(n + 255) / 256, 256, 0, st>>>(n, qv, qw, q, scale, hi, lo, g);
    return cudaGetLastError();
}

cudaError_t elemff_sum(const GridGeom& geo, const CellGrid& cg, const ElemLists32& L,
                       const float4* hi, const float4* lo, const float4* g, const int4* qvs,
                       double near, const SortedSources<double>& tgt, const double* nrm, int layer,
                       double* out, int out_stride, cudaStream_t st) {
    if (tgt.n <= 0) return cudaSuccess;
    const double pi = 3.14159265358979323846, lam = ff_scale(geo.alpha);
    FFArgs a;
    a.n_tgt = tgt.n;
    a.tpos = tgt.pos;
    a.tcell = tgt.cell;
    a.tperm = tgt.perm;
    a.nstart = L.nstart;
    a.nbr = L.nbr;
    a.noff = L.noff;
    a.hi = hi;
    a.lo = lo;
    a.g = g;
    a.qvs = qvs;
    a.nrm = nrm;
    a.out = out;
    a.out_stride = out_stride;
    a.lam = lam;
    a.mag = ff_mag(cg, lam);
    a.hx = cg.hx * lam;
    a.hy = cg.hy * lam;
    a.hz = cg.hz * lam;
    const double rc2 = geo.rcut * geo.rcut * lam * lam;
    a.rc2.hi = (float)rc2;
    a.rc2.lo = (float)(rc2 - (double)a.rc2.hi);
    a.rc2_up = (float)(rc2 * (1.0 + 1e-5));
    a.near2_up = (float)(near * near * lam * lam * (1.0 + 1e-5));
    a.fac = (layer == 0 ? lam : 6.0 * lam * lam) / (8.0 * pi * geo.mu);
    const dim3 b(FW * 32), gr((tgt.n + FW - 1) / FW);
    if (layer == 0) k_local_elem_ff<0><<<gr, b, 0, st>>>(a);
    else k_local_elem_ff<1><<<gr, b, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace ggem
