// PCG of the MIXED field solve with a fast-diagonalisation preconditioner (Lynch,
// Rice and Thomas 1964): in MIXED the default for single field solves of
// FD_MIN_NODES nodes or more and on batches' clusters, where the x-y plane fits in
// shared memory.  (Sec. 2.5: the matrix solve is a PCG iteration stopped on the
// relative residual; the paper names no preconditioner.)
//
// A context's own steps stay with Jacobi (multigrid beyond the registers), though
// this solver is faster there too (0.33 against 0.69 ms a solve at 64^3, 3.1 against
// 3.9 at 160 x 160 x 80): solvers that stop at the same residual differ by up to 2e-5
// of the largest potential, and the object's mean potential is smaller than that is
// when it passes through zero, so that a run's first steps differed there by 1e-3 of
// it (50^3 eighth sphere) from what they were.
//
// Preconditioner.  The free nodes of the box (Dirichlet faces removed) form a
// tensor grid, and the 7-point operator on it with a permittivity that depends
// on z alone is
//     P = h (Kx My Mz + Mx Ky Mz + Mx My Kz),
// K the 1D stiffness and M the lumped 1D mass along an axis (Mz, Kz weighted
// with the permittivity profile).  With V the M-orthonormal eigenvectors of
// K v = lambda M v along x and y (sines and cosines for every pair of Dirichlet
// / Neumann ends), P^-1 r is: the transform r^ = Vy^T r Vx of every plane, one
// tridiagonal system (lx + ly) Mz + Kz along z per mode, and the transform back
// Vy r^ Vx^T.  On a mesh without object the 5-tet operator A lies between 2/3 P
// and 7/6 P (its odd rows are 2/3 of the 7-point row, its even rows add the
// face diagonals), so the iteration count does not grow with the mesh.  The
// object enters through a diagonal scaling S, z = S P^-1 S r with
// S = (eps_n / sqrt(profile))^(-1/4), eps_n the node's diagonal over the
// plasma's, and the profile's square root in P: the exponents that needed the
// fewest iterations on the sphere (eps 4, 10), crater and layered set-ups (12,
// 18, 14 and 15 for 1e-6 from a random start on 32^3 to 60 x 30 x 30 cells; 17,
// 28, 17 and 27 without S and profile; Jacobi 84, 93, 170 and 227).
//
// Layout.  A plane's transform is two small matrix products (for half a plane of
// a 64^3 box 63 x 63 x 32), on the tensor cores: every FP32 operand is split into
// two BF16 parts, head and tail (16 bits), and a product takes three mma.sync
// (head head, head tail, tail head) with FP32 accumulation.  The preconditioner
// only shapes the search directions -- the vectors, products with A, dot
// products and the FP64 residual that ends the solve are not touched by the
// split, and the iteration counts equal those of an FP32 transform.  (3xTF32
// needs twice the products and splits in the inner loop: 33 against 22 us an
// iteration at 64^3, on the node layout.)  A block takes one plane and a chunk of its output columns, so
// both products of a transform stay in the block: the plane split on its way into
// shared memory, the first product's result split again next to it; the basis
// matrices come split and in fragment order from L1 (16 bytes per lane).
//
// The tridiagonal pass holds 32 modes in a block's registers, a run of z rows per
// warp; the warps' runs are joined through their end values (a two-level
// recurrence), so the dependent chain is a run plus one step per warp instead of
// 2 mz steps.
//
// Vectors.  The solve's vectors live in a box of their own: the free nodes, rows
// padded to 16 bytes with at least one zero, one zero row after each plane and a
// zero guard plane on either side.  Every access is then a 16-byte load of four
// nodes, absent neighbours (Dirichlet or beyond a Neumann face) read as zero, and a
// row's coefficients depend on position only through the number of cubes on either
// side (1 on a Neumann face, else 2).  On the node layout, one node at a time, the
// passes issued about 830 instructions a node and iteration, bound by issue: 22 us
// an iteration at 64^3, 18 in the box.
//
// One iteration is four team barriers, two of which carry the reductions
// (Chronopoulos and Gear's form: both dot products after one matrix product):
//   A  q = w + beta q, r -= alpha q, p = z + beta p, x += alpha p (folded into the
//      load of the plane), transform; r.r
//   B  tridiagonal systems
//   C  transform back: z
//   D  w = A z; r.z and w.z
#include <math.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "field_common.cuh"
#include "internal.h"
#include "pcg_team.cuh"

namespace pf {

constexpr int FD_THREADS = 512;
constexpr int FD_WARPS = FD_THREADS / 32;
constexpr int FD_MAX_OUTER = 12;           // refinement steps at most
constexpr int FD_MAX_RUN = 16;             // z rows of a warp in the tridiagonal pass at most
constexpr double FD_MARGIN = 0.2;          // with Neumann faces: the inner solves' target below the tolerance (at most)
constexpr double FD_INNER_RED = 1e-6;      // an inner solve's reduction between Dirichlet faces (at most)
// node kinds (FdPlan::kind)
enum : unsigned {
    FK_INNER = 1,                          // inside the object
    FK_PATCH = 2,                          // row next to interface tets (explicit coefficients)
    FK_PAD = 4,                            // no node
    FK_CX = 8, FK_CY = 16, FK_CZ = 32,     // cubes on one side only along the axis (a Neumann face)
    FK_ODD = 64
};

struct FdArgs {
    FieldArgs f;
    const double* b;              // FP64 right-hand side (nodes)
    const double* g;              // Dirichlet values (nodes)
    double* phi;                  // potential out (nodes)
    FdPlan d;
    int npatch;
    double tol2, inner_red2, margin2;
    int maxit;
    double* val;
    unsigned long long* arrivals;
    unsigned long long* fx;       // fixed-point exchange words: r.r, r.z and w.z
    const int* hold;
    PcgState* S;
    long long* it_total;
    long long* outer_total;
    int* err;
};
static_assert(sizeof(FdArgs) <= 4096, "the solve arguments travel as a kernel parameter");

// the reductions of a team: over the grid the fixed-point exchange (its words
// are used in turn with other exchanges, as it requires), over a cluster the
// plain one
struct FdGrid : GridTeam<FdArgs> {
    unsigned long long prev_rr = 0, prev_gd = 0;
    __device__ FdGrid(const FdArgs& a, int& e, ExchShared& xs) : GridTeam<FdArgs>{a, e, xs} {
        if (threadIdx.x < 2) {
            prev_rr = ld_relaxed(a.fx);
            prev_gd = ld_relaxed(a.fx + (1 + threadIdx.x) * FX_LINE);
        }
    }
    __device__ bool sum_rr(float (&v)[1], const float (&ref)[1], float (&tot)[1]) {
        return exchange_f32<1, true, 8>(a, e, a.fx, prev_rr, ref, fx_ref_ok(ref[0]), v, tot, xs);
    }
    __device__ bool sum_gd(float (&v)[2], const float (&ref)[2], float (&tot)[2]) {
        return exchange_f32<2, true, 8>(a, e, a.fx + FX_LINE, prev_gd, ref, fx_ref_ok(ref[0]) && fx_ref_ok(ref[1]), v,
                                        tot, xs);
    }
};

struct FdCluster : ClusterTeam {
    __device__ FdCluster(cg::cluster_group& cl, int C, ClusterSlots& cs)
        : ClusterTeam{cl, C, (int)cl.block_rank(), 0, cs} {}
    __device__ bool sum_rr(float (&v)[1], const float (&)[1], float (&tot)[1]) { return reduce<float, 1>(v, tot); }
    __device__ bool sum_gd(float (&v)[2], const float (&)[2], float (&tot)[2]) { return reduce<float, 2>(v, tot); }
};

// ---- split products ----------------------------------------------------------------
// head and tail of two neighbouring values, packed as the products take them
static __device__ __forceinline__ uint2 bf16_split(float x0, float x1) {
    uint2 o;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(o.x) : "f"(x1), "f"(x0));
    const float t0 = x0 - __uint_as_float(o.x << 16), t1 = x1 - __uint_as_float(o.x & 0xFFFF0000u);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(o.y) : "f"(t1), "f"(t0));
    return o;
}
static __device__ __forceinline__ void mma_bf16(float (&c)[4], const uint4& a, unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// one block's product C = A B: mt 16-row tiles of A (fragments fa: head and tail of
// tile (m, k) at 64 (m ks + k) + lane, + 32), nt 8-column tiles of B ([column][ld]
// split pairs along the depth, in shared memory), ks 16-deep steps; a warp takes 16
// rows and NT column tiles at a time.  out(m, n, c): rows g, g + 8 and columns 2t,
// 2t + 1 of tile (m, n), g = lane / 4, t = lane % 4.
template <int NT, class OUT>
static __device__ __forceinline__ void fd_product_nt(int mt, int nt, int ks, const uint4* fa, const uint2* B, int ld,
                                                     OUT out) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int ng = (nt + NT - 1) / NT;
    for (int unit = threadIdx.x >> 5; unit < mt * ng; unit += FD_WARPS) {
        const int gi = unit / mt, m = unit - gi * mt, n0 = gi * NT;
        constexpr int NA = NT == 1 ? 3 : 1;    // one tile alone: an accumulator per part, for shorter chains
        float c[NT * NA][4];
#pragma unroll
        for (int n = 0; n < NT * NA; ++n)
#pragma unroll
            for (int q = 0; q < 4; ++q) c[n][q] = 0.0f;
        const uint4* ap = fa + (size_t)m * ks * 64 + lane;
        const uint2* bp[NT];                   // (a column tile past the end repeats the last one)
#pragma unroll
        for (int n = 0; n < NT; ++n) bp[n] = B + (min(n0 + n, nt - 1) * 8 + g) * ld + t;
#pragma unroll 4
        for (int k = 0; k < ks; ++k) {
            const uint4 ah = ap[k * 64], al = ap[k * 64 + 32];
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                const uint2 b0 = bp[n][k * 8], b1 = bp[n][k * 8 + 4];
                mma_bf16(c[n * NA], ah, b0.x, b1.x);
                mma_bf16(c[n * NA + (NA > 1)], ah, b0.y, b1.y);
                mma_bf16(c[n * NA + 2 * (NA > 1)], al, b0.x, b1.x);
            }
        }
#pragma unroll
        for (int n = 0; n < NT; ++n)
            if (n0 + n < nt) {
                if (NA > 1)
#pragma unroll
                    for (int q = 0; q < 4; ++q) c[0][q] += c[NA > 1][q] + c[2 * (NA > 1)][q];
                out(m, n0 + n, c[n * NA]);
            }
    }
}
template <class OUT>
static __device__ __forceinline__ void fd_product(int ntw, int mt, int nt, int ks, const uint4* fa, const uint2* B,
                                                  int ld, OUT out) {
    if (ntw == 1) fd_product_nt<1>(mt, nt, ks, fa, B, ld, out);
    else if (ntw == 2) fd_product_nt<2>(mt, nt, ks, fa, B, ld, out);
    else fd_product_nt<4>(mt, nt, ks, fa, B, ld, out);
}

// a block's share of the transforms: chunk c of the planes k0, k0 + dk, ... (every
// plane's chunks go to nch different blocks), and its fragments, in shared memory
// where they fit (a barrier empties L1, and an L2 round trip is as long as a small
// product)
struct FdShare {
    int c, k0, dk, m0, mta;
    uint2 *X, *Y;
    const uint4 *fxF, *fxI, *fyF, *fyI;
};
template <class Team>
static __device__ FdShare fd_share(const FdPlan& d, const Team& team, uint2* sm) {
    FdShare h;
    h.dk = team.ctas() / d.nch;
    h.c = team.rank_of() % d.nch;
    h.k0 = team.rank_of() / d.nch;
    if (h.k0 >= h.dk) h.k0 = d.mz;         // (a rank beyond the last whole group has no plane)
    h.m0 = h.c * d.mta;
    h.mta = min(d.mta, d.ksx - h.m0);
    h.X = sm;
    h.Y = h.X + d.pb * d.ksy * 16 * d.ldX;
    h.fxF = d.fxF + (size_t)h.m0 * d.ksx * 64;
    h.fxI = d.fxI + (size_t)h.m0 * d.ksx * 64;
    h.fyF = d.fyF;
    h.fyI = d.fyI;
    if (d.stage) {
        uint4* f = reinterpret_cast<uint4*>(sm + d.stage);
        const int nx = d.mta * d.ksx * 64, nxh = h.mta * d.ksx * 64, ny = d.ksy * d.ksy * 64;
        for (int e = threadIdx.x; e < nxh; e += FD_THREADS) { f[e] = h.fxF[e]; f[nx + e] = h.fxI[e]; }
        for (int e = threadIdx.x; e < ny; e += FD_THREADS) { f[2 * nx + e] = h.fyF[e]; f[2 * nx + ny + e] = h.fyI[e]; }
        h.fxF = f; h.fxI = f + nx; h.fyF = f + 2 * nx; h.fyI = f + 2 * nx + ny;
    }
    return h;                              // (the first reduction's barrier comes before any use)
}

// the transform of np planes in X, the block's chunk of columns: Y = fx X (to shared
// memory, transposed and split), then out(plane, m, n, c) = fy Y
template <class OUT>
static __device__ __forceinline__ void fd_transform(const FdPlan& d, const FdShare& h, int np, const uint4* fx,
                                                    const uint4* fy, OUT out) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    fd_product(d.nt1, h.mta, 2 * d.ksy * np, d.ksx, fx, h.X, d.ldX, [&](int m, int n, const float (&c)[4]) {
        const int pl = n / (2 * d.ksy);
        uint2* yp = h.Y + ((pl * h.mta + m) * 16 + g) * d.ldY + (n - pl * 2 * d.ksy) * 4 + t;
        yp[0] = bf16_split(c[0], c[1]);
        yp[8 * d.ldY] = bf16_split(c[2], c[3]);
    });
    __syncthreads();
    fd_product(d.nt2, d.ksy, 2 * h.mta * np, d.ksy, fy, h.Y, d.ldY, [&](int m, int n, const float (&c)[4]) {
        const int pl = n / (2 * h.mta);
        out(pl, m, n - pl * 2 * h.mta, c);
    });
}

// ---- the passes of one iteration -------------------------------------------------------
static __device__ __forceinline__ float4 ld4(const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }
static __device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
static __device__ __forceinline__ float4 axpy4(float a, float4 x, float4 y) {
    return make_float4(y.x + a * x.x, y.y + a * x.y, y.z + a * x.z, y.w + a * x.w);
}

// the rows of a group of np planes, 16-byte columns spread over the block: f(row of X,
// plane, row, column / 4) for the columns [0, nc4)
template <class F>
static __device__ __forceinline__ void fd_rows(int rows, int np, int nc4, F f) {
    int row = threadIdx.x / nc4, c4 = threadIdx.x - row * nc4;
    const int dr = FD_THREADS / nc4, dc = FD_THREADS - dr * nc4;
#pragma unroll 2
    while (row < rows * np) {
        const int pl = np == 1 ? 0 : row / rows;
        f(row, pl, row - pl * rows, c4);
        c4 += dc;
        row += dr;
        if (c4 >= nc4) { c4 -= nc4; row += 1; }
    }
}

// A: T = Vy^T (S r) Vx per plane.  upd: q = w + beta q and r -= alpha q first, from one
// copy of q and r to the other (every block of a plane forms them; the rows of its
// share are written here, with p = z + beta p and x += alpha p); rr gets this thread's
// partial of r.r
static __device__ void fd_forward(const FdArgs& a, const FdShare& h, bool upd, int cur, float alpha, float beta,
                                  float& rr) {
    const FdPlan& d = a.d;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const float *ro = d.r[cur], *qo = d.q[cur];
    float *rn = d.r[cur ^ 1], *qn = d.q[cur ^ 1];
    const bool old = beta != 0.0f;         // (the first update has no old q and p)
    for (int kb = h.k0; kb < d.mz; kb += h.dk * d.pb) {
        const int np = min(d.pb, (d.mz - 1 - kb) / h.dk + 1);
        fd_rows(d.ksy * 16, np, d.ksx * 4, [&](int row, int pl, int j, int c4) {
            uint4 o = make_uint4(0u, 0u, 0u, 0u);
            if (j < d.my && c4 * 4 < d.ldv) {
                const int n = (kb + pl * h.dk) * d.PV + j * d.ldv + c4 * 4;
                float4 r = ld4(ro + n);
                const float4 s = __ldg(reinterpret_cast<const float4*>(d.s + n));
                if (upd) {
                    const bool own = d.nch == 1 || j % d.nch == h.c;
                    const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    const float4 w = ld4(d.w + n), q0 = old ? ld4(qo + n) : zero;
                    const float4 z = own ? ld4(d.z + n) : zero, p0 = own && old ? ld4(d.p + n) : zero;
                    const float4 x = own ? ld4(d.x + n) : zero;
                    const float4 q = axpy4(beta, q0, w);
                    r = axpy4(-alpha, q, r);
                    if (own) {
                        const float4 p = axpy4(beta, p0, z);
                        st4(qn + n, q);
                        st4(rn + n, r);
                        st4(d.p + n, p);
                        st4(d.x + n, axpy4(alpha, p, x));
                        rr += (r.x * r.x + r.y * r.y) + (r.z * r.z + r.w * r.w);
                    }
                }
                const uint2 lo = bf16_split(r.x * s.x, r.y * s.y), hi = bf16_split(r.z * s.z, r.w * s.w);
                o = make_uint4(lo.x, lo.y, hi.x, hi.y);
            }
            *reinterpret_cast<uint4*>(h.X + row * d.ldX + c4 * 2) = o;
        });
        __syncthreads();
        fd_transform(d, h, np, h.fxF, h.fyF, [&](int pl, int m, int n, const float (&v)[4]) {
            const int b = m * 16 + g;
            float* Tk = d.T + (size_t)(kb + pl * h.dk) * d.PT + b * d.ldT + h.m0 * 16 + n * 8 + 2 * t;
            if (b < d.my) *reinterpret_cast<float2*>(Tk) = make_float2(v[0], v[1]);
            if (b + 8 < d.my) *reinterpret_cast<float2*>(Tk + 8 * d.ldT) = make_float2(v[2], v[3]);
        });
        __syncthreads();
    }
}

// B: the tridiagonal systems along z.  WT warps take 32 modes at a time, each a run of RW
// rows: y_k = f_k i_k + (e_{k-1} i_k) y_{k-1} down and x_k = y_k + (e_k i_k) x_{k+1} up,
// each run first from a zero start, then corrected with the value that enters it times
// the run's products; i the inverted pivots.
template <int WT, int RW, class Team>
static __device__ void fd_tridiag_runs(const FdArgs& a, const Team& team, float2* sm) {
    const FdPlan& d = a.d;
    constexpr int NG = FD_WARPS / WT;      // tiles of 32 modes a block works on at once
    const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5, w = wb % WT, k0 = w * RW;
    const int tiles = (int)(d.PT / 32), step = team.ctas() * NG;
    float em[RW + 1];                      // couplings e_{k0-1} .. e_{k0+RW-1}
#pragma unroll
    for (int r = 0; r <= RW; ++r) em[r] = (k0 + r >= 1 && k0 + r < d.mz) ? __ldg(d.ez + k0 + r - 1) : 0.0f;
    float2* ends = sm + (wb / WT) * 4 * WT * 32 + lane;
    int par = 0;
    for (int t0 = team.rank_of(); t0 < tiles; t0 += step) {
        const int tile = t0 + (wb / WT) * team.ctas();
        float y[RW], iv[RW], pr[RW];
        const int at = k0 * (int)d.PT + tile * 32 + lane;
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            const bool ok = tile < tiles && k0 + r < d.mz;
            y[r] = ok ? __ldcg(d.T + at + r * (int)d.PT) : 0.0f;
            iv[r] = ok ? __ldg(d.inv + at + r * (int)d.PT) : 0.0f;
        }
        float2* dn = ends + par * 2 * WT * 32;   // run ends, down then up
        float2* up = dn + WT * 32;
        par ^= 1;
        float v = 0.0f, c = 1.0f;
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            const float ci = em[r] * iv[r];
            v = y[r] * iv[r] + ci * v;
            c = ci * c;
            y[r] = v;
            pr[r] = c;
        }
        dn[w * 32] = make_float2(v, c);
        __syncthreads();
        v = 0.0f;
        for (int q = 0; q < w; ++q) {
            const float2 s = dn[q * 32];
            v = s.x + s.y * v;
        }
#pragma unroll
        for (int r = 0; r < RW; ++r) y[r] += pr[r] * v;
        v = 0.0f;
        c = 1.0f;
#pragma unroll
        for (int r = RW - 1; r >= 0; --r) {
            const float ci = em[r + 1] * iv[r];
            v = y[r] + ci * v;
            c = ci * c;
            y[r] = v;
            pr[r] = c;
        }
        up[w * 32] = make_float2(v, c);
        __syncthreads();
        v = 0.0f;
        for (int q = WT - 1; q > w; --q) {
            const float2 s = up[q * 32];
            v = s.x + s.y * v;
        }
#pragma unroll
        for (int r = 0; r < RW; ++r)
            if (tile < tiles && k0 + r < d.mz) d.T[at + r * (int)d.PT] = y[r] + pr[r] * v;
    }
}
template <class Team>
static __device__ __forceinline__ void fd_tridiag(const FdArgs& a, const Team& team, float2* sm) {
    if (a.d.mz <= 64) fd_tridiag_runs<8, 8>(a, team, sm);
    else if (a.d.mz <= 128) fd_tridiag_runs<16, 8>(a, team, sm);
    else fd_tridiag_runs<16, 16>(a, team, sm);
}

// C: z = S Vy T Vx^T per plane
static __device__ void fd_backward(const FdArgs& a, const FdShare& h) {
    const FdPlan& d = a.d;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    for (int kb = h.k0; kb < d.mz; kb += h.dk * d.pb) {
        const int np = min(d.pb, (d.mz - 1 - kb) / h.dk + 1);
        fd_rows(d.ksy * 16, np, d.ksx * 4, [&](int row, int pl, int j, int c4) {
            uint4 o = make_uint4(0u, 0u, 0u, 0u);
            if (j < d.my) {
                const float4 v = ld4(d.T + (size_t)(kb + pl * h.dk) * d.PT + j * d.ldT + c4 * 4);
                const uint2 lo = bf16_split(v.x, v.y), hi = bf16_split(v.z, v.w);
                o = make_uint4(lo.x, lo.y, hi.x, hi.y);
            }
            *reinterpret_cast<uint4*>(h.X + row * d.ldX + c4 * 2) = o;
        });
        __syncthreads();
        fd_transform(d, h, np, h.fxI, h.fyI, [&](int pl, int m, int n, const float (&v)[4]) {
            const int i = h.m0 * 16 + n * 8 + 2 * t;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int j = m * 16 + g + 8 * q;
                if (j < d.my && i < d.mx) {
                    const int l = (kb + pl * h.dk) * d.PV + j * d.ldv + i;
                    const float2 s = __ldg(reinterpret_cast<const float2*>(d.s + l));
                    *reinterpret_cast<float2*>(d.z + l) =
                        make_float2(s.x * v[2 * q], i + 1 < d.mx ? s.y * v[2 * q + 1] : 0.0f);
                }
            }
        });
        __syncthreads();
    }
}

// A pass over the nodes and the patch rows, in chunks of a warp: every block takes an
// equal, contiguous share of either, the patch chunks first.  (The patch rows' gathered
// loads keep a warp busy several times as long as a regular chunk; dealt out after the
// regular chunks they all fell to the last few blocks, which the others then waited for:
// 8 us of a 64^3 solve, 18 of a 37^3 one)
template <class Team, class N, class P>
static __device__ __forceinline__ void fd_deal(const Team& team, int nw, int np, N nodes, P rows) {
    const int C = team.ctas(), b = team.rank_of();
    const int n0 = (int)((long long)nw * b / C), n1 = (int)((long long)nw * (b + 1) / C);
    const int p0 = (int)((long long)np * b / C), p1 = (int)((long long)np * (b + 1) / C);
    for (int c = threadIdx.x >> 5; c < n1 - n0 + p1 - p0; c += FD_WARPS) {
        if (c < p1 - p0) rows(p0 + c);
        else nodes(n0 + c - (p1 - p0));
    }
}

// D: w = A z, v gets this thread's partials of r.z and w.z.  A thread takes four nodes of
// a row: with cx, cy, cz the cubes on either side along the axes (1 on a Neumann face)
// and Sx, Sy, Sz, Dxy, Dxz, Dyz the sums over the axis and face-diagonal neighbours, a
// regular row is
//   eps (cx (c0 cy cz h z - h/6 (cz Sy + cy Sz) - h/12 Dyz) - h/6 cy cz Sx
//        - h/12 (cz Dxy + cy Dxz)),
// c0 = 3/4 and the diagonals on even nodes, c0 = 1/2 and none on odd ones.  The patch
// rows are a list of their own, 32 to a warp, before the regular ones (fd_deal): met among
// these they would set the pace of every warp that has some.  z goes through L1: the team's
// last barrier ordered the writers before these reads.
template <class Team>
static __device__ void fd_matvec(const FdArgs& a, const Team& team, int cur, float (&v)[2]) {
    const FdPlan& d = a.d;
    const float *r = d.r[cur], *z = d.z;
    const int ldv = d.ldv, PV = d.PV;
    const int nv = d.mz * PV / 4, nw = (nv + 31) / 32, np = (a.npatch + 31) / 32, lane = threadIdx.x & 31;
    const float h = (float)a.f.m.h, h6 = a.f.m.h6f, h12 = a.f.m.h12f;
    const float ep = (float)a.f.o.eps_plus, ei = (float)a.f.o.eps_minus;
    fd_deal(team, nw, np,
        [&](int c) {
            const int e4 = c * 32 + lane;
            if (e4 >= nv) return;
            const int n = e4 * 4;
            const unsigned kd = __ldg(reinterpret_cast<const unsigned*>(d.kind) + e4);
            const bool ev = !(kd & FK_ODD);      // the first and third node are even, else the second and fourth
            const float* cp = z + n;
            auto row = [&](int o) { return *reinterpret_cast<const float4*>(cp + o); };
            const int so = ev ? -1 : 4;          // the even nodes' fourth column of a neighbouring row
            const float4 v0 = row(0), vym = row(-ldv), vyp = row(ldv), vzm = row(-PV), vzp = row(PV);
            const float4 d0 = row(-ldv - PV), d1 = row(ldv - PV), d2 = row(-ldv + PV), d3 = row(ldv + PV);
            const float xl = cp[-1], xr = cp[4];
            const float sym = cp[so - ldv], syp = cp[so + ldv], szm = cp[so - PV], szp = cp[so + PV];
            const float4 rv = ld4(r + n);
            const float cy = (kd & FK_CY) ? 1.0f : 2.0f, cz = (kd & FK_CZ) ? 1.0f : 2.0f;
            // the even nodes' diagonal sums, first and second
            auto pair = [&](const float4& q, float sc, float& s0, float& s1) {
                const float lft = ev ? sc : q.x, mid = ev ? q.y : q.z, rgt = ev ? q.w : sc;
                s0 += lft + mid;
                s1 += mid + rgt;
            };
            float dxy0 = 0.0f, dxy1 = 0.0f, dxz0 = 0.0f, dxz1 = 0.0f;
            pair(vym, sym, dxy0, dxy1);
            pair(vyp, syp, dxy0, dxy1);
            pair(vzm, szm, dxz0, dxz1);
            pair(vzp, szp, dxz0, dxz1);
            const float dyz0 = ev ? (d0.x + d1.x) + (d2.x + d3.x) : (d0.y + d1.y) + (d2.y + d3.y);
            const float dyz1 = ev ? (d0.z + d1.z) + (d2.z + d3.z) : (d0.w + d1.w) + (d2.w + d3.w);
            const float ed0 = h12 * (cz * dxy0 + cy * dxz0), ed1 = h12 * (cz * dxy1 + cy * dxz1);
            const float zc[4] = {v0.x, v0.y, v0.z, v0.w};
            const float sx[4] = {xl + v0.y, v0.x + v0.z, v0.y + v0.w, v0.z + xr};
            const float sy[4] = {vym.x + vyp.x, vym.y + vyp.y, vym.z + vyp.z, vym.w + vyp.w};
            const float sz[4] = {vzm.x + vzp.x, vzm.y + vzp.y, vzm.z + vzp.z, vzm.w + vzp.w};
            const float rr[4] = {rv.x, rv.y, rv.z, rv.w};
            const float ce = 0.75f * h * cy * cz, co = 0.5f * h * cy * cz;
            float wv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned kq = kd >> (8 * q);
                const bool even = ev == ((q & 1) == 0);
                float t = (even ? ce : co) * zc[q] - h6 * (cz * sy[q] + cy * sz[q]);
                if (even) t -= h12 * (q < 2 ? dyz0 : dyz1);
                float y = ((kq & FK_CX) ? 1.0f : 2.0f) * t - h6 * cy * cz * sx[q];
                if (even) y -= q < 2 ? ed0 : ed1;
                y *= (kq & FK_INNER) ? ei : ep;
                wv[q] = (kq & (FK_PAD | FK_PATCH)) ? 0.0f : y;
                v[1] += wv[q] * zc[q];
                v[0] += (kq & FK_PATCH) ? 0.0f : rr[q] * zc[q];
            }
            if (!(kd & (FK_PATCH * 0x01010101u))) {
                st4(d.w + n, make_float4(wv[0], wv[1], wv[2], wv[3]));
            } else {                             // (a patch row's w is another warp's)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (!((kd >> (8 * q)) & FK_PATCH)) d.w[n + q] = wv[q];
            }
        },
        [&](int c) {
            const int row = c * 32 + lane;
            if (row >= a.npatch) return;
            const int n = __ldg(d.patch + row);
            const float* k = a.f.coeff + (size_t)row * 19;   // (zero where a neighbour is absent, and on the
            const float* cp = z + n;                         // diagonals of an odd node)
            const int off[19] = {0, -1, 1, -ldv, ldv, -PV, PV, -1 - ldv, 1 - ldv, -1 + ldv, 1 + ldv, -1 - PV, 1 - PV,
                                 -1 + PV, 1 + PV, -ldv - PV, ldv - PV, -ldv + PV, ldv + PV};
            float y = 0.0f;
#pragma unroll
            for (int q = 0; q < 19; ++q) y += __ldg(k + q) * cp[off[q]];
            d.w[n] = y;
            v[0] += __ldcg(r + n) * cp[0];
            v[1] += y * cp[0];
        });
}

// the FP64 residual b - A u of every node, in the same form (two nodes of a row per
// lane, so that a warp mostly holds one parity at a time: FP64 issues slowly here):
// r gets it in FP32, x zero; v2 the partials of b.b (first: only then) and r.r
template <class Team>
static __device__ void fd_residual(const FdArgs& a, const Team& team, bool first, double (&v2)[2]) {
    const FdPlan& d = a.d;
    const Mesh& m = a.f.m;
    const double* u = d.u;
    const int ldv = d.ldv, PV = d.PV, lane = threadIdx.x & 31;
    const int nw = (d.mz * PV + 63) / 64, np = (a.npatch + 31) / 32;
    const double h6[2] = {m.h6, 2.0 * m.h6}, h12[2] = {m.h12, 2.0 * m.h12};   // times 1 or 2 cubes
    const double h66 = 4.0 * m.h6;
    auto take = [&](int n, double bn, double rn) {
        d.r[0][n] = (float)rn;
        d.x[n] = 0.0f;
        v2[1] += rn * rn;
        if (first) v2[0] += bn * bn;
    };
    auto node = [&](int n) {
        const int k = n / PV, l = n - k * PV, j = l / ldv;
        return node_id(m, d.x0 + l - j * ldv, d.y0 + j, d.z0 + k);
    };
    fd_deal(team, nw, np,
        [&](int c) {
            const int n0 = c * 64 + 2 * lane;
            if (n0 >= d.mz * PV) return;
            const unsigned kd2 = __ldg(reinterpret_cast<const unsigned short*>(d.kind + n0));
            const long long nn = node(n0);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const unsigned kd = kd2 >> (8 * e);
                if (kd & (FK_PAD | FK_PATCH)) continue;
                const int n = n0 + e;
                const double* cp = u + n;
                const double bn = a.b[nn + e], zc = cp[0];
                const double sx = cp[-1] + cp[1], sy = cp[-ldv] + cp[ldv], sz = cp[-PV] + cp[PV];
                const int iy = (kd & FK_CY) ? 0 : 1, iz = (kd & FK_CZ) ? 0 : 1;
                const double hx = (iy & iz) ? h66 : h6[iy | iz];        // h/6 cy cz
                const double eps = (kd & FK_INNER) ? a.f.o.eps_minus : a.f.o.eps_plus;
                const double cx = (kd & FK_CX) ? 1.0 : 2.0;
                double y;
                if (kd & FK_ODD) {
                    // c0 cy cz h = 3 (h/6) cy cz
                    y = cx * (3.0 * hx * zc - h6[iz] * sy - h6[iy] * sz) - hx * sx;
                } else {
                    const double dxy = (cp[-1 - ldv] + cp[1 - ldv]) + (cp[-1 + ldv] + cp[1 + ldv]);
                    const double dxz = (cp[-1 - PV] + cp[1 - PV]) + (cp[-1 + PV] + cp[1 + PV]);
                    const double dyz = (cp[-ldv - PV] + cp[ldv - PV]) + (cp[-ldv + PV] + cp[ldv + PV]);
                    y = cx * (4.5 * hx * zc - h6[iz] * sy - h6[iy] * sz - h12[0] * dyz) - hx * sx - h12[iz] * dxy -
                        h12[iy] * dxz;
                }
                take(n, bn, bn - eps * y);
            }
        },
        [&](int c) {
            const int row = c * 32 + lane;
            if (row >= a.npatch) return;
            const int n = __ldg(d.patch + row);
            const double* k = a.f.coef + (size_t)row * 19;
            const double* cp = u + n;
            const int off[19] = {0, -1, 1, -ldv, ldv, -PV, PV, -1 - ldv, 1 - ldv, -1 + ldv, 1 + ldv, -1 - PV, 1 - PV,
                                 -1 + PV, 1 + PV, -ldv - PV, ldv - PV, -ldv + PV, ldv + PV};
            double y = 0.0;
#pragma unroll
            for (int q = 0; q < 19; ++q) y += k[q] * cp[off[q]];
            const double bn = a.b[node(n)];
            take(n, bn, bn - y);
        });
}

// the refined PCG of one system, by one team
template <class Team>
static __device__ void fd_pcg(const FdArgs& a, Team& team, uint2* sm) {
    const FdPlan& d = a.d;
    const Mesh& m = a.f.m;
    const int TT = (int)team.size(), t0 = (int)team.t0();
    const FdShare h = fd_share(d, team, sm);
    const double tol2 = a.tol2;
    // An inner solve that reduces the residual 1e-6-fold meets the tolerance after one
    // refinement step, but leaves the FP32 rounding of its whole correction in the
    // smoothest modes.  Between Dirichlet faces that is 5e-7 of the potential (64^3
    // sphere; the Jacobi solver leaves 2e-5).  With Neumann faces the smoothest modes
    // are far softer (7e-4 on the 160 x 160 x 80 crater), so there the context's
    // reduction splits the solve into two refinement steps and the second corrects the
    // first's rounding; a margin of 0.2 at most (one iteration more) leaves 2e-6 there.
    const double inner_red2 = d.deep ? fmin(a.inner_red2, FD_INNER_RED * FD_INNER_RED) : a.inner_red2;
    const double margin2 = d.deep ? a.margin2 : fmin(a.margin2, FD_MARGIN * FD_MARGIN);
    const int maxit = a.maxit;
    int it = 0, outer = 0;
    double bb = 0.0, rr = 0.0;
    bool conv = false, alive = true;
    for (;;) {
        // true residual of u in FP64, rounded to the FP32 inner solve; x = 0
        double v2[2] = {0.0, 0.0}, t2[2];
        fd_residual(a, team, outer == 0, v2);
        if (!(alive = team.template reduce<double, 2>(v2, t2))) break;
        if (outer == 0) bb = t2[0];
        rr = t2[1];
        conv = (bb == 0.0) || (rr <= tol2 * bb);
        if (conv || it >= maxit || outer >= FD_MAX_OUTER) break;
        // inner target: max(margin tol |b|, reduction |r0|) (set_refinement)
        const float rr_stop = (float)fmax(margin2 * tol2 * bb, inner_red2 * rr);
        ++outer;
        int cur = 0;
        float alpha = 0.0f, beta = 0.0f;
        float rr_in[1] = {(float)rr}, gd[2] = {0.0f, 0.0f};   // r.r; r.z and w.z
        bool first = true;
        for (;;) {
            float v1[1] = {0.0f}, t1[1];
            fd_forward(a, h, !first, cur, alpha, beta, v1[0]);
            if (first) {
                if (!(alive = team.sync())) break;
            } else {
                cur ^= 1;
                if (!(alive = team.sum_rr(v1, rr_in, t1))) break;
                rr_in[0] = t1[0];
                if (t1[0] <= rr_stop || it >= maxit) break;
            }
            fd_tridiag(a, team, reinterpret_cast<float2*>(sm));
            if (!(alive = team.sync())) break;
            fd_backward(a, h);
            if (!(alive = team.sync())) break;
            float vg[2] = {0.0f, 0.0f}, tg[2];
            fd_matvec(a, team, cur, vg);
            if (!(alive = team.sum_gd(vg, gd, tg))) break;
            beta = first ? 0.0f : tg[0] / gd[0];
            alpha = tg[0] / (first ? tg[1] : tg[1] - beta * tg[0] / alpha);
            gd[0] = tg[0];
            gd[1] = tg[1];
            ++it;
            // rounding broke the recurrence: restart from the true residual (x as it is)
            if (!(alpha > 0.0f && alpha < 1e30f && fabsf(beta) < 1e30f)) break;
            first = false;
        }
        if (!alive) break;
        for (int n = t0; n < d.mz * d.PV; n += TT) d.u[n] = d.u[n] + (double)__ldcg(d.x + n);
        // the next residual reads the neighbours' new u
        if (!(alive = team.sync())) break;
    }
    for (int n = t0; n < (int)m.nnodes; n += TT) {
        int i, j, k;
        node_ijk(m, n, i, j, k);
        i -= d.x0; j -= d.y0; k -= d.z0;
        const bool in = (unsigned)i < (unsigned)d.mx && (unsigned)j < (unsigned)d.my && (unsigned)k < (unsigned)d.mz;
        a.phi[n] = (!in || bb == 0.0) ? a.g[n] : __ldcg(d.u + k * d.PV + j * d.ldv + i) + a.g[n];
    }
    if (team.leader() && threadIdx.x == 0) {
        PcgState* S = a.S;
        S->bb = bb; S->rr = rr; S->it = it; S->outer_it = outer;
        S->converged = alive && conv;
        S->relres = bb > 0.0 ? sqrt(rr / bb) : 0.0;
        *a.it_total += it;
        *a.outer_total += outer;
    }
}

__global__ void __launch_bounds__(FD_THREADS, 1) k_pcg_fd(const __grid_constant__ FdArgs a) {
    extern __shared__ __align__(16) uint2 fd_dyn[];
    __shared__ ExchShared xs;
    int e = 0;
    FdGrid team(a, e, xs);
    fd_pcg(a, team, fd_dyn);
}

// batched: one system on one cluster of C CTAs (the grid is that cluster)
__global__ void __launch_bounds__(FD_THREADS, 1) k_pcg_fd_cluster(const __grid_constant__ FdArgs a, int C) {
    extern __shared__ __align__(16) uint2 fd_dyn[];
    __shared__ ClusterSlots cs;
    cg::cluster_group cl = cg::this_cluster();
    FdCluster team(cl, C, cs);
    fd_pcg(a, team, fd_dyn);
    cl.sync();   // (no CTA leaves while a peer may still read its shared slots)
}

// ---- set-up -------------------------------------------------------------------------
// permittivity of a node's row relative to the plasma's: its diagonal over the
// regular diagonal of the same node
static __device__ __forceinline__ double fd_eps(const Mesh& m, const double* invdiag, int i, int j, int k) {
    const long long n = node_id(m, i, j, k);
    const int c = ((i > 0) + (i < m.nx)) * ((j > 0) + (j < m.ny)) * ((k > 0) + (k < m.nz));
    return 1.0 / (invdiag[n] * ((double)c * (((i + j + k) & 1) ? 0.5 : 0.75) * m.h));
}
// mean over the free nodes of each plane, one block per plane
__global__ void k_fd_profile(Mesh m, const double* invdiag, FdPlan d, double* prof) {
    __shared__ double sh[32];
    double v[1] = {0.0};
    for (int e = threadIdx.x; e < d.mx * d.my; e += blockDim.x)
        v[0] += fd_eps(m, invdiag, d.x0 + e % d.mx, d.y0 + e / d.mx, d.z0 + (int)blockIdx.x);
    block_sum_f64<1>(v, sh);
    if (threadIdx.x == 0) prof[blockIdx.x] = v[0] / ((double)d.mx * d.my);
}
// the box's scaling and node kinds, and the patch rows' places
__global__ void k_fd_box(Mesh m, const double* invdiag, const int* ntype, FdPlan d, const double* prof, float* s,
                         unsigned char* kind, int* patch) {
    const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (e >= (long long)d.mz * d.PV) return;
    const int k = (int)(e / d.PV), l = (int)(e - (long long)k * d.PV), j = l / d.ldv, i = l - j * d.ldv;
    const int ni = d.x0 + i, nj = d.y0 + j, nk = d.z0 + k;
    unsigned kd = ((ni + nj + nk) & 1) ? FK_ODD : 0;
    float sv = 0.0f;
    if (i >= d.mx || j >= d.my) {
        kd |= FK_PAD;
    } else {
        const int ty = ntype[node_id(m, ni, nj, nk)];
        if (ty == -2) kd |= FK_INNER;
        if (ty >= 0) { kd |= FK_PATCH; patch[ty] = (int)e; }
        if (ni == 0 || ni == m.nx) kd |= FK_CX;
        if (nj == 0 || nj == m.ny) kd |= FK_CY;
        if (nk == 0 || nk == m.nz) kd |= FK_CZ;
        sv = (float)pow(fd_eps(m, invdiag, ni, nj, nk) / sqrt(prof[k]), -0.25);
    }
    kind[e] = (unsigned char)kd;
    s[e] = sv;
}

// eigenvector k (node index j counted from the face) of K v = lambda M v on n
// cells: sines from a Dirichlet end, cosines from a Neumann end, half-integer
// wave numbers where the ends differ; M-orthonormal
struct FdAxis {
    int n, lo, hi;   // cells; 1 where the end is Dirichlet
};
static __device__ __forceinline__ double fd_wave(const FdAxis& x, int k) {
    if (x.lo && x.hi) return (double)(k + 1) / x.n;
    return x.lo == x.hi ? (double)k / x.n : ((double)k + 0.5) / x.n;
}
static __device__ double fd_basis(const FdAxis& x, int j, int k) {
    const int m = x.n + 1 - x.lo - x.hi;
    if (j >= m || k >= m) return 0.0;
    const double c = (x.lo == 0 && x.hi == 0 && (k == 0 || k == x.n)) ? sqrt(1.0 / x.n) : sqrt(2.0 / x.n);
    const double a = fd_wave(x, k) * (double)(j + x.lo);
    return c * (x.lo ? sinpi(a) : cospi(a));
}
static __device__ __forceinline__ double fd_lambda(const FdAxis& x, int k) { return 2.0 - 2.0 * cospi(fd_wave(x, k)); }

// split fragments of a basis matrix, 16 x 16 tiles: rows modes and columns nodes
// (to modes) or the other way round (back)
static __device__ uint4 fd_fragment(const FdAxis& x, bool back, int r, int k, int half) {
    unsigned o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {          // (r, k), (r + 8, k), (r, k + 8), (r + 8, k + 8), two columns each
        const int rr = r + 8 * (q & 1), kk = k + 8 * (q >> 1);
        float v[2];
        for (int e = 0; e < 2; ++e) v[e] = (float)(back ? fd_basis(x, rr, kk + e) : fd_basis(x, kk + e, rr));
        const uint2 s = bf16_split(v[0], v[1]);
        o[q] = half ? s.y : s.x;
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}
__global__ void k_fd_fragments(FdAxis x, int ks, uint4* F, uint4* B) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x, lane = e & 31, half = (e >> 5) & 1, tile = e >> 6;
    if (tile >= ks * ks) return;
    const int r = (tile / ks) * 16 + (lane >> 2), k = (tile % ks) * 16 + 2 * (lane & 3);
    F[e] = fd_fragment(x, false, r, k, half);
    B[e] = fd_fragment(x, true, r, k, half);
}
// inverted pivots of ((lx + ly) Mz + Kz) per mode; mk: [mz] Mz, then [mz] the diagonal of Kz
__global__ void k_fd_pivots(FdAxis x, FdAxis y, FdPlan d, const double* mk, const double* ez, float* inv) {
    const long long col = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (col >= d.PT) return;
    const int a = (int)(col % d.ldT), b = (int)(col / d.ldT);
    const bool in = a < d.mx && b < d.my;
    const double lam = in ? fd_lambda(x, a) + fd_lambda(y, b) : 0.0;
    double v = 0.0;
    for (int k = 0; k < d.mz; ++k) {
        const double e = k > 0 ? ez[k - 1] : 0.0;
        v = 1.0 / (lam * mk[k] + mk[d.mz + k] - e * e * v);
        inv[(size_t)k * d.PT + col] = in ? (float)v : 0.0f;
    }
}
__global__ void k_fd_narrow(int n, const double* in, float* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (float)in[i];
}

void free_fd(Ctx& c) {
    FdPlan& d = c.fd;
    lib_free(c.fd_mem);
    c.fd_mem = nullptr;
    d = FdPlan{};
}

// shared memory of the passes: the planes of a group and their first product's chunks,
// or the tridiagonal runs' ends; then the fragments if they are staged
static size_t fd_pass_smem(const FdPlan& d) {
    const size_t tr = (size_t)d.pb * ((size_t)d.ksy * 16 * d.ldX + (size_t)d.mta * 16 * d.ldY);
    return sizeof(uint2) * ((std::max(tr, (size_t)4 * FD_WARPS * 32) + 1) & ~(size_t)1);
}
static size_t fd_frag_smem(const FdPlan& d) {
    return sizeof(uint4) * 64 * 2 * ((size_t)d.mta * d.ksx + (size_t)d.ksy * d.ksy);
}
static size_t fd_smem(const FdPlan& d) { return fd_pass_smem(d) + (d.stage ? fd_frag_smem(d) : 0); }

// the split of the planes for a team of G blocks: chunks of mta 16-column tiles, pb
// planes of a block at a time, and the two products' tiles over the warps -- the least
// time of a block's rounds, counted in tile products of a warp plus the plane's load,
// among the splits that fit in shared memory (false: none)
static bool fd_split(FdPlan& d, int G, size_t limit) {
    double best = 0.0;
    const int widths[3] = {1, 2, 4};
    auto rounds = [](int m, int n, int w) { return std::ceil((double)m * ((n + w - 1) / w) / FD_WARPS) * (w + 0.7); };
    FdPlan p = d;
    p.stage = 0;
    for (int mta = 1; mta <= std::min(d.ksx, 8); ++mta) {
        p.mta = mta;
        p.nch = (d.ksx + mta - 1) / mta;
        if (p.nch > G) continue;
        const int planes = (d.mz + G / p.nch - 1) / (G / p.nch);   // a block's planes
        for (p.pb = 1; p.pb <= std::min(planes, 4); ++p.pb) {
            if (fd_pass_smem(p) > limit) break;
            double c1 = 0.0, c2 = 0.0;
            for (int w : widths) {
                const double r1 = d.ksx * rounds(mta, 2 * d.ksy * p.pb, w), r2 = d.ksy * rounds(d.ksy, 2 * mta * p.pb, w);
                if (c1 == 0.0 || r1 < c1) { c1 = r1; p.nt1 = w; }
                if (c2 == 0.0 || r2 < c2) { c2 = r2; p.nt2 = w; }
            }
            const double cost =
                std::ceil((double)planes / p.pb) * (c1 + c2 + 10.0 + 1.0 * d.ksx * d.ksy * p.pb);
            if (best == 0.0 || cost < best) { best = cost; d = p; }
        }
    }
    if (best > 0.0 && fd_pass_smem(d) + fd_frag_smem(d) <= limit) d.stage = (int)(fd_pass_smem(d) / sizeof(uint2));
    return best > 0.0;
}

// The plan for the context's mesh, boundaries and operator, in MIXED mode with AUTO,
// once pifepic_solve_field (from FD_MIN_NODES nodes) or a batch has asked for it; not
// where no node is free, where every face is Neumann (P is singular), where a plane
// does not fit in shared memory or beyond FD_MAX_CONTRAST.
cudaError_t plan_pcg_fd(Ctx& c) {
    free_fd(c);
    const Mesh& m = c.mesh;
    if (c.precision != PIFEPIC_MIXED || c.precond != PIFEPIC_PRECOND_AUTO || !c.fd_wanted ||
        m.nnodes < FD_CLUSTER_MIN_NODES)
        return cudaSuccess;
    double lo = std::min(c.obj.eps_plus, c.obj.eps_minus), hi = std::max(c.obj.eps_plus, c.obj.eps_minus);
    if (c.obj.bed) { lo = std::min(lo, c.obj.eps_bed); hi = std::max(hi, c.obj.eps_bed); }
    if (!(hi <= FD_MAX_CONTRAST * lo)) return cudaSuccess;
    int dir[6], any = 0;
    for (int f = 0; f < 6; ++f) any |= dir[f] = c.bc[f].kind == PIFEPIC_BC_DIRICHLET;
    FdPlan d;
    d.x0 = dir[0]; d.y0 = dir[2]; d.z0 = dir[4];
    const int mx = m.NX - dir[0] - dir[1], my = m.NY - dir[2] - dir[3], mz = m.NZ - dir[4] - dir[5];
    if (!any || mx < 1 || my < 1 || mz < 1 || mz > FD_MAX_RUN * FD_WARPS)
        return cudaSuccess;
    d.mx = mx; d.my = my; d.mz = mz;
    d.deep = dir[0] && dir[1] && dir[2] && dir[3] && dir[4] && dir[5];
    d.ksx = (mx + 15) / 16; d.ksy = (my + 15) / 16;
    d.ldX = d.ksx * 8 + 4;                // (pairs; 4 mod 8: a fragment's rows fall into different banks)
    d.ldY = d.ksy * 8 + 4;
    d.ldT = d.ksx * 16;
    d.PT = ((long long)my * d.ldT + 31) / 32 * 32;
    d.ldv = (mx + 1 + 3) / 4 * 4;
    d.PV = (my + 1) * d.ldv;
    int nsm = 0, optin = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c.device);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c.device);
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, k_pcg_fd);
    if (e != cudaSuccess) return e;
    const size_t limit = (size_t)(optin - (int)fa.sharedSizeBytes);
    if ((long long)d.PT * mz > INT32_MAX || ((long long)d.PV + 64) * (mz + 2) > INT32_MAX ||
        !fd_split(d, std::min(nsm, 255), limit))
        return cudaSuccess;
    e = cudaFuncSetAttribute(k_pcg_fd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit);
    if (e != cudaSuccess) return e;
    // one allocation, every array on a 256-byte boundary and zero to begin with
    const size_t LV = (size_t)d.PV * d.mz;                      // box entries (a multiple of 4)
    const size_t guard = ((size_t)d.PV + d.ldv + 4 + 63) / 64 * 64;
    const size_t TN = (size_t)d.PT * d.mz;
    const int ex = 64 * d.ksx * d.ksx, ey = 64 * d.ksy * d.ksy;   // fragments of a basis matrix
    size_t bytes = 0;
    auto room = [&](size_t n) {
        const size_t at = bytes;
        bytes += (n + 255) / 256 * 256;
        return at;
    };
    const size_t o_u = room(sizeof(double) * (LV + 2 * guard)), o_z = room(sizeof(float) * (LV + 2 * guard));
    size_t o_v[7], o_f[4];
    for (size_t& o : o_v) o = room(sizeof(float) * LV);
    const size_t o_s = room(sizeof(float) * LV), o_k = room(LV), o_p = room(sizeof(int) * (c.npatch > 0 ? c.npatch : 1));
    const size_t o_T = room(sizeof(float) * TN), o_i = room(sizeof(float) * TN), o_e = room(sizeof(float) * d.mz);
    for (int q = 0; q < 4; ++q) o_f[q] = room(sizeof(uint4) * (q < 2 ? ex : ey));
    const size_t o_w = room(sizeof(double) * 4 * d.mz);         // profile, then Mz, diag(Kz) and the couplings
    char* mem = nullptr;
    e = lib_malloc(&mem, bytes);
    if (e != cudaSuccess) return e;
    c.fd_mem = mem;
    d.u = (double*)(mem + o_u) + guard;
    d.z = (float*)(mem + o_z) + guard;
    float** vec[7] = {&d.r[0], &d.r[1], &d.q[0], &d.q[1], &d.w, &d.p, &d.x};
    for (int q = 0; q < 7; ++q) *vec[q] = (float*)(mem + o_v[q]);
    float *s = (float*)(mem + o_s), *inv = (float*)(mem + o_i), *ez = (float*)(mem + o_e);
    unsigned char* kind = (unsigned char*)(mem + o_k);
    int* patch = (int*)(mem + o_p);
    uint4* frag[4];
    for (int q = 0; q < 4; ++q) frag[q] = (uint4*)(mem + o_f[q]);
    double* work = (double*)(mem + o_w);
    d.T = (float*)(mem + o_T);
    d.s = s; d.kind = kind; d.patch = patch; d.inv = inv; d.ez = ez;
    d.fxF = frag[0]; d.fxI = frag[1]; d.fyF = frag[2]; d.fyI = frag[3];
    c.fd = d;
    e = cudaMemsetAsync(mem, 0, bytes, c.stream);
    std::vector<double> prof(d.mz), mk(3 * d.mz);
    if (e == cudaSuccess) {
        k_fd_profile<<<d.mz, 256, 0, c.stream>>>(m, c.invdiag, d, work);
        e = scopy(c.stream, prof.data(), work, sizeof(double) * d.mz, cudaMemcpyDeviceToHost);
    }
    if (e == cudaSuccess) {
        // cell permittivities of P: the square root of the profile, constant beyond the free planes
        auto cell = [&](int K) {          // between node planes K and K + 1
            const double lo = prof[std::max(K - d.z0, 0)], hi = prof[std::min(K + 1 - d.z0, d.mz - 1)];
            return std::sqrt(0.5 * (lo + hi));
        };
        for (int k = 0; k < d.mz; ++k) {
            const int K = d.z0 + k;
            const double lo = K > 0 ? cell(K - 1) : 0.0, hi = K < m.nz ? cell(K) : 0.0;
            mk[k] = 0.5 * (lo + hi);
            mk[d.mz + k] = lo + hi;
            mk[2 * d.mz + k] = hi;
        }
        k_fd_box<<<(unsigned)((LV + 255) / 256), 256, 0, c.stream>>>(m, c.invdiag, c.ntype, d, work, s, kind, patch);
        e = scopy(c.stream, work + d.mz, mk.data(), sizeof(double) * 3 * d.mz, cudaMemcpyHostToDevice);
    }
    if (e == cudaSuccess) {
        const FdAxis ax{m.nx, dir[0], dir[1]}, ay{m.ny, dir[2], dir[3]};
        k_fd_fragments<<<(ex + 255) / 256, 256, 0, c.stream>>>(ax, d.ksx, frag[0], frag[1]);
        k_fd_fragments<<<(ey + 255) / 256, 256, 0, c.stream>>>(ay, d.ksy, frag[2], frag[3]);
        k_fd_pivots<<<(unsigned)((d.PT + 127) / 128), 128, 0, c.stream>>>(ax, ay, d, work + d.mz, work + 3 * d.mz, inv);
        k_fd_narrow<<<(d.mz + 255) / 256, 256, 0, c.stream>>>(d.mz, work + 3 * d.mz, ez);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(c.stream);
    }
    if (e != cudaSuccess) free_fd(c);
    return e;
}

static FdArgs fd_args(Ctx& c) {
    FdArgs a;
    a.f.m = c.mesh; a.f.o = c.obj; a.f.ntype = c.ntype; a.f.coef = c.patch_coef; a.f.coeff = c.patch_coeff;
    a.f.invdiag = c.invdiag; a.f.invdiagf = c.invdiagf;
    a.b = c.b; a.g = c.gdir; a.phi = c.phi;
    a.d = c.fd;
    a.npatch = (int)c.npatch;
    a.tol2 = c.tol * c.tol;
    a.inner_red2 = c.inner_red * c.inner_red;
    a.margin2 = c.inner_margin * c.inner_margin;
    a.maxit = c.maxit;
    a.val = c.coop_partial;
    a.arrivals = c.bar64 + BAR64_FD;
    a.fx = c.bar64 + BAR64_FD + FX_LINE;
    a.hold = (const int*)(c.scal + 45);
    a.S = (PcgState*)c.scal;
    a.it_total = (long long*)(c.scal + 40);
    a.outer_total = (long long*)(c.scal + 41);
    a.err = c.err_word;
    return a;
}

// the cluster kernel's launch for the plan d, split for a team of C CTAs (1..16);
// ok: the device runs it (a split exists and the cluster fits)
static cudaError_t fd_cluster_config(const Ctx& c, FdPlan& d, int C, cudaLaunchConfig_t& cfg,
                                     cudaLaunchAttribute& attr, bool& ok) {
    void* kern = (void*)k_pcg_fd_cluster;
    ok = false;
    int optin = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c.device);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    // (the whole opt-in budget for every member, as the other cluster solvers)
    const int limit = optin - (int)fa.sharedSizeBytes;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
    if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess || !fd_split(d, C, (size_t)limit)) return e;
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3(FD_THREADS);
    cfg.dynamicSmemBytes = fd_smem(d);
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)C;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    e = cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg);
    ok = e == cudaSuccess && nclusters >= 1;
    return e;
}

// The CTAs of a member's cluster (0: none can run it): the smallest power of two
// that keeps each CTA at or under cta_nodes nodes and whose CTAs take a plane's
// columns between them (a long x axis has more 16-column tiles than few CTAs hold).
int fd_cluster_size(const Ctx& c, long long cta_nodes) {
    for (int C = 1; C <= 16; C *= 2) {
        if (C < 16 && (c.mesh.nnodes + C - 1) / C > cta_nodes) continue;
        FdPlan d = c.fd;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr = {};
        bool ok;
        if (fd_cluster_config(c, d, C, cfg, attr, ok) != cudaSuccess) cudaGetLastError();
        else if (ok) return C;
    }
    return 0;
}

// a batched solve: the system of c on one cluster of C CTAs (fd_cluster_size)
cudaError_t launch_pcg_fd_cluster(Ctx& c, int C, cudaStream_t st) {
    FdArgs a = fd_args(c);
    // A batch's clusters solve in one refinement step, as the Jacobi clusters do, with Neumann
    // faces too: on members of 15,000 to 50,000 nodes, craters and layers with five Neumann
    // faces among them, the potential is then 2e-7 to 1.5e-6 from a tight solve's, where the
    // Jacobi clusters leave 4e-7 to 4e-6 (and 2e-3 where their 150 iterations are too few).
    a.d.deep = true;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr = {};
    bool ok;
    cudaError_t e = fd_cluster_config(c, a.d, C, cfg, attr, ok);
    if (e != cudaSuccess) return e;
    if (!ok) return cudaErrorInvalidConfiguration;
    cfg.stream = st;
    void* args[] = {(void*)&a, (void*)&C};
    return cudaLaunchKernelExC(&cfg, (void*)k_pcg_fd_cluster, args);
}

cudaError_t launch_pcg_fd(Ctx& c, cudaStream_t st) {
    FdArgs a = fd_args(c);
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c.device);
    void* args[] = {&a};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min(nsm, 255));   // the fixed-point exchange counts arrivals in 8 bits
    cfg.blockDim = dim3(FD_THREADS);
    cfg.dynamicSmemBytes = fd_smem(c.fd);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, (void*)k_pcg_fd, args);
}

}  // namespace pf
