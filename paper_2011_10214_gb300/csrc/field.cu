// IFE field solve on the GPU: right-hand side with the flux-jump term, the solve
// graph around the persistent PCG kernels (pcg_coop.cu, pcg_mg.cu, pcg_fd.cu),
// node field, and the statistics of a call.
//
// Sec. 2.1 (Eqs. 2.1-2.5): weak form a(phi, v) = (rho, v) - int_Gamma q v; the
// non-homogeneous IFE solution is phi_h = u_h + phi_J (phi_J the element-wise
// jump function) with a_h(u_h, psi_i) = F_i - int_Gamma q psi_i - a_h(phi_J,
// psi_i), i.e. F_i + sum_T q_T c_{T,i} (c the unit-jump load of interface tet
// T).  Sec. 2.5: the matrix solve is a PCG iteration stopped on the relative
// residual (Sec. 3.2, Sec. 4, Sec. 5.2.2 give tolerance 1e-6 and caps 60/150).
// Preconditioners (unstated in the paper): pcg_coop.cu, pcg_mg.cu and pcg_fd.cu.
//
// The whole solve of a step is one CUDA graph: q_T, RHS and start vector, one
// persistent PCG kernel, node field.  The iteration count and convergence test
// live on the device; no host round trip.
#include <math.h>
#include <stdio.h>
#include <atomic>

#include "internal.h"
#include "field_common.cuh"

namespace pf {

__constant__ TetTables cTf;
// Interior-regular nodes (all eight cubes present, none holding an interface
// tet): every tet around the node lies on one side, so the node field is one
// fixed 27-point stencil per node parity P, cFold[P][3 nb + d] with
// nb = (dx + 1) + 3 (dy + 1) + 9 (dz + 1): minus the sum over the node's tets of
// vol_t grad_t (h = 1) at neighbour nb, over the sum of vol_t; E = cFold phi / h.
__constant__ float cFold[2][81];

// ---- right-hand side ----------------------------------------------------------
// the surface charge density of each interface tet's object, from its cut cell
__global__ void k_qtets(long long nit, const int* it_acc, RhsArgs a, const double* area, double* qT) {
    long long T = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (T >= nit) return;
    const int c = it_acc[T];
    double q = 0.0;
    if (c >= 0) {
        double Q = 0.0;
        int ns = *a.nspec;
        for (int s = 0; s < ns; ++s) Q = Q + a.coefs[s] * (double)(long long)a.surf[(long long)s * a.ncut + c];
        q = -(Q / area[c]);
    }
    qT[T] = q;
}

// the flux-jump terms of a node's right-hand side (the node rows of the set-up)
struct FluxRows {
    const int* row;
    const int* qoff;
    const int4* q;
    const double* qc;
};

// The solve's start vector: the last potential, or once two earlier solves exist
// its linear extrapolation 2 phi_{n-1} - phi_{n-2} (particles move the charge
// smoothly from step to step, so this start is closer), less the Dirichlet
// values; phi_prev <- phi.  The solve still stops on the same relative residual.
struct StartArgs {
    const double* phi;
    double* phi_prev;
    const double* g;
    double* u;                // null: the start goes into the box of the fast-diagonalisation solve
    const long long* hist;    // solves before this one (3: three or more; counted by the node field's kernel)
    FdPlan d;
};
static __device__ __forceinline__ void start_vector(const StartArgs& a, const Mesh& m, long long n, bool dirichlet) {
    const double p = a.phi[n];
    const double start = *a.hist >= 2 ? 2.0 * p - a.phi_prev[n] : p;
    if (a.u) {
        a.u[n] = dirichlet ? 0.0 : start - a.g[n];
    } else {
        int i, j, k;
        node_ijk(m, n, i, j, k);
        i -= a.d.x0; j -= a.d.y0; k -= a.d.z0;
        if ((unsigned)i < (unsigned)a.d.mx && (unsigned)j < (unsigned)a.d.my && (unsigned)k < (unsigned)a.d.mz)
            a.d.u[k * a.d.PV + j * a.d.ldv + i] = start - a.g[n];
    }
    a.phi_prev[n] = p;
}

// right-hand side, and the start vector in the same pass (START)
template <bool START>
__global__ void k_rhs(FieldArgs f, RhsArgs a, FluxRows fr, const double* qT, const double* lift, double* b,
                      const double* Fext, const __grid_constant__ StartArgs start) {
    const Mesh& m = f.m;
    long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (n >= m.nnodes) return;
    int ty = f.ntype[n];
    if (START) start_vector(start, m, n, ty == -3);
    if (ty == -3) { b[n] = 0.0; return; }
    double F = 0.0;
    if (Fext) {
        F = Fext[n];
    } else {
        int ns = *a.nspec;
        for (int s = 0; s < ns; ++s)
            F = F + (a.coefs[s] * 2.3283064365386963e-10) * (double)(long long)a.W[(long long)s * m.nnodes + n];
    }
    if (ty >= 0 && qT) {   // touches interface tets: flux-jump load (none when qT is NULL)
        const int r = fr.row[n];
        if (r >= 0) {
            const int e1 = fr.qoff[r + 1];
            for (int e = fr.qoff[r]; e < e1; ++e) F += qT[fr.q[e].x] * fr.qc[e];
        }
    }
    b[n] = F - lift[n];
}

// one more solve done (k_node_E and k_node_E_f: the last kernel of every solve)
static __device__ __forceinline__ void count_solve(long long* hist) {
    if (hist && *hist < 3) *hist += 1;
}

// ---- PCG kernels ------------------------------------------------------------------
__global__ void k_matvec(FieldArgs f, const double* x, double* y) {
    long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (n >= f.m.nnodes) return;
    int i, j, k;
    node_ijk(f.m, n, i, j, k);
    y[n] = apply_row<double>(f, n, i, j, k, x, f.coef);
}

// phi = u + g; a zero right-hand side has the lift alone as its solution
__global__ void k_phi_from_u(long long N, const double* u, const double* g, double* phi, const PcgState* S) {
    long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (n < N) phi[n] = S->bb == 0.0 ? g[n] : u[n] + g[n];
}
// ---- node field ---------------------------------------------------------------------
// Minus the volume-weighted mean of the element gradients around a node, the
// plasma-side pieces if there are any.  A block takes 4 x 4 x 4 nodes: first each
// tet of its 5 x 5 x 5 cells once, into shared memory (its volume times gradient
// and its volume, plasma side and whole), then each node's eight sums over its 8
// or 32 tets, in cell order, one sum per thread (a warp takes nodes of one parity,
// which have the same tets).  FP64-bound: about 310 operations a node, where a
// thread per node spent 770 on its 20 tets and the interface's nodes in turn
// made one thread the tail.  16^3 cells: 107 -> 23 us, 40^3: 219 -> 75.
constexpr int N64_T = 4, N64_C = N64_T + 1, N64_TETS = N64_C * N64_C * N64_C * 5, N64_GRAD = 13;
__global__ void __launch_bounds__(256) k_node_E(FieldArgs f, const double* L, const unsigned char* imask, const int* ibase,
                                                const double* it_data, const double* qT, const double* phi, double4* E,
                                                float4* Ef, long long* hist) {
    enum { APL = 0, VPL = 3, AAL = 4, VAL = 7 };
    __shared__ double ct[8][N64_TETS];
    __shared__ double res[8][N64_T * N64_T * N64_T];
    __shared__ double grad[2 * 5 * N64_GRAD], vol[5], s_ih;
    __shared__ int vert[2 * 5 * 4], has[2 * 8];   // has: the tets of a cell of parity p at its corner c8, as bits
    const Mesh& m = f.m;
    const int tid = threadIdx.x;
    const int i0 = blockIdx.x * N64_T, j0 = blockIdx.y * N64_T, k0 = blockIdx.z * N64_T;
    if (tid == 0 && i0 + j0 + k0 == 0) count_solve(hist);
    if (tid < 120) grad[(tid / 12) * N64_GRAD + tid % 12] = (&cTf.grad[0][0][0][0])[tid];
    else if (tid >= 128 && tid < 133) vol[tid - 128] = cTf.vol[tid - 128];
    else if (tid >= 160 && tid < 200) vert[tid - 160] = (&cTf.vert[0][0][0])[tid - 160];
    else if (tid >= 224 && tid < 240) {
        int bits = 0;
        for (int t = 0; t < 5; ++t)
            for (int v = 0; v < 4; ++v)
                if (cTf.vert[(tid - 224) >> 3][t][v] == (tid & 7)) bits |= 1 << t;
        has[tid - 224] = bits;
    } else if (tid == 255) {
        s_ih = 1.0 / m.h;   // (once: an FP64 division is some ten instructions)
    }
    __syncthreads();
    const double ih = s_ih, V3 = m.h * m.h * m.h;
    for (int q = tid; q < N64_TETS; q += 256) {
        const int t = q % 5, cell = q / 5;
        const int ci = i0 - 1 + cell % N64_C, cj = j0 - 1 + cell / N64_C % N64_C, ck = k0 - 1 + cell / (N64_C * N64_C);
        if (ci < 0 || cj < 0 || ck < 0 || ci >= m.nx || cj >= m.ny || ck >= m.nz) continue;
        const long long id = cell_id(m, ci, cj, ck);
        const unsigned mk = imask[id];
        const int tet = ((ci + cj + ck) & 1) * 5 + t;
        double ph[4];
        long long nd0 = 0;
        for (int v = 0; v < 4; ++v) {
            int av, bv, cv; loff(vert[tet * 4 + v], av, bv, cv);
            const long long nd = node_id(m, ci + av, cj + bv, ck + cv);
            if (v == 0) nd0 = nd;
            ph[v] = phi[nd];
        }
        double o[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if ((mk >> t) & 1) {
            const int T = ibase[id] + __popc(mk & ((1u << t) - 1));
            const double* rec = it_data + (long long)T * IT_STRIDE;
            const double qt = qT[T], vp = rec[IT_VOLP], vm = rec[IT_VOLM];
            // the + piece is plasma on the object's surface only (not on the bedrock plane)
            const bool plasma = vp > 0.0 && rec[IT_KIND] == 0.0;
            for (int d = 0; d < 3; ++d) {
                const double gp = ph[0] * rec[IT_GP + d] + ph[1] * rec[IT_GP + 3 + d] + ph[2] * rec[IT_GP + 6 + d] +
                                  ph[3] * rec[IT_GP + 9 + d] + qt * rec[IT_GP + 12 + d];
                const double gm = ph[0] * rec[IT_GM + d] + ph[1] * rec[IT_GM + 3 + d] + ph[2] * rec[IT_GM + 6 + d] +
                                  ph[3] * rec[IT_GM + 9 + d] + qt * rec[IT_GM + 12 + d];
                if (plasma) o[APL + d] = vp * gp;
                o[AAL + d] = vp * gp + vm * gm;
            }
            if (plasma) o[VPL] = vp;
            o[VAL] = vp + vm;
        } else {
            const double* gr = grad + tet * N64_GRAD;
            const double V = vol[t] * V3;
            const bool plasma = L[nd0] >= 0.0;
            for (int d = 0; d < 3; ++d) {
                const double g = (ph[0] * gr[d] + ph[1] * gr[3 + d] + ph[2] * gr[6 + d] + ph[3] * gr[9 + d]) * ih;
                o[AAL + d] = V * g;
                if (plasma) o[APL + d] = V * g;
            }
            if (plasma) o[VPL] = V;
            o[VAL] = V;
        }
#pragma unroll
        for (int d = 0; d < 8; ++d) ct[d][q] = o[d];
    }
    __syncthreads();
    for (int half = 0; half < 2; ++half) {
        const int lane = tid & 31, odd = (tid >> 5) & 1, d = 4 * half + (tid >> 6);   // (a warp: one sum of the 32 nodes of a parity)
        const int z = lane >> 3, y = (lane >> 1) & 3, x = 2 * (lane & 1) + ((odd + y + z + i0 + j0 + k0) & 1);
        const int i = i0 + x, j = j0 + y, k = k0 + z;
        double sum = 0.0;
        // (the sums over all pieces only where there is no plasma)
        if (i <= m.nx && j <= m.ny && k <= m.nz && !(half && res[VPL][x + N64_T * (y + N64_T * z)] > 0.0))
            for (int c8 = 0; c8 < 8; ++c8) {
                int a, b, c; loff(c8, a, b, c);
                const int ci = i - a, cj = j - b, ck = k - c;
                if (ci < 0 || cj < 0 || ck < 0 || ci >= m.nx || cj >= m.ny || ck >= m.nz) continue;
                const double* tets = ct[d] + 5 * ((x + 1 - a) + N64_C * ((y + 1 - b) + N64_C * (z + 1 - c)));
                const int bits = has[((ci + cj + ck) & 1) * 8 + c8];
                for (int t = 0; t < 5; ++t)
                    if ((bits >> t) & 1) sum += tets[t];
            }
        res[d][x + N64_T * (y + N64_T * z)] = sum;
        __syncthreads();
    }
    if (tid >= N64_T * N64_T * N64_T) return;
    const int i = i0 + tid % N64_T, j = j0 + tid / N64_T % N64_T, k = k0 + tid / (N64_T * N64_T);
    if (i > m.nx || j > m.ny || k > m.nz) return;
    const bool plasma = res[VPL][tid] > 0.0;
    const int g = plasma ? APL : AAL;
    const double w = res[plasma ? VPL : VAL][tid];
    double4 e;
    e.x = -res[g][tid] / w; e.y = -res[g + 1][tid] / w; e.z = -res[g + 2][tid] / w;
    e.w = 0.0;
    const long long n = node_id(m, i, j, k);
    E[n] = e;
    if (Ef) Ef[n] = make_float4((float)e.x, (float)e.y, (float)e.z, 0.0f);
}

static void launch_node_E(const FieldArgs& f, const Ctx& c, float4* Ef, long long* hist, cudaStream_t st) {
    const Mesh& m = c.mesh;
    const dim3 grid((m.NX + N64_T - 1) / N64_T, (m.NY + N64_T - 1) / N64_T, (m.NZ + N64_T - 1) / N64_T);
    k_node_E<<<grid, 256, 0, st>>>(f, c.Lnode, c.imask, c.ibase, c.it_data, c.qT, c.phi, c.E, Ef, hist);
}

// Node field in FP32 (MIXED steps; the push reads only this copy).  Same
// reading as k_node_E: minus the volume-weighted mean of the element
// gradients around the node, plasma-side pieces preferred.  A block covers a
// 32 x 4 x 2 brick of nodes and stages phi of the brick and a one-node halo
// (34 x 6 x 4) in shared memory, converted to FP32 once.  An interior-regular
// node applies its parity's 27-point stencil (cFold); any other node its row of
// the set-up (27 x 3 coefficients and the q_T terms of its interface tets).
constexpr int NE_BX = 32, NE_BY = 4, NE_BZ = 2;
constexpr int NE_TX = NE_BX + 2, NE_TY = NE_BY + 2, NE_TZ = NE_BZ + 2;
constexpr int NE_FOLD = 97;   // the parity tables' stride in shared memory (not a multiple of the 32 banks)
__global__ void __launch_bounds__(NE_BX * NE_BY * NE_BZ) k_node_E_f(Mesh m, const int* row, long long R,
                                                                    const float* coef, const int* qoff,
                                                                    const int4* qent, const double* qT,
                                                                    const double* phi, float4* Ef, long long* hist) {
    __shared__ float ph[NE_TX * NE_TY * NE_TZ];
    __shared__ float sF[2 * NE_FOLD];
    const int i0 = blockIdx.x * NE_BX, j0 = blockIdx.y * NE_BY, k0 = blockIdx.z * NE_BZ;
    const int tid = threadIdx.x + NE_BX * (threadIdx.y + NE_BY * threadIdx.z);
    const int i = i0 + threadIdx.x, j = j0 + threadIdx.y, k = k0 + threadIdx.z;
    if (tid == 0 && i0 + j0 + k0 == 0) count_solve(hist);
    const bool mine = i < m.NX && j < m.NY && k < m.NZ;
    const long long n = mine ? node_id(m, i, j, k) : 0;
    const int r = mine ? row[n] : -1;
    for (int q = tid; q < 2 * 81; q += NE_BX * NE_BY * NE_BZ) sF[(q / 81) * NE_FOLD + q % 81] = (&cFold[0][0])[q];
    for (int q = tid; q < NE_TX * NE_TY * NE_TZ; q += NE_BX * NE_BY * NE_BZ) {
        const int gi = i0 - 1 + q % NE_TX, gj = j0 - 1 + (q / NE_TX) % NE_TY, gk = k0 - 1 + q / (NE_TX * NE_TY);
        const bool in = gi >= 0 && gj >= 0 && gk >= 0 && gi < m.NX && gj < m.NY && gk < m.NZ;
        ph[q] = in ? (float)phi[node_id(m, gi, gj, gk)] : 0.0f;
    }
    __syncthreads();
    if (!mine) return;
    // the node in the staged brick; neighbour nb at ph[c + off(nb)]
    const float* c = ph + (threadIdx.x + 1) + NE_TX * ((threadIdx.y + 1) + NE_TY * (threadIdx.z + 1));
    float e0 = 0.f, e1 = 0.f, e2 = 0.f;
    if (r < 0) {
        const float* F = sF + ((i + j + k) & 1) * NE_FOLD;
#pragma unroll
        for (int nb = 0; nb < 27; ++nb) {
            const float f = c[(nb % 3 - 1) + NE_TX * ((nb / 3 % 3 - 1) + NE_TY * (nb / 9 - 1))];
            e0 += F[3 * nb] * f;
            e1 += F[3 * nb + 1] * f;
            e2 += F[3 * nb + 2] * f;
        }
        const float ih = 1.0f / (float)m.h;
        e0 *= ih; e1 *= ih; e2 *= ih;
    } else {
        const float* cf = coef + r;
#pragma unroll
        for (int nb = 0; nb < 27; ++nb) {
            const float f = c[(nb % 3 - 1) + NE_TX * ((nb / 3 % 3 - 1) + NE_TY * (nb / 9 - 1))];
            e0 += cf[(3 * nb) * R] * f;
            e1 += cf[(3 * nb + 1) * R] * f;
            e2 += cf[(3 * nb + 2) * R] * f;
        }
        const int q1 = qoff[r + 1];
        for (int q = qoff[r]; q < q1; ++q) {
            const int4 w = qent[q];
            const float qt = (float)qT[w.x];
            e0 += __int_as_float(w.y) * qt;
            e1 += __int_as_float(w.z) * qt;
            e2 += __int_as_float(w.w) * qt;
        }
    }
    Ef[n] = make_float4(e0, e1, e2, 0.f);
}

static void launch_node_E_f(const Ctx& c, long long* hist, cudaStream_t st) {
    const Mesh& m = c.mesh;
    dim3 grid((m.NX + NE_BX - 1) / NE_BX, (m.NY + NE_BY - 1) / NE_BY, (m.NZ + NE_BZ - 1) / NE_BZ);
    k_node_E_f<<<grid, dim3(NE_BX, NE_BY, NE_BZ), 0, st>>>(m, c.ne_row, c.ne_nrows, c.ne_coef, c.ne_qoff, c.ne_q,
                                                          c.qT, c.phi, c.Ef, hist);
}


// ------------------------------------------------------------------------------------
static unsigned nb(long long n) { return (unsigned)((n + 255) / 256); }
// device count of solves (PCG start extrapolation), scalar slot 43
static long long* solve_hist(Ctx& c) { return (long long*)(c.scal + 43); }

// one node per thread: 256-thread blocks, or 64-thread ones for a mesh whose
// 256-thread grid would leave most SMs idle (these kernels are FP64-bound)
static int node_threads(long long N) { return N < 152LL * 256 ? 64 : 256; }
static unsigned node_blocks(long long N) {
    const int t = node_threads(N);
    return (unsigned)((N + t - 1) / t);
}

static FieldArgs fargs(Ctx& c) {
    FieldArgs f;
    f.m = c.mesh; f.o = c.obj; f.ntype = c.ntype; f.coef = c.patch_coef; f.coeff = c.patch_coeff;
    f.invdiag = c.invdiag; f.invdiagf = c.invdiagf;
    return f;
}

// device scratch layout in c.scal: [0..15] PcgState, [16..23] species coefs,
// [24] nspec (as int), [32..] diag outputs
static PcgState* pcg_state(Ctx& c) { return (PcgState*)c.scal; }
static double* coefs_dev(Ctx& c) { return c.scal + 16; }
static int* nspec_dev(Ctx& c) { return (int*)(c.scal + 24); }

static RhsArgs rargs(Ctx& c) {
    RhsArgs a;
    a.W = c.Wall;
    a.surf = c.surfall;
    a.coefs = coefs_dev(c);
    a.nspec = nspec_dev(c);
    a.ncut = c.ncut;
    return a;
}

static FluxRows flux_rows(const Ctx& c) { return FluxRows{c.ne_row, c.ne_qoff, c.ne_q, c.ne_qc}; }

cudaError_t launch_field_lift(Ctx& c) {
    FieldArgs f = fargs(c);
    k_matvec<<<nb(c.mesh.nnodes), 256, 0, c.stream>>>(f, c.gdir, c.lift);
    return cudaGetLastError();
}

cudaError_t launch_pcg_coop(Ctx& c, cudaStream_t st);   // pcg_coop.cu

// q_T, RHS, warm start, then the persistent PCG and the node field
// hybrid grid: the PIC nodes are the IFE nodes (r i, r j, r k); the push reads
// the node field there
__global__ void k_E_to_pic(Mesh pm, Mesh fm, int r, const double4* E, const float4* Ef, double4* Ep, float4* Efp,
                           int both) {
    long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (n >= pm.nnodes) return;
    int i = (int)(n % pm.NX), j = (int)((n / pm.NX) % pm.NY), k = (int)(n / ((long long)pm.NX * pm.NY));
    long long f = node_id(fm, r * i, r * j, r * k);
    Efp[n] = Ef[f];
    if (both) Ep[n] = E[f];
}

cudaError_t launch_E_to_pic(const Ctx& c, cudaStream_t st, bool both) {
    if (c.refine == 1) return cudaSuccess;
    k_E_to_pic<<<nb(c.pmesh.nnodes), 256, 0, st>>>(c.pmesh, c.mesh, c.refine, c.E, c.Ef, c.Ep, c.Efp, both ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t plan_pcg_fd(Ctx& c);                      // pcg_fd.cu
cudaError_t launch_pcg_fd(Ctx& c, cudaStream_t st);
// q_T, right-hand side and start vector (where the solver keeps it)
static cudaError_t launch_rhs(Ctx& c, cudaStream_t st, bool fd, const double* Fext) {
    const long long N = c.mesh.nnodes;
    const RhsArgs a = rargs(c);
    if (!Fext && c.nit > 0) k_qtets<<<nb(c.nit), 256, 0, st>>>(c.nit, c.it_acc, a, c.cut_area, c.qT);
    const StartArgs start{c.phi, c.phi_prev, c.gdir, fd ? nullptr : c.u, solve_hist(c), c.fd};
    k_rhs<true><<<node_blocks(N), node_threads(N), 0, st>>>(fargs(c), a, flux_rows(c), c.qT, c.lift, c.b, Fext, start);
    return cudaGetLastError();
}

static cudaError_t solve_sequence(Ctx& c, cudaStream_t st, const double* Fext) {
    FieldArgs f = fargs(c);
    const bool fd = Fext && c.fd.mx > 0 && c.mesh.nnodes >= FD_MIN_NODES;   // (the steps: Jacobi or multigrid)
    cudaError_t e = launch_rhs(c, st, fd, Fext);
    if (e != cudaSuccess) return e;
    e = fd ? launch_pcg_fd(c, st) : launch_pcg_coop(c, st);
    if (e != cudaSuccess) return e;
    if (c.precision == PIFEPIC_MIXED) launch_node_E_f(c, solve_hist(c), st);
    else launch_node_E(f, c, c.Ef, solve_hist(c), st);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_E_to_pic(c, st, c.precision != PIFEPIC_MIXED);
}

// the solve's pieces around the PCG, for the batched step (batch.cu); fd: the
// member's solve is the fast-diagonalisation one
cudaError_t launch_solve_prefix(Ctx& c, cudaStream_t st, bool fd) { return launch_rhs(c, st, fd, nullptr); }
cudaError_t launch_solve_suffix(Ctx& c, cudaStream_t st) {
    FieldArgs f = fargs(c);
    if (c.precision == PIFEPIC_MIXED) launch_node_E_f(c, solve_hist(c), st);
    else launch_node_E(f, c, c.Ef, solve_hist(c), st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_E_to_pic(c, st, c.precision != PIFEPIC_MIXED);
}

// kernels launched per solve
int solve_graph_fixed_kernels(const Ctx& c) { return (c.nit > 0) + 3 + (c.refine > 1); }

// The solve as one CUDA graph (both precisions): q_T -> RHS -> warm start ->
// persistent PCG -> node field
cudaError_t build_pcg_graph(Ctx& c) {
    plan_pcg(c);
    if (c.pcg_exec) { cudaGraphExecDestroy(c.pcg_exec); c.pcg_exec = nullptr; }
    if (c.pcg_graph) { cudaGraphDestroy(c.pcg_graph); c.pcg_graph = nullptr; }
    cudaStream_t cs;
    cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    cudaGraph_t g = nullptr;
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        cudaError_t e2 = solve_sequence(c, cs, nullptr);
        e = cudaStreamEndCapture(cs, &g);
        if (e == cudaSuccess) e = e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&c.pcg_exec, g, 0);
    if (e == cudaSuccess) c.pcg_graph = g;
    else if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cs);
    return e;
}

// the solver's limits on the device: sent when they change (every solve writes the
// rest of the state, and a copy per solve was 3 us of a step)
static cudaError_t set_pcg_state(Ctx& c) {
    const double lim[4] = {c.tol, (double)c.maxit, c.inner_red, c.inner_margin};
    if (c.limits_sent && memcmp(lim, c.limits, sizeof(lim)) == 0) return cudaSuccess;
    memcpy(c.limits, lim, sizeof(lim));
    c.limits_sent = true;
    PcgState h = {};
    h.tol2 = c.tol * c.tol;
    h.maxit = c.maxit;
    h.inner_red2 = c.inner_red * c.inner_red;
    h.margin2 = c.inner_margin * c.inner_margin;
    cudaError_t e = cudaMemcpyAsync(c.scal, &h, sizeof(PcgState), cudaMemcpyHostToDevice, c.stream);
    if (e != cudaSuccess) c.limits_sent = false;
    return e;
}

cudaError_t launch_pcg(Ctx& c) {
    cudaError_t e = set_pcg_state(c);
    if (e != cudaSuccess) return e;
    return cudaGraphLaunch(c.pcg_exec, c.stream);
}


// standalone solve with an external node load (solver parity)
cudaError_t launch_solve_external(Ctx& c, const double* Fdev, int* iters, double* relres) {
    if (!c.fd_wanted && c.mesh.nnodes >= FD_MIN_NODES) {
        c.fd_wanted = true;
        if (plan_pcg_fd(c) != cudaSuccess) cudaGetLastError();   // (no plan: the context's own solver)
    }
    cudaError_t e = set_pcg_state(c);
    if (e == cudaSuccess) e = solve_sequence(c, c.stream, Fdev);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c.stream);
    if (e != cudaSuccess) return e;
    PcgState hs;
    e = scopy(c.stream, &hs, pcg_state(c), sizeof(PcgState), cudaMemcpyDeviceToHost);
    if (iters) *iters = hs.it;
    if (relres) *relres = hs.relres;
    c.last_iters = hs.it; c.last_relres = hs.relres; c.last_conv = hs.converged;
    return e;
}

// ---- statistics of a call -------------------------------------------------------
constexpr int ST_THREADS = 256, ST_BLOCKS = 304;   // (two blocks per SM; bounds the partials in c.red)

// The packs are written straight into the contexts' pinned host blocks (some
// 700 bytes, by one block at its end): no copy to queue, and the host waits for
// the stream once per call.  The kernels take up to STAT_GROUP contexts.
struct StatGroup {
    StatArgs a[STAT_GROUP];
};
static_assert(sizeof(StatGroup) <= 4096, "kernel parameters");

// the counters before the call's first step, one block per context
__global__ void k_stat_mark(const __grid_constant__ StatGroup g) {
    const StatArgs& a = g.a[blockIdx.x];
    const int t = threadIdx.x;
    if (t < MAX_SPECIES * NCTR) a.out[1].ctr[t] = a.ctrall[t];
    if (t < MAX_SPECIES) a.count[t] = 0ull;
    if (t == 0) {
        a.out[1].it_total = ((const long long*)a.scal)[40];
        a.out[1].outer_total = ((const long long*)a.scal)[41];
    }
}

// After it, gridDim.y contexts: the object's area-mean potential on Gamma_h and
// its collected charge, the species' particle counts, the solver's state.  One
// pass over the interface tets, the cut cells and the bins, block partials, and
// the last block to arrive packs the result.  The counts are integers (added
// to cleared words): eight more FP64 sums made the launch 23-33 us, not 12-15.
// Two reductions and a one-block count were three launches of 5-10 us each (the
// count alone 64-169 us with 250,000 bins).
__global__ void k_stat_pack(const __grid_constant__ StatGroup g) {
    const StatArgs& a = g.a[blockIdx.y];
    double v[3] = {0.0, 0.0, 0.0};
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, dt = (long long)gridDim.x * blockDim.x;
    const int ns = a.nspecies < MAX_SPECIES ? a.nspecies : MAX_SPECIES;
    if (a.diag) {
        const Mesh& m = a.m;
        for (long long T = t0; T < a.nit; T += dt) {
            // the object's surface only: a bedrock-plane tet lies inside the object
            const double* rec = a.it_data + T * IT_STRIDE;
            if (rec[IT_KIND] != 0.0) continue;
            int c = a.it_cell[T], t = a.it_t[T];
            int i = c % m.nx, j = (c / m.nx) % m.ny, k = c / (m.nx * m.ny);
            int p = (i + j + k) & 1;
            double s = a.qT[T] * rec[IT_SJ];
            for (int q = 0; q < 4; ++q) {
                int av, bv, cv; loff(cTf.vert[p][t][q], av, bv, cv);
                s += a.phi[node_id(m, i + av, j + bv, k + cv)] * rec[IT_S + q];
            }
            v[0] += s; v[1] += rec[IT_AREA];
        }
        for (long long c = t0; c < a.rhs.ncut; c += dt) {
            const int nsp = *a.rhs.nspec;
            for (int s = 0; s < nsp; ++s)
                v[2] += a.rhs.coefs[s] * (double)(long long)a.rhs.surf[(long long)s * a.rhs.ncut + c];
        }
    }
#pragma unroll
    for (int s = 0; s < MAX_SPECIES; ++s)
        if (s < ns && a.bcount[s]) {
            // (a warp's sum stays below 2^32: 32 lanes, nblocks / dt bins each, BIN_MAX particles a bin)
            unsigned n = 0;
            for (long long b = t0; b < a.nblocks; b += dt) n += (unsigned)a.bcount[s][b];
            n = __reduce_add_sync(0xffffffffu, n);
            if ((threadIdx.x & 31) == 0 && n) atomicAdd(a.count + s, (unsigned long long)n);
        }
    double tot[3];
    if (!grid_sum<3>(v, a.partial, a.ticket, tot)) return;   // (fences behind the counts too)
    StatPack* out = a.out;
    if (threadIdx.x >= 128 && threadIdx.x < 128 + MAX_SPECIES) {
        const int s = threadIdx.x - 128;
        out->count[s] = (long long)__ldcg(a.count + s) + (s < ns && a.mov_n[s] ? (long long)a.mov_n[s][0] : 0);
    }
    if (threadIdx.x < MAX_SPECIES * NCTR) out->ctr[threadIdx.x] = a.ctrall[threadIdx.x];
    if (threadIdx.x == 0) {
        const PcgState* S = (const PcgState*)a.scal;
        out->it = S->it;
        out->converged = S->converged;
        out->relres = S->relres;
        out->it_total = ((const long long*)a.scal)[40];
        out->outer_total = ((const long long*)a.scal)[41];
        out->surface_charge = tot[2];
        out->surface_potential = tot[1] > 0.0 ? tot[0] / tot[1] : 0.0;
        out->err = *a.err;
    }
}

static StatArgs stat_args(Ctx& c, bool diag) {
    StatArgs a = {};
    a.m = c.mesh;
    a.diag = diag;
    a.nit = c.nit; a.it_cell = c.it_cell; a.it_t = c.it_t; a.it_data = c.it_data; a.qT = c.qT; a.phi = c.phi;
    a.rhs = rargs(c);
    a.ctrall = c.ctrall;
    a.nspecies = (int)c.sp.size();
    for (int s = 0; s < a.nspecies && s < MAX_SPECIES; ++s) {
        a.bcount[s] = c.sp[s].bcount;
        a.mov_n[s] = c.sp[s].mov_n;
    }
    a.nblocks = c.nblocks;
    a.scal = c.scal;
    a.err = c.err_word;
    a.count = (unsigned long long*)c.red;
    a.partial = c.red + MAX_SPECIES;
    a.ticket = c.red_ticket;
    a.out = c.stat_host;
    long long work = c.nblocks;
    if (diag) work = std::max(work, std::max(c.nit, c.ncut));
    a.blocks = (int)std::max(1ll, std::min((long long)ST_BLOCKS, (work + ST_THREADS - 1) / ST_THREADS));
    return a;
}

cudaError_t mark_stats(Ctx* const* c, int n, cudaStream_t st) {
    for (int i = 0; i < n; i += STAT_GROUP) {
        StatGroup g = {};
        const int k = std::min(STAT_GROUP, n - i);
        for (int q = 0; q < k; ++q) g.a[q] = stat_args(*c[i + q], false);
        k_stat_mark<<<k, MAX_SPECIES * NCTR, 0, st>>>(g);
    }
    return cudaGetLastError();
}

cudaError_t queue_stats(Ctx* const* c, int n, cudaStream_t st) {
    for (int i = 0; i < n; i += STAT_GROUP) {
        StatGroup g = {};
        const int k = std::min(STAT_GROUP, n - i);
        int blocks = 1;   // (a context with less work than the largest: its last blocks find none)
        for (int q = 0; q < k; ++q) {
            g.a[q] = stat_args(*c[i + q], c[i + q]->have_object);
            blocks = std::max(blocks, g.a[q].blocks);
        }
        k_stat_pack<<<dim3(blocks, k), ST_THREADS, 0, st>>>(g);
    }
    return cudaGetLastError();
}

// FP64 node field from the current phi into E only (the FP32 copy the MIXED
// push reads is left as the step made it)
cudaError_t launch_node_E64(Ctx& c) {
    launch_node_E(fargs(c), c, nullptr, nullptr, c.stream);
    return cudaGetLastError();
}

cudaError_t set_field_tables(const TetTables& t) {
    // per cube of parity p holding the node at its local corner c8: G = sum
    // over the cube's tets containing it of vol_t grad_t at each corner (h = 1),
    // V = sum of their vol_t; summed in FP64
    double G[2][8][8][3] = {}, V[2][8] = {};
    for (int p = 0; p < 2; ++p)
        for (int q = 0; q < 5; ++q)
            for (int a = 0; a < 4; ++a) {
                const int c8 = t.vert[p][q][a];   // the tet contains local corner c8
                V[p][c8] += t.vol[q];
                for (int b = 0; b < 4; ++b)
                    for (int d = 0; d < 3; ++d) G[p][c8][t.vert[p][q][b]][d] += t.vol[q] * t.grad[p][q][b][d];
            }
    // the eight cubes around a node of parity P: the cube with the node at its
    // corner c8 = (a, b, c) has parity P + a + b + c, and its corner (x, y, z) is
    // the node's neighbour (x - a, y - b, z - c)
    double F[2][27][3] = {}, W[2] = {};
    for (int P = 0; P < 2; ++P)
        for (int c8 = 0; c8 < 8; ++c8) {
            const int a = c8 & 1, b = (c8 >> 1) & 1, cc = (c8 >> 2) & 1, pc = (P + a + b + cc) & 1;
            W[P] += V[pc][c8];
            for (int cn = 0; cn < 8; ++cn) {
                const int nb = ((cn & 1) - a + 1) + 3 * (((cn >> 1) & 1) - b + 1) + 9 * (((cn >> 2) & 1) - cc + 1);
                for (int d = 0; d < 3; ++d) F[P][nb][d] += G[pc][c8][cn][d];
            }
        }
    float Ff[2][81];
    for (int P = 0; P < 2; ++P)
        for (int nb = 0; nb < 27; ++nb)
            for (int d = 0; d < 3; ++d) Ff[P][3 * nb + d] = (float)(-F[P][nb][d] / W[P]);
    cudaError_t e = cudaMemcpyToSymbol(cTf, &t, sizeof(TetTables));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(cFold, Ff, sizeof(Ff));
    return e;
}

// ======================================================================================
// Field solve that allocates nothing (pifepic_solve_field_noalloc).
//
// Some callers cannot call cudaMalloc once their run is under way: a serving
// loop whose device memory is handed out by a pool it does not own (a
// cudaMalloc there can fail or stall the whole process on a device
// synchronisation), or an embedding that forbids allocation after start-up.
// pifepic_solve_field allocates a staging buffer on every call and its solver's
// plan on the first, so those callers need this variant.  It reuses the context's
// operator (read only), takes the load F, the flux jumps q (NULL: none) and
// the output phi as caller-owned device arrays, and keeps every work vector of
// the PCG in one file-scope device array of fixed size, found once per device
// with cudaGetSymbolAddress.  It always runs the FP64 PCG, whatever the
// context's precision.
// ======================================================================================
constexpr long long NOALLOC_MAX_NODES = 131072;                  // 2^17 mesh nodes
constexpr long long NOALLOC_PARTIALS = 4 * (NOALLOC_MAX_NODES / 256 + 1);
constexpr long long NOALLOC_DOUBLES = 5 * NOALLOC_MAX_NODES + NOALLOC_PARTIALS + 32;
// layout: u, b, r, p, q (NOALLOC_MAX_NODES each) | partials | PcgState + ticket
static __device__ __align__(256) double g_noalloc_scratch[NOALLOC_DOUBLES];

// the PCG steps of the graph version without the conditional handle; every
// launch after convergence returns at once, so the host can queue the
// iteration cap without waiting for the device
__global__ void k_na_init(FieldArgs f, const double* b, const double* q, double* r, double* p, double* partial,
                          unsigned* ticket, PcgState* S) {
    long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    double v[3] = {0, 0, 0};
    if (n < f.m.nnodes) {
        double bn = b[n];
        double rn = (f.ntype[n] == -3) ? 0.0 : bn - q[n];
        double zn = f.invdiag[n] * rn;
        r[n] = rn;
        p[n] = zn;
        v[0] = bn * bn; v[1] = rn * rn; v[2] = rn * zn;
    }
    double tot[3];
    if (grid_sum<3>(v, partial, ticket, tot) && threadIdx.x == 0) {
        S->bb = tot[0]; S->rr = tot[1]; S->rz = tot[2];
        S->it = 0;
        S->converged = (tot[0] == 0.0) || (tot[1] <= S->tol2 * tot[0]);
        S->done = S->converged || (S->maxit <= 0);
        S->relres = tot[0] > 0.0 ? sqrt(tot[1] / tot[0]) : 0.0;
    }
}

__global__ void k_na_spmv(FieldArgs f, const double* p, double* q, double* partial, unsigned* ticket, PcgState* S) {
    if (S->done) return;
    long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    double v[1] = {0.0};
    if (n < f.m.nnodes) {
        int i, j, k;
        node_ijk(f.m, n, i, j, k);
        double y = apply_row<double>(f, n, i, j, k, p, f.coef);
        q[n] = y;
        v[0] = p[n] * y;
    }
    double tot[1];
    if (grid_sum<1>(v, partial, ticket, tot) && threadIdx.x == 0) {
        S->pq = tot[0];
        S->alpha = S->rz / tot[0];
    }
}

__global__ void k_na_update(FieldArgs f, double* u, double* r, const double* p, const double* q, double* partial,
                            unsigned* ticket, PcgState* S) {
    if (S->done) return;
    long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    double alpha = S->alpha;
    double v[2] = {0, 0};
    if (n < f.m.nnodes) {
        double rn = r[n] - alpha * q[n];
        u[n] = u[n] + alpha * p[n];
        r[n] = rn;
        v[0] = rn * rn; v[1] = rn * f.invdiag[n] * rn;
    }
    double tot[2];
    if (grid_sum<2>(v, partial, ticket, tot) && threadIdx.x == 0) {
        S->rr = tot[0];
        S->beta = tot[1] / S->rz;
        S->rz = tot[1];
        S->it = S->it + 1;
        S->converged = tot[0] <= S->tol2 * S->bb;
        S->relres = sqrt(tot[0] / S->bb);
        S->done = S->converged || (S->it >= S->maxit);
    }
}

__global__ void k_na_dir(FieldArgs f, const double* r, double* p, const PcgState* S) {
    if (S->done) return;
    long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (n < f.m.nnodes) p[n] = f.invdiag[n] * r[n] + S->beta * p[n];
}

__global__ void k_na_state(PcgState* S, unsigned* ticket, double tol2, int maxit) {
    PcgState s = {};
    s.tol2 = tol2;
    s.maxit = maxit;
    *S = s;
    *ticket = 0u;
}

// set-up once per device (with that device current): in host code the name of
// a __device__ array is a host-side stand-in, not a device address, so the
// address is looked up with cudaGetSymbolAddress and cached per device.  Two
// threads doing the first call on one device at once both look it up and
// store the same value (an atomic store, so neither sees a torn pointer).
static std::atomic<void*> g_noalloc_dev[64];

pifepic_status solve_field_noalloc(Ctx& c, const double* F, const double* q, double* phi, int* iters,
                                   double* relres) {
    long long N = c.mesh.nnodes;
    if (N > NOALLOC_MAX_NODES) {
        char b[256];
        snprintf(b, sizeof(b), "solve_field_noalloc: mesh has %lld nodes; the fixed scratch holds at most %lld",
                 N, NOALLOC_MAX_NODES);
        c.err = b;
        log_error(b);
        return PIFEPIC_EINVAL;
    }
    // the scratch address is per device and the kernels run on the context's
    // stream, so the context's device must be the current one
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        c.err = "solve_field_noalloc: no current device";
        log_error(c.err.c_str());
        return PIFEPIC_ECUDA;
    }
    if (dev != c.device || dev < 0 || dev >= 64) {
        char b[160];
        snprintf(b, sizeof(b), "solve_field_noalloc: current device %d is not the context's device %d", dev,
                 c.device);
        c.err = b;
        log_error(b);
        return PIFEPIC_EINVAL;
    }
    void* base_ptr = g_noalloc_dev[dev].load(std::memory_order_acquire);
    if (!base_ptr) {
        cudaError_t e = cudaGetSymbolAddress(&base_ptr, g_noalloc_scratch);
        if (e != cudaSuccess || !base_ptr) {
            c.err = std::string("solve_field_noalloc: cudaGetSymbolAddress failed: ") + cudaGetErrorString(e);
            log_error(c.err.c_str());
            return PIFEPIC_ECUDA;
        }
        g_noalloc_dev[dev].store(base_ptr, std::memory_order_release);
    }
    double* base = (double*)base_ptr;
    double* u = base;
    double* bvec = base + NOALLOC_MAX_NODES;
    double* r = base + 2 * NOALLOC_MAX_NODES;
    double* p = base + 3 * NOALLOC_MAX_NODES;
    double* qv = base + 4 * NOALLOC_MAX_NODES;
    double* partial = base + 5 * NOALLOC_MAX_NODES;
    PcgState* S = (PcgState*)(partial + NOALLOC_PARTIALS);
    unsigned* ticket = (unsigned*)(partial + NOALLOC_PARTIALS + 24);
    FieldArgs f = fargs(c);
    RhsArgs a = rargs(c);
    unsigned gb = nb(N);
    cudaStream_t st = c.stream;
    k_na_state<<<1, 1, 0, st>>>(S, ticket, c.tol * c.tol, c.maxit);
    k_rhs<false><<<gb, 256, 0, st>>>(f, a, flux_rows(c), q, c.lift, bvec, F, StartArgs{});
    cudaMemsetAsync(u, 0, sizeof(double) * N, st);
    k_matvec<<<gb, 256, 0, st>>>(f, u, qv);
    k_na_init<<<gb, 256, 0, st>>>(f, bvec, qv, r, p, partial, ticket, S);
    for (int it = 0; it < c.maxit; ++it) {
        k_na_spmv<<<gb, 256, 0, st>>>(f, p, qv, partial, ticket, S);
        k_na_update<<<gb, 256, 0, st>>>(f, u, r, p, qv, partial, ticket, S);
        k_na_dir<<<gb, 256, 0, st>>>(f, r, p, S);
    }
    k_phi_from_u<<<gb, 256, 0, st>>>(N, u, c.gdir, phi, S);
    cudaError_t e = cudaGetLastError();
    PcgState hs;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hs, S, sizeof(PcgState), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        c.err = std::string("solve_field_noalloc: ") + cudaGetErrorString(e);
        log_error(c.err.c_str());
        return PIFEPIC_ECUDA;
    }
    if (iters) *iters = hs.it;
    if (relres) *relres = hs.relres;
    return PIFEPIC_OK;
}

}  // namespace pf
