// Shared by the PCG kernels whose vectors live in global memory (pcg_mg.cu,
// pcg_fd.cu): the team of blocks that solves one system -- a whole cooperative
// grid or one thread-block cluster -- the four-nodes-at-a-time pass and the
// FP32 row of the fine operator.
#pragma once
#include <cooperative_groups.h>

#include "pcg_sync.cuh"

namespace cg = cooperative_groups;

namespace pf {

// ---- the team that solves one system ---------------------------------------------------
// GridTeam: the whole cooperative grid (one system per launch; grid barriers and
// exchanges over the arrival counter, bounded waits).  ClusterTeam: one
// thread-block cluster per system (a batch of independent systems per launch;
// the hardware cluster barrier orders global memory within the cluster, and a
// reduction reads the C block partials through distributed shared memory).
template <class Args>
struct GridTeam {
    const Args& a;
    int& e;
    ExchShared& xs;
    __device__ long long t0() const { return (long long)blockIdx.x * blockDim.x + threadIdx.x; }
    __device__ long long size() const { return (long long)gridDim.x * blockDim.x; }
    __device__ int rank_of() const { return (int)blockIdx.x; }
    __device__ int ctas() const { return (int)gridDim.x; }
    __device__ bool leader() const { return blockIdx.x == 0; }
    __device__ bool sync() { return grid_barrier(a, e, xs); }
    template <typename A, int NV>
    __device__ bool reduce(A (&v)[NV], A (&tot)[NV]) { return exchange<A, NV>(a, e, v, tot, xs); }
};

struct ClusterSlots {
    double sh[4 * 32];
    double bc[4];
    double slot[2][4];    // this CTA's partials, by reduction parity
};

struct ClusterTeam {
    cg::cluster_group& cl;
    int C, rank;
    int e;
    ClusterSlots& cs;
    __device__ long long t0() const { return (long long)rank * blockDim.x + threadIdx.x; }
    __device__ long long size() const { return (long long)C * blockDim.x; }
    __device__ int rank_of() const { return rank; }
    __device__ int ctas() const { return C; }
    __device__ bool leader() const { return rank == 0; }
    __device__ bool sync() {
        cl.sync();
        return true;
    }
    // every CTA of the cluster gets the same totals (the partials summed in rank order)
    template <typename A, int NV>
    __device__ bool reduce(A (&v)[NV], A (&tot)[NV]) {
        A* sh = (A*)cs.sh;
        block_sum_t<A, NV>(v, sh);
        A* slot = (A*)cs.slot[e & 1];
        if (threadIdx.x == 0)
#pragma unroll
            for (int q = 0; q < NV; ++q) slot[q] = v[q];
        cl.sync();
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                A x = (A)0;
                if (lane < C) x = cl.map_shared_rank(slot, lane)[q];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
                if (lane == 0) ((A*)cs.bc)[q] = x;
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NV; ++q) tot[q] = ((A*)cs.bc)[q];
        ++e;
        return true;
    }
};

// A pass over the nodes [0, N) of a level, strided over the grid, four nodes
// at a time: every node's value (its loads) before any node's store, so the
// L2 round trips of a group overlap.
constexpr int PASS_UNROLL = 4;
template <class F, class S>
static __device__ __forceinline__ void pass4(long long N, long long t0, long long TT, F value, S store) {
    for (long long n0 = t0; n0 < N; n0 += PASS_UNROLL * TT) {
        float v[PASS_UNROLL];
#pragma unroll
        for (int u = 0; u < PASS_UNROLL; ++u) {
            const long long n = n0 + u * TT;
            v[u] = n < N ? value(n) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < PASS_UNROLL; ++u) {
            const long long n = n0 + u * TT;
            if (n < N) store(n, v[u]);
        }
    }
}

// a fine row times v (v inside a zeroed guard: the masked stencil reads the
// absent neighbours of boundary nodes and multiplies them by zero)
static __device__ __forceinline__ float fine_row_f(const FieldArgs& f, const float* v, long long n, unsigned kd) {
    if (kd & RK_DIRICHLET) return 0.0f;
    if (kd & RK_GENERAL) {
        int i, j, k;
        node_ijk(f.m, n, i, j, k);
        return apply_row<float, true>(f, n, i, j, k, v, f.coeff);
    }
    const int NX = f.m.NX, NXY = f.m.NX * f.m.NY;
    return regular_row_masked_ld<float>([&](int o) { return __ldcg(v + n + o); }, NX, NXY, kd, (float)f.m.h,
                                        h_over6<float>(f.m), h_over12<float>(f.m), (float)f.o.eps_plus,
                                        (float)f.o.eps_minus);
}

}  // namespace pf
