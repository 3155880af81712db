// MIXED-precision particle cycle: the same steps as particles.cu (Sec. 2.1
// gather / push / scatter, Sec. 3.1.3 and Sec. 5.2.2 injection, absorption and
// collection) with the state a particle carries cut to 28 bytes: a packed
// int32 cell (i | j<<11 | k<<22), the FP32 offset inside the cell and the
// FP32 velocity.  Positions never lose precision far from the origin because
// the offset is relative to the cell.  Node charges stay int64 with exactly
// 2^32 units per particle; the weights are FP32, rounded to 2^-19 of a particle
// inside a bin (2^-32 for movers).  Injection samples in FP32 from the same
// random streams as the FP64 path.
#include <math.h>

#include "internal.h"
#include "sampling.cuh"

namespace pf {

// kernels defined in particles.cu (bin construction and count clamping do not
// depend on the particle representation)
__global__ void k_bin_count(Launch L, PArr a, long long n, int* cnt);
__global__ void k_bin_caps(int nb, const int* cnt, int* cap, int* cnt_copy);
__global__ void k_bin_scan(int nb, const int* cap, long long* start, long long* total);
__global__ void k_clamp_counts(Launch L, long long* step);
cudaError_t launch_push_prep(Ctx& c);

// Which product of a b + c d is rounded before the fused sum: ROUND 1 the first, 2 the
// second, 0 either, as the compiler likes.  The bins' push pins it, 2 at a move's start
// and 1 at its end (its order when one pass did all): it takes the level set of a particle
// in two places, and left to the compiler 1 hit in 2 million (sphere; 1 in 700,000 on a
// plane, 1 in 12 million on a cap crater) within rounding of the surface or of a cell's
// face was decided differently than before the leavers had a pass of their own.
template <int ROUND>
PF_D float sum2(float a, float b, float c, float d) {
    return ROUND == 1 ? fmaf(c, d, a * b) : ROUND == 2 ? fmaf(a, b, c * d) : a * b + c * d;
}

template <int ROUND = 0>
PF_D float level_set_f(const ObjF& o, float x, float y, float z) {
    if (o.kind == 1) {
        float dx = x - o.a0, dy = y - o.a1, dz = z - o.a2;
        if (ROUND) return fmaf(dz, dz, sum2<ROUND>(dx, dx, dy, dy)) - o.a3;
        return (dx * dx + dy * dy + dz * dz) - o.a3;
    } else if (o.kind == 2) {
        float dx = x - o.a1, dy = y - o.a2;
        float r2 = sum2<ROUND>(dx, dx, dy, dy);
        float zs = (r2 < o.a3) ? o.a5 - sqrtf(o.a4 - r2) : o.a0;
        return z - zs;
    } else if (o.kind == 3) {
        if (ROUND) return fmaf(o.a2, z, sum2<ROUND>(o.a0, x, o.a1, y)) - o.a3;
        return o.a0 * x + o.a1 * y + o.a2 * z - o.a3;
    } else if (o.kind == 4) {   // rim crater, parameters as in level_set
        const float dx = x - o.a0, dy = y - o.a1;
        const float r = sqrtf(sum2<ROUND>(dx, dx, dy, dy));
        float zs;
        if (r <= o.a2) {
            zs = o.a5;
        } else if (r <= o.a3) {
            const float t = (r - o.a2) / o.a9;
            zs = o.a5 + o.a7 * ((t * t) * (3.0f - 2.0f * t));
        } else if (r < o.a4) {
            const float t = (r - o.a3) / o.a10;
            zs = o.a6 - o.a8 * ((t * t) * (3.0f - 2.0f * t));
        } else {
            zs = o.a11;
        }
        return z - zs;
    }
    return 1.0f;
}

PF_D int pack_cell(int i, int j, int k) { return i | (j << 11) | (k << 22); }
PF_D void unpack_cell(int c, int& i, int& j, int& k) {
    unsigned u = (unsigned)c;
    i = (int)(u & 2047u);
    j = (int)((u >> 11) & 2047u);
    k = (int)(u >> 22);
}

struct WF {
    float w[8];
};
PF_D WF weights_f(float fx, float fy, float fz) {
    WF r;
    float wx[2] = {1.0f - fx, fx}, wy[2] = {1.0f - fy, fy}, wz[2] = {1.0f - fz, fz};
#pragma unroll
    for (int l = 0; l < 8; ++l) r.w[l] = (wx[l & 1] * wy[(l >> 1) & 1]) * wz[(l >> 2) & 1];
    return r;
}

PF_D void fixed_weights_f(const WF& w, long long W[8]) {
    long long rest = 1ll << 32;
#pragma unroll
    for (int l = 0; l < 7; ++l) {
        // w < 1 except at a cell corner; 2^32 saturates to 2^32 - 1 and the
        // remainder weight below restores the exact total
        W[l] = (long long)__float2uint_rn(w.w[l] * 4294967296.0f);
        rest -= W[l];
    }
    W[7] = rest;
}

struct EGlobalF {
    const float4* E;
    Mesh m;
    PF_D float4 operator()(int i, int j, int k) const { return E[node_id(m, i, j, k)]; }
};

template <class EA>
PF_D void gather_f(int i, int j, int k, const WF& w, const EA& ea, float& ex, float& ey, float& ez) {
    ex = 0.f; ey = 0.f; ez = 0.f;
#pragma unroll
    for (int l = 0; l < 8; ++l) {
        float4 e = ea(i + (l & 1), j + ((l >> 1) & 1), k + ((l >> 2) & 1));
        ex += w.w[l] * e.x;
        ey += w.w[l] * e.y;
        ez += w.w[l] * e.z;
    }
}

// one particle: kick, drift in cell-relative coordinates, cell change,
// boundary test, object test (codes as in particles.cu)
enum { ALIVE = 0, ABSORBED = 1, COLLECTED = 2, NONE = 3 };

struct PF32 {
    int i, j, k;
    float fx, fy, fz, vx, vy, vz;
};

PF_D void advance_axis(float& f, int& c) {
    float s = floorf(f);
    f -= s;
    c += (int)s;
    if (f >= 1.0f) { f = 0.0f; c += 1; }   // -tiny - (-1) rounded up to 1
}

// reflecting faces (bit f = face f, minus face first per axis) on the cell +
// offset state: the mirror of c + f is -c - f at the minus face and 2n - c - f
// at the plus face, split again into a cell and an offset in [0, 1); a mirror
// that rounds onto n takes the last offset below 1 of cell n - 1
PF_D void reflect_axis_f(int& c, float& f, float& v, int n, int lo, int hi) {
    if (lo && c < 0) {
        if (f == 0.0f) {
            c = -c;
        } else {
            c = -c - 1; f = 1.0f - f;
            if (f >= 1.0f) { f = 0.0f; c += 1; }
        }
        v = -v;
    }
    if (hi && c >= n) {
        if (f == 0.0f) {
            c = 2 * n - c;
        } else {
            c = 2 * n - c - 1; f = 1.0f - f;
            if (f >= 1.0f) { f = 0.0f; c += 1; }
        }
        if (c >= n) { c = n - 1; f = 0.99999994f; }
        v = -v;
    }
}
PF_D void reflect_cell(const Mesh& m, int mask, PF32& p) {
    reflect_axis_f(p.i, p.fx, p.vx, m.nx, mask & 1, mask & 2);
    reflect_axis_f(p.j, p.fy, p.vy, m.ny, mask & 4, mask & 8);
    reflect_axis_f(p.k, p.fz, p.vz, m.nz, mask & 16, mask & 32);
}
// the same on a plain FP32 coordinate (injected particles, before the cell split)
PF_D void reflect_axis_pf(float& x, float& v, int n, int lo, int hi) {
    const float nf = (float)n;
    if (lo && x < 0.0f) { x = -x; v = -v; }
    if (hi && x >= nf) {
        x = (2.0f * nf) - x;
        if (x >= nf) x = __int_as_float(__float_as_int(nf) - 1);
        v = -v;
    }
}

template <bool PIN = false>
PF_D int hit_cell_f(const Launch& L, const ObjF& of, float xo, float yo, float zo, float xn, float yn, float zn) {
    float Lo = level_set_f<PIN ? 2 : 0>(of, xo, yo, zo), Ln = level_set_f<PIN ? 1 : 0>(of, xn, yn, zn);
    float t = Lo / (Lo - Ln);
    float xc = xo + t * (xn - xo), yc = yo + t * (yn - yo), zc = zo + t * (zn - zo);
    // the crossing point's cell on the IFE mesh (refine times finer; exact scaling)
    const float r = (float)L.refine;
    int ci = min(max((int)floorf(r * xc), 0), L.fmesh.nx - 1);
    int cj = min(max((int)floorf(r * yc), 0), L.fmesh.ny - 1);
    int ck = min(max((int)floorf(r * zc), 0), L.fmesh.nz - 1);
    return L.cell_acc[cell_id(L.fmesh, ci, cj, ck)];
}

template <bool PIN = false, class EA>
PF_D int push_one(const Launch& L, const ObjF& of, float kf, float dthf, int refl, PF32& p, const EA& ea, int& acc) {
    WF w = weights_f(p.fx, p.fy, p.fz);
    float ex, ey, ez;
    gather_f(p.i, p.j, p.k, w, ea, ex, ey, ez);
    p.vx += kf * ex; p.vy += kf * ey; p.vz += kf * ez;
    float xo = (float)p.i + p.fx, yo = (float)p.j + p.fy, zo = (float)p.k + p.fz;
    p.fx += p.vx * dthf; p.fy += p.vy * dthf; p.fz += p.vz * dthf;
    advance_axis(p.fx, p.i); advance_axis(p.fy, p.j); advance_axis(p.fz, p.k);
    if (refl) reflect_cell(L.mesh, refl, p);
    if (p.i < 0 || p.i >= L.mesh.nx || p.j < 0 || p.j >= L.mesh.ny || p.k < 0 || p.k >= L.mesh.nz) return ABSORBED;
    float xn = (float)p.i + p.fx, yn = (float)p.j + p.fy, zn = (float)p.k + p.fz;
    if (level_set_f<PIN ? 1 : 0>(of, xn, yn, zn) < 0.0f) {
        acc = hit_cell_f<PIN>(L, of, xo, yo, zo, xn, yn, zn);
        return COLLECTED;
    }
    return ALIVE;
}

// deposit on the IFE mesh: with refine r the IFE cell of (i + f) is r i +
// floor(r f) and its offset frac(r f) (exact in FP32: r is a power of two)
PF_D void global_deposit_f(const Launch& L, unsigned long long* W, const PF32& p) {
    long long Wf[8];
    int i = p.i, j = p.j, k = p.k;
    float fx = p.fx, fy = p.fy, fz = p.fz;
    if (L.refine != 1) {
        const float r = (float)L.refine;
        const float sx = floorf(r * fx), sy = floorf(r * fy), sz = floorf(r * fz);
        i = L.refine * i + (int)sx; j = L.refine * j + (int)sy; k = L.refine * k + (int)sz;
        fx = r * fx - sx; fy = r * fy - sy; fz = r * fz - sz;
    }
    fixed_weights_f(weights_f(fx, fy, fz), Wf);
#pragma unroll
    for (int l = 0; l < 8; ++l)
        atomicAdd(&W[node_id(L.fmesh, i + (l & 1), j + ((l >> 1) & 1), k + ((l >> 2) & 1))],
                  (unsigned long long)Wf[l]);
}

PF_D void load_p(const PArrF& a, long long g, PF32& p) {
    const unsigned* w = a.w + pword(g);
    unpack_cell((int)w[0], p.i, p.j, p.k);
    p.fx = __uint_as_float(w[32]); p.fy = __uint_as_float(w[64]); p.fz = __uint_as_float(w[96]);
    p.vx = __uint_as_float(w[128]); p.vy = __uint_as_float(w[160]); p.vz = __uint_as_float(w[192]);
}
PF_D void store_v(const PArrF& a, long long g, float vx, float vy, float vz) {
    unsigned* w = a.w + pword(g);
    w[128] = __float_as_uint(vx); w[160] = __float_as_uint(vy); w[192] = __float_as_uint(vz);
}
PF_D void store_p(const PArrF& a, long long g, const PF32& p, long long id, bool track) {
    unsigned* w = a.w + pword(g);
    w[0] = (unsigned)pack_cell(p.i, p.j, p.k);
    w[32] = __float_as_uint(p.fx); w[64] = __float_as_uint(p.fy); w[96] = __float_as_uint(p.fz);
    w[128] = __float_as_uint(p.vx); w[160] = __float_as_uint(p.vy); w[192] = __float_as_uint(p.vz);
    if (track) a.id[g] = id;
}

PF_D void count_event(unsigned long long* sctr, bool ev) {
    unsigned m = __ballot_sync(0xffffffffu, ev);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(sctr, (unsigned long long)__popc(m));
}

PF_D long long list_len(const unsigned long long* n, long long cap) {
    long long v = (long long)*n;
    return v < cap ? v : cap;
}

// the bin of a cell inside the mesh (non-negative indices; bin edge 2^bsh)
PF_D int block_of(const Launch& L, int ci, int cj, int ck) {
    return (ci >> L.bsh) + L.nbx * ((cj >> L.bsh) + L.nby * (ck >> L.bsh));
}

// ------------------------------------------------------------------------------------
// fused gather + push + boundary + collection + deposit + compaction (one bin per CTA)
// ------------------------------------------------------------------------------------
// A bin of B^3 cells reads and deposits through a TL^3 node tile, TL = B + 1.
// The node-field tile holds each node with its neighbour along x, P = (Ex, Ex', Ey, Ey') and
// Q = (Ez, Ez'): a cell's field is 4 x (16 + 8) bytes, 24 shared-memory wavefronts a warp at
// least, against 32 for eight float4 nodes.  t0 = tile index of the cell's corner 0; the sums
// run over the corners in their order, as gather_f's.
template <int TL>
PF_D void gather_tile(const float4* P, const float2* Q, int t0, const WF& w, float& ex, float& ey, float& ez) {
    ex = 0.f; ey = 0.f; ez = 0.f;
#pragma unroll
    for (int l = 0; l < 8; l += 2) {
        const float4 p = P[t0 + tile_corner<TL>(l)];
        const float2 q = Q[t0 + tile_corner<TL>(l)];
        ex += w.w[l] * p.x; ex += w.w[l + 1] * p.y;
        ey += w.w[l] * p.z; ey += w.w[l + 1] * p.w;
        ez += w.w[l] * q.x; ez += w.w[l + 1] * q.y;
    }
}

template <int TL>
PF_D int tile_index(int i, int j, int k, int x0, int y0, int z0) {
    return (i - x0) + TL * ((j - y0) + TL * (k - z0));
}

// a bin's deposit tile: NC interleaved 32-bit copies per node (copy = lane % NC),
// units of 2^-19 particle (see k_push_bins_m).  One particle: 7 rounded
// weights and the remainder, so it adds exactly 2^19.  (The scale, a power of
// two, goes into the z weights: the products round the same.)
template <int TL, int NC>
PF_D void tile_deposit19(unsigned* Wt, int t0, float fx, float fy, float fz) {
    const float wx[2] = {1.0f - fx, fx}, wy[2] = {1.0f - fy, fy}, wz[2] = {(1.0f - fz) * 524288.0f, fz * 524288.0f};
    unsigned rest = 1u << 19;
#pragma unroll
    for (int l = 0; l < 7; ++l) {
        const unsigned W = __float2uint_rn((wx[l & 1] * wy[(l >> 1) & 1]) * wz[(l >> 2) & 1]);
        rest -= W;
        atomicAdd(&Wt[t0 + NC * tile_corner<TL>(l)], W);
    }
    atomicAdd(&Wt[t0 + NC * tile_corner<TL>(7)], rest);
}
// add the tile to the node charges (2^32 units per particle), all threads of the block
// (a node's copies are read from a different one on by each lane: NC = 32 would put every
// lane's first copy into one bank)
template <int TL, int NC>
PF_D void tile_flush19(const Launch& L, unsigned long long* W, const unsigned* Wt, int x0, int y0, int z0) {
    for (int t = threadIdx.x; t < TL * TL * TL; t += blockDim.x) {
        long long v = 0;
        for (int c = 0; c < NC; ++c) {
            long long u = (long long)Wt[t * NC + ((c + t) & (NC - 1))];
            if (u >= (3ll << 30)) u -= 1ll << 32;     // a (small) negative copy total
            v += u;
        }
        if (!v) continue;
        int tx = t % TL, ty = (t / TL) % TL, tz = t / (TL * TL);
        int gi = x0 + tx, gj = y0 + ty, gk = z0 + tz;
        if (gi <= L.mesh.nx && gj <= L.mesh.ny && gk <= L.mesh.nz)
            atomicAdd(&W[node_id(L.mesh, gi, gj, gk)], (unsigned long long)(v * 8192));
    }
}

// One CTA of NW warps per (bin, species); warps take chunks of 32 particles in turn (chunk
// c to warp c mod NW) and meet at a block barrier only at the end.
//
// What bounds it is instruction issue (the state's 56 bytes a particle alone take 0.27 ms
// at 32.6M particles), so the pass over the chunks does only what every particle needs:
// kick, drift, and the test that it is still in the bin.  A particle that is (about 94 %
// on the 64^3 sphere) is written back to its own slot and deposits; in a bin that the
// object cannot reach and that touches no reflecting face no other test is due.  Any other
// particle only leaves its slot number in its warp's list, and 32 of them at a time go
// through the whole push again (push_leavers: reflection, faces, object, hit cell, mover
// list), so that the rare paths run on full warps.  The slots they leave are filled at the
// end from the bin's last stayers, matched by their ranks over the chunks' stayer masks.
// Against the pass that tested every particle for everything and compacted the stayers in
// order (a look-back over the chunks' counts), one launch of 32.6M particles (64^3 cells,
// bins of 4,096) went from 522 to 326 warp instructions a chunk and from 0.600 to 0.416 ms:
// 0.65 of the measured copy rate for the 56 bytes a particle, 0.56 on the 160 x 160 x 80
// crater (8.2 -> 5.8 ms).  Issue slots are then 67 % taken and the shared-memory pipe 60 %.
//
// A warp's next PUSH_DEPTH chunks are in flight at any time: one lane copies a chunk's 896
// bytes into the warp's stage with a bulk copy (bins start on whole groups of 32 slots), so
// the particles cost no address arithmetic and no registers while they travel.
// RF (instantiations of their own keep the common path's registers): 0, the IFE mesh is the PIC
// mesh; 2, it is twice as fine and B = 4: stayers deposit into a tile of its 9^3 nodes, in the
// 2^32 units a particle of the direct deposit (low and high halves, 8 copies a node, 47 KB), so
// the sums are the same integers; 1, any finer mesh, whose tile has no room (17^3 nodes): eight
// 64-bit atomics a particle straight onto its nodes.  4.1M particles in 32^3 cells of two IFE
// cells a side: 189 us directly, 96 by the tile.
constexpr int PUSH_DEPTH = 3;   // chunks in flight per warp
constexpr int PUSH_CHUNKS = (BIN_MAX + 31) / 32;

// the push's dynamic shared memory for bins of edge B: node-field pairs, deposit tile (first
// the landing place of the node-field tile), stages, stayer masks (in that order).  The
// stages' room later holds the masks' prefix counts and the list of slots to fill.
// 16 deposit copies a node halve the atomics' bank conflicts against 8 (32, without any, were
// no faster at 4,096 particles a bin and slower at 1,024); at B = 8 they would take 47 KB.
template <int RF, int B, int NW>
struct PushSmem {
    static constexpr int TL = B + 1, TN = TL * TL * TL;
    static constexpr int NC = B == 4 ? 16 : 8;
    static constexpr size_t pp = sizeof(float4) * TN, pq = (pp + sizeof(float2) * TN + 127) / 128 * 128;
    static constexpr int TL2 = 2 * B + 1, TN2 = TL2 * TL2 * TL2;   // IFE nodes of a bin, refine 2
    static constexpr int wn = RF == 2 ? 2 * 8 * TN2 : NC * TN;      // words of the deposit tile
    static constexpr size_t wt = (sizeof(unsigned) * wn + 127) / 128 * 128;
    static constexpr size_t stg = sizeof(unsigned) * NW * PUSH_DEPTH * 7 * 32;
    static constexpr size_t mask = sizeof(unsigned) * PUSH_CHUNKS;
    static constexpr size_t bytes = pq + wt + stg + mask;
    static constexpr int holes = (int)((stg - mask) / sizeof(unsigned short));   // slots to fill at a time
    static_assert(mask % 16 == 0 && stg > mask, "the prefix counts fit in the stages");
    static_assert(sizeof(float4) * TN <= wt, "the node-field tile lands in the deposit tile's room");
};

// the whole push of up to 32 particles of the bin that did not simply stay in it (act: the
// lanes that have one, in slot start + i): as push_one, then the survivors go to the mover
// list and deposit in the rebin, with every mover of the step
template <int TL>
static __device__ __noinline__ void push_leavers(const Launch& L, const SpeciesDev& S, const ObjF& of, float dthf,
                                                 const float4* P, const float2* Q, int x0, int y0, int z0, long long g,
                                                 bool act, unsigned* sctr) {
    int code = NONE, acc = -1;
    PF32 p;
    long long id = 0;
    if (act) {
        load_p(S.binsF, g, p);
        if (L.track) id = S.binsF.id[g];
        struct Tile {             // (a node as the neighbour of the one before it, but for the first of a row)
            const float4* P;
            const float2* Q;
            int x0, y0, z0;
            PF_D float4 operator()(int i, int j, int k) const {
                const int second = i > x0, t = tile_index<TL>(i - second, j, k, x0, y0, z0);
                const float4 p = P[t];
                const float2 q = Q[t];
                return second ? make_float4(p.y, p.w, q.y, 0.0f) : make_float4(p.x, p.z, q.x, 0.0f);
            }
        };
        code = push_one<true>(L, of, (float)S.k, dthf, S.reflect, p, Tile{P, Q, x0, y0, z0}, acc);
        if (code == COLLECTED && acc >= 0) atomicAdd(&S.surf[acc], 1ull);
    }
    count_event32(&sctr[C_ABSORBED], code == ABSORBED);
    count_event32(&sctr[C_COLLECTED], code == COLLECTED);
    count_event32(&sctr[C_LOST], code == COLLECTED && acc < 0);
    const bool alive = code == ALIVE;
    const long long slot = warp_reserve(S.mov_out_n, alive);
    if (alive) {
        if (slot < S.mcap) store_p(S.movF_out, slot, p, id, L.track);
        else atomicAdd(&S.ctr[C_DROPPED], 1ull);
    }
}

// a bulk copy to shared memory, counted on an mbarrier
PF_D void bulk_copy(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

template <int RF, int B, int NW>
__global__ void __launch_bounds__(32 * NW, RF == 2 ? 3 : 32 / NW) k_push_bins_m(const __grid_constant__ Launch L, const __grid_constant__ ObjF of,
                                                     float dthf, const __grid_constant__ CUtensorMap tmE) {
    using SM = PushSmem<RF, B, NW>;
    constexpr int NT = 32 * NW;
    constexpr int TL = SM::TL, TN = SM::TN;
    extern __shared__ __align__(128) unsigned char push_smem[];
    float4* Ep = reinterpret_cast<float4*>(push_smem);   // the bin's node field in pairs along x
    float2* Eq = reinterpret_cast<float2*>(push_smem + SM::pp);
    // deposits of the bin's stayers in units of 2^-19 particle, NC interleaved
    // copies per node (copy = lane % NC) so that the lanes of one atomic
    // instruction spread over the banks.  A particle adds 7 rounded weights and
    // the remainder 2^19 - sum (at least -4), so a copy, reached by at most
    // BIN_MAX / 8 + 1 particles, holds a value in [-2^14, 2^31]: exact in 32
    // bits modulo 2^32.  The flush multiplies by 2^13 (2^32 units per particle).
    unsigned* Wt = reinterpret_cast<unsigned*>(push_smem + SM::pq);
    float4* Et = reinterpret_cast<float4*>(Wt);          // the node-field tile (TMA destination) before
    // per warp and stage: cell, fx, fy, fz, vx, vy, vz of 32 particles
    typedef unsigned Stage[PUSH_DEPTH][7][32];
    Stage* stg = reinterpret_cast<Stage*>(push_smem + SM::pq + SM::wt);
    unsigned* stay_mask = reinterpret_cast<unsigned*>(push_smem + SM::pq + SM::wt + SM::stg);   // [chunk]
    __shared__ alignas(8) unsigned long long bar, sbar[NW][PUSH_DEPTH];
    __shared__ unsigned sctr[NCTR];
    __shared__ unsigned short list[NW][64];   // slots that wait for push_leavers, per warp
    __shared__ unsigned short rest[NW * 32];  // what the warps have left over at the end
    __shared__ int s_ok, s_rest, s_sum[NW];
    const int s = blockIdx.y;
    const int b = blockIdx.x;
    const SpeciesDev& S = L.sp[s];
    const int n = S.bcount[b];
    if (n == 0) {
        if (threadIdx.x == 0) S.bstay[b] = 0;
        return;
    }
    const int bx = b % L.nbx, by = (b / L.nbx) % L.nby, bz = b / (L.nbx * L.nby);
    const int x0 = bx * B, y0 = by * B, z0 = bz * B;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nch = (n + 31) >> 5;
    const long long start = S.bstart[b];
    unsigned* const bin = S.binsF.w + (start >> 5) * PGROUP;   // (bins start on whole groups)
    // one lane copies chunk cc (this warp's) into stage slot sl
    auto stage = [&](int cc, int sl) {
        if (cc < nch && lane == 0) {
            mbar_expect_tx(&sbar[wid][sl], 4 * PGROUP);
            bulk_copy(stg[wid][sl], bin + cc * PGROUP, 4 * PGROUP, &sbar[wid][sl]);
        }
    };
    if (tid == 0) {
        mbar_init(&bar, 1);
        for (int q = 0; q < NW * PUSH_DEPTH; ++q) mbar_init(&sbar[0][q], 1);
        fence_barrier_init();
        s_rest = 0;
    }
    if (tid < NCTR) sctr[tid] = 0u;
    __syncthreads();
    if (tid == 0) {
        mbar_expect_tx(&bar, TN * (unsigned)sizeof(float4));
        tma_load_4d(Et, &tmE, &bar, 0, x0, y0, z0);
    }
#pragma unroll
    for (int d = 0; d < PUSH_DEPTH; ++d) stage(wid + d * NW, d);
    if (tid == 0) {
        bool ok = mbar_wait_bounded(&bar, 0);
        if (!ok) {
            atomicOr(L.err, ERR_TMA_TIMEOUT);
            mbar_wait_bounded(&bar, 0);
        }
        s_ok = ok;
    }
    __syncthreads();
    for (int t = tid; t < TN; t += NT)
        if (t % TL < TL - 1) {
            const float4 u = Et[t], v = Et[t + 1];
            Ep[t] = make_float4(u.x, v.x, u.y, v.y);
            Eq[t] = make_float2(u.z, v.z);
        }
    __syncthreads();
    for (int t = tid; t < SM::wn; t += NT) Wt[t] = 0u;
    __syncthreads();
    const float kf = (float)S.k;
    // the bin's cells inside the mesh, the reflecting faces it touches, and whether the
    // object reaches it
    const int lx = min(B, L.mesh.nx - x0), ly = min(B, L.mesh.ny - y0), lz = min(B, L.mesh.nz - z0);
    const int refl = S.reflect & ((x0 == 0 ? 1 : 0) | (x0 + lx == L.mesh.nx ? 2 : 0) | (y0 == 0 ? 4 : 0) |
                                  (y0 + ly == L.mesh.ny ? 8 : 0) | (z0 == 0 ? 16 : 0) | (z0 + lz == L.mesh.nz ? 32 : 0));
    const bool clear = box_clear(of, (float)x0, (float)(x0 + lx), (float)y0, (float)(y0 + ly), (float)z0, (float)(z0 + lz));
    const int cell0 = pack_cell(x0, y0, z0);
    const int copy = lane & (SM::NC - 1);
    unsigned short* mine = list[wid];
    int waiting = 0;                       // slots in this warp's list
    bool fail = !s_ok;
    int sl = 0;                            // stage slot of the current chunk
    unsigned phase = 0;                    // its parity
    for (int c = wid; c < nch; c += NW) {
        const int i = c * 32 + lane;
        const bool live = i < n;
        if (!mbar_try_wait(&sbar[wid][sl], phase) && !mbar_wait_bounded(&sbar[wid][sl], phase)) {
            if (lane == 0) atomicOr(L.err, ERR_TMA_TIMEOUT);
            fail = true;
        }
        if (fail) {   // (one more bounded wait for each copy in flight, so that none lands after the block has left)
            for (int d = 0; d < PUSH_DEPTH && c + d * NW < nch; ++d) {
                mbar_wait_bounded(&sbar[wid][sl], phase);
                if (++sl == PUSH_DEPTH) { sl = 0; phase ^= 1; }
            }
            break;
        }
        // the cell relative to the bin, until the end
        int ri, rj, rk;
        float fx, fy, fz, vx, vy, vz;
        {
            const unsigned(&d)[7][32] = stg[wid][sl];
            unpack_cell(live ? (int)d[0][lane] : cell0, ri, rj, rk);
            ri -= x0; rj -= y0; rk -= z0;
            fx = __uint_as_float(d[1][lane]); fy = __uint_as_float(d[2][lane]); fz = __uint_as_float(d[3][lane]);
            vx = __uint_as_float(d[4][lane]); vy = __uint_as_float(d[5][lane]); vz = __uint_as_float(d[6][lane]);
        }
        // kick with the field gathered at the old position, then drift
        {
            const WF w = weights_f(fx, fy, fz);
            float ex, ey, ez;
            gather_tile<TL>(Ep, Eq, ri + TL * (rj + TL * rk), w, ex, ey, ez);
            vx += kf * ex; vy += kf * ey; vz += kf * ez;
        }
        fx += vx * dthf; fy += vy * dthf; fz += vz * dthf;
        advance_axis(fx, ri); advance_axis(fy, rj); advance_axis(fz, rk);
        if (refl) {
            PF32 p{ri + x0, rj + y0, rk + z0, fx, fy, fz, vx, vy, vz};
            reflect_cell(L.mesh, refl, p);
            ri = p.i - x0; rj = p.j - y0; rk = p.k - z0;
            fx = p.fx; fy = p.fy; fz = p.fz; vx = p.vx; vy = p.vy; vz = p.vz;
        }
        bool stay = live & ((unsigned)ri < (unsigned)lx) & ((unsigned)rj < (unsigned)ly) & ((unsigned)rk < (unsigned)lz);
        if (!clear)
            stay = stay &&
                   !(level_set_f<1>(of, (float)(ri + x0) + fx, (float)(rj + y0) + fy, (float)(rk + z0) + fz) < 0.0f);
        const unsigned bal = __ballot_sync(0xffffffffu, stay);
        // refill the stage slot: the bulk copy is not ordered after the reads of the slot by
        // itself, but the vote above has waited for what every lane made of its seven words
        stage(c + PUSH_DEPTH * NW, sl);
        if (++sl == PUSH_DEPTH) { sl = 0; phase ^= 1; }
        if (stay) {
            unsigned* o = bin + (c * PGROUP + lane);
            o[0] = (unsigned)(cell0 + ri + (rj << 11) + (rk << 22));
            o[32] = __float_as_uint(fx); o[64] = __float_as_uint(fy); o[96] = __float_as_uint(fz);
            o[128] = __float_as_uint(vx); o[160] = __float_as_uint(vy); o[192] = __float_as_uint(vz);
            if (RF == 2) {         // hybrid grid, two IFE cells a cell
                const float gx = 2.0f * fx, gy = 2.0f * fy, gz = 2.0f * fz, sx = floorf(gx), sy = floorf(gy),
                            sz = floorf(gz);
                const int t0 = 2 * ri + (int)sx + SM::TL2 * (2 * rj + (int)sy + SM::TL2 * (2 * rk + (int)sz));
                long long Wf[8];
                fixed_weights_f(weights_f(gx - sx, gy - sy, gz - sz), Wf);
                const long long W7[7] = {Wf[0], Wf[1], Wf[2], Wf[3], Wf[4], Wf[5], Wf[6]};
                int* lo = reinterpret_cast<int*>(Wt);
                tile_deposit<long long, SM::TL2>(lo, lo + 8 * SM::TN2, 8 * t0 + (lane & 7), W7);
            } else if (RF == 1) {  // finer: straight onto the IFE nodes
                global_deposit_f(L, S.W, PF32{ri + x0, rj + y0, rk + z0, fx, fy, fz, vx, vy, vz});
            } else {               // (movers deposit in the rebin, with every mover of the step)
                tile_deposit19<TL, SM::NC>(Wt, SM::NC * (ri + TL * (rj + TL * rk)) + copy, fx, fy, fz);
            }
        }
        if (lane == 0) stay_mask[c] = bal;
        const unsigned gone = __ballot_sync(0xffffffffu, live && !stay);
        if (gone) {
            if (live && !stay) mine[waiting + __popc(gone & ((1u << lane) - 1))] = (unsigned short)i;
            waiting += __popc(gone);
            __syncwarp();
            if (waiting >= 32) {
                push_leavers<TL>(L, S, of, dthf, Ep, Eq, x0, y0, z0, start + mine[lane], true, sctr);
                waiting -= 32;
                const unsigned short up = mine[32 + lane];
                __syncwarp();
                mine[lane] = up;
                __syncwarp();
            }
        }
    }
    // what the warps have left, 32 to a warp again
    {
        int at = 0;
        if (lane == 0 && waiting) at = atomicAdd(&s_rest, waiting);
        at = __shfl_sync(0xffffffffu, at, 0);
        if (lane < waiting) rest[at + lane] = mine[lane];
    }
    // (a warp that gave up: the bin's particles are dropped, the error flag reports it; a
    // tile that never came: the bin is left as it was)
    if (__syncthreads_or(fail)) {
        if (tid == 0) {
            const int left = s_ok ? 0 : n;
            S.bcount[b] = left;
            S.bstay[b] = left;
        }
        return;
    }
    for (int q = wid * 32; q < s_rest; q += NW * 32) {
        const bool act = q + lane < s_rest;
        push_leavers<TL>(L, S, of, dthf, Ep, Eq, x0, y0, z0, start + (act ? (int)rest[q + lane] : 0), act, sctr);
    }
    // the stayers' count before each chunk
    int* pre = reinterpret_cast<int*>(stg);
    int total;
    {
        constexpr int PER = (PUSH_CHUNKS + NT - 1) / NT;
        int cnt[PER], sum = 0;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            cnt[q] = tid * PER + q < nch ? __popc(stay_mask[tid * PER + q]) : 0;
            sum += cnt[q];
        }
        int inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) s_sum[wid] = inc;
        __syncthreads();
        int run = inc - sum;
        total = 0;
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            if (q < wid) run += s_sum[q];
            total += s_sum[q];
        }
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            if (tid * PER + q < nch) pre[tid * PER + q] = run;
            run += cnt[q];
        }
    }
    __syncthreads();   // (also: the leavers have been read from their slots)
    // the stayers in slots from `total` on move to the slots below it that leavers left,
    // in order of their ranks, SM::holes at a time
    unsigned short* hole = reinterpret_cast<unsigned short*>(push_smem + SM::pq + SM::wt + SM::mask);
    const int c1 = total >> 5;
    const int below = c1 < nch ? pre[c1] + __popc(stay_mask[c1] & ((1u << (total & 31)) - 1)) : total;
    const unsigned lt = (1u << lane) - 1;
    for (int h0 = 0; h0 < total - below; h0 += SM::holes) {
        for (int c = tid; c * 32 < total; c += NT) {
            unsigned m = ~stay_mask[c];
            if (total - c * 32 < 32) m &= (1u << (total - c * 32)) - 1;
            for (int rank = c * 32 - pre[c] - h0; m; ++rank, m &= m - 1)
                if (rank >= 0 && rank < SM::holes) hole[rank] = (unsigned short)(c * 32 + __ffs(m) - 1);
        }
        __syncthreads();
        for (int c = c1 + wid; c < nch; c += NW) {
            const unsigned m = stay_mask[c];
            const int slot = c * 32 + lane, rank = pre[c] + __popc(m & lt) - below - h0;
            if (slot >= total && ((m >> lane) & 1) && rank >= 0 && rank < SM::holes) {
                const int to = hole[rank];
                unsigned* o = bin + pword(to);
                const unsigned* f = bin + pword(slot);
#pragma unroll
                for (int d = 0; d < 7; ++d) o[32 * d] = f[32 * d];
                if (L.track) S.binsF.id[start + to] = S.binsF.id[start + slot];
            }
        }
        __syncthreads();
    }
    if (tid == 0) {
        S.bcount[b] = total;
        S.bstay[b] = total;
        sctr[C_PUSHED] = (unsigned)n;
    }
    if (RF == 2) {
        const int* lo = reinterpret_cast<const int*>(Wt);
        const int* hi = lo + 8 * SM::TN2;
        for (int t = tid; t < SM::TN2; t += NT) {
            long long v = 0;
            for (int c = 0; c < 8; ++c) {
                const int at = 8 * t + ((c + t) & 7);
                v += tile_value(lo[at], hi[at]);
            }
            const int gi = 2 * x0 + t % SM::TL2, gj = 2 * y0 + t / SM::TL2 % SM::TL2, gk = 2 * z0 + t / (SM::TL2 * SM::TL2);
            if (v && gi <= L.fmesh.nx && gj <= L.fmesh.ny && gk <= L.fmesh.nz)
                atomicAdd(&S.W[node_id(L.fmesh, gi, gj, gk)], (unsigned long long)v);
        }
    } else if (RF == 0) {
        tile_flush19<TL, SM::NC>(L, S.W, Wt, x0, y0, z0);
    }
    __syncthreads();
    if (tid < NCTR && sctr[tid]) atomicAdd(&S.ctr[tid], (unsigned long long)sctr[tid]);
}

__global__ void k_push_movers_m(Launch L, ObjF of, float dthf) {
    __shared__ unsigned long long sctr[NCTR];
    const int s = blockIdx.y;
    const SpeciesDev& S = L.sp[s];
    if (threadIdx.x < NCTR) sctr[threadIdx.x] = 0ull;
    __syncthreads();
    const long long n = list_len(S.mov_in_n, S.mcap);
    const EGlobalF ea{L.Ef, L.mesh};
    const bool track = L.track;
    const float kf = (float)S.k;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long base = blockIdx.x * (long long)blockDim.x; base < n; base += stride) {
        long long i = base + threadIdx.x;
        int code = NONE, acc = -1;
        PF32 p;
        long long id = 0;
        if (i < n) {
            load_p(S.movF_in, i, p);
            if (track) id = S.movF_in.id[i];
            code = push_one(L, of, kf, dthf, S.reflect, p, ea, acc);
            if (code == COLLECTED && acc >= 0) atomicAdd(&S.surf[acc], 1ull);
        }
        count_event(&sctr[C_PUSHED], code != NONE);
        count_event(&sctr[C_ABSORBED], code == ABSORBED);
        count_event(&sctr[C_COLLECTED], code == COLLECTED);
        count_event(&sctr[C_LOST], code == COLLECTED && acc < 0);
        bool alive = code == ALIVE;
        long long slot = warp_reserve(S.mov_out_n, alive);
        if (alive) {
            if (slot < S.mcap) store_p(S.movF_out, slot, p, id, track);
            else atomicAdd(&S.ctr[C_DROPPED], 1ull);
        }
    }
    __syncthreads();
    if (threadIdx.x < NCTR && sctr[threadIdx.x]) atomicAdd(&S.ctr[threadIdx.x], sctr[threadIdx.x]);
    list_read(S);
}

// injection: FP32 sampling (same random streams as the FP64 path) and FP32
// tests, stored as cell + FP32 offset
__global__ void k_inject_m(Launch L, InjArgs a, ObjF of, float dthf) {
    __shared__ unsigned long long sctr[NCTR];
    const int q = blockIdx.y;
    const InjectDev d = a.st[q];
    const int s = d.species;
    const SpeciesDev& S = L.sp[s];
    if (threadIdx.x < NCTR) sctr[threadIdx.x] = 0ull;
    __syncthreads();
    const int cnt = a.count[q];
    const long long idb = a.idbase[q];
    const bool track = L.track;
    const float nxf = (float)L.mesh.nx, nyf = (float)L.mesh.ny, nzf = (float)L.mesh.nz;
    for (int base = blockIdx.x * blockDim.x; base < cnt; base += gridDim.x * blockDim.x) {
        int mm = base + threadIdx.x;
        int code = NONE, acc = -1;
        bool rejected = false;
        PF32 p;
        if (mm < cnt) {
            // FP32 sample (the MIXED state is FP32); tests on the FP32 level set
            InjSampleF sm = inject_sample_f(d, mm, *a.step, s, L.mesh, dthf);
            if (S.reflect) {
                reflect_axis_pf(sm.p[0], sm.v[0], L.mesh.nx, S.reflect & 1, S.reflect & 2);
                reflect_axis_pf(sm.p[1], sm.v[1], L.mesh.ny, S.reflect & 4, S.reflect & 8);
                reflect_axis_pf(sm.p[2], sm.v[2], L.mesh.nz, S.reflect & 16, S.reflect & 32);
            }
            if (!sm.ok || level_set_f(of, sm.p0[0], sm.p0[1], sm.p0[2]) < 0.0f) {
                rejected = true;
            } else if (sm.p[0] < 0.0f || sm.p[0] >= nxf || sm.p[1] < 0.0f || sm.p[1] >= nyf || sm.p[2] < 0.0f ||
                       sm.p[2] >= nzf) {
                code = ABSORBED;
            } else {
                const float fi = floorf(sm.p[0]), fj = floorf(sm.p[1]), fk = floorf(sm.p[2]);
                p.i = (int)fi; p.j = (int)fj; p.k = (int)fk;
                p.fx = sm.p[0] - fi; p.fy = sm.p[1] - fj; p.fz = sm.p[2] - fk;
                if (p.fx >= 1.0f) p.fx = 0.99999994f;
                if (p.fy >= 1.0f) p.fy = 0.99999994f;
                if (p.fz >= 1.0f) p.fz = 0.99999994f;
                p.vx = sm.v[0]; p.vy = sm.v[1]; p.vz = sm.v[2];
                if (level_set_f(of, sm.p[0], sm.p[1], sm.p[2]) < 0.0f) {
                    acc = hit_cell_f(L, of, sm.p0[0], sm.p0[1], sm.p0[2], sm.p[0], sm.p[1], sm.p[2]);
                    code = COLLECTED;
                    if (acc >= 0) atomicAdd(&S.surf[acc], 1ull);
                } else {
                    code = ALIVE;   // deposits in the rebin
                }
            }
        }
        count_event(&sctr[C_INJECTED], code != NONE);
        count_event(&sctr[C_REJECTED], rejected);
        count_event(&sctr[C_ABSORBED], code == ABSORBED);
        count_event(&sctr[C_COLLECTED], code == COLLECTED);
        count_event(&sctr[C_LOST], code == COLLECTED && acc < 0);
        bool alive = code == ALIVE;
        long long slot = warp_reserve(S.mov_out_n, alive);
        if (alive) {
            if (slot < S.mcap) store_p(S.movF_out, slot, p, idb + mm, track);
            else atomicAdd(&S.ctr[C_DROPPED], 1ull);
        }
    }
    __syncthreads();
    if (threadIdx.x < NCTR && sctr[threadIdx.x]) atomicAdd(&S.ctr[threadIdx.x], sctr[threadIdx.x]);
}

// rebin: every particle of this step's mover list (bin leavers of the push,
// survivors of the spill list, injected and photoemitted particles) deposits
// its charge here, in one warp-coherent pass, then joins its bin or, if the
// bin is full, next step's spill list
// DEFER: a mover stored into a bin deposits later with the bin's other arrivals
// (k_deposit_arrivals_m); one that waits in the list deposits here
template <bool DEFER>
__global__ void k_rebin_m(Launch L) {
    const int s = blockIdx.y;
    const SpeciesDev& S = L.sp[s];
    const long long n = list_len(S.mov_out_n, S.mcap);
    const bool track = L.track;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long base = blockIdx.x * (long long)blockDim.x; base < n; base += stride) {
        long long i = base + threadIdx.x;
        bool spill = false;
        PF32 p;
        long long id = 0;
        if (i < n) {
            load_p(S.movF_out, i, p);
            if (track) id = S.movF_out.id[i];
            int b = block_of(L, p.i, p.j, p.k);
            int slot = warp_inc(&S.bcount[b]);
            if (slot < S.bcap[b]) store_p(S.binsF, S.bstart[b] + slot, p, id, track);
            else spill = true;
            if (!DEFER || spill) global_deposit_f(L, S.W, p);
        }
        long long slot = warp_reserve(S.mov_in_n, spill);
        if (spill) {
            if (slot < S.mcap) store_p(S.movF_in, slot, p, id, track);
            else atomicAdd(&S.ctr[C_DROPPED], 1ull);
        }
    }
}

// FP64 flat list -> MIXED bins (load, explicit particles, rebuild)
__global__ void k_bin_scatter_m(Launch L, int s, PArr a, long long n, bool track) {
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const SpeciesDev& S = L.sp[s];
    double fi = floor(a.x[i]), fj = floor(a.y[i]), fk = floor(a.z[i]);
    PF32 p;
    p.i = (int)fi; p.j = (int)fj; p.k = (int)fk;
    p.fx = (float)(a.x[i] - fi); p.fy = (float)(a.y[i] - fj); p.fz = (float)(a.z[i] - fk);
    if (p.fx >= 1.0f) p.fx = 0.99999994f;
    if (p.fy >= 1.0f) p.fy = 0.99999994f;
    if (p.fz >= 1.0f) p.fz = 0.99999994f;
    p.vx = (float)a.vx[i]; p.vy = (float)a.vy[i]; p.vz = (float)a.vz[i];
    int b = block_of(L, p.i, p.j, p.k);
    int slot = warp_inc(&S.bcount[b]);
    long long id = track ? a.id[i] : 0;
    if (slot < S.bcap[b]) {
        store_p(S.binsF, S.bstart[b] + slot, p, id, track);
    } else {   // a full bin: the particle waits in the mover list
        unsigned long long q = atomicAdd(S.mov_in_n, 1ull);
        if ((long long)q < S.mcap) store_p(S.movF_in, (long long)q, p, id, track);
        else atomicAdd(&S.ctr[C_DROPPED], 1ull);
    }
}

PF_D void put_d(const PArr& o, long long g, const PF32& p, long long id, bool track) {
    o.x[g] = (double)p.i + (double)p.fx; o.y[g] = (double)p.j + (double)p.fy; o.z[g] = (double)p.k + (double)p.fz;
    o.vx[g] = p.vx; o.vy[g] = p.vy; o.vz[g] = p.vz;
    if (track) o.id[g] = id;
}

__global__ void k_flatten_m(Launch L, int s, PArr out, unsigned long long* nout) {
    const SpeciesDev& S = L.sp[s];
    int b = blockIdx.x;
    int n = S.bcount[b];
    __shared__ unsigned long long base;
    if (threadIdx.x == 0) base = n ? atomicAdd(nout, (unsigned long long)n) : 0ull;
    __syncthreads();
    long long st = S.bstart[b];
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        PF32 p;
        load_p(S.binsF, st + i, p);
        put_d(out, (long long)base + i, p, L.track ? S.binsF.id[st + i] : 0, true);
    }
}

__global__ void k_flatten_list_m(Launch L, int s, PArr out, unsigned long long* nout) {
    const SpeciesDev& S = L.sp[s];
    long long n = list_len(S.mov_in_n, S.mcap);
    __shared__ unsigned long long base;
    if (threadIdx.x == 0) base = n ? atomicAdd(nout, (unsigned long long)n) : 0ull;
    __syncthreads();
    for (long long i = threadIdx.x; i < n; i += blockDim.x) {
        PF32 p;
        load_p(S.movF_in, i, p);
        put_d(out, (long long)base + i, p, L.track ? S.movF_in.id[i] : 0, true);
    }
}

// every binned particle's deposit (a full recount of the node charges) with
// the 2^-32 weights of global_deposit_f: on the PIC mesh through a shared tile
// of split 32-bit counters (tile_deposit; integer sums, so the node charges
// equal those of one global atomic per weight), on a finer IFE mesh straight
// to its nodes
template <bool HYBRID, int B>
__global__ void k_deposit_bins_m(Launch L) {
    constexpr int TL = B + 1, TN = TL * TL * TL;
    __shared__ int Wlo[8 * TN];
    __shared__ int Whi[8 * TN];
    const SpeciesDev& S = L.sp[blockIdx.y];
    const int b = blockIdx.x;
    const int n = S.bcount[b];
    if (n == 0) return;
    const long long st = S.bstart[b];
    if (HYBRID) {
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            PF32 p;
            load_p(S.binsF, st + i, p);
            global_deposit_f(L, S.W, p);
        }
        return;
    }
    const int bx = b % L.nbx, by = (b / L.nbx) % L.nby, bz = b / (L.nbx * L.nby);
    const int x0 = bx * B, y0 = by * B, z0 = bz * B;
    for (int t = threadIdx.x; t < 8 * TN; t += blockDim.x) { Wlo[t] = 0; Whi[t] = 0; }
    __syncthreads();
    const int copy = threadIdx.x & 7;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        PF32 p;
        load_p(S.binsF, st + i, p);
        long long Wf[8];
        fixed_weights_f(weights_f(p.fx, p.fy, p.fz), Wf);
        unsigned W7[7];
#pragma unroll
        for (int l = 0; l < 7; ++l) W7[l] = (unsigned)Wf[l];
        tile_deposit<unsigned, TL>(Wlo, Whi, 8 * tile_index<TL>(p.i, p.j, p.k, x0, y0, z0) + copy, W7);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < TN; t += blockDim.x) {
        long long v = 0;
        for (int c = 0; c < 8; ++c) v += tile_value(Wlo[t * 8 + c], Whi[t * 8 + c]);
        if (!v) continue;
        const int tx = t % TL, ty = (t / TL) % TL, tz = t / (TL * TL);
        const int gi = x0 + tx, gj = y0 + ty, gk = z0 + tz;
        if (gi <= L.mesh.nx && gj <= L.mesh.ny && gk <= L.mesh.nz)
            atomicAdd(&S.W[node_id(L.mesh, gi, gj, gk)], (unsigned long long)v);
    }
}
__global__ void k_deposit_list_m(Launch L) {
    const SpeciesDev& S = L.sp[blockIdx.y];
    long long n = list_len(S.mov_in_n, S.mcap);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        PF32 p;
        load_p(S.movF_in, i, p);
        global_deposit_f(L, S.W, p);
    }
}

__global__ void k_half_kick_bins_m(Launch L) {
    const SpeciesDev& S = L.sp[blockIdx.y];
    int b = blockIdx.x;
    int n = S.bcount[b];
    long long st = S.bstart[b];
    const EGlobalF ea{L.Ef, L.mesh};
    const float kh = (float)S.khalf;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        PF32 p;
        load_p(S.binsF, st + i, p);
        float ex, ey, ez;
        gather_f(p.i, p.j, p.k, weights_f(p.fx, p.fy, p.fz), ea, ex, ey, ez);
        store_v(S.binsF, st + i, p.vx - kh * ex, p.vy - kh * ey, p.vz - kh * ez);
    }
}
__global__ void k_half_kick_list_m(Launch L) {
    const SpeciesDev& S = L.sp[blockIdx.y];
    long long n = list_len(S.mov_in_n, S.mcap);
    const EGlobalF ea{L.Ef, L.mesh};
    const float kh = (float)S.khalf;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        PF32 p;
        load_p(S.movF_in, i, p);
        float ex, ey, ez;
        gather_f(p.i, p.j, p.k, weights_f(p.fx, p.fy, p.fz), ea, ex, ey, ez);
        store_v(S.movF_in, i, p.vx - kh * ex, p.vy - kh * ey, p.vz - kh * ez);
    }
}

// ------------------------------------------------------------------------------------
// host launchers
// ------------------------------------------------------------------------------------
static unsigned nb(long long n) { return (unsigned)((n + 255) / 256); }

cudaError_t set_mixed_tables(const TetTables&) { return cudaSuccess; }

static InjArgs inj_args_m(Ctx& c) {
    InjArgs a;
    a.st = c.inj_dev; a.nst = (int)c.inj.size();
    a.count = c.inj_count; a.idbase = c.inj_base; a.carry = c.inj_carry; a.next_id = c.next_id;
    a.step = (const long long*)(c.scal + 42);
    return a;
}

__global__ void k_inject_counts(InjArgs a);   // particles.cu

// one push launch; the kernel's dynamic shared-memory limit is raised once to what it
// needs (above the 48 KB default)
template <int RF, int B, int NW>
static cudaError_t push_bins_m(dim3 grid, cudaStream_t st, const Launch& L, const ObjF& of, float dthf,
                               const CUtensorMap& tm) {
    using SM = PushSmem<RF, B, NW>;
    static_assert(SM::bytes <= 200 * 1024, "push shared memory");
    void* kern = (void*)k_push_bins_m<RF, B, NW>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM::bytes);
    if (e != cudaSuccess) return e;
    k_push_bins_m<RF, B, NW><<<grid, 32 * NW, SM::bytes, st>>>(L, of, dthf, tm);
    return cudaGetLastError();
}
// Warps per block by the slots of a bin (particles and a quarter more, of the fullest
// species).  A block spends about 8 us outside the pass over its chunks (tile, leavers,
// filled slots, flush), so small bins want many small blocks in an SM to hide one's ends
// behind the others, large ones long passes that many warps share.  Push of the 64^3 sphere
// in ms: 4^3-cell bins of 512 particles 0.107 with 4 warps and 0.138 with 8, 2,048 0.236
// and 0.255, 3,072 0.336 and 0.332, 8,000 0.901 and 0.790; 8^3-cell bins of 4,096 particles
// 0.0944 with 8 warps and 0.0954 with 16, 8,192 0.151 and 0.143, 24,576 0.397 and 0.359.
constexpr long long PUSH_SMALL = 3700, PUSH_LARGE = 6200;   // slots of a bin, at B = 4 and 8
template <int B>
static cudaError_t push_bins_by_fill(dim3 grid, cudaStream_t st, const Launch& L, const ObjF& of, float dthf,
                                     const CUtensorMap& tm, long long slots) {
    if (slots < (B == 4 ? PUSH_SMALL : PUSH_LARGE)) return push_bins_m<0, B, B == 4 ? 4 : 8>(grid, st, L, of, dthf, tm);
    return push_bins_m<0, B, B == 4 ? 8 : 16>(grid, st, L, of, dthf, tm);
}

// what precedes a push: the step's mover-list counts and node charges start at zero
cudaError_t launch_push_prep_mixed(Ctx& c) { return launch_push_prep(c); }

cudaError_t launch_push_mixed(Ctx& c) {
    cudaError_t e = launch_push_prep_mixed(c);
    return e == cudaSuccess ? launch_push_bins_mixed(c) : e;
}

cudaError_t launch_push_bins_mixed(Ctx& c) {
    Launch L = make_launch(c);
    int ns = (int)c.sp.size();
    const dim3 grid(c.nblocks, ns);
    const ObjF of = obj_f(c.obj);
    const float dthf = (float)c.dth;
    long long slots = 0;
    for (const Species& q : c.sp) slots = q.cap > slots ? q.cap : slots;
    slots /= c.nblocks;
    cudaError_t e;
    if (c.bin_edge == 8)
        e = c.refine == 1 ? push_bins_by_fill<8>(grid, c.stream, L, of, dthf, c.tmapEf, slots)
                          : push_bins_m<1, 8, 8>(grid, c.stream, L, of, dthf, c.tmapEf);
    else
        e = c.refine == 1 ? push_bins_by_fill<4>(grid, c.stream, L, of, dthf, c.tmapEf, slots)
                          : c.refine == 2 ? push_bins_m<2, 4, 8>(grid, c.stream, L, of, dthf, c.tmapEf)
                                          : push_bins_m<1, 4, 8>(grid, c.stream, L, of, dthf, c.tmapEf);
    c.launches += 1;
    return e;
}

cudaError_t launch_movers_mixed(Ctx& c) {
    Launch L = make_launch(c);
    int ns = (int)c.sp.size();
    k_push_movers_m<<<dim3(152, ns), 256, 0, c.stream>>>(L, obj_f(c.obj), (float)c.dth);
    c.launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_photo_mixed(Ctx& c);

cudaError_t launch_inject_mixed(Ctx& c) {
    if (!c.inj.empty()) {
        Launch L = make_launch(c);
        InjArgs a = inj_args_m(c);
        k_inject_counts<<<1, 32, 0, c.stream>>>(a);
        int maxc = 1;
        for (auto& d : c.inj) maxc = d.maxcnt > maxc ? d.maxcnt : maxc;
        unsigned gx = (unsigned)((maxc + 255) / 256);
        if (gx > 1024) gx = 1024;
        k_inject_m<<<dim3(gx, (unsigned)c.inj.size()), 256, 0, c.stream>>>(L, a, obj_f(c.obj), (float)c.dth);
        c.launches += 2;
    }
    return launch_photo_mixed(c);
}

// ---- photoelectron emission (MIXED state) ----------------------------------
// The emitted counts are small, so the sample is taken in FP64 exactly as on the
// FP64 path and then stored as cell + FP32 offset.
PhotoArgs photo_args(Ctx& c);                 // particles.cu
cudaError_t launch_photo_counts(Ctx& c);
__global__ void k_photo_ids(long long* next_id, const long long* total);

__global__ void k_photo_m(Launch L, PhotoArgs a) {
    __shared__ unsigned long long sctr[NCTR];
    const SpeciesDev& S = L.sp[a.species];
    if (threadIdx.x < NCTR) sctr[threadIdx.x] = 0ull;
    __syncthreads();
    const long long total = *a.total;
    const long long idb = a.next_id[a.species];
    const unsigned long long key1 = stream_key(3, a.species, 0, *a.step);
    const bool track = L.track;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long base = blockIdx.x * (long long)blockDim.x; base < total; base += stride) {
        const long long m = base + threadIdx.x;
        bool emitted = false, alive = false, out = false;
        PF32 p;
        double vn = 0.0;
        const bool drawn = flux_normal(m < total, (unsigned long long)m, a.seed, key1, 0.0, vn);
        if (m < total) {
            const PhotoDev& d = a.tets[photo_tet_of(a.base, a.ne, m)];
            PhotoSample sm = photo_sample(d, (unsigned long long)m, a.seed, key1, a.vth, a.dth, drawn, vn);
            for (int c = 0; c < 3; ++c) sm.p[c] *= a.inv_r;   // IFE to PIC cell units (exact)
            if (S.reflect) reflect_d(L.mesh, S.reflect, sm.p[0], sm.p[1], sm.p[2], sm.v[0], sm.v[1], sm.v[2]);
            emitted = sm.ok && !(level_set(L.obj, sm.p[0], sm.p[1], sm.p[2]) < 0.0);
            if (emitted) {
                atomicAdd(&S.surf[d.acc], (unsigned long long)-1ll);   // the electron leaves +e behind
                out = (sm.p[0] < 0.0) | (sm.p[0] >= (double)L.mesh.nx) | (sm.p[1] < 0.0) |
                      (sm.p[1] >= (double)L.mesh.ny) | (sm.p[2] < 0.0) | (sm.p[2] >= (double)L.mesh.nz);
                alive = !out;
                if (alive) {
                    const double fi = floor(sm.p[0]), fj = floor(sm.p[1]), fk = floor(sm.p[2]);
                    p.i = (int)fi; p.j = (int)fj; p.k = (int)fk;
                    p.fx = (float)(sm.p[0] - fi); p.fy = (float)(sm.p[1] - fj); p.fz = (float)(sm.p[2] - fk);
                    if (p.fx >= 1.0f) p.fx = 0.99999994f;
                    if (p.fy >= 1.0f) p.fy = 0.99999994f;
                    if (p.fz >= 1.0f) p.fz = 0.99999994f;
                    p.vx = (float)sm.v[0]; p.vy = (float)sm.v[1]; p.vz = (float)sm.v[2];   // deposits in the rebin
                }
            }
        }
        count_event(&sctr[C_INJECTED], emitted);
        count_event(&sctr[C_REJECTED], m < total && !emitted);
        count_event(&sctr[C_ABSORBED], out);
        long long slot = warp_reserve(S.mov_out_n, alive);
        if (alive) {
            if (slot < S.mcap) store_p(S.movF_out, slot, p, idb + m, track);
            else atomicAdd(&S.ctr[C_DROPPED], 1ull);
        }
    }
    __syncthreads();
    if (threadIdx.x < NCTR && sctr[threadIdx.x]) atomicAdd(&S.ctr[threadIdx.x], sctr[threadIdx.x]);
}

cudaError_t launch_photo_mixed(Ctx& c) {
    if (c.ph_species < 0 || c.ph_ne <= 0) return cudaSuccess;
    cudaError_t e = launch_photo_counts(c);
    if (e != cudaSuccess) return e;
    k_photo_m<<<4 * 152, 256, 0, c.stream>>>(make_launch(c), photo_args(c));
    k_photo_ids<<<1, 1, 0, c.stream>>>(c.next_id + c.ph_species, c.ph_total);
    c.launches += 2;
    return cudaGetLastError();
}

// the bin's arrivals of this step, slots [bstay, bcount), deposit through a
// shared tile of split 32-bit counters with the 2^-32 weights of
// global_deposit_f (integer sums: the node charges equal those of one global
// atomic per weight, with an eighth of the global atomics or fewer)
template <int B>
__global__ void k_deposit_arrivals_m(Launch L) {
    constexpr int TL = B + 1, TN = TL * TL * TL;
    __shared__ int Wlo[8 * TN];
    __shared__ int Whi[8 * TN];
    const SpeciesDev& S = L.sp[blockIdx.y];
    const int b = blockIdx.x;
    const int n0 = S.bstay[b], n1 = S.bcount[b];   // (bcount clamped to the capacity)
    if (n1 <= n0) return;
    const long long st = S.bstart[b];
    const int bx = b % L.nbx, by = (b / L.nbx) % L.nby, bz = b / (L.nbx * L.nby);
    const int x0 = bx * B, y0 = by * B, z0 = bz * B;
    for (int t = threadIdx.x; t < 8 * TN; t += blockDim.x) { Wlo[t] = 0; Whi[t] = 0; }
    __syncthreads();
    const int copy = threadIdx.x & 7;
    for (int i = n0 + threadIdx.x; i < n1; i += blockDim.x) {
        PF32 p;
        load_p(S.binsF, st + i, p);
        long long Wf[8];
        fixed_weights_f(weights_f(p.fx, p.fy, p.fz), Wf);
        unsigned W7[7];
#pragma unroll
        for (int l = 0; l < 7; ++l) W7[l] = (unsigned)Wf[l];
        tile_deposit<unsigned, TL>(Wlo, Whi, 8 * tile_index<TL>(p.i, p.j, p.k, x0, y0, z0) + copy, W7);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < TN; t += blockDim.x) {
        long long v = 0;
        for (int c = 0; c < 8; ++c) v += tile_value(Wlo[t * 8 + c], Whi[t * 8 + c]);
        if (!v) continue;
        const int tx = t % TL, ty = (t / TL) % TL, tz = t / (TL * TL);
        const int gi = x0 + tx, gj = y0 + ty, gk = z0 + tz;
        if (gi <= L.mesh.nx && gj <= L.mesh.ny && gk <= L.mesh.nz)
            atomicAdd(&S.W[node_id(L.mesh, gi, gj, gk)], (unsigned long long)v);
    }
}

cudaError_t launch_rebin_mixed(Ctx& c) {
    Launch L = make_launch(c);
    int ns = (int)c.sp.size();
    const bool defer = c.refine == 1;   // (a finer IFE mesh takes the deposits node by node)
    if (defer) k_rebin_m<true><<<dim3(4 * 152, ns), 256, 0, c.stream>>>(L);
    else k_rebin_m<false><<<dim3(4 * 152, ns), 256, 0, c.stream>>>(L);
    k_clamp_counts<<<dim3(nb(c.nblocks), ns), 256, 0, c.stream>>>(L, (long long*)(c.scal + 42));
    if (defer) {
        if (c.bin_edge == 8) k_deposit_arrivals_m<8><<<dim3(c.nblocks, ns), 256, 0, c.stream>>>(L);
        else k_deposit_arrivals_m<4><<<dim3(c.nblocks, ns), 256, 0, c.stream>>>(L);
    }
    c.launches += defer ? 3 : 2;
    return cudaGetLastError();
}

cudaError_t launch_deposit_all_mixed(Ctx& c) {
    Launch L = make_launch(c);
    int ns = (int)c.sp.size();
    cudaMemsetAsync(c.Wall, 0, sizeof(unsigned long long) * MAX_SPECIES * c.mesh.nnodes, c.stream);
    if (ns == 0) return cudaGetLastError();
    const dim3 grid(c.nblocks, ns);
    if (c.bin_edge == 8) {
        if (c.refine > 1) k_deposit_bins_m<true, 8><<<grid, 256, 0, c.stream>>>(L);
        else k_deposit_bins_m<false, 8><<<grid, 256, 0, c.stream>>>(L);
    } else {
        if (c.refine > 1) k_deposit_bins_m<true, 4><<<grid, 256, 0, c.stream>>>(L);
        else k_deposit_bins_m<false, 4><<<grid, 256, 0, c.stream>>>(L);
    }
    k_deposit_list_m<<<dim3(64, ns), 256, 0, c.stream>>>(L);
    c.launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_half_kick_mixed(Ctx& c) {
    Launch L = make_launch(c);
    int ns = (int)c.sp.size();
    if (ns == 0) return cudaSuccess;
    k_half_kick_bins_m<<<dim3(c.nblocks, ns), 256, 0, c.stream>>>(L);
    k_half_kick_list_m<<<dim3(64, ns), 256, 0, c.stream>>>(L);
    c.launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_flatten_mixed_to_f64(Ctx& c, int s, PArr flat, unsigned long long* nflat) {
    Launch L = make_launch(c);
    if (c.sp[s].bcount) k_flatten_m<<<c.nblocks, 256, 0, c.stream>>>(L, s, flat, nflat);
    if (c.sp[s].mov_n) k_flatten_list_m<<<1, 256, 0, c.stream>>>(L, s, flat, nflat);
    return cudaGetLastError();
}

void free_parrf(PArrF& a) {
    lib_free(a.base);
    a = PArrF{};
}

// the groups of 32 particles, then the ids, in one allocation
cudaError_t alloc_parrf(PArrF& a, long long n, bool id) {
    free_parrf(a);
    const size_t groups = (size_t)(n > 0 ? n + 31 : 32) / 32;
    char* b = nullptr;
    cudaError_t e = lib_malloc(&b, groups * (sizeof(unsigned) * PGROUP + (id ? sizeof(long long) * 32 : 0)));
    if (e != cudaSuccess) return e;
    a.base = b;
    a.w = (unsigned*)b;
    if (id) a.id = (long long*)(b + groups * sizeof(unsigned) * PGROUP);
    return cudaSuccess;
}

// (re)build MIXED bins of species s from a flat FP64 list of n particles
cudaError_t launch_build_bins_mixed(Ctx& c, int s, PArr flat, long long n, bool) {
    Species& q = c.sp[s];
    cudaError_t e;
    int* cnt = nullptr;
    long long* tot = nullptr;
    long long total = 0;
    e = lib_malloc(&cnt, sizeof(int) * c.nblocks);
    if (e != cudaSuccess) return e;
    e = lib_malloc(&tot, sizeof(long long));
    if (e != cudaSuccess) { lib_free(cnt); return e; }
    cudaMemsetAsync(cnt, 0, sizeof(int) * c.nblocks, c.stream);
    Launch L = make_launch(c);
    if (n > 0) k_bin_count<<<nb(n), 256, 0, c.stream>>>(L, flat, n, cnt);
    if (!q.bcap) {
        lib_malloc(&q.bcap, sizeof(int) * c.nblocks);
        lib_malloc(&q.bcount, sizeof(int) * c.nblocks);
        lib_malloc(&q.bstart, sizeof(long long) * c.nblocks);
        lib_malloc(&q.bstay, sizeof(int) * c.nblocks);
    }
    cudaMemsetAsync(q.bstay, 0, sizeof(int) * c.nblocks, c.stream);
    k_bin_caps<<<nb(c.nblocks), 256, 0, c.stream>>>(c.nblocks, cnt, q.bcap, q.bcount);
    k_bin_scan<<<1, BIN_SCAN_THREADS, 0, c.stream>>>(c.nblocks, q.bcap, q.bstart, tot);
    e = cudaMemcpyAsync(&total, tot, sizeof(long long), cudaMemcpyDeviceToHost, c.stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c.stream);
    if (e != cudaSuccess) { lib_free(cnt); lib_free(tot); return e; }
    if (total > q.cap) {
        e = alloc_parrf(q.binsF, total, c.track != 0);
        if (e != cudaSuccess) { lib_free(cnt); lib_free(tot); return e; }
        q.cap = total;
    }
    L = make_launch(c);
    cudaMemsetAsync(q.mov_n, 0, 2 * sizeof(unsigned long long), c.stream);
    if (n > 0) k_bin_scatter_m<<<nb(n), 256, 0, c.stream>>>(L, s, flat, n, c.track != 0);
    k_clamp_counts<<<dim3(nb(c.nblocks), (unsigned)c.sp.size()), 256, 0, c.stream>>>(L, nullptr);
    e = cudaStreamSynchronize(c.stream);
    lib_free(cnt);
    lib_free(tot);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace pf
