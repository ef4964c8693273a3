// p2g_tiles.cuh -- the lane-per-cell P2G kernel of 1, 4 and 8 modes, and of the
// fused transfer's movers (its per-particle pieces are in p2g_kernel.cuh), and
// its launcher.  Each
// instantiation is compiled in one of the p2g_tiles_*.cu translation units.
//
// Work decomposition (no float atomics, bit-identical from run to run): one
// CTA per 8x8x4-cell tile, one warp per 4x4x2-cell block, one lane per cell;
// a lane accumulates its cell's 4 x 3 x 3 footprint of face grid A in
// registers over the rounds of the three component passes, the warp adds the
// 32 footprints into its block region in 36 node-offset phases, and the CTA
// adds the 8 block regions into the tile region in ascending block order.
#pragma once
#include "p2g_kernel.cuh"

namespace polypic {

constexpr int kP2GWarps = 8;

template <int A> struct Reg {
    static constexpr int X = reg_x(A), Y = reg_y(A), Z = reg_z(A);
};

// Index in block region A of node (ix, iy, iz) relative to the region origin.
template <int A>
__device__ __forceinline__ int region_index(int ix, int iy, int iz) {
    return (iz * Reg<A>::Y + iy) * Reg<A>::X + ix;
}

template <int R, bool AFF = false, int FMT = POLYPIC_COEFF_F32> constexpr int p2g_smem_bytes() {
    return (kP2GWarps * kRegionFloats + kP2GWarps * kStages * Stage<R, AFF, FMT>::NV * 32) * 4;
}
static_assert(p2g_smem_bytes<8, true>() <= 227 * 1024,
              "P2G staging exceeds the shared memory of a CTA");

// The rounds of the three component passes form one stream (pass 0 rounds
// 0 .. maxn-1, then pass 1, then pass 2) that flows through the stage ring
// without draining: while a pass finishes and merges, the first rounds of the
// next one are already in flight.  `ia` / `ir` name the next round to issue,
// `sn` / `pn` its slot and particle index (loaded one round ahead).
struct Pipe {
    int ia;
    uint32_t ir, sn, pn;
    uint32_t before;  // slots of the block before round ir
    int ring;  // stage holding the next round to consume

    // Slot of the lane's particle in round ir (every lane must call it); the
    // rounds come in order, so the slots before one are a running sum.
    __device__ __forceinline__ void locate(const uint32_t *perm, uint32_t bs, uint32_t n_c,
                                           unsigned lt) {
        const unsigned mask = __ballot_sync(0xffffffffu, n_c > ir);
        sn = bs + before + __popc(mask & lt);
        before += __popc(mask);
        pn = n_c > ir ? perm[sn] : 0u;
    }
};

template <int R, int FMT, bool ADJ, bool AFF>
__device__ __forceinline__ void pipe_issue(const P2GArgs &P, Pipe &q, uint32_t bs, uint32_t n_c,
                                           uint32_t maxn, unsigned lt, float *st, int lane) {
    if (q.ia < 3 && n_c > q.ir)  // q.ia is warp-uniform
        stage_particle<R, FMT, ADJ, AFF>(P, q.ia, q.pn, q.sn, st, lane);
    cp_async_commit();
    if (q.ia < 3 && ++q.ir == maxn) {
        q.ir = 0;
        q.before = 0;
        ++q.ia;
    }
    if (q.ia < 3) q.locate(P.perm, bs, n_c, lt);
}

template <int R, int FMT, int A, bool ADJ, bool AFF>
__device__ __forceinline__ void p2g_pass(const P2GArgs &P, Pipe &q, uint32_t bs, uint32_t n_c,
                                         uint32_t maxn, int ci, int cj, int ck, int gi, int gj,
                                         int gk, int lane, float *reg, float *stage, bool &bad) {
    using S = Stage<R, AFF, FMT>;
    // being in a cell of 1 .. n - 2 on every axis is the valid region 1 <= v < n - 1
    const bool valid = gi >= 1 && gi <= P.g.n[0] - 2 && gj >= 1 && gj <= P.g.n[1] - 2 &&
                       gk >= 1 && gk <= P.g.n[2] - 2;
    const float fi = (float)gi, fj = (float)gj, fk = (float)gk;
    Foot F;
    F.zero();
    const unsigned lt = (1u << lane) - 1u;
    for (uint32_t r = 0; r < maxn; ++r) {
        float *st = stage + q.ring * S::NV * 32;
        cp_async_wait<kStages - 1>();
        if (n_c > r) {
            const float px = st[S::kX * 32 + lane], py = st[S::kY * 32 + lane],
                        pz = st[S::kZ * 32 + lane];
            float mt = st[S::kM * 32 + lane];
            if (!ADJ && P.mass_abs) mt += st[S::kMabs * 32 + lane];
            const float v0 = cell_coord(px, P.g.inv_dx), v1 = cell_coord(py, P.g.inv_dx),
                        v2 = cell_coord(pz, P.g.inv_dx);
            const bool ok = valid && floorf(v0) == fi && floorf(v1) == fj && floorf(v2) == fk;
            if (ok) {
                const float vu = A == 0 ? v0 : (A == 1 ? v1 : v2);
                const float vv = A == 0 ? v1 : v0;
                const float vw = A == 2 ? v1 : v2;
                const Axis au = axis_decide(vu, true), av_ = axis_decide(vv, false),
                           aw = axis_decide(vw, false);
                const int cu = A == 0 ? gi : (A == 1 ? gj : gk);
                const int shift = au.base - (cu - 1);
                accumulate<R, FMT, A, ADJ, AFF>(P, st, lane, mt, shift, stencil_1d_scaled(au.t, P.s1, P.s2),
                                           stencil_1d_scaled(av_.t, P.s1, P.s2), stencil_1d_scaled(aw.t, P.s1, P.s2), au.guard,
                                           av_.guard, aw.guard, F);
            } else {
                bad = true;
            }
        }
        // refill the stage just consumed with the next round of the stream
        pipe_issue<R, FMT, ADJ, AFF>(P, q, bs, n_c, maxn, lt, st, lane);
        q.ring = q.ring + 1 == kStages ? 0 : q.ring + 1;
    }
    // merge the 32 footprints into the block region, one node offset per phase
    const int cu = A == 0 ? ci : (A == 1 ? cj : ck);
    const int cv = A == 0 ? cj : ci;
    const int cw = A == 2 ? cj : ck;
    float *rm = reg + reg_off(A, 0);
    float *rv = reg + reg_off(A, 1);
#pragma unroll
    for (int d = 0; d < 4; ++d)
#pragma unroll
        for (int kv = 0; kv < 3; ++kv)
#pragma unroll
            for (int kw = 0; kw < 3; ++kw) {
                const int nu = cu + d, nv = cv + kv, nw = cw + kw;
                const int ix = A == 0 ? nu : nv;
                const int iy = A == 0 ? nv : (A == 1 ? nu : nw);
                const int iz = A == 2 ? nu : nw;
                const int idx = region_index<A>(ix, iy, iz);
                rm[idx] += F.m(d, kv, kw);
                rv[idx] += F.v(d, kv, kw);
                __syncwarp();
            }
}

// All three passes of one block: the prologue fills the ring once.
template <int R, int FMT, bool ADJ, bool AFF>
__device__ __forceinline__ void p2g_block(const P2GArgs &P, uint32_t bs, uint32_t n_c,
                                          uint32_t maxn, int ci, int cj, int ck, int gi, int gj,
                                          int gk, int lane, float *reg, float *stage, bool &bad) {
    const unsigned lt = (1u << lane) - 1u;
    Pipe q;
    q.ia = 0;
    q.ir = 0;
    q.ring = 0;
    q.before = 0;
    q.locate(P.perm, bs, n_c, lt);
#pragma unroll
    for (int k = 0; k < kStages; ++k)
        pipe_issue<R, FMT, ADJ, AFF>(P, q, bs, n_c, maxn, lt, stage + k * Stage<R, AFF, FMT>::NV * 32,
                                     lane);
    p2g_pass<R, FMT, 0, ADJ, AFF>(P, q, bs, n_c, maxn, ci, cj, ck, gi, gj, gk, lane, reg, stage, bad);
    p2g_pass<R, FMT, 1, ADJ, AFF>(P, q, bs, n_c, maxn, ci, cj, ck, gi, gj, gk, lane, reg, stage, bad);
    p2g_pass<R, FMT, 2, ADJ, AFF>(P, q, bs, n_c, maxn, ci, cj, ck, gi, gj, gk, lane, reg, stage, bad);
    cp_async_wait<0>();
}

// Adds block region A of warp w into the tile region (written to dst).
template <int A>
__device__ __forceinline__ void merge_tile(const float *smem_regions, const bool *empty,
                                           float *dst) {
    constexpr int N = TileReg<A>::X * TileReg<A>::Y * TileReg<A>::Z;
    for (int i = threadIdx.x; i < N; i += kP2GWarps * 32) {
        const int lx = i % TileReg<A>::X, ly = (i / TileReg<A>::X) % TileReg<A>::Y,
                  lz = i / (TileReg<A>::X * TileReg<A>::Y);
        float sm = 0.0f, sv = 0.0f;
#pragma unroll
        for (int w = 0; w < kP2GWarps; ++w) {
            if (empty[w]) continue;
            const int bx = lx - 4 * (w & 1), by = ly - 4 * ((w >> 1) & 1), bz = lz - 2 * (w >> 2);
            if (bx < 0 || bx >= Reg<A>::X || by < 0 || by >= Reg<A>::Y || bz < 0 || bz >= Reg<A>::Z)
                continue;
            const float *r = smem_regions + w * kRegionFloats;
            const int idx = region_index<A>(bx, by, bz);
            sm += r[reg_off(A, 0) + idx];
            sv += r[reg_off(A, 1) + idx];
        }
        dst[tile_off(A, 0) + i] = sm;
        dst[tile_off(A, 1) + i] = sv;
    }
}

template <int R, int FMT, bool ADJ, bool AFF>
// two CTAs per SM fit without spills, but with 27 modes (one measured faster)
__global__ void __launch_bounds__(kP2GWarps * 32, R == 27 ? 1 : 2)
    k_p2g_tiles(P2GArgs P) {
    extern __shared__ float smem[];
    __shared__ bool s_empty[kP2GWarps];
    float *s_reg = smem;                                     // [8][kRegionFloats]
    float *s_stage = smem + kP2GWarps * kRegionFloats;        // [8][kStages][NV][32]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t tile = blockIdx.x;
    const bool tile_empty = P.cell_start[tile * 256] == P.cell_start[tile * 256 + 256];
    if (threadIdx.x == 0) P.tile_live[tile] = tile_empty ? 0 : 1;
    if (tile_empty) return;  // CTA-uniform

    const uint32_t b = tile * kP2GWarps + warp;
    const uint32_t k = b * 32 + lane;
    const uint32_t cs0 = P.cell_start[k];
    const uint32_t n_c = P.cell_start[k + 1] - cs0;
    const uint32_t bs = P.cell_start[b * 32];
    const uint32_t maxn = __reduce_max_sync(0xffffffffu, n_c);
    float *reg = s_reg + warp * kRegionFloats;
    float *stage = s_stage + warp * kStages * Stage<R, AFF, FMT>::NV * 32;
    if (lane == 0) s_empty[warp] = maxn == 0;
    if (maxn > 0) {
        for (int i = lane; i < kRegionFloats; i += 32) reg[i] = 0.0f;
        __syncwarp();
        int i0, j0, k0;
        block_origin(P.g, b, i0, j0, k0);
        const int ci = lane & 3, cj = (lane >> 2) & 3, ck = lane >> 4;
        const int gi = i0 + ci, gj = j0 + cj, gk = k0 + ck;
        bool bad = false;
        p2g_block<R, FMT, ADJ, AFF>(P, bs, n_c, maxn, ci, cj, ck, gi, gj, gk, lane, reg, stage,
                                    bad);
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(P.status, kFlagOutOfDomain);
    }
    __syncthreads();
    float *dst = P.scratch + (size_t)tile * kTileFloats;
    merge_tile<0>(s_reg, s_empty, dst);
    merge_tile<1>(s_reg, s_empty, dst);
    merge_tile<2>(s_reg, s_empty, dst);
}

template <int R, int FMT, bool ADJ, bool AFF = false>
cudaError_t launch_tiles(const P2GArgs &P, int grid, cudaStream_t s) {
    const int smem = p2g_smem_bytes<R, AFF, FMT>();
    // the attribute is a property of the kernel in the current context; it is
    // set on every launch (a cheap host call), which keeps no state shared
    // between host threads or devices
    const cudaError_t e = cudaFuncSetAttribute(k_p2g_tiles<R, FMT, ADJ, AFF>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_p2g_tiles<R, FMT, ADJ, AFF><<<grid, kP2GWarps * 32, smem, s>>>(P);
    return cudaGetLastError();
}

// Launchers of the instantiations, one per translation unit.
cudaError_t launch_tiles_f32(const P2GArgs &P, int R, int grid, cudaStream_t s);
cudaError_t launch_tiles_16(const P2GArgs &P, int R, int fmt, int grid, cudaStream_t s);
cudaError_t launch_tiles_adj(const P2GArgs &P, int R, int grid, cudaStream_t s);
cudaError_t launch_tiles_aff4(const P2GArgs &P, int grid, cudaStream_t s);

}  // namespace polypic
