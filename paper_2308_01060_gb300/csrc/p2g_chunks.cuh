// p2g_chunks.cuh -- the P2G kernel of 27 modes, of the node-by-node affine map
// and of solid phases, and its launcher.  Each instantiation is compiled in
// one of the p2g_chunks_*.cu translation units.
//
// Work decomposition (no float atomics, bit-identical from run to run): one
// CTA per 8x8x4-cell tile.  The tile's 8 blocks of 4x4x2 cells are split into
// G contiguous groups, and every (group, face grid) is one warp, which walks
// the slots of its blocks in chunks of 32 in two phases:
//   * lane = slot: the lane's particle is contracted into its 9 stencil
//     columns on the face grid (sum factorisation), 4 padded nodes along its
//     axis each, and the columns go to the warp's exchange buffer with the
//     particle's mass weights;
//   * lane = cell: each lane adds the chunk's particles of its cell, in slot
//     order, to the cell's 4 x 3 x 3 footprint held in registers (mass and
//     momentum).
// After a block's last chunk the warp adds the 32 footprints into its group
// region in 36 node-offset phases (distinct cells hit distinct nodes), and at
// the end the CTA adds the G group regions into the tile region in order.
//
// Only the second phase runs with the lanes of emptier cells idle; the
// lane-per-cell kernel of p2g_tiles.cuh idles them through the contraction as
// well (Poisson-filled cells: 55% of its lanes work).  What that is worth
// depends on the contraction, see launch_p2g in p2g.cu.
//
// What bounds it: the latency of 12 warps a SM (168 registers: 72 hold the
// footprint) and the shared-memory exchange, ~890 instructions a chunk and
// face grid at 40% issue.  Two choices were worth more than any other:
//   * the face grid is a run-time value, so that the SM's warps share one
//     code: three unrolled copies missed the instruction cache (891 us against
//     674 in the runs that compared them, 3.8 million particles, 27 modes FP32);
//   * L1 holds the lines of the loads in flight: the two CTAs of 27 modes FP32
//     of a fluid, and of the 16-bit formats, stay under the 164 KB carve-out of
//     shared memory by 384 bytes and more; the next step up (60 KB of L1 instead
//     of 92) cost 10%, two stages of coefficients (28 KB) 50%.  With two groups
//     a solid phase's absorbed mass and the affine map's six words take them
//     above it.
// In the form kept, P2G of those 3.8 million takes 697 us (lane per cell: 856).
#pragma once
#include <type_traits>

#include "p2g_kernel.cuh"

namespace polypic {

// Region of one group of 8 / G blocks on face grid A, in role order: u = the
// axis A (fastest), v and w = the two other axes in ascending order, so that
// one code serves the three face grids.
template <int G, int A> struct GroupReg {
    static constexpr int CX = G >= 8 ? 4 : 8, CY = G >= 4 ? 4 : 8, CZ = G >= 2 ? 2 : 4;
    static constexpr int U = (A == 0 ? CX : A == 1 ? CY : CZ) + 3, V = (A == 0 ? CY : CX) + 2,
                         W = (A == 2 ? CY : CZ) + 2, N = U * V * W;
};
template <int G> constexpr int group_floats() {
    return 2 * (GroupReg<G, 0>::N + GroupReg<G, 1>::N + GroupReg<G, 2>::N);
}
// Floats before region (A, mass | momentum) of a group.
template <int G, int A> constexpr int group_off(int which) {
    return (A >= 1 ? 2 * GroupReg<G, 0>::N : 0) + (A >= 2 ? 2 * GroupReg<G, 1>::N : 0) +
           which * GroupReg<G, A>::N;
}
template <class T> __device__ __forceinline__ T by_role(int a, T t0, T t1, T t2) {
    return a == 0 ? t0 : (a == 1 ? t1 : t2);
}

// Exchange buffer of a warp: rows of 32 float4 (one per slot of the chunk).
// Rows 0..8: the momentum column (kv, kw) = row, 4 nodes along A; row 9: the
// mass weight of the 4 nodes; rows 10, 11: the weights along the other axes.
constexpr int kExRows = 12;

// Staged words of a particle ([word][lane]): the coefficients, one per mode for
// FP32, one per pair of modes for the 16-bit formats; with the affine map the
// linear modes of the two other components; x, y, z, m, s_p (16-bit formats),
// m_abs (a solid phase).
template <int R, int FMT, bool AFF> struct ChunkStage {
    static constexpr int kL = FMT == POLYPIC_COEFF_F32 ? R : (R + 1) / 2;
    static constexpr int kX = kL + (AFF ? 6 : 0), kM = kX + 3, kS = kM + 1,
                         kMabs = kM + (FMT == POLYPIC_COEFF_F32 ? 1 : 2);
};
template <int R, int FMT, bool AFF> __host__ __device__ constexpr int stage_floats(bool solid) {
    return (ChunkStage<R, FMT, AFF>::kMabs + (solid ? 1 : 0)) * 32;
}
template <int R, int FMT, bool ADJ, bool AFF, int G> constexpr int chunks_smem_bytes(bool solid) {
    return (3 * G * ((ADJ ? 9 : kExRows) * 128 + stage_floats<R, FMT, AFF>(solid)) +
            G * group_floats<G>()) * 4;
}

// Column values of one particle on face grid A, written by `put(col, float4)`.
// Fu, Fv, Fw: the axis factors along A and the two other axes; the momentum
// weight is in Gp, Fu padded along A to 4 nodes (node = k + shift).
template <int R> struct Contraction {
    static constexpr int D = axis_degrees(R);
    // after the contraction along w: [dv][kw], du = 0, 1 as a packed pair
    float2 p[D][3];
    float s[D][3];  // du = 2 (27 modes)
};

template <int R, int A, class C>
__device__ __forceinline__ void contract_w(const C &coef, const float (&Fw)[axis_degrees(R)][3],
                                           Contraction<R> &T) {
    constexpr int D = axis_degrees(R);
#pragma unroll
    for (int dv = 0; dv < D; ++dv) {
#pragma unroll
        for (int kw = 0; kw < 3; ++kw) T.p[dv][kw] = make_float2(0.0f, 0.0f);
        // du = 0, 1 packed: the pair's coefficients sit in neighbouring
        // registers, only the axis factor is broadcast
#pragma unroll
        for (int dw = 0; dw < D; ++dw) {
            const bool h0 = has_mode(R, deg_x<A>(0, dv, dw), deg_y<A>(0, dv, dw), deg_z<A>(0, dv, dw));
            const bool h1 = has_mode(R, deg_x<A>(1, dv, dw), deg_y<A>(1, dv, dw), deg_z<A>(1, dv, dw));
            if (h0 && h1) {
                const float2 c = make_float2(
                    coef(mode_index(deg_x<A>(0, dv, dw), deg_y<A>(0, dv, dw), deg_z<A>(0, dv, dw))),
                    coef(mode_index(deg_x<A>(1, dv, dw), deg_y<A>(1, dv, dw), deg_z<A>(1, dv, dw))));
#pragma unroll
                for (int kw = 0; kw < 3; ++kw)
                    T.p[dv][kw] = dw == 0 ? __fmul2_rn(c, bcast(Fw[dw][kw]))
                                          : __ffma2_rn(c, bcast(Fw[dw][kw]), T.p[dv][kw]);
            } else if (h0) {  // 4 modes: no product modes
                const float c = coef(mode_index(deg_x<A>(0, dv, dw), deg_y<A>(0, dv, dw), deg_z<A>(0, dv, dw)));
#pragma unroll
                for (int kw = 0; kw < 3; ++kw) T.p[dv][kw].x = fmaf(c, Fw[dw][kw], T.p[dv][kw].x);
            }
        }
        if constexpr (D == 3) {
#pragma unroll
            for (int dw = 0; dw < 3; ++dw) {
                const float c = coef(mode_index(deg_x<A>(2, dv, dw), deg_y<A>(2, dv, dw), deg_z<A>(2, dv, dw)));
#pragma unroll
                for (int kw = 0; kw < 3; ++kw)
                    T.s[dv][kw] = dw == 0 ? c * Fw[dw][kw] : fmaf(c, Fw[dw][kw], T.s[dv][kw]);
            }
        }
    }
}

// Column (kv, kw): contract v, then u into the 4 padded nodes.
template <int R>
__device__ __forceinline__ float4 contract_column(const Contraction<R> &T,
                                                  const float (&Fv)[axis_degrees(R)][3],
                                                  const float2 (&Gp)[axis_degrees(R)][2], int kv,
                                                  int kw) {
    constexpr int D = axis_degrees(R);
    float2 t = __fmul2_rn(T.p[0][kw], bcast(Fv[0][kv]));
    if constexpr (R == 4) {  // only du = 0 has a mode with dv = 1
        t.x = fmaf(T.p[1][kw].x, Fv[1][kv], t.x);
    } else {
#pragma unroll
        for (int dv = 1; dv < D; ++dv) t = __ffma2_rn(T.p[dv][kw], bcast(Fv[dv][kv]), t);
    }
    float2 a = __fmul2_rn(bcast(t.x), Gp[0][0]), b = __fmul2_rn(bcast(t.x), Gp[0][1]);
    a = __ffma2_rn(bcast(t.y), Gp[1][0], a);
    b = __ffma2_rn(bcast(t.y), Gp[1][1], b);
    if constexpr (D == 3) {
        float u = T.s[0][kw] * Fv[0][kv];
        u = fmaf(T.s[1][kw], Fv[1][kv], u);
        u = fmaf(T.s[2][kw], Fv[2][kv], u);
        a = __ffma2_rn(bcast(u), Gp[2][0], a);
        b = __ffma2_rn(bcast(u), Gp[2][1], b);
    }
    return make_float4(a.x, a.y, b.x, b.y);
}

// Eq 12's affine map: M = (I + dt C)^-1 with C_ab = c_{a, 1+b} (the linear
// modes of all three components; stage rows R.. hold the other two
// components').  In role order: rows and columns u, v, w (the inverse permutes
// with the matrix).
template <int R, int A>
__device__ __forceinline__ void affine_inverse(const float *st, float dt,
                                               float (&M)[3][3]) {
    constexpr int ax[3] = {A, A == 0 ? 1 : 0, A == 2 ? 1 : 2};  // u, v, w
    float C[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int row = a == 0 ? 1 + ax[b] : R + 3 * (a - 1) + ax[b];
            C[a][b] = fmaf(dt, st[row * 32], a == b ? 1.0f : 0.0f);
        }
    inverse_or_identity(C, M);
}

// 8 and 27 modes under the map are not separable per axis: every stencil node
// evaluates s_r(xi) = f_a(xi_u) f_b(xi_v) f_c(xi_w) at xi = M z, with
// f_2(xi) = xi^2 - kappa xi - mu2 from the particle's own (unmapped) axis
// constants kappa = dx t (1 - 4t^2), mu2 = dx^2 / 4.  All in role order.
template <int R> struct Mapped {
    static constexpr int D = axis_degrees(R);
    float c[D][D][D], M[3][3];
    float kap[3], mu2;
    float Mz[3][3][3];  // [axis u/v/w][node k][component of xi]

    template <int A> __device__ __forceinline__ void load(const P2GArgs &P, const float *st) {
        affine_inverse<R, A>(st, P.map_dt, M);
#pragma unroll
        for (int du = 0; du < D; ++du)
#pragma unroll
            for (int dv = 0; dv < D; ++dv)
#pragma unroll
                for (int dw = 0; dw < D; ++dw)
                    c[du][dv][dw] = st[mode_index(deg_x<A>(du, dv, dw), deg_y<A>(du, dv, dw),
                                                  deg_z<A>(du, dv, dw)) * 32];
    }
    __device__ __forceinline__ void offsets(const P2GArgs &P, const float (&t3)[3]) {
        const float dx = P.dxpow[1];
        mu2 = 0.25f * P.dxpow[2];
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const float t = t3[e];
            kap[e] = dx * t * ((1.0f - 2.0f * t) * (1.0f + 2.0f * t));
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float z = ((float)(k - 1) - t) * dx;
#pragma unroll
                for (int g = 0; g < 3; ++g) Mz[e][k][g] = M[g][e] * z;
            }
        }
    }
    // sum_r c_r s_r at node (ku, kv, kw)
    __device__ __forceinline__ float node(int ku, int kv, int kw) const {
        float f[3][3];  // [axis][degree]
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            const float xi = Mz[0][ku][g] + Mz[1][kv][g] + Mz[2][kw][g];
            f[g][1] = xi;
            f[g][2] = fmaf(xi, xi - kap[g], -mu2);
        }
        float Sn = 0.0f;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            float Sa = 0.0f;
#pragma unroll
            for (int b = 0; b < D; ++b) {
                float Sb = c[a][b][0];
#pragma unroll
                for (int cc = 1; cc < D; ++cc) Sb = fmaf(c[a][b][cc], f[2][cc], Sb);
                Sa = b == 0 ? Sb : fmaf(Sb, f[1][b], Sa);
            }
            Sn = a == 0 ? Sa : fmaf(Sa, f[0][a], Sn);
        }
        return Sn;
    }
};

// A run of at most 32 slots of one block; ib == number of blocks: none left.
struct Chunk {
    int ib;
    uint32_t j0, je;  // first slot, end of the block's slots
};

// The work of one warp: face grid a over the blocks of group g.  `a` is a
// run-time value: the three face grids share one code (all but the reads of
// the coefficients), which has to stay in the instruction cache.
template <int R, int FMT, bool ADJ, bool AFF, int G>
__device__ __forceinline__ void p2g_item(const P2GArgs &P, uint32_t tile, int g, int a, int lane,
                                         float *ex, float *st, float *reg) {
    static_assert(R == 4 || R == 8 || R == 27, "one mode has no use for the exchange");
    static_assert(!AFF || R > 4, "the affine map of 4 modes is separable: k_p2g_tiles");
    constexpr int D = axis_degrees(R);
    constexpr int NB = 8 / G;
    constexpr bool F32 = FMT == POLYPIC_COEFF_F32;
    const unsigned full = 0xffffffffu;
    const uint32_t b0 = tile * 8 + g * NB;
    // lane l holds the first slot of block l (l = NB: the end)
    const uint32_t bound = P.cell_start[(b0 + (uint32_t)min(lane, NB)) * 32];
    // the next chunk; after the last one ib = NB and the slots stay valid
    auto advance = [&](Chunk &c) {
        if (c.j0 + 32 < c.je) {
            c.j0 += 32;
            return;
        }
        uint32_t j0, je;
        do {
            if (++c.ib >= NB) {
                c.ib = NB;
                return;
            }
            j0 = __shfl_sync(full, bound, c.ib);
            je = __shfl_sync(full, bound, c.ib + 1);
        } while (j0 >= je);
        c.j0 = j0;
        c.je = je;
    };
    Chunk cur{-1, 0, 0};
    advance(cur);
    if (cur.ib == NB) return;  // warp-uniform

    const uint32_t cnt = (uint32_t)P.count;  // rows are count words apart; count < 2^31
    // rows of face grid a
    using S = ChunkStage<R, FMT, AFF>;
    constexpr int H = S::kL;
    const uint32_t *rows = ADJ ? reinterpret_cast<const uint32_t *>(P.mu)
                               : reinterpret_cast<const uint32_t *>(P.coeff);
    rows += (uint64_t)cnt * (uint32_t)(a * H);
    const int ov = a == 0 ? 1 : 0, ow = a == 2 ? 1 : 2;  // the two other components / axes
    st += lane;
    auto stage = [&](uint32_t p, uint32_t slot) {
        cp_async4(st + S::kX * 32, P.x + p);
        cp_async4(st + (S::kX + 1) * 32, P.y + p);
        cp_async4(st + (S::kX + 2) * 32, P.z + p);
        if constexpr (!ADJ) {
            cp_async4(st + S::kM * 32, P.mass + p);
            if (P.mass_abs) cp_async4(st + S::kMabs * 32, P.mass_abs + p);
            if constexpr (!F32) cp_async4(st + S::kS * 32, P.scale + p);
        }
        // adjoint scatter: coefficients mu in slot order
        const uint32_t *c = rows + (ADJ ? slot : p);
#pragma unroll
        for (int r = ADJ ? 1 : 0; r < H; ++r)
            cp_async4(st + r * 32, c + (uint64_t)cnt * (uint32_t)r);
        if constexpr (ADJ) cp_async4(st, P.mu0 + (uint64_t)cnt * (uint32_t)a + slot);
        if constexpr (AFF) {
            const float *cf = reinterpret_cast<const float *>(P.coeff) + p;
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const float *co = cf + (uint64_t)cnt * (uint32_t)((o == 0 ? ov : ow) * R);
#pragma unroll
                for (int b = 0; b < 3; ++b)
                    cp_async4(st + (S::kL + 3 * o + b) * 32, co + (uint64_t)cnt * (uint32_t)(1 + b));
            }
        }
    };
    // a lane past the end of a chunk repeats its last slot (and is not counted)
    auto slot_of = [&](const Chunk &c) { return min(c.j0 + (uint32_t)lane, c.je - 1u); };

    // the stream of chunks: a lane stages its particle of the next chunk as soon
    // as it has consumed its stage column (cp.async throughout: the compiler
    // sinks loads into registers to their uses)
    Chunk nxt = cur;
    advance(nxt);
    stage(P.perm[slot_of(cur)], slot_of(cur));
    cp_async_commit();

    float2 accv[9][2], accm[ADJ ? 1 : 9][2];
    auto clear = [&]() {
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            accv[c][0] = accv[c][1] = make_float2(0.0f, 0.0f);
            if constexpr (!ADJ) accm[c][0] = accm[c][1] = make_float2(0.0f, 0.0f);
        }
    };
    clear();
    bool bad = false;
    // face grid 0 checks that the slots follow the order of polypic_sort: the
    // (rank in cell, cell) of a block's slots ascend and every cell has its count
    uint32_t seen = 0, want0 = 0, want1 = 0;  // the cell's slots: [want0, want1)
    int last = -1;
    {
        const uint32_t k = (b0 + cur.ib) * 32 + lane;
        want0 = P.cell_start[k];
        want1 = P.cell_start[k + 1];
    }
    float4 *ex4 = reinterpret_cast<float4 *>(ex) + lane;
    int ti, tj, tk;  // first cell of the group
    block_origin(P.g, b0, ti, tj, tk);

    for (;;) {
        const bool more = nxt.ib < NB;  // warp-uniform
        const uint32_t pn = P.perm[slot_of(nxt)];
        cp_async_wait<0>();
        struct {
            float x, y, z, m;
        } q;
        q.x = st[S::kX * 32];
        q.y = st[(S::kX + 1) * 32];
        q.z = st[(S::kX + 2) * 32];
        q.m = 1.0f;  // adjoint scatter: unit weight
        if constexpr (!ADJ) {
            q.m = st[S::kM * 32];
            if (P.mass_abs) q.m += st[S::kMabs * 32];
        }

        // ---- lane = slot: decisions and stencils
        const int fb = g * NB + cur.ib;  // block in tile
        const int bx = G >= 8 ? 0 : (fb & 1) * 4, by = G >= 4 ? 0 : (fb & 2) * 2,
                  bz = G >= 2 ? 0 : (fb & 4) >> 1;
        const int i0 = ti + bx, j0 = tj + by, k0 = tk + bz;
        const float v0 = cell_coord(q.x, P.g.inv_dx), v1 = cell_coord(q.y, P.g.inv_dx),
                    v2 = cell_coord(q.z, P.g.inv_dx);
        const int gi = (int)floorf(v0), gj = (int)floorf(v1), gk = (int)floorf(v2);
        // in the block and in the valid region 1 <= v < n - 1
        const bool in = cur.j0 + lane < cur.je;
        auto inside = [](int v, int lo, int hi) {  // lo <= v <= hi (none if hi < lo)
            return (unsigned)(v - lo) < (unsigned)max(hi - lo + 1, 0);
        };
        const bool ok = in && inside(gi, max(i0, 1), min(i0 + 3, P.g.n[0] - 2)) &&
                        inside(gj, max(j0, 1), min(j0 + 3, P.g.n[1] - 2)) &&
                        inside(gk, max(k0, 1), min(k0 + 1, P.g.n[2] - 2));
        bad |= in && !ok;
        const int cell = (gi & 3) | ((gj & 3) << 2) | ((gk & 1) << 4);
        const Axis au = axis_decide(by_role(a, v0, v1, v2), true),
                   av = axis_decide(a == 0 ? v1 : v0, false),
                   aw = axis_decide(a == 2 ? v1 : v2, false);
        const bool shift = au.base != by_role(a, gi, gj, gk) - 1;
        const Stencil1D su = stencil_1d_scaled(au.t, P.s1, P.s2),
                        sv = stencil_1d_scaled(av.t, P.s1, P.s2),
                        sw = stencil_1d_scaled(aw.t, P.s1, P.s2);
        float Fu[D][3], Fv[D][3], Fw[D][3];
        if constexpr (ADJ) {
            fit_rows<D>(su, au.guard, P.inv_dx, P.inv_dx2, Fu);
            fit_rows<D>(sv, av.guard, P.inv_dx, P.inv_dx2, Fv);
            fit_rows<D>(sw, aw.guard, P.inv_dx, P.inv_dx2, Fw);
        } else {
            axis_factors<D>(su, Fu);
            axis_factors<D>(sv, Fv);
            axis_factors<D>(sw, Fw);
        }
        auto pad = [&](float w, const float (&f)[3], float2 (&o)[2]) {
            const float f0 = w * f[0], f1 = w * f[1], f2 = w * f[2];
            o[0] = make_float2(shift ? 0.0f : f0, shift ? f0 : f1);
            o[1] = make_float2(shift ? f1 : f2, shift ? f2 : 0.0f);
        };
        auto put = [&](int row, float4 v) { ex4[row * 32] = v; };
        if constexpr (!ADJ) {
            float2 wm[2];
            pad(q.m, su.W, wm);
            put(9, make_float4(wm[0].x, wm[0].y, wm[1].x, wm[1].y));
            put(10, make_float4(sv.W[0], sv.W[1], sv.W[2], sw.W[0]));
            put(11, make_float4(sw.W[1], sw.W[2], 0.0f, 0.0f));
        }
        // once the lane's stage column is consumed
        auto refill = [&]() {
            stage(pn, slot_of(nxt));
            cp_async_commit();
        };
        if constexpr (AFF) {
            Mapped<R> E;
            if (a == 0) E.template load<0>(P, st);
            else if (a == 1) E.template load<1>(P, st);
            else E.template load<2>(P, st);
            refill();
            const float t3[3] = {au.t, av.t, aw.t};
            E.offsets(P, t3);
#pragma unroll
            for (int kv = 0; kv < 3; ++kv)
#pragma unroll
                for (int kw = 0; kw < 3; ++kw) {
                    const float w = q.m * sv.W[kv] * sw.W[kw];
                    float f[3];
#pragma unroll
                    for (int ku = 0; ku < 3; ++ku) f[ku] = su.W[ku] * E.node(ku, kv, kw);
                    float2 o[2];
                    pad(w, f, o);
                    put(kv * 3 + kw, make_float4(o[0].x, o[0].y, o[1].x, o[1].y));
                }
        } else {
            Contraction<R> T;
            auto contract = [&](auto axis) {
                constexpr int A = decltype(axis)::value;
                // the coefficient of mode r (16-bit codes: the low or high half of
                // word r / 2)
                auto coef = [&](int r) {
                    if constexpr (F32) {
                        return st[r * 32];
                    } else {
                        const uint32_t word = reinterpret_cast<const uint32_t *>(st)[(r / 2) * 32];
                        return Codec<FMT>::decode((uint16_t)((r & 1) ? word >> 16 : word));
                    }
                };
                contract_w<R, A>(coef, Fw, T);
            };
            if (a == 0) contract(std::integral_constant<int, 0>{});
            else if (a == 1) contract(std::integral_constant<int, 1>{});
            else contract(std::integral_constant<int, 2>{});
            const float mom = F32 ? q.m : q.m * st[S::kS * 32];
            refill();
            float2 Gp[D][2];
#pragma unroll
            for (int d = 0; d < D; ++d) pad(mom, Fu[d], Gp[d]);
#pragma unroll
            for (int kv = 0; kv < 3; ++kv)
#pragma unroll
                for (int kw = 0; kw < 3; ++kw)
                    put(kv * 3 + kw, contract_column<R>(T, Fv, Gp, kv, kw));
        }
        __syncwarp();

        // ---- lane = cell: the chunk's slots that hold a particle of the lane's cell
        unsigned mine = __ballot_sync(full, ok);
#pragma unroll
        for (int b = 0; b < 5; ++b) {
            const unsigned with = __ballot_sync(full, (cell >> b) & 1);
            mine &= (lane >> b) & 1 ? with : ~with;
        }
        if (a == 0) {  // warp-uniform
            const uint32_t rank = __shfl_sync(full, seen, cell) +
                                  __popc(__shfl_sync(full, mine, cell) & ((1u << lane) - 1u));
            const int place = (int)(rank * 32) + cell;
            int before = __shfl_up_sync(full, place, 1);
            if (lane == 0) before = last;
            bad |= ok && place <= before;
            last = __shfl_sync(full, place, 31);  // read only while the block goes on
            seen += __popc(mine);
        }
        const float4 *row0 = ex4 - lane;
        while (__any_sync(full, mine != 0)) {
            if (mine) {
                const float4 *row = row0 + (__ffs(mine) - 1);
                mine &= mine - 1;
#pragma unroll
                for (int c = 0; c < 9; ++c) {
                    const float4 v = row[c * 32];
                    accv[c][0] = __fadd2_rn(accv[c][0], make_float2(v.x, v.y));
                    accv[c][1] = __fadd2_rn(accv[c][1], make_float2(v.z, v.w));
                }
                if constexpr (!ADJ) {
                    const float4 m = row[9 * 32], e = row[10 * 32], f = row[11 * 32];
                    const float Wv[3] = {e.x, e.y, e.z}, Ww[3] = {e.w, f.x, f.y};
                    const float2 m01 = make_float2(m.x, m.y), m23 = make_float2(m.z, m.w);
#pragma unroll
                    for (int kv = 0; kv < 3; ++kv)
#pragma unroll
                        for (int kw = 0; kw < 3; ++kw) {
                            const float2 w = bcast(Wv[kv] * Ww[kw]);
                            accm[kv * 3 + kw][0] = __ffma2_rn(w, m01, accm[kv * 3 + kw][0]);
                            accm[kv * 3 + kw][1] = __ffma2_rn(w, m23, accm[kv * 3 + kw][1]);
                        }
                }
            }
        }
        __syncwarp();

        if (nxt.ib != cur.ib) {
            // the block is done: its 32 footprints into the group region, one
            // node offset per phase
            const int x = bx + (lane & 3), y = by + ((lane >> 2) & 3), z = bz + (lane >> 4);
            const int sv_ = by_role(a, GroupReg<G, 0>::U, GroupReg<G, 1>::U, GroupReg<G, 2>::U);
            const int sw_ = sv_ * by_role(a, GroupReg<G, 0>::V, GroupReg<G, 1>::V, GroupReg<G, 2>::V);
            const int half = by_role(a, GroupReg<G, 0>::N, GroupReg<G, 1>::N, GroupReg<G, 2>::N);
            float *rm = reg + by_role(a, x, y, z) + (a == 0 ? y : x) * sv_ + (a == 2 ? y : z) * sw_;
#pragma unroll
            for (int c = 0; c < 9; ++c) {
                float *m = rm + (c / 3) * sv_ + (c % 3) * sw_, *v = m + half;
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    const float2 v2_ = accv[c][d >> 1];
                    v[d] += (d & 1) ? v2_.y : v2_.x;
                    if constexpr (!ADJ) {
                        const float2 m2_ = accm[c][d >> 1];
                        m[d] += (d & 1) ? m2_.y : m2_.x;
                    }
                    __syncwarp();
                }
            }
            clear();
            if (a == 0) {
                bad |= seen != want1 - want0;
                seen = 0;
                last = -1;
                if (more) {
                    const uint32_t k = (b0 + nxt.ib) * 32 + lane;
                    want0 = P.cell_start[k];
                    want1 = P.cell_start[k + 1];
                }
            }
        }
        if (!more) break;
        cur = nxt;
        advance(nxt);
    }
    cp_async_wait<0>();
    if (__any_sync(full, bad) && lane == 0) atomicOr(P.status, kFlagOutOfDomain);
}

// The G group regions of face grid A added into the tile region (dst).
template <int G, int A, bool ADJ>
__device__ __forceinline__ void merge_groups(const float *regions, float *dst) {
    using Reg = GroupReg<G, A>;
    constexpr int X = TileReg<A>::X, Y = TileReg<A>::Y, Z = TileReg<A>::Z;
    for (int i = threadIdx.x; i < X * Y * Z; i += 96 * G) {
        const int lx = i % X, ly = (i / X) % Y, lz = i / (X * Y);
        float sm = 0.0f, sv = 0.0f;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int fb = g * (8 / G);  // first block of the group
            const int x = lx - (fb & 1) * 4, y = ly - ((fb >> 1) & 1) * 4, z = lz - (fb >> 2) * 2;
            const int u = A == 0 ? x : (A == 1 ? y : z), v = A == 0 ? y : x, w = A == 2 ? y : z;
            if (u < 0 || u >= Reg::U || v < 0 || v >= Reg::V || w < 0 || w >= Reg::W) continue;
            const float *r = regions + g * group_floats<G>() + (w * Reg::V + v) * Reg::U + u;
            if constexpr (!ADJ) sm += r[group_off<G, A>(0)];
            sv += r[group_off<G, A>(1)];
        }
        if constexpr (!ADJ) dst[tile_off(A, 0) + i] = sm;
        dst[tile_off(A, 1) + i] = sv;
    }
}

template <int R, int FMT, bool ADJ, bool AFF, int G>
// 12 warps an SM: the footprint (72 registers) beside the contraction
__global__ void __launch_bounds__(96 * G, 4 / G) k_p2g_chunks(P2GArgs P) {
    extern __shared__ float4 smem4[];
    float *regions = reinterpret_cast<float *>(smem4);  // after the buffers below
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t tile = blockIdx.x;
    const bool tile_empty = P.cell_start[tile * 256] == P.cell_start[tile * 256 + 256];
    if (threadIdx.x == 0) P.tile_live[tile] = tile_empty ? 0 : 1;
    if (tile_empty) return;  // CTA-uniform
    const int kEx = (ADJ ? 9 : kExRows) * 128,
              kSt = stage_floats<R, FMT, AFF>(P.mass_abs != nullptr);
    float *ex = regions + warp * (kEx + kSt), *st = ex + kEx;
    regions += 3 * G * (kEx + kSt);
    const int g = warp / 3, a = warp - 3 * g;
    float *mine = regions + g * group_floats<G>();
    for (int i = threadIdx.x; i < G * group_floats<G>(); i += 96 * G) regions[i] = 0.0f;
    __syncthreads();
    p2g_item<R, FMT, ADJ, AFF, G>(P, tile, g, a, lane, ex, st,
                                  mine + by_role(a, group_off<G, 0>(0), group_off<G, 1>(0), group_off<G, 2>(0)));
    __syncthreads();
    float *dst = P.scratch + (size_t)tile * kTileFloats;
    merge_groups<G, 0, ADJ>(regions, dst);
    merge_groups<G, 1, ADJ>(regions, dst);
    merge_groups<G, 2, ADJ>(regions, dst);
}

template <int R, int FMT, bool ADJ, bool AFF, int G>
cudaError_t launch_chunks_g(const P2GArgs &P, int grid, cudaStream_t s) {
    // The limit belongs to the kernel, not to the launch: every caller sets the
    // same value, the largest that a launch of this kernel needs (a solid phase's),
    // so that a host thread never lowers it between another's setting and launch.
    constexpr int limit = chunks_smem_bytes<R, FMT, ADJ, AFF, G>(true);
    static_assert(limit <= 227 * 1024, "P2G exceeds the shared memory of a CTA");
    const cudaError_t e = cudaFuncSetAttribute(k_p2g_chunks<R, FMT, ADJ, AFF, G>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
    if (e != cudaSuccess) return e;
    const int smem = chunks_smem_bytes<R, FMT, ADJ, AFF, G>(P.mass_abs != nullptr);
    k_p2g_chunks<R, FMT, ADJ, AFF, G><<<grid, 96 * G, smem, s>>>(P);
    return cudaGetLastError();
}

// Two groups (two CTAs of 6 warps on an SM) overlap one tile's prologue and
// merge with the other's work; four groups (one CTA of 12) give a tile twice the
// warps.  With fewer than about four tiles of 2048 particles per SM the last
// wave decides: the P2G call takes 62 us with 4 groups and 92 with 2 (33x29x45
// cells, 119 thousand particles, 27 modes), 200 and 210 (64^3, 863 thousand); on
// 128^3 and 3.8 million the kernel takes 697 us with 2 and 729 with 4.  A sparse
// phase has more tiles than its count says (half of 128^3 with 0.5 million: 661
// us with 4, 539 with 2); no call knows that.
constexpr int64_t kWideTiles = 152 * 4 * 2048;
template <int R, int FMT, bool ADJ, bool AFF = false>
cudaError_t launch_chunks(const P2GArgs &P, int grid, cudaStream_t s) {
    return P.count < kWideTiles ? launch_chunks_g<R, FMT, ADJ, AFF, 4>(P, grid, s)
                                : launch_chunks_g<R, FMT, ADJ, AFF, 2>(P, grid, s);
}

// Launchers of the instantiations, one per translation unit.
cudaError_t launch_chunks_f32(const P2GArgs &P, int R, int grid, cudaStream_t s);
cudaError_t launch_chunks_16(const P2GArgs &P, int fmt, int grid, cudaStream_t s);
cudaError_t launch_chunks_adj(const P2GArgs &P, int grid, cudaStream_t s);
cudaError_t launch_chunks_aff(const P2GArgs &P, int R, int grid, cudaStream_t s);

}  // namespace polypic
