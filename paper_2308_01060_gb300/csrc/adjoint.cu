// adjoint.cu -- adjoint (transposed) transfers for differentiating through
// steps of PolyPIC (constant map, single phase, FP32 coefficients).
//
// Forward, per particle p and face grid a (physical units, z = x_i - x_p):
//   P2G  m_ia  += mt W_ia,   mv_ia += mt sum_abc c_abc Fx_a Fy_b Fz_c
//   G2P  c'_abc = sum_i Gx_a Gy_b Gz_c v_ia,   x'_a = clamp(x_a + dt c'_000)
// with per-axis factors (t = particle offset from the middle node in cells,
// q = 1 - 4t^2, F^1 and phi the dimensionless closed forms of polypic_internal):
//   F0 = W, F1 = dx F^1, F2 = dx^2 phi (1, -2, 1)          (P2G, W f_a)
//   G0 = W, G1 = 4 F^1 / dx, G2 = (1, -2, 1) / (2 dx^2)   (fit, W f_a / d_a)
// and their x-derivatives (dt/dx = 1/dx):
//   dW/dt = (t - 1/2, -2t, t + 1/2)
//   dF^1/dt = (3q/8, (12t^2 - 3)/4, 3q/8)
//   dphi/dt = -t q (7 - 12 t^2) / 4,   dG2/dx = 0 (the quadratic fit weights
//   do not depend on t).
//
// G2P adjoint: mu_abc = lc'_abc (+ dt lx'_a on the constant mode if x'_a was
// not clamped);  lv_ia += sum_abc mu_abc G_a G_b G_c  (a P2G-shaped scatter,
// done by the deterministic P2G kernel);  lx_b += (lx'_b if not clamped)
// + sum_a sum_abc mu_abc sum_i d/dx_b(G_a G_b G_c) v_ia  (gathered here).
// P2G adjoint: lc_abc = mt sum_i F_a F_b F_c lmv_ia;  lx_b += mt sum_a sum_i
// [d/dx_b(W W W) lm_ia + sum_abc c_abc d/dx_b(F_a F_b F_c) lmv_ia].
#include <type_traits>

#include "adjoint.cuh"
#include "cp_async.cuh"
#include "p2g.cuh"

namespace polypic {

constexpr int kAdjThreads = 256;
// CTAs of an SM that a gather's registers are limited for.  A phase of at most
// one tile an SM (2048 particles each at 8 a cell) has no use for a second CTA,
// only for the registers: on 119 thousand particles (33x29x45 cells) the P2G
// adjoint of 8 modes takes 45 us with one and 53 with two, of 4 modes 38 and 47,
// the G2P adjoint with its scatter of 27 modes 97 and 111.  Larger phases take
// two (863 thousand particles: P2G adjoint of 8 modes 124 us, 157 with one; G2P
// adjoint of 27 modes 307, 319 with one), but for the P2G adjoint of 27 modes,
// which would spill 376 bytes a thread (262 -> 275 us).  One mode is small
// enough for two and, above two tiles an SM, three (2.9 million particles: P2G
// adjoint 210 -> 184 us; 364 thousand: 39 us with two, 51 with three).  A sparse
// phase has more tiles than its count says, so the grid's count as well (62
// thousand particles in half of 64^3, G2P adjoint of 27 modes: 133 us with one,
// 121 with two; grids up to 48^3 are below the line).
constexpr bool adj_few(int R, int64_t count, int64_t tiles) {
    return count <= (R == 1 ? 2 : 1) * 152 * 2048 && tiles <= 152 * 4;
}
template <int R, bool FEW> constexpr int g2p_adj_ctas() { return (R == 1 ? 2 : 1) + (FEW ? 0 : 1); }
template <int R, bool FEW> constexpr int p2g_adj_ctas() {
    return R == 27 ? 1 : g2p_adj_ctas<R, FEW>();
}
template <int A> struct ATile {
    static constexpr int X = A == 0 ? 11 : 10, Y = A == 1 ? 11 : 10, Z = A == 2 ? 7 : 6;
    static constexpr int N = X * Y * Z;
};
constexpr int kATileOff1 = ATile<0>::N, kATileOff2 = ATile<0>::N + ATile<1>::N;
constexpr int kATileFloats = ATile<0>::N + ATile<1>::N + ATile<2>::N;

struct AxisFac {
    float W[3], dW[3];    // W and dW/dx
    float F1[3], dF1[3];  // dimensionless F^1 and dF^1/dt
    float phi, dphi;      // phi and dphi/dt
    bool guard;
};

__device__ __forceinline__ AxisFac axis_fac(const Axis &ax) {
    AxisFac f;
    const float t = ax.t;
    const Stencil1D s = stencil_1d(t);
    const float q = (1.0f - 2.0f * t) * (1.0f + 2.0f * t);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        f.W[k] = s.W[k];
        f.F1[k] = s.F1[k];
    }
    f.dW[0] = t - 0.5f;
    f.dW[1] = -2.0f * t;
    f.dW[2] = t + 0.5f;
    f.dF1[0] = 0.375f * q;
    f.dF1[1] = (12.0f * t * t - 3.0f) * 0.25f;
    f.dF1[2] = 0.375f * q;
    f.phi = s.phi;
    f.dphi = -t * q * (7.0f - 12.0f * t * t) * 0.25f;
    f.guard = ax.guard;
    return f;
}

// P2G factor rows (physical) and their x-derivatives.
template <int D>
__device__ __forceinline__ void p2g_rows(const AxisFac &f, float dx, float inv_dx, float (&F)[D][3],
                                         float (&dF)[D][3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        F[0][k] = f.W[k];
        dF[0][k] = f.dW[k] * inv_dx;
    }
    if constexpr (D > 1) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            F[1][k] = dx * f.F1[k];
            dF[1][k] = f.dF1[k];
        }
    }
    if constexpr (D > 2) {
        const float p = dx * dx * f.phi, dp = dx * f.dphi;
        F[2][0] = p;
        F[2][1] = -2.0f * p;
        F[2][2] = p;
        dF[2][0] = dp;
        dF[2][1] = -2.0f * dp;
        dF[2][2] = dp;
    }
}

// Fit factor rows (physical) and their x-derivatives.
template <int D>
__device__ __forceinline__ void fit_rows_d(const AxisFac &f, float inv_dx, float (&G)[D][3],
                                           float (&dG)[D][3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        G[0][k] = f.W[k];
        dG[0][k] = f.dW[k] * inv_dx;
    }
    if constexpr (D > 1) {
        const float a = 4.0f * inv_dx, b = 4.0f * inv_dx * inv_dx;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            G[1][k] = a * f.F1[k];
            dG[1][k] = b * f.dF1[k];
        }
    }
    if constexpr (D > 2) {
        const float h = f.guard ? 0.0f : 0.5f * inv_dx * inv_dx;
        G[2][0] = h;
        G[2][1] = -2.0f * h;
        G[2][2] = h;
        dG[2][0] = dG[2][1] = dG[2][2] = 0.0f;
    }
}

// sum_abc mu_abc sum_i d/dx_b (X_a Y_b Z_c)(i) v(i) for b = x, y, z, with the
// contraction over x first, then y, then z, streamed over a.  A factor and its
// derivative meet the same operand, so the two run as one packed FP32 FMA (each
// half rounds as fmaf does).  ZERO2: the degree-2 derivative rows are 0 (the
// fit's), and their terms are left out: 126 of 648 FMAs of a component.
template <int R, int D, bool ZERO2, class Mu>
__device__ __forceinline__ void adj_position(const float (&X)[D][3], const float (&dX)[D][3],
                                             const float (&Y)[D][3], const float (&dY)[D][3],
                                             const float (&Z)[D][3], const float (&dZ)[D][3],
                                             const float (&v)[3][3][3], const Mu &mu, float &Dx,
                                             float &Dy, float &Dz) {
    auto bc = [](float f) { return make_float2(f, f); };
#pragma unroll
    for (int a = 0; a < D; ++a) {
        float U1[3][3], U1d[3][3];  // [ky][kz]
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
            for (int kz = 0; kz < 3; ++kz) {
                if (ZERO2 && a == 2) {
                    U1[ky][kz] = fmaf(X[a][0], v[0][ky][kz], fmaf(X[a][1], v[1][ky][kz], X[a][2] * v[2][ky][kz]));
                    U1d[ky][kz] = 0.0f;
                } else {
                    float2 t = __fmul2_rn(make_float2(X[a][2], dX[a][2]), bc(v[2][ky][kz]));
                    t = __ffma2_rn(make_float2(X[a][1], dX[a][1]), bc(v[1][ky][kz]), t);
                    t = __ffma2_rn(make_float2(X[a][0], dX[a][0]), bc(v[0][ky][kz]), t);
                    U1[ky][kz] = t.x;
                    U1d[ky][kz] = t.y;
                }
            }
#pragma unroll
        for (int b = 0; b < D; ++b) {
            float m[D];
#pragma unroll
            for (int c = 0; c < D; ++c) m[c] = has_mode(R, a, b, c) ? mu(a, b, c) : 0.0f;
#pragma unroll
            for (int kz = 0; kz < 3; ++kz) {
                float2 u;  // U1 contracted with Y_b and dY_b
                if (ZERO2 && b == 2) {
                    u = make_float2(fmaf(Y[b][0], U1[0][kz], fmaf(Y[b][1], U1[1][kz], Y[b][2] * U1[2][kz])), 0.0f);
                } else {
                    u = __fmul2_rn(make_float2(Y[b][2], dY[b][2]), bc(U1[2][kz]));
                    u = __ffma2_rn(make_float2(Y[b][1], dY[b][1]), bc(U1[1][kz]), u);
                    u = __ffma2_rn(make_float2(Y[b][0], dY[b][0]), bc(U1[0][kz]), u);
                }
                float2 M = make_float2(0.0f, 0.0f);  // the modes (a, b, *) with Z and dZ
#pragma unroll
                for (int c = 0; c < D; ++c)
                    if (has_mode(R, a, b, c)) {
                        if (ZERO2 && c == 2) M.x = fmaf(m[c], Z[c][kz], M.x);
                        else M = __ffma2_rn(bc(m[c]), make_float2(Z[c][kz], dZ[c][kz]), M);
                    }
                if (!(ZERO2 && a == 2)) {
                    const float ux = fmaf(Y[b][0], U1d[0][kz], fmaf(Y[b][1], U1d[1][kz], Y[b][2] * U1d[2][kz]));
                    Dx = fmaf(M.x, ux, Dx);
                }
                if (!(ZERO2 && b == 2)) Dy = fmaf(M.x, u.y, Dy);
                Dz = fmaf(M.y, u.x, Dz);
            }
        }
    }
}

// out(r) = sum_i X_a Y_b Z_c v(i) for the modes r = (a, b, c) of the set, handed
// out degree a by degree a (at most 9 values live).
template <int R, int D, class Out>
__device__ __forceinline__ void contract_modes(const float (&X)[D][3], const float (&Y)[D][3],
                                               const float (&Z)[D][3], const float (&v)[3][3][3],
                                               const Out &out) {
#pragma unroll
    for (int a = 0; a < D; ++a) {
        float U1[3][3], m[D][D];
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
            for (int kz = 0; kz < 3; ++kz)
                U1[ky][kz] = fmaf(X[a][0], v[0][ky][kz], fmaf(X[a][1], v[1][ky][kz], X[a][2] * v[2][ky][kz]));
#pragma unroll
        for (int b = 0; b < D; ++b) {
            float U2[3];
#pragma unroll
            for (int kz = 0; kz < 3; ++kz)
                U2[kz] = fmaf(Y[b][0], U1[0][kz], fmaf(Y[b][1], U1[1][kz], Y[b][2] * U1[2][kz]));
#pragma unroll
            for (int c = 0; c < D; ++c)
                m[b][c] = fmaf(Z[c][0], U2[0], fmaf(Z[c][1], U2[1], Z[c][2] * U2[2]));
        }
        out(a, m);
    }
}

// Stage the footprints (three face grids) of `src` around tile (tx, ty, tz).
__device__ __forceinline__ void stage_tile(const GridGeom &g, const float *const src[3], int ox,
                                           int oy, int oz, float *dst) {
    const int dims[3][3] = {{ATile<0>::X, ATile<0>::Y, ATile<0>::Z},
                            {ATile<1>::X, ATile<1>::Y, ATile<1>::Z},
                            {ATile<2>::X, ATile<2>::Y, ATile<2>::Z}};
    const int off[3] = {0, kATileOff1, kATileOff2};
    for (int a = 0; a < 3; ++a) {
        const int X = dims[a][0], Y = dims[a][1], Z = dims[a][2];
        const int dX = g.n[0] + (a == 0), dY = g.n[1] + (a == 1), dZ = g.n[2] + (a == 2);
        for (int i = threadIdx.x; i < X * Y * Z; i += kAdjThreads) {
            const int lx = i % X, ly = (i / X) % Y, lz = i / (X * Y);
            const int gx = ox + lx, gy = oy + ly, gz = oz + lz;
            float v = 0.0f;
            if (gx >= 0 && gx < dX && gy >= 0 && gy < dY && gz >= 0 && gz < dZ)
                v = src[a][((int64_t)gz * dY + gy) * dX + gx];
            dst[off[a] + i] = v;
        }
    }
}

template <int A>
__device__ __forceinline__ void read_stencil(const float *tile, int lx, int ly, int lz,
                                             float (&v)[3][3][3]) {
    const float *t = tile + (A == 0 ? 0 : A == 1 ? kATileOff1 : kATileOff2);
#pragma unroll
    for (int kz = 0; kz < 3; ++kz)
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
            for (int kx = 0; kx < 3; ++kx)
                v[kx][ky][kz] = t[((lz + kz) * ATile<A>::Y + (ly + ky)) * ATile<A>::X + lx + kx];
}

struct ParticleAxes {
    bool ok;
    int cell[3];
    Axis ctr[3], fce[3];
};

__device__ __forceinline__ ParticleAxes particle_axes(const GridGeom &g, float px, float py,
                                                      float pz, int tx, int ty, int tz) {
    ParticleAxes P;
    const float v[3] = {cell_coord(px, g.inv_dx), cell_coord(py, g.inv_dx), cell_coord(pz, g.inv_dx)};
    P.ok = coord_valid(v[0], g.n[0]) && coord_valid(v[1], g.n[1]) && coord_valid(v[2], g.n[2]);
    const int org[3] = {8 * tx, 8 * ty, 4 * tz}, ext[3] = {8, 8, 4};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        P.cell[b] = cell_index(v[b], g.n[b]);
        P.ok = P.ok && P.cell[b] >= org[b] && P.cell[b] < org[b] + ext[b];
        P.ctr[b] = axis_decide(v[b], false);
        P.fce[b] = axis_decide(v[b], true);
    }
    return P;
}

// ---------------------------------------------------------------- coefficient stages
// A thread's R coefficients of one component ([mode][thread], its own column
// only): two stages of shared memory filled by cp.async one component ahead of
// their use: loaded into registers when a component began, they cost a memory
// latency each time with 8 warps an SM to hide it.
template <int R> struct CoeffStage {
    float *at;      // the thread's column of the stage in use
    int other = R * kAdjThreads;  // the other stage, from here
    __device__ __forceinline__ CoeffStage(float *smem) : at(smem + threadIdx.x) {}
    __device__ __forceinline__ void fill(bool ahead, const float *src, int64_t cnt) {
        float *to = at + (ahead ? other : 0);
#pragma unroll
        for (int r = 0; r < R; ++r, src += cnt) cp_async4(to + r * kAdjThreads, src);
    }
    __device__ __forceinline__ void next() {
        at += other;
        other = -other;
    }
    __device__ __forceinline__ float operator()(int a, int b, int c) const {
        return at[mode_index(a, b, c) * kAdjThreads];
    }
};
template <int R> constexpr int stage_bytes() { return 2 * R * kAdjThreads * (int)sizeof(float); }

// ---------------------------------------------------------------- G2P adjoint gather
template <int R, int A>
__device__ __forceinline__ void g2p_adj_component(const AdjG2PArgs &G, const ParticleAxes &pa,
                                                  const float *tile, int ox, int oy, int oz,
                                                  uint32_t j, float px_a, const CoeffStage<R> &bar,
                                                  float (&lx)[3]) {
    constexpr int D = axis_degrees(R);
    const Axis &ax = A == 0 ? pa.fce[0] : pa.ctr[0];
    const Axis &ay = A == 1 ? pa.fce[1] : pa.ctr[1];
    const Axis &az = A == 2 ? pa.fce[2] : pa.ctr[2];
    float X[D][3], dX[D][3], Y[D][3], dY[D][3], Z[D][3], dZ[D][3];
    fit_rows_d<D>(axis_fac(ax), G.inv_dx, X, dX);
    fit_rows_d<D>(axis_fac(ay), G.inv_dx, Y, dY);
    fit_rows_d<D>(axis_fac(az), G.inv_dx, Z, dZ);
    float v[3][3][3];
    read_stencil<A>(tile, ax.base - ox, ay.base - oy, az.base - oz, v);
    // the forward velocity fit (constant mode) decides whether x'_A was clamped
    float c0 = 0.0f;
#pragma unroll
    for (int kz = 0; kz < 3; ++kz)
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
            const float yz = Y[0][ky] * Z[0][kz];
#pragma unroll
            for (int kx = 0; kx < 3; ++kx) c0 = fmaf(X[0][kx] * yz, v[kx][ky][kz], c0);
        }
    const float xn = fmaf(G.dt, c0, px_a);
    const bool clamped = xn < G.g.lo[A] || xn > G.g.hi[A];
    const float lxo = __ldg(G.bar_x[A] + j);
    // the effective coefficient adjoint mu is bar c' but for the constant mode,
    // which also gets the advection's term: only that mode is written for the
    // scatter, which reads the others where they are (all 27 written and read
    // again were 560 MB at 863 thousand particles, now 311)
    const float mu0 = clamped ? bar(0, 0, 0) : fmaf(G.dt, lxo, bar(0, 0, 0));
    G.mu0[(int64_t)A * G.count + j] = mu0;
    auto mu = [&](int a, int b, int c) { return a + b + c == 0 ? mu0 : bar(a, b, c); };
    float Dx = 0.0f, Dy = 0.0f, Dz = 0.0f;
    adj_position<R, D, true>(X, dX, Y, dY, Z, dZ, v, mu, Dx, Dy, Dz);
    lx[0] += Dx;
    lx[1] += Dy;
    lx[2] += Dz;
    if (!clamped) lx[A] += lxo;
}

template <int R, bool FEW>
__global__ void __launch_bounds__(kAdjThreads, g2p_adj_ctas<R, FEW>()) k_g2p_adjoint(AdjG2PArgs G) {
    __shared__ float s_tile[kATileFloats];
    const GridGeom &g = G.g;
    const uint32_t tile = blockIdx.x;
    const uint32_t jb = G.cell_start[tile * 256], je = G.cell_start[tile * 256 + 256];
    if (jb == je) return;
    const int tx = (int)(tile % (uint32_t)g.tiles[0]);
    const int ty = (int)((tile / (uint32_t)g.tiles[0]) % (uint32_t)g.tiles[1]);
    const int tz = (int)(tile / ((uint32_t)g.tiles[0] * (uint32_t)g.tiles[1]));
    const int ox = 8 * tx - 1, oy = 8 * ty - 1, oz = 4 * tz - 1;
    stage_tile(g, G.vel, ox, oy, oz, s_tile);
    __syncthreads();
    // software pipeline: the next particle's index and position load while
    // this one is computed, every component's coefficients one ahead
    extern __shared__ float s_stage[];
    CoeffStage<R> bar(s_stage);
    const int64_t cnt = G.count;
    uint32_t j = jb + threadIdx.x;
    uint32_t pn = j < je ? G.perm[j] : 0u;
    float nx = 0.0f, ny = 0.0f, nz = 0.0f;
    if (j < je) {
        nx = G.x[0][pn];
        ny = G.x[1][pn];
        nz = G.x[2][pn];
        bar.fill(false, G.bar_c + j, cnt);
    }
    cp_async_commit();
    for (; j < je; j += kAdjThreads) {
        const uint32_t p = pn;
        const float px = nx, py = ny, pz = nz;
        const uint32_t jn = j + kAdjThreads;
        if (jn < je) {
            pn = G.perm[jn];
            nx = G.x[0][pn];
            ny = G.x[1][pn];
            nz = G.x[2][pn];
        }
        const ParticleAxes pa = particle_axes(g, px, py, pz, tx, ty, tz);
        float lx[3] = {0.0f, 0.0f, 0.0f};
        auto component = [&](auto axis, float pos) {
            constexpr int A = decltype(axis)::value;
            if (A < 2) bar.fill(true, G.bar_c + (int64_t)(A + 1) * R * cnt + j, cnt);
            else if (jn < je) bar.fill(true, G.bar_c + jn, cnt);
            cp_async_commit();
            cp_async_wait<1>();
            if (pa.ok) g2p_adj_component<R, A>(G, pa, s_tile, ox, oy, oz, j, pos, bar, lx);
            else G.mu0[(int64_t)A * cnt + j] = 0.0f;
            bar.next();
        };
        component(std::integral_constant<int, 0>{}, px);
        component(std::integral_constant<int, 1>{}, py);
        component(std::integral_constant<int, 2>{}, pz);
        if (!pa.ok) atomicOr(G.status, kFlagOutOfDomain);
        if (G.accumulate) {  // three loads, then three stores
            const float o0 = G.out_x[0][p], o1 = G.out_x[1][p], o2 = G.out_x[2][p];
            lx[0] += o0;
            lx[1] += o1;
            lx[2] += o2;
        }
#pragma unroll
        for (int b = 0; b < 3; ++b) G.out_x[b][p] = lx[b];
    }
}

// ---------------------------------------------------------------- P2G adjoint gather
template <int R, int A>
__device__ __forceinline__ void p2g_adj_component(const AdjP2GArgs &Q, const ParticleAxes &pa,
                                                  const float *tile_m, const float *tile_v, int ox,
                                                  int oy, int oz, uint32_t p, float mt,
                                                  const CoeffStage<R> &coef,
                                                  const CoeffStage<R> &old, float (&lx)[3]) {
    constexpr int D = axis_degrees(R);
    const Axis &ax = A == 0 ? pa.fce[0] : pa.ctr[0];
    const Axis &ay = A == 1 ? pa.fce[1] : pa.ctr[1];
    const Axis &az = A == 2 ? pa.fce[2] : pa.ctr[2];
    const AxisFac fx = axis_fac(ax), fy = axis_fac(ay), fz = axis_fac(az);
    float X[D][3], dX[D][3], Y[D][3], dY[D][3], Z[D][3], dZ[D][3];
    p2g_rows<D>(fx, Q.dx, Q.inv_dx, X, dX);
    p2g_rows<D>(fy, Q.dx, Q.inv_dx, Y, dY);
    p2g_rows<D>(fz, Q.dx, Q.inv_dx, Z, dZ);
    const int lx0 = ax.base - ox, ly0 = ay.base - oy, lz0 = az.base - oz;
    const int64_t cnt = Q.count;
    float *__restrict__ cout = Q.out_c + (int64_t)A * R * cnt + p;
    float Dx = 0.0f, Dy = 0.0f, Dz = 0.0f;
    {  // position terms of the mass, through the weights
        float lm[3][3][3];
        read_stencil<A>(tile_m, lx0, ly0, lz0, lm);
        float Wx[1][3], dWx[1][3], Wy[1][3], dWy[1][3], Wz[1][3], dWz[1][3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            Wx[0][k] = X[0][k]; dWx[0][k] = dX[0][k];
            Wy[0][k] = Y[0][k]; dWy[0][k] = dY[0][k];
            Wz[0][k] = Z[0][k]; dWz[0][k] = dZ[0][k];
        }
        auto one = [](int, int, int) { return 1.0f; };
        adj_position<1, 1, false>(Wx, dWx, Wy, dWy, Wz, dWz, lm, one, Dx, Dy, Dz);
    }
    float lmv[3][3][3];
    read_stencil<A>(tile_v, lx0, ly0, lz0, lmv);
    contract_modes<R, D>(X, Y, Z, lmv, [&](int a, const float (&m)[D][D]) {
#pragma unroll
        for (int b = 0; b < D; ++b)
#pragma unroll
            for (int cc = 0; cc < D; ++cc)
                if (has_mode(R, a, b, cc))
                    cout[mode_index(a, b, cc) * cnt] =
                        Q.accumulate ? fmaf(mt, m[b][cc], old(a, b, cc)) : mt * m[b][cc];
    });
    // position terms of the momentum, through the modes
    adj_position<R, D, false>(X, dX, Y, dY, Z, dZ, lmv, coef, Dx, Dy, Dz);
    lx[0] = fmaf(mt, Dx, lx[0]);
    lx[1] = fmaf(mt, Dy, lx[1]);
    lx[2] = fmaf(mt, Dz, lx[2]);
}

// With 27 modes, tiles of at most this many particles are walked in memory order
// (below): the three adjoints of 863 thousand particles take 577 us instead of
// 581.  With fewer modes the list costs more than it gives (P2G adjoint of the
// same particles without it: 8 modes 129 -> 127 us, 4 modes 119 -> 109, one mode
// 71 -> 66).
constexpr int kAdjList = 3072;
constexpr int kAdjWords = 128;  // bitmap words: a window of 4096 indices

// The tile's particle indices perm[jb .. je) into `idx` in ascending order:
// those inside a window of 4096 around the median of three samples ranked by a
// bitmap, the others behind them in any order (every particle reads and writes
// only its own entries, so the order changes no result).  The arrays are in
// the slot order of the step before: ascending indices read and write whole
// sectors of their 162 coefficient rows where slot order, moved by a rank
// wherever a particle left or entered a cell, touched them in pieces.  A perm
// that names a particle twice ranks it once; the entries this leaves over keep
// the particle of their slot.
__device__ __forceinline__ void list_in_memory_order(const uint32_t *__restrict__ perm, uint32_t jb,
                                                     uint32_t je, uint32_t *idx, uint32_t *bits) {
    uint32_t *pre = bits + kAdjWords, *far = pre + kAdjWords;
    const uint32_t n = je - jb;
    const uint32_t a = perm[jb + n / 4], b = perm[jb + n / 2], c = perm[jb + (n - 1) - n / 4];
    const uint32_t mid = max(min(a, b), min(max(a, b), c));
    constexpr uint32_t W = 32 * kAdjWords;
    const uint32_t base = mid > W / 2 ? (mid - W / 2) & ~31u : 0u;
    for (int i = threadIdx.x; i < kAdjWords; i += blockDim.x) bits[i] = 0;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
        const uint32_t p = perm[jb + i], off = p - base;
        idx[i] = p;
        if (off < W) atomicOr(&bits[off >> 5], 1u << (off & 31u));
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        uint32_t run = 0;
        for (int w0 = 0; w0 < kAdjWords; w0 += 32) {
            const uint32_t v = (uint32_t)__popc(bits[w0 + lane]);
            uint32_t x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            pre[w0 + lane] = run + x - v;
            run += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) *far = run;
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
        const uint32_t p = perm[jb + i], off = p - base;
        const uint32_t at = off < W ? pre[off >> 5] + (uint32_t)__popc(bits[off >> 5] &
                                                                     ((1u << (off & 31u)) - 1u))
                                    : atomicAdd(far, 1u);
        if (at < n) idx[at] = p;
    }
    __syncthreads();
}

template <int R, bool FEW>
__global__ void __launch_bounds__(kAdjThreads, p2g_adj_ctas<R, FEW>()) k_p2g_adjoint(AdjP2GArgs Q) {
    extern __shared__ float s_adj[];
    constexpr bool kList = R == 27;
    __shared__ uint32_t s_idx[kList ? kAdjList : 1], s_bits[kList ? 2 * kAdjWords + 1 : 1];
    float *tile_m = s_adj, *tile_v = s_adj + kATileFloats;
    const GridGeom &g = Q.g;
    const uint32_t tile = blockIdx.x;
    const uint32_t jb = Q.cell_start[tile * 256], je = Q.cell_start[tile * 256 + 256];
    if (jb == je) return;
    const int tx = (int)(tile % (uint32_t)g.tiles[0]);
    const int ty = (int)((tile / (uint32_t)g.tiles[0]) % (uint32_t)g.tiles[1]);
    const int tz = (int)(tile / ((uint32_t)g.tiles[0] * (uint32_t)g.tiles[1]));
    const int ox = 8 * tx - 1, oy = 8 * ty - 1, oz = 4 * tz - 1;
    stage_tile(g, Q.lm, ox, oy, oz, tile_m);
    stage_tile(g, Q.lmv, ox, oy, oz, tile_v);
    const bool listed = kList && je - jb <= (uint32_t)kAdjList;  // CTA-uniform
    if (listed) list_in_memory_order(Q.perm, jb, je, s_idx, s_bits);
    else __syncthreads();
    auto particle = [&](uint32_t j) { return listed ? s_idx[j - jb] : Q.perm[j]; };
    // software pipeline: the next particle's index, position and mass load
    // while this one is computed, every component's coefficients one ahead, and
    // its old outputs when they are added to (loaded where they are used, they
    // cost a component three memory latencies)
    CoeffStage<R> coef(s_adj + 2 * kATileFloats);
    CoeffStage<R> old(s_adj + 2 * kATileFloats + 2 * R * kAdjThreads);
    const bool add = Q.accumulate;
    const int64_t cnt = Q.count;
    uint32_t j = jb + threadIdx.x;
    uint32_t pn = j < je ? particle(j) : 0u;
    float nx = 0.0f, ny = 0.0f, nz = 0.0f, nm = 0.0f;
    if (j < je) {
        nx = Q.x[0][pn];
        ny = Q.x[1][pn];
        nz = Q.x[2][pn];
        nm = Q.mass[pn] + (Q.mass_abs ? Q.mass_abs[pn] : 0.0f);
        coef.fill(false, Q.coeff + pn, cnt);
        if (add) old.fill(false, Q.out_c + pn, cnt);
    }
    cp_async_commit();
    for (; j < je; j += kAdjThreads) {
        const uint32_t p = pn;
        const float px = nx, py = ny, pz = nz, mt = nm;
        const bool more = j + kAdjThreads < je;
        if (more) {
            pn = particle(j + kAdjThreads);
            nx = Q.x[0][pn];
            ny = Q.x[1][pn];
            nz = Q.x[2][pn];
            nm = Q.mass[pn] + (Q.mass_abs ? Q.mass_abs[pn] : 0.0f);
        }
        const ParticleAxes pa = particle_axes(g, px, py, pz, tx, ty, tz);
        float lx[3] = {0.0f, 0.0f, 0.0f};
        auto component = [&](auto axis) {
            constexpr int A = decltype(axis)::value;
            if (A < 2 || more) {
                const int64_t at = A < 2 ? (int64_t)(A + 1) * R * cnt + p : (int64_t)pn;
                coef.fill(true, Q.coeff + at, cnt);
                if (add) old.fill(true, Q.out_c + at, cnt);
            }
            cp_async_commit();
            cp_async_wait<1>();
            if (pa.ok) p2g_adj_component<R, A>(Q, pa, tile_m, tile_v, ox, oy, oz, p, mt, coef, old, lx);
            coef.next();
            old.next();
        };
        component(std::integral_constant<int, 0>{});
        component(std::integral_constant<int, 1>{});
        component(std::integral_constant<int, 2>{});
        if (!pa.ok) {
            atomicOr(Q.status, kFlagOutOfDomain);
            for (int a = 0; a < 3; ++a)
                for (int r = 0; r < R; ++r) {
                    float *o = Q.out_c + ((int64_t)a * R + r) * Q.count + p;
                    if (!Q.accumulate) *o = 0.0f;
                }
        }
        if (Q.accumulate) {  // three loads, then three stores
            const float o0 = Q.out_x[0][p], o1 = Q.out_x[1][p], o2 = Q.out_x[2][p];
            lx[0] += o0;
            lx[1] += o1;
            lx[2] += o2;
        }
#pragma unroll
        for (int b = 0; b < 3; ++b) Q.out_x[b][p] = lx[b];
    }
}

// ---------------------------------------------------------------- drivers
size_t adjoint_scratch_bytes(int64_t count) {
    return (size_t)count * 3 * sizeof(float) + 512;
}

template <int R>
static cudaError_t launch_g2p_adjoint(const AdjG2PArgs &G, int64_t tiles, cudaStream_t s) {
    constexpr int smem = stage_bytes<R>();
    const auto kernel = adj_few(R, G.count, tiles) ? k_g2p_adjoint<R, true> : k_g2p_adjoint<R, false>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    kernel<<<(int)tiles, kAdjThreads, smem, s>>>(G);
    return cudaGetLastError();
}

template <int R>
static cudaError_t launch_p2g_adjoint(const AdjP2GArgs &Q, int64_t tiles, cudaStream_t s) {
    constexpr int tiles_bytes = 2 * kATileFloats * (int)sizeof(float);
    constexpr int limit = tiles_bytes + 2 * stage_bytes<R>();  // the kernel's, whatever the call
    static_assert(limit <= 200 * 1024, "the P2G adjoint exceeds the shared memory of a CTA");
    const int smem = tiles_bytes + (Q.accumulate ? 2 : 1) * stage_bytes<R>();
    const bool few = R == 27 || adj_few(R, Q.count, tiles);
    const auto kernel = few ? k_p2g_adjoint<R, true> : k_p2g_adjoint<R, R == 27>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
    if (e != cudaSuccess) return e;
    kernel<<<(int)tiles, kAdjThreads, smem, s>>>(Q);
    return cudaGetLastError();
}

cudaError_t adjoint_g2p(const GridGeom &g, int64_t num_keys, int R, float dx,
                        const polypic_grid *grid, const polypic_particles *in, float dt,
                        const polypic_particles *bar_out, polypic_grid *bar_grid,
                        polypic_particles *bar_in, bool accumulate, uint32_t *status,
                        Workspace &ws, cudaStream_t s) {
    const int64_t tiles = num_keys / 256;
    if (in->count == 0) {  // nothing scatters: the grid adjoint is 0 (or unchanged)
        if (!accumulate)
            for (int a = 0; a < 3; ++a) {
                const size_t n = (size_t)(g.n[0] + (a == 0)) * (g.n[1] + (a == 1)) * (g.n[2] + (a == 2));
                cudaError_t e = cudaMemsetAsync(bar_grid->vel[a], 0, n * sizeof(float), s);
                if (e != cudaSuccess) return e;
            }
        return cudaSuccess;
    }
    float *mu0 = ws.take<float>((size_t)in->count * 3);
    P2GArgs P{};
    P.scratch = ws.take<float>((size_t)tiles * kTileFloats);
    P.tile_live = ws.take<uint8_t>((size_t)tiles);
    if (ws.overflow) return cudaErrorInvalidValue;

    AdjG2PArgs G{};
    G.g = g;
    G.count = in->count;
    G.dt = dt;
    G.inv_dx = 1.0f / dx;
    for (int a = 0; a < 3; ++a) {
        G.vel[a] = grid->vel[a];
        G.x[a] = in->x[a];
        G.bar_x[a] = bar_out->x[a];
        G.out_x[a] = bar_in->x[a];
    }
    G.bar_c = static_cast<const float *>(bar_out->coeff);
    G.perm = in->perm;
    G.cell_start = in->cell_start;
    G.mu0 = mu0;
    G.status = status;
    G.accumulate = accumulate;
    cudaError_t e = cudaErrorInvalidValue;
    if (R == 1) e = launch_g2p_adjoint<1>(G, tiles, s);
    if (R == 4) e = launch_g2p_adjoint<4>(G, tiles, s);
    if (R == 8) e = launch_g2p_adjoint<8>(G, tiles, s);
    if (R == 27) e = launch_g2p_adjoint<27>(G, tiles, s);
    if (e != cudaSuccess) return e;

    P.g = g;
    P.count = in->count;
    P.x = in->x[0];
    P.y = in->x[1];
    P.z = in->x[2];
    P.perm = in->perm;
    P.cell_start = in->cell_start;
    P.status = status;
    P.nblocks = (uint32_t)(num_keys / 32);
    P.s1 = P.s2 = 1.0f;  // the scatter's fit rows carry their own 1/dx powers
    P.mu = static_cast<const float *>(bar_out->coeff);
    P.mu0 = mu0;
    P.inv_dx = 1.0f / dx;
    P.inv_dx2 = 1.0f / (dx * dx);
    return p2g_adjoint_scatter(P, bar_grid->vel, accumulate, R, s);
}

cudaError_t adjoint_p2g(const GridGeom &g, int64_t num_keys, int R, float dx,
                        const polypic_particles *in, const polypic_grid *bar_grid,
                        polypic_particles *bar_in, bool accumulate, uint32_t *status,
                        Workspace &ws, cudaStream_t s) {
    (void)ws;
    if (in->count == 0) return cudaSuccess;
    AdjP2GArgs Q{};
    Q.g = g;
    Q.count = in->count;
    Q.dx = dx;
    Q.inv_dx = 1.0f / dx;
    for (int a = 0; a < 3; ++a) {
        Q.lm[a] = bar_grid->mass[a];
        Q.lmv[a] = bar_grid->mom[a];
        Q.x[a] = in->x[a];
        Q.out_x[a] = bar_in->x[a];
    }
    Q.mass = in->mass;
    Q.mass_abs = in->mass_abs;
    Q.coeff = static_cast<const float *>(in->coeff);
    Q.out_c = static_cast<float *>(bar_in->coeff);
    Q.perm = in->perm;
    Q.cell_start = in->cell_start;
    Q.status = status;
    Q.accumulate = accumulate;
    const int64_t tiles = num_keys / 256;
    if (R == 1) return launch_p2g_adjoint<1>(Q, tiles, s);
    if (R == 4) return launch_p2g_adjoint<4>(Q, tiles, s);
    if (R == 8) return launch_p2g_adjoint<8>(Q, tiles, s);
    if (R == 27) return launch_p2g_adjoint<27>(Q, tiles, s);
    return cudaErrorInvalidValue;
}

}  // namespace polypic
