// pcg.cu -- pressure projection of the fluid grid velocity.
//
// The paper delegates the pressure solve to the host simulator (Section 3);
// this is the stated minimal form.  Cells holding fluid particles are fluid;
// other cells have p = 0; walls have zero normal velocity.  For a fluid cell c
//   sum_{non-wall neighbours n} (p_c - p_n) = -(rho dx^2 / dt) div_c,
//   div_c = sum_a (v_a(c + e_a) - v_a(c)) / dx,
// solved by conjugate gradients with FP32 vectors and FP64 dot products and
// norms (two-stage deterministic reductions), preconditioned by one
// multigrid V-cycle; then v_a -= dt / (rho dx) (p_hi - p_lo) on every non-wall
// face next to a fluid cell.  alpha and beta are formed on the device with the
// dot products; the host reads the residual norm every kCheckEvery iterations.
//
// The V-cycle (an aggregation multigrid): a coarse cell is the 2x2x2 block of
// fine cells, fluid if any child is; the coarse operator is the Galerkin
// product P^T A P with P the injection of a coarse value into its fluid
// children, so every level is again a 7-point operator (diagonal and one
// coupling per +x/+y/+z face).  Two damped-Jacobi sweeps (omega 2/3) from zero
// before the coarse correction and two after it, the residual restricted by
// P^T, the coarsest level (at most 512 cells) swept 32 times in one CTA.  The
// cycle is a fixed symmetric linear operator, positive definite because the
// sweeps converge and the Galerkin correction is an A-orthogonal projection,
// so CG keeps its guarantees.
//
// Launches: the large levels (more than kMgSmall cells, and always the finest)
// run one kernel per pass over a list of their fluid cells, in ascending order;
// all smaller levels run in one CTA from shared memory.  The working set stays in L2
// (60 MB at 128^3); a pass is bound by its loads' latency and by launching.
// The grid update of 128^3 with 476 thousand fluid cells, 24 iterations, takes
// 1.97 ms; 4.68 ms before, with a thread per cell of the box on every level,
// 23 launches per iteration and the coarsest level's operator read from memory
// on each of its 32 sweeps.
#include <algorithm>
#include <cmath>
#include <new>

#include "pcg.cuh"

namespace polypic {

constexpr int kPcgThreads = 256;
constexpr int kPcgMaxBlocks = 1024;
constexpr int kCheckEvery = 8;

struct PcgBuffers {
    float *x, *r, *z, *d, *d2, *Ap, *diag;  // d / d2: directions (ping-pong)
    uint8_t *fluid;
    double *sums, *rr;  // block sums of the running kernel; of |r|^2
    double *scal;       // the scalars named by the enum below
    uint32_t *arrived;  // blocks of the running kernel that have left their sum
};

// scal[]: |r|^2 and |b|^2 for the host, r . z by the iteration's parity, and
// CG's alpha and beta (rounded to FP32)
enum { kRr = 0, kBb = 1, kRz = 3, kAlpha = 5, kBeta = 6 };

__device__ __forceinline__ int64_t cidx(const GridGeom &g, int i, int j, int k) {
    return ((int64_t)k * g.n[1] + j) * g.n[0] + i;
}

// Sum over the block, in a fixed order; the value is valid in thread 0.  FP64
// adds are the cost (a warp's takes the SM's FP64 unit 16 cycles or so): one
// warp adds the 8 warps' values and shuffles, 12 of them a block where a
// shuffle tree in every warp takes 48 (k_mg_sweep 9.2 -> 8.4 us at 128^3).
__device__ __forceinline__ double block_sum(double a) {
    __shared__ double sa[kPcgThreads];
    __syncthreads();  // sa may still be read from the block's last sum
    sa[threadIdx.x] = a;
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int i = 1; i < kPcgThreads / 32; ++i) a += sa[threadIdx.x + 32 * i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    }
    return a;
}

// Total of nb block sums in a fixed order; valid in thread 0.
__device__ __forceinline__ double block_total(const double *sums, int nb) {
    double a = 0.0;
    for (int i = threadIdx.x; i < nb; i += kPcgThreads) a += sums[i];
    return block_sum(a);
}

// Sum of `a` over the grid into *out: the block that arrives last adds the
// block sums, in block order whatever the order of arrival, so that the total
// needs no launch of its own and no block waits for another.  Its thread 0
// also calls done(total): the FP64 quotients of CG are formed there, once,
// instead of by every thread that uses them (k_apply 10.9 -> 9.7, k_update 8.0
// -> 6.6, k_mg_sweep 8.3 -> 8.9 us at 128^3).
template <class Done>
__device__ __forceinline__ void grid_sum(double a, const PcgBuffers &B, const Done &done) {
    __shared__ bool last;
    a = block_sum(a);
    if (threadIdx.x == 0) {
        B.sums[blockIdx.x] = a;
        __threadfence();
        last = atomicInc(B.arrived, gridDim.x - 1) == gridDim.x - 1;  // wraps to 0
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const volatile double *sums = B.sums;
    double t = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += kPcgThreads) t += sums[i];
    t = block_sum(t);
    if (threadIdx.x == 0) done(t);
}

// r . z of iteration `odd`, and beta of the direction that follows (0 if the
// previous r . z is 0; the first direction has none and ignores it).
__device__ __forceinline__ void put_rz(const PcgBuffers &B, int odd, double rz) {
    const double prev = B.scal[kRz + (odd ^ 1)];
    B.scal[kRz + odd] = rz;
    B.scal[kBeta] = prev == 0.0 ? 0.0f : (float)(rz / prev);
}

__global__ void __launch_bounds__(kPcgThreads) k_total(const double *sums, int nb, double *out) {
    const double t = block_total(sums, nb);
    if (threadIdx.x == 0) *out = t;
}

// ---------------------------------------------------------------- multigrid levels
constexpr int kMgMaxLevels = 12;
constexpr int kMgCoarsest = 512;      // cells of the level swept in one CTA
constexpr int kMgCoarseSweeps = 32;
constexpr float kMgOmega = 2.0f / 3.0f;
// Levels of at most this many cells run in one CTA (16^3 fits): a thread keeps
// the operator of its five cells of the first one in registers, 64 of them at
// 1024 threads (the shared memory would hold more).
constexpr int64_t kMgSmall = 4608;
constexpr int kMgSmallThreads = 1024;
// All the shared memory a CTA can have.  The levels of 128^3 take 64 KB, no
// grid's more than 112 KB (thin ones, whose levels shrink least).
constexpr int kMgSmallLimit = 227 * 1024;
constexpr int kListTile = 2048;  // cells per CTA of the list's compaction

// One level of the hierarchy.  Level 0 is the fine system: couplings are -1
// between fluid neighbours (ox == nullptr).  Coarse levels store the Galerkin
// diagonal and the coupling of each cell to its +x, +y, +z neighbour.
struct MgLevel {
    int n[3];
    int64_t cells;
    uint8_t *fluid;
    float *diag, *wd, *ox, *oy, *oz;  // wd = omega / diag, the damped Jacobi scale
    float *x, *b, *t;
    // the large levels' fluid cells in ascending order, the coarse cell of each,
    // and their number; cell info of the finest level (see kInfo*)
    uint32_t *idx, *par, *count, *blocks;
    uint16_t *info;
};

// Info word of a finest-level cell: bits 0..5 a fluid neighbour across -x, +x,
// -y, +y, -z, +z, bits 6..8 the diagonal (number of non-wall faces), bit 9
// fluid, bits 10..12 the parity of i, j, k.
constexpr unsigned kInfoFluid = 1u << 9;
__device__ __forceinline__ float info_diag(unsigned w) { return (float)((w >> 6) & 7u); }

__host__ __device__ inline int mg_coarse_dim(int n) { return (n + 1) / 2; }

// Coupling of fluid cell c to neighbour m across face (axis a, side +1/-1).
__device__ __forceinline__ float mg_off(const MgLevel &L, int64_t c, int64_t m, int a, int side) {
    if (!L.ox) return L.fluid[m] ? -1.0f : 0.0f;
    const float *o = a == 0 ? L.ox : (a == 1 ? L.oy : L.oz);
    return side > 0 ? o[c] : o[m];
}

// (A v)(c) for fluid cell c at (i, j, k); v(m, i, j, k) gives the vector at
// cell m with coordinates (i, j, k) (called for c and its in-domain
// neighbours, so no functor divides an index).
template <class V>
__device__ __forceinline__ float mg_apply(const MgLevel &L, int64_t c, int i, int j, int k,
                                          const V &v) {
    float s = L.diag[c] * v(c, i, j, k);
    const int64_t sx = 1, sy = L.n[0], sz = (int64_t)L.n[0] * L.n[1];
    if (i > 0) s = fmaf(mg_off(L, c, c - sx, 0, -1), v(c - sx, i - 1, j, k), s);
    if (i < L.n[0] - 1) s = fmaf(mg_off(L, c, c + sx, 0, +1), v(c + sx, i + 1, j, k), s);
    if (j > 0) s = fmaf(mg_off(L, c, c - sy, 1, -1), v(c - sy, i, j - 1, k), s);
    if (j < L.n[1] - 1) s = fmaf(mg_off(L, c, c + sy, 1, +1), v(c + sy, i, j + 1, k), s);
    if (k > 0) s = fmaf(mg_off(L, c, c - sz, 2, -1), v(c - sz, i, j, k - 1), s);
    if (k < L.n[2] - 1) s = fmaf(mg_off(L, c, c + sz, 2, +1), v(c + sz, i, j, k + 1), s);
    return s;
}

// Cell coordinates of a linear index (32-bit division where the index fits).
__device__ __forceinline__ void cell_ijk(int64_t c, int n0, int n1, int &i, int &j, int &k) {
    if (c < 0x7fffffffLL) {
        const uint32_t u = (uint32_t)c, q = u / (uint32_t)n0;
        i = (int)(u - q * (uint32_t)n0);
        j = (int)(q % (uint32_t)n1);
        k = (int)(q / (uint32_t)n1);
    } else {
        const int64_t q = c / n0;
        i = (int)(c - q * n0);
        j = (int)(q % n1);
        k = (int)(q / n1);
    }
}

__device__ __forceinline__ void mg_ijk(const MgLevel &L, int64_t c, int &i, int &j, int &k) {
    cell_ijk(c, L.n[0], L.n[1], i, j, k);
}

#define MG_CELLS(L, c) \
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < (L).cells; \
         c += (int64_t)gridDim.x * blockDim.x)

// Coarse level from fine: fluid flags, Galerkin diagonal and couplings.
__global__ void __launch_bounds__(kPcgThreads) k_mg_coarsen(MgLevel F, MgLevel C) {
    MG_CELLS(C, cc) {
        int I, J, K;
        mg_ijk(C, cc, I, J, K);
        bool fl = false;
        float d = 0.0f, ox = 0.0f, oy = 0.0f, oz = 0.0f;
        for (int q = 0; q < 8; ++q) {
            const int a = q & 1, b = (q >> 1) & 1, e = q >> 2;
            const int i = 2 * I + a, j = 2 * J + b, k = 2 * K + e;
            if (i >= F.n[0] || j >= F.n[1] || k >= F.n[2]) continue;
            const int64_t c = ((int64_t)k * F.n[1] + j) * F.n[0] + i;
            if (!F.fluid[c]) continue;
            fl = true;
            d += F.diag[c];
            // the child's +x / +y / +z couplings: inside the block they fold
            // into the diagonal (both orderings), across it they couple blocks
            if (i + 1 < F.n[0]) {
                const float o = mg_off(F, c, c + 1, 0, +1);
                if (a == 0) d += 2.0f * o; else ox += o;
            }
            if (j + 1 < F.n[1]) {
                const float o = mg_off(F, c, c + F.n[0], 1, +1);
                if (b == 0) d += 2.0f * o; else oy += o;
            }
            if (k + 1 < F.n[2]) {
                const float o = mg_off(F, c, c + (int64_t)F.n[0] * F.n[1], 2, +1);
                if (e == 0) d += 2.0f * o; else oz += o;
            }
        }
        C.fluid[cc] = fl ? 1 : 0;
        C.diag[cc] = fl ? d : 1.0f;
        C.wd[cc] = fl ? kMgOmega / d : 0.0f;
        C.ox[cc] = ox;
        C.oy[cc] = oy;
        C.oz[cc] = oz;
    }
}

// ---------------------------------------------------------------- fluid-cell lists
__global__ void __launch_bounds__(kPcgThreads) k_list_count(MgLevel L) {
    const int64_t base = (int64_t)blockIdx.x * kListTile;
    int n = 0;
#pragma unroll
    for (int i = 0; i < kListTile / kPcgThreads; ++i) {
        const int64_t c = base + i * kPcgThreads + threadIdx.x;
        n += __syncthreads_count(c < L.cells && L.fluid[c]);
    }
    if (threadIdx.x == 0) L.blocks[blockIdx.x] = (uint32_t)n;
}

// Exclusive scan of a warp's values.
__device__ __forceinline__ uint32_t warp_exclusive(uint32_t v, uint32_t &total) {
    const int lane = threadIdx.x & 31;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    total = __shfl_sync(0xffffffffu, x, 31);
    return x - v;
}

__global__ void __launch_bounds__(32) k_list_scan(MgLevel L, int nblocks) {
    uint32_t run = 0;
    for (int i0 = 0; i0 < nblocks; i0 += 32) {
        const int i = i0 + threadIdx.x;
        uint32_t total;
        const uint32_t at = warp_exclusive(i < nblocks ? L.blocks[i] : 0u, total);
        if (i < nblocks) L.blocks[i] = run + at;
        run += total;
    }
    if (threadIdx.x == 0) *L.count = run;
}

// The list in ascending cell order; on the finest level also the info words.
template <bool TOP>
__global__ void __launch_bounds__(kPcgThreads) k_list_write(MgLevel L, int c0, int c1) {
    __shared__ uint32_t s_w[kPcgThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * kListTile;
    uint32_t at = L.blocks[blockIdx.x];
    for (int i = 0; i < kListTile / kPcgThreads; ++i) {
        const int64_t c = base + i * kPcgThreads + threadIdx.x;
        const bool fl = c < L.cells && L.fluid[c];
        const unsigned bal = __ballot_sync(0xffffffffu, fl);
        if (lane == 0) s_w[warp] = (uint32_t)__popc(bal);
        __syncthreads();
        uint32_t before = 0, all = 0;
#pragma unroll
        for (int w = 0; w < kPcgThreads / 32; ++w) {
            before += w < warp ? s_w[w] : 0u;
            all += s_w[w];
        }
        if (fl) {
            int x, y, z;
            mg_ijk(L, c, x, y, z);
            const uint32_t t = at + before + (uint32_t)__popc(bal & ((1u << lane) - 1u));
            L.idx[t] = (uint32_t)c;
            L.par[t] = (uint32_t)(((z >> 1) * c1 + (y >> 1)) * c0 + (x >> 1));
            if constexpr (TOP) {
                const int64_t sy = L.n[0], sz = sy * L.n[1];
                unsigned w = kInfoFluid | ((unsigned)L.diag[c] << 6) | ((x & 1) << 10) |
                             ((y & 1) << 11) | ((z & 1) << 12);
                if (x > 0 && L.fluid[c - 1]) w |= 1u;
                if (x < L.n[0] - 1 && L.fluid[c + 1]) w |= 2u;
                if (y > 0 && L.fluid[c - sy]) w |= 4u;
                if (y < L.n[1] - 1 && L.fluid[c + sy]) w |= 8u;
                if (z > 0 && L.fluid[c - sz]) w |= 16u;
                if (z < L.n[2] - 1 && L.fluid[c + sz]) w |= 32u;
                L.info[c] = (uint16_t)w;
            }
        } else if (TOP && c < L.cells) {
            L.info[c] = 0;
        }
        at += all;
        __syncthreads();
    }
}

// (A v)(c) on a large level, with the terms in mg_apply's order.  w: the info
// word on the finest level (elsewhere its parity bits alone); v(m, e): the
// vector at cell m, whose coarse cell is e cells from c's; csy, csz: the
// coarse strides.  A zero coupling (also the one that a row's end stores
// towards the next row) adds nothing.  AHEAD: v may be read at any cell of the
// box, so that its loads wait for neither the info word nor the couplings
// (what a cell that is not fluid holds is read and not used).  With the lists
// and vectors read by __ldg, which lets a pass's next cell start before this
// one's store, an iteration at 128^3 goes from 88 to 85 us.
template <bool TOP, bool AHEAD, class V>
__device__ __forceinline__ float list_apply(const MgLevel &L, int c, unsigned w, int csy, int csz,
                                            const V &v) {
    const int sy = L.n[0], sz = L.n[0] * L.n[1], end = (int)L.cells - 1;
    const int px = (w >> 10) & 1, py = (w >> 11) & 1, pz = (w >> 12) & 1;
    const int m[6] = {c - 1, c + 1, c - sy, c + sy, c - sz, c + sz};
    const int e[6] = {px - 1, px, py ? 0 : -csy, py ? csy : 0, pz ? 0 : -csz, pz ? csz : 0};
    float n[6];
    if constexpr (AHEAD) {
#pragma unroll
        for (int q = 0; q < 6; ++q) n[q] = v(q & 1 ? min(m[q], end) : max(m[q], 0), 0);
    }
    if constexpr (TOP) {
        float s = info_diag(w) * v(c, 0);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            if constexpr (AHEAD) s = w & (1u << q) ? s - n[q] : s;
            else if (w & (1u << q)) s -= v(m[q], e[q]);
        }
        return s;
    } else {
        const float o[6] = {c >= 1 ? __ldg(L.ox + c - 1) : 0.0f,   __ldg(L.ox + c),
                            c >= sy ? __ldg(L.oy + c - sy) : 0.0f, __ldg(L.oy + c),
                            c >= sz ? __ldg(L.oz + c - sz) : 0.0f, __ldg(L.oz + c)};
        float s = __ldg(L.diag + c) * v(c, 0);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            if constexpr (AHEAD) s = o[q] != 0.0f ? fmaf(o[q], n[q], s) : s;
            else if (o[q] != 0.0f) s = fmaf(o[q], v(m[q], e[q]), s);
        }
        return s;
    }
}

template <bool TOP> __device__ __forceinline__ float list_wd(const MgLevel &L, int c, unsigned w) {
    if constexpr (TOP) return kMgOmega / info_diag(w);
    else return __ldg(L.wd + c);
}

#define LIST_CELLS(L, t) \
    for (uint32_t t = blockIdx.x * kPcgThreads + threadIdx.x, t##n = *(L).count; t < t##n; \
         t += gridDim.x * kPcgThreads)

// Two damped-Jacobi sweeps from x = 0: x1 = w b / D, x = x1 + w (b - A x1) / D.
// On the finest level x1 is in L.t (k_setup and k_update leave it there).
template <bool TOP> __global__ void __launch_bounds__(kPcgThreads) k_mg_pre(MgLevel L) {
    auto x1 = [&](int m, int) { return TOP ? __ldg(L.t + m) : __ldg(L.wd + m) * __ldg(L.b + m); };
    LIST_CELLS(L, t) {
        const int c = (int)__ldg(L.idx + t);
        const unsigned w = TOP ? __ldg(L.info + c) : 0u;
        const float ax = list_apply<TOP, true>(L, c, w, 0, 0, x1);
        L.x[c] = fmaf(list_wd<TOP>(L, c, w), __ldg(L.b + c) - ax, x1(c, 0));
    }
}

// Coarse right-hand side: the fine residual b - A x summed over each block's
// fluid children (P^T r).  8 lanes per coarse cell, one child each, added in
// the children's order.
template <bool TOP>
__global__ void __launch_bounds__(kPcgThreads) k_mg_restrict(MgLevel F, MgLevel C, bool list) {
    auto xf = [&](int m, int) { return __ldg(F.x + m); };
    const int64_t total = 8 * (list ? (int64_t)*C.count : C.cells);
    const int lane = threadIdx.x & 31;
    const unsigned group = 0xffu << (lane & 24);
    for (int64_t u = (int64_t)blockIdx.x * kPcgThreads + threadIdx.x; u < total;
         u += (int64_t)gridDim.x * kPcgThreads) {
        const int64_t cc = list ? (int64_t)__ldg(C.idx + (u >> 3)) : u >> 3;
        const int q = (int)(u & 7);
        int I, J, K;
        mg_ijk(C, cc, I, J, K);
        const int i = 2 * I + (q & 1), j = 2 * J + ((q >> 1) & 1), k = 2 * K + (q >> 2);
        float r = 0.0f;
        if (i < F.n[0] && j < F.n[1] && k < F.n[2]) {
            const int c = (k * F.n[1] + j) * F.n[0] + i;
            const unsigned w = TOP ? __ldg(F.info + c) : 0u;
            const float a = __ldg(F.b + c) - list_apply<TOP, true>(F, c, w, 0, 0, xf);
            if (TOP ? (w & kInfoFluid) != 0 : __ldg(F.fluid + c) != 0) r = a;
        }
        float s = 0.0f;
#pragma unroll
        for (int e = 0; e < 8; ++e) s += __shfl_sync(group, r, (lane & 24) + e);
        if (q == 0) C.b[cc] = s;
    }
}

// Coarse correction and the first post-sweep: x' = x + P x_c (formed on the
// fly), t = x' + w (b - A x') / D.
template <bool TOP>
__global__ void __launch_bounds__(kPcgThreads) k_mg_post(MgLevel F, MgLevel C) {
    const int csy = C.n[0], csz = C.n[0] * C.n[1];
    LIST_CELLS(F, t) {
        const int c = (int)__ldg(F.idx + t), pc = (int)__ldg(F.par + t);
        unsigned w;
        if constexpr (TOP) {
            w = __ldg(F.info + c);
        } else {
            int i, j, k;
            mg_ijk(F, c, i, j, k);
            w = ((i & 1) << 10) | ((j & 1) << 11) | ((k & 1) << 12);
        }
        auto xp = [&](int m, int e) { return __ldg(F.x + m) + __ldg(C.x + pc + e); };
        const float ax = list_apply<TOP, false>(F, c, w, csy, csz, xp);
        F.t[c] = fmaf(list_wd<TOP>(F, c, w), __ldg(F.b + c) - ax, xp(c, 0));
    }
}

// The second post-sweep: x = t + w (b - A t) / D.  On the finest level it also
// forms b . x = r . z for CG.
template <bool TOP>
__global__ void __launch_bounds__(kPcgThreads) k_mg_sweep(MgLevel L, PcgBuffers B, int odd) {
    auto tv = [&](int m, int) { return __ldg(L.t + m); };
    double rz = 0.0;
    LIST_CELLS(L, t) {
        const int c = (int)__ldg(L.idx + t);
        const unsigned w = TOP ? __ldg(L.info + c) : 0u;
        const float b = __ldg(L.b + c);
        const float out = fmaf(list_wd<TOP>(L, c, w), b - list_apply<TOP, true>(L, c, w, 0, 0, tv), tv(c, 0));
        if (TOP) rz += (double)b * (double)out;
        L.x[c] = out;
    }
    if constexpr (TOP) grid_sum(rz, B, [&](double t) { put_rz(B, odd, t); });
}

// ---------------------------------------------------------------- small levels
struct MgSmall {
    int levels;  // the coarsest is levels - 1
    MgLevel L[kMgMaxLevels];
};

// Words of shared memory per cell of a small level: the operator and three
// vectors (the first of several levels: the vectors alone).
constexpr int kMgWords = 8;

struct SmallLevel {
    int n0, n1, n2, cells;
    float *diag, *wd, *ox, *oy, *oz, *x, *b, *t;
    // (A v)(c), the terms in mg_apply's order; couplings of 0 (towards cells
    // that are not fluid, and from a row's end to the next row) add nothing
    __device__ __forceinline__ float apply(int c, const float *v) const {
        const int sy = n0, sz = n0 * n1;
        float s = diag[c] * v[c];
        if (c >= 1) s = fmaf(ox[c - 1], v[c - 1], s);
        if (c + 1 < cells) s = fmaf(ox[c], v[c + 1], s);
        if (c >= sy) s = fmaf(oy[c - sy], v[c - sy], s);
        if (c + sy < cells) s = fmaf(oy[c], v[c + sy], s);
        if (c >= sz) s = fmaf(oz[c - sz], v[c - sz], s);
        if (c + sz < cells) s = fmaf(oz[c], v[c + sz], s);
        return s;
    }
};

// A thread's cells tid + 1024 k of the first small level, their operator in
// registers (a neighbour outside is the cell itself, times 0): its passes then
// read shared memory for the vector alone, 8 words a cell instead of 15, and
// all the operator's loads are in flight at once: 18.1 -> 16.7 us a cycle with
// 4,032 and 504 cells.
constexpr int kMgOwn = (int)((kMgSmall + kMgSmallThreads - 1) / kMgSmallThreads);
struct OwnCells {
    float diag[kMgOwn], wd[kMgOwn], o[kMgOwn][6];
    __device__ __forceinline__ void load(const MgLevel &G, int tid) {
        const int sy = G.n[0], sz = G.n[0] * G.n[1], cells = (int)G.cells;
#pragma unroll
        for (int q = 0; q < kMgOwn; ++q) {
            const int c = tid + q * kMgSmallThreads;
            const bool in = c < cells;
            diag[q] = in ? G.diag[c] : 0.0f;
            wd[q] = in ? G.wd[c] : 0.0f;
            o[q][0] = in && c >= 1 ? G.ox[c - 1] : 0.0f;
            o[q][1] = in && c + 1 < cells ? G.ox[c] : 0.0f;
            o[q][2] = in && c >= sy ? G.oy[c - sy] : 0.0f;
            o[q][3] = in && c + sy < cells ? G.oy[c] : 0.0f;
            o[q][4] = in && c >= sz ? G.oz[c - sz] : 0.0f;
            o[q][5] = in && c + sz < cells ? G.oz[c] : 0.0f;
        }
    }
    __device__ __forceinline__ float apply(int q, int c, int sy, int sz, int cells,
                                           const float *v) const {
        float s = diag[q] * v[c];
        s = fmaf(o[q][0], v[max(c - 1, 0)], s);
        s = fmaf(o[q][1], v[min(c + 1, cells - 1)], s);
        s = fmaf(o[q][2], v[c >= sy ? c - sy : c], s);
        s = fmaf(o[q][3], v[c + sy < cells ? c + sy : c], s);
        s = fmaf(o[q][4], v[c >= sz ? c - sz : c], s);
        s = fmaf(o[q][5], v[c + sz < cells ? c + sz : c], s);
        return s;
    }
};

#define OWN_CELLS(S, q, c)                                                            \
    _Pragma("unroll") for (int q = 0, c = tid; q < kMgOwn; ++q, c += kMgSmallThreads) \
        if (c < (S).cells)

// The rest of the cycle below the large levels, in one CTA: the vectors of all
// small levels in shared memory, the first one's operator in registers and the
// others' in shared memory (16^3 cells and below: 64 KB), the passes separated
// by the CTA's barrier; the coarsest level keeps each cell's operator and value
// in registers for its sweeps.  Cells that are not fluid have wd = b = 0 and
// only zero couplings: they are computed like the others, and stay finite.
// (Launched one by one, the three smallest levels of 128^3 took 38 us a cycle;
// a cluster of 8 CTAs on data in L2 took 26 us for the two smallest.)
__global__ void __launch_bounds__(kMgSmallThreads) k_mg_small(MgSmall M) {
    extern __shared__ float s_mg[];
    const int tid = (int)threadIdx.x;
    const int top = M.levels - 1;
    auto level = [&](int l) {  // the level's place: levels follow one another
        SmallLevel S;
        int at = 0;
        for (int k = 0; k < l; ++k) at += (int)M.L[k].cells * (k == 0 ? 3 : kMgWords);
        S.n0 = M.L[l].n[0];
        S.n1 = M.L[l].n[1];
        S.n2 = M.L[l].n[2];
        S.cells = (int)M.L[l].cells;
        float *p = s_mg + at;
        S.x = p;
        S.b = p + S.cells;
        S.t = p + 2 * S.cells;
        S.diag = p + 3 * S.cells;  // these not on the first of several levels
        S.wd = p + 4 * S.cells;
        S.ox = p + 5 * S.cells;
        S.oy = p + 6 * S.cells;
        S.oz = p + 7 * S.cells;
        return S;
    };
    // The first of several levels: b first, its two loads independent (b of a
    // cell that is not fluid may be anything), then the other levels, then the
    // operator into registers, in flight until the first pass.
    OwnCells own;
    float b0[kMgOwn];
    uint8_t f0[kMgOwn];
    if (top > 0) {
#pragma unroll
        for (int q = 0; q < kMgOwn; ++q) {
            const int c = min(tid + q * kMgSmallThreads, (int)M.L[0].cells - 1);
            b0[q] = M.L[0].b[c];
            f0[q] = M.L[0].fluid[c];
        }
    }
    for (int l = top > 0 ? 1 : 0; l <= top; ++l) {
        const MgLevel &G = M.L[l];
        const SmallLevel S = level(l);
        for (int c = tid; c < S.cells; c += kMgSmallThreads) {
            const float d = G.diag[c];
            S.diag[c] = d;
            if (l == 0) S.b[c] = G.fluid[c] ? G.b[c] : 0.0f;
            if (G.ox) {
                S.wd[c] = G.wd[c];
                S.ox[c] = G.ox[c];
                S.oy[c] = G.oy[c];
                S.oz[c] = G.oz[c];
            } else {  // a one-level cycle: the finest system itself
                int i, j, k;
                mg_ijk(G, c, i, j, k);
                const bool fl = G.fluid[c];
                S.wd[c] = fl ? kMgOmega / d : 0.0f;
                S.ox[c] = fl && i + 1 < S.n0 && G.fluid[c + 1] ? -1.0f : 0.0f;
                S.oy[c] = fl && j + 1 < S.n1 && G.fluid[c + S.n0] ? -1.0f : 0.0f;
                S.oz[c] = fl && k + 1 < S.n2 && G.fluid[c + S.n0 * S.n1] ? -1.0f : 0.0f;
            }
        }
    }
    if (top > 0) {
        const SmallLevel S = level(0);
        OWN_CELLS(S, q, c) S.b[c] = f0[q] ? b0[q] : 0.0f;
        own.load(M.L[0], tid);
    }
    __syncthreads();
    for (int l = 0; l < top; ++l) {
        const SmallLevel S = level(l), C = level(l + 1);
        // two sweeps from 0 (t: the first), the residual (t), its sums over the children
        if (l == 0) {
            const int sy = S.n0, sz = S.n0 * S.n1;
            OWN_CELLS(S, q, c) S.t[c] = own.wd[q] * S.b[c];
            __syncthreads();
            OWN_CELLS(S, q, c)
                S.x[c] = fmaf(own.wd[q], S.b[c] - own.apply(q, c, sy, sz, S.cells, S.t), S.t[c]);
            __syncthreads();
            OWN_CELLS(S, q, c) S.t[c] = S.b[c] - own.apply(q, c, sy, sz, S.cells, S.x);
        } else {
            for (int c = tid; c < S.cells; c += kMgSmallThreads) S.t[c] = S.wd[c] * S.b[c];
            __syncthreads();
            for (int c = tid; c < S.cells; c += kMgSmallThreads)
                S.x[c] = fmaf(S.wd[c], S.b[c] - S.apply(c, S.t), S.t[c]);
            __syncthreads();
            for (int c = tid; c < S.cells; c += kMgSmallThreads) S.t[c] = S.b[c] - S.apply(c, S.x);
        }
        __syncthreads();
        for (int cc = tid; cc < C.cells; cc += kMgSmallThreads) {
            const int I = cc % C.n0, J = (cc / C.n0) % C.n1, K = cc / (C.n0 * C.n1);
            float r = 0.0f;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int i = 2 * I + (q & 1), j = 2 * J + ((q >> 1) & 1), k = 2 * K + (q >> 2);
                if (i < S.n0 && j < S.n1 && k < S.n2) r += S.t[(k * S.n1 + j) * S.n0 + i];
            }
            C.b[cc] = r;
        }
        __syncthreads();
    }
    {
        // the coarsest level, x = 0: the operator of the thread's cell in
        // registers (a neighbour outside reads the cell itself, times 0)
        const SmallLevel S = level(top);
        const int c = tid, sy = S.n0, sz = S.n0 * S.n1;
        const bool in = c < S.cells;
        float o[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, diag = 0.0f, wd = 0.0f, b = 0.0f, v = 0.0f;
        int m[6] = {c, c, c, c, c, c};
        if (in) {
            const int st[3] = {1, sy, sz};
            const float *oo[3] = {S.ox, S.oy, S.oz};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (c >= st[a]) {
                    m[2 * a] = c - st[a];
                    o[2 * a] = oo[a][c - st[a]];
                }
                if (c + st[a] < S.cells) {
                    m[2 * a + 1] = c + st[a];
                    o[2 * a + 1] = oo[a][c];
                }
            }
            diag = S.diag[c];
            wd = S.wd[c];
            b = S.b[c];
            S.x[c] = 0.0f;
        }
        __syncthreads();
        for (int it = 0; it < kMgCoarseSweeps; ++it) {
            if (c < kMgCoarsest) {  // whole warps; x and t alternate (an even number of sweeps)
                const float *from = (it & 1) ? S.t : S.x;
                float *to = (it & 1) ? S.x : S.t;
                if (in) {
                    float s = diag * v;
#pragma unroll
                    for (int e = 0; e < 6; ++e) s = fmaf(o[e], from[m[e]], s);
                    to[c] = v = fmaf(wd, b - s, v);
                }
                // the sweeps' own barrier: only the warps that take part
                asm volatile("bar.sync 1, %0;" ::"n"(kMgCoarsest) : "memory");
            }
        }
        __syncthreads();
    }
    for (int l = top - 1; l >= 0; --l) {
        const SmallLevel S = level(l), C = level(l + 1);
        // two threads a coarse cell, four children each: the divisions of the
        // index once for the four (a thread per child: 4,250 cycles of 32,000;
        // with the loads of b and of the operator reordered 16.7 -> 15.0 us)
        for (int u = tid; u < 2 * C.cells; u += kMgSmallThreads) {
            const int up = u >= C.cells, cc = u - up * C.cells;
            const int I = cc % C.n0, J = (cc / C.n0) % C.n1, K = cc / (C.n0 * C.n1);
            const float x = C.x[cc];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = 2 * I + (q & 1), j = 2 * J + (q >> 1), k = 2 * K + up;
                if (i < S.n0 && j < S.n1 && k < S.n2) S.x[(k * S.n1 + j) * S.n0 + i] += x;
            }
        }
        __syncthreads();
        if (l == 0) {
            const int sy = S.n0, sz = S.n0 * S.n1;
            OWN_CELLS(S, q, c)
                S.t[c] = fmaf(own.wd[q], S.b[c] - own.apply(q, c, sy, sz, S.cells, S.x), S.x[c]);
            __syncthreads();
            OWN_CELLS(S, q, c)
                S.x[c] = fmaf(own.wd[q], S.b[c] - own.apply(q, c, sy, sz, S.cells, S.t), S.t[c]);
        } else {
            for (int c = tid; c < S.cells; c += kMgSmallThreads)
                S.t[c] = fmaf(S.wd[c], S.b[c] - S.apply(c, S.x), S.x[c]);
            __syncthreads();
            for (int c = tid; c < S.cells; c += kMgSmallThreads)
                S.x[c] = fmaf(S.wd[c], S.b[c] - S.apply(c, S.t), S.t[c]);
        }
        __syncthreads();
    }
    const SmallLevel S = level(0);
    for (int c = tid; c < S.cells; c += kMgSmallThreads) M.L[0].x[c] = S.x[c];
}
#undef OWN_CELLS

// b . x = r . z over the fluid cells, for a one-level cycle.
__global__ void __launch_bounds__(kPcgThreads) k_mg_dot(MgLevel L, PcgBuffers B, int odd) {
    double rz = 0.0;
    LIST_CELLS(L, t) {
        const uint32_t c = L.idx[t];
        rz += (double)L.b[c] * (double)L.x[c];
    }
    grid_sum(rz, B, [&](double t) { put_rz(B, odd, t); });
}

struct Multigrid {
    int levels;  // the coarsest is levels - 1
    int large;   // levels 0 .. large - 1 have lists, the others run in one CTA
    MgLevel L[kMgMaxLevels];
};

static int list_blocks(int64_t cells) { return (int)((cells + kListTile - 1) / kListTile); }

// Level dimensions: halve (rounding up) until at most kMgCoarsest cells.
static int mg_dims(const GridGeom &g, int dims[kMgMaxLevels][3]) {
    int n[3] = {g.n[0], g.n[1], g.n[2]};
    int lv = 0;
    for (;;) {
        for (int a = 0; a < 3; ++a) dims[lv][a] = n[a];
        ++lv;
        if ((int64_t)n[0] * n[1] * n[2] <= kMgCoarsest || lv == kMgMaxLevels) break;
        for (int a = 0; a < 3; ++a) n[a] = mg_coarse_dim(n[a]);
    }
    return lv;
}

static bool mg_large(int l, int64_t cells) { return l == 0 || cells > kMgSmall; }

static size_t mg_scratch_bytes(const GridGeom &g) {
    int dims[kMgMaxLevels][3];
    const int lv = mg_dims(g, dims);
    size_t bytes = 0;
    for (int l = 0; l < lv; ++l) {
        const size_t cells = (size_t)dims[l][0] * dims[l][1] * dims[l][2];
        if (l > 0) bytes += cells * (8 * sizeof(float) + 1) + 9 * 256;
        if (mg_large(l, (int64_t)cells))
            bytes += cells * (2 * sizeof(uint32_t) + (l == 0 ? sizeof(uint16_t) : 0)) +
                     ((size_t)list_blocks((int64_t)cells) + 1) * sizeof(uint32_t) + 5 * 256;
    }
    return bytes;
}

__global__ void __launch_bounds__(kPcgThreads) k_setup(GridGeom g, int64_t num_keys,
                                                       const uint32_t *__restrict__ cs,
                                                       const float *__restrict__ v0,
                                                       const float *__restrict__ v1,
                                                       const float *__restrict__ v2, float scale,
                                                       PcgBuffers B) {
    const int64_t nc = (int64_t)g.n[0] * g.n[1] * g.n[2];
    double bb = 0.0;
    for (int64_t c = (int64_t)blockIdx.x * kPcgThreads + threadIdx.x; c < nc;
         c += (int64_t)gridDim.x * kPcgThreads) {
        int i, j, k;
        cell_ijk(c, g.n[0], g.n[1], i, j, k);
        const uint32_t key = cell_key(g, i, j, k);
        const bool fl = cs[key + 1] > cs[key];
        B.fluid[c] = fl ? 1 : 0;
        float b = 0.0f, dg = 1.0f;
        if (fl) {
            const int d0 = g.n[0] + 1, d1 = g.n[1] + 1;
            const float div = (v0[((int64_t)k * g.n[1] + j) * d0 + i + 1] - v0[((int64_t)k * g.n[1] + j) * d0 + i]) +
                              (v1[((int64_t)k * d1 + j + 1) * g.n[0] + i] - v1[((int64_t)k * d1 + j) * g.n[0] + i]) +
                              (v2[((int64_t)(k + 1) * g.n[1] + j) * g.n[0] + i] - v2[((int64_t)k * g.n[1] + j) * g.n[0] + i]);
            b = -scale * div;
            int nn = 0;
            nn += (i > 0) + (i < g.n[0] - 1) + (j > 0) + (j < g.n[1] - 1) + (k > 0) + (k < g.n[2] - 1);
            dg = (float)nn;
        }
        B.diag[c] = dg;
        B.Ap[c] = fl ? (kMgOmega / dg) * b : 0.0f;  // the first sweep of the cycle
        B.x[c] = 0.0f;
        B.r[c] = b;
        B.d[c] = 0.0f;
        bb += (double)b * (double)b;
    }
    grid_sum(bb, B, [&](double t) { B.scal[kBb] = t; });
}

// The new direction and its product with A in one pass: d_out = z + beta d_in
// (beta = rz / rz_prev, 0 for the first direction), formed on the fly for
// the neighbours, Ap = A d_out, and d_out . Ap.
__global__ void __launch_bounds__(kPcgThreads) k_apply(MgLevel L, PcgBuffers B, int odd,
                                                       const float *d_in, float *d_out,
                                                       bool first) {
    const float beta = first ? 0.0f : (float)B.scal[kBeta];
    auto dn = [&](int m, int) { return fmaf(beta, __ldg(d_in + m), __ldg(B.z + m)); };
    double pap = 0.0;
    LIST_CELLS(L, t) {
        const int c = (int)__ldg(L.idx + t);
        const float dc = dn(c, 0);
        const float s = list_apply<true, true>(L, c, __ldg(L.info + c), 0, 0, dn);
        d_out[c] = dc;
        B.Ap[c] = s;
        pap += (double)dc * (double)s;
    }
    grid_sum(pap, B, [&](double t) {  // alpha of the step along the direction
        B.scal[kAlpha] = t != 0.0 ? (float)(B.scal[kRz + odd] / t) : 0.0f;
    });
}

// The step along d, the residual and its block sums, and in Ap's place the
// first sweep of the cycle that follows, w r / D.
__global__ void __launch_bounds__(kPcgThreads) k_update(MgLevel L, PcgBuffers B,
                                                        const float *__restrict__ d) {
    const float alpha = (float)B.scal[kAlpha];
    double rr = 0.0;
    const uint32_t n = *L.count, step = gridDim.x * kPcgThreads;
    for (uint32_t t = blockIdx.x * kPcgThreads + threadIdx.x; t < n; t += 2 * step) {
        // two cells at a time, their loads ahead of either's stores (9.1 -> 8.1 us at 128^3)
        const bool two = step < n - t;
        const int c[2] = {(int)__ldg(L.idx + t), (int)__ldg(L.idx + (two ? t + step : t))};
        float x[2], r[2], wd[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            x[q] = fmaf(alpha, __ldg(d + c[q]), B.x[c[q]]);
            r[q] = fmaf(-alpha, B.Ap[c[q]], B.r[c[q]]);
            wd[q] = kMgOmega / info_diag(__ldg(L.info + c[q]));
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (q == 1 && !two) break;
            B.x[c[q]] = x[q];
            B.r[c[q]] = r[q];
            B.Ap[c[q]] = wd[q] * r[q];
            rr += (double)r[q] * (double)r[q];
        }
    }
    rr = block_sum(rr);
    if (threadIdx.x == 0) B.rr[blockIdx.x] = rr;
}

__global__ void k_latch(uint32_t *status, uint32_t flag) { atomicOr(status, flag); }

struct Velocity {
    float *v[3];
};

// v_a -= dt/(rho dx) (p_hi - p_lo) on non-wall faces next to a fluid cell: a
// fluid cell takes its upper faces, and a lower one when the cell below is not
// fluid (p is 0 there).
__global__ void __launch_bounds__(kPcgThreads) k_velocity(GridGeom g, MgLevel L, float coef,
                                                          const float *__restrict__ p,
                                                          Velocity V) {
    LIST_CELLS(L, t) {
        const int c = (int)L.idx[t];
        const unsigned w = L.info[c];
        int at[3];
        mg_ijk(L, c, at[0], at[1], at[2]);
        const float pc = p[c];
        const int st[3] = {1, g.n[0], g.n[0] * g.n[1]};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int64_t dX = g.n[0] + (a == 0), dY = g.n[1] + (a == 1);
            const int64_t f = ((int64_t)at[2] * dY + at[1]) * dX + at[0];
            const int64_t up = a == 0 ? 1 : (a == 1 ? dX : dX * dY);
            if (at[a] < g.n[a] - 1) V.v[a][f + up] -= coef * (p[c + st[a]] - pc);
            if (at[a] > 0 && !(w & (1u << (2 * a)))) V.v[a][f] -= coef * (pc - p[c - st[a]]);
        }
    }
}

size_t pcg_scratch_bytes(const GridGeom &g) {
    const size_t nc = (size_t)g.n[0] * g.n[1] * g.n[2];
    return nc * (7 * sizeof(float) + 1) + (2 * kPcgMaxBlocks + 16) * sizeof(double) + 16 + 15 * 256 +
           mg_scratch_bytes(g);
}

// z = V-cycle(r): level 0 reads B.r, writes B.z, sweeps through B.Ap (which
// holds the first sweep on entry); its last sweep also leaves r . z in
// scal[kRz + odd].
static cudaError_t mg_vcycle(const Multigrid &M, const PcgBuffers &B, int odd, int nb,
                             cudaStream_t s) {
    auto blocks = [](int64_t cells) {
        return (int)std::min<int64_t>(152 * 8, (cells + kPcgThreads - 1) / kPcgThreads);
    };
    const int top = M.levels - 1, large = M.large;
    if (top > 0) {
        for (int l = 0; l < large; ++l) {
            const MgLevel &L = M.L[l], &C = M.L[l + 1];
            const int nf = blocks(L.cells), nc = blocks(8 * C.cells);
            if (l == 0) {
                k_mg_pre<true><<<nf, kPcgThreads, 0, s>>>(L);
                k_mg_restrict<true><<<nc, kPcgThreads, 0, s>>>(L, C, l + 1 < large);
            } else {
                k_mg_pre<false><<<nf, kPcgThreads, 0, s>>>(L);
                k_mg_restrict<false><<<nc, kPcgThreads, 0, s>>>(L, C, l + 1 < large);
            }
        }
    }
    MgSmall S;
    const int from = top > 0 ? large : 0;
    S.levels = M.levels - from;
    for (int l = 0; l < S.levels; ++l) S.L[l] = M.L[from + l];
    int64_t words = 0;  // the first of several levels: its vectors alone
    for (int l = 0; l < S.levels; ++l)
        words += S.L[l].cells * (l == 0 && S.levels > 1 ? 3 : kMgWords);
    const int smem = (int)(words * (int64_t)sizeof(float));
    // the kernel's limit, the same whatever the grid: contexts of other grids may
    // be launching it from other host threads
    const cudaError_t e = cudaFuncSetAttribute(k_mg_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               kMgSmallLimit);
    if (e != cudaSuccess) return e;
    k_mg_small<<<1, kMgSmallThreads, smem, s>>>(S);
    if (top > 0) {
        for (int l = large - 1; l >= 1; --l) {
            k_mg_post<false><<<blocks(M.L[l].cells), kPcgThreads, 0, s>>>(M.L[l], M.L[l + 1]);
            k_mg_sweep<false><<<blocks(M.L[l].cells), kPcgThreads, 0, s>>>(M.L[l], B, 0);
        }
        k_mg_post<true><<<blocks(M.L[0].cells), kPcgThreads, 0, s>>>(M.L[0], M.L[1]);
        k_mg_sweep<true><<<nb, kPcgThreads, 0, s>>>(M.L[0], B, odd);
    } else {  // one level: the coarsest sweeps are the whole cycle
        k_mg_dot<<<nb, kPcgThreads, 0, s>>>(M.L[0], B, odd);
    }
    return cudaGetLastError();
}

// Iterations it0 .. it0 + batch - 1 of the CG loop: the new direction and
// its product with A, the step, the residual norm, the V-cycle, r . z; then
// the last residual norm for the host.
static cudaError_t launch_batch(PcgBuffers &B, const Multigrid &M, int nb, int it0, int batch,
                                cudaStream_t s) {
    for (int b = 0; b < batch; ++b) {
        // directions alternate between d and d2, r . z between its two scalars
        const int odd = (it0 + b) & 1;
        float *d_in = odd ? B.d2 : B.d, *d_out = odd ? B.d : B.d2;
        k_apply<<<nb, kPcgThreads, 0, s>>>(M.L[0], B, odd, d_in, d_out, it0 + b == 0);
        k_update<<<nb, kPcgThreads, 0, s>>>(M.L[0], B, d_out);
        const cudaError_t e = mg_vcycle(M, B, odd ^ 1, nb, s);
        if (e != cudaSuccess) return e;
    }
    k_total<<<1, kPcgThreads, 0, s>>>(B.rr, nb, B.scal + kRr);
    return cudaGetLastError();
}

// Two workspace layouts are kept (the forward projection and the adjoint's,
// whose vectors sit behind three face arrays), the older one replaced.
struct PcgGraphs {
    cudaStream_t side = nullptr;   // capture stream (the caller's may be the legacy one)
    struct Entry {
        const float *key = nullptr;                    // B.x of the captured layout
        cudaGraphExec_t exec[2] = {nullptr, nullptr};  // [1]: the batch from iteration 0
        uint64_t used = 0;
    } entry[2];
    uint64_t clock = 0;
};

static void drop(PcgGraphs::Entry &E) {
    for (auto &e : E.exec)
        if (e) {
            cudaGraphExecDestroy(e);
            e = nullptr;
        }
    E.key = nullptr;
}

void pcg_graphs_free(PcgGraphs *G) {
    if (!G) return;
    for (auto &E : G->entry) drop(E);
    if (G->side) cudaStreamDestroy(G->side);
    delete G;
}

// The captured graph of a full batch (kCheckEvery iterations from an even
// iteration count), captured on first use for this workspace; nullptr if the
// capture is not possible here (the batch is then launched directly).
static cudaGraphExec_t batch_graph(PcgGraphs *&G, PcgBuffers &B, const Multigrid &M, int nb,
                                   bool first) {
    if (!G) G = new (std::nothrow) PcgGraphs;
    if (!G) return nullptr;
    PcgGraphs::Entry *E = G->entry[0].key == B.x ? &G->entry[0]
                          : G->entry[1].key == B.x ? &G->entry[1] : nullptr;
    if (!E) {
        E = G->entry[0].used <= G->entry[1].used ? &G->entry[0] : &G->entry[1];
        drop(*E);
        E->key = B.x;
    }
    E->used = ++G->clock;
    cudaGraphExec_t &ex = E->exec[first ? 1 : 0];
    if (ex) return ex;
    if (!G->side && cudaStreamCreateWithFlags(&G->side, cudaStreamNonBlocking) != cudaSuccess) {
        G->side = nullptr;
        (void)cudaGetLastError();
        return nullptr;
    }
    if (cudaStreamBeginCapture(G->side, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        (void)cudaGetLastError();
        return nullptr;
    }
    // a later batch is the loop from any even iteration count but 0: the same
    // kernels with k_apply's `first` off
    const cudaError_t e0 = launch_batch(B, M, nb, first ? 0 : kCheckEvery, kCheckEvery, G->side);
    cudaGraph_t graph = nullptr;
    const cudaError_t e1 = cudaStreamEndCapture(G->side, &graph);
    if (e0 != cudaSuccess || e1 != cudaSuccess || !graph) {
        if (graph) cudaGraphDestroy(graph);
        (void)cudaGetLastError();
        return nullptr;
    }
    const cudaError_t e2 = cudaGraphInstantiate(&ex, graph, 0);
    cudaGraphDestroy(graph);
    if (e2 != cudaSuccess) {
        ex = nullptr;
        (void)cudaGetLastError();
        return nullptr;
    }
    return ex;
}

polypic_status pcg_project(const GridGeom &g, int64_t num_keys, const uint32_t *cell_start,
                           float *vel[3], float dt, float rho, int maxiter, double rtol,
                           uint32_t *status, Workspace &ws, cudaStream_t s, PcgGraphs **graphs) {
    (void)num_keys;
    const int64_t nc = (int64_t)g.n[0] * g.n[1] * g.n[2];  // < 2^28 (polypic_create)
    PcgBuffers B;
    B.x = ws.take<float>(nc);
    B.r = ws.take<float>(nc);
    B.z = ws.take<float>(nc);
    B.d = ws.take<float>(nc);
    B.d2 = ws.take<float>(nc);
    B.Ap = ws.take<float>(nc);
    B.diag = ws.take<float>(nc);
    B.fluid = ws.take<uint8_t>(nc);
    B.sums = ws.take<double>(kPcgMaxBlocks);
    B.rr = ws.take<double>(kPcgMaxBlocks);
    B.arrived = ws.take<uint32_t>(1);
    B.scal = ws.take<double>(16);
    // the multigrid hierarchy: level 0 reads r, writes z, sweeps through Ap
    Multigrid M;
    {
        int dims[kMgMaxLevels][3];
        M.levels = mg_dims(g, dims);
        M.large = 0;
        for (int l = 0; l < M.levels; ++l) {
            MgLevel &L = M.L[l];
            L = MgLevel{};
            for (int a = 0; a < 3; ++a) L.n[a] = dims[l][a];
            L.cells = (int64_t)L.n[0] * L.n[1] * L.n[2];
            if (l == 0) {
                L.fluid = B.fluid;
                L.diag = B.diag;
                L.x = B.z;
                L.b = B.r;
                L.t = B.Ap;
            } else {
                L.fluid = ws.take<uint8_t>(L.cells);
                L.diag = ws.take<float>(L.cells);
                L.wd = ws.take<float>(L.cells);
                L.ox = ws.take<float>(L.cells);
                L.oy = ws.take<float>(L.cells);
                L.oz = ws.take<float>(L.cells);
                L.x = ws.take<float>(L.cells);
                L.b = ws.take<float>(L.cells);
                L.t = ws.take<float>(L.cells);
            }
            if (mg_large(l, L.cells)) {
                ++M.large;
                L.idx = ws.take<uint32_t>(L.cells);
                L.par = ws.take<uint32_t>(L.cells);
                L.count = ws.take<uint32_t>(1);
                L.blocks = ws.take<uint32_t>(list_blocks(L.cells));
                if (l == 0) L.info = ws.take<uint16_t>(L.cells);
            }
        }
    }
    if (ws.overflow) return POLYPIC_ERR_WORKSPACE;
    // the coarsest level is swept by one CTA of kMgCoarsest threads
    if (M.L[M.levels - 1].cells > kMgCoarsest) return POLYPIC_ERR_UNSUPPORTED;
    const int nb = (int)std::min<int64_t>(152 * 3, (nc + kPcgThreads - 1) / kPcgThreads);
    const double gdx = (double)g.dx;
    // rhs = -(rho dx^2 / dt) div with div = (sum of face differences) / dx
    const float scale = (float)((double)rho * gdx / (double)dt);

    auto ok = [&]() { return cudaGetLastError() == cudaSuccess; };
    if (cudaMemsetAsync(B.arrived, 0, sizeof(uint32_t), s) != cudaSuccess) return POLYPIC_ERR_CUDA;
    k_setup<<<nb, kPcgThreads, 0, s>>>(g, num_keys, cell_start, vel[0], vel[1], vel[2], scale, B);
    for (int l = 1; l < M.levels; ++l) {
        const int blocks = (int)std::min<int64_t>(152 * 8, (M.L[l].cells + kPcgThreads - 1) / kPcgThreads);
        k_mg_coarsen<<<blocks, kPcgThreads, 0, s>>>(M.L[l - 1], M.L[l]);
    }
    for (int l = 0; l < M.large; ++l) {
        const MgLevel &L = M.L[l];
        const int blocks = list_blocks(L.cells);
        const int c0 = mg_coarse_dim(L.n[0]), c1 = mg_coarse_dim(L.n[1]);
        k_list_count<<<blocks, kPcgThreads, 0, s>>>(L);
        k_list_scan<<<1, 32, 0, s>>>(L, blocks);
        if (l == 0) k_list_write<true><<<blocks, kPcgThreads, 0, s>>>(L, c0, c1);
        else k_list_write<false><<<blocks, kPcgThreads, 0, s>>>(L, c0, c1);
    }
    // z = M^-1 r and rz = r . z (the first direction is z: k_apply's `first`)
    if (mg_vcycle(M, B, 0, nb, s) != cudaSuccess) return POLYPIC_ERR_CUDA;
    if (!ok()) return POLYPIC_ERR_CUDA;
    double host[2];
    if (cudaMemcpyAsync(host, B.scal, 2 * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return POLYPIC_ERR_CUDA;
    const double bnorm = std::sqrt(host[kBb]);
    bool converged = bnorm == 0.0;
    int it = 0;
    while (!converged && it < maxiter) {
        const int batch = std::min(kCheckEvery, maxiter - it);
        // a full batch replays its captured graph (its kernels and arguments
        // depend only on the workspace and on whether it is the first)
        cudaGraphExec_t ex = batch == kCheckEvery && graphs
                                 ? batch_graph(*graphs, B, M, nb, it == 0)
                                 : nullptr;
        if (ex) {
            if (cudaGraphLaunch(ex, s) != cudaSuccess) return POLYPIC_ERR_CUDA;
        } else {
            if (launch_batch(B, M, nb, it, batch, s) != cudaSuccess) return POLYPIC_ERR_CUDA;
        }
        if (!ok()) return POLYPIC_ERR_CUDA;
        it += batch;
        if (cudaMemcpyAsync(host, B.scal, 2 * sizeof(double), cudaMemcpyDeviceToHost, s) !=
                cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return POLYPIC_ERR_CUDA;
        converged = std::sqrt(host[kRr]) <= rtol * bnorm;
    }
    const float coef = (float)((double)dt / ((double)rho * gdx));
    Velocity V;
    for (int a = 0; a < 3; ++a) V.v[a] = vel[a];
    k_velocity<<<nb, kPcgThreads, 0, s>>>(g, M.L[0], coef, B.x, V);
    if (!ok()) return POLYPIC_ERR_CUDA;
    if (!converged) {
        k_latch<<<1, 1, 0, s>>>(status, kFlagNotConverged);
        return POLYPIC_ERR_NOT_CONVERGED;
    }
    return POLYPIC_OK;
}

}  // namespace polypic
