// Coulomb elastic collisions (1)-(6) of Table 1 (e-e, O- - O-, O2+ - O2+,
// e - O2+, e - O-, O- - O2+), by the binary collision model of Takizuka & Abe
// (J. Comput. Phys. 25, 205, 1977), on ion steps with dt_ion, after the
// species' pushes and collisions and before the reactive pairs (22), (16),
// (17); reactions in the order (1)..(6).
//
// Within a cell each pair's relative velocity u (|u| = g) turns by theta,
// tan(theta/2) = delta ~ N(0, sigma^2), sigma^2 = K N / g^3 with
// K = q_a^2 q_b^2 w lnL dt_ion / (8 pi eps0^2 mu^2 A dx), and an azimuth phi
// uniform on [0, 2 pi); the pair's momentum and energy are kept.  Pairs from
// the cell lists in array order: like species the rotated list (r a random
// shift per cell) in consecutive pairs (an odd one sits out), N = the
// species' count in the cell; unlike species the i-th of the shorter list
// with member (i + r) mod M of the longer, N = M.  delta from the first
// member's stream (tag 12 + reaction index): one polar normal, then phi as
// the double angle of a uniform point of the unit disk (no trigonometric
// function: the same rounding as the oracle's).
//
// GPU form: on a Coulomb step each species taking part is sorted by cell
// (stable: array order within a cell) in three passes over its tiles of
// TILE slots: per-tile cell counts, a scan of each cell's counts over the
// tiles (and of the cell totals), and a scatter that ranks the slots of a
// tile per cell warp by warp (each warp owns a contiguous chunk, its rounds
// of 32 in slot order, ranks within a round from __match_any_sync).  The
// scatter moves velocities and ids into 16-byte entries in cell order, the
// reactions work on those, and a last pass brings the velocities back: a
// particle meets up to three reactions, and its four words lie in four arrays
// some hundred slots from its neighbours in the cell, so pairs read from the
// arrays cost 13 sectors of L2 traffic each; sorted, both lists of a cell are
// read and written in line.  The pairs of a reaction are disjoint and spread
// over several blocks per cell, about one pair per thread, because a pair is a
// chain of dependent loads, draws and divisions.  The species are sorted by
// the same launches (blockIdx.y); (1), (2) and (3) touch different species and
// share one.  What bounds it now is that chain and L2.  Per ion step of 4e5 e,
// 4e5 O-, 8e5 O2+ on 301 cells (a species or reaction per launch, a block per
// cell, pairs from the arrays -> now): sort 115 -> 51 us, reactions 366 -> 82 us.
#include "common.cuh"

namespace o2 {

namespace {

constexpr int CT = 256;                       // threads of the pair kernel
constexpr int ST = 512;                       // threads of the count kernel
constexpr int SCAN_T = 1024;                  // threads of the column scan (32 cells x 32 warps)
// Warps of a scatter block: each holds a 16-bit count per cell in shared
// memory, so 16 warps up to 4096 cells (128 KB), 8 beyond.
constexpr int SW_MANY = 16, SW_FEW = 8, SW_CELLS = 4096;

constexpr unsigned NOWHERE = 0xffffffffu;     // place of a dead slot

// The species a launch sorts, one per blockIdx.y.
struct SortSet {
    int s[NSP];
};

// Per-tile cell counts of the live particles of a species: hist[tile][cell].
__global__ void __launch_bounds__(ST) k_cell_count(Params P, SortSet set) {
    extern __shared__ unsigned cnt[];         // [Nc]
    const int Nc = P.Nc, S = set.s[blockIdx.y];
    for (int c = threadIdx.x; c < Nc; c += ST) cnt[c] = 0u;
    pdl_wait();
    DevCtrl* C = P.ctrl;
    const unsigned long long ns = C->slots[S] < P.sp[S].cap ? C->slots[S] : P.sp[S].cap;
    const unsigned ntiles = (unsigned)ceil_div(ns, TILE);
    const float* __restrict__ X = P.sp[S].x[C->cur[S]];
    const float inv_dx = P.inv_dx, limit = cell_limit(Nc);
    unsigned* __restrict__ H = P.chist[S];
    for (unsigned t = blockIdx.x; t < ntiles; t += gridDim.x) {
        __syncthreads();
        const unsigned long long base = (unsigned long long)t * TILE + threadIdx.x;
        float x[TILE / ST];
#pragma unroll
        for (int k = 0; k < TILE / ST; ++k) x[k] = base + k * ST < ns ? X[base + k * ST] : dead_marker();
#pragma unroll
        for (int k = 0; k < TILE / ST; ++k) {
            if (is_dead(x[k])) continue;
            int c; float f;
            cell_of_inside(x[k], inv_dx, limit, c, f);
            atomicAdd(&cnt[c], 1u);
        }
        __syncthreads();
        for (int c = threadIdx.x; c < Nc; c += ST) { H[(size_t)t * Nc + c] = cnt[c]; cnt[c] = 0u; }
    }
    pdl_trigger();
}

// Each cell's counts over the tiles turned into offsets (exclusive scan
// along the tiles, in place), and the cell totals.  A block takes 32 cells
// (lane = cell), its 32 warps contiguous ranges of tiles.
__global__ void __launch_bounds__(SCAN_T) k_cell_colscan(Params P, SortSet set) {
    __shared__ unsigned part[32][33];
    pdl_wait();
    DevCtrl* C = P.ctrl;
    const int Nc = P.Nc, S = set.s[blockIdx.y];
    const unsigned long long ns = C->slots[S] < P.sp[S].cap ? C->slots[S] : P.sp[S].cap;
    const unsigned T = (unsigned)ceil_div(ns, TILE);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * 32 + lane;
    const unsigned per = (T + 31) / 32;
    const unsigned t0 = warp * per < T ? warp * per : T, t1 = t0 + per < T ? t0 + per : T;
    unsigned* __restrict__ H = P.chist[S];
    unsigned sum = 0;
    if (c < Nc) {
#pragma unroll 4
        for (unsigned t = t0; t < t1; ++t) sum += H[(size_t)t * Nc + c];
    }
    part[warp][lane] = sum;
    __syncthreads();
    if (warp == 0) {
        unsigned run = 0;
        for (int w = 0; w < 32; ++w) { const unsigned v = part[w][lane]; part[w][lane] = run; run += v; }
        if (c < Nc) P.ctot[S][c] = run;
    }
    __syncthreads();
    if (c < Nc) {
        unsigned run = part[warp][lane];
        for (unsigned t = t0; t < t1; ++t) {
            const unsigned v = H[(size_t)t * Nc + c];
            H[(size_t)t * Nc + c] = run;
            run += v;
        }
    }
    pdl_trigger();
}

// Start of each cell's list: exclusive scan of the cell totals (one block per
// species).
__global__ void __launch_bounds__(SCAN_T) k_cell_start(Params P, SortSet set) {
    __shared__ unsigned ws[32];
    pdl_wait();
    const int Nc = P.Nc, S = set.s[blockIdx.y];
    const int per = (Nc + SCAN_T - 1) / SCAN_T;
    const int c0 = threadIdx.x * per;
    unsigned local = 0;
    for (int i = 0; i < per; ++i) if (c0 + i < Nc) local += P.ctot[S][c0 + i];
    unsigned total;
    unsigned run = block_excl_scan<SCAN_T>(local, ws, &total);
    for (int i = 0; i < per; ++i)
        if (c0 + i < Nc) { P.cstart[S][c0 + i] = run; run += P.ctot[S][c0 + i]; }
    pdl_trigger();
}

// Rows of the per-warp counts have an even length, so that the 32-bit
// shared-memory atomics on pairs of 16-bit counts stay 4-byte aligned.
__host__ __device__ inline int even(int n) { return (n + 1) & ~1; }

// Stable scatter of the slots of a species into cell order.
template <int SW>
__global__ void __launch_bounds__(SW * 32) k_cell_scatter(Params P, SortSet set) {
    constexpr int THREADS = SW * 32, CHUNK_W = TILE / SW, SR = CHUNK_W / 32;   // slots, rounds of a warp
    extern __shared__ unsigned short wcnt[];  // [SW][even(Nc)]: per-warp counts, then offsets
    const int Nc = P.Nc, NcE = even(P.Nc), S = set.s[blockIdx.y];
    pdl_wait();
    DevCtrl* C = P.ctrl;
    const unsigned long long ns = C->slots[S] < P.sp[S].cap ? C->slots[S] : P.sp[S].cap;
    const unsigned ntiles = (unsigned)ceil_div(ns, TILE);
    const float* __restrict__ X = P.sp[S].x[C->cur[S]];
    const float inv_dx = P.inv_dx, limit = cell_limit(Nc);
    const unsigned* __restrict__ H = P.chist[S];
    const unsigned* __restrict__ cst = P.cstart[S];
    float4* __restrict__ out = P.csort[S];
    unsigned* __restrict__ place = P.cplace[S];
    const unsigned cb = C->cur[S];
    const float* __restrict__ VX = P.sp[S].vx[cb];
    const float* __restrict__ VY = P.sp[S].vy[cb];
    const float* __restrict__ VZ = P.sp[S].vz[cb];
    const uint32_t* __restrict__ ID = P.sp[S].id[cb];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    unsigned short* mine = wcnt + warp * NcE;
    for (unsigned t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const unsigned long long base = (unsigned long long)t * TILE + (unsigned long long)warp * CHUNK_W + lane;
        float x[SR];
#pragma unroll
        for (int r = 0; r < SR; ++r) x[r] = base + 32 * r < ns ? X[base + 32 * r] : dead_marker();
        unsigned* w32 = reinterpret_cast<unsigned*>(wcnt);
        for (int k = threadIdx.x; k < SW * NcE / 2; k += THREADS) w32[k] = 0u;
        __syncthreads();
        int cell[SR];
#pragma unroll
        for (int r = 0; r < SR; ++r) {
            cell[r] = -1;
            if (!is_dead(x[r])) {
                float f;
                cell_of_inside(x[r], inv_dx, limit, cell[r], f);
                atomicAdd(reinterpret_cast<unsigned*>(&mine[cell[r] & ~1]), (cell[r] & 1) ? 0x10000u : 1u);
            }
        }
        __syncthreads();
        // per cell: offsets of the warps' chunks within the tile
        for (int c = threadIdx.x; c < Nc; c += THREADS) {
            unsigned run = 0;
#pragma unroll
            for (int w = 0; w < SW; ++w) {
                const unsigned v = wcnt[w * NcE + c];
                wcnt[w * NcE + c] = (unsigned short)run;
                run += v;
            }
        }
        __syncthreads();
        unsigned to[SR];      // start of the cell's slots of this tile
#pragma unroll
        for (int r = 0; r < SR; ++r) to[r] = cell[r] >= 0 ? cst[cell[r]] + H[(size_t)t * Nc + cell[r]] : 0u;
        constexpr int G = 4;  // rounds whose velocities are in flight together
#pragma unroll
        for (int r0 = 0; r0 < SR; r0 += G) {
            float4 v[G];
#pragma unroll
            for (int k = 0; k < G; ++k) {
                const unsigned long long p = base + 32 * (r0 + k);
                if (cell[r0 + k] >= 0) v[k] = make_float4(VX[p], VY[p], VZ[p], __uint_as_float(ID[p]));
            }
#pragma unroll
            for (int k = 0; k < G; ++k) {
                const int r = r0 + k, c = cell[r];
                const unsigned peers = __match_any_sync(0xffffffffu, c);
                unsigned off = 0;
                if (c >= 0) off = mine[c];
                __syncwarp();
                unsigned q = NOWHERE;
                if (c >= 0) {
                    const unsigned rank = __popc(peers & lt);
                    q = to[r] + off + rank;
                    out[q] = v[k];
                    if (rank == 0) mine[c] = (unsigned short)(off + __popc(peers));
                }
                if (base + 32 * r < ns) place[base + 32 * r] = q;
                __syncwarp();
            }
        }
        __syncthreads();
    }
    pdl_trigger();
}

// The velocities of the sorted entries back to their slots.
__global__ void __launch_bounds__(ST) k_cell_unsort(Params P, SortSet set) {
    pdl_wait();
    const int S = set.s[blockIdx.y];
    DevCtrl* C = P.ctrl;
    const unsigned long long ns = C->slots[S] < P.sp[S].cap ? C->slots[S] : P.sp[S].cap;
    const unsigned cb = C->cur[S];
    float* __restrict__ VX = P.sp[S].vx[cb];
    float* __restrict__ VY = P.sp[S].vy[cb];
    float* __restrict__ VZ = P.sp[S].vz[cb];
    const float4* __restrict__ E = P.csort[S];
    const unsigned* __restrict__ place = P.cplace[S];
    constexpr int G = 4;
    for (unsigned long long p0 = (unsigned long long)blockIdx.x * ST * G + threadIdx.x; p0 < ns;
         p0 += (unsigned long long)gridDim.x * ST * G) {
        unsigned q[G];
        float4 v[G];
#pragma unroll
        for (int k = 0; k < G; ++k) q[k] = p0 + k * ST < ns ? place[p0 + k * ST] : NOWHERE;
#pragma unroll
        for (int k = 0; k < G; ++k)
            if (q[k] != NOWHERE) v[k] = E[q[k]];
#pragma unroll
        for (int k = 0; k < G; ++k)
            if (q[k] != NOWHERE) { VX[p0 + k * ST] = v[k].x; VY[p0 + k * ST] = v[k].y; VZ[p0 + k * ST] = v[k].z; }
    }
    pdl_trigger();
}

// One pair of reaction r: sorted entries A of species a and B of species b.
// The deflection's normal and the azimuth's point of the disk are drawn by one
// rejection loop from pairs of words (0, 1), (2, 3) of block 0, (0, 1) of block
// 1, ..., so that lanes need a new block at the same tries.
__device__ __forceinline__ void coulomb_pair(const Params& P, int r, float4* A, float4* B, float N,
                                             unsigned long long n, unsigned& wtries, unsigned& npairs) {
    const float4 a = *A, b = *B;
    const float ux = a.x - b.x, uy = a.y - b.y, uz = a.z - b.z;
    const float g2 = dot3(ux, uy, uz, ux, uy, uz);
    if (!(g2 > 0.0f)) return;
    const float g = sqrtf(g2);
    const uint32_t id = __float_as_uint(a.w), tag = TAG_COUL + (uint32_t)r;
    uint4 buf = philox4x32_10(make_uint4((uint32_t)n, tag, 0u, (uint32_t)(n >> 32)), make_uint2(id, P.seed));
    float an = 0.0f, sn2 = 0.5f;                  // the normal's point
    float e1 = 1.0f, e2 = 0.0f, s2 = 1.0f;        // the azimuth's point
    int task = 0, tries = 0;
    for (uint32_t t = 0; task < 2; ++t) {
        if (t > 0u && (t & 1u) == 0u)
            buf = philox4x32_10(make_uint4((uint32_t)n, tag, t >> 1, (uint32_t)(n >> 32)), make_uint2(id, P.seed));
        const float p = 2.0f * uniform((t & 1u) ? buf.z : buf.x) - 1.0f;
        const float q = 2.0f * uniform((t & 1u) ? buf.w : buf.y) - 1.0f;
        const float s = task == 0 ? fmaf(p, p, q * q) : p * p + q * q;
        const bool in = s > 0.0f && s < 1.0f;
        if (!in && ++tries < MAX_TRIES) continue;
        if (!in) ++wtries;                        // gives up: normal 0, azimuth 0
        else if (task == 0) { an = p; sn2 = s; }
        else { e1 = p; e2 = q; s2 = s; }
        ++task;
        tries = 0;
    }
    const float z0 = an * sqrtf((-2.0f * ln_series(sn2)) / sn2);
    const float sig2 = P.coul_K[r] * N / (g2 * g);
    const float d = sqrtf(sig2) * z0;
    float sn, omc;
    if (fabsf(d) < 1e18f) {
        const float q = 1.0f / (1.0f + d * d);
        sn = 2.0f * d * q;
        omc = 2.0f * (d * d) * q;
    } else {
        sn = 0.0f; omc = 2.0f;
    }
    const float cp = (e1 * e1 - e2 * e2) / s2, spn = (2.0f * e1 * e2) / s2;
    const float up2 = ux * ux + uy * uy;
    float dx, dy, dz;
    if (up2 > 0.0f) {
        const float up = sqrtf(up2);
        const float sc = sn * cp, ss = sn * spn;
        dx = (ux * uz / up) * sc - (uy * g / up) * ss - ux * omc;
        dy = (uy * uz / up) * sc + (ux * g / up) * ss - uy * omc;
        dz = -up * sc - uz * omc;
    } else {
        dx = g * (sn * cp);
        dy = g * (sn * spn);
        dz = -uz * omc;
    }
    const float fa = P.coul_fa[r], fb = P.coul_fb[r];
    *A = make_float4(a.x + fa * dx, a.y + fa * dy, a.z + fa * dz, a.w);
    *B = make_float4(b.x - fb * dx, b.y - fb * dy, b.z - fb * dz, b.w);
    ++npairs;
}

// Reactions r[blockIdx.z] (species a, b) of one launch; a cell (blockIdx.x,
// grid-stride) has gridDim.y blocks, its pairs spread over their threads
// (disjoint particles: no two threads touch one).
struct ReactionSet {
    int r[3], a[3], b[3];
};

__global__ void __launch_bounds__(CT) k_coulomb(Params P, ReactionSet set) {
    __shared__ unsigned sh_tries, sh_pairs;
    const int r = set.r[blockIdx.z], a = set.a[blockIdx.z], b = set.b[blockIdx.z];
    if (threadIdx.x == 0) { sh_tries = 0u; sh_pairs = 0u; }
    pdl_wait();
    __syncthreads();
    DevCtrl* C = P.ctrl;
    const unsigned long long n = C->step;
    const int Nc = P.Nc;
    const unsigned t0 = blockIdx.y * CT + threadIdx.x, nt = gridDim.y * CT;
    unsigned wtries = 0, npairs = 0;
    for (int c = blockIdx.x; c < Nc; c += gridDim.x) {
        const unsigned na = P.ctot[a][c], nb = (a == b) ? na : P.ctot[b][c];
        if (a == b ? na < 2u : (na == 0u || nb == 0u)) continue;   // block-uniform
        const unsigned M = na > nb ? na : nb, m = na < nb ? na : nb;
        if (blockIdx.y * CT >= (a == b ? na / 2u : m)) continue;
        // the cell's shift, drawn by every thread (no barrier)
        const uint4 w = philox4x32_10(make_uint4((uint32_t)n, TAG_SHIFT_COUL + (uint32_t)r, 0u, (uint32_t)(n >> 32)),
                                      make_uint2((uint32_t)c, P.seed));
        const unsigned rs = w.x % M;
        float4* LA = P.csort[a] + P.cstart[a][c];
        float4* LB = P.csort[b] + P.cstart[b][c];
        // (i + rs) mod M with i, rs < M: sums below 2^32 (lists below 2^31)
        auto wrap = [M](unsigned q) { return q >= M ? q - M : q; };
        if (a == b) {
            for (unsigned j = t0; 2u * j + 1u < na; j += nt)
                coulomb_pair(P, r, LA + wrap(rs + 2u * j), LA + wrap(rs + 2u * j + 1u), (float)na, n, wtries, npairs);
        } else {
            const bool a_short = na <= nb;
            for (unsigned i = t0; i < m; i += nt) {
                const unsigned q = wrap(i + rs);
                coulomb_pair(P, r, LA + (a_short ? i : q), LB + (a_short ? q : i), (float)M, n, wtries, npairs);
            }
        }
    }
    pdl_trigger();
    if (wtries) atomicAdd(&sh_tries, wtries);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) npairs += __shfl_down_sync(0xffffffffu, npairs, o);
    if ((threadIdx.x & 31) == 0 && npairs) atomicAdd(&sh_pairs, npairs);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (sh_tries) atomicAdd(&C->cnt.warn_tries, (unsigned long long)sh_tries);
        if (sh_pairs) atomicAdd(&C->cnt.coulomb_pairs, (unsigned long long)sh_pairs);
    }
}

}  // namespace

const int COUL_SPECIES[6][2] = {{SP_E, SP_E}, {SP_OM, SP_OM}, {SP_OP, SP_OP}, {SP_E, SP_OP}, {SP_E, SP_OM},
                                {SP_OM, SP_OP}};

static size_t scatter_smem(int warps, int Nc) { return sizeof(unsigned short) * warps * (size_t)even(Nc); }

cudaError_t configure_coulomb_smem(int Nc) {
    cudaError_t e = Nc <= SW_CELLS ? cudaFuncSetAttribute(k_cell_scatter<SW_MANY>,
                                                          cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                          (int)scatter_smem(SW_MANY, SW_CELLS))
                                   : cudaFuncSetAttribute(k_cell_scatter<SW_FEW>,
                                                          cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                          (int)scatter_smem(SW_FEW, MAX_NODES));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_cell_count, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(unsigned) * (size_t)MAX_NODES));
    return e;
}

// The Coulomb collisions of one ion step (mask bit r-1 = reaction r): the
// species taking part sorted by cell, then the reactions in order.  `grid`
// blocks per species sort its tiles; reactions get about `grid` blocks, 1 to 16
// per cell.  Returns the number of kernels launched.
int launch_coulomb(const Params& P, unsigned mask, int grid, cudaStream_t s) {
    int launches = 0;
    unsigned need = 0;
    for (int r = 0; r < 6; ++r)
        if ((mask >> r) & 1u) need |= (1u << COUL_SPECIES[r][0]) | (1u << COUL_SPECIES[r][1]);
    const int Nc = P.Nc;
    SortSet set = {};
    int ns = 0;
    unsigned long long cap = 0;
    for (int sp = 0; sp < NSP; ++sp)
        if ((need >> sp) & 1u) { set.s[ns++] = sp; cap = cap > P.sp[sp].cap ? cap : P.sp[sp].cap; }
    if (ns > 0) {
        const int tiles = (int)(ceil_div(cap, TILE) < (unsigned long long)grid ? ceil_div(cap, TILE) : grid);
        const dim3 gt(tiles > 0 ? tiles : 1, ns);
        launch_pdl(k_cell_count, gt, ST, sizeof(unsigned) * (size_t)Nc, s, P, set);
        launch_pdl(k_cell_colscan, dim3((Nc + 31) / 32, ns), SCAN_T, 0, s, P, set);
        launch_pdl(k_cell_start, dim3(1, ns), SCAN_T, 0, s, P, set);
        if (Nc <= SW_CELLS) launch_pdl(k_cell_scatter<SW_MANY>, gt, SW_MANY * 32, scatter_smem(SW_MANY, Nc), s, P, set);
        else launch_pdl(k_cell_scatter<SW_FEW>, gt, SW_FEW * 32, scatter_smem(SW_FEW, Nc), s, P, set);
        launches += 4;
    }
    const int cells = Nc < 4096 ? Nc : 4096;
    const int split = 2 * grid / cells < 1 ? 1 : (2 * grid / cells > 16 ? 16 : 2 * grid / cells);
    auto react = [&](const ReactionSet& R, int n) {
        if (n == 0) return;
        launch_pdl(k_coulomb, dim3(cells, split, n), CT, 0, s, P, R);
        ++launches;
    };
    ReactionSet like = {};
    int nl = 0;
    for (int r = 0; r < 6; ++r) {
        if (r == 3) { react(like, nl); nl = 0; }   // (1)-(3): different species, one launch
        if (!((mask >> r) & 1u)) continue;
        if (r < 3) {
            like.r[nl] = r;
            like.a[nl] = like.b[nl] = COUL_SPECIES[r][0];
            ++nl;
        } else {
            ReactionSet R = {};
            R.r[0] = r;
            R.a[0] = COUL_SPECIES[r][0];
            R.b[0] = COUL_SPECIES[r][1];
            react(R, 1);
        }
    }
    if (ns > 0) {
        launch_pdl(k_cell_unsort, dim3(grid, ns), ST, 0, s, P, set);
        ++launches;
    }
    return launches;
}

}  // namespace o2
