// Ion-ion neutralization (17), O- + O2+ -> O + O2, on ion steps: a binary,
// cell-local (DSMC-like) process at the post-push positions.
//
// Pairing (the reading used by the oracle): in cell c take the surviving O-
// and O2+ in array order, n- and n+ of them, m = min, M = max, and a shift
// r_c drawn per cell and step; the i-th member of the shorter list (O- on a
// tie), i < m, is paired with member (i + r_c) mod M of the longer one.  A
// pair reacts with probability P = M w sigma_n(E_rel) g dt_ion / (A dx).
//
// GPU form.  The acceptance draw u of a pair needs only the O- id, and
// P <= K_max M pf (pf = w dt_ion / (A dx)), so an O- can react only if
// u < K_max M pf; at the method's weights and time steps that bound is
// ~1e-6 and only a handful of O- per step pass it.  So:
//   * k_pair_count, O- part: streams x and id of the O- once; per tile of 8192
//     slots the live O- per cell (and their totals n-), and u against the
//     bound with M replaced by the number of slots in use: the ~1e-3 that pass
//     go to a candidate list.  O2+ part: the same counts of the O2+.  Neither
//     part needs the other, so each runs behind its own species' chain and the
//     draws (ALU) beside the O2+ push (HBM), off the step's critical path;
//   * k_pair, once both are there: the candidates against the bound with the
//     cell's M, one per thread; for each one left the whole block finds its
//     rank k in the cell list (counts of the earlier tiles + same-cell slots
//     before it in its tile), the partner rank q, the O2+ tile holding rank q
//     (block scan of that cell's per-tile counts) and the partner's slot there
//     (the warp whose slots hold it, by ballots), each step with all of the
//     block's loads in flight; one thread then does the reaction test with the
//     exact P.
// Both streams are bound by HBM on large arrays and by latency on small ones.
// Reactions only append (O- slot, O2+ slot) to the removal list and take the
// pair out of the fresh deposit; both are order-independent, so flagged ions
// may be resolved in any order.
//
// The kernels take the two species, tables and lists as a PairSpec: the same
// code runs (22) e + O- -> O + 2e (A = O-, B = e, only A removed; its
// kinematics and births in k_edet_apply) and (16) e + O2+ -> O + O (A = e)
// before (17) (A = O-); the removals of (22) and (16) are applied before the
// next process counts its particles.
#include "common.cuh"

namespace o2 {

namespace {

constexpr int HIST_T = 512;                  // threads of k_pair_count
constexpr int HIST_V = TILE / HIST_T / 4;    // 16-byte loads of an array per thread and tile
constexpr int PAIR_T = 256;                  // threads of k_pair
constexpr int PER_T = TILE / PAIR_T;         // 32 slots of a tile per thread
static_assert(PER_T == 32, "one 32-bit hit mask per thread");

// Four slots from p on of an array of n (p a multiple of 4); `fill` beyond n.
template <class V, class T>
__device__ __forceinline__ V load4(const T* __restrict__ A, unsigned long long p, unsigned long long n, T fill) {
    V v;
    if (p + 4 <= n) {
        v = *reinterpret_cast<const V*>(A + p);
    } else {
        v.x = p < n ? A[p] : fill;
        v.y = p + 1 < n ? A[p + 1] : fill;
        v.z = p + 2 < n ? A[p + 2] : fill;
        v.w = fill;
    }
    return v;
}

// Live particles per cell (post-push positions) of each tile of one of the two
// species (`first`: A): hist[tile][cell], and the totals per cell (zero on
// entry; the end-of-step kernel clears them), added once per block at the end.
// A also draws: the particles whose acceptance number is below the bound for
// as many partners as there are slots go to the candidate list.  With the
// counts behind the chains instead of after their join: RF cycle of 512 cells
// 36.0 -> 35.4 ms, 2048 cells 25.5 -> 24.8, 128 cells 14.0 -> 13.3.
template <bool FIRST>
__device__ __forceinline__ void pair_count_body(const Params& P, const PairSpec& Sp, unsigned blk, unsigned nblk) {
    extern __shared__ unsigned hsm[];   // [Nc] tile counts, [Nc] block totals
    DevCtrl* C = P.ctrl;
    const int Nc = P.Nc;
    const float inv_dx = P.inv_dx, limit = cell_limit(P.Nc);
    unsigned* bt = hsm + Nc;
    for (int c = threadIdx.x; c < Nc; c += HIST_T) { hsm[c] = 0u; bt[c] = 0u; }
    pdl_wait();
    const int S = FIRST ? Sp.A : Sp.B;
    const unsigned long long n = C->slots[S];
    const unsigned ntiles = (unsigned)ceil_div(n, TILE);
    if (blk >= ntiles) return;          // block-uniform
    const unsigned cb = C->cur[S];
    const float* __restrict__ X = P.sp[S].x[cb];
    const uint32_t* __restrict__ ID = P.sp[S].id[cb];
    const unsigned long long step = C->step;
    const PhiloxPre pre = philox_pre((uint32_t)step, Sp.tag_pair, (uint32_t)(step >> 32), P.seed);
    // P <= K_max M pf with M at most the slots in use of either species
    const unsigned long long mb = C->slots[Sp.A] > C->slots[Sp.B] ? C->slots[Sp.A] : C->slots[Sp.B];
    const float bound = Sp.Kmax_hi * (P.pair_factor * (float)mb);
    __syncthreads();
    for (unsigned tile = blk; tile < ntiles; tile += nblk) {
        const unsigned long long base = (unsigned long long)tile * TILE + 4u * threadIdx.x;
        float4 x[HIST_V];
        uint4 id[FIRST ? HIST_V : 1];
#pragma unroll
        for (int i = 0; i < HIST_V; ++i) x[i] = load4<float4>(X, base + 4ull * HIST_T * i, n, dead_marker());
        if (FIRST) {
#pragma unroll
            for (int i = 0; i < HIST_V; ++i) id[i] = load4<uint4>(ID, base + 4ull * HIST_T * i, n, 0u);
        }
#pragma unroll
        for (int i = 0; i < HIST_V; ++i) {
            const float xs[4] = {x[i].x, x[i].y, x[i].z, x[i].w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (is_dead(xs[k])) continue;
                int c; float fr;
                cell_of_inside(xs[k], inv_dx, limit, c, fr);
                atomicAdd(&hsm[c], 1u);
            }
        }
        if constexpr (FIRST) {
            const int lane = threadIdx.x & 31;
#pragma unroll
            for (int i = 0; i < HIST_V; ++i) {
                if (base + 4ull * HIST_T * i >= n) break;
                const float xs[4] = {x[i].x, x[i].y, x[i].z, x[i].w};
                const uint32_t ids[4] = {id[i].x, id[i].y, id[i].z, id[i].w};
                uint32_t w[4];
                bool any = false;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    w[k] = philox_id(pre, ids[k]).x;
                    any |= uniform(w[k]) < bound;
                }
                if (!any) continue;
                // the lanes that are here add their candidates with one atomic:
                // one by one, 4e6 O- that all pass took 76-90 us for the counts
                // of both species, now 35 (27 where next to none passes)
                const unsigned act = __activemask();
                unsigned in[4];                 // of them, those whose slot k is a candidate
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    in[k] = __ballot_sync(act, uniform(w[k]) < bound && !is_dead(xs[k]));
                const int first = __ffs(act) - 1;
                unsigned q = 0u;
                if (lane == first)              // at most the slots of A
                    q = atomicAdd(Sp.ncand, __popc(in[0]) + __popc(in[1]) + __popc(in[2]) + __popc(in[3]));
                q = __shfl_sync(act, q, first);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if ((in[k] >> lane) & 1u)
                        Sp.cand[q + __popc(in[k] & ((1u << lane) - 1u))] =
                            make_uint2((unsigned)(base + 4ull * HIST_T * i) + k, w[k]);
                    q += __popc(in[k]);
                }
            }
        }
        __syncthreads();
        unsigned* H = (FIRST ? Sp.histA : Sp.histB) + (size_t)tile * Nc;
        for (int c = threadIdx.x; c < Nc; c += HIST_T) {
            const unsigned v = hsm[c];
            H[c] = v;
            bt[c] += v;
            hsm[c] = 0u;
        }
        __syncthreads();
    }
    pdl_trigger();
    for (int c = threadIdx.x; c < Nc; c += HIST_T)
        if (bt[c]) atomicAdd(&Sp.tot[FIRST ? c : Nc + c], bt[c]);
}

__device__ __forceinline__ unsigned block_sum(unsigned v, unsigned* ws) {
    unsigned total;
    (void)block_excl_scan<PAIR_T>(v, ws, &total);
    return total;
}

// Exclusive scan over the block (PAIR_T threads) with one barrier; ws = PAIR_T / 32 words.
__device__ __forceinline__ unsigned scan_once(unsigned v, unsigned* ws, unsigned* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    unsigned before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < PAIR_T / 32; ++w) {
        if (w < warp) before += ws[w];
        all += ws[w];
    }
    *total = all;
    return before + x - v;
}

// Resolve one flagged O- (slot p, acceptance number u, in cell c).  Every
// thread of the block calls it; all return at the same point except at the
// very end.  Bound by a chain of L2 round trips, so loads that do not depend on
// one another go out together: the earlier tiles' counts with the own tile's
// slots (rank k), eight tiles of a group at a time (the partner's tile), the
// partner tile's slots as 32 neighbours per warp (its slot, found with ballots).
// Measured per RF cycle: 512 cells 34.58 -> 34.08 ms, 2048 cells 24.13 -> 24.02;
// with the groups read before the rank is known 33.99 but 24.24, and with a tile's
// slots as 32 in a row per thread besides 34.56 and 24.35.  ws: PAIR_T / 32 words, sh: 2
// words, wc: PAIR_T / 32 words of shared memory.
__device__ void resolve_one(const Params& P, const PairSpec& Sp, unsigned p, float u, unsigned c,
                            unsigned* ws, unsigned* sh, unsigned* wc, unsigned long long step,
                            unsigned long long nsp, unsigned ntp, unsigned cm, unsigned cp, unsigned& gt1) {
    DevCtrl* C = P.ctrl;
    const int Nc = P.Nc;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float inv_dx = P.inv_dx, limit = cell_limit(Nc);
    const unsigned tile = p / TILE;
    const unsigned* __restrict__ H0 = Sp.histA;
    const unsigned* __restrict__ H1 = Sp.histB;
    const float* __restrict__ XM = P.sp[Sp.A].x[cm];
    const float* __restrict__ XP = P.sp[Sp.B].x[cp];
    float xa[PER_T];
#pragma unroll
    for (int i = 0; i < PER_T; ++i) {
        const unsigned q = tile * TILE + (unsigned)i * PAIR_T + tid;
        xa[i] = q < p ? XM[q] : dead_marker();
    }
    const unsigned nm = Sp.tot[c], npl = Sp.tot[Nc + c];
    unsigned cnt = 0, gs = 0;
#pragma unroll 8
    for (unsigned t = tid; t < tile; t += PAIR_T) cnt += H0[(size_t)t * Nc + c];
    // tiles of B: thread t sums a contiguous group
    const unsigned per = (ntp + PAIR_T - 1) / PAIR_T;
    const unsigned t0 = (unsigned)tid * per, t1 = (t0 + per < ntp) ? t0 + per : ntp;
#pragma unroll
    for (int i = 0; i < PER_T; ++i) {
        if (is_dead(xa[i])) continue;
        int j; float fr;
        cell_of_inside(xa[i], inv_dx, limit, j, fr);
        cnt += (unsigned)j == c ? 1u : 0u;
    }
    unsigned k;
    (void)scan_once(cnt, ws, &k);
    const unsigned m = nm < npl ? nm : npl, M = nm < npl ? npl : nm;
    if (m == 0 || k >= nm) return;   // block-uniform
    const uint4 wr = philox4x32_10(make_uint4((uint32_t)step, Sp.tag_shift, 0u, (uint32_t)(step >> 32)),
                                   make_uint2(c, P.seed));
    const unsigned r = wr.x % M;
    unsigned q;
    if (nm <= npl) {
        q = k + r; if (q >= M) q -= M;
    } else {
        unsigned i = k + (M - r); if (i >= M) i -= M;   // the O2+ of rank i has this O- as partner
        if (i >= m) return;                              // block-uniform
        q = i;
    }
    __syncthreads();   // ws is written again
#pragma unroll 8
    for (unsigned t = t0; t < t1; ++t) gs += H1[(size_t)t * Nc + c];
    unsigned gtot;
    const unsigned gex = scan_once(gs, ws, &gtot);
    if (q >= gtot) return;   // block-uniform (inconsistent counts; never expected)
    // the O2+ tile holding rank q
    if (gex <= q && q < gex + gs) {
        // eight tiles' counts in flight (one by one, each compare waits for its load)
        unsigned run = gex, at = t0;
        bool in = false;
        for (unsigned t = t0; t < t1 && !in; t += 8) {
            unsigned v[8];
#pragma unroll
            for (unsigned i = 0; i < 8; ++i) v[i] = t + i < t1 ? H1[(size_t)(t + i) * Nc + c] : 0u;
#pragma unroll
            for (unsigned i = 0; i < 8; ++i) {
                if (in) continue;
                if (q < run + v[i]) { in = true; at = t + i; }
                else run += v[i];
            }
        }
        sh[0] = at;
        sh[1] = q - run;
    }
    __syncthreads();
    const unsigned lo = sh[0], want = sh[1];
    // the partner's slot: rank `want` among the tile's live O2+ of cell c; warp w
    // takes the w-th eighth of the tile, 32 neighbouring slots per round
    const unsigned long long bb = (unsigned long long)lo * TILE + (unsigned)(warp * PER_T * 32 + lane);
    float xb[PER_T];
#pragma unroll
    for (int i = 0; i < PER_T; ++i) xb[i] = (bb + 32u * i < nsp) ? XP[bb + 32u * i] : dead_marker();
    unsigned hits = 0;      // bit i: round i's slot is one of them
#pragma unroll
    for (int i = 0; i < PER_T; ++i) {
        int j = -1; float fr;
        if (!is_dead(xb[i])) cell_of_inside(xb[i], inv_dx, limit, j, fr);
        if (j == (int)c) hits |= 1u << i;
    }
    unsigned mine = __popc(hits);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if (lane == 0) wc[warp] = mine;
    __syncthreads();
    unsigned before = 0;
#pragma unroll
    for (int w = 0; w < PAIR_T / 32; ++w) before += w < warp ? wc[w] : 0u;
    if (want < before || want >= before + mine) return;   // warp-uniform
    unsigned left = want - before, b_slot = 0;
    bool found = false;
    for (int i = 0; i < PER_T; ++i) {
        const unsigned h = __ballot_sync(0xffffffffu, (hits >> i) & 1u), n = __popc(h);
        if (left < n) {
            found = ((hits >> i) & 1u) && (unsigned)__popc(h & ((1u << lane) - 1u)) == left;
            b_slot = (unsigned)(bb + 32u * i);
            break;
        }
        left -= n;
    }
    if (!found) return;
    // reaction test with the exact probability
    const SpeciesBuf& SM = P.sp[Sp.A];
    const SpeciesBuf& SPp = P.sp[Sp.B];
    const float gx = SM.vx[cm][p] - SPp.vx[cp][b_slot];
    const float gy = SM.vy[cm][p] - SPp.vy[cp][b_slot];
    const float gz = SM.vz[cm][p] - SPp.vz[cp][b_slot];
    const float E = Sp.kappa * dot3(gx, gy, gz, gx, gy, gz);
    int gi; float gw; bool above;
    grid_locate(E, gi, gw, above);
    if (above) atomicAdd(&C->cnt.warn_emax, 1ull);
    const float K = grid_interp(Sp.K, 1, 0, gi, gw);
    const float Pp = K * (P.pair_factor * (float)M);
    if (Pp > 1.0f) ++gt1;
    if (u < Pp && E >= Sp.thr) {
        const unsigned idx = atomicAdd(Sp.nremovals, 1u);
        if (idx < Sp.max_removals) {
            Sp.removal[2 * idx] = p;
            Sp.removal[2 * idx + 1] = b_slot;
        }
        // take both out of the fresh deposit
        int j; float f;
        cell_of(SM.x[cm][p], P.inv_dx, Nc, j, f);
        uint32_t rr = cic_r(f);
        atomicAdd(&P.Qf[Sp.A][j], 0ull - (unsigned long long)(65536u - rr));
        atomicAdd(&P.Qf[Sp.A][j + 1], 0ull - (unsigned long long)rr);
        if (!Sp.b_survives) {
            cell_of(XP[b_slot], inv_dx, Nc, j, f);
            rr = cic_r(f);
            atomicAdd(&P.Qf[Sp.B][j], 0ull - (unsigned long long)(65536u - rr));
            atomicAdd(&P.Qf[Sp.B][j + 1], 0ull - (unsigned long long)rr);
        }
    }
}

// The candidates, one per thread, against the bound with their cell's M; those
// left are resolved one after another by the block.  Block 0 also adds
// sum_c min(n-, n+) to the pair counter.
__device__ __forceinline__ void pair_body(const Params& P, const PairSpec& Sp, unsigned blk, unsigned nblk) {
    __shared__ unsigned list[PAIR_T], cell[PAIR_T];
    __shared__ float draw[PAIR_T];
    __shared__ unsigned ws[32], wc[PAIR_T / 32];
    __shared__ unsigned sh[2];
    __shared__ unsigned nflag;
    DevCtrl* C = P.ctrl;
    const int Nc = P.Nc;
    const int tid = threadIdx.x;
    const unsigned long long step = C->step;
    const unsigned long long nsm = C->slots[Sp.A], nsp = C->slots[Sp.B];
    const unsigned ntp = (unsigned)ceil_div(nsp, TILE);
    const unsigned cm = C->cur[Sp.A], cp = C->cur[Sp.B];
    const float* __restrict__ XM = P.sp[Sp.A].x[cm];
    const unsigned* __restrict__ tot = Sp.tot;
    const unsigned n = *Sp.ncand < nsm ? *Sp.ncand : (unsigned)nsm;
    unsigned gt1 = 0;

    if (blk == 0) {
        unsigned pairs = 0;   // at most 2^32 ions in all
        for (int c = tid; c < Nc; c += PAIR_T) {
            const unsigned a = tot[c], b = tot[Nc + c];
            pairs += a < b ? a : b;
        }
        const unsigned s = block_sum(pairs, ws);
        if (tid == 0 && s) atomicAdd(Sp.tested, (unsigned long long)s);
    }
    for (unsigned e0 = 0; e0 < n; e0 += nblk * PAIR_T) {
        if (tid == 0) nflag = 0u;
        __syncthreads();
        const unsigned e = e0 + (unsigned)tid * nblk + blk;
        if (e < n) {
            const uint2 r = Sp.cand[e];
            int c; float fr;
            cell_of(XM[r.x], P.inv_dx, Nc, c, fr);
            const unsigned a = tot[c], b = tot[Nc + c];
            const unsigned M = a < b ? b : a;
            const float u = uniform(r.y);
            if (u < Sp.Kmax_hi * (P.pair_factor * (float)M)) {
                const unsigned i = atomicAdd(&nflag, 1u);
                list[i] = r.x;
                cell[i] = (unsigned)c;
                draw[i] = u;
            }
        }
        __syncthreads();
        const unsigned nf = nflag;
        for (unsigned j = 0; j < nf; ++j) {
            resolve_one(P, Sp, list[j], draw[j], cell[j], ws, sh, wc, step, nsp, ntp, cm, cp, gt1);
            __syncthreads();   // before the next one writes the shared words
        }
        __syncthreads();
    }
    pdl_trigger();
    if (gt1) atomicAdd(&C->cnt.warn_pair_gt1, (unsigned long long)gt1);
}

// The removals of a pair process that runs before another (16 before 17):
// mark both particles of every listed pair dead, count them, clear the list.
__device__ __forceinline__ void pair_apply_body(const Params& P, const PairSpec& Sp) {
    DevCtrl* C = P.ctrl;
    const unsigned listed = *Sp.nremovals;
    const unsigned n = listed < Sp.max_removals ? listed : Sp.max_removals;
    const unsigned ca = C->cur[Sp.A], cb = C->cur[Sp.B];
    for (unsigned r = threadIdx.x; r < n; r += blockDim.x) {
        P.sp[Sp.A].x[ca][Sp.removal[2 * r]] = dead_marker();
        P.sp[Sp.B].x[cb][Sp.removal[2 * r + 1]] = dead_marker();
    }
    pdl_trigger();
    if (threadIdx.x == 0 && n) {
        atomicAdd(&C->removed[Sp.A], (unsigned long long)n);
        atomicAdd(&C->removed[Sp.B], (unsigned long long)n);
        atomicAdd(Sp.reacted, (unsigned long long)n);
    }
}

// (22) e + O- -> O + 2e: the reacted pairs (O- slot, e slot), listed in any
// order by k_pair, in one block.  Each pair's kinematics continue the O-'s
// stream after its acceptance number: the share u of E_rel - E_th taken by
// the detached electron, then one isotropic direction for each electron; the
// electron keeps going from the O-'s velocity with the rest, the O- is marked
// dead (its charge was taken out by k_pair), and the newborn is staged at the
// rank of its O- parent's slot among the listed pairs (the method's order),
// its charge into the births' deposit.  The end-of-step kernel places the
// newborns after the step's other electron births.
__device__ __forceinline__ void edet_apply_body(const Params& P, const PairSpec& Sp) {
    __shared__ unsigned sh_wtries;
    DevCtrl* C = P.ctrl;
    if (threadIdx.x == 0) sh_wtries = 0u;
    __syncthreads();
    const unsigned listed = *Sp.nremovals;
    const unsigned n = listed < Sp.max_removals ? listed : Sp.max_removals;
    const unsigned long long step = C->step;
    const unsigned ca = C->cur[Sp.A], cb = C->cur[Sp.B];
    const SpeciesBuf& SA = P.sp[Sp.A];
    const SpeciesBuf& SB = P.sp[Sp.B];
    unsigned wtries = 0;
    for (unsigned r = threadIdx.x; r < n; r += blockDim.x) {
        const unsigned a = Sp.removal[2 * r], b = Sp.removal[2 * r + 1];
        unsigned rank = 0;   // slots of the O- are distinct: each reacts once
        for (unsigned q = 0; q < n; ++q) rank += (Sp.removal[2 * q] < a) ? 1u : 0u;
        const float ax = SA.x[ca][a], avx = SA.vx[ca][a], avy = SA.vy[ca][a], avz = SA.vz[ca][a];
        const uint32_t id = SA.id[ca][a];
        const float gx = avx - SB.vx[cb][b], gy = avy - SB.vy[cb][b], gz = avz - SB.vz[cb][b];
        const float E = Sp.kappa * dot3(gx, gy, gz, gx, gy, gz);
        const float Er = E - Sp.thr;
        Stream st;
        st.init(id, P.seed, step, Sp.tag_pair);
        (void)st.next();                         // the acceptance number
        const float us = uniform(st.next());
        const float Es = us * Er;
        const float Ep = Er - Es;
        float n1x, n1y, n1z, n2x, n2y, n2z;
        isotropic(st, n1x, n1y, n1z, wtries);
        isotropic(st, n2x, n2y, n2z, wtries);
        const float vp = sqrtf(Ep / P.kappa[SP_E]);
        const float vs = sqrtf(Es / P.kappa[SP_E]);
        SB.vx[cb][b] = avx + vp * n1x;
        SB.vy[cb][b] = avy + vp * n1y;
        SB.vz[cb][b] = avz + vp * n1z;
        SA.x[ca][a] = dead_marker();
        P.stage22[rank] = make_float4(ax, avx + vs * n2x, avy + vs * n2y, avz + vs * n2z);
        int j; float f;
        cell_of(ax, P.inv_dx, P.Nc, j, f);
        const uint32_t rr = cic_r(f);
        atomicAdd(&P.Qb[SP_E][j], (unsigned long long)(65536u - rr));
        if (rr) atomicAdd(&P.Qb[SP_E][j + 1], (unsigned long long)rr);
    }
    pdl_trigger();
    if (wtries) atomicAdd(&sh_wtries, wtries);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (n) {
            atomicAdd(&C->removed[Sp.A], (unsigned long long)n);
            atomicAdd(Sp.reacted, (unsigned long long)n);
        }
        C->births22 = n;
        if (sh_wtries) atomicAdd(&C->cnt.warn_tries, (unsigned long long)sh_wtries);
    }
}

// Blocks [0, na) count A, the others B.
__global__ void __launch_bounds__(HIST_T, 2) k_pair_count(Params P, PairSpec Sp, unsigned na) {
    if (blockIdx.x < na) pair_count_body<true>(P, Sp, blockIdx.x, na);
    else pair_count_body<false>(P, Sp, blockIdx.x - na, gridDim.x - na);
}

__global__ void __launch_bounds__(PAIR_T) k_pair(Params P, PairSpec Sp) {
    pdl_wait();
    pair_body(P, Sp, blockIdx.x, gridDim.x);
}

// one block: the lists are short
__global__ void k_pair_apply(Params P, PairSpec Sp) {
    pdl_wait();
    pair_apply_body(P, Sp);
}

// batched: block b works for discharge map[b].x (block map[b].y of map[b].z)
// batched: map[b].w = 0 counts A, 1 B
__global__ void __launch_bounds__(HIST_T, 2) k_pair_count_b(const Params* __restrict__ all,
                                                            const PairSpec* __restrict__ specs,
                                                            const uint4* __restrict__ map) {
    __shared__ Params sP;
    const uint4 m = map[blockIdx.x];
    const PairSpec Sp = specs[m.x];
    if (!Sp.active) {         // block-uniform; no block may end before the predecessor has
        pdl_wait();
        return;
    }
    load_params(sP, all + m.x);
    if (m.w == 0u) pair_count_body<true>(sP, Sp, m.y, m.z);
    else pair_count_body<false>(sP, Sp, m.y, m.z);
}

__global__ void __launch_bounds__(PAIR_T) k_pair_b(const Params* __restrict__ all, const PairSpec* __restrict__ specs,
                                                    const uint4* __restrict__ map) {
    __shared__ Params sP;
    pdl_wait();
    const uint4 m = map[blockIdx.x];
    const PairSpec Sp = specs[m.x];
    if (!Sp.active) return;
    load_params(sP, all + m.x);
    pair_body(sP, Sp, m.y, m.z);
}

__global__ void k_edet_apply(Params P, PairSpec Sp) {
    pdl_wait();
    edet_apply_body(P, Sp);
}

// batched: block d applies discharge d's (22) list
__global__ void k_edet_apply_b(const Params* __restrict__ all, const PairSpec* __restrict__ specs) {
    __shared__ Params sP;
    pdl_wait();
    const PairSpec Sp = specs[blockIdx.x];
    if (!Sp.active) return;
    load_params(sP, all + blockIdx.x);
    edet_apply_body(sP, Sp);
}

// batched: block d applies discharge d's list
__global__ void k_pair_apply_b(const Params* __restrict__ all, const PairSpec* __restrict__ specs) {
    __shared__ Params sP;
    pdl_wait();
    const PairSpec Sp = specs[blockIdx.x];
    if (!Sp.active) return;
    load_params(sP, all + blockIdx.x);
    pair_apply_body(sP, Sp);
}

}  // namespace

size_t pair_count_smem_bytes(int Nc) { return 2 * sizeof(unsigned) * (size_t)Nc; }

cudaError_t configure_pair_count_smem(int Nc) {
    cudaError_t e = cudaFuncSetAttribute(k_pair_count, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)pair_count_smem_bytes(Nc));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_pair_count_b, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)pair_count_smem_bytes(Nc));
    return e;
}

void launch_pair_count(const Params& P, const PairSpec& S, int na, int nb, cudaStream_t s) {
    launch_pdl(k_pair_count, na + nb, HIST_T, pair_count_smem_bytes(P.Nc), s, P, S, (unsigned)na);
}

void launch_pair(const Params& P, const PairSpec& S, int grid, cudaStream_t s) {
    launch_pdl(k_pair, grid, PAIR_T, 0, s, P, S);
}

// the list counter is cleared by the end-of-step kernel
void launch_pair_apply(const Params& P, const PairSpec& S, cudaStream_t s) {
    launch_pdl(k_pair_apply, 1, 256, 0, s, P, S);
}

void launch_edet_apply(const Params& P, const PairSpec& S, cudaStream_t s) {
    launch_pdl(k_edet_apply, 1, 256, 0, s, P, S);
}

void launch_edet_apply_batched(const Params* all, const PairSpec* specs, int n, cudaStream_t s) {
    launch_pdl(k_edet_apply_b, n, 256, 0, s, all, specs);
}

void launch_pair_count_batched(const Params* all, const PairSpec* specs, const uint4* map, int nblocks, size_t smem,
                               cudaStream_t s) {
    launch_pdl(k_pair_count_b, nblocks, HIST_T, smem, s, all, specs, map);
}

void launch_pair_batched(const Params* all, const PairSpec* specs, const uint4* map, int nblocks, cudaStream_t s) {
    launch_pdl(k_pair_b, nblocks, PAIR_T, 0, s, all, specs, map);
}

void launch_pair_apply_batched(const Params* all, const PairSpec* specs, int n, cudaStream_t s) {
    launch_pdl(k_pair_apply_b, n, 256, 0, s, all, specs);
}

}  // namespace o2
