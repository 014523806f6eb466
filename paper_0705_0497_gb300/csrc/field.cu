// End-of-step kernel (two clusters of blocks): charge commit, cycle moments,
// Poisson solve and E on the nodes; placement of the step's births, removals of (17) and the
// commit of the step; plus the stable compaction of dead slots and small
// utility kernels.
//
// Poisson (Sec. 2): interior nodes satisfy
//     -phi_{j-1} + 2 phi_j - phi_{j+1} = rho_j dx^2 / eps0,
// phi_0 = U sin(2 pi f t) (driven electrode at x = 0), phi_N = 0 (grounded).
// With the net fixed-point charge R_j (2^16 per macro-particle, exact int64)
// and c = e w dx / (A eps0 2^16), the system is solved in closed form by
// exact integer prefix sums (one scan of the pair S, U over a cluster):
//     S_m = sum_{k=1..m} R_k,  U_m = sum_{k=1..m} k R_k,
//     T_j = sum_{m<j} S_m = j S_{j-1} - U_{j-1},
//     D_0 = phi_1 - phi_0 = (c T_N - V0) / N,  phi_j = V0 + j D_0 - c T_j,
//     E_j = (c (S_j + S_{j-1}) - 2 D_0) [1/(2 dx)]         (1 <= j <= N-1),
//     E_0 = (-D_0 - c R_0) [1/dx],  E_N = (c S_{N-1} - D_0 + c R_N) [1/dx]
// (wall nodes from Gauss's law over the half cell next to the wall).  This is
// the exact solution of the linear system a Thomas sweep would solve; it
// needs no serial FP64 recurrence (FP64 throughput on this GPU is low), its
// only rounding is in the final FP64 expressions, each evaluated in the order
// written here.  |S| <= 2^47 and |T| <= 2^58 for up to 2^31 particles and 8192
// cells, so int64 holds both exactly.
#include <algorithm>

#include "compact.cuh"

namespace o2 {

namespace {

// The end-of-step kernel is two independent clusters of FC blocks of FT threads
// (one pair per discharge of a batched launch): cluster 0 commits the charge
// and solves the field, cluster 1 places the births and commits the step.  They
// share nothing; cluster 0 keeps its own copy of the step counter (field_step)
// for U sin(2 pi f t).
//
// Bound by latency (a few dependent L2 round trips of 0.45 us) and, in a
// single block, by one SM's FP64 and int64 conversion rate (513 nodes: 0.8
// us) and outstanding misses.  So the nodes, and the births, are spread over
// the FC SMs of a cluster; the field's blocks exchange their partial sums
// once through distributed shared memory, and the births' blocks each scan
// all counts (a thread takes whole particle-kernel blocks of 8 warps).  512
// cells: 13.3 us between events (two blocks of 512 threads) -> 10.5, of which
// the launch is about 4.8; 2048 cells 26 -> 12.6.
constexpr int FT = 256;
constexpr int FC = 8;                             // blocks of a cluster
constexpr int FW = FT / 32;
constexpr int FN = (MAX_NODES + FC * FT - 1) / (FC * FT);   // nodes per thread, at most (5)
constexpr int PW = BLOCK / 32;                    // warps of a particle-kernel block

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Cluster barrier (not the .aligned form, which needs a converged warp: the
// loops before a barrier diverge).
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// v into the same shared-memory word of block `rank` of the cluster
__device__ __forceinline__ void store_remote(long long* p, unsigned rank, long long v) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("{ .reg .b32 r; mapa.shared::cluster.u32 r, %0, %1; st.shared::cluster.s64 [r], %2; }" ::"r"(a),
                 "r"(rank), "l"(v)
                 : "memory");
}

// Births of one step, placed in the order the method defines (source species
// e then O-, parent order, e before O2+ for an ionization): each warp of a
// particle kernel staged the births of its slot range [u R, ...) with their
// count (their charge already went to Qb there).  The counts are scanned into
// per-block offsets in shared memory, and every thread of the births cluster
// then places single births (found by a binary search over the offsets and the
// counts of the block's warps), so the work spreads however the births cluster.
// A newborn of step n starts a free flight at its first push after n (step
// n + 1 for electrons, the next ion step for ions), drawn from its own stream
// at step n with tag TAG_FLIGHT + d.
__device__ void place_birth(const Params& P, DevCtrl* C, const unsigned cur[NSP], int d, unsigned long long slot,
                            unsigned long long id64, float4 b, unsigned long long n) {
    const SpeciesBuf& B = P.sp[d];
    if (slot >= B.cap) { atomicOr(&C->error_flags, ERR_CAPACITY); return; }
    // ids are 32-bit: a birth whose id would be 2^32 or more overflows
    // (counted per birth; the particle keeps the low 32 bits)
    if (id64 > 0xFFFFFFFFull) {
        atomicOr(&C->error_flags, ERR_ID);
        atomicAdd(&C->cnt.id_overflow, 1ull);
    }
    const unsigned cb = cur[d];
    const uint32_t id = (uint32_t)id64;
    const unsigned sub = P.sub[d];
    const uint32_t nf = (uint32_t)((n + sub) / sub * sub);
    const uint4 w = philox4x32_10(make_uint4((uint32_t)n, TAG_FLIGHT + (uint32_t)d, 0u, (uint32_t)(n >> 32)),
                                  make_uint2(id, P.seed));
    B.x[cb][slot] = b.x;
    B.vx[cb][slot] = b.y;
    B.vy[cb][slot] = b.z;
    B.vz[cb][slot] = b.w;
    B.id[cb][slot] = id;
    B.tc[cb][slot] = nf + sub * flight_gap(w.x, P.inv_lnq[d], P.kcap[d]);
}

// Exclusive scan over the block of two 64-bit values per thread (words: two
// 32-bit counts each), with the totals.
__device__ __forceinline__ void block_excl_scan_pair(unsigned long long v, unsigned long long w,
                                                     unsigned long long* ws, unsigned long long& ev,
                                                     unsigned long long& ew, unsigned long long& tv,
                                                     unsigned long long& tw) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long x = v, y = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long xo = __shfl_up_sync(0xffffffffu, x, o);
        const unsigned long long yo = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= o) { x += xo; y += yo; }
    }
    if (lane == 31) { ws[warp] = x; ws[FW + warp] = y; }
    __syncthreads();
    ev = x - v;
    ew = y - w;
    tv = tw = 0ull;
#pragma unroll
    for (int k = 0; k < FW; ++k) {
        const unsigned long long a = ws[k], b = ws[FW + k];
        if (k < warp) { ev += a; ew += b; }
        tv += a;
        tw += b;
    }
}

// The birth counts of one particle-kernel block's PW warps.
struct WarpCounts {
    uint4 a, b;
    __device__ __forceinline__ void load(const unsigned* c, unsigned blk) {
        const uint4* p = reinterpret_cast<const uint4*>(c + (size_t)blk * PW);
        a = p[0];
        b = p[1];
    }
    __device__ __forceinline__ unsigned sum() const { return a.x + a.y + a.z + a.w + b.x + b.y + b.z + b.w; }
    // the warp that staged the block's birth number r (r < sum()); r becomes its
    // rank among that warp's
    __device__ __forceinline__ unsigned warp_of(unsigned& r) const {
        const unsigned n[PW] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        unsigned u = 0;
        bool found = false;
#pragma unroll
        for (int k = 0; k < PW; ++k) {
            if (!found && r < n[k]) { u = k; found = true; }
            if (!found) r -= n[k];
        }
        return u;
    }
};
static_assert(PW == 8, "two 16-byte words of counts per block");

// The block whose births hold number b (largest u with p[u] <= b).
__device__ __forceinline__ unsigned find_unit(const unsigned* p, unsigned nu, unsigned b) {
    unsigned lo = 0, hi = nu;
    while (hi - lo > 1) {
        const unsigned mid = (lo + hi) >> 1;
        if (p[mid] <= b) lo = mid; else hi = mid;
    }
    return lo;
}

struct CtrlSnap {
    unsigned long long step, epoch, acc_steps, slots[NSP], live[NSP], removed[NSP];
    unsigned long long next_id[NSP];
    unsigned cur[NSP], removals, births22;
};

// The charge commit, cycle moments and field solve of one block (rank cr) of
// the field cluster: nodes [cr per, (cr + 1) per), a few neighbouring ones per
// thread.  mode 0: end of a step (pushed_mask = species pushed this step);
// mode 1: after a load (all species freshly deposited into Qf).
__device__ __forceinline__ void field_solve(const Params& P, int mode, int pushed_mask, unsigned cr) {
    __shared__ long long ws[2 * FW];
    __shared__ long long part[2 * FC];     // the cluster's partial sums, written by its blocks
    DevCtrl* C = P.ctrl;
    const int N = P.Nc, Ng = P.Ng;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int per = (Ng + FC - 1) / FC, pt = (per + FT - 1) / FT;
    const int c0 = (int)cr * per, c1 = min(Ng, c0 + per), j0 = c0 + t * pt;
    cluster_arrive();                      // this block runs (before others write to its shared memory)
    // U sin(2 pi f t) at t^{n+1} (end of step) or t^n (after a load), evaluated
    // on the host in FP64 and staged in a ring indexed by the step; D0 needs it
    // in one lane per warp
    unsigned long long fstep = 0ull;
    double V0 = 0.0;
    if (lane == 0) fstep = C->field_step;
    // Q = (this step's deposit Qf, or the kept Q of a species not pushed) + the
    // births' deposit Qb, and the cycle moments Qacc += Q
    long long r[FN], net[FN];
#pragma unroll
    for (int i = 0; i < FN; ++i) {
        const int j = j0 + i;
        r[i] = 0;
        net[i] = 0;
        if (i >= pt || j >= c1) continue;
        unsigned long long q[NSP], qa[NSP];
#pragma unroll
        for (int s = 0; s < NSP; ++s) {
            qa[s] = (mode == 0) ? P.Qacc[s][j] : 0ull;
            unsigned long long v = P.Qb[s][j];
            if ((mode == 1) || ((pushed_mask >> s) & 1)) {
#pragma unroll
                for (int k = 0; k < QCOPIES; ++k) v += P.Qf[s][(size_t)k * Ng + j];
            } else {
                v += P.Q[s][j];
            }
            q[s] = v;
        }
#pragma unroll
        for (int s = 0; s < NSP; ++s) {
            P.Q[s][j] = q[s];
            if (mode == 0) P.Qacc[s][j] = qa[s] + q[s];
            P.Qf[s][j] = 0ull;
            if ((mode == 1) || ((pushed_mask >> s) & 1)) {   // only pushes fill copies 1..
#pragma unroll
                for (int k = 1; k < QCOPIES; ++k) P.Qf[s][(size_t)k * Ng + j] = 0ull;
            }
            P.Qb[s][j] = 0ull;
            net[i] += (s == SP_OP) ? (long long)q[s] : -(long long)q[s];
        }
        if (j >= 1 && j < N) r[i] = net[i];
    }
    // the scans of R_j and j R_j (j = 1 .. N - 1) over the cluster
    long long a = 0, b = 0;
#pragma unroll
    for (int i = 0; i < FN; ++i) { a += r[i]; b += (long long)(j0 + i) * r[i]; }
    long long xa = a, xb = b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long ya = __shfl_up_sync(0xffffffffu, xa, o);
        const long long yb = __shfl_up_sync(0xffffffffu, xb, o);
        if (lane >= o) { xa += ya; xb += yb; }
    }
    if (lane == 31) { ws[warp] = xa; ws[FW + warp] = xb; }
    if (lane == 0) V0 = P.vring[(mode == 0 ? fstep + 1 : fstep) & P.vring_mask];
    __syncthreads();
    long long sa = xa - a, sb = xb - b;    // exclusive, over the block
#pragma unroll
    for (int k = 0; k < FW - 1; ++k)
        if (k < warp) { sa += ws[k]; sb += ws[FW + k]; }
    cluster_wait();
    if (t < 2 * FC) {
        const int h = t & 1;               // 0: S, 1: U
        long long tot = 0;
#pragma unroll
        for (int k = 0; k < FW; ++k) tot += ws[h * FW + k];
        store_remote(&part[h * FC + cr], (unsigned)t >> 1, tot);
    }
    cluster_arrive();
    cluster_wait();
    long long ta = 0, tb = 0;              // over the cluster: S_{N-1}, U_{N-1}
#pragma unroll
    for (int k = 0; k < FC; ++k) {
        const long long pa = part[k], pb = part[FC + k];
        if (k < (int)cr) { sa += pa; sb += pb; }
        ta += pa;
        tb += pb;
    }
    // D0 in one lane per warp: FP64 throughput on this GPU is low
    const double c = P.c_field;
    double D0 = 0.0;
    if (lane == 0) {
        const long long TN = (long long)N * ta - tb;
        // a power-of-two N divides exactly by its reciprocal (same IEEE
        // result as the division, which is slow in FP64 here)
        const double num = c * (double)TN - V0;
        D0 = (P.inv_Nc64 != 0.0) ? num * P.inv_Nc64 : num / (double)N;
        if (cr == 0 && warp == 0) {
            P.fVD[0] = V0;
            P.fVD[1] = D0;
            if (mode == 0) C->field_step = fstep + 1;   // read by this cluster only, before its barrier
        }
    }
    D0 = __shfl_sync(0xffffffffu, D0, 0);
    // E on the nodes (what the next push gathers).  The potential needs as
    // much FP64 work again and only diagnostics read it: S, U, V0 and D0
    // are kept so that k_phi evaluates it with the same expressions.
    const double D2 = 2.0 * D0;            // exact
#pragma unroll
    for (int i = 0; i < FN; ++i) {
        const int j = j0 + i;
        if (i >= pt || j >= c1) continue;
        const long long below = sa;        // S_{j-1}
        sa += r[i];
        sb += (long long)j * r[i];
        double E;
        if (j == 0) E = (-D0 - c * (double)net[i]) * P.inv_dx64;
        else if (j == N) E = (c * (double)ta - D0 + c * (double)net[i]) * P.inv_dx64;
        else E = (c * (double)(sa + below) - D2) * P.inv_2dx64;
        P.Ef[j] = (float)E;
        P.fS[j] = sa;
        P.fU[j] = sb;
    }
}

// Births, (17) removals and the commit of the step, by one block (rank cr) of
// the births cluster.  Dynamic shared memory: three u32 [units + 1].
__device__ __forceinline__ void step_commit(const Params& P, int mode, int pushed_mask, unsigned cr) {
    __shared__ unsigned long long ws[2 * FW];
    __shared__ CtrlSnap cs;
    extern __shared__ unsigned fsm[];
    DevCtrl* C = P.ctrl;
    const int N = P.Nc, t = threadIdx.x;
    const unsigned ct = cr * FT + (unsigned)t;            // thread of the cluster
    constexpr unsigned CT = FC * FT;
    unsigned* p1 = fsm;
    unsigned* p2 = p1 + (P.max_push_warps / PW + 1);
    unsigned* p3 = p2 + (P.max_push_warps / PW + 1);
    const bool births_e = mode == 0 && P.births_possible[SP_E];
    const bool births_om = mode == 0 && ((pushed_mask >> SP_OM) & 1) && P.births_possible[SP_OM];
    if (t < NSP) {
        cs.slots[t] = C->slots[t]; cs.live[t] = C->live[t]; cs.removed[t] = C->removed[t];
        cs.next_id[t] = C->next_id[t]; cs.cur[t] = C->cur[t];
    } else if (t == 32) {
        cs.step = C->step;
        cs.epoch = C->epoch;
        cs.acc_steps = C->acc_steps;
        cs.removals = C->removals;
        cs.births22 = C->births22;
    }
    // births of the step: n1 ionizations (e + O2+) and n2 attachments (O-)
    // staged by the electron kernel, n3 detachment electrons staged by the O-
    // kernel (ion steps), placed after the electrons' own, then n4 electrons
    // of (22) staged in order by its apply kernel (ion steps).  Offsets of the
    // particle-kernel blocks' counts by one scan: a thread owns `ub`
    // neighbouring blocks
    const unsigned nu1 = births_e ? P.push_warps[SP_E] / PW : 0u, nu3 = births_om ? P.push_warps[SP_OM] / PW : 0u;
    const unsigned nu = nu1 > nu3 ? nu1 : nu3, ub = (nu + FT - 1) / FT, u0 = (unsigned)t * ub;
    unsigned long long m12 = 0, m3 = 0, t12 = 0, t3 = 0;
    for (unsigned i = 0; i < ub; ++i) {
        const unsigned u = u0 + i;
        WarpCounts a, b, d;
        if (u < nu1) { a.load(P.wcount[B_E_FROM_E], u); b.load(P.wcount[B_OM_FROM_E], u); }
        if (u < nu3) d.load(P.wcount[B_E_FROM_OM], u);
        if (u < nu1) {
            const unsigned sa = a.sum(), sb = b.sum();
            p1[u] = sa;
            p2[u] = sb;
            m12 += (unsigned long long)sa | ((unsigned long long)sb << 32);
        }
        if (u < nu3) { const unsigned sd = d.sum(); p3[u] = sd; m3 += sd; }
    }
    unsigned long long e12, e3;
    block_excl_scan_pair(m12, m3, ws, e12, e3, t12, t3);
    cluster_arrive();                      // every block has its snapshot of the step state
    {
        unsigned r1 = (unsigned)e12, r2 = (unsigned)(e12 >> 32), r3 = (unsigned)e3;
        for (unsigned i = 0; i < ub; ++i) {
            const unsigned u = u0 + i;
            if (u < nu1) { const unsigned x = p1[u], y = p2[u]; p1[u] = r1; p2[u] = r2; r1 += x; r2 += y; }
            if (u < nu3) { const unsigned z = p3[u]; p3[u] = r3; r3 += z; }
        }
    }
    __syncthreads();
    const unsigned n1 = (unsigned)t12, n2 = (unsigned)(t12 >> 32), n3 = (unsigned)t3;
    const unsigned n4 = (mode == 0) ? cs.births22 : 0u;
    const unsigned ntot = n1 + n2 + n3 + n4;
    const unsigned ns1 = (unsigned)(cs.slots[SP_E] < P.sp[SP_E].cap ? cs.slots[SP_E] : P.sp[SP_E].cap);
    const unsigned ns3 = (unsigned)(cs.slots[SP_OM] < P.sp[SP_OM].cap ? cs.slots[SP_OM] : P.sp[SP_OM].cap);
    const unsigned R1 = warp_range_len(ns1, nu1 ? nu1 * PW : 1u), R3 = warp_range_len(ns3, nu3 ? nu3 * PW : 1u);
    // one birth per thread and pass: which list, its rank there, the warp that
    // staged it and its staging slot; all loads of the birth before its stores
    for (unsigned b = ct; b < ntot; b += CT) {
        if (b >= n1 + n2 + n3) {   // (22): staged in place order
            const unsigned r = b - n1 - n2 - n3;
            place_birth(P, C, cs.cur, SP_E, cs.slots[SP_E] + n1 + n3 + r,
                        (unsigned long long)cs.next_id[SP_E] + n1 + n3 + r, P.stage22[r], cs.step);
            continue;
        }
        const int kind = b < n1 ? 0 : (b < n1 + n2 ? 1 : 2);
        const unsigned r = kind == 0 ? b : (kind == 1 ? b - n1 : b - n1 - n2);
        const unsigned* p = kind == 0 ? p1 : (kind == 1 ? p2 : p3);
        const unsigned R = kind == 2 ? R3 : R1, ns = kind == 2 ? ns3 : ns1;
        const unsigned blk = find_unit(p, kind == 2 ? nu3 : nu1, r);
        WarpCounts wc;
        wc.load(P.wcount[kind == 0 ? B_E_FROM_E : (kind == 1 ? B_OM_FROM_E : B_E_FROM_OM)], blk);
        unsigned rank = r - p[blk];
        const unsigned long long u = (unsigned long long)blk * PW + wc.warp_of(rank);
        const unsigned long long sb = (u * R < ns ? u * R : ns) + rank;
        if (kind == 0) {
            const float4 be = P.stage[B_E_FROM_E][sb], bo = P.stage[B_OP_FROM_E][sb];
            place_birth(P, C, cs.cur, SP_E, cs.slots[SP_E] + r, (unsigned long long)cs.next_id[SP_E] + r, be,
                        cs.step);
            place_birth(P, C, cs.cur, SP_OP, cs.slots[SP_OP] + r, (unsigned long long)cs.next_id[SP_OP] + r, bo,
                        cs.step);
        } else if (kind == 1) {
            place_birth(P, C, cs.cur, SP_OM, cs.slots[SP_OM] + r, (unsigned long long)cs.next_id[SP_OM] + r,
                        P.stage[B_OM_FROM_E][sb], cs.step);
        } else {
            place_birth(P, C, cs.cur, SP_E, cs.slots[SP_E] + n1 + r, (unsigned long long)cs.next_id[SP_E] + n1 + r,
                        P.stage[B_E_FROM_OM][sb], cs.step);
        }
    }
    const unsigned long long btot[NB] = {n1, n1, n2, n3 + n4};   // by BirthSlot
    // (17) removals: mark both ions of every reacted pair dead
    const unsigned nrem = (mode != 0) ? 0u : (cs.removals < P.max_removals) ? cs.removals : P.max_removals;
    for (unsigned r = ct; r < nrem; r += CT) {
        P.sp[SP_OM].x[cs.cur[SP_OM]][P.removal[2 * r]] = dead_marker();
        P.sp[SP_OP].x[cs.cur[SP_OP]][P.removal[2 * r + 1]] = dead_marker();
    }
    // per-cell totals of the pair processes: zero for the next ion step
    if (mode != 0 || pushed_mask != 1)
        for (unsigned k = ct; k < 2u * N; k += CT) { P.ptot[k] = 0u; P.rtot[k] = 0u; P.dtot[k] = 0u; }
    if (mode != 0)   // the ring of conduction-current sums restarts
        for (unsigned k = ct; k < JRING * NSP; k += CT) P.jring[k] = 0ull;
    cluster_wait();
    if (cr != 0) return;
    const int tB = t;
    if (mode == 0) {
        // commit of the step: one thread per species, then the step counters
        if (tB < NSP) {
            const int s = tB;
            const unsigned long long bs = (s == SP_E) ? btot[B_E_FROM_E] + btot[B_E_FROM_OM]
                                                      : (s == SP_OP ? btot[B_OP_FROM_E] : btot[B_OM_FROM_E]);
            const unsigned long long rem = cs.removed[s] + ((s != SP_E) ? (unsigned long long)nrem : 0ull);
            unsigned long long ns = cs.slots[s] + bs;
            unsigned long long nl = cs.live[s] + bs - rem;
            if (ns > P.sp[s].cap) {   // births beyond the capacity were dropped
                atomicOr(&C->error_flags, ERR_CAPACITY);
                nl -= (ns - P.sp[s].cap) < nl ? (ns - P.sp[s].cap) : nl;
                ns = P.sp[s].cap;
            }
            C->slots[s] = ns;
            C->live[s] = nl;
            C->next_id[s] = cs.next_id[s] + bs;
            C->removed[s] = 0ull;
            if (bs) atomicAdd(&C->cnt.born[s], bs);
        } else if (tB == 32) {
            if (nrem) atomicAdd(&C->cnt.neutralized, (unsigned long long)nrem);
            // this block is the only writer of the step state: plain stores
            C->removals = 0u;
            C->rremovals = 0u;
            C->dremovals = 0u;
            C->births22 = 0u;
            C->pcand[0] = C->pcand[1] = C->pcand[2] = 0u;
            C->acc_steps = cs.acc_steps + 1;
            C->step = cs.step + 1;
            C->epoch = cs.epoch + 1;
        } else if (tB >= 64 && tB < 64 + NSP) {
            C->ticket[tB - 64] = 0u;
        }
    }
    // conduction-current sums: at the end of step n the ions' entries of a step
    // without an ion push repeat those of step n-1, and the slot of step n+1 is
    // cleared for its pushes
    if (mode != 0) {
        if (tB < NSP) C->ticket[tB] = 0u;
    } else if (tB >= 96 && tB < 96 + NSP) {
        const int sp = tB - 96;
        const unsigned long long n = cs.step;
        if (sp != SP_E && !((pushed_mask >> sp) & 1))
            P.jring[(n & (JRING - 1)) * NSP + sp] = P.jring[((n - 1) & (JRING - 1)) * NSP + sp];
        P.jring[((n + 1) & (JRING - 1)) * NSP + sp] = 0ull;
    }
}

// Stable compaction of the live slots of one species into the other buffer,
// when more than a fraction of the slots is dead.
__device__ __forceinline__ void compact_body(const Params& P, int S, CompactShared& sh) {
    DevCtrl* C = P.ctrl;
    // One thread decides for the block: the block of the last tile writes the
    // new counts while blocks may still be starting, and the threads of one of
    // those must not differ.  (Such a block claims no tile, whatever mixture of
    // counts it sees: all tiles are claimed by then.)
    if (threadIdx.x == 0) {
        const unsigned long long n = C->slots[S];
        const unsigned long long dead = n - C->live[S];
        const bool many_dead = (double)dead > (double)P.compact_dead_frac * (double)n;
        const bool near_full = dead > 0 && 4 * n > 3 * P.sp[S].cap;
        sh.excl = n;
        sh.tile = C->cur[S];
        sh.ok = (many_dead || near_full) ? 1 : 0;
    }
    __syncthreads();
    const unsigned long long nslots = sh.excl;
    const unsigned cb = sh.tile, nb = cb ^ 1u;
    const bool go = sh.ok != 0;
    __syncthreads();
    if (!go) return;
    const SpeciesBuf& B = P.sp[S];
    const unsigned long long cap = B.cap;
    compact_tiles(
        sh, B.x[cb], nslots, &C->ticket[S], P.lb_flag[S], P.lb_val[S], C->epoch, &C->error_flags,
        [&](unsigned long long p) {
            prefetch_l2(B.vx[cb] + p); prefetch_l2(B.vy[cb] + p); prefetch_l2(B.vz[cb] + p);
            prefetch_l2(B.id[cb] + p); prefetch_l2(B.tc[cb] + p);
        },
        [&](const float (&x)[CMP_I], unsigned long long base, unsigned long long d, const unsigned (&off)[CMP_I],
            unsigned in) {
#pragma unroll
            for (int i = 0; i < CMP_I; ++i)
                if (((in >> i) & 1u) && d + off[i] < cap) B.x[nb][d + off[i]] = x[i];
            move_array(B.vx[nb], B.vx[cb], base, d, off, in, cap);
            move_array(B.vy[nb], B.vy[cb], base, d, off, in, cap);
            move_array(B.vz[nb], B.vz[cb], base, d, off, in, cap);
            move_array(B.id[nb], B.id[cb], base, d, off, in, cap);
            move_array(B.tc[nb], B.tc[cb], base, d, off, in, cap);
        },
        [&](unsigned long long kept) {
            C->slots[S] = kept;
            C->live[S] = kept;
            C->cur[S] = nb;
        });
}

__device__ __forceinline__ void field_body(const Params& P, int mode, int pushed_mask, unsigned cluster) {
    if (cluster == 0) field_solve(P, mode, pushed_mask, cluster_rank());
    else step_commit(P, mode, pushed_mask, cluster_rank());
}

__global__ void __cluster_dims__(FC, 1, 1) __launch_bounds__(FT) k_field(Params P, int mode, int pushed_mask) {
    pdl_wait();
    pdl_trigger();   // a few SMs: the next step's push may take the others
    field_body(P, mode, pushed_mask, blockIdx.x / FC);
}

// batched: clusters 2d and 2d + 1 are the end-of-step kernel of discharge d
__global__ void __cluster_dims__(FC, 1, 1) __launch_bounds__(FT) k_field_b(const Params* __restrict__ all, int mode,
                                                                           int pushed_mask) {
    __shared__ Params sP;
    load_params(sP, all + blockIdx.x / (2 * FC));
    pdl_wait();
    pdl_trigger();
    field_body(sP, mode, pushed_mask, (blockIdx.x / FC) & 1u);
}

// The compaction check of all species: blockIdx.y is the species.
__global__ void __launch_bounds__(CMP_T, 2) k_compact(Params P) {
    __shared__ CompactShared sh;
    pdl_wait();
    compact_body(P, (int)blockIdx.y, sh);
}

// batched: the blocks of map[b].x claim that discharge's tiles of species
// map[b].w by its own ticket
__global__ void __launch_bounds__(CMP_T, 2) k_compact_b(const Params* __restrict__ all, const uint4* __restrict__ map) {
    __shared__ CompactShared sh;
    pdl_wait();
    const uint4 m = map[blockIdx.x];
    compact_body(all[m.x], (int)m.w, sh);
}

// Stable copy of the live particles of a species into caller buffers (a
// caller may ask for the flights alone).
__global__ void __launch_bounds__(CMP_T, 2) k_gather(Params P, int S, unsigned long long epoch, unsigned* ticket,
                                                     unsigned long long* flag, unsigned long long* val, float* ox,
                                                     float* ovx, float* ovy, float* ovz, uint32_t* oid, uint32_t* otc,
                                                     unsigned long long ocap, unsigned long long* out_count) {
    __shared__ CompactShared sh;
    DevCtrl* C = P.ctrl;
    const SpeciesBuf& B = P.sp[S];
    const unsigned cb = C->cur[S];
    compact_tiles(
        sh, B.x[cb], C->slots[S], ticket, flag, val, epoch, &C->error_flags,
        [&](unsigned long long p) {
            if (ox) {
                prefetch_l2(B.vx[cb] + p); prefetch_l2(B.vy[cb] + p); prefetch_l2(B.vz[cb] + p);
                prefetch_l2(B.id[cb] + p);
            }
            if (otc) prefetch_l2(B.tc[cb] + p);
        },
        [&](const float (&x)[CMP_I], unsigned long long base, unsigned long long d, const unsigned (&off)[CMP_I],
            unsigned in) {
            if (ox) {
#pragma unroll
                for (int i = 0; i < CMP_I; ++i)
                    if (((in >> i) & 1u) && d + off[i] < ocap) ox[d + off[i]] = x[i];
                move_array(ovx, B.vx[cb], base, d, off, in, ocap);
                move_array(ovy, B.vy[cb], base, d, off, in, ocap);
                move_array(ovz, B.vz[cb], base, d, off, in, ocap);
                move_array(oid, B.id[cb], base, d, off, in, ocap);
            }
            if (otc) move_array(otc, B.tc[cb], base, d, off, in, ocap);
        },
        [&](unsigned long long kept) { *out_count = kept; });
}

// Validation of freshly loaded particles (x in [0, L), finite velocities)
// and the largest id (+1) for the species' next id.  Bound by HBM (20 B per
// particle, the five loads of a particle in flight together) as long as one
// thread per block touches the two words: with one atomic per thread on the
// same word 0.73 ms for 1.4e6 and for 5.7e6 particles alike.  Reading and
// loading a 512-cell discharge from the host 4.94 -> 3.38 ms.
constexpr int LOAD_T = 256, LOAD_BLOCKS = 8 * 152;   // one wave of 152 SMs, 2048 threads each

template <int S>
__global__ void __launch_bounds__(LOAD_T) k_load_check(Params P, unsigned long long n) {
    __shared__ unsigned wmax[LOAD_T / 32];
    DevCtrl* C = P.ctrl;
    const unsigned cb = C->cur[S];
    const float* __restrict__ X = P.sp[S].x[cb];
    const float* __restrict__ VX = P.sp[S].vx[cb];
    const float* __restrict__ VY = P.sp[S].vy[cb];
    const float* __restrict__ VZ = P.sp[S].vz[cb];
    const uint32_t* __restrict__ ID = P.sp[S].id[cb];
    unsigned mx = 0;
    bool bad = false;
    const unsigned long long first = blockIdx.x * (unsigned long long)LOAD_T;
#pragma unroll 2
    for (unsigned long long i = first + threadIdx.x; i < n; i += (unsigned long long)gridDim.x * LOAD_T) {
        const float x = X[i], vx = VX[i], vy = VY[i], vz = VZ[i];
        const unsigned id = ID[i];
        bad |= !(x >= 0.0f && x < P.Lf) | !isfinite(vx) | !isfinite(vy) | !isfinite(vz);
        mx = id > mx ? id : mx;
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mx;
    const int any_bad = __syncthreads_or(bad);
    if (threadIdx.x != 0 || first >= n) return;   // first < n: the block has a particle
    for (int w = 1; w < LOAD_T / 32; ++w) mx = wmax[w] > mx ? wmax[w] : mx;
    if (any_bad) atomicOr(&C->error_flags, ERR_NONFINITE);
    atomicMax(&C->next_id[S], (unsigned long long)mx + 1ull);
}

__global__ void k_philox(const uint32_t* ctr, const uint32_t* key, uint32_t* out, unsigned long long n) {
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
        const uint4 r = philox4x32_10(c, make_uint2(key[2 * i], key[2 * i + 1]));
        out[4 * i] = r.x; out[4 * i + 1] = r.y; out[4 * i + 2] = r.z; out[4 * i + 3] = r.w;
    }
}

__global__ void k_ln(const float* x, float* out, unsigned long long n) {
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x)
        out[i] = ln_series(x[i]);
}

}  // namespace

size_t field_smem_bytes(const Params& P) {
    return 3 * sizeof(unsigned) * ((size_t)P.max_push_warps / PW + 1);
}

// The potential of the last field solve: phi_0 = V0, phi_N = 0,
// phi_j = V0 + j D0 - c T_j with T_j = j S_{j-1} - U_{j-1} (FP64, the
// expressions of the closed-form solve).
__global__ void k_phi(Params P) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int N = P.Nc;
    if (j > N) return;
    const double V0 = P.fVD[0], D0 = P.fVD[1], c = P.c_field;
    const long long Tj = (j >= 1) ? (long long)j * P.fS[j - 1] - P.fU[j - 1] : 0;
    P.phi[j] = (j == 0) ? V0 : (j == N ? 0.0 : V0 + (double)j * D0 - c * (double)Tj);
}

void launch_phi(const Params& P, cudaStream_t s) {
    k_phi<<<(P.Ng + 255) / 256, 256, 0, s>>>(P);
}

void launch_field_batched(const Params* all, int n, size_t smem, int mode, int pushed_mask, cudaStream_t s) {
    launch_pdl(k_field_b, 2 * FC * n, FT, smem, s, all, mode, pushed_mask);
}

void launch_compact_batched(const Params* all, const uint4* map, int nblocks, cudaStream_t s) {
    launch_pdl(k_compact_b, nblocks, CMP_T, 0, s, all, map);
}

void launch_field(const Params& P, int mode, int pushed_mask, cudaStream_t s) {
    launch_pdl(k_field, 2 * FC, FT, field_smem_bytes(P), s, P, mode, pushed_mask);
}

cudaError_t configure_field_smem(size_t bytes) {
    cudaError_t e = cudaFuncSetAttribute(k_field, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_field_b, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    return e;
}

// `grid` blocks per species (two per SM are resident)
void launch_compact(const Params& P, int grid, cudaStream_t s) {
    launch_pdl(k_compact, dim3(grid, NSP), CMP_T, 0, s, P);
}

void launch_gather(int species, const Params& P, int grid, unsigned long long epoch, unsigned* ticket,
                   unsigned long long* flag, unsigned long long* val, float* x, float* vx, float* vy, float* vz,
                   uint32_t* id, uint32_t* tc, unsigned long long cap, unsigned long long* out_count, cudaStream_t s) {
    k_gather<<<grid, CMP_T, 0, s>>>(P, species, epoch, ticket, flag, val, x, vx, vy, vz, id, tc, cap, out_count);
}

void launch_load_check(int species, const Params& P, unsigned long long n, cudaStream_t s) {
    const int grid = (int)std::min<unsigned long long>(ceil_div(n, LOAD_T), LOAD_BLOCKS);
    if (species == SP_E) k_load_check<SP_E><<<grid, LOAD_T, 0, s>>>(P, n);
    else if (species == SP_OM) k_load_check<SP_OM><<<grid, LOAD_T, 0, s>>>(P, n);
    else k_load_check<SP_OP><<<grid, LOAD_T, 0, s>>>(P, n);
}

void launch_philox(const uint32_t* ctr, const uint32_t* key, uint32_t* out, unsigned long long n, cudaStream_t s) {
    const int grid = (int)(n / 256 + 1 < 4096 ? n / 256 + 1 : 4096);
    k_philox<<<grid, 256, 0, s>>>(ctr, key, out, n);
}

void launch_ln(const float* x, float* out, unsigned long long n, cudaStream_t s) {
    const int grid = (int)(n / 256 + 1 < 4096 ? n / 256 + 1 : 4096);
    k_ln<<<grid, 256, 0, s>>>(x, out, n);
}

}  // namespace o2
