// Particle kernel of one species for one time step (Sec. 2 of the paper):
// field gather, leapfrog push in x (v_x accelerated, v_y and v_z carried),
// absorbing electrodes, null-collision Monte Carlo against the O2 / O2(a)
// background, births, and the CIC charge deposit of the pushed particles.
//
// Layout and flow (GB300-first):
//   * SoA FP32 arrays x, vx, vy, vz + u32 id, updated IN PLACE: a particle
//     keeps its slot, removed particles are marked (x = NaN) and dropped by a
//     periodic stable compaction, births are appended after the last slot.
//     The common path reads x, vx, tc (12 B) and writes x, vx (8 B); id,
//     vy, vz are read for collision candidates only.
//   * a persistent grid; each warp owns one contiguous, 128-aligned slot range
//     (O2+: takes rounds of the whole array in turn) and walks it in rounds of
//     128, a lane taking four neighbouring slots with one 16-byte load and
//     store per array, the next round's loads in flight while it works on this
//     one.  No block-wide barrier between the set-up and the end of the ranges.
//   * what bounds it: on large arrays HBM (20 B per particle; 4.65e7 O2+ on
//     2048 cells 198 -> 180 us, 5.2 TB/s against 6.8 of a plain copy), on small ones the
//     instructions (80 per 32 particles, before 122: integer deposit counters
//     of 32 bits instead of a 64-bit compare-and-swap loop, no conversion on
//     the FP64 unit, one branch per round for all that is rare) and the tail
//     of collisions;
//   * the gather field and the deposit live in shared memory; the deposit is
//     a count and a sum of CIC weights per cell, turned into node charges when
//     the block flushes (one 64-bit add per node);
//   * free flights (Sec. 2: "the durations of the free flights ... from
//     elementary kinetic considerations"): each particle carries the step of
//     its next null-collision candidate (tc, read with x and v_x), so the
//     common path draws no random number; candidates are queued per warp in
//     shared memory and handled 32 at a time (all lanes busy): one Philox
//     block (the id-free first round hoisted) draws the next free flight and
//     the rest of the collision;
//   * electrons: a candidate is filtered at once (energy against the total
//     rate, the total-rate column in shared memory), only the real
//     collisions are recorded (32 B each: slot, id, v, the Philox block's
//     rest), and the block runs their kinematics once all its warps' ranges
//     are pushed, pooled over the warps (no second kernel on electron steps);
//   * ions: candidates are recorded (slot, id, v and the Philox block's rest) and
//     a second kernel filters them (target sampled from the gas Maxwellian,
//     energy against the total rate) and runs the kinematics of the real ones
//     (inside the particle kernel the target draws cost registers and time);
//   * births are ranked with warp ballots and staged at the warp's range;
//     the end-of-step kernel places them in parent order.
#include "common.cuh"

// Launch shape of the particle kernels: minimum resident blocks per SM, which
// caps the registers (80 at 3: room for the round in flight).  Per launch, 4, 3
// and 2 blocks: electrons 24.7, 22.4, 22.8 us (1.5e6 on 512 cells) and 207, 206,
// 228 us (2.6e7 on 2048 cells), O2+ 183, 180, 195 us (4.65e7 on 2048 cells).
#ifndef O2PIC_PUSH_MIN_BLOCKS
#define O2PIC_PUSH_MIN_BLOCKS 3
#endif
// The electron kernel also runs the kinematics of its real collisions.
#ifndef O2PIC_PUSH_E_MIN_BLOCKS
#define O2PIC_PUSH_E_MIN_BLOCKS 3
#endif
// Minimum resident blocks per SM of the ion collision kernel (caps its
// registers; the particle kernel's grid then runs in one wave).
#ifndef O2PIC_ION_MIN_BLOCKS
#define O2PIC_ION_MIN_BLOCKS 3
#endif

namespace o2 {

namespace {

template <int S> struct SpeciesTraits;
template <> struct SpeciesTraits<SP_E> { static constexpr uint32_t tag = TAG_E; };
template <> struct SpeciesTraits<SP_OM> { static constexpr uint32_t tag = TAG_OM; };
template <> struct SpeciesTraits<SP_OP> { static constexpr uint32_t tag = TAG_OP; };

constexpr int WARPS = BLOCK / 32;           // 8
constexpr int ROUND = 128;                  // slots per warp round (4 per lane)

struct PushShared {
    unsigned long long jsum;     // block's sum of trunc(256 v_x^{n+1/2})
    unsigned absorbed[2];
    unsigned removed;
    unsigned psteps;
    unsigned nonfinite;
    unsigned wtries;
};

// A block's real collisions and their births (see collide_tail).
struct CollideShared {
    unsigned events[MAXPROC];                  // per process
    unsigned start[WARPS + 1];                 // place of each warp's first record in the pool
    unsigned nb1[WARPS], nb2[WARPS];           // births of each warp's own passes, by bkind
    unsigned m1[WARPS], m2[WARPS];             // births of the pool, by thread
};

// The last records of each warp, record i of a warp at place i mod 32 (what is
// pooled is read from here, without a trip to the list in memory).
struct PushPool {
    uint4 a[WARPS][32], b[WARPS][32];
};

// First record of particle-kernel warp gw (of W) in its species' candidate list:
// the warp's first slot, or, where warps take rounds in turn (O2+), the number
// of slots in the rounds of the warps before it; never fewer records than the
// slots it handles lie between two warps' starts.
template <int S>
__device__ __forceinline__ unsigned list_start(unsigned gw, unsigned W, unsigned nslots) {
    if (S == SP_OP) {
        const unsigned rounds = (nslots + ROUND - 1) / ROUND, q = rounds / W, rem = rounds % W;
        return ROUND * (gw * q + (gw < rem ? gw : rem));
    }
    const unsigned R = warp_range_len(nslots, W);
    return (gw * (unsigned long long)R < nslots) ? gw * R : nslots;
}

__host__ __device__ inline size_t align16(size_t v) { return (v + 15) & ~(size_t)15; }

// Process of a real collision (a candidate its filter kept): the total rate is
// above u1 nu_max, and the first process whose cumulative rate exceeds it is
// chosen (the last one if rounding leaves none).  -1: null (rounding).  The
// cumulative rates are read four processes at a time (loads in flight
// together); each value is grid_interp(cum, np, kk, i, w).
__device__ __forceinline__ int select_process(const float* __restrict__ cum, int np, float target, int i, float w) {
    const bool last = i >= NGRID - 1;
    const float* row = cum + (size_t)(last ? NGRID - 1 : i) * np;
    auto interp = [&](float a, float b) { return last ? a : fmaf(w, b - a, a); };
    const float ta = row[np - 1], tb = last ? 0.0f : row[2 * np - 1];
    float a[4], b[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        a[j] = (j < np - 1) ? row[j] : 0.0f;
        b[j] = (j < np - 1 && !last) ? row[np + j] : 0.0f;
    }
    if (!(target < interp(ta, tb))) return -1;
    for (int k0 = 0; k0 < np - 1; k0 += 4) {
        if (k0 > 0) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int kk = k0 + j;
                a[j] = (kk < np - 1) ? row[kk] : 0.0f;
                b[j] = (kk < np - 1 && !last) ? row[np + kk] : 0.0f;
            }
        }
        int f = -1;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int kk = k0 + j;
            if (f < 0 && kk < np - 1 && target < interp(a[j], b[j])) f = kk;
        }
        if (f >= 0) return f;
    }
    return np - 1;
}

// One real collision of an electron: process selection and kinematics, with the
// random words and the arithmetic in the order of the oracle.  w0: block 0 of
// its stream (word 0, the candidate draw, is spent).  Returns the event index,
// or -1 for a null collision (the selected process's threshold above E; the
// rate test itself repeats the filter's).  bkind: 0 none, 1 ionization (two
// births), 2 attachment (one).
//
// The directions (Marsaglia 1972: points of the unit disk) and normals
// (Marsaglia-Bray polar method: the same without the centre) a lane needs are
// drawn by one rejection loop, task after task: 0, 1 directions, 2, 3 pairs of
// normals; elastic and excited electrons need task 0, an ionization 0-3 (after
// the share of the energy), an attachment 2-3.  A warp passes the loop as often
// as its longest lane needs in all, not in each task, and the code holds one
// Philox block instead of nine.
__device__ __forceinline__ int collide_electron(const Params& P, const float* __restrict__ cum, int np,
                                                unsigned long long step, uint32_t id, uint4 w0, float x, float& vx,
                                                float& vy, float& vz, bool& alive, int& bkind, float4& b1, float4& b2,
                                                unsigned& warn_tries) {
    alive = true;
    bkind = 0;
    const float E = P.kappa[SP_E] * dot3(vx, vy, vz, vx, vy, vz);
    int i; float w; bool above;
    grid_locate(E, i, w, above);
    const int k = select_process(cum, np, uniform(w0.y) * P.numax[SP_E], i, w);
    if (k < 0) return -1;
    const float thr = P.thr[SP_E][k];
    if (E < thr) return -1;
    const int kind = P.kind[SP_E][k];
    const bool ionize = kind == K_IONIZE, attach = kind == K_ATTACH;
    // words come from a window of one block (w0) or two (the next ones, drawn
    // together so that their rounds overlap); pos: the next word in it
    uint4 lo = w0, hi = w0;
    uint32_t block = 0;
    int pos = 2, words = 4;
    float u = 0.0f;
    if (ionize) { u = uniform(lo.z); pos = 3; }
    float a0 = 0.0f, c0 = 0.0f, s0 = 0.0f, a1 = 0.0f, c1 = 0.0f, s1 = 0.0f, a2 = 0.0f, c2 = 0.0f, s2 = 0.5f,
          a3 = 0.0f, s3 = 0.5f;
    const int last_task = (ionize || attach) ? 4 : 1;
    int task = attach ? 2 : 0, tries = 0;
    auto word = [&](int i) {
        const uint4 q = i < 4 ? lo : hi;
        const uint32_t e = (i & 1) ? q.y : q.x, f = (i & 1) ? q.w : q.z;
        return (i & 2) ? f : e;
    };
    while (task < last_task) {
        // the next two words (the second may be the first of the next window)
        uint32_t wa = word(pos), wb;
        if (pos + 1 < words) {
            wb = word(pos + 1);
            pos += 2;
        } else {
            const uint4 ctr = make_uint4((uint32_t)step, SpeciesTraits<SP_E>::tag, block + 1, (uint32_t)(step >> 32));
            lo = philox4x32_10(ctr, make_uint2(id, P.seed));
            hi = philox4x32_10(make_uint4(ctr.x, ctr.y, block + 2, ctr.w), make_uint2(id, P.seed));
            block += 2;
            if (pos < words) { wb = lo.x; pos = 1; }
            else { wa = lo.x; wb = lo.y; pos = 2; }
            words = 8;
        }
        float a = 2.0f * uniform(wa) - 1.0f;
        float b = 2.0f * uniform(wb) - 1.0f;
        float s = fmaf(a, a, b * b);
        if (!(s < 1.0f && (task < 2 || s > 0.0f))) {
            if (++tries < MAX_TRIES) continue;
            ++warn_tries;              // gives up: direction (0, 0, 1), normals 0
            a = 0.0f; b = 0.0f; s = task < 2 ? 0.0f : 0.5f;
        }
        if (task == 0) { a0 = a; c0 = b; s0 = s; }
        else if (task == 1) { a1 = a; c1 = b; s1 = s; }
        else if (task == 2) { a2 = a; c2 = b; s2 = s; }
        else { a3 = a; s3 = s; }
        ++task;
        tries = 0;
    }
    if (ionize || attach) {
        const float sig = P.sig_birth[ionize ? SP_OP : SP_OM];
        const float f2 = sqrtf((-2.0f * ln_series(s2)) / s2), f3 = sqrtf((-2.0f * ln_series(s3)) / s3);
        b2 = make_float4(x, sig * (a2 * f2), sig * (c2 * f2), sig * (a3 * f3));
        if (attach) {
            b1 = b2;
            bkind = 2;
            alive = false;
            return k;
        }
    }
    const float h0 = 2.0f * sqrtf(1.0f - s0);
    const float nx = a0 * h0, ny = c0 * h0, nz = 1.0f - 2.0f * s0;
    float vn;
    if (kind == K_ELASTIC) {
        const float vm = sqrtf(dot3(vx, vy, vz, vx, vy, vz));
        const float cosx = (vm > 0.0f) ? dot3(nx, ny, nz, vx, vy, vz) / vm : 0.0f;
        const float fac = 1.0f - P.delta_el * (1.0f - cosx);
        vn = vm * sqrtf(fac);
    } else {
        const float Er = E - thr;
        float Ep = Er;
        if (ionize) {
            const float Es = u * Er;
            Ep = Er - Es;
            const float h1 = 2.0f * sqrtf(1.0f - s1);
            const float vs = sqrtf(Es / P.kappa[SP_E]);
            b1 = make_float4(x, vs * (a1 * h1), vs * (c1 * h1), vs * (1.0f - 2.0f * s1));
            bkind = 1;
        }
        vn = sqrtf(Ep / P.kappa[SP_E]);
    }
    vx = vn * nx; vy = vn * ny; vz = vn * nz;
    return k;
}

// An ion's random words after u1: pairs of words, (2, 3) of block 0 (w0), then
// (0, 1), (2, 3) of block 1, and so on; try t takes pair t.  All that an ion
// draws is drawn in pairs (normals, directions), so the lanes of a warp need a
// new block at the same tries.
struct IonPairs {
    uint4 buf;
    uint32_t id, t;
    template <int S>
    __device__ __forceinline__ void next(const Params& P, unsigned long long step, float& a, float& b) {
        uint32_t wa = buf.z, wb = buf.w;
        if (t & 1u) {
            buf = philox4x32_10(make_uint4((uint32_t)step, SpeciesTraits<S>::tag, (t + 1u) >> 1, (uint32_t)(step >> 32)),
                                make_uint2(id, P.seed));
            wa = buf.x;
            wb = buf.y;
        }
        ++t;
        a = 2.0f * uniform(wa) - 1.0f;
        b = 2.0f * uniform(wb) - 1.0f;
    }
};

// The gas molecule an ion meets, a Maxwellian: both pairs of normals
// (Marsaglia-Bray polar method) drawn by one rejection loop, transformed once
// at its end.
template <int S>
__device__ __forceinline__ void gas_target(const Params& P, unsigned long long step, IonPairs& r, float& vx, float& vy,
                                           float& vz, unsigned& warn) {
    float a0 = 0.0f, b0 = 0.0f, s0 = 0.5f, a1 = 0.0f, s1 = 0.5f;
    int task = 0, tries = 0;
    while (task < 2) {
        float a, b;
        r.next<S>(P, step, a, b);
        float s = fmaf(a, a, b * b);
        if (!(s > 0.0f && s < 1.0f)) {
            if (++tries < MAX_TRIES) continue;
            ++warn;                    // gives up: normals 0
            a = 0.0f; b = 0.0f; s = 0.5f;
        }
        if (task == 0) { a0 = a; b0 = b; s0 = s; }
        else { a1 = a; s1 = s; }
        ++task;
        tries = 0;
    }
    const float f0 = sqrtf((-2.0f * ln_series(s0)) / s0), f1 = sqrtf((-2.0f * ln_series(s1)) / s1);
    vx = P.sig_gas * (a0 * f0); vy = P.sig_gas * (b0 * f0); vz = P.sig_gas * (a1 * f1);
}

// One real collision of an ion, exactly in the order of the oracle (its filter
// already counted the warnings of the target sample and the energy).  Returns
// as collide_electron; bkind 2: detachment (the electron in b1).
template <int S>
__device__ __forceinline__ int collide_ion(const Params& P, const float* __restrict__ cum, int np,
                                           unsigned long long step, uint32_t id, uint4 w0, float x, float& vx,
                                           float& vy, float& vz, bool& alive, int& bkind, float4& b1,
                                           unsigned& warn_tries) {
    alive = true;
    bkind = 0;
    IonPairs r = {w0, id, 0u};
    float vtx, vty, vtz;
    unsigned counted_by_filter = 0;
    gas_target<S>(P, step, r, vtx, vty, vtz, counted_by_filter);
    const float gx = vx - vtx, gy = vy - vty, gz = vz - vtz;
    const float E = P.kappa[S] * dot3(gx, gy, gz, gx, gy, gz);
    int i; float w; bool above;
    grid_locate(E, i, w, above);
    const int k = select_process(cum, np, uniform(w0.y) * P.numax[S], i, w);
    if (k < 0) return -1;
    const float thr = P.thr[S][k];
    if (E < thr) return -1;
    const int kind = P.kind[S][k];
    if (kind == K_CX) {
        vx = vtx; vy = vty; vz = vtz;
        return k;
    }
    float nx = 0.0f, ny = 0.0f, nz = 1.0f;     // isotropic()
    int t = 0;
    for (; t < MAX_TRIES; ++t) {
        float a, b;
        r.next<S>(P, step, a, b);
        const float s = fmaf(a, a, b * b);
        if (s < 1.0f) {
            const float h = 2.0f * sqrtf(1.0f - s);
            nx = a * h; ny = b * h; nz = 1.0f - 2.0f * s;
            break;
        }
    }
    if (t == MAX_TRIES) ++warn_tries;
    if (kind == K_ELASTIC) {
        const float gm = sqrtf(dot3(gx, gy, gz, gx, gy, gz));
        const float cmx = fmaf(P.a_m[S], vx, P.a_M[S] * vtx);
        const float cmy = fmaf(P.a_m[S], vy, P.a_M[S] * vty);
        const float cmz = fmaf(P.a_m[S], vz, P.a_M[S] * vtz);
        const float f = P.a_M[S] * gm;
        vx = fmaf(f, nx, cmx); vy = fmaf(f, ny, cmy); vz = fmaf(f, nz, cmz);
    } else if (S == SP_OM && kind == K_DETACH) {
        const float vn = sqrtf((E - thr) / P.kappa[SP_E]);
        b1 = make_float4(x, vn * nx, vn * ny, vn * nz);
        bkind = 2;
        alive = false;
    }
    return k;
}

__device__ __forceinline__ void deposit_add(unsigned* hist, float x, float inv_dx, int Nc) {
    int j; float frac;
    cell_of(x, inv_dx, Nc, j, frac);
    const uint32_t r = cic_r(frac);
    atomicAdd(&hist[j], 65536u - r);
    atomicAdd(&hist[j + 1], r);
}

__device__ __forceinline__ void deposit_sub_global(unsigned long long* Q, float x, float inv_dx, int Nc) {
    int j; float frac;
    cell_of(x, inv_dx, Nc, j, frac);
    const uint32_t r = cic_r(frac);
    atomicAdd(&Q[j], 0ull - (unsigned long long)(65536u - r));
    atomicAdd(&Q[j + 1], 0ull - (unsigned long long)r);
}

// A birth's CIC charge, into the births' accumulator Qb of its species.
__device__ __forceinline__ void deposit_add_global(unsigned long long* Q, float x, float inv_dx, int Nc) {
    int j; float frac;
    cell_of(x, inv_dx, Nc, j, frac);
    const uint32_t r = cic_r(frac);
    atomicAdd(&Q[j], (unsigned long long)(65536u - r));
    if (r) atomicAdd(&Q[j + 1], (unsigned long long)r);
}

__device__ __forceinline__ void flush_hist(unsigned* hist, unsigned long long* Q, int Ng) {
    for (int j = threadIdx.x; j < Ng; j += BLOCK) {
        const unsigned v = hist[j];
        if (v) {
            atomicAdd(&Q[j], (unsigned long long)v);
            hist[j] = 0u;
        }
    }
}

// Filter of an electron candidate: is it a real collision?  The same
// arithmetic as the start of collide(): energy of the particle, the total
// rate on the table grid (column `tot` = the last cumulative column) and the
// comparison with u1 nu_max.
__device__ __forceinline__ bool electron_is_real(const Params& P, const float* tot, uint32_t w1, float vx, float vy,
                                                 float vz, unsigned& wemax, unsigned& wnumax) {
    const float u1 = uniform(w1);
    const float E = P.kappa[SP_E] * dot3(vx, vy, vz, vx, vy, vz);
    int i; float w; bool above;
    grid_locate(E, i, w, above);
    if (above) ++wemax;
    const float total = grid_interp(tot, 1, 0, i, w);
    if (total > P.numax[SP_E]) ++wnumax;   // above a capped majorant
    return (u1 * P.numax[SP_E]) < total;
}

// Total-rate column (the last cumulative column) of species S into shared memory.
__device__ __forceinline__ void stage_total(const Params& P, int S, float* tot) {
    const float* __restrict__ g = P.tot[S];
    constexpr int K = (NGRID + BLOCK - 1) / BLOCK;
    float v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int i = (int)threadIdx.x + k * BLOCK;
        v[k] = i < NGRID ? g[i] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int i = (int)threadIdx.x + k * BLOCK;
        if (i < NGRID) tot[i] = v[k];
    }
}

// (long long)v for |v| >= 2^31 (and infinities, NaN) in integer arithmetic: a
// 64-bit conversion runs on the FP64 unit, also where its predicate is false.
__device__ __forceinline__ long long trunc_s64_large(float v) {
    const uint32_t b = __float_as_uint(v);
    const int e = (int)((b >> 23) & 0xFFu) - 150;                  // v = +-m 2^e, e >= 8
    if (e > 39) return (v > 0.0f) ? 0x7FFFFFFFFFFFFFFFll : (long long)0x8000000000000000ull;
    const long long m = (long long)((b & 0x007FFFFFu) | 0x00800000u) << e;
    return (b >> 31) ? -m : m;
}

// The block's deposit: per cell the count of its particles and the sum of
// their CIC weights r (32-bit counters: shared memory adds 32-bit words in one
// instruction, 64-bit words in a compare-and-swap loop).  A weight sum that
// wraps hands its 2^32 to the node charges at once: the one operation that
// wrapped sees it in the old value, so no block is too large for the counters.
__device__ __forceinline__ void weight_wrapped(unsigned long long* Q, int c, int sign) {
    const unsigned long long w = (unsigned long long)((long long)sign << 32);
    atomicAdd(&Q[c], 0ull - w);
    atomicAdd(&Q[c + 1], w);
}

__device__ __forceinline__ void cell_sub(unsigned* cnt, unsigned* rsum, int c, uint32_t r, unsigned long long* Q) {
    atomicSub(&cnt[c], 1u);
    const unsigned old = atomicSub(&rsum[c], r);
    if (old < r) weight_wrapped(Q, c, -1);
}

// Set bits [a, b) of the 32-bit words in m (b - a <= 32).
__device__ __forceinline__ unsigned bits_between(const unsigned* m, unsigned a, unsigned b) {
    if (a >= b) return 0u;
    const unsigned wa = a >> 5, wb = (b - 1u) >> 5;
    const unsigned lo = 0xffffffffu << (a & 31u), hi = 0xffffffffu >> (31u - ((b - 1u) & 31u));
    return wa == wb ? __popc(m[wa] & lo & hi) : __popc(m[wa] & lo) + __popc(m[wb] & hi);
}

// The kinematics of a block's real collisions: nrec records of this warp
// {slot, id, vx, vy}{vz, w1, w2, w3} from CAND[2 rec0] on, in slot order, the
// last ones also in `pool`.  Each warp takes its own records 32 at a time, and
// what is left (fewer than 32 per warp) is pooled over the block, in warp
// order, one record per thread, so that short lists still fill their warps
// (1.5e6 electrons: 14 records per warp).  A removed particle's charge comes
// off the block's deposit when `cnt` is given (the particle kernel), else off
// the step's deposit in memory.  The filter counted the warnings of the part
// it shares with the kinematics.  Births are staged at their warp's slot range
// [gw R, ...) in slot order (those of its own passes, then those of its pooled
// records), with their number per warp, for the end-of-step kernel, which
// places them; their charge goes to Qb now.
template <int S>
__device__ __forceinline__ void collide_tail(const Params& P, CollideShared& sh, PushPool& pool, unsigned blk,
                                             unsigned long long step, unsigned cb, unsigned R, unsigned rec0,
                                             unsigned nrec, unsigned* cnt, unsigned* rsum, unsigned long long* Qcopy,
                                             unsigned& nrm, unsigned& wtries) {
    const int np = P.nproc[S];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    float* __restrict__ X = P.sp[S].x[cb];
    float* __restrict__ VX = P.sp[S].vx[cb];
    float* __restrict__ VY = P.sp[S].vy[cb];
    float* __restrict__ VZ = P.sp[S].vz[cb];
    const uint4* CAND = P.cand[S];             // written by this warp just now
    const float inv_dx = P.inv_dx;
    const int Nc = P.Nc;
    const unsigned own = nrec & ~31u;
    unsigned nb1 = 0, nb2 = 0;   // warp-uniform: births of its own passes
    if (lane == 0) sh.start[warp + 1] = nrec - own;
    __syncthreads();
    if (warp == 0) {
        unsigned v = lane < WARPS ? sh.start[lane + 1] : 0u;
#pragma unroll
        for (int o = 1; o < WARPS; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        if (lane < WARPS) sh.start[lane + 1] = v;
        if (lane == 0) sh.start[0] = 0u;
    }
    __syncthreads();
    const unsigned pooled = sh.start[WARPS];
    const bool births = S != SP_OP && P.births_possible[S] != 0;
    unsigned u = (unsigned)warp;              // the warp whose record this is
    for (unsigned c = 0;; c += 32u) {
        const bool last = c >= own;           // the pool
        bool has = true;
        if (last) {
            has = (unsigned)tid < pooled;
            for (u = 0; u < WARPS - 1 && (unsigned)tid >= sh.start[u + 1]; ++u) {}
        }
        int bkind = 0;
        float4 b1 = make_float4(0.f, 0.f, 0.f, 0.f), b2 = b1;
        if (has) {
            const unsigned i = (unsigned)tid - sh.start[u];   // (pool)
            const uint4 a = last ? pool.a[u][i] : CAND[2 * (size_t)(rec0 + c + lane)];
            const uint4 b = last ? pool.b[u][i] : CAND[2 * (size_t)(rec0 + c + lane) + 1];
            const unsigned slot = a.x;
            const float x = S != SP_OP ? X[slot] : 0.0f;      // needed late: births, removals
            float vx = __uint_as_float(a.z), vy = __uint_as_float(a.w), vz = __uint_as_float(b.x);
            bool alive;
            const int k = S == SP_E ? collide_electron(P, P.cum[S], np, step, a.y, b, x, vx, vy, vz, alive, bkind, b1,
                                                       b2, wtries)
                                    : collide_ion<S>(P, P.cum[S], np, step, a.y, b, x, vx, vy, vz, alive, bkind, b1,
                                                     wtries);
            if (k >= 0) {
                atomicAdd(&sh.events[k], 1u);
                if (S == SP_OP || alive) {
                    VX[slot] = vx; VY[slot] = vy; VZ[slot] = vz;
                } else {
                    X[slot] = dead_marker();
                    if (S == SP_E) {
                        int j; float f;
                        cell_of(x, inv_dx, Nc, j, f);
                        cell_sub(cnt, rsum, j, cic_r(f), Qcopy);
                    } else {
                        deposit_sub_global(P.Qf[S], x, inv_dx, Nc);
                    }
                    ++nrm;
                }
            }
        }
        if (S == SP_OP) {
            if (last) break;
            continue;
        }
        const unsigned m1 = __ballot_sync(0xffffffffu, bkind == 1), m2 = __ballot_sync(0xffffffffu, bkind == 2);
        unsigned rank1 = nb1 + __popc(m1 & lt_mask), rank2 = nb2 + __popc(m2 & lt_mask), w = blk * WARPS + warp;
        if (last) {
            if (lane == 0) { sh.nb1[warp] = nb1; sh.nb2[warp] = nb2; sh.m1[warp] = m1; sh.m2[warp] = m2; }
            __syncthreads();
            if (bkind) {
                rank1 = sh.nb1[u] + bits_between(sh.m1, sh.start[u], (unsigned)tid);
                rank2 = sh.nb2[u] + bits_between(sh.m2, sh.start[u], (unsigned)tid);
                w = blk * WARPS + u;
            }
        }
        const unsigned s0 = w * R;
        if (bkind == 1) {
            P.stage[B_E_FROM_E][s0 + rank1] = b1;
            P.stage[B_OP_FROM_E][s0 + rank1] = b2;
            deposit_add_global(P.Qb[SP_E], b1.x, inv_dx, Nc);
            deposit_add_global(P.Qb[SP_OP], b2.x, inv_dx, Nc);
        } else if (bkind == 2) {
            P.stage[S == SP_E ? B_OM_FROM_E : B_E_FROM_OM][s0 + rank2] = b1;
            deposit_add_global(P.Qb[S == SP_E ? SP_OM : SP_E], b1.x, inv_dx, Nc);
        }
        if (last) break;
        nb1 += __popc(m1);
        nb2 += __popc(m2);
    }
    if (births && tid < WARPS) {
        const unsigned w = blk * WARPS + tid, a = sh.start[tid], b = sh.start[tid + 1];
        if (S == SP_E) P.wcount[B_E_FROM_E][w] = sh.nb1[tid] + bits_between(sh.m1, a, b);
        P.wcount[S == SP_E ? B_OM_FROM_E : B_E_FROM_OM][w] = sh.nb2[tid] + bits_between(sh.m2, a, b);
    }
}

// Candidate queue of one warp of the particle kernel (shared memory): the slots
// of its candidates in slot order.  Fewer than 32 stay from one round to the
// next and a round adds at most ROUND.
constexpr int QN = 32 + ROUND;
struct PushQueue {
    unsigned slot[WARPS][QN];
};

// Body of the particle kernel for block blk of nblk blocks (the launch's own
// block, or a block a batched launch maps to this discharge).
template <int S>
__device__ __forceinline__ void push_body(const Params& P, unsigned blk, unsigned nblk) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int np = P.nproc[S];
    PushShared& sh = *reinterpret_cast<PushShared*>(smem);
    PushPool& pool = *reinterpret_cast<PushPool*>(smem + align16(sizeof(PushShared)));   // electrons only
    CollideShared& ch = *reinterpret_cast<CollideShared*>(&pool + 1);                    // electrons only
    unsigned char* rest = smem + align16(sizeof(PushShared)) +
                          (S == SP_E ? sizeof(PushPool) + align16(sizeof(CollideShared)) : 0);
    float* Es = reinterpret_cast<float*>(rest);
    unsigned* cnt = reinterpret_cast<unsigned*>(Es + P.Ng);
    unsigned* rsum = cnt + P.Ng;
    PushQueue& Q = *reinterpret_cast<PushQueue*>(rsum + P.Ng);
    float* Tt = reinterpret_cast<float*>(&Q + 1);        // electrons: total-rate column
    constexpr bool electrons = S == SP_E;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    unsigned* qs = Q.slot[warp];
    const int Nc = P.Nc, Ng = P.Ng;

    // what no earlier kernel writes, before waiting for the one before
    for (int j = tid; j < Ng; j += BLOCK) { cnt[j] = 0u; rsum[j] = 0u; }
    if (electrons) stage_total(P, S, Tt);
    if (tid == 0) {
        sh.absorbed[0] = sh.absorbed[1] = 0u; sh.removed = 0u; sh.psteps = 0u; sh.nonfinite = 0u; sh.wtries = 0u;
        sh.jsum = 0ull;
    }
    if (electrons && tid < MAXPROC) ch.events[tid] = 0u;
    pdl_wait();

    DevCtrl* C = P.ctrl;
    const unsigned long long step = C->step;
    const uint32_t step_lo = (uint32_t)step;
    const unsigned cb = C->cur[S];
    const unsigned nslots = (unsigned)((C->slots[S] < P.sp[S].cap) ? C->slots[S] : P.sp[S].cap);
    float* __restrict__ X = P.sp[S].x[cb];
    float* __restrict__ VX = P.sp[S].vx[cb];
    float* __restrict__ VY = P.sp[S].vy[cb];
    float* __restrict__ VZ = P.sp[S].vz[cb];
    const uint32_t* __restrict__ ID = P.sp[S].id[cb];
    uint32_t* __restrict__ TC = P.sp[S].tc[cb];
    uint4* CAND = P.cand[S];
    const float qmdt = P.qmdt[S], dts = P.dt_s[S], inv_dx = P.inv_dx, Lf = P.Lf;
    const float inv_lnq = P.inv_lnq[S], kcap = P.kcap[S];
    const unsigned sub = P.sub[S];
    const float jmax = cell_limit(Nc);
    unsigned long long* __restrict__ Qcopy = P.Qf[S] + (size_t)(blk & (QCOPIES - 1)) * Ng;
    const PhiloxPre pre = philox_pre(step_lo, SpeciesTraits<S>::tag, (uint32_t)(step >> 32), P.seed);

    // this warp's contiguous slot range, and its first round of x, v_x, tc
    // requested before the block's set-up (their latency overlaps it).  A lane
    // takes four neighbouring slots of a round, one 16-byte word per array
    // (ranges start on multiples of 128 slots); the last round of the slots in
    // use is read slot by slot.
    const unsigned W = nblk * WARPS;
    const unsigned gw = blk * WARPS + warp;
    const unsigned R = warp_range_len(nslots, W);
    const unsigned r0 = (gw * (unsigned long long)R < nslots) ? gw * R : nslots;
    const unsigned r1 = (r0 + R < nslots) ? r0 + R : nslots;
    // O2+ have no births, so nothing asks for their order: their warps take the
    // rounds of the whole array in turn, and the grid sweeps it front to back
    // (5.1 against 4.7 TB/s for 4.65e7 O2+ on 2048 cells).  Births are placed in
    // parent order, so the other species' warps keep contiguous ranges.
    constexpr bool in_turn = S == SP_OP;
    const unsigned stride = in_turn ? W * ROUND : ROUND;
    const unsigned ga = in_turn ? gw * ROUND : r0, gz = in_turn ? nslots : r1;
    const unsigned rec0 = in_turn ? list_start<S>(gw, W, nslots) : r0;
    float xs[4], vxs[4];
    uint32_t tcs[4];
    auto load_round = [&](unsigned g0, float (&xs)[4], float (&vxs)[4], uint32_t (&tcs)[4]) {
        const unsigned i0 = g0 + 4u * lane;
        if (g0 + ROUND <= gz) {
            const float4 a = *reinterpret_cast<const float4*>(X + i0);
            const float4 b = *reinterpret_cast<const float4*>(VX + i0);
            const uint4 c = *reinterpret_cast<const uint4*>(TC + i0);
            xs[0] = a.x; xs[1] = a.y; xs[2] = a.z; xs[3] = a.w;
            vxs[0] = b.x; vxs[1] = b.y; vxs[2] = b.z; vxs[3] = b.w;
            tcs[0] = c.x; tcs[1] = c.y; tcs[2] = c.z; tcs[3] = c.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool inr = i0 + k < gz;
                xs[k] = inr ? X[i0 + k] : dead_marker();
                vxs[k] = inr ? VX[i0 + k] : 0.0f;
                tcs[k] = inr ? TC[i0 + k] : 0u;
            }
        }
    };
    if (ga < gz) load_round(ga, xs, vxs, tcs);

    for (int j0 = tid; j0 < Ng; j0 += 4 * BLOCK) {       // four loads in flight
        float e[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) e[k] = j0 + k * BLOCK < Ng ? P.Ef[j0 + k * BLOCK] : 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (j0 + k * BLOCK < Ng) Es[j0 + k * BLOCK] = e[k];
    }
    __syncthreads();

    unsigned nabs0 = 0, nabs1 = 0, nnf = 0, wemax = 0, wtries = 0, wnumax = 0;
    long long jacc = 0;   // conduction current: sum of trunc(256 v_x^{n+1/2}) (exact)
    unsigned nrec = 0;    // warp-uniform: records of this warp so far
    unsigned qn = 0;      // warp-uniform: queued candidates

    // m (<= 32) queued candidates from entry h on, one per lane: the candidate's
    // stream at this step (block 0) draws its next free flight (word 0) and
    // the electrons' real/null test (word 1 against the total rate at the
    // particle's energy); records go to the warp's list in slot order, two uint4
    // each: {slot, id, vx, vy}{vz, w1, w2, w3}, electrons per real collision,
    // ions per candidate.
    auto flush = [&](unsigned h, unsigned m) {
        const bool has = (unsigned)lane < m;
        const unsigned slot = has ? qs[h + lane] : 0u;
        uint32_t id = 0u;
        float cvx = 0.0f, cvy = 0.0f, cvz = 0.0f;
        if (has) { id = ID[slot]; cvx = VX[slot]; cvy = VY[slot]; cvz = VZ[slot]; }   // (v_x: as this warp stored it)
        bool rec = false;
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (has) {
            w = philox_id(pre, id);
            TC[slot] = step_lo + sub * (1u + flight_gap(w.x, inv_lnq, kcap));
            rec = !electrons || electron_is_real(P, Tt, w.y, cvx, cvy, cvz, wemax, wnumax);
        }
        const unsigned cm = __ballot_sync(0xffffffffu, rec);
        if (rec) {
            const unsigned i = nrec + __popc(cm & lt_mask);
            const size_t q = rec0 + i;
            const uint4 a = make_uint4(slot, id, __float_as_uint(cvx), __float_as_uint(cvy));
            const uint4 b = make_uint4(__float_as_uint(cvz), w.y, w.z, w.w);
            CAND[2 * q] = a;
            CAND[2 * q + 1] = b;
            if (electrons) { pool.a[warp][i & 31u] = a; pool.b[warp][i & 31u] = b; }
        }
        nrec += __popc(cm);
    };

    for (unsigned g0 = ga; g0 < gz; g0 += stride) {
        float xn[4], vxn[4];
        uint32_t tcn[4];
        if (g0 + stride < gz) load_round(g0 + stride, xn, vxn, tcn);   // in flight meanwhile
        const unsigned i0 = g0 + 4u * lane;
        // the four slots without branches (a dead slot's NaN falls through the
        // arithmetic and takes part in nothing); what is rare is flagged and
        // handled once per round: bit k of `out`: the particle left the gap,
        // `wrap`: its weight sum wrapped, `cand`: its free flight ends at this
        // step; vmax: a current term may not fit 32 bits
        unsigned cand = 0u, out = 0u, wrap = 0u;
        float vmax = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float x = xs[k], vx = vxs[k];
            const bool live = !is_dead(x);
            int j; float frac;
            cell_of_inside(x, inv_dx, jmax, j, frac);
            const float Ep = fmaf(frac, Es[j + 1] - Es[j], Es[j]);
            vx = fmaf(qmdt, Ep, vx);
            x = fmaf(vx, dts, x);
            // exact scaling by 2^8, then truncation
            const float jv = vx * 256.0f;
            jacc += (long long)__float2int_rz(jv);       // 0 for a dead slot's NaN
            vmax = fmaxf(vmax, fabsf(jv));               // (leaves a NaN out)
            if (x >= 0.0f && x < Lf) {
                // (a finite x here has a finite v_x.)  CIC deposit as (count,
                // sum of r) per cell: node c gets 2^16 count_c - rsum_c, node
                // c+1 gets rsum_c
                int j2; float f2;
                cell_of_inside(x, inv_dx, jmax, j2, f2);
                const uint32_t r = cic_r_inside(f2);
                atomicAdd(&cnt[j2], 1u);
                const unsigned old = atomicAdd(&rsum[j2], r);
                if (old + r < old) wrap |= 1u << k;
                if (tcs[k] == step_lo) cand |= 1u << k;
            } else if (live) {
                out |= 1u << k;
            }
            xs[k] = x;
            vxs[k] = vx;
        }
        if ((out | wrap) || !(vmax < 2147483648.0f)) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                // (a NaN here is a particle's, not a dead slot's, if it is in `out`)
                const float jv = vxs[k] * 256.0f;
                if (fabsf(jv) >= 2147483648.0f || (((out >> k) & 1u) && is_dead(jv)))
                    jacc += trunc_s64_large(jv) - (long long)__float2int_rz(jv);
                if ((wrap >> k) & 1u) {
                    int j2; float f2;
                    cell_of_inside(xs[k], inv_dx, jmax, j2, f2);
                    weight_wrapped(Qcopy, j2, 1);
                }
                if ((out >> k) & 1u) {
                    if (xs[k] < 0.0f) ++nabs0;
                    else if (xs[k] >= Lf) ++nabs1;
                    else ++nnf;
                    xs[k] = dead_marker();
                }
            }
        }
        if (g0 + ROUND <= gz) {
            *reinterpret_cast<float4*>(X + i0) = make_float4(xs[0], xs[1], xs[2], xs[3]);
            *reinterpret_cast<float4*>(VX + i0) = make_float4(vxs[0], vxs[1], vxs[2], vxs[3]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (i0 + k < gz) { X[i0 + k] = xs[k]; VX[i0 + k] = vxs[k]; }
        }
        const unsigned some = np > 0 ? __ballot_sync(0xffffffffu, cand != 0u) : 0u;
        if (some) {
            // queue them in slot order (lane by lane, four slots each); most
            // rounds have at most one in a lane
            if (!__any_sync(0xffffffffu, (cand & (cand - 1u)) != 0u)) {
                if (cand) qs[qn + __popc(some & lt_mask)] = i0 + (unsigned)__ffs(cand) - 1u;
                qn += __popc(some);
            } else {
                unsigned below = 0u, all = 0u;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const unsigned b = __ballot_sync(0xffffffffu, (cand >> k) & 1u);
                    below += __popc(b & lt_mask);
                    all += __popc(b);
                }
                unsigned q = qn + below;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if ((cand >> k) & 1u) qs[q++] = i0 + k;
                qn += all;
            }
            if (qn >= 32u) {
                __syncwarp();
                unsigned h = 0u;
                do { flush(h, 32u); h += 32u; } while (qn - h >= 32u);
                const unsigned rest = qn - h;      // < 32: lane q moves entry h + q
                const unsigned s0 = ((unsigned)lane < rest) ? qs[h + lane] : 0u;
                __syncwarp();
                if ((unsigned)lane < rest) qs[lane] = s0;
                qn = rest;
                __syncwarp();
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) { xs[k] = xn[k]; vxs[k] = vxn[k]; tcs[k] = tcn[k]; }
    }
    __syncwarp();
    if (qn > 0u) flush(0u, qn);
    unsigned nrm = 0;
    if (electrons) {
        collide_tail<S>(P, ch, pool, blk, step, cb, R, rec0, nrec, cnt, rsum, Qcopy, nrm, wtries);
    } else if (lane == 0) {
        P.ccount[S][gw] = nrec;
    }
    pdl_trigger();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) jacc += __shfl_down_sync(0xffffffffu, jacc, o);
    if (lane == 0 && jacc) atomicAdd(&sh.jsum, (unsigned long long)jacc);
    if (nabs0) atomicAdd(&sh.absorbed[0], nabs0);
    if (nabs1) atomicAdd(&sh.absorbed[1], nabs1);
    if (nabs0 + nabs1 + nnf + nrm) atomicAdd(&sh.removed, nabs0 + nabs1 + nnf + nrm);
    if (nnf) atomicAdd(&sh.nonfinite, nnf);
    if (wtries) atomicAdd(&sh.wtries, wtries);
    if (wemax) atomicAdd(&C->cnt.warn_emax, (unsigned long long)wemax);
    if (wnumax) atomicAdd(&C->cnt.warn_numax, (unsigned long long)wnumax);
    __syncthreads();
    if (electrons && tid < np && ch.events[tid]) atomicAdd(&C->cnt.events[S][tid], (unsigned long long)ch.events[tid]);
    // one 64-bit add per node: what its two cells give it
    unsigned kept = 0;
    for (int j = tid; j < Ng; j += BLOCK) {
        unsigned long long v = 0ull;
        if (j < Nc) { v = ((unsigned long long)cnt[j] << 16) - rsum[j]; kept += cnt[j]; }
        if (j > 0) v += rsum[j - 1];
        if (v) atomicAdd(&Qcopy[j], v);
    }
    // pushed: those still in the deposit and those removed since
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kept += __shfl_down_sync(0xffffffffu, kept, o);
    if (lane == 0 && kept) atomicAdd(&sh.psteps, kept);
    __syncthreads();
    if (tid == 0) sh.psteps += sh.removed;
    if (tid == 0) {
        if (sh.absorbed[0]) atomicAdd(&C->cnt.absorbed[S][0], (unsigned long long)sh.absorbed[0]);
        if (sh.absorbed[1]) atomicAdd(&C->cnt.absorbed[S][1], (unsigned long long)sh.absorbed[1]);
        if (sh.removed) atomicAdd(&C->removed[S], (unsigned long long)sh.removed);
        if (sh.psteps) {
            atomicAdd(&C->cnt.particle_steps, (unsigned long long)sh.psteps);
            atomicAdd(&C->cnt.psteps[S], (unsigned long long)sh.psteps);
        }
        if (sh.nonfinite) atomicOr(&C->error_flags, ERR_NONFINITE);
        if (sh.wtries) atomicAdd(&C->cnt.warn_tries, (unsigned long long)sh.wtries);
        if (sh.jsum) atomicAdd(&P.jring[(step & (JRING - 1)) * NSP + S], sh.jsum);
    }
}

// Free flights of the particles of species S drawn afresh at the current step
// n (after a load, or when new tables change nu_max): the first push at or
// after n plus sub K, K from word 0 of the particle's stream with tag
// TAG_FLIGHT + S at step n.
template <int S>
__global__ void k_flight_init(Params P) {
    DevCtrl* C = P.ctrl;
    const unsigned long long n = C->step;
    const unsigned cb = C->cur[S];
    const unsigned long long ns = (C->slots[S] < P.sp[S].cap) ? C->slots[S] : P.sp[S].cap;
    const float* __restrict__ X = P.sp[S].x[cb];
    const uint32_t* __restrict__ ID = P.sp[S].id[cb];
    uint32_t* __restrict__ TC = P.sp[S].tc[cb];
    const unsigned sub = P.sub[S];
    const uint32_t nf = (uint32_t)((n + sub - 1) / sub * sub);
    const PhiloxPre pre = philox_pre((uint32_t)n, TAG_FLIGHT + (uint32_t)S, (uint32_t)(n >> 32), P.seed);
    const float inv_lnq = P.inv_lnq[S], kcap = P.kcap[S];
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < ns;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        if (is_dead(X[i])) continue;
        TC[i] = nf + sub * flight_gap(philox_id(pre, ID[i]).x, inv_lnq, kcap);
    }
}

// Collisions of one ion species: block b of the particle kernel's grid takes the
// candidate lists of that kernel's block b, a warp each.  The filter: target
// sampled from the gas Maxwellian, relative energy and total rate against u1
// nu_max, the same arithmetic as the start of collide_ion(); it reads the
// records only (they carry the velocities and the Philox words).  The real
// collisions (some in ten) keep their records, compacted in place at the start
// of the list (a record is written only over one already read), then run
// through the kinematics, pooled over the block.  Bound by latency (draws,
// table reads) at a few records per lane, so one launch instead of a filter and
// a kinematics kernel: RF cycle of 128 cells 13.3 -> 12.1 ms, 512 cells 35.4 ->
// 34.7, 2048 cells 24.8 -> 24.2 (with the O2+ counted beside it).
template <int S>
__device__ __forceinline__ void ion_body(const Params& P, unsigned blk) {
    __shared__ float tot[NGRID];
    __shared__ PushPool pool;
    __shared__ CollideShared ch;
    __shared__ unsigned sh_wtries, sh_wemax, sh_removed;
    const int np = P.nproc[S];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    if (tid == 0) { sh_wtries = 0u; sh_wemax = 0u; sh_removed = 0u; }
    if (tid < MAXPROC) ch.events[tid] = 0u;
    stage_total(P, S, tot);
    __syncthreads();
    pdl_wait();
    DevCtrl* C = P.ctrl;
    const unsigned long long step = C->step;
    const unsigned cb = C->cur[S];
    const unsigned nslots = (unsigned)((C->slots[S] < P.sp[S].cap) ? C->slots[S] : P.sp[S].cap);
    uint4* CAND = P.cand[S];
    const unsigned W = P.push_warps[S], gw = blk * WARPS + (unsigned)warp;
    const float numax = P.numax[S], kap = P.kappa[S];
    unsigned wtries = 0, wemax = 0, wnumax = 0, nremoved = 0;
    const unsigned r0 = list_start<S>(gw, W, nslots);
    const unsigned n = P.ccount[S][gw];
    unsigned nreal = 0;   // warp-uniform
    for (unsigned c0 = 0; c0 < n; c0 += 64) {
        uint4 a[2], b[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const unsigned ci = c0 + 32u * k + lane;
            const bool in = ci < n;
            a[k] = in ? CAND[2 * (size_t)(r0 + ci)] : make_uint4(0u, 0u, 0u, 0u);
            b[k] = in ? CAND[2 * (size_t)(r0 + ci) + 1] : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (c0 + 32u * k >= n) break;   // warp-uniform
            bool real = false;
            if (c0 + 32u * k + lane < n) {
                IonPairs r = {b[k], a[k].y, 0u};
                float vtx, vty, vtz;
                gas_target<S>(P, step, r, vtx, vty, vtz, wtries);
                const float gx = __uint_as_float(a[k].z) - vtx, gy = __uint_as_float(a[k].w) - vty,
                            gz = __uint_as_float(b[k].x) - vtz;
                const float E = kap * dot3(gx, gy, gz, gx, gy, gz);
                int i; float w; bool above;
                grid_locate(E, i, w, above);
                if (above) ++wemax;
                const float total = grid_interp(tot, 1, 0, i, w);
                if (total > numax) ++wnumax;   // above a capped majorant
                real = (uniform(b[k].y) * numax) < total;
            }
            const unsigned m = __ballot_sync(0xffffffffu, real);
            if (real) {
                const unsigned i = nreal + __popc(m & lt_mask);
                CAND[2 * (size_t)(r0 + i)] = a[k];
                CAND[2 * (size_t)(r0 + i) + 1] = b[k];
                pool.a[warp][i & 31u] = a[k];
                pool.b[warp][i & 31u] = b[k];
            }
            nreal += __popc(m);
        }
        __syncwarp();
    }
    collide_tail<S>(P, ch, pool, blk, step, cb, warp_range_len(nslots, W), r0, nreal, nullptr, nullptr, nullptr,
                    nremoved, wtries);
    pdl_trigger();
    if (wtries) atomicAdd(&sh_wtries, wtries);
    if (wemax) atomicAdd(&sh_wemax, wemax);
    if (nremoved) atomicAdd(&sh_removed, nremoved);
    if (wnumax) atomicAdd(&C->cnt.warn_numax, (unsigned long long)wnumax);
    __syncthreads();
    if (tid < np && ch.events[tid]) atomicAdd(&C->cnt.events[S][tid], (unsigned long long)ch.events[tid]);
    if (tid == 0) {
        if (sh_removed) atomicAdd(&C->removed[S], (unsigned long long)sh_removed);
        if (sh_wtries) atomicAdd(&C->cnt.warn_tries, (unsigned long long)sh_wtries);
        if (sh_wemax) atomicAdd(&C->cnt.warn_emax, (unsigned long long)sh_wemax);
    }
}

template <int S>
constexpr int push_min_blocks() { return S == SP_E ? O2PIC_PUSH_E_MIN_BLOCKS : O2PIC_PUSH_MIN_BLOCKS; }

template <int S>
__global__ void __launch_bounds__(BLOCK, push_min_blocks<S>()) k_push(Params P) {
    push_body<S>(P, blockIdx.x, gridDim.x);
}

template <int S>
__global__ void __launch_bounds__(BLOCK, O2PIC_ION_MIN_BLOCKS) k_ion(Params P) {
    ion_body<S>(P, blockIdx.x);
}

// Batched launches: block b works for discharge map[b].x as its block
// map[b].y of map[b].z, with that discharge's parameters copied to shared
// memory (load_params).
template <int S>
__global__ void __launch_bounds__(BLOCK, push_min_blocks<S>()) k_push_b(const Params* __restrict__ all,
                                                                        const uint4* __restrict__ map) {
    __shared__ Params sP;
    const uint4 m = map[blockIdx.x];
    load_params(sP, all + m.x);
    push_body<S>(sP, m.y, m.z);
}

template <int S>
__global__ void __launch_bounds__(BLOCK, O2PIC_ION_MIN_BLOCKS) k_ion_b(const Params* __restrict__ all,
                                                                      const uint4* __restrict__ map) {
    __shared__ Params sP;
    const uint4 m = map[blockIdx.x];
    load_params(sP, all + m.x);
    if (sP.nproc[S] == 0) {   // block-uniform; no block may end before the predecessor has
        pdl_wait();
        return;
    }
    ion_body<S>(sP, m.y);
}

// Deposit of all live particles of one species into Qf (used after a load).
template <int S>
__global__ void __launch_bounds__(BLOCK) k_deposit(Params P) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned* hist = reinterpret_cast<unsigned*>(smem);
    const int Ng = P.Ng, Nc = P.Nc;
    DevCtrl* C = P.ctrl;
    const unsigned cb = C->cur[S];
    const unsigned long long n = C->slots[S];
    const float* X = P.sp[S].x[cb];
    for (int j = threadIdx.x; j < Ng; j += BLOCK) hist[j] = 0u;
    __syncthreads();
    // each block deposits at most 2^16 - 1 particles between flushes
    const unsigned long long per = (unsigned long long)gridDim.x * BLOCK;
    unsigned long long count = 0;
    for (unsigned long long b = (unsigned long long)blockIdx.x * BLOCK; b < n; b += per) {
        const unsigned long long i = b + threadIdx.x;
        if (i < n) {
            const float x = X[i];
            if (!is_dead(x)) deposit_add(hist, x, P.inv_dx, Nc);
        }
        count += BLOCK;
        if (count >= 65536ull - BLOCK) {
            __syncthreads();
            flush_hist(hist, P.Qf[S], Ng);
            __syncthreads();
            count = 0;
        }
    }
    __syncthreads();
    flush_hist(hist, P.Qf[S], Ng);
}

}  // namespace

size_t push_smem_bytes(int species, const Params& P) {
    const size_t base = align16(sizeof(PushShared)) + (sizeof(float) + 2 * sizeof(unsigned)) * P.Ng + sizeof(PushQueue);
    return base + (species == SP_E ? sizeof(float) * NGRID + sizeof(PushPool) + align16(sizeof(CollideShared)) : 0);
}

void launch_flight_init(int species, const Params& P, cudaStream_t s) {
    const unsigned long long cap = P.sp[species].cap;
    const int grid = (int)(cap / 256 + 1 < 4096 ? cap / 256 + 1 : 4096);
    if (species == SP_E) k_flight_init<SP_E><<<grid, 256, 0, s>>>(P);
    else if (species == SP_OM) k_flight_init<SP_OM><<<grid, 256, 0, s>>>(P);
    else k_flight_init<SP_OP><<<grid, 256, 0, s>>>(P);
}

void launch_push(int species, const Params& P, int grid, cudaStream_t s) {
    const size_t sm = push_smem_bytes(species, P);
    if (species == SP_E) launch_pdl(k_push<SP_E>, grid, BLOCK, sm, s, P);
    else if (species == SP_OM) launch_pdl(k_push<SP_OM>, grid, BLOCK, sm, s, P);
    else launch_pdl(k_push<SP_OP>, grid, BLOCK, sm, s, P);
}

void launch_push_batched(int species, const Params* all, const uint4* map, int nblocks, size_t smem, cudaStream_t s) {
    if (species == SP_E) launch_pdl(k_push_b<SP_E>, nblocks, BLOCK, smem, s, all, map);
    else if (species == SP_OM) launch_pdl(k_push_b<SP_OM>, nblocks, BLOCK, smem, s, all, map);
    else launch_pdl(k_push_b<SP_OP>, nblocks, BLOCK, smem, s, all, map);
}

// one block per block of the species' particle kernel
void launch_ion(int species, const Params& P, int grid, cudaStream_t s) {
    if (species == SP_OM) launch_pdl(k_ion<SP_OM>, grid, BLOCK, 0, s, P);
    else if (species == SP_OP) launch_pdl(k_ion<SP_OP>, grid, BLOCK, 0, s, P);
}

void launch_ion_batched(int species, const Params* all, const uint4* map, int nblocks, cudaStream_t s) {
    if (species == SP_OM) launch_pdl(k_ion_b<SP_OM>, nblocks, BLOCK, 0, s, all, map);
    else if (species == SP_OP) launch_pdl(k_ion_b<SP_OP>, nblocks, BLOCK, 0, s, all, map);
}

void launch_deposit(int species, const Params& P, int grid, cudaStream_t s) {
    const size_t sm = sizeof(unsigned) * (size_t)P.Ng;
    if (species == SP_E) k_deposit<SP_E><<<grid, BLOCK, sm, s>>>(P);
    else if (species == SP_OM) k_deposit<SP_OM><<<grid, BLOCK, sm, s>>>(P);
    else k_deposit<SP_OP><<<grid, BLOCK, sm, s>>>(P);
}

// Opt every particle kernel into the shared memory it needs (once per device).
cudaError_t configure_push_smem(size_t max_bytes) {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_push<SP_E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_bytes))) return e;
    if ((e = cudaFuncSetAttribute(k_push<SP_OM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_bytes))) return e;
    if ((e = cudaFuncSetAttribute(k_push<SP_OP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_bytes))) return e;
    if ((e = cudaFuncSetAttribute(k_push_b<SP_E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_bytes))) return e;
    if ((e = cudaFuncSetAttribute(k_push_b<SP_OM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_bytes))) return e;
    if ((e = cudaFuncSetAttribute(k_push_b<SP_OP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_bytes))) return e;
    if ((e = cudaFuncSetAttribute(k_deposit<SP_E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_bytes))) return e;
    if ((e = cudaFuncSetAttribute(k_deposit<SP_OM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_bytes))) return e;
    return cudaFuncSetAttribute(k_deposit<SP_OP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_bytes);
}

int push_occupancy(int species, const Params& P, int* blocks_per_sm) {
    const size_t sm = push_smem_bytes(species, P);
    cudaError_t e;
    if (species == SP_E) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_push<SP_E>, BLOCK, sm);
    else if (species == SP_OM) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_push<SP_OM>, BLOCK, sm);
    else e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_push<SP_OP>, BLOCK, sm);
    return e == cudaSuccess ? 0 : -1;
}

}  // namespace o2
