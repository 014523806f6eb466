// Stable compaction of particle arrays: the slots whose x is not NaN are moved
// to the front of other arrays in their order.  One pass over tiles of TILE
// slots claimed in increasing order by running blocks; each tile's live count
// is combined with the earlier tiles' by a decoupled look-back.
//
// Bound by memory (read and write of every live particle, plus x of the dead
// ones).  A thread keeps the x of its 16 slots in registers from the count to
// the move, the tile's lines of the other arrays are requested into L2 before
// the look-back, and the moves of an array are 16 independent loads and stores
// per thread, coalesced (a warp's 32 lanes take neighbouring slots).  The
// look-back reads 32 earlier tiles at a time, one per lane.  2e7 particles with
// a twentieth removed (764 MB) 378 -> 254 us, 3.0 TB/s; a tile's blocks still wait
// between its count and its move.
#pragma once

#include "common.cuh"

namespace o2 {

constexpr int CMP_T = 512;                    // threads of the compaction kernels
constexpr int CMP_I = TILE / CMP_T;           // slots of a tile per thread (16)
constexpr int CMP_W = CMP_T / 32;

struct CompactShared {
    unsigned wsum[CMP_W];
    unsigned tile, total;
    unsigned long long excl;
    int ok;
};

// The look-back of one tile by one warp (all lanes call it).  Publishes the
// tile's aggregate, walks back to the nearest inclusive prefix, publishes the
// tile's own inclusive prefix and returns the exclusive prefix.  Per tile: a
// flag word = (epoch << 2) | state (1 = aggregate published, 2 = inclusive
// prefix published) and two value words (val[2t] = aggregate, val[2t+1] =
// inclusive prefix).  A value is stored before its flag (release) and read
// after the flag (acquire); the aggregate word is never rewritten, so a reader
// that saw state 1 reads the aggregate even if the tile has meanwhile
// published its prefix.  Tiles are claimed in increasing order by running
// blocks, so every predecessor is being processed; the wait is still bounded:
// on giving up the error flag is set, *ok = false and the caller skips its
// writes.
constexpr unsigned LOOKBACK_SPIN_LIMIT = 1u << 22;

__device__ __forceinline__ unsigned long long lookback(unsigned long long* flag, unsigned long long* val,
                                                       unsigned tile, unsigned long long agg,
                                                       unsigned long long epoch, unsigned long long* err, bool* ok) {
    const int lane = threadIdx.x & 31;
    *ok = true;
    if (lane == 0) {
        st_relaxed(&val[2 * (size_t)tile + (tile == 0 ? 1 : 0)], agg);
        st_release(&flag[tile], (epoch << 2) | (tile == 0 ? 2ull : 1ull));
    }
    if (tile == 0) return 0ull;
    unsigned long long excl = 0ull;
    for (int j = (int)tile - 1; j >= 0; j -= 32) {
        const int i = j - lane;
        unsigned long long f = 2ull, v = 0ull;    // before tile 0: an empty prefix
        bool gave_up = false;
        if (i >= 0) {
            unsigned spins = 0;
            while (((f = ld_acquire(&flag[i])) >> 2) != epoch) {
                if (++spins > LOOKBACK_SPIN_LIMIT) { gave_up = true; break; }
                if (spins > 64) __nanosleep(64);
            }
            if (!gave_up) v = ld_relaxed(&val[2 * (size_t)i + ((f & 3ull) == 2ull ? 1 : 0)]);
        }
        if (__any_sync(0xffffffffu, gave_up)) {
            if (lane == 0) atomicOr(err, ERR_TIMEOUT);
            *ok = false;
            return 0ull;
        }
        // lanes up to the nearest tile with an inclusive prefix
        const unsigned m = __ballot_sync(0xffffffffu, (f & 3ull) == 2ull);
        if (m && lane > __ffs(m) - 1) v = 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        excl += v;
        if (m) break;
    }
    if (lane == 0) {
        st_relaxed(&val[2 * (size_t)tile + 1], excl + agg);
        st_release(&flag[tile], (epoch << 2) | 2ull);
    }
    return excl;
}

// The tiles that this block claims from *ticket.  request(slot): prefetch of
// the other arrays at a slot; move(x, base, d, off, in): copy of one thread's
// slots (x[i] and slot base + 32 i of the other arrays to d + off[i] where bit i
// of `in` is set); total(n): called once, with the number kept, by the block of
// the last tile.
template <class Request, class Move, class Total>
__device__ __forceinline__ void compact_tiles(CompactShared& sh, const float* __restrict__ X, unsigned long long n,
                                              unsigned* ticket, unsigned long long* flag, unsigned long long* val,
                                              unsigned long long epoch, unsigned long long* err, Request&& request,
                                              Move&& move, Total&& total) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const unsigned ntiles = (unsigned)ceil_div(n, TILE);
    for (;;) {
        if (tid == 0) sh.tile = atomicAdd(ticket, 1u);
        __syncthreads();
        const unsigned tile = sh.tile;
        if (tile >= ntiles) break;
        // warp w: CMP_I rounds of 32 slots from its part of the tile
        const unsigned long long base = (unsigned long long)tile * TILE + (unsigned)(warp * CMP_I * 32 + lane);
        // one line (32 slots) of the other arrays per thread
        if ((tid & 1) == 0 && (unsigned long long)tile * TILE + 16ull * tid < n)
            request((unsigned long long)tile * TILE + 16ull * tid);
        float x[CMP_I];
        unsigned in = 0u, cnt = 0u;
#pragma unroll
        for (int i = 0; i < CMP_I; ++i) x[i] = (base + 32u * i < n) ? X[base + 32u * i] : dead_marker();
#pragma unroll
        for (int i = 0; i < CMP_I; ++i) {
            if (!is_dead(x[i])) in |= 1u << i;
            cnt += __popc(__ballot_sync(0xffffffffu, !is_dead(x[i])));
        }
        if (lane == 0) sh.wsum[warp] = cnt;
        __syncthreads();
        if (warp == 0) {
            unsigned v = lane < CMP_W ? sh.wsum[lane] : 0u;
            const unsigned own = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += y;
            }
            const unsigned all = __shfl_sync(0xffffffffu, v, 31);
            if (lane < CMP_W) sh.wsum[lane] = v - own;
            bool ok;
            const unsigned long long excl = lookback(flag, val, tile, all, epoch, err, &ok);
            if (lane == 0) {
                sh.excl = excl;
                sh.ok = ok ? 1 : 0;
                if (ok && tile == ntiles - 1) total(excl + all);
            }
        }
        __syncthreads();
        if (sh.ok) {
            unsigned long long d = sh.excl + sh.wsum[warp];
            unsigned off[CMP_I], run = 0u;
#pragma unroll
            for (int i = 0; i < CMP_I; ++i) {
                const unsigned b = __ballot_sync(0xffffffffu, !is_dead(x[i]));
                off[i] = run + __popc(b & lt);
                run += __popc(b);
            }
            move(x, base, d, off, in);
        }
    }
}

// One array's part of a move: CMP_I loads, then CMP_I stores; destinations
// at or beyond `cap` are left out.
template <class T>
__device__ __forceinline__ void move_array(T* __restrict__ D, const T* __restrict__ A, unsigned long long base,
                                           unsigned long long d, const unsigned (&off)[CMP_I], unsigned in,
                                           unsigned long long cap) {
    T v[CMP_I];
#pragma unroll
    for (int i = 0; i < CMP_I; ++i) v[i] = ((in >> i) & 1u) ? A[base + 32u * i] : T(0);
#pragma unroll
    for (int i = 0; i < CMP_I; ++i)
        if (((in >> i) & 1u) && d + off[i] < cap) D[d + off[i]] = v[i];
}

template <class T>
__device__ __forceinline__ void prefetch_l2(const T* p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

}  // namespace o2
