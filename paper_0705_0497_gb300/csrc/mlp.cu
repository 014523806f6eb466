// Small multilayer perceptron for the learned warm start of a discharge:
// (U, p, L, C) -> cycle-averaged log-density profiles.  Weights bf16 (an
// fp32 master copy is what Adam updates), every product accumulated in fp32,
// tanh on the hidden layers, linear output; mean-squared-error loss.
//
// Shapes are small (widths of a few hundred, batches of a few to a few
// thousand rows): a call is a chain of short launches, bound by their latency
// up to some hundred rows and by the fp32 FMA rate and shared memory beyond.
// Every output is one chain of fused multiply-adds in the order of k
// (deterministic, the same for every tile shape), so the contractions are
// tiled FMA kernels, not the tensor cores, whose sums round in another order.
// Tiles are chosen by size so that a contraction has a block for every SM;
// the gradients of all layers' weights and biases (and the Adam update of a
// training step, in their epilogue) are one launch.
//
// Parameter layout (fp32 master, gradients, Adam moments): for each layer l,
// W_l as [in_l][out_l] row-major, then b_l[out_l].  The bf16 copy of the
// weights uses the same offsets.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>
#include <new>
#include <vector>

#include "common.cuh"

namespace o2 {
namespace {

enum Epi { EPI_NONE = 0, EPI_TANH = 1, EPI_DTANH = 2 };

__device__ __forceinline__ float ldf(const float* p) { return *p; }
__device__ __forceinline__ float ldf(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// Adam (Kingma & Ba 2015) on the fp32 master parameters with gradients g[k] at
// indices i[k] (where in[k]), then the bf16 copies of weights; all loads before
// the first store.
struct Adam {
    float *P, *Mo, *Ve;
    __nv_bfloat16* Wb;
    float lr, b1, b2, eps, c1, c2;
    template <int N>
    __device__ __forceinline__ void step(const size_t (&i)[N], const float (&g)[N], const bool (&in)[N],
                                         bool weight) const {
        float mo[N], ve[N], p[N];
#pragma unroll
        for (int k = 0; k < N; ++k) {
            mo[k] = in[k] ? Mo[i[k]] : 0.0f;
            ve[k] = in[k] ? Ve[i[k]] : 0.0f;
            p[k] = in[k] ? P[i[k]] : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < N; ++k) {
            if (!in[k]) continue;
            const float m = fmaf(b1, mo[k], (1.0f - b1) * g[k]);
            const float v = fmaf(b2, ve[k], (1.0f - b2) * g[k] * g[k]);
            Mo[i[k]] = m;
            Ve[i[k]] = v;
            const float q = p[k] - lr * (m / c1) / (sqrtf(v / c2) + eps);
            P[i[k]] = q;
            if (weight) Wb[i[k]] = __float2bfloat16_rn(q);
        }
    }
};

// One output tile (TM x TN at m0, n0) of C[m][n] = epi( sum_k A(m,k) B(k,n) +
// bias[n] ), summed over k in order by one chain of FMAs per output.
// A(m,k) = TA ? A[k lda + m] : A[m lda + k];  B(k,n) = TB ? B[n ldb + k] : B[k ldb + n].
// Each of the (TM/4)(TN/4) threads owns 4 x 4 neighbouring outputs; k-slices of
// KS go through shared memory in two stages, the next slice's global loads in
// flight while this one is summed (a slice is long enough to cover an L2 round
// trip).  Shared rows are k; SWIZZLE permutes their groups of four columns by k,
// so that an operand whose k is contiguous in memory is stored without bank
// conflicts while fragments stay 16-byte words.
template <int TM, int TN, int KS, bool SWIZZLE>
struct Tile {
    static constexpr int RM = 4, RN = 4;
    static constexpr int TX = TN / RN, NT = (TM / RM) * TX;
    static_assert(KS % 8 == 0 && TM % 32 == 0 && TN % 32 == 0, "whole groups");
    struct Shared {
        __align__(16) float A[2][KS][TM];
        __align__(16) float B[2][KS][TN];
    };
    static __device__ __forceinline__ int col(int k, int x) {
        return SWIZZLE ? ((((x >> 2) ^ ((k ^ (k >> 2)) & 7)) << 2) | (x & 3)) : x;
    }
    // element e of a slice of T columns: its k and column
    template <bool KFAST, int T>
    static __device__ __forceinline__ void place(int e, int& k, int& x) {
        if (KFAST) {
            const int hi = e >> 5;
            k = (hi % (KS / 8)) * 8 + (e & 7);
            x = (hi / (KS / 8)) * 4 + ((e >> 3) & 3);
        } else {
            k = e / T;
            x = e % T;
        }
    }

    // One operand's part of a slice, CNT columns of KS k, in registers between
    // its global loads and its stores to shared memory.  VEC: 16-byte loads (4
    // floats or 8 bf16) along the direction contiguous in memory, which needs
    // base, row length and extent to be multiples of that.
    template <int CNT, bool KFAST, bool VEC, typename T>
    struct Part {
        static constexpr int V = VEC ? 16 / (int)sizeof(T) : 1;
        static constexpr int L = CNT * KS / NT / V;           // loads per thread
        static_assert(L * V * NT == CNT * KS, "whole loads per thread");
        float v[L][V];
        static __device__ __forceinline__ void where(int i, int& k, int& x) {
            const int e = (int)threadIdx.x + i * NT;
            if (!VEC) place<KFAST, CNT>(e, k, x);
            else if (KFAST) { k = (e % (KS / V)) * V; x = e / (KS / V); }
            else { x = (e % (CNT / V)) * V; k = e / (CNT / V); }
        }
        __device__ __forceinline__ void load(const T* __restrict__ g, int ld, int k0, int x0, int K, int X) {
#pragma unroll
            for (int i = 0; i < L; ++i) {
                int kk, xx;
                where(i, kk, xx);
                const int k = k0 + kk, x = x0 + xx;
                const bool in = k < K && x < X;
                const T* p = g + (KFAST ? (size_t)x * ld + k : (size_t)k * ld + x);
                if (VEC) {
                    const uint4 q = in ? *reinterpret_cast<const uint4*>(p) : make_uint4(0u, 0u, 0u, 0u);
                    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                    for (int j = 0; j < V; ++j)
                        v[i][j] = sizeof(T) == 4 ? __uint_as_float(w[j % 4])
                                                 : __uint_as_float((j & 1) ? w[j / 2] & 0xFFFF0000u : w[j / 2] << 16);
                } else {
                    v[i][0] = in ? ldf(p) : 0.0f;
                }
            }
        }
        __device__ __forceinline__ void stage(float (&dst)[KS][CNT]) const {
#pragma unroll
            for (int i = 0; i < L; ++i) {
                int kk, xx;
                where(i, kk, xx);
                if (VEC && !KFAST) {
#pragma unroll
                    for (int j = 0; j < V; j += 4)
                        *reinterpret_cast<float4*>(&dst[kk][col(kk, xx + j)]) =
                            make_float4(v[i][j], v[i][(j + 1) % V], v[i][(j + 2) % V], v[i][(j + 3) % V]);
                } else {
#pragma unroll
                    for (int j = 0; j < V; ++j) dst[kk + j][col(kk + j, xx)] = v[i][j];
                }
            }
        }
    };

    // the thread's outputs: rows m0 + ty RM + i, columns n0 + tx RN + j
    template <bool TA, bool TB, bool VEC, typename BT>
    static __device__ __forceinline__ void run(Shared& sh, const float* __restrict__ A, int lda,
                                               const BT* __restrict__ B, int ldb, int M, int N, int K, int m0, int n0,
                                               float (&acc)[RM][RN]) {
        const int t = threadIdx.x, tx = t % TX, ty = t / TX;
        Part<TM, !TA, VEC, float> pa;
        Part<TN, TB, VEC, BT> pb;
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
            for (int j = 0; j < RN; ++j) acc[i][j] = 0.0f;
        pa.load(A, lda, 0, m0, K, M);
        pb.load(B, ldb, 0, n0, K, N);
        pa.stage(sh.A[0]);
        pb.stage(sh.B[0]);
        __syncthreads();
        int s = 0;
        for (int k0 = 0; k0 < K; k0 += KS, s ^= 1) {
            const bool more = k0 + KS < K;
            if (more) {
                pa.load(A, lda, k0 + KS, m0, K, M);
                pb.load(B, ldb, k0 + KS, n0, K, N);
            }
            constexpr int UN = SWIZZLE ? KS : 16;
#pragma unroll UN
            for (int kk = 0; kk < KS; ++kk) {
                const float4 av = *reinterpret_cast<const float4*>(&sh.A[s][kk][col(kk, 4 * ty)]);
                const float4 bv = *reinterpret_cast<const float4*>(&sh.B[s][kk][col(kk, 4 * tx)]);
                const float a[RM] = {av.x, av.y, av.z, av.w}, b[RN] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                for (int i = 0; i < RM; ++i)
#pragma unroll
                    for (int j = 0; j < RN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
            }
            if (more) {
                pa.stage(sh.A[s ^ 1]);   // last read in the slice before this one
                pb.stage(sh.B[s ^ 1]);
                __syncthreads();
            }
        }
    }
};

// Whether an operand can be read 16 bytes at a time: `fast` is the extent along
// its contiguous direction.
template <typename T>
__host__ __device__ inline bool in_words(const T* p, int ld, int fast) {
    constexpr int V = 16 / (int)sizeof(T);
    return ((size_t)p & 15) == 0 && ld % V == 0 && fast % V == 0;
}

// Forward contractions and gradients at the pre-activations of many rows.
using Large = Tile<64, 64, 32, true>;
// Weight gradients (outputs in x out, sums over the batch rows).
using Grad = Tile<64, 32, 48, false>;

// EPI_TANH: tanh of the sum; EPI_DTANH: the sum times (1 - H[m][n]^2).
__device__ __forceinline__ float epilogue(float v, int epi, const float* __restrict__ bias,
                                          const float* __restrict__ H, int m, int n, int N) {
    if (bias) v += bias[n];
    if (epi == EPI_TANH) v = tanhf(v);
    else if (epi == EPI_DTANH) { const float h = H[(size_t)m * N + n]; v = v * (1.0f - h * h); }
    return v;
}

template <bool TB, bool VEC>
__global__ void __launch_bounds__(Large::NT) k_gemm(const float* __restrict__ A, int lda,
                                                    const __nv_bfloat16* __restrict__ B, int ldb,
                                                    float* __restrict__ C, int M, int N, int K,
                                                    const float* __restrict__ bias, int epi,
                                                    const float* __restrict__ H) {
    __shared__ Large::Shared sh;
    pdl_wait();
    pdl_trigger();
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    float acc[4][4];
    Large::run<false, TB, VEC>(sh, A, lda, B, ldb, M, N, K, m0, n0, acc);
    const int tx = threadIdx.x % Large::TX, ty = threadIdx.x / Large::TX;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int m = m0 + ty * 4 + i, n = n0 + tx * 4 + j;
            if (m < M && n < N) C[(size_t)m * N + n] = epilogue(acc[i][j], epi, bias, H, m, n, N);
        }
}

// The same for few rows: a block has 8 rows (a warp each) and 32 columns (a lane
// each), one output and one chain of FMAs per thread, so that even 32 x 256
// outputs use 32 SMs.  What bounds it is latency: the launch, one L2 round trip
// per panel of 256 k (the next panel's loads in flight while this one is
// summed) and the chain itself (4 cycles per k; 4 k take one 16-byte broadcast
// load of A and two words of B, each a pair of bf16 at neighbouring k).
constexpr int RM_ = 8, RN_ = 32, RK = 256, RT = 256;
struct FewShared {
    __align__(16) float A[RM_][RK + 4];
    uint32_t B[RK / 2][RN_ + 1];
};

template <bool TB>
__global__ void __launch_bounds__(RT) k_gemm_few(const float* __restrict__ A, int lda,
                                                 const __nv_bfloat16* __restrict__ B, int ldb, float* __restrict__ C,
                                                 int M, int N, int K, const float* __restrict__ bias, int epi,
                                                 const float* __restrict__ H) {
    __shared__ FewShared sh;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int m0 = blockIdx.y * RM_, n0 = blockIdx.x * RN_;
    constexpr int PA = RM_ * RK / RT, PB = RN_ * RK / RT;   // 8 and 32 per thread
    float pa[PA];
    unsigned short pb[PB];
    const unsigned short* __restrict__ Bu = reinterpret_cast<const unsigned short*>(B);
    // panel [k0, k0 + RK): thread t loads k0 + t of each row of A, and of B
    // column t (TB: k contiguous in memory) or lane's column of rows k0 + warp +
    // 8 i (n contiguous)
    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < PA; ++i) pa[i] = (m0 + i < M && k0 + t < K) ? A[(size_t)(m0 + i) * lda + k0 + t] : 0.0f;
#pragma unroll
        for (int i = 0; i < PB; ++i) {
            if (TB) pb[i] = (n0 + i < N && k0 + t < K) ? Bu[(size_t)(n0 + i) * ldb + k0 + t] : (unsigned short)0;
            else pb[i] = (n0 + lane < N && k0 + warp + 8 * i < K) ? Bu[(size_t)(k0 + warp + 8 * i) * ldb + n0 + lane]
                                                                  : (unsigned short)0;
        }
    };
    pdl_wait();
    pdl_trigger();
    load(0);
    float acc = 0.0f;
    for (int k0 = 0; k0 < K; k0 += RK) {
        if (k0 > 0) __syncthreads();
#pragma unroll
        for (int i = 0; i < PA; ++i) sh.A[i][t] = pa[i];
        unsigned short* b16 = reinterpret_cast<unsigned short*>(sh.B);
#pragma unroll
        for (int i = 0; i < PB; ++i) {
            const int k = TB ? t : warp + 8 * i, n = TB ? i : lane;
            b16[2 * ((k >> 1) * (RN_ + 1) + n) + (k & 1)] = pb[i];
        }
        __syncthreads();
        if (k0 + RK < K) load(k0 + RK);
        const int kn = min(RK, K - k0);
#pragma unroll 8
        for (int k = 0; k < kn; k += 4) {              // beyond K: zeros
            const float4 a = *reinterpret_cast<const float4*>(&sh.A[warp][k]);
            const uint32_t b0 = sh.B[k / 2][lane], b1 = sh.B[k / 2 + 1][lane];
            acc = fmaf(a.x, __uint_as_float(b0 << 16), acc);
            acc = fmaf(a.y, __uint_as_float(b0 & 0xFFFF0000u), acc);
            acc = fmaf(a.z, __uint_as_float(b1 << 16), acc);
            acc = fmaf(a.w, __uint_as_float(b1 & 0xFFFF0000u), acc);
        }
    }
    const int m = m0 + warp, n = n0 + lane;
    if (m < M && n < N) C[(size_t)m * N + n] = epilogue(acc, epi, bias, H, m, n, N);
}

// dY = 2 (Y - T) / (B N); per-block partial sums of (Y - T)^2 (fixed order).
// Eight elements are loaded before the first is used.
__global__ void k_mse(const float* __restrict__ Y, const float* __restrict__ T, float* __restrict__ dY, size_t n,
                      float scale, float* __restrict__ partial) {
    __shared__ float red[256];
    pdl_wait();
    pdl_trigger();
    float s = 0.0f;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += 8 * stride) {
        float y[8], t[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const bool in = i + k * stride < n;
            y[k] = in ? Y[i + k * stride] : 0.0f;
            t[k] = in ? T[i + k * stride] : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (i + k * stride >= n) break;
            const float d = y[k] - t[k];
            dY[i + k * stride] = 2.0f * d * scale;
            s = fmaf(d, d, s);
        }
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

// All layers' weight and bias gradients, and the loss, in one launch: the
// tiles of dW_l = H_{l-1}^T dZ_l first (layer by layer), then blocks of NT
// columns of db_l = column sums of dZ_l (rows in order), then one block for the
// loss.  Written to G (parameter layout), or applied at once (Adam).
constexpr int MAX_LAYERS = 15;
struct GradJobs {
    const float* H[MAX_LAYERS];
    const float* dZ[MAX_LAYERS];
    int K[MAX_LAYERS], N[MAX_LAYERS];
    bool vec[MAX_LAYERS];                    // both operands in 16-byte words
    size_t offW[MAX_LAYERS], offB[MAX_LAYERS];
    int first_w[MAX_LAYERS + 1], first_b[MAX_LAYERS + 1];   // block numbers
    int layers, B;
    float* G;
    const float* partial;
    float* loss;
    int npartial;
    float scale;
};

template <bool UPDATE>
__global__ void __launch_bounds__(Grad::NT) k_grads(GradJobs J, Adam ad) {
    __shared__ Grad::Shared sh;
    pdl_wait();
    pdl_trigger();
    const int blk = (int)blockIdx.x;
    const int B = J.B;
    if (blk < J.first_w[J.layers]) {
        int l = 0;
        while (blk >= J.first_w[l + 1]) ++l;
        const int K = J.K[l], N = J.N[l], tiles_n = (N + 31) / 32, r = blk - J.first_w[l];
        const int m0 = (r / tiles_n) * 64, n0 = (r % tiles_n) * 32;
        float acc[4][4];
        if (J.vec[l]) Grad::run<true, false, true>(sh, J.H[l], K, J.dZ[l], N, K, N, B, m0, n0, acc);
        else Grad::run<true, false, false>(sh, J.H[l], K, J.dZ[l], N, K, N, B, m0, n0, acc);
        const int tx = threadIdx.x % Grad::TX, ty = threadIdx.x / Grad::TX;
        size_t idx[16];
        float g[16];
        bool in[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int m = m0 + ty * 4 + k / 4, n = n0 + tx * 4 + k % 4;
            in[k] = m < K && n < N;
            idx[k] = J.offW[l] + (size_t)m * N + n;
            g[k] = acc[k / 4][k % 4];
            if (!UPDATE && in[k]) J.G[idx[k]] = g[k];
        }
        if (UPDATE) ad.step<16>(idx, g, in, true);
    } else if (blk < J.first_b[J.layers]) {
        int l = 0;
        while (blk >= J.first_b[l + 1]) ++l;
        const int N = J.N[l], n = (blk - J.first_b[l]) * Grad::NT + (int)threadIdx.x;
        if (n >= N) return;
        const float* __restrict__ dZ = J.dZ[l];
        float s = 0.0f;
        int m = 0;
        for (; m + 16 <= B; m += 16) {
            float v[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = dZ[(size_t)(m + k) * N + n];
#pragma unroll
            for (int k = 0; k < 16; ++k) s += v[k];
        }
        for (; m < B; ++m) s += dZ[(size_t)m * N + n];
        const size_t idx[1] = {J.offB[l] + n};
        const float g[1] = {s};
        const bool in[1] = {true};
        if (UPDATE) ad.step<1>(idx, g, in, false);
        else J.G[idx[0]] = s;
    } else if (threadIdx.x == 0) {
        float s = 0.0f;
#pragma unroll 8
        for (int i = 0; i < J.npartial; ++i) s += J.partial[i];
        *J.loss = s * J.scale;
    }
}

__global__ void k_to_bf16(const float* __restrict__ P, __nv_bfloat16* __restrict__ Wb,
                          const unsigned char* __restrict__ is_w, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        if (is_w[i]) Wb[i] = __float2bfloat16_rn(P[i]);
}

// C = epi(A B + bias) with A [M][K] fp32, B bf16 [K][N] (or its transpose
// [N][K]: TB).  The large tile when its grid fills three quarters of the SMs,
// else k_gemm_few.  2000 rows of 256 to 256 (128 large tiles): 17 us (the
// former 64 x 64 kernel without prefetch 31); 81 rows of 256 to 256 (88 blocks
// of 8 x 32): 5.4 us by k_gemm_few, 13 by such a tile with short slices, 38
// before.
template <bool TB>
void gemm(const float* A, int lda, const __nv_bfloat16* B, int ldb, float* C, int M, int N, int K, const float* bias,
          int epi, const float* H, int sms, cudaStream_t s) {
    const long long large = (long long)((N + 63) / 64) * ((M + 63) / 64);
    if (4 * large >= 3 * sms) {
        const dim3 grid((N + 63) / 64, (M + 63) / 64);
        if (in_words(A, lda, K) && in_words(B, ldb, TB ? K : N))
            launch_pdl(k_gemm<TB, true>, grid, Large::NT, 0, s, A, lda, B, ldb, C, M, N, K, bias, epi, H);
        else
            launch_pdl(k_gemm<TB, false>, grid, Large::NT, 0, s, A, lda, B, ldb, C, M, N, K, bias, epi, H);
    } else {
        const dim3 grid((N + RN_ - 1) / RN_, (M + RM_ - 1) / RM_);
        launch_pdl(k_gemm_few<TB>, grid, RT, 0, s, A, lda, B, ldb, C, M, N, K, bias, epi, H);
    }
}

}  // namespace
}  // namespace o2

using namespace o2;

struct o2pic_mlp {
    int device = 0;
    std::vector<int> w;                    // widths, w[0] = inputs, w[L] = outputs
    std::vector<size_t> offW, offB;        // parameter offsets per layer
    size_t nparams = 0;
    float *P = nullptr, *G = nullptr, *Mo = nullptr, *Ve = nullptr;
    __nv_bfloat16* Wb = nullptr;
    unsigned char* is_w = nullptr;
    // for a batch of up to cap rows: activations H[l] (l = 1..L-1); of up to
    // gcap rows: output Y, gradients at the pre-activations dZ[l] (l = 1..L)
    int cap = 0, gcap = 0;
    std::vector<float*> H, dZ;
    float *Y = nullptr, *partial = nullptr;
    int sms = 0;
    unsigned long long t = 0;              // Adam steps taken
};

namespace {

constexpr int MSE_BLOCKS = 120;
constexpr int CARVEOUT = 30;   // per cent shared memory (about two blocks of the large tile)

int layers(const o2pic_mlp* m) { return (int)m->w.size() - 1; }

void free_rows(std::vector<float*>& v) {
    for (float* p : v) if (p) cudaFree(p);
    v.clear();
}

void free_acts(o2pic_mlp* m) {
    free_rows(m->H);
    m->cap = 0;
}

void free_grads(o2pic_mlp* m) {
    free_rows(m->dZ);
    if (m->Y) cudaFree(m->Y);
    m->Y = nullptr;
    m->gcap = 0;
}

// v[l] = B rows of layer l's width, l = 1..last.
int alloc_rows(o2pic_mlp* m, std::vector<float*>& v, int last, int B) {
    v.assign(last + 1, nullptr);
    for (int l = 1; l <= last; ++l)
        if (cudaMalloc((void**)&v[l], sizeof(float) * (size_t)B * m->w[l]) != cudaSuccess) return O2PIC_E_CUDA;
    return O2PIC_OK;
}

int ensure_acts(o2pic_mlp* m, int B) {
    if (B <= m->cap) return O2PIC_OK;
    free_acts(m);
    if (int rc = alloc_rows(m, m->H, layers(m) - 1, B)) return rc;
    m->cap = B;
    return O2PIC_OK;
}

// What a backward pass needs besides (a caller who only runs forward does not
// hold it).
int ensure_grads(o2pic_mlp* m, int B) {
    if (B <= m->gcap) return O2PIC_OK;
    free_grads(m);
    const int L = layers(m);
    if (int rc = alloc_rows(m, m->dZ, L, B)) return rc;
    if (cudaMalloc((void**)&m->Y, sizeof(float) * (size_t)B * m->w[L]) != cudaSuccess) return O2PIC_E_CUDA;
    m->gcap = B;
    return O2PIC_OK;
}

// Forward pass of B rows of X into m->H and out (the output layer).
void forward(o2pic_mlp* m, const float* X, float* out, int B, cudaStream_t s) {
    const int L = layers(m);
    const float* in = X;
    for (int l = 1; l <= L; ++l) {
        const int K = m->w[l - 1], N = m->w[l];
        float* dst = (l == L) ? out : m->H[l];
        gemm<false>(in, K, m->Wb + m->offW[l - 1], N, dst, B, N, K, m->P + m->offB[l - 1],
                    l == L ? EPI_NONE : EPI_TANH, nullptr, m->sms, s);
        in = dst;
    }
}

// Loss and gradients of the mean-squared error over B rows into G, or (adam)
// applied to the parameters as they are formed: nothing after the gradients at
// the pre-activations reads the weights.
void backward(o2pic_mlp* m, const float* X, const float* T, int B, float* loss, float* G, const Adam* adam,
              cudaStream_t s) {
    const int L = layers(m);
    const size_t nout = (size_t)B * m->w[L];
    const float scale = 1.0f / (float)nout;
    launch_pdl(k_mse, MSE_BLOCKS, 256, 0, s, m->Y, T, m->dZ[L], nout, scale, m->partial);
    for (int l = L; l > 1; --l) {
        // dZ_{l-1} = (dZ_l W_l^T) (1 - H_{l-1}^2)
        const int K = m->w[l - 1], N = m->w[l];
        gemm<true>(m->dZ[l], N, m->Wb + m->offW[l - 1], N, m->dZ[l - 1], B, K, N, nullptr, EPI_DTANH, m->H[l - 1],
                   m->sms, s);
    }
    GradJobs J = {};
    J.layers = L;
    J.B = B;
    J.G = G;
    J.partial = m->partial;
    J.npartial = MSE_BLOCKS;
    J.loss = loss;
    J.scale = scale;
    int blk = 0;
    for (int i = 0; i < L; ++i) {
        J.H[i] = i == 0 ? X : m->H[i];
        J.dZ[i] = m->dZ[i + 1];
        J.K[i] = m->w[i];
        J.N[i] = m->w[i + 1];
        J.vec[i] = in_words(J.H[i], J.K[i], J.K[i]) && in_words(J.dZ[i], J.N[i], J.N[i]);
        J.offW[i] = m->offW[i];
        J.offB[i] = m->offB[i];
        J.first_w[i] = blk;
        blk += ((J.K[i] + 63) / 64) * ((J.N[i] + 31) / 32);
    }
    J.first_w[L] = blk;
    for (int i = 0; i < L; ++i) {
        J.first_b[i] = blk;
        blk += (J.N[i] + Grad::NT - 1) / Grad::NT;
    }
    J.first_b[L] = blk;
    if (adam) launch_pdl(k_grads<true>, blk + 1, Grad::NT, 0, s, J, *adam);
    else launch_pdl(k_grads<false>, blk + 1, Grad::NT, 0, s, J, Adam{});
}

// One division of the SM's memory between L1 and shared memory for all of the
// network's kernels: an SM changes it only when it is empty, so kernels that ask
// for different ones cannot overlap and cost some microseconds at each change
// (gradients over 2000 rows: 317 -> 262 us).
cudaError_t configure_carveout() {
    const void* k[] = {(const void*)k_gemm<false, false>, (const void*)k_gemm<false, true>,
                       (const void*)k_gemm<true, false>,  (const void*)k_gemm<true, true>,
                       (const void*)k_gemm_few<false>,    (const void*)k_gemm_few<true>,
                       (const void*)k_grads<false>,       (const void*)k_grads<true>,
                       (const void*)k_mse,                (const void*)k_to_bf16};
    for (const void* f : k)
        if (cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, CARVEOUT)) return e;
    return cudaSuccess;
}

// SplitMix64 (Steele, Lea & Flood 2014) for the initial weights.
uint64_t splitmix64(uint64_t& x) {
    uint64_t z = (x += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

}  // namespace

extern "C" {

int o2pic_mlp_create(const int32_t* widths, int32_t n_widths, uint64_t seed, o2pic_mlp** out) {
    if (!out) return O2PIC_E_INVALID_ARG;
    *out = nullptr;
    if (!widths || n_widths < 2 || n_widths > 16) return O2PIC_E_INVALID_ARG;
    for (int i = 0; i < n_widths; ++i)
        if (widths[i] < 1 || widths[i] > 8192) return O2PIC_E_INVALID_ARG;
    o2pic_mlp* m = new (std::nothrow) o2pic_mlp;
    if (!m) return O2PIC_E_CUDA;
    cudaGetDevice(&m->device);
    cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, m->device);
    m->w.assign(widths, widths + n_widths);
    const int L = n_widths - 1;
    for (int l = 0; l < L; ++l) {
        m->offW.push_back(m->nparams);
        m->nparams += (size_t)m->w[l] * m->w[l + 1];
        m->offB.push_back(m->nparams);
        m->nparams += (size_t)m->w[l + 1];
    }
    // Glorot-uniform weights U(-a, a), a = sqrt(6 / (in + out)); zero biases
    std::vector<float> P(m->nparams, 0.0f);
    std::vector<unsigned char> isw(m->nparams, 0);
    uint64_t st = seed;
    for (int l = 0; l < L; ++l) {
        const double a = std::sqrt(6.0 / (double)(m->w[l] + m->w[l + 1]));
        const size_t n = (size_t)m->w[l] * m->w[l + 1];
        for (size_t i = 0; i < n; ++i) {
            const double u = (double)(splitmix64(st) >> 11) * (1.0 / 9007199254740992.0);
            P[m->offW[l] + i] = (float)((2.0 * u - 1.0) * a);
            isw[m->offW[l] + i] = 1;
        }
    }
    bool ok = cudaMalloc((void**)&m->P, sizeof(float) * m->nparams) == cudaSuccess &&
              cudaMalloc((void**)&m->G, sizeof(float) * m->nparams) == cudaSuccess &&
              cudaMalloc((void**)&m->Mo, sizeof(float) * m->nparams) == cudaSuccess &&
              cudaMalloc((void**)&m->Ve, sizeof(float) * m->nparams) == cudaSuccess &&
              cudaMalloc((void**)&m->Wb, sizeof(__nv_bfloat16) * m->nparams) == cudaSuccess &&
              cudaMalloc((void**)&m->is_w, m->nparams) == cudaSuccess &&
              cudaMalloc((void**)&m->partial, sizeof(float) * MSE_BLOCKS) == cudaSuccess;
    ok = ok && cudaMemcpy(m->is_w, isw.data(), m->nparams, cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemset(m->G, 0, sizeof(float) * m->nparams) == cudaSuccess &&
         cudaMemset(m->Mo, 0, sizeof(float) * m->nparams) == cudaSuccess &&
         cudaMemset(m->Ve, 0, sizeof(float) * m->nparams) == cudaSuccess &&
         cudaMemset(m->Wb, 0, sizeof(__nv_bfloat16) * m->nparams) == cudaSuccess;
    ok = ok && configure_carveout() == cudaSuccess;
    if (!ok) { o2pic_mlp_destroy(m); return O2PIC_E_CUDA; }
    *out = m;
    return o2pic_mlp_set_params(m, P.data());
}

uint64_t o2pic_mlp_num_params(o2pic_mlp* m) { return m ? m->nparams : 0; }

int o2pic_mlp_set_params(o2pic_mlp* m, const float* host) {
    if (!m || !host) return O2PIC_E_INVALID_ARG;
    if (cudaSetDevice(m->device) != cudaSuccess) return O2PIC_E_CUDA;
    if (cudaMemcpy(m->P, host, sizeof(float) * m->nparams, cudaMemcpyHostToDevice) != cudaSuccess) return O2PIC_E_CUDA;
    k_to_bf16<<<120, 256>>>(m->P, m->Wb, m->is_w, m->nparams);
    if (cudaDeviceSynchronize() != cudaSuccess) return O2PIC_E_CUDA;
    m->t = 0;
    cudaMemset(m->Mo, 0, sizeof(float) * m->nparams);
    cudaMemset(m->Ve, 0, sizeof(float) * m->nparams);
    return cudaGetLastError() == cudaSuccess ? O2PIC_OK : O2PIC_E_CUDA;
}

int o2pic_mlp_get_params(o2pic_mlp* m, float* host) {
    if (!m || !host) return O2PIC_E_INVALID_ARG;
    if (cudaSetDevice(m->device) != cudaSuccess) return O2PIC_E_CUDA;
    return cudaMemcpy(host, m->P, sizeof(float) * m->nparams, cudaMemcpyDeviceToHost) == cudaSuccess ? O2PIC_OK
                                                                                                   : O2PIC_E_CUDA;
}

int o2pic_mlp_forward(o2pic_mlp* m, const float* X, float* Y, int32_t B, void* stream) {
    if (!m || B < 0 || (B > 0 && (!X || !Y))) return O2PIC_E_INVALID_ARG;
    if (B == 0) return O2PIC_OK;
    if (cudaSetDevice(m->device) != cudaSuccess) return O2PIC_E_CUDA;
    if (int rc = ensure_acts(m, B)) return rc;
    forward(m, X, Y, B, (cudaStream_t)stream);
    return cudaGetLastError() == cudaSuccess ? O2PIC_OK : O2PIC_E_CUDA;
}

int o2pic_mlp_gradients(o2pic_mlp* m, const float* X, const float* T, int32_t B, float* grad, float* loss,
                        void* stream) {
    if (!m || B < 1 || !X || !T || !loss) return O2PIC_E_INVALID_ARG;
    if (cudaSetDevice(m->device) != cudaSuccess) return O2PIC_E_CUDA;
    if (int rc = ensure_acts(m, B)) return rc;
    if (int rc = ensure_grads(m, B)) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    forward(m, X, m->Y, B, s);
    backward(m, X, T, B, loss, grad ? grad : m->G, nullptr, s);
    return cudaGetLastError() == cudaSuccess ? O2PIC_OK : O2PIC_E_CUDA;
}

int o2pic_mlp_train_step(o2pic_mlp* m, const float* X, const float* T, int32_t B, float lr, float* loss,
                         void* stream) {
    if (!m || B < 1 || !X || !T || !loss || !(lr >= 0.0f)) return O2PIC_E_INVALID_ARG;
    if (cudaSetDevice(m->device) != cudaSuccess) return O2PIC_E_CUDA;
    if (int rc = ensure_acts(m, B)) return rc;
    if (int rc = ensure_grads(m, B)) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    const unsigned long long t = m->t + 1;
    const Adam ad = {m->P, m->Mo, m->Ve, m->Wb, lr, 0.9f, 0.999f, 1e-8f, (float)(1.0 - std::pow(0.9, (double)t)),
                     (float)(1.0 - std::pow(0.999, (double)t))};
    forward(m, X, m->Y, B, s);
    backward(m, X, T, B, loss, nullptr, &ad, s);
    if (cudaGetLastError() != cudaSuccess) return O2PIC_E_CUDA;
    m->t = t;
    return O2PIC_OK;
}

void o2pic_mlp_destroy(o2pic_mlp* m) {
    if (!m) return;
    cudaSetDevice(m->device);
    cudaDeviceSynchronize();
    free_acts(m);
    free_grads(m);
    for (void* p : {(void*)m->P, (void*)m->G, (void*)m->Mo, (void*)m->Ve, (void*)m->Wb, (void*)m->is_w,
                    (void*)m->partial})
        if (p) cudaFree(p);
    delete m;
}

}  // extern "C"
