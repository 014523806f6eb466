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

// Adam (Kingma & Ba 2015) on the fp32 master parameter i with gradient g, then
// the bf16 copy if it is a weight.
struct Adam {
    float *P, *Mo, *Ve;
    __nv_bfloat16* Wb;
    float lr, b1, b2, eps, c1, c2;
    __device__ __forceinline__ void step(size_t i, float g, bool weight) const {
        const float m = fmaf(b1, Mo[i], (1.0f - b1) * g);
        const float v = fmaf(b2, Ve[i], (1.0f - b2) * g * g);
        Mo[i] = m;
        Ve[i] = v;
        const float p = P[i] - lr * (m / c1) / (sqrtf(v / c2) + eps);
        P[i] = p;
        if (weight) Wb[i] = __float2bfloat16_rn(p);
    }
};

// One output tile (TM x TN at m0, n0) of C[m][n] = epi( sum_k A(m,k) B(k,n) +
// bias[n] ), summed over k in order by one chain of FMAs per output.
// A(m,k) = TA ? A[k lda + m] : A[m lda + k];  B(k,n) = TB ? B[n ldb + k] : B[k ldb + n].
// Each of the (TM/RM)(TN/RN) threads owns RM x RN neighbouring outputs; k-slices
// of KS go through shared memory in two stages, the next slice's global loads
// in flight while this one is summed.
template <int TM, int TN, int RM, int RN, int KS>
struct Tile {
    static constexpr int TX = TN / RN, NT = (TM / RM) * TX, LA = TM + 4, LB = TN + 4;
    static constexpr int PA = TM * KS / NT, PB = TN * KS / NT;
    static_assert(TM * KS % NT == 0 && TN * KS % NT == 0, "whole loads per thread");
    struct Shared {
        __align__(16) float A[2][KS][LA];
        __align__(16) float B[2][KS][LB];
    };

    template <int R>
    static __device__ __forceinline__ void fragment(float (&r)[R], const float* p) {
        if constexpr (R == 4) {
            const float4 v = *reinterpret_cast<const float4*>(p);
            r[0] = v.x; r[1] = v.y; r[2] = v.z; r[3] = v.w;
        } else {
#pragma unroll
            for (int i = 0; i < R; ++i) r[i] = p[i];
        }
    }

    template <bool TA, bool TB, typename BT, typename Store>
    static __device__ __forceinline__ void run(Shared& sh, const float* __restrict__ A, int lda,
                                               const BT* __restrict__ B, int ldb, int M, int N, int K, int m0, int n0,
                                               Store&& store) {
        const int t = threadIdx.x, tx = t % TX, ty = t / TX;
        float pa[PA], pb[PB];
        auto load = [&](int k0) {
#pragma unroll
            for (int i = 0; i < PA; ++i) {
                const int e = t + i * NT;
                const int mm = TA ? e % TM : e / KS, kk = TA ? e / TM : e % KS;
                const int m = m0 + mm, k = k0 + kk;
                pa[i] = (m < M && k < K) ? (TA ? A[(size_t)k * lda + m] : A[(size_t)m * lda + k]) : 0.0f;
            }
#pragma unroll
            for (int i = 0; i < PB; ++i) {
                const int e = t + i * NT;
                const int nn = TB ? e / KS : e % TN, kk = TB ? e % KS : e / TN;
                const int n = n0 + nn, k = k0 + kk;
                pb[i] = (n < N && k < K) ? (TB ? ldf(&B[(size_t)n * ldb + k]) : ldf(&B[(size_t)k * ldb + n])) : 0.0f;
            }
        };
        auto stage = [&](int s) {
#pragma unroll
            for (int i = 0; i < PA; ++i) {
                const int e = t + i * NT;
                sh.A[s][TA ? e / TM : e % KS][TA ? e % TM : e / KS] = pa[i];
            }
#pragma unroll
            for (int i = 0; i < PB; ++i) {
                const int e = t + i * NT;
                sh.B[s][TB ? e % KS : e / TN][TB ? e / KS : e % TN] = pb[i];
            }
        };
        float acc[RM][RN];
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
            for (int j = 0; j < RN; ++j) acc[i][j] = 0.0f;
        load(0);
        stage(0);
        __syncthreads();
        int s = 0;
        for (int k0 = 0; k0 < K; k0 += KS, s ^= 1) {
            const bool more = k0 + KS < K;
            if (more) load(k0 + KS);
#pragma unroll 16
            for (int kk = 0; kk < KS; ++kk) {
                float a[RM], b[RN];
                fragment<RM>(a, &sh.A[s][kk][ty * RM]);
                fragment<RN>(b, &sh.B[s][kk][tx * RN]);
#pragma unroll
                for (int i = 0; i < RM; ++i)
#pragma unroll
                    for (int j = 0; j < RN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
            }
            if (more) {
                stage(s ^ 1);   // last read in the slice before this one
                __syncthreads();
            }
        }
#pragma unroll
        for (int i = 0; i < RM; ++i) {
            const int m = m0 + ty * RM + i;
#pragma unroll
            for (int j = 0; j < RN; ++j) {
                const int n = n0 + tx * RN + j;
                if (m < M && n < N) store(m, n, acc[i][j]);
            }
        }
    }
};

// The forward contractions and the gradients at the pre-activations take the
// large tile when it gives every SM a block, else the small one (Small: a few
// rows, 64 threads, so that even 32 x 256 outputs spread over 32 SMs).
using Large = Tile<64, 64, 4, 4, 16>;
using Small = Tile<8, 32, 1, 4, 64>;
// Weight gradients (outputs in x out, sums over the batch rows).
using Grad = Tile<64, 32, 4, 4, 16>;

// EPI_TANH: tanh of the sum; EPI_DTANH: the sum times (1 - H[m][n]^2).
template <class T, bool TB>
__global__ void __launch_bounds__(T::NT) k_gemm(const float* __restrict__ A, int lda,
                                                const __nv_bfloat16* __restrict__ B, int ldb, float* __restrict__ C,
                                                int M, int N, int K, const float* __restrict__ bias, int epi,
                                                const float* __restrict__ H) {
    __shared__ typename T::Shared sh;
    pdl_wait();
    pdl_trigger();
    const int m0 = blockIdx.y * (T::LA - 4), n0 = blockIdx.x * (T::LB - 4);
    T::template run<false, TB>(sh, A, lda, B, ldb, M, N, K, m0, n0, [&](int m, int n, float v) {
        if (bias) v += bias[n];
        if (epi == EPI_TANH) v = tanhf(v);
        else if (epi == EPI_DTANH) { const float h = H[(size_t)m * N + n]; v = v * (1.0f - h * h); }
        C[(size_t)m * N + n] = v;
    });
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
        const size_t off = J.offW[l];
        Grad::run<true, false>(sh, J.H[l], K, J.dZ[l], N, K, N, B, (r / tiles_n) * 64, (r % tiles_n) * 32,
                               [&](int m, int n, float v) {
                                   const size_t i = off + (size_t)m * N + n;
                                   if (UPDATE) ad.step(i, v, true);
                                   else J.G[i] = v;
                               });
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
        if (UPDATE) ad.step(J.offB[l] + n, s, false);
        else J.G[J.offB[l] + n] = s;
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
// [N][K]: TB).  The large tile from one block per SM on: 2000 x 256 outputs
// (128 blocks) 8x faster than the former 64 x 64 kernel without prefetch, 81 x
// 256 (44 small blocks) 10x.
template <bool TB>
void gemm(const float* A, int lda, const __nv_bfloat16* B, int ldb, float* C, int M, int N, int K, const float* bias,
          int epi, const float* H, int sms, cudaStream_t s) {
    const long long large = (long long)((N + 63) / 64) * ((M + 63) / 64);
    if (4 * large >= 3 * sms) {
        const dim3 grid((N + 63) / 64, (M + 63) / 64);
        launch_pdl(k_gemm<Large, TB>, grid, Large::NT, 0, s, A, lda, B, ldb, C, M, N, K, bias, epi, H);
    } else {
        const dim3 grid((N + 31) / 32, (M + 7) / 8);
        launch_pdl(k_gemm<Small, TB>, grid, Small::NT, 0, s, A, lda, B, ldb, C, M, N, K, bias, epi, H);
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
    // for a batch of up to cap rows: activations H[l] (l = 1..L-1), output Y,
    // gradients at the pre-activations dZ[l] (l = 1..L)
    int cap = 0;
    std::vector<float*> H, dZ;
    float *Y = nullptr, *partial = nullptr;
    int sms = 0;
    unsigned long long t = 0;              // Adam steps taken
};

namespace {

constexpr int MSE_BLOCKS = 120;

int layers(const o2pic_mlp* m) { return (int)m->w.size() - 1; }

void free_acts(o2pic_mlp* m) {
    for (float* h : m->H) if (h) cudaFree(h);
    for (float* d : m->dZ) if (d) cudaFree(d);
    m->H.clear();
    m->dZ.clear();
    if (m->Y) cudaFree(m->Y);
    m->Y = nullptr;
    m->cap = 0;
}

int ensure_acts(o2pic_mlp* m, int B) {
    if (B <= m->cap) return O2PIC_OK;
    free_acts(m);
    const int L = layers(m);
    m->H.assign(L, nullptr);
    m->dZ.assign(L + 1, nullptr);
    for (int l = 1; l < L; ++l)
        if (cudaMalloc((void**)&m->H[l], sizeof(float) * (size_t)B * m->w[l]) != cudaSuccess) return O2PIC_E_CUDA;
    for (int l = 1; l <= L; ++l)
        if (cudaMalloc((void**)&m->dZ[l], sizeof(float) * (size_t)B * m->w[l]) != cudaSuccess) return O2PIC_E_CUDA;
    if (cudaMalloc((void**)&m->Y, sizeof(float) * (size_t)B * m->w[L]) != cudaSuccess) return O2PIC_E_CUDA;
    m->cap = B;
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
    for (void* p : {(void*)m->P, (void*)m->G, (void*)m->Mo, (void*)m->Ve, (void*)m->Wb, (void*)m->is_w,
                    (void*)m->partial})
        if (p) cudaFree(p);
    delete m;
}

}  // extern "C"
