// Stable compaction of a caller's particle arrays (the removal half of the
// method's births/removal step): particles whose x is NaN (the library's
// marker of a removed particle) are dropped, the others are written in their
// original order to the output arrays (compact_tiles).  The look-back state
// and the tile ticket are the kernel's scratch memory.
#include "compact.cuh"

namespace o2 {

namespace {

__global__ void __launch_bounds__(CMP_T, 2) k_compact_arrays(const float* __restrict__ X, const float* __restrict__ VX,
                                                            const float* __restrict__ VY, const float* __restrict__ VZ,
                                                            const uint32_t* __restrict__ ID, unsigned long long n,
                                                            float* OX, float* OVX, float* OVY, float* OVZ,
                                                            uint32_t* OID, unsigned long long* n_out,
                                                            unsigned long long* ticket, unsigned long long* count,
                                                            unsigned long long* flag, unsigned long long* val,
                                                            unsigned long long epoch, unsigned long long* err) {
    __shared__ CompactShared sh;
    compact_tiles(
        sh, X, n, reinterpret_cast<unsigned*>(ticket), flag, val, epoch, err,
        [&](unsigned long long p) {
            prefetch_l2(VX + p); prefetch_l2(VY + p); prefetch_l2(VZ + p); prefetch_l2(ID + p);
        },
        [&](const float (&x)[CMP_I], unsigned long long base, unsigned long long d, const unsigned (&off)[CMP_I],
            unsigned in) {
#pragma unroll
            for (int i = 0; i < CMP_I; ++i)
                if ((in >> i) & 1u) OX[d + off[i]] = x[i];
            move_array(OVX, VX, base, d, off, in, ~0ull);
            move_array(OVY, VY, base, d, off, in, ~0ull);
            move_array(OVZ, VZ, base, d, off, in, ~0ull);
            move_array(OID, ID, base, d, off, in, ~0ull);
        },
        [&](unsigned long long kept) { *count = kept; *n_out = kept; });
}

// One warp waits, as tile 1 of a look-back, for tile 0, whose flag nothing
// ever sets (epoch 1 against the zeroed flag): the bounded wait must give up,
// set the timeout bit and return.  words = [err, flag[2], val[4]].
__global__ void k_lookback_probe(unsigned long long* words) {
    bool ok;
    (void)lookback(words + 1, words + 3, 1u, 1ull, 1ull, words, &ok);
}

}  // namespace

size_t compact_scratch_words(unsigned long long n) {
    const unsigned long long tiles = ceil_div(n, TILE) + 1;
    return 3 + 3 * tiles;   // ticket, count, error word, flags, values
}

// Scratch laid out in `words` (u64): [ticket, count, err, flag[tiles], val[2 tiles]].
void launch_compact_arrays(const float* x, const float* vx, const float* vy, const float* vz, const uint32_t* id,
                           unsigned long long n, float* ox, float* ovx, float* ovy, float* ovz, uint32_t* oid,
                           unsigned long long* n_out, unsigned long long* words, unsigned long long tiles,
                           unsigned long long epoch, int sms, cudaStream_t s) {
    // two blocks per SM are resident; fewer where there are fewer tiles
    const int grid = (int)(ceil_div(n, TILE) < 2ull * sms ? ceil_div(n, TILE) : 2ull * sms);
    k_compact_arrays<<<grid, CMP_T, 0, s>>>(x, vx, vy, vz, id, n, ox, ovx, ovy, ovz, oid, n_out, &words[0], &words[1],
                                            &words[3], &words[3 + tiles], epoch, &words[2]);
}

}  // namespace o2

using namespace o2;

extern "C" int o2pic_check_bounded_wait(double* seconds, void* stream) {
    cudaStream_t s = (cudaStream_t)stream;
    unsigned long long* w = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaMalloc((void**)&w, 7 * sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMemsetAsync(w, 0, 7 * sizeof(unsigned long long), s);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e == cudaSuccess) e = cudaEventRecord(e0, s);
    if (e == cudaSuccess) {
        k_lookback_probe<<<1, 32, 0, s>>>(w);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaEventRecord(e1, s);
    unsigned long long err = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&err, w, sizeof(err), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (seconds) *seconds = 1e-3 * ms;
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (w) cudaFree(w);
    if (e != cudaSuccess) return O2PIC_E_CUDA;
    return (err & ERR_TIMEOUT) ? O2PIC_E_TIMEOUT : O2PIC_OK;
}

extern "C" int o2pic_compact_particles(const float* x, const float* vx, const float* vy, const float* vz,
                                       const uint32_t* id, uint64_t n, float* ox, float* ovx, float* ovy, float* ovz,
                                       uint32_t* oid, uint64_t* n_out, void* stream) {
    if (!n_out || (n > 0 && (!x || !vx || !vy || !vz || !id || !ox || !ovx || !ovy || !ovz || !oid)))
        return O2PIC_E_INVALID_ARG;
    if (n > (1ull << 31)) return O2PIC_E_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const unsigned long long tiles = ceil_div(n, TILE) + 1;
    const size_t words = compact_scratch_words(n);
    unsigned long long* scratch = nullptr;
    cudaError_t e = cudaMalloc((void**)&scratch, sizeof(unsigned long long) * words);
    if (e != cudaSuccess) return O2PIC_E_CUDA;
    e = cudaMemsetAsync(scratch, 0, sizeof(unsigned long long) * words, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(n_out, 0, sizeof(uint64_t), s);
    int dev = 0, sms = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && n > 0) {
        launch_compact_arrays(x, vx, vy, vz, id, n, ox, ovx, ovy, ovz, oid, (unsigned long long*)n_out, scratch, tiles,
                              1ull, sms, s);
        e = cudaGetLastError();
    }
    unsigned long long err = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&err, &scratch[2], sizeof(err), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(scratch);
    if (e != cudaSuccess) return O2PIC_E_CUDA;
    return (err & ERR_TIMEOUT) ? O2PIC_E_TIMEOUT : O2PIC_OK;
}
