// Launch interface of the BF16 tensor-core GEMM (no_gemm.cu) used by the neural operator.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

namespace cmlbm {

// Raises the kernel's limit of dynamic shared memory to `bytes` on the current device, once per device
// (`done`: a bit for each where it is raised).  A failure is not kept: the next call tries again.
inline cudaError_t opt_in_smem(const void* kernel, int bytes, std::atomic<uint64_t>& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? 1ull << dev : 0;
    if (done.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

// C[b] (+)= alpha * A[b] x B[b].  Element (m, k) of A[b] is A[b * sab + m * sam + k * sak], likewise
// B (k, n) and C (m, n).  A and B are BF16; C is FP32, or BF16 when out_bf16 is set.  beta != 0
// adds to the existing C.  err: device flag set to 1 if an mbarrier wait timed out.  After a
// timeout the block that gave up has freed its tensor memory and returned while MMAs it had
// committed may still be running: C and every buffer downstream of it are undefined, and the
// owner (the neural operator) must be destroyed rather than used again.
struct GemmArgs {
    int M, N, K;
    const __nv_bfloat16* A;
    long long sam, sak, sab;
    const __nv_bfloat16* B;
    long long sbk, sbn, sbb;
    void* C;
    long long scm, scn, scb;
    int out_bf16;
    float alpha;
    int beta;
    unsigned int* err;
    // set by launch_gemm_bf16 from the strides and alignment: staging mode of A and B in the
    // register-staged kernel (0 element by element, 1 K-contiguous 16-byte rows, 2 row-contiguous
    // 8 x 8 blocks); C stored as 16-byte vectors (1 FP32, 2 BF16) or element by element (0)
    int a_mode, b_mode, c_vec;
    // split-K into partial products (copy-engine path only): item b's K range is cut into ksplit
    // slices of kchunk elements (a multiple of 64; the last slice shorter), slice j of item b
    // written to C item b * ksplit + j.  ksplit = 1: the plain product.
    int ksplit = 1;
    int kchunk = 0;
};

cudaError_t launch_gemm_bf16(const GemmArgs& g, int batch, cudaStream_t st);

// The 1x1 map of a hidden layer of width 32 with what follows it, in one pass over the activations:
//   z[b][o][s] += sum_c Wc[o][c] h[b][c][s];   v = act(z + bias[o]);   hb[b][o][s] = bf16(v)
// and the sums of v per row: part[(b 32 + o) map_parts(S) + k], the row's parts in FP64.  h, Wc and hb BF16,
// act = GELU.  cudaErrorNotSupported where the kernel does not apply (S no multiple of 128, alignment).
constexpr int MAP_W = 32;
inline int map_parts(long long S) { return (int)((S + 8191) / 8192) * 32; }
cudaError_t launch_map_act(const __nv_bfloat16* h, const __nv_bfloat16* Wc, const float* bias, int B, long long S, float* z,
                           __nv_bfloat16* hb, double* part, unsigned int* err, cudaStream_t st);

}  // namespace cmlbm
