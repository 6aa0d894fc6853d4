// Internal interfaces between the C-ABI layer (api.cu) and the kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lpk {

// Per-stage twiddle tables of one Stockham chain: table s (s >= 1) holds
// exp(-i 2 pi k m / (Ns R_s)) at [(m-1) Ns + k], k < Ns, 1 <= m < R_s,
// with Ns = R_0 ... R_{s-1}.
struct TwChain {
    const float2* p[6];
};

// Twiddle tables of one length's block transform N = R0 R1 R2 (N1 = R1 R2):
// w1[m R1P + l] = exp(-i 2 pi l m / (R0 R1)), m < R0, l < R1 (R1P: R1 rounded
// up to even), and w2[m N1 + k R2 + i] = exp(-i 2 pi i (m + R0 k) / N), k < R1,
// i < R2.
struct BlkTw {
    const float2* w1;
    const float2* w2;
};

struct P1Args;
struct P2Args;
struct P3Args;
struct P2MArgs;
struct P2TcArgs;

// One supported FFT length with its compiled FP32 kernels.
struct SizeKernels {
    int N;
    int geo[3];          // R0, R1, R2 of the FP32 passes' block transforms
    int vk;              // consecutive frequencies a spectrum run is read in (Geo::VK)
    int nstages;
    int radices[6];      // forward order of the tensor-core column pass's chain
    int batch;           // several spectra: one forward column transform, parked
    int park_multi;      // the batched pass parks its column in global memory
    int park_class;      // the Eq. (4) pass keeps its sums in global memory
    int park_cols;       // columns side by side in a block's parked set
    cudaError_t (*set_attrs)();
    cudaError_t (*p1)(const P1Args&, cudaStream_t);
    cudaError_t (*p2)(const P2Args&, bool kreal, cudaStream_t);
    cudaError_t (*p2m)(const P2MArgs&, bool kreal, cudaStream_t);
    cudaError_t (*p3)(const P3Args&, int nspec, cudaStream_t);
    // split-precision (BF16 hi/lo) tensor-core column pass, one spectrum per
    // launch; tc_smem = 0 where this length has none
    int tc_threads;
    int tc_smem;
    cudaError_t (*p2tc)(const P2TcArgs&, bool kreal, cudaStream_t);
};

// generated registry (one translation unit per size)
extern const SizeKernels* const kAllSizes[];
extern const int kNumSizes;

// Order of the frequencies within a stored spectrum column: frequency
// u = m + r0 (k1 + r1 k2) at ((m (r2 / vk) + k2 / vk) r1 + k1) vk + k2 mod vk
// (r0 = 0: natural order).
struct SpecOrder {
    int r0, r1, r2, vk;
    unsigned inv0, inv1;  // ceil(2^32 / r0), ceil(2^32 / r1) (r > 1): quotients by multiplication
};

// FP64 spectrum pipeline (spectrum.cu)
bool fft64_supported(int N);
// *d_out += the fingerprint of K's values; *d_asym |= 1 where K is not point-symmetric, |= 2 where its rows are not
// mirror-symmetric
cudaError_t psf_inspect_launch(const double* K, int hk, int wk, unsigned long long* d_out, int* d_asym, cudaStream_t st);
// *d_diff |= 1 where a[i] and b[i] differ in any bit (i < n)
cudaError_t psf_compare_launch(const double* a, const double* b, long long n, int* d_diff, cudaStream_t st);
size_t psf_scratch_bytes(int hk, int wk, int Ny, int Nx, int real_only);
cudaError_t psf_spectrum_build(const double* K, int hk, int wk, int Ny, int Nx, int real_only, int mirror, void* dst,
                               long long ldK, SpecOrder order, void* scratch, cudaStream_t st);
// a stored spectrum's columns in natural order, packed (ny values each)
cudaError_t spectrum_copy_natural(const void* data, long long ldK, int ny, int ncols, int is_real, SpecOrder order,
                                  float* dst, cudaStream_t st);

}  // namespace lpk
