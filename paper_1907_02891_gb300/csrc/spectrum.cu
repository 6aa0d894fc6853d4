// PSF spectrum (step S0): K^ = DFT of the zero-padded PSF, Sec. 2.3 Eq. (10),
// computed once per (PSF, padded size) in FP64 and stored in FP32 in the
// column-major layout the column pass reads.
//
// The PSF is placed with its centre pixel at index (0,0) of the Ny x Nx
// padded grid (negative offsets wrap to the far end).  With that placement
// the circular convolution of Sec. 2.5 needs no crop offset for the
// same-size output, and the spectrum of a point-symmetric PSF is real.
//
// Pipeline (all on the caller's stream, FP64; the card's FP64 rate, two
// multiply-adds per SM and clock, is what bounds it, so every step is there
// to spend fewer of them):
//   * two real rows of K share one complex row transform; of a
//     point-symmetric K only the rows y >= 0 are transformed (row -y is the
//     conjugate of row y);
//   * the columns of a point-symmetric K have real transforms, so two of
//     them share one complex transform;
//   * of a K that is mirror-symmetric too (a radial PSF), every transform is
//     even, so only the residues m <= R / 2 below are transformed and their
//     mirror images stored with them;
//   * a transform of length N = R M of k < N non-zero samples is, per residue
//     m < R, the M-point transform of the samples times exp(-i 2 pi n m / N)
//     folded modulo M: X[m + R k'] = sum_j w_M^{j k'} sum_{n = j mod M} x[n]
//     w_N^{n m}.  R is chosen so that the folding and the M-point transform
//     cost least (fft64_split); one block per (transform, m), in place in
//     shared memory;
//   * twiddles come from a table of N values made once per build; sincospi
//     per element and stage had taken most of the build's time.
// For the 541 x 541 PSF at 4704 x 4704 (radial) the transforms took 4.3 ms as
// one global-memory pass per radix with sincospi twiddles, and take 0.32 ms
// (columns 254 us, 0.68 of the FP64 rate; rows 36, transposition 28 us); the
// fingerprint took 190 us with an atomic per PSF value, and takes 6.
#include "fft_core.cuh"
#include "lp_internal.h"

namespace lpk {

constexpr int kMaxStages64 = 16;
constexpr int kMaxM64 = 4608;  // points of one in-place transform: 72 KB, three blocks per SM

// An M-point transform in shared memory: radices in stage order
struct Fft64 {
    int N, R, M, ns;
    int radix[kMaxStages64];
};

static int pick_radix64(int rem)
{
    for (int r : {8, 4, 2, 3, 5, 7})
        if (rem % r == 0) return r;
    return 0;
}

static int fft64_stages(int n, int* radix)
{
    int ns = 0;
    while (n > 1) {
        const int r = pick_radix64(n);
        if (r == 0 || ns == kMaxStages64) return -1;
        if (radix) radix[ns] = r;
        ++ns;
        n /= r;
    }
    return ns;
}

bool fft64_supported(int N) { return N >= 1 && fft64_stages(N, nullptr) >= 0; }

// Split N = R M for k non-zero samples: the fewest FP64 instructions per
// output (butterflies and twiddles by prime factor, four per folded sample),
// with M points (16 bytes each) in at most 72 KB of shared memory, and enough
// of them to fill a block.
static Fft64 fft64_split(int N, int k)
{
    Fft64 best{};
    double best_cost = 0.0;
    for (int R = 1; R <= N; ++R) {
        if (N % R != 0 || N / R > kMaxM64 || (N / R < 192 && R > 1)) continue;
        Fft64 f{N, R, N / R, 0, {}};
        f.ns = fft64_stages(f.M, f.radix);
        if (f.ns < 0) continue;
        double cost = 4.0 * (double)k / f.M;
        for (int s = 0; s < f.ns; ++s) {
            const int r = f.radix[s];
            cost += 4.0 * (r - 1) / r + (r == 8 ? 6.5 : r == 4 ? 4.0 : r == 2 ? 2.0 : r == 3 ? 4.7 : r == 5 ? 7.2 : 9.4);
        }
        if (best.N == 0 || cost < best_cost) {
            best = f;
            best_cost = cost;
        }
    }
    return best;
}

// table[t] = exp(-i 2 pi t / N), t < N, and perm[p] = the frequency k' that
// the in-place stages leave at position p of M
__global__ void fft64_tables(Fft64 f, double2* table, unsigned short* perm)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < f.N) {
        double s, c;
        sincospi(2.0 * (double)t / (double)f.N, &s, &c);
        table[t] = mk<double2>(c, -s);
    }
    if (t < f.M) {
        int L = f.M, p = t, k = 0, w = 1;
        for (int s = 0; s < f.ns; ++s) {
            L /= f.radix[s];
            const int d = p / L;
            p -= d * L;
            k += d * w;
            w *= f.radix[s];
        }
        perm[t] = (unsigned short)k;
    }
}

// one decimation-in-frequency stage on blocks of length L: outputs m of
// butterfly j to sub-block m, times w_L^{j m} = table[j m N / L]
template <int R>
__device__ __forceinline__ void stage64(double2* sm, int M, int L, int N, const double2* __restrict__ table)
{
    const int S = L / R, step = N / L;
    for (int b = threadIdx.x; b < M / R; b += blockDim.x) {
        const int g = b / S, j = b - g * S;
        double2* x = sm + g * L + j;
        double2 v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = x[q * S];
        Dft<R, -1, double2>::run(v);
        x[0] = v[0];
#pragma unroll
        for (int m = 1; m < R; ++m) x[m * S] = S > 1 ? cmul(v[m], __ldg(table + j * m * step)) : v[m];
    }
    __syncthreads();
}

__device__ __forceinline__ void fft64_inplace(double2* sm, const Fft64& f, const double2* __restrict__ table)
{
    int L = f.M;
    for (int s = 0; s < f.ns; ++s) {
        switch (f.radix[s]) {
        case 2: stage64<2>(sm, f.M, L, f.N, table); break;
        case 3: stage64<3>(sm, f.M, L, f.N, table); break;
        case 4: stage64<4>(sm, f.M, L, f.N, table); break;
        case 5: stage64<5>(sm, f.M, L, f.N, table); break;
        case 7: stage64<7>(sm, f.M, L, f.N, table); break;
        default: stage64<8>(sm, f.M, L, f.N, table); break;
        }
        L /= f.radix[s];
    }
}

// bin j of the folded input: samples i of the window (position i - c) with
// i - c = j mod M, times w_N^{(i - c) m}
template <class Sample>
__device__ __forceinline__ double2 fold64(const Fft64& f, const double2* __restrict__ table, int j, int m, int k, int c,
                                          Sample&& sample)
{
    double2 acc = mk<double2>(0.0, 0.0);
    for (int i = (j + c) % f.M; i < k; i += f.M) {
        const double2 x = sample(i);
        const int n = i - c < 0 ? i - c + f.N : i - c;
        const double2 w = __ldg(table + (int)((long long)n * m % f.N));
        acc.x = fma(x.x, w.x, fma(-x.y, w.y, acc.x));
        acc.y = fma(x.x, w.y, fma(x.y, w.x, acc.y));
    }
    return acc;
}

extern __shared__ __align__(16) double2 sm64[];

// Row pair p (rows y0 + 2p, y0 + 2p + 1 of K packed as a + i b), residue m
// = blockIdx.x: frequencies m + R k' to W[p][.]; mirror: the rows are even,
// and so are their transforms (grid: residues 0 .. R / 2).
__global__ void __launch_bounds__(256) psf_rows(const double* __restrict__ K, int hk, int wk, int y0, int mirror, Fft64 f,
                                                const double2* __restrict__ table, const unsigned short* __restrict__ perm,
                                                double2* __restrict__ W)
{
    const int m = blockIdx.x, p = blockIdx.y;
    const int ya = y0 + 2 * p;
    const double* a = K + (long long)ya * wk;
    const bool vb = ya + 1 < hk;
    for (int j = threadIdx.x; j < f.M; j += blockDim.x)
        sm64[j] = fold64(f, table, j, m, wk, (wk - 1) / 2, [&](int i) { return mk<double2>(a[i], vb ? a[wk + i] : 0.0); });
    __syncthreads();
    fft64_inplace(sm64, f, table);
    double2* dst = W + (long long)p * f.N;
    const bool both = mirror && m != 0 && 2 * m != f.R;
    for (int t = threadIdx.x; t < f.M; t += blockDim.x) {
        const int u = m + f.R * perm[t];
        dst[u] = sm64[t];
        if (both) dst[f.N - u] = sm64[t];
    }
}

// G_y[c] from the packed row transforms: rows a = 2p, b = 2p + 1 of pair p,
// G_a = (Z[c] + conj Z[N-c]) / 2, G_b = -i (Z[c] - conj Z[N-c]) / 2
__device__ __forceinline__ double2 row_spectrum(const double2* __restrict__ W, int Nx, int r, int c)
{
    const double2* row = W + (long long)(r >> 1) * Nx;
    const double2 z = row[c], zm = row[c == 0 ? 0 : Nx - c];
    return (r & 1) ? mk<double2>(0.5 * (z.y + zm.y), -0.5 * (z.x - zm.x)) : mk<double2>(0.5 * (z.x + zm.x), 0.5 * (z.y - zm.y));
}

// position of frequency u in a spectrum column (SpecOrder)
__device__ __forceinline__ int spec_pos(SpecOrder o, int u)
{
    if (o.r0 == 0) return u;
    // (u r < 2^32, so the high half of u ceil(2^32 / r) is u / r)
    const int k = o.r0 > 1 ? (int)__umulhi((unsigned)u, o.inv0) : u, m = u - k * o.r0;
    const int k2 = (int)__umulhi((unsigned)k, o.inv1), k1 = k - k2 * o.r1;
    const int run = o.vk == 4 ? k2 >> 2 : o.vk == 2 ? k2 >> 1 : k2;
    return ((m * (o.vk == 4 ? o.r2 >> 2 : o.vk == 2 ? o.r2 >> 1 : o.r2) + run) * o.r1 + k1) * o.vk + (k2 & (o.vk - 1));
}

// Inputs of the column transforms, transposed: unit u's samples i < hk at
// X[u hk + i].  SYM (point-symmetric K): the unit is columns c = 2u and c + 1
// packed as G_c + i G_{c+1}, W holds the rows y >= 0, and G_{-y} = conj G_y.
// Else the unit is column u, and W holds all rows.
template <bool SYM>
__global__ void __launch_bounds__(256) psf_pack(const double2* __restrict__ W, int hk, int Nx, int ncols, int units,
                                                double2* __restrict__ X)
{
    __shared__ double2 tile[32][33];
    const int u0 = blockIdx.x * 32, i0 = blockIdx.y * 32, cy = (hk - 1) / 2;
    for (int q = threadIdx.y; q < 32; q += 8) {
        const int i = i0 + q, u = u0 + threadIdx.x;
        if (i >= hk || u >= units) continue;
        if constexpr (SYM) {
            const int r = i < cy ? cy - i : i - cy, c = 2 * u;
            double2 g = row_spectrum(W, Nx, r, c);
            double2 h = c + 1 < ncols ? row_spectrum(W, Nx, r, c + 1) : mk<double2>(0.0, 0.0);
            if (i < cy) {
                g.y = -g.y;
                h.y = -h.y;
            }
            tile[q][threadIdx.x] = mk<double2>(g.x - h.y, g.y + h.x);
        } else {
            tile[q][threadIdx.x] = row_spectrum(W, Nx, i, u);
        }
    }
    __syncthreads();
    for (int q = threadIdx.y; q < 32; q += 8) {
        const int u = u0 + q, i = i0 + threadIdx.x;
        if (i < hk && u < units) X[(long long)u * hk + i] = tile[threadIdx.x][q];
    }
}

// Column transforms of unit blockIdx.y, residue m = blockIdx.x.  SYM: the real
// and imaginary parts of the result are the real spectra of columns 2u, 2u + 1
// (mirror: both are even; grid: residues 0 .. R / 2).
template <bool SYM>
__global__ void __launch_bounds__(256) psf_cols(const double2* __restrict__ X, int hk, int ncols, int mirror, Fft64 f,
                                                const double2* __restrict__ table, const unsigned short* __restrict__ perm,
                                                double scale, void* dst, long long ldK, SpecOrder order)
{
    const int m = blockIdx.x, u = blockIdx.y;
    const double2* x = X + (long long)u * hk;
    for (int j = threadIdx.x; j < f.M; j += blockDim.x)
        sm64[j] = fold64(f, table, j, m, hk, (hk - 1) / 2, [&](int i) { return __ldg(x + i); });
    __syncthreads();
    fft64_inplace(sm64, f, table);
    const bool both = SYM && mirror && m != 0 && 2 * m != f.R;
    for (int t = threadIdx.x; t < f.M; t += blockDim.x) {
        const double2 z = sm64[t];
        const int v = m + f.R * perm[t];
        if constexpr (SYM) {
            float* d = static_cast<float*>(dst) + (long long)(2 * u) * ldK;
            for (int side = 0; side <= (both ? 1 : 0); ++side) {
                const int p = spec_pos(order, side ? f.N - v : v);
                d[p] = (float)(z.x * scale);
                if (2 * u + 1 < ncols) d[ldK + p] = (float)(z.y * scale);
            }
        } else {
            static_cast<float2*>(dst)[(long long)u * ldK + spec_pos(order, v)] =
                make_float2((float)(z.x * scale), (float)(z.y * scale));
        }
    }
}

// order-independent 64-bit fingerprint of the PSF values (cache key).  mix64
// is the SplitMix64 output finaliser (Steele, Lea and Flood, "Fast
// splittable pseudorandom number generators", OOPSLA 2014): its published
// shift and multiplier constants, applied to value bits and index.
__device__ __forceinline__ unsigned long long mix64(unsigned long long z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// out[0] += the fingerprint, *asym |= 1 where K is not point-symmetric, |= 2
// where its rows are not mirror-symmetric
__global__ void __launch_bounds__(256) psf_inspect(const double* __restrict__ K, int hk, int wk, unsigned long long* out,
                                                   int* asym)
{
    const long long n = (long long)hk * wk;
    unsigned long long sum = 0;
    int differs = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double v = K[i];
        sum += mix64((unsigned long long)__double_as_longlong(v) ^ mix64((unsigned long long)i));
        const long long y = i / wk;
        if (v != K[n - 1 - i]) differs |= 1;
        if (v != K[(hk - 1 - y) * wk + (i - y * wk)]) differs |= 2;
    }
    differs = __syncthreads_or(differs & 1) ? 1 | (differs & 2) : differs & 2;
    differs = __syncthreads_or(differs & 2) ? 2 | (differs & 1) : differs & 1;
    __shared__ unsigned long long part[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) sum += part[w];
        atomicAdd(out, sum);
        if (differs) atomicOr(asym, differs);
    }
}

cudaError_t psf_inspect_launch(const double* K, int hk, int wk, unsigned long long* d_out, int* d_asym, cudaStream_t st)
{
    const long long blocks = ((long long)hk * wk + 255) / 256;
    psf_inspect<<<(unsigned)(blocks < 304 ? blocks : 304), 256, 0, st>>>(K, hk, wk, d_out, d_asym);
    return cudaGetLastError();
}

__global__ void psf_compare(const double* __restrict__ a, const double* __restrict__ b, long long n,
                            int* diff)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (__double_as_longlong(a[i]) != __double_as_longlong(b[i])) atomicOr(diff, 1);
}

cudaError_t psf_compare_launch(const double* a, const double* b, long long n, int* d_diff, cudaStream_t st)
{
    psf_compare<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, b, n, d_diff);
    return cudaGetLastError();
}

// scratch of a build: the packed row transforms, the column transforms'
// inputs, then the tables
size_t psf_scratch_bytes(int hk, int wk, int Ny, int Nx, int real_only)
{
    const size_t rows = real_only ? (hk + 1) / 2 : hk, ncols = Nx / 2 + 1, units = real_only ? (ncols + 1) / 2 : ncols;
    (void)wk;
    return 16ull * ((rows + 1) / 2 * (size_t)Nx + units * hk + (size_t)Nx + (size_t)Ny) + 2ull * ((size_t)Nx + (size_t)Ny) + 64;
}

// Full spectrum build in `scratch` (16-byte aligned).
cudaError_t psf_spectrum_build(const double* K, int hk, int wk, int Ny, int Nx, int real_only, int mirror, void* dst,
                               long long ldK, SpecOrder order, void* scratch, cudaStream_t st)
{
    const int ncols = Nx / 2 + 1, units = real_only ? (ncols + 1) / 2 : ncols;
    const Fft64 fx = fft64_split(Nx, wk), fy = fft64_split(Ny, hk);
    if (fx.N == 0 || fy.N == 0) return cudaErrorInvalidValue;
    const int rows = real_only ? (hk + 1) / 2 : hk, pairs = (rows + 1) / 2;
    double2* W = static_cast<double2*>(scratch);
    double2* X = W + (size_t)pairs * Nx;
    double2* tx = X + (size_t)units * hk;
    double2* ty = tx + Nx;
    unsigned short* px = reinterpret_cast<unsigned short*>(ty + Ny);
    unsigned short* py = px + Nx;
    const int sx = 16 * fx.M, sy = 16 * fy.M;
    if (sx > 48 * 1024 || sy > 48 * 1024) {  // (one value for all builds: they may run side by side)
        constexpr auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
        cudaError_t e = cudaFuncSetAttribute(psf_rows, attr, 16 * kMaxM64);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(psf_cols<true>, attr, 16 * kMaxM64);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(psf_cols<false>, attr, 16 * kMaxM64);
        if (e != cudaSuccess) return e;
    }
    fft64_tables<<<(Nx + 127) / 128, 128, 0, st>>>(fx, tx, px);
    if (Ny == Nx && fy.R == fx.R) {
        ty = tx;
        py = px;
    } else {
        fft64_tables<<<(Ny + 127) / 128, 128, 0, st>>>(fy, ty, py);
    }
    // (threads: about one radix-8 butterfly each, whole warps)
    const auto threads = [](int M) { return M >= 2048 ? 256 : M >= 512 ? 128 : 64; };
    mirror = mirror && real_only;
    const auto residues = [mirror](int R) { return mirror ? R / 2 + 1 : R; };
    psf_rows<<<dim3(residues(fx.R), pairs), threads(fx.M), sx, st>>>(K, hk, wk, real_only ? (hk - 1) / 2 : 0, mirror, fx,
                                                                    tx, px, W);
    const dim3 gp((units + 31) / 32, (hk + 31) / 32), bp(32, 8), gc(residues(fy.R), units);
    const double scale = 1.0 / (2.0 * (double)Ny * (double)Nx);
    if (real_only) {
        psf_pack<true><<<gp, bp, 0, st>>>(W, hk, Nx, ncols, units, X);
        psf_cols<true><<<gc, threads(fy.M), sy, st>>>(X, hk, ncols, mirror, fy, ty, py, scale, dst, ldK, order);
    } else {
        psf_pack<false><<<gp, bp, 0, st>>>(W, hk, Nx, ncols, units, X);
        psf_cols<false><<<gc, threads(fy.M), sy, st>>>(X, hk, ncols, mirror, fy, ty, py, scale, dst, ldK, order);
    }
    return cudaGetLastError();
}

// One stored column to natural order, by way of shared memory (reading the
// gathered order straight from memory took 52 us at 4704 x 4704, this 28).
// The destination is written as D: whole values, or the floats of complex ones
// where it is not aligned for them.
template <class V, class D>
__global__ void __launch_bounds__(256) spectrum_natural(const V* __restrict__ src, long long ldK, int ny, SpecOrder order,
                                                        D* __restrict__ dst)
{
    extern __shared__ __align__(16) unsigned char smn[];
    constexpr int PER = sizeof(V) / sizeof(D);
    V* col = reinterpret_cast<V*>(smn);
    src += (long long)blockIdx.x * ldK;
    dst += (long long)blockIdx.x * ny * PER;
    // (one element of padding per 32: a step of one in m may be a multiple of
    // 32 positions)
    for (int p = threadIdx.x; p < ny; p += blockDim.x) col[p + (p >> 5)] = src[p];
    __syncthreads();
    const D* val = reinterpret_cast<const D*>(smn);
    for (int i = threadIdx.x; i < ny * PER; i += blockDim.x) {
        const int p = spec_pos(order, i / PER);
        dst[i] = val[(p + (p >> 5)) * PER + i % PER];
    }
}

template <class V, class D>
static cudaError_t natural_launch(const void* data, long long ldK, int ny, int ncols, SpecOrder order, float* dst,
                                  cudaStream_t st)
{
    // (the attribute's value does not depend on the length: copies of
    // different lengths may be launched side by side)
    const cudaError_t e = cudaFuncSetAttribute(spectrum_natural<V, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)(sizeof(V) * 28 * 1024));
    if (e != cudaSuccess) return e;
    spectrum_natural<V, D><<<ncols, 256, sizeof(V) * (size_t)(ny + ny / 32 + 1), st>>>(static_cast<const V*>(data), ldK, ny, order,
                                                                       reinterpret_cast<D*>(dst));
    return cudaGetLastError();
}

cudaError_t spectrum_copy_natural(const void* data, long long ldK, int ny, int ncols, int is_real, SpecOrder order,
                                  float* dst, cudaStream_t st)
{
    if (is_real) return natural_launch<float, float>(data, ldK, ny, ncols, order, dst, st);
    return reinterpret_cast<uintptr_t>(dst) % sizeof(float2) == 0
               ? natural_launch<float2, float2>(data, ldK, ny, ncols, order, dst, st)
               : natural_launch<float2, float>(data, ldK, ny, ncols, order, dst, st);
}

}  // namespace lpk
