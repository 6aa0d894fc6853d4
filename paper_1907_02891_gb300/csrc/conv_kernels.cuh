// The three FP32 passes of the Fourier-domain convolution (Sec. 2.3 Eq. (9),
// workflow of Sec. 2.5 / Fig. 1): zero padding is implicit, the spectrum
// product sits between the forward and inverse column transforms, and the
// crop is a predicate on the last stores.
//
//   P1  rows:    two real rows a, b packed as z = a + i b, length-Nx forward
//                FFT, split into the half spectra of a and b (Hermitian
//                symmetry), stored by column c in [0, Nx/2] (column-blocked
//                layout, below).
//   P2  columns: per column c, length-Ny forward FFT of T[c][0..H) (rows
//                >= H are the zero padding), multiply by the PSF spectrum
//                K^[c][.] (pre-scaled by 1/(2 Ny Nx)), inverse FFT, keep the
//                output rows of the crop window.  With n spectra the batched
//                kernel parks the forward result in shared memory and reuses
//                it n times; plans may instead run one pass per spectrum.
//   P3  rows:    Hermitian extension of two rows' half spectra packed as
//                Z = A + i B, length-Nx inverse FFT, real part -> row a,
//                imaginary part -> row b, keep the crop columns.
//
// Layouts (element = complex64 unless stated):
//   L    FP32, row-major H x W, leading dimension ldl (elements)
//   T    the row pass's half spectra, column-blocked (below): ldT >= 2 ceil(H/2)
//        elements per column, Nx/2+1 columns rounded up to a multiple of kTCB
//   K^   (Nx/2+1) rows of ldK elements: FP32 (point-symmetric PSF, real
//        spectrum) or complex64
//   U    per spectrum, column-blocked (below): ldU >= 2 ceil(Hout/2) elements per
//        column, Nx/2+1 columns rounded up to a multiple of kUCB
//   out  FP32 row-major Hout x Wout, leading dimension ldo
#pragma once

#include "fft_core.cuh"

namespace lpk {

// Column-blocked layout of the intermediate half spectra T and U.  Element
// (column c, row pair p) is a float4 {row 2p, row 2p+1} of column c; the
// columns are grouped in blocks of CB, and within a block the CB columns'
// float4 of one row pair sit side by side:
//   float4 index ((c / CB) * ldq + p) * CB + c mod CB,  ldq = ld / 2,
// with ld the (even) number of rows stored per column.  The row passes,
// which handle all columns of one row pair, then move 16 CB contiguous
// bytes per column block instead of 16 scattered ones; the column pass
// reads / writes a column at a 16 CB-byte stride.  Measured at 4704^2 with
// blocks of 1 / 2 / 4 / 8 for T: row pass 73 / 43.4 / 40.0 / 37.0 us; column
// pass, T and U alike, 51.6 / 55.0 / 67.1 / 86.0 us.  The CB-1 columns past the last one that
// padding adds to a partial last block are allocated and never touched.
template <int CB>
__host__ __device__ constexpr long long blk_cols_alloc(long long ncols) { return (ncols + CB - 1) / CB * CB; }
template <int CB>
__host__ __device__ __forceinline__ long long blk_index4(int c, long long p, long long ldq)
{
    return ((long long)(c / CB) * ldq + p) * CB + (c % CB);
}
// row r of a column, in float2 from the column's row 0
template <int CB>
__host__ __device__ __forceinline__ long long blk_row(int r) { return (long long)(r >> 1) * (2 * CB) + (r & 1); }

constexpr int kTCB = 2;  // T: written by the forward row pass, read by the column pass
// U: written by the column pass, read by the inverse row pass.  Measured at
// 4704^2, blocks of 1 / 2 / 4 / 8 (T in blocks of 2 for 2 and 4): inverse row
// pass 56.2 / 45.9 / 39.6 / 37.3 us, column pass 51.6 / 55.0 / 59.7 / 86.0 us.
constexpr int kUCB = 4;
__host__ __device__ constexpr long long t_cols_alloc(long long ncols) { return blk_cols_alloc<kTCB>(ncols); }
__host__ __device__ constexpr long long u_cols_alloc(long long ncols) { return blk_cols_alloc<kUCB>(ncols); }
__host__ __device__ __forceinline__ long long t_index4(int c, long long p, long long ldq) { return blk_index4<kTCB>(c, p, ldq); }
__host__ __device__ __forceinline__ long long u_index4(int c, long long p, long long ldq) { return blk_index4<kUCB>(c, p, ldq); }
__host__ __device__ __forceinline__ long long t_row(int r) { return blk_row<kTCB>(r); }
// offset of row j + m S from row j's when S is even (the pair index moves by
// m S / 2, the row parity stays): a compile-time multiple of m
template <int S>
__host__ __device__ constexpr long long t_row_step() { return (long long)(S / 2) * 2 * kTCB; }
__host__ __device__ __forceinline__ long long u_row(int r) { return blk_row<kUCB>(r); }
// float2 pointer to row 0 of column c
__host__ __device__ __forceinline__ const float2* t_column(const float2* T, long long ldT, int c)
{
    return T + 2 * t_index4(c, 0, ldT / 2);
}
__host__ __device__ __forceinline__ float2* u_column(float2* U, long long ldU, int c)
{
    return U + 2 * u_index4(c, 0, ldU / 2);
}

constexpr int kMaxSpectraPerLaunch = 32;

struct P1Args {
    const float* L[kMaxSpectraPerLaunch];  // map i of the launch, into T + i specT
    int nmaps;
    long long ldl;
    int H, W;
    float2* T;
    long long ldT;
    long long specT;
    int pair0;   // first row pair of this launch (pairs pair0 .. npairs-1)
    int npairs;  // ceil(H/2)
    int ncols;   // Nx/2 + 1
    BlkTw tw;    // of the row length
    int* err;            // device status word (debug builds: bounds checks)
    long long t_elems;   // float2 elements of the T buffer (of one map)
};

struct P2Args {
    const float2* T;
    long long ldT;
    int H;
    const void* K[kMaxSpectraPerLaunch];
    long long ldK;
    int nspec;
    float2* U;
    long long ldU;
    long long specU;  // elements between consecutive spectra's U blocks
    int r0;           // first kept row (mod Ny) of the inverse output
    int Hout;         // kept rows
    int HoutPad;      // 2 ceil(Hout/2): rows written (the extra one is zero)
    int ncols;
    BlkTw tw;          // of the column length
    float2* park;      // batched pass: forward column spectra, N per column
    int* err;              // device status word (debug builds: bounds checks)
    long long t_elems;     // float2 elements of the T buffer
    long long u_elems;     // float2 elements of U from a.U on (all spectra of the launch)
    long long k_elems;     // spectrum values (floats or float2) of each spectrum
    long long park_elems;  // float2 elements of the park area (0 without one)
};

struct P3Args {
    const float2* U;
    long long ldU;
    long long specU;
    int Hout, npairs;
    int pair0;  // first output row pair of this launch
    float* out[kMaxSpectraPerLaunch];
    long long ldo;
    int c0;  // first kept column (mod Nx)
    int Wout;
    int ncols;
    BlkTw tw;  // of the row length
    int* err;           // device status word (debug builds: bounds checks)
    long long u_elems;  // float2 elements of U from a.U on (all spectra of the launch)
};

// Debug builds (LP_DEBUG=1, a library of their own): before a work unit
// touches global memory, its block checks the unit's whole extent in every
// buffer against the sizes the host passed; a unit outside them sets bit 3
// of the device status word and is skipped (no assert or trap, so the
// context stays usable).  Release builds compile the checks away.
#ifndef LP_DEBUG
#define LP_DEBUG 0
#endif
constexpr int kDevErrBounds = 8;

__device__ __forceinline__ bool lp_checked(int* err, bool ok)
{
#if LP_DEBUG
    if (!ok && threadIdx.x == 0) atomicOr(err, kDevErrBounds);
    return ok;
#else
    (void)err;
    (void)ok;
    return true;
#endif
}

// P1 unit: rows 2 pair, 2 pair + 1 of L, and row pair `pair` of every column of T
__device__ __forceinline__ bool p1_unit_ok(const P1Args& a, int pair)
{
#if LP_DEBUG
    const long long ldq = a.ldT / 2;
    return lp_checked(a.err, pair >= 0 && 2 * pair < a.H && pair < ldq && a.W <= a.ldl &&
                                 2 * (t_index4(a.ncols - 1, pair, ldq) + 1) <= a.t_elems);
#else
    (void)a;
    (void)pair;
    return true;
#endif
}

// P2 unit: column c of T (all ldT rows), of each spectrum, of each of the
// launch's U blocks (HoutPad rows), and the park area up to column park_end
// (a block's columns are parked interleaved, those past the last one too)
__device__ __forceinline__ bool p2_column_ok(const P2Args& a, int c, int n, int kw, int park_end)
{
#if LP_DEBUG
    const bool t_ok = 2 * t_index4(c, 0, a.ldT / 2) + t_row((int)a.ldT - 1) < a.t_elems && a.H <= a.ldT;
    const bool k_ok = (long long)(c + 1) * a.ldK <= a.k_elems && n <= a.ldK;
    const bool u_ok = a.HoutPad <= a.ldU &&
                      (long long)(a.nspec - 1) * a.specU + 2 * u_index4(c, 0, a.ldU / 2) + u_row(a.HoutPad - 1) <
                          a.u_elems;
    const bool p_ok = a.park == nullptr || (long long)park_end * n <= a.park_elems;
    (void)kw;
    return lp_checked(a.err, c >= 0 && c < a.ncols && t_ok && k_ok && u_ok && p_ok);
#else
    (void)a;
    (void)c;
    (void)n;
    (void)kw;
    (void)park_end;
    return true;
#endif
}

// P3 unit: row pair `pair` of every column of U block sidx, rows 2 pair,
// 2 pair + 1 of out[sidx]
__device__ __forceinline__ bool p3_unit_ok(const P3Args& a, int pair, int sidx)
{
#if LP_DEBUG
    const long long ldq = a.ldU / 2;
    return lp_checked(a.err, pair >= 0 && 2 * pair < a.Hout && pair < ldq && a.out[sidx] != nullptr &&
                                 a.Wout <= a.ldo &&
                                 (long long)sidx * a.specU + 2 * (u_index4(a.ncols - 1, pair, ldq) + 1) <=
                                     a.u_elems);
#else
    (void)a;
    (void)pair;
    (void)sidx;
    return true;
#endif
}

// Radix order of a length's self-sorting chain (the tensor-core column pass).
template <int N, class FwdSeq>
struct Plan {
    using Fwd = FwdSeq;
    using Inv = Reverse<FwdSeq>;
    static_assert(SeqInfo<Fwd>::product == N, "radices must multiply to N");
    static constexpr int R0 = SeqInfo<Fwd>::first;   // first forward radix
    static constexpr int RL = SeqInfo<Fwd>::last;    // last forward radix
};

// Programmatic dependent launch.  The pass kernels are launched with the
// programmatic-stream-serialization attribute and begin with pdl_begin():
// the wait holds this grid until the previous grid on the stream has
// completed with its memory visible, and the trigger after it lets the next
// kernel on the stream start launching once every block of this grid has got
// so far (its blocks then wait in their own pdl_begin) -- so no pass touches
// its predecessor's results before they are there, everything older is
// complete when a block starts, and the launch latency of each pass overlaps
// the tail of the one before.  Without the attribute (or after a non-kernel
// operation) the wait returns at once.  With LATE the block does not
// trigger, so the next kernel launches only as this grid's blocks exit:
// measured faster for the forward row pass at three resident blocks per SM
// (the next pass's early blocks otherwise share its last wave's SMs), a plan
// knob per pass.
//
// What the previous grid wrote (L, T, U) is read by plain loads or TMA, never
// by __ldg: a non-coherent load may be moved above the wait, its data being
// constant as far as the compiler knows.
template <bool LATE = false>
__device__ __forceinline__ void pdl_begin()
{
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    if constexpr (!LATE) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

template <class... KArgs, class... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}


// ---------------------------------------------------------------------------
// A pass kernel's shape: geometry of the length, NT transforms per block (row
// pairs or columns), TH threads (per group in the batched column pass),
// minimum resident blocks per SM (register cap), late launch trigger.
// ---------------------------------------------------------------------------
template <class Ge_, int NT_, int TH_, int MINB_, bool LATE_>
struct PassCfg {
    using Ge = Ge_;
    using La = Lay<Ge_>;
    static constexpr int NT = NT_, TH = TH_, MINB = MINB_;
    static constexpr bool LATE = LATE_;
    static_assert(TH % 32 == 0 && TH <= 1024, "whole warps");
    static constexpr int WORK = NT * La::ELEMS;          // float2 of one working set
    static constexpr int SMEM = 8 * (Ge::W1 + WORK);     // w1, then the working set
    static constexpr int U1 = Ge::N1 * NT;               // stage-1 butterflies
    static constexpr int E1 = (U1 + TH - 1) / TH;
    static constexpr int GROUPS = TH / 32 * Ge::GPW;     // sub-transforms in flight
    static constexpr int UB = Ge::R0 * NT;               // sub-transforms
    static constexpr int EB = (UB + GROUPS - 1) / GROUPS;
    static constexpr int US = Ge::R0 * Ge::R1 * NT;      // stage-3 runs
    static constexpr int ES = (US + TH - 1) / TH;
};

// shared memory of the FP32 passes (namespace scope, so that functions that
// are not inlined address it as shared memory)
extern __shared__ __align__(16) float2 lp_dsmem[];

// ---------------------------------------------------------------------------
// Row passes.  A transform packs two real rows, z = a + i b, so the half
// spectra of a and b need each frequency k = m + R0 (k1 + R1 k2) together
// with N - k.  That partner lies in sub-transform R0 - m (m = 0: in itself),
// at k1' = R1 - 1 - k1, k2' = R2 - 1 - k2 (m = 0: k1' = (R1 - k1) mod R1, and
// for k1 = 0 the run's own element (R2 - k2) mod R2).  Where a transform is
// one sub-transform (R0 = 1) its lanes exchange the partners by shuffles
// (RowSub), each handing over the upper half of its run; else a sweep through
// shared memory combines them (shuffles between the lanes of m and R0 - m were
// slower at 4704: forward 44 -> 58-65, inverse 41 -> 43-50 us, T and U then
// being accessed in 16-byte pieces of distinct lines).
// ---------------------------------------------------------------------------
// A lane's place in round `round` of the transforms of a block, R0 = 1
template <class C>
struct RowSub {
    using Ge = typename C::Ge;
    static constexpr int G = Ge::G;
    static constexpr int FLIGHT = C::TH / G;  // transforms at a time
    static constexpr int ROUNDS = (C::NT + FLIGHT - 1) / FLIGHT;
    int tr, li, partner;  // transform, lane in the group, partner's lane in the warp
    bool live, origin;    // origin: the run k1 = 0
    __device__ __forceinline__ RowSub(int t, int round)
    {
        tr = t / G + round * FLIGHT;
        li = t % G;
        live = ROUNDS * FLIGHT == C::NT || tr < C::NT;
        origin = li == 0;
        const int lane = t & 31;
        partner = lane - li + (origin || li >= Ge::R1 ? li : Ge::R1 - li);
    }
};

// {2 X_a[c], 2 X_b[c]} of the packed transform's Z[c] and Z[N - c]
__device__ __forceinline__ float4 split_rows(float2 zc, float2 zm)
{
    float4 o;
    o.x = zc.x + zm.x;       // 2 X_a = Z[c] + conj Z[N-c]
    o.y = zc.y - zm.y;
    o.z = zc.y + zm.y;       // 2 X_b = -i (Z[c] - conj Z[N-c])
    o.w = -(zc.x - zm.x);
    return o;
}
// Z[c] and Z[N - c] from the half spectra {A, B} of c
__device__ __forceinline__ float2 join_lo(float4 q) { return make_float2(q.x - q.w, q.y + q.z); }
__device__ __forceinline__ float2 join_hi(float4 q) { return make_float2(q.x + q.w, q.z - q.y); }

// ---------------------------------------------------------------------------
// P1: row R2C of two packed rows per transform, NT transforms per block.
// The maps of several classes are one launch: the last wave of each map's
// blocks (1024 blocks on 304 places at 4704) is filled by the next map's.
// Three classes of 4096^2: 290.3 -> 280.1 us with one launch for three.
// ---------------------------------------------------------------------------
struct RowInput {
    const float *pa, *pb;
    int wa, wb;  // columns to read of each row (0: none)
    __device__ __forceinline__ RowInput(const P1Args& a, int pair)
    {
        const int ra = 2 * pair;
        pa = a.L[blockIdx.y] + (long long)ra * a.ldl;
        pb = pa + a.ldl;
        wa = pair < a.npairs && ra < a.H ? a.W : 0;
        wb = pair < a.npairs && ra + 1 < a.H ? a.W : 0;
    }
    __device__ __forceinline__ float2 operator()(int col) const
    {
        return make_float2(col < wa ? pa[col] : 0.f, col < wb ? pb[col] : 0.f);
    }
};

template <class C>
__global__ void __launch_bounds__(C::TH, C::MINB) p1_rows(const __grid_constant__ P1Args a)
{
    pdl_begin<C::LATE>();
    using Ge = typename C::Ge;
    using La = typename C::La;
    using RS = RowSub<C>;
    constexpr int R0 = Ge::R0, R1 = Ge::R1, R2 = Ge::R2, N1 = Ge::N1, UR = R0 * R1;
    const int pair0 = a.pair0 + blockIdx.x * C::NT;
    for (int tr = 0; tr < C::NT; ++tr)
        if (pair0 + tr < a.npairs && !p1_unit_ok(a, pair0 + tr)) return;  // (whole block: before any barrier)
    const int t = threadIdx.x;
    float2* work = lp_dsmem + Ge::W1;
    if constexpr (R0 > 1) {
        load_w1<Ge>(lp_dsmem, a.tw.w1, t, C::TH);
#pragma unroll 1
        for (int e = 0; e < C::E1; ++e) {
            const int u = t + e * C::TH;
            if (C::E1 * C::TH != C::U1 && u >= C::U1) break;
            const int tr = C::NT == 1 ? 0 : u / N1;
            const int j = u - tr * N1;
            const RowInput in(a, pair0 + tr);
            float2 v[R0];
#pragma unroll
            for (int q = 0; q < R0; ++q) v[q] = in(j + q * N1);
            Dft<R0, -1, float2>::run(v);
            float2* w = work + tr * La::ELEMS + stage1_addr<Ge>(j);
#pragma unroll
            for (int m = 0; m < R0; ++m) w[m * La::S0] = v[m];
        }
        __syncthreads();
    }
    const long long ldq = a.ldT / 2;
    float4* Tq = reinterpret_cast<float4*>(a.T + blockIdx.y * a.specT);
    if constexpr (R0 == 1) {
#pragma unroll 1
        for (int e = 0; e < RS::ROUNDS; ++e) {
            const RS s(t, e);
            float2* b = work + s.tr * La::ELEMS;
            if (s.live && s.li < R2) {
                float2 x[R1];
                const RowInput in(a, pair0 + s.tr);
#pragma unroll
                for (int l = 0; l < R1; ++l) x[l] = in(s.li + l * R2);
                stage2_fwd<Ge>(x, b, 0, s.li, lp_dsmem, a.tw.w2);
            }
            __syncwarp();
            float2 f[R2];
            if (s.live && s.li < R1) {
                load_run<Ge>(f, b, s.li);
                Dft<R2, -1, float2>::run(f);
            }
            const int pair = pair0 + s.tr;
            const bool store = s.live && s.li < R1 && pair < a.npairs;
            const int u = s.li;
            float4* dst = Tq + t_index4(u, pair, ldq);
#pragma unroll
            for (int k = 0; k <= R2 / 2; ++k) {
                float2 zm;
                constexpr int last = R2 - 1;
                zm.x = __shfl_sync(0xffffffffu, f[last - k].x, s.partner);
                zm.y = __shfl_sync(0xffffffffu, f[last - k].y, s.partner);
                if (s.origin) zm = f[k == 0 ? 0 : R2 - k];
                const int c = u + k * UR;
                if (store && (k < R2 / 2 || c < a.ncols)) {
                    const float4 o = split_rows(f[k], zm);
                    if constexpr (UR % kTCB == 0) dst[k * (UR / kTCB) * (ldq * kTCB)] = o;
                    else Tq[t_index4(c, pair, ldq)] = o;
                }
            }
        }
    } else {
        const int li = t % Ge::G;
#pragma unroll 1
        for (int e = 0; e < C::EB; ++e) {
            const int q = t / Ge::G + e * C::GROUPS;
            const bool live = C::EB * C::GROUPS == C::UB || q < C::UB;
            const int tr = C::NT == 1 ? 0 : q / R0;
            const int m = q - tr * R0;
            float2* b = work + tr * La::ELEMS + m * La::S0;
            if (live && li < R2) {
                float2 x[R1];
#pragma unroll
                for (int l = 0; l < R1; ++l) x[l] = b[li + l * La::S1];
                stage2_fwd<Ge>(x, b, m, li, lp_dsmem, a.tw.w2);
            }
            __syncwarp();
            if (live && li < R1) {
                float2 f[R2];
                load_run<Ge>(f, b, li);
                Dft<R2, -1, float2>::run(f);
                store_run<Ge>(f, b, li);
            }
        }
        __syncthreads();
        // The run u = m + R0 k1 holds the frequencies c = u + R0 R1 k2, its
        // partners N - c are the run R0 R1 - u backwards, so both addresses
        // are a base plus a constant.
#pragma unroll 1
        for (int e = 0; e < C::ES; ++e) {
            const int v = t + e * C::TH;
            if (C::ES * C::TH != C::US && v >= C::US) break;
            const int tr = v % C::NT, u = v / C::NT;
            const int pair = pair0 + tr;
            if (pair >= a.npairs) continue;
            const int up = u == 0 ? 0 : UR - u;
            const float2* z = work + tr * La::ELEMS + (u % R0) * La::S0 + (u / R0) * La::S1;
            const float2* zp = work + tr * La::ELEMS + (up % R0) * La::S0 + (up / R0) * La::S1;
            float4* dst = Tq + t_index4(u, pair, ldq);
            auto put = [&](int k, float2 zc, float2 zm) {
                if constexpr (UR % kTCB == 0) dst[k * (UR / kTCB) * (ldq * kTCB)] = split_rows(zc, zm);
                else Tq[t_index4(u + k * UR, pair, ldq)] = split_rows(zc, zm);
            };
            if (La::VEC && u > 0) {
                // R2 even: k2 < R2 / 2, two at a time
#pragma unroll
                for (int k = 0; k < R2 / 2; k += 2) {
                    const float4 c2 = *reinterpret_cast<const float4*>(z + k);
                    const float4 p2 = *reinterpret_cast<const float4*>(zp + (R2 - 2 - k));
                    put(k, make_float2(c2.x, c2.y), make_float2(p2.z, p2.w));
                    if (k + 1 < R2 / 2) put(k + 1, make_float2(c2.z, c2.w), make_float2(p2.x, p2.y));
                }
            } else {
#pragma unroll
                for (int k = 0; k <= R2 / 2; ++k)
                    if (k < R2 / 2 || u + k * UR < a.ncols)
                        put(k, z[k], zp[u > 0 ? R2 - 1 - k : k == 0 ? 0 : R2 - k]);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// P2: per column forward FFT, spectrum product, inverse FFT, row crop.
// ---------------------------------------------------------------------------
// Stage 1 of NT columns from T (rows >= H are the zero padding) into sm.
// Consecutive lanes take the block's columns, then rows, so that the pieces
// of a column block of T are read together.
template <class C>
__device__ __forceinline__ void column_stage1(const float2* T, long long ldT, int H, int c0, int ncols,
                                              float2* sm, int t, int th)
{
    using Ge = typename C::Ge;
    using La = typename C::La;
    constexpr int R0 = Ge::R0, N1 = Ge::N1, NT = C::NT;
#pragma unroll 1
    for (int u = t; u < C::U1; u += th) {
        const int cl = u % NT, j = u / NT;
        const int c = c0 + cl;
        const float2* col = t_column(T, ldT, c);
        float2 v[R0];
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            const int row = j + q * N1;
            const long long off = (N1 % 2 == 0) ? t_row(j) + q * t_row_step<N1>() : t_row(row);
            v[q] = (row < H && (NT == 1 || c < ncols)) ? ld_once<Ge>(col + off) : make_float2(0.f, 0.f);
        }
        Dft<R0, -1, float2>::run(v);
        float2* w = sm + cl * La::ELEMS + stage1_addr<Ge>(j);
#pragma unroll
        for (int m = 0; m < R0; ++m) w[m * La::S0] = v[m];
    }
}

// Inverse stage 1 of NT columns: rows of the crop window to U.
template <class C>
__device__ __forceinline__ void column_out(const P2Args& a, float2* U, int c0, const float2* sm, int t)
{
    using Ge = typename C::Ge;
    using La = typename C::La;
    constexpr int R0 = Ge::R0, N1 = Ge::N1, NT = C::NT;
#pragma unroll 1
    for (int u = t; u < C::U1; u += C::TH) {
        const int cl = u % NT, j = u / NT;
        const int c = c0 + cl;
        const float2* w = sm + cl * La::ELEMS + stage1_addr<Ge>(j);
        float2 v[R0];
#pragma unroll
        for (int m = 0; m < R0; ++m) v[m] = w[m * La::S0];
        Dft<R0, 1, float2>::run(v);
        if (NT > 1 && c >= a.ncols) continue;
        float2* Uc = u_column(U, a.ldU, c);
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            int rr = j + q * N1 - a.r0;
            if (rr < 0) rr += Ge::N;
            if (rr < a.Hout) Uc[u_row(rr)] = v[q];
        }
    }
}

// the zero row that completes the last row pair when Hout is odd
template <class C>
__device__ __forceinline__ void column_pad(const P2Args& a, float2* U, int c0, int t)
{
    if (a.HoutPad != a.Hout && t < C::NT && c0 + t < a.ncols)
        u_column(U, a.ldU, c0 + t)[u_row(a.Hout)] = make_float2(0.f, 0.f);
}

// Spectrum values of frequencies (m, k1, 0..R2-1) of one column (stored in
// the order Geo::kpos).
template <class Ge, bool KREAL>
__device__ __forceinline__ void load_spectrum(typename std::conditional<KREAL, float, float2>::type (&k)[Ge::R2],
                                              const void* kcol, int m, int k1)
{
    constexpr int R2 = Ge::R2, VK = Ge::VK;
    if constexpr (KREAL) {
        const float* p = static_cast<const float*>(kcol) + Ge::kpos(m, k1, 0);
#pragma unroll
        for (int i = 0; i < R2; i += VK) {
            const float* q = p + i * Ge::R1;
            if constexpr (VK == 4) {
                const float4 x = ld_spectrum<Ge>(reinterpret_cast<const float4*>(q));
                k[i] = x.x;
                k[i + 1] = x.y;
                k[i + 2] = x.z;
                k[i + 3] = x.w;
            } else if constexpr (VK == 2) {
                const float2 x = ld_spectrum<Ge>(reinterpret_cast<const float2*>(q));
                k[i] = x.x;
                k[i + 1] = x.y;
            } else {
                k[i] = ld_spectrum<Ge>(q);
            }
        }
    } else {
        const float2* p = static_cast<const float2*>(kcol) + Ge::kpos(m, k1, 0);
#pragma unroll
        for (int i = 0; i < R2; i += VK) {
            const float2* q = p + i * Ge::R1;
            if constexpr (VK >= 2) {
#pragma unroll
                for (int h = 0; h < VK; h += 2) {
                    const float4 x = ld_spectrum<Ge>(reinterpret_cast<const float4*>(q + h));
                    k[i + h] = make_float2(x.x, x.y);
                    k[i + h + 1] = make_float2(x.z, x.w);
                }
            } else {
                k[i] = ld_spectrum<Ge>(q);
            }
        }
    }
}

// Bulk prefetch of the spectrum columns c0 .. of one spectrum into L2 by NT
// threads: a batched block's next spectrum, while it works on this one.
template <class C, bool KREAL>
__device__ __forceinline__ void prefetch_spectrum(const P2Args& a, const void* K, int c0, int t)
{
    if (t < C::NT && c0 + t < a.ncols) {
        const float* p = static_cast<const float*>(K) + (long long)(c0 + t) * a.ldK * (KREAL ? 1 : 2);
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p),
                     "r"(16u * ((C::Ge::N * (KREAL ? 1 : 2) + 3) / 4)) : "memory");
    }
}

template <bool KREAL, int R>
__device__ __forceinline__ void spectrum_product(float2 (&f)[R],
                                                 const typename std::conditional<KREAL, float, float2>::type (&k)[R])
{
#pragma unroll
    for (int i = 0; i < R; ++i) {
        if constexpr (KREAL) f[i] = cscale(f[i], k[i]);
        else f[i] = cmul(f[i], k[i]);
    }
}

// Where R0 = 1 a column is one sub-transform: rows li + l R2 of T, read by
// stage 2 itself.
template <class Ge>
__device__ __forceinline__ void column_direct(float2 (&x)[Ge::R1], const float2* T, long long ldT, int H, int c,
                                              int li)
{
    const float2* col = t_column(T, ldT, c);
#pragma unroll
    for (int l = 0; l < Ge::R1; ++l) {
        const int row = li + l * Ge::R2;
        x[l] = row < H ? ld_once<Ge>(col + t_row(row)) : make_float2(0.f, 0.f);
    }
}
template <class Ge>
__device__ __forceinline__ void column_direct_out(const float2 (&x)[Ge::R1], const P2Args& a, float2* U, int c, int li)
{
    float2* Uc = u_column(U, a.ldU, c);
#pragma unroll
    for (int l = 0; l < Ge::R1; ++l) {
        int rr = li + l * Ge::R2 - a.r0;
        if (rr < 0) rr += Ge::N;
        if (rr < a.Hout) Uc[u_row(rr)] = x[l];
    }
}

// One spectrum.
template <class C, bool KREAL>
__global__ void __launch_bounds__(C::TH, C::MINB) p2_cols(const __grid_constant__ P2Args a)
{
    pdl_begin<C::LATE>();
    using Ge = typename C::Ge;
    using La = typename C::La;
    constexpr int R0 = Ge::R0, R1 = Ge::R1, R2 = Ge::R2, NT = C::NT;
    const int c0 = blockIdx.x * NT;
    const int t = threadIdx.x;
    float2* work = lp_dsmem + Ge::W1;
    for (int cl = 0; cl < NT; ++cl)
        if (c0 + cl < a.ncols && !p2_column_ok(a, c0 + cl, Ge::N, KREAL ? 1 : 2, c0 + cl + 1)) return;
    if constexpr (R0 > 1) {
        load_w1<Ge>(lp_dsmem, a.tw.w1, t, C::TH);
        column_stage1<C>(a.T, a.ldT, a.H, c0, a.ncols, work, t, C::TH);
        __syncthreads();
    }
    const int li = t % Ge::G;
#pragma unroll 1
    for (int e = 0; e < C::EB; ++e) {
        const int q = t / Ge::G + e * C::GROUPS;
        const int cl = q % NT, m = q / NT;
        const int c = c0 + cl;
        const bool live = (C::EB * C::GROUPS == C::UB || q < C::UB) && (NT == 1 || c < a.ncols);
        float2* b = work + cl * La::ELEMS + m * La::S0;
        if (live && li < R2) {
            float2 x[R1];
            if constexpr (R0 > 1) {
#pragma unroll
                for (int l = 0; l < R1; ++l) x[l] = b[li + l * La::S1];
            } else {
                column_direct<Ge>(x, a.T, a.ldT, a.H, c, li);
            }
            stage2_fwd<Ge>(x, b, m, li, lp_dsmem, a.tw.w2);
        }
        typename std::conditional<KREAL, float, float2>::type k[R2];
        if (live && li < R1)
            load_spectrum<Ge, KREAL>(k, static_cast<const float*>(a.K[0]) + (long long)c * a.ldK * (KREAL ? 1 : 2), m, li);
        __syncwarp();
        if (live && li < R1) {
            float2 f[R2];
            load_run<Ge>(f, b, li);
            Dft<R2, -1, float2>::run(f);
            spectrum_product<KREAL>(f, k);
            Dft<R2, 1, float2>::run(f);
            store_run<Ge>(f, b, li);
        }
        __syncwarp();
        if (live && li < R2) {
            float2 x[R1];
            stage2_inv<Ge>(x, b, m, li, lp_dsmem, a.tw.w2);
            if constexpr (R0 > 1) {
#pragma unroll
                for (int l = 0; l < R1; ++l) b[li + l * La::S1] = x[l];
            } else {
                column_direct_out<Ge>(x, a, a.U, c, li);
            }
        }
    }
    if constexpr (R0 > 1) {
        __syncthreads();
        column_out<C>(a, a.U, c0, work, t);
    }
    column_pad<C>(a, a.U, c0, t);
}

// ---------------------------------------------------------------------------
// Several spectra (lp_map, n > 1) and several source classes (Sec. 2.2
// Eq. (4)): the frequencies of a column are parked in the order the threads
// of stage 3 hold them -- run (m, k1) of column cl, elements k2 -- in shared
// memory, or in global memory (PARKG) for the lengths that leave no room.
// Every element is read back by the thread that wrote it or after a barrier.
// ---------------------------------------------------------------------------
template <class C>
__device__ __forceinline__ void park_store(float2* F, int run, const float2 (&f)[C::Ge::R2])
{
    constexpr int R2 = C::Ge::R2, RUNS = C::US;
    if constexpr (R2 % 2 == 0) {
        float4* p = reinterpret_cast<float4*>(F) + run;
#pragma unroll
        for (int k = 0; k < R2; k += 2)
            p[(k / 2) * RUNS] = make_float4(f[k].x, f[k].y, f[k + 1].x, f[k + 1].y);
    } else {
#pragma unroll
        for (int k = 0; k < R2; ++k) F[k * RUNS + run] = f[k];
    }
}
template <class C>
__device__ __forceinline__ void park_load(float2 (&f)[C::Ge::R2], const float2* F, int run)
{
    constexpr int R2 = C::Ge::R2, RUNS = C::US;
    if constexpr (R2 % 2 == 0) {
        const float4* p = reinterpret_cast<const float4*>(F) + run;
#pragma unroll
        for (int k = 0; k < R2; k += 2) {
            const float4 q = p[(k / 2) * RUNS];
            f[k] = make_float2(q.x, q.y);
            f[k + 1] = make_float2(q.z, q.w);
        }
    } else {
#pragma unroll
        for (int k = 0; k < R2; ++k) f[k] = F[k * RUNS + run];
    }
}

// barrier of one group of TH threads (the whole block where there is one group)
template <int TH, int GRP>
__device__ __forceinline__ void group_sync(int grp)
{
    if constexpr (GRP == 1) __syncthreads();
    else asm volatile("barrier.cta.sync %0, %1;\n" ::"r"(grp + 1), "n"(TH) : "memory");
}

// Forward transform of columns c0.. of T by all `th` threads of the block,
// each frequency run handed to `sink(cl, m, k1, f)`.
template <class C, class Sink>
__device__ __forceinline__ void columns_forward(const float2* T, long long ldT, int H, int c0, int ncols,
                                                BlkTw tw, float2* sm, int t, int th, Sink&& sink)
{
    using Ge = typename C::Ge;
    using La = typename C::La;
    constexpr int R0 = Ge::R0, R1 = Ge::R1, R2 = Ge::R2, NT = C::NT;
    if constexpr (R0 > 1) {
        column_stage1<C>(T, ldT, H, c0, ncols, sm, t, th);
        __syncthreads();
    }
    const int li = t % Ge::G;
    const int groups = th / Ge::G;
#pragma unroll 1
    for (int q0 = 0; q0 < C::UB; q0 += groups) {
        const int q = t / Ge::G + q0;
        const int cl = q % NT, m = q / NT;
        const bool live = q < C::UB && (NT == 1 || c0 + cl < ncols);
        float2* b = sm + cl * La::ELEMS + m * La::S0;
        if (live && li < R2) {
            float2 x[R1];
            if constexpr (R0 > 1) {
#pragma unroll
                for (int l = 0; l < R1; ++l) x[l] = b[li + l * La::S1];
            } else {
                column_direct<Ge>(x, T, ldT, H, c0 + cl, li);
            }
            stage2_fwd<Ge>(x, b, m, li, lp_dsmem, tw.w2);
        }
        __syncwarp();
        if (live && li < R1) {
            float2 f[R2];
            load_run<Ge>(f, b, li);
            Dft<R2, -1, float2>::run(f);
            sink(cl, m, li, f);
        }
    }
}

// Inverse of columns c0.. by the TH threads of one group (thread t of it):
// `source(cl, m, k1, f)` gives each frequency run (live columns only).
template <class C, int GRP, class Source>
__device__ __forceinline__ void columns_inverse(const P2Args& a, float2* U, int c0, float2* sm, int t, int grp,
                                                Source&& source)
{
    using Ge = typename C::Ge;
    using La = typename C::La;
    constexpr int R0 = Ge::R0, R1 = Ge::R1, R2 = Ge::R2, NT = C::NT;
    const int li = t % Ge::G;
#pragma unroll 1
    for (int e = 0; e < C::EB; ++e) {
        const int q = t / Ge::G + e * C::GROUPS;
        const int cl = q % NT, m = q / NT;
        const bool live = (C::EB * C::GROUPS == C::UB || q < C::UB) && (NT == 1 || c0 + cl < a.ncols);
        float2* b = sm + cl * La::ELEMS + m * La::S0;
        if (live && li < R1) {
            float2 f[R2];
            source(cl, m, li, f);
            Dft<R2, 1, float2>::run(f);
            store_run<Ge>(f, b, li);
        }
        __syncwarp();
        if (live && li < R2) {
            float2 x[R1];
            stage2_inv<Ge>(x, b, m, li, lp_dsmem, a.tw.w2);
            if constexpr (R0 > 1) {
#pragma unroll
                for (int l = 0; l < R1; ++l) b[li + l * La::S1] = x[l];
            } else {
                column_direct_out<Ge>(x, a, U, c0 + cl, li);
            }
        }
        if constexpr (R0 == 1) __syncwarp();
    }
    if constexpr (R0 > 1) {
        group_sync<C::TH, GRP>(grp);
        column_out<C>(a, U, c0, sm, t);
    }
    column_pad<C>(a, U, c0, t);
}

// One spectrum of the batched pass.  Not inlined: as a loop body it would
// let the compiler keep constants and addresses of the whole inverse live
// across iterations.
template <class C, int GRP, bool PARKG, bool KREAL>
__device__ __noinline__ void p2_spectrum_pass(const P2Args& a, int c0, int s, int work, int t, int grp)
{
    using Ge = typename C::Ge;
    constexpr int R2 = Ge::R2;
    const float2* F = PARKG ? a.park + (size_t)c0 * Ge::N : lp_dsmem + Ge::W1 + GRP * C::WORK;
    columns_inverse<C, GRP>(a, a.U + (long long)s * a.specU, c0, lp_dsmem + Ge::W1 + work, t, grp,
                            [&](int cl, int m, int k1, float2(&f)[R2]) {
                                typename std::conditional<KREAL, float, float2>::type k[R2];
                                load_spectrum<Ge, KREAL>(k, static_cast<const float*>(a.K[s]) +
                                                                (long long)(c0 + cl) * a.ldK * (KREAL ? 1 : 2), m, k1);
                                park_load<C>(f, F, (cl * Ge::R0 + m) * Ge::R1 + k1);
                                spectrum_product<KREAL>(f, k);
                            });
}

// Several spectra: GRP groups of TH threads take the spectra in turn, each
// with a working set of its own beside the one parked column (set).
template <class C, int GRP, bool PARKG, bool KREAL>
__global__ void __launch_bounds__(C::TH * GRP, C::MINB) p2_cols_multi(const __grid_constant__ P2Args a)
{
    pdl_begin<C::LATE>();
    using Ge = typename C::Ge;
    constexpr int NT = C::NT;
    const int c0 = blockIdx.x * NT;
    for (int cl = 0; cl < NT; ++cl)
        if (c0 + cl < a.ncols && !p2_column_ok(a, c0 + cl, Ge::N, KREAL ? 1 : 2, c0 + NT)) return;
    float2* F = PARKG ? a.park + (size_t)c0 * Ge::N : lp_dsmem + Ge::W1 + GRP * C::WORK;
    const int grp = GRP == 1 ? 0 : threadIdx.x / C::TH;
    const int t = GRP == 1 ? threadIdx.x : threadIdx.x % C::TH;
    if (grp < a.nspec) prefetch_spectrum<C, KREAL>(a, a.K[grp], c0, t);
    load_w1<Ge>(lp_dsmem, a.tw.w1, threadIdx.x, C::TH * GRP);
    columns_forward<C>(a.T, a.ldT, a.H, c0, a.ncols, a.tw, lp_dsmem + Ge::W1, threadIdx.x, C::TH * GRP,
                       [&](int cl, int m, int k1, float2(&f)[Ge::R2]) {
                           park_store<C>(F, (cl * Ge::R0 + m) * Ge::R1 + k1, f);
                       });
    __syncthreads();
#pragma unroll 1
    for (int s = grp; s < a.nspec; s += GRP) {
        if (s + GRP < a.nspec) prefetch_spectrum<C, KREAL>(a, a.K[s + GRP], c0, t);
        p2_spectrum_pass<C, GRP, PARKG, KREAL>(a, c0, s, grp * C::WORK, t, grp);
        if constexpr (Ge::R0 > 1) group_sync<C::TH, GRP>(grp);  // the working set has been read
    }
}

// ---------------------------------------------------------------------------
// P2 for Sec. 2.2 Eq. (4): several source classes, one PSF each.  The
// forward column transform of each class's T is multiplied by its spectrum
// and accumulated; one inverse transform follows.
// ---------------------------------------------------------------------------
struct P2MArgs {
    P2Args a;  // output side, twiddles, ncols; T and K unused
    const float2* T[kMaxSpectraPerLaunch];
    const void* K[kMaxSpectraPerLaunch];
    int nclass;
};

// multiclass unit: column c of every class's T, of every spectrum, of U and of the sums
__device__ __forceinline__ bool p2m_column_ok(const P2MArgs& m, int c, int n, int kw, int park_end)
{
    return p2_column_ok(m.a, c, n, kw, park_end);
}

// One class: forward transform of the class's columns, product with its
// spectrum, summed into F (the first class writes it).  Each thread adds only
// to elements it owns, so the sum needs no barrier.
template <class C, bool PARKG, bool KREAL>
__device__ __noinline__ void p2_class_pass(const P2MArgs& M, int c0, int q)
{
    using Ge = typename C::Ge;
    constexpr int R2 = Ge::R2;
    const P2Args& a = M.a;
    float2* F = PARKG ? a.park + (size_t)c0 * Ge::N : lp_dsmem + Ge::W1 + C::WORK;
    columns_forward<C>(M.T[q], a.ldT, a.H, c0, a.ncols, a.tw, lp_dsmem + Ge::W1, threadIdx.x, C::TH,
                       [&](int cl, int m, int k1, float2(&f)[R2]) {
                           typename std::conditional<KREAL, float, float2>::type k[R2];
                           load_spectrum<Ge, KREAL>(k, static_cast<const float*>(M.K[q]) +
                                                           (long long)(c0 + cl) * a.ldK * (KREAL ? 1 : 2), m, k1);
                           spectrum_product<KREAL>(f, k);
                           const int run = (cl * Ge::R0 + m) * Ge::R1 + k1;
                           if (q > 0) {
                               float2 s[R2];
                               park_load<C>(s, F, run);
#pragma unroll
                               for (int i = 0; i < R2; ++i) f[i] = cadd(s[i], f[i]);
                           }
                           park_store<C>(F, run, f);
                       });
}

template <class C, bool PARKG, bool KREAL>
__global__ void __launch_bounds__(C::TH, C::MINB) p2_multiclass(const __grid_constant__ P2MArgs M)
{
    pdl_begin<C::LATE>();
    using Ge = typename C::Ge;
    constexpr int NT = C::NT;
    const P2Args& a = M.a;
    const int c0 = blockIdx.x * NT;
    for (int cl = 0; cl < NT; ++cl)
        if (c0 + cl < a.ncols && !p2m_column_ok(M, c0 + cl, Ge::N, KREAL ? 1 : 2, c0 + NT)) return;
    const float2* F = PARKG ? a.park + (size_t)c0 * Ge::N : lp_dsmem + Ge::W1 + C::WORK;
    load_w1<Ge>(lp_dsmem, a.tw.w1, threadIdx.x, C::TH);
#pragma unroll 1
    for (int q = 0; q < M.nclass; ++q) {
        p2_class_pass<C, PARKG, KREAL>(M, c0, q);
        __syncthreads();  // the working set has been read
    }
    // (groups of one round are the same in both directions: TH threads, one
    // group; every run is read back by the thread that summed it)
    columns_inverse<C, 1>(a, a.U, c0, lp_dsmem + Ge::W1, threadIdx.x, 0, [&](int cl, int m, int k1, float2(&f)[Ge::R2]) {
        park_load<C>(f, F, (cl * Ge::R0 + m) * Ge::R1 + k1);
    });
}

// ---------------------------------------------------------------------------
// P3: row C2R of two packed rows per transform, NT transforms per block,
// blockIdx.y selects the spectrum.  P1 backwards.
// ---------------------------------------------------------------------------
template <class C>
__global__ void __launch_bounds__(C::TH, C::MINB) p3_rows(const __grid_constant__ P3Args a)
{
    pdl_begin<C::LATE>();
    using Ge = typename C::Ge;
    using La = typename C::La;
    using RS = RowSub<C>;
    constexpr int R0 = Ge::R0, R1 = Ge::R1, R2 = Ge::R2, N1 = Ge::N1, N = Ge::N, UR = R0 * R1;
    const int pair0 = a.pair0 + blockIdx.x * C::NT;
    const int sidx = blockIdx.y;
    for (int tr = 0; tr < C::NT; ++tr)
        if (pair0 + tr < a.npairs && !p3_unit_ok(a, pair0 + tr, sidx)) return;
    const int t = threadIdx.x;
    float2* work = lp_dsmem + Ge::W1;
    const long long ldq = a.ldU / 2;
    const float4* Uq = reinterpret_cast<const float4*>(a.U + (long long)sidx * a.specU);
    auto store2 = [&](int tr, int col, float2 o) {
        const int pair = pair0 + tr;
        int cc = col - a.c0;
        if (cc < 0) cc += N;
        if (cc < a.Wout && pair < a.npairs) {
            float* oa = a.out[sidx] + (long long)(2 * pair) * a.ldo + cc;
            oa[0] = o.x;
            if (2 * pair + 1 < a.Hout) oa[a.ldo] = o.y;
        }
    };
    // lane li of sub-transform m at b: inverse stage 2, kept in place or (R0 = 1) stored
    auto finish = [&](int tr, int m, int li, float2* b) {
        float2 x[R1];
        stage2_inv<Ge>(x, b, m, li, lp_dsmem, a.tw.w2);
        if constexpr (R0 > 1) {
#pragma unroll
            for (int l = 0; l < R1; ++l) b[li + l * La::S1] = x[l];
        } else {
#pragma unroll
            for (int l = 0; l < R1; ++l) store2(tr, li + l * R2, x[l]);
        }
    };
    if constexpr (R0 > 1) load_w1<Ge>(lp_dsmem, a.tw.w1, t, C::TH);
    if constexpr (R0 == 1) {
#pragma unroll 1
        for (int e = 0; e < RS::ROUNDS; ++e) {
            const RS s(t, e);
            float2* b = work + s.tr * La::ELEMS;
            const int pair = pair0 + s.tr;
            const bool load = s.live && s.li < R1 && pair < a.npairs;
            const bool vb = 2 * pair + 1 < a.Hout;
            const int u = s.li;
            const float4* src = Uq + u_index4(u, pair, ldq);
            float4 q[R2 / 2 + 1];
#pragma unroll
            for (int k = 0; k <= R2 / 2; ++k) {
                const int c = u + k * UR;
                q[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (load && (k < R2 / 2 || c < a.ncols)) {
                    if constexpr (UR % kUCB == 0) q[k] = ld_once<Ge>(src + k * (UR / kUCB) * (ldq * kUCB));
                    else q[k] = ld_once<Ge>(Uq + u_index4(c, pair, ldq));
                }
                if (!vb) q[k].z = q[k].w = 0.f;
            }
            // own lower half; the upper half from the partner (the origin
            // run holds its own, one element further on)
            float2 f[R2];
#pragma unroll
            for (int k = 0; k < R2 / 2; ++k) f[k] = join_lo(q[k]);
#pragma unroll
            for (int k = 0; k < (R2 + 1) / 2; ++k) {
                float2 h = join_hi(q[k]);
                h.x = __shfl_sync(0xffffffffu, h.x, s.partner);
                h.y = __shfl_sync(0xffffffffu, h.y, s.partner);
                if (k == R2 / 2) {  // R2 odd: the middle element, whichever side of N / 2 it is on
                    f[k] = u + k * UR < a.ncols ? join_lo(q[k]) : h;
                } else {
                    const float2 own = (R2 % 2 == 0 && k + 1 == R2 / 2) ? join_lo(q[R2 / 2]) : join_hi(q[k + 1]);
                    f[R2 - 1 - k] = s.origin ? own : h;
                }
            }
            if (s.live && s.li < R1) {
                Dft<R2, 1, float2>::run(f);
                store_run<Ge>(f, b, s.li);
            }
            __syncwarp();
            if (s.live && s.li < R2) finish(s.tr, 0, s.li, b);
        }
    } else {
#pragma unroll 1
        for (int e = 0; e < C::ES; ++e) {
            const int v = t + e * C::TH;
            if (C::ES * C::TH != C::US && v >= C::US) break;
            const int tr = v % C::NT, u = v / C::NT;
            const int pair = pair0 + tr;
            if (pair >= a.npairs) continue;
            const bool vb = 2 * pair + 1 < a.Hout;
            const int up = u == 0 ? 0 : UR - u;
            float2* z = work + tr * La::ELEMS + (u % R0) * La::S0 + (u / R0) * La::S1;
            float2* zp = work + tr * La::ELEMS + (up % R0) * La::S0 + (up / R0) * La::S1;
            const float4* src = Uq + u_index4(u, pair, ldq);
            float4 q[R2 / 2 + 1];
#pragma unroll
            for (int k = 0; k <= R2 / 2; ++k) {
                const int c = u + k * UR;
                if (k == R2 / 2 && c >= a.ncols) break;
                if constexpr (UR % kUCB == 0) q[k] = ld_once<Ge>(src + k * (UR / kUCB) * (ldq * kUCB));
                else q[k] = ld_once<Ge>(Uq + u_index4(c, pair, ldq));
                if (!vb) q[k].z = q[k].w = 0.f;
            }
            if (La::VEC && u > 0) {
#pragma unroll
                for (int k = 0; k < R2 / 2; k += 2) {
                    const float2 l0 = join_lo(q[k]), h0 = join_hi(q[k]);
                    if (k + 1 < R2 / 2) {
                        const float2 l1 = join_lo(q[k + 1]), h1 = join_hi(q[k + 1]);
                        *reinterpret_cast<float4*>(z + k) = make_float4(l0.x, l0.y, l1.x, l1.y);
                        *reinterpret_cast<float4*>(zp + (R2 - 2 - k)) = make_float4(h1.x, h1.y, h0.x, h0.y);
                    } else {
                        z[k] = l0;
                        zp[R2 - 1 - k] = h0;
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k <= R2 / 2; ++k) {
                    const int c = u + k * UR;
                    if (k == R2 / 2 && c >= a.ncols) break;
                    z[k] = join_lo(q[k]);
                    if (k == 0 ? u != 0 : (k != R2 / 2 || 2 * c != N)) zp[u > 0 ? R2 - 1 - k : R2 - k] = join_hi(q[k]);
                }
            }
        }
        __syncthreads();
        const int li = t % Ge::G;
#pragma unroll 1
        for (int e = 0; e < C::EB; ++e) {
            const int q = t / Ge::G + e * C::GROUPS;
            const bool live = C::EB * C::GROUPS == C::UB || q < C::UB;
            const int tr = C::NT == 1 ? 0 : q / R0;
            const int m = q - tr * R0;
            float2* b = work + tr * La::ELEMS + m * La::S0;
            if (live && li < R1) {
                float2 f[R2];
                load_run<Ge>(f, b, li);
                Dft<R2, 1, float2>::run(f);
                store_run<Ge>(f, b, li);
            }
            __syncwarp();
            if (live && li < R2) finish(tr, m, li, b);
        }
    }
    if constexpr (R0 > 1) {
        __syncthreads();
#pragma unroll 1
        for (int e = 0; e < C::E1; ++e) {
            const int u = t + e * C::TH;
            if (C::E1 * C::TH != C::U1 && u >= C::U1) break;
            const int tr = C::NT == 1 ? 0 : u / N1;
            const int j = u - tr * N1;
            const float2* w = work + tr * La::ELEMS + stage1_addr<Ge>(j);
            float2 v[R0];
#pragma unroll
            for (int m = 0; m < R0; ++m) v[m] = w[m * La::S0];
            Dft<R0, 1, float2>::run(v);
            const int pair = pair0 + tr;
            if (pair >= a.npairs) continue;
            const bool vb = 2 * pair + 1 < a.Hout;
            float* oa = a.out[sidx] + (long long)(2 * pair) * a.ldo;
            float* ob = oa + a.ldo;
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                int cc = j + q * N1 - a.c0;
                if (cc < 0) cc += N;
                if (cc < a.Wout) {
                    oa[cc] = v[q].x;
                    if (vb) ob[cc] = v[q].y;
                }
            }
        }
    }
}

}  // namespace lpk
