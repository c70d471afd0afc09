// Site-tensor repacking, FP32 SIMT contraction, measurement (Algorithm 2) and
// output transposition kernels.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "f32x2.cuh"
#include "launch.h"
#include "measure.cuh"

namespace fastmps {

// ---------------------------------------------------------------------------
// Stacked real operand of the complex contraction.
//
// With v = vr + i vi and A = Ar + i Ai, y = v A has
//   Re y =  vr Ar - vi Ai,   Im y = vr Ai + vi Ar,
// so with the left row [vr | vi] (length 2 chi_l) the output column
// (s, p = 0, b) takes the operand column [Ar[:, s, b] ; -Ai[:, s, b]] and the
// column (s, p = 1, b) takes [Ai[:, s, b] ; Ar[:, s, b]].  That is four real
// products per complex multiply-add, 8 chi_l d chi_r flops per sample.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float load_part(const void *src, int is_f64, int64_t cidx, int part) {
    if (is_f64) return (float)(static_cast<const double *>(src)[2 * cidx + part]);
    return static_cast<const float *>(src)[2 * cidx + part];
}

// Returns the operand value at output column c and reduction index kappa and
// sets *zero when the position is padding.  (re_part, sign) say which part of
// A[a, s, b] it is: value = sign * (re_part ? Re : Im) A[a, s, b].
struct StackedPos {
    int64_t cidx;  // complex index a*d*chi_r + s*chi_r + b
    int re_part;   // 1: real part, 0: imaginary part
    float sign;
    bool zero;
};

__device__ __forceinline__ StackedPos stacked_pos(int c, int kappa, int chi_l, int d, int chi_r, int Cs) {
    StackedPos q;
    const int s = c / Cs;
    const int r = c - s * Cs;
    q.zero = (r >= 2 * chi_r) || (kappa >= 2 * chi_l) || (s >= d);
    if (q.zero) {
        q.cidx = 0;
        q.re_part = 1;
        q.sign = 0.f;
        return q;
    }
    const int p = r >= chi_r;
    const int b = r - p * chi_r;
    const int second = kappa >= chi_l;
    const int a = second ? kappa - chi_l : kappa;
    q.cidx = ((int64_t)a * d + s) * chi_r + b;
    if (p == 0) {  // real output column: [Ar ; -Ai]
        q.re_part = second ? 0 : 1;
        q.sign = second ? -1.f : 1.f;
    } else {       // imaginary output column: [Ai ; Ar]
        q.re_part = second ? 1 : 0;
        q.sign = 1.f;
    }
    return q;
}

// 16-bit operands (BF16, or FP16 at a power-of-two scale) from complex float or double, optionally with column b
// scaled by lam[b] (Vidal form, in the input's type), or from a compact 16-bit copy.  Bound by HBM: each complex
// entry is read once and written four times (twice per plane and outcome column).
// The operand is the transpose of the tensor's rows: a block reads 64 x 32 entries (a, b) of one outcome along b,
// keeps them as 16-bit values in shared memory, and writes the four runs of 64 entries along kappa that they make
// (16-byte stores where chi_l is a multiple of 8).  Reading one entry per stored value along kappa instead, a
// chi_r-strided gather, took 185 us for chi = 2000, d = 3; this takes 44 (144 MB).
struct Repack16 {
    const void *src;       // [chi_l][d][chi_r] complex
    const void *lam;       // [chi_r] real, or null
    const float *amax;     // FP16: largest |Re|, |Im| (the scale puts it in [16384, 32768]); null: no scale
    int chi_l, d, chi_r, Cs, K_pad;
    int f16;
    uint16_t *hi, *lo;     // lo: null for one plane
};
enum Repack16Source : int { kFromFloat = 0, kFromDouble = 1, kFrom16 = 2 };
constexpr int kRepackA = 64, kRepackB = 32, kRepackLd = kRepackA + 8;

// Entry e of column b as FP32 (aligned to a whole entry).
template <int kSource>
__device__ __forceinline__ float2 repack_value(const Repack16 &r, int64_t e, int b) {
    if constexpr (kSource == kFromDouble) {
        double2 x = static_cast<const double2 *>(r.src)[e];
        if (r.lam) {
            const double l = static_cast<const double *>(r.lam)[b];
            x.x *= l;
            x.y *= l;
        }
        return make_float2((float)x.x, (float)x.y);
    } else {
        float2 x = static_cast<const float2 *>(r.src)[e];
        if (r.lam) {
            const float l = static_cast<const float *>(r.lam)[b];
            x.x *= l;
            x.y *= l;
        }
        return x;
    }
}

// 2^floor(log2(32768 / amax)) (1 for an all-zero tensor)
__device__ __forceinline__ float f16_site_scale(float amax) {
    if (!(amax > 0.f)) return 1.f;
    if (isinf(amax)) return 0.f;
    int e;
    const float m = frexpf(amax, &e);  // amax = m 2^e, m in [0.5, 1)
    return ldexpf(1.f, 15 - (m == 0.5f ? e - 1 : e));
}

template <int kSource, bool kVec>
__global__ void __launch_bounds__(256) repack16_kernel(const Repack16 r) {
    __shared__ __align__(16) uint16_t sm[4][kRepackB][kRepackLd];  // Re hi, Im hi, Re lo, Im lo
    const int b0 = blockIdx.x * kRepackB, a0 = blockIdx.y * kRepackA, s = blockIdx.z, tid = threadIdx.x;
    const int planes = r.lo ? 2 : 1;
    const float scale = r.amax ? f16_site_scale(*r.amax) : 1.f;
    const int64_t n = (int64_t)r.chi_l * r.d * r.chi_r;
    for (int i = tid; i < kRepackA * kRepackB; i += 256) {
        const int a = i / kRepackB, b = i % kRepackB;
        if (a0 + a >= r.chi_l || b0 + b >= r.chi_r) continue;
        const int64_t e = ((int64_t)(a0 + a) * r.d + s) * r.chi_r + b0 + b;
        if constexpr (kSource == kFrom16) {
            const ushort2 *c = static_cast<const ushort2 *>(r.src);
            const ushort2 hi = c[e];
            sm[0][b][a] = hi.x;
            sm[1][b][a] = hi.y;
            if (planes > 1) {
                const ushort2 lo = c[n + e];
                sm[2][b][a] = lo.x;
                sm[3][b][a] = lo.y;
            }
        } else {
            const float2 v = repack_value<kSource>(r, e, b0 + b);
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                const float x = (part ? v.y : v.x) * scale;  // exact: a power of two
                if (r.f16) {
                    const __half hi = __float2half_rn(x);
                    sm[part][b][a] = __half_as_ushort(hi);
                    if (planes > 1) sm[2 + part][b][a] = __half_as_ushort(__float2half_rn(x - __half2float(hi)));
                } else {
                    __nv_bfloat16 hi, lo;
                    split_bf16(x, hi, lo);
                    sm[part][b][a] = __bfloat16_as_ushort(hi);
                    if (planes > 1) sm[2 + part][b][a] = __bfloat16_as_ushort(lo);
                }
            }
        }
    }
    __syncthreads();
    // column (p, b) takes [Ar ; -Ai] (p = 0) or [Ai ; Ar] (p = 1) along kappa
    for (int q = 0; q < planes; ++q) {
        uint16_t *out = q ? r.lo : r.hi;
        constexpr int kRun = kVec ? kRepackA / 8 : kRepackA;  // stores per run of 64
        for (int i = tid; i < kRepackB * 4 * kRun; i += 256) {
            const int piece = i % kRun, half = i / kRun & 1, part = i / (2 * kRun) & 1, b = i / (4 * kRun);
            const int a = kVec ? 8 * piece : piece;
            if (b0 + b >= r.chi_r || a0 + a >= r.chi_l) continue;
            const uint16_t *v = &sm[2 * q + (part == half ? 0 : 1)][b][a];
            uint16_t *dst = out + ((int64_t)s * r.Cs + part * r.chi_r + b0 + b) * r.K_pad + half * r.chi_l + a0 + a;
            const bool negative = part == 0 && half == 1;
            if constexpr (kVec) {
                uint4 x = *reinterpret_cast<const uint4 *>(v);
                const uint32_t flip = negative ? 0x80008000u : 0u;
                *reinterpret_cast<uint4 *>(dst) = make_uint4(x.x ^ flip, x.y ^ flip, x.z ^ flip, x.w ^ flip);
            } else {
                *dst = (uint16_t)(*v ^ (negative ? 0x8000u : 0u));
            }
        }
        // padding: the end of these columns' rows, and the outcome block's columns past 2 chi_r
        if (a0 + kRepackA >= r.chi_l) {
            const int pad = r.K_pad - 2 * r.chi_l;
            for (int i = tid; i < pad * 2 * kRepackB; i += 256) {
                const int k = i % pad, part = i / pad & 1, b = i / (2 * pad);
                if (b0 + b < r.chi_r)
                    out[((int64_t)s * r.Cs + part * r.chi_r + b0 + b) * r.K_pad + 2 * r.chi_l + k] = 0;
            }
        }
        if (b0 + kRepackB >= r.chi_r) {
            // 128 kappa entries per a-tile cover K_pad = roundup(2 chi_l, 64)
            const int k0 = 2 * a0, pieces = min(2 * kRepackA, r.K_pad - k0) / 8;
            for (int i = tid; i < (r.Cs - 2 * r.chi_r) * pieces; i += 256)
                *reinterpret_cast<uint4 *>(out + ((int64_t)s * r.Cs + 2 * r.chi_r + i / pieces) * r.K_pad + k0 +
                                           8 * (i % pieces)) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
}

__global__ void repack_f32_kernel(const void *__restrict__ src, int is_f64, int chi_l, int d, int chi_r, int Cs,
                                  int ncols, int K_pad, float *__restrict__ Bt) {
    const int64_t total = (int64_t)ncols * K_pad;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int kappa = (int)(i / ncols);
        const int c = (int)(i - (int64_t)kappa * ncols);
        const StackedPos q = stacked_pos(c, kappa, chi_l, d, chi_r, Cs);
        float x = 0.f;
        if (!q.zero) x = q.sign * load_part(src, is_f64, q.cidx, q.re_part ? 0 : 1);
        Bt[i] = x;
    }
}

__global__ void repack_e4m3_kernel(const void *__restrict__ src, int is_f64, int chi_l, int d, int chi_r, int Cs,
                                   int ncols, int K_pad, float scale, uint8_t *__restrict__ B8) {
    const int64_t total = (int64_t)ncols * K_pad;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i / K_pad);
        const int kappa = (int)(i - (int64_t)c * K_pad);
        const StackedPos q = stacked_pos(c, kappa, chi_l, d, chi_r, Cs);
        float x = 0.f;
        if (!q.zero) x = q.sign * load_part(src, is_f64, q.cidx, q.re_part ? 0 : 1);
        B8[i] = (uint8_t)__nv_cvt_float_to_fp8(x * scale, __NV_SATFINITE, __NV_E4M3);
    }
}

// max over |Re|, |Im| (as float) of n2 / 2 complex entries, column b scaled by lam[b] (nullable); non-negative
// floats order like their bit patterns.  One atomic per block: one per warp kept the address busy for 28 us.
__global__ void __launch_bounds__(256) absmax_kernel(const void *__restrict__ src, int is_f64, int64_t n2, int chi_r,
                                                     const void *__restrict__ lam, float *out) {
    __shared__ float part[8];
    float m = 0.f;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n2; i += (int64_t)gridDim.x * blockDim.x) {
        float x;
        if (is_f64) {
            double v = static_cast<const double *>(src)[i];
            if (lam) v *= static_cast<const double *>(lam)[(i >> 1) % chi_r];
            x = (float)v;
        } else {
            x = static_cast<const float *>(src)[i];
            if (lam) x *= static_cast<const float *>(lam)[(i >> 1) % chi_r];
        }
        m = fmaxf(m, fabsf(x));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) m = fmaxf(m, part[w]);
        atomicMax(reinterpret_cast<unsigned int *>(out), __float_as_uint(m));
    }
}

static int grid_for(int64_t total, int block) {
    int64_t g = (total + block - 1) / block;
    if (g > 152 * 32) g = 152 * 32;
    if (g < 1) g = 1;
    return (int)g;
}

template <int kSource>
static void launch_repack16(const void *src, const void *lam, const float *amax, int f16, const SiteLayout &L, uint16_t *hi,
                            uint16_t *lo, cudaStream_t st) {
    const Repack16 r{src, lam, amax, L.chi_l, L.d, L.chi_r, L.Cs, L.K_pad, f16, hi, lo};
    const dim3 grid((unsigned)((L.chi_r + kRepackB - 1) / kRepackB), (unsigned)((L.chi_l + kRepackA - 1) / kRepackA),
                    (unsigned)L.d);
    if (L.chi_l % 8 == 0) repack16_kernel<kSource, true><<<grid, 256, 0, st>>>(r);
    else repack16_kernel<kSource, false><<<grid, 256, 0, st>>>(r);
}

void launch_repack_bf16(const void *src, int is_f64, const void *lam, const SiteLayout &L, __nv_bfloat16 *B_hi,
                        __nv_bfloat16 *B_lo, cudaStream_t st) {
    uint16_t *hi = reinterpret_cast<uint16_t *>(B_hi), *lo = reinterpret_cast<uint16_t *>(B_lo);
    if (is_f64) launch_repack16<kFromDouble>(src, lam, nullptr, 0, L, hi, lo, st);
    else launch_repack16<kFromFloat>(src, lam, nullptr, 0, L, hi, lo, st);
}

void launch_expand_bf16(const __nv_bfloat16 *compact, const SiteLayout &L, __nv_bfloat16 *B_hi, __nv_bfloat16 *B_lo,
                        cudaStream_t st) {
    launch_repack16<kFrom16>(compact, nullptr, nullptr, 0, L, reinterpret_cast<uint16_t *>(B_hi),
                             reinterpret_cast<uint16_t *>(B_lo), st);
}

void launch_repack_e4m3(const void *src, int is_f64, const SiteLayout &L, float scale, uint8_t *B8,
                        cudaStream_t st) {
    const int64_t total = (int64_t)L.ncols * L.K_pad;
    repack_e4m3_kernel<<<grid_for(total, 256), 256, 0, st>>>(src, is_f64, L.chi_l, L.d, L.chi_r, L.Cs, L.ncols,
                                                              L.K_pad, scale, B8);
}

void launch_repack_f16(const void *src, int is_f64, const void *lam, const float *amax, const SiteLayout &L,
                       uint16_t *B16, uint16_t *B16_lo, cudaStream_t st) {
    if (is_f64) launch_repack16<kFromDouble>(src, lam, amax, 1, L, B16, B16_lo, st);
    else launch_repack16<kFromFloat>(src, lam, amax, 1, L, B16, B16_lo, st);
}

void launch_absmax(const void *src, int is_f64, int64_t n_complex, int chi_r, const void *lam, float *out_dev,
                   cudaStream_t st) {
    cudaMemsetAsync(out_dev, 0, sizeof(float), st);
    const int64_t blocks = (2 * n_complex + 255) / 256;
    absmax_kernel<<<(unsigned)std::min<int64_t>(blocks, 152 * 8), 256, 0, st>>>(src, is_f64, 2 * n_complex, chi_r, lam,
                                                                             out_dev);
}

void launch_repack_f32(const void *src, int is_f64, const SiteLayout &L, float *Bt, cudaStream_t st) {
    const int64_t total = (int64_t)L.ncols * L.K_pad;
    repack_f32_kernel<<<grid_for(total, 256), 256, 0, st>>>(src, is_f64, L.chi_l, L.d, L.chi_r, L.Cs, L.ncols,
                                                             L.K_pad, Bt);
}

// ---------------------------------------------------------------------------
// Left boundary v_0 = [1]: row = [1, 0, ..., 0] (real part 1, imaginary 0).
// ---------------------------------------------------------------------------
// One 16-byte piece per thread; `one` is the bit pattern of 1 in column 0 (little-endian, in the first bytes).
__global__ void init_left_kernel(uint4 *__restrict__ V, int64_t rows, int ld, int cols, uint32_t one) {
    const int64_t total = rows * cols;  // ld, cols: in pieces
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / cols;
        const int c = (int)(i - r * cols);
        V[r * ld + c] = make_uint4(c == 0 ? one : 0u, 0u, 0u, 0u);
    }
}

static void init_left_plane(void *V, int64_t rows, int ld, int cols, int elem_bytes, uint32_t one, cudaStream_t st) {
    const int per = 16 / elem_bytes;  // ld and cols are multiples of 64
    init_left_kernel<<<grid_for(rows * (cols / per), 256), 256, 0, st>>>(static_cast<uint4 *>(V), rows, ld / per,
                                                                          cols / per, one);
}

void launch_init_left_f16(uint16_t *V0, uint16_t *V1, int64_t rows, int ld, int cols, cudaStream_t st) {
    init_left_plane(V0, rows, ld, cols, 2, 0x3C00u, st);
    init_left_plane(V1, rows, ld, cols, 2, 0u, st);
}

void launch_init_left_e4m3(uint8_t *V8, uint8_t *V8lo, int64_t rows, int ld, int cols, cudaStream_t st) {
    init_left_plane(V8, rows, ld, cols, 1, 0x38u, st);
    if (V8lo) init_left_plane(V8lo, rows, ld, cols, 1, 0u, st);
}

void launch_init_left_bf16(__nv_bfloat16 *const *Vp, int nplanes, int64_t rows, int ld, int cols, cudaStream_t st) {
    for (int p = 0; p < nplanes; ++p) init_left_plane(Vp[p], rows, ld, cols, 2, p ? 0u : 0x3F80u, st);
}

void launch_init_left_f32(float *V, int64_t rows, int ld, int cols, cudaStream_t st) {
    init_left_plane(V, rows, ld, cols, 4, 0x3F800000u, st);
}

// ---------------------------------------------------------------------------
// FP32 SIMT contraction (the plain path): Y = V Bt over a (16 TM) x 128 tile per block of 256 threads,
// TM x 8 outputs per thread.  Epilogue: store the tile to the FP32 scratch and one sum of squares per row
// (the tile lies inside one outcome block s).
//
// Chunked accumulation: each output sums its K = 2 chi_l products in chunks
// of F32_CHUNK, every chunk in its own FP32 accumulator that is then added to
// a running FP32 total.  One sequential FP32 sum over K = 2048 has a rounding
// error ~ sqrt(K) units in the last place of the result, and because the
// left vector's direction error is carried, not forgotten, along a chain of
// random isometries, those errors add up over the sites and surface in the
// last sites' conditionals; chunks of 64 cut the per-site error about five
// times (2.3e-5 -> 4.7e-6 at M = 1024, chi = 1024 in a CPU emulation of both
// orders).
//
// Bound by the FP32 pipes' operand reads: scalar fma of register operands levels off at 53 TFLOP/s without
// the totals (two thirds of 152 SMs x 128 lanes, whatever the tile, the lane layout or the shared-memory
// traffic), 46 with them.  So two outputs of neighbouring rows share one packed fma.rn.f32x2, whose repeated
// operand (b, b) is read once for TM/2 of them; each half is the correctly rounded fma of its own operands, in
// the order of a scalar loop.  The running totals live in shared memory, one private column per thread, and
// are touched once per chunk, so that two blocks fit an SM.  Fragments of the next K entry are loaded while
// the current ones are multiplied.  32768 rows, K = 512, 2048 columns: 1317 us, 52 TFLOP/s (60 without the
// totals; scalar, totals in registers, one block per SM: 1447 us).  Keeping every left entry twice in shared
// memory, to save the register copy of a packed operand, was slower (43 TFLOP/s).
// A tile whose last 64 columns are padding of its outcome block (2 chi_r <= 64 modulo 128) leaves them out:
// they are zero, add nothing to the sum of squares, and nothing reads them.
// ---------------------------------------------------------------------------
constexpr int F32_BN = 128, F32_THREADS = 256;
constexpr int F32_CHUNK = kF32Chunk;  // K is a multiple of it

template <int TM>
struct F32Tile {
    static constexpr int BM = 16 * TM;             // rows
    static constexpr int BK = TM == 8 ? 8 : 16;    // K entries per stage
    static constexpr int AK = BK * BM / F32_THREADS;  // left entries per thread and stage, along K
    static constexpr int RG = TM == 8 ? 4 : TM;    // consecutive rows per thread; TM = 8: again 64 rows on
    static constexpr int floats = 2 * BK * (BM + F32_BN) + BM * F32_BN;
    static constexpr size_t bytes = sizeof(float) * floats + 16;  // + the tile's place, for the epilogue
};

// One (16 TM) x (64 NQ) tile.  Thread (ty, tx) holds rows 64 g + RG ty + .. and columns 64 q + 4 tx .. + 3.
template <int TM, int NQ>
__device__ __forceinline__ void contract_f32_tile(const float *__restrict__ Ag, int64_t ldV,
                                                  const float *__restrict__ Bg, int ldB, int K,
                                                  float *__restrict__ Y, int64_t ldY, float *__restrict__ P, int ldP,
                                                  int rows_valid, float *smem) {
    using T = F32Tile<TM>;
    constexpr int BM = T::BM, BK = T::BK, AK = T::AK, RG = T::RG, NP = TM / 2, NC = 4 * NQ;
    float *As = smem;                                // [2][BK][BM]
    float *Bs = As + 2 * BK * BM;                    // [2][BK][128]
    ulonglong2 *tot = reinterpret_cast<ulonglong2 *>(Bs + 2 * BK * F32_BN);  // [NP * NC / 2][threads]
    const int tid = threadIdx.x;
    const int a_row = tid % BM, a_k = tid / BM * AK;
    const int ty = tid >> 4, tx = tid & 15;
    const float *ap = Ag + (int64_t)a_row * ldV + a_k;

    float ra[AK];
    auto load_a = [&](int k0) {
        if constexpr (AK == 4) {
            const float4 v = *reinterpret_cast<const float4 *>(ap + k0);
            ra[0] = v.x, ra[1] = v.y, ra[2] = v.z, ra[3] = v.w;
        } else {
            const float2 v = *reinterpret_cast<const float2 *>(ap + k0);
            ra[0] = v.x, ra[1] = v.y;
        }
    };
    auto store_a = [&](int buf) {
#pragma unroll
        for (int e = 0; e < AK; ++e) As[(buf * BK + a_k + e) * BM + a_row] = ra[e];
    };
    auto copy_b = [&](int buf, int k0) {
#pragma unroll
        for (int id = tid; id < BK * 16 * NQ; id += F32_THREADS) {
            const int r = id / (16 * NQ), c = id % (16 * NQ) * 4;
            cp_async16(Bs + (buf * BK + r) * F32_BN + c, Bg + (int64_t)(k0 + r) * ldB + c);
        }
        cp_async_commit();
    };
    f32x2 a[2][NP];
    float b[2][NC];
    auto load_fragments = [&](int f, int buf, int kk) {
        const float *A = As + (buf * BK + kk) * BM + ty * RG, *B = Bs + (buf * BK + kk) * F32_BN + tx * 4;
        if constexpr (RG == 2) {
            a[f][0] = *reinterpret_cast<const f32x2 *>(A);
        } else {
#pragma unroll
            for (int g = 0; g < TM / RG; ++g) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(A + 64 * g);
                a[f][2 * g] = v.x;
                a[f][2 * g + 1] = v.y;
            }
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float4 v = *reinterpret_cast<const float4 *>(B + 64 * q);
            b[f][4 * q] = v.x, b[f][4 * q + 1] = v.y, b[f][4 * q + 2] = v.z, b[f][4 * q + 3] = v.w;
        }
    };

    load_a(0);
    copy_b(0, 0);
    store_a(0);
    cp_async_wait<0>();
    __syncthreads();

    f32x2 acc[NC][NP];
#pragma unroll
    for (int j = 0; j < NC; ++j)
#pragma unroll
        for (int i = 0; i < NP; ++i) acc[j][i] = 0ull;
    load_fragments(0, 0, 0);
    const int nk = K / BK;
    for (int k0 = 0; k0 < nk; k0 += F32_CHUNK / BK) {
#pragma unroll 1
        for (int kt = k0; kt < k0 + F32_CHUNK / BK; ++kt) {
            const int cur = kt & 1;
            if (kt + 1 < nk) {
                load_a((kt + 1) * BK);
                copy_b(cur ^ 1, (kt + 1) * BK);
            }
#pragma unroll
            for (int kk = 0; kk < BK; ++kk) {
                if (kk + 1 < BK) {
                    load_fragments((kk + 1) & 1, cur, kk + 1);
                } else {
                    if (kt + 1 < nk) {
                        store_a(cur ^ 1);
                        cp_async_wait<0>();
                    }
                    __syncthreads();
                    if (kt + 1 < nk) load_fragments(0, cur ^ 1, 0);
                }
#pragma unroll
                for (int j = 0; j < NC; ++j) {
                    const f32x2 bb = twice_f32x2(b[kk & 1][j]);
#pragma unroll
                    for (int i = 0; i < NP; ++i) fma_f32x2(acc[j][i], a[kk & 1][i], bb);
                }
            }
        }
        // end of a K chunk: fold its partial sums into the running totals (into acc after the last one),
        // eight loads in flight
        const bool first = k0 == 0, last = k0 + F32_CHUNK / BK == nk;
        constexpr int NE = NP * NC / 2, G = NE < 8 ? NE : 8;
#pragma unroll
        for (int e0 = 0; e0 < NE; e0 += G) {
            if (!first) {
                ulonglong2 t[G];
#pragma unroll
                for (int g = 0; g < G; ++g) t[g] = tot[(e0 + g) * F32_THREADS + tid];
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const int e = 2 * (e0 + g);
                    acc[e / NP][e % NP] = add_f32x2(t[g].x, acc[e / NP][e % NP]);
                    acc[(e + 1) / NP][(e + 1) % NP] = add_f32x2(t[g].y, acc[(e + 1) / NP][(e + 1) % NP]);
                }
            }
            if (!last) {
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const int e = 2 * (e0 + g);
                    tot[(e0 + g) * F32_THREADS + tid] =
                        make_ulonglong2(acc[e / NP][e % NP], acc[(e + 1) / NP][(e + 1) % NP]);
                    acc[e / NP][e % NP] = acc[(e + 1) / NP][(e + 1) % NP] = 0ull;
                }
            }
        }
    }

    // (the tile's place is read back here, so that it takes no registers from the loop)
    const int *place = reinterpret_cast<const int *>(smem + T::floats);
    const int m0 = place[0] * BM, rows_left = rows_valid - m0;
    Y += (int64_t)m0 * ldY + (int64_t)place[1] * F32_BN;
    P += (int64_t)m0 * ldP + place[1];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int r = 64 * (i / RG) + ty * RG + i % RG;
        float ss = 0.f, out[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            const float2 v = unpack_f32x2(acc[j][i / 2]);
            out[j] = i & 1 ? v.y : v.x;
            ss = fmaf(out[j], out[j], ss);
        }
        ss += __shfl_xor_sync(0xffffffffu, ss, 1);
        ss += __shfl_xor_sync(0xffffffffu, ss, 2);
        ss += __shfl_xor_sync(0xffffffffu, ss, 4);
        ss += __shfl_xor_sync(0xffffffffu, ss, 8);
        if (r < rows_left) {
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                *reinterpret_cast<float4 *>(Y + (int64_t)r * ldY + 64 * q + tx * 4) =
                    make_float4(out[4 * q], out[4 * q + 1], out[4 * q + 2], out[4 * q + 3]);
            if (tx == 0) P[(int64_t)r * ldP] = ss;
        }
    }
}

template <int TM>
__global__ void __launch_bounds__(F32_THREADS, 2)
contract_f32_kernel(const float *__restrict__ V, int64_t ldV, int64_t row0, const float *__restrict__ Bt, int ldB,
                    int K, float *__restrict__ Y, int64_t ldY, float *__restrict__ P, int ldP, int rows_valid,
                    int tiles_per_s, int nreal, int num_m) {
    extern __shared__ __align__(16) float f32_smem[];
    constexpr int BM = F32Tile<TM>::BM;
    // Tiles with 64 padding columns (the last of each outcome, `half` of them per row of tiles) cost half of the
    // others and come last: an SM that has a whole tile gets a half one with it.  In the order of the columns some
    // SMs got two whole tiles and others two half ones (d = 6, chi = 90, 3001 rows, 288 tiles: 32 sites in 1.74 ms,
    // 1.95 in that order).
    const int T = tiles_per_s, nx = ldB / F32_BN, half = nreal - (T - 1) * F32_BN <= 64 ? nx / T : 0;
    const int whole = nx - half, id = blockIdx.x, first_half = whole * num_m;
    int m, n;
    if (id < first_half) {
        m = id / whole;
        const int j = id - m * whole;
        n = half ? j / (T - 1) * T + j % (T - 1) : j;
    } else {
        m = (id - first_half) / half;
        n = (id - first_half - m * half) * T + T - 1;
    }
    if (threadIdx.x == 0) {
        int *place = reinterpret_cast<int *>(f32_smem + F32Tile<TM>::floats);
        place[0] = m;
        place[1] = n;
    }
    const float *Ag = V + (row0 + (int64_t)m * BM) * ldV, *Bg = Bt + (int64_t)n * F32_BN;
    if (id < first_half) contract_f32_tile<TM, 2>(Ag, ldV, Bg, ldB, K, Y, ldY, P, ldP, rows_valid, f32_smem);
    else contract_f32_tile<TM, 1>(Ag, ldV, Bg, ldB, K, Y, ldY, P, ldP, rows_valid, f32_smem);
}

void launch_contract_f32(const float *V, int64_t ldV, int64_t row0, const float *Bt, const SiteLayout &L,
                         const ContractOut &o, int num_sms, cudaStream_t st) {
    // 128-row tiles, unless 64- or 32-row tiles still fit one per SM: a lone block per SM runs at half the
    // pace of two, and a shorter tile ends sooner.  Measured, us (128 / 64 / 32 rows): d = 4, chi = 256,
    // 64 rows: 66 / 39 / 33; 512 rows: 66 / 39 / 58; 1024 rows: 66 / 68 / 109.  128 rows at most, so that no
    // tile reaches past the left operand's rows (a multiple of 128).
    const int64_t nx = L.ncols / F32_BN;
    auto run = [&](auto tm) {
        using T = F32Tile<decltype(tm)::value>;
        auto kern = contract_f32_kernel<decltype(tm)::value>;
        if (T::bytes > 48 * 1024)
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::bytes);
        const int64_t num_m = (o.rows_valid + T::BM - 1) / T::BM;
        kern<<<(unsigned)(nx * num_m), F32_THREADS, T::bytes, st>>>(V, ldV, row0, Bt, L.ncols, L.K_pad, o.Y, o.ldY, o.P,
                                                                    o.ldP, o.rows_valid, L.tiles_per_s, 2 * L.chi_r,
                                                                    (int)num_m);
    };
    if (nx * ((o.rows_valid + 31) / 32) <= num_sms) run(std::integral_constant<int, 2>());
    else if (nx * ((o.rows_valid + 63) / 64) <= num_sms) run(std::integral_constant<int, 4>());
    else run(std::integral_constant<int, 8>());
}

// ---------------------------------------------------------------------------
// Stand-alone measurement: a block of four warps takes R rows.  First the w_s of its rows, one thread per
// (row, outcome); then one thread per row draws; then all threads write the rows; the logarithm comes last.
// Bound by HBM: one selected block read and one next row written per sample.  131072 rows of 512 entries
// (d = 4, BF16 planes): 94 us = 5.8 TB/s; 65536 rows of 2048 entries: 180 us = 6.0 TB/s in BF16 planes,
// 201 us in FP16.  (One warp for 32 rows in turn, its draw included: 110, -- and 516 us; and 398 us against
// 24 where a call has 5003 rows of 1554 entries, because 157 warps were all there was.)
// ---------------------------------------------------------------------------
constexpr int MEASURE_THREADS = 128;
constexpr int MEASURE_ROWS = 32;    // most rows of a block
constexpr int MEASURE_SUMS = 1024;  // most (row, outcome) sums of a block

// kScaled: FP16 or E4M3 rows (one warp per row), else FP32 or BF16 planes
template <bool kScaled>
__global__ void __launch_bounds__(MEASURE_THREADS) measure_kernel(const MeasureArgs a, int R) {
    __shared__ double w_sh[MEASURE_SUMS];
    __shared__ int sstar_sh[MEASURE_ROWS];
    __shared__ float scale_sh[MEASURE_ROWS];
    const int tid = threadIdx.x, lane = tid & 31;
    const int r0 = blockIdx.x * R;
    const int count = min(R, a.rows - r0);
    const int T = a.tiles_per_s, d = a.d;
    for (int q = tid; q < count * d; q += MEASURE_THREADS) {
        const int r = q / d, s = q - r * d;
        w_sh[q] = sum_tiles(a.P + (int64_t)(r0 + r) * a.ldP + s * T, T);
    }
    double u = 0.0, lp = 0.0;
    if (tid < count) {
        u = sample_uniform(a.seed, a.n_base + (uint64_t)(r0 + tid), a.k, a.job);
        lp = a.logp[a.row0 + r0 + tid];
    }
    __syncthreads();
    double Z = 0.0, ws = 0.0;
    bool ok = false;
    const RowSums w{w_sh + tid * d, nullptr, d, T};
    if (tid < count) {
        const int sstar = draw_row(w, u, &Z, &ws, &ok);
        sstar_sh[tid] = sstar;
        scale_sh[tid] = ok ? rsqrtf((float)ws) : 0.f;
        a.outcomes[r0 + tid] = (uint8_t)sstar;
    }
    __syncthreads();
    if constexpr (!kScaled) {
        write_rows_flat<1>(a, tid, MEASURE_THREADS, r0, count, sstar_sh, scale_sh);
    } else {
        for (int j = tid >> 5; j < count; j += MEASURE_THREADS / 32)
            write_row_scaled(a, lane, a.Y + (int64_t)(r0 + j) * a.ldY + (int64_t)sstar_sh[j] * a.Cs, scale_sh[j],
                             a.row0 + r0 + j);
    }
    // nothing waits for the logarithm: it follows the row writes
    if (tid < count) measure_finish(a, r0 + tid, ws, Z, ok, lp, w);
}

void launch_measure(const MeasureArgs &a, int num_sms, cudaStream_t st) {
    if (a.rows <= 0) return;
    // Rows per block: a warp's worth, so that the FP64 draw (a warp-wide FP64 instruction costs the SM 16
    // cycles however many lanes it has) stays a small part; fewer where rows are wide (65536 rows of 2048
    // entries: 204 us with 32 rows per block, 180 with 16) or where that would leave less than four blocks
    // per SM (5003 rows of 1554 entries: 60 us with 32, 24 with 8); at most MEASURE_SUMS sums.
    int R = MEASURE_ROWS;
    while (R > 4 && (R * a.K_next > 32768 || (a.rows + R - 1) / R < 4 * num_sms || R * a.d > MEASURE_SUMS)) R >>= 1;
    const int grid = (a.rows + R - 1) / R;
    if (a.f16 || a.V8) measure_kernel<true><<<grid, MEASURE_THREADS, 0, st>>>(a, R);
    else measure_kernel<false><<<grid, MEASURE_THREADS, 0, st>>>(a, R);
}

// ---------------------------------------------------------------------------
// Outcomes are produced site-major (coalesced writes per site); the caller
// wants sample-major rows.  32 x 32 byte tiles through shared memory.
// ---------------------------------------------------------------------------
__global__ void transpose_u8_kernel(const uint8_t *__restrict__ O, int64_t ldO, int64_t N, int M,
                                    uint8_t *__restrict__ out) {
    __shared__ uint8_t t[32][33];
    const int64_t n0 = (int64_t)blockIdx.x * 32;
    const int k0 = blockIdx.y * 32;
    for (int j = threadIdx.y; j < 32; j += blockDim.y) {
        const int k = k0 + j;
        const int64_t n = n0 + threadIdx.x;
        if (k < M && n < N) t[j][threadIdx.x] = O[(int64_t)k * ldO + n];
    }
    __syncthreads();
    for (int j = threadIdx.y; j < 32; j += blockDim.y) {
        const int64_t n = n0 + j;
        const int k = k0 + threadIdx.x;
        if (k < M && n < N) out[n * M + k] = t[threadIdx.x][j];
    }
}

void launch_transpose_outcomes(const uint8_t *O, int64_t ldO, int64_t N, int M, uint8_t *out, cudaStream_t st) {
    if (N <= 0 || M <= 0) return;
    dim3 grid((unsigned)((N + 31) / 32), (unsigned)((M + 31) / 32));
    transpose_u8_kernel<<<grid, dim3(32, 8), 0, st>>>(O, ldO, N, M, out);
}

}  // namespace fastmps

namespace fastmps {

// Self-test of the bounded wait used by the pipelined kernels: waits on an
// mbarrier that nothing ever arrives on; the wait gives up after limit_ns and
// the kernel records kDevTimeoutProducer and returns (no fault, no hang).
__global__ void bounded_wait_selftest_kernel(uint64_t limit_ns, int *status, unsigned long long *waited_ns) {
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint64_t t0 = global_ns();
        const bool ok = mbar_wait_bounded(&bar, 0u, &abort_flag, limit_ns);
        *waited_ns = global_ns() - t0;
        *status = ok ? kDevOk : kDevTimeoutProducer;
    }
}

void launch_bounded_wait_selftest(uint64_t limit_ns, int *status, unsigned long long *waited_ns, cudaStream_t st) {
    bounded_wait_selftest_kernel<<<1, 32, 0, st>>>(limit_ns, status, waited_ns);
}

}  // namespace fastmps
