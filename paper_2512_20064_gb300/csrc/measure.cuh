// Measurement step shared by the stand-alone measurement kernel and the
// measurement warps fused into the tcgen05 contraction (device code, internal).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <stdint.h>

#include "common.cuh"
#include "launch.h"

namespace fastmps {

// ---------------------------------------------------------------------------
// Measurement (Algorithm 2 with the exact per-sample rescaling of Sec. 3.3.1).
// Phase 1, one thread per sample (draw_row, measure_finish):
//  * w_s = sum of the FP32 per-tile sums of squares of outcome block s,
//    accumulated in FP64;
//  * C_s = w_0 + ... + w_s in s order (FP64), Z = C_{d-1}, Philox uniform u,
//    s* = #{s < d-1 : C_s < u Z}: the decision is taken in FP64 as in the
//    oracle;
//  * log p accumulates log(w_{s*} / Z) in FP64: the ratio and its logarithm
//    are taken in FP64 (one log per sample per site, O(N M) work), since a
//    rare outcome has w_{s*} << 1 and the absolute error of an FP32 log
//    there would add up over thousands of sites.
// Phase 2, a group of warps for a group of rows (measure_write_rows): the selected block y_{s*} of
// each row is scaled by 1/sqrt(w_{s*}) (FP32; the scale cancels in every later ratio w/Z) and
// written as the next left row -- FP32, or BF16 planes of successive residuals -- with coalesced
// 32-byte loads.  FP16 and E4M3 rows, whose power-of-two scale comes from the row's largest entry, are
// read twice by one warp.
// GB300's FP64 pipes are narrow, so FP64 is kept to the O(d) per-sample
// operations of the draw and the accumulation, one sample per lane.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void write_planes(float x, int nplanes, __nv_bfloat16 &h0, __nv_bfloat16 &h1,
                                             __nv_bfloat16 &h2) {
    h0 = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(h0);
    h1 = __float2bfloat16_rn(r1);
    h2 = __float2bfloat16_rn(r1 - __bfloat162float(h1));
    if (nplanes < 3) h2 = __float2bfloat16_rn(0.f);
}

// Eight entries (columns i .. i+7, i a multiple of 8) of a selected block; zero at and beyond nreal.
// One 32-byte load through L2 (the block may have been written by other thread blocks of the same
// kernel).  A block's columns are padded to a multiple of 32 (SiteLayout::Cs), so the load at i < nreal
// stays inside the block, and is 32-byte aligned, for any nreal.
struct Entries8 {
    float x[8];
};

__device__ __forceinline__ Entries8 load_block8(const float *ysrc, int i, int nreal) {
    Entries8 v;
    if (i >= nreal) {
#pragma unroll
        for (int e = 0; e < 8; ++e) v.x[e] = 0.f;
        return v;
    }
    asm volatile("ld.global.cg.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v.x[0]), "=f"(v.x[1]), "=f"(v.x[2]), "=f"(v.x[3]), "=f"(v.x[4]), "=f"(v.x[5]), "=f"(v.x[6]),
                   "=f"(v.x[7])
                 : "l"(ysrc + i)
                 : "memory");
    if (i + 7 >= nreal) {
#pragma unroll
        for (int e = 1; e < 8; ++e)
            if (i + e >= nreal) v.x[e] = 0.f;
    }
    return v;
}

// Entries i .. i+7 of a next left row in FP32 or BF16 planes (off: element offset of entry i).
__device__ __forceinline__ void store_row8(const MeasureArgs &a, int64_t off, const Entries8 &v, float scale) {
    if (a.V32) {
        float4 *dst = reinterpret_cast<float4 *>(a.V32 + off);
        dst[0] = make_float4(v.x[0] * scale, v.x[1] * scale, v.x[2] * scale, v.x[3] * scale);
        dst[1] = make_float4(v.x[4] * scale, v.x[5] * scale, v.x[6] * scale, v.x[7] * scale);
        return;
    }
    __align__(16) __nv_bfloat16 p0[8], p1[8], p2[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) write_planes(v.x[e] * scale, a.nplanes, p0[e], p1[e], p2[e]);
    *reinterpret_cast<uint4 *>(a.Vp[0] + off) = *reinterpret_cast<const uint4 *>(p0);
    *reinterpret_cast<uint4 *>(a.Vp[1] + off) = *reinterpret_cast<const uint4 *>(p1);
    if (a.nplanes > 2) *reinterpret_cast<uint4 *>(a.Vp[2] + off) = *reinterpret_cast<const uint4 *>(p2);
}

// Next left rows of micro-batch rows r0 .. r0+count-1 (FP32 or BF16 planes) by `nt` threads: the rows'
// 8-entry pieces are dealt to the threads in order, U of them in flight per thread, so threads stay busy
// whether rows are 64 or 4096 entries wide.  sstar, scale: per row.  Pieces of 8 entries make every load 32
// bytes and every BF16 plane store 16 bytes.
// U = 1 where many blocks share an SM: more in flight per thread costs registers, so resident warps, and
// gains nothing (131072 rows of 512 entries, 32 rows per block: 94 us, 98 with two; 137 us with four pieces
// of 4 entries).  U = 8 where four warps are all an SM has for the measurement.
template <int U>
__device__ __forceinline__ void write_rows_flat(const MeasureArgs &a, int tid, int nt, int r0, int count,
                                                const int *sstar, const float *scale) {
    const int nreal = 2 * a.chi_r;
    const int per_row = a.K_next >> 3;
    const int step_r = nt / per_row, step_c = nt - step_r * per_row;
    int r = tid / per_row, c = tid - r * per_row;
    while (r < count) {
        Entries8 v[U];
        int rr[U], cc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            rr[u] = r;
            cc[u] = 8 * c;
            if (r < count)
                v[u] = load_block8(a.Y + (int64_t)(r0 + r) * a.ldY + (int64_t)sstar[r] * a.Cs, 8 * c, nreal);
            r += step_r;
            c += step_c;
            if (c >= per_row) {
                c -= per_row;
                ++r;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (rr[u] >= count) break;
            store_row8(a, (a.row0 + r0 + rr[u]) * (int64_t)a.ld_next + cc[u], v[u], scale[rr[u]]);
        }
    }
}

// One FP16 or E4M3 next left row by one warp, read twice (for its largest entry, then for the entries;
// the second read hits L2) in pieces of 512 entries; a row of one piece stays in registers.  Holding up to
// 2048 entries in registers instead takes 229 us, not 201, for 65536 rows of 2048 entries: fewer warps are
// resident.  The unit-norm row is scaled by the power of two that puts its largest entry in [top/2, top] -- top = 32768 for binary16, 448 for E4M3 -- which cancels
// in w/Z at the next site and keeps small entries normal; then
//   FP16: two binary16 planes of successive residuals, each rounded to nearest even;
//   E4M3: one plane, or two with the residual at the same scale (the products add up to (V0 + V1) B).
__device__ __forceinline__ void store_scaled8(const MeasureArgs &a, int64_t off, const Entries8 &v, float s2) {
    if (a.f16) {
        __align__(16) uint16_t h0[8], h1[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float x = v.x[e] * s2;
            const __half h = __float2half_rn(x);
            h0[e] = __half_as_ushort(h);
            h1[e] = __half_as_ushort(__float2half_rn(x - __half2float(h)));
        }
        *reinterpret_cast<uint4 *>(a.Vp[0] + off) = *reinterpret_cast<const uint4 *>(h0);
        *reinterpret_cast<uint4 *>(a.Vp[1] + off) = *reinterpret_cast<const uint4 *>(h1);
        return;
    }
    __align__(8) uint8_t q0[8], q1[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const float x = v.x[e] * s2;
        const __nv_fp8_storage_t h = __nv_cvt_float_to_fp8(x, __NV_SATFINITE, __NV_E4M3);
        q0[e] = (uint8_t)h;
        const float hv = __half2float(__half(__nv_cvt_fp8_to_halfraw(h, __NV_E4M3)));
        q1[e] = (uint8_t)__nv_cvt_float_to_fp8(x - hv, __NV_SATFINITE, __NV_E4M3);
    }
    *reinterpret_cast<uint2 *>(a.V8 + off) = *reinterpret_cast<const uint2 *>(q0);
    if (a.V8lo) *reinterpret_cast<uint2 *>(a.V8lo + off) = *reinterpret_cast<const uint2 *>(q1);
}

__device__ __forceinline__ void write_row_scaled(const MeasureArgs &a, int lane, const float *ysrc, float scale,
                                                 int64_t grow) {
    constexpr int NV = 2;  // 8-entry pieces per lane
    const int nreal = 2 * a.chi_r;
    const int64_t off = grow * a.ld_next;
    Entries8 v[NV];
    float m = 0.f;
    auto take = [&](int base) {
#pragma unroll
        for (int u = 0; u < NV; ++u) v[u] = load_block8(ysrc, base + 8 * lane + 256 * u, nreal);
#pragma unroll
        for (int u = 0; u < NV; ++u)
#pragma unroll
            for (int e = 0; e < 8; ++e) v[u].x[e] *= scale;
    };
    auto put = [&](int base, float s2) {
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int i = base + 8 * lane + 256 * u;
            if (i >= a.K_next) break;
            store_scaled8(a, off + i, v[u], s2);
        }
    };
    const bool one_piece = a.K_next <= 256 * NV;
    for (int base = 0; base < nreal; base += 256 * NV) {
        take(base);
#pragma unroll
        for (int u = 0; u < NV; ++u)
#pragma unroll
            for (int e = 0; e < 8; ++e) m = fmaxf(m, fabsf(v[u].x[e]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const float s2 = m > 0.f ? exp2f(floorf(log2f((a.f16 ? 32768.f : 448.f) / m))) : 1.f;
    if (one_piece) {
        put(0, s2);
    } else {
        for (int base = 0; base < a.K_next; base += 256 * NV) {
            take(base);
            put(base, s2);
        }
    }
}

// Next left rows of micro-batch rows r0 .. r0+count-1 by `nt` threads (whole warps), any precision.
__device__ __forceinline__ void measure_write_rows(const MeasureArgs &a, int tid, int nt, int r0, int count,
                                                   const int *sstar, const float *scale) {
    if (a.f16 || a.V8) {
        for (int j = tid >> 5; j < count; j += nt >> 5)
            write_row_scaled(a, tid & 31, a.Y + (int64_t)(r0 + j) * a.ldY + (int64_t)sstar[j] * a.Cs, scale[j],
                                a.row0 + r0 + j);
        return;
    }
    write_rows_flat<8>(a, tid, nt, r0, count, sstar, scale);
}

// w_s of one row: the FP64 sum, in tile order, of its T per-tile sums of squares.  P is read through L2
// (it may have been written by other thread blocks of the same kernel), eight loads in flight.
__device__ __forceinline__ double sum_tiles(const float *P, int T) {
    double acc = 0.0;
    for (int j = 0; j < T; j += 8) {
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = j + e < T ? __ldcg(P + j + e) : 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (j + e < T) acc += (double)x[e];
    }
    return acc;
}

// Calls f(s, w_s) for s = 0 .. d-1 until it returns true, the sums as in sum_tiles.  The d T values of a row are
// contiguous: 16 loads in flight, whatever T is (one thread has the whole row, and each load takes most of a
// microsecond).
template <class F>
__device__ __forceinline__ void each_outcome_sum(const float *P, int d, int T, F f) {
    const int n = d * T;
    double acc = 0.0;
    int s = 0, left = T;
    for (int j = 0; j < n; j += 16) {
        float x[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) x[e] = j + e < n ? __ldcg(P + j + e) : 0.f;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            if (j + e >= n) break;
            acc += (double)x[e];
            if (--left == 0) {
                if (f(s, acc)) return;
                acc = 0.0;
                left = T;
                ++s;
            }
        }
    }
}

// The sums w_s of one row: in shared memory (w), or still as per-tile sums in P.
struct RowSums {
    const double *w;
    const float *P;
    int d, T;
    template <class F>
    __device__ __forceinline__ void each(F f) const {
        if (w) {
            for (int s = 0; s < d; ++s)
                if (f(s, w[s])) return;
        } else {
            each_outcome_sum(P, d, T, f);
        }
    }
};

// The draw of one row (FP64, in s order): Z = w_0 + ... + w_{d-1}; s* is the first s < d-1 with
// C_s >= u Z (else d-1), which equals #{s < d-1 : C_s < u Z} because C is non-decreasing.
__device__ __forceinline__ int draw_row(const RowSums &row, double u, double *Z_out, double *ws_out, bool *ok_out) {
    double Z = 0.0;
    row.each([&](int, double w) {
        Z += w;
        return false;
    });
    const double t = u * Z;
    double C = 0.0, ws = 0.0;
    int sstar = row.d - 1;
    row.each([&](int s, double w) {
        C += w;
        if (s < row.d - 1 && !(C >= t)) return false;
        sstar = s;
        ws = w;
        return true;
    });
    *Z_out = Z;
    *ws_out = ws;
    *ok_out = (Z > 0.0) && isfinite(Z) && (ws > 0.0);
    return sstar;
}

// Log-probability, numeric check and optional trace of one drawn row.
__device__ __forceinline__ void measure_finish(const MeasureArgs &a, int row, double ws, double Z, bool ok, double lp,
                                               const RowSums &w) {
    const int64_t grow = a.row0 + row;
    if (ok) a.logp[grow] = lp + log(ws / Z);
    else atomicExch(a.err, (int)kDevNumeric);
    const int64_t slot = a.trace ? (a.trace_slot ? (int64_t)a.trace_slot[grow] : (grow < a.trace_rows ? grow : -1))
                                 : -1;
    if (slot >= 0)
        w.each([&](int s, double x) {
            a.trace[slot * a.d + s] = ok ? x / Z : 0.0;
            return false;
        });
}

// Phase 1 for sample `row` of the micro-batch (row < a.rows) by one thread: draw, outcome,
// log-probability, optional trace.  Returns the outcome and sets *scale to 1/sqrt(w_{s*}).
__device__ __forceinline__ int measure_draw(const MeasureArgs &a, int row, float *scale_out) {
    const RowSums w{nullptr, a.P + (int64_t)row * a.ldP, a.d, a.tiles_per_s};
    double Z, ws;
    bool ok;
    const int sstar = draw_row(w, sample_uniform(a.seed, a.n_base + (uint64_t)row, a.k, a.job), &Z, &ws, &ok);
    a.outcomes[row] = (uint8_t)sstar;
    measure_finish(a, row, ws, Z, ok, a.logp[a.row0 + row], w);
    *scale_out = ok ? rsqrtf((float)ws) : 0.f;
    return sstar;
}

}  // namespace fastmps
