// FP32 sampling of a whole chain in one launch, for calls whose sites are too small to pay for two launches
// each.
//
// A block of 256 threads takes 32 rows through every site.  Its left rows, the contracted rows and the
// per-tile sums of squares stay in shared memory; only the site tensors are read (from L2, by every block)
// and only the outcomes and log-probabilities are written.  No block waits for another.
//
// Bound by latency for narrow chains (three barriers, an FP64 draw and at least one pipeline stage per site:
// 3 to 5 us), by shared-memory reads of the site operand for wider ones.  The site operand is copied with
// cp.async in stages of 16 K-entries x 128 columns, four in flight, and the copies run ahead over tiles and
// sites: a site's tensor does not depend on what was drawn.  Each thread holds two neighbouring rows x 8
// columns (packed fma.rn.f32x2, see contract_f32_tile).
//
// Same bits as the two-kernel path (contract_f32_kernel, measure_kernel): every output sums its products in
// the same order in the same chunks, every tile's sum of squares has the same tree, the draw takes the same
// FP64 sums.  K entries that are padding (zeros on both sides) are left out.  The FP64 logarithms are taken
// for 32 sites at a time, one per thread, and added in site order.
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "f32x2.cuh"
#include "launch.h"

namespace fastmps {

namespace {

constexpr int kRows = 32;        // rows per block
constexpr int kThreads = 256;
constexpr int kBK = 16;          // K entries per stage
constexpr int kStages = 4;
constexpr int kVld = kRows + 2;  // left rows, transposed: [K][kVld] (8-byte aligned row pairs)
constexpr int kLogs = 32;        // sites whose logarithms are taken together

// Byte offsets of the block's shared-memory arrays.
struct ChainSmem {
    int v, y, p, w, u, sums, sstar, scale, total;
};

__host__ __device__ inline ChainSmem chain_smem(int k_max, int y_ld, int p_ld, int d) {
    ChainSmem s;
    int at = kStages * kBK * 128 * 4;  // the stages come first
    s.w = at, at += d * kRows * 8;
    s.u = at, at += 2 * kRows * 8;
    s.sums = at, at += kLogs * 2 * kRows * 8;
    s.y = at, at += kRows * y_ld * 4;
    s.v = at, at += k_max * kVld * 4;
    s.p = at, at += kRows * p_ld * 4;
    s.sstar = at, at += kRows * 4;
    s.scale = at, at += kRows * 4;
    s.total = at;
    return s;
}

struct ChainParams {
    const ChainSite *sites;
    int M, d, k_max, y_ld, p_ld;
    int64_t rows;
    uint64_t seed, n0;
    uint32_t job;
    uint8_t *samples;  // [rows][M] or null
    double *logp;      // [rows]
    double *trace;     // [M][trace_rows][d] or null
    int64_t trace_rows;
    const int *trace_slot;
    int *err;
};

// A unit is 128 columns of work: one 128-column tile of the operand (the last tile of an outcome block may
// need its first 64 columns only), or, where an outcome block has at most 64 columns that are not padding,
// 128 / Wb outcome blocks side by side, Wb = 16, 32 or 64 columns each.
struct Units {
    int Wb;     // columns of an outcome block in a unit, 0: one tile per unit
    int count;  // units of the site
};

__host__ __device__ inline Units units_of(const ChainSite &s, int d) {
    Units u;
    u.Wb = s.nreal > 64 ? 0 : s.nreal > 32 ? 64 : s.nreal > 16 ? 32 : 16;
    u.count = u.Wb ? (d * u.Wb + 127) / 128 : d * s.tiles_per_s;
    return u;
}
// Whether columns 64 .. 127 of unit j hold anything.
__host__ __device__ inline bool unit_is_wide(const ChainSite &s, const Units &u, int d, int j) {
    return u.Wb ? d * u.Wb - j * 128 > 64 : s.nreal - (j % s.tiles_per_s) * 128 > 64;
}

// The block's copies of the site operands, in the order they are used: (site, unit, K stage).
struct Copier {
    const ChainSite *sites;
    float *ring;
    int M, d;
    int k = 0, j = 0, t = 0, slot = 0;
    ChainSite s, ahead;  // the site being copied, and the one after it
    Units u;

    __device__ __forceinline__ void start() {
        s = sites[0];
        ahead = sites[M > 1 ? 1 : 0];
        u = units_of(s, d);
    }
    // One stage (nothing past the last one); always commits a group.
    __device__ __forceinline__ void next() {
        if (k < M) {
            const int r = threadIdx.x >> 4, c = (threadIdx.x & 15) * 4;
            float *dst = ring + (slot * kBK + r) * 128 + c;
            const float *src = s.Bt + (int64_t)(t * kBK + r) * s.ldB;
            if (u.Wb) {
                const int c0 = j * 128 + c, c1 = c0 + 64, s0 = c0 / u.Wb, s1 = c1 / u.Wb;
                if (s0 < d) cp_async16(dst, src + s0 * 128 + (c0 & (u.Wb - 1)));
                if (s1 < d) cp_async16(dst + 64, src + s1 * 128 + (c1 & (u.Wb - 1)));
            } else {
                cp_async16(dst, src + j * 128 + c);
                if (unit_is_wide(s, u, d, j)) cp_async16(dst + 64, src + j * 128 + c + 64);
            }
            if (++t == s.K / kBK) {
                t = 0;
                if (++j == u.count) {
                    j = 0;
                    ++k;
                    s = ahead;
                    ahead = sites[k + 1 < M ? k + 1 : M - 1];
                    u = units_of(s, d);
                }
            }
            slot = slot + 1 == kStages ? 0 : slot + 1;
        }
        cp_async_commit();
    }
};

// One 32 x (64 NQ) unit from V (shared, transposed) and the staged operand; leaves the outputs in out[row][col]
// of the thread's rows 2 ty, 2 ty + 1 and columns 64 q + 4 tx .. + 3.
template <int NQ>
__device__ __forceinline__ void chain_tile(Copier &copier, int &slot, const float *ring, const float *V, int K, int ty,
                                           int tx, float (&out)[2][8]) {
    f32x2 acc[4 * NQ], tot[4 * NQ];
#pragma unroll
    for (int j = 0; j < 4 * NQ; ++j) acc[j] = tot[j] = 0ull;
    for (int t = 0; t < K / kBK; ++t) {
        cp_async_wait<kStages - 2>();
        __syncthreads();  // this stage has landed for everyone; the previous one has been read by everyone
        copier.next();
        const float *B = ring + slot * kBK * 128 + 4 * tx, *A = V + t * kBK * kVld + 2 * ty;
        slot = slot + 1 == kStages ? 0 : slot + 1;
#pragma unroll
        for (int kk = 0; kk < kBK; ++kk) {
            const f32x2 a = *reinterpret_cast<const f32x2 *>(A + kk * kVld);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const float4 b = *reinterpret_cast<const float4 *>(B + kk * 128 + 64 * q);
                fma_f32x2(acc[4 * q], a, twice_f32x2(b.x));
                fma_f32x2(acc[4 * q + 1], a, twice_f32x2(b.y));
                fma_f32x2(acc[4 * q + 2], a, twice_f32x2(b.z));
                fma_f32x2(acc[4 * q + 3], a, twice_f32x2(b.w));
            }
        }
        if ((t + 1) % (kF32Chunk / kBK) == 0 || t + 1 == K / kBK) {
#pragma unroll
            for (int j = 0; j < 4 * NQ; ++j) {
                tot[j] = add_f32x2(tot[j], acc[j]);
                acc[j] = 0ull;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 4 * NQ; ++j) {
        const float2 v = unpack_f32x2(tot[j]);
        out[0][j] = v.x;
        out[1][j] = v.y;
    }
}

__global__ void __launch_bounds__(kThreads, kChainBlocksPerSm) chain_f32_kernel(const ChainParams p) {
    extern __shared__ __align__(16) uint8_t smem[];
    const ChainSmem L = chain_smem(p.k_max, p.y_ld, p.p_ld, p.d);
    float *ring = reinterpret_cast<float *>(smem);
    double *w_sh = reinterpret_cast<double *>(smem + L.w);          // [d][kRows]
    double *u_sh = reinterpret_cast<double *>(smem + L.u);          // [kRows]: this site's uniforms
    double *u_next = u_sh + kRows;                                  // [kRows]: the next site's
    double *sums = reinterpret_cast<double *>(smem + L.sums);       // [kLogs][w_{s*}, Z][kRows]
    float *Y = reinterpret_cast<float *>(smem + L.y);               // [kRows][y_ld]
    float *V = reinterpret_cast<float *>(smem + L.v);               // [k_max][kVld]
    float *P = reinterpret_cast<float *>(smem + L.p);               // [kRows][p_ld]
    int *sstar_sh = reinterpret_cast<int *>(smem + L.sstar);
    float *scale_sh = reinterpret_cast<float *>(smem + L.scale);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ty = tid >> 4, tx = tid & 15;
    const int64_t row0 = (int64_t)blockIdx.x * kRows;
    const int d = p.d;

    Copier copier{p.sites, ring, p.M, d};
    copier.start();
    for (int s = 0; s < kStages - 1; ++s) copier.next();
    for (int e = tid; e < kBK * kRows; e += kThreads) V[e / kRows * kVld + e % kRows] = e < kRows ? 1.f : 0.f;

    if (warp == 7) u_sh[lane] = sample_uniform(p.seed, p.n0 + (uint64_t)(row0 + lane), 0u, p.job);

    int slot = 0, nlog = 0;
    double lp = 0.0;  // of row `lane`, in warp 0
    ChainSite s = p.sites[0];
    for (int k = 0; k < p.M; ++k) {
        const ChainSite s_next = p.sites[k + 1 < p.M ? k + 1 : k];
        const Units un = units_of(s, d);
        const int T = s.tiles_per_s, bs = (s.nreal + 3) & ~3;  // columns of an outcome block in Y
        for (int j = 0; j < un.count; ++j) {
            float out[2][8];
            const bool wide = unit_is_wide(s, un, d, j);
            if (wide) chain_tile<2>(copier, slot, ring, V, s.K, ty, tx, out);
            else chain_tile<1>(copier, slot, ring, V, s.K, ty, tx, out);
            // where the thread's four columns at 64 q lie: tile `tile`, columns c .. c + 3 of outcome block so
            int tile[2], so[2], c[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int col = 64 * q + 4 * tx;
                if (un.Wb) {
                    tile[q] = so[q] = (j * 128 + col) / un.Wb;
                    c[q] = col & (un.Wb - 1);
                } else {
                    tile[q] = j;
                    so[q] = j / T;
                    c[q] = (j - so[q] * T) * 128 + col;
                }
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = 2 * ty + i;
                float *y = Y + r * p.y_ld;
                // sums of squares in the order of contract_f32_kernel: a thread's 4 or 8 columns of the tile,
                // then a tree over the 16 threads of the row (those of another outcome block, or of padding,
                // would add zeros)
                float ss[2] = {0.f, 0.f};
#pragma unroll
                for (int e = 0; e < 4; ++e) ss[0] = fmaf(out[i][e], out[i][e], ss[0]);
                if (wide) {
                    ss[1] = un.Wb ? 0.f : ss[0];
#pragma unroll
                    for (int e = 4; e < 8; ++e) ss[1] = fmaf(out[i][e], out[i][e], ss[1]);
                    if (!un.Wb) ss[0] = ss[1];
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    if (q == 1 && !(un.Wb && wide)) break;
                    ss[q] += __shfl_xor_sync(0xffffffffu, ss[q], 1);
                    ss[q] += __shfl_xor_sync(0xffffffffu, ss[q], 2);
                    if (un.Wb != 16) ss[q] += __shfl_xor_sync(0xffffffffu, ss[q], 4);
                    if (un.Wb == 0 || un.Wb == 64) ss[q] += __shfl_xor_sync(0xffffffffu, ss[q], 8);
                    if ((un.Wb ? c[q] == 0 : tx == 0) && so[q] < d) P[r * p.p_ld + tile[q]] = ss[q];
                }
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    if ((q == 0 || wide) && so[q] < d && c[q] < s.nreal)
                        *reinterpret_cast<float4 *>(y + so[q] * bs + c[q]) =
                            make_float4(out[i][4 * q], out[i][4 * q + 1], out[i][4 * q + 2], out[i][4 * q + 3]);
            }
        }
        __syncthreads();
        // w_s in FP64, in tile order; with one tile per outcome that is the tile's sum itself
        if (T > 1) {
            for (int e = tid; e < kRows * d; e += kThreads) {
                const float *src = P + (e % kRows) * p.p_ld + e / kRows * T;
                double acc = 0.0;
                for (int j = 0; j < T; ++j) acc += (double)src[j];
                w_sh[e] = acc;
            }
            __syncthreads();
        }
        if (warp == 0) {
            const int64_t row = row0 + lane;
            auto w_of = [&](int q) { return T > 1 ? w_sh[q * kRows + lane] : (double)P[lane * p.p_ld + q]; };
            double Z = 0.0;
            for (int q = 0; q < d; ++q) Z += w_of(q);
            const double t = u_sh[lane] * Z;
            double C = 0.0, ws = 0.0;
            int sstar = d - 1;
            for (int q = 0; q < d; ++q) {
                const double w = w_of(q);
                C += w;
                if (q == d - 1 || C >= t) {
                    sstar = q;
                    ws = w;
                    break;
                }
            }
            const bool ok = (Z > 0.0) && isfinite(Z) && (ws > 0.0);
            sstar_sh[lane] = sstar;
            scale_sh[lane] = ok ? rsqrtf((float)ws) : 0.f;
            sums[(2 * nlog) * kRows + lane] = ok ? ws : 1.0;
            sums[(2 * nlog + 1) * kRows + lane] = ok ? Z : 1.0;
            if (row < p.rows) {
                if (p.samples) p.samples[row * p.M + k] = (uint8_t)sstar;
                if (!ok) atomicExch(p.err, (int)kDevNumeric);
                const int64_t ts = !p.trace ? -1 : p.trace_slot ? (int64_t)p.trace_slot[row] : row < p.trace_rows ? row : -1;
                if (ts >= 0)
                    for (int q = 0; q < d; ++q)
                        p.trace[((int64_t)k * p.trace_rows + ts) * d + q] = ok ? w_of(q) / Z : 0.0;
            }
            // the next site's uniforms are drawn by another warp meanwhile, into the other half
        } else if (warp == 7) {
            u_next[lane] = sample_uniform(p.seed, p.n0 + (uint64_t)(row0 + lane), (uint32_t)k + 1u, p.job);
        }
        __syncthreads();
        if (k + 1 < p.M) {
            // the selected block, scaled, is the next left row; zeros up to the next site's last stage
            const int K_next = (s.nreal + kBK - 1) / kBK * kBK;
            for (int r = warp; r < kRows; r += kThreads / 32) {
                const float sc = scale_sh[r];
                const float *src = Y + r * p.y_ld + sstar_sh[r] * bs;
                for (int i = lane; i < K_next; i += 32) V[i * kVld + r] = i < s.nreal ? src[i] * sc : 0.f;
            }
        }
        if (++nlog == kLogs || k + 1 == p.M) {
            for (int e = tid; e < nlog * kRows; e += kThreads) {
                double *w = sums + e / kRows * 2 * kRows + e % kRows;
                w[0] = log(w[0] / w[kRows]);
            }
            __syncthreads();
            if (warp == 0)
                for (int q = 0; q < nlog; ++q) lp += sums[2 * q * kRows + lane];
            __syncthreads();
            nlog = 0;
        }
        double *swap = u_sh;
        u_sh = u_next;
        u_next = swap;
        s = s_next;
    }
    if (warp == 0 && p.logp && row0 + lane < p.rows) p.logp[row0 + lane] = lp;
    cp_async_wait<0>();
}

}  // namespace

void chain_f32_units(const ChainSite &s, int d, int *wide, int *narrow) {
    const Units u = units_of(s, d);
    *wide = 0;
    for (int j = 0; j < u.count; ++j) *wide += unit_is_wide(s, u, d, j) ? 1 : 0;
    *narrow = u.count - *wide;
}

int64_t chain_f32_blocks(int64_t rows) { return (rows + kRows - 1) / kRows; }

size_t chain_f32_smem(int k_max, int y_ld, int p_ld, int d) { return (size_t)chain_smem(k_max, y_ld, p_ld, d).total; }

cudaError_t launch_chain_f32(const ChainArgs &a, cudaStream_t st) {
    if (a.rows <= 0 || a.M <= 0) return cudaSuccess;
    ChainParams p;
    p.sites = a.sites;
    p.M = a.M;
    p.d = a.d;
    p.k_max = a.k_max;
    p.y_ld = a.y_ld;
    p.p_ld = a.p_ld;
    p.rows = a.rows;
    p.seed = a.seed;
    p.n0 = a.n0;
    p.job = a.job;
    p.samples = a.samples;
    p.logp = a.logp;
    p.trace = a.trace;
    p.trace_rows = a.trace_rows;
    p.trace_slot = a.trace_slot;
    p.err = a.err;
    const size_t smem = chain_f32_smem(a.k_max, a.y_ld, a.p_ld, a.d);
    cudaError_t e = cudaFuncSetAttribute(chain_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    chain_f32_kernel<<<(unsigned)chain_f32_blocks(a.rows), kThreads, smem, st>>>(p);
    return cudaGetLastError();
}

}  // namespace fastmps
