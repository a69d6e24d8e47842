// Prompt prefill on the 5th-generation tensor cores.
//
// The decode kernels stream every weight once per pass of at most 64 rows, which is the right trade for a
// round (1..13 rows) and the wrong one for a prompt: hundreds of positions can share one pass over the
// weights.  Here the four projections of a layer run as tiled GEMMs over up to PF_ROWS prompt positions
// at a time,  Y[M, N] = X[M, K] * W[N, K]^T,  with the layer's element-wise work fused into the epilogue:
//   QKV     1/rms of the row, rotary embedding on q and k, q -> Q buffer, k and v -> paged cache
//   OPROJ   + residual (in place), ffn-norm input, per-tile sums of squares
//   GATEUP  1/rms, SiLU(gate) * up -> activation buffer (the tile holds 128 gate and the same 128 up rows)
//   DOWN    + residual (in place), next layer's attention-norm input, per-tile sums of squares
// Of most prompt positions only the KV cache is needed later.  The last window of positions also seeds
// the acceptance statistics: the hidden state of those rows after every layer (and their embedding) is
// copied into the hidden stack, where the stacked LM head finds it.
//
// The activations enter every GEMM as a pair of bf16 values (high + low part, see common.cuh): each k-block is
// two MMAs on the same weight tile, one per part, into the same accumulator, so that the prompt's keys, values
// and hidden states carry the same accuracy as those the decode kernels make.
//
// CTA tile 128 rows x 256 or 128 output features (prefill_tc_split chooses per launch), K blocks of 64 (one 128-byte
// swizzle span), same roles as the stacked LM head: warp 0 issues TMA loads into a shared-memory ring (3 stages of 64 KB or 4
// of 48 KB), warp 1 issues tcgen05.mma into one of two 256-column accumulators in tensor memory, warps 2-9 read their own
// row with tcgen05.ld, each half of the columns, and run the epilogue while the next tile's MMAs proceed.  A launch
// with fewer tiles than half of the SMs (short prompts) cuts K into up to 4 parts: each CTA leaves its partial sums in the
// workspace, takes a ticket, and the last one of a tile adds the parts in K order and runs the epilogue.
// Ragged shapes (rows, N, K) rely on TMA zero fill plus store masks.  Every mbarrier wait is bounded.
#include <cuda.h>

#include <algorithm>
#include <initializer_list>

#include "kernels.h"
#include "tc_common.cuh"

namespace {

using namespace tc;

constexpr int BM = 128, BK = 64, ACC = 256;      // ACC: columns of an accumulator
// a stage: high parts of the activation tile, their low parts, the weight tile
constexpr int A_BYTES = BM * BK * 2, RING_BYTES = 3 * (2 * A_BYTES + 256 * BK * 2), MAX_STAGES = 4;
constexpr int PF_THREADS = 320, EPI_WARPS = 8;
static_assert(RING_BYTES == 4 * (2 * A_BYTES + 128 * BK * 2), "both tile widths fill the ring");

struct PfMaps {
    CUtensorMap a, a_lo;       // activations [chunk rows, K], high and low parts, box 64 x 128
    CUtensorMap b0, b1, b2;    // weights [N, K]: QKV Wq / Wk / Wv (box 64 x 128); GATEUP gate / up (box 64 x 64); else b0 (64 x 128)
};

// where a tile's sums are: an accumulator in tensor memory, or the partial sums of a tile whose K was cut
struct Sums {
    uint32_t taddr;
    const float *part;         // [parts][columns / 32][128 rows][32], this thread's row; nullptr: tensor memory
    int parts, stride;         // floats between two parts
    __device__ __forceinline__ void load32(int col, uint32_t (&r)[32]) const {
        if (part == nullptr) {
            tmem_ld32(taddr + (uint32_t)col, r);
            return;
        }
        float s[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) s[e] = 0.f;
        const float *p = part + (size_t)(col >> 5) * BM * 32;
        for (int i = 0; i < parts; ++i, p += stride)                  // ascending K
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float4 v = __ldcg(reinterpret_cast<const float4 *>(p) + e);
                s[4 * e] += v.x; s[4 * e + 1] += v.y; s[4 * e + 2] += v.z; s[4 * e + 3] += v.w;
            }
#pragma unroll
        for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(s[e]);
    }
};

// 1/rms of a row from the producer's per-tile sums of squares
__device__ __forceinline__ float row_rscale(const float *ssp, int n_part, int d, float eps) {
    float s = 0.f;
    if ((n_part & 3) == 0) {       // (then every row starts on 16 bytes)
#pragma unroll 4
        for (int i = 0; i < n_part; i += 4) {
            const float4 v = __ldcg(reinterpret_cast<const float4 *>(ssp + i));
            s = (((s + v.x) + v.y) + v.z) + v.w;
        }
    } else {
        for (int i = 0; i < n_part; ++i) s += ldg_cg_f32(ssp + i);
    }
    return rsqrtf(s / (float)d + eps);
}

__device__ __forceinline__ void store_bf16x32(bf16 *dst, const float (&v)[32]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint4 w;
        w.x = pack_bf16(v[8 * q + 0], v[8 * q + 1]);
        w.y = pack_bf16(v[8 * q + 2], v[8 * q + 3]);
        w.z = pack_bf16(v[8 * q + 4], v[8 * q + 5]);
        w.w = pack_bf16(v[8 * q + 6], v[8 * q + 7]);
        *reinterpret_cast<uint4 *>(dst + 8 * q) = w;
    }
}
// Whole 32-byte sectors per lane: the lanes' rows are far apart, so a 16-byte store writes half of a sector, and the other
// half is a second transaction (7B shape, 1000 rows, us: O-projection 63 -> 57, down 136 -> 130)
__device__ __forceinline__ void store32(void *dst, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t e, uint32_t f, uint32_t g, uint32_t h) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(a), "r"(b), "r"(c), "r"(d), "r"(e), "r"(f), "r"(g), "r"(h) : "memory");
}
__device__ __forceinline__ void load32(const float *src, float *v) {
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "l"(src) : "memory");
}
__device__ __forceinline__ void store_f32x32(float *dst, const float (&v)[32]) {
#pragma unroll
    for (int q = 0; q < 32; q += 8)
        store32(dst + q, __float_as_uint(v[q]), __float_as_uint(v[q + 1]), __float_as_uint(v[q + 2]), __float_as_uint(v[q + 3]),
                __float_as_uint(v[q + 4]), __float_as_uint(v[q + 5]), __float_as_uint(v[q + 6]), __float_as_uint(v[q + 7]));
}
// the same values as high parts to `hi` and low parts to `lo` (both 32-byte aligned: rows of the workspace)
__device__ __forceinline__ void store_split_x32(bf16 *hi, bf16 *lo, const float (&v)[32]) {
#pragma unroll
    for (int q = 0; q < 32; q += 16) {
        uint32_t wh[8], wl[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) split_bf16x2(v[q + 2 * i], v[q + 2 * i + 1], wh[i], wl[i]);
        store32(hi + q, wh[0], wh[1], wh[2], wh[3], wh[4], wh[5], wh[6], wh[7]);
        store32(lo + q, wl[0], wl[1], wl[2], wl[3], wl[4], wl[5], wl[6], wl[7]);
    }
}

// Four entries of a rotary table.  Every lane reads another position's row, so an access costs as many passes through L1 as
// lanes: 16 bytes at a time where the tables are aligned (the caller's pointers need not be) take a quarter of them
// (7B shape, 1000 rows: the QKV launch 178 us with 4-byte loads, 165 with these).
__device__ __forceinline__ void load_rope4(const float *q, int vec, float (&v)[4]) {
    if (vec) {
        const float4 f = __ldg(reinterpret_cast<const float4 *>(q));
        v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = __ldg(q + i);
    }
}

// 32 features of this lane's row, scaled and rounded to bf16, transposed among the 8 lanes of a block of rows: w[k] =
// feature 8 k + (lane & 7) of the block's 8 rows
__device__ __forceinline__ void transpose8(const uint32_t (&r)[32], float scale, bool live, int lane, uint4 (&w)[4]) {
    uint32_t a[16], b[8][2];
    const bool b0 = lane & 1, b1 = lane & 2, b2 = lane & 4;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float x = live ? scale * __uint_as_float(r[2 * i]) : 0.f, y = live ? scale * __uint_as_float(r[2 * i + 1]) : 0.f;
        const float got = __shfl_xor_sync(0xffffffffu, b0 ? x : y, 1);
        a[i] = b0 ? pack_bf16(got, y) : pack_bf16(x, got);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t got = __shfl_xor_sync(0xffffffffu, b1 ? a[2 * i] : a[2 * i + 1], 2);
        b[i][0] = b1 ? got : a[2 * i];
        b[i][1] = b1 ? a[2 * i + 1] : got;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t g0 = __shfl_xor_sync(0xffffffffu, b2 ? b[2 * i][0] : b[2 * i + 1][0], 4);
        const uint32_t g1 = __shfl_xor_sync(0xffffffffu, b2 ? b[2 * i][1] : b[2 * i + 1][1], 4);
        w[i] = b2 ? make_uint4(g0, g1, b[2 * i + 1][0], b[2 * i + 1][1]) : make_uint4(b[2 * i][0], b[2 * i][1], g0, g1);
    }
}

// ---- epilogues: one thread owns one row of the tile and, of its columns, the blocks of 32 (rotary and gate / up partners:
// the pairs of blocks) with half = 0 the first, 1 the second half; rs: the row's 1/rms (QKV, GATEUP)
template <int EPI>
__device__ __forceinline__ void epilogue(const PfArgs &p, const Sums &src, int row, int nt, int half_id, float rs) {
    const int BN = p.bn;
    const bool live = row < p.M;
    const int lane = threadIdx.x & 31;
    const Dims &D = p.D;
    uint32_t r0[32], r1[32];
    if (EPI == PF_QKV) {
        const int hd = D.hd, half = hd >> 1;
        const int n_qt = (D.nh * hd + BN - 1) / BN, n_kt = (D.nkv * hd + BN - 1) / BN;
        const int which = nt < n_qt ? 0 : (nt < n_qt + n_kt ? 1 : 2);
        const int n0 = (nt - (which == 0 ? 0 : (which == 1 ? n_qt : n_qt + n_kt))) * BN;   // feature offset in its matrix
        const int n_out = which == 0 ? D.nh * hd : D.nkv * hd;
        const int pos = p.pos0 + min(row, p.M - 1);              // (rows past the chunk: the last live row's page)
        const int pg = p.PT[p.seq * D.pages_per_seq + (pos >> 4)], sl = pos & 15;
        if (which < 2) {
            const float *cs = p.rope_cos + (size_t)pos * half, *sn = p.rope_sin + (size_t)pos * half;
            const int per = half >> 5, n_pair = BN >> 6;             // pairs of blocks per head, per tile
            for (int u = half_id * (n_pair >> 1); u < (half_id + 1) * (n_pair >> 1); ++u) {
                {
                    const int h0 = (per == 2 ? u >> 1 : u) * hd, jj = per == 2 ? (u & 1) * 32 : 0;     // head inside the tile
                    __syncwarp();
                    src.load32(h0 + jj, r0);
                    src.load32(h0 + half + jj, r1);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    const int n = n0 + h0;                       // first feature of the head
                    if (!live || n >= n_out) continue;
                    float lo[32], hi[32];
#pragma unroll
                    for (int e4 = 0; e4 < 32; e4 += 4) {
                        float c[4], s[4];
                        load_rope4(cs + jj + e4, p.rope_vec, c);
                        load_rope4(sn + jj + e4, p.rope_vec, s);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int e = e4 + i;
                            const float a = rs * __uint_as_float(r0[e]), b = rs * __uint_as_float(r1[e]);
                            lo[e] = a * c[i] - b * s[i];
                            hi[e] = b * c[i] + a * s[i];
                        }
                    }
                    if (which == 0) {
                        const size_t qo = (size_t)row * (D.nh * hd) + n + jj;
                        store_split_x32(p.Q + qo, p.QL + qo, lo);
                        store_split_x32(p.Q + qo + half, p.QL + qo + half, hi);
                    } else {
                        bf16 *dst = p.KP + ((((size_t)pg * D.L + (p.layer - 1)) * D.nkv + n / hd) * 16 + sl) * hd + jj;
                        store_bf16x32(dst, lo);
                        store_bf16x32(dst + half, hi);
                    }
                }
            }
        } else {
            for (int c0 = half_id * (BN >> 1); c0 < (half_id + 1) * (BN >> 1); c0 += 32) {
                __syncwarp();
                src.load32(c0, r0);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                const int n = n0 + c0;                           // 32 features of one head (n_out is a multiple of 64)
                if (n >= n_out) continue;
                const int kvh = n / hd, dim = n - kvh * hd;
                if (p.vp_vec) {
                    // transposed in blocks of 8 positions x 8 features across lanes: 4 stores of 16 bytes instead of 32 of 2
                    // (positions past the prompt that share a block with it get zeros)
                    uint4 w[4];
                    transpose8(r0, live ? rs : 0.f, live, lane, w);
                    if ((row & ~7) < p.M) {
                        bf16 *dst = p.VP + ((((size_t)pg * D.L + (p.layer - 1)) * D.nkv + kvh) * hd + dim + (lane & 7)) * 16 + (sl & 8);
#pragma unroll
                        for (int k = 0; k < 4; ++k) *reinterpret_cast<uint4 *>(dst + (size_t)k * 8 * 16) = w[k];
                    }
                } else if (live) {
                    bf16 *dst = p.VP + ((((size_t)pg * D.L + (p.layer - 1)) * D.nkv + kvh) * hd + dim) * 16 + sl;
#pragma unroll
                    for (int e = 0; e < 32; ++e) dst[e * 16] = __float2bfloat16_rn(rs * __uint_as_float(r0[e]));
                }
            }
        }
    } else if (EPI == PF_GATEUP) {
        for (int c0 = half_id * (BN >> 2); c0 < (half_id + 1) * (BN >> 2); c0 += 32) {
            __syncwarp();
            src.load32(c0, r0);
            src.load32(BN / 2 + c0, r1);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            const int f0 = nt * (BN / 2) + c0;
            if (!live || f0 >= D.F) continue;
            float act[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                const float g = rs * __uint_as_float(r0[e]), u = rs * __uint_as_float(r1[e]);
                act[e] = g / (1.f + __expf(-g)) * u;
            }
            bf16 *dst = p.ACT + (size_t)row * D.F + f0, *dlo = p.ACTL + (size_t)row * D.F + f0;
            if (f0 + 32 <= D.F) {
                store_split_x32(dst, dlo, act);
            } else {
                for (int e = 0; e < 32 && f0 + e < D.F; ++e) split_bf16(act[e], dst[e], dlo[e]);
            }
        }
    } else {   // PF_OPROJ, PF_DOWN: residual update in place, next norm input, sums of squares of the new h
        float ss = 0.f;
        bf16 *xo = EPI == PF_OPROJ ? p.XM : p.XS, *xl = EPI == PF_OPROJ ? p.XML : p.XSL;
        for (int c0 = half_id * (BN >> 1); c0 < (half_id + 1) * (BN >> 1); c0 += 32) {
            __syncwarp();
            src.load32(c0, r0);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            const int n = nt * BN + c0;
            if (!live || n >= D.d) continue;                     // d is a multiple of 32
            float *hp = p.H + (size_t)row * D.d + n;
            float h[32];
#pragma unroll
            for (int q = 0; q < 32; q += 8) load32(hp + q, h + q);
#pragma unroll
            for (int e = 0; e < 32; ++e) h[e] += __uint_as_float(r0[e]);
            store_f32x32(hp, h);
            if (EPI == PF_DOWN && p.pos0 + row >= p.win0)
                store_f32x32(p.stackH + stack_row(D, p.layer, p.seq, p.pos0 + row - p.win0) * D.d + n, h);
            float x[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                ss += h[e] * h[e];
                x[e] = p.gain ? h[e] * bf16_to_f(p.gain[n + e]) : 0.f;
            }
            if (p.gain) store_split_x32(xo + (size_t)row * D.d + n, xl + (size_t)row * D.d + n, x);
            // one partial sum of squares per 64 columns, whatever the tile width: results do not depend on it
            if ((c0 & 63) == 32 || n + 32 >= D.d) {
                (EPI == PF_OPROJ ? p.SSPM : p.SSP)[(size_t)row * p.n_ssp + (n >> 6)] = ss;
                ss = 0.f;
            }
        }
    }
}

template <int EPI>
__global__ void __launch_bounds__(PF_THREADS, 1) prefill_gemm_kernel(const __grid_constant__ PfMaps maps, const PfArgs p) {
    extern __shared__ unsigned char smem_dyn[];
    __shared__ __align__(8) uint64_t full_bar[MAX_STAGES], empty_bar[MAX_STAGES], tfull_bar[2], tempty_bar[2];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int s_err;
    __shared__ int s_last;
    // 1024-byte alignment for the 128-byte swizzle atoms
    unsigned char *tiles = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&tfull_bar[b], 1); mbar_init(&tempty_bar[b], EPI_WARPS); }
        s_err = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_base_s;

    pdl_launch();
    pdl_wait();

    const int bn = p.bn, n_stages = bn == 256 ? 3 : 4, b_bytes = bn * BK * 2, stage_bytes = 2 * A_BYTES + b_bytes;
    const int n_kb_all = (p.K + BK - 1) / BK;
    const int n_mt = (p.M + BM - 1) / BM;
    const int n_tiles = n_mt * p.n_ntiles;
    // with K cut into parts every CTA has one (tile, part); otherwise tiles go round
    const int part = p.k_parts > 1 ? (int)blockIdx.x / n_tiles : 0, tile0 = (int)blockIdx.x - part * n_tiles;
    const int kb_first = n_kb_all * part / p.k_parts, n_kb = n_kb_all * (part + 1) / p.k_parts - kb_first;
    const int my_tiles = p.k_parts > 1 ? 1 : (n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;

    if (warp == 0) {
        if (lane == 0) {
            // With up to two row tiles the weights are most of what a launch reads, each tile at about the same time by both: it goes
            // first from L2, and activations and code stay.  ms per prompt without / with, 7B shape: 45 positions 6.01 / 5.44, 128:
            // 6.38 / 5.97, 160: 8.98 / 8.82, 256: 9.44 / 9.27; 1B 45: 2.01 / 1.92, 256: 2.42 / 2.35; 8B and 13B 1 to 7 % less; tiny (all
            // weights stay in L2 anyway) 0 to 1 % more.  With more row tiles (tried up to four) 257 to 384 positions would gain 2 % at the 1B shape, 1 % at
            // 7B and 0 to 1.5 % at 8B and 13B, 385 to 512 -1 to 2 %, longer ones nothing or -1 %; a load with the normal policy given
            // explicitly costs the latter too.  Those load without one.
            const bool few = n_mt <= 2;
            const uint64_t pol = l2_evict_first();
            auto load_w = [&](void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
                if (few) tma_load_2d(dst, map, x, y, bar, pol);
                else tma_load_2d(dst, map, x, y, bar);
            };
            const int n_qt = (p.D.nh * p.D.hd + bn - 1) / bn, n_kt = (p.D.nkv * p.D.hd + bn - 1) / bn;
            int s = 0;
            uint32_t phase = 1;
            for (int i = 0; i < my_tiles && !s_err; ++i) {
                const int tile = tile0 + i * gridDim.x;
                const int nt = tile / n_mt, mt = tile - nt * n_mt;      // row tiles of one weight tile run together
                const CUtensorMap *mb = &maps.b0;
                int y = nt * bn;
                if (EPI == PF_QKV) {
                    mb = nt < n_qt ? &maps.b0 : (nt < n_qt + n_kt ? &maps.b1 : &maps.b2);
                    y = (nt - (nt < n_qt ? 0 : (nt < n_qt + n_kt ? n_qt : n_qt + n_kt))) * bn;
                }
                for (int kb = kb_first; kb < kb_first + n_kb; ++kb) {
                    if (!mbar_wait(&empty_bar[s], phase)) { s_err = 1; break; }
                    mbar_expect_tx(&full_bar[s], stage_bytes);
                    unsigned char *sa = tiles + (size_t)s * stage_bytes, *sb = sa + 2 * A_BYTES;
                    tma_load_2d(sa, &maps.a, kb * BK, mt * BM, &full_bar[s]);
                    tma_load_2d(sa + A_BYTES, &maps.a_lo, kb * BK, mt * BM, &full_bar[s]);
                    if (EPI == PF_GATEUP) {
                        // accumulator columns 0 .. bn/2 - 1: gate rows of this tile, bn/2 .. bn - 1: the same rows of W_up
                        for (int r = 0; r < bn / 2; r += 64) {
                            load_w(sb + r * 128, &maps.b0, kb * BK, nt * (bn / 2) + r, &full_bar[s]);
                            load_w(sb + (bn / 2 + r) * 128, &maps.b1, kb * BK, nt * (bn / 2) + r, &full_bar[s]);
                        }
                    } else {
                        for (int r = 0; r < bn; r += 128) load_w(sb + r * 128, mb, kb * BK, y + r, &full_bar[s]);
                    }
                    if (++s == n_stages) { s = 0; phase ^= 1; }
                }
            }
            if (s_err) drain(full_bar, n_stages, s, phase ^ 1);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // instruction descriptor: fp32 accumulate, bf16 x bf16, both operands K-major, N = tile width, M = 128
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            int s = 0;
            uint32_t phase = 0;
            for (int i = 0; i < my_tiles && !s_err; ++i) {
                const int buf = i & 1;
                if (!mbar_wait(&tempty_bar[buf], ((i >> 1) & 1) ^ 1)) { s_err = 2; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t d_tmem = tmem_base + (uint32_t)buf * ACC;
                bool ok = true;
                for (int kb = 0; kb < n_kb; ++kb) {
                    if (!mbar_wait(&full_bar[s], phase)) { s_err = 3; ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t sa = smem_u32(tiles + (size_t)s * stage_bytes);
                    const uint64_t da = umma_desc(sa), dl = umma_desc(sa + A_BYTES), db = umma_desc(sa + 2 * A_BYTES);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        umma_bf16(d_tmem, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
                        umma_bf16(d_tmem, dl + 2 * k, db + 2 * k, idesc, 1u);
                    }
                    umma_commit(&empty_bar[s]);      // the stage may be refilled once these MMAs have read it
                    if (++s == n_stages) { s = 0; phase ^= 1; }
                }
                if (!ok) break;
                umma_commit(&tfull_bar[buf]);        // accumulator complete
            }
            if (s_err) drain(empty_bar, n_stages, s, phase);
        }
    } else {
        const int q = warp & 3, half_id = (warp - 2) >> 2;   // TMEM lane quarter this warp may read, half of the columns
        for (int i = 0; i < my_tiles; ++i) {
            const int tile = tile0 + i * gridDim.x;
            const int nt = tile / n_mt, mt = tile - nt * n_mt;
            const int buf = i & 1, rr = q * 32 + lane, row = mt * BM + rr;
            float rs = 0.f;
            if ((EPI == PF_QKV || EPI == PF_GATEUP) && row < p.M)
                rs = row_rscale((EPI == PF_QKV ? p.SSP : p.SSPM) + (size_t)row * p.n_ssp, p.n_ssp, p.D.d, p.D.eps);
            bool ok = !s_err;
            if (ok && !mbar_wait(&tfull_bar[buf], (i >> 1) & 1)) { s_err = 4; ok = false; }
            if (p.k_parts == 1 && !ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            Sums src{tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * ACC), nullptr, 1, 0};
            if (p.k_parts > 1) {
                // this part's sums -> workspace; the last of the tile's CTAs goes on
                const int tile_floats = BM * bn;
                if (ok) {
                    float *o = p.part + ((size_t)part * n_tiles + tile) * tile_floats + rr * 32;
                    for (int c0 = half_id * (bn >> 1); c0 < (half_id + 1) * (bn >> 1); c0 += 32) {
                        uint32_t r[32];
                        __syncwarp();
                        tmem_ld32(src.taddr + (uint32_t)c0, r);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        uint4 *d = reinterpret_cast<uint4 *>(o + (size_t)(c0 >> 5) * BM * 32);
#pragma unroll
                        for (int e = 0; e < 8; ++e) __stcg(d + e, make_uint4(r[4 * e], r[4 * e + 1], r[4 * e + 2], r[4 * e + 3]));
                    }
                }
                asm volatile("bar.sync 1, 256;" ::: "memory");
                if (threadIdx.x == 64) {
                    int old = -1;
                    if (!s_err) asm volatile("atom.add.acq_rel.gpu.s32 %0, [%1], 1;" : "=r"(old) : "l"(p.ticket + tile) : "memory");
                    s_last = old == p.k_parts - 1;
                    if (old == p.k_parts - 1) p.ticket[tile] = 0;
                }
                asm volatile("bar.sync 1, 256;" ::: "memory");
                if (!s_last) break;
                src.part = p.part + (size_t)tile * tile_floats + rr * 32;
                src.parts = p.k_parts;
                src.stride = n_tiles * tile_floats;
            }
            epilogue<EPI>(p, src, row, nt, half_id, rs);
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty_bar[buf]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
    if (threadIdx.x == 0 && s_err) atomicMax(p.err, (int)s_err);
}

// h^0 of the chunk's rows: embedding as fp32, layer 1's attention-norm input, sum of squares in partial 0
__global__ void __launch_bounds__(256) prefill_embed_kernel(const PfArgs p, const bf16 *tok_emb, const int32_t *prompt, const bf16 *gain0) {
    __shared__ float s_red[8];
    pdl_launch();
    pdl_wait();
    const int row = blockIdx.x, d = p.D.d;
    const bf16 *e = tok_emb + (size_t)prompt[p.pos0 + row] * d;
    float *sp = p.pos0 + row >= p.win0 ? p.stackH + stack_row(p.D, 0, p.seq, p.pos0 + row - p.win0) * d : nullptr;
    float ss = 0.f;
    for (int o = threadIdx.x; o < d; o += 256) {
        const float h = bf16_to_f(e[o]);
        p.H[(size_t)row * d + o] = h;
        if (sp) sp[o] = h;
        split_bf16(h * bf16_to_f(gain0[o]), p.XS[(size_t)row * d + o], p.XSL[(size_t)row * d + o]);
        ss += h * h;
    }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = ss;
    __syncthreads();
    for (int i = threadIdx.x; i < p.n_ssp; i += 256) {
        float t = 0.f;
        if (i == 0)
            for (int w = 0; w < 8; ++w) t += s_red[w];
        p.SSP[(size_t)row * p.n_ssp + i] = t;
    }
}

constexpr size_t SMEM_BYTES = (size_t)RING_BYTES + 1024;

template <int EPI> cudaError_t prepare_epi() {
    static SmemAttrOnce attr;
    return attr.set(prefill_gemm_kernel<EPI>, (int)SMEM_BYTES);
}

template <int EPI>
cudaError_t launch_epi(const PfMaps &maps, const PfArgs &p, int n_sms, cudaStream_t st, bool pdl) {
    auto kern = prefill_gemm_kernel<EPI>;
    {
        cudaError_t e = prepare_epi<EPI>();
        if (e != cudaSuccess) return e;
    }
    const int n_tiles = ((p.M + BM - 1) / BM) * p.n_ntiles * p.k_parts;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_tiles < n_sms ? n_tiles : n_sms);
    cfg.blockDim = dim3(PF_THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, maps, p);
}

}  // namespace

int prefill_tc_nssp(const Dims &D) { return (D.d + 63) / 64; }

namespace {

int n_tiles_of(int epi, const Dims &D, int bn) {
    switch (epi) {
        case PF_QKV: return (D.nh * D.hd + bn - 1) / bn + 2 * ((D.nkv * D.hd + bn - 1) / bn);
        case PF_GATEUP: return (D.F + bn / 2 - 1) / (bn / 2);
        default: return (D.d + bn - 1) / bn;
    }
}

// Tile width and parts of K of a launch: the choice with the smallest estimated time, waves of tiles on the SMs x (K blocks of
// a tile x what a block takes) + the last tile's epilogue + the merge of the parts.  The constants are microseconds fitted to 897
// launches of six layer shapes (50 to 635 MB) at 48 to 2048 rows: 6 % rms, and no launch whose choice is more than 7 % slower
// than the best of the five.  That holds for launches of up to two row tiles with their weights marked evict-first, too: seven shapes
// at 48 to 512 rows measured again, choices at most 4 % from the best.  Measured, us, 256 wide / 128 wide / 128 wide with K
// in 2, 3, 4 parts (1024 rows: before that):
//   7B shape,   48 rows: QKV 49 / 35,  O 48 / 34 / 30, 29, 29,  gate/up 53 / 66,  down 112 / 78 / 52, 44, 41
//   7B shape,  160 rows: QKV 54 / 60,  O 53 / 36 / 33,          gate/up 90 / 91,  down 114 / 78 / 56
//   7B shape,  512 rows: QKV 89 / 92,  O 54 / 39,               gate/up 137 / 153, down 118 / 85
//   7B shape, 1024 rows: QKV 142 / 188, O 59 / 71,              gate/up 232 / 315, down 134 / 169
//   13B shape, 1024 rows: QKV 223 / 272, O 119 / 123,           gate/up 352 / 471, down 308 / 312
//   1B shape,  160 rows: QKV 31 / 22 / 24, 26,  O 34 / 23 / 25, 26, 27,  gate/up 32 / 37,  down 88 / 60 / 44, 39, 38
// (a merge costs as much as 25 to 40 K blocks, so K of 2048 is not cut)
struct Split { int bn, parts; double us; };
Split choose_split(int epi, const Dims &D, int M, int n_sms) {
    const int K = epi == PF_OPROJ ? D.nh * D.hd : (epi == PF_DOWN ? D.F : D.d);
    const int n_mt = (M + BM - 1) / BM, n_kb = (K + BK - 1) / BK;
    Split best{0, 0, 0.0};
    for (int bn = 256; bn >= 128; bn -= 128)
        for (int parts = 1; parts <= (bn == 128 ? 4 : 1); ++parts) {
            const int tiles = n_mt * n_tiles_of(epi, D, bn) * parts;
            if (parts > 1 && (tiles > n_sms || tiles > rowgemm_tc_ctas(D) || n_kb < 4 * parts)) continue;
            const double us = (tiles + n_sms - 1) / n_sms * ((double)n_kb / parts * (bn == 256 ? 0.667 : 0.452)) + (bn == 256 ? 12 : 8.3) + (parts > 1 ? 5 + 2.3 * parts : 0);
            if (best.bn == 0 || us < best.us) best = Split{bn, parts, us};
        }
    return best;
}

}  // namespace

void prefill_tc_split(int epi, const Dims &D, int M, int n_sms, int *bn, int *parts) {
    const Split s = choose_split(epi, D, M, n_sms);
    *bn = s.bn;
    *parts = s.parts;
}

// Positions per chunk of a prompt of n: the whole number of 128-row tiles, at most max_rows, with the smallest estimated
// time of the four GEMMs over all chunks (a wave of tiles that is nearly empty costs as much as a full one: the 13B shape's
// down projection has 160 tiles of 256 at 1024 rows, 240 at 1536, on 148 SMs; its 3072-position prompt
// takes 3494 us per layer in chunks of 1024 and 3079 in chunks of 1536)
int prefill_tc_chunk(const Dims &D, int n, int n_sms, int max_rows) {
    int best = 0;
    double best_us = 0.0;
    for (int c = std::min((n + BM - 1) / BM * BM, max_rows / BM * BM); c >= BM; c -= BM) {
        double us = 0.0;
        for (int p = 0; p < n; p += c) {
            us += 10.0;                                                 // launches, the attention's ragged blocks
            for (int epi = PF_QKV; epi <= PF_DOWN; ++epi) us += choose_split(epi, D, std::min(c, n - p), n_sms).us;
        }
        if (best == 0 || us < best_us) { best = c; best_us = us; }
    }
    return best;
}

cudaError_t prefill_tc_prepare() {
    for (cudaError_t e : {prepare_epi<PF_QKV>(), prepare_epi<PF_OPROJ>(), prepare_epi<PF_GATEUP>(), prepare_epi<PF_DOWN>()})
        if (e != cudaSuccess) return e;
    cudaFuncAttributes a;
    return cudaFuncGetAttributes(&a, prefill_embed_kernel);
}

// map_a / map_b*: 128-byte CUtensorMap blobs made by lmhead_tc_make_map (boxes of 128 rows, W_gate / W_up 64)
cudaError_t launch_prefill_gemm(int epi, const void *map_a, const void *map_a_lo, const void *map_b0, const void *map_b1,
                                const void *map_b2, const PfArgs &args, int n_sms, cudaStream_t st, bool pdl) {
    PfArgs p = args;
    const Split s = choose_split(epi, p.D, p.M, n_sms);
    p.bn = s.bn;
    p.k_parts = s.parts;
    p.n_ntiles = n_tiles_of(epi, p.D, s.bn);
    p.rope_vec = ((reinterpret_cast<uintptr_t>(p.rope_cos) | reinterpret_cast<uintptr_t>(p.rope_sin)) & 15) == 0;      // rows are whole multiples of 16 bytes
    p.vp_vec = (reinterpret_cast<uintptr_t>(p.VP) & 15) == 0;
    PfMaps maps;
    maps.a = *reinterpret_cast<const CUtensorMap *>(map_a);
    maps.a_lo = *reinterpret_cast<const CUtensorMap *>(map_a_lo);
    maps.b0 = *reinterpret_cast<const CUtensorMap *>(map_b0);
    maps.b1 = *reinterpret_cast<const CUtensorMap *>(map_b1 ? map_b1 : map_b0);
    maps.b2 = *reinterpret_cast<const CUtensorMap *>(map_b2 ? map_b2 : map_b0);
    switch (epi) {
        case PF_QKV: return launch_epi<PF_QKV>(maps, p, n_sms, st, pdl);
        case PF_OPROJ: return launch_epi<PF_OPROJ>(maps, p, n_sms, st, pdl);
        case PF_GATEUP: return launch_epi<PF_GATEUP>(maps, p, n_sms, st, pdl);
        case PF_DOWN: return launch_epi<PF_DOWN>(maps, p, n_sms, st, pdl);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_prefill_embed(const PfArgs &p, const bf16 *tok_emb, const int32_t *prompt, const bf16 *gain0, cudaStream_t st) {
    prefill_embed_kernel<<<p.M, 256, 0, st>>>(p, tok_emb, prompt, gain0);
    return cudaGetLastError();
}
