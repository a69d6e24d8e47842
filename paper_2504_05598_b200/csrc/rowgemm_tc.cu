// Layer GEMMs of passes with many rows:  Y[m, N] = X[m, K] * W[N, K]^T  on tcgen05, weights as the M operand.
//
// What bounds it: HBM, like the register-streaming form in rowgemm.cu (every weight byte once per launch).  That form
// holds the activation fragments of a burst in registers, so with more rows fewer weight bytes are in flight: its
// gate/up launch of the 7B shape (180 MB) takes 30 us for up to 4 rows, but 51 us for 9..16 and 102 us (two
// launches) for 17..64.  Here neither operand passes through registers.
//
// Tile: 128 weight rows (MMA M) x NP activation rows (16..64), K blocks of 128 (two 128-byte swizzle spans).  The
// activations' high and low parts lie behind one another in shared memory and are the 2 NP columns of one MMA; the
// two column halves are added when the accumulator is read, so the product carries the precision of the pair.
//
// Split: all (tile, K block) units of a launch are cut into one contiguous range per CTA, so that every SM streams
// the same number of bytes whatever the number of tiles (the 32 tiles of a d x d projection would otherwise leave 116
// of 148 SMs idle).  A tile cut by a range boundary is finished by whichever of its CTAs arrives last: each leaves its
// partial sums in the workspace, takes a ticket, and the last one adds all parts in K order.  Results depend
// neither on timing nor on the number of rows of such a pass; nobody waits for another CTA.
//
// Roles (384 threads): warp 0 streams weight blocks with TMA (the ring is filled before the kernel waits for its
// producer: weights depend on nobody), warp 2 the activation rows (for QKV they lie scattered over the hidden stack:
// groups of 8 consecutive rows), warp 1 issues the MMAs, warps 4-11 run the epilogues, one thread per weight row
// and half of the columns, accumulators double-buffered.  Rotary and gate / up partners sit in other lanes; they
// change places through shared memory.  One thread's issue latency paces each of the first three roles: with K blocks
// of 64, two rings and ring positions by division the same loop took 0.85 us per 16 KB of weights instead of 0.33.
// What bounds it now: HBM between a launch's first round trip and the ticket and merge at its end.  16 rows of the 7B shape,
// launches one at a time: QKV 26, O 14, gate/up 35 (180 MB, 5.2 TB/s), down 23 us; the layer, chained and with attention,
// takes 102 us (streaming form: 141; 32 rows: 124, 258).
#include <cuda.h>

#include <cstring>
#include <initializer_list>

#include "kernels.h"
#include "tc_common.cuh"

namespace {

using namespace tc;

constexpr int BM = 128, BK = 128, W_BYTES = BM * BK * 2;
constexpr int WT_THREADS = 384;
constexpr int WT_PIECES = 8;                // partial sums of a cut tile that are loaded at once

template <int NP> __host__ __device__ constexpr int x_bytes() { return 2 * NP * BK * 2; }
template <int NP> __host__ __device__ constexpr int stages() { return NP <= 16 ? 5 : (NP <= 32 ? 4 : 3); }

struct WtMaps {
    CUtensorMap w0, w1, w2;      // QKV: Wq, Wk, Wv; GATEUP: gate, up (boxes of 64 rows); else W.  Boxes of 128 rows
    CUtensorMap x, xl;           // activations, high and low parts (QKV: the hidden stack, boxes of 8 rows; else 16)
};

struct WtArgs {
    GemmArgs g;
    bf16 *xd, *xdl;              // DOWN: the next layer's input once more, by row of the pass (high / low part)
    float *part;                 // [CTA][2][NP / 8][128][8] partial sums of the cut tiles
    int32_t *ticket;             // [tiles] arrivals at a cut tile; zero between launches
    int32_t n_tiles, nkb;
    // 8 MMA columns each: the pass's rows row .. row + n - 1 (QKV: consecutive rows of the stack from src)
    int32_t n_grp, dense;        // dense: the input lies by row of the pass (always so but for some QKV launches)
    struct { int32_t src, row, n; } grp[DEL_ROWS_MAX / 8];
};

__device__ __forceinline__ void bar_epi() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void bar_half(int half) { asm volatile("bar.sync %0, 128;" ::"r"(2 + half) : "memory"); }
// barrier of the epilogue warps that also tells whether all of them said yes (so that they give up together)
__device__ __forceinline__ bool bar_epi_and(bool yes) {
    uint32_t all;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, 1, 256, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(all) : "r"((uint32_t)yes) : "memory");
    return all != 0;
}

// eight columns of the products with the high parts plus the same columns of those with the low parts
__device__ __forceinline__ void tmem_ld_sum8(uint32_t taddr, uint32_t low, float (&v)[8]) {
    uint32_t r[8], s[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr) : "memory");
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3]), "=r"(s[4]), "=r"(s[5]), "=r"(s[6]), "=r"(s[7])
                 : "r"(taddr + low) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(r[e]) + __uint_as_float(s[e]);
}

// position in the ring: stage and the parity of its current use
template <int N> struct Ring {
    int s = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void next() {
        if (++s == N) { s = 0; phase ^= 1; }
    }
};

// CTA c's units are [start(c), start(c + 1)); the CTA that holds unit u
// (units x CTAs stay below 2^31: rowgemm_tc_supported)
__device__ __forceinline__ int unit_start(int c, int U, int G) { return (int)((uint32_t)c * (uint32_t)U / (uint32_t)G); }
__device__ __forceinline__ int unit_cta(int u, int U, int G) { return (int)(((uint32_t)(u + 1) * (uint32_t)G - 1) / (uint32_t)U); }

// matrix of a QKV tile (0, 1, 2: q, k, v) and the tile's number inside it
__device__ __forceinline__ int qkv_tile(const Dims &D, int tile, int &local) {
    const int nq = (D.nh * D.hd + BM - 1) >> 7, nk = (D.nkv * D.hd + BM - 1) >> 7;
    const int which = tile < nq ? 0 : (tile < nq + nk ? 1 : 2);
    local = tile - (which == 0 ? 0 : (which == 1 ? nq : nq + nk));
    return which;
}

// per column (row of the pass): where its outputs go; filled once per launch
template <int NP> struct ColInfo {
    int src[NP], dst[NP];        // rows of the hidden stack: residual of the O-projection, output of DOWN
    int er[NP];                  // row of the exit buffers
    int kv[NP];                  // QKV: (page * L + layer - 1) * nkv
    int pos[NP];
    float rs[NP];                // 1/rms
};

// what an epilogue reads for 8 columns at this thread's feature, requested before the sums are there: the residual
// (O-projection, DOWN) or the rotation's cos and sin (QKV)
template <int NP, int EPI>
__device__ __forceinline__ void epi_loads(const WtArgs &w, const ColInfo<NP> &ci, int tile, int rr, int col, float (&p)[8], float (&p2)[8]) {
    const GemmArgs &a = w.g;
    const Dims &D = a.D;
    const int c0 = w.grp[col >> 3].row, n = w.grp[col >> 3].n;
    if (EPI == EPI_OPROJ || EPI == EPI_DOWN) {
        const int o = tile * BM + rr;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float *h = EPI == EPI_OPROJ ? a.B.H + (size_t)ci.src[col + e] * D.d + o : a.B.HM + (size_t)(c0 + e) * D.d + o;
            p[e] = e < n && o < D.d ? ldg_cg_f32(h) : 0.f;
        }
    } else if (EPI == EPI_QKV) {
        int local;
        const bool rot = qkv_tile(D, tile, local) < 2;
        const int hh = D.hd >> 1, j = rr & (hh - 1);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const size_t at = (size_t)ci.pos[col + e] * hh + j;
            p[e] = e < n && rot ? __ldg(a.B.rope_cos + at) : 0.f;
            p2[e] = e < n && rot ? __ldg(a.B.rope_sin + at) : 0.f;
        }
    }
}

// 8 finished columns of a tile: rr = weight row of the tile, ga / gb = the norm gains of its feature, xch = exchange
// buffer of this half's 4 warps
template <int NP, int EPI>
__device__ __forceinline__ void finish(const WtArgs &w, const ColInfo<NP> &ci, int tile, int rr, int half, int col, const float (&acc)[8],
                                       const float (&p)[8], const float (&p2)[8], float ga, float gb, float (*xch)[BM]) {
    const GemmArgs &a = w.g;
    const Dims &D = a.D;
    const int c0 = w.grp[col >> 3].row, n = w.grp[col >> 3].n;       // rows c0 .. c0 + n - 1 of the pass
    if (EPI == EPI_OPROJ || EPI == EPI_DOWN) {
        const int o = tile * BM + rr;
        const bool in = o < D.d;
        float v[8], ss[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            v[e] = in ? p[e] + acc[e] : 0.f;
            ss[e] = v[e] * v[e];
        }
#pragma unroll
        for (int s = 8; s > 0; s >>= 1)                               // sums over the 16 features of a partial
#pragma unroll
            for (int e = 0; e < 8; ++e) ss[e] += __shfl_xor_sync(0xffffffffu, ss[e], s);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            if (e >= n || !in) continue;
            const int c = c0 + e;
            bf16 hi, lo;
            split_bf16(v[e] * ga, hi, lo);
            const size_t i = (size_t)c * D.d + o;
            if (EPI == EPI_OPROJ) {
                a.B.HM[i] = v[e];
                a.B.XM[i] = hi;
                a.B.XML[i] = lo;
                if ((rr & 15) == 0) a.B.SSM[(size_t)c * D.n_sst + (o >> 4)] = ss[e];
            } else {
                const size_t sr = ci.dst[col + e], er = ci.er[col + e];
                a.B.H[sr * D.d + o] = v[e];
                if (a.gain_a) {
                    a.B.XS[sr * D.d + o] = hi;
                    a.B.XSL[sr * D.d + o] = lo;
                    w.xd[i] = hi;
                    w.xdl[i] = lo;
                }
                if (a.gain_b) a.B.XE[er * D.d + o] = __float2bfloat16_rn(v[e] * gb);
                if ((rr & 15) == 0) {
                    a.B.SS[sr * D.n_sst + (o >> 4)] = ss[e];
                    if (a.gain_b) a.B.SSE[er * D.n_sst + (o >> 4)] = ss[e];
                }
            }
        }
        return;
    }
    int local = 0;
    const int which = EPI == EPI_QKV ? qkv_tile(D, tile, local) : 0;
    float mine[8], other[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) mine[e] = ci.rs[col + e] * acc[e];
    if (EPI == EPI_GATEUP || which < 2) {
        const int partner = rr ^ (EPI == EPI_GATEUP ? 64 : D.hd >> 1);
#pragma unroll
        for (int e = 0; e < 8; ++e) xch[e][rr] = mine[e];
        bar_half(half);
#pragma unroll
        for (int e = 0; e < 8; ++e) other[e] = xch[e][partner];
    }
    if (EPI == EPI_GATEUP) {
        // rows 0..63: gate, 64..127: the same rows of W_up; the gate threads finish columns 0..3, the up threads 4..7
        const int f = tile * 64 + (rr & 63);
        const bool up = rr >= 64;
        if (f >= D.F) return;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = up ? 4 + i : i, c = c0 + e;
            if (e >= n) continue;
            const float g = up ? other[4 + i] : mine[i], u = up ? mine[4 + i] : other[i];
            const float act = g / (1.f + __expf(-g)) * u;
            split_bf16(act, a.B.ACT[(size_t)c * D.F + f], a.B.ACTL[(size_t)c * D.F + f]);
        }
        return;
    }
    const int f = local * BM + rr, hs = D.hd == 128 ? 7 : 6, head = f >> hs, dim = f & (D.hd - 1);
    if (f >= (which == 0 ? D.nh : D.nkv) * D.hd) return;
    const bool lo = dim < (D.hd >> 1);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        if (e >= n) continue;
        // first half: v_j cos - v_(j + half) sin; second half: v_(j + half) cos + v_j sin
        const float out = which == 2 ? mine[e] : (lo ? mine[e] * p[e] - other[e] * p2[e] : mine[e] * p[e] + other[e] * p2[e]);
        const bf16 v = __float2bfloat16_rn(out);
        const size_t page = (size_t)(ci.kv[col + e] + head);
        const int sl = ci.pos[col + e] & 15;
        if (which == 0) a.B.Q[(size_t)(c0 + e) * (D.nh * D.hd) + f] = v;
        else if (which == 1) a.B.KP[(page * 16 + sl) * D.hd + dim] = v;
        else a.B.VP[(page * D.hd + dim) * 16 + sl] = v;
    }
}

template <int NP, int EPI>
__global__ void __launch_bounds__(WT_THREADS, 1) rowgemm_tc_kernel(const __grid_constant__ WtMaps maps, const __grid_constant__ WtArgs w) {
    constexpr int X_BYTES = x_bytes<NP>(), STAGES = stages<NP>(), STAGE_BYTES = W_BYTES + X_BYTES;
    constexpr uint32_t TM_COLS = NP <= 16 ? 64 : (NP <= 32 ? 128 : 256);
    constexpr bool XCH = EPI == EPI_QKV || EPI == EPI_GATEUP;
    extern __shared__ unsigned char smem_dyn[];
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int s_err;
    __shared__ int s_last;
    __shared__ ColInfo<NP> ci;
    __shared__ float xch[XCH ? 4 : 1][8][BM];                         // [half][turn & 1]: one barrier per exchange is enough
    unsigned char *ring = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
    const GemmArgs &a = w.g;
    const Dims &D = a.D;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nkb = w.nkb, U = w.n_tiles * nkb, G = (int)gridDim.x, cta = (int)blockIdx.x;
    const int u_begin = unit_start(cta, U, G), u_end = unit_start(cta + 1, U, G);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 2); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], 8); }
        s_err = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(TM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_base_s;
    pdl_launch();

    if (warp == 0) {
        if (lane == 0) {
            // as in rowgemm.cu; ms per round, 7B shape, 13-row verify passes 7.41 -> 7.21, 8B shape, 8 sequences (48 rows) 8.58 -> 8.18
            const uint64_t pol = l2_evict_first();
            Ring<STAGES> r;
            int tile = u_begin / nkb, kb = u_begin - tile * nkb, cur = -1, which = 0, local = 0;
            for (int u = u_begin; u < u_end && !s_err; ++u, r.next()) {
                if (!mbar_wait(&empty[r.s], r.phase ^ 1)) { s_err = 1; break; }
                mbar_expect_tx(&full[r.s], W_BYTES);
                unsigned char *dst = ring + (size_t)r.s * STAGE_BYTES;
                if (EPI == EPI_QKV && tile != cur) { cur = tile; which = qkv_tile(D, tile, local); }
#pragma unroll
                for (int k = 0; k < 2; ++k, dst += W_BYTES / 2) {
                    const int x = kb * BK + 64 * k;
                    if (EPI == EPI_QKV) {
                        tma_load_2d(dst, which == 0 ? &maps.w0 : (which == 1 ? &maps.w1 : &maps.w2), x, local * BM, &full[r.s], pol);
                    } else if (EPI == EPI_GATEUP) {
                        tma_load_2d(dst, &maps.w0, x, tile * 64, &full[r.s], pol);
                        tma_load_2d(dst + W_BYTES / 4, &maps.w1, x, tile * 64, &full[r.s], pol);
                    } else {
                        tma_load_2d(dst, &maps.w0, x, tile * BM, &full[r.s], pol);
                    }
                }
                if (++kb == nkb) { kb = 0; ++tile; }
            }
            if (s_err) drain(full, STAGES, r.s, r.phase);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // fp32 accumulate, bf16 x bf16, both operands K-major, N = 2 NP, M = 128
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NP >> 2) << 17) | ((uint32_t)(BM >> 4) << 24);
            const uint32_t ring0 = smem_u32(ring);
            Ring<STAGES> r;
            int piece = 0, kb0 = u_begin % nkb;
            for (int u = u_begin; u < u_end && !s_err; ++piece, kb0 = 0) {
                const int n = min(nkb - kb0, u_end - u), buf = piece & 1;
                if (!mbar_wait(&tempty[buf], ((piece >> 1) & 1) ^ 1)) { s_err = 2; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * 2 * NP);
                bool ok = true;
                for (int i = 0; i < n; ++i, r.next()) {
                    if (!mbar_wait(&full[r.s], r.phase)) { s_err = 3; ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t sa = ring0 + (uint32_t)r.s * STAGE_BYTES;
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        const uint64_t dw = umma_desc(sa + (k >> 2) * (W_BYTES / 2)), dx = umma_desc(sa + W_BYTES + (k >> 2) * (X_BYTES / 2));
                        umma_bf16(d_tmem, dw + 2 * (k & 3), dx + 2 * (k & 3), idesc, (i | k) != 0);
                    }
                    umma_commit(&empty[r.s]);
                }
                if (!ok) break;
                umma_commit(&tfull[buf]);
                u += n;
            }
            if (s_err) drain(empty, STAGES, r.s, r.phase);
        }
    } else if (warp == 2) {
        if (lane == 0) {
            pdl_wait();
            Ring<STAGES> r;
            int kb = u_begin % nkb;
            const int n_grp = w.n_grp;
            const bool dense = EPI != EPI_QKV || w.dense;
            for (int u = u_begin; u < u_end && !s_err; ++u, r.next()) {
                if (!mbar_wait(&empty[r.s], r.phase ^ 1)) { s_err = 4; break; }
                unsigned char *dst = ring + (size_t)r.s * STAGE_BYTES + W_BYTES;
                mbar_expect_tx(&full[r.s], dense ? X_BYTES : n_grp * 4096);
#pragma unroll
                for (int k = 0; k < 2; ++k, dst += X_BYTES / 2) {
                    const int x = kb * BK + 64 * k;
                    if (!dense) {
                        for (int g = 0; g < n_grp; ++g) {
                            const int src = w.grp[g].src;
                            tma_load_2d(dst + g * 1024, &maps.x, x, src, &full[r.s]);
                            tma_load_2d(dst + X_BYTES / 4 + g * 1024, &maps.xl, x, src, &full[r.s]);
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < NP; q += 16) {
                            tma_load_2d(dst + q * 128, &maps.x, x, q, &full[r.s]);
                            tma_load_2d(dst + X_BYTES / 4 + q * 128, &maps.xl, x, q, &full[r.s]);
                        }
                    }
                }
                if (++kb == nkb) kb = 0;
            }
            if (s_err) drain(full, STAGES, r.s, r.phase);
        }
    } else if (warp >= 4) {
        const int q = warp & 3, half = (warp - 4) >> 2, et = threadIdx.x - 128, rr = q * 32 + lane;
        pdl_wait();
        for (int col = warp - 4; col < NP; col += 8) {
            const int g = col >> 3, c = w.grp[g].row + (col & 7);
            const bool live = g < w.n_grp && (col & 7) < w.grp[g].n;
            const RowDesc rd = a.plan.rows[live ? c : 0];
            const int src = (int)stack_row(D, a.layer - 1, rd.seq, rd.slot);
            float s = 0.f;
            if (XCH && live) {
                // 1/rms from the producer's partial sums of squares
                const float *ss = EPI == EPI_GATEUP ? a.B.SSM + (size_t)c * D.n_sst : a.B.SS + (size_t)src * D.n_sst;
                for (int i = lane; i < D.n_sst; i += 32) s += ldg_cg_f32(ss + i);
            }
            s = warp_sum(s);
            if (lane == 0) {
                ci.src[col] = src;
                ci.dst[col] = src + D.B * D.S;
                ci.er[col] = rd.seq * D.S + rd.slot;
                ci.pos[col] = rd.pos;
                if (EPI == EPI_QKV) ci.kv[col] = (a.B.PT[rd.seq * D.pages_per_seq + (rd.pos >> 4)] * D.L + (a.layer - 1)) * D.nkv;
                ci.rs[col] = rsqrtf(s / (float)D.d + D.eps);
            }
        }
        bar_epi();
        const int c_lo = half * (NP / 2), c_hi = min(c_lo + NP / 2, 8 * w.n_grp);
        int piece = 0, turn = 0;
        for (int u = u_begin; u < u_end; ++piece) {
            const int tile = u / nkb, kb0 = u - tile * nkb, n = min(nkb - kb0, u_end - u), buf = piece & 1;
            const bool whole = n == nkb;
            // the CTAs that share a cut tile, and where the first of them leaves its part: a CTA's cut tiles are the one its
            // range starts in (slot 0) and the one it ends in (slot 1)
            int first = cta, last = cta, slot0 = 0;
            if (!whole) {
                first = unit_cta(tile * nkb, U, G);
                last = unit_cta(tile * nkb + nkb - 1, U, G);
                slot0 = unit_start(first, U, G) != tile * nkb;
            }
            float p[8], p2[8], ga = 0.f, gb = 0.f;
            if (EPI == EPI_OPROJ || EPI == EPI_DOWN) {
                const int o = min(tile * BM + rr, D.d - 1);
                if (a.gain_a) ga = bf16_to_f(a.gain_a[o]);
                if (EPI == EPI_DOWN && a.gain_b) gb = bf16_to_f(a.gain_b[o]);
            }
            if (c_lo < c_hi) epi_loads<NP, EPI>(w, ci, tile, rr, c_lo, p, p2);
            bool ok = !s_err;
            if (ok && !mbar_wait(&tfull[buf], (piece >> 1) & 1)) { s_err = 5; ok = false; }
            if (!bar_epi_and(ok)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 2 * NP);
            if (whole) {
                for (int c0 = c_lo; c0 < c_hi; c0 += 8, ++turn) {
                    float v[8];
                    if (c0 != c_lo) epi_loads<NP, EPI>(w, ci, tile, rr, c0, p, p2);
                    __syncwarp();
                    tmem_ld_sum8(taddr + (uint32_t)c0, NP, v);
                    finish<NP, EPI>(w, ci, tile, rr, half, c0, v, p, p2, ga, gb, xch[XCH ? 2 * half + (turn & 1) : 0]);
                }
            } else {
                float *mine = w.part + ((size_t)(2 * cta + (u == u_begin ? 0 : 1)) * NP) * BM + rr * 8;
                for (int c0 = c_lo; c0 < c_hi; c0 += 8) {
                    float v[8];
                    __syncwarp();
                    tmem_ld_sum8(taddr + (uint32_t)c0, NP, v);
                    float4 *o = reinterpret_cast<float4 *>(mine + (size_t)c0 * BM);
                    __stcg(o, make_float4(v[0], v[1], v[2], v[3]));
                    __stcg(o + 1, make_float4(v[4], v[5], v[6], v[7]));
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[buf]);
            if (!whole) {
                bar_epi();                                            // (also: everybody has read the last cut tile's s_last)
                if (et == 0) {
                    int old;
                    asm volatile("atom.add.acq_rel.gpu.s32 %0, [%1], 1;" : "=r"(old) : "l"(w.ticket + tile) : "memory");
                    s_last = old == last - first;
                    if (old == last - first) w.ticket[tile] = 0;
                }
                bar_epi();
                if (s_last) {
                    for (int c0 = c_lo; c0 < c_hi; c0 += 8, ++turn) {
                        float v[8];
                        if (c0 != c_lo) epi_loads<NP, EPI>(w, ci, tile, rr, c0, p, p2);
#pragma unroll
                        for (int e = 0; e < 8; ++e) v[e] = 0.f;
                        for (int b = first; b <= last; b += WT_PIECES) {      // ascending K; one latency per WT_PIECES parts
                            float4 x[WT_PIECES][2];
#pragma unroll
                            for (int i = 0; i < WT_PIECES; ++i) {
                                const int c = b + i;
                                const int slot = c == first ? slot0 : 0;
                                const float4 *s = reinterpret_cast<const float4 *>(w.part + ((size_t)(2 * c + slot) * NP + c0) * BM + rr * 8);
                                x[i][0] = c <= last ? __ldcg(s) : make_float4(0.f, 0.f, 0.f, 0.f);
                                x[i][1] = c <= last ? __ldcg(s + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
                            }
#pragma unroll
                            for (int i = 0; i < WT_PIECES; ++i) {
                                v[0] += x[i][0].x; v[1] += x[i][0].y; v[2] += x[i][0].z; v[3] += x[i][0].w;
                                v[4] += x[i][1].x; v[5] += x[i][1].y; v[6] += x[i][1].z; v[7] += x[i][1].w;
                            }
                        }
                        finish<NP, EPI>(w, ci, tile, rr, half, c0, v, p, p2, ga, gb, xch[XCH ? 2 * half + (turn & 1) : 0]);
                    }
                }
            }
            u += n;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TM_COLS) : "memory");
    }
    if (threadIdx.x == 0 && s_err) atomicMax(a.B.ERR, (int)s_err);
}

template <int NP> constexpr size_t smem_bytes() { return (size_t)stages<NP>() * (W_BYTES + x_bytes<NP>()) + 1024; }

template <int NP, int EPI> cudaError_t prepare_np() {
    static SmemAttrOnce attr;
    return attr.set(rowgemm_tc_kernel<NP, EPI>, (int)smem_bytes<NP>());
}

template <int NP> cudaError_t prepare_rows() {
    for (cudaError_t e : {prepare_np<NP, EPI_QKV>(), prepare_np<NP, EPI_OPROJ>(), prepare_np<NP, EPI_GATEUP>(), prepare_np<NP, EPI_DOWN>()})
        if (e != cudaSuccess) return e;
    return cudaSuccess;
}

template <int NP, int EPI>
cudaError_t launch_np(const WtMaps &maps, const WtArgs &w, int n_sms, cudaStream_t st, bool pdl) {
    const size_t smem = smem_bytes<NP>();
    auto kern = rowgemm_tc_kernel<NP, EPI>;
    {
        cudaError_t e = prepare_np<NP, EPI>();
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(min(min(n_sms, DEL_WT_CTAS), w.n_tiles * w.nkb));
    cfg.blockDim = dim3(WT_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, maps, w);
}

template <int EPI>
cudaError_t launch_epi(const WtMaps &maps, const WtArgs &w, int n_sms, cudaStream_t st, bool pdl) {
    if (w.n_grp <= 2) return launch_np<16, EPI>(maps, w, n_sms, st, pdl);
    if (w.n_grp <= 4) return launch_np<32, EPI>(maps, w, n_sms, st, pdl);
    if (w.n_grp <= 6) return launch_np<48, EPI>(maps, w, n_sms, st, pdl);
    return launch_np<64, EPI>(maps, w, n_sms, st, pdl);
}

// column groups of a launch: for QKV 8 consecutive rows of one sequence each; false if they are more than fit
bool make_groups(const GemmArgs &a, bool dense, WtArgs &w) {
    const PassPlan &p = a.plan;
    w.n_grp = 0;
    w.dense = dense;
    if (dense) {
        for (int r = 0; r < p.m; r += 8) w.grp[w.n_grp++] = {r, r, min(8, p.m - r)};
        return true;
    }
    for (int s = 0; s < p.n_seg; ++s)
        for (int r = 0; r < p.seg[s].nrows; r += 8) {
            if (w.n_grp == DEL_ROWS_MAX / 8) return false;
            const int row = p.seg[s].row0 + r;
            const size_t src = ((size_t)(a.layer - 1) * a.D.B + p.rows[row].seq) * a.D.S + p.rows[row].slot;
            w.grp[w.n_grp++] = {(int32_t)src, row, min(8, p.seg[s].nrows - r)};
        }
    return true;
}

}  // namespace

int rowgemm_tc_tiles(int epi, const Dims &D) {
    switch (epi) {
        case EPI_QKV: return (D.nh * D.hd + BM - 1) / BM + 2 * ((D.nkv * D.hd + BM - 1) / BM);
        case EPI_GATEUP: return (D.F + 63) / 64;
        default: return (D.d + BM - 1) / BM;
    }
}

int rowgemm_tc_ctas(const Dims &D) {
    int most = 0;
    for (int epi = EPI_QKV; epi <= EPI_DOWN; ++epi) {
        const int K = epi == EPI_OPROJ ? D.nh * D.hd : (epi == EPI_DOWN ? D.F : D.d);
        most = max(most, min(DEL_WT_CTAS, rowgemm_tc_tiles(epi, D) * ((K + BK - 1) / BK)));
    }
    return most;
}

bool rowgemm_tc_supported(const Dims &D) {
    const int k = D.F > D.nh * D.hd ? D.F : D.nh * D.hd, kmax = k > D.d ? k : D.d;
    const long long tiles = rowgemm_tc_tiles(EPI_QKV, D) > rowgemm_tc_tiles(EPI_GATEUP, D) ? rowgemm_tc_tiles(EPI_QKV, D) : rowgemm_tc_tiles(EPI_GATEUP, D);
    const long long rows = tiles > rowgemm_tc_tiles(EPI_DOWN, D) ? tiles : rowgemm_tc_tiles(EPI_DOWN, D);
    return (rows * ((kmax + BK - 1) / BK) + 1) * DEL_WT_CTAS < (1ll << 31);
}

cudaError_t rowgemm_tc_prepare() {
    for (cudaError_t e : {prepare_rows<16>(), prepare_rows<32>(), prepare_rows<48>(), prepare_rows<64>()})
        if (e != cudaSuccess) return e;
    return cudaSuccess;
}

bool rowgemm_tc_fits(const GemmArgs &a) {
    WtArgs w;
    return make_groups(a, false, w);
}

// map_w*: 128-byte CUtensorMap blobs made by lmhead_tc_make_map (boxes of 128 rows, W_gate / W_up 64); map_x / map_xl: the
// input's high and low parts by row of the pass (boxes of 16 rows), or, with dense false, the hidden stack (8 rows)
cudaError_t launch_rowgemm_tc(int epi, const GemmArgs &a, const void *map_w0, const void *map_w1, const void *map_w2, const void *map_x,
                              const void *map_xl, bool dense, const WtBuffers &b, int n_sms, cudaStream_t st, bool pdl) {
    WtMaps maps;
    maps.w0 = *reinterpret_cast<const CUtensorMap *>(map_w0);
    maps.w1 = *reinterpret_cast<const CUtensorMap *>(map_w1 ? map_w1 : map_w0);
    maps.w2 = *reinterpret_cast<const CUtensorMap *>(map_w2 ? map_w2 : map_w0);
    maps.x = *reinterpret_cast<const CUtensorMap *>(map_x);
    maps.xl = *reinterpret_cast<const CUtensorMap *>(map_xl);
    WtArgs w;
    memset(&w, 0, sizeof(w));
    w.g = a;
    w.xd = b.xd;
    w.xdl = b.xdl;
    w.part = b.part;
    w.ticket = b.ticket;
    w.n_tiles = rowgemm_tc_tiles(epi, a.D);
    w.nkb = (a.K + BK - 1) / BK;
    if (!make_groups(a, dense, w)) return cudaErrorInvalidValue;
    switch (epi) {
        case EPI_QKV: return launch_epi<EPI_QKV>(maps, w, n_sms, st, pdl);
        case EPI_OPROJ: return launch_epi<EPI_OPROJ>(maps, w, n_sms, st, pdl);
        case EPI_GATEUP: return launch_epi<EPI_GATEUP>(maps, w, n_sms, st, pdl);
        case EPI_DOWN: return launch_epi<EPI_DOWN>(maps, w, n_sms, st, pdl);
    }
    return cudaErrorInvalidValue;
}
