// A whole pass of up to 64 rows through layers l_begin .. l_end in ONE kernel: QKV, attention, O-projection, gate / up and
// down of every layer, on tcgen05 with the weights as the M operand.
//
// What bounds it: HBM (every weight byte once per pass), and the chain of dependences through it.  Launched one by one, the
// five kernels of a layer stop the weight stream five times: a launch drains, the next one's first loads, its wait for the
// producer and its merge run with HBM idle.  Here one thread per SM requests the CTA's weight blocks of all layers in order,
// as far ahead as the ring holds (144-192 KB per SM, about 4 us of HBM's time): weights depend on nobody, so HBM works while
// a phase's last sums are merged and while attention runs.
//
// GEMM phases.  Tile: 128 weight rows (MMA M) x NP activation rows (8..64), K blocks of 128 (two 128-byte swizzle spans).
// The activations' high and low parts lie behind one another in shared memory and are the 2 NP columns of one MMA; the two
// column halves are added when the accumulator is read.  All (tile, K block) units of a phase are cut into one contiguous
// range per CTA; a tile cut by a range boundary is finished by whichever of its CTAs arrives last: each leaves its partial
// sums in the workspace, takes a ticket, and the last one adds all parts in K order.  One accumulator takes 32 steps of the
// tensor core's running sum; the epilogue warps add the accumulators of a part in fp32.
//
// Attention: the 8 epilogue warps run the tasks (segment, kv head, key range) of attention_body.cuh, one or more per CTA.
//
// Order: a counter per kind of phase counts finished tiles (attention: finished (segment, kv head) pairs); whoever reads a
// phase's outputs waits until the count says that all are there (release by the finishing CTA, acquire by the reader, with
// proxy fences on both sides where TMA reads them).  The counts only grow; the host passes their values before the launch.
// Partial sums alternate between two buffers from phase to phase: a CTA that starts phase p + 2 has seen an output of
// phase p + 1, which needed every output of phase p, so nobody still reads the parts of phase p.  All CTAs must be resident
// at once: the launch is cooperative.  Every wait is bounded; a CTA that gives up drains what it has in flight and leaves.
//
// Roles (384 threads): warp 0 streams weight blocks with TMA, warp 2 the activation rows, warp 1 issues the MMAs, warps
// 4-11 run the epilogues (one thread per weight row; groups of 8 columns alternate between their two halves) and attention.
#pragma once

#include <cuda.h>

#include <cstring>
#include <initializer_list>

#include "attention_body.cuh"
#include "kernels.h"
#include "tc_common.cuh"

namespace pass {

using namespace tc;

constexpr int BM = 128, BK = 128, W_BYTES = BM * BK * 2;
constexpr int THREADS = 384;
constexpr int PIECES = 8;                   // partial sums of a cut tile that are loaded at once
// A part's running sums: NI accumulators take its MMA steps in turn, 32 steps each, so SUB K blocks at a time; NACC such sets in
// tensor memory
template <int NP> __host__ __device__ constexpr int n_ileave() { return NP <= 32 ? 4 : 2; }
template <int NP> __host__ __device__ constexpr int n_acc() { return NP <= 16 ? 4 : 2; }
template <int NP> __host__ __device__ constexpr int sub_blocks() { return 4 * n_ileave<NP>(); }
// registers per thread: 168 at launch; the roles keep 72, the epilogue warps take 216 (128 * 72 + 256 * 216 = 384 * 168)
constexpr int REGS_LAUNCH = 168;

template <int NP> __host__ __device__ constexpr int x_bytes() { return 2 * NP * BK * 2; }
template <int NP> __host__ __device__ constexpr int stages() { return NP <= 8 ? 5 : (NP <= 32 ? 4 : 3); }

struct Maps {                    // PassTcMaps
    CUtensorMap x[4], xl[4];
};
static_assert(sizeof(Maps) == sizeof(PassTcMaps), "");

__device__ __forceinline__ void bar_epi() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void bar_half(int half) { asm volatile("bar.sync %0, 128;" ::"r"(2 + half) : "memory"); }
// barrier of the epilogue warps that also tells whether all of them said yes (so that they give up together)
__device__ __forceinline__ bool bar_epi_and(bool yes) {
    uint32_t all;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, 1, 256, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(all) : "r"((uint32_t)yes) : "memory");
    return all != 0;
}
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ void count_up(int32_t *p) { asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p) : "memory"); }
// bounded waits: false when the limit is reached or another role of the CTA has given up
__device__ __forceinline__ bool wait_bar(uint64_t *b, uint32_t parity, const volatile int &err) {
    for (uint32_t i = 0; i < WAIT_LIMIT; ++i) {
        if (mbar_try(b, parity)) return true;
        if ((i & 31) == 31 && err) return false;
    }
    return false;
}
__device__ __forceinline__ bool wait_count(const int32_t *p, int32_t want, const volatile int &err) {
    for (int i = 0; i < (1 << 21); ++i) {
        int32_t v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        if (v - want >= 0) return true;
        if ((i & 31) == 31 && err) return false;
    }
    return false;
}

// eight columns of the products with the high parts plus the same columns of those with the low parts
__device__ __forceinline__ void tmem_add_sum8(uint32_t taddr, uint32_t low, float (&v)[8]) {
    uint32_t r[8], s[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr) : "memory");
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3]), "=r"(s[4]), "=r"(s[5]), "=r"(s[6]), "=r"(s[7])
                 : "r"(taddr + low) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] += __uint_as_float(r[e]) + __uint_as_float(s[e]);
}

// position in the ring: stage and the parity of its current use
template <int N> struct Ring {
    int s = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void next() {
        if (++s == N) { s = 0; phase ^= 1; }
    }
};

// A phase's U units are cut among the first G = min(CTAs, U) of the CTAs: CTA c's are [start(c), start(c + 1)); the CTA that
// holds unit u (units x CTAs stay below 2^31: rowgemm_tc_supported)
__device__ __forceinline__ int unit_start(int c, int U, int G) { return (int)((uint32_t)min(c, G) * (uint32_t)U / (uint32_t)G); }
__device__ __forceinline__ int unit_cta(int u, int U, int G) { return (int)(((uint32_t)(u + 1) * (uint32_t)G - 1) / (uint32_t)U); }

// matrix of a QKV tile (0, 1, 2: q, k, v) and the tile's number inside it
__device__ __forceinline__ int qkv_tile(const Dims &D, int tile, int &local) {
    const int nq = (D.nh * D.hd + BM - 1) >> 7, nk = (D.nkv * D.hd + BM - 1) >> 7;
    const int which = tile < nq ? 0 : (tile < nq + nk ? 1 : 2);
    local = tile - (which == 0 ? 0 : (which == 1 ? nq : nq + nk));
    return which;
}

// a CTA's units through all layers and phases of the launch, in order
struct Units {
    int l, ph, u, end, tile, kb, nkb;
    __device__ __forceinline__ void seek(const PassTcArgs &w, int cta, int n_cta) {
        for (; l <= w.l_end; step()) {
            nkb = w.nkb[ph];
            const int U = w.tiles[ph] * nkb, G = min(n_cta, U);
            u = unit_start(cta, U, G);
            end = unit_start(cta + 1, U, G);
            if (u < end) {
                tile = u / nkb;
                kb = u - tile * nkb;
                return;
            }
        }
    }
    __device__ __forceinline__ void step() {
        if (++ph == 4) { ph = 0; ++l; }
    }
    __device__ __forceinline__ void next(const PassTcArgs &w, int cta, int n_cta) {
        if (++kb == nkb) { kb = 0; ++tile; }
        if (++u == end) {
            step();
            seek(w, cta, n_cta);
        }
    }
};

// the weight block of unit `it`
__device__ __forceinline__ void load_weights(const PassTcArgs &w, const Units &it, unsigned char *dst, uint64_t *bar) {
    const PassLayer &L = w.layers[it.l - 1];
    int which, row;
    if (it.ph == EPI_QKV) {
        which = qkv_tile(w.D, it.tile, row);
        row *= BM;
    } else {
        which = it.ph == EPI_OPROJ ? 3 : (it.ph == EPI_GATEUP ? 4 : 6);
        row = it.tile * (it.ph == EPI_GATEUP ? BM / 2 : BM);
    }
    const CUtensorMap *map = reinterpret_cast<const CUtensorMap *>(L.w[which]);
#pragma unroll
    for (int k = 0; k < 2; ++k, dst += W_BYTES / 2) {
        const int x = it.kb * BK + 64 * k;
        tma_load_2d(dst, map, x, row, bar);
        if (it.ph == EPI_GATEUP) tma_load_2d(dst + W_BYTES / 4, map + 1, x, row, bar);      // boxes of 64 rows: gate, then the same rows of up
    }
}

// per column = row of the pass: where its outputs go; filled once per launch (rs: per phase)
template <int NP> struct ColInfo {
    int er[NP];                  // row of the exit buffers, and of a layer's part of the hidden stack
    int kv[NP];                  // page * L * nkv
    int pos[NP];
    float rs[NP];                // 1/rms
};

// what an epilogue reads for 8 columns at this thread's feature, requested before the sums are there: the residual
// (O-projection, DOWN) or the rotation's cos and sin (QKV)
template <int NP, int HD, int EPI>
__device__ __forceinline__ void epi_loads(const PassTcArgs &w, const ColInfo<NP> &ci, int layer, int tile, int rr, int col, float (&p)[8], float (&p2)[8]) {
    const Dims &D = w.D;
    const int n = w.plan.m - col;
    if (EPI == EPI_OPROJ || EPI == EPI_DOWN) {
        const int o = tile * BM + rr;
        const size_t base = (size_t)(layer - 1) * D.B * D.S;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float *h = EPI == EPI_OPROJ ? w.B.H + (base + (e < n ? ci.er[col + e] : 0)) * D.d + o : w.B.HM + (size_t)(col + e) * D.d + o;
            p[e] = e < n && o < D.d ? ldg_cg_f32(h) : 0.f;
        }
    } else if (EPI == EPI_QKV) {
        int local;
        const bool rot = qkv_tile(D, tile, local) < 2;
        constexpr int hh = HD >> 1;
        const int j = rr & (hh - 1);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const size_t at = (size_t)(e < n ? ci.pos[col + e] : 0) * hh + j;
            p[e] = e < n && rot ? __ldg(w.B.rope_cos + at) : 0.f;
            p2[e] = e < n && rot ? __ldg(w.B.rope_sin + at) : 0.f;
        }
    }
}

// 8 finished columns of a tile: rr = weight row of the tile, ga / gb = the norm gains of its feature, xch = exchange buffer
// of this half's 4 warps
template <int NP, int HD, int EPI>
__device__ __forceinline__ void finish(const PassTcArgs &w, const ColInfo<NP> &ci, int layer, int tile, int rr, int half, int col, const float (&acc)[8],
                                       const float (&p)[8], const float (&p2)[8], const bf16 *gain_a, float ga, const bf16 *gain_b, float gb, float (*xch)[BM]) {
    const Dims &D = w.D;
    const Buffers &B = w.B;
    const int n = w.plan.m - col;
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
            bf16 hi, lo;
            split_bf16(v[e] * ga, hi, lo);
            const size_t i = (size_t)(col + e) * D.d + o;
            if (EPI == EPI_OPROJ) {
                B.HM[i] = v[e];
                B.XM[i] = hi;
                B.XML[i] = lo;
                if ((rr & 15) == 0) B.SSM[(size_t)(col + e) * D.n_sst + (o >> 4)] = ss[e];
            } else {
                const size_t er = ci.er[col + e], sr = (size_t)layer * D.B * D.S + er;
                B.H[sr * D.d + o] = v[e];
                if (gain_a) {
                    if (layer == w.l_end) {                           // the next pass gathers its rows from the stack
                        B.XS[sr * D.d + o] = hi;
                        B.XSL[sr * D.d + o] = lo;
                    } else {
                        w.xd[i] = hi;
                        w.xdl[i] = lo;
                    }
                }
                if (gain_b) B.XE[er * D.d + o] = __float2bfloat16_rn(v[e] * gb);
                if ((rr & 15) == 0) {
                    B.SS[sr * D.n_sst + (o >> 4)] = ss[e];
                    if (gain_b) B.SSE[er * D.n_sst + (o >> 4)] = ss[e];
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
        const int partner = rr ^ (EPI == EPI_GATEUP ? 64 : HD >> 1);
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
            const int e = up ? 4 + i : i;
            if (e >= n) continue;
            const float g = up ? other[4 + i] : mine[i], u = up ? mine[4 + i] : other[i];
            const float act = g / (1.f + __expf(-g)) * u;
            split_bf16(act, B.ACT[(size_t)(col + e) * D.F + f], B.ACTL[(size_t)(col + e) * D.F + f]);
        }
        return;
    }
    const int f = local * BM + rr, head = f / HD, dim = f & (HD - 1);
    if (f >= (which == 0 ? D.nh : D.nkv) * HD) return;
    const bool lo = dim < (HD >> 1);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        if (e >= n) continue;
        // first half: v_j cos - v_(j + half) sin; second half: v_(j + half) cos + v_j sin
        const float out = which == 2 ? mine[e] : (lo ? mine[e] * p[e] - other[e] * p2[e] : mine[e] * p[e] + other[e] * p2[e]);
        const bf16 v = __float2bfloat16_rn(out);
        const size_t page = (size_t)ci.kv[col + e] + (size_t)(layer - 1) * D.nkv + head;
        const int sl = ci.pos[col + e] & 15;
        if (which == 0) B.Q[(size_t)(col + e) * (D.nh * HD) + f] = v;
        else if (which == 1) B.KP[(page * 16 + sl) * HD + dim] = v;
        else B.VP[(page * HD + dim) * 16 + sl] = v;
    }
}

// attention_body.cuh on the 8 epilogue warps
template <int NP> struct EpiWarps {
    static constexpr int T0 = THREADS - 256;
    static constexpr int FEW = NP <= 16 ? 1 : 2, MANY = NP <= 16 ? 2 : 4;
    const int32_t *count;        // finished QKV tiles
    int32_t want;
    volatile int *err;
    __device__ __forceinline__ void sync() const { bar_epi(); }
    __device__ __forceinline__ bool ready(const AttnView &) const {
        bool ok = true;
        if (threadIdx.x == T0 && !wait_count(count, want, *err)) {
            *err = 7;
            ok = false;
        }
        return bar_epi_and(ok);
    }
};
// the epilogue warps' shared memory: merge of attention's outputs, or the exchange buffers [half][turn & 1][8][128]
template <int NP, int HD> __host__ __device__ constexpr size_t scratch_bytes() {
    const size_t a = attn::merge_bytes<EpiWarps<NP>>(HD), x = sizeof(float) * 4 * 8 * BM;
    return ((a > x ? a : x) + 15) & ~(size_t)15;
}

// state of an epilogue thread that runs on from phase to phase
struct EpiState { int acc = 0, turn = 0; };

// The epilogue of one phase.  false: the CTA gives up.
template <int NP, int HD, int EPI>
__device__ __forceinline__ bool epilogue(const PassTcArgs &w, const ColInfo<NP> &ci, float (*xch)[8][BM], int layer, EpiState &es, uint32_t tmem_base,
                                         uint64_t *tfull, uint64_t *tempty, volatile int &s_err, int &s_last) {
    constexpr int NG = (NP / 8 + 1) / 2;                              // groups of 8 columns of a half
    constexpr int SUB = sub_blocks<NP>(), NACC = n_acc<NP>(), NI = n_ileave<NP>();
    constexpr bool XCH = EPI == EPI_QKV || EPI == EPI_GATEUP;
    const Dims &D = w.D;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp & 3, half = (warp - 4) >> 2, et = threadIdx.x - 128, rr = q * 32 + lane;
    const int cta = (int)blockIdx.x, nkb = w.nkb[EPI], U = w.tiles[EPI] * nkb, G = min((int)gridDim.x, U);
    const int u_begin = unit_start(cta, U, G), u_end = unit_start(cta + 1, U, G);
    const bf16 *gain_a = EPI == EPI_OPROJ ? w.layers[layer - 1].ffn_gain : w.layers[layer - 1].next_gain;
    const bf16 *gain_b = EPI == EPI_DOWN && layer == w.l_end ? w.exit_gain : nullptr;
    const int m = w.plan.m;
    for (int u = u_begin; u < u_end;) {
        const int tile = u / nkb, kb0 = u - tile * nkb, n = min(nkb - kb0, u_end - u);
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
            if (gain_a) ga = bf16_to_f(gain_a[o]);
            if (gain_b) gb = bf16_to_f(gain_b[o]);
        }
        if (8 * half < m) epi_loads<NP, HD, EPI>(w, ci, layer, tile, rr, 8 * half, p, p2);
        float v[NG][8];
#pragma unroll
        for (int g = 0; g < NG; ++g)
#pragma unroll
            for (int e = 0; e < 8; ++e) v[g][e] = 0.f;
        bool ok = true;
        for (int i = 0; i < n; i += SUB, ++es.acc) {
            const int buf = es.acc % NACC;
            if (ok && !wait_bar(&tfull[buf], (es.acc / NACC) & 1, s_err)) { s_err = 5; ok = false; }
            if (!ok) continue;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            __syncwarp();
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const int c0 = 8 * (2 * g + half);
                if (c0 >= m) continue;
#pragma unroll
                for (int j = 0; j < NI; ++j) tmem_add_sum8(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)((buf * NI + j) * 2 * NP + c0), NP, v[g]);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[buf]);
        }
        bool fin = whole;
        if (!whole) {
            float *mine = w.part + ((size_t)((EPI & 1) * (int)gridDim.x * 2 + 2 * cta + (u == u_begin ? 0 : 1)) * NP) * BM + rr * 8;
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const int c0 = 8 * (2 * g + half);
                if (c0 >= m) continue;
                float4 *o = reinterpret_cast<float4 *>(mine + (size_t)c0 * BM);
                __stcg(o, make_float4(v[g][0], v[g][1], v[g][2], v[g][3]));
                __stcg(o + 1, make_float4(v[g][4], v[g][5], v[g][6], v[g][7]));
            }
        }
        if (!bar_epi_and(ok)) return false;                           // (also: everybody has read the last cut tile's s_last)
        if (!whole) {
            if (et == 0) {
                int32_t *ticket = w.ticket + EPI * w.n_tickets + tile;
                int old;
                asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(old) : "l"(ticket) : "memory");
                s_last = old == last - first;
                if (old == last - first) *ticket = 0;
            }
            bar_epi();
            fin = s_last;
        }
        if (fin) {
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const int c0 = 8 * (2 * g + half);
                if (c0 >= m) continue;
                if (!whole) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[g][e] = 0.f;
                    for (int b = first; b <= last; b += PIECES) {     // ascending K; one latency per PIECES parts
                        float4 x[PIECES][2];
#pragma unroll
                        for (int i = 0; i < PIECES; ++i) {
                            const int c = b + i;
                            const int slot = c == first ? slot0 : 0;
                            const float4 *s = reinterpret_cast<const float4 *>(w.part + ((size_t)((EPI & 1) * (int)gridDim.x * 2 + 2 * c + slot) * NP + c0) * BM + rr * 8);
                            x[i][0] = c <= last ? __ldcg(s) : make_float4(0.f, 0.f, 0.f, 0.f);
                            x[i][1] = c <= last ? __ldcg(s + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
#pragma unroll
                        for (int i = 0; i < PIECES; ++i) {
                            v[g][0] += x[i][0].x; v[g][1] += x[i][0].y; v[g][2] += x[i][0].z; v[g][3] += x[i][0].w;
                            v[g][4] += x[i][1].x; v[g][5] += x[i][1].y; v[g][6] += x[i][1].z; v[g][7] += x[i][1].w;
                        }
                    }
                }
                if (g != 0) epi_loads<NP, HD, EPI>(w, ci, layer, tile, rr, c0, p, p2);
                finish<NP, HD, EPI>(w, ci, layer, tile, rr, half, c0, v[g], p, p2, gain_a, ga, gain_b, gb, xch[XCH ? 2 * half + (es.turn & 1) : 0]);
                ++es.turn;
            }
            proxy_fence();                                            // the next phase reads these outputs with TMA
            bar_epi();
            if (et == 0) count_up(w.count + EPI);
        }
        u += n;
    }
    return true;
}

template <int NP, int HD>
__global__ void __launch_bounds__(THREADS, 1) pass_kernel(const __grid_constant__ Maps maps, const __grid_constant__ PassTcArgs w) {
    constexpr int X_BYTES = x_bytes<NP>(), STAGES = stages<NP>(), STAGE_BYTES = W_BYTES + X_BYTES;
    constexpr int SUB = sub_blocks<NP>(), NACC = n_acc<NP>(), NI = n_ileave<NP>();
    constexpr uint32_t ACC_COLS = 2 * NP * NACC * NI, TM_COLS = ACC_COLS <= 256 ? 256 : 512;
    extern __shared__ unsigned char smem_dyn[];
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], tfull[NACC], tempty[NACC];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int s_err;
    __shared__ int s_last;
    __shared__ ColInfo<NP> ci;
    unsigned char *ring = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
    float *scratch = reinterpret_cast<float *>(ring + (size_t)STAGES * STAGE_BYTES);
    const Dims &D = w.D;
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;      // (the same in all lanes, visibly)
    const int G = (int)gridDim.x, cta = (int)blockIdx.x;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 2); mbar_init(&empty[s], 1); }
        for (int b = 0; b < NACC; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], 8); }
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

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
        if (warp == 0 && lane == 0) {
            Ring<STAGES> r;
            Units it;
            it.l = w.l_begin;
            it.ph = 0;
            it.seek(w, cta, G);
            for (; it.l <= w.l_end && !s_err; it.next(w, cta, G), r.next()) {
                if (!wait_bar(&empty[r.s], r.phase ^ 1, s_err)) { s_err = 1; break; }
                mbar_expect_tx(&full[r.s], W_BYTES);
                load_weights(w, it, ring + (size_t)r.s * STAGE_BYTES, &full[r.s]);
            }
            if (s_err) drain(full, STAGES, r.s, r.phase);
        } else if (warp == 1) {
            // The whole warp runs this loop and one lane issues: addresses and descriptors then stay in uniform registers (issue
            // by a single thread's code takes 0.64 us for a unit's 8 MMAs, about as long as HBM takes for the unit).
            // fp32 accumulate, bf16 x bf16, both operands K-major, N = 2 NP, M = 128
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NP >> 2) << 17) | ((uint32_t)(BM >> 4) << 24);
            const uint32_t ring0 = smem_u32(ring);
            Ring<STAGES> r;
            Units it;
            it.l = w.l_begin;
            it.ph = 0;
            it.seek(w, cta, G);
            bool ok = true;
            for (int acc = 0; it.l <= w.l_end && ok; ++acc) {
                // (a part of a tile starts new accumulators: the epilogue counts in the same way)
                const int n = min(min(it.nkb - it.kb, it.end - it.u), SUB), buf = acc % NACC;
                if (!__all_sync(0xffffffffu, wait_bar(&tempty[buf], ((acc / NACC) & 1) ^ 1, s_err))) { s_err = 2; ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * NI * 2 * NP);
                for (int i = 0; i < n; ++i, it.next(w, cta, G), r.next()) {
                    if (!__all_sync(0xffffffffu, wait_bar(&full[r.s], r.phase, s_err))) { s_err = 3; ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t sa = ring0 + (uint32_t)r.s * STAGE_BYTES;
                    const uint64_t dw = umma_desc(sa), dx = umma_desc(sa + W_BYTES);       // (addresses in units of 16 bytes)
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k)
                            umma_bf16(d_tmem + (k % NI) * 2 * NP, dw + (k >> 2) * (W_BYTES / 32) + 2 * (k & 3), dx + (k >> 2) * (X_BYTES / 32) + 2 * (k & 3),
                                      idesc, i != 0 || k >= NI);
                        umma_commit(&empty[r.s]);
                    }
                    __syncwarp();
                }
                if (!ok) break;
                if (elect_one()) umma_commit(&tfull[buf]);
                __syncwarp();
            }
            if (s_err) drain(empty, STAGES, r.s, r.phase);
        } else if (warp == 2 && lane == 0) {
            pdl_wait();
            Ring<STAGES> r;
            Units it;
            it.l = w.l_begin;
            it.ph = 0;
            it.seek(w, cta, G);
            int seen = -1;
            for (; it.l <= w.l_end && !s_err; it.next(w, cta, G), r.next()) {
                const int at = 4 * it.l + it.ph;
                if (at != seen) {
                    // all outputs of the phase before: QKV reads DOWN's (of the layer before), O attention's, gate / up O's, ...
                    seen = at;
                    const int c = it.ph == EPI_QKV ? EPI_DOWN : (it.ph == EPI_OPROJ ? PASS_ATT : it.ph - 1);
                    if (!wait_count(w.count + c, w.base[c] + (it.l - w.l_begin + 1) * w.step[c], s_err)) { s_err = 6; break; }
                    proxy_fence();
                }
                if (!wait_bar(&empty[r.s], r.phase ^ 1, s_err)) { s_err = 4; break; }
                unsigned char *dst = ring + (size_t)r.s * STAGE_BYTES + W_BYTES;
                mbar_expect_tx(&full[r.s], X_BYTES);
#pragma unroll
                for (int k = 0; k < 2; ++k, dst += X_BYTES / 2) {
                    const int x = it.kb * BK + 64 * k;
                    tma_load_2d(dst, &maps.x[it.ph], x, 0, &full[r.s]);
                    tma_load_2d(dst + X_BYTES / 4, &maps.xl[it.ph], x, 0, &full[r.s]);
                }
            }
            if (s_err) drain(full, STAGES, r.s, r.phase);
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        const int et = threadIdx.x - 128, ew = warp - 4, m = w.plan.m;
        float (*xch)[8][BM] = reinterpret_cast<float (*)[8][BM]>(scratch);
        const AttnPrefetch no_pf = {};
        pdl_wait();
        // the input of the first layer, by row of the pass
        const size_t stack0 = (size_t)(w.l_begin - 1) * D.B * D.S;
        for (int t = cta; t < w.tiles[EPI_DOWN]; t += G) {
            const int f = t * BM + (et & 15) * 8;
            if (f < D.d)
                for (int c = et >> 4; c < m; c += 16) {
                    const size_t src = (stack0 + (size_t)w.plan.rows[c].seq * D.S + w.plan.rows[c].slot) * D.d + f, dst = (size_t)c * D.d + f;
                    *reinterpret_cast<uint4 *>(w.xd + dst) = ldg_act16(w.B.XS + src);
                    *reinterpret_cast<uint4 *>(w.xdl + dst) = ldg_act16(w.B.XSL + src);
                }
            proxy_fence();
            bar_epi();
            if (et == 0) count_up(w.count + EPI_DOWN);
        }
        for (int c = et; c < m; c += 256) {
            const RowDesc rd = w.plan.rows[c];
            ci.er[c] = rd.seq * D.S + rd.slot;
            ci.pos[c] = rd.pos;
            ci.kv[c] = w.B.PT[rd.seq * D.pages_per_seq + (rd.pos >> 4)] * D.L * D.nkv;
        }
        // waits until counter c stands where its k-th layer of this launch leaves it
        auto done = [&](int c, int k, int code) {
            bool ok = true;
            if (et == 0 && !wait_count(w.count + c, w.base[c] + k * w.step[c], s_err)) {
                s_err = code;
                ok = false;
            }
            return bar_epi_and(ok);
        };
        // 1/rms of every row from the producer's partial sums of squares
        auto scales = [&](const float *ss, bool by_row) {
            for (int c = ew; c < m; c += 8) {
                const float *s = ss + (size_t)(by_row ? c : ci.er[c]) * D.n_sst;
                float sum = 0.f;
                for (int i = lane; i < D.n_sst; i += 32) sum += ldg_cg_f32(s + i);
                sum = warp_sum(sum);
                if (lane == 0) ci.rs[c] = rsqrtf(sum / (float)D.d + D.eps);
            }
            bar_epi();
        };
        const int n_units = w.plan.n_seg * D.nkv * w.n_splits;
        EpiState es;
        for (int l = w.l_begin; l <= w.l_end; ++l) {
            const int k = l - w.l_begin + 1;
            // committed cache pages of this CTA's attention task go to L2 while the QKV weights stream
            if (cta < n_units) {
                const int split = cta % w.n_splits, rest = cta / w.n_splits, kvh = rest % D.nkv, z = rest / D.nkv;
                const Segment seg = w.plan.seg[z];
                const int n_pages = (seg.pos0 + seg.nrows + 15) >> 4, pps = (n_pages + w.n_splits - 1) / w.n_splits;
                const int p_end = min(min(n_pages, (split + 1) * pps), w.early_pos[z] >> 4);
                for (int p = split * pps + et; p < p_end; p += 256) {
                    const size_t off = (((size_t)w.B.PT[seg.seq * D.pages_per_seq + p] * D.L + (l - 1)) * D.nkv + kvh) * 16 * HD;
                    l2_prefetch_bulk(w.B.KP + off, 16 * HD * 2);
                    l2_prefetch_bulk(w.B.VP + off, 16 * HD * 2);
                }
            }
            if (!done(EPI_DOWN, k, 8)) break;
            scales(w.B.SS + (size_t)(l - 1) * D.B * D.S * D.n_sst, false);
            if (!epilogue<NP, HD, EPI_QKV>(w, ci, xch, l, es, tmem_base, tfull, tempty, s_err, s_last)) break;
            bool ok = true;
            for (int i = cta; i < n_units; i += G) {
                const int split = i % w.n_splits, rest = i / w.n_splits, kvh = rest % D.nkv, z = rest / D.nkv;
                const Segment seg = w.plan.seg[z];
                const AttnView av{D, w.B, l, w.early_pos[z], &no_pf};
                const EpiWarps<NP> pol{w.count + EPI_QKV, w.base[EPI_QKV] + k * w.step[EPI_QKV], &s_err};
                const int n_pages = (seg.pos0 + seg.nrows + 15) >> 4, pps = (n_pages + w.n_splits - 1) / w.n_splits;
                ok = attn::partial<HD>(pol, av, scratch, seg, kvh, split * pps, min(n_pages, (split + 1) * pps), 0, 0x7fffffff, split, w.n_splits);
                if (!ok) break;
                bool fin = true;
                if (w.n_splits > 1) {
                    // (tile_end ends with a barrier: all partial states are stored)
                    if (et == 0) {
                        int32_t *ticket = w.B.ACNT + z * D.nkv + kvh;
                        int old;
                        asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(old) : "l"(ticket) : "memory");
                        s_last = old == w.n_splits - 1;
                        if (old == w.n_splits - 1) *ticket = 0;
                    }
                    bar_epi();
                    fin = s_last;
                    if (fin) attn::merge_slots<HD, EpiWarps<NP>>(av, seg, kvh, w.n_splits);
                }
                proxy_fence();
                bar_epi();
                if (fin && et == 0) count_up(w.count + PASS_ATT);
            }
            if (!ok) break;
            if (!epilogue<NP, HD, EPI_OPROJ>(w, ci, xch, l, es, tmem_base, tfull, tempty, s_err, s_last)) break;
            if (!done(EPI_OPROJ, k, 9)) break;
            scales(w.B.SSM, true);
            if (!epilogue<NP, HD, EPI_GATEUP>(w, ci, xch, l, es, tmem_base, tfull, tempty, s_err, s_last)) break;
            if (!epilogue<NP, HD, EPI_DOWN>(w, ci, xch, l, es, tmem_base, tfull, tempty, s_err, s_last)) break;
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TM_COLS) : "memory");
    }
    if (threadIdx.x == 0 && s_err) atomicMax(w.B.ERR, (int)s_err);
}

template <int NP, int HD> constexpr size_t smem_bytes() { return (size_t)stages<NP>() * (W_BYTES + x_bytes<NP>()) + 1024 + scratch_bytes<NP, HD>(); }

// raises the shared-memory limit, and checks that the registers at launch cover the split among the warps (a larger sum would
// wait for ever)
template <int NP, int HD> cudaError_t prepare_np() {
    static SmemAttrOnce attr;
    cudaError_t e = attr.set(pass_kernel<NP, HD>, (int)smem_bytes<NP, HD>());
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, pass_kernel<NP, HD>);
    if (e != cudaSuccess) return e;
    return fa.numRegs == REGS_LAUNCH ? cudaSuccess : cudaErrorInvalidConfiguration;
}

template <int HD> cudaError_t prepare_hd() {
    for (cudaError_t e : {prepare_np<8, HD>(), prepare_np<16, HD>(), prepare_np<32, HD>(), prepare_np<48, HD>(), prepare_np<64, HD>()})
        if (e != cudaSuccess) return e;
    return cudaSuccess;
}

template <int NP, int HD>
cudaError_t launch_np(const Maps &maps, const PassTcArgs &w, int grid, cudaStream_t st, bool pdl) {
    static SmemAttrOnce attr;
    cudaError_t e = attr.set(pass_kernel<NP, HD>, (int)smem_bytes<NP, HD>());
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = smem_bytes<NP, HD>();
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, pass_kernel<NP, HD>, maps, w);
}

template <int HD>
cudaError_t launch_hd(const PassTcMaps &m, const PassTcArgs &w, int np, int grid, cudaStream_t st, bool pdl) {
    Maps maps;
    memcpy(&maps, &m, sizeof(maps));
    switch (np) {
        case 8: return launch_np<8, HD>(maps, w, grid, st, pdl);
        case 16: return launch_np<16, HD>(maps, w, grid, st, pdl);
        case 32: return launch_np<32, HD>(maps, w, grid, st, pdl);
        case 48: return launch_np<48, HD>(maps, w, grid, st, pdl);
        case 64: return launch_np<64, HD>(maps, w, grid, st, pdl);
    }
    return cudaErrorInvalidValue;
}

}  // namespace pass
