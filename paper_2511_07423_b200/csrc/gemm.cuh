// Projection GEMM of the verification step for sm_100a, "swap-AB" orientation:
//   D[feature][token] = sum_k W[feature][k] * X[token][k]
// The weight matrix is the UMMA A operand (M = 128 output features per tile; a CTA normally owns a
// PAIR of such tiles that share one token tile), the ragged token batch is the UMMA B operand
// (N = 16..256 tokens), so a batch of T tokens pads to a multiple of 16 instead of 128.  Weights are
// stored pre-tiled and pre-swizzled ([feature pair][k-block][2][128 x 64] images of the
// 128-byte-swizzled shared-memory tile), so a stage's weights are ONE contiguous bulk copy;
// activations come through a TMA tensor map.  One persistent CTA per SM walks a static schedule.
// Three variants of the kernel (template parameter):
//   GEMM_WAVES  : whole pair tiles in full waves, leftovers as single 128-feature tiles;
//   GEMM_KSPLIT : as above, but the pair tiles left over after the full waves are cut along K into
//                 parts on different CTAs (the "helper" parts run first and store their fp32
//                 accumulators, the "owner" part runs last on another CTA, adds them in part order
//                 and finishes the tile);
//   GEMM_RSPLIT : projections with fewer pair tiles than SMs (o, down, qkv at a few hundred tokens):
//                 every tile's K range is split over S CTAs that run at the same time; each CTA
//                 keeps a contiguous share of the tile's token columns, hands the accumulators of
//                 the other columns to their keepers through global memory, adds what it receives
//                 in split order (so the sum does not depend on timing) and runs the epilogue on
//                 its own columns: a reduce-scatter, after which all S CTAs share the epilogue.
// Every CTA starts its k loop at a different k-block, so the CTAs that share a token tile do not
// ask L2 for the same lines at the same moment.  Accumulation is tcgen05.mma into TMEM, read back
// with tcgen05.ld by twelve or sixteen epilogue warps; a thread then holds one output feature for sixteen
// tokens; a warp turns its 32 x 16 block round in shared memory, so that every lane reads and writes
// 16-byte pieces of token-major rows:
//   EPI_QKV    : RMSNorm scale, RoPE on q and k (the partner dimension sits 16 lanes away), q store,
//                paged-KV append
//   EPI_RESID  : x += D (the residual stream, fp32), the next projection's operand half(x * gain) and
//                the sums of x^2 over each group of 32 features that the next RMSNorm needs
//   EPI_SWIGLU : RMSNorm scale, silu(gate) * up (a gate feature and its up feature sit 16 lanes apart)
//   EPI_LMHEAD : RMSNorm scale, optional logits, vocabulary argmax (warp reduction, packed 64-bit atomicMax)
//   EPI_PLAIN  : fp32 store (test hook)
// RMSNorm is split between producer and consumer: the kernel that writes the residual stream
// (EPI_RESID, or prep_kernel for the first layer) stores half(x * gain) and partial sums of x^2; the
// projection that consumes it multiplies its accumulators by the token's 1/sqrt(mean(x^2) + eps),
// a per-column scalar in this orientation, which its epilogue warps work out from the partial sums
// while the main loop runs.
#pragma once
#include "ptx.cuh"

namespace syn {

enum { EPI_PLAIN = 0, EPI_QKV = 1, EPI_RESID = 2, EPI_SWIGLU = 3, EPI_LMHEAD = 4 };
enum { GEMM_WAVES = 0, GEMM_KSPLIT = 1, GEMM_RSPLIT = 2 };

struct EpiParams {
    int mode;
    int T;  // valid tokens
    int N;  // valid output features (rows of W)
    // PLAIN
    float* y;
    int ldy;
    // QKV
    op16* q;
    int q_dim, kv_dim, hd, n_kv_heads, page_size;
    const float2* rope;  // [T][hd/2] (cos, sin)
    op16* pool;          // this layer's pool: [page][kvh][K|V][row][hd]
    const int* slot;     // [T] page * page_size + row
    // RMSNorm scale of the token operand (QKV, SWIGLU, LMHEAD; NULL: the operand is used as it is)
    const float* ssq_in; // [T][n_ssq] partial sums of x^2 of the operand's source rows
    int n_ssq;           // a multiple of 4
    float inv_d, eps;
    // RESID
    float* x;            // [T][d] residual stream, updated in place
    const __nv_bfloat16* gain;   // [d] gain of the NEXT RMSNorm
    op16* xg;            // [T][d] half(x * gain): the next projection's operand
    float* ssq_out;      // [T][d / 32]
    int d;
    // SWIGLU
    op16* act;
    int f_pad;
    // LMHEAD
    float* logits;
    int vocab;
    unsigned long long* best;
    uint32_t* warp_max;   // NULL, or [T][n_warp_max]: the ordered bit pattern of the largest logit of every
    int n_warp_max;       // 32-feature group of a token (0 for a group without a valid feature)
};

__device__ __forceinline__ uint32_t orderable_f32(float v) {   // monotone map of a float to unsigned
    uint32_t u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ unsigned long long pack_argmax_key(uint32_t key, int idx) {
    return ((unsigned long long)key << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)idx);
}

// Row order inside one packed 128-feature tile.  TMEM lane l of the tile belongs to warp quarter
// q = l / 32; partners that an epilogue combines (the two RoPE halves of a head dimension, a gate
// feature and its up feature) sit 16 lanes apart in the same warp, so they meet by one shuffle.
//   rope tiles (q and k rows): quarter q covers head q / (hd/32) of the tile, dims
//     [16 s, 16 s + 16) for lanes 0..15 and the same dims + hd/2 for lanes 16..31, s = q % (hd/32)
//   gate/up tiles: quarter q lanes 0..15 = gate features 64 b + 16 q + lane, lanes 16..31 = the up
//     features of the same indices (b = tile index)
//   every other tile: feature = tile base + lane
__host__ __device__ __forceinline__ int rope_tile_feature(int l, int hd) {   // offset inside the tile's 128 features
    const int half = hd >> 1, groups = half >> 4, q = l >> 5, ll = l & 31;
    return (q / groups) * hd + 16 * (q % groups) + (ll & 15) + ((ll & 16) ? half : 0);
}

constexpr int GEMM_EPI_WARPS = 16;               // at most: four groups of four (one warp per TMEM lane quarter)

// Epilogue of one 16-token chunk of one warp: a[j] = D[feature of this lane][token t0 + j] (tokens
// j >= ncols are padding), already summed and scaled.  In this orientation a lane holds ONE output
// feature for sixteen tokens, while every output is token-major in memory, so the 32 x 16 block is
// first turned round in a shared-memory scratch of the warp (16 rows of 36 floats: no bank conflicts
// either way).  Afterwards the lanes walk the block row by row: eight neighbouring lanes cover the 32
// columns of one token with four columns each, so that a warp-wide access touches whole 32-byte
// sectors of four tokens' rows (the cost of these epilogues is the number of sectors and of memory
// instructions they issue, not their arithmetic).
// `m0` = first packed row of the tile, `quarter` = warp's TMEM lane quarter.
constexpr int EPI_COLS = 16;
constexpr int EPI_SCR_STRIDE = 36;   // floats: rows stay 16-byte aligned, so that a lane reads its four columns with one load
constexpr int EPI_SCR_FLOATS = EPI_COLS * EPI_SCR_STRIDE;   // per epilogue warp

__device__ __forceinline__ uint2 pack4_op(float a, float b, float c, float d) { return make_uint2(pack_op(a, b), pack_op(c, d)); }

// What an epilogue reads besides the accumulators: the residual rows and the gains (EPI_RESID) or the RoPE rows and KV
// slots (EPI_QKV).  Loaded on its own so that a caller can have it in flight while it waits for the accumulators.
template <int MODE>
struct EpiOperand {
    float4 v[MODE == EPI_QKV ? 8 : (MODE == EPI_RESID ? 4 : 1)];
    uint2 gain;
    int slot;
};

// Loads of data that no kernel beside this one writes, issued where they stand: the compiler moves a plain __ldg down to its
// use, behind the barriers whose wait is to hide it (the o projection of the 1B shape, 5 tokens: a gain that came from HBM held
// the last 1 400 cycles of the kernel).
__device__ __forceinline__ float4 ldg_here(const float4* p) {
    float4 v;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ldg_here(const uint2* p) {
    uint2 v;
    asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ int ldg_here(const int* p) {
    int v;
    asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

template <int MODE>
__device__ __forceinline__ void epi_load_rope(const EpiParams& p, EpiOperand<MODE>& o, int t0, int ncols, int quarter, int lane) {
    const int tq = lane >> 3, c0 = (lane & 7) * 4;
    const int half = p.hd >> 1, dim = 16 * (quarter & ((half >> 4) - 1)) + (c0 & 15);   // lower dim of the pair
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4* cs = reinterpret_cast<const float4*>(p.rope + (size_t)(t0 + tq + 4 * i) * half + dim);   // 4 x (cos, sin)
        const bool tv = tq + 4 * i < ncols;
        o.v[(2 * i) & (MODE == EPI_QKV ? 7 : 0)] = tv ? ldg_here(cs) : make_float4(1.f, 0.f, 1.f, 0.f);
        o.v[(2 * i + 1) & (MODE == EPI_QKV ? 7 : 0)] = tv ? ldg_here(cs + 1) : make_float4(1.f, 0.f, 1.f, 0.f);
    }
}

template <int MODE>
__device__ __forceinline__ void epi_load(const EpiParams& p, EpiOperand<MODE>& o, int m0, int t0, int ncols, int quarter, int lane) {
    const int tq = lane >> 3, c0 = (lane & 7) * 4;
    if (MODE == EPI_RESID) {
        const int f = m0 + quarter * 32 + c0;
        o.gain = ldg_here(reinterpret_cast<const uint2*>(p.gain + f));
#pragma unroll
        for (int i = 0; i < 4; ++i)
            o.v[i & (MODE == EPI_RESID ? 3 : 0)] = tq + 4 * i < ncols ? *reinterpret_cast<const float4*>(p.x + (size_t)(t0 + tq + 4 * i) * p.d + f)
                                                                      : make_float4(0.f, 0.f, 0.f, 0.f);
    } else if (MODE == EPI_QKV) {
        const int which = m0 < p.q_dim ? 0 : (m0 < p.q_dim + p.kv_dim ? 1 : 2);
        // KV slot (page * 16 + row) of token lane & 15, handed round by shuffles
        o.slot = (which > 0 && (lane & 15) < ncols) ? ldg_here(p.slot + t0 + (lane & 15)) : 0;
        if (which < 2) epi_load_rope<MODE>(p, o, t0, ncols, quarter, lane);
    }
}

// The chunk into the warp's scratch, one feature per lane ...
__device__ __forceinline__ void epi_stage(const float (&a)[EPI_COLS], float* scr, int lane) {
    __syncwarp();   // the previous chunk's rows have been read
#pragma unroll
    for (int j = 0; j < EPI_COLS; ++j) scr[j * EPI_SCR_STRIDE + lane] = a[j];
    __syncwarp();
}

// ... and out of it: the lane's four columns of the four tokens tq, tq + 4, ...  All loads stand before the first store (to the
// compiler a store may change the scratch, and a token at a time the four round trips follow one another: 1 000 cycles of a
// residual unit, 350 together).
__device__ __forceinline__ void epi_rows(const float* scr, float4 (&rows)[4], int tq, int c0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) rows[i] = *reinterpret_cast<const float4*>(scr + (tq + 4 * i) * EPI_SCR_STRIDE + c0);
}

// The chunk that a warp finishes next: what it reads is requested as soon as the operand's registers are free, and arrives while
// the present chunk is stored and the next one staged.
struct EpiNext {
    bool any;
    int m0, t0, ncols;
};

// The chunks of an item that a warp finishes, in turn: every NGRP-th of the chunks [c_lo, c_hi) of its tiles, from the grp-th on
// (carried along instead of divided out for every chunk).
template <int NGRP>
struct EpiCursor {
    int mt, c, left, c_lo, c_hi;   // left: chunks from this one on, over all groups (<= 0: none for this warp)
    __device__ __forceinline__ EpiCursor(int grp, int mt_lo, int lo, int hi, int total) : mt(mt_lo), c(lo + grp), left(total - grp), c_lo(lo), c_hi(hi) { wrap(); }
    __device__ __forceinline__ void advance() { c += NGRP; left -= NGRP; wrap(); }
    __device__ __forceinline__ void wrap() {
        while (left > 0 && c >= c_hi) { c -= c_hi - c_lo; ++mt; }
    }
};

// ... `o` holds what epi_load brought.  SWIGLU and LMHEAD have ways of their own (below).
template <int MODE>
__device__ __forceinline__ void epi_unit(const EpiParams& p, EpiOperand<MODE>& o, const float (&a)[EPI_COLS], float* scr, int m0,
                                         int t0, int ncols, int quarter, int lane, const EpiNext& next) {
    if (MODE != EPI_SWIGLU && (MODE != EPI_LMHEAD || p.logits)) epi_stage(a, scr, lane);
    const int tq = lane >> 3, c0 = (lane & 7) * 4;   // token (+ 4 i) and first of four columns of this lane
    if (MODE == EPI_PLAIN) {
        const int f = m0 + quarter * 32 + c0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = tq + 4 * i;
            const float4 r4 = *reinterpret_cast<const float4*>(scr + t * EPI_SCR_STRIDE + c0);
            const float row[4] = {r4.x, r4.y, r4.z, r4.w};
            if (t < ncols) {
                float* dst = p.y + (size_t)(t0 + t) * p.ldy + f;
                if ((p.ldy & 3) == 0 && f + 4 <= p.N) {
                    *reinterpret_cast<float4*>(dst) = make_float4(row[0], row[1], row[2], row[3]);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (f + k < p.N) dst[k] = row[k];
                }
            }
        }
    } else if (MODE == EPI_RESID) {
        // x += D; operand of the next projection half(x * gain); sum of x^2 over this warp's 32 features
        const int f = m0 + quarter * 32 + c0;
        const uint2 gain = o.gain;
        const __nv_bfloat162 g01 = *reinterpret_cast<const __nv_bfloat162*>(&gain.x);
        const __nv_bfloat162 g23 = *reinterpret_cast<const __nv_bfloat162*>(&gain.y);
        float4 nx[4];
        float ss[4];
        epi_rows(scr, nx, tq, c0);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 xv = o.v[i & (MODE == EPI_RESID ? 3 : 0)];
            nx[i] = make_float4(xv.x + nx[i].x, xv.y + nx[i].y, xv.z + nx[i].z, xv.w + nx[i].w);
            ss[i] = tq + 4 * i < ncols ? (nx[i].x * nx[i].x + nx[i].y * nx[i].y) + (nx[i].z * nx[i].z + nx[i].w * nx[i].w) : 0.f;
        }
        if (next.any) epi_load<MODE>(p, o, next.m0, next.t0, next.ncols, quarter, lane);
#pragma unroll
        for (int k = 1; k < 8; k <<= 1)   // the eight lanes of the token, a fixed order
#pragma unroll
            for (int i = 0; i < 4; ++i) ss[i] += __shfl_xor_sync(0xFFFFFFFFu, ss[i], k);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = tq + 4 * i;
            if (t < ncols) {
                const size_t at = (size_t)(t0 + t) * p.d + f;
                *reinterpret_cast<float4*>(p.x + at) = nx[i];
                *reinterpret_cast<uint2*>(p.xg + at) = pack4_op(nx[i].x * __low2float(g01), nx[i].y * __high2float(g01),
                                                                  nx[i].z * __low2float(g23), nx[i].w * __high2float(g23));
                if ((lane & 7) == 0) p.ssq_out[(size_t)(t0 + t) * (p.d >> 5) + ((m0 >> 5) + quarter)] = ss[i];
            }
        }
    } else if (MODE == EPI_QKV) {
        const int which = m0 < p.q_dim ? 0 : (m0 < p.q_dim + p.kv_dim ? 1 : 2);
        const int region0 = which == 0 ? 0 : (which == 1 ? p.q_dim : p.q_dim + p.kv_dim);
        const int half = p.hd >> 1, hd_log = p.hd == 128 ? 7 : 6;   // head_dim is 64 or 128
        const size_t page_stride = (size_t)p.n_kv_heads * 2 * 16 * p.hd;
        const int my_slot = o.slot;
        if (which < 2) {
            // q and k tiles: columns 0..15 of the block are the dims [d0, d0 + 16) of one head, columns 16..31
            // the same dims + hd/2 (rope_tile_feature); a lane rotates its four columns with their partners
            const int g_log = hd_log - 5;                                   // 16-dim groups of a half
            const int fhead = (m0 - region0) + ((quarter >> g_log) << hd_log);   // first feature of the head, inside q or k
            const bool hi = c0 >= 16;
            const int dim = 16 * (quarter & ((1 << g_log) - 1)) + (c0 & 15);            // lower dim of the pair
            const float sg = hi ? 1.f : -1.f;   // dim i: x cos - y sin; dim i + hd/2: y cos + x sin
            float4 mine[4], part[4];
            uint2 rot[4];
            epi_rows(scr, mine, tq, c0);
            epi_rows(scr, part, tq, c0 ^ 16);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 w0 = o.v[(2 * i) & (MODE == EPI_QKV ? 7 : 0)], w1 = o.v[(2 * i + 1) & (MODE == EPI_QKV ? 7 : 0)];
                rot[i] = pack4_op(mine[i].x * w0.x + sg * part[i].x * w0.y, mine[i].y * w0.z + sg * part[i].y * w0.w,
                                  mine[i].z * w1.x + sg * part[i].z * w1.y, mine[i].w * w1.z + sg * part[i].w * w1.w);
            }
            if (next.any) epi_load<MODE>(p, o, next.m0, next.t0, next.ncols, quarter, lane);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int t = tq + 4 * i;
                const int sl = __shfl_sync(0xFFFFFFFFu, my_slot, t);
                if (t < ncols) {
                    op16* dst;
                    if (which == 0) dst = p.q + (size_t)(t0 + t) * p.q_dim + fhead;
                    else dst = p.pool + (size_t)(sl >> 4) * page_stride + ((size_t)(fhead >> hd_log) * 2) * 16 * p.hd + (size_t)(sl & 15) * p.hd;
                    *reinterpret_cast<uint2*>(dst + dim + (hi ? half : 0)) = rot[i];
                }
            }
        } else {
            // v tiles: features in natural order
            const int fr = (m0 - region0) + quarter * 32 + c0;
            float4 rows[4];
            epi_rows(scr, rows, tq, c0);
            if (next.any) epi_load<MODE>(p, o, next.m0, next.t0, next.ncols, quarter, lane);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int t = tq + 4 * i;
                const float4 row = rows[i];
                const int sl = __shfl_sync(0xFFFFFFFFu, my_slot, t);
                if (t < ncols) {
                    op16* dst = p.pool + (size_t)(sl >> 4) * page_stride + ((size_t)(fr >> hd_log) * 2 + 1) * 16 * p.hd +
                                         (size_t)(sl & 15) * p.hd + (fr & (p.hd - 1));
                    *reinterpret_cast<uint2*>(dst) = pack4_op(row.x, row.y, row.z, row.w);
                }
            }
        }
    } else if (MODE == EPI_SWIGLU) {
        // Lanes 0..15 hold gate features, lanes 16..31 the matching up features.  The two exchange halves of their tokens,
        // so that each lane has gate and up of its feature for eight tokens; the results, already half precision, go
        // through a [16 features][16 tokens] tile (rows of 48 bytes) and come out of ldmatrix.trans with four consecutive
        // features of a token per lane.  (Half the instructions of the fp32 transposition that the other epilogues need.)
        const bool hi = lane & 16;
        float h[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float other = __shfl_xor_sync(0xFFFFFFFFu, hi ? a[k] : a[k + 8], 16);
            const float g = hi ? other : a[k], u = hi ? a[k + 8] : other;
            h[k] = __fdividef(g, 1.0f + __expf(-g)) * u;
        }
        uint8_t* const tile = reinterpret_cast<uint8_t*>(scr);
        __syncwarp();   // the previous chunk's tile has been read
        *reinterpret_cast<uint4*>(tile + (lane & 15) * 48 + (lane >> 4) * 16) =
            make_uint4(pack_op(h[0], h[1]), pack_op(h[2], h[3]), pack_op(h[4], h[5]), pack_op(h[6], h[7]));
        __syncwarp();
        // matrix j of the four: tokens 8 (j / 2) .., features 4 q + 2 (j & 1) + {0, 1} for q = 0 .. 3
        const int i = lane & 7, j = lane >> 3;
        uint32_t r0, r1, r2, r3;
        ldsm_x4_t(smem_u32(tile + (4 * (i >> 1) + 2 * (j & 1) + (i & 1)) * 48 + (j >> 1) * 16), r0, r1, r2, r3);
        const int t = lane >> 2;
        op16* dst = p.act + (size_t)(t0 + t) * p.f_pad + (m0 >> 1) + 16 * quarter + (lane & 3) * 4;
        if (t < ncols) *reinterpret_cast<uint2*>(dst) = make_uint2(r0, r1);
        if (t + 8 < ncols) *reinterpret_cast<uint2*>(dst + (size_t)8 * p.f_pad) = make_uint2(r2, r3);
    } else {  // EPI_LMHEAD
        // Largest logit of each token among the warp's 32 features, lowest id on ties, before any transposition: a maximum over
        // the warp and a ballot of the lanes that have it; lane j then speaks for token j.
        const int fl = m0 + quarter * 32;
        const bool fv = fl + lane < p.vocab;
        uint32_t top = 0u, who = 0u;
#pragma unroll
        for (int j = 0; j < EPI_COLS; ++j) {
            const uint32_t key = fv ? orderable_f32(a[j]) : 0u;
            const uint32_t mx = __reduce_max_sync(0xFFFFFFFFu, key);
            const uint32_t eq = __ballot_sync(0xFFFFFFFFu, key == mx && fv);
            if (lane == j) { top = mx; who = eq; }
        }
        if (lane < ncols) {
            if (who) atomicMax(p.best + t0 + lane, pack_argmax_key(top, fl + __ffs(who) - 1));
            // the group's maximum of the token (0: no valid feature): a threshold source for a later top-k
            if (p.warp_max) p.warp_max[(size_t)(t0 + lane) * p.n_warp_max + (m0 >> 5) + quarter] = top;
        }
        if (p.logits) {
            const int f = fl + c0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {   // (a token at a time: with all four rows first an item's epilogue took 23.5 k cycles against 19.5 k)
                const int t = tq + 4 * i;
                const float4 v = *reinterpret_cast<const float4*>(scr + t * EPI_SCR_STRIDE + c0);
                if (t < ncols) {
                    float* dst = p.logits + (size_t)(t0 + t) * p.vocab + f;
                    if ((p.vocab & 3) == 0 && f + 4 <= p.vocab) {
                        *reinterpret_cast<float4*>(dst) = v;
                    } else {
                        if (f < p.vocab) dst[0] = v.x;
                        if (f + 1 < p.vocab) dst[1] = v.y;
                        if (f + 2 < p.vocab) dst[2] = v.z;
                        if (f + 3 < p.vocab) dst[3] = v.w;
                    }
                }
            }
        }
    }
}

// Whether an epilogue multiplies by the RMSNorm scale of its tokens.
__host__ __device__ constexpr bool epi_scaled(int mode) { return mode == EPI_QKV || mode == EPI_SWIGLU || mode == EPI_LMHEAD; }

// Epilogue warps of the kernels that take a whole SM: 16 (four groups of four warps, one to a TMEM lane quarter) with 96 registers
// each; 12 with 128 where a chunk's operand is in flight beside it, which does not fit into 96 (8B shape, cycles from the last MMA
// to the end with 12 and 16 warps: o 27.4 and 30.9 k, down 27.1 and 30.4 k at 2 048 tokens, down 20.2 and 24.9 k at 544).  Where a
// CTA finishes few chunks a warp's share is rounded up more often with three groups: o of the 8B shape at 320 to 512 tokens, K in
// parts, 33.1 < 35.0 us between events; the steps of those sizes are 1.02 to 1.04 times as fast all the same.
__host__ __device__ constexpr int gemm_epi_warps(int mode) { return mode == EPI_QKV || mode == EPI_RESID ? 12 : GEMM_EPI_WARPS; }
__host__ __device__ constexpr int gemm_threads(int mode) { return (2 + gemm_epi_warps(mode)) * 32; }

// A chunk's accumulators, summed, through the epilogue.
template <int MODE>
__device__ __forceinline__ void epi_chunk(const EpiParams& p, EpiOperand<MODE>& o, const uint32_t (&r)[EPI_COLS], const float* rs, float* scr,
                                          int m0, int t0, int ncols, int quarter, int lane, const EpiNext& next) {
    float a[EPI_COLS];
#pragma unroll
    for (int j = 0; j < EPI_COLS; j += 4) {
        const float4 k = epi_scaled(MODE) ? *reinterpret_cast<const float4*>(rs + j) : make_float4(1.f, 1.f, 1.f, 1.f);
        a[j] = __uint_as_float(r[j]); a[j + 1] = __uint_as_float(r[j + 1]); a[j + 2] = __uint_as_float(r[j + 2]); a[j + 3] = __uint_as_float(r[j + 3]);
        if (epi_scaled(MODE)) { a[j] *= k.x; a[j + 1] *= k.y; a[j + 2] *= k.z; a[j + 3] *= k.w; }
    }
    epi_unit<MODE>(p, o, a, scr, m0, t0, ncols, quarter, lane, next);
}

// Accumulators of another part of K that its CTA left in global memory, added to (or, `first`, put into) a chunk.
__device__ __forceinline__ void epi_add_part(uint32_t (&r)[EPI_COLS], const float4* src, bool first) {
    float4 q[EPI_COLS / 4];
#pragma unroll
    for (int v = 0; v < EPI_COLS / 4; ++v) q[v] = __ldcg(src + v * 32);
#pragma unroll
    for (int v = 0; v < EPI_COLS / 4; ++v) {
        r[4 * v] = first ? __float_as_uint(q[v].x) : __float_as_uint(__uint_as_float(r[4 * v]) + q[v].x);
        r[4 * v + 1] = first ? __float_as_uint(q[v].y) : __float_as_uint(__uint_as_float(r[4 * v + 1]) + q[v].y);
        r[4 * v + 2] = first ? __float_as_uint(q[v].z) : __float_as_uint(__uint_as_float(r[4 * v + 2]) + q[v].z);
        r[4 * v + 3] = first ? __float_as_uint(q[v].w) : __float_as_uint(__uint_as_float(r[4 * v + 3]) + q[v].w);
    }
}

// RMSNorm scales of the tokens n0 .. n0 + n_valid - 1 from the partial sums of x^2 their source rows
// carry: one warp per token (warp `e` of NW takes every NW-th), a fixed reduction
// order, so every CTA that needs a token's scale gets the same bits.
template <int NW>
__device__ __forceinline__ void epi_rms_scales(const EpiParams& p, float* dst, int n0, int n_valid, int e, int lane) {
    const int nq = p.n_ssq >> 2;
    for (int t = e; t < n_valid; t += NW) {
        const float4* row = reinterpret_cast<const float4*>(p.ssq_in + (size_t)(n0 + t) * p.n_ssq);
        float sum = 0.f;
        for (int i = lane; i < nq; i += 32) {
            const float4 v = __ldcg(row + i);
            sum += (v.x + v.y) + (v.z + v.w);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        if (lane == 0) dst[t] = rsqrtf(sum * p.inv_d + p.eps);
    }
}

// ------------------------------------------------------------------------------------------
// Weight packing: row-major sources -> [pair][k-block][2][128 rows x 64 cols], each 16 KB tile
// stored as the 128-byte-swizzled shared-memory image (16-byte chunk c of row r at chunk c ^ (r & 7)).
// mode 0: packed row pr = row pr of the concatenation of up to three matrices.
// mode 1: gate/up: tile b holds gate and up features [64 b, 64 b + 64) in the lane order of
//         epi_unit (quarter q: lanes 0..15 gate 64 b + 16 q + lane, lanes 16..31 the same up rows).
// mode 2: q | k | v concatenation; q and k tiles in the RoPE lane order (rope_tile_feature), v plain.
// ------------------------------------------------------------------------------------------
struct PackSrc {
    const __nv_bfloat16* p[3];
    int rows[3];
    int mode;
    int src_k;   // valid columns of the sources (row pitch)
    int hd;      // mode 2: head dimension
};

__global__ void pack_weight_kernel(PackSrc src, op16* __restrict__ out, int num_kb) {
    const int mtile = blockIdx.x, kb = blockIdx.y;
    op16* tile = out + (((size_t)(mtile >> 1) * num_kb + kb) * 2 + (mtile & 1)) * (128 * 64);
    for (int i = threadIdx.x; i < 128 * 8; i += blockDim.x) {
        const int r = i >> 3, c = i & 7;
        const __nv_bfloat16* row = nullptr;
        if (src.mode == 0) {
            int q = mtile * 128 + r;
            for (int k = 0; k < 3 && !row; ++k) {
                if (q < src.rows[k]) row = src.p[k] + (size_t)q * src.src_k;
                q -= src.rows[k];
            }
        } else if (src.mode == 1) {
            const int sr = mtile * 64 + 16 * (r >> 5) + (r & 15);
            if (sr < src.rows[0]) row = src.p[(r & 16) ? 1 : 0] + (size_t)sr * src.src_k;
        } else {
            int base = mtile * 128, k = 0;   // region of this tile (regions are multiples of 128 rows)
            while (k < 2 && base >= src.rows[k]) base -= src.rows[k++];
            const int q = base + (k < 2 ? rope_tile_feature(r, src.hd) : r);
            if (q < src.rows[k]) row = src.p[k] + (size_t)q * src.src_k;
        }
        uint4 v = make_uint4(0, 0, 0, 0);
        const int col = kb * 64 + c * 8;
        if (row) {
            __nv_bfloat16 tmp[8];
            if (col + 8 <= src.src_k && (((uintptr_t)(row + col)) & 15) == 0) {
                *reinterpret_cast<uint4*>(tmp) = *reinterpret_cast<const uint4*>(row + col);
            } else {
                for (int e = 0; e < 8; ++e) tmp[e] = col + e < src.src_k ? row[col + e] : __float2bfloat16(0.f);
            }
            // bf16 -> half: exact for every weight of magnitude >= 2^-17
            v = make_uint4(pack_op(__bfloat162float(tmp[0]), __bfloat162float(tmp[1])), pack_op(__bfloat162float(tmp[2]), __bfloat162float(tmp[3])),
                           pack_op(__bfloat162float(tmp[4]), __bfloat162float(tmp[5])), pack_op(__bfloat162float(tmp[6]), __bfloat162float(tmp[7])));
        }
        *reinterpret_cast<uint4*>(tile + r * 64 + ((c ^ (r & 7)) << 3)) = v;
    }
}

// ------------------------------------------------------------------------------------------
// The kernel.  One persistent CTA per SM, 576 threads (448 with 12 epilogue warps): warp 0 = producer (bulk copy of the weight
// tiles + TMA boxes of the token tile), warp 1 = TMEM owner and MMA issuer, warps 2..17 (2..13) = epilogue
// (four or three groups of four; a group covers the four TMEM lane quarters; draining TMEM is limited per
// warp, so many warps share it).
// ------------------------------------------------------------------------------------------
constexpr int GEMM_BK = 64;                        // 16-bit elements per k-block = one 128-byte swizzle row
constexpr int GEMM_TILE_BYTES = 128 * GEMM_BK * 2; // 16 KB: one 128-feature tile of one k-block
constexpr int GEMM_A_BYTES = 2 * GEMM_TILE_BYTES;  // stage room for a pair
constexpr int GEMM_BOX_ROWS = 32;                  // token rows per B box
constexpr int GEMM_BOX_BYTES = GEMM_BOX_ROWS * GEMM_BK * 2;
constexpr int GEMM_MAX_STAGES = 8;
constexpr int GEMM_SMEM_MAX = 232448;
constexpr int GEMM_BAR_BYTES = 256;                // mbarriers and the TMEM address word

__host__ __device__ inline int gemm_stage_bytes(int TN) { return GEMM_A_BYTES + ((TN + 31) / 32) * GEMM_BOX_BYTES; }
// RMSNorm scales of an item's tokens, two buffers (items alternate); rounded up so that an epilogue
// that takes 32 columns at a time stays inside the buffer
__host__ __device__ inline int gemm_rs_stride(int TN) { return (TN + 31) & ~31; }
__host__ __device__ inline int gemm_scr_offset(int TN) { return GEMM_BAR_BYTES + 2 * gemm_rs_stride(TN) * 4; }   // from the barriers
__host__ inline int gemm_fixed_smem(int TN) { return 1024 /*align*/ + gemm_scr_offset(TN) + GEMM_EPI_WARPS * EPI_SCR_FLOATS * 4; }
__host__ inline int gemm_stages(int TN) {
    int s = (GEMM_SMEM_MAX - gemm_fixed_smem(TN)) / gemm_stage_bytes(TN);
    return s > GEMM_MAX_STAGES ? GEMM_MAX_STAGES : s;
}

struct GemmParams {
    const op16* w;              // packed weights
    int num_kb;                 // k-blocks of 64
    int n_pairs;                // 256-feature pairs
    int n_tt, TN;               // token tiles of TN columns (multiple of 16, <= 256)
    int n_stages;
    int splits, kb_per_split;   // splits > 1 (GEMM_RSPLIT): every CTA owns one (pair tile, k range)
    int pair_mode;              // 1: pair tiles in full waves + remainder as singles; 0: all singles;
                                // 2: one wave of n_cta items, pair tiles first, the rest as singles
    int ksplit;                 // pair mode, > 1: the remainder's pair tiles are cut along K into this many parts
    int kper;                   // ksplit: k-blocks of a helper part, (ksplit - 1) * kper < num_kb
    float* fix_part;            // ksplit: fp32 partial accumulators of the helper parts, [slot][2][TN/16][4][32][16];
                                // splits > 1: the exchange slots of the CTAs, same layout, slot = CTA index
    int* fix_flag;              // ksplit: per remainder tile, epilogue warps of helpers that have stored; then
                                // [n_sm + tile]: owner warps that are done reading (the last one clears both);
                                // splits > 1: the same two counters per pair tile
    int n_sm;
    int* status;
    long long spin_limit;       // SM cycles after which a wait gives up and sets *status
};

struct GemmWork {
    int pair, tt, mt_lo, mt_hi, kb0, kb1, split;
    int role;    // 0: the item's whole K; 1: helper part (accumulators go to fix_part); 2: owner part (adds the helpers')
    int rtile;   // role 1, 2: index of the remainder tile
    int hpart;   // role 1: which helper part
};

// Static schedule: work item i of CTA `cta`.  Returns false when the CTA is done.
// KSPLIT: the kernel variant that cuts the remainder's pair tiles along K (launched only when
// GemmParams::ksplit > 1; the plain variant carries none of that code).
template <bool KSPLIT>
__host__ __device__ __forceinline__ bool gemm_work(const GemmParams& g, int cta, int n_cta, int i, GemmWork& w) {
    const int n_tiles = g.n_pairs * g.n_tt;
    w.split = 0; w.kb0 = 0; w.kb1 = g.num_kb; w.mt_lo = 0; w.mt_hi = 2;
    w.role = 0; w.rtile = 0; w.hpart = 0;
    if (g.splits > 1) {
        if (i > 0 || cta >= n_tiles * g.splits) return false;
        const int tile = cta / g.splits;
        w.split = cta - tile * g.splits;
        w.pair = tile / g.n_tt; w.tt = tile - w.pair * g.n_tt;
        w.kb0 = w.split * g.kb_per_split;
        w.kb1 = w.kb0 + g.kb_per_split < g.num_kb ? w.kb0 + g.kb_per_split : g.num_kb;
        return true;
    }
    if (KSPLIT) {
        // Full waves of pair tiles; the R tiles of the remainder are cut along K into ksplit parts on
        // different CTAs.  The helper parts run FIRST on CTAs 0 .. R (ksplit - 1) - 1, the owner part
        // (the last k range) runs LAST on the last R CTAs and adds the helpers' stored accumulators,
        // which by then have long been written.
        const int fw = n_tiles / n_cta, R = n_tiles - fw * n_cta, H = g.ksplit - 1;
        const int kper = g.kper;   // k-blocks of a helper part; the owner takes the (shorter) rest
        const bool helper = cta < R * H, owner = cta >= n_cta - R;
        int wave = i;
        if (helper) {
            if (i == 0) {
                w.role = 1; w.rtile = cta / H; w.hpart = cta - w.rtile * H;
                const int tile = fw * n_cta + w.rtile;
                w.pair = tile / g.n_tt; w.tt = tile - w.pair * g.n_tt;
                w.kb0 = w.hpart * kper; w.kb1 = w.kb0 + kper;
                return true;
            }
            wave = i - 1;
        }
        if (wave < fw) {
            const int tile = wave * n_cta + cta;
            w.pair = tile / g.n_tt; w.tt = tile - w.pair * g.n_tt;
            return true;
        }
        if (owner && wave == fw) {
            w.role = 2; w.rtile = cta - (n_cta - R);
            const int tile = fw * n_cta + w.rtile;
            w.pair = tile / g.n_tt; w.tt = tile - w.pair * g.n_tt;
            w.kb0 = H * kper; w.kb1 = g.num_kb;
            return true;
        }
        return false;
    }
    if (g.pair_mode == 1) {
        const int fw = n_tiles / n_cta;
        if (i < fw) {
            const int tile = i * n_cta + cta;
            w.pair = tile / g.n_tt; w.tt = tile - w.pair * g.n_tt;
            return true;
        }
        const int r = (i - fw) * n_cta + cta;
        if (r >= (n_tiles - fw * n_cta) * 2) return false;
        const int tile = fw * n_cta + (r >> 1);
        w.pair = tile / g.n_tt; w.tt = tile - w.pair * g.n_tt;
        w.mt_lo = r & 1; w.mt_hi = w.mt_lo + 1;
        return true;
    }
    if (g.pair_mode == 2) {
        // One item per CTA and more single tiles than CTAs: the first 2 n_tiles - n_cta pair tiles stay
        // whole, the others run as two single tiles, so that n_cta CTAs cover everything in one wave.
        if (i > 0) return false;
        const int whole = 2 * n_tiles - n_cta;
        if (cta < whole) {
            w.pair = cta / g.n_tt; w.tt = cta - w.pair * g.n_tt;
            return true;
        }
        const int r = cta - whole, tile = whole + (r >> 1);
        w.pair = tile / g.n_tt; w.tt = tile - w.pair * g.n_tt;
        w.mt_lo = r & 1; w.mt_hi = w.mt_lo + 1;
        return true;
    }
    const int sidx = i * n_cta + cta;
    if (sidx >= n_tiles * 2) return false;
    const int mtile = sidx / g.n_tt;
    w.tt = sidx - mtile * g.n_tt;
    w.pair = mtile >> 1;
    w.mt_lo = mtile & 1; w.mt_hi = w.mt_lo + 1;
    return true;
}

// Every CTA walks its k-blocks from a different starting point (and wraps): at any moment the CTAs
// that share a token tile then ask L2 for different lines of it instead of all for the same ones.
// The schedule is static, so the summation order of a given output is the same in every run.
__device__ __forceinline__ int gemm_k_rotation(int cta, int n_cta, int nk) {
    return (int)(((long long)cta * nk) / n_cta);
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

template <int VARIANT, int MODE>
__global__ void __launch_bounds__(gemm_threads(MODE), 1)
gemm_kernel(const __grid_constant__ CUtensorMap tmB, GemmParams g, EpiParams p) {
    constexpr bool KSPLIT = VARIANT == GEMM_KSPLIT;
    constexpr bool RSPLIT = VARIANT == GEMM_RSPLIT;
    constexpr int EW = gemm_epi_warps(MODE);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int stage_bytes = gemm_stage_bytes(g.TN);
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + g.n_stages * stage_bytes);
    uint64_t* empty_bar = full_bar + GEMM_MAX_STAGES;
    uint64_t* accf_bar = empty_bar + GEMM_MAX_STAGES;   // accumulators complete (MMA -> epilogue)
    uint64_t* acce_bar = accf_bar + 1;                  // accumulators drained (epilogue -> MMA)
    uint64_t* rs_bar = acce_bar + 1;                    // RMSNorm scales of the item's tokens are in rs_s
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(rs_bar + 1);
    float* rs_s = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(full_bar) + GEMM_BAR_BYTES);   // [2][rs stride]
    float* scr_s = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(full_bar) + gemm_scr_offset(g.TN));   // [epilogue warp][16][36]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_cta = gridDim.x, cta = blockIdx.x;
    const long long limit = g.spin_limit;
    pdl_launch_dependents();
    uint32_t acc_stride = 32;
    while ((int)acc_stride < g.TN) acc_stride <<= 1;
    const uint32_t tmem_cols = 2 * acc_stride;

    if (threadIdx.x == 0) {
        tma_prefetch_desc(&tmB);
        for (int s = 0; s < g.n_stages; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(accf_bar, 1);
        mbar_init(acce_bar, EW);
        mbar_init(rs_bar, EW);
        mbar_fence_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (elect_one()) {
            // (stage and k-block indices are carried along: a remainder costs this one thread more than its requests do)
            int s = 0;
            uint32_t ph = 1;   // parity of the use of stage s that the MMAs have to release; nothing to wait for in the first round
            bool ok = true, first = true;
            GemmWork w;
            for (int i = 0; ok && gemm_work<KSPLIT>(g, cta, n_cta, i, w); ++i) {
                const int n0 = w.tt * g.TN;
                const int nbox = (((min(g.TN, p.T - n0) + 15) & ~15) + 31) >> 5;
                const uint32_t a_bytes = (uint32_t)(w.mt_hi - w.mt_lo) * GEMM_TILE_BYTES;
                const op16* wsrc = g.w + ((size_t)w.pair * g.num_kb) * (2 * 128 * 64) + (size_t)w.mt_lo * (128 * 64);
                const int nk = w.kb1 - w.kb0, rot = gemm_k_rotation(cta, n_cta, nk);
                // The weights never depend on an earlier kernel: the first item's weight tiles of the
                // whole ring are requested before waiting for the predecessor, whose output is only the
                // token operand.
                const int n_early = i == 0 ? min(nk, g.n_stages) : 0;
                int kb = w.kb0 + rot;
                for (int j = 0; j < n_early; ++j) {
                    uint8_t* a_s = smem + j * stage_bytes;
                    mbar_expect_tx(&full_bar[j], a_bytes + nbox * GEMM_BOX_BYTES);
                    bulk_load(a_s + w.mt_lo * GEMM_TILE_BYTES, wsrc + (size_t)kb * (2 * 128 * 64), a_bytes, &full_bar[j]);
                    if (++kb == w.kb1) kb = w.kb0;
                }
                if (i == 0) pdl_wait();
                kb = w.kb0 + rot;
                for (int j = 0; j < nk; ++j) {
                    if (!first && !mbar_wait(&empty_bar[s], ph, g.status, limit)) {
                        ok = false;
                        break;
                    }
                    uint8_t* a_s = smem + s * stage_bytes;
                    uint8_t* b_s = a_s + GEMM_A_BYTES;
                    if (j >= n_early) {
                        mbar_expect_tx(&full_bar[s], a_bytes + nbox * GEMM_BOX_BYTES);
                        bulk_load(a_s + w.mt_lo * GEMM_TILE_BYTES, wsrc + (size_t)kb * (2 * 128 * 64), a_bytes, &full_bar[s]);
                    }
                    for (int b = 0; b < nbox; ++b)
                        tma_load_2d(b_s + b * GEMM_BOX_BYTES, &tmB, &full_bar[s], kb * GEMM_BK, n0 + b * GEMM_BOX_ROWS);
                    if (++kb == w.kb1) kb = w.kb0;
                    if (++s == g.n_stages) { s = 0; ph ^= 1; first = false; }
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (elect_one()) {
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            GemmWork w;
            for (int i = 0; ok && gemm_work<KSPLIT>(g, cta, n_cta, i, w); ++i) {
                const uint32_t nn = (uint32_t)((min(g.TN, p.T - w.tt * g.TN) + 15) & ~15);
                const uint32_t idesc = umma_idesc_f16(128, nn);
                if (i > 0) {   // the epilogue must have drained the previous item's accumulators
                    ok = mbar_wait(acce_bar, (i - 1) & 1, g.status, limit);
                    if (!ok) break;
                    tc_fence_after();
                }
                const int nk = w.kb1 - w.kb0;
                for (int j = 0; j < nk; ++j) {
                    ok = mbar_wait(&full_bar[s], ph, g.status, limit);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a_addr = smem_u32(smem + s * stage_bytes);
                    const uint64_t db = umma_desc_k128(a_addr + GEMM_A_BYTES);
                    // consecutive MMAs alternate between the two accumulators: back-to-back MMAs into
                    // one accumulator wait for each other
#pragma unroll
                    for (int k = 0; k < GEMM_BK / 16; ++k)  // 16 halves = 32 bytes = 2 descriptor address units
                        for (int mt = w.mt_lo; mt < w.mt_hi; ++mt) {
                            const uint64_t da = umma_desc_k128(a_addr + mt * GEMM_TILE_BYTES);
                            umma_bf16(tmem_base + mt * acc_stride, da + 2 * k, db + 2 * k, idesc, j > 0 || k > 0);
                        }
                    umma_commit(&empty_bar[s]);
                    if (++s == g.n_stages) { s = 0; ph ^= 1; }
                }
                if (ok) umma_commit(accf_bar);
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ epilogue
        const int e = warp - 2;
        const int grp = e >> 2;               // the groups take the 16-token chunks round robin
        constexpr int NGRP = EW / 4;
        const int quarter = warp & 3;         // TMEM lane quarter this warp may read
        constexpr bool scaled = epi_scaled(MODE);
        float* const scr = scr_s + e * EPI_SCR_FLOATS;
        bool ok = true;
        GemmWork w;
        pdl_wait();   // the epilogues read and write buffers of earlier kernels
        for (int i = 0; ok && gemm_work<KSPLIT>(g, cta, n_cta, i, w); ++i) {
            const int n0 = w.tt * g.TN;
            const int n_valid = min(g.TN, p.T - n0);
            const int nchunks = (n_valid + EPI_COLS - 1) / EPI_COLS;
            float* const rsi = rs_s + (i & 1) * gemm_rs_stride(g.TN);
            if (scaled) {   // while the main loop runs: the scales of this item's tokens
                epi_rms_scales<EW>(p, rsi, n0, n_valid, e, lane);
                __syncwarp();
                if (lane == 0) mbar_arrive(rs_bar);
            }
            // The chunks [c_lo, c_hi) of this CTA's tiles are finished here, the warp's group takes every NGRP-th of them.
            const int S = RSPLIT ? g.splits : 1, sp = RSPLIT ? w.split : 0;
            const int c_lo = sp * nchunks / S, c_hi = (sp + 1) * nchunks / S;
            const int total_chunks = (w.mt_hi - w.mt_lo) * (c_hi - c_lo);
            EpiCursor<NGRP> cur(grp, w.mt_lo, c_lo, c_hi, total_chunks);
            auto unit_here = [&]() {
                EpiNext u;
                u.m0 = w.pair * 256 + cur.mt * 128;
                u.t0 = n0 + cur.c * EPI_COLS;
                u.ncols = min(EPI_COLS, n_valid - cur.c * EPI_COLS);
                u.any = cur.left > 0 && u.m0 < p.N;
                return u;
            };
            EpiOperand<MODE> opnd;   // of the warp's first chunk: in flight while the main loop runs
            EpiNext unit = unit_here();
            if (unit.any && (!KSPLIT || w.role != 1)) epi_load<MODE>(p, opnd, unit.m0, unit.t0, unit.ncols, quarter, lane);
            ok = mbar_wait(accf_bar, i & 1, g.status, limit);
            if (ok && scaled) ok = mbar_wait(rs_bar, i & 1, g.status, limit);
            if (!ok) break;
            tc_fence_after();
            if (RSPLIT) {
                // ---- reduce-scatter over the S CTAs that share this tile.  CTA `split` keeps the
                // chunks [c_lo, c_hi) of both 128-feature tiles.  Exchange slot of a CTA:
                // [tile of the pair][chunk][lane quarter][4][lane][4 floats], so that one 16-byte access
                // per lane covers 512 contiguous bytes per warp.
                const int tile = cta / S;
                const int cpt = g.TN / EPI_COLS;
                const size_t slot_elems = (size_t)2 * cpt * 128 * EPI_COLS;
                float* const mine = g.fix_part + (size_t)cta * slot_elems;
                int nth = 0;
                for (int mt = 0; mt < 2; ++mt)
                    for (int c = 0; c < nchunks; ++c) {
                        if (c >= c_lo && c < c_hi) continue;
                        if (nth++ % NGRP != grp) continue;
                        uint32_t r[EPI_COLS];
                        tmem_ld16(tmem_base + mt * acc_stride + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(c * EPI_COLS), r);
                        tmem_ld_wait();
                        uint4* dst = reinterpret_cast<uint4*>(mine + (((size_t)mt * cpt + c) * 4 + quarter) * 32 * EPI_COLS) + lane;
#pragma unroll
                        for (int v = 0; v < EPI_COLS / 4; ++v) dst[v * 32] = make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
                    }
                __threadfence();        // this warp's share of the accumulators is in memory
                __syncwarp();
                if (lane == 0) atomicAdd(g.fix_flag + tile, 1);
                // all warps of all S CTAs must have stored before anyone reads; the CTAs of a tile are
                // neighbours in the grid and the grid is at most one CTA per SM, so they run together
                if (lane == 0) {
                    const int want = S * EW;
                    const long long t_end = clock64() + limit;
                    while (ld_acquire_gpu(g.fix_flag + tile) < want) {
                        if (clock64() > t_end) {
                            atomicExch(g.status, 1);
                            break;
                        }
                    }
                }
                __syncwarp();
                while (cur.left > 0) {
                    const int mt = cur.mt, c = cur.c;
                    uint32_t own[EPI_COLS], r[EPI_COLS];
                    tmem_ld16(tmem_base + mt * acc_stride + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(c * EPI_COLS), own);
                    tmem_ld_wait();
                    const size_t at = (((size_t)mt * cpt + c) * 4 + quarter) * 32 * EPI_COLS;
                    for (int q = 0; q < S; ++q) {   // fixed order: the parts in split order
                        if (q == sp) {
#pragma unroll
                            for (int v = 0; v < EPI_COLS; ++v)
                                r[v] = q == 0 ? own[v] : __float_as_uint(__uint_as_float(r[v]) + __uint_as_float(own[v]));
                        } else {
                            epi_add_part(r, reinterpret_cast<const float4*>(g.fix_part + (size_t)(tile * S + q) * slot_elems + at) + lane, q == 0);
                        }
                    }
                    cur.advance();
                    const EpiNext next = unit_here();
                    if (unit.any) epi_chunk<MODE>(p, opnd, r, rsi + c * EPI_COLS, scr, unit.m0, unit.t0, unit.ncols, quarter, lane, next);
                    unit = next;
                }
                // the last warp of the tile's CTAs to finish reading clears the counters for the next launch
                __syncwarp();
                if (lane == 0 && atomicAdd(g.fix_flag + g.n_sm + tile, 1) == S * EW - 1) {
                    g.fix_flag[tile] = 0;
                    g.fix_flag[g.n_sm + tile] = 0;
                }
                continue;
            }
            if (!KSPLIT || w.role == 0) {
                while (cur.left > 0) {
                    const int mt = cur.mt, c = cur.c;
                    uint32_t r[EPI_COLS];
                    tmem_ld16(tmem_base + mt * acc_stride + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(c * EPI_COLS), r);
                    tmem_ld_wait();
                    if (cur.left <= NGRP) {   // last TMEM read of this warp for this item
                        tc_fence_before();
                        if (lane == 0) mbar_arrive(acce_bar);
                    }
                    cur.advance();
                    const EpiNext next = unit_here();
                    if (unit.any) epi_chunk<MODE>(p, opnd, r, rsi + c * EPI_COLS, scr, unit.m0, unit.t0, unit.ncols, quarter, lane, next);
                    unit = next;
                }
                if (grp >= total_chunks) {   // a group without any chunk still releases the accumulators
                    tc_fence_before();
                    if (lane == 0) mbar_arrive(acce_bar);
                }
                continue;
            }
            // ---- a part of a K-split remainder tile.  Stored accumulators:
            // [part][tile of the pair][chunk][lane quarter][4][lane][4 floats], so that one 16-byte access
            // per lane covers 512 contiguous bytes per warp.
            const int H = g.ksplit - 1, cpt = g.TN / EPI_COLS;   // helper parts per tile, chunk slots per tile
            const size_t part_elems = (size_t)2 * cpt * 128 * EPI_COLS;
            if (w.role == 1) {
                float* mine = g.fix_part + (size_t)(w.rtile * H + w.hpart) * part_elems;
                while (cur.left > 0) {
                    const int mt = cur.mt, c = cur.c;
                    uint32_t r[EPI_COLS];
                    tmem_ld16(tmem_base + mt * acc_stride + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(c * EPI_COLS), r);
                    tmem_ld_wait();
                    if (cur.left <= NGRP) {
                        tc_fence_before();
                        if (lane == 0) mbar_arrive(acce_bar);
                    }
                    uint4* dst = reinterpret_cast<uint4*>(mine + (((size_t)mt * cpt + c) * 4 + quarter) * 32 * EPI_COLS) + lane;
#pragma unroll
                    for (int v = 0; v < EPI_COLS / 4; ++v) dst[v * 32] = make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
                    cur.advance();
                }
                if (grp >= total_chunks) {
                    tc_fence_before();
                    if (lane == 0) mbar_arrive(acce_bar);
                }
                __threadfence();        // this warp's part of the accumulators is in memory
                __syncwarp();
                if (lane == 0) atomicAdd(g.fix_flag + w.rtile, 1);
                continue;
            }
            // owner: the helpers ran first; the wait is bounded all the same
            if (lane == 0) {
                const int want = H * EW;
                const long long t_end = clock64() + limit;
                while (ld_acquire_gpu(g.fix_flag + w.rtile) < want) {
                    if (clock64() > t_end) {
                        atomicExch(g.status, 1);
                        break;
                    }
                }
            }
            __syncwarp();
            while (cur.left > 0) {
                const int mt = cur.mt, c = cur.c;
                uint32_t r[EPI_COLS];
                tmem_ld16(tmem_base + mt * acc_stride + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(c * EPI_COLS), r);
                tmem_ld_wait();
                if (cur.left <= NGRP) {
                    tc_fence_before();
                    if (lane == 0) mbar_arrive(acce_bar);
                }
                const size_t at = (((size_t)mt * cpt + c) * 4 + quarter) * 32 * EPI_COLS;
                for (int h = 0; h < H; ++h)   // fixed order: own k range, then the helpers' in part order
                    epi_add_part(r, reinterpret_cast<const float4*>(g.fix_part + (size_t)(w.rtile * H + h) * part_elems + at) + lane, false);
                cur.advance();
                const EpiNext next = unit_here();
                if (unit.any) epi_chunk<MODE>(p, opnd, r, rsi + c * EPI_COLS, scr, unit.m0, unit.t0, unit.ncols, quarter, lane, next);
                unit = next;
            }
            if (grp >= total_chunks) {
                tc_fence_before();
                if (lane == 0) mbar_arrive(acce_bar);
            }
            // the last warp to finish reading clears the tile's counters for the next launch
            __syncwarp();
            if (lane == 0 && atomicAdd(g.fix_flag + g.n_sm + w.rtile, 1) == EW - 1) {
                g.fix_flag[w.rtile] = 0;
                g.fix_flag[g.n_sm + w.rtile] = 0;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, tmem_cols);
    }
}

}  // namespace syn
