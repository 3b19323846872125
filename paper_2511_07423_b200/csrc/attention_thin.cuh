// Ragged multi-query attention over the paged KV cache (paper Sec. 3.2, 3.4) for batches with few (request, kv head)
// units, where a layer's keys are read in 10 to 30 us and what counts is that every SM has an equal share of them and
// that the fixed part of the kernel is short.  Same work items, arithmetic and partial results as attention.cuh; the
// differences:
//   - a CTA takes half an SM (160 threads, about 100 KB of shared memory), two of them run side by side: one loads
//     while the other merges, and the CTAs start while the projection before them drains;
//   - one consumer warp takes a whole stage (two pages of 128-dim heads, four of 64-dim ones), the four warps take
//     stages in turn (fewer row tiles than four) or row tiles; so a stage costs one warp's barrier wait and softmax
//     and not four;
//   - queries go straight from L2 to registers: no Q tile, no barrier for it;
//   - K and V that no chunk of the batch writes (AttnItem::kv_safe) are requested before the projection that
//     writes the chunks' K and V has finished.
// What bounds it: with 64-dim heads the arithmetic of a stage on one warp and the last CTA's merge (1B shape, contexts
// 256-2048, chunks 1-8: 150 requests 71 us a layer against 88 of the full-SM kernel, 40 requests 33.0 against 33.4 and a step of 4
// layers 385 us against 395); with 128-dim heads and many units the warps' arithmetic (8B shape, 64 requests of 512-4096,
// chunks 1-16: 174 us against 137), so those keep the full-SM kernel.
#pragma once
#include "attention.cuh"

namespace syn {

constexpr int ATTN_THIN_WARPS = 4;
constexpr int ATTN_THIN_THREADS = (ATTN_THIN_WARPS + 1) * 32;
constexpr int ATTN_THIN_STAGES = 5;
constexpr int ATTN_THIN_MAX_PARTS = 32;   // of one row group
constexpr int ATTN_THIN_ROWS = 64;        // of an item's tile (AttnParams::row_cap): row stride of the parts

template <int HD>
struct AttnThinSmem {
    static constexpr int PAGES = HD == 128 ? 2 : 4;                // per stage
    static constexpr int PAGE_BYTES = 2 * 16 * HD * 2;             // K and V of one page, one head
    static constexpr int STAGE_BYTES = PAGES * PAGE_BYTES;         // 16 KB
    // two slots of O[16][HD] + (m, l)[16], or a weight for every part of the rows and one over their sums
    static constexpr int WEIGHT_BYTES = (ATTN_THIN_MAX_PARTS + 1) * ATTN_THIN_ROWS * 4, SLOT_BYTES = 2 * 16 * (HD + 4) * 4;
    static constexpr int MERGE_BYTES = WEIGHT_BYTES > SLOT_BYTES ? WEIGHT_BYTES : SLOT_BYTES;
    static constexpr int TOTAL = 1024 + ATTN_THIN_STAGES * STAGE_BYTES + MERGE_BYTES + 512;
    static_assert(2 * (TOTAL + 1024) <= 233472, "two CTAs per SM");
};

__device__ __forceinline__ void mbar_arrive_n(uint64_t* bar, uint32_t n) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(n) : "memory");
}
__device__ __forceinline__ void l2_prefetch(const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<uint64_t>(src)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void l1_prefetch(const void* src) { asm volatile("prefetch.global.L1 [%0];" ::"l"(src)); }
__device__ __forceinline__ void attn_thin_bar() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

template <int HD>
__global__ void __launch_bounds__(ATTN_THIN_THREADS, 2)
attn_thin_kernel(const __grid_constant__ CUtensorMap tmKV, AttnParams p) {
    using SM = AttnThinSmem<HD>;
    constexpr int HALVES = HD / 64, NS = ATTN_THIN_STAGES, KEYS = 16 * SM::PAGES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* stages = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    float* merge = reinterpret_cast<float*>(stages + NS * SM::STAGE_BYTES);
    // Stage st lies in slot st % NS and completes full_bar[st % 4][st % NS]: a warp that takes every stage, every second
    // or every fourth one then sees the phases of each of its barriers one by one (a parity wait must never be two
    // phases behind, and loads land out of order).
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(merge) + SM::MERGE_BYTES);
    uint64_t* empty_bar = full_bar + 4 * NS;
    int* last_flag = reinterpret_cast<int*>(empty_bar + NS);
    static_assert(5 * NS * 8 + 8 <= 512 && NS % 2 == 1, "barrier area; slots and classes must be coprime");

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int it_begin = p.cta_begin[blockIdx.x], it_end = p.cta_begin[blockIdx.x + 1];
    const int G = p.group;
    const bool list_ok = it_begin >= 0 && it_begin <= it_end && it_end <= p.n_items;

    if (threadIdx.x == 0) {
        tma_prefetch_desc(&tmKV);
        for (int s = 0; s < 4 * NS; ++s) mbar_init(&full_bar[s], 1);
        for (int s = 0; s < NS; ++s) mbar_init(&empty_bar[s], 4);
        mbar_fence_init();
    }
    __syncthreads();

    if (warp == ATTN_THIN_WARPS) {
        // ------------------------------------------------------------ producer
        uint32_t st = 0;
        bool ok = list_ok, waited = false;
        const int my_pg = lane / HALVES, my_half = lane % HALVES;
        for (int it = it_begin; it < it_end && ok; ++it) {
            const AttnItem item = p.items[it];
            if (!attn_item_ok(item, p)) break;   // the consumers flag it and stop waiting
            const int* pt = p.page_tables + (size_t)item.req * p.max_pages;
            const int first_page = item.kv_begin >> 4, last_page = (item.kv_end - 1) >> 4;
            constexpr int PER = 32 / SM::PAGES;   // stages whose page-table entries the warp holds, one per lane
            int ent_cur = first_page + lane <= last_page ? pt[first_page + lane] : 0;
            int ent_next = first_page + 32 + lane <= last_page ? pt[first_page + 32 + lane] : 0;
            int k = 0;   // stage of the item
            for (int kv0 = item.kv_begin; kv0 < item.kv_end; kv0 += KEYS, ++st, ++k) {
                const int s = st % NS;
                if (k > 0 && (k & (PER - 1)) == 0) {
                    ent_cur = ent_next;
                    const int nidx = first_page + (k / PER) * 32 + 32 + lane;
                    ent_next = nidx <= last_page ? pt[nidx] : 0;
                }
                int page = __shfl_sync(0xFFFFFFFFu, ent_cur, ((k & (PER - 1)) * SM::PAGES + my_pg) & 31);
                const int npg = min(SM::PAGES, (item.kv_end - kv0 + 15) >> 4);
                if (!waited && kv0 + KEYS > item.kv_safe) {   // keys that the projection before this kernel may still write
                    pdl_wait();
                    waited = true;
                }
                uint64_t* fb = &full_bar[(st & 3u) * NS + s];
                if (lane == 0) {
                    if (st >= (uint32_t)NS) ok = mbar_wait(&empty_bar[s], ((st / NS) - 1) & 1, p.status);
                    if (ok) mbar_expect_tx(fb, npg * SM::PAGE_BYTES);
                }
                ok = __shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0) != 0;
                if (!ok) break;
                if (my_pg < npg && (unsigned)page >= (unsigned)p.n_pages) {
                    atomicExch(p.status, 2);
                    page = 0;
                }
                if (my_pg < npg) {
                    const int row0 = (p.layer_block0 + 2 * (page * p.n_kv_heads + item.kvh)) * 16;
                    tma_load_2d(stages + s * SM::STAGE_BYTES + my_pg * SM::PAGE_BYTES + my_half * 4096, &tmKV, fb, my_half * 64, row0);
                }
            }
        }
        // HBM would idle while the last parts are finished and merged: ask L2 for weights of the projections behind, where
        // there are many keys only once this CTA's own are here (sooner, the requests delay the CTAs that are behind)
        if (p.ahead_late)
            for (uint32_t q = st > (uint32_t)NS ? st - NS : 0u; ok && q < st; ++q)
                if (lane == 0) ok = mbar_wait(&empty_bar[q % NS], (q / NS) & 1, p.status);
        if (lane == 0 && ok)
            for (int i = 0; i < 2; ++i) {
                const WeightsAhead& a = p.ahead[i];
                for (int b = blockIdx.x; b < a.n_tiles * a.splits * a.count; b += gridDim.x) {
                    const int unit = b / a.count, j = a.skip + b - unit * a.count, tile = unit / a.splits, part = unit - tile * a.splits;
                    const int k0 = (int)((long long)part * a.num_kb / a.splits), nk = (int)((long long)(part + 1) * a.num_kb / a.splits) - k0;
                    if (j < nk)
                        l2_prefetch(a.w + (((size_t)(tile >> 1) * a.num_kb + k0 + (j + tile * a.n_tt % nk) % nk) * 2 + (tile & 1)) * (128 * 64), 128 * 64 * 2);
                }
            }
        return;
    }

    // ---------------------------------------------------------------- consumers (warps 0..3)
    // A wait that runs out sets `ok` = false; the warp then skips all further waits and arithmetic but still walks the
    // items and takes part in every named barrier, so no other warp is left waiting for it.
    if (list_ok && it_begin < it_end && lane < 2) l1_prefetch(reinterpret_cast<const uint8_t*>(p.items + it_begin) + lane * (sizeof(AttnItem) - 4));
    pdl_wait();   // Q and the chunk's K/V come from the preceding projection kernel
    if (threadIdx.x == 0) pdl_launch_dependents();
    const int g = lane >> 2, c = lane & 3;
    uint32_t st = 0;
    bool ok = true;
    if (!list_ok && threadIdx.x == 0) atomicExch(p.status, 2);
    for (int it = it_begin; list_ok && it < it_end; ++it) {
        const AttnItem item = p.items[it];
        if (!attn_item_ok(item, p)) {   // uniform over the CTA: every warp leaves here together
            if (threadIdx.x == 0) atomicExch(p.status, 2);
            break;
        }
        const int rows = item.nj * G;
        const int n_mt = (rows + 15) >> 4;
        const int npw = n_mt >= 3 ? 4 : n_mt;             // row-tile slots (1, 2 or 4)
        const int nph = 4 / npw;                          // the warps of a row tile take stages in turn
        const int mt = warp % npw, ph = warp / npw;
        const bool active = mt < n_mt;

        uint32_t qf[HD / 16][4];
        {
            const int r0 = mt * 16 + g, r1 = r0 + 8;
            const op16* q0 = p.q + (size_t)(item.q_tok + r0 / G) * p.q_dim + (item.kvh * G + r0 % G) * HD + 2 * c;
            const op16* q1 = p.q + (size_t)(item.q_tok + r1 / G) * p.q_dim + (item.kvh * G + r1 % G) * HD + 2 * c;
#pragma unroll
            for (int ks = 0; ks < HD / 16; ++ks) {
                qf[ks][0] = r0 < rows ? __ldcg(reinterpret_cast<const unsigned int*>(q0 + 16 * ks)) : 0u;
                qf[ks][1] = r1 < rows ? __ldcg(reinterpret_cast<const unsigned int*>(q1 + 16 * ks)) : 0u;
                qf[ks][2] = r0 < rows ? __ldcg(reinterpret_cast<const unsigned int*>(q0 + 16 * ks + 8)) : 0u;
                qf[ks][3] = r1 < rows ? __ldcg(reinterpret_cast<const unsigned int*>(q1 + 16 * ks + 8)) : 0u;
            }
        }
        float o[HD / 8][4];
#pragma unroll
        for (int nt = 0; nt < HD / 8; ++nt) o[nt][0] = o[nt][1] = o[nt][2] = o[nt][3] = 0.f;
        float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
        const int lim0 = item.q_pos0 + (mt * 16 + g) / G, lim1 = item.q_pos0 + (mt * 16 + g + 8) / G;

        for (int kv0 = item.kv_begin; kv0 < item.kv_end; kv0 += KEYS, ++st) {
            if ((int)(st & (uint32_t)(nph - 1)) != ph) continue;
            const int s = st % NS;
            if (ok) ok = mbar_wait(&full_bar[(st & 3u) * NS + s], (st / (4 * NS)) & 1, p.status);
            if (active && ok) {
                const int npg = min(SM::PAGES, (item.kv_end - kv0 + 15) >> 4);
                const bool need_mask = kv0 + KEYS - 1 > item.q_pos0;
                const uint8_t* sp = stages + s * SM::STAGE_BYTES;
                if (npg == SM::PAGES)
                    attn_consume_stage<HD, SM::PAGES, true>(sp, 0, npg, kv0, qf, o, m, l, lim0, lim1, p.scale_log2, need_mask, lane);
                else
                    attn_consume_stage<HD, SM::PAGES, false>(sp, 0, npg, kv0, qf, o, m, l, lim0, lim1, p.scale_log2, need_mask, lane);
            }
            __syncwarp();
            if (lane == 0 && ok) mbar_arrive_n(&empty_bar[s], nph);   // npw warps arrive, 4 in all
        }

        // row sums across the quad
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            l[r] += __shfl_xor_sync(0xFFFFFFFFu, l[r], 1);
            l[r] += __shfl_xor_sync(0xFFFFFFFFu, l[r], 2);
        }
        int part0 = 0, n_parts = 0;   // of the item's merge group
        if (item.part >= 0) { part0 = p.groups[item.grp].part0; n_parts = p.groups[item.grp].n_parts; }
        // the warps of a row tile, in a fixed order: (0 + 2) + (1 + 3), or 0 + 1
        if (nph > 1) {
            attn_thin_bar();   // slots free: the previous item's readers are done
            const int half = nph / 2;
            if (ph >= half) attn_store_slot<HD>(merge + ((ph - half) * npw + mt) * 16 * (HD + 4), o, m, l, g, c);
            attn_thin_bar();
            if (ph < half) attn_fold_slot<HD>(merge + (ph * npw + mt) * 16 * (HD + 4), o, m, l, g, c);
            if (nph == 4) {
                attn_thin_bar();
                if (ph == 1) attn_store_slot<HD>(merge + mt * 16 * (HD + 4), o, m, l, g, c);
                attn_thin_bar();
                if (ph == 0) attn_fold_slot<HD>(merge + mt * 16 * (HD + 4), o, m, l, g, c);
            }
        }
        // write: final output (half precision) or fp32 partial
        if (active && ph == 0 && ok) {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int row = mt * 16 + g + 8 * r;
                if (row < rows) {
                    const int j = row / G, gq = row - j * G;
                    if (item.part < 0) {
                        const float inv = l[r] > 0.f ? 1.f / l[r] : 0.f;
                        op16* dst = p.out + (size_t)(item.q_tok + j) * p.q_dim + (item.kvh * G + gq) * HD;
#pragma unroll
                        for (int nt = 0; nt < HD / 8; ++nt)
                            *reinterpret_cast<uint32_t*>(dst + nt * 8 + 2 * c) = pack_op(o[nt][2 * r] * inv, o[nt][2 * r + 1] * inv);
                    } else {
                        float* dst = p.part_o + ((size_t)item.part * ATTN_THIN_ROWS + row) * HD;
#pragma unroll
                        for (int nt = 0; nt < HD / 8; ++nt)
                            *reinterpret_cast<float2*>(dst + nt * 8 + 2 * c) = make_float2(o[nt][2 * r], o[nt][2 * r + 1]);
                        if (c == 0) p.part_ml[(size_t)item.part * ATTN_THIN_ROWS + row] = make_float2(m[r], l[r]);
                    }
                }
            }
        }
        // a partial item: count it; the CTA that completes the group combines the partials in part order
        if (item.part >= 0) {
            attn_thin_bar();
            // (one thread's release covers what the barrier ordered before it, its acquire what the barrier orders behind it)
            if (threadIdx.x == 0) *last_flag = atomic_add_acq_rel(p.group_count + item.grp, 1) == n_parts - 1;
            attn_thin_bar();
            if (*last_flag) {
                // What this costs is round trips, on the step's critical path: the (m, l) pairs and the first UK parts of the
                // outputs (NU places of the rows each) are in flight together, and the weights wait for the pairs alone.  (Loads
                // past the last part repeat it: left out under a condition they cost 600 bytes of spills in the stage loop.)
                if (threadIdx.x == 0) p.group_count[item.grp] = 0;   // ready for the next launch
                const int np = min(n_parts, ATTN_THIN_MAX_PARTS);
                float* w_s = merge;                                             // [part][row]
                float* inv_s = merge + ATTN_THIN_MAX_PARTS * ATTN_THIN_ROWS;    // [row]
                constexpr int VR = HD / 4, NU = HD == 128 ? 5 : 3, UK = HD == 128 ? 3 : 5, CAP = ATTN_THIN_ROWS;
                static_assert(CAP == 64, "two lanes of 128 threads take a row; row / G below");
                const int n_vec = rows * VR, by_g = 4096 / G + 1;   // row / G = row * by_g >> 12 for rows up to 64
                const float4* src = reinterpret_cast<const float4*>(p.part_o) + (size_t)part0 * (CAP * VR);
                float4 v[UK][NU];
                auto fetch = [&](int u0, int k0) {
#pragma unroll
                    for (int k = 0; k < UK; ++k)
#pragma unroll
                        for (int i = 0; i < NU; ++i) v[k][i] = __ldcg(src + min(k0 + k, np - 1) * (CAP * VR) + min(u0 + i * 128, n_vec - 1));
                };
                {   // lanes 2 r and 2 r + 1 take the even and the odd parts of row r, eight of them at a time
                    const int row = threadIdx.x >> 1, odd = threadIdx.x & 1;
                    const float2* ml = p.part_ml + (size_t)part0 * CAP + min(row, rows - 1);
                    float2 t[8];
                    auto pairs = [&](int k0) {
#pragma unroll
                        for (int k = 0; k < 8; ++k) t[k] = k0 + odd + 2 * k < np ? __ldcg(ml + (k0 + odd + 2 * k) * CAP) : make_float2(-INFINITY, 0.f);
                    };
                    pairs(0);
                    fetch(threadIdx.x, 0);
                    float mx = -INFINITY, lsum = 0.f;
                    for (int k0 = 0; k0 < np; k0 += 16) {
                        if (k0) pairs(k0);
#pragma unroll
                        for (int k = 0; k < 8; ++k) mx = fmaxf(mx, t[k].x);
                    }
                    mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 1));
                    const float bs = mx == -INFINITY ? 0.f : mx;
                    // the sum goes through the parts in their order, whoever holds them (a part past the last adds zero), and a
                    // weight is divided by it before it meets the outputs: both are part of what a step's logits are, bit for bit.
                    // (8B shape, eight requests, whole steps: 3 708 us; 3 723 with the weights divided in shared memory before the
                    // barrier and a branch for every part; 3 706 with the sums of even and of odd parts added, in other bits.)
                    for (int k0 = 0; k0 < np; k0 += 16) {
                        if (np > 16) pairs(k0);
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            if (k % 2 == 0 && k0 + 2 * k >= np) break;
                            const float w = ex2_approx(t[k].x - bs), w_of = __shfl_xor_sync(0xFFFFFFFFu, w, 1);
                            const float l_of = __shfl_xor_sync(0xFFFFFFFFu, t[k].y, 1);
                            lsum += (odd ? l_of : t[k].y) * (odd ? w_of : w);
                            lsum += (odd ? t[k].y : l_of) * (odd ? w : w_of);
                            w_s[(k0 + odd + 2 * k) * CAP + row] = w;
                        }
                    }
                    const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
                    if (!odd) inv_s[row] = inv;
                }
                attn_thin_bar();
                op16* const out0 = p.out + (size_t)item.q_tok * p.q_dim + item.kvh * G * HD;
                for (int u0 = threadIdx.x; u0 < n_vec; u0 += NU * 128) {
                    float4 acc[NU];
                    float inv[NU];
#pragma unroll
                    for (int i = 0; i < NU; ++i) {
                        acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                        inv[i] = inv_s[min(u0 + i * 128, n_vec - 1) / VR];
                    }
                    for (int k0 = 0; k0 < np; k0 += UK) {
                        if (k0 > 0 || u0 != (int)threadIdx.x) fetch(u0, k0);
#pragma unroll
                        for (int k = 0; k < UK; ++k) {
                            if (k0 + k >= np) break;
#pragma unroll
                            for (int i = 0; i < NU; ++i) {
                                const float w = w_s[(k0 + k) * CAP + min(u0 + i * 128, n_vec - 1) / VR] * inv[i];
                                acc[i].x += v[k][i].x * w; acc[i].y += v[k][i].y * w; acc[i].z += v[k][i].z * w; acc[i].w += v[k][i].w * w;
                            }
                        }
                    }
#pragma unroll
                    for (int i = 0; i < NU; ++i) {
                        const int u = u0 + i * 128, row = u / VR, j = row * by_g >> 12, gq = row - j * G;
                        if (u < n_vec)
                            *reinterpret_cast<uint2*>(out0 + (size_t)j * p.q_dim + gq * HD + 4 * (u % VR)) =
                                make_uint2(pack_op(acc[i].x, acc[i].y), pack_op(acc[i].z, acc[i].w));
                    }
                }
                attn_thin_bar();   // the weights' area is the next item's merge slots
            }
        }
    }
}

}  // namespace syn
