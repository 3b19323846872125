// The projection GEMM for batches of few tokens (sm_100a), where a step is a chain of short dependent
// kernels that stream the weights once: what counts is that the weights keep coming from HBM across
// the kernel boundaries and that the part of a kernel that depends on its predecessor is short.
//   - A CTA takes HALF an SM (at most 113 KB of shared memory, 256 TMEM columns, 320 threads of at most
//     102 registers), so that the CTAs of two consecutive kernels are resident together: while a
//     kernel drains, its successor has set up its barriers and filled its operand ring with weights
//     (they depend on nothing).  This kernel lets its successor start once its own predecessor is
//     complete, so that of a chain of such kernels at most two are unfinished (the full-SM kernels
//     let theirs start before they wait; it cannot become resident beside them anyway).
//   - Work item = 128 output features x one token tile (all tokens up to 128, else equal tiles) x one of
//     S parts of K.  The S CTAs of an item are a cluster: they hand each other fp32 accumulators
//     through distributed shared memory (a reduce-scatter over units of 32 features x 16 tokens, added in
//     part order): asynchronous remote stores that count their bytes on an mbarrier of the receiver, no
//     global memory and no counters.
//   - Same orientation, weight tiles and epilogues (epi_unit) as gemm.cuh.  Two accumulators take
//     alternate k-steps (an MMA into the accumulator of its predecessor waits for it).
// Whole steps, every projection on the one-CTA kernel -> with this one: 1B shape, 5 tokens 1 187 -> 821 us; 135 tokens
// 1 611 -> 1 340 us; 8B shape, 40 tokens 4 600 -> 3 820 us (the weights alone take 2 325 us at the copy rate), 119 tokens
// 6 100 -> 5 760 us.  The 8B o projection (33.5 MB) at 40 tokens: 26.1 -> 15.5 us between events in the step.  What bounds
// it: HBM while it streams (4.5 - 5 TB/s in a launch of its own), and about 3 us per launch that depend on the
// predecessor (its results visible, token operand, exchange, epilogue).  With the epilogues that load ahead and the shorter
// attention merges those steps take 759, 1 240, 3 740 and 5 770 us.  Tried and dropped: 256 CTAs instead of 148 and fewer with one
// token tile (14 % slower at the 8B shape), asking L2 for the next projection's weights (1 to 5 % slower: the
// requests compete with the loads that the step waits for), two cluster barriers around plain remote
// stores instead of the counted asynchronous ones.
#pragma once
#include "gemm.cuh"

namespace syn {

constexpr int THIN_EPI_WARPS = 8;
constexpr int THIN_THREADS = (2 + THIN_EPI_WARPS) * 32;
constexpr int THIN_MAX_TN = 128;
constexpr int THIN_MAX_SPLITS = 8;
constexpr int THIN_SMEM_MAX = 113 * 1024;       // two CTAs (of one kernel or of two consecutive ones) per SM
constexpr int THIN_UNIT_FLOATS = 32 * EPI_COLS; // exchange unit: 32 features x 16 tokens
constexpr int THIN_MAX_STAGES = 6;
constexpr int THIN_RECV_OWN_MAX = 20 * 1024;    // a receive area of its own up to this size costs at most one stage of the ring

struct ThinParams {
    const op16* w;              // packed weights
    int num_kb;                 // k-blocks of 64
    int n_tiles;                // 128-feature tiles
    int n_tt, TN;               // token tiles of TN columns (multiple of 16, <= THIN_MAX_TN)
    int n_stages, splits;       // splits = cluster size
    int recv_own;               // 1: the receive area is shared memory of its own, 0: it is the operand ring's
    int* status;
    long long spin_limit;
};

// Shared memory: operand ring | receive area, if it is of its own | barriers | RMSNorm scales.  After the main loop the
// ring also holds the epilogue warps' scratch (at its end) and, unless it is of its own, the receive area (at its start).
constexpr int THIN_SCR_BYTES = THIN_EPI_WARPS * EPI_SCR_FLOATS * 4;
__host__ __device__ inline int thin_stage_bytes(int TN) { return GEMM_TILE_BYTES + TN * GEMM_BK * 2; }
__host__ __device__ inline int thin_recv_bytes(int TN, int S) {   // the S parts of the most units a CTA finishes
    return (TN / EPI_COLS * 4 + S - 1) / S * S * THIN_UNIT_FLOATS * 4;
}
__host__ inline int thin_fixed_smem(int TN) { return 1024 /*align*/ + GEMM_BAR_BYTES + TN * 4; }
__host__ inline int thin_stages(int TN, int recv) {
    const int s = (THIN_SMEM_MAX - thin_fixed_smem(TN) - recv) / thin_stage_bytes(TN);
    return s > THIN_MAX_STAGES ? THIN_MAX_STAGES : s;
}

// Unit u = chunk * 4 + lane quarter of U = 4 * nchunks belongs to rank r with first(r) <= u < first(r + 1).
__host__ __device__ __forceinline__ int thin_unit_first(int r, int U, int S) { return r * U / S; }
__host__ __device__ __forceinline__ int thin_unit_owner(int u, int U, int S) { return ((u + 1) * S - 1) / U; }

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void sts_v4(uint32_t addr, float a, float b, float c, float d) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
__device__ __forceinline__ float4 lds_v4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
// 16 bytes into another CTA's shared memory, counted on an mbarrier there
__device__ __forceinline__ void st_async_v4(uint32_t addr, uint32_t bar, float a, float b, float c, float d) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d), "r"(bar) : "memory");
}

// RMSNorm scales of the tokens t_lo .. t_hi - 1 of the tile at n0 (see epi_rms_scales; the same bits): four
// tokens of a warp at a time, so that their loads overlap.
__device__ __forceinline__ void thin_rms_scales(const EpiParams& p, float* dst, int n0, int t_lo, int t_hi, int e, int lane) {
    const int nq = p.n_ssq >> 2;
    for (int t = t_lo + e; t < t_hi; t += 4 * THIN_EPI_WARPS) {
        float sum[4] = {0.f, 0.f, 0.f, 0.f};
        for (int i = lane; i < nq; i += 32) {
            float4 v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int tk = min(t + k * THIN_EPI_WARPS, t_hi - 1);
                v[k] = __ldcg(reinterpret_cast<const float4*>(p.ssq_in + (size_t)(n0 + tk) * p.n_ssq) + i);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) sum[k] += (v[k].x + v[k].y) + (v[k].z + v[k].w);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < 4; ++k) sum[k] += __shfl_xor_sync(0xFFFFFFFFu, sum[k], o);
        if (lane < 4) {
            const int tk = t + lane * THIN_EPI_WARPS;
            const float s = lane == 0 ? sum[0] : (lane == 1 ? sum[1] : (lane == 2 ? sum[2] : sum[3]));
            if (tk < t_hi) dst[tk] = rsqrtf(s * p.inv_d + p.eps);
        }
    }
}

template <int MODE>
__global__ void __launch_bounds__(THIN_THREADS, 2)
thin_kernel(const __grid_constant__ CUtensorMap tmB, ThinParams g, EpiParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int stage_bytes = thin_stage_bytes(g.TN);
    const int recv_bytes = g.splits > 1 ? thin_recv_bytes(g.TN, g.splits) : 0;
    uint8_t* recv = g.recv_own ? smem + g.n_stages * stage_bytes : smem;
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + g.n_stages * stage_bytes + (g.recv_own ? recv_bytes : 0));
    uint64_t* empty_bar = full_bar + THIN_MAX_STAGES;
    uint64_t* accf_bar = empty_bar + THIN_MAX_STAGES;
    uint64_t* recv_bar = accf_bar + 1;      // everything the other parts send has arrived
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(recv_bar + 1);
    float* rs_s = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(full_bar) + GEMM_BAR_BYTES);   // [TN]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S = g.splits, item = blockIdx.x / S, split = blockIdx.x - item * S;   // split = rank in the cluster
    const int tile = item / g.n_tt, tt = item - tile * g.n_tt;
    const int n0 = tt * g.TN, n_valid = min(g.TN, p.T - n0);
    const int nchunks = (n_valid + EPI_COLS - 1) / EPI_COLS;
    const int kb0 = (int)((long long)split * g.num_kb / S), nk = (int)((long long)(split + 1) * g.num_kb / S) - kb0;
    const int U = nchunks * 4, u_lo = thin_unit_first(split, U, S), u_hi = thin_unit_first(split + 1, U, S);   // units this CTA finishes
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
        mbar_init(recv_bar, 1);
        mbar_fence_init();
        if (S > 1) mbar_expect_tx(recv_bar, (uint32_t)((u_hi - u_lo) * (S - 1) * (THIN_UNIT_FLOATS * 4)));
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // A CTA may send once every receiver has its barrier and, where the receive area is the operand ring's, has
    // completed its MMAs: the arrival on the cluster's barrier says so.
    if (S > 1 && g.recv_own) cluster_arrive();

    bool ok = true;
    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (elect_one()) {
            // (stage and k-block indices are carried along: a remainder costs this one thread more than its requests do)
            const op16* wsrc = g.w + ((size_t)(tile >> 1) * g.num_kb * 2 + (tile & 1)) * (128 * 64);
            const int kb1 = kb0 + nk;
            int kb = kb0 + item % nk;   // CTAs that share a token tile walk it from different places
            const int kb_first = kb;
            const uint32_t bytes = (uint32_t)stage_bytes;
            const int n_early = min(nk, g.n_stages);
            for (int j = 0; j < n_early; ++j) {
                mbar_expect_tx(&full_bar[j], bytes);
                bulk_load(smem + j * stage_bytes, wsrc + (size_t)kb * (2 * 128 * 64), GEMM_TILE_BYTES, &full_bar[j]);
                if (++kb == kb1) kb = kb0;
            }
            pdl_wait();
            pdl_launch_dependents();
            kb = kb_first;
            for (int j = 0; j < n_early; ++j) {
                tma_load_2d(smem + j * stage_bytes + GEMM_TILE_BYTES, &tmB, &full_bar[j], kb * GEMM_BK, n0);
                if (++kb == kb1) kb = kb0;
            }
            int s = 0;
            uint32_t ph = 0;   // parity of the use of stage s that the MMAs have to release
            for (int j = n_early; j < nk; ++j) {
                if (!mbar_wait(&empty_bar[s], ph, g.status, g.spin_limit)) break;
                uint8_t* a_s = smem + s * stage_bytes;
                mbar_expect_tx(&full_bar[s], bytes);
                bulk_load(a_s, wsrc + (size_t)kb * (2 * 128 * 64), GEMM_TILE_BYTES, &full_bar[s]);
                tma_load_2d(a_s + GEMM_TILE_BYTES, &tmB, &full_bar[s], kb * GEMM_BK, n0);
                if (++kb == kb1) kb = kb0;
                if (++s == g.n_stages) { s = 0; ph ^= 1; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (elect_one()) {
            const uint32_t idesc = umma_idesc_f16(128, (uint32_t)(nchunks * EPI_COLS));
            int s = 0;
            uint32_t ph = 0;
            for (int j = 0; j < nk; ++j) {
                ok = mbar_wait(&full_bar[s], ph, g.status, g.spin_limit);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a_addr = smem_u32(smem + s * stage_bytes);
                const uint64_t da = umma_desc_k128(a_addr), db = umma_desc_k128(a_addr + GEMM_TILE_BYTES);
#pragma unroll
                for (int k = 0; k < GEMM_BK / 16; ++k)   // 16 halves = 32 bytes = 2 descriptor address units
                    umma_bf16(tmem_base + (k & 1) * acc_stride, da + 2 * k, db + 2 * k, idesc, j > 0 || k >= 2);
                umma_commit(&empty_bar[s]);
                if (++s == g.n_stages) { s = 0; ph ^= 1; }
            }
            if (ok) umma_commit(accf_bar);
        }
        __syncwarp();
    }
    if (warp < 2) {
        if (S > 1) {   // the cluster's barrier counts every thread
            if (!g.recv_own) cluster_arrive();
            cluster_wait();
            cluster_arrive();
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int e = warp - 2, grp = e >> 2;   // two groups take the 16-token chunks in turn
        const int quarter = warp & 3;           // TMEM lane quarter this warp may read
        constexpr bool scaled = epi_scaled(MODE);
        float* const scr = reinterpret_cast<float*>(smem + g.n_stages * stage_bytes - THIN_SCR_BYTES) + e * EPI_SCR_FLOATS;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const int m0 = tile * 128;
        // the chunks of this warp whose units this CTA finishes: c = c_first, c_first + 2, ... while 4 c + quarter < u_hi
        int c_first = grp;
        while (4 * c_first + quarter < u_lo) c_first += 2;
        pdl_wait();   // the epilogues read and write buffers of earlier kernels
        EpiOperand<MODE> opnd;   // of the first unit: in flight while the main loop runs
        if (4 * c_first + quarter < u_hi) epi_load<MODE>(p, opnd, m0, n0 + c_first * EPI_COLS, min(EPI_COLS, n_valid - c_first * EPI_COLS), quarter, lane);
        if (scaled && u_hi > u_lo) {   // and the scales of the tokens this CTA finishes
            thin_rms_scales(p, rs_s, n0, (u_lo >> 2) * EPI_COLS, min(n_valid, ((u_hi - 1) >> 2) * EPI_COLS + EPI_COLS), e, lane);
            asm volatile("bar.sync 1, 256;" ::: "memory");
        }
        ok = mbar_wait(accf_bar, 0, g.status, g.spin_limit);
        ok = __all_sync(0xFFFFFFFFu, ok) != 0;
        tc_fence_after();
        auto read_acc = [&](int c, float (&a)[EPI_COLS]) {   // both accumulators of chunk c, this warp's quarter
            uint32_t r[EPI_COLS], r2[EPI_COLS];
            tmem_ld16(t_lane + (uint32_t)(c * EPI_COLS), r);
            tmem_ld16(t_lane + acc_stride + (uint32_t)(c * EPI_COLS), r2);
            tmem_ld_wait();
#pragma unroll
            for (int v = 0; v < EPI_COLS; ++v) a[v] = __uint_as_float(r[v]) + __uint_as_float(r2[v]);
        };
        if (S > 1) {
            if (!g.recv_own) cluster_arrive();
            cluster_wait();
            if (ok)
                for (int c = grp; c < nchunks; c += 2) {
                    const int u = c * 4 + quarter, owner = thin_unit_owner(u, U, S);
                    float a[EPI_COLS];
                    read_acc(c, a);
                    // receive area: [unit of the receiver][part][4][lane][4 floats]
                    const int slot = (u - thin_unit_first(owner, U, S)) * S + split;
                    const uint32_t at = smem_u32(recv + (size_t)slot * (THIN_UNIT_FLOATS * 4)) + lane * 16;
                    if (owner == split) {
#pragma unroll
                        for (int v = 0; v < EPI_COLS / 4; ++v) sts_v4(at + v * 512, a[4 * v], a[4 * v + 1], a[4 * v + 2], a[4 * v + 3]);
                    } else {
                        const uint32_t dst = mapa_rank(at, owner), bar = mapa_rank(smem_u32(recv_bar), owner);
#pragma unroll
                        for (int v = 0; v < EPI_COLS / 4; ++v) st_async_v4(dst + v * 512, bar, a[4 * v], a[4 * v + 1], a[4 * v + 2], a[4 * v + 3]);
                    }
                }
            __syncwarp();
            cluster_arrive();
            if (ok && 4 * c_first + quarter < u_hi) {
                ok = mbar_wait(recv_bar, 0, g.status, g.spin_limit);
                ok = __all_sync(0xFFFFFFFFu, ok) != 0;
            }
        }
        for (int c = c_first; ok && 4 * c + quarter < u_hi; c += 2) {
            float a[EPI_COLS];
            if (S == 1) {
                read_acc(c, a);
            } else {   // the parts in split order
                const uint32_t src = smem_u32(recv + (size_t)(4 * c + quarter - u_lo) * S * (THIN_UNIT_FLOATS * 4)) + lane * 16;
                // (the next part's four loads in flight while one is added)
                float4 f[2][EPI_COLS / 4];
#pragma unroll
                for (int v = 0; v < EPI_COLS / 4; ++v) {
                    f[0][v] = lds_v4(src + v * 512);
                    a[4 * v] = a[4 * v + 1] = a[4 * v + 2] = a[4 * v + 3] = 0.f;
                }
#pragma unroll
                for (int q = 0; q < THIN_MAX_SPLITS; ++q) {
                    if (q >= S) break;
                    if (q + 1 < S) {
#pragma unroll
                        for (int v = 0; v < EPI_COLS / 4; ++v) f[(q + 1) & 1][v] = lds_v4(src + (q + 1) * (THIN_UNIT_FLOATS * 4) + v * 512);
                    }
#pragma unroll
                    for (int v = 0; v < EPI_COLS / 4; ++v) {
                        const float4 t = f[q & 1][v];
                        a[4 * v] += t.x; a[4 * v + 1] += t.y; a[4 * v + 2] += t.z; a[4 * v + 3] += t.w;
                    }
                }
            }
            if (scaled) {
#pragma unroll
                for (int v = 0; v < EPI_COLS; ++v) a[v] *= rs_s[c * EPI_COLS + v];
            }
            const int tc = n0 + c * EPI_COLS, ncols = min(EPI_COLS, n_valid - c * EPI_COLS);
            const EpiNext next = {4 * (c + 2) + quarter < u_hi, m0, tc + 2 * EPI_COLS, min(EPI_COLS, n_valid - (c + 2) * EPI_COLS)};
            epi_unit<MODE>(p, opnd, a, scr, m0, tc, ncols, quarter, lane, next);
        }
    }
    if (S > 1) cluster_wait();   // nobody leaves while another part may still send to it
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, tmem_cols);
    }
}

}  // namespace syn
