// Host side of the library: C ABI, weight packing, KV pool, step planner and the launch
// sequence of one verification step.  See include/synera.h for the contract of every entry point.
#include "../../include/synera.h"

#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "attention2.cuh"
#include "attention_thin.cuh"
#include "gemm.cuh"
#include "gemm2.cuh"
#include "gemm_thin.cuh"
#include "pieces.h"
#include "sampling.cuh"

using namespace syn;
typedef __nv_bfloat16 bf16;
// Slot of one helper part's stored accumulators: two tiles of 128 features x up to 256 tokens, fp32.
constexpr size_t GEMM_FIX_SLOT_BYTES = (size_t)2 * 128 * 256 * 4;
constexpr int GEMM_FLAG_INTS = 4;   // arrival / release counters of the exchanges: ints per SM
constexpr int GEMM_MAX_SPLITS = 8;   // most CTAs that share one pair tile's K range
// Limit of the kernels' bounded waits in SM cycles (syn_debug_set_spin_limit; tests shorten it).
static long long g_spin_limit = SYN_SPIN_LIMIT_CYCLES;
// 0: every projection takes the kernel its shape calls for; 1: the one-CTA kernel always (syn_debug_set_schedule).
static int g_schedule = 0;
// Attention kernel: 0 = whichever the planner makes cheaper for the batch, 1 = warp-level MMAs (64-row tiles),
// 2 = tcgen05 (128-row tiles), 3 = warp-level MMAs in CTAs of half an SM.
static int g_attention = 0;

// Name of the last CUDA error a call of this library met on this thread (for syn_last_cuda_error).
static thread_local const char* g_last_cuda_error = "";
static inline cudaError_t note_cuda(cudaError_t e) {
    if (e != cudaSuccess) g_last_cuda_error = cudaGetErrorName(e);
    return e;
}
// cudaGetLastError after a launch, recorded like any other failing call
static inline bool launch_ok() { return note_cuda(cudaGetLastError()) == cudaSuccess; }

#define CU_OK(expr)                              \
    do {                                         \
        cudaError_t _e = note_cuda(expr);        \
        if (_e != cudaSuccess) {                 \
            (void)cudaGetLastError();            \
            return _e == cudaErrorMemoryAllocation ? SYN_E_OOM : SYN_E_CUDA; \
        }                                        \
    } while (0)

// Launch, with `pdl` with programmatic stream serialization: the kernel may then start while its predecessor in the
// stream still runs; every kernel of the step calls pdl_wait() before it touches anything an earlier
// kernel produces or still reads.
template <typename... KArgs, typename... Args>
static cudaError_t launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl, Args... args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr;
    memset(&attr, 0, sizeof(attr));
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return note_cuda(cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...));
}
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    return launch(kernel, grid, block, smem, st, true, args...);
}

// The same for a kernel whose CTAs form clusters of `cluster` neighbours.
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl_clusters(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster, Args... args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    memset(attr, 0, sizeof(attr));
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return note_cuda(cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...));
}

// ------------------------------------------------------------------------------------------ small kernels

// Token embedding (paper Sec. 4.5: the flattened batch enters the transformer), the first layer's
// GEMM operand half(x * gain) with the sums of x^2 per 32 features its RMSNorm scale is made of,
// RoPE table, argmax reset.
__global__ void __launch_bounds__(256)
prep_kernel(const bf16* __restrict__ embed, const int* __restrict__ tokens, const int* __restrict__ pos,
            const bf16* __restrict__ gain, const double* __restrict__ inv_freq, float* __restrict__ x,
            op16* __restrict__ xg, float* __restrict__ ssq, float2* __restrict__ rope, unsigned long long* __restrict__ best,
            int d, int half) {
    const int t = blockIdx.x, lane = threadIdx.x & 31;
    pdl_launch_dependents();
    pdl_wait();
    const bf16* e = embed + (size_t)tokens[t] * d;
    for (int f0 = (threadIdx.x >> 5) * 32; f0 < d; f0 += blockDim.x) {   // one warp per group of 32 features
        const int f = f0 + lane;
        const float v = __bfloat162float(e[f]);
        x[(size_t)t * d + f] = v;
        xg[(size_t)t * d + f] = to_op(v * __bfloat162float(gain[f]));
        float ss = v * v;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, o);
        if (lane == 0) ssq[(size_t)t * (d >> 5) + (f0 >> 5)] = ss;
    }
    if (threadIdx.x == 0) best[t] = 0ull;
    for (int i = threadIdx.x; i < half; i += blockDim.x) {
        double sn, cs;
        sincos((double)pos[t] * inv_freq[i], &sn, &cs);
        rope[(size_t)t * half + i] = make_float2((float)cs, (float)sn);
    }
}

// The lm_head's operand of the rows that verification looks at, side by side (one block a row).
__global__ void __launch_bounds__(256)
judging_rows_kernel(const op16* xg, const float* ssq, const int* __restrict__ rows, op16* xj, float* ssqj, int d) {
    pdl_launch_dependents();
    const size_t from = (size_t)rows[blockIdx.x], to = blockIdx.x;   // (the plan is older than the step)
    pdl_wait();
    for (int i = threadIdx.x * 8; i < d; i += blockDim.x * 8) *reinterpret_cast<uint4*>(xj + to * d + i) = *reinterpret_cast<const uint4*>(xg + from * d + i);
    for (int i = threadIdx.x; i < d >> 5; i += blockDim.x) ssqj[to * (d >> 5) + i] = ssq[from * (d >> 5) + i];
}

// Greedy verification (paper Sec. 3.1 "draft & verify", Sec. 4.5): one thread per request.  The blocking calls have the results and
// the kernels' status written straight to pinned host memory (with three copies behind the kernel a call of four requests of
// the two-layer shape took 84.6 us and takes 69.7; one on four layers of the 1B shape 243.7 and 230.0).
__global__ void verify_kernel(const unsigned long long* __restrict__ best, const int* __restrict__ tokens,
                              const int* __restrict__ offsets, const int* __restrict__ n_uncached, int n_req,
                              int* __restrict__ accept_len, int* __restrict__ correction, int* __restrict__ top1_out,
                              const int* __restrict__ first_row, const int* status, int* status_out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    if (i == 0 && status_out) *status_out = *status;
    if (i >= n_req) return;
    const int b = offsets[i], n = offsets[i + 1] - b, u = n_uncached[i];
    if (top1_out)
        for (int j = 0; j < n; ++j) top1_out[b + j] = (int)(0xFFFFFFFFu - (uint32_t)(best[b + j] & 0xFFFFFFFFull));
    const unsigned long long* mine = best + (first_row ? first_row[i] : b + u - 1);   // the row that judges the first draft
    int a = 0;
    while (a < n - u && (int)(0xFFFFFFFFu - (uint32_t)(mine[a] & 0xFFFFFFFFull)) == tokens[b + u + a]) ++a;
    accept_len[i] = a;
    correction[i] = (int)(0xFFFFFFFFu - (uint32_t)(mine[a] & 0xFFFFFFFFull));
}

// Copy K/V of logical positions between a dense bf16 [n_pos][Hkv][hd] buffer and the paged pool (half precision).  The
// page ids travel as a launch parameter, so that a transfer is one launch: no device buffer, no copy, no memory that
// callers on several streams or threads would share.  A thread moves VEC elements of K and of V (8: 16 bytes each
// way) of KV_COPY_POS positions, all loads before the first store.  A blocking call of 2 600 positions of the 8B shape
// (10.6 MB each way) takes 20 us, of 100 positions 16: launch and synchronisation bound it (59 us when the slots went
// through a device buffer of the call's own; 1 or 4 positions a thread measured the same).
constexpr int KV_COPY_POS = 2;
template <int CAP>
struct KvPages {
    int id[CAP];   // pages of the positions [16 * first page, ...)
};
template <int CAP, int VEC>
__global__ void __launch_bounds__(256)
kv_copy_kernel(op16* pool_layer, const __grid_constant__ KvPages<CAP> pages, int pos0, int n_pos, bf16* k, bf16* v, int kv_dim, int hd_log,
               int to_pool) {
    const int per_pos = kv_dim / VEC;   // threads of a position
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int i0 = t / per_pos * KV_COPY_POS, e = (t % per_pos) * VEC;
    if (i0 >= n_pos) return;
    struct alignas(2 * VEC) Src { bf16 x[VEC]; };
    struct alignas(2 * VEC) Dst { op16 x[VEC]; };
    Src sk[KV_COPY_POS], sv[KV_COPY_POS];
    Dst dk[KV_COPY_POS], dv[KV_COPY_POS];
    const int hd = 1 << hd_log, head = e >> hd_log;
    op16* at[KV_COPY_POS];
#pragma unroll
    for (int i = 0; i < KV_COPY_POS; ++i) {
        const int ii = min(i0 + i, n_pos - 1), row = (pos0 & 15) + ii;
        at[i] = pool_layer + ((size_t)pages.id[row >> 4] * kv_dim * 2 + (size_t)head * 2 * hd) * 16 + (size_t)(row & 15) * hd + (e & (hd - 1));
        const size_t oi = (size_t)ii * kv_dim + e;
        if (to_pool) {
            sk[i] = *reinterpret_cast<const Src*>(k + oi);
            sv[i] = *reinterpret_cast<const Src*>(v + oi);
        } else {
            dk[i] = *reinterpret_cast<const Dst*>(at[i]);
            dv[i] = *reinterpret_cast<const Dst*>(at[i] + 16 * hd);
        }
    }
#pragma unroll
    for (int i = 0; i < KV_COPY_POS; ++i) {
        if (i0 + i >= n_pos) break;
        const size_t oi = (size_t)(i0 + i) * kv_dim + e;
        if (to_pool) {
#pragma unroll
            for (int c = 0; c < VEC; ++c) {
                dk[i].x[c] = to_op(__bfloat162float(sk[i].x[c]));
                dv[i].x[c] = to_op(__bfloat162float(sv[i].x[c]));
            }
            *reinterpret_cast<Dst*>(at[i]) = dk[i];
            *reinterpret_cast<Dst*>(at[i] + 16 * hd) = dv[i];
        } else {
#pragma unroll
            for (int c = 0; c < VEC; ++c) {
                sk[i].x[c] = __float2bfloat16(__half2float(dk[i].x[c]));
                sv[i].x[c] = __float2bfloat16(__half2float(dv[i].x[c]));
            }
            *reinterpret_cast<Src*>(k + oi) = sk[i];
            *reinterpret_cast<Src*>(v + oi) = sv[i];
        }
    }
}

// ------------------------------------------------------------------------------------------ objects

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn g_encode = nullptr;

static int load_driver_entry() {
    if (g_encode) return SYN_OK;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    CU_OK(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres));
    if (!fn || qres != cudaDriverEntryPointSuccess) return SYN_E_CUDA;
    g_encode = reinterpret_cast<EncodeTiledFn>(fn);
    return SYN_OK;
}

// 2-D 16-bit row-major [rows][cols] (pitch in elements), box = box_rows x 64 columns, 128-byte swizzle.
static int make_map_2d(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t cols, uint64_t pitch, uint32_t box_rows) {
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {pitch * 2};
    cuuint32_t box[2] = {64, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = g_encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? SYN_OK : SYN_E_CUDA;
}

// 2-D view of a packed weight matrix for the CTA-pair kernel: rows of 128 bytes (64 bf16), no
// swizzle (the tiles already are shared-memory images); one box = the two 128-row tiles of a
// feature pair for one k-block (QUAD items) or one of them (DUO items).
struct WMaps {
    CUtensorMap quad, duo;
};
static int make_wmaps(const void* packed, int packed_rows, int K, WMaps* out) {
    const uint64_t n_pairs = (uint64_t)((packed_rows + 511) / 512 * 2), nkb = (uint64_t)((K + 63) / 64);
    cuuint64_t dims[2] = {64, n_pairs * nkb * 256};
    cuuint64_t strides[1] = {128};
    cuuint32_t estr[2] = {1, 1};
    for (int k = 0; k < 2; ++k) {
        cuuint32_t box[2] = {64, k == 0 ? 256u : 128u};
        if (g_encode(k == 0 ? &out->quad : &out->duo, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(packed), dims, strides,
                     box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return SYN_E_CUDA;
    }
    return SYN_OK;
}

// The token operand of a projection, [tokens][K] half precision, as boxes of 32 rows (the kernels of gemm.cuh and
// gemm2.cuh) and, for the thin kernel, of 16, 32, ... THIN_MAX_TN rows: one box is a whole token tile.
struct XMaps {
    CUtensorMap box, thin[THIN_MAX_TN / 16];
};
static int make_xmaps(XMaps* out, const void* base, uint64_t rows, uint64_t K) {
    int r = make_map_2d(&out->box, base, rows, K, K, GEMM_BOX_ROWS);
    for (int i = 0; i < THIN_MAX_TN / 16 && !r; ++i) r = make_map_2d(&out->thin[i], base, rows, K, K, 16 * (i + 1));
    return r;
}

struct syn_model {
    syn_model_desc desc;
    int f_pad, n_sm, gu_rows, qkv_rows, v_rows;
    bf16 *embed = nullptr, *final_norm = nullptr;
    op16* lm_head = nullptr;
    std::vector<op16*> wqkv, wo, wgu, wd;                 // projections in the packed tile layout (half precision)
    std::vector<bf16*> norm1, norm2;
    std::vector<WMaps> tm_wqkv, tm_wo, tm_wgu, tm_wd;      // their tensor maps
    WMaps tm_lm_head;
    double* inv_freq = nullptr;
    int* status_dev = nullptr;
    // workspace (grow-only)
    int t_cap = 0;
    float *x = nullptr, *ssq = nullptr;   // residual stream; sums of x^2 per token and 32 features
    op16 *xn = nullptr,   // half(x * gain of the next RMSNorm): the operand of the qkv, gate/up and lm_head projections
         *q = nullptr, *attn = nullptr, *act = nullptr;
    float2* rope = nullptr;
    unsigned long long* best = nullptr;
    op16* xj = nullptr;      // operand and sums of the rows that verification looks at, where the lm_head runs over those alone
    float* ssqj = nullptr;
    XMaps tm_xn, tm_attn, tm_act, tm_xj;
    CUtensorMap tm_q, tm_q4;
    float* fix_part = nullptr;      // stored accumulators of K-split remainder tiles (one slot per SM)
    int* fix_flag = nullptr;        // their arrival / release counters, [GEMM_FLAG_INTS * n_sm], zero between launches
    float* part_o = nullptr;
    float2* part_ml = nullptr;
    int* group_count = nullptr;     // per merge group: partial items completed (zero between launches)
    int part_cap = 0;
    syn_plan* scratch_plan = nullptr;
    // sampling-based verification (grow-only): logits of a step, the rows' top-k lists, the
    // transmitted SLM distributions and the uniform draws
    struct SampleWs {
        float *logits = nullptr, *topk_logit = nullptr, *slm_prob = nullptr, *rand_accept = nullptr, *rand_sample = nullptr;
        int *topk_id = nullptr, *slm_id = nullptr;
        uint32_t* warp_max = nullptr;   // [t_cap][v_rows / 32]: per-group maxima stored by the lm_head epilogue
        size_t logits_cap = 0;
        int t_cap = 0, b_cap = 0, slm_cap = 0;
    } sw;
    int* pinned_out = nullptr;
    int pinned_out_cap = 0;
    // what syn_last_step_stats reports: the counters of the last step launched on this model and,
    // with profiling on, its device time (events around the whole step) and the wall time of the
    // blocking call
    syn_step_stats last_stats;
    bool have_last = false, step_timed = false;
    cudaEvent_t step_a = nullptr, step_b = nullptr;
    double last_wall_ms = 0.0;
    // per-class event timing
    bool profile = false;
    struct Ev { cudaEvent_t a, b; int cls; };
    std::vector<Ev> ev_used, ev_free;
};

// Brackets one launch with events when profiling is on.
struct ProfScope {
    syn_model* m; cudaStream_t st; syn_model::Ev ev; bool on;
    ProfScope(syn_model* m_, int cls, cudaStream_t st_) : m(m_), st(st_), on(m_ && m_->profile) {
        if (!on) return;
        if (!m->ev_free.empty()) { ev = m->ev_free.back(); m->ev_free.pop_back(); }
        else if (cudaEventCreate(&ev.a) != cudaSuccess || cudaEventCreate(&ev.b) != cudaSuccess) { on = false; return; }
        ev.cls = cls;
        cudaEventRecord(ev.a, st);
    }
    ~ProfScope() {
        if (!on) return;
        cudaEventRecord(ev.b, st);
        m->ev_used.push_back(ev);
    }
};

struct syn_kv {
    syn_model* model;
    op16* pool = nullptr;   // half precision (K and V enter and leave through syn_kv_import / syn_kv_export as bf16)
    uint32_t n_pages, page_size;
    size_t layer_elems;
    CUtensorMap tm_kv, tm_kv5;   // boxes of 32 rows (K and V of a page and head); of 16 rows (K or V) with both 64-dim halves
};

// The attention kernels a work list can be made for.
enum { ATTN_WARP = 1, ATTN_TENSOR = 2, ATTN_THIN = 3 };
static int attn_rows(int kind) { return kind == ATTN_TENSOR ? 128 : kind == ATTN_THIN ? ATTN_THIN_ROWS : 64; }

struct syn_plan {
    syn_step_stats stats;
    int n_req = 0, T = 0, max_pages = 0, n_items = 0, n_cta = 0, n_groups = 0, n_parts = 0;
    int attn = ATTN_WARP;   // which attention kernel the work list was made for
    // one device buffer and its pinned host mirror
    uint8_t *dev = nullptr, *host = nullptr;
    size_t cap = 0, used = 0;
    // offsets into the buffer
    size_t o_tokens, o_pos, o_slot, o_offsets, o_uncached, o_tables, o_items, o_cta, o_groups;
    size_t o_row, o_first;   // the judging rows, and where a request's begin among them
    int n_judging = 0;       // rows whose argmax verification looks at: a request's from its last uncached token on
    // the cache the page ids and slots were validated against
    const syn_kv* kv = nullptr;
    const void* kv_pool = nullptr;
    uint32_t kv_pages = 0;
    template <class Tp> Tp* d(size_t off) const { return reinterpret_cast<Tp*>(dev + off); }
    template <class Tp> Tp* h(size_t off) const { return reinterpret_cast<Tp*>(host + off); }
};

static void free_workspace(syn_model* m) {
    cudaFree(m->x); cudaFree(m->ssq); cudaFree(m->xn); cudaFree(m->q); cudaFree(m->attn); cudaFree(m->act);
    cudaFree(m->rope); cudaFree(m->best); cudaFree(m->xj); cudaFree(m->ssqj);
    m->xj = nullptr; m->ssqj = nullptr;
    m->x = m->ssq = nullptr; m->xn = m->q = m->attn = m->act = nullptr; m->rope = nullptr; m->best = nullptr;
    m->t_cap = 0;
}

static int ensure_workspace(syn_model* m, int T, int n_parts) {
    const syn_model_desc& c = m->desc;
    const int q_dim = c.n_q_heads * c.head_dim;
    if (T > m->t_cap) {
        free_workspace(m);
        const int cap = (T + 255) / 256 * 256;
        CU_OK(cudaMalloc(&m->x, (size_t)cap * c.d_model * 4));
        CU_OK(cudaMalloc(&m->ssq, (size_t)cap * (c.d_model / 32) * 4));
        CU_OK(cudaMalloc(&m->xn, (size_t)cap * c.d_model * 2));
        CU_OK(cudaMalloc(&m->q, (size_t)cap * q_dim * 2));
        CU_OK(cudaMalloc(&m->attn, (size_t)cap * q_dim * 2));
        CU_OK(cudaMalloc(&m->act, (size_t)cap * m->f_pad * 2));
        CU_OK(cudaMalloc(&m->rope, (size_t)cap * (c.head_dim / 2) * 8));
        CU_OK(cudaMalloc(&m->best, (size_t)cap * 8));
        CU_OK(cudaMalloc(&m->xj, (size_t)(cap / 2) * c.d_model * 2));
        CU_OK(cudaMalloc(&m->ssqj, (size_t)(cap / 2) * (c.d_model / 32) * 4));
        CU_OK(cudaMemset(m->xj, 0, (size_t)(cap / 2) * c.d_model * 2));
        CU_OK(cudaMemset(m->xn, 0, (size_t)cap * c.d_model * 2));
        CU_OK(cudaMemset(m->q, 0, (size_t)cap * q_dim * 2));
        CU_OK(cudaMemset(m->attn, 0, (size_t)cap * q_dim * 2));
        CU_OK(cudaMemset(m->act, 0, (size_t)cap * m->f_pad * 2));
        m->t_cap = cap;
        int r;
        if ((r = make_xmaps(&m->tm_xn, m->xn, cap, c.d_model))) return r;
        if ((r = make_xmaps(&m->tm_xj, m->xj, cap / 2, c.d_model))) return r;
        if ((r = make_xmaps(&m->tm_attn, m->attn, cap, q_dim))) return r;
        if ((r = make_xmaps(&m->tm_act, m->act, cap, m->f_pad))) return r;
        // Q tile of the attention kernel: [token][128-byte line][64]; box = min(16, 64/G) tokens x (G * hd/64) lines
        const uint32_t G = c.n_q_heads / c.n_kv_heads, halves = c.head_dim / 64;
        const uint32_t box_tokens = std::min(16u, 64u / G);
        cuuint64_t dims[3] = {64, (cuuint64_t)q_dim / 64, (cuuint64_t)cap};
        cuuint64_t strides[2] = {128, (cuuint64_t)q_dim * 2};
        cuuint32_t box[3] = {64, G * halves, box_tokens};
        cuuint32_t estr[3] = {1, 1, 1};
        if (g_encode(&m->tm_q, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, m->q, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return SYN_E_CUDA;
        // Q tile of the tensor-memory attention kernel: [token][head][64-dim half][64]; one box = one half of the
        // G heads of a kv head for min(32, 128 / G) tokens, i.e. rows (token, head) of 128 bytes
        cuuint64_t dims4[4] = {64, halves, c.n_q_heads, (cuuint64_t)cap};
        cuuint64_t strides4[3] = {128, (cuuint64_t)c.head_dim * 2, (cuuint64_t)q_dim * 2};
        cuuint32_t box4[4] = {64, 1, G, std::min((uint32_t)SYN_MAX_CHUNK, 128u / G)};
        cuuint32_t estr4[4] = {1, 1, 1, 1};
        if (g_encode(&m->tm_q4, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, m->q, dims4, strides4, box4, estr4,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return SYN_E_CUDA;
    }
    if (!m->fix_part) {
        CU_OK(cudaMalloc(&m->fix_part, (size_t)m->n_sm * GEMM_FIX_SLOT_BYTES));
        CU_OK(cudaMalloc(&m->fix_flag, (size_t)GEMM_FLAG_INTS * m->n_sm * 4));
        CU_OK(cudaMemset(m->fix_flag, 0, (size_t)GEMM_FLAG_INTS * m->n_sm * 4));
    }
    if (n_parts > m->part_cap) {
        cudaFree(m->part_o); cudaFree(m->part_ml); cudaFree(m->group_count);
        m->part_o = nullptr; m->part_ml = nullptr; m->group_count = nullptr; m->part_cap = 0;
        const int cap = (n_parts + 255) / 256 * 256;
        CU_OK(cudaMalloc(&m->part_o, (size_t)cap * 128 * c.head_dim * 4));   // rows of the larger tile
        CU_OK(cudaMalloc(&m->part_ml, (size_t)cap * 128 * 8));
        CU_OK(cudaMalloc(&m->group_count, (size_t)cap * 4));   // a group has >= 2 parts: cap/2 would do
        CU_OK(cudaMemset(m->group_count, 0, (size_t)cap * 4));
        m->part_cap = cap;
    }
    return SYN_OK;
}

// Dynamic shared memory of every kernel that needs more than the default, and the same carveout for all kernels of
// the step: an SM has to drain before it can change its carveout, which would keep neighbours apart.
template <typename K>
static cudaError_t kernel_smem(K kernel, int bytes) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess && bytes > 0) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return e;
}
// Which variants of the one-CTA projection kernel an epilogue meets (gemm_plan): leftover tiles of a residual projection are
// not cut along K, only qkv and residual projections share K.
constexpr bool gemm_variant_used(int variant, int mode) {
    return variant == GEMM_KSPLIT ? mode != EPI_RESID : (variant == GEMM_RSPLIT ? mode != EPI_SWIGLU && mode != EPI_LMHEAD : true);
}
template <int VARIANT, int MODE>
static cudaError_t gemm_kernel_smem() {
    if constexpr (gemm_variant_used(VARIANT, MODE)) return kernel_smem(gemm_kernel<VARIANT, MODE>, GEMM_SMEM_MAX);
    else return cudaSuccess;
}
template <int MODE>
static cudaError_t projection_smem() {   // the projection kernels with one epilogue
    const cudaError_t all[] = {gemm_kernel_smem<GEMM_WAVES, MODE>(), gemm_kernel_smem<GEMM_KSPLIT, MODE>(), gemm_kernel_smem<GEMM_RSPLIT, MODE>(),
                               kernel_smem(gemm2_kernel<false, MODE>, GEMM_SMEM_MAX), kernel_smem(gemm2_kernel<true, MODE>, GEMM_SMEM_MAX),
                               kernel_smem(thin_kernel<MODE>, THIN_SMEM_MAX)};
    for (cudaError_t e : all)
        if (e != cudaSuccess) return e;
    return cudaSuccess;
}
static cudaError_t set_kernel_attributes() {
    const cudaError_t all[] = {
        projection_smem<EPI_PLAIN>(), projection_smem<EPI_QKV>(), projection_smem<EPI_RESID>(), projection_smem<EPI_SWIGLU>(), projection_smem<EPI_LMHEAD>(),
        kernel_smem(attn_kernel<128>, AttnSmem<128>::TOTAL), kernel_smem(attn_kernel<64>, AttnSmem<64>::TOTAL),
        kernel_smem(attn2_kernel<128>, Attn2Smem<128>::TOTAL), kernel_smem(attn2_kernel<64>, Attn2Smem<64>::TOTAL),
        kernel_smem(attn_thin_kernel<128>, AttnThinSmem<128>::TOTAL), kernel_smem(attn_thin_kernel<64>, AttnThinSmem<64>::TOTAL),
        kernel_smem(prep_kernel, 0), kernel_smem(verify_kernel, 0), kernel_smem(judging_rows_kernel, 0), kernel_smem(topk_rows_kernel, 0), kernel_smem(sample_verify_kernel, 0)};
    for (cudaError_t e : all)
        if (e != cudaSuccess) return e;
    return cudaSuccess;
}

// ------------------------------------------------------------------------------------------ model

extern "C" void syn_model_free(syn_model* m) {
    if (!m) return;
    for (auto& v : {&m->wqkv, &m->wo, &m->wgu, &m->wd})
        for (op16* p : *v) cudaFree(p);
    for (auto& v : {&m->norm1, &m->norm2})
        for (bf16* p : *v) cudaFree(p);
    cudaFree(m->embed); cudaFree(m->lm_head); cudaFree(m->final_norm); cudaFree(m->inv_freq); cudaFree(m->status_dev);
    free_workspace(m);
    cudaFree(m->part_o); cudaFree(m->part_ml); cudaFree(m->group_count);
    cudaFree(m->fix_part); cudaFree(m->fix_flag);
    if (m->pinned_out) cudaFreeHost(m->pinned_out);
    cudaFree(m->sw.logits); cudaFree(m->sw.topk_logit); cudaFree(m->sw.topk_id); cudaFree(m->sw.slm_id);
    cudaFree(m->sw.slm_prob); cudaFree(m->sw.rand_accept); cudaFree(m->sw.rand_sample); cudaFree(m->sw.warp_max);
    if (m->scratch_plan) syn_plan_free(m->scratch_plan);
    for (auto* v : {&m->ev_used, &m->ev_free})
        for (auto& e : *v) { cudaEventDestroy(e.a); cudaEventDestroy(e.b); }
    if (m->step_a) cudaEventDestroy(m->step_a);
    if (m->step_b) cudaEventDestroy(m->step_b);
    delete m;
}

static int syn_model_load_impl(const syn_model_desc* desc, const syn_weights* w, syn_model** out) {
    if (!desc || !w || !out) return SYN_E_INVALID_ARG;
    const syn_model_desc c = *desc;
    if (c.flags != 0 || c.n_layers == 0 || c.vocab == 0 || c.d_ffn == 0) return SYN_E_INVALID_ARG;
    if (c.head_dim != 64 && c.head_dim != 128) return SYN_E_INVALID_ARG;
    if (c.d_model == 0 || c.d_model % 128 != 0 || c.d_ffn % 8 != 0) return SYN_E_INVALID_ARG;
    if (c.n_kv_heads == 0 || c.n_q_heads % c.n_kv_heads != 0 || c.n_q_heads / c.n_kv_heads > 8) return SYN_E_INVALID_ARG;
    if ((c.n_q_heads * c.head_dim) % 128 != 0 || (c.n_kv_heads * c.head_dim) % 128 != 0) return SYN_E_INVALID_ARG;
    if (!(c.rope_base > 0.f) || !(c.rms_eps >= 0.f)) return SYN_E_INVALID_ARG;
    if (!w->embed || !w->lm_head || !w->final_norm || !w->wq || !w->wk || !w->wv || !w->wo || !w->wg || !w->wu ||
        !w->wd || !w->norm1 || !w->norm2 || (w->location != 0 && w->location != 1))
        return SYN_E_INVALID_ARG;
    for (uint32_t l = 0; l < c.n_layers; ++l)
        if (!w->wq[l] || !w->wk[l] || !w->wv[l] || !w->wo[l] || !w->wg[l] || !w->wu[l] || !w->wd[l] || !w->norm1[l] ||
            !w->norm2[l])
            return SYN_E_INVALID_ARG;
    int dev = 0;
    cudaDeviceProp prop;
    CU_OK(cudaGetDevice(&dev));
    CU_OK(cudaGetDeviceProperties(&prop, dev));
    if (prop.major != 10) return SYN_E_ARCH;
    int r = load_driver_entry();
    if (r) return r;

    syn_model* m = new (std::nothrow) syn_model();
    if (!m) return SYN_E_OOM;
    m->desc = c;
    m->n_sm = prop.multiProcessorCount;
    m->f_pad = (c.d_ffn + 63) / 64 * 64;
    const int d = c.d_model, q_dim = c.n_q_heads * c.head_dim, kv_dim = c.n_kv_heads * c.head_dim, f = c.d_ffn;
    m->qkv_rows = q_dim + 2 * kv_dim;
    m->gu_rows = 2 * m->f_pad;
    m->v_rows = (c.vocab + 127) / 128 * 128;
    const int loc = w->location;
    const cudaMemcpyKind kind = loc ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;

#define LOAD_FAIL(code)        \
    do {                       \
        syn_model_free(m);     \
        return (code);         \
    } while (0)
#define CU_M(expr)                                                                        \
    do {                                                                                  \
        cudaError_t _e = (expr);                                                          \
        if (_e != cudaSuccess) {                                                          \
            (void)cudaGetLastError();                                                     \
            LOAD_FAIL(_e == cudaErrorMemoryAllocation ? SYN_E_OOM : SYN_E_CUDA);          \
        }                                                                                 \
    } while (0)

    CU_M(cudaMalloc(&m->embed, (size_t)c.vocab * d * 2));
    CU_M(cudaMemcpy(m->embed, w->embed, (size_t)c.vocab * d * 2, kind));
    CU_M(cudaMalloc(&m->final_norm, (size_t)d * 2));
    CU_M(cudaMemcpy(m->final_norm, w->final_norm, (size_t)d * 2, kind));
    // staging buffer for host-resident sources (largest single matrix)
    bf16* stage[3] = {nullptr, nullptr, nullptr};
    if (!loc) {
        const size_t big = std::max((size_t)c.vocab * d, std::max((size_t)f * d, (size_t)q_dim * d));
        for (int k = 0; k < 3; ++k) {
            const size_t n = k == 0 ? big : (k == 1 ? std::max((size_t)f * d, (size_t)kv_dim * d) : (size_t)kv_dim * d);
            cudaError_t e = cudaMalloc(&stage[k], n * 2);
            if (e != cudaSuccess) {
                (void)cudaGetLastError();
                for (int j = 0; j < k; ++j) cudaFree(stage[j]);
                LOAD_FAIL(SYN_E_OOM);
            }
        }
    }
    // pack `n` row-major sources (rows[i] x src_k each) into a new tile-layout buffer of `packed_rows` x K
    auto pack = [&](const void* const* srcs, const int* rows, int n, int mode, int src_k, int packed_rows,
                    op16** out_ptr) -> int {
        const int n_mt = (packed_rows + 511) / 512 * 4, nkb = (src_k + 63) / 64;   // an even number of feature pairs (zero rows at the end)
        op16* outp = nullptr;
        cudaError_t e = cudaMalloc(&outp, (size_t)n_mt * nkb * 128 * 64 * 2);
        if (e != cudaSuccess) { (void)cudaGetLastError(); return SYN_E_OOM; }
        *out_ptr = outp;
        PackSrc ps;
        memset(&ps, 0, sizeof(ps));
        ps.mode = mode; ps.src_k = src_k; ps.hd = (int)c.head_dim;
        for (int i = 0; i < n; ++i) {
            ps.rows[i] = rows[i];
            if (loc) ps.p[i] = (const bf16*)srcs[i];
            else {
                if (cudaMemcpy(stage[i], srcs[i], (size_t)rows[i] * src_k * 2, cudaMemcpyHostToDevice) != cudaSuccess) {
                    cudaFree(outp);
                    *out_ptr = nullptr;
                    return SYN_E_CUDA;
                }
                ps.p[i] = stage[i];
            }
        }
        pack_weight_kernel<<<dim3(n_mt, nkb), 256>>>(ps, outp, nkb);
        if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) {
            cudaFree(outp);
            *out_ptr = nullptr;
            return SYN_E_CUDA;
        }
        return SYN_OK;
    };
#define PACK_OR_FAIL(call)                                  \
    do {                                                    \
        int _r = (call);                                    \
        if (_r) {                                           \
            for (int j = 0; j < 3; ++j) cudaFree(stage[j]); \
            LOAD_FAIL(_r);                                  \
        }                                                   \
    } while (0)
    {
        const void* srcs[1] = {w->lm_head};
        const int rows[1] = {(int)c.vocab};
        PACK_OR_FAIL(pack(srcs, rows, 1, 0, d, c.vocab, &m->lm_head));
        PACK_OR_FAIL(make_wmaps(m->lm_head, m->v_rows, d, &m->tm_lm_head));
    }
    for (uint32_t l = 0; l < c.n_layers; ++l) {
        bf16 *n1 = nullptr, *n2 = nullptr;
        op16* pk = nullptr;
        {
            const void* srcs[3] = {w->wq[l], w->wk[l], w->wv[l]};
            const int rows[3] = {q_dim, kv_dim, kv_dim};
            PACK_OR_FAIL(pack(srcs, rows, 3, 2, d, m->qkv_rows, &pk));
            m->wqkv.push_back(pk);
            WMaps wm;
            PACK_OR_FAIL(make_wmaps(pk, m->qkv_rows, d, &wm));
            m->tm_wqkv.push_back(wm);
        }
        {
            const void* srcs[1] = {w->wo[l]};
            const int rows[1] = {d};
            PACK_OR_FAIL(pack(srcs, rows, 1, 0, q_dim, d, &pk));
            m->wo.push_back(pk);
            WMaps wm;
            PACK_OR_FAIL(make_wmaps(pk, d, q_dim, &wm));
            m->tm_wo.push_back(wm);
        }
        {   // a tile holds the gate and the up rows of the same 64 features; rows of the padded tail are zero
            const void* srcs[2] = {w->wg[l], w->wu[l]};
            const int rows[2] = {f, f};
            PACK_OR_FAIL(pack(srcs, rows, 2, 1, d, m->gu_rows, &pk));
            m->wgu.push_back(pk);
            WMaps wm;
            PACK_OR_FAIL(make_wmaps(pk, m->gu_rows, d, &wm));
            m->tm_wgu.push_back(wm);
        }
        {   // down projection: K = d_ffn, zero-padded to f_pad by the k-block tail
            const void* srcs[1] = {w->wd[l]};
            const int rows[1] = {d};
            PACK_OR_FAIL(pack(srcs, rows, 1, 0, f, d, &pk));
            m->wd.push_back(pk);
            WMaps wm;
            PACK_OR_FAIL(make_wmaps(pk, d, m->f_pad, &wm));
            m->tm_wd.push_back(wm);
        }
        CU_M(cudaMalloc(&n1, (size_t)d * 2)); m->norm1.push_back(n1);
        CU_M(cudaMalloc(&n2, (size_t)d * 2)); m->norm2.push_back(n2);
        CU_M(cudaMemcpy(n1, w->norm1[l], (size_t)d * 2, kind));
        CU_M(cudaMemcpy(n2, w->norm2[l], (size_t)d * 2, kind));
    }
    for (int j = 0; j < 3; ++j) cudaFree(stage[j]);
#undef PACK_OR_FAIL
    std::vector<double> inv(c.head_dim / 2);
    for (uint32_t i = 0; i < c.head_dim / 2; ++i) inv[i] = std::pow((double)c.rope_base, -2.0 * (double)i / (double)c.head_dim);
    CU_M(cudaMalloc(&m->inv_freq, inv.size() * 8));
    CU_M(cudaMemcpy(m->inv_freq, inv.data(), inv.size() * 8, cudaMemcpyHostToDevice));
    CU_M(cudaMalloc(&m->status_dev, 4));
    CU_M(cudaMemset(m->status_dev, 0, 4));
    CU_M(set_kernel_attributes());
    CU_M(cudaDeviceSynchronize());
    *out = m;
    return SYN_OK;
#undef CU_M
#undef LOAD_FAIL
}

// ------------------------------------------------------------------------------------------ KV pool

extern "C" void syn_kv_free(syn_kv* kv) {
    if (!kv) return;
    cudaFree(kv->pool);
    delete kv;
}

extern "C" int syn_kv_alloc(syn_model* m, uint32_t n_pages, uint32_t page_size, syn_kv** out) {
    if (!m || !out || n_pages == 0 || page_size != 16) return SYN_E_INVALID_ARG;
    const syn_model_desc& c = m->desc;
    const uint64_t blocks = (uint64_t)c.n_layers * n_pages * c.n_kv_heads * 2;
    if (blocks > 0x7FFFFFFFull) return SYN_E_INVALID_ARG;
    syn_kv* kv = new (std::nothrow) syn_kv();
    if (!kv) return SYN_E_OOM;
    kv->model = m;
    kv->n_pages = n_pages;
    kv->page_size = page_size;
    kv->layer_elems = (size_t)n_pages * c.n_kv_heads * 2 * page_size * c.head_dim;
    const size_t bytes = kv->layer_elems * c.n_layers * 2;
    cudaError_t e = cudaMalloc(&kv->pool, bytes);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        delete kv;
        return e == cudaErrorMemoryAllocation ? SYN_E_OOM : SYN_E_CUDA;
    }
    if (cudaMemset(kv->pool, 0, bytes) != cudaSuccess) {
        syn_kv_free(kv);
        return SYN_E_CUDA;
    }
    // pool as a 2-D tensor [blocks * 16 rows][head_dim]; a box of 32 rows x 64 columns is one
    // 64-element half of the K rows and the V rows of one (page, kv head)
    if (make_map_2d(&kv->tm_kv, kv->pool, blocks * page_size, c.head_dim, c.head_dim, 2 * page_size) != SYN_OK) {
        syn_kv_free(kv);
        return SYN_E_CUDA;
    }
    {
        // The 16 K rows (or the 16 V rows) of a page and head as one box for the tensor-memory attention
        // kernel, landing in shared memory as [rows 0-7: dims 0-63][rows 0-7: dims 64-127][rows 8-15: ...]:
        // the 8-row groups of consecutive boxes are then evenly spaced for either 64-dim half, which a tcgen05
        // operand descriptor needs.  Dimensions: dim in a half, row in a group, half, group, 16-row block.
        const cuuint64_t hd2 = (cuuint64_t)c.head_dim * 2;
        cuuint64_t dims[5] = {64, 8, c.head_dim / 64, 2, (cuuint64_t)blocks};
        cuuint64_t strides[4] = {hd2, 128, 8 * hd2, 16 * hd2};
        cuuint32_t box[5] = {64, 8, c.head_dim / 64, 2, 1};
        cuuint32_t estr[5] = {1, 1, 1, 1, 1};
        if (g_encode(&kv->tm_kv5, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 5, kv->pool, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            syn_kv_free(kv);
            return SYN_E_CUDA;
        }
    }
    if (cudaDeviceSynchronize() != cudaSuccess) {
        syn_kv_free(kv);
        return SYN_E_CUDA;
    }
    *out = kv;
    return SYN_OK;
}

constexpr int KV_COPY_PAGES_SMALL = 192, KV_COPY_PAGES = 960;   // page ids a launch carries (parameters of 0.8 and 3.8 KB)

template <int CAP, int VEC>
static int kv_copy_launch(syn_kv* kv, uint32_t layer, const int32_t* pages, int n_pages, int pos0, int n_pos, bf16* k, bf16* v,
                          cudaStream_t st, int to_pool) {
    const syn_model_desc& c = kv->model->desc;
    KvPages<CAP> pg;
    memcpy(pg.id, pages, (size_t)n_pages * 4);
    const int kv_dim = (int)(c.n_kv_heads * c.head_dim);
    const int64_t threads = (int64_t)((n_pos + KV_COPY_POS - 1) / KV_COPY_POS) * (kv_dim / VEC);
    kv_copy_kernel<CAP, VEC><<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(kv->pool + kv->layer_elems * layer, pg, pos0, n_pos, k, v, kv_dim,
                                                                                 c.head_dim == 128 ? 7 : 6, to_pool);
    return launch_ok() ? SYN_OK : SYN_E_CUDA;
}

static int kv_copy(syn_kv* kv, uint32_t layer, const int32_t* page_table, int32_t pos0, int32_t n_pos, void* k, void* v,
                   void* stream, int to_pool) {
    if (!kv || !page_table || !k || !v || pos0 < 0 || n_pos <= 0 || layer >= kv->model->desc.n_layers)
        return SYN_E_INVALID_ARG;
    const int P = (int)kv->page_size, first = pos0 / P, last = (int)(((int64_t)pos0 + n_pos - 1) / P);
    for (int i = first; i <= last; ++i)
        if (page_table[i] < 0 || (uint32_t)page_table[i] >= kv->n_pages) return SYN_E_PAGE_OOB;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // launches of at most KV_COPY_PAGES pages; short transfers carry the smaller parameter
    const size_t kv_dim = (size_t)kv->model->desc.n_kv_heads * kv->model->desc.head_dim;
    return for_pieces(
        pos0, n_pos, P, KV_COPY_PAGES,
        [&](int at, int n, int64_t done) {
            const int p0 = at / P, n_pg = (at % P + n + P - 1) / P;
            bf16 *kk = (bf16*)k + (size_t)done * kv_dim, *vv = (bf16*)v + (size_t)done * kv_dim;
            const bool vec = (((uintptr_t)kk | (uintptr_t)vv) & 15) == 0;
            return n_pg <= KV_COPY_PAGES_SMALL
                       ? (vec ? kv_copy_launch<KV_COPY_PAGES_SMALL, 8>(kv, layer, page_table + p0, n_pg, at, n, kk, vv, st, to_pool)
                              : kv_copy_launch<KV_COPY_PAGES_SMALL, 1>(kv, layer, page_table + p0, n_pg, at, n, kk, vv, st, to_pool))
                       : (vec ? kv_copy_launch<KV_COPY_PAGES, 8>(kv, layer, page_table + p0, n_pg, at, n, kk, vv, st, to_pool)
                              : kv_copy_launch<KV_COPY_PAGES, 1>(kv, layer, page_table + p0, n_pg, at, n, kk, vv, st, to_pool));
        },
        [&]() -> int {
            CU_OK(cudaStreamSynchronize(st));
            return SYN_OK;
        });
}

static int syn_kv_import_impl(syn_kv* kv, uint32_t layer, const int32_t* page_table, int32_t pos0, int32_t n_pos,
                             const void* k, const void* v, void* stream) {
    return kv_copy(kv, layer, page_table, pos0, n_pos, const_cast<void*>(k), const_cast<void*>(v), stream, 1);
}
static int syn_kv_export_impl(syn_kv* kv, uint32_t layer, const int32_t* page_table, int32_t pos0, int32_t n_pos, void* k,
                             void* v, void* stream) {
    return kv_copy(kv, layer, page_table, pos0, n_pos, k, v, stream, 0);
}

// ------------------------------------------------------------------------------------------ planner

extern "C" void syn_plan_free(syn_plan* p) {
    if (!p) return;
    cudaFree(p->dev);
    if (p->host) cudaFreeHost(p->host);
    delete p;
}

static size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// CTAs of the half-SM attention kernel that a device of n_sm SMs holds at a time.
static int thin_attention_ctas(int n_sm) { return 2 * n_sm; }

// Host-side result of planning one batch (no device involved).
struct HostPlan {
    int T = 0, n_cta = 0, n_parts = 0, kind = ATTN_WARP;
    std::vector<int> pos, slot, cta_begin;
    std::vector<AttnItem> items;          // sorted by CTA
    std::vector<MergeGroup> groups;
    syn_step_stats stats;
};

// Validate the batch, then build token positions, KV slots and the attention work list
// (the "flatten" of paper Sec. 4.5).  Pure host code.  thin_ctas: CTAs to plan for when the half-SM kernel is taken.
static int plan_compute(const syn_model_desc& c, int P, uint32_t n_pages, int n_sm, int32_t n_req,
                        const int32_t* chunk_tokens, const int32_t* chunk_offsets, const int32_t* page_tables,
                        int32_t max_pages, const int32_t* ctx_lens, const int32_t* n_uncached, int attention, int thin_ctas, HostPlan& hp) {
    if (n_req <= 0 || !chunk_tokens || !chunk_offsets || !page_tables || !ctx_lens || max_pages <= 0 || n_sm <= 0)
        return SYN_E_INVALID_ARG;
    const int G = c.n_q_heads / c.n_kv_heads, Hkv = c.n_kv_heads;
    if (chunk_offsets[0] != 0) return SYN_E_INVALID_ARG;
    int64_t ctx_sum = 0, keys_seen = 0, kv_units = 0;
    int max_chunk = 0;
    for (int i = 0; i < n_req; ++i) {
        const int64_t n = (int64_t)chunk_offsets[i + 1] - chunk_offsets[i];
        if (n < 1 || n > SYN_MAX_CHUNK) return SYN_E_CHUNK_LEN;
        const int u = n_uncached ? n_uncached[i] : 1;
        if (u < 1 || u > n) return SYN_E_UNCACHED;
        if (ctx_lens[i] < 0) return SYN_E_INVALID_ARG;
        if ((int64_t)ctx_lens[i] + n > (int64_t)max_pages * P) return SYN_E_CAPACITY;
        const int used = (int)((ctx_lens[i] + n + P - 1) / P);
        const int32_t* row = page_tables + (size_t)i * max_pages;
        uint32_t worst = 0;   // a negative id is a large unsigned one
        for (int k = 0; k < used; ++k) worst = std::max(worst, (uint32_t)row[k]);
        if (worst >= n_pages) return SYN_E_PAGE_OOB;
        ctx_sum += ctx_lens[i];
        max_chunk = std::max(max_chunk, (int)n);
        kv_units += ctx_lens[i] + n;
        keys_seen += n * (int64_t)ctx_lens[i] + n * (n + 1) / 2;
    }
    const int T = chunk_offsets[n_req];
    for (int t = 0; t < T; ++t)
        if (chunk_tokens[t] < 0 || (uint32_t)chunk_tokens[t] >= c.vocab) return SYN_E_TOKEN_OOB;
    std::vector<int>& pos = hp.pos;
    std::vector<int>& slot = hp.slot;
    pos.assign(T, 0);
    slot.assign(T, 0);
    for (int i = 0; i < n_req; ++i)
        for (int j = 0, b = chunk_offsets[i]; b + j < chunk_offsets[i + 1]; ++j) {
            const int pp = ctx_lens[i] + j;
            pos[b + j] = pp;
            slot[b + j] = page_tables[(size_t)i * max_pages + pp / P] * P + pp % P;
        }
    {
        // Two chunk tokens may not share a KV slot.  Inside a request the chunk's slots differ unless
        // two of its (at most three) pages are the same page; between requests they can only meet in
        // a page both chunks write.  So look at the pages first, and at the slots only if a page
        // is written twice.
        std::vector<int> pg;
        pg.reserve((size_t)n_req * 3);
        for (int i = 0; i < n_req; ++i) {
            const int first = ctx_lens[i] / P, last = (ctx_lens[i] + (chunk_offsets[i + 1] - chunk_offsets[i]) - 1) / P;
            for (int k = first; k <= last; ++k) pg.push_back(page_tables[(size_t)i * max_pages + k]);
        }
        std::sort(pg.begin(), pg.end());
        if (std::adjacent_find(pg.begin(), pg.end()) != pg.end()) {
            std::vector<int> s2(slot);
            std::sort(s2.begin(), s2.end());
            if (std::adjacent_find(s2.begin(), s2.end()) != s2.end()) return SYN_E_PAGE_ALIAS;
        }
    }
    // Attention work list: (request, kv head, token group, key range).  Cost of an item, in SM cycles: its blocks of
    // 64 keys times a time per block that grows with the number of 16-row query tiles (more tensor work per key byte),
    // plus a fixed overhead per item, plus one more if it covers only part of its unit's keys (an fp32 partial); `fixed` is the
    // kernel's own, `merge` and `merge_tile` (per part and query tile) what the CTA that ends a unit's last part has still to
    // do.  Fitted to per-CTA durations of some twenty batches of the 1B, 8B and 32B shapes (rms error 7 to 10 %); the half-SM
    // kernel's are 5 to 15 % above its fit, which was taken where HBM was not yet the bound.
    struct AttnCost { int kind, block[5], item, part, fixed, merge, merge_tile; };
    static const AttnCost COSTS[2][3] = {
        {{ATTN_WARP, {0, 760, 820, 965, 1050}, 3400, 1600, 4000, 5000, 400}, {ATTN_TENSOR, {0, 1100, 1100, 1100, 1100}, 2800, 3900, 7100, 12000, 200},
         {ATTN_THIN, {0, 1050, 1170, 2080, 2200}, 4700, 2800, 4500, 4000, 350}},
        {{ATTN_WARP, {0, 1110, 1200, 1600, 1650}, 6500, 2400, 5600, 6000, 800}, {ATTN_TENSOR, {0, 1300, 1300, 1300, 1300}, 3400, 6500, 11400, 25000, 200},
         {ATTN_THIN, {0, 2600, 2800, 4500, 4800}, 3700, 2200, 6500, 4500, 700}}};
    const AttnCost* costs = COSTS[c.head_dim == 128 ? 1 : 0];
    struct Unit { int req, j0, nj, L, nb; int64_t bc; };   // the same for every kv head
    struct Layout {
        const AttnCost* ac = nullptr;
        std::vector<Unit> units;
        int slots = 0;             // CTAs
        int64_t n_units = 0, total = 0, longest = 0;
        int64_t limit = 0;         // of an item in equal parts; wrapped: of a CTA
        bool merge_counts = true;  // the merge of a unit's parts has to end by `limit` too
        bool wrapped = false;
        int64_t estimate = 0;
    };
    auto tiles = [&](const Unit& u) { return (u.nj * G + 15) / 16; };
    // equal parts that end by `limit`, where it counts with a merge of a few of them
    auto parts_of = [&](const Layout& y, const Unit& u, int64_t limit) {
        if (u.nb * u.bc + y.ac->item <= limit) return 1;
        const int min_blocks = y.ac->kind == ATTN_THIN ? 1 : 4, max_parts = y.ac->kind == ATTN_THIN ? ATTN_THIN_MAX_PARTS : 64;
        const int64_t tail = y.merge_counts ? y.ac->part + y.ac->merge + 4 * tiles(u) * y.ac->merge_tile : 0;
        const int64_t most = std::max<int64_t>(min_blocks, (limit - y.ac->item - tail) / u.bc);   // blocks of a part
        return (int)std::min<int64_t>(std::min<int64_t>(max_parts, std::max(1, u.nb / min_blocks)), (u.nb + most - 1) / most);
    };
    // The units one after the other, longest first, each CTA filled up to `limit`: what does not fit goes on in the next CTA
    // (so at most two partials a CTA).  emit(unit, head, first block, one past the last, cta); false if the CTAs do not suffice.
    auto wrap = [&](const Layout& y, int64_t limit, auto&& emit) {
        const AttnCost& k = *y.ac;
        const int min_blocks = 2, max_parts = k.kind == ATTN_THIN ? ATTN_THIN_MAX_PARTS : 64;
        int cta = 0;
        int64_t load = 0;
        for (const Unit& u : y.units)
            for (int h = 0; h < Hkv; ++h) {
                int at = 0, np = 0;
                while (at < u.nb) {
                    const int64_t room = limit - load - k.item;
                    const int left = u.nb - at;
                    int take = left * u.bc + (at ? k.part : 0) <= room ? left : (int)std::min<int64_t>(left - 1, (room - k.part) / u.bc);
                    if (take < left && (take < min_blocks || room < k.part)) take = 0;
                    if (take == 0 && load == 0) return false;
                    if (take) {
                        emit(u, h, at, at + take, cta);
                        load += take * u.bc + k.item + (take < u.nb ? k.part : 0);
                        at += take;
                        if (++np > max_parts) return false;
                    }
                    if (at < u.nb) {
                        load = 0;
                        if (++cta >= y.slots) return false;
                    }
                }
            }
        return true;
    };
    auto lay_out = [&](const AttnCost& k, int slots) {
        Layout y;
        y.ac = &k;
        y.slots = slots;
        const int tpg = k.kind == ATTN_TENSOR ? std::min(SYN_MAX_CHUNK, 128 / G) : std::min(16, 64 / G);
        y.units.reserve(n_req);
        for (int i = 0; i < n_req; ++i) {
            const int n = chunk_offsets[i + 1] - chunk_offsets[i];
            for (int j0 = 0; j0 < n; j0 += tpg) {
                const int nj = std::min(tpg, n - j0), L = ctx_lens[i] + j0 + nj, nb = (L + 63) / 64;
                y.units.push_back({i, j0, nj, L, nb, 0});
                const int64_t bc = y.units.back().bc = k.block[std::min(4, tiles(y.units.back()))];
                y.total += (nb * bc + k.item) * Hkv;
                y.longest = std::max(y.longest, nb * bc + k.item);
            }
        }
        y.n_units = (int64_t)y.units.size() * Hkv;
        const int64_t mean = (y.total + slots - 1) / slots;
        if (y.n_units > 2 * slots) {
            // Many units to a CTA: whole, unless one alone exceeds a CTA's fair share by so much that parts of it pay for
            // themselves.  The merge of a unit's parts runs beside other items and counts as work, not as time that a part has to
            // leave free (with the merge inside the share, three requests of 6 000 keys among 58 of the 8B shape were cut into
            // parts of 4 blocks: 528 parts and 520 us a layer; 96 and 58 with this).
            y.merge_counts = false;
            y.estimate = INT64_MAX;
            for (int64_t limit = std::max(mean, 8 * (int64_t)k.block[4] + k.item);; limit += limit / 4) {
                int64_t total = 0, longest = 0;
                for (const Unit& u : y.units) {
                    const int np = parts_of(y, u, limit);
                    total += u.nb * u.bc + k.item;
                    if (np > 1) total += (int64_t)np * (k.item + k.part) - k.item + k.merge + std::min(np, 8) * tiles(u) * k.merge_tile;
                    longest = std::max(longest, (u.nb + np - 1) / np * u.bc + k.item + (np > 1 ? k.part : 0));
                }
                const int64_t estimate = std::max((total * Hkv + slots - 1) / slots, longest) + k.fixed;
                if (estimate < y.estimate) { y.estimate = estimate; y.limit = limit; }
                if (limit >= y.longest) break;   // nothing is cut
            }
            return y;
        }
        // Few: whole units (as good as their number divides), equal parts of which there are no more than CTAs, or wrapped; with
        // two CTAs or more to a unit equal parts are as even and have fewer merges (64 units of the 8B shape on 296 CTAs: 29.5 us
        // wrapped, 28.8 in equal parts).
        int64_t best = y.n_units <= slots ? y.longest : std::max(y.longest, (y.n_units + slots - 1) / slots * (y.total / y.n_units));
        y.limit = y.longest;
        if (y.n_units <= slots) {
            auto fits = [&](int64_t lim) {
                int64_t n = 0;
                for (const Unit& u : y.units) n += (int64_t)parts_of(y, u, lim) * Hkv;
                return n <= slots;
            };
            int64_t lo = k.item, hi = y.longest;
            while (hi - lo > 256) {   // the number of parts falls with the limit; at `hi` nothing is cut
                const int64_t mid = (lo + hi) / 2;
                if (fits(mid)) hi = mid; else lo = mid;
            }
            int64_t part = 0;
            for (const Unit& u : y.units) {
                const int np = parts_of(y, u, hi);
                part = std::max(part, (u.nb + np - 1) / np * u.bc + k.item + (np > 1 ? k.part + k.merge + std::min(np, 8) * tiles(u) * k.merge_tile : 0));
            }
            if (part < best) {
                best = part;
                y.limit = hi;
            }
        }
        if (2 * y.n_units > slots) {
            std::sort(y.units.begin(), y.units.end(), [](const Unit& p, const Unit& q) {
                return p.nb * p.bc != q.nb * q.bc ? p.nb * p.bc > q.nb * q.bc : (p.req != q.req ? p.req < q.req : p.j0 < q.j0);
            });
            auto nothing = [](const Unit&, int, int, int, int) {};
            int64_t lo = mean, hi = mean + 2 * (k.item + k.part) + 2 * (int64_t)k.block[4];
            int64_t merge = 0;   // a cut unit has two or three parts
            for (const Unit& u : y.units) merge = std::max<int64_t>(merge, k.merge + 2 * tiles(u) * k.merge_tile);
            if (lo + merge < best && wrap(y, hi, nothing)) {
                while (hi - lo > 64 + mean / 64) {
                    const int64_t mid = (lo + hi) / 2;
                    if (wrap(y, mid, nothing)) hi = mid; else lo = mid;
                }
                if (hi + merge < best) { best = hi + merge; y.limit = hi; y.wrapped = true; }
            }
        }
        y.estimate = best + k.fixed;
        return y;
    };
    // Three kernels; the estimated time decides.  The tensor-memory one (row tiles of 128: the same time per block whatever the
    // number of rows; a chunk of more than 64 / G tokens is one item there and several items that each read the request's keys
    // in the others) is looked at if some chunk fills more than two row tiles of 16 (below, it was 2 to 12 us behind the better of
    // the others in every batch tried), and has to be 3 % better, 12 % where there are more than two units (request, token group, kv head) to an SM:
    // it draws more power, and under the power cap a step that uses it runs its other kernels at a lower clock (544 tokens of the
    // 8B shape: 109 us against 112 a layer, and the step takes as long).
    Layout lay;
    if (attention) {
        const int slots = attention == ATTN_THIN ? thin_ctas : n_sm;
        lay = lay_out(costs[attention - 1], slots);
    } else {
        // Whole units, one to an SM at most: left to the half-SM kernel, whose parts let the next projection in as they end.
        lay = lay_out(costs[0], n_sm);
        if (lay.n_units <= n_sm && !lay.wrapped) lay.estimate = INT64_MAX / 256;
        const int64_t lead = lay.n_units > 2 * n_sm ? 112 : 103;
        Layout other = lay_out(costs[2], thin_attention_ctas(n_sm));
        if (other.estimate < lay.estimate) lay = std::move(other);
        if (max_chunk * G > 32) {
            other = lay_out(costs[1], n_sm);
            if (other.estimate * lead < lay.estimate * 100) lay = std::move(other);
        }
        if (lay.ac->kind == ATTN_THIN && thin_ctas != lay.slots) lay = lay_out(costs[2], thin_ctas);
    }
    const int kind = lay.ac->kind;
    hp.kind = kind;
    // Positions that no chunk of the batch writes, for the kernel that requests keys before the chunks' are written: up
    // to the first page of the request that holds a written slot, of whichever request.
    std::vector<int> safe;
    if (kind == ATTN_THIN) {
        std::vector<uint8_t> written(n_pages, 0);
        for (int i = 0; i < n_req; ++i)
            for (int k = ctx_lens[i] / P; k <= (ctx_lens[i] + (chunk_offsets[i + 1] - chunk_offsets[i]) - 1) / P; ++k)
                written[page_tables[(size_t)i * max_pages + k]] = 1;
        safe.resize(n_req);
        for (int i = 0; i < n_req; ++i) {
            int k = 0;
            while (k < ctx_lens[i] / P && !written[page_tables[(size_t)i * max_pages + k]]) ++k;
            safe[i] = k * P;
        }
    }
    std::vector<AttnItem> items;
    std::vector<int> item_cost, owner;
    std::vector<MergeGroup>& groups = hp.groups;
    groups.clear();
    int n_parts = 0;
    auto add_item = [&](const Unit& u, int h, int b0, int b1) {
        const bool whole = b0 == 0 && b1 == u.nb;
        const int q_tok = chunk_offsets[u.req] + u.j0;
        if (!whole && b0 == 0) groups.push_back({q_tok, u.nj, h, n_parts, 0, 0, 0, 0});
        if (!whole) groups.back().n_parts++;
        items.push_back({q_tok, u.nj, h, u.req, b0 * 64, std::min(u.L, b1 * 64), ctx_lens[u.req] + u.j0, whole ? -1 : n_parts++,
                         whole ? -1 : (int)groups.size() - 1, kind == ATTN_THIN ? safe[u.req] : 0, 0, 0});
        item_cost.push_back((int)((b1 - b0) * u.bc) + lay.ac->item + (whole ? 0 : lay.ac->part));
    };
    if (lay.wrapped) {
        wrap(lay, lay.limit, [&](const Unit& u, int h, int b0, int b1, int cta) {
            add_item(u, h, b0, b1);
            owner.push_back(cta);
        });
    } else {
        for (const Unit& u : lay.units) {
            const int np = parts_of(lay, u, lay.limit);
            for (int h = 0; h < Hkv; ++h)
                for (int k = 0; k < np; ++k) add_item(u, h, (int)((int64_t)k * u.nb / np), (int)((int64_t)(k + 1) * u.nb / np));
        }
    }
    const int n_items = (int)items.size();
    const int n_cta = lay.wrapped ? owner.back() + 1 : std::min(lay.slots, n_items);
    std::vector<int> order(n_items);
    for (int i = 0; i < n_items; ++i) order[i] = i;
    std::vector<int>& count = hp.cta_begin;
    count.assign(n_cta + 1, 0);
    auto cost = [&](int i) { return item_cost[i]; };
    if (lay.wrapped) {
        for (int k : owner) count[k + 1]++;
    } else {
        // longest first (equal costs: lower index first), each to the least loaded CTA (ties: lower CTA);
        // both orders are carried in one 64-bit key
        owner.assign(n_items, 0);
        {
            // stable radix sort of the indices by decreasing cost, 11 bits a pass
            int top = 0;
            for (int i = 0; i < n_items; ++i) top = std::max(top, item_cost[i]);
            std::vector<int> tmp(n_items);
            int hist[2048];
            for (int shift = 0; shift < 32 && (top >> shift) != 0; shift += 11) {
                memset(hist, 0, sizeof(hist));
                for (int i = 0; i < n_items; ++i) hist[2047 - ((item_cost[order[i]] >> shift) & 2047)]++;
                int run = 0;
                for (int b = 0; b < 2048; ++b) { const int h = hist[b]; hist[b] = run; run += h; }
                for (int i = 0; i < n_items; ++i) tmp[hist[2047 - ((item_cost[order[i]] >> shift) & 2047)]++] = order[i];
                order.swap(tmp);
            }
        }
        {
            std::vector<uint64_t> heap(n_cta);   // (load << 16) | cta, smallest at the root
            for (int k = 0; k < n_cta; ++k) heap[k] = (uint64_t)k;   // all loads 0: already a heap
            for (int i : order) {
                const uint64_t top = heap[0];
                const int k = (int)(top & 0xFFFFu);
                owner[i] = k;
                count[k + 1]++;
                const uint64_t v = (((top >> 16) + (uint64_t)cost(i)) << 16) | (uint64_t)k;
                int at = 0;   // the root grows: sift it down
                for (;;) {
                    int ch = 2 * at + 1;
                    if (ch >= n_cta) break;
                    if (ch + 1 < n_cta && heap[ch + 1] < heap[ch]) ++ch;
                    if (heap[ch] >= v) break;
                    heap[at] = heap[ch];
                    at = ch;
                }
                heap[at] = v;
            }
        }
        // Local search on the greedy result: relieve the most loaded CTA by moving one of its items to
        // another CTA, or by exchanging it for a cheaper one, as long as that lowers the larger of the
        // two loads; partners are the least loaded CTAs.  Only when CTAs hold more than one item and the greedy result is more
        // than 1 % above the mean; stops within 0.3 % of it.
        if (n_cta < n_items) {
            std::vector<int64_t> load(n_cta, 0);
            int64_t sum = 0;
            for (int i = 0; i < n_items; ++i) {
                load[owner[i]] += cost(i);
                sum += cost(i);
            }
            const int64_t mean = sum / n_cta;
            if (*std::max_element(load.begin(), load.end()) > mean + mean / 100) {
                std::vector<std::vector<int>> held(n_cta);
                for (int i = 0; i < n_items; ++i) held[owner[i]].push_back(i);
                std::vector<int> by_load(n_cta);   // CTAs by increasing load, kept sorted
                for (int k = 0; k < n_cta; ++k) by_load[k] = k;
                auto lighter = [&](int x, int y) { return load[x] != load[y] ? load[x] < load[y] : x < y; };
                std::sort(by_load.begin(), by_load.end(), lighter);
                auto resort = [&](int k) {   // k's load changed: move it to its place
                    int at = (int)(std::find(by_load.begin(), by_load.end(), k) - by_load.begin());
                    while (at + 1 < n_cta && lighter(by_load[at + 1], k)) { by_load[at] = by_load[at + 1]; ++at; }
                    while (at > 0 && lighter(k, by_load[at - 1])) { by_load[at] = by_load[at - 1]; --at; }
                    by_load[at] = k;
                };
                const int64_t good = mean + mean / 333;
                const int n_cand = std::min(n_cta - 1, 16);
                for (int round = 0; round < 128; ++round) {
                    const int hi = by_load[n_cta - 1];
                    if (load[hi] <= good) break;
                    int64_t best = load[hi];
                    int bi = -1, bk = -1, bj = -1;   // position in held[hi], the other CTA, position in held[bk] (-1: move)
                    for (int a = 0; a < (int)held[hi].size(); ++a) {
                        const int64_t ca = cost(held[hi][a]);
                        for (int q = 0; q < n_cand; ++q) {
                            const int k = by_load[q];
                            if (std::max(load[hi] - ca, load[k] + ca) < best) {
                                best = std::max(load[hi] - ca, load[k] + ca);
                                bi = a; bk = k; bj = -1;
                            }
                            for (int b2 = 0; b2 < (int)held[k].size(); ++b2) {
                                const int64_t dlt = ca - cost(held[k][b2]);
                                if (dlt > 0 && std::max(load[hi] - dlt, load[k] + dlt) < best) {
                                    best = std::max(load[hi] - dlt, load[k] + dlt);
                                    bi = a; bk = k; bj = b2;
                                }
                            }
                        }
                    }
                    if (bi < 0 || load[hi] - best < mean / 1000) break;   // nothing, or next to nothing, to gain
                    const int ia = held[hi][bi];
                    if (bj < 0) {
                        load[hi] -= cost(ia); load[bk] += cost(ia);
                        owner[ia] = bk;
                        held[bk].push_back(ia);
                        held[hi].erase(held[hi].begin() + bi);
                    } else {
                        const int ib = held[bk][bj];
                        const int64_t dlt = cost(ia) - cost(ib);
                        load[hi] -= dlt; load[bk] += dlt;
                        owner[ia] = bk; owner[ib] = hi;
                        held[hi][bi] = ib; held[bk][bj] = ia;
                    }
                    resort(hi);
                    resort(bk);
                }
                std::fill(count.begin(), count.end(), 0);
                for (int i = 0; i < n_items; ++i) count[owner[i] + 1]++;
            }
        }
    }
    for (int k = 0; k < n_cta; ++k) count[k + 1] += count[k];
    hp.items.assign(n_items, AttnItem());
    {
        std::vector<int> cur(count.begin(), count.end() - 1);
        for (int i : order) hp.items[cur[owner[i]]++] = items[i];
    }
    hp.T = T; hp.n_cta = n_cta; hp.n_parts = n_parts;

    syn_step_stats& s = hp.stats;
    memset(&s, 0, sizeof(s));
    const double d = c.d_model, qd = (double)c.n_q_heads * c.head_dim, kd = (double)Hkv * c.head_dim;
    const double params = c.n_layers * (d * (qd + 2 * kd) + qd * d + 3.0 * d * c.d_ffn) + d * c.vocab;
    s.n_req = n_req; s.n_tokens = T; s.ctx_tokens = ctx_sum;
    s.weight_bytes = (int64_t)(params * 2);
    s.kv_read_bytes = kv_units * (int64_t)(2 * kd * 2) * c.n_layers;
    s.kv_write_bytes = (int64_t)T * (int64_t)(2 * kd * 2) * c.n_layers;
    s.dense_flops = 2.0 * T * params;
    s.attn_flops = 4.0 * qd * c.n_layers * (double)keys_seen;
    s.attn_items = n_items; s.attn_split_items = n_parts;
    s.kernel_launches = 1 + c.n_layers * 5 + 2;
    s.attn_rows = attn_rows(kind);
    return SYN_OK;
}

// plan_compute, then pack everything into the plan's pinned buffer (grown on demand).
static int plan_build(syn_plan* p, syn_model* m, syn_kv* kv, int32_t n_req, const int32_t* chunk_tokens,
                      const int32_t* chunk_offsets, const int32_t* page_tables, int32_t max_pages, const int32_t* ctx_lens,
                      const int32_t* n_uncached) {
    if (!m || !kv || kv->model != m) return SYN_E_INVALID_ARG;
    HostPlan hp;
    int r = plan_compute(m->desc, (int)kv->page_size, kv->n_pages, m->n_sm, n_req, chunk_tokens, chunk_offsets, page_tables,
                         max_pages, ctx_lens, n_uncached, g_attention, thin_attention_ctas(m->n_sm), hp);
    if (r) return r;
    const int T = hp.T, n_items = (int)hp.items.size(), n_cta = hp.n_cta;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
    p->o_tokens = take((size_t)T * 4);
    p->o_pos = take((size_t)T * 4);
    p->o_slot = take((size_t)T * 4);
    p->o_offsets = take((size_t)(n_req + 1) * 4);
    p->o_uncached = take((size_t)n_req * 4);
    p->o_tables = take((size_t)n_req * max_pages * 4);
    p->o_row = take((size_t)T * 4);
    p->o_first = take((size_t)n_req * 4);
    p->o_items = take((size_t)n_items * sizeof(AttnItem));
    p->o_cta = take((size_t)(n_cta + 1) * 4);
    p->o_groups = take(std::max<size_t>(1, hp.groups.size()) * sizeof(MergeGroup));
    if (off > p->cap) {
        cudaFree(p->dev);
        if (p->host) cudaFreeHost(p->host);
        p->dev = p->host = nullptr;
        p->cap = 0;
        const size_t cap = align_up(off + off / 2, 4096);
        CU_OK(cudaMalloc(&p->dev, cap));
        CU_OK(cudaMallocHost(&p->host, cap));
        p->cap = cap;
    }
    p->used = off;
    memcpy(p->h<int>(p->o_tokens), chunk_tokens, (size_t)T * 4);
    memcpy(p->h<int>(p->o_pos), hp.pos.data(), (size_t)T * 4);
    memcpy(p->h<int>(p->o_slot), hp.slot.data(), (size_t)T * 4);
    memcpy(p->h<int>(p->o_offsets), chunk_offsets, (size_t)(n_req + 1) * 4);
    p->n_judging = 0;
    for (int i = 0; i < n_req; ++i) {
        const int u = n_uncached ? n_uncached[i] : 1;
        p->h<int>(p->o_uncached)[i] = u;
        p->h<int>(p->o_first)[i] = p->n_judging;
        for (int t = chunk_offsets[i] + u - 1; t < chunk_offsets[i + 1]; ++t) p->h<int>(p->o_row)[p->n_judging++] = t;
    }
    memcpy(p->h<int>(p->o_tables), page_tables, (size_t)n_req * max_pages * 4);
    memcpy(p->h<AttnItem>(p->o_items), hp.items.data(), (size_t)n_items * sizeof(AttnItem));
    memcpy(p->h<int>(p->o_cta), hp.cta_begin.data(), (size_t)(n_cta + 1) * 4);
    if (!hp.groups.empty()) memcpy(p->h<MergeGroup>(p->o_groups), hp.groups.data(), hp.groups.size() * sizeof(MergeGroup));
    p->n_req = n_req; p->T = T; p->max_pages = max_pages; p->n_items = n_items; p->n_cta = n_cta;
    p->n_groups = (int)hp.groups.size(); p->n_parts = hp.n_parts;
    p->attn = hp.kind;
    p->stats = hp.stats;
    p->stats.h2d_bytes = (int64_t)off;
    p->kv = kv; p->kv_pool = kv->pool; p->kv_pages = kv->n_pages;
    return SYN_OK;
}

// The planner without a device, for `thin_ctas` CTAs of the half-SM attention kernel; the work list goes to caller-provided HOST
// arrays, `fields` ints an item.
static int plan_host(const syn_model_desc* desc, uint32_t n_pages, uint32_t page_size, int32_t n_sm, int thin_ctas, int32_t n_req,
                     const int32_t* chunk_tokens, const int32_t* chunk_offsets, const int32_t* page_tables, int32_t max_pages,
                     const int32_t* ctx_lens, const int32_t* n_uncached, int32_t* items, int32_t items_cap, int fields,
                     int32_t* n_items, int32_t* cta_begin, int32_t* n_cta, HostPlan& hp) {
    if (!desc || page_size != 16 || !n_items || !n_cta) return SYN_E_INVALID_ARG;
    if (desc->n_kv_heads == 0 || desc->n_q_heads % desc->n_kv_heads != 0 || desc->n_q_heads / desc->n_kv_heads > 8)
        return SYN_E_INVALID_ARG;
    int r = plan_compute(*desc, (int)page_size, n_pages, n_sm, n_req, chunk_tokens, chunk_offsets, page_tables, max_pages,
                         ctx_lens, n_uncached, g_attention, thin_ctas, hp);
    if (r) return r;
    *n_items = (int)hp.items.size();
    *n_cta = hp.n_cta;
    if (items) {
        if (items_cap < *n_items) return SYN_E_CAPACITY;
        for (int i = 0; i < *n_items; ++i) {
            const AttnItem& it = hp.items[i];
            const int32_t row[SYN_WORK_ITEM_FIELDS] = {it.q_tok, it.nj, it.kvh, it.req, it.kv_begin, it.kv_end, it.q_pos0,
                                                       it.part, it.grp, it.kv_safe};
            memcpy(items + (size_t)i * fields, row, fields * sizeof(int32_t));
        }
    }
    if (cta_begin) memcpy(cta_begin, hp.cta_begin.data(), (size_t)(hp.n_cta + 1) * 4);
    return SYN_OK;
}

static int syn_plan_host_impl(const syn_model_desc* desc, uint32_t n_pages, uint32_t page_size, int32_t n_sm, int32_t n_req,
                             const int32_t* chunk_tokens, const int32_t* chunk_offsets, const int32_t* page_tables,
                             int32_t max_pages, const int32_t* ctx_lens, const int32_t* n_uncached, int32_t* pos,
                             int32_t* slot, int32_t* items, int32_t items_cap, int32_t* n_items, int32_t* cta_begin,
                             int32_t* n_cta, syn_step_stats* stats) {
    HostPlan hp;
    // n_sm CTAs whatever the kernel: callers pass a cta_begin of that size
    const int r = plan_host(desc, n_pages, page_size, n_sm, n_sm, n_req, chunk_tokens, chunk_offsets, page_tables, max_pages, ctx_lens,
                            n_uncached, items, items_cap, SYN_PLAN_ITEM_FIELDS, n_items, cta_begin, n_cta, hp);
    if (r && r != SYN_E_CAPACITY) return r;
    if (pos) memcpy(pos, hp.pos.data(), hp.pos.size() * 4);
    if (slot) memcpy(slot, hp.slot.data(), hp.slot.size() * 4);
    if (r) return r;
    if (stats) *stats = hp.stats;
    return SYN_OK;
}

static int syn_plan_work_host_impl(const syn_model_desc* desc, uint32_t n_pages, uint32_t page_size, int32_t n_sm, int32_t n_req,
                                   const int32_t* chunk_tokens, const int32_t* chunk_offsets, const int32_t* page_tables,
                                   int32_t max_pages, const int32_t* ctx_lens, const int32_t* n_uncached, int32_t* items,
                                   int32_t items_cap, int32_t* n_items, int32_t* cta_begin, int32_t* n_cta, int32_t* attention,
                                   syn_step_stats* stats) {
    if (n_sm <= 0 || n_sm > 32767) return SYN_E_INVALID_ARG;
    HostPlan hp;
    const int r = plan_host(desc, n_pages, page_size, n_sm, thin_attention_ctas(n_sm), n_req, chunk_tokens, chunk_offsets, page_tables,
                            max_pages, ctx_lens, n_uncached, items, items_cap, SYN_WORK_ITEM_FIELDS, n_items, cta_begin, n_cta, hp);
    if (r) return r;
    if (attention) *attention = hp.kind;
    if (stats) *stats = hp.stats;
    return SYN_OK;
}

static int syn_plan_create_impl(syn_model* m, syn_kv* kv, int32_t n_req, const int32_t* chunk_tokens,
                               const int32_t* chunk_offsets, const int32_t* page_tables, int32_t max_pages,
                               const int32_t* ctx_lens, const int32_t* n_uncached, syn_plan** out) {
    if (!out) return SYN_E_INVALID_ARG;
    syn_plan* p = new (std::nothrow) syn_plan();
    if (!p) return SYN_E_OOM;
    int r = plan_build(p, m, kv, n_req, chunk_tokens, chunk_offsets, page_tables, max_pages, ctx_lens, n_uncached);
    if (r == SYN_OK) {
        cudaError_t e = cudaMemcpy(p->dev, p->host, p->used, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) r = SYN_E_CUDA;
    }
    if (r == SYN_OK) r = ensure_workspace(m, p->T, p->n_parts);
    if (r != SYN_OK) {
        syn_plan_free(p);
        return r;
    }
    *out = p;
    return SYN_OK;
}

extern "C" int syn_plan_attention(const syn_plan* p) { return p ? p->attn : SYN_E_INVALID_ARG; }

extern "C" int syn_plan_stats(const syn_plan* p, syn_step_stats* out) {
    if (!p || !out) return SYN_E_INVALID_ARG;
    *out = p->stats;
    return SYN_OK;
}

extern "C" int syn_last_step_stats(syn_model* m, syn_step_stats* out) {
    if (!m || !out || !m->have_last) return SYN_E_INVALID_ARG;
    *out = m->last_stats;
    if (m->step_timed) {
        float ms = 0.f;
        CU_OK(cudaEventSynchronize(m->step_b));
        CU_OK(cudaEventElapsedTime(&ms, m->step_a, m->step_b));
        out->t_gpu_ms = ms;
        out->t_wall_ms = m->last_wall_ms;
    }
    return SYN_OK;
}

// A plan's page ids and KV slots were checked against one cache: only that cache may run it.
static bool plan_matches(const syn_plan* p, const syn_kv* kv) {
    return p->kv == kv && p->kv_pool == kv->pool && p->kv_pages == kv->n_pages;
}

// ------------------------------------------------------------------------------------------ launches

// The launch shape of one projection D[rows][T] = Wpacked[rows][K] * X[T][K]^T: token tiling, work
// decomposition, CTA count.  Host arithmetic only (also exported as syn_gemm_plan_host so that the
// schedule can be checked without a device).  `mode` = the epilogue the schedule is made for.
static int gemm_plan(int T, int packed_rows, int K, int n_sm, int mode, bool may_ksplit, GemmParams& g, int& n_cta) {
    g.num_kb = (K + 63) / 64;
    g.n_pairs = (packed_rows + 255) / 256;
    g.n_tt = (T + 255) / 256;
    // A projection with fewer pair tiles than SMs can share a tile's K range between CTAs (reduce-
    // scatter, GEMM_RSPLIT): always for the residual projections, whose K is long and whose output is
    // narrow; for qkv from a few hundred tokens on, where single 128-feature tiles would ask L2 for
    // the token tile twice as often; parts of at least 4 (residual) or 8 (qkv) k-blocks.
    const int tiles_nat = g.n_pairs * g.n_tt;
    const bool qkv_split = mode == EPI_QKV && T >= 256 && n_sm / tiles_nat >= 2 && g.num_kb >= 16;
    if (mode != EPI_RESID) {
        // Few feature tiles and few tokens: narrower token tiles (32 tokens at least) put more SMs to
        // work; the weights are then read by several CTAs, which costs only L2 bandwidth.
        const int want = n_sm / std::max(1, 2 * g.n_pairs), most = (T + 31) / 32;
        if (!qkv_split) g.n_tt = std::max(g.n_tt, std::min(want, most));
    } else if (g.n_pairs * g.n_tt < n_sm && n_sm / (g.n_pairs * g.n_tt) < 2) {
        // Residual projection whose pair tiles cover more than half of the SMs but not all: K cannot be
        // split, so narrower token tiles (64 tokens at least) fill the machine instead; every CTA still
        // walks the whole K, on a smaller item.
        const int fit = n_sm / g.n_pairs, most = (T + 63) / 64;
        g.n_tt = std::max(g.n_tt, std::min(fit, most));
    }
    g.TN = (((T + g.n_tt - 1) / g.n_tt) + 15) / 16 * 16;
    g.n_tt = (T + g.TN - 1) / g.TN;   // rounding the width up may leave the last tiles without tokens
    g.n_stages = gemm_stages(g.TN);
    g.ksplit = 1; g.kper = 0; g.n_sm = n_sm;
    g.splits = 1;
    g.kb_per_split = g.num_kb;
    // every token tile must hold a token: an empty one would issue an MMA of width 0
    if (g.n_stages < 2 || g.TN < 16 || g.TN > 256 || (g.n_tt - 1) * g.TN >= T) return SYN_E_INVALID_ARG;
    const int tiles = g.n_pairs * g.n_tt;
    g.pair_mode = tiles >= n_sm;
    if ((mode == EPI_RESID || qkv_split) && tiles < n_sm) {
        const int min_kb = mode == EPI_RESID ? 4 : 8;
        int sp = std::min(GEMM_MAX_SPLITS, std::min(n_sm / tiles, std::max(1, g.num_kb / min_kb)));
        g.kb_per_split = (g.num_kb + sp - 1) / sp;
        g.splits = (g.num_kb + g.kb_per_split - 1) / g.kb_per_split;
        g.pair_mode = 1;
    }
    if (g.splits > 1) n_cta = tiles * g.splits;
    else n_cta = std::min(n_sm, g.pair_mode ? tiles : 2 * tiles);
    // fewer pair tiles than SMs but more single tiles: one wave that mixes whole pair tiles and single tiles
    // (two waves of single tiles would take longer than one pair tile)
    if (g.splits == 1 && !g.pair_mode && 2 * tiles > n_sm) g.pair_mode = 2;
    if (g.splits == 1 && g.pair_mode == 1 && may_ksplit) {
        // The tiles left after the full waves: cut along K over otherwise idle CTAs (parts of at
        // least 8 k-blocks; helpers and owners are different CTAs, so R * parts <= n_cta).
        const int rem = tiles % n_cta;
        if (rem > 0) {
            const int parts = std::min(std::min(8, n_cta / rem), g.num_kb / 8);
            if (parts >= 2) {
                // the owner part also adds the others and finishes the tile: about half a helper's k range
                const int H = parts - 1;
                int kper = (2 * g.num_kb + 2 * H) / (2 * H + 1);
                while (H * kper >= g.num_kb) --kper;
                g.ksplit = parts;
                g.kper = kper;
            }
        }
    }
    return SYN_OK;
}

// The instance of a projection kernel for the epilogue `mode`.
#define EPI_SWITCH(mode, call)                                           \
    switch (mode) {                                                      \
        case EPI_QKV: { constexpr int MODE = EPI_QKV; call; break; }       \
        case EPI_RESID: { constexpr int MODE = EPI_RESID; call; break; }   \
        case EPI_SWIGLU: { constexpr int MODE = EPI_SWIGLU; call; break; } \
        case EPI_LMHEAD: { constexpr int MODE = EPI_LMHEAD; call; break; } \
        default: { constexpr int MODE = EPI_PLAIN; call; break; }          \
    }

template <int VARIANT, int MODE>
static cudaError_t launch_gemm_variant(const GemmParams& g, int n_cta, const CUtensorMap& tmB, const EpiParams& ep, cudaStream_t st) {
    const int smem = gemm_fixed_smem(g.TN) + g.n_stages * gemm_stage_bytes(g.TN);
    if constexpr (gemm_variant_used(VARIANT, MODE)) return launch_pdl(gemm_kernel<VARIANT, MODE>, dim3(n_cta), dim3(gemm_threads(MODE)), smem, st, tmB, g, ep);
    else return note_cuda(cudaErrorInvalidDeviceFunction);
}
template <int MODE>
static cudaError_t launch_gemm_mode(const GemmParams& g, int n_cta, const CUtensorMap& tmB, const EpiParams& ep, cudaStream_t st) {
    return g.splits > 1 ? launch_gemm_variant<GEMM_RSPLIT, MODE>(g, n_cta, tmB, ep, st)
           : g.ksplit > 1 ? launch_gemm_variant<GEMM_KSPLIT, MODE>(g, n_cta, tmB, ep, st)
                          : launch_gemm_variant<GEMM_WAVES, MODE>(g, n_cta, tmB, ep, st);
}

// One projection with the epilogue `ep`; `plan_mode` = the epilogue its schedule is made for (the
// same, except in the test hook, which runs any schedule with the plain store epilogue).
static int launch_gemm(syn_model* prof_m, int cls, int n_sm, int* status, const op16* w_packed, int packed_rows, int K,
                       const CUtensorMap& tmB, const EpiParams& ep, cudaStream_t st, float* fix_part, int* fix_flag,
                       int plan_mode) {
    ProfScope prof(cls >= 0 ? prof_m : nullptr, cls, st);
    GemmParams g;
    memset(&g, 0, sizeof(g));
    int n_cta = 0;
    if (!fix_part || !fix_flag) return SYN_E_INVALID_ARG;
    const int pr = gemm_plan(ep.T, packed_rows, K, n_sm, plan_mode, plan_mode != EPI_RESID, g, n_cta);
    if (pr) return pr;
    g.w = w_packed;
    g.status = status;
    g.fix_part = fix_part; g.fix_flag = fix_flag;
    g.spin_limit = g_spin_limit;
    cudaError_t le;
    EPI_SWITCH(ep.mode, le = launch_gemm_mode<MODE>(g, n_cta, tmB, ep, st));
    return le == cudaSuccess ? SYN_OK : SYN_E_CUDA;
}

// Schedules of the CTA-pair kernel (gemm2.cuh).
enum { PAIR_NONE = 0, PAIR_QUAD = 1, PAIR_DUO = 2 };

// Estimated time, in SM cycles, of a projection on the one-CTA kernel (kind PAIR_NONE) or on CTA pairs: the work of its first
// and of its last CTA or cluster, whichever is more.  An item costs its k-blocks times the larger of its tensor-core
// cycles and of its operands at 57 bytes a cycle and SM from L2, its epilogue per output element, the accumulators it
// stores and reads of others, and a fixed part; the coefficients are a least-squares fit to 540 event times (264 to 2 048 tokens,
// all projections of the 1B, 8B and 32B shapes, three kernels; rms error 5, 5 and 9 %).
static int gemm2_plan(int T, int packed_rows, int K, int n_sm, int mode, int force, Gemm2Params& g, int& n_cl);
static double proj_cost(int T, int packed_rows, int K, int n_sm, int mode, int kind) {
    struct Fit { double main, epi[5], exch, item, fixed; };   // epi: PLAIN, QKV, RESID, SWIGLU, LMHEAD
    static const Fit QUAD = {1.292, {0.07, 0.302, 0.190, 0.073, 0.283}, 0.302, -1650, 21300}, DUO = {1.152, {0.0, 0.302, 0.057, -0.093, 0.165}, 0.369, 5080, 20200},
                     ONE = {1.138, {0.09, 0.362, 0.213, 0.086, 0.319}, 0.276, -2420, 20400};
    const Fit& f = kind == PAIR_QUAD ? QUAD : (kind == PAIR_DUO ? DUO : ONE);
    auto width = [&](int TN, int tt) { return (double)((std::min(TN, T - tt * TN) + 15) / 16 * 16); };
    auto item = [&](int kb, int mt, double n, double mma, double bytes, double epi_share, double exch) {
        return f.main * kb * std::max(mma, bytes / 57.0) + 128.0 * mt * n * (f.epi[mode] * epi_share + f.exch * exch) + f.item;
    };
    double worst = 0.0;
    if (kind == PAIR_NONE) {
        GemmParams g;
        memset(&g, 0, sizeof(g));
        int n_cta = 0;
        if (gemm_plan(T, packed_rows, K, n_sm, mode, mode != EPI_RESID, g, n_cta)) return 1e30;
        for (int cta : {0, n_cta - 1}) {
            double sum = f.fixed;
            GemmWork w;
            for (int i = 0; g.ksplit > 1 ? gemm_work<true>(g, cta, n_cta, i, w) : gemm_work<false>(g, cta, n_cta, i, w); ++i) {
                const int mt = w.mt_hi - w.mt_lo, S = g.splits;
                const double n = width(g.TN, w.tt);
                const double share = w.role == 1 ? 0.0 : 1.0 / S;
                const double exch = w.role == 1 ? 1.0 : (w.role == 2 ? g.ksplit - 1.0 : 2.0 * (S - 1) / S);
                sum += item(w.kb1 - w.kb0, mt, n, mt == 2 ? 4 * n : 576.0, 16384.0 * mt + 128 * n, share, exch);   // one accumulator: 144 cycles an MMA
            }
            worst = std::max(worst, sum);
        }
        return worst;
    }
    Gemm2Params g;
    int n_cl = 0;
    if (gemm2_plan(T, packed_rows, K, n_sm, mode, kind, g, n_cl) != kind) return 1e30;
    const int mt = kind == PAIR_QUAD ? 2 : 1;
    for (int cl : {0, n_cl - 1}) {
        double sum = f.fixed;
        Gemm2Work w;
        for (int i = 0; gemm2_work(g, cl, n_cl, i, w); ++i) {
            const double n = width(g.TN, w.tt);
            sum += item(w.kb1 - w.kb0, mt, n, 2 * n * mt, 16384.0 * mt + 64 * n, 1.0 / w.nsplit, 2.0 * (w.nsplit - 1) / w.nsplit);
        }
        worst = std::max(worst, sum);
    }
    // 256-feature items left after the full waves and cut along K: 84 of them between 264 and 2 040 tokens took 1.09 times the
    // estimate, up to 1.25 (qkv of the 32B shape at 544 tokens: 61 us estimated, 71 measured, 62 on the one-CTA kernel)
    return kind == PAIR_DUO && g.rem_base > 1 ? 1.15 * worst : worst;
}

// Launch shape of a projection on CTA pairs, or PAIR_NONE when the one-CTA kernel serves it better
// (few tokens: the pair kernel's token tiles are the natural 256-token cut, it has no narrow tiles).
// Host arithmetic only.  `force`: PAIR_QUAD / PAIR_DUO to take that item shape regardless (test hook).
static int gemm2_plan_by_rule(int T, int packed_rows, int K, int n_sm, int mode, int force, Gemm2Params& g, int& n_cl) {
    memset(&g, 0, sizeof(g));
    const int n_pairs = (packed_rows + 255) / 256, n_cl_max = n_sm / 2;
    g.num_kb = (K + 63) / 64;
    g.n_tt = (T + 255) / 256;
    g.TN = (((T + g.n_tt - 1) / g.n_tt) + 15) / 16 * 16;
    g.n_tt = (T + g.TN - 1) / g.TN;
    g.splits = 1; g.kb_per_split = g.num_kb; g.n_sm = n_sm;
    if (n_cl_max < 1 || (force == PAIR_NONE && T < 256)) return PAIR_NONE;
    const int quad_items = (n_pairs + 1) / 2 * g.n_tt, duo_items = n_pairs * g.n_tt;
    int kind = force;
    const bool may_split = mode == EPI_RESID;
    if (kind == PAIR_NONE) {
        if (quad_items >= n_cl_max) kind = PAIR_QUAD;                                   // full waves of 512-feature items
        else if (4 * quad_items >= 3 * n_cl_max) kind = PAIR_QUAD;                      // one wave, at least three quarters full: measured
                                                                                        // 7-9 % ahead of 256-feature items in two rounds
        else if (!may_split && 8 * quad_items >= 5 * n_cl_max) kind = PAIR_QUAD;        // (without a residual epilogue already from five
                                                                                        // eighths: qkv at 921 tokens 94 us against 102)
        else if (may_split && g.num_kb >= 96 && n_cl_max / quad_items >= 2) kind = PAIR_QUAD;   // long K: shared between clusters
        else if (2 * duo_items >= n_cl_max) kind = PAIR_DUO;
        else return PAIR_NONE;
    }
    const int items = kind == PAIR_QUAD ? quad_items : duo_items;
    g.n_groups = kind == PAIR_QUAD ? (n_pairs + 1) / 2 : n_pairs;
    if (may_split && items < n_cl_max && n_cl_max / items >= 2) {
        const int sp = std::min(GEMM_MAX_SPLITS, std::min(n_cl_max / items, std::max(1, g.num_kb / 8)));
        g.kb_per_split = (g.num_kb + sp - 1) / sp;
        g.splits = (g.num_kb + g.kb_per_split - 1) / g.kb_per_split;
    }
    n_cl = g.splits > 1 ? items * g.splits : std::min(n_cl_max, items);
    // Fewer than three full waves and a last round that fills less than half of the clusters: the one-CTA kernel,
    // whose leftover tiles cost less (helper parts first, short owner parts last), is the faster one there
    // (gate/up at 544 tokens: 168 items on 74 clusters, 2.27 waves: 130 us here against 118 us).
    if (force == PAIR_NONE && g.splits == 1 && items > n_cl && items / n_cl < 3 && items % n_cl != 0 && 2 * (items % n_cl) < n_cl)
        return PAIR_NONE;
    if (g.splits == 1 && items > n_cl) {
        // items left after the full waves: cut along K into one part per cluster (parts of at least 8 k-blocks,
        // at most GEMM_MAX_SPLITS of them), so that the last round takes a fraction of an item's time.  (Helper
        // parts that run first and an owner part that runs last, as in the one-CTA kernel, measured slower here:
        // gate/up 138 against 130 us at 544 tokens, 241 against 201 us at 921: the owner adds up to seven stored
        // parts alone, where the reduce-scatter shares that work between all the tile's clusters.)
        const int rem = items % n_cl;
        if (rem > 0 && n_cl / rem >= 2) {
            int base = n_cl / rem, extra = n_cl % rem;
            const int most = std::min(GEMM_MAX_SPLITS, g.num_kb / 8);
            if (base + (extra > 0 ? 1 : 0) > most) { base = most; extra = 0; }
            if (base >= 2) { g.rem_base = base; g.rem_extra = extra; }
        }
    }
    g.n_stages = gemm2_stages(g.TN, kind == PAIR_DUO);
    if (g.n_stages < 2 || g.TN < 16 || g.TN > 256 || (g.n_tt - 1) * g.TN >= T) return PAIR_NONE;
    return kind;
}

// The rule above, unless another kernel is estimated at least 8 % faster.  Measured at 28 sizes of 264 to 2 040 tokens, the
// projections of a layer of the three shapes, all three kernels (316 points): the choice costs 1.4 % more time than the best
// kernel everywhere would, the rule alone 4.3 %; at worst 29 and 92 % (the 32B o at 1 536 tokens, 88 us on the rule's 512-feature
// items against 69 on the one-CTA kernel; the 32B down at 2 040, 849 us on the one-CTA kernel against 442).  It is never more
// than 3 % behind the rule.  Gate/up of the 8B shape at 688 to 768 tokens stays on the one-CTA kernel by the 8 % (158 us
// against 130).
static int gemm2_plan(int T, int packed_rows, int K, int n_sm, int mode, int force, Gemm2Params& g, int& n_cl) {
    const int by_rule = gemm2_plan_by_rule(T, packed_rows, K, n_sm, mode, force, g, n_cl);
    if (force != PAIR_NONE || T < 256 || n_sm < 2) return by_rule;
    int best = by_rule;
    double limit = proj_cost(T, packed_rows, K, n_sm, mode, by_rule) / 1.08;
    for (int kind : {PAIR_NONE, PAIR_QUAD, PAIR_DUO}) {
        const double c = kind == by_rule ? limit : proj_cost(T, packed_rows, K, n_sm, mode, kind);
        if (c < limit) { best = kind; limit = c; }
    }
    if (best == by_rule || best == PAIR_NONE) return best;
    return gemm2_plan_by_rule(T, packed_rows, K, n_sm, mode, best, g, n_cl);
}

constexpr int THIN_MAX_TOKENS = 512, THIN_MAX_TOKENS_QKV = 1024;

// Launch shape of a projection on the thin kernel (gemm_thin.cuh): at most one CTA per SM where K is shared, so that the
// other half of every SM is free for the next kernel, but for the case below; at least two k-blocks each.
static void thin_plan(int T, int packed_rows, int K, int n_sm, ThinParams& g) {
    memset(&g, 0, sizeof(g));
    g.num_kb = (K + 63) / 64;
    g.n_tiles = (packed_rows + 127) / 128;
    g.n_tt = (T + THIN_MAX_TN - 1) / THIN_MAX_TN;
    g.TN = ((T + g.n_tt - 1) / g.n_tt + 15) / 16 * 16;
    g.n_tt = (T + g.TN - 1) / g.TN;
    const int items = g.n_tiles * g.n_tt;
    g.splits = std::max(1, std::min(std::min(THIN_MAX_SPLITS, n_sm / items), g.num_kb / 2));
    // Two CTAs to an SM where several token tiles make L2 -> SM traffic the bound (the operands in flight of one CTA, 96 KB, bring
    // 36 bytes a cycle of the 63 that an SM can take), K leaves every part 16 k-blocks, and clusters of four fill the slots
    // (larger clusters and those of three or six do not all fit at a time: 1B down at 320 tokens 29.5 < 35.5 us with six).  Event
    // times, one CTA to an SM and two: 1B down at 448 tokens 33.3 > 29.2 us, at 512 34.6 > 31.4; 8B o at 160 tokens 23.0 > 21.0.
    // By items, o and down (128 k-blocks) of models of that many tiles, 144 to 256 tokens (three or four token tiles: 384 and 512):
    // 56 items 25.0 > 23.5 and 37.3 > 31.5, 60 36.5 > 31.4 (down), 68 24.8 > 22.9 and 37.3 > 29.1; from 72 on a last cluster of
    // four waits for a whole round of the others: 72 29.2 < 34.2 and 38.6 < 44.6, 74 27.1 < 36.2 and 39.4 < 46.2; steps of 69 and 70
    // items are 1.04 to 1.14 times as fast, so the line is at 70 of the 74 that two CTAs to an SM would make.
    if (g.n_tt >= 2 && 4 * items <= 2 * n_sm - 16 && 4 * items >= 3 * n_sm / 2 && g.num_kb >= 64) g.splits = 4;
    const int recv = g.splits > 1 ? thin_recv_bytes(g.TN, g.splits) : 0;
    g.recv_own = recv > 0 && recv <= THIN_RECV_OWN_MAX;
    g.n_stages = thin_stages(g.TN, g.recv_own ? recv : 0);
}

// Whether a projection takes the thin kernel.  Measured against the other kernels, event times of a class in us, other >
// thin, at 8 layers and fewer of the three model widths:
//   one token tile (128 tokens and fewer): 1B shape o 20.8 > 14.3 and down 26.8 > 18.5 at 40 tokens, 8B shape qkv 27.4 > 20.9,
//   o 28.2 > 16.9, gate/up 55.2 > 48.2 (128 tokens), 32B shape o 31.0 > 20.5; not a projection with so many tiles that the
//   launch is many rounds of CTAs (lm_head of the 8B shape 182 < 188 at 80 tokens), unless the tokens are very few (173 > 170 at 40);
//   several token tiles read the weights once each, which only pays while every CTA has little work: 1B shape at 256 tokens
//   qkv 31.1 > 20.9 (16 k-blocks a CTA), gate/up 29.1 > 28.1 (32), down 36.9 > 25.0 (32), 8B shape o 35.1 > 27.0 (32); but
//   8B shape qkv 31.1 < 36.3 (176 tokens, 64 k-blocks), down 46 < 54 (112), 1B gate/up 35 < 41 at 320 tokens (384 CTAs).
//   Beyond 512 tokens qkv of a narrow model (32 k-blocks, two CTAs to an SM): 1B 30.5 > 23.0 at 576 tokens, 33.1 > 23.2 at 640,
//   29.0 > 24.5 at 768, 29.0 = 28.8 at 1 024; its o would gain little (24.4 > 22.8 at 576) and is left to the other kernels.
static bool thin_takes(int T, int packed_rows, int K, int n_sm, int mode) {
    if (T > (mode == EPI_QKV ? THIN_MAX_TOKENS_QKV : THIN_MAX_TOKENS)) return false;
    ThinParams g;
    thin_plan(T, packed_rows, K, n_sm, g);
    const int items = g.n_tiles * g.n_tt, S = std::min(g.splits, std::max(1, n_sm / items));   // (one CTA to an SM)
    const int ctas = items * S, nk = (g.num_kb + S - 1) / S;
    if (g.n_tt == 1) return T <= 64 || ctas <= 3 * n_sm;
    return mode == EPI_RESID ? ctas <= n_sm && nk <= 64 : ctas <= 2 * n_sm && nk <= 32;
}

static int thin_smem(const ThinParams& g) {
    return thin_fixed_smem(g.TN) + g.n_stages * thin_stage_bytes(g.TN) + (g.recv_own ? thin_recv_bytes(g.TN, g.splits) : 0);
}

template <int MODE>
static cudaError_t launch_thin_mode(const ThinParams& g, const XMaps& xm, const EpiParams& ep, cudaStream_t st) {
    return launch_pdl_clusters(thin_kernel<MODE>, dim3(g.n_tiles * g.n_tt * g.splits), dim3(THIN_THREADS), thin_smem(g), st, g.splits,
                               xm.thin[g.TN / 16 - 1], g, ep);
}

static int launch_thin(syn_model* prof_m, int cls, int n_sm, int* status, const op16* w_packed, int packed_rows, int K, const XMaps& xm,
                       const EpiParams& ep, cudaStream_t st) {
    ProfScope prof(cls >= 0 ? prof_m : nullptr, cls, st);
    ThinParams g;
    thin_plan(ep.T, packed_rows, K, n_sm, g);
    g.w = w_packed; g.status = status; g.spin_limit = g_spin_limit;
    cudaError_t e;
    EPI_SWITCH(ep.mode, e = launch_thin_mode<MODE>(g, xm, ep, st));
    return e == cudaSuccess ? SYN_OK : SYN_E_CUDA;
}

// What a caller may ask of launch_proj instead of the kernel the shape calls for (test hook).
enum { PROJ_AUTO = 0, PROJ_QUAD = PAIR_QUAD, PROJ_DUO = PAIR_DUO, PROJ_THIN, PROJ_NOT_THIN };

// Which kernel a projection takes and how, worked out once for the layers of a step.
struct ProjPlan {
    bool thin;
    int kind;   // PAIR_NONE: the one-CTA kernel
    Gemm2Params g2;
    int n_cl;
};
static ProjPlan proj_plan(int T, int packed_rows, int K, int n_sm, int plan_mode, int force = PROJ_AUTO) {
    ProjPlan pl;
    pl.thin = force == PROJ_THIN || (force == PROJ_AUTO && g_schedule != 1 && thin_takes(T, packed_rows, K, n_sm, plan_mode));
    const int force_pair = force == PROJ_QUAD || force == PROJ_DUO ? force : PAIR_NONE;
    pl.n_cl = 0;
    pl.kind = !pl.thin && (g_schedule != 1 || force_pair != PAIR_NONE) ? gemm2_plan(T, packed_rows, K, n_sm, plan_mode, force_pair, pl.g2, pl.n_cl) : PAIR_NONE;
    return pl;
}

// One projection with the epilogue `ep` on the kernel its plan says.  `plan_mode` = the epilogue the schedule is made for (the
// same, except in the test hook).
static int launch_proj(syn_model* prof_m, int cls, int n_sm, int* status, const op16* w_packed, const WMaps* wm, int packed_rows,
                       int K, const XMaps& xm, const EpiParams& ep, cudaStream_t st, float* fix_part, int* fix_flag, const ProjPlan& pl,
                       int plan_mode = -1) {
    if (plan_mode < 0) plan_mode = ep.mode;
    if (pl.thin) return launch_thin(prof_m, cls, n_sm, status, w_packed, packed_rows, K, xm, ep, st);
    if (pl.kind == PAIR_NONE) return launch_gemm(prof_m, cls, n_sm, status, w_packed, packed_rows, K, xm.box, ep, st, fix_part, fix_flag, plan_mode);
    if (!fix_part || !fix_flag) return SYN_E_INVALID_ARG;
    Gemm2Params g2 = pl.g2;
    const int n_cl = pl.n_cl, kind = pl.kind;
    ProfScope prof(cls >= 0 ? prof_m : nullptr, cls, st);
    g2.status = status; g2.spin_limit = g_spin_limit;
    g2.fix_part = fix_part; g2.fix_flag = fix_flag;
    const bool duo = kind == PAIR_DUO;
    const int smem = gemm_fixed_smem(g2.TN) + g2.n_stages * gemm2_stage_bytes(g2.TN, duo);
    cudaError_t le;
    EPI_SWITCH(ep.mode, le = duo ? launch_pdl_clusters(gemm2_kernel<true, MODE>, dim3(2 * n_cl), dim3(gemm_threads(MODE)), smem, st, 2, wm->duo, xm.box, g2, ep)
                                 : launch_pdl_clusters(gemm2_kernel<false, MODE>, dim3(2 * n_cl), dim3(gemm_threads(MODE)), smem, st, 2, wm->quad, xm.box, g2, ep));
    return le == cudaSuccess ? SYN_OK : SYN_E_CUDA;
}

static void attn_params(AttnParams& ap, const syn_model* m, const syn_kv* kv, const syn_plan* p, uint32_t layer, op16* out,
                        float* part_o, float2* part_ml, int* group_count) {
    const syn_model_desc& c = m->desc;
    ap.items = p->d<AttnItem>(p->o_items);
    ap.cta_begin = p->d<int>(p->o_cta);
    ap.page_tables = p->d<int>(p->o_tables);
    ap.max_pages = p->max_pages;
    ap.n_kv_heads = c.n_kv_heads;
    ap.group = c.n_q_heads / c.n_kv_heads;
    ap.q_dim = c.n_q_heads * c.head_dim;
    ap.row_cap = attn_rows(p->attn);
    ap.q_box_tokens = p->attn == ATTN_TENSOR ? std::min(SYN_MAX_CHUNK, 128 / ap.group) : std::min(16, 64 / ap.group);
    ap.layer_block0 = (int)(2ull * layer * kv->n_pages * c.n_kv_heads);
    ap.scale_log2 = (float)(1.4426950408889634 / std::sqrt((double)c.head_dim));
    ap.q = m->q;
    memset(ap.ahead, 0, sizeof(ap.ahead));
    ap.ahead_late = 0;
    ap.out = out;
    ap.part_o = part_o;
    ap.part_ml = part_ml;
    ap.groups = p->d<MergeGroup>(p->o_groups);
    ap.group_count = group_count;
    ap.status = m->status_dev;
    ap.n_items = p->n_items; ap.n_req = p->n_req; ap.n_tokens = p->T; ap.n_pages = (int)kv->n_pages;
    ap.n_parts = p->n_parts; ap.n_groups = p->n_groups;
}

// Weights that the half-SM attention asks of L2 for the projections behind it, while HBM would idle: 24 MB, at most ten tiles
// of 16 KB per CTA (more, and a CTA with few keys outlasts the merge).  Measured, us a step at 0 / 16 / 24 / 40 MB: 1B shape,
// one request 840 / 830 / - / 883 (104 CTAs), 1B shape, two requests 878 / 870 / 863 / 844, 8B shape, eight requests
// 4 048 / 3 956 / 3 939 / 3 922, 16 requests 2 414 / 2 400 / 2 403 / 2 440 (16 layers).  Where a layer has more than 16 MB of
// keys a CTA waits for its own first (8B shape, eight requests, without that: 3 974).
// Only where most items are parts: while those are merged HBM idles, whereas whole units of unequal length keep some CTAs loading
// to the end, and these the requests delay (1B shape, with and without: 32 requests of 256 - 2 048 keys 1 300 and 1 268 us a step,
// 26 of 380 - 474 keys 894 and 863, 4 of 78 - 125 keys 787 and 755; one request in 104 parts 774 and 788; 8B shape, eight requests in
// 288 parts 3 764 and 3 818).  Where the line lies, over 176 batches of 3 to 32 requests, steps with the requests over those without:
// no item a part 1B 1.02 - 1.08 and 8B 1.01 - 1.02; up to half of them 1B 1.02 - 1.04, 8B 1.00 - 1.01; half to 0.8 1B 0.99 - 1.03,
// 8B 0.99 - 1.01; above that 1B 0.98 - 1.03, 8B 0.98 - 1.01.
constexpr int64_t ATTN_AHEAD_BYTES = 24 << 20, ATTN_AHEAD_TILES = 10, ATTN_AHEAD_LATE_BYTES = 16 << 20;

// What the attention may ask of L2 ahead: `budget` bytes (taken off) of a projection's weights beyond what the operand rings
// of its CTAs hold anyway.
static WeightsAhead weights_ahead(const op16* w, int T, int packed_rows, int K, int n_sm, int mode, int64_t& budget) {
    WeightsAhead a;
    memset(&a, 0, sizeof(a));
    ThinParams g;
    if (budget <= 0 || g_schedule == 1 || !thin_takes(T, packed_rows, K, n_sm, mode)) return a;
    thin_plan(T, packed_rows, K, n_sm, g);
    const int units = g.n_tiles * g.splits, nk = (g.num_kb + g.splits - 1) / g.splits;
    a.w = w; a.num_kb = g.num_kb; a.n_tiles = g.n_tiles; a.n_tt = g.n_tt; a.splits = g.splits;
    a.skip = std::min(g.n_stages, nk);
    a.count = (int)std::min<int64_t>(nk - a.skip, budget / ((int64_t)units * GEMM_TILE_BYTES));
    budget -= (int64_t)units * a.count * GEMM_TILE_BYTES;
    return a;
}

// The kernel the plan was made for; `pdl`: may start while its predecessor in the stream still runs.
static cudaError_t attention_kernel(const syn_model* m, const syn_kv* kv, const syn_plan* p, const AttnParams& ap, const CUtensorMap& tmQ, bool pdl,
                                    cudaStream_t st) {
    const bool wide_head = m->desc.head_dim == 128;
    const dim3 grid(p->n_cta);
    switch (p->attn) {
        case ATTN_TENSOR:
            return wide_head ? launch(attn2_kernel<128>, grid, dim3(ATT2_THREADS), Attn2Smem<128>::TOTAL, st, pdl, m->tm_q4, kv->tm_kv5, ap)
                             : launch(attn2_kernel<64>, grid, dim3(ATT2_THREADS), Attn2Smem<64>::TOTAL, st, pdl, m->tm_q4, kv->tm_kv5, ap);
        case ATTN_THIN:
            return wide_head ? launch(attn_thin_kernel<128>, grid, dim3(ATTN_THIN_THREADS), AttnThinSmem<128>::TOTAL, st, pdl, kv->tm_kv, ap)
                             : launch(attn_thin_kernel<64>, grid, dim3(ATTN_THIN_THREADS), AttnThinSmem<64>::TOTAL, st, pdl, kv->tm_kv, ap);
        default:
            return wide_head ? launch(attn_kernel<128>, grid, dim3(ATT_THREADS), AttnSmem<128>::TOTAL, st, pdl, tmQ, kv->tm_kv, ap)
                             : launch(attn_kernel<64>, grid, dim3(ATT_THREADS), AttnSmem<64>::TOTAL, st, pdl, tmQ, kv->tm_kv, ap);
    }
}

static int launch_attention(syn_model* m, syn_kv* kv, const syn_plan* p, uint32_t layer, const CUtensorMap& tmQ,
                            op16* out, cudaStream_t st) {
    AttnParams ap;
    attn_params(ap, m, kv, p, layer, out, m->part_o, m->part_ml, m->group_count);
    if (p->attn == ATTN_THIN && 2 * p->n_parts > p->n_items) {
        const syn_model_desc& c = m->desc;
        const int d = c.d_model, q_dim = c.n_q_heads * c.head_dim;
        int64_t budget = std::min(ATTN_AHEAD_BYTES, (int64_t)p->n_cta * ATTN_AHEAD_TILES * GEMM_TILE_BYTES);
        ap.ahead_late = p->stats.kv_read_bytes / c.n_layers > ATTN_AHEAD_LATE_BYTES;
        ap.ahead[0] = weights_ahead(m->wo[layer], p->T, d, q_dim, m->n_sm, EPI_RESID, budget);
        ap.ahead[1] = weights_ahead(m->wgu[layer], p->T, m->gu_rows, d, m->n_sm, EPI_SWIGLU, budget);
    }
    {
        ProfScope prof(m, 2, st);
        if (attention_kernel(m, kv, p, ap, tmQ, true, st) != cudaSuccess) return SYN_E_CUDA;
    }
    return SYN_OK;
}

static int run_step(syn_model* m, syn_kv* kv, const syn_plan* p, int* acc_dev, int* corr_dev, int* top1_dev,
                    float* logits_out, cudaStream_t st, uint32_t* warp_max = nullptr, int* status_out = nullptr) {
    const syn_model_desc& c = m->desc;
    const int T = p->T, d = c.d_model, q_dim = c.n_q_heads * c.head_dim, kv_dim = c.n_kv_heads * c.head_dim;
    if (T > m->t_cap || p->n_parts > m->part_cap) return SYN_E_INVALID_ARG;
    const int* tokens = p->d<int>(p->o_tokens);
    const float inv_d = 1.0f / (float)d;
    // Where nobody asked for logits or argmaxes, the lm_head runs over the rows that verification looks at, if they are at most
    // half of more than 128 (up to there its time is that of its weights: 1B shape 37 us at 128 tokens, 105 at 768; a
    // prefill iteration of 768 tokens of 24 requests needs 24 rows).  At the edge, steps of two layers with all rows and with
    // those: 1B shape 129 tokens, 64 rows 162.7 > 158.7 us, 160 and 80 163.0 = 162.9, 192 and 96 177.2 = 177.1, 256 and 128
    // 205.8 > 197.6; 8B shape 129 and 64 449 > 431, 160 and 80 462 > 437, 256 and 128 578 > 521; 32B width, one layer, 129 and 64
    // 545 > 511, 256 and 128 664 > 593.
    const bool judging_only = !logits_out && !top1_dev && T > 128 && 2 * p->n_judging <= T;
    const int T_lm = judging_only ? p->n_judging : T;
    m->last_stats = p->stats;
    m->last_stats.dense_flops -= 2.0 * (T - T_lm) * (double)d * c.vocab;
    m->last_stats.kernel_launches += judging_only;
    m->have_last = true;
    m->step_timed = false;
    m->last_wall_ms = 0.0;
    if (m->profile) {
        if (!m->step_a) CU_OK(cudaEventCreate(&m->step_a));
        if (!m->step_b) CU_OK(cudaEventCreate(&m->step_b));
        CU_OK(cudaEventRecord(m->step_a, st));
    }
    {
        ProfScope prof(m, 0, st);
        if (launch_pdl(prep_kernel, dim3(T), dim3(256), 0, st, m->embed, tokens, p->d<int>(p->o_pos), m->norm1[0], m->inv_freq,
                       m->x, m->xn, m->ssq, m->rope, m->best, d, (int)(c.head_dim / 2)) != cudaSuccess)
            return SYN_E_CUDA;
    }
    EpiParams base;
    memset(&base, 0, sizeof(base));
    base.T = T;
    // the consumers of a normalised operand: RMSNorm scale from the partial sums of x^2
    EpiParams scaled = base;
    scaled.ssq_in = m->ssq; scaled.n_ssq = d / 32; scaled.inv_d = inv_d; scaled.eps = c.rms_eps;
    // the writers of the residual stream: x += D, next operand half(x * gain), new partial sums
    EpiParams resid = base;
    resid.mode = EPI_RESID; resid.N = d; resid.d = d; resid.x = m->x; resid.xg = m->xn; resid.ssq_out = m->ssq;
    // (the projections' plans, some 6 us each, are made in the first layer, while the kernels before run)
    ProjPlan pl_qkv, pl_o, pl_gu, pl_d;
    int r;
    for (uint32_t l = 0; l < c.n_layers; ++l) {
        EpiParams e = scaled;
        e.mode = EPI_QKV; e.N = m->qkv_rows;
        e.q = m->q; e.q_dim = q_dim; e.kv_dim = kv_dim; e.hd = c.head_dim; e.n_kv_heads = c.n_kv_heads;
        e.page_size = kv->page_size; e.rope = m->rope; e.pool = kv->pool + kv->layer_elems * l;
        e.slot = p->d<int>(p->o_slot);
        if (l == 0) pl_qkv = proj_plan(T, m->qkv_rows, d, m->n_sm, EPI_QKV);
        if ((r = launch_proj(m, 1, m->n_sm, m->status_dev, m->wqkv[l], &m->tm_wqkv[l], m->qkv_rows, d, m->tm_xn, e, st, m->fix_part, m->fix_flag, pl_qkv)))
            return r;
        if ((r = launch_attention(m, kv, p, l, m->tm_q, m->attn, st))) return r;
        e = resid;
        e.gain = m->norm2[l];
        if (l == 0) pl_o = proj_plan(T, d, q_dim, m->n_sm, EPI_RESID);
        if ((r = launch_proj(m, 4, m->n_sm, m->status_dev, m->wo[l], &m->tm_wo[l], d, q_dim, m->tm_attn, e, st, m->fix_part, m->fix_flag, pl_o)))
            return r;
        e = scaled;
        e.mode = EPI_SWIGLU; e.N = m->gu_rows; e.act = m->act; e.f_pad = m->f_pad;
        if (l == 0) pl_gu = proj_plan(T, m->gu_rows, d, m->n_sm, EPI_SWIGLU);
        if ((r = launch_proj(m, 5, m->n_sm, m->status_dev, m->wgu[l], &m->tm_wgu[l], m->gu_rows, d, m->tm_xn, e, st, m->fix_part, m->fix_flag, pl_gu)))
            return r;
        e = resid;
        e.gain = l + 1 < c.n_layers ? m->norm1[l + 1] : m->final_norm;
        if (l == 0) pl_d = proj_plan(T, d, m->f_pad, m->n_sm, EPI_RESID);
        if ((r = launch_proj(m, 6, m->n_sm, m->status_dev, m->wd[l], &m->tm_wd[l], d, m->f_pad, m->tm_act, e, st, m->fix_part, m->fix_flag, pl_d)))
            return r;
    }
    EpiParams e = scaled;
    if (judging_only) {
        ProfScope prof(m, 9, st);
        if (launch_pdl(judging_rows_kernel, dim3(T_lm), dim3(256), 0, st, m->xn, m->ssq, p->d<int>(p->o_row), m->xj, m->ssqj, d) != cudaSuccess)
            return SYN_E_CUDA;
        e.T = T_lm;
        e.ssq_in = m->ssqj;
    }
    e.mode = EPI_LMHEAD; e.N = m->v_rows; e.vocab = c.vocab; e.logits = logits_out; e.best = m->best;
    e.warp_max = warp_max; e.n_warp_max = m->v_rows / 32;
    const ProjPlan pl_lm = proj_plan(T_lm, m->v_rows, d, m->n_sm, EPI_LMHEAD);
    if ((r = launch_proj(m, 7, m->n_sm, m->status_dev, m->lm_head, &m->tm_lm_head, m->v_rows, d, judging_only ? m->tm_xj : m->tm_xn, e, st, m->fix_part, m->fix_flag, pl_lm)))
        return r;
    {
        ProfScope prof(m, 8, st);
        if (launch_pdl(verify_kernel, dim3((p->n_req + 127) / 128), dim3(128), 0, st, m->best, tokens, p->d<int>(p->o_offsets),
                       p->d<int>(p->o_uncached), p->n_req, acc_dev, corr_dev, top1_dev, judging_only ? p->d<int>(p->o_first) : nullptr,
                       m->status_dev, status_out) != cudaSuccess)
            return SYN_E_CUDA;
    }
    if (m->profile) {
        CU_OK(cudaEventRecord(m->step_b, st));
        m->step_timed = true;
    }
    return SYN_OK;
}

static int syn_verify_run_impl(syn_model* m, syn_kv* kv, const syn_plan* p, int32_t* accept_len_dev, int32_t* correction_dev,
                              int32_t* top1_dev, float* logits_out, void* cuda_stream) {
    if (!m || !kv || !p || kv->model != m || !plan_matches(p, kv) || !accept_len_dev || !correction_dev) return SYN_E_INVALID_ARG;
    return run_step(m, kv, p, accept_len_dev, correction_dev, top1_dev, logits_out, reinterpret_cast<cudaStream_t>(cuda_stream));
}

extern "C" int syn_set_profile(syn_model* m, int on) {
    if (!m) return SYN_E_INVALID_ARG;
    m->profile = on != 0;
    return SYN_OK;
}

static int syn_get_profile_impl(syn_model* m, double* ms, int32_t* launches) {
    if (!m || !ms || !launches) return SYN_E_INVALID_ARG;
    CU_OK(cudaDeviceSynchronize());
    for (int i = 0; i < SYN_N_KERNEL_CLASSES; ++i) { ms[i] = 0.0; launches[i] = 0; }
    for (auto& e : m->ev_used) {
        float t = 0.f;
        if (cudaEventElapsedTime(&t, e.a, e.b) == cudaSuccess && e.cls >= 0 && e.cls < SYN_N_KERNEL_CLASSES) {
            ms[e.cls] += t;
            launches[e.cls] += 1;
        }
        m->ev_free.push_back(e);
    }
    m->ev_used.clear();
    return SYN_OK;
}

extern "C" int syn_model_status(syn_model* m) {
    if (!m) return SYN_E_INVALID_ARG;
    int s = 0;
    if (cudaMemcpy(&s, m->status_dev, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return SYN_E_CUDA;
    if (s) {
        cudaMemset(m->status_dev, 0, 4);
        if (m->group_count) cudaMemset(m->group_count, 0, (size_t)m->part_cap * 4);   // an aborted step may leave counts
        if (m->fix_flag) cudaMemset(m->fix_flag, 0, (size_t)GEMM_FLAG_INTS * m->n_sm * 4);
        return SYN_E_DEVICE_TIMEOUT;
    }
    return SYN_OK;
}

static int syn_verify_batch_impl(syn_model* m, syn_kv* kv, int32_t n_req, const int64_t* req_ids, const int32_t* chunk_tokens,
                                const int32_t* chunk_offsets, const int32_t* page_tables, int32_t max_pages,
                                const int32_t* ctx_lens, const int32_t* n_uncached, int32_t* accept_len,
                                int32_t* correction_token, float* logits_out, void* cuda_stream) {
    (void)req_ids;
    if (!m || !accept_len || !correction_token) return SYN_E_INVALID_ARG;
    if (!m->scratch_plan) {
        m->scratch_plan = new (std::nothrow) syn_plan();
        if (!m->scratch_plan) return SYN_E_OOM;
    }
    syn_plan* p = m->scratch_plan;
    int r = plan_build(p, m, kv, n_req, chunk_tokens, chunk_offsets, page_tables, max_pages, ctx_lens, n_uncached);
    if (r) return r;
    if ((r = ensure_workspace(m, p->T, p->n_parts))) return r;
    if (n_req > m->pinned_out_cap) {
        if (m->pinned_out) cudaFreeHost(m->pinned_out);
        m->pinned_out = nullptr; m->pinned_out_cap = 0;
        const int cap = (n_req + 255) / 256 * 256;
        CU_OK(cudaMallocHost(&m->pinned_out, (size_t)cap * 12));
        m->pinned_out_cap = cap;
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
    CU_OK(cudaMemcpyAsync(p->dev, p->host, p->used, cudaMemcpyHostToDevice, st));
    int *const po = m->pinned_out, *const po_corr = po + m->pinned_out_cap, *const po_status = po + 2 * m->pinned_out_cap;
    if ((r = run_step(m, kv, p, po, po_corr, nullptr, logits_out, st, nullptr, po_status))) return r;
    CU_OK(cudaStreamSynchronize(st));
    if (*po_status) {
        cudaMemset(m->status_dev, 0, 4);
        if (m->group_count) cudaMemset(m->group_count, 0, (size_t)m->part_cap * 4);
        if (m->fix_flag) cudaMemset(m->fix_flag, 0, (size_t)GEMM_FLAG_INTS * m->n_sm * 4);
        return SYN_E_DEVICE_TIMEOUT;
    }
    memcpy(accept_len, po, (size_t)n_req * 4);
    memcpy(correction_token, po_corr, (size_t)n_req * 4);
    return SYN_OK;
}

// ------------------------------------------------------------------------------------------ sampling-based verification

static int check_sampling(const syn_sampling* cfg, int vocab, int T, int n_req, const int32_t* slm_ids, const float* slm_probs,
                          const float* rand_accept, const float* rand_sample) {
    if (!cfg || !slm_ids || !slm_probs || !rand_accept || !rand_sample) return SYN_E_INVALID_ARG;
    if (cfg->top_k < 1 || cfg->top_k > SYN_SAMPLE_MAX_K || cfg->slm_k < 1 || cfg->slm_k > SYN_SAMPLE_MAX_K) return SYN_E_INVALID_ARG;
    if (!(cfg->top_p > 0.f && cfg->top_p <= 1.f) || !(cfg->temperature > 0.f)) return SYN_E_INVALID_ARG;
    for (size_t i = 0; i < (size_t)T * cfg->slm_k; ++i) {
        if (slm_ids[i] < -1 || slm_ids[i] >= vocab) return SYN_E_TOKEN_OOB;
        if (!(slm_probs[i] >= 0.f && slm_probs[i] <= 1.f)) return SYN_E_INVALID_ARG;
    }
    for (int t = 0; t < T; ++t)
        if (!(rand_accept[t] >= 0.f && rand_accept[t] < 1.f)) return SYN_E_INVALID_ARG;
    for (int i = 0; i < n_req; ++i)
        if (!(rand_sample[i] >= 0.f && rand_sample[i] < 1.f)) return SYN_E_INVALID_ARG;
    return SYN_OK;
}

// The two kernels behind the lm_head; every pointer is device memory.
static int sample_stage(syn_model* prof_m, cudaStream_t st, const float* logits, int T, int V, int n_req, const int* tokens,
                        const int* offsets, const int* uncached, const syn_sampling& cfg, int* topk_id, float* topk_logit,
                        const int* slm_id, const float* slm_prob, const float* rand_accept, const float* rand_sample,
                        int* acc_dev, int* corr_dev, const uint32_t* warp_max = nullptr, int n_warp_max = 0) {
    ProfScope prof(prof_m, 8, st);
    if (launch_pdl(topk_rows_kernel, dim3(T), dim3(TOPK_THREADS), 0, st, logits, V, offsets, uncached, n_req, (int)cfg.top_k,
                   warp_max, n_warp_max, topk_id, topk_logit) != cudaSuccess)
        return SYN_E_CUDA;
    SampleParams sp;
    sp.tokens = tokens; sp.offsets = offsets; sp.uncached = uncached;
    sp.topk_id = topk_id; sp.topk_logit = topk_logit;
    sp.slm_id = slm_id; sp.slm_prob = slm_prob; sp.rand_accept = rand_accept; sp.rand_sample = rand_sample;
    sp.accept_len = acc_dev; sp.correction = corr_dev;
    sp.n_req = n_req; sp.top_k = cfg.top_k; sp.slm_k = cfg.slm_k;
    sp.top_p = cfg.top_p; sp.inv_temperature = 1.0f / cfg.temperature;
    if (launch_pdl(sample_verify_kernel, dim3(n_req), dim3(SAMPLE_MAX_K), 0, st, sp) != cudaSuccess) return SYN_E_CUDA;
    return SYN_OK;
}

static int ensure_sample_ws(syn_model* m, int T, int B, int slm_k, bool own_logits) {
    syn_model::SampleWs& w = m->sw;
    const size_t need_logits = own_logits ? (size_t)T * m->desc.vocab : 0;
    if (need_logits > w.logits_cap) {
        cudaFree(w.logits); w.logits = nullptr; w.logits_cap = 0;
        CU_OK(cudaMalloc(&w.logits, need_logits * 4));
        w.logits_cap = need_logits;
    }
    if (T > w.t_cap) {
        cudaFree(w.topk_id); cudaFree(w.topk_logit); cudaFree(w.rand_accept); cudaFree(w.warp_max);
        w.topk_id = nullptr; w.topk_logit = nullptr; w.rand_accept = nullptr; w.warp_max = nullptr; w.t_cap = 0;
        const int cap = (T + 255) / 256 * 256;
        CU_OK(cudaMalloc(&w.warp_max, (size_t)cap * (m->v_rows / 32) * 4));
        CU_OK(cudaMalloc(&w.topk_id, (size_t)cap * SAMPLE_MAX_K * 4));
        CU_OK(cudaMalloc(&w.topk_logit, (size_t)cap * SAMPLE_MAX_K * 4));
        CU_OK(cudaMalloc(&w.rand_accept, (size_t)cap * 4));
        w.t_cap = cap;
        w.slm_cap = 0;
    }
    if (T * slm_k > w.slm_cap) {
        cudaFree(w.slm_id); cudaFree(w.slm_prob);
        w.slm_id = nullptr; w.slm_prob = nullptr; w.slm_cap = 0;
        const int cap = w.t_cap * slm_k;
        CU_OK(cudaMalloc(&w.slm_id, (size_t)cap * 4));
        CU_OK(cudaMalloc(&w.slm_prob, (size_t)cap * 4));
        w.slm_cap = cap;
    }
    if (B > w.b_cap) {
        cudaFree(w.rand_sample); w.rand_sample = nullptr; w.b_cap = 0;
        const int cap = (B + 255) / 256 * 256;
        CU_OK(cudaMalloc(&w.rand_sample, (size_t)cap * 4));
        w.b_cap = cap;
    }
    return SYN_OK;
}

static int syn_verify_batch_sampled_impl(syn_model* m, syn_kv* kv, int32_t n_req, const int64_t* req_ids,
                                        const int32_t* chunk_tokens, const int32_t* chunk_offsets, const int32_t* page_tables,
                                        int32_t max_pages, const int32_t* ctx_lens, const int32_t* n_uncached,
                                        const syn_sampling* cfg, const int32_t* slm_ids, const float* slm_probs,
                                        const float* rand_accept, const float* rand_sample, int32_t* accept_len,
                                        int32_t* correction_token, float* logits_out, void* cuda_stream) {
    (void)req_ids;
    if (!m || !accept_len || !correction_token) return SYN_E_INVALID_ARG;
    if (!m->scratch_plan) {
        m->scratch_plan = new (std::nothrow) syn_plan();
        if (!m->scratch_plan) return SYN_E_OOM;
    }
    syn_plan* p = m->scratch_plan;
    int r = plan_build(p, m, kv, n_req, chunk_tokens, chunk_offsets, page_tables, max_pages, ctx_lens, n_uncached);
    if (r) return r;
    if ((r = check_sampling(cfg, (int)m->desc.vocab, p->T, n_req, slm_ids, slm_probs, rand_accept, rand_sample))) return r;
    if ((r = ensure_workspace(m, p->T, p->n_parts))) return r;
    if ((r = ensure_sample_ws(m, p->T, n_req, cfg->slm_k, logits_out == nullptr))) return r;
    if (n_req > m->pinned_out_cap) {
        if (m->pinned_out) cudaFreeHost(m->pinned_out);
        m->pinned_out = nullptr; m->pinned_out_cap = 0;
        const int cap = (n_req + 255) / 256 * 256;
        CU_OK(cudaMallocHost(&m->pinned_out, (size_t)cap * 12));
        m->pinned_out_cap = cap;
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
    syn_model::SampleWs& w = m->sw;
    float* logits = logits_out ? logits_out : w.logits;
    CU_OK(cudaMemcpyAsync(p->dev, p->host, p->used, cudaMemcpyHostToDevice, st));
    CU_OK(cudaMemcpyAsync(w.slm_id, slm_ids, (size_t)p->T * cfg->slm_k * 4, cudaMemcpyHostToDevice, st));
    CU_OK(cudaMemcpyAsync(w.slm_prob, slm_probs, (size_t)p->T * cfg->slm_k * 4, cudaMemcpyHostToDevice, st));
    CU_OK(cudaMemcpyAsync(w.rand_accept, rand_accept, (size_t)p->T * 4, cudaMemcpyHostToDevice, st));
    CU_OK(cudaMemcpyAsync(w.rand_sample, rand_sample, (size_t)n_req * 4, cudaMemcpyHostToDevice, st));
    int *const po = m->pinned_out, *const po_corr = po + m->pinned_out_cap, *const po_status = po + 2 * m->pinned_out_cap;
    if ((r = run_step(m, kv, p, po, po_corr, nullptr, logits, st, w.warp_max, po_status))) return r;
    // the greedy results of the step are replaced by the sampled ones
    if ((r = sample_stage(m, st, logits, p->T, (int)m->desc.vocab, n_req, p->d<int>(p->o_tokens), p->d<int>(p->o_offsets),
                          p->d<int>(p->o_uncached), *cfg, w.topk_id, w.topk_logit, w.slm_id, w.slm_prob, w.rand_accept,
                          w.rand_sample, po, po_corr, w.warp_max, m->v_rows / 32)))
        return r;
    CU_OK(cudaStreamSynchronize(st));
    if (*po_status) {
        cudaMemset(m->status_dev, 0, 4);
        if (m->group_count) cudaMemset(m->group_count, 0, (size_t)m->part_cap * 4);
        if (m->fix_flag) cudaMemset(m->fix_flag, 0, (size_t)GEMM_FLAG_INTS * m->n_sm * 4);
        return SYN_E_DEVICE_TIMEOUT;
    }
    memcpy(accept_len, po, (size_t)n_req * 4);
    memcpy(correction_token, po_corr, (size_t)n_req * 4);
    return SYN_OK;
}

// ------------------------------------------------------------------------------------------ single ops

// The sampling stage alone on logits the caller supplies (device, fp32 [T][vocab]).
static int syn_op_sample_verify_impl(const float* logits, int32_t T, int32_t vocab, int32_t n_req, const int32_t* chunk_tokens,
                                    const int32_t* chunk_offsets, const int32_t* n_uncached, const syn_sampling* cfg,
                                    const int32_t* slm_ids, const float* slm_probs, const float* rand_accept,
                                    const float* rand_sample, int32_t* accept_len, int32_t* correction_token,
                                    void* cuda_stream) {
    if (!logits || T <= 0 || vocab <= 0 || n_req <= 0 || !chunk_tokens || !chunk_offsets || !n_uncached || !accept_len ||
        !correction_token)
        return SYN_E_INVALID_ARG;
    if (chunk_offsets[0] != 0 || chunk_offsets[n_req] != T) return SYN_E_INVALID_ARG;
    for (int i = 0; i < n_req; ++i) {
        const int n = chunk_offsets[i + 1] - chunk_offsets[i];
        if (n < 1 || n > SYN_MAX_CHUNK) return SYN_E_CHUNK_LEN;
        if (n_uncached[i] < 1 || n_uncached[i] > n) return SYN_E_UNCACHED;
    }
    for (int t = 0; t < T; ++t)
        if (chunk_tokens[t] < 0 || chunk_tokens[t] >= vocab) return SYN_E_TOKEN_OOB;
    int r = check_sampling(cfg, vocab, T, n_req, slm_ids, slm_probs, rand_accept, rand_sample);
    if (r) return r;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
    const size_t n_slm = (size_t)T * cfg->slm_k;
    // one device block: tokens, offsets, uncached, slm ids | slm probs, draws | top-k lists | results
    const size_t n_i = (size_t)T + (n_req + 1) + n_req + n_slm + (size_t)T * SAMPLE_MAX_K + 2 * (size_t)n_req;
    const size_t n_f = n_slm + T + n_req + (size_t)T * SAMPLE_MAX_K;
    int* di = nullptr;
    float* df = nullptr;
    CU_OK(cudaMalloc(&di, n_i * 4));
    if (note_cuda(cudaMalloc(&df, n_f * 4)) != cudaSuccess) { cudaFree(di); return SYN_E_OOM; }
    int *d_tok = di, *d_off = d_tok + T, *d_unc = d_off + n_req + 1, *d_sid = d_unc + n_req, *d_tid = d_sid + n_slm,
        *d_acc = d_tid + (size_t)T * SAMPLE_MAX_K, *d_cor = d_acc + n_req;
    float *d_sp = df, *d_ra = d_sp + n_slm, *d_rs = d_ra + T, *d_tl = d_rs + n_req;
    std::vector<int> out(2 * (size_t)n_req);
    bool ok = cudaMemcpyAsync(d_tok, chunk_tokens, (size_t)T * 4, cudaMemcpyHostToDevice, st) == cudaSuccess &&
              cudaMemcpyAsync(d_off, chunk_offsets, (size_t)(n_req + 1) * 4, cudaMemcpyHostToDevice, st) == cudaSuccess &&
              cudaMemcpyAsync(d_unc, n_uncached, (size_t)n_req * 4, cudaMemcpyHostToDevice, st) == cudaSuccess &&
              cudaMemcpyAsync(d_sid, slm_ids, n_slm * 4, cudaMemcpyHostToDevice, st) == cudaSuccess &&
              cudaMemcpyAsync(d_sp, slm_probs, n_slm * 4, cudaMemcpyHostToDevice, st) == cudaSuccess &&
              cudaMemcpyAsync(d_ra, rand_accept, (size_t)T * 4, cudaMemcpyHostToDevice, st) == cudaSuccess &&
              cudaMemcpyAsync(d_rs, rand_sample, (size_t)n_req * 4, cudaMemcpyHostToDevice, st) == cudaSuccess;
    r = ok ? sample_stage(nullptr, st, logits, T, vocab, n_req, d_tok, d_off, d_unc, *cfg, d_tid, d_tl, d_sid, d_sp, d_ra, d_rs,
                          d_acc, d_cor)
           : SYN_E_CUDA;
    if (r == SYN_OK && (note_cuda(cudaMemcpyAsync(out.data(), d_acc, 2 * (size_t)n_req * 4, cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
                        note_cuda(cudaStreamSynchronize(st)) != cudaSuccess))
        r = SYN_E_CUDA;
    cudaFree(di);
    cudaFree(df);
    if (r) return r;
    memcpy(accept_len, out.data(), (size_t)n_req * 4);
    memcpy(correction_token, out.data() + n_req, (size_t)n_req * 4);
    return SYN_OK;
}

// Process-wide context of the single-projection test hook: status word, exchange workspace, and the
// packed copy of the last weight matrix seen.
struct LinearCtx {
    int n_sm = 0;
    int* status = nullptr;
    float* fix_part = nullptr;
    int* fix_flag = nullptr;
    op16* packed = nullptr;
    const void* packed_src = nullptr;
    int packed_n = 0, packed_k = 0;
    WMaps wm;
};
static LinearCtx g_lin;

static int linear_ctx_init() {
    if (g_lin.status) return SYN_OK;
    int dev = 0;
    cudaDeviceProp prop;
    CU_OK(cudaGetDevice(&dev));
    CU_OK(cudaGetDeviceProperties(&prop, dev));
    if (prop.major != 10) return SYN_E_ARCH;
    g_lin.n_sm = prop.multiProcessorCount;
    CU_OK(set_kernel_attributes());
    CU_OK(cudaMalloc(&g_lin.fix_part, (size_t)g_lin.n_sm * GEMM_FIX_SLOT_BYTES));
    CU_OK(cudaMalloc(&g_lin.fix_flag, (size_t)GEMM_FLAG_INTS * g_lin.n_sm * 4));
    CU_OK(cudaMemset(g_lin.fix_flag, 0, (size_t)GEMM_FLAG_INTS * g_lin.n_sm * 4));
    CU_OK(cudaMalloc(&g_lin.status, 4));
    CU_OK(cudaMemset(g_lin.status, 0, 4));
    return SYN_OK;
}

extern "C" int syn_op_linear_reset(void) {
    if (g_lin.packed) {
        CU_OK(cudaDeviceSynchronize());
        cudaFree(g_lin.packed);
    }
    g_lin.packed = nullptr; g_lin.packed_src = nullptr; g_lin.packed_n = g_lin.packed_k = 0;
    return SYN_OK;
}

extern "C" int syn_op_linear_as(const void* x, const void* w, float* y, int32_t T, int32_t N, int32_t K, int32_t schedule_as,
                                void* cuda_stream) {
    if (!x || !w || !y || T <= 0 || N <= 0 || K <= 0 || K % 8 != 0 || schedule_as < EPI_PLAIN || schedule_as > EPI_LMHEAD + 5)
        return SYN_E_INVALID_ARG;
    int r = load_driver_entry();
    if (r) return r;
    if ((r = linear_ctx_init())) return r;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
    const int n_mt = (N + 511) / 512 * 4, nkb = (K + 63) / 64;
    if (g_lin.packed_src != w || g_lin.packed_n != N || g_lin.packed_k != K) {
        if ((r = syn_op_linear_reset())) return r;
        CU_OK(cudaMalloc(&g_lin.packed, (size_t)n_mt * nkb * 128 * 64 * 2));
        PackSrc ps;
        memset(&ps, 0, sizeof(ps));
        ps.p[0] = (const bf16*)w; ps.rows[0] = N; ps.src_k = K;
        pack_weight_kernel<<<dim3(n_mt, nkb), 256, 0, st>>>(ps, g_lin.packed, nkb);
        if (!launch_ok()) return SYN_E_CUDA;
        CU_OK(cudaStreamSynchronize(st));   // the GEMM requests weight tiles before it waits for its predecessor
        g_lin.packed_src = w; g_lin.packed_n = N; g_lin.packed_k = K;
        if ((r = make_wmaps(g_lin.packed, n_mt * 128, K, &g_lin.wm))) return r;
    }
    XMaps xm;
    if ((r = make_xmaps(&xm, x, T, K))) return r;
    EpiParams e;
    memset(&e, 0, sizeof(e));
    e.mode = EPI_PLAIN; e.T = T; e.N = N; e.y = y; e.ldy = N;
    // 0..4: the one-CTA or CTA-pair schedule for that epilogue; 5, 6: CTA pairs with QUAD / DUO items; 7, 8: the same as
    // residual projections (K shared between clusters where the shape allows it); 9: the thin kernel
    const int force = schedule_as <= EPI_LMHEAD ? PROJ_NOT_THIN : (schedule_as == 9 ? PROJ_THIN : (schedule_as == 5 || schedule_as == 7 ? PROJ_QUAD : PROJ_DUO));
    const int plan_mode = schedule_as <= EPI_LMHEAD ? schedule_as : (schedule_as == 7 || schedule_as == 8 ? EPI_RESID : EPI_PLAIN);
    r = launch_proj(nullptr, -1, g_lin.n_sm, g_lin.status, g_lin.packed, &g_lin.wm, (N + 127) / 128 * 128, K, xm, e, st, g_lin.fix_part,
                    g_lin.fix_flag, proj_plan(T, (N + 127) / 128 * 128, K, g_lin.n_sm, plan_mode, force), plan_mode);
    if (r) return r;
    CU_OK(cudaStreamSynchronize(st));
    int sflag = 0;
    CU_OK(cudaMemcpy(&sflag, g_lin.status, 4, cudaMemcpyDeviceToHost));
    if (sflag) {
        cudaMemset(g_lin.status, 0, 4);
        cudaMemset(g_lin.fix_flag, 0, (size_t)GEMM_FLAG_INTS * g_lin.n_sm * 4);
        return SYN_E_DEVICE_TIMEOUT;
    }
    return SYN_OK;
}

extern "C" int syn_op_linear(const void* x, const void* w, float* y, int32_t T, int32_t N, int32_t K, void* cuda_stream) {
    return syn_op_linear_as(x, w, y, T, N, K, EPI_PLAIN, cuda_stream);
}

extern "C" int syn_debug_set_spin_limit(int64_t cycles) {
    if (cycles < 0) return SYN_E_INVALID_ARG;
    g_spin_limit = cycles == 0 ? SYN_SPIN_LIMIT_CYCLES : (long long)cycles;
    return SYN_OK;
}

extern "C" int syn_debug_set_schedule(int32_t which) {
    if (which < 0 || which > 1) return SYN_E_INVALID_ARG;
    g_schedule = which;
    return SYN_OK;
}

extern "C" int syn_debug_set_attention(int32_t which) {
    if (which < 0 || which > 3) return SYN_E_INVALID_ARG;
    g_attention = which;
    return SYN_OK;
}

extern "C" int syn_debug_linear_counter(int32_t index, int32_t value) {
    int r = linear_ctx_init();
    if (r) return r;
    if (index < 0 || index >= GEMM_FLAG_INTS * g_lin.n_sm) return SYN_E_INVALID_ARG;
    CU_OK(cudaDeviceSynchronize());
    CU_OK(cudaMemcpy(g_lin.fix_flag + index, &value, 4, cudaMemcpyHostToDevice));
    return SYN_OK;
}

static int syn_op_attention_impl(syn_model* m, syn_kv* kv, const syn_plan* p, uint32_t layer, const void* q, void* out,
                                void* cuda_stream) {
    if (!m || !kv || !p || kv->model != m || !plan_matches(p, kv) || !q || !out || layer >= m->desc.n_layers)
        return SYN_E_INVALID_ARG;
    const syn_model_desc& c = m->desc;
    const int q_dim = c.n_q_heads * c.head_dim;
    if (p->T > m->t_cap || p->n_parts > m->part_cap) return SYN_E_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
    // the Q tensor map is bound to the workspace buffer: stage the caller's q there
    CU_OK(cudaMemcpyAsync(m->q, q, (size_t)p->T * q_dim * 2, cudaMemcpyDeviceToDevice, st));
    return launch_attention(m, kv, p, layer, m->tm_q, (op16*)out, st);
}

// ------------------------------------------------------------------------------------------ no-allocation attention

// Scratch of syn_op_attention_static: the fp32 partial outputs and (max, sum) pairs of attention
// work items that cover only part of a request's keys, and the per-group completion counters.  File-scope device memory, so every GPU that
// loads the library holds these ~19.7 MB from load to exit: two partials of 64 rows for each of 296 CTAs (work lists cut where a
// CTA is full; half as many of 128 rows).  Host code may not pass these names to a
// kernel (on the host they are stand-ins, not device addresses): static_scratch() asks the runtime
// for the device addresses once per device.
static __device__ __align__(256) float g_static_part_o[(size_t)SYN_STATIC_MAX_PARTS * 64 * 128];
static __device__ __align__(256) float2 g_static_part_ml[(size_t)SYN_STATIC_MAX_PARTS * 64];
static __device__ __align__(256) int g_static_group_count[SYN_STATIC_MAX_PARTS];

static int static_scratch(float** part_o, float2** part_ml, int** group_count) {
    constexpr int MAX_DEV = 64;
    static float* o_of[MAX_DEV];
    static float2* ml_of[MAX_DEV];
    static int* cnt_of[MAX_DEV];
    static std::mutex lock;   // two host threads may make the first call on a device together
    int dev = -1;
    CU_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= MAX_DEV) return SYN_E_INVALID_ARG;
    std::lock_guard<std::mutex> hold(lock);
    if (!o_of[dev]) {   // first call on this device (which is current): resolve the symbols
        void *a = nullptr, *b = nullptr, *cn = nullptr;
        CU_OK(cudaGetSymbolAddress(&a, g_static_part_o));
        CU_OK(cudaGetSymbolAddress(&b, g_static_part_ml));
        CU_OK(cudaGetSymbolAddress(&cn, g_static_group_count));
        if (!a || !b || !cn) return SYN_E_CUDA;
        ml_of[dev] = static_cast<float2*>(b);
        cnt_of[dev] = static_cast<int*>(cn);
        o_of[dev] = static_cast<float*>(a);
    }
    *part_o = o_of[dev];
    *part_ml = ml_of[dev];
    *group_count = cnt_of[dev];
    return SYN_OK;
}

static int syn_op_attention_static_impl(syn_model* m, syn_kv* kv, const syn_plan* p, uint32_t layer, const void* q,
                                       void* out, void* cuda_stream) {
    if (!m || !kv || !p || kv->model != m || !plan_matches(p, kv) || !q || !out || layer >= m->desc.n_layers)
        return SYN_E_INVALID_ARG;
    const syn_model_desc& c = m->desc;
    const int q_dim = c.n_q_heads * c.head_dim;
    if (p->T > m->t_cap) return SYN_E_INVALID_ARG;
    if ((int64_t)p->n_parts * attn_rows(p->attn) > (int64_t)SYN_STATIC_MAX_PARTS * 64) return SYN_E_CAPACITY;
    float* part_o = nullptr;
    float2* part_ml = nullptr;
    int* group_count = nullptr;
    int r = static_scratch(&part_o, &part_ml, &group_count);
    if (r) return r;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
    CU_OK(cudaMemcpyAsync(m->q, q, (size_t)p->T * q_dim * 2, cudaMemcpyDeviceToDevice, st));
    // the group counters must start at zero; every partial row that is read is written first
    CU_OK(cudaMemsetAsync(group_count, 0, (size_t)SYN_STATIC_MAX_PARTS * 4, st));
    AttnParams ap;
    attn_params(ap, m, kv, p, layer, (op16*)out, part_o, part_ml, group_count);
    return attention_kernel(m, kv, p, ap, m->tm_q, false, st) == cudaSuccess ? SYN_OK : SYN_E_CUDA;
}

// The projection schedule without a device (tests): the launch shape, and work item i of CTA `cta`.
extern "C" int syn_gemm_plan_host(int32_t T, int32_t N, int32_t K, int32_t n_sm, int32_t epilogue, int32_t* out) {
    if (T <= 0 || N <= 0 || K <= 0 || n_sm <= 0 || n_sm > 65535 || epilogue < EPI_PLAIN || epilogue > EPI_LMHEAD || !out)
        return SYN_E_INVALID_ARG;
    GemmParams g;
    memset(&g, 0, sizeof(g));
    int n_cta = 0;
    const int r = gemm_plan(T, (N + 255) / 256 * 256, K, n_sm, epilogue, epilogue != EPI_RESID, g, n_cta);
    if (r) return r;
    const int v[SYN_GEMM_PLAN_FIELDS] = {g.n_pairs, g.n_tt, g.TN, g.num_kb, n_cta, g.pair_mode, g.splits, g.kb_per_split, g.ksplit, g.kper};
    memcpy(out, v, sizeof(v));
    return SYN_OK;
}

extern "C" int syn_gemm_work_host(int32_t T, int32_t N, int32_t K, int32_t n_sm, int32_t epilogue, int32_t cta, int32_t i,
                                  int32_t* out) {
    if (T <= 0 || N <= 0 || K <= 0 || n_sm <= 0 || n_sm > 65535 || epilogue < EPI_PLAIN || epilogue > EPI_LMHEAD || !out || i < 0)
        return SYN_E_INVALID_ARG;
    GemmParams g;
    memset(&g, 0, sizeof(g));
    int n_cta = 0;
    const int r = gemm_plan(T, (N + 255) / 256 * 256, K, n_sm, epilogue, epilogue != EPI_RESID, g, n_cta);
    if (r) return r;
    if (cta < 0 || cta >= n_cta) return SYN_E_INVALID_ARG;
    GemmWork w;
    const bool have = g.ksplit > 1 ? gemm_work<true>(g, cta, n_cta, i, w) : gemm_work<false>(g, cta, n_cta, i, w);
    if (!have) return 0;
    const int v[SYN_GEMM_WORK_FIELDS] = {w.pair, w.tt, w.mt_lo, w.mt_hi, w.kb0, w.kb1, w.split, w.role, w.rtile, w.hpart};
    memcpy(out, v, sizeof(v));
    return 1;
}


// ------------------------------------------------------------------------------------------ exported wrappers
// No C++ exception crosses the C ABI: the host code behind these entry points uses std::vector.
#define SYN_GUARD(call)                  \
    try {                                \
        return (call);                   \
    } catch (const std::bad_alloc&) {    \
        return SYN_E_OOM;                \
    } catch (...) {                      \
        return SYN_E_INVALID_ARG;        \
    }

extern "C" int syn_model_load(const syn_model_desc* desc, const syn_weights* w, syn_model** out) {
    SYN_GUARD(syn_model_load_impl(desc, w, out));
}

extern "C" int syn_kv_import(syn_kv* kv, uint32_t layer, const int32_t* page_table, int32_t pos0, int32_t n_pos, const void* k, const void* v, void* stream) {
    SYN_GUARD(syn_kv_import_impl(kv, layer, page_table, pos0, n_pos, k, v, stream));
}

extern "C" int syn_kv_export(syn_kv* kv, uint32_t layer, const int32_t* page_table, int32_t pos0, int32_t n_pos, void* k, void* v, void* stream) {
    SYN_GUARD(syn_kv_export_impl(kv, layer, page_table, pos0, n_pos, k, v, stream));
}

extern "C" int syn_plan_host(const syn_model_desc* desc, uint32_t n_pages, uint32_t page_size, int32_t n_sm, int32_t n_req, const int32_t* chunk_tokens, const int32_t* chunk_offsets, const int32_t* page_tables, int32_t max_pages, const int32_t* ctx_lens, const int32_t* n_uncached, int32_t* pos, int32_t* slot, int32_t* items, int32_t items_cap, int32_t* n_items, int32_t* cta_begin, int32_t* n_cta, syn_step_stats* stats) {
    SYN_GUARD(syn_plan_host_impl(desc, n_pages, page_size, n_sm, n_req, chunk_tokens, chunk_offsets, page_tables, max_pages, ctx_lens, n_uncached, pos, slot, items, items_cap, n_items, cta_begin, n_cta, stats));
}

extern "C" int syn_plan_work_host(const syn_model_desc* desc, uint32_t n_pages, uint32_t page_size, int32_t n_sm, int32_t n_req, const int32_t* chunk_tokens, const int32_t* chunk_offsets, const int32_t* page_tables, int32_t max_pages, const int32_t* ctx_lens, const int32_t* n_uncached, int32_t* items, int32_t items_cap, int32_t* n_items, int32_t* cta_begin, int32_t* n_cta, int32_t* attention, syn_step_stats* stats) {
    SYN_GUARD(syn_plan_work_host_impl(desc, n_pages, page_size, n_sm, n_req, chunk_tokens, chunk_offsets, page_tables, max_pages, ctx_lens, n_uncached, items, items_cap, n_items, cta_begin, n_cta, attention, stats));
}

extern "C" int syn_plan_create(syn_model* m, syn_kv* kv, int32_t n_req, const int32_t* chunk_tokens, const int32_t* chunk_offsets, const int32_t* page_tables, int32_t max_pages, const int32_t* ctx_lens, const int32_t* n_uncached, syn_plan** out) {
    SYN_GUARD(syn_plan_create_impl(m, kv, n_req, chunk_tokens, chunk_offsets, page_tables, max_pages, ctx_lens, n_uncached, out));
}

extern "C" int syn_verify_run(syn_model* m, syn_kv* kv, const syn_plan* p, int32_t* accept_len_dev, int32_t* correction_dev, int32_t* top1_dev, float* logits_out, void* cuda_stream) {
    SYN_GUARD(syn_verify_run_impl(m, kv, p, accept_len_dev, correction_dev, top1_dev, logits_out, cuda_stream));
}

extern "C" int syn_get_profile(syn_model* m, double* ms, int32_t* launches) {
    SYN_GUARD(syn_get_profile_impl(m, ms, launches));
}

extern "C" int syn_verify_batch(syn_model* m, syn_kv* kv, int32_t n_req, const int64_t* req_ids, const int32_t* chunk_tokens, const int32_t* chunk_offsets, const int32_t* page_tables, int32_t max_pages, const int32_t* ctx_lens, const int32_t* n_uncached, int32_t* accept_len, int32_t* correction_token, float* logits_out, void* cuda_stream) {
    const auto t0 = std::chrono::steady_clock::now();
    int r;
    try {
        r = syn_verify_batch_impl(m, kv, n_req, req_ids, chunk_tokens, chunk_offsets, page_tables, max_pages, ctx_lens, n_uncached, accept_len, correction_token, logits_out, cuda_stream);
    } catch (const std::bad_alloc&) {
        return SYN_E_OOM;
    } catch (...) {
        return SYN_E_INVALID_ARG;
    }
    if (m && m->profile) m->last_wall_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return r;
}

extern "C" int syn_verify_batch_sampled(syn_model* m, syn_kv* kv, int32_t n_req, const int64_t* req_ids, const int32_t* chunk_tokens, const int32_t* chunk_offsets, const int32_t* page_tables, int32_t max_pages, const int32_t* ctx_lens, const int32_t* n_uncached, const syn_sampling* cfg, const int32_t* slm_ids, const float* slm_probs, const float* rand_accept, const float* rand_sample, int32_t* accept_len, int32_t* correction_token, float* logits_out, void* cuda_stream) {
    const auto t0 = std::chrono::steady_clock::now();
    int r;
    try {
        r = syn_verify_batch_sampled_impl(m, kv, n_req, req_ids, chunk_tokens, chunk_offsets, page_tables, max_pages, ctx_lens, n_uncached, cfg, slm_ids, slm_probs, rand_accept, rand_sample, accept_len, correction_token, logits_out, cuda_stream);
    } catch (const std::bad_alloc&) {
        return SYN_E_OOM;
    } catch (...) {
        return SYN_E_INVALID_ARG;
    }
    if (m && m->profile) m->last_wall_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return r;
}

extern "C" int syn_op_sample_verify(const float* logits, int32_t T, int32_t vocab, int32_t n_req, const int32_t* chunk_tokens, const int32_t* chunk_offsets, const int32_t* n_uncached, const syn_sampling* cfg, const int32_t* slm_ids, const float* slm_probs, const float* rand_accept, const float* rand_sample, int32_t* accept_len, int32_t* correction_token, void* cuda_stream) {
    SYN_GUARD(syn_op_sample_verify_impl(logits, T, vocab, n_req, chunk_tokens, chunk_offsets, n_uncached, cfg, slm_ids, slm_probs, rand_accept, rand_sample, accept_len, correction_token, cuda_stream));
}

extern "C" int syn_op_attention(syn_model* m, syn_kv* kv, const syn_plan* p, uint32_t layer, const void* q, void* out, void* cuda_stream) {
    SYN_GUARD(syn_op_attention_impl(m, kv, p, layer, q, out, cuda_stream));
}

extern "C" int syn_op_attention_static(syn_model* m, syn_kv* kv, const syn_plan* p, uint32_t layer, const void* q, void* out, void* cuda_stream) {
    SYN_GUARD(syn_op_attention_static_impl(m, kv, p, layer, q, out, cuda_stream));
}

// The CTA-pair schedule without a device (tests).
extern "C" int syn_gemm2_plan_host(int32_t T, int32_t N, int32_t K, int32_t n_sm, int32_t epilogue, int32_t force, int32_t* out) {
    if (T <= 0 || N <= 0 || K <= 0 || n_sm <= 0 || n_sm > 65535 || epilogue < EPI_PLAIN || epilogue > EPI_LMHEAD || force < PAIR_NONE ||
        force > PAIR_DUO || !out)
        return SYN_E_INVALID_ARG;
    Gemm2Params g;
    int n_cl = 0;
    const int kind = gemm2_plan(T, (N + 255) / 256 * 256, K, n_sm, epilogue, force, g, n_cl);
    const int v[SYN_GEMM2_PLAN_FIELDS] = {kind, g.n_groups, g.n_tt, g.TN, g.num_kb, n_cl, g.splits, g.kb_per_split, g.rem_base, g.rem_extra};
    memcpy(out, v, sizeof(v));
    return SYN_OK;
}

extern "C" int syn_gemm2_work_host(int32_t T, int32_t N, int32_t K, int32_t n_sm, int32_t epilogue, int32_t force, int32_t cluster,
                                   int32_t i, int32_t* out) {
    if (T <= 0 || N <= 0 || K <= 0 || n_sm <= 0 || n_sm > 65535 || epilogue < EPI_PLAIN || epilogue > EPI_LMHEAD || force < PAIR_NONE ||
        force > PAIR_DUO || !out || i < 0)
        return SYN_E_INVALID_ARG;
    Gemm2Params g;
    int n_cl = 0;
    const int kind = gemm2_plan(T, (N + 255) / 256 * 256, K, n_sm, epilogue, force, g, n_cl);
    if (kind == PAIR_NONE || cluster < 0 || cluster >= n_cl) return SYN_E_INVALID_ARG;
    Gemm2Work w;
    if (!gemm2_work(g, cluster, n_cl, i, w)) return 0;
    const int v[SYN_GEMM2_WORK_FIELDS] = {w.grp, w.tt, w.kb0, w.kb1, w.tile, w.split, w.nsplit, w.first_cl, w.counter};
    memcpy(out, v, sizeof(v));
    return 1;
}

extern "C" int syn_thin_plan_host(int32_t T, int32_t N, int32_t K, int32_t n_sm, int32_t epilogue, int32_t* out) {
    if (T <= 0 || N <= 0 || K <= 0 || n_sm <= 0 || n_sm > 65535 || epilogue < EPI_PLAIN || epilogue > EPI_LMHEAD || !out) return SYN_E_INVALID_ARG;
    ThinParams g;
    thin_plan(T, (N + 127) / 128 * 128, K, n_sm, g);
    const int v[SYN_THIN_PLAN_FIELDS] = {thin_takes(T, (N + 127) / 128 * 128, K, n_sm, epilogue) ? 1 : 0, g.n_tiles, g.n_tt, g.TN, g.num_kb, g.splits, g.n_stages,
                                         g.n_stages * thin_stage_bytes(g.TN) - (g.splits > 1 && !g.recv_own ? thin_recv_bytes(g.TN, g.splits) : 0) - THIN_SCR_BYTES};
    memcpy(out, v, sizeof(v));
    return SYN_OK;
}

extern "C" const char* syn_last_cuda_error(void) { return g_last_cuda_error; }

extern "C" const char* syn_strerror(int code) {
    switch (code) {
        case SYN_OK: return "ok";
        case SYN_E_INVALID_ARG: return "invalid argument";
        case SYN_E_CHUNK_LEN: return "chunk length outside [1, 32]";
        case -20: return "scheduler: no live request with this id";
        case -21: return "scheduler: a live request with this id exists already";
        case -22: return "scheduler: the request cannot take this call in its present state";
        case -23: return "scheduler: commit without a peeked batch";
        case SYN_E_UNCACHED: return "n_uncached outside [1, chunk length]";
        case SYN_E_PAGE_OOB: return "page id out of range";
        case SYN_E_CAPACITY: return "context + chunk exceeds the page table";
        case SYN_E_TOKEN_OOB: return "token id out of range";
        case SYN_E_PAGE_ALIAS: return "two chunk tokens map to the same KV slot";
        case SYN_E_OOM: return "out of memory";
        case SYN_E_ARCH: return "device is not sm_100";
        case SYN_E_CUDA: return "CUDA call failed";
        case SYN_E_DEVICE_TIMEOUT: return "bounded device-side wait ran out";
        default: return "unknown error";
    }
}
