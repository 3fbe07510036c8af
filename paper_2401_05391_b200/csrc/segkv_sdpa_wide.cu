// Decode attention for work groups of many query columns (beams * query heads per kv head from 9 to 32) on the
// fifth-generation tensor cores (tcgen05 + tensor memory), head_dim 64, 128 or 256.  Same contract as the
// tiled kernel's separate form (paper Sections 3.2, 3.3): the prompt segment is read once for all columns of
// a (request, kv head), the response rows through the request's list of distinct rows, one softmax over both.
//
// What bounds it: HBM, once the columns share every key.  The tiled kernel keeps O^T of all columns in one
// warp's registers (mma.sync), which ends at 16 columns (8 at head_dim 256); beyond that the only kernel
// was the row-wise one, which reads the prompt once per beam and query head.
//
//  * one persistent CTA per SM walks the items (work group, split) round-robin;
//  * S[128 rows, KEYS] = Q.K^T with M = 128: the at most 32 query columns are the rows, REPEATED FOUR TIMES, so
//    that each of the four softmax warps finds all columns in its own tensor-memory lanes and takes a
//    quarter of the tile's keys (one column per lane, KEYS/4 keys per thread: no shuffles).  The repeated
//    rows cost MMA time the tensor pipe has to spare: 8 MMAs of 64 keys and 4 of 128 columns per 32 KB of keys
//    and values, 512 clocks of math in a tile of about 1250, the longer part of which is their issue and the waits
//    between; an SM's share of HBM bandwidth takes about 1300;
//  * the four warps agree on a column's maximum through shared memory (one barrier per tile, which also
//    carries the "a wait ran out" flag, so that all warps leave together) and write the weights P into ONE
//    shared-memory tile, the A operand of O[128, D] += P.V.  The weights keep what fp32 has of them: they go as the
//    sum of two fp16 or three bf16 parts, each part 32 rows of the same MMA, which has rows to spare, and the
//    parts of O are added up in the epilogue.  (One fp16 part: error against 64 bits 2.9e-4 of the result instead
//    of the 2.1e-4 that rounding the output takes; two bf16 parts: 1.65e-3, which is that rounding, but five times
//    as many outputs are not the nearest number, 0.25 %.)  Rows past the parts' are never read;
//  * O stays in tensor memory and is rescaled only when a column's maximum has grown by more than 2^8 over
//    the reference in use (sum and weights use the same reference, so the result is exact);
//  * prompt tiles arrive by TMA in one ring; response tiles are gathered row by row (cp.async into the same
//    128-byte-swizzled layout) by two groups of two warps, one stage each, so that two gathers are in
//    flight; the gather warps also stage the query block, which the softmax warps place in tensor memory;
//  * splits of a work group meet in the global workspace, the parts of each added up: the last CTA to arrive folds
//    them (as in the tiled kernel).
//  * an Inf or a NaN in a value row would reach the columns that do not read the row (their weight there is zero, and
//    zero times Inf is NaN), and a weight in parts makes a NaN of an Inf.  So the columns of a finished work group
//    whose output is not finite are worked out again one by one, from the rows that they read (segkv_rowwise.cuh), by
//    the softmax warps.  Without splits that is done at the end of the CTA's next item, where the warps meet anyhow.
// Every mbarrier is waited on phase by phase and every wait is bounded; on expiry the kernel flags
// SEGKV_DEV_WAIT_LIMIT, leaves the output alone and still releases its tensor memory and its tickets.
#include "segkv_internal.h"
#include "segkv_ptx.cuh"
#include "segkv_rowwise.cuh"
#include "segkv_tc5.cuh"

namespace segkv_impl {

namespace {

using namespace ptx;

constexpr int kTicketAbortedW = 1 << 16;     // same marker as the tiled kernel's
constexpr int kCols = kMaxCols;              // query columns of a work group, padded: one tensor-memory lane each

// Loads of the split merge, from the L2 (other SMs wrote the data), issued in program order.
__device__ __forceinline__ float4 ldcg4(const float4* a) {
    float4 v;
    asm volatile("ld.global.cg.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(a));
    return v;
}
__device__ __forceinline__ float2 ldcg2(const float2* a) {
    float2 v;
    asm volatile("ld.global.cg.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(a));
    return v;
}

struct WideParams {
    const void* q;
    void* out;
    const float* slopes;
    const char* kr;                // response K (V row = K row + vdelta)
    const char* const* k_chunks;   // growing capacity: chunk base pointers, chunk_steps steps each
    long long vdelta;
    const URow* ulist;
    const int32_t* ucount;
    const int32_t* plens;
    float* ws_o;                   // [item][ncols][D] un-normalised partial outputs
    float* ws_ml;                  // [item][ncols][2] reference maximum (base-2 domain) and sum
    int* tickets;
    int* err_word;
    int P, steps, S, W, G, H, Hkv, rows, max_steps, ncols, chunk_steps, items;
    int early_prompt, dbg_skip;
    unsigned long long wait_ns;
    float scale2;
    uint32_t idesc_qk, idesc_pv;
    rowwise::Args row;             // the same call, for columns that are not finite
};

// A softmax weight as a sum of 16-bit parts for the tensor cores, with what fp32 has of it: fp16 in two (22 bits), bf16
// in three cut off one behind the other (8 bits each: all 24).  fp16 weights carry a factor of 2^7 (the sum does
// too), so that parts below fp16's smallest number are 2^-31 of the largest weight and not 2^-24.
template <typename T> struct Parts;
template <> struct Parts<__half> {
    static constexpr int kNum = 2;
    static constexpr float kShift = 7.f;              // the largest weight is 2^8 times this factor: 2^15
    static __device__ __forceinline__ void split(float a, float c, uint32_t* w) {
        const __half2 h = __floats2half2_rn(a, c);
        const float2 f = __half22float2(h);
        w[0] = *reinterpret_cast<const uint32_t*>(&h);
        w[1] = ptx::Mma<__half>::pack(a - f.x, c - f.y);
    }
};
template <> struct Parts<__nv_bfloat16> {
    static constexpr int kNum = 3;
    static constexpr float kShift = 0.f;
    static __device__ __forceinline__ void split(float a, float c, uint32_t* w) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint32_t x = __float_as_uint(a), y = __float_as_uint(c);
            w[i] = __byte_perm(x, y, 0x7632);
            a -= __uint_as_float(x & 0xFFFF0000u);
            c -= __uint_as_float(y & 0xFFFF0000u);
        }
        w[2] = ptx::Mma<__nv_bfloat16>::pack(a, c);
    }
};

template <typename T, int D_>
struct WideLayout {
    static constexpr int D = D_;
    static constexpr int kParts = Parts<T>::kNum;
    static constexpr int KEYS = D == 256 ? 32 : 64;              // keys of a tile: one box of the prompt's tensor map
    static constexpr int KW = KEYS / 4;                          // keys of a softmax warp
    static constexpr int kDBoxes = D / 64;                       // 128-byte column blocks of a row
    static constexpr int kColTile = KEYS * 128;
    static constexpr int kTile = kDBoxes * kColTile;             // bytes of a K (or a V) tile
    static constexpr int kStage = 2 * kTile;
    static constexpr int SP = D == 64 ? 8 : 4;                   // prompt stages
    static constexpr int SR = 2;                                 // response stages: one per gather group
    static constexpr int kPRows = kParts * 32 * 128;             // weights of a tile: 32 rows of each part, 128 bytes each
    // two buffers of weights: tiles of 32 keys fill half a row each, and the other half is the other buffer
    static constexpr int kPBuf = KEYS == 32 ? 64 : kPRows;
    static constexpr int kP = KEYS == 32 ? kPRows : 2 * kPRows;
    static constexpr int kQ = kCols * D * 2;                     // the next query block, on its way to tensor memory
    static constexpr int kMeta = SR * KEYS * (int)sizeof(URow);
    static constexpr int kMax = 2 * 4 * kCols * 4, kSum = 4 * kCols * 4;
    static constexpr int kBars = 3 * SP + 2 * SR + 3 + 6 + 1;    // rings, query, S/P/O x 2, wind-down
    // the small arrays first, then, on a swizzle atom's boundary, weights, rings and the query block
    static constexpr int kSmall = (kMeta + kMax + kSum + 8 * kBars + 32 + 1023) & ~1023;
    static constexpr size_t kBytes = (size_t)kSmall + kP + (SP + SR) * kStage + kQ;
    // the parts of O meet in shared memory, where the weights were, XC of D at a time in two buffers in turn
    static constexpr int kXch = (kParts - 1) * kCols * 4;        // bytes of one of D
    static constexpr int XC = kP >= 64 * kXch ? 32 : 16;
    static_assert(2 * XC * kXch <= kP, "exchange of the parts");
    static_assert(rowwise::kScratch<D> * 4 <= kP, "columns that are worked out again");
    // tensor memory: two S buffers, O, and the query block (16-bit, two elements per column)
    static constexpr int kColO = 2 * KEYS, kColQ = kColO + D, kColEnd = kColQ + D / 2;
    static constexpr int kTmemCols = kColEnd <= 256 ? 256 : 512;
    static constexpr int kThreads = 320;                         // 4 softmax warps, TMA, MMA, 2 x 2 gather warps
    static_assert(kColEnd <= kTmemCols, "tensor memory");
    static_assert(kBytes <= 232448, "shared memory");
};

// The columns `mask` of a finished work group again, each from its own rows; all four softmax warps, the weights' place
// (s) free.  (Out of line: inlined it cost every launch about 1 us.)
template <typename T, int D>
__device__ __noinline__ void redo_columns(const rowwise::Args& a, int slab, uint32_t mask, float* s) {
    const int b = slab / a.Hkv, kvh = slab - b * a.Hkv;
    for (; mask; mask &= mask - 1) {
        const int col = __ffs(mask) - 1;
        rowwise::attend<T, D>(a, b * a.W + col / a.group, kvh * a.group + col % a.group, threadIdx.x >> 5, threadIdx.x & 31, s,
                              [] { bar_sync_n(1, 128); });
        bar_sync_n(1, 128);
    }
}

template <typename T, int D>
__global__ void __launch_bounds__(320, 1)
sdpa_wide_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ WideParams p) {
    using L = WideLayout<T, D>;
    constexpr int KEYS = L::KEYS, KW = L::KW, SP = L::SP, SR = L::SR;
    constexpr int kParts = L::kParts;
    extern __shared__ __align__(1024) uint8_t smem[];
    URow* meta = reinterpret_cast<URow*>(smem);
    float* s_max = reinterpret_cast<float*>(meta + SR * KEYS);    // [2][4 warps][kCols]
    float* s_sum = s_max + 2 * 4 * kCols;                         // [4 warps][kCols]
    uint64_t* bars = reinterpret_cast<uint64_t*>(s_sum + 4 * kCols);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + L::kBars);
    volatile int* s_flags = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int &s_abort = s_flags[0], &s_ticket = s_flags[1];
    uint32_t* s_bad = tmem_slot + 3;                              // [2] columns of an item that are not finite: item parity
    uint8_t* p_smem = smem + L::kSmall;                           // two buffers; their A operands reach into the ring behind
    uint8_t* p_ring = p_smem + L::kP;
    uint8_t* r_ring = p_ring + (size_t)SP * L::kStage;
    uint8_t* q_smem = r_ring + (size_t)SR * L::kStage;            // [32 rows][D], 16-byte chunks XOR-swizzled by the row
    const uint32_t pfull = smem_u32(bars), kempty = pfull + 8 * SP, vempty = kempty + 8 * SP;
    const uint32_t rfull = vempty + 8 * SP, rempty = rfull + 8 * SR, qfull = rempty + 8 * SR;
    const uint32_t sfull = qfull + 8, sempty = sfull + 8;         // the query block in shared memory
    const uint32_t bar_s = sempty + 8, bar_p = bar_s + 16, bar_o = bar_p + 16;     // two each: tile parity
    const uint32_t bar_end = bar_o + 16;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // One item: the split's share of a work group (prompt tiles, and a range of the request's distinct rows)
    struct Item { int slab, split, b, kvh, P, pt0, npt; };
    auto item_of = [&](int it) {
        Item x;
        x.slab = it / p.S;
        x.split = it - x.slab * p.S;
        x.b = x.slab / p.Hkv;
        x.kvh = x.slab - x.b * p.Hkv;
        x.P = p.plens ? __ldg(p.plens + x.b) : p.P;
        const int ntp = (x.P + KEYS - 1) / KEYS;
        x.pt0 = (int)((long long)x.split * ntp / p.S);
        x.npt = (int)((long long)(x.split + 1) * ntp / p.S) - x.pt0;
        return x;
    };
    // the distinct rows of an item's request; asked for one item ahead
    auto count_of = [&](int it) { return p.steps > 0 && it < p.items ? p.ucount[it / p.S / p.Hkv] : 0; };
    auto rows_of = [&](const Item& x, int n_b, int& e0, int& e1) {
        const int each = n_b / p.S, left = n_b - each * p.S;      // beams that stay apart have up to beams * steps rows
        e0 = x.split * each + min(x.split, left);
        e1 = e0 + each + (x.split < left ? 1 : 0);
    };
    // the K (or V) part of the item's prompt tile k
    auto issue_part = [&](const CUtensorMap* tm, const Item& x, int k, uint32_t dst, uint32_t full) {
        mbar_arrive_expect_tx(full, (uint32_t)L::kTile);
#pragma unroll
        for (int bx = 0; bx < L::kDBoxes; ++bx) tma_load_4d(dst + bx * L::kColTile, tm, bx * 64, x.kvh, (x.pt0 + k) * KEYS, x.b, full);
    };
    const uint32_t p_ring_u = smem_u32(p_ring), r_ring_u = smem_u32(r_ring);

    // Set-up by the TMA warp, which then goes straight to its prompt tiles (when nothing can still be writing the
    // prompt, before the previous kernel has finished).
    if (warp == 4) {
        if (lane == 0) {
            for (int s = 0; s < SP; ++s) {
                mbar_init(pfull + 8 * s, 2);                      // the K part and the V part
                mbar_init(kempty + 8 * s, 1);
                mbar_init(vempty + 8 * s, 1);
            }
            for (int s = 0; s < SR; ++s) {
                mbar_init(rfull + 8 * s, 1);
                mbar_init(rempty + 8 * s, 1);
            }
            mbar_init(qfull, 128);
            mbar_init(sfull, 128);
            mbar_init(sempty, 128);
            for (int i = 0; i < 2; ++i) {
                mbar_init(bar_s + 8 * i, 1);
                mbar_init(bar_p + 8 * i, 128);
                mbar_init(bar_o + 8 * i, 1);
            }
            mbar_init(bar_end, 1);
            s_abort = 0;
            s_bad[0] = s_bad[1] = 0u;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            fence_proxy_async();
        }
        __syncwarp();
        asm volatile("barrier.cta.arrive 5, %0;" ::"n"(L::kThreads) : "memory");    // the others go on; this warp needs nothing of theirs
    } else {
        if (warp == 5) {                 // this warp owns the tensor memory
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                         ::"r"(smem_u32(tmem_slot)), "n"(L::kTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        tc_fence_before();
        bar_sync_n(5, L::kThreads);
        tc_fence_after();
    }
    const uint32_t tmem = warp == 4 ? 0u : *tmem_slot;
    if (warp != 4) {
        // everything but the prompt tiles follows the previous kernel; its successors are let go only after that
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }

    if (warp == 4) {
        // ------------------------------- prompt tiles (TMA) -------------------------------
        if (lane == 0) {
            uint32_t pos = 0;
            bool ok = true;
            if (!p.early_prompt) asm volatile("griddepcontrol.wait;" ::: "memory");
            for (int it = blockIdx.x; it < p.items && ok; it += gridDim.x) {
                const Item x = item_of(it);
                for (int k = 0; k < x.npt; ++k, ++pos) {
                    const uint32_t st = pos % SP, ph = ((pos / SP) & 1) ^ 1, dst = p_ring_u + st * (uint32_t)L::kStage;
                    ok = mbar_wait(kempty + 8 * st, ph, p.wait_ns);
                    if (!ok) break;
                    issue_part(&tm_k, x, k, dst, pfull + 8 * st);
                    ok = mbar_wait(vempty + 8 * st, ph, p.wait_ns);
                    if (!ok) break;
                    issue_part(&tm_v, x, k, dst + L::kTile, pfull + 8 * st);
                }
            }
            if (!ok) {
                s_abort = 1;
                // copies in flight land first (or the limit runs out: a K part may have been asked for without its V part)
                for (uint32_t k = pos > (uint32_t)SP ? pos - SP : 0; k <= pos; ++k)
                    (void)mbar_wait(pfull + 8 * (k % SP), (k / SP) & 1, p.wait_ns);
            }
        }
    } else if (warp == 5) {
        // -------------------------------- MMA issuer --------------------------------
        // (the whole warp runs this, converged: see tc_mma_ss_if.  What decides the control flow is made uniform by
        // a warp reduction or vote.)
        const uint32_t lead = elect_one();
        const uint32_t p_lo = (smem_u32(p_smem) & 0x3FFFFu) >> 4, ring_lo = (p_ring_u & 0x3FFFFu) >> 4, resp_lo = (r_ring_u & 0x3FFFFu) >> 4;
        const uint64_t dk = smem_desc(0, 16, 1024), dv = smem_desc(0, L::kColTile, 1024);     // descriptors without an address
        uint32_t n = 0, qi = 0, ps = 0, pph = 0, rs = 0, rph = 0;   // tiles, items; prompt / response stage and phase of the next tile
        bool ok = true;
        auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
            return __all_sync(0xffffffffu, mbar_wait_hot(bar, parity, p.wait_ns));
        };
        int n_next = count_of((int)blockIdx.x);
        for (int it = blockIdx.x; it < p.items && ok; it += gridDim.x) {
            const Item x = item_of(it);
            int e0, e1;
            rows_of(x, n_next, e0, e1);
            n_next = count_of(it + (int)gridDim.x);
            const int npt = (int)__reduce_max_sync(0xffffffffu, (unsigned)x.npt);
            const int tiles = npt + (int)__reduce_max_sync(0xffffffffu, (unsigned)((e1 - e0 + KEYS - 1) / KEYS));
            if (tiles == 0) continue;
            uint32_t v_lo = 0, v_empty = 0;                       // the V part of the tile whose scores were issued last
            auto issue_qk = [&](int t, uint32_t buf) -> bool {
                const bool prompt = t < npt;
                const uint32_t lo = prompt ? ring_lo + ps * (uint32_t)(L::kStage >> 4) : resp_lo + rs * (uint32_t)(L::kStage >> 4);
                const uint32_t full = prompt ? pfull + 8 * ps : rfull + 8 * rs, par = prompt ? pph : rph;
                v_lo = lo + (uint32_t)(L::kTile >> 4);
                v_empty = prompt ? vempty + 8 * ps : rempty + 8 * rs;
                if (!wait(full, par)) return false;
                tc_fence_after();
                const uint64_t kd = dk + lo;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks)
                    tc_mma_ts_if(lead, tmem + buf * KEYS, tmem + L::kColQ + ks * 8,
                                 kd + (uint64_t)(((ks >> 2) * L::kColTile + (ks & 3) * 32) >> 4), p.idesc_qk, ks > 0);
                tc_commit_if(lead, bar_s + 8 * buf);
                if (prompt) {
                    tc_commit_if(lead, kempty + 8 * ps);
                    if (++ps == SP) { ps = 0; pph ^= 1u; }
                } else if (++rs == SR) { rs = 0; rph ^= 1u; }
                return true;
            };
            ok = wait(qfull, qi & 1);
            ++qi;
            if (ok) ok = issue_qk(0, n & 1);
            if (!ok) break;
            for (int t = 0; t < tiles; ++t, ++n) {
                const uint32_t buf = n & 1, lo = v_lo, empty = v_empty;
                if (t + 1 < tiles) {                              // the next scores run under this tile's softmax
                    ok = issue_qk(t + 1, buf ^ 1);
                    if (!ok) break;
                }
                ok = wait(bar_p + 8 * buf, (n >> 1) & 1);
                if (!ok) break;
                tc_fence_after();
                const uint64_t pd = dk + (p_lo + buf * (uint32_t)(L::kPBuf >> 4)), vd = dv + lo;
#pragma unroll
                for (int kk = 0; kk < KEYS / 16; ++kk)            // O += P[:, 16 keys] . V[16 keys, :]
                    tc_mma_ss_if(lead, tmem + L::kColO, pd + (uint64_t)((kk * 32) >> 4), vd + (uint64_t)((kk * 2048) >> 4),
                                 p.idesc_pv, t > 0 || kk > 0);
                tc_commit_if(lead, bar_o + 8 * buf);
                tc_commit_if(lead, empty);
            }
        }
        if (!ok && lane == 0) s_abort = 1;
    } else if (warp >= 6) {
        // ------------------- the query block, and response tiles: index select fused into the load -------------------
        const int grp = (warp - 6) >> 1, gt = tid - 192 - grp * 64, bid = 2 + grp;
        constexpr int CPR = D / 8;                                // 16-byte chunks per row
        constexpr int RW = KEYS / 2, RPI = 32 / CPR;              // rows of a tile that a warp fetches, and how many at once
        const size_t slab_bytes = (size_t)p.rows * p.Hkv * (size_t)(D * 2);
        uint8_t* stage = r_ring + (size_t)grp * L::kStage;        // the group's stage
        const int wrow = (gt >> 5) * RW;                          // the warp's first row
        URow* meta_g = meta + grp * KEYS;
        uint32_t rn = 0, qi = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < p.items && ok; it += gridDim.x) {
            const Item x = item_of(it);
            const int n_b = count_of(it);
            // this thread's share of the query block: whole rows side by side; rows past the last column are zeros
            constexpr int QI = kCols * CPR / 128;
            uint4 w[QI];
#pragma unroll
            for (int i = 0; i < QI; ++i) {
                const int col = (i * 128 + tid - 192) / CPR, c = (tid - 192) % CPR;
                w[i] = make_uint4(0u, 0u, 0u, 0u);
                if (col < p.ncols)
                    w[i] = *reinterpret_cast<const uint4*>(reinterpret_cast<const T*>(p.q) +
                               ((size_t)(x.b * p.W + col / p.G) * p.H + x.kvh * p.G + col % p.G) * D + c * 8);
            }
            ok = mbar_wait(sempty, (qi & 1) ^ 1, p.wait_ns);
            ok = bar_and(bid, 64, ok);
            if (!ok) break;
            ++qi;
#pragma unroll
            for (int i = 0; i < QI; ++i) {
                const int col = (i * 128 + tid - 192) / CPR, c = (tid - 192) % CPR;
                *reinterpret_cast<uint4*>(q_smem + (size_t)col * (D * 2) + ((c ^ (col & 7)) << 4)) = w[i];
            }
            mbar_arrive(sfull);
            int e0, e1;
            rows_of(x, n_b, e0, e1);
            const int nrt = (e1 - e0 + KEYS - 1) / KEYS;
            const URow* list = p.ulist + (size_t)x.b * p.W * p.max_steps;
            for (int r = 0; r < nrt; ++r) {
                const uint32_t pos = rn + (uint32_t)r;
                if ((pos & 1) != (uint32_t)grp) continue;         // the other group's tile
                const int eb = e0 + r * KEYS, cnt = min(KEYS, e1 - eb);
                URow u = {0, 0u};                                 // lane i < RW: the warp's row i
                if (lane < RW && wrow + lane < cnt) u = list[eb + wrow + lane];
                ok = mbar_wait(rempty + 8 * grp, ((pos >> 1) & 1) ^ 1, p.wait_ns);
                ok = bar_and(bid, 64, ok);
                if (!ok) break;
                unsigned long long row_at;
                {
                    const int s = u.row / p.rows;
                    const char* base = p.chunk_steps == 0 ? p.kr + (size_t)s * slab_bytes
                                                          : p.k_chunks[s / p.chunk_steps] + (size_t)(s % p.chunk_steps) * slab_bytes;
                    row_at = (unsigned long long)(base + ((size_t)(u.row - s * p.rows) * p.Hkv + x.kvh) * (size_t)(D * 2));
                    u.row = s;                                    // the softmax threads need the step only
                    if (lane < RW) meta_g[wrow + lane] = u;       // (no beam reads the padding of the last tile)
                }
                const int c = lane % CPR;
                uint8_t* dst0 = stage + (size_t)(c >> 3) * L::kColTile;
#pragma unroll 4
                for (int i = 0; i < RW / RPI; ++i) {
                    const int row = i * RPI + lane / CPR, key = wrow + row;
                    const char* src = reinterpret_cast<const char*>(__shfl_sync(0xffffffffu, row_at, row)) + c * 16;
                    uint8_t* dst = dst0 + key * 128 + (((c & 7) ^ (key & 7)) << 4);
                    if (key < cnt) {
                        cp_async_16(smem_u32(dst), src);
                        cp_async_16(smem_u32(dst + L::kTile), src + p.vdelta);
                    } else {                                      // a weight of zero times whatever was here need not be zero
                        *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
                        *reinterpret_cast<uint4*>(dst + L::kTile) = make_uint4(0u, 0u, 0u, 0u);
                    }
                }
                cp_async_wait_all();
                fence_proxy_async();
                bar_sync_n(bid, 64);
                if (gt == 0) mbar_arrive(rfull + 8 * grp);
            }
            rn += (uint32_t)nrt;
        }
        if (!ok && gt == 0) s_abort = 1;
    } else {
        // ---------------------- softmax warps: one column per lane, a quarter of the keys per warp ----------------------
        const uint32_t tm_lane = tmem + ((uint32_t)(warp * 32) << 16);
        const uint32_t tm_o = tm_lane + (uint32_t)L::kColO;
        const bool owns_o = warp < kParts;                        // the first part's rows of O are 0..31, the second's 32..63, ...
        const bool real = lane < p.ncols;
        const int beam = real ? lane / p.G : 0, hg = real ? lane % p.G : 0;
        const uint32_t beambit = real ? 1u << beam : 0u;
        uint32_t n = 0, rn = 0, qi = 0;                           // tiles, response tiles and items so far
        // The next item's query block, from shared memory into this warp's lanes of tensor memory (one column's row per
        // lane).  An item without any tile (a split beyond a request's keys) uses none.
        auto place_query = [&](bool used) -> bool {
            bool got = mbar_wait_hot(sfull, qi & 1, p.wait_ns);
            got = __all_sync(0xffffffffu, got);
            if (!got) return false;
            ++qi;
            if (used) {
#pragma unroll 1
                for (int c0 = 0; c0 < D / 8; c0 += 8) {           // 8 chunks of 16 bytes (32 columns) at a time
                    uint4 w[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        w[i] = *reinterpret_cast<const uint4*>(q_smem + (size_t)lane * (D * 2) + (((c0 + i) ^ (lane & 7)) << 4));
                    tc_st32(tm_lane + L::kColQ + c0 * 4, reinterpret_cast<const uint32_t*>(w));
                }
                tc_wait_st();
                tc_fence_before();
                mbar_arrive(qfull);
            }
            mbar_arrive(sempty);
            return true;
        };
        auto share_of = [&](int i, int n_b, Item& x) {            // item i and its response tiles
            x = item_of(i);
            int e0, e1;
            rows_of(x, n_b, e0, e1);
            return (e1 - e0 + KEYS - 1) / KEYS;
        };
        uint32_t items_done = 0;
        int slab_before = 0;                                      // work group of the item before, without splits
        bool gone = false;                                        // the four warps have agreed to leave: a wait ran out
        int it = blockIdx.x;
        Item x;
        int nrt = share_of(it, count_of(it), x);
        bool ok = place_query(x.npt + nrt > 0);
        while (it < p.items) {
            const int tiles = x.npt + nrt, it_next = it + (int)gridDim.x;
            const int n_next = count_of(it_next);
            const float slope2 = (p.slopes && real) ? p.slopes[x.kvh * p.G + hg] * 1.4426950408889634f : 0.f;
            const int qpos = x.P + (p.steps > 0 ? p.steps - 1 : -1);
            float m_ref = -INFINITY, l_run = 0.f;
            for (int t = 0; t < tiles; ++t, ++n) {
                const uint32_t buf = n & 1;
                const bool resp = t >= x.npt;
                const uint32_t rpos = rn + (uint32_t)(t - x.npt);
                if (ok && resp) ok = mbar_wait_hot(rfull + 8 * (rpos % SR), (rpos / SR) & 1, p.wait_ns);   // the tile's records
                if (ok) ok = mbar_wait_hot(bar_s + 8 * buf, (n >> 1) & 1, p.wait_ns);
                ok = __all_sync(0xffffffffu, ok);
                float v[KW];
                float tmax = -INFINITY;
                if (ok) {
                    tc_fence_after();
                    uint32_t sr[KW];
                    if (KW == 16) tc_ld16(tm_lane + buf * KEYS + warp * KW, sr);
                    else tc_ld8(tm_lane + buf * KEYS + warp * KW, sr);
                    tc_wait_ld();
                    pin<KW>(sr);
                    if (!resp) {
                        const int key0 = (x.pt0 + t) * KEYS + warp * KW, left = x.P - key0;      // keys past the prompt are masked
                        const float bias0 = slope2 * (float)(key0 - qpos);
#pragma unroll
                        for (int i = 0; i < KW; ++i) {
                            v[i] = fmaf(__uint_as_float(sr[i]), p.scale2, fmaf(slope2, (float)i, bias0));
                            if (i >= left) v[i] = -INFINITY;
                        }
                    } else {
                        const URow* mt = meta + (rpos % SR) * KEYS + warp * KW;
#pragma unroll
                        for (int i = 0; i < KW; ++i) {
                            const int2 u = *reinterpret_cast<const int2*>(mt + i);                  // {step, beams that read the row}
                            v[i] = fmaf(__uint_as_float(sr[i]), p.scale2, slope2 * (float)(x.P + u.x - qpos));
                            if (!((uint32_t)u.y & beambit)) v[i] = -INFINITY;
                        }
                    }
                    float tm[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
                    for (int i = 4; i < KW; ++i) tm[i & 3] = fmaxf(tm[i & 3], v[i]);
                    tmax = fmaxf(fmaxf(tm[0], tm[1]), fmaxf(tm[2], tm[3]));
                }
                // The reference in use nearly always stands, so the weights are worked out with it before the warps
                // meet; that one of them needs a new one is found at the meeting.
                float ls[2];
                uint32_t wp[kParts][KW / 2];
                auto weigh = [&]() {
                    const float m_use = m_ref == -INFINITY ? 0.f : m_ref - Parts<T>::kShift;    // no key of this column so far
                    ls[0] = ls[1] = 0.f;
#pragma unroll
                    for (int i = 0; i < KW; i += 2) {
                        const float a = exp2f(v[i] - m_use), c = exp2f(v[i + 1] - m_use);
                        ls[(i >> 1) & 1] += a + c;
                        uint32_t w[kParts];
                        Parts<T>::split(a, c, w);
#pragma unroll
                        for (int k = 0; k < kParts; ++k) wp[k][i >> 1] = w[k];
                    }
                };
                if (ok) weigh();
                bool need = tmax > m_ref + 8.f;
                float alpha = 1.f;
                if (!bar_and(1, 128, ok && !need)) {
                    s_max[(buf * 4 + warp) * kCols + lane] = tmax;
                    ok = bar_and(1, 128, ok);                     // everybody's maxima are there, or everybody leaves
                    gone = !ok;
                    if (gone) break;
#pragma unroll
                    for (int w = 0; w < 4; ++w) tmax = fmaxf(tmax, s_max[(buf * 4 + w) * kCols + lane]);
                    need = tmax > m_ref + 8.f;
                    if (need) {
                        alpha = exp2f(m_ref - tmax);              // 0 on the first keys
                        m_ref = tmax;
                    }
                    weigh();
                }
                l_run = l_run * alpha + (ls[0] + ls[1]);
                // (The buffer the weights go to is free: these scores were issued behind P.V of the tile before last.)
                if (t > 0 && owns_o && __any_sync(0xffffffffu, need)) {
                    ok = mbar_wait_hot(bar_o + 8 * (buf ^ 1), ((n - 1) >> 1) & 1, p.wait_ns);
                    ok = __all_sync(0xffffffffu, ok);
                    if (ok) {
                        tc_fence_after();
#pragma unroll 1
                        for (int c = 0; c < D / 32; ++c) {
                            uint32_t o[32];
                            tc_ld32(tm_o + c * 32, o);
                            tc_wait_ld();
                            pin<32>(o);
#pragma unroll
                            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                            tc_st32(tm_o + c * 32, o);
                        }
                        tc_wait_st();
                    }
                }
                if (ok) {
                    uint8_t* dst = p_smem + (KEYS == 32 ? 0 : buf * L::kPBuf) + lane * 128;
#pragma unroll
                    for (int c = 0; c < KW / 8; ++c) {
                        const int ch = (((KEYS == 32 ? 4 * (int)buf : 0) + warp * (KW / 8) + c) ^ (lane & 7)) << 4;
#pragma unroll
                        for (int k = 0; k < kParts; ++k)
                            *reinterpret_cast<uint4*>(dst + k * (32 * 128) + ch) = make_uint4(wp[k][4 * c], wp[k][4 * c + 1], wp[k][4 * c + 2], wp[k][4 * c + 3]);
                    }
                    fence_proxy_async();
                    tc_fence_before();
                    if (!(p.dbg_skip && tid == 0 && n == 0)) mbar_arrive(bar_p + 8 * buf);
                }
            }
            if (gone) break;
            // the next item's query, whose first scores then run under this item's epilogue (this item's scores are all done)
            ok = __all_sync(0xffffffffu, ok);
            const Item done = x;
            const int done_nrt = nrt;
            if (it_next < p.items) {
                nrt = share_of(it_next, n_next, x);
                if (ok) ok = place_query(x.npt + nrt > 0);
            }
            // ---- the item's result: sums over the warps, O once its last P.V is done ----
            s_sum[warp * kCols + lane] = l_run;
            if (tiles > 0 && ok) ok = mbar_wait_hot(bar_o + 8 * ((n - 1) & 1), ((n - 1) >> 1) & 1, p.wait_ns);
            ok = bar_and(1, 128, ok);
            gone = !ok;
            if (gone) break;
            tc_fence_after();
            float l = 0.f;
#pragma unroll
            for (int w = 0; w < 4; ++w) l += s_sum[w * kCols + lane];
            rn += (uint32_t)done_nrt;
            if (p.S == 1 && s_bad[(items_done & 1) ^ 1]) {
                redo_columns<T, D>(p.row, slab_before, s_bad[(items_done & 1) ^ 1], reinterpret_cast<float*>(p_smem));
                if (tid == 0) s_bad[(items_done & 1) ^ 1] = 0u;
            }
            slab_before = done.slab;
            // One row per lane: the parts come over to the first warp, the small ones first (they are worked out from what
            // the larger ones left), and go out as the output rows, or as a split's partial.
            if (owns_o) {
                T* orow = reinterpret_cast<T*>(p.out) + ((size_t)(done.b * p.W + beam) * p.H + done.kvh * p.G + hg) * D;
                float* wrow = p.ws_o + ((size_t)it * p.ncols + lane) * D;
                const float inv = 1.f / l;
                bool bad = false;
                if (p.S > 1 && warp == 0 && real)
                    *reinterpret_cast<float2*>(p.ws_ml + ((size_t)it * p.ncols + lane) * 2) = make_float2(m_ref, l);
#pragma unroll 1
                for (int d0 = 0; d0 < D; d0 += L::XC) {
                    float* xch = reinterpret_cast<float*>(p_smem) + ((d0 / L::XC) & 1) * (L::XC * L::kXch / 4);   // [part][XC][32 columns]
                    uint32_t o[L::XC];
                    if constexpr (L::XC == 32) tc_ld32(tm_o + d0, o);
                    else tc_ld16(tm_o + d0, o);
                    tc_wait_ld();
                    pin<L::XC>(o);
                    if (warp > 0) {
#pragma unroll
                        for (int i = 0; i < L::XC; ++i) xch[((warp - 1) * L::XC + i) * kCols + lane] = __uint_as_float(o[i]);
                    }
                    bar_sync_n(4, 32 * kParts);
                    if (warp > 0) continue;
                    float f[L::XC];
#pragma unroll
                    for (int i = 0; i < L::XC; ++i) {
                        float low = 0.f;
#pragma unroll
                        for (int k = kParts - 2; k >= 0; --k) low += xch[(k * L::XC + i) * kCols + lane];
                        f[i] = tiles > 0 ? __uint_as_float(o[i]) + low : 0.f;              // (a split without keys has no O)
                    }
                    if (real && p.S > 1) {
#pragma unroll
                        for (int i = 0; i < L::XC; i += 4) *reinterpret_cast<float4*>(wrow + d0 + i) = make_float4(f[i], f[i + 1], f[i + 2], f[i + 3]);
                    } else if (real) {
#pragma unroll
                        for (int i = 0; i < L::XC; ++i) {
                            f[i] *= inv;
                            bad |= !(fabsf(f[i]) < INFINITY);
                        }
#pragma unroll
                        for (int i = 0; i < L::XC; i += 8)
                            *reinterpret_cast<uint4*>(orow + d0 + i) = make_uint4(Mma<T>::pack(f[i], f[i + 1]), Mma<T>::pack(f[i + 2], f[i + 3]),
                                                                                  Mma<T>::pack(f[i + 4], f[i + 5]), Mma<T>::pack(f[i + 6], f[i + 7]));
                    }
                }
                const uint32_t mask = __ballot_sync(0xffffffffu, bad);
                if (p.S == 1 && tid == 0 && mask) s_bad[items_done & 1] = mask;     // read behind the next meeting
            }
            ++items_done;
            const int it_done = it;
            it = it_next;
            if (p.S == 1) continue;
            // ---- split merge: the last CTA of the work group to arrive folds all partials ----
            bar_sync_n(1, 128);
            if (tid == 0) {
                // (the partials are ordered before by the barrier; acq_rel publishes them)
                int ticket;
                asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(ticket) : "l"(p.tickets + done.slab) : "memory");
                const bool last = (ticket & (kTicketAbortedW - 1)) == p.S - 1;
                s_ticket = last ? 1 + (ticket >= kTicketAbortedW ? 1 : 0) : 0;
                if (last) p.tickets[done.slab] = 0;              // everybody has arrived: ready for the next launch
            }
            bar_sync_n(1, 128);
            const int verdict = s_ticket;
            bar_sync_n(1, 128);
            if (verdict != 1) continue;                       // not the last, or a CTA of the group gave up: no merge
            const int it0 = it_done - done.split;
            const float2* ml0 = reinterpret_cast<const float2*>(p.ws_ml + (size_t)it0 * p.ncols * 2);
            const float* o0 = p.ws_o + (size_t)it0 * p.ncols * D;
            const int parts = p.S;
            // A CTA without further items has its prompt ring free (all tiles in it have been used): if they fit, all partials are
            // on their way there at once while the factors are worked out.  (Merging four splits of 32 columns at D 128, 64 KB,
            // by 16 loads per thread at a time took 4.6 us, by 8 6.4: the loads' latency.)
            constexpr int D4 = D / 4, NE = 4;
            const int n4 = p.ncols * D4;
            const bool landed = it >= p.items && (size_t)parts * n4 * 16 <= (size_t)SP * L::kStage;
            const float4* land = reinterpret_cast<const float4*>(p_ring);
            if (landed)
                for (int i = tid; i < parts * n4; i += 128) cp_async_16(p_ring_u + 16 * i, reinterpret_cast<const float4*>(o0) + i);
            // Two passes: each part's factor per column, then 16 loads in flight per thread.  (One float4 of one column at
            // a time, its parts' loads ordered by the use of each, cost most of the about 7 us that merging four splits took.)
            float* fac = reinterpret_cast<float*>(p_smem);        // [part][32 columns]: 2^(m_part - m) / sum
            if (warp == 0 && real) {
                float mm = -INFINITY, ll = 0.f;
                for (int s0 = 0; s0 < parts; s0 += 8) {
                    float2 ml[8];
                    float bm = mm;
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        ml[u] = ldcg2(ml0 + (size_t)min(s0 + u, parts - 1) * p.ncols + lane);
                        if (s0 + u >= parts) ml[u] = make_float2(-INFINITY, 0.f);
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) bm = fmaxf(bm, ml[u].x);
                    ll *= mm == -INFINITY ? 0.f : exp2f(mm - bm);
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        ll += ml[u].x == -INFINITY ? 0.f : ml[u].y * exp2f(ml[u].x - bm);
                        if (s0 + u < parts) fac[(s0 + u) * kCols + lane] = ml[u].x;
                    }
                    mm = bm;
                }
                const float inv = 1.f / ll;
                for (int u = 0; u < parts; ++u) {
                    const float m = fac[u * kCols + lane];
                    fac[u * kCols + lane] = m == -INFINITY ? 0.f : exp2f(m - mm) * inv;
                }
            }
            if (landed) cp_async_wait_all();
            bar_sync_n(1, 128);
            for (int e0 = tid; e0 < n4; e0 += 128 * NE) {
                float4 o[NE];
#pragma unroll
                for (int i = 0; i < NE; ++i) o[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
                for (int s0 = 0; s0 < parts && landed; ++s0)
#pragma unroll
                    for (int i = 0; i < NE; ++i) {
                        const int e = min(e0 + 128 * i, n4 - 1);
                        const float4 w = land[s0 * n4 + e];
                        const float f = fac[s0 * kCols + e / D4];
                        o[i].x += w.x * f; o[i].y += w.y * f; o[i].z += w.z * f; o[i].w += w.w * f;
                    }
#pragma unroll 1
                for (int s0 = 0; s0 < parts && !landed; s0 += 4) {
                    float4 w[NE][4];
#pragma unroll
                    for (int i = 0; i < NE; ++i)
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            w[i][u] = ldcg4(reinterpret_cast<const float4*>(o0) + (size_t)min(s0 + u, parts - 1) * n4 + min(e0 + 128 * i, n4 - 1));
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (s0 + u >= parts) break;
#pragma unroll
                        for (int i = 0; i < NE; ++i) {
                            const float f = fac[(s0 + u) * kCols + min(e0 + 128 * i, n4 - 1) / D4];
                            o[i].x += w[i][u].x * f; o[i].y += w[i][u].y * f; o[i].z += w[i][u].z * f; o[i].w += w[i][u].w * f;
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < NE; ++i) {
                    const int e = e0 + 128 * i, col = e / D4, d = (e % D4) * 4;
                    if (e >= n4) break;
                    if (!(fabsf(o[i].x) + fabsf(o[i].y) + fabsf(o[i].z) + fabsf(o[i].w) < INFINITY)) atomicOr(&s_bad[0], 1u << col);
                    T* orow = reinterpret_cast<T*>(p.out) + ((size_t)(done.b * p.W + col / p.G) * p.H + done.kvh * p.G + col % p.G) * D + d;
                    *reinterpret_cast<uint2*>(orow) = make_uint2(Mma<T>::pack(o[i].x, o[i].y), Mma<T>::pack(o[i].z, o[i].w));
                }
            }
            bar_sync_n(1, 128);                                   // the factors' place takes weights again
            if (const uint32_t mask = s_bad[0]) {
                redo_columns<T, D>(p.row, done.slab, mask, reinterpret_cast<float*>(p_smem));
                if (tid == 0) s_bad[0] = 0u;
                bar_sync_n(1, 128);
            }
        }
        if (!gone && p.S == 1) {                                  // the last item's
            bar_sync_n(1, 128);
            if (const uint32_t mask = s_bad[(items_done & 1) ^ 1]) redo_columns<T, D>(p.row, slab_before, mask, reinterpret_cast<float*>(p_smem));
        }
        if (gone) {
            if (tid == 0) {
                s_abort = 1;
                // the arrival counters must still come back to zero: marked tickets for what this CTA leaves undone
                for (; it < p.items && p.S > 1; it += gridDim.x) {
                    int* tk = p.tickets + it / p.S;
                    int ticket;
                    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(ticket) : "l"(tk), "r"(kTicketAbortedW + 1) : "memory");
                    if ((ticket & (kTicketAbortedW - 1)) == p.S - 1) *tk = 0;
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 5) {
        if (s_abort) {
            // MMAs may still be in flight: let them finish (bounded) before the tensor memory goes back
            if (lane == 0) {
                tc_commit(bar_end);
                (void)mbar_wait(bar_end, 0, p.wait_ns);
                atomicOr(p.err_word, SEGKV_DEV_WAIT_LIMIT);
            }
            __syncwarp();
        }
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(L::kTmemCols) : "memory");
    }
}

template <typename T, int D>
cudaError_t launch_one(const Dims& d, const SdpaArgs& a, const CUtensorMap& tmk, const CUtensorMap& tmv, int sms, cudaStream_t st) {
    using L = WideLayout<T, D>;
    // never two CTAs on one SM: the second would wait for tensor memory inside its allocation
    constexpr size_t smem = L::kBytes > 120 * 1024 ? L::kBytes : 120 * 1024;
    auto kern = sdpa_wide_kernel<T, D>;
    static bool configured[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    WideParams p;
    p.q = a.q; p.out = a.out; p.slopes = a.slopes;
    p.kr = (const char*)a.kr; p.k_chunks = (const char* const*)a.k_chunks; p.vdelta = a.vdelta; p.chunk_steps = d.chunk_steps;
    p.ulist = a.ulist; p.ucount = a.ucount; p.plens = a.plens;
    p.tickets = a.tickets; p.err_word = a.err_word;
    p.P = a.prompt_len; p.steps = a.steps; p.S = a.splits; p.W = d.beams; p.G = d.group; p.H = d.heads; p.Hkv = d.kv_heads;
    p.rows = d.rows; p.max_steps = d.max_steps; p.ncols = d.beams * d.group;
    p.items = d.batch * d.kv_heads * a.splits;
    p.ws_o = a.ws;
    p.ws_ml = a.ws + (size_t)p.items * p.ncols * D;
    p.early_prompt = (a.pdl && a.prompt_immutable) ? 1 : 0;
    p.row = rowwise::make_args(d, a);
    p.dbg_skip = a.dbg_skip ? 1 : 0;
    p.wait_ns = a.wait_ns ? a.wait_ns : kWaitLimitNs;
    p.scale2 = 1.4426950408889634f / sqrtf((float)D);
    // instruction descriptors: fp32 accumulate, A/B format, N >> 3, M = 128; V is the MN-major operand
    const uint32_t fmt = d.dtype == SEGKV_BF16 ? 1u : 0u;
    const uint32_t common = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(128 >> 4) << 24);
    p.idesc_qk = common | ((uint32_t)(L::KEYS >> 3) << 17);
    p.idesc_pv = common | (1u << 16) | ((uint32_t)(D >> 3) << 17);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.items < sms ? p.items : sms), 1, 1);
    cfg.blockDim = dim3(L::kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (a.pdl) {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    return cudaLaunchKernelEx(&cfg, kern, tmk, tmv, p);
}

template <typename T>
cudaError_t dispatch(const Dims& d, const SdpaArgs& a, const CUtensorMap& tmk, const CUtensorMap& tmv, int sms, cudaStream_t st) {
    switch (d.head_dim) {
        case 64: return launch_one<T, 64>(d, a, tmk, tmv, sms, st);
        case 128: return launch_one<T, 128>(d, a, tmk, tmv, sms, st);
        case 256: return launch_one<T, 256>(d, a, tmk, tmv, sms, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// The split merge keeps one factor per split and column where the weights were.  (bf16 at head_dim 256: the 32 that the
// segkv_get_splits of such a handle has always answered at most.)
int wide_max_splits(const Dims& d) {
    static_assert(WideLayout<__half, 256>::kP >= kMaxSplits * kCols * 4, "factors of the split merge");
    return d.head_dim == 256 && d.dtype == SEGKV_BF16 ? 32 : kMaxSplits;
}

int wide_tile_keys(const Dims& d) { return d.head_dim == 256 ? WideLayout<__half, 256>::KEYS : WideLayout<__half, 128>::KEYS; }

cudaError_t launch_sdpa_wide(const Dims& d, const SdpaArgs& a, const CUtensorMap& tmk, const CUtensorMap& tmv, int sms, cudaStream_t st) {
    if (a.splits < 1 || a.splits > wide_max_splits(d) || d.beams * d.group > kCols) return cudaErrorInvalidValue;
    return d.dtype == SEGKV_BF16 ? dispatch<__nv_bfloat16>(d, a, tmk, tmv, sms, st) : dispatch<__half>(d, a, tmk, tmv, sms, st);
}

}  // namespace segkv_impl
