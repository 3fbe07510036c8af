// Prefill attention on the fifth-generation tensor cores (tcgen05 + tensor memory), head_dim 64,
// 128 or 256 (paper Section 3.1 / 3.3: the prefill kernel is the special case of the customised
// SDPA kernel that sees only the query and the prompt key/value, batch-first in and out):
//     out[b,i,h,:] = softmax_{j<=i}( q[b,i,h,:] . K[b,j,:] / sqrt(D) + bias ) . V[b,j,:].
//
//   * one persistent CTA per SM walks a static list of work items (one or two groups of 128
//     query rows of one (request, head)), longest first; a group's rows are one per TMEM lane and
//     per TWO softmax threads (four where one group of head_dim 64 or 128 runs), which share a tile's keys;
//   * an item's keys are gone through from the newest back, so that its two groups end together and the second's diagonal
//     tile does not run alone at the end (from the oldest forward: 4 % slower at 64 x 56 x 2048, and under an ALiBi
//     bias a row's maximum grew with every tile, so that most of Bloom's heads took two passes over each and rescaled O).
//     Without a bias the oldest tile comes before them all: every row sees all of it, and the reference is the exact score
//     of one of its keys, whose weight is then not rounded (with a reference from the diagonal tile, of which some
//     rows see a few keys, the error against 64 bits was 1 % larger);
//   * Q of each group arrives by TMA (a per-call tensor map over [B, N, H, D]) in the
//     128-byte-swizzled K-major layout; K and V tiles (128 keys; 64 at head_dim 256) arrive by TMA
//     in the same layout through separate rings: a K tile is needed one step before the V tile
//     of the same keys.  They come from the prompt segment, or (fused prefill) from the caller's
//     arrays, and are then also stored on into the segment, each tile by one CTA;
//   * one warp, converged, issues one lane's MMAs: S = Q.K^T (M 128, N = keys of a tile, K-steps of 16)
//     into a TMEM buffer and O += P.V (M 128, N = head_dim) into a TMEM accumulator.  P never
//     touches shared memory: the softmax threads write it, rounded to the 16-bit type, over
//     the scores it came from (16 keys' weights over the first half of their columns), and the MMA
//     takes its A operand from tensor memory.  V is consumed as an MN-major B operand straight from
//     its row-major tile;
//   * the softmax threads read S with tcgen05.ld (no shuffles for the row max / sum) and
//     rescale O in tensor memory only when a row's maximum has grown by more than about 2^8 over the
//     reference it is using (the sum uses the same reference, so the result is exact).  Weights are worked out with the
//     reference in use in one pass over the scores, 16 keys at a time with the next 16 on their way; what they add up to
//     decides whether they stand;
//   * with two groups per CTA each has one S buffer and the tensor cores work for one group
//     while the other is in its softmax; with one group S is double-buffered so that Q.K^T of
//     tile j+1 runs under the softmax of tile j.  The tail of one item overlaps the head of the
//     next (loads, and the first Q.K^T while the previous output is stored).
//
// What bounds it: a group's chain softmax -> P.V -> Q.K^T (1024 clocks of MMAs and as many of exponentials a tile), which two
// groups overlap in part, and the issue slots of the softmax; with a few items the start as well.  (Large launches run at 1.5 to
// 1.65 GHz where a lone call runs at 1.9, so compare queued times with queued ones: these are.)  Measured in turn with the form that went from the oldest keys forward throughout, held P back until the row's two
// threads had met, spilled and was launched behind the whole kernel before (before / now in us, attention alone): with ALiBi
// 32 x 112 heads x 1024 at D 128 bf16 1922 / 1607 (fp16 1825 / 1335), D 64, 16 x 64 x 2048, bf16 1515 / 1053, D 256, 2 x 8 x 2000, bf16
// 61.6 / 42.1; without 64 x 56 x 2048 at D 128 fp16 4810 / 4789, bf16 5118 / 4787, 1 x 32 x 1024 20.6 / 18.9, 4 x 40 x 700 49.3 / 44.6,
// D 64, 16 x 64 x 2048, 992 / 978, D 256, 16 x 16 x 1003, 182 / 185 (with the store fused 228 / 225).  Putting a share of the
// exponentials on the FMA pipes as a polynomial was measured slower (4.42 against 4.17 ms): the issue slots it costs are on
// the same chain.
//
// Tensor memory (all 512 columns are allocated): S buffers first, then one O accumulator per
// group.  Every mbarrier is waited on phase by phase (a parity wait cannot tell phases two
// apart) and every wait is bounded; on expiry the kernel flags SEGKV_DEV_WAIT_LIMIT, skips
// the output and still releases its tensor memory.
#include <type_traits>

#include "segkv_internal.h"
#include "segkv_ptx.cuh"
#include "segkv_tc5.cuh"

namespace segkv_impl {

namespace {

using namespace ptx;

constexpr int kRows = 128;     // query rows per group (TMEM lanes)
constexpr int kBoxQ = kRows * 128;           // 64 head-dim elements of a group's Q rows (one 128-byte swizzle span wide)
constexpr int kTmemCols = 512;

struct Tc5Params {
    void* out;
    const float* slopes;
    int* err_word;
    const int32_t* plens;    // per-request prompt lengths (rows and keys past them are skipped), or NULL
    int N, H, G, B, snake;
    int paired, rounds;      // item order: see round_item; rounds = items a CTA walks through (some may be empty)
    float scale2;
    uint32_t idesc_qk, idesc_pv;
    int dbg_skip;            // test aid: one softmax thread leaves out one barrier arrival, so that a wait runs out
    unsigned long long wait_ns;   // limit of every bounded wait
};

template <typename T> struct SplitP { typedef char yes; static constexpr bool value = false; };
template <> struct SplitP<__nv_bfloat16> { typedef char yes; static constexpr bool value = true; };
// Factor of the weights, as a power of two: fp16 weights are at most 2^8 of the reference times 2^7, which keeps what is
// far below the maximum above fp16's smallest numbers.
template <typename T> constexpr float kWeightShift = SplitP<T>::value ? 0.f : 7.f;
template <typename T> constexpr float kWeightMax = SplitP<T>::value ? 256.f : 32768.f;    // 2^8 of the reference

// Shape of one instantiation: head_dim D (64, 128 or 256), KEYS keys per K/V tile, NG groups of
// 128 query rows per CTA.  head_dim 256 leaves tensor memory for one group and 64-key tiles only.
template <int D_, int KEYS_, int NG_>
struct Tc5Layout {
    static constexpr int D = D_, KEYS = KEYS_, NG = NG_;
    static constexpr int NB = NG == 1 ? 2 : 1;                   // S buffers per group
    static constexpr int TPR = D == 256 ? 2 : 4 / NG;            // softmax threads per query row
    static constexpr int kSoftWarps = 4 * TPR * NG;
    static constexpr int kThreads = 32 * (kSoftWarps + 4);       // and TMA loads, MMAs, TMA stores, one idle (it costs no registers)
    static constexpr int kDBoxes = D / 64;                       // 64-element (128-byte) column blocks of a row
    static constexpr int kBoxRows = D == 256 ? 32 : 64;          // rows of one TMA box of the prompt segment's tensor map
    static constexpr int kBoxBytes = kBoxRows * 128;
    static constexpr int kColTile = KEYS * 128;                  // one column block of all keys of a tile
    static constexpr int kTileKV = kDBoxes * kColTile;           // bytes of a K (or a V) tile
    static constexpr int kStagesK = 3;
    static constexpr int kStagesV = (NG == 1 && D <= 128) ? 3 : 2;
    static constexpr int kRingK = kStagesK * kTileKV;
    static constexpr int kRingV = kStagesV * kTileKV;
    static constexpr int kQGroup = kDBoxes * kBoxQ;              // bytes of one group's Q
    static constexpr int kQ = NG * kQGroup;
    static constexpr int kBars = 2 * kStagesK + 2 * kStagesV + 6 * NG + 1;   // K full/empty, V full/empty, per group: S0 S1 P O Qfull Qempty; wind-down
    static constexpr size_t kBytes = (size_t)kRingK + kRingV + kQ + 8 * kBars + NG * TPR * kRows * 4 + 16;
    // tensor memory: S buffers of KEYS columns first, then one O accumulator of D columns per group
    static constexpr int kColO = NG * NB * KEYS;
    static_assert(kColO + NG * D <= kTmemCols, "tensor memory");
    static_assert(kBytes <= 232448, "shared memory");
};

// Maximum of 16 scores of a row, in log2 units with BIAS (s * scale2 + bias0 + slope2 * i), else raw dot products;
// MASK: keys above the row (i > lim) do not count.
template <bool BIAS, bool MASK>
__device__ __forceinline__ float max16(const uint32_t* sr, float scale2, float slope2, float bias0, int lim) {
    float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
        float v[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            v[u] = __uint_as_float(sr[i + u]);
            if (BIAS) v[u] = fmaf(v[u], scale2, fmaf(slope2, (float)(i + u), bias0));
            if (MASK && i + u > lim) v[u] = -INFINITY;
        }
        asm("max.f32 %0, %0, %1, %2;" : "+f"(mx[(i >> 1) & 1]) : "f"(v[0]), "f"(v[1]));
    }
    return fmaxf(mx[0], mx[1]);
}

// bf16 keeps 8 significant bits of a softmax weight.  Where a few keys carry a row's whole weight
// and their values cancel, that rounding alone exceeds the path's tolerance, so where it can
// happen the weights go to the tensor cores as TWO bf16 parts, p = hi + lo (hi = p cut to bf16,
// lo = bf16(p - hi): 16 significant bits together), lo in the second half of the S buffer's
// columns, and O takes a second P.V MMA for those keys.  Which keys is known from the launch
// shape: the first key tile of the rows that start the prompt (a handful of keys in all), and,
// under an ALiBi slope steep enough to put a row's weight on its nearest neighbours, the keys
// within kSplitWindow of the group's rows.  fp16 weights (11 bits) never need it.
constexpr float kSplitSlope = 0.0625f;   // weights fall by e^-slope per key: below this, dozens of keys share a row's weight
constexpr int kSplitWindow = 64;
// Do the `nkeys` keys from `key0` on get two-part weights, for the group whose first row is row0?
__device__ __forceinline__ bool split_p_keys(int row0, int key0, int nkeys, bool steep) {
    if (row0 == 0 && key0 < kRows) return true;
    return steep && key0 + nkeys - 1 >= row0 - kSplitWindow;
}

// Two fp32 values in one 64-bit register pair, for the packed fp32 instructions.
__device__ __forceinline__ uint64_t f2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float f2_lo(uint64_t v) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return a;
}
__device__ __forceinline__ float f2_hi(uint64_t v) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return b;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Weights of 16 keys of a row from their scores: 2^(s * scale2 + c0 + slope2 * i), c0 = bias minus the row's reference;
// packed in 16 bits (SPLIT: a second set of 8 words with the low parts).  Returns their sum.
template <typename T, bool BIAS, bool MASK, bool SPLIT>
__device__ __forceinline__ uint64_t weigh16(const uint32_t* sr, float scale2, float slope2, float c0, int lim, uint32_t* hi, uint32_t* lo) {
    const uint64_t sc = f2(scale2, scale2), sl = f2(slope2, slope2), cc = f2(c0, c0);
    uint64_t ls[2] = {0ull, 0ull};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint64_t x = f2_fma(f2(__uint_as_float(sr[2 * k]), __uint_as_float(sr[2 * k + 1])), sc,
                                  BIAS ? f2_fma(sl, f2((float)(2 * k), (float)(2 * k + 1)), cc) : cc);
        const float xa = MASK && 2 * k > lim ? -INFINITY : f2_lo(x), xb = MASK && 2 * k + 1 > lim ? -INFINITY : f2_hi(x);
        const float ea = exp2f(xa), eb = exp2f(xb);
        ls[k & 1] = k < 2 ? f2(ea, eb) : f2_add(ls[k & 1], f2(ea, eb));
        if (!SPLIT) {
            hi[k] = Mma<T>::pack(ea, eb);
        } else {
            const uint32_t b0 = __float_as_uint(ea), b1 = __float_as_uint(eb);
            hi[k] = __byte_perm(b0, b1, 0x7632);
            lo[k] = Mma<T>::pack(ea - __uint_as_float(b0 & 0xFFFF0000u), eb - __uint_as_float(b1 & 0xFFFF0000u));
        }
    }
    return f2_add(ls[0], ls[1]);
}

// One CTA per SM walks a static list of work items (128*NG query rows of one (request, head)),
// longest first and dealt round-robin, so that the tail of one item overlaps the head of the
// next: the producer runs ahead through the K/V rings and reloads a group's Q as soon as the
// group's last Q.K^T has been read, and the first Q.K^T of the next item executes while the
// softmax threads are still storing the previous output.
// MODE 0: K/V from the prompt segment, one prompt length; 1: fused prefill (K/V from the caller's arrays,
// every tile stored into the segment); 2: per-request prompt lengths (kept out of the other two: the
// lengths as run-time values cost registers that the softmax threads of the two-group shape do not have).
template <typename T, typename L, int MODE>
__global__ void __launch_bounds__(L::kThreads, 1)
prefill_tc5_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                   const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_k_seg,
                   const __grid_constant__ CUtensorMap tm_v_seg, const Tc5Params p) {
    constexpr int NG = L::NG, NB = L::NB, TPR = L::TPR, SK = L::kStagesK, SV = L::kStagesV;
    constexpr bool STORE = MODE == 1, RAGGED = MODE == 2;
    constexpr bool kSplitP = sizeof(typename SplitP<T>::yes) != 0 && SplitP<T>::value;
    constexpr int kD = L::D, kKeys = L::KEYS, kTileKV = L::kTileKV, kColTile = L::kColTile;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* k_ring = smem;                                       // tile: two halves [128 keys][64 elements]
    uint8_t* v_ring = k_ring + L::kRingK;
    uint8_t* q_smem = v_ring + L::kRingV;                         // per group two halves [128 rows][64 elements]
    uint64_t* bars = reinterpret_cast<uint64_t*>(q_smem + L::kQ);
    const uint32_t kfull0 = smem_u32(bars), kempty0 = kfull0 + 8 * SK;
    const uint32_t vfull0 = kempty0 + 8 * SK, vempty0 = vfull0 + 8 * SV;
    const uint32_t gbar0 = vempty0 + 8 * SV;                      // group g: + kGB g; S buffer 0, S buffer 1, P, O, Q full, Q empty
    constexpr uint32_t kGB = 48;
    const uint32_t bar_end = gbar0 + kGB * NG;
    float* s_row = reinterpret_cast<float*>(bars + L::kBars);     // [group][thread of the row][row]: one value, for the row's other threads
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_row + NG * TPR * kRows);
    volatile int& s_abort = *reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nqt = (p.N + kRows * NG - 1) / (kRows * NG);
    const int hb_count = p.H * p.B;
    const int n_items = nqt * hb_count;
    // The CTA's item of round j: the list is sorted longest first and dealt out round-robin; with
    // only a few rounds, in snake order (every other round reversed), which evens out the total
    // length per CTA.
    auto round_item = [&](int j) -> int {
        const int G = (int)gridDim.x, c = (int)blockIdx.x;
        if (p.paired) {
            // Long prompts, many (request, head)s: the query tiles of one (request, head) run at the same
            // time on neighbouring CTAs, so that its K/V crosses HBM once and is found in the L2 by the
            // others (dealt longest-first over all (request, head)s, every query tile re-reads its keys
            // from HBM: 2.3x the unique bytes).  CTA c takes the pr-th longest tile, then the pr-th
            // shortest, of the same (request, head): every CTA gets the same number of key tiles.
            const int ppb = (nqt + 1) / 2;            // CTAs per (request, head)
            const int bpw = G / ppb;                  // (request, head)s in flight
            if (c >= bpw * ppb) return n_items;       // (a few CTAs idle when ppb does not divide the grid)
            const int hb = (j >> 1) * bpw + c / ppb, pr = c % ppb;
            if (hb >= hb_count) return n_items;
            const int qt = (j & 1) ? pr : nqt - 1 - pr;
            if ((j & 1) && 2 * pr == nqt - 1) return n_items;   // the middle tile of an odd count came first
            return (nqt - 1 - qt) * hb_count + hb;
        }
        const int w = j * G + ((p.snake && (j & 1)) ? G - 1 - c : c);
        return w < n_items ? w : n_items;
    };
    // item w -> query tile (longest first), head, request
    auto item_qt = [&](int w) { return nqt - 1 - w / hb_count; };
    // key tiles of group g of query tile qt: up to its diagonal tile (causal); none past the prompt
    // Order of an item's tiles (see the head of this file): position i of n tiles
    const bool back = p.slopes != nullptr;
    auto tile_at = [&](int i, int n) -> int { return back ? n - 1 - i : i == 0 ? 0 : n - i; };
    // nb = the request's own prompt length: with ragged prompts the items are still laid out for the
    // longest one, and a shorter request leaves its later items (and the tail of one) without work.  (Lengths and slopes are read
    // by plain loads: the kernel before may write them, and a read-only load need not stay behind the wait for it below.)
    auto request_len = [&](int b) -> int { return RAGGED ? p.plens[b] : p.N; };
    auto group_tiles = [&](int qt, int g, int nb) -> int {
        const int base = (qt * NG + g) * kRows;
        return base < nb ? min((nb + kKeys - 1) / kKeys, (base + kRows - 1) / kKeys + 1) : 0;
    };

    if (tid == 0) {
        // a stage is released by the MMAs that read it and, when tiles are stored on, by the store thread
        for (int s = 0; s < SK; ++s) {
            mbar_init(kfull0 + 8 * s, 1);
            mbar_init(kempty0 + 8 * s, STORE ? 2 : 1);
        }
        for (int s = 0; s < SV; ++s) {
            mbar_init(vfull0 + 8 * s, 1);
            mbar_init(vempty0 + 8 * s, STORE ? 2 : 1);
        }
        for (int g = 0; g < NG; ++g) {
            mbar_init(gbar0 + kGB * g, 1);
            mbar_init(gbar0 + kGB * g + 8, 1);
            mbar_init(gbar0 + kGB * g + 16, 4 * TPR);             // a lane of each of the group's warps
            mbar_init(gbar0 + kGB * g + 24, 1);
            mbar_init(gbar0 + kGB * g + 32, 1);
            mbar_init(gbar0 + kGB * g + 40, 1);
        }
        mbar_init(bar_end, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    if (warp == L::kSoftWarps + 1) {                                     // this warp owns the tensor memory
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "n"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // Set up while the previous kernel ends: everything it may have written is read from here on.  (The launch of one
    // prefill behind another took up to 6 us of an idle GPU.)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == L::kSoftWarps) {
        // ------------------------------- TMA producer -------------------------------
        if (lane == 0) {
            prefetch_tmap(&tm_q);
            prefetch_tmap(&tm_k);
            prefetch_tmap(&tm_v);
            auto load_tile = [&](const CUtensorMap* tm, uint8_t* dst_tile, int kt, int kvh, int b, uint32_t full) {
                const uint32_t dst = smem_u32(dst_tile);
                mbar_arrive_expect_tx(full, (uint32_t)kTileKV);
#pragma unroll
                for (int cb = 0; cb < L::kDBoxes; ++cb)
#pragma unroll
                    for (int rb = 0; rb < kKeys / L::kBoxRows; ++rb)
                        tma_load_4d(dst + cb * kColTile + rb * L::kBoxBytes, tm, cb * 64, kvh,
                                    kt * kKeys + rb * L::kBoxRows, b, full);
            };
            uint32_t tp = 0, tk = 0;                               // K/V tiles requested so far (ring position); K tiles alone
            uint32_t qi[NG];                                      // items group g has taken part in: Q barrier phases
#pragma unroll
            for (int g = 0; g < NG; ++g) qi[g] = 0;
            bool ok = true;
            for (int j = 0; j < p.rounds && ok; ++j) {
                const int w = round_item(j);
                if (w >= n_items) continue;
                const int qt = item_qt(w), hb = w % hb_count, h = hb % p.H, b = hb / p.H;
                const int kvh = h / p.G;
                int nkt = 0;
#pragma unroll
                for (int g = 0; g < NG; ++g) nkt = max(nkt, group_tiles(qt, g, request_len(b)));
#pragma unroll
                for (int x = 0; x < NG; ++x) {                    // the group that begins first
                    const int g = back ? NG - 1 - x : x;
                    if (!ok || group_tiles(qt, g, request_len(b)) == 0) continue;
                    // the group's Q rows (past the prompt: zeros), once its previous Q is no longer read
                    ok = mbar_wait(gbar0 + kGB * g + 40, (qi[g] & 1) ^ 1, p.wait_ns);
                    if (!ok) break;
                    ++qi[g];
                    const uint32_t qfull = gbar0 + kGB * g + 32;
                    const uint32_t dst = smem_u32(q_smem) + (uint32_t)g * L::kQGroup;
                    mbar_arrive_expect_tx(qfull, (uint32_t)L::kQGroup);
#pragma unroll
                    for (int cb = 0; cb < L::kDBoxes; ++cb)
                        tma_load_4d(dst + cb * kBoxQ, &tm_q, cb * 64, h, (qt * NG + g) * kRows, b, qfull);
                }
                for (int i = 0; i < nkt && ok; ++i, ++tp) {
                    const int kt = tile_at(i, nkt);
                    const uint32_t sk = tp % SK, sv = tp % SV;
                    ok = mbar_wait(kempty0 + 8 * sk, ((tp / SK) & 1) ^ 1, p.wait_ns);
                    if (!ok) break;
                    load_tile(&tm_k, k_ring + (size_t)sk * kTileKV, kt, kvh, b, kfull0 + 8 * sk);
                    tk = tp + 1;
                    ok = mbar_wait(vempty0 + 8 * sv, ((tp / SV) & 1) ^ 1, p.wait_ns);
                    if (!ok) break;
                    load_tile(&tm_v, v_ring + (size_t)sv * kTileKV, kt, kvh, b, vfull0 + 8 * sv);
                }
            }
            if (!ok) s_abort = 1;
            // no copy may land after the CTA has gone (all have, unless a wait ran out somewhere)
            for (uint32_t k = tk > (uint32_t)SK ? tk - SK : 0; k < tk; ++k) (void)mbar_wait(kfull0 + 8 * (k % SK), (k / SK) & 1, p.wait_ns);
            for (uint32_t k = tp > (uint32_t)SV ? tp - SV : 0; k < tp; ++k) (void)mbar_wait(vfull0 + 8 * (k % SV), (k / SV) & 1, p.wait_ns);
#pragma unroll
            for (int g = 0; g < NG; ++g)
                if (qi[g] > 0) (void)mbar_wait(gbar0 + kGB * g + 32, (qi[g] - 1) & 1, p.wait_ns);
        }
    } else if (warp == L::kSoftWarps + 2) {
        if (STORE && lane == 0) {
            // ---- fused prefill: the tiles just read from the caller's K/V also become the prompt segment
            // (paper Section 3.2: the prompt is kept once per request).  Tile kt of a kv head is stored by
            // exactly one item: the first query head of the group, at the query tile whose rows start the
            // tile's keys.  The thread follows the producer's tile sequence, waits for a tile to land,
            // stores it if this item owns it (TMA store from the same swizzled tile), and adds its
            // release of the stage to the MMAs' once the store has read shared memory.
            prefetch_tmap(&tm_k_seg);
            prefetch_tmap(&tm_v_seg);
            auto store_tile = [&](const CUtensorMap* tm, uint8_t* src_tile, int kt, int kvh, int b) {
                const uint32_t src = smem_u32(src_tile);
#pragma unroll
                for (int cb = 0; cb < L::kDBoxes; ++cb)
#pragma unroll
                    for (int rb = 0; rb < kKeys / L::kBoxRows; ++rb)
                        tma_store_4d(tm, src + cb * kColTile + rb * L::kBoxBytes, cb * 64, kvh,
                                     kt * kKeys + rb * L::kBoxRows, b);
                bulk_commit_group();
                bulk_wait_read_all();
            };
            uint32_t tp = 0;
            bool ok = true;
            for (int j = 0; j < p.rounds && ok; ++j) {
                const int w = round_item(j);
                if (w >= n_items) continue;
                const int qt = item_qt(w), hb = w % hb_count, h = hb % p.H, b = hb / p.H;
                const int kvh = h / p.G;
                int nkt = 0;
#pragma unroll
                for (int g = 0; g < NG; ++g) nkt = max(nkt, group_tiles(qt, g, request_len(b)));
                for (int i = 0; i < nkt && ok; ++i, ++tp) {
                    const int kt = tile_at(i, nkt);
                    const bool mine = (h % p.G) == 0 && (kt * kKeys) / (kRows * NG) == qt;
                    const uint32_t sk = tp % SK, sv = tp % SV;
                    ok = mbar_wait(kfull0 + 8 * sk, (tp / SK) & 1, p.wait_ns);
                    if (!ok) break;
                    if (mine) store_tile(&tm_k_seg, k_ring + (size_t)sk * kTileKV, kt, kvh, b);
                    mbar_arrive(kempty0 + 8 * sk);
                    ok = mbar_wait(vfull0 + 8 * sv, (tp / SV) & 1, p.wait_ns);
                    if (!ok) break;
                    if (mine) store_tile(&tm_v_seg, v_ring + (size_t)sv * kTileKV, kt, kvh, b);
                    mbar_arrive(vempty0 + 8 * sv);
                }
            }
            bulk_wait_all();                                      // the stores themselves, before the CTA may exit
            if (!ok) s_abort = 1;
        }
    } else if (warp == L::kSoftWarps + 1) {
        // -------------------------------- MMA issuer --------------------------------
        // (the whole warp runs this, converged, and one lane's MMAs are issued: see tc_mma_ss_if.  What decides the
        // control flow is made uniform by a warp reduction or vote.)
        {
            // Ring positions are counted, not computed with remainders, so that descriptors stay in uniform
            // registers: MMAs follow each other at 64 clocks then, and at about 108 with remainders.
            const uint32_t lead = elect_one();
            auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
                return __all_sync(0xffffffffu, mbar_wait_hot(bar, parity, p.wait_ns));
            };
            const uint32_t q_lo = (smem_u32(q_smem) & 0x3FFFFu) >> 4, k_lo0 = (smem_u32(k_ring) & 0x3FFFFu) >> 4;
            const uint32_t v_lo0 = (smem_u32(v_ring) & 0x3FFFFu) >> 4;
            const uint64_t dk = smem_desc(0, 16, 1024), dv = smem_desc(0, kColTile, 1024);   // descriptors without an address
            uint32_t kst = 0, kph = 0, vst = 0, vph = 0;          // stage and phase of the next K and V tile
            uint32_t n[NG], qi[NG];                               // tiles / items of group g so far: barrier phases
#pragma unroll
            for (int g = 0; g < NG; ++g) n[g] = qi[g] = 0;
            bool ok = true;
            // S_g[buf] = Q_g . K^T for the K tile of stage kst; after the group's last one its Q may be replaced
            auto issue_qk = [&](int g, uint32_t buf, bool last) {
                const uint64_t qd = dk + (q_lo + (uint32_t)g * (uint32_t)(L::kQGroup >> 4));
                const uint64_t kd = dk + (k_lo0 + kst * (uint32_t)(kTileKV >> 4));
                const uint32_t d_tmem = tmem + (uint32_t)kKeys * ((uint32_t)(g * NB) + buf);
#pragma unroll
                for (int ks = 0; ks < kD / 16; ++ks)
                    tc_mma_ss_if(lead, d_tmem, qd + (uint64_t)(((ks >> 2) * kBoxQ + (ks & 3) * 32) >> 4),
                                 kd + (uint64_t)(((ks >> 2) * kColTile + (ks & 3) * 32) >> 4), p.idesc_qk, ks > 0);
                tc_commit_if(lead, gbar0 + kGB * g + 8 * buf);
                if (last) tc_commit_if(lead, gbar0 + kGB * g + 40);
            };
            auto wait_k = [&]() -> bool {
                const bool r = wait(kfull0 + 8 * kst, kph);
                tc_fence_after();
                return r;
            };
            auto release_k = [&]() {                              // K stage free once these MMAs are done
                tc_commit_if(lead, kempty0 + 8 * kst);
                if (++kst == SK) { kst = 0; kph ^= 1u; }
            };
            for (int j = 0; j < p.rounds && ok; ++j) {
                const int w = round_item(j);
                if (w >= n_items) continue;
                const int qt = item_qt(w), nb = RAGGED ? (int)__reduce_max_sync(0xffffffffu, (unsigned)request_len((w % hb_count) / p.H)) : p.N;
                // is the head's slope one of those whose weights go in two parts next to the diagonal?
                const bool steep = kSplitP && p.slopes && __any_sync(0xffffffffu, p.slopes[(w % hb_count) % p.H] >= kSplitSlope);
                int gt[NG], nkt = 0;
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    gt[g] = group_tiles(qt, g, nb);
                    nkt = max(nkt, gt[g]);
                }
                if (nkt == 0) continue;                           // the request ends before this item's rows
                // The first of two groups does not see the item's last tile: the position that it leaves out, and its first and
                // last one.
                int skip[NG], first[NG], last[NG];
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    skip[g] = gt[g] == nkt ? -1 : back ? 0 : 1;
                    first[g] = skip[g] == 0 ? 1 : 0;
                    last[g] = skip[g] == nkt - 1 ? nkt - 2 : nkt - 1;
                }
                // the scores of position i of group g, the K tile waited for
                auto scores = [&](int g, int i) -> bool {
                    if (i == first[g]) {
                        if (!wait(gbar0 + kGB * g + 32, qi[g]++ & 1)) return false;   // Q_g landed
                        tc_fence_after();
                    }
                    issue_qk(g, NB == 2 ? (n[g] + (i == first[g] ? 0u : 1u)) & 1 : 0u, i == last[g]);
                    return true;
                };
                ok = wait_k();
#pragma unroll
                for (int g = 0; g < NG; ++g)
                    if (gt[g] > 0 && skip[g] != 0 && ok) ok = scores(g, 0);
                if (!ok) break;
                release_k();
                for (int i = 0; i < nkt && ok; ++i) {
                    const int kt = tile_at(i, nkt);
                    if (NB == 2 && i + 1 < nkt) {                 // next tile's scores run under this tile's softmax
                        ok = wait_k();
                        if (!ok) break;
                        (void)scores(0, i + 1);
                        release_k();
                    }
                    const uint64_t vd = dv + (v_lo0 + vst * (uint32_t)(kTileKV >> 4));
                    ok = wait(vfull0 + 8 * vst, vph);
                    if (!ok) break;
                    bool k_next = false;
#pragma unroll
                    for (int g = 0; g < NG; ++g) {
                        if (gt[g] == 0) continue;
                        if (i != skip[g]) {
                            ok = wait(gbar0 + kGB * g + 16, n[g] & 1);   // P_g written over its S buffer
                            if (!ok) break;
                            tc_fence_after();
                            const uint32_t p_tmem = tmem + (uint32_t)kKeys * ((uint32_t)(g * NB) + (NB == 2 ? n[g] & 1 : 0u));
#pragma unroll
                            for (int kk = 0; kk < kKeys / 16; ++kk)   // O_g += P_g[:, 16 keys] . V[16 keys, :]
                                tc_mma_ts_if(lead, tmem + (uint32_t)(L::kColO + kD * g), p_tmem + kk * 16,
                                             vd + (uint64_t)((kk * 2048) >> 4), p.idesc_pv, (i != first[g] || kk > 0));
                            if (kSplitP && split_p_keys((qt * NG + g) * kRows, kt * kKeys, kKeys, steep)) {
#pragma unroll
                                for (int kk = 0; kk < kKeys / 16; ++kk)   // ... and the low parts of the weights that have one
                                    if (split_p_keys((qt * NG + g) * kRows, kt * kKeys + 16 * kk, 16, steep))
                                        tc_mma_ts_if(lead, tmem + (uint32_t)(L::kColO + kD * g), p_tmem + kk * 16 + 8,
                                                     vd + (uint64_t)((kk * 2048) >> 4), p.idesc_pv, 1u);
                            }
                            tc_commit_if(lead, gbar0 + kGB * g + 24);
                            ++n[g];
                        }
                        if (NB == 1 && i + 1 < nkt && i + 1 != skip[g]) {        // the group's next scores, behind its P.V in the pipe
                            if (!k_next) {
                                ok = wait_k();
                                if (!ok) break;
                                k_next = true;
                            }
                            ok = scores(g, i + 1);
                            if (!ok) break;
                        }
                    }
                    if (!ok) break;
                    tc_commit_if(lead, vempty0 + 8 * vst);        // stage free once every MMA so far is done
                    if (++vst == SV) { vst = 0; vph ^= 1u; }
                    if (NB == 1 && i + 1 < nkt) release_k();
                }
            }
            if (!ok && lane == 0) s_abort = 1;
        }
    } else if (warp < L::kSoftWarps) {
        // ------------------------------ softmax warps: two or four threads per row ------------------------------
        // Each takes its part of a tile's keys, and at the end of an item its part of the output row.  (One thread per row
        // spent 2200 clocks on a tile of 128 keys, of which 1170 are hidden behind the other group's MMAs: the
        // chain softmax -> P.V -> next Q.K^T bound the kernel.  More warps hide each other's latencies: a lone group's
        // tile took 1890 clocks with two threads per row.)
        constexpr int KH = kKeys / TPR, DH = kD / TPR;
        // keys at a time: 32 where the registers are there (with one group a tile's latency counts), else 16
        constexpr int PC = NG == 1 && KH >= 32 ? 32 : 16;
        const int g = warp / (4 * TPR), part = (warp >> 2) % TPR, r = (warp & 3) * 32 + lane;
        const int rows_bar = 1 + g * 4 + (warp & 3);              // barrier of the warps that share these rows
        const uint32_t bar_s0 = gbar0 + kGB * g, bar_p = bar_s0 + 16, bar_o = bar_s0 + 24;
        const uint32_t tm_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);     // this warp's TMEM lanes
        const uint32_t tm_o = tm_lane + (uint32_t)(L::kColO + kD * g + DH * part);
        float* xrow = s_row + g * TPR * kRows + r;                // + kRows x thread of the row
        const size_t qstride = (size_t)p.H * kD;
        uint32_t n = 0;                                           // tiles of this group so far: barrier phases
        bool ok = true, gone = false;                             // a wait of this thread ran out; the row's warps have agreed to leave
        for (int j = 0; j < p.rounds && !gone; ++j) {
            const int w = round_item(j);
            if (w >= n_items) continue;
            const int qt = item_qt(w), hb = w % hb_count, h = hb % p.H, b = hb / p.H;
            const int my_tiles = group_tiles(qt, g, request_len(b));
            if (my_tiles == 0) continue;
            const int row0 = (qt * NG + g) * kRows, row = row0 + r;
            const float slope_nat = p.slopes ? p.slopes[h] : 0.f;
            const float slope2 = slope_nat * 1.4426950408889634f;
            const bool biased = back;
            float m_ref = -INFINITY, l_run = 0.f;
            for (int t = 0; t < my_tiles; ++t, ++n) {
                const int kt = tile_at(t, my_tiles);
                const int buf = NB == 2 ? (int)(n & 1) : 0;
                const uint32_t tm_s = tm_lane + (uint32_t)(kKeys * (g * NB + buf) + KH * part);
                if (ok) ok = mbar_wait_hot(bar_s0 + 8 * buf, (NB == 2 ? (n >> 1) : n) & 1, p.wait_ns);
                ok = __all_sync(0xffffffffu, ok);
                // One tile of the group, from the scores in tensor memory to the weights handed to the MMA thread.
                // P goes in place of the scores: 16 keys' weights, two to a column, over the first half of those
                // keys' columns, low parts (bf16, where the weights go in two parts) over the second half.
                const int key0 = kt * kKeys + part * KH;
                const int lim = row - key0;                        // key index i is visible iff i <= lim
                const float bias0 = slope2 * (float)(key0 - row);
                const bool two = kSplitP && split_p_keys(row0, kt * kKeys, kKeys, slope_nat >= kSplitSlope);
                float alpha = 1.f;
                uint64_t ls = 0ull;
                int kept = 0;                                     // keys whose weights are stored
                // The reference in use nearly always stands behind the first tile: the weights are worked out and stored
                // with it in one pass over the scores; 16 (32) keys whose weights add up to more than 2^8 end the pass.  (That they
                // do is seen from their sum, which is needed anyhow: noting the maximum cost an instruction for every
                // two scores, on the chain that sets the pace.  Not where no key has been visible to a
                // row so far, nor under a negative slope, whose maximum grows from tile to tile towards the oldest key: there the
                // reference follows it exactly, so that the weight of the key that counts most is not rounded.)
                const bool fresh = t == 0 || slope2 < 0.f || __any_sync(0xffffffffu, m_ref == -INFINITY);
                const int seen = row0 + (warp & 3) * 32 + 32 - key0;       // keys that some row of the warp sees
                const bool mask = key0 + KH - 1 > row0 + (warp & 3) * 32;  // keys that some row of the warp does not see
                bool stands = false;
                if (!fresh) {
                    if (ok) {
                        tc_fence_after();
                        const float m_use = m_ref - kWeightShift<T>;
                        auto pass = [&](auto with_bias, auto masked, auto in_two) {
                            constexpr bool BIAS = decltype(with_bias)::value, MASK = decltype(masked)::value, SPLIT = decltype(in_two)::value;
                            uint32_t sr[KH > PC ? 2 : 1][PC];     // the next scores are on their way while these are worked on
                            if constexpr (PC == 32) tc_ld32(tm_s, sr[0]);
                            else tc_ld16(tm_s, sr[0]);
#pragma unroll
                            for (int c = 0; c < KH; c += PC) {
                                uint32_t* cur = sr[(c / PC) & 1];
                                tc_wait_ld();
                                pin<PC>(cur);
                                if (c + PC < KH) {
                                    if constexpr (PC == 32) tc_ld32(tm_s + c + PC, sr[KH > PC ? ((c / PC) & 1) ^ 1 : 0]);
                                    else tc_ld16(tm_s + c + PC, sr[KH > PC ? ((c / PC) & 1) ^ 1 : 0]);
                                }
                                uint32_t hi[PC / 2], lo[PC / 2];
                                uint64_t lp = 0ull;
#pragma unroll
                                for (int u = 0; u < PC; u += 16) {
                                    if (MASK && c + u >= seen) {  // keys beyond the warp's last row
#pragma unroll
                                        for (int i = 0; i < 8; ++i) hi[u / 2 + i] = lo[u / 2 + i] = 0u;
                                        continue;
                                    }
                                    const float c0 = (BIAS ? bias0 + slope2 * (float)(c + u) : 0.f) - m_use;
                                    const uint64_t ln = weigh16<T, BIAS, MASK, SPLIT>(cur + u, p.scale2, slope2, c0, lim - c - u, hi + u / 2, lo + u / 2);
                                    lp = u ? f2_add(lp, ln) : ln;
                                }
                                if (__any_sync(0xffffffffu, f2_lo(lp) + f2_hi(lp) > kWeightMax<T>)) break;
                                ls = f2_add(ls, lp);
#pragma unroll
                                for (int u = 0; u < PC; u += 16) {
                                    tc_st8(tm_s + c + u, hi + u / 2);
                                    if (SPLIT) tc_st8(tm_s + c + u + 8, lo + u / 2);
                                }
                                kept = c + PC;
                            }
                            tc_wait_ld();
                        };
                        // (with a bias there is no mask behind the first tile, see above)
                        constexpr std::integral_constant<bool, kSplitP> parts{};
                        constexpr std::true_type yes{};
                        constexpr std::false_type no{};
                        if (kSplitP && two) {
                            if (biased) pass(yes, no, parts);
                            else if constexpr (kKeys < kRows) pass(no, yes, parts);      // (else only the first tile's)
                        } else {
                            if (biased) pass(yes, no, no);
                            else if (mask) pass(no, yes, no);
                            else pass(no, no, no);
                        }
                    }
                    stands = bar_and(rows_bar, 32 * TPR, ok && kept == KH);
                }
                if (!stands) {
                    // A new reference, where the maximum of the keys that have no weights yet has grown by more than 2^4, or at all under a negative slope (those
                    // that have are below 2^8 of the one in use): the sum and O use the same reference, so the
                    // result is exact.  Keys beyond the last row of the warp take no part.
                    float tmax = -INFINITY;
                    if (ok) {
                        tc_fence_after();
#pragma unroll 1
                        for (int c = kept; c < KH && c < seen; c += 16) {
                            uint32_t sr[16];
                            tc_ld16(tm_s + c, sr);
                            tc_wait_ld();
                            pin<16>(sr);
                            // in log2 units; without a bias the scale is folded into the exponent's FMA
                            float m;
                            if (biased) m = mask ? max16<true, true>(sr, p.scale2, slope2, bias0 + slope2 * (float)c, lim - c)
                                                 : max16<true, false>(sr, p.scale2, slope2, bias0 + slope2 * (float)c, lim - c);
                            else m = (mask ? max16<false, true>(sr, p.scale2, slope2, 0.f, lim - c)
                                           : max16<false, false>(sr, p.scale2, slope2, 0.f, lim - c)) * p.scale2;
                            tmax = fmaxf(tmax, m);
                        }
                    }
                    xrow[part * kRows] = tmax;
                    ok = bar_and(rows_bar, 32 * TPR, ok);
                    gone = !ok;
                    if (gone) break;
#pragma unroll
                    for (int i = 0; i < TPR; ++i) tmax = fmaxf(tmax, xrow[i * kRows]);
                    const bool none = bar_and(rows_bar, 32 * TPR, kept == 0);
                    const bool need = tmax > m_ref + (slope2 < 0.f ? 0.f : 4.f), rescale = need && m_ref > -INFINITY;   // (O is zero so far, else)
                    if (need && none) {
                        alpha = exp2f(m_ref - tmax);              // 0 on the first keys
                        m_ref = tmax;
                    } else if (need) {
                        // Some of the rows' weights are stored: a whole number of powers of two further up, so that they move by
                        // their exponents alone and none is rounded a second time (read back, scaled by 2^(m_ref - tmax) and
                        // rounded again their error was half as large again).
                        const float up = ceilf(tmax - m_ref);
                        alpha = up < 127.f ? __uint_as_float((uint32_t)(127 - (int)up) << 23) : 0.f;
                        m_ref += up;
                    }
                    // (no visible key of this row so far: its weights are zeros with any reference)
                    const float m_use = (m_ref == -INFINITY ? 0.f : m_ref) - kWeightShift<T>;
                    // weights that are stored already, with the reference before
                    if (kept > 0) tc_wait_st();
                    ls = f2_mul(ls, f2(alpha, alpha));
#pragma unroll 1
                    for (int c = 0; c < kept; c += 16) {
                        uint32_t u[16];
                        tc_ld16(tm_s + c, u);
                        tc_wait_ld();
                        pin<16>(u);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float2 a = Mma<T>::unpack(u[i]);
                            u[i] = Mma<T>::pack(a.x * alpha, a.y * alpha);
                            if (kSplitP && two) {
                                const float2 e = Mma<T>::unpack(u[8 + i]);
                                u[8 + i] = Mma<T>::pack(e.x * alpha, e.y * alpha);
                            }
                        }
                        tc_st8(tm_s + c, u);
                        if (kSplitP && two) tc_st8(tm_s + c + 8, u + 8);
                    }
#pragma unroll 1
                    for (int c = kept; c < KH; c += 16) {
                        uint32_t sr[16], hi[8], lo[8];
                        if (c < seen) {
                            tc_ld16(tm_s + c, sr);
                            tc_wait_ld();
                            pin<16>(sr);
                            const float c0 = (biased ? bias0 + slope2 * (float)c : 0.f) - m_use;
                            uint64_t lp;
                            if (kSplitP && two) {
                                if (biased) lp = weigh16<T, true, true, kSplitP>(sr, p.scale2, slope2, c0, lim - c, hi, lo);
                                else lp = weigh16<T, false, true, kSplitP>(sr, p.scale2, slope2, c0, lim - c, hi, lo);
                            } else {
                                if (biased) lp = mask ? weigh16<T, true, true, false>(sr, p.scale2, slope2, c0, lim - c, hi, lo)
                                                      : weigh16<T, true, false, false>(sr, p.scale2, slope2, c0, lim - c, hi, lo);
                                else lp = mask ? weigh16<T, false, true, false>(sr, p.scale2, slope2, c0, lim - c, hi, lo)
                                               : weigh16<T, false, false, false>(sr, p.scale2, slope2, c0, lim - c, hi, lo);
                            }
                            ls = f2_add(ls, lp);
                        } else {
#pragma unroll
                            for (int i = 0; i < 8; ++i) hi[i] = lo[i] = 0u;
                        }
                        tc_st8(tm_s + c, hi);
                        if (kSplitP && two) tc_st8(tm_s + c + 8, lo);
                    }
                    // O is rescaled, a part of the row per thread, before this thread hands over its weights (the MMA thread waits
                    // for all of them), once P.V of the previous tile is done: after the weights, under which that P.V runs
                    if (t > 0 && __any_sync(0xffffffffu, rescale)) {
                        ok = mbar_wait_hot(bar_o, (n - 1) & 1, p.wait_ns);
                        ok = __all_sync(0xffffffffu, ok);
                        if (ok) {
                            tc_fence_after();
#pragma unroll 1
                            for (int c = 0; c < DH / 16; ++c) {
                                uint32_t orr[16];
                                tc_ld16(tm_o + c * 16, orr);
                                tc_wait_ld();
                                pin<16>(orr);
#pragma unroll
                                for (int i = 0; i < 16; ++i) orr[i] = __float_as_uint(__uint_as_float(orr[i]) * alpha);
                                tc_st16(tm_o + c * 16, orr);
                            }
                        }
                    }
                }
                l_run = l_run * alpha + (f2_lo(ls) + f2_hi(ls));
                // With one S buffer these scores were issued behind P.V of the previous tile, which keeps the O and P
                // barriers at the phases waited for; with two, where a thread could run two phases ahead of the
                // MMA thread, every phase of the O barrier is waited for in turn.
                if (NB == 2 && t > 0 && ok) {
                    ok = mbar_wait_hot(bar_o, (n - 1) & 1, p.wait_ns);
                    ok = __all_sync(0xffffffffu, ok);
                }
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0 && ok && !(p.dbg_skip && tid == 0 && n == 0)) mbar_arrive(bar_p);
            }
            if (gone) break;
            // the item's output: O / l, once the last P.V has landed.  The next item's first P.V
            // cannot overwrite O before these loads: it waits for this warp's next P arrival.
            if (ok) ok = mbar_wait_hot(bar_o, (n - 1) & 1, p.wait_ns);
            ok = __all_sync(0xffffffffu, ok);
            xrow[part * kRows] = l_run;
            ok = bar_and(rows_bar, 32 * TPR, ok);
            gone = !ok;
            if (gone) break;
            tc_fence_after();
            l_run = 0.f;
#pragma unroll
            for (int i = 0; i < TPR; ++i) l_run += xrow[i * kRows];
            bar_sync_n(rows_bar, 32 * TPR);
            const float inv = 1.f / l_run;
            // NP lanes trade 16-byte pieces of their rows, so that a store instruction writes 64 (32) bytes of each of 8 (16) rows
            // instead of 16 of 32: with one row per lane the stores of an item took 3400 clocks (6500 at head_dim 256).
            constexpr int EC = DH < 32 ? DH : 32, NP = EC / 8;    // columns at a time; pieces of a row and lanes that trade
            const int len = request_len(b), rowq = row0 + (r & ~(NP - 1));
            T* oq = reinterpret_cast<T*>(p.out) + ((size_t)b * p.N * p.H + h) * kD + (size_t)rowq * qstride + DH * part + (lane & (NP - 1)) * 8;
#pragma unroll 1
            for (int c = 0; c < DH / EC; ++c) {
                uint32_t orr[EC];
                if constexpr (EC == 32) tc_ld32(tm_o + c * EC, orr);
                else tc_ld16(tm_o + c * EC, orr);
                tc_wait_ld();
                pin<EC>(orr);
                uint32_t v[NP][4];                                // [piece][word]
#pragma unroll
                for (int i = 0; i < NP; ++i)
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        v[i][u] = Mma<T>::pack(__uint_as_float(orr[8 * i + 2 * u]) * inv, __uint_as_float(orr[8 * i + 2 * u + 1]) * inv);
#pragma unroll
                for (int x = 1; x < NP; x <<= 1) {                // an NP x NP transposition, an exchange per bit
                    const bool up = (lane & x) != 0;
#pragma unroll
                    for (int i = 0; i < NP; ++i) {
                        if (i & x) continue;
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const uint32_t t = __shfl_xor_sync(0xffffffffu, up ? v[i][u] : v[i | x][u], x);
                            if (up) v[i][u] = t;
                            else v[i | x][u] = t;
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < NP; ++i)
                    if (rowq + i < len)
                        *reinterpret_cast<uint4*>(oq + (size_t)i * qstride + c * EC) = make_uint4(v[i][0], v[i][1], v[i][2], v[i][3]);
            }
        }
        if (!ok && lane == 0) s_abort = 1;
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == L::kSoftWarps + 1) {
        if (s_abort && lane == 0) {
            // MMAs may still be in flight: let them finish (bounded) before the tensor memory goes back
            tc_commit(bar_end);
            (void)mbar_wait(bar_end, 0, p.wait_ns);
        }
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmemCols) : "memory");
        if (lane == 0 && s_abort) atomicOr(p.err_word, SEGKV_DEV_WAIT_LIMIT);
    }
}

// Are a launch's items dealt in pairs of query tiles of one (request, head) (round_item)?  What that gains is K and V found in the
// L2 by the other query tiles instead of read from HBM again: nothing where all of them stay there anyhow, little where a tile's
// arithmetic hides the reads.  What it costs is balance: the middle one of an odd number of query tiles has a CTA to itself, and
// whole rounds of bpw (request, head)s are dealt.  `share` is the busiest CTA's work in hundredths of the mean.  Pairs against
// longest-first, times of the attention alone in us: head_dim 128, 3 query tiles 16 x 56 x 768 294 / 235, 11 x 96 x 549 291 / 215; 5, 20 x 56 x
// 1280 740 / 690; 4, 32 x 56 x 1024 751 / 741; 8, 8 x 56 x 2048 606 / 643; 16, 6 x 56 x 4096 1548 / 1731; two query heads per kv head 8, 8 x 56 x
// 2048 592 / 598, four (117 MB of K and V) 587 / 576.  head_dim 256 (128-row items), 4, 16 x 32 x 500 150 / 166; 5, 125 x 16 x 640 913 / 864; 7, 16 x 16 x
// 900 207 / 251; 8, 16 x 16 x 1003 220 / 265; 32, 20 x 16 x 4096 3120 / 3916; eight query heads per kv head, 9, 16 x 56 x 1100 907 / 844, 16, 8 x 56 x
// 2048 1193 / 1236.  head_dim 64, 2, 36 x 56 x 500 213 / 205; 6, 15 x 56 x 1500 513 / 505; 8, 8 x 56 x 2048 (share 107) 458 / 453, 12 x 40 x 2048 with
// the store (share 100) 467 / 502; 12, 6 x 56 x 3072 684 / 719.  bf16 with ALiBi: head_dim 64
// 6 x 56 x 4096 1312 / 1265, 128 32 x 56 x 1024 837 / 840, 8 x 56 x 2048 640 / 660, 4 x 56 x 4000 1059 / 1137, 256 8 x 32 x 1024 211 / 248.
bool deal_in_pairs(const Dims& d, int prompt_len, bool biased, int nqt, int bpw, int sms) {
    const long hb = (long)d.heads * d.batch;
    const long share = 200L * sms * ((hb + bpw - 1) / bpw) / (hb * nqt);
    const bool in_l2 = 4LL * d.batch * d.kv_heads * prompt_len * d.head_dim < 150000000LL;      // (126 MB of it)
    const bool two_part = d.dtype == SEGKV_BF16 && biased;        // more work next to the diagonal
    switch (d.head_dim) {
        case 64: return nqt >= 4 && !in_l2 && !two_part && share <= (nqt >= 8 ? 104 : 102);
        case 128: return !in_l2 && (nqt >= 6 ? share <= 115 : !two_part && share <= 104);
        default: return share <= (in_l2 || nqt < 4 ? 104 : 120);
    }
}

template <typename T, typename L>
cudaError_t launch_tc5(const Dims& d, const PrefillArgs& a, Tc5Params p, int sms, cudaStream_t st) {
    constexpr int NG = L::NG;
    // Never two CTAs on one SM: each allocates all of tensor memory and keeps it while it walks
    // its items, so a second one would wait for it inside tcgen05.alloc.
    constexpr size_t smem = L::kBytes > 120 * 1024 ? L::kBytes : 120 * 1024;
    static bool configured[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(prefill_tc5_kernel<T, L, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(prefill_tc5_kernel<T, L, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(prefill_tc5_kernel<T, L, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    // instruction descriptors: fp32 accumulate, A/B format (the same for both operands: a P in fp16
    // against a V in bf16 is not a pair the f16 kind takes), operand majors, N >> 3, M >> 4
    const uint32_t fmt = d.dtype == SEGKV_BF16 ? 1u : 0u;
    const uint32_t common = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(kRows >> 4) << 24);
    p.idesc_qk = common | ((uint32_t)(L::KEYS >> 3) << 17);               // A, B both K-major; N = keys of a tile
    p.idesc_pv = common | (1u << 16) | ((uint32_t)(L::D >> 3) << 17);     // B (= V) MN-major; N = head_dim
    p.scale2 = 1.4426950408889634f / sqrtf((float)L::D);
    const long items = (long)((a.prompt_len + kRows * NG - 1) / (kRows * NG)) * d.heads * d.batch;
    const unsigned grid = (unsigned)(items < sms ? items : sms);  // one CTA per SM
    p.snake = items < 8L * sms;
    {
        const int nqt = (a.prompt_len + kRows * NG - 1) / (kRows * NG), ppb = (nqt + 1) / 2;
        const long hb_count = (long)d.heads * d.batch;
        const int bpw = ppb <= sms ? sms / ppb : 0;
        p.paired = (grid == (unsigned)sms && bpw > 0 && hb_count >= 4L * bpw && deal_in_pairs(d, a.prompt_len, p.slopes != nullptr, nqt, bpw, sms)) ? 1 : 0;
        p.rounds = p.paired ? 2 * (int)((hb_count + bpw - 1) / bpw) : (int)((items + grid - 1) / grid);
    }
    // fused prefill: load through the maps over the caller's arrays, store through the segment's
    const bool store = a.tm_k_src && a.tm_v_src;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(L::kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = a.pdl ? 1 : 0;
    if (store) return cudaLaunchKernelEx(&cfg, prefill_tc5_kernel<T, L, 1>, *a.tm_q, *a.tm_k_src, *a.tm_v_src, *a.tm_k, *a.tm_v, p);
    if (p.plens) return cudaLaunchKernelEx(&cfg, prefill_tc5_kernel<T, L, 2>, *a.tm_q, *a.tm_k, *a.tm_v, *a.tm_k, *a.tm_v, p);
    return cudaLaunchKernelEx(&cfg, prefill_tc5_kernel<T, L, 0>, *a.tm_q, *a.tm_k, *a.tm_v, *a.tm_k, *a.tm_v, p);
}

template <typename T>
cudaError_t dispatch_tc5(const Dims& d, const PrefillArgs& a, const Tc5Params& p, int sms, cudaStream_t st) {
    // two row groups per CTA once there are enough 256-row items to fill the machine a few times over
    const long items2 = (long)((a.prompt_len + 2 * kRows - 1) / (2 * kRows)) * d.heads * d.batch;
    const bool two = a.row_groups ? a.row_groups == 2 : items2 >= 2L * sms;
    switch (d.head_dim) {
        case 64:
            return two ? launch_tc5<T, Tc5Layout<64, 128, 2>>(d, a, p, sms, st)
                       : launch_tc5<T, Tc5Layout<64, 128, 1>>(d, a, p, sms, st);
        case 128:
            return two ? launch_tc5<T, Tc5Layout<128, 128, 2>>(d, a, p, sms, st)
                       : launch_tc5<T, Tc5Layout<128, 128, 1>>(d, a, p, sms, st);
        case 256:   // O alone takes 256 of the 512 columns: one group, 64-key tiles, S double-buffered
            return launch_tc5<T, Tc5Layout<256, 64, 1>>(d, a, p, sms, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

bool prefill_tc5_supported(const Dims& d) { return d.head_dim == 64 || d.head_dim == 128 || d.head_dim == 256; }

cudaError_t launch_prefill_tc5(const Dims& d, const PrefillArgs& a, cudaStream_t st) {
    if (!prefill_tc5_supported(d) || !a.tm_q) return cudaErrorInvalidValue;
    Tc5Params p;
    p.out = a.out; p.slopes = a.slopes; p.err_word = a.err_word;
    p.plens = a.plens;
    p.N = a.prompt_len; p.H = d.heads; p.G = d.group; p.B = d.batch;
    p.scale2 = 0.f; p.idesc_qk = p.idesc_pv = 0; p.snake = 0; p.paired = 0; p.rounds = 0;
    p.dbg_skip = a.dbg_skip ? 1 : 0;
    p.wait_ns = a.wait_ns ? a.wait_ns : kWaitLimitNs;
    int sms = 148;
    {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    return d.dtype == SEGKV_BF16 ? dispatch_tc5<__nv_bfloat16>(d, a, p, sms, st) : dispatch_tc5<__half>(d, a, p, sms, st);
}

}  // namespace segkv_impl
