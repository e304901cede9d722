// Placement constraints Phi_C: node-label loading and batched node-selector
// evaluation (Sec. 3.3 satisfaction (i); Sec. 4.1 placement directives;
// Sec. 5.5 compute check; Sec. 6.3 hallucinated identifiers; Sec. 5.3
// fail-closed unenforceable intents).
//
// Two exact kernels compute the same feasible-node bitsets:
//  * sel_cmp_kernel: label columns of a node tile are staged in shared
//    memory; a warp per pod sweeps 32 nodes at a time, tests each
//    expression against the node's value and emits one bitset word per
//    sweep with __ballot_sync.
//  * sel_rows_kernel: pv_load_cluster builds, for every (key, carried
//    value), the bitset of nodes carrying it, plus one "key present" row
//    per key.  An In expression is then the OR of its values' rows, NotIn
//    its complement, Exists / DoesNotExist the present row or its
//    complement, and a pod's row the AND over its expressions (in the term
//    form the OR of its terms' ANDs) -- 32 nodes per word operation, rows
//    read from L2 with 128-bit loads.  Warps own ranges of pods and resolve
//    the expressions of several pods at once, one per lane.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "pv_internal.cuh"

namespace {

constexpr uint32_t kInvWords = 2048;                  // 65536 value ids / 32
constexpr uint64_t kRowBudgetBytes = 2ull << 30;      // value-row memory budget
constexpr uint32_t kMaxKeys = 4096;

__host__ __device__ inline uint32_t words_for(uint32_t n) { return ((n + 127) / 128) * 4; }

// ---------------------------------------------------------------------------
// loading
// ---------------------------------------------------------------------------
__global__ void build_inventory_kernel(uint32_t N, uint32_t K, const uint16_t *__restrict__ labels,
                                       uint32_t *__restrict__ inv) {
    size_t total = (size_t)N * K;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        uint32_t k = (uint32_t)(i / N);
        uint16_t v = labels[i];
        if (v != PV_ABSENT) atomicOr(&inv[(size_t)k * kInvWords + (v >> 5)], 1u << (v & 31));
    }
}

// One block (1024 threads) per key: exclusive prefix popcount over the key's
// 2048 inventory words, stored beside them (a value's row then takes one
// load); count[k] = number of carried values.
__global__ void __launch_bounds__(1024) inventory_rank_kernel(const uint32_t *__restrict__ inv,
                                                              uint2 *__restrict__ ranked,
                                                              uint32_t *__restrict__ count) {
    __shared__ uint32_t s_warp[32];
    const uint32_t k = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t *w = inv + (size_t)k * kInvWords;
    uint32_t a = __popc(w[2 * t]), b = __popc(w[2 * t + 1]);
    uint32_t x = a + b, incl = x;
    for (int d = 1; d < 32; d <<= 1) {
        uint32_t y = __shfl_up_sync(PV_FULL_MASK, incl, d);
        if (lane >= (uint32_t)d) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t v = s_warp[lane], vi = v;
        for (int d = 1; d < 32; d <<= 1) {
            uint32_t y = __shfl_up_sync(PV_FULL_MASK, vi, d);
            if (lane >= (uint32_t)d) vi += y;
        }
        s_warp[lane] = vi - v;
        if (lane == 31) count[k] = vi;
    }
    __syncthreads();
    uint32_t excl = s_warp[warp] + incl - x;
    ranked[(size_t)k * kInvWords + 2 * t] = make_uint2(w[2 * t], excl);
    ranked[(size_t)k * kInvWords + 2 * t + 1] = make_uint2(w[2 * t + 1], excl + a);
}

// Single block: key_base = exclusive scan of count[0..K), key_base[K] = total.
__global__ void __launch_bounds__(1024) key_base_kernel(uint32_t K, const uint32_t *__restrict__ count,
                                                        uint32_t *__restrict__ base) {
    __shared__ uint32_t s_carry;
    __shared__ uint32_t s_warp[32];
    const uint32_t t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) s_carry = 0;
    __syncthreads();
    for (uint32_t c0 = 0; c0 < K; c0 += 1024) {
        uint32_t i = c0 + t;
        uint32_t x = i < K ? count[i] : 0, incl = x;
        for (int d = 1; d < 32; d <<= 1) {
            uint32_t y = __shfl_up_sync(PV_FULL_MASK, incl, d);
            if (lane >= (uint32_t)d) incl += y;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            uint32_t v = s_warp[lane], vi = v;
            for (int d = 1; d < 32; d <<= 1) {
                uint32_t y = __shfl_up_sync(PV_FULL_MASK, vi, d);
                if (lane >= (uint32_t)d) vi += y;
            }
            s_warp[lane] = vi - v;
        }
        __syncthreads();
        uint32_t excl = s_carry + s_warp[warp] + incl - x;
        if (i < K) base[i] = excl;
        __syncthreads();
        if (t == 1023) s_carry = excl + x;
        __syncthreads();
    }
    if (t == 0) base[K] = s_carry;
}

// The row of value v of key k, if some node carries it: the key's first row
// plus the carried values below v.
__device__ __forceinline__ uint32_t value_row(const uint2 *__restrict__ ranked,
                                              const uint32_t *__restrict__ key_base, uint32_t k, uint32_t v,
                                              bool *carried) {
    const uint2 w = __ldg(ranked + (size_t)k * kInvWords + (v >> 5));
    const uint32_t bit = v & 31;
    *carried = (w.x >> bit) & 1u;
    return __ldg(key_base + k) + w.y + __popc(w.x & ((1u << bit) - 1u));
}

// Value rows and present rows.  One warp covers 32 consecutive nodes of one
// key; present rows are written with a ballot, value rows with atomicOr.
__global__ void build_rows_kernel(uint32_t N, uint32_t K, const uint16_t *__restrict__ labels,
                                  const uint2 *__restrict__ ranked, const uint32_t *__restrict__ key_base,
                                  uint32_t num_value_rows, uint32_t row_words, uint32_t *__restrict__ rows) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t words = (N + 31) / 32;
    const size_t total_warps = (size_t)K * words;
    const size_t gw = (blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5;
    const size_t nw = ((size_t)gridDim.x * blockDim.x) >> 5;
    for (size_t i = gw; i < total_warps; i += nw) {
        uint32_t k = (uint32_t)(i / words), wd = (uint32_t)(i % words);
        uint32_t n = wd * 32 + lane;
        uint16_t v = n < N ? labels[(size_t)k * N + n] : (uint16_t)PV_ABSENT;
        uint32_t pres = __ballot_sync(PV_FULL_MASK, v != PV_ABSENT);
        if (lane == 0) rows[((size_t)num_value_rows + k) * row_words + wd] = pres;
        if (v != PV_ABSENT) {
            bool carried;
            uint32_t r = value_row(ranked, key_base, k, v, &carried);
            atomicOr(&rows[(size_t)r * row_words + wd], 1u << lane);
        }
    }
}

// ---------------------------------------------------------------------------
// expression checks shared by both kernels
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool expr_valid(const pv_expr &x, uint32_t K) {
    if (x.key >= K) return false;
    if (x.op == PV_IN || x.op == PV_NOTIN) {
        if (x.nvals < 1 || x.nvals > 8) return false;
        for (int j = 0; j < 8; ++j)
            if (j < x.nvals && x.vals[j] == PV_ABSENT) return false;
        return true;
    }
    if (x.op == PV_EXISTS || x.op == PV_DOESNOTEXIST) return x.nvals == 0;
    return false;
}

// Lane-parallel validation and hallucinated-value scan of pod p's list.
// Returns bit0 = bad, bit1 = unknown value.
__device__ __forceinline__ uint32_t pod_prescan(uint32_t lo, uint32_t hi, uint32_t num_exprs,
                                                const pv_expr *__restrict__ exprs, uint32_t K,
                                                const uint32_t *__restrict__ inv, uint32_t lane) {
    bool bad = hi < lo || hi > num_exprs;
    bool unknown = false;
    if (!bad) {
        for (uint32_t e = lo + lane; e < hi; e += 32) {
            pv_expr x = exprs[e];
            if (!expr_valid(x, K)) {
                bad = true;
                continue;
            }
            if (x.op == PV_IN)
                for (int j = 0; j < 8; ++j)
                    if (j < x.nvals) {
                        uint32_t v = x.vals[j];
                        if (!((inv[(size_t)x.key * kInvWords + (v >> 5)] >> (v & 31)) & 1u)) unknown = true;
                    }
        }
    }
    bad = __any_sync(PV_FULL_MASK, bad);
    unknown = __any_sync(PV_FULL_MASK, unknown);
    return (bad ? 1u : 0u) | (unknown ? 2u : 0u);
}

__device__ __forceinline__ uint8_t pod_flags(bool nonempty, bool unknown, bool has_assign, bool assign_ok) {
    uint8_t f = 0;
    if (!nonempty) f |= PV_F_EMPTY;
    if (unknown) f |= PV_F_UNKNOWN_VALUE;
    if (has_assign && assign_ok) {
        f |= PV_F_ASSIGN_OK;
        if (!unknown) f |= PV_F_PASS;
    }
    return f;
}

// ---------------------------------------------------------------------------
// kernel 1: per-node comparison over shared-memory label tiles
// ---------------------------------------------------------------------------
constexpr int kCmpThreads = 512;
constexpr int kCmpWarps = kCmpThreads / 32;
constexpr int kCmpPods = 128;   // pods per block
constexpr int kCmpCache = 8;    // expressions cached per warp

__global__ void __launch_bounds__(kCmpThreads) sel_cmp_kernel(
    uint32_t N, uint32_t K, const uint16_t *__restrict__ labels, uint32_t tile, uint32_t P,
    const uint32_t *__restrict__ offs, uint32_t num_exprs, const pv_expr *__restrict__ exprs,
    const uint32_t *__restrict__ assign, uint32_t *__restrict__ bits, uint32_t W, uint8_t *__restrict__ flags,
    const uint32_t *__restrict__ inv, const uint32_t *__restrict__ rep_of) {
    extern __shared__ uint16_t s_lab[];   // [K][tile]
    __shared__ uint8_t s_state[kCmpPods]; // bit0 nonempty, bit1 assign ok, bit2 bad, bit3 unknown
    __shared__ pv_expr s_ex[kCmpWarps][kCmpCache];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t p0 = blockIdx.x * kCmpPods;
    if (p0 >= P) return;
    const uint32_t np = min((uint32_t)kCmpPods, P - p0);
    const uint32_t nvalid_words = (N + 31) / 32;

    // per-pod validation / unknown scan (warp per pod)
    for (uint32_t pl = warp; pl < np; pl += kCmpWarps) {
        uint32_t p = p0 + pl;
        if (rep_of && rep_of[p] != p) continue;   // a duplicate: sel_copy_kernel writes it
        uint32_t r = pod_prescan(offs[p], offs[p + 1], num_exprs, exprs, K, inv, lane);
        if (lane == 0) s_state[pl] = (uint8_t)(((r & 1u) ? 4u : 0u) | ((r & 2u) ? 8u : 0u));
    }

    for (uint32_t n0 = 0; n0 < N; n0 += tile) {
        const uint32_t tn = min(tile, N - n0);
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < K * tile; i += kCmpThreads) {
            uint32_t k = i / tile, j = i - k * tile;
            s_lab[i] = j < tn ? labels[(size_t)k * N + n0 + j] : (uint16_t)PV_ABSENT;
        }
        __syncthreads();
        const uint32_t groups = (tn + 31) / 32;
        for (uint32_t pl = warp; pl < np; pl += kCmpWarps) {
            const uint32_t p = p0 + pl;
            if (rep_of && rep_of[p] != p) continue;
            const uint8_t st = s_state[pl];
            uint32_t *row = bits + (size_t)p * W + (n0 >> 5);
            if (st & 4u) {
                for (uint32_t g = lane; g < groups; g += 32) row[g] = 0;
                continue;
            }
            const uint32_t lo = offs[p], E = offs[p + 1] - lo;
            const bool cached = E <= (uint32_t)kCmpCache;
            if (cached) {
                if (lane < E) s_ex[warp][lane] = exprs[lo + lane];
                __syncwarp();
            }
            const uint32_t a = assign ? assign[p] : PV_UNPLACED;
            bool any = false, aok = false;
            for (uint32_t gb = 0; gb < groups; gb += 32) {
                uint32_t mine = 0;
                const uint32_t gend = min(groups, gb + 32);
                for (uint32_t g = gb; g < gend; ++g) {
                    const uint32_t j = g * 32 + lane;   // node offset within the tile
                    bool ok = j < tn;
                    for (uint32_t e = 0; e < E; ++e) {
                        const pv_expr &x = cached ? s_ex[warp][e] : exprs[lo + e];
                        const uint16_t v = s_lab[(uint32_t)x.key * tile + j];
                        const bool present = v != PV_ABSENT;
                        bool inset = false;
                        const uint32_t nv = x.nvals;
                        for (uint32_t q = 0; q < nv; ++q) inset |= (v == x.vals[q]);
                        bool m;
                        switch (x.op) {
                        case PV_IN: m = present && inset; break;
                        case PV_NOTIN: m = !present || !inset; break;
                        case PV_EXISTS: m = present; break;
                        default: m = !present; break;
                        }
                        ok = ok && m;
                    }
                    const uint32_t w = __ballot_sync(PV_FULL_MASK, ok);
                    if (lane == g - gb) mine = w;
                    const uint32_t node_base = n0 + g * 32;
                    if (a >= node_base && a < node_base + 32) aok = (w >> (a - node_base)) & 1u;
                }
                if (lane < gend - gb) row[gb + lane] = mine;
                any = any || __any_sync(PV_FULL_MASK, mine != 0);
            }
            __syncwarp();
            if (lane == 0) s_state[pl] = st | (any ? 1u : 0u) | (aok ? 2u : 0u);
        }
    }
    __syncthreads();
    // padding words and flags
    for (uint32_t pl = warp; pl < np; pl += kCmpWarps) {
        const uint32_t p = p0 + pl;
        if (rep_of && rep_of[p] != p) continue;
        for (uint32_t w = nvalid_words + lane; w < W; w += 32) bits[(size_t)p * W + w] = 0;
        if (lane == 0) {
            const uint8_t st = s_state[pl];
            flags[p] = (st & 4u) ? (uint8_t)PV_F_BAD_EXPR
                                 : pod_flags(st & 1u, st & 8u, assign != nullptr, st & 2u);
        }
    }
}

// ---------------------------------------------------------------------------
// kernel 2: per-(key, value) node-bitset rows
// ---------------------------------------------------------------------------

// A warp takes as many of its pods as have 32 expressions together and first
// resolves those, one per lane: validated, In values that no node carries
// flagged, and every expression turned into words of the warp's list in shared
// memory, one per row to OR; then it sweeps pod after pod,
// reading only the list and rows.  (Resolving one pod at a time kept most lanes
// idle in code of 300 instructions.)
// Threads per block: in the term form the pods' lengths differ more, and with
// half the block the first ones to finish leave room sooner (5,500 pods on
// 5,000 nodes 16.7 us with 256 threads, 15.8 with 128; the single-list form at
// 100,000 pods 68.7 and 72.8).  Three blocks of 256 per SM, or as much: 80
// registers without a spill; with four the term form at 100,000 pods took 113.8
// us instead of 97.1, with two of 128 registers 129.
template <bool kTerms>
constexpr int kRowsThreads = kTerms ? 128 : 256;
// A row's word is its byte offset (a multiple of 16 below 2^32) and the flags
// below.
constexpr uint32_t kRowLast = 1u;   // the expression's last row
constexpr uint32_t kRowNot = 2u;    // complement of the OR (NotIn, DoesNotExist)
constexpr uint32_t kRowTerm = 4u;   // the term's last row
constexpr int kAhead = 4;   // rows in flight (2: 72.1 us for the 100,000 pods, 3: 70.1, 4: 68.7, 6: 75.8)
constexpr uint32_t kListWords = 32 * 8;   // a group's rows at most
static_assert(kRowBudgetBytes < 1ull << 32, "rows and the row of no node have 32-bit byte offsets");

// One expression of at most eight rows, resolved by one lane.
struct LaneExpr {
    uint32_t off[8];       // byte offset of each listed value's row; off[0] alone for Exists / DoesNotExist
    uint32_t carried;      // bit j: off[j] is a row to OR
    uint32_t op;
    bool bad, unknown;
};

__device__ __forceinline__ void resolve_expr(LaneExpr &r, const pv_expr *__restrict__ x, uint32_t K,
                                             const uint2 *__restrict__ ranked,
                                             const uint32_t *__restrict__ key_base, uint32_t num_value_rows,
                                             uint32_t row_bytes) {
    uint32_t w[5];   // 20-byte records: 32-bit loads unless the caller's array is only 2-byte aligned
    if (((uintptr_t)x & 3) == 0) {
#pragma unroll
        for (int i = 0; i < 5; ++i) w[i] = __ldg(reinterpret_cast<const uint32_t *>(x) + i);
    } else {
        const uint16_t *h = reinterpret_cast<const uint16_t *>(x);
#pragma unroll
        for (int i = 0; i < 5; ++i) w[i] = (uint32_t)__ldg(h + 2 * i) | (uint32_t)__ldg(h + 2 * i + 1) << 16;
    }
    const uint32_t k = w[0] & 0xFFFFu, op = (w[0] >> 16) & 0xFFu, nv = w[0] >> 24;
    const bool listed = op == PV_IN || op == PV_NOTIN;
    r.op = op;
    r.bad = k >= K || (listed ? nv < 1 || nv > 8 : (op == PV_EXISTS || op == PV_DOESNOTEXIST) ? nv != 0 : true);
    r.unknown = false;
    r.carried = 0;
    if (r.bad) return;
    if (!listed) {
        r.off[0] = (num_value_rows + k) * row_bytes;
        r.carried = 1;
        return;
    }
    uint2 e[8];   // the values' inventory words, all in flight
#pragma unroll
    for (uint32_t j = 0; j < 8; ++j) {
        const uint32_t v = (w[1 + j / 2] >> (16 * (j & 1))) & 0xFFFFu;
        e[j] = j < nv ? __ldg(ranked + (size_t)k * kInvWords + (v >> 5)) : make_uint2(0, 0);
    }
    const uint32_t base = __ldg(key_base + k);
#pragma unroll
    for (uint32_t j = 0; j < 8; ++j) {
        const uint32_t v = (w[1 + j / 2] >> (16 * (j & 1))) & 0xFFFFu, bit = v & 31;
        const bool used = j < nv, has = used && ((e[j].x >> bit) & 1u);
        r.bad = r.bad || (used && v == PV_ABSENT);
        r.unknown = r.unknown || (used && !has && op == PV_IN);
        r.carried |= has ? 1u << j : 0u;
        r.off[j] = (base + e[j].y + __popc(e[j].x & ((1u << bit) - 1u))) * row_bytes;
    }
}

// Clears the bits of nodes >= N in the four words from w0.
__device__ __forceinline__ void clip_rows4(uint4 &acc, uint32_t w0, uint32_t N) {
    const uint32_t full_words = N >> 5, tail_bits = N & 31;
    uint32_t *aw = &acc.x;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t w = w0 + i;
        if (w > full_words || (w == full_words && tail_bits == 0)) aw[i] = 0;
        else if (w == full_words) aw[i] &= (1u << tail_bits) - 1u;
    }
}

struct SelArgs {
    uint32_t N, K, P;
    const uint32_t *offs;        // pod -> expressions (or terms)
    const uint32_t *term_offs;   // term -> expressions (multi-term form)
    uint32_t num_terms, num_exprs;
    const pv_expr *exprs;
    const uint32_t *assign;
    uint32_t *bits;
    uint32_t W;
    uint8_t *flags;
    const uint32_t *inv;
    const uint2 *ranked;
    const uint32_t *key_base, *rows;
    uint32_t row_words, num_value_rows, zero_row;   // zero_row: byte offset of the row of no node
    const uint32_t *pod_list, *list_len;   // with a list: only the pods it names
};

// A lane's share of the 160-word span from word sb: byte offsets of its chunk
// and its word within a row, and the bits of theirs that are nodes (a lane past
// the rows reads a word of theirs and keeps nothing).
struct RowSpan {
    uint4 m0;
    uint32_t m1, b0, b1;
};
__device__ __forceinline__ RowSpan row_span(uint32_t sb, uint32_t lane, uint32_t N, uint32_t W, uint32_t row_words) {
    const uint32_t q = sb / 4 + lane, w = sb + 128 + lane;
    const bool in0 = q * 4 < row_words && q * 4 < W, in1 = w < row_words && w < W;
    RowSpan s;
    s.b0 = in0 ? q * 16 : 0u;
    s.b1 = in1 ? w * 4 : 0u;
    s.m0 = in0 ? make_uint4(~0u, ~0u, ~0u, ~0u) : make_uint4(0, 0, 0, 0);
    if (in0 && q * 4 + 4 > N >> 5) clip_rows4(s.m0, q * 4, N);
    s.m1 = !in1 || w > N >> 5 ? 0u : w == N >> 5 ? (1u << (N & 31)) - 1u : ~0u;
    return s;
}

// Expressions first .. first + count - 1 (at most 32), resolved one per lane into
// the warp's list as they are given; bit e of term_ends: expression e is its term's
// last.  Returns the list's words; adds 1 (bad) and 2 (unknown value) to pre.
__device__ __forceinline__ uint32_t resolve_list(const SelArgs &g, uint32_t first, uint32_t count, uint32_t term_ends,
                                                 uint32_t lane, uint32_t *list, uint32_t &pre) {
    LaneExpr r;
    r.carried = 0;
    r.op = 0;
    r.bad = r.unknown = false;
    const bool on = lane < count;
    if (on) resolve_expr(r, g.exprs + first + lane, g.K, g.ranked, g.key_base, g.num_value_rows, g.row_words * 4);
    const uint32_t n = on ? max(__popc(r.carried), 1) : 0u;
    uint32_t incl = n;
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(PV_FULL_MASK, incl, d);
        if (lane >= (uint32_t)d) incl += y;
    }
    pre |= __any_sync(PV_FULL_MASK, r.bad) ? 1u : 0u;
    pre |= __any_sync(PV_FULL_MASK, r.unknown) ? 2u : 0u;
    __syncwarp();   // the list before is done with
    if (on) {
        uint32_t pos = incl - n;
        const uint32_t fl = r.op == PV_NOTIN || r.op == PV_DOESNOTEXIST ? kRowNot : 0u;
        const uint32_t last = kRowLast | ((term_ends >> lane) & 1u ? kRowTerm : 0u);
        if (r.carried == 0) list[pos] = g.zero_row | fl | last;
#pragma unroll
        for (uint32_t j = 0; j < 8; ++j)
            if ((r.carried >> j) & 1u) list[pos++] = r.off[j] | fl | (r.carried >> j == 1u ? last : 0u);
    }
    __syncwarp();
    return __shfl_sync(PV_FULL_MASK, incl, 31);
}

// A list's expressions ANDed into the lane's words a, and a into r at each
// term's last one (kTerms), kBatch rows loaded at once.
template <bool kTerms, int kBatch>
__device__ __forceinline__ void fold_list(const SelArgs &g, const uint32_t *list, uint32_t total, const RowSpan &sp,
                                          uint4 &a0, uint32_t &a1, uint4 &r0, uint32_t &r1) {
    const uint8_t *rb = reinterpret_cast<const uint8_t *>(g.rows);
    uint4 v0 = make_uint4(0, 0, 0, 0);   // the OR of the expression's rows
    uint32_t v1 = 0;
    for (uint32_t x = 0; x < total; x += kBatch) {
        uint4 n0[kBatch];
        uint32_t n1[kBatch], ent[kBatch];
#pragma unroll
        for (uint32_t i = 0; i < kBatch; ++i) {
            ent[i] = list[min(x + i, total - 1)];
            const uint32_t off = ent[i] & ~15u;
            n0[i] = __ldg(reinterpret_cast<const uint4 *>(rb + (size_t)(off + sp.b0)));
            n1[i] = __ldg(reinterpret_cast<const uint32_t *>(rb + (size_t)(off + sp.b1)));
        }
#pragma unroll
        for (uint32_t i = 0; i < kBatch; ++i) {
            if (x + i >= total) break;
            v0.x |= n0[i].x; v0.y |= n0[i].y; v0.z |= n0[i].z; v0.w |= n0[i].w;
            v1 |= n1[i];
            if (!(ent[i] & kRowLast)) continue;
            const uint32_t inv = ent[i] & kRowNot ? ~0u : 0u;
            a0.x &= v0.x ^ inv; a0.y &= v0.y ^ inv; a0.z &= v0.z ^ inv; a0.w &= v0.w ^ inv;
            a1 &= v1 ^ inv;
            v0 = make_uint4(0, 0, 0, 0);
            v1 = 0;
            if (kTerms && (ent[i] & kRowTerm)) {
                r0.x |= a0.x; r0.y |= a0.y; r0.z |= a0.z; r0.w |= a0.w;
                r1 |= a1;
                a0 = sp.m0;
                a1 = sp.m1;
            }
        }
    }
}

// The AND into the lane's words of the expressions [first, past), 32 at a time.
template <int kBatch>
__device__ __forceinline__ void and_exprs(const SelArgs &g, uint32_t first, uint32_t past, const RowSpan &sp, uint32_t lane,
                                          uint32_t *list, uint4 &a0, uint32_t &a1) {
    for (uint32_t left = past - first; left; first += 32, left -= min(left, 32u)) {
        uint32_t pre = 0, none = 0;
        const uint32_t total = resolve_list(g, first, min(left, 32u), 0u, lane, list, pre);
        uint4 unused = make_uint4(0, 0, 0, 0);
        fold_list<false, kBatch>(g, list, total, sp, a0, a1, unused, none);
        if (!__any_sync(PV_FULL_MASK, (a0.x | a0.y | a0.z | a0.w | a1) != 0)) break;
    }
}

// Stores a pod's row in one span; true when the lane's words hold the assigned
// node a and it is in the row.
__device__ __forceinline__ bool put_span(uint32_t *row, uint32_t sb, uint32_t lane, uint32_t W, uint32_t N, uint32_t a,
                                         const uint4 &r0, uint32_t r1) {
    const uint32_t q = sb / 4 + lane, w = sb + 128 + lane;
    if (q * 4 < W) reinterpret_cast<uint4 *>(row)[q] = r0;
    if (w < W) row[w] = r1;
    const uint32_t at = (a >> 5) - sb;   // the assigned node's word in the span
    if (a >= N || at >= 160 || lane != (at < 128 ? at >> 2 : at - 128)) return false;
    const uint32_t word = at >= 128 ? r1 : at & 2u ? (at & 1u ? r0.w : r0.z) : (at & 1u ? r0.y : r0.x);
    return (word >> (a & 31)) & 1u;
}

// A pod with a malformed list, a bad expression or more than 32 of them:
// validated and scanned for unknown values, then evaluated by and_exprs.
// (After a warp's other pods, so that its code costs them no registers; kPodLeft
// in the flags marks it until then.)  Expression by expression, each value's row
// found as it was read, 5,000 pods of 33 to 64 expressions on 5,000 nodes took 253 us,
// 69 resolved 32 at a time.
constexpr uint8_t kPodLeft = 0x80;
// kPodWarp: the copy of sel_terms_kernel, which has fewer registers (one copy for both
// cost sel_rows_kernel 1 to 2%).
template <bool kTerms, bool kPodWarp>
__device__ __noinline__ void unresolved_pod(const SelArgs &g, uint32_t p, uint32_t *list) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t o0 = g.offs[p], o1 = g.offs[p + 1], W = g.W, N = g.N, a = g.assign ? g.assign[p] : PV_UNPLACED;
    uint32_t pre;
    if (!kTerms) {
        pre = pod_prescan(o0, o1, g.num_exprs, g.exprs, g.K, g.inv, lane);
    } else {
        pre = o1 < o0 || o1 > g.num_terms ? 1u : 0u;
        for (uint32_t k = o0; k < o1 && !(pre & 1u); ++k)
            pre |= pod_prescan(g.term_offs[k], g.term_offs[k + 1], g.num_exprs, g.exprs, g.K, g.inv, lane);
    }
    const uint4 none = make_uint4(0, 0, 0, 0);
    uint32_t *row = g.bits + (size_t)p * W;
    bool any = false, aok = false;
    for (uint32_t sb = 0; sb < W; sb += 160) {
        const RowSpan sp = row_span(sb, lane, N, W, g.row_words);
        uint4 r0 = pre & 1u ? none : sp.m0;   // an empty row, or every node
        uint32_t r1 = pre & 1u ? 0u : sp.m1;
        if (pre & 1u) {
        } else if (!kTerms) {
            and_exprs<4>(g, o0, o1, sp, lane, list, r0, r1);
        } else if (o1 > o0) {
            r0 = none;
            r1 = 0;
            for (uint32_t k = o0; k < o1; ++k) {
                const uint32_t first = g.term_offs[k], past = g.term_offs[k + 1];
                if (past <= first) continue;
                uint4 a0 = sp.m0;
                uint32_t a1 = sp.m1;
                and_exprs<1>(g, first, past, sp, lane, list, a0, a1);   // (more rows at once: sel_rows_kernel spills)
                r0.x |= a0.x; r0.y |= a0.y; r0.z |= a0.z; r0.w |= a0.w;
                r1 |= a1;
            }
        }
        any = any || (r0.x | r0.y | r0.z | r0.w | r1) != 0;
        aok = put_span(row, sb, lane, W, N, a, r0, r1) || aok;
    }
    any = __any_sync(PV_FULL_MASK, any);
    aok = __any_sync(PV_FULL_MASK, aok);
    if (lane == 0)
        g.flags[p] = pre & 1u ? (uint8_t)PV_F_BAD_EXPR : pod_flags(any, pre & 2u, g.assign != nullptr, aok);
}

// The term form with one pod to a warp and 40 warps an SM, for as many pods as
// that many warps and more than sel_rows_kernel has warps for: there some of its
// warps take two pods and the launch waits for them.  3,700 / 4,500 / 5,400 / 6,000
// pods, us, a pod a warp against sel_rows_kernel: 5,000 nodes 12.8 / 12.8 / 14.3 /
// 16.7 against 16.3 / 16.6 / 16.5 / 18.6, 1,000 nodes 12.8 / 12.8 / 12.8 / 14.8 against
// 14.7 / 16.7 / 16.0 / 16.9, 12,000 29.0 / 29.0 / 29.1 / 35.2 against 31.0 / 35.1 /
// 33.2 / 39.3.  Bound by one pod's chain of loads; three rows at once are what 48
// registers hold without spilling in the loop.
constexpr int kPodThreads = 128;
__global__ void __launch_bounds__(kPodThreads, 1280 / kPodThreads) sel_terms_kernel(const __grid_constant__ SelArgs g) {
    __shared__ uint32_t s_list[kPodThreads / 32][kListWords];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, p = blockIdx.x * (kPodThreads / 32) + warp;
    if (p >= g.P) return;
    uint32_t *list = s_list[warp];
    const uint32_t o0 = g.offs[p], o1 = g.offs[p + 1], n = o1 - o0;
    const uint32_t a = g.assign ? g.assign[p] : PV_UNPLACED;
    // lane i: start of term i (lane n: the last one's end); a pod of more than 31
    // terms, with decreasing offsets or more than 32 expressions is left
    bool left = o1 < o0 || o1 > g.num_terms || n > 31;
    uint32_t off = 0, pre = 0, first = 0, count = 0, ends = 0;
    if (!left && n) {
        off = g.term_offs[o0 + min(lane, n)];
        const uint32_t before = __shfl_up_sync(PV_FULL_MASK, off, 1);
        first = __shfl_sync(PV_FULL_MASK, off, 0);
        const uint32_t past = __shfl_sync(PV_FULL_MASK, off, n);
        left = __any_sync(PV_FULL_MASK, lane && off < before) || past > g.num_exprs || past - first > 32;
        count = past - first;
        if (!left) ends = __reduce_or_sync(PV_FULL_MASK, lane && off > before ? 1u << (off - first - 1) : 0u);
    }
    uint32_t total = 0;
    if (!left) {
        total = resolve_list(g, first, count, ends, lane, list, pre);
        left = pre & 1u;   // a bad expression: validated again, in order
    }
    if (left) {   // (warp-uniform, as every condition above)
        unresolved_pod<true, true>(g, p, list);
        return;
    }
    bool any = false, aok = false;
    for (uint32_t sb = 0; sb < g.W; sb += 160) {
        const RowSpan sp = row_span(sb, lane, g.N, g.W, g.row_words);
        uint4 a0 = sp.m0, r0 = n ? make_uint4(0, 0, 0, 0) : sp.m0;   // no terms: every node
        uint32_t a1 = sp.m1, r1 = n ? 0u : sp.m1;
        fold_list<true, 3>(g, list, total, sp, a0, a1, r0, r1);
        any = any || (r0.x | r0.y | r0.z | r0.w | r1) != 0;
        aok = put_span(g.bits + (size_t)p * g.W, sb, lane, g.W, g.N, a, r0, r1) || aok;
    }
    any = __any_sync(PV_FULL_MASK, any);
    aok = __any_sync(PV_FULL_MASK, aok);
    if (lane == 0) g.flags[p] = pod_flags(any, pre & 2u, g.assign != nullptr, aok);
}

// A pod's row is the AND over its expressions, or, with kTerms (Kubernetes
// required node affinity), the OR over its terms of the AND over each term's
// expressions: a pod without terms admits every node, a term without
// expressions matches none.  The AND does not depend on the order: In
// expressions with the fewest carried values first, then DoesNotExist, Exists
// and NotIn, the sparsest sets first, so that a pod whose row empties early
// stops reading rows.
// kOneSpan: rows of at most 160 words (5,120 nodes), one pass over a pod's
// entries.
// What bounds it: instruction issue with many pods (about two thirds of the
// slots at 100,000 pods, the rows coming from L2), with few the chain offsets
// -> expressions -> inventory -> rows of one pod.  On 5,000 nodes against a
// warp per pod that resolved one pod at a time and loaded two rows ahead:
// 100,000 pods 101.8 -> 72.4 us, 10,000 19.0 -> 15.6, 777 12.2 -> 10.3; in the
// term form 129.6 -> 97, 22.1 -> 18.9 and 14.0 -> 11.1.
template <bool kTerms, bool kOneSpan>
__global__ void __launch_bounds__(kRowsThreads<kTerms>, 768 / kRowsThreads<kTerms>)
    sel_rows_kernel(const __grid_constant__ SelArgs g) {
    constexpr int kWarps = kRowsThreads<kTerms> / 32;
    __shared__ uint32_t s_list[kWarps][kListWords];
    __shared__ uint4 s_pod[kWarps][32];
    __shared__ uint32_t s_word[kWarps][32];   // the word of each pod's row that holds its assigned node
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, N = g.N, W = g.W;
    uint32_t *list = s_list[warp];
    const uint32_t total = g.pod_list ? *g.list_len : g.P;
    const uint32_t gw = blockIdx.x * kWarps + warp, nw = gridDim.x * kWarps;
    const uint32_t end = (uint32_t)(((uint64_t)total * (gw + 1)) / nw);
    uint32_t take = 0;
    RowSpan sp = row_span(0, lane, N, W, g.row_words);
    const uint32_t begin = (uint32_t)(((uint64_t)total * gw) / nw);
    bool left_over = false;
    for (uint32_t at = begin; at < end; at += take) {
        // lane i: pod at + i, its expressions [lo, lo + cnt); a pod with a
        // malformed list or more than 32 takes no slots and is evaluated
        // unresolved
        uint32_t p = 0, o0 = 0, o1 = 0, lo = 0, cnt = 0, a = PV_UNPLACED;
        uint32_t t1 = 0, t2 = 0, t3 = 0;   // kTerms: ends of the first three terms
        bool slow = false;
        if (at + lane < end) {
            p = g.pod_list ? g.pod_list[at + lane] : at + lane;
            o0 = lo = g.offs[p];
            o1 = g.offs[p + 1];
            if (g.assign) a = g.assign[p];
            uint32_t hi = o1;
            slow = o1 < o0 || o1 > (kTerms ? g.num_terms : g.num_exprs);
            if (kTerms) {
                // the terms' expressions form one range when their offsets do not decrease
                lo = hi = 0;
                if (o1 > o0 && !slow) {
                    // up to four terms' ends in flight (the last one's repeated)
                    const uint32_t last = o1;
                    lo = g.term_offs[o0];
                    t1 = g.term_offs[o0 + 1];
                    t2 = g.term_offs[min(o0 + 2, last)];
                    t3 = g.term_offs[min(o0 + 3, last)];
                    hi = g.term_offs[min(o0 + 4, last)];
                    slow = t1 < lo || t2 < t1 || t3 < t2 || hi < t3;
                    for (uint32_t k = o0 + 4; k < o1 && !slow; ++k) {
                        const uint32_t x = g.term_offs[k + 1];
                        slow = x < hi;
                        hi = x;
                    }
                    slow = slow || hi > g.num_exprs;
                }
            }
            slow = slow || hi - lo > 32;
            cnt = slow ? 0u : hi - lo;
        }
        uint32_t incl = cnt;
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(PV_FULL_MASK, incl, d);
            if (lane >= (uint32_t)d) incl += y;
        }
        const uint32_t fit = __ballot_sync(PV_FULL_MASK, at + lane < end && incl <= 32);   // leading lanes, the first always
        take = fit == PV_FULL_MASK ? 32u : (uint32_t)__ffs(~fit) - 1u;
        const uint32_t slots = __shfl_sync(PV_FULL_MASK, incl, take - 1), excl = incl - cnt;
        // lane t: expression t of the group, of pod `pod`
        uint32_t pod = 0;   // the first whose expressions end past t
#pragma unroll
        for (uint32_t step = 16; step; step >>= 1)
            if (__shfl_sync(PV_FULL_MASK, incl, pod + step - 1) <= lane) pod += step;
        pod = min(pod, 31u);   // lanes past the slots: unused
        const uint32_t f = __shfl_sync(PV_FULL_MASK, excl, pod), c = __shfl_sync(PV_FULL_MASK, cnt, pod);
        const uint32_t e = __shfl_sync(PV_FULL_MASK, lo, pod) + lane - f;
        uint32_t term = 0;   // e's term among the pod's
        if (kTerms) {
            const uint32_t tm0 = __shfl_sync(PV_FULL_MASK, o0, pod), tm1 = __shfl_sync(PV_FULL_MASK, o1, pod);
            term = (e >= __shfl_sync(PV_FULL_MASK, t1, pod) ? 1u : 0u) + (e >= __shfl_sync(PV_FULL_MASK, t2, pod) ? 1u : 0u) +
                   (e >= __shfl_sync(PV_FULL_MASK, t3, pod) ? 1u : 0u);
            if (lane < slots && tm1 - tm0 > 4 && term == 3)
                while (g.term_offs[tm0 + term + 1] <= e) ++term;
        }
        LaneExpr r;
        r.carried = 0;
        r.op = 0;
        r.bad = r.unknown = false;
        uint32_t key = 0, n = 0;
        if (lane < slots) {
            resolve_expr(r, g.exprs + e, g.K, g.ranked, g.key_base, g.num_value_rows, g.row_words * 4);
            const uint32_t cls = r.op == PV_IN ? 0u : r.op == PV_DOESNOTEXIST ? 1u : r.op == PV_EXISTS ? 2u : 3u;
            const uint32_t rows = __popc(r.carried);
            n = max(rows, 1u);   // (no value carried: the row of no node)
            key = term << 6 | cls << 4 | rows;
        }
        const uint32_t bad = __ballot_sync(PV_FULL_MASK, r.bad), unknown = __ballot_sync(PV_FULL_MASK, r.unknown);
        // the list: pods in order, each one's expressions in evaluation order
        uint32_t ni = n;
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(PV_FULL_MASK, ni, d);
            if (lane >= (uint32_t)d) ni += y;
        }
        uint32_t pos = __shfl_sync(PV_FULL_MASK, ni - n, f & 31u);   // the pod's first word
        bool term_end = true;
        const uint32_t most = __reduce_max_sync(PV_FULL_MASK, lane < slots ? c : 0u);
        for (uint32_t j = 0; j < most; ++j) {
            const uint32_t y = (f + j) & 31u, ky = __shfl_sync(PV_FULL_MASK, key, y), ny = __shfl_sync(PV_FULL_MASK, n, y);
            if (j < c && y != lane) {
                const bool before = ky < key || (ky == key && y < lane);
                if (before) pos += ny;
                else if (kTerms && ky >> 6 == term) term_end = false;
            }
        }
        if (lane < slots) {
            const uint32_t fl = r.op == PV_NOTIN || r.op == PV_DOESNOTEXIST ? kRowNot : 0u;
            const uint32_t last = kRowLast | (kTerms && term_end ? kRowTerm : 0u);
            if (r.carried == 0) list[pos] = g.zero_row | fl | last;
#pragma unroll
            for (uint32_t j = 0; j < 8; ++j)
                if ((r.carried >> j) & 1u) list[pos++] = r.off[j] | fl | (r.carried >> j == 1u ? last : 0u);
        }
        // lane i: pod i {index, words first | past << 16, assigned node, it has terms}
        const uint32_t ent0 = __shfl_sync(PV_FULL_MASK, ni - n, excl & 31u);
        const uint32_t ent1 = __shfl_sync(PV_FULL_MASK, ni, (incl - 1u) & 31u);
        const uint32_t span = cnt >= 32 ? PV_FULL_MASK : ((1u << cnt) - 1u) << (excl & 31u);
        uint32_t pre = (cnt && (bad & span) ? 1u : 0u) | (cnt && (unknown & span) ? 2u : 0u);
        s_pod[warp][lane] = make_uint4(p, cnt ? ent0 | ent1 << 16 : 0u, a, o1 > o0 ? 1u : 0u);
        s_word[warp][lane] = 0;
        const uint32_t group = take == 32 ? PV_FULL_MASK : (1u << take) - 1u;
        const uint32_t plain = __ballot_sync(PV_FULL_MASK, !slow && !(pre & 1u)) & group;
        uint32_t feasible = 0;   // pods with a feasible node
        __syncwarp();
        for (uint32_t todo = plain; todo; todo &= todo - 1u) {
            const uint32_t i = (uint32_t)__ffs(todo) - 1u;
            const uint4 pod = s_pod[warp][i];
            uint32_t *row = g.bits + (size_t)pod.x * W;
            bool any = false;
            // of each 160-word span a lane takes chunk lane (words 4 lane ..
            // 4 lane + 3) and word 128 + lane: five words per lane, so a row of
            // up to 5,120 nodes keeps every lane busy in one pass
            for (uint32_t sb = 0; kOneSpan ? sb == 0 : sb < W; sb += 160) {
                if (!kOneSpan) sp = row_span(sb, lane, N, W, g.row_words);
                uint4 a0 = sp.m0;   // the AND of the expressions, from the words' nodes
                uint32_t a1 = sp.m1;
                uint4 r0 = a0;      // kTerms: the OR of the terms; no terms: every node
                uint32_t r1 = a1;
                if (kTerms && pod.w) {
                    r0 = make_uint4(0, 0, 0, 0);
                    r1 = 0;
                }
                bool left = true;   // some node of the span is left
                const uint8_t *rb = reinterpret_cast<const uint8_t *>(g.rows);
                uint32_t x = pod.y & 0xFFFFu;
                const uint32_t x1 = pod.y >> 16;
                // rows are loaded kAhead entries ahead, across expressions
                uint4 n0[kAhead];
                uint32_t n1[kAhead];
                auto load = [&](int s, uint32_t at) {
                    if (at < x1) {
                        const uint32_t off = list[at] & ~15u;
                        n0[s] = __ldg(reinterpret_cast<const uint4 *>(rb + (size_t)(off + sp.b0)));
                        n1[s] = __ldg(reinterpret_cast<const uint32_t *>(rb + (size_t)(off + sp.b1)));
                    }
                };
                while (x < x1) {
#pragma unroll
                    for (int s = 0; s < kAhead; ++s) {
                        n0[s] = make_uint4(0, 0, 0, 0);
                        n1[s] = 0;
                        load(s, x + s);
                    }
                    uint4 v0 = make_uint4(0, 0, 0, 0);   // the OR of the expression's rows
                    uint32_t v1 = 0;
                    bool on = true;
                    while (on) {
#pragma unroll
                        for (int s = 0; s < kAhead; ++s) {
                            const uint32_t ent = list[x];
                            v0.x |= n0[s].x; v0.y |= n0[s].y; v0.z |= n0[s].z; v0.w |= n0[s].w;
                            v1 |= n1[s];
                            load(s, x + kAhead);
                            ++x;
                            if (!(ent & kRowLast)) continue;
                            const uint32_t inv = ent & kRowNot ? ~0u : 0u;
                            a0.x &= v0.x ^ inv; a0.y &= v0.y ^ inv; a0.z &= v0.z ^ inv; a0.w &= v0.w ^ inv;
                            a1 &= v1 ^ inv;
                            v0 = make_uint4(0, 0, 0, 0);
                            v1 = 0;
                            left = __any_sync(PV_FULL_MASK, (a0.x | a0.y | a0.z | a0.w | a1) != 0);
                            on = x < x1;
                            if (!kTerms) {
                                if (!left) x = x1;
                                on = on && left;
                            } else if (!left || (ent & kRowTerm)) {
                                r0.x |= a0.x; r0.y |= a0.y; r0.z |= a0.z; r0.w |= a0.w;
                                r1 |= a1;
                                a0 = sp.m0;
                                a1 = sp.m1;
                                if (!(ent & kRowTerm)) {
                                    // no node is left and the term's other sets cannot add
                                    // one back: the next term comes first
                                    while (!(list[x++] & kRowTerm)) {}
                                    on = false;
                                }
                            }
                            if (!on) break;
                        }
                    }
                }
                if (kTerms) {
                    left = __any_sync(PV_FULL_MASK, (r0.x | r0.y | r0.z | r0.w | r1) != 0);
                } else {
                    r0 = a0;
                    r1 = a1;
                }
                any = any || left;
                const uint32_t q = sb / 4 + lane, w = sb + 128 + lane;
                if (q * 4 < W) reinterpret_cast<uint4 *>(row)[q] = r0;
                if (w < W) row[w] = r1;
                const uint32_t at_word = (pod.z >> 5) - sb;   // of the assigned node, in the span
                if (at_word < 160 && lane == (at_word < 128 ? at_word >> 2 : at_word - 128))
                    s_word[warp][i] = at_word >= 128 ? r1
                                      : at_word & 2u ? (at_word & 1u ? r0.w : r0.z) : (at_word & 1u ? r0.y : r0.x);
            }
            if (any) feasible |= 1u << i;
        }
        // lane i: pod i's flags.  Malformed lists, bad expressions and lists
        // without slots are left to the pass below.
        __syncwarp();
        if (lane < take) {
            const bool aok = a < N && ((s_word[warp][lane] >> (a & 31)) & 1u);
            g.flags[p] = (plain >> lane) & 1u ? pod_flags((feasible >> lane) & 1u, pre & 2u, g.assign != nullptr, aok)
                                              : kPodLeft;
        }
        left_over = left_over || plain != group;
        __syncwarp();   // the list is rebuilt for the next pods
    }
    if (!left_over) return;
    for (uint32_t at = begin; at < end; at += 32) {
        const uint32_t pl = at + lane < end ? (g.pod_list ? g.pod_list[at + lane] : at + lane) : 0u;
        const bool mine = at + lane < end && *(volatile uint8_t *)(g.flags + pl) == kPodLeft;
        for (uint32_t todo = __ballot_sync(PV_FULL_MASK, mine); todo; todo &= todo - 1u)
            unresolved_pod<kTerms, false>(g, __shfl_sync(PV_FULL_MASK, pl, __ffs(todo) - 1), s_list[threadIdx.x >> 5]);
    }
}

// ---------------------------------------------------------------------------
// identical selectors evaluated once (pods sharing an expression list, such
// as the replicas of one deployment, or intents with the same selector)
// ---------------------------------------------------------------------------
// A list's canonical form: per expression its key / operator / count word
// and its value words with the unused value slots zeroed (evaluation never
// reads them), so equal canonical lists give equal rows and flags.  Each
// pod's list is hashed (splitmix64's finalizer over the words, mixed with
// the expression's position) into an open-addressing table whose entries
// keep the smallest pod with that hash; every other pod with the hash is
// compared word by word with it, so a hash collision costs only an extra
// evaluation, never a wrong row.  Representatives are evaluated as usual;
// each duplicate then copies its representative's row and flags and redoes
// its own placement check.
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ void canon_expr(const pv_expr *x, uint32_t w[5]) {
    const uint32_t *raw = reinterpret_cast<const uint32_t *>(x);   // 20-byte records, 4-byte aligned
    w[0] = raw[0];
    const bool listed = (x->op == PV_IN || x->op == PV_NOTIN) && x->nvals <= 8;
    const uint32_t nv = listed ? x->nvals : 0u;
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i) {
        const uint32_t v = raw[1 + i];
        w[1 + i] = (2 * i < nv ? (v & 0xFFFFu) : 0u) | (2 * i + 1 < nv ? (v & 0xFFFF0000u) : 0u);
    }
}

__device__ __forceinline__ uint64_t warp_sum64(uint64_t v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(PV_FULL_MASK, v, o);
    return v;
}

// Warp per pod: hashes[p] (0 for a malformed range, which is never shared)
// and the pod's entry in the table (keys: hash, 0 = free; reps: smallest pod).
__global__ void __launch_bounds__(256) sel_hash_kernel(uint32_t P, const uint32_t *__restrict__ offs,
                                                       uint32_t num_exprs, const pv_expr *__restrict__ exprs,
                                                       unsigned long long *__restrict__ keys,
                                                       uint32_t *__restrict__ reps, uint32_t cap_mask,
                                                       uint32_t weak, unsigned long long *__restrict__ hashes) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t p = gw; p < P; p += nw) {
        const uint32_t lo = offs[p], hi = offs[p + 1];
        if (hi < lo || hi > num_exprs) {
            if (lane == 0) hashes[p] = 0;
            continue;
        }
        const uint32_t E = hi - lo;
        uint64_t acc = 0;
        for (uint32_t e = lane; e < E; e += 32) {
            uint32_t w[5];
            canon_expr(exprs + lo + e, w);
            uint64_t h = mix64(((uint64_t)e << 32) ^ w[0]);
#pragma unroll
            for (uint32_t i = 1; i < 5; ++i) h = mix64(h ^ ((uint64_t)i << 40) ^ w[i]);
            acc += h;
        }
        acc = warp_sum64(acc);
        uint64_t h = mix64(acc ^ ((uint64_t)E * 0x9E3779B97F4A7C15ull)) | 1ull;
        if (weak) h = (h & 7ull) + 1ull;   // test mode: eight hash values, so most lists collide
        if (lane == 0) {
            hashes[p] = h;
            // popular lists share a slot: read first, and take an atomic only
            // to claim a free slot or to lower the slot's pod
            uint32_t slot = (uint32_t)(h * 0x9E3779B97F4A7C15ull >> 32) & cap_mask;
            for (uint32_t probe = 0; probe <= cap_mask; ++probe) {   // the table has room for every pod
                unsigned long long k = *(volatile unsigned long long *)(keys + slot);
                if (k == 0ull) k = atomicCAS(keys + slot, 0ull, (unsigned long long)h);
                if (k == 0ull || k == h) {
                    if (*(volatile uint32_t *)(reps + slot) > p) atomicMin(reps + slot, p);
                    break;
                }
                slot = (slot + 1) & cap_mask;
            }
        }
    }
}

// Warp per pod: rep_of[p] = the table's pod for p's hash when its canonical
// list equals p's, else p.
__global__ void __launch_bounds__(256) sel_rep_kernel(uint32_t P, const uint32_t *__restrict__ offs,
                                                      const pv_expr *__restrict__ exprs,
                                                      const unsigned long long *__restrict__ keys,
                                                      const uint32_t *__restrict__ reps, uint32_t cap_mask,
                                                      const unsigned long long *__restrict__ hashes,
                                                      uint32_t *__restrict__ rep_of, uint32_t *__restrict__ rep_list,
                                                      uint32_t *__restrict__ rep_count) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t p = gw; p < P; p += nw) {
        const uint64_t h = hashes[p];
        uint32_t r = p;
        if (h != 0) {
            uint32_t slot = (uint32_t)(h * 0x9E3779B97F4A7C15ull >> 32) & cap_mask;
            for (uint32_t probe = 0; probe <= cap_mask && keys[slot] != h; ++probe) slot = (slot + 1) & cap_mask;
            r = keys[slot] == h ? reps[slot] : p;
        }
        if (r != p) {
            const uint32_t lo = offs[p], E = offs[p + 1] - lo, lr = offs[r], Er = offs[r + 1] - lr;
            bool same = E == Er;
            for (uint32_t e = lane; same && e < E; e += 32) {
                uint32_t a[5], b[5];
                canon_expr(exprs + lo + e, a);
                canon_expr(exprs + lr + e, b);
#pragma unroll
                for (int i = 0; i < 5; ++i) same = same && a[i] == b[i];
            }
            if (!__all_sync(PV_FULL_MASK, same)) r = p;
        }
        if (lane == 0) {
            rep_of[p] = r;
            if (r == p) rep_list[atomicAdd(rep_count, 1u)] = p;
        }
    }
}

// Warp per duplicate pod: its representative's row, flags without the
// placement bits, and its own placement check.
__global__ void __launch_bounds__(256) sel_copy_kernel(uint32_t P, uint32_t N, uint32_t W,
                                                       const uint32_t *__restrict__ rep_of,
                                                       const uint32_t *__restrict__ assign, uint32_t *__restrict__ bits,
                                                       uint8_t *__restrict__ flags) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t p = gw; p < P; p += nw) {
        const uint32_t r = rep_of[p];
        if (r == p) continue;
        const uint4 *src = reinterpret_cast<const uint4 *>(bits + (size_t)r * W);
        uint4 *dst = reinterpret_cast<uint4 *>(bits + (size_t)p * W);
        for (uint32_t q = lane; q < W / 4; q += 32) dst[q] = src[q];
        if (lane == 0) {
            uint8_t f = flags[r] & (uint8_t)(PV_F_EMPTY | PV_F_UNKNOWN_VALUE | PV_F_BAD_EXPR);
            const uint32_t a = assign ? assign[p] : PV_UNPLACED;
            if (a < N && ((bits[(size_t)r * W + (a >> 5)] >> (a & 31)) & 1u)) {
                f |= PV_F_ASSIGN_OK;
                if (!(f & PV_F_UNKNOWN_VALUE)) f |= PV_F_PASS;
            }
            flags[p] = f;
        }
    }
}

}  // namespace

// -----------------------------------------------------------------------------
// C ABI
// -----------------------------------------------------------------------------
extern "C" int pv_load_cluster(pv_ctx *ctx, uint32_t num_nodes, uint32_t num_keys, const uint16_t *labels) {
    if (!ctx) return PV_EINVAL;
    if (num_nodes == 0 || num_keys == 0 || !labels)
        return pv_fail(ctx, PV_EINVAL, "pv_load_cluster: empty cluster or NULL labels");
    if (num_keys > kMaxKeys) return pv_fail(ctx, PV_EINVAL, "pv_load_cluster: num_keys > %u", kMaxKeys);
    if (int rc0 = pv_load_begin(ctx)) return rc0;
    cudaStream_t ls = ctx->load_stream;
    pv_cluster_state c;   // the new state (the loaded one stays in use until it is complete)
    const size_t nl = (size_t)num_nodes * num_keys;
    int rc;
    if ((rc = pv_pool_alloc(ctx, (void **)&c.d_labels, nl * 2, "labels")) ||
        (rc = pv_pool_alloc(ctx, (void **)&c.d_inv, (size_t)num_keys * kInvWords * 4, "inventory")) ||
        (rc = pv_pool_alloc(ctx, (void **)&c.d_ranked, (size_t)num_keys * kInvWords * 8, "inventory rank")) ||
        (rc = pv_pool_alloc(ctx, (void **)&c.d_key_base, ((size_t)num_keys + 1) * 4 * 2, "key base"))) {
        pv_free_cluster(ctx, c);
        return rc;
    }
    uint32_t *d_count = c.d_key_base + (num_keys + 1);
    PV_TRY_CUDA(ctx, cudaMemcpyAsync(c.d_labels, labels, nl * 2, cudaMemcpyHostToDevice, ls), "labels upload");
    PV_TRY_CUDA(ctx, cudaMemsetAsync(c.d_inv, 0, (size_t)num_keys * kInvWords * 4, ls), "inventory clear");
    build_inventory_kernel<<<ctx->num_sms * 8, 256, 0, ls>>>(num_nodes, num_keys, c.d_labels, c.d_inv);
    inventory_rank_kernel<<<num_keys, 1024, 0, ls>>>(c.d_inv, c.d_ranked, d_count);
    key_base_kernel<<<1, 1024, 0, ls>>>(num_keys, d_count, c.d_key_base);
    if ((rc = pv_check_launch(ctx, "inventory kernels"))) { pv_free_cluster(ctx, c); return rc; }
    uint32_t nvr = 0;
    cudaError_t e = cudaMemcpyAsync(&nvr, c.d_key_base + num_keys, 4, cudaMemcpyDeviceToHost, ls);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ls);
    if (e != cudaSuccess) {
        pv_free_cluster(ctx, c);
        return pv_cuda_fail(ctx, e, "value count");
    }
    c.num_nodes = num_nodes;
    c.num_keys = num_keys;
    c.row_words = words_for(num_nodes);
    c.num_value_rows = nvr;
    const uint64_t row_bytes = ((uint64_t)nvr + num_keys + 1) * c.row_words * 4;   // and the row of no node
    if (row_bytes - c.row_words * 4ull <= kRowBudgetBytes) {
        if (pv_pool_alloc(ctx, (void **)&c.d_rows, row_bytes, "value rows") == PV_OK) {
            if ((e = cudaMemsetAsync(c.d_rows, 0, row_bytes, ls)) != cudaSuccess) {
                pv_free_cluster(ctx, c);
                return pv_cuda_fail(ctx, e, "value rows clear");
            }
            build_rows_kernel<<<ctx->num_sms * 8, 256, 0, ls>>>(num_nodes, num_keys, c.d_labels, c.d_ranked, c.d_key_base,
                                                          nvr, c.row_words, c.d_rows);
            if ((rc = pv_check_launch(ctx, "value rows"))) { pv_free_cluster(ctx, c); return rc; }
            c.rows_built = true;
        } else {
            ctx->err.clear();   // rows are optional; fall back to the comparison kernel
        }
    }
    c.loaded = true;
    pv_retire_begin(ctx);
    pv_free_cluster(ctx, ctx->cl);
    pv_retire_end(ctx);
    ctx->cl = c;
    return pv_load_end(ctx);
}

namespace {

// The loaded cluster's part of the kernels' arguments.
SelArgs cluster_args(const pv_ctx *ctx, SelArgs g) {
    const pv_cluster_state &c = ctx->cl;
    g.N = c.num_nodes;
    g.K = c.num_keys;
    g.inv = c.d_inv;
    g.ranked = c.d_ranked;
    g.key_base = c.d_key_base;
    g.rows = c.d_rows;
    g.row_words = c.row_words;
    g.num_value_rows = c.num_value_rows;
    g.zero_row = (c.num_value_rows + c.num_keys) * c.row_words * 4;
    return g;
}

// The rows kernel's grid: a warp per pod until the GPU is full, then the pods
// shared out.
template <bool kTerms>
void launch_rows(pv_ctx *ctx, const SelArgs &g, cudaStream_t st) {
    void (*fn)(SelArgs) = g.W <= 160 ? sel_rows_kernel<kTerms, true> : sel_rows_kernel<kTerms, false>;
    const int per_sm = std::max(1, pv_blocks_per_sm(ctx, (const void *)fn, kRowsThreads<kTerms>, 0));
    constexpr uint32_t warps = kRowsThreads<kTerms> / 32;
    const uint32_t blocks = std::min((g.P + warps - 1) / warps, (uint32_t)(ctx->num_sms * per_sm));
    fn<<<blocks, kRowsThreads<kTerms>, 0, st>>>(g);
}

// The term form: a pod to a warp where that many warps fit at once and the rows
// kernel's do not.
void launch_terms(pv_ctx *ctx, const SelArgs &g, cudaStream_t st) {
    constexpr uint32_t pods = kPodThreads / 32, warps = kRowsThreads<true> / 32;
    const uint32_t sms = (uint32_t)ctx->num_sms;
    const void *rows = g.W <= 160 ? (const void *)sel_rows_kernel<true, true> : (const void *)sel_rows_kernel<true, false>;
    if (g.P > sms * warps * (uint32_t)pv_blocks_per_sm(ctx, rows, kRowsThreads<true>, 0) &&
        g.P <= sms * pods * (uint32_t)pv_blocks_per_sm(ctx, (const void *)sel_terms_kernel, kPodThreads, 0))
        sel_terms_kernel<<<(g.P + pods - 1) / pods, kPodThreads, 0, st>>>(g);
    else
        launch_rows<true>(ctx, g, st);
}

}  // namespace

extern "C" int pv_eval_selectors(pv_ctx *ctx, uint32_t num_pods, const uint32_t *d_expr_offs, uint32_t num_exprs,
                                 const pv_expr *d_exprs, const uint32_t *d_assign, uint32_t *d_bits,
                                 uint32_t words_per_row, uint8_t *d_flags, pv_stream stream) {
    if (!ctx) return PV_EINVAL;
    const pv_cluster_state &c = ctx->cl;
    if (!c.loaded) return pv_fail(ctx, PV_ESTATE, "pv_eval_selectors: no cluster loaded");
    if (num_pods == 0) return PV_OK;
    if (!d_expr_offs || !d_bits || !d_flags || (num_exprs > 0 && !d_exprs))
        return pv_fail(ctx, PV_EINVAL, "pv_eval_selectors: NULL device pointer");
    if (words_per_row % 4 != 0 || words_per_row < (c.num_nodes + 31) / 32)
        return pv_fail(ctx, PV_EINVAL, "pv_eval_selectors: words_per_row must be >= ceil(N/32) and a multiple of 4");
    if (((uintptr_t)d_bits & 15) != 0) return pv_fail(ctx, PV_EINVAL, "pv_eval_selectors: d_bits must be 16-byte aligned");
    if (((uintptr_t)d_exprs & 3) != 0)   // expressions are read a 32-bit word at a time
        return pv_fail(ctx, PV_EINVAL, "pv_eval_selectors: d_exprs must be 4-byte aligned");
    int which = ctx->opt_selector;
    if (which == 0) which = c.rows_built ? 2 : 1;
    if (which == 2 && !c.rows_built)
        return pv_fail(ctx, PV_EINVAL, "pv_eval_selectors: value rows were not built for this cluster");
    cudaStream_t st = (cudaStream_t)stream;
    const uint32_t wblocks = std::min<uint32_t>((num_pods + 7) / 8, (uint32_t)ctx->num_sms * 16);   // warp per pod
    // comparison kernel: node tiles of as many nodes (multiple of 32) as fit 96 KB of label columns
    uint32_t tile = (uint32_t)((96 * 1024) / (2ull * c.num_keys)) / 32 * 32;
    if (which == 1 && tile < 32)
        return pv_fail(ctx, PV_EINVAL, "pv_eval_selectors: too many keys for the comparison kernel");
    tile = min(tile, ((c.num_nodes + 31) / 32) * 32);
    uint32_t *rep_of = nullptr, *rep_list = nullptr, *rep_count = nullptr;
    pv_use_begin(ctx, st);
    const int pr = pv_prof_start(ctx, st, PV_K_SELECTOR);
    if (ctx->opt_selector_dedupe && num_pods <= (1u << 30)) {
        uint32_t cap = 1;
        while ((uint64_t)cap < 2ull * num_pods) cap <<= 1;
        const size_t o_reps = (size_t)cap * 8, o_hash = o_reps + (((size_t)cap * 4 + 255) & ~(size_t)255);
        const size_t o_rep = o_hash + (size_t)num_pods * 8, o_list = o_rep + (((size_t)num_pods * 4 + 255) & ~(size_t)255);
        const size_t total = o_list + (size_t)num_pods * 4 + 256;
        uint8_t *base = (uint8_t *)pv_scratch(ctx, total);
        if (!base) {
            pv_prof_stop(ctx, st, pr, 0);
            return PV_ENOMEM;
        }
        auto *keys = reinterpret_cast<unsigned long long *>(base);
        auto *reps = reinterpret_cast<uint32_t *>(base + o_reps);
        auto *hashes = reinterpret_cast<unsigned long long *>(base + o_hash);
        rep_of = reinterpret_cast<uint32_t *>(base + o_rep);
        rep_list = reinterpret_cast<uint32_t *>(base + o_list);
        rep_count = rep_list + num_pods;
        PV_TRY_CUDA(ctx, cudaMemsetAsync(rep_count, 0, 4, st), "selector list clear");
        PV_TRY_CUDA(ctx, cudaMemsetAsync(keys, 0, (size_t)cap * 8, st), "selector table clear");
        PV_TRY_CUDA(ctx, cudaMemsetAsync(reps, 0xFF, (size_t)cap * 4, st), "selector table clear");
        sel_hash_kernel<<<wblocks, 256, 0, st>>>(num_pods, d_expr_offs, num_exprs, d_exprs, keys, reps, cap - 1,
                                                  ctx->opt_selector_dedupe == 2 ? 1u : 0u, hashes);
        sel_rep_kernel<<<wblocks, 256, 0, st>>>(num_pods, d_expr_offs, d_exprs, keys, reps, cap - 1, hashes, rep_of,
                                                 rep_list, rep_count);
    }
    if (which == 2) {
        SelArgs g = {};
        g.P = num_pods;
        g.offs = d_expr_offs;
        g.num_exprs = num_exprs;
        g.exprs = d_exprs;
        g.assign = d_assign;
        g.bits = d_bits;
        g.W = words_per_row;
        g.flags = d_flags;
        g.pod_list = rep_list;
        g.list_len = rep_count;
        launch_rows<false>(ctx, cluster_args(ctx, g), st);
    } else {
        const size_t smem = (size_t)tile * c.num_keys * 2;
        PV_TRY_CUDA(ctx, cudaFuncSetAttribute(sel_cmp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                    "sel_cmp_kernel smem");
        const uint32_t blocks = (num_pods + kCmpPods - 1) / kCmpPods;
        sel_cmp_kernel<<<blocks, kCmpThreads, smem, st>>>(c.num_nodes, c.num_keys, c.d_labels, tile, num_pods,
                                                          d_expr_offs, num_exprs, d_exprs, d_assign, d_bits,
                                                          words_per_row, d_flags, c.d_inv, rep_of);
    }
    if (rep_of)
        sel_copy_kernel<<<wblocks, 256, 0, st>>>(num_pods, c.num_nodes, words_per_row, rep_of, d_assign, d_bits,
                                                 d_flags);
    pv_prof_stop(ctx, st, pr, rep_of ? 4 : 1);
    pv_mark_use(ctx, st);
    return pv_check_launch(ctx, "selector kernels");
}

extern "C" int pv_eval_selector_terms(pv_ctx *ctx, uint32_t num_pods, const uint32_t *d_pod_terms, uint32_t num_terms,
                                      const uint32_t *d_term_offs, uint32_t num_exprs, const pv_expr *d_exprs,
                                      const uint32_t *d_assign, uint32_t *d_bits, uint32_t words_per_row,
                                      uint8_t *d_flags, pv_stream stream) {
    if (!ctx) return PV_EINVAL;
    const pv_cluster_state &c = ctx->cl;
    if (!c.loaded) return pv_fail(ctx, PV_ESTATE, "pv_eval_selector_terms: no cluster loaded");
    if (num_pods == 0) return PV_OK;
    if (!d_pod_terms || !d_bits || !d_flags || (num_terms > 0 && !d_term_offs) || (num_exprs > 0 && !d_exprs))
        return pv_fail(ctx, PV_EINVAL, "pv_eval_selector_terms: NULL device pointer");
    if (words_per_row % 4 != 0 || words_per_row < (c.num_nodes + 31) / 32)
        return pv_fail(ctx, PV_EINVAL,
                       "pv_eval_selector_terms: words_per_row must be >= ceil(N/32) and a multiple of 4");
    if (((uintptr_t)d_bits & 15) != 0)
        return pv_fail(ctx, PV_EINVAL, "pv_eval_selector_terms: d_bits must be 16-byte aligned");
    if (!c.rows_built)
        return pv_fail(ctx, PV_EINVAL, "pv_eval_selector_terms: value rows were not built for this cluster");
    cudaStream_t st = (cudaStream_t)stream;
    SelArgs g = {};
    g.P = num_pods;
    g.offs = d_pod_terms;
    g.num_terms = num_terms;
    g.term_offs = d_term_offs;
    g.num_exprs = num_exprs;
    g.exprs = d_exprs;
    g.assign = d_assign;
    g.bits = d_bits;
    g.W = words_per_row;
    g.flags = d_flags;
    pv_use_begin(ctx, st);
    const int pr = pv_prof_start(ctx, st, PV_K_SELECTOR);
    launch_terms(ctx, cluster_args(ctx, g), st);
    pv_prof_stop(ctx, st, pr, 1);
    pv_mark_use(ctx, st);
    return pv_check_launch(ctx, "selector kernels");
}
