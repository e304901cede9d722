// Jurisdiction-masked reachability (Sec. 3.3 forbidden-vertex policy over
// G = (V, E); Sec. 4.2 graph search over the current topology).
//
// R(s, m) is the least set that contains s when region(s) is permitted by m
// and is closed under edges u -> v into permitted v.  One block computes it
// for one mask and a batch of 64 sources at once: vertex v holds a 64-bit
// word whose bit j says "v is in R(src_j, m)" (multi-source, bit-parallel
// frontier propagation).  Sweeps pull over in-edges,
//     vis[v] |= OR_{u -> v} vis[u]      for permitted v,
// in place, until a sweep changes nothing; in-place updates only speed up
// convergence and the fixpoint is exactly the closure, so the result equals
// a breadth-first search per source.  At most V + 1 sweeps run (each sweep
// extends every search by at least one level).  The vertex-major words are
// transposed with __ballot_sync into the caller's source-major bitset rows,
// written with 128-bit stores.
//
// Symmetric graphs (every edge u -> v has its reverse v -> u) take an exact
// shortcut: there a path s -> v inside the permitted vertices exists iff s
// and v lie in the same connected component of the subgraph induced by the
// permitted vertices, so R(s, m) is that component (or empty when s itself
// is not permitted).  One block labels the components of one mask with a
// lock-free union-find in shared memory and writes the bitset of each to a
// table; a source's row is then a copy of its component's.  A device-side check decides per call which of
// the two paths runs; both are launched and the other one returns at once.
//
// Other graphs seldom need a search per source either: most permitted
// vertices lie in one strongly connected component.  Per mask, a hub vertex h
// is taken and its forward set F and backward set B are searched once; a
// source in F and B has R(s, m) = F, and only the others are searched (those
// in B from F on: F is part of their sets).
//
// A row of a source that is not permitted is empty on either path, so those
// rows are cleared by blocks of their own in the check's and the labels'
// launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "pv_internal.cuh"

namespace {

constexpr uint32_t kReachMaxV = 16384;
constexpr int kReachThreads = 512;
constexpr int kGridThreads = 256;

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// A CSR whose offsets are malformed (some row with offs[u + 1] < offs[u] or
// offs[u + 1] > E) counts as having no edges at all: its well-formed rows
// could overlap, so their lengths could add up past E, the size of every
// edge-indexed scratch array.  A per-call flag says so (kBadOffs of the
// context's flags; the no-allocation call's is indeg[V]); every later kernel
// of the call reads it before it touches an edge.
enum { kAsym = 0, kBadOffs = 1, kPairs = 2, kReachFlags = 3 };   // words of pv_ctx::d_reach_flags

// The call's rows come from components: the graph is symmetric (no edges at
// all included).
__device__ __forceinline__ bool component_path(const uint32_t *flags) {
    const volatile uint32_t *f = flags;
    return f[kAsym] == 0 || f[kBadOffs] != 0;
}

__device__ __forceinline__ bool csr_offsets_bad(const uint32_t *bad) {
    return *(volatile const uint32_t *)bad != 0;
}

// In-degree count with validation of the caller's CSR, eight lanes to a
// vertex (a vertex's loads then overlap).  An out-of-range column skips that
// edge; malformed offsets set the flag at indeg[V] (the counts of this pass
// are then unused).
constexpr uint32_t kEdgeLanes = 8;
__global__ void reach_indeg_kernel(uint32_t V, uint32_t E, const uint32_t *__restrict__ offs,
                                   const uint32_t *__restrict__ cols, const uint8_t *__restrict__ region,
                                   uint32_t *__restrict__ indeg, int32_t *status) {
    const uint32_t sub = threadIdx.x % kEdgeLanes, groups = gridDim.x * blockDim.x / kEdgeLanes;
    for (uint32_t u = (blockIdx.x * blockDim.x + threadIdx.x) / kEdgeLanes; u < V; u += groups) {
        if (sub == 0 && region[u] >= 32) pv_device_error(status, PV_EINVAL);
        const uint32_t a = offs[u], b = offs[u + 1];
        if (b < a || b > E) {
            pv_device_error(status, PV_EINVAL);
            atomicOr(&indeg[V], 1u);
            continue;
        }
        for (uint32_t e = a + sub; e < b; e += kEdgeLanes) {
            const uint32_t v = cols[e];
            if (v >= V) {
                pv_device_error(status, PV_EINVAL);
                continue;
            }
            atomicAdd(&indeg[v], 1u);
        }
    }
}

// indeg and the call's flags cleared in one launch.
__global__ void reach_clear_kernel(uint32_t V, uint32_t *__restrict__ indeg, uint32_t *__restrict__ flags) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < V) indeg[i] = 0;
    if (i < kReachFlags) flags[i] = 0;
}

// Single block: in_offs = exclusive scan of indeg (V+1 entries); cursor copy.
// With malformed offsets every in-edge list is empty.
__global__ void __launch_bounds__(1024) reach_scan_kernel(uint32_t V, const uint32_t *__restrict__ indeg,
                                                          uint32_t *__restrict__ in_offs,
                                                          uint32_t *__restrict__ cursor, const uint32_t *flags,
                                                          const uint32_t *bad_offs) {
    if (flags && component_path(flags)) return;   // in-edges unused
    __shared__ uint32_t s_warp[32];
    __shared__ uint32_t s_carry;
    const bool bad = csr_offsets_bad(bad_offs);
    const uint32_t t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) s_carry = 0;
    __syncthreads();
    for (uint32_t c0 = 0; c0 < V; c0 += 1024) {
        const uint32_t i = c0 + t;
        const uint32_t x = i < V && !bad ? indeg[i] : 0;
        uint32_t incl = x;
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
        const uint32_t excl = s_carry + s_warp[warp] + incl - x;
        if (i < V) {
            in_offs[i] = excl;
            cursor[i] = excl;
        }
        __syncthreads();
        if (t == 1023) s_carry = excl + x;
        __syncthreads();
    }
    if (t == 0) in_offs[V] = s_carry;
}

__global__ void reach_fill_kernel(uint32_t V, uint32_t E, const uint32_t *__restrict__ offs,
                                  const uint32_t *__restrict__ cols, uint32_t *__restrict__ cursor,
                                  uint32_t *__restrict__ in_cols, const uint32_t *flags, const uint32_t *bad) {
    if (flags && component_path(flags)) return;   // in-edges unused
    if (csr_offsets_bad(bad)) return;             // no edges
    const uint32_t sub = threadIdx.x % kEdgeLanes, groups = gridDim.x * blockDim.x / kEdgeLanes;
    for (uint32_t u = (blockIdx.x * blockDim.x + threadIdx.x) / kEdgeLanes; u < V; u += groups) {
        const uint32_t a = offs[u], b = offs[u + 1];
        if (b < a || b > E) continue;
        for (uint32_t e = a + sub; e < b; e += kEdgeLanes) {
            const uint32_t v = cols[e];
            if (v < V) in_cols[atomicAdd(&cursor[v], 1u)] = u;
        }
    }
}

__device__ __forceinline__ bool source_permitted(uint32_t s, uint32_t V, const uint8_t *__restrict__ region,
                                                 uint32_t mask) {
    const uint32_t r = s < V ? region[s] : 32u;
    return r < 32 && ((mask >> r) & 1u);
}

// Rows of the sources that are not permitted or out of range (empty on either
// path), a warp to 32 (mask, source) rows at a time.  Two thirds of a WAN's
// rows are, and checking and labelling the graph leave most SMs and the memory
// idle, so blocks of their own in those two launches write them.  [lo, hi):
// this launch's share of the rows.
struct ClearArgs {
    const uint32_t *masks, *src;
    uint32_t num_src, W;
    uint32_t *reach;
    uint64_t lo, hi;
};
__device__ __forceinline__ void clear_rows(const ClearArgs &c, uint32_t block, uint32_t blocks, uint32_t V,
                                           const uint8_t *__restrict__ region) {
    const uint32_t lane = threadIdx.x & 31, warps = blockDim.x / 32;
    for (uint64_t i0 = c.lo + ((uint64_t)block * warps + threadIdx.x / 32) * 32; i0 < c.hi;
         i0 += (uint64_t)blocks * warps * 32) {
        const uint64_t i = i0 + lane;
        const uint32_t m = (uint32_t)(i / c.num_src);
        const bool clear = i < c.hi && !source_permitted(c.src[i - (uint64_t)m * c.num_src], V, region, c.masks[m]);
        for (uint32_t todo = __ballot_sync(PV_FULL_MASK, clear); todo; todo &= todo - 1u) {
            uint4 *out = reinterpret_cast<uint4 *>(c.reach + (i0 + (uint32_t)(__ffs(todo) - 1)) * c.W);
            for (uint32_t q = lane; q < c.W / 4; q += 32) out[q] = make_uint4(0, 0, 0, 0);
        }
    }
}

// Validation, in-degrees and symmetry of the caller's out-edge CSR in one
// pass, one warp per vertex.  kAsym is set unless every edge u -> v (v < V)
// has its reverse v -> u; vertices whose list is longer than kSymScanMax make
// the graph count as asymmetric (the search path then runs; still exact).
// Each undirected edge is listed once, as pairs[] = u << 16 | v with v < u, in
// no particular order.  With malformed offsets the counts and pairs of this
// pass are unused (rows that overlap could list more than E pairs: those past
// the array are dropped).
constexpr uint32_t kSymScanMax = 64;

__global__ void reach_check_kernel(uint32_t V, uint32_t E, const uint32_t *__restrict__ offs,
                                   const uint32_t *__restrict__ cols, const uint8_t *__restrict__ region,
                                   uint32_t *__restrict__ indeg, uint32_t *flags, uint32_t *__restrict__ pairs,
                                   int32_t *status, uint32_t check_blocks, ClearArgs clear) {
    if (blockIdx.x >= check_blocks) {
        clear_rows(clear, blockIdx.x - check_blocks, gridDim.x - check_blocks, V, region);
        return;
    }
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t nwarps = check_blocks * (blockDim.x / 32);
    for (uint32_t u = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; u < V; u += nwarps) {
        const uint32_t a = offs[u], b = offs[u + 1];
        if (lane == 0 && region[u] >= 32) pv_device_error(status, PV_EINVAL);
        if (b < a || b > E) {
            if (lane == 0) {
                pv_device_error(status, PV_EINVAL);
                atomicOr(flags + kBadOffs, 1u);
            }
            continue;
        }
        // once the graph is known to be asymmetric only the counts matter
        // (warp-uniform: lane 0's read decides)
        bool sym = __shfl_sync(PV_FULL_MASK, *(volatile uint32_t *)(flags + kAsym), 0) == 0;
        if (sym && b - a > kSymScanMax) {
            if (lane == 0) atomicOr(flags + kAsym, 1u);
            sym = false;
        }
        for (uint32_t e0 = a; e0 < b; e0 += 32) {
            const uint32_t e = e0 + lane;
            uint32_t v = V;
            if (e < b) {
                v = cols[e];
                if (v < V) atomicAdd(&indeg[v], 1u);
                else pv_device_error(status, PV_EINVAL);
            }
            if (!sym) continue;
            bool ok = true;
            if (v < V && v != u) {
                const uint32_t c = offs[v], d = offs[v + 1];
                bool found = false;
                if (!(d < c || d > E) && d - c <= kSymScanMax)
                    for (uint32_t f = c; f < d && !found; f += 4) {   // four columns in flight
                        uint32_t x[4];
#pragma unroll
                        for (uint32_t j = 0; j < 4; ++j) x[j] = f + j < d ? cols[f + j] : V;
                        found = x[0] == u || x[1] == u || x[2] == u || x[3] == u;
                    }
                ok = found;
            }
            if (__any_sync(PV_FULL_MASK, !ok)) {
                if (lane == 0) atomicOr(flags + kAsym, 1u);
                sym = false;
                continue;
            }
            const bool keep = v < u;   // v < V too
            const uint32_t bal = __ballot_sync(PV_FULL_MASK, keep);
            uint32_t base = 0;
            if (lane == 0 && bal) base = atomicAdd(flags + kPairs, (uint32_t)__popc(bal));
            base = __shfl_sync(PV_FULL_MASK, base, 0) + __popc(bal & ((1u << lane) - 1u));
            if (keep && base < E) pairs[base] = (u << 16) | v;
        }
    }
}

// Union-find over shared memory with parent[x] <= x at all times: roots are
// hooked under smaller roots by compare-and-swap, finds halve paths (a
// racing write only ever stores an ancestor).  A failed hook means the root
// gained a parent, so the next attempt starts from a smaller root: at most
// 2V attempts.
__device__ __forceinline__ uint32_t uf_find(volatile uint32_t *parent, uint32_t x) {
    for (;;) {
        const uint32_t p = parent[x];
        if (p == x) return x;
        const uint32_t gp = parent[p];
        if (gp != p) parent[x] = gp;
        x = gp;
    }
}

__device__ __forceinline__ void uf_union(volatile uint32_t *parent, uint32_t a, uint32_t b, uint32_t limit,
                                         int32_t *status) {
    for (uint32_t it = 0; it < limit; ++it) {
        a = uf_find(parent, a);
        b = uf_find(parent, b);
        if (a == b) return;
        if (a < b) {
            const uint32_t x = a;
            a = b;
            b = x;
        }
        if (atomicCAS(const_cast<uint32_t *>(parent + a), a, b) == a) return;
    }
    // not reachable by the argument above; should it happen all the same,
    // the row would be wrong, so the call reports it rather than pass
    pv_device_error(status, PV_ETIMEOUT);
}

// Component table at most.  Rows past it come from the labels by ballots: 4,096
// sources on 16,384 vertices, 64 masks and some 2,700 components a mask 364 us
// with 64 MB, 247 with 128.
constexpr size_t kTableBytes = (size_t)128 << 20;

constexpr uint16_t kNoLabel = 0xFFFF;
constexpr uint16_t kSlotNone = 0xFFFF, kSlotOverflow = 0xFFFE, kSlotSingle = 0xFFFD;   // table rows stay below these

__host__ __device__ inline uint32_t up16u(uint32_t x) { return (x + 15u) & ~15u; }

// Component labels of one mask per block: lab[m][v] = the smallest vertex
// of v's component in the permitted subgraph, kNoLabel for a vertex whose
// region the mask does not permit.  One pass over the pair list (from L2)
// points every permitted vertex at its smallest permitted neighbour below
// it (a valid forest of the same components, so most unions then find one
// root) and copies the pairs inside the permitted subgraph, usually a small
// share of them, to shared memory; the union pass then runs over that
// compact list (over the whole list again when it did not fit).  Each
// component of several vertices then takes a row of the mask's table, if one is
// left: slots[m][v] = v's row, kSlotOverflow past the table, kSlotSingle for a
// vertex alone in its component, kSlotNone for one that is not permitted.  With few masks several blocks (parts) label the
// same mask and each writes a share of its table (4,096 sources on 16,000 vertices
// of average degree 0.6, one mask: the call takes 101 us with four, 89 with eight,
// 156 with one).
constexpr int kLabelThreads = 1024;
constexpr uint32_t kLabelParts = 8;               // most blocks that label one mask
constexpr size_t kLabelSmemTarget = 100 * 1024;   // two label blocks per SM

// Layout of the labels kernel's dynamic shared memory for V vertices:
// parent[V], the permitted-vertex bitmap, then the compact pair list.
struct LabelSmem {
    uint32_t allow, pairs, cap;
    size_t total;
    __host__ __device__ explicit LabelSmem(uint32_t V) {
        allow = up16u(V * 4);
        pairs = allow + up16u(((V + 31) / 32) * 4);
        const size_t left = kLabelSmemTarget > pairs ? kLabelSmemTarget - pairs : 0;
        cap = (uint32_t)(left / 4) & ~3u;
        total = (size_t)pairs + (size_t)cap * 4;
    }
};

__global__ void __launch_bounds__(kLabelThreads) reach_labels_kernel(
    uint32_t V, const uint32_t *__restrict__ pairs, const uint8_t *__restrict__ region,
    const uint32_t *__restrict__ masks, uint16_t *__restrict__ lab, uint16_t *__restrict__ slots,
    uint32_t *__restrict__ table, uint32_t cap, uint32_t W, const uint32_t *flags, int32_t *status,
    uint32_t label_blocks, uint32_t parts, ClearArgs clear) {
    if (blockIdx.x >= label_blocks) {
        clear_rows(clear, blockIdx.x - label_blocks, gridDim.x - label_blocks, V, region);
        return;
    }
    if (!component_path(flags)) return;       // the search path runs
    extern __shared__ __align__(16) uint8_t s_dyn[];
    __shared__ uint32_t s_np, s_comps;                                             // compact pairs, components
    const LabelSmem L(V);
    volatile uint32_t *parent = reinterpret_cast<uint32_t *>(s_dyn);              // [V]
    uint32_t *s_allow = reinterpret_cast<uint32_t *>(s_dyn + L.allow);            // [ceil(V / 32)]
    uint32_t *s_pairs = reinterpret_cast<uint32_t *>(s_dyn + L.pairs);            // [L.cap]
    const uint32_t t = threadIdx.x, lane = t & 31, warp = t >> 5, nt = blockDim.x;
    const uint32_t m = blockIdx.x / parts, part = blockIdx.x - m * parts, mask = masks[m];
    auto allowed = [&](uint32_t v) { return (s_allow[v >> 5] >> (v & 31)) & 1u; };
    // every vertex its own root; permitted-vertex bitmap
    for (uint32_t v0 = 0; v0 < V; v0 += nt) {
        const uint32_t v = v0 + t;
        bool ok = false;
        if (v < V) {
            const uint32_t r = region[v];
            ok = r < 32 && ((mask >> r) & 1u);
            parent[v] = v;
        }
        const uint32_t bal = __ballot_sync(PV_FULL_MASK, ok);
        if (lane == 0 && v0 + warp * 32 < V) s_allow[(v0 >> 5) + warp] = bal;
    }
    if (t == 0) s_np = s_comps = 0;
    __syncthreads();
    // each permitted vertex under its smallest permitted neighbour; the
    // pairs inside the permitted subgraph copied to the compact list
    const uint32_t np = csr_offsets_bad(flags + kBadOffs) ? 0u : flags[kPairs];
    for (uint32_t i0 = 0; i0 < np; i0 += 4 * nt) {
        const uint32_t i = i0 + 4 * t;
        uint32_t pq[4] = {0, 0, 0, 0};
        if (i < np) {
            const uint4 q = *reinterpret_cast<const uint4 *>(pairs + i);
            pq[0] = q.x;
            pq[1] = q.y;
            pq[2] = q.z;
            pq[3] = q.w;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t u = pq[k] >> 16, v = pq[k] & 0xFFFFu;   // v < u
            const bool in = i + k < np && allowed(u) && allowed(v);
            if (in) atomicMin(const_cast<uint32_t *>(parent + u), v);
            const uint32_t bal = __ballot_sync(PV_FULL_MASK, in);
            uint32_t base = 0;
            if (lane == 0 && bal) base = atomicAdd(&s_np, (uint32_t)__popc(bal));
            base = __shfl_sync(PV_FULL_MASK, base, 0) + __popc(bal & ((1u << lane) - 1u));
            if (in && base < L.cap) s_pairs[base] = pq[k];
        }
    }
    __syncthreads();
    // union the endpoints of every undirected edge inside the permitted
    // vertices (each pair once): from the compact list, or from the whole
    // list again when the compact one overflowed
    const uint32_t nc = s_np;
    if (nc <= L.cap) {
        for (uint32_t i = t; i < nc; i += nt) {
            const uint32_t p = s_pairs[i];
            uf_union(parent, p >> 16, p & 0xFFFFu, 2 * V + 2, status);
        }
    } else {
        for (uint32_t i = 4 * t; i < np; i += 4 * nt) {
            const uint4 q = *reinterpret_cast<const uint4 *>(pairs + i);
            const uint32_t pq[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t u = pq[k] >> 16, v = pq[k] & 0xFFFFu;
                if (i + k < np && allowed(u) && allowed(v)) uf_union(parent, u, v, 2 * V + 2, status);
            }
        }
    }
    __syncthreads();
    uint16_t *s_slot = reinterpret_cast<uint16_t *>(s_pairs);   // [V]: the pairs are done with
    uint32_t *s_rank = s_pairs + (V + 1) / 2;                   // [ceil(V / 32)]: roots with company before the word
    const uint32_t words = (V + 31) / 32;
    for (uint32_t v = t; v < V; v += nt) s_slot[v] = 0;
    __syncthreads();
    for (uint32_t v = t; v < V; v += nt) {
        const uint32_t r = uf_find(parent, v);
        if (part == 0) lab[(size_t)m * V + v] = allowed(v) ? (uint16_t)r : kNoLabel;
        if (r != v) s_slot[r] = 1;   // r has company
    }
    __syncthreads();
    if (parts == 1) {
        for (uint32_t v = t; v < V; v += nt)
            if (parent[v] == v && allowed(v)) {
                const uint32_t k = s_slot[v] ? atomicAdd(&s_comps, 1u) : 0u;
                s_slot[v] = !s_slot[v] ? kSlotSingle : k < cap ? (uint16_t)k : kSlotOverflow;
            }
    } else {   // rows in the order of the labels, the same in every part
        for (uint32_t v0 = warp * 32; v0 < V; v0 += nt) {
            const uint32_t bal = __ballot_sync(PV_FULL_MASK, v0 + lane < V && s_slot[v0 + lane] != 0);
            if (lane == 0) s_rank[v0 >> 5] = __popc(bal);
        }
        __syncthreads();
        if (warp == 0) {
            uint32_t run = 0;
            for (uint32_t w0 = 0; w0 < words; w0 += 32) {
                const uint32_t c = w0 + lane < words ? s_rank[w0 + lane] : 0u;
                uint32_t incl = c;
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(PV_FULL_MASK, incl, d);
                    if (lane >= (uint32_t)d) incl += y;
                }
                if (w0 + lane < words) s_rank[w0 + lane] = run + incl - c;
                run += __shfl_sync(PV_FULL_MASK, incl, 31);
            }
            if (lane == 0) s_comps = run;
        }
        __syncthreads();
        for (uint32_t v0 = warp * 32; v0 < V; v0 += nt) {
            const uint32_t v = v0 + lane;
            const bool has = v < V && s_slot[v] != 0;
            const uint32_t k = s_rank[v0 >> 5] + __popc(__ballot_sync(PV_FULL_MASK, has) & ((1u << lane) - 1u));
            if (v < V) s_slot[v] = !has ? kSlotSingle : k < cap ? (uint16_t)k : kSlotOverflow;   // (used for roots)
        }
    }
    __syncthreads();
    // the part's rows of the table: cleared, then every word written once, by
    // the first of the component's vertices among its 32
    const uint32_t rows = min(s_comps, cap), k0 = rows * part / parts, k1 = rows * (part + 1) / parts;
    uint32_t *tab = table + (size_t)m * cap * W;
    for (uint32_t q = t; q < (k1 - k0) * (W / 4); q += nt)
        reinterpret_cast<uint4 *>(tab + (size_t)k0 * W)[q] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    for (uint32_t v0 = warp * 32; v0 < V; v0 += nt) {
        const uint32_t v = v0 + lane;
        const uint32_t k = v < V && allowed(v) ? s_slot[uf_find(parent, v)] : kSlotNone;
        if (v < V && part == 0) slots[(size_t)m * V + v] = (uint16_t)k;
        const uint32_t peers = __match_any_sync(PV_FULL_MASK, k);
        if (k - k0 < k1 - k0 && lane == (uint32_t)(__ffs(peers) - 1)) tab[(size_t)k * W + (v0 >> 5)] = peers;
    }
}

// The bitset row of component c (all v < V with lab[v] == c; words past V
// are zero), written by one warp: for components past the table.
__device__ __forceinline__ void comp_row(const uint16_t *lab, uint32_t V, uint32_t W, uint32_t c, uint4 *dst,
                                         uint32_t lane) {
    const uint32_t groups = W / 4;
    for (uint32_t g0 = 0; g0 < groups; g0 += 32) {
        uint4 mine = make_uint4(0, 0, 0, 0);
        const uint32_t n = min(32u, groups - g0);
        for (uint32_t i = 0; i < n; ++i) {
            const uint32_t base = (g0 + i) * 128 + lane;
            uint32_t bits[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t v = base + 32 * k;
                bits[k] = __ballot_sync(PV_FULL_MASK, v < V && __ldg(lab + v) == c);
            }
            if (lane == i) mine = make_uint4(bits[0], bits[1], bits[2], bits[3]);
        }
        if (lane < n) dst[g0 + lane] = mine;
    }
}

// R(s, m) = the row of s's component (clear_rows writes the rows
// of the other sources): a warp takes per_warp (mask, source) rows, finds their
// table rows at once and copies them one after the other from L2.
// Bound by the row writes.  A block per mask and slice of sources used to
// rebuild the labels and the rows of its components, up to 90 of them, in
// shared memory (a 4,096-vertex WAN has some 150 a mask, so that many rows
// came from ballots): 22-32 us of the call's 70.
constexpr int kRowThreads = 256;
__global__ void __launch_bounds__(kRowThreads) reach_rows_kernel(
    uint32_t V, const uint16_t *__restrict__ lab, const uint16_t *__restrict__ slots,
    const uint32_t *__restrict__ table, uint32_t cap, uint32_t num_masks, uint32_t num_src,
    const uint32_t *__restrict__ src, uint32_t *__restrict__ reach, uint32_t W, uint32_t per_warp,
    const uint32_t *flags) {
    if (!component_path(flags)) return;
    const uint32_t lane = threadIdx.x & 31, warps = kRowThreads / 32;
    const uint64_t rows = (uint64_t)num_masks * num_src, step = (uint64_t)gridDim.x * warps * per_warp;
    for (uint64_t i0 = ((uint64_t)blockIdx.x * warps + threadIdx.x / 32) * per_warp; i0 < rows; i0 += step) {
        const uint64_t i = i0 + lane;
        const uint32_t m = (uint32_t)(i / num_src);
        const uint32_t s = lane < per_warp && i < rows ? src[i - (uint64_t)m * num_src] : V;
        const uint32_t slot = s < V ? __ldg(slots + (size_t)m * V + s) : kSlotNone;
        // four rows in flight
        for (uint32_t todo = __ballot_sync(PV_FULL_MASK, slot < kSlotSingle); todo;) {
            const uint4 *row[4];
            uint4 *out[4];
#pragma unroll
            for (uint32_t r = 0; r < 4; ++r) {
                out[r] = nullptr;
                row[r] = nullptr;
                if (todo) {   // warp-uniform
                    const uint32_t j = (uint32_t)(__ffs(todo) - 1);
                    todo &= todo - 1u;
                    out[r] = reinterpret_cast<uint4 *>(reach + (i0 + j) * W);
                    row[r] = reinterpret_cast<const uint4 *>(
                        table + ((size_t)__shfl_sync(PV_FULL_MASK, m, j) * cap + __shfl_sync(PV_FULL_MASK, slot, j)) * W);
                }
            }
            for (uint32_t q = lane; q < W / 4; q += 32) {
                uint4 x[4];
#pragma unroll
                for (uint32_t r = 0; r < 4; ++r) x[r] = row[r] ? __ldg(row[r] + q) : make_uint4(0, 0, 0, 0);
#pragma unroll
                for (uint32_t r = 0; r < 4; ++r)
                    if (out[r]) out[r][q] = x[r];
            }
        }
        for (uint32_t todo = __ballot_sync(PV_FULL_MASK, slot == kSlotSingle); todo; todo &= todo - 1u) {
            const uint32_t j = (uint32_t)(__ffs(todo) - 1), v = __shfl_sync(PV_FULL_MASK, s, j), bit = 1u << (v & 31);
            uint4 *out = reinterpret_cast<uint4 *>(reach + (i0 + j) * W);
            for (uint32_t q = lane; q < W / 4; q += 32) {
                const uint32_t w = q == v >> 7 ? (v >> 5) & 3u : 4u;
                out[q] = make_uint4(w == 0 ? bit : 0u, w == 1 ? bit : 0u, w == 2 ? bit : 0u, w == 3 ? bit : 0u);
            }
        }
        for (uint32_t todo = __ballot_sync(PV_FULL_MASK, slot == kSlotOverflow); todo; todo &= todo - 1u) {
            const uint32_t j = (uint32_t)(__ffs(todo) - 1);
            const uint16_t *l = lab + (size_t)__shfl_sync(PV_FULL_MASK, m, j) * V;
            comp_row(l, V, W, __ldg(l + __shfl_sync(PV_FULL_MASK, s, j)),
                     reinterpret_cast<uint4 *>(reach + (i0 + j) * W), lane);
        }
    }
}

// Permitted-vertex bitmap of a mask, by the whole block.
__device__ __forceinline__ void block_allow(uint32_t V, const uint8_t *__restrict__ region, uint32_t mask,
                                            uint32_t *s_allow) {
    const uint32_t t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (uint32_t v0 = 0; v0 < V; v0 += blockDim.x) {
        const uint32_t b = __ballot_sync(PV_FULL_MASK, source_permitted(v0 + t, V, region, mask));
        if (lane == 0 && v0 + warp * 32 < V) s_allow[(v0 >> 5) + warp] = b;
    }
}

// Sweeps of up to 64 sources to the fixpoint from the words in s_vis (bit j of
// s_vis[v]: v is known to be in source j's set), then source j's row to row_of(j)
// for those in `write`.
// The loops stay plain: four in-edges at a time made graphs of one or two edges a
// vertex half as slow again, and a transposition that stops at the last source
// used in place of 64 unrolled steps cost 6 us of 19 at 1,000 vertices (3,000
// vertices of one edge each, 24 masks, no cycles: the call 130 us, 104 plain).
template <typename RowOf>
__device__ __forceinline__ void msbfs_sweeps(uint32_t V, const uint32_t *__restrict__ in_offs,
                                             const uint32_t *__restrict__ in_cols, uint64_t write,
                                             uint32_t W, uint64_t *s_vis, const uint32_t *s_allow, RowOf row_of) {
    const uint32_t t = threadIdx.x, lane = t & 31, warp = t >> 5;
    volatile uint64_t *vis = s_vis;
    for (uint32_t iter = 0; iter <= V; ++iter) {
        int changed = 0;
        for (uint32_t v = t; v < V; v += kReachThreads) {
            if (!((s_allow[v >> 5] >> (v & 31)) & 1u)) continue;
            const uint64_t old = vis[v];
            uint64_t acc = old;
            const uint32_t a = __ldg(in_offs + v), b = __ldg(in_offs + v + 1);
            for (uint32_t e = a; e < b; ++e) acc |= vis[__ldg(in_cols + e)];
            if (acc != old) {
                vis[v] = acc;
                changed = 1;
            }
        }
        if (!__syncthreads_or(changed)) break;
    }
    // transpose: warp handles 128 vertices (4 words) per step
    const uint32_t groups = W / 4;
    for (uint32_t q = warp; q < groups; q += kReachThreads / 32) {
        uint64_t x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t v = q * 128 + i * 32 + lane;
            x[i] = v < V ? vis[v] : 0ull;
        }
        uint4 lo = make_uint4(0, 0, 0, 0), hi = make_uint4(0, 0, 0, 0);
        for (uint32_t j = 0; j < 64; ++j) {   // (unrolled: all 64, used or not)
            uint32_t b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) b[i] = __ballot_sync(PV_FULL_MASK, (x[i] >> j) & 1ull);
            if (lane == (j & 31)) {
                if (j < 32) lo = make_uint4(b[0], b[1], b[2], b[3]);
                else hi = make_uint4(b[0], b[1], b[2], b[3]);
            }
        }
        if ((write >> lane) & 1ull) reinterpret_cast<uint4 *>(row_of(lane))[q] = lo;
        if ((write >> (lane + 32)) & 1ull) reinterpret_cast<uint4 *>(row_of(lane + 32))[q] = hi;
    }
}

__global__ void __launch_bounds__(kReachThreads) reach_msbfs_kernel(
    uint32_t V, const uint32_t *__restrict__ in_offs, const uint32_t *__restrict__ in_cols,
    const uint8_t *__restrict__ region, uint32_t num_src, const uint32_t *__restrict__ src, uint32_t num_masks,
    const uint32_t *__restrict__ masks, uint32_t *__restrict__ reach, uint32_t W, const uint32_t *flags) {
    if (flags && component_path(flags)) return;
    extern __shared__ uint64_t s_vis[];                 // [V]
    __shared__ uint32_t s_allow[kReachMaxV / 32], s_on[2];   // s_on: the permitted sources
    const uint32_t nbatch = (num_src + 63) / 64, t = threadIdx.x;
    const uint64_t items = (uint64_t)nbatch * num_masks;   // (mask, source batch) pairs
    for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const uint32_t m = (uint32_t)(item / nbatch), j0 = (uint32_t)(item % nbatch) * 64;
        const uint32_t nb = min(64u, num_src - j0);
        block_allow(V, region, masks[m], s_allow);
        for (uint32_t v = t; v < V; v += kReachThreads) s_vis[v] = 0;
        __syncthreads();
        if (t < 64) {
            const uint32_t s = t < nb ? src[j0 + t] : V;
            const bool on = s < V && ((s_allow[s >> 5] >> (s & 31)) & 1u);
            if (on) atomicOr((unsigned long long *)&s_vis[s], 1ull << t);
            const uint32_t bal = __ballot_sync(PV_FULL_MASK, on);
            if ((t & 31) == 0) s_on[t >> 5] = bal;
        }
        __syncthreads();
        // with flags, blocks of other launches write the empty rows
        const uint64_t on = (uint64_t)s_on[1] << 32 | s_on[0], used = nb == 64 ? ~0ull : (1ull << nb) - 1ull;
        if (on || !flags)   // (block-uniform)
            msbfs_sweeps(V, in_offs, in_cols, flags ? on : used, W, s_vis, s_allow,
                         [&](uint32_t j) { return reach + ((size_t)m * num_src + j0 + j) * W; });
        __syncthreads();
    }
}

// Hub of a mask (search path, one block per mask): the permitted vertex with
// the most edges both in and out inside the permitted subgraph (the smaller of
// the two counts; ties to the lower id) and the vertices it reaches and is
// reached from there, searched level by level, half of the block each way.
// Any hub is exact; one inside the largest strongly connected component
// leaves the fewest sources to search, so a second is tried when the first
// one's component holds less than a quarter of the permitted vertices (unless both
// sets hold a quarter, or neither a sixteenth: then no large component is near),
// and the better is kept.  Last, the permitted sources outside the kept component
// are listed: rest[m][0 .. rest_n[m]), in no particular order.
constexpr int kHubThreads = 1024;
constexpr uint32_t kHubTries = 2;
// Most levels of a search where some permitted vertex has no edge in or none out.
// There a long search mostly ends without a component (a path of 3,000 vertices, 64
// masks: the call 13.2 ms without the limit, 5.3 by sweeps alone); a ring, where
// every level is needed, has no such vertex (1.7 ms, 5.3 by sweeps alone).
constexpr uint32_t kHubLevels = 256;
constexpr uint32_t kHubMinV = 1000;   // smallest graph (see the call)

struct HubSmem {   // two visited bitmaps, the permitted bitmap, two queues
    uint32_t allow, queue, total;
    __host__ __device__ explicit HubSmem(uint32_t V) {
        const uint32_t words = (V + 31) / 32;
        allow = 2 * words * 4;
        queue = allow + words * 4;
        total = queue + 2 * V * 2;
    }
};

__global__ void __launch_bounds__(kHubThreads) reach_hub_kernel(
    uint32_t V, const uint32_t *__restrict__ offs, const uint32_t *__restrict__ cols,
    const uint32_t *__restrict__ in_offs, const uint32_t *__restrict__ in_cols, const uint8_t *__restrict__ region,
    const uint32_t *__restrict__ masks, uint32_t *__restrict__ sets,
    uint32_t num_src, const uint32_t *__restrict__ src, uint32_t *__restrict__ rest, uint2 *__restrict__ rest_n,
    const uint32_t *flags) {
    if (component_path(flags)) return;
    extern __shared__ __align__(16) uint8_t s_dyn[];
    __shared__ uint32_t s_best, s_tail[2], s_core, s_all, s_rest;
    const HubSmem L(V);
    const uint32_t words = (V + 31) / 32, t = threadIdx.x, way = t / (kHubThreads / 2), m = blockIdx.x;
    uint32_t *s_sets = reinterpret_cast<uint32_t *>(s_dyn), *s_seen = s_sets + way * words;   // this half's visited set
    uint32_t *s_allow = reinterpret_cast<uint32_t *>(s_dyn + L.allow);
    uint16_t *queue = reinterpret_cast<uint16_t *>(s_dyn + L.queue) + way * V;
    const uint32_t *o = way ? in_offs : offs, *c = way ? in_cols : cols;
    if (t == 0) s_all = s_rest = 0;
    block_allow(V, region, masks[m], s_allow);
    __syncthreads();
    auto allowed = [&](uint32_t v) { return v < V && ((s_allow[v >> 5] >> (v & 31)) & 1u); };
    auto degree = [&](const uint32_t *off, const uint32_t *col, uint32_t v) {   // inside the permitted subgraph
        uint32_t n = 0;
        for (uint32_t e = __ldg(off + v), e1 = __ldg(off + v + 1); e < e1; e += 8) {   // eight columns in flight
            uint32_t x[8];
#pragma unroll
            for (uint32_t j = 0; j < 8; ++j) x[j] = e + j < e1 ? __ldg(col + e + j) : V;
#pragma unroll
            for (uint32_t j = 0; j < 8; ++j) n += allowed(x[j]) ? 1u : 0u;
        }
        return n;
    };
    for (uint32_t w = t; w < words; w += kHubThreads)
        if (s_allow[w]) atomicAdd(&s_all, (uint32_t)__popc(s_allow[w]));
    uint32_t tried[kHubTries], kept = 0;
    bool ends = false;   // this thread has seen a permitted vertex without edges in or out
    for (uint32_t attempt = 0; attempt < kHubTries; ++attempt) {
        if (t == 0) s_best = s_core = 0;
        __syncthreads();
        uint32_t best = 0;
        for (uint32_t v = t; v < V; v += kHubThreads) {
            bool skip = !allowed(v);
            for (uint32_t i = 0; i < attempt; ++i) skip = skip || v == tried[i];
            if (!skip) {
                const uint32_t d = min(min(degree(offs, cols, v), degree(in_offs, in_cols, v)), 0xFFFEu);
                ends = ends || d == 0;
                best = max(best, (d + 1u) << 16 | (0xFFFFu - v));
            }
        }
        best = __reduce_max_sync(PV_FULL_MASK, best);
        if ((t & 31) == 0) atomicMax(&s_best, best);
        const uint32_t most = __syncthreads_or(ends) ? kHubLevels : V;
        // a vertex that is not permitted counts as seen
        for (uint32_t w = t; w < 2 * words; w += kHubThreads) s_sets[w] = ~s_allow[w < words ? w : w - words];
        __syncthreads();
        const uint32_t hub = 0xFFFFu - (s_best & 0xFFFFu);
        tried[attempt] = hub;
        if (t % (kHubThreads / 2) == 0) {
            s_tail[way] = s_best != 0 ? 1u : 0u;   // 0: no permitted vertex is left to try
            if (s_best != 0) {
                queue[0] = (uint16_t)hub;
                s_seen[hub >> 5] |= 1u << (hub & 31);
            }
        }
        __syncthreads();
        uint32_t head = 0, levels = 0;
        const uint32_t sub = t % kEdgeLanes, lane8 = t % (kHubThreads / 2) / kEdgeLanes;
        while (true) {
            const uint32_t tail = *(volatile uint32_t *)&s_tail[way];
            // also: everyone has read the tail before it moves
            if (!__syncthreads_or(head < tail) || ++levels > most) break;
            for (uint32_t i = head + lane8; i < tail; i += kHubThreads / 2 / kEdgeLanes) {
                const uint32_t u = queue[i], b = __ldg(o + u + 1);
                for (uint32_t e = __ldg(o + u) + sub; e < b; e += kEdgeLanes) {
                    const uint32_t v = __ldg(c + e);
                    if (v >= V) continue;
                    const uint32_t bit = 1u << (v & 31);
                    if (!(*(volatile uint32_t *)&s_seen[v >> 5] & bit) && !(atomicOr(&s_seen[v >> 5], bit) & bit))
                        queue[atomicAdd(&s_tail[way], 1u)] = (uint16_t)v;
                }
            }
            head = tail;
            __syncthreads();
        }
        if (levels > most) {   // given up (block-uniform): an earlier hub's sets or none
            if (attempt == 0)
                for (uint32_t w = t; w < 2 * words; w += kHubThreads) sets[(size_t)m * 2 * words + w] = 0;
            __syncthreads();
            break;
        }
        for (uint32_t w = t; w < words; w += kHubThreads) {
            const uint32_t n = __popc(s_sets[w] & s_sets[words + w] & s_allow[w]);
            if (n) atomicAdd(&s_core, n);
        }
        __syncthreads();
        const uint32_t core = s_core;
        if (attempt == 0 || core > kept) {   // sets[m]: forward, then backward, words each
            for (uint32_t w = t; w < 2 * words; w += kHubThreads)
                sets[(size_t)m * 2 * words + w] = s_sets[w] & s_allow[w < words ? w : w - words];
            kept = core;
        }
        __syncthreads();
        // (block-uniform) large enough, both sets large and yet little in common,
        // or both small: no large component is near
        if (kept * 4 >= s_all || min(s_tail[0], s_tail[1]) * 4 >= s_all || max(s_tail[0], s_tail[1]) * 16 < s_all) break;
        __syncthreads();
    }
    const uint32_t lane = t & 31;
    const uint32_t *fwd = sets + (size_t)m * 2 * words, *bwd = fwd + words;   // written by this block
    for (uint32_t b = t - lane; b < num_src; b += kHubThreads) {
        const uint32_t s = b + lane < num_src ? src[b + lane] : V;
        const bool listed = allowed(s) && !((fwd[s >> 5] & bwd[s >> 5]) >> (s & 31) & 1u);
        const uint32_t bal = __ballot_sync(PV_FULL_MASK, listed);
        uint32_t base = 0;
        if (lane == 0 && bal) base = atomicAdd(&s_rest, (uint32_t)__popc(bal));
        base = __shfl_sync(PV_FULL_MASK, base, 0) + __popc(bal & ((1u << lane) - 1u));
        if (listed) rest[(size_t)m * num_src + base] = b + lane;
    }
    __syncthreads();
    if (t == 0) rest_n[m] = make_uint2(s_rest, kept * 4 >= s_all ? 1u : 0u);   // y: the component is large
}

// Rows of the search path.  Item (m, x) copies the hub's forward set to the
// rows of those of sources 64 x .. 64 x + 63 that lie in its strongly connected
// component, then takes 64 of the listed others.  When the component is large
// they are few and what they reach outside it is little: a warp searches each
// from its own queue, a source that reaches the hub over the forward set it
// starts with.  Searches past kOwnQueue vertices, and all of them when the
// component is small, are swept together.
// (3,001 vertices, 18,006 one-way edges, 24 masks, all sources: sweeps for
// every 64 sources took 311 of the call's 330 us; hub and rows take 60 of its
// 100, most of it the hub's levels.)
constexpr uint32_t kOwnQueue = 128;
struct HubRowSmem {   // vis[V] first
    uint32_t sets, allow, seen, queue, total;
    __host__ __device__ explicit HubRowSmem(uint32_t V) {
        const uint32_t words = (V + 31) / 32;
        sets = V * 8;
        allow = sets + 2 * words * 4;
        seen = allow + words * 4;                             // a warp's own set each
        queue = seen + kReachThreads / 32 * words * 4;        // and queue
        total = queue + kReachThreads / 32 * kOwnQueue * 2;
    }
};

__global__ void __launch_bounds__(kReachThreads) reach_hub_rows_kernel(
    uint32_t V, const uint32_t *__restrict__ offs, const uint32_t *__restrict__ cols,
    const uint32_t *__restrict__ in_offs, const uint32_t *__restrict__ in_cols, const uint8_t *__restrict__ region,
    uint32_t num_src, const uint32_t *__restrict__ src, uint32_t num_masks, const uint32_t *__restrict__ masks,
    const uint32_t *__restrict__ sets, const uint32_t *__restrict__ rest, const uint2 *__restrict__ rest_n,
    uint32_t *__restrict__ reach, uint32_t W, const uint32_t *flags) {
    if (component_path(flags)) return;
    extern __shared__ uint64_t s_vis[];
    __shared__ uint32_t s_list[64], s_sweep;   // sources (as row numbers) to sweep
    __shared__ uint64_t s_back;
    const HubRowSmem L(V);
    uint8_t *s_dyn = reinterpret_cast<uint8_t *>(s_vis);
    const uint32_t words = (V + 31) / 32, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t *fwd = reinterpret_cast<uint32_t *>(s_dyn + L.sets), *bwd = fwd + words;
    uint32_t *s_allow = reinterpret_cast<uint32_t *>(s_dyn + L.allow);
    uint32_t *seen = reinterpret_cast<uint32_t *>(s_dyn + L.seen) + warp * words;
    uint16_t *queue = reinterpret_cast<uint16_t *>(s_dyn + L.queue) + warp * kOwnQueue;
    const uint32_t batches = (num_src + 63) / 64;
    const uint64_t items = (uint64_t)batches * num_masks;
    for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const uint32_t m = (uint32_t)(item / batches), x = (uint32_t)(item % batches);
        __syncthreads();   // the item before is done with the shared state
        uint32_t *rows = reach + (size_t)m * num_src * W;
        const uint2 listed = rest_n[m];
        const uint32_t j0 = x * 64, n = j0 < listed.x ? min(64u, listed.x - j0) : 0u;
        const uint32_t *list = rest + (size_t)m * num_src + j0;
        if (t == 0) {
            s_sweep = 0;
            s_back = 0;
        }
        for (uint32_t w = t; w < 2 * words; w += kReachThreads) fwd[w] = sets[(size_t)m * 2 * words + w];
        if (n) block_allow(V, region, masks[m], s_allow);
        __syncthreads();
        auto in = [](const uint32_t *set, uint32_t v) { return (set[v >> 5] >> (v & 31)) & 1u; };
        if (warp < 2) {
            const uint32_t j = j0 + warp * 32 + lane, s = j < num_src ? src[j] : V;
            uint32_t todo = __ballot_sync(PV_FULL_MASK, s < V && in(fwd, s) && in(bwd, s));
            if (lane == 0) s_list[warp] = todo;
        }
        __syncthreads();
        for (uint32_t half = 0; half < 2; ++half) {
            uint32_t todo = s_list[half];
            for (uint32_t i = 0; todo; ++i, todo &= todo - 1u) {
                uint32_t *row = rows + (size_t)(j0 + half * 32 + (uint32_t)(__ffs(todo) - 1)) * W;
                if (i % (kReachThreads / 32) == warp)
                    for (uint32_t w = lane; w < W; w += 32) row[w] = w < words ? fwd[w] : 0u;
            }
        }
        if (n == 0) continue;   // block-uniform
        __syncthreads();        // s_list is free
        if (!listed.y) {
            if (t < n) s_list[t] = list[t];
            if (t == 0) s_sweep = n;
        } else {
            const uint32_t sub = lane % kEdgeLanes, lt = (1u << lane) - 1u;
            for (uint32_t i = warp; i < n; i += kReachThreads / 32) {
                const uint32_t j = list[i], s = src[j];
                const bool back = in(bwd, s) != 0;
                for (uint32_t w = lane; w < words; w += 32) seen[w] = back ? fwd[w] : 0u;
                __syncwarp();
                if (lane == 0) {
                    seen[s >> 5] |= 1u << (s & 31);
                    queue[0] = (uint16_t)s;
                }
                __syncwarp();
                uint32_t head = 0, tail = 1;
                bool over = false;
                while (head < tail && !over) {
                    // four vertices of the queue, eight lanes to each
                    const uint32_t q = head + lane / kEdgeLanes;
                    uint32_t e = 0, e1 = 0;
                    if (q < tail) {
                        const uint32_t u = queue[q];
                        e = __ldg(offs + u) + sub;
                        e1 = __ldg(offs + u + 1);
                    }
                    head = min(head + 32 / kEdgeLanes, tail);
                    while (__any_sync(PV_FULL_MASK, e < e1) && !over) {
                        bool push = false;
                        uint32_t v = 0;
                        if (e < e1) {
                            v = __ldg(cols + e);
                            e += kEdgeLanes;
                            if (v < V && in(s_allow, v)) {
                                const uint32_t bit = 1u << (v & 31);
                                push = !(atomicOr(&seen[v >> 5], bit) & bit);
                            }
                        }
                        const uint32_t pushed = __ballot_sync(PV_FULL_MASK, push);
                        over = tail + __popc(pushed) > kOwnQueue;
                        if (push && !over) queue[tail + __popc(pushed & lt)] = (uint16_t)v;
                        tail += over ? 0u : __popc(pushed);
                        __syncwarp();
                    }
                }
                if (over) {
                    if (lane == 0) s_list[atomicAdd(&s_sweep, 1u)] = j;
                } else {
                    uint32_t *row = rows + (size_t)j * W;
                    for (uint32_t w = lane; w < W; w += 32) row[w] = w < words ? seen[w] : 0u;
                }
                __syncwarp();
            }
        }
        __syncthreads();
        const uint32_t nb = s_sweep;
        if (nb == 0) continue;   // block-uniform
        // a source that reaches the hub starts with the hub's whole forward set
        if (t < nb && in(bwd, src[s_list[t]])) atomicOr((unsigned long long *)&s_back, 1ull << t);
        __syncthreads();
        const uint64_t back = s_back;
        for (uint32_t v = t; v < V; v += kReachThreads) s_vis[v] = in(fwd, v) ? back : 0ull;
        __syncthreads();
        if (t < nb) atomicOr((unsigned long long *)&s_vis[src[s_list[t]]], 1ull << t);
        __syncthreads();
        const uint64_t used = nb == 64 ? ~0ull : (1ull << nb) - 1ull;   // listed sources are permitted
        msbfs_sweeps(V, in_offs, in_cols, used, W, s_vis, s_allow,
                     [&](uint32_t j) { return rows + (size_t)s_list[j] * W; });
    }
}

// The dynamic shared-memory limits of the block-wide kernels are
// process-wide settings per device.  They are raised once per device to the
// largest size any call can ask for (under a mutex), so that no call lowers
// the limit between another thread's setting and launch.
constexpr int kSmemAttrMaxDevices = 64;
std::mutex g_smem_attr_mutex;
bool g_smem_attr_set[kSmemAttrMaxDevices] = {};

cudaError_t reach_smem_limits() {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kSmemAttrMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_smem_attr_mutex);
    if (g_smem_attr_set[dev]) return cudaSuccess;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    const int rows_max = optin - 1024;
    const int lab_max = (int)LabelSmem(kReachMaxV).total;
    const int bfs_max = (int)(kReachMaxV * 8), hub_max = (int)HubSmem(kReachMaxV).total;
    if ((e = cudaFuncSetAttribute(reach_labels_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  std::min(lab_max, rows_max))) != cudaSuccess ||
        (e = cudaFuncSetAttribute(reach_msbfs_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  std::min(bfs_max, rows_max))) != cudaSuccess ||
        (e = cudaFuncSetAttribute(reach_hub_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  std::min(hub_max, rows_max))) != cudaSuccess ||
        (e = cudaFuncSetAttribute(reach_hub_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, rows_max)) !=
            cudaSuccess)
        return e;
    g_smem_attr_set[dev] = true;
    return cudaSuccess;
}

}  // namespace

extern "C" int pv_compliant_reach(pv_ctx *ctx, uint32_t V, const uint32_t *d_offs, uint32_t num_edges,
                                  const uint32_t *d_cols, const uint8_t *d_region, uint32_t num_src,
                                  const uint32_t *d_src, uint32_t num_masks, const uint32_t *d_masks,
                                  uint32_t *d_reach, uint32_t words_per_row, pv_stream stream) {
    if (!ctx) return PV_EINVAL;
    if (V == 0 || V > kReachMaxV) return pv_fail(ctx, PV_EINVAL, "pv_compliant_reach: V must be 1..%u", kReachMaxV);
    if (words_per_row % 4 != 0 || words_per_row < (V + 31) / 32)
        return pv_fail(ctx, PV_EINVAL, "pv_compliant_reach: words_per_row must be >= ceil(V/32) and a multiple of 4");
    if (num_src == 0 || num_masks == 0) return PV_OK;
    if (!d_offs || !d_region || !d_src || !d_masks || !d_reach || (num_edges && !d_cols))
        return pv_fail(ctx, PV_EINVAL, "pv_compliant_reach: NULL device pointer");
    if (((uintptr_t)d_reach & 15) != 0) return pv_fail(ctx, PV_EINVAL, "pv_compliant_reach: d_reach must be 16-byte aligned");
    if (num_masks > 65535) return pv_fail(ctx, PV_EINVAL, "pv_compliant_reach: num_masks must be <= 65535");
    const size_t o_indeg = 0, o_in_offs = align256((size_t)(V + 1) * 4);
    const size_t o_cursor = o_in_offs + align256((size_t)(V + 1) * 4);
    const size_t o_cols = o_cursor + align256((size_t)V * 4);
    const size_t o_pairs = o_cols + align256((size_t)num_edges * 4 + 4);   // undirected pairs
    const size_t o_lab = o_pairs + align256((size_t)num_edges * 4 + 16);   // component labels, or the hubs' sets
    bool comp = ctx->opt_reach == 0;
    const size_t set_words = 2 * (((size_t)V + 31) / 32);                  // a hub's two sets
    const size_t o_slots = o_lab + align256((size_t)num_masks * std::max<size_t>((size_t)V * 2, set_words * 4));
    const size_t o_table = o_slots + align256((size_t)num_masks * V * 2);
    // table rows a mask: every component's (of two vertices or more) when they
    // fit kTableBytes; past the table rows come from the labels
    const size_t mask_row = (size_t)num_masks * words_per_row * 4;
    const uint32_t cap = (uint32_t)std::min<size_t>(V / 2, kTableBytes / mask_row);
    // search path: the sources to search of every mask and their counts, in the table's place
    const size_t o_rest_n = o_table + align256((size_t)num_masks * num_src * 4);
    const size_t total = std::max(o_table + cap * mask_row, o_rest_n + (size_t)num_masks * 8);
    uint8_t *base = (uint8_t *)pv_scratch(ctx, comp ? total : o_lab);
    if (!base && comp) {   // little memory is left beside the caller's rows: the sweeps need the least
        ctx->err.clear();
        comp = false;
        base = (uint8_t *)pv_scratch(ctx, o_lab);
    }
    if (!base) return PV_ENOMEM;
    uint32_t *indeg = (uint32_t *)(base + o_indeg), *in_offs = (uint32_t *)(base + o_in_offs);
    uint32_t *cursor = (uint32_t *)(base + o_cursor), *in_cols = (uint32_t *)(base + o_cols);
    uint32_t *pairs = (uint32_t *)(base + o_pairs);
    cudaStream_t st = (cudaStream_t)stream;
    uint16_t *lab = (uint16_t *)(base + o_lab);     // [num_masks][V] (component path)
    uint32_t *sets = (uint32_t *)(base + o_lab);    // [num_masks][2][ceil(V / 32)] (search path): never both
    uint16_t *slots = (uint16_t *)(base + o_slots);   // [num_masks][V]
    uint32_t *table = (uint32_t *)(base + o_table);   // [num_masks][cap][words_per_row]
    uint32_t *rest = (uint32_t *)(base + o_table);    // [num_masks][num_src] (search path)
    uint2 *rest_n = (uint2 *)(base + o_rest_n);       // [num_masks] (search path)
    PV_TRY_CUDA(ctx, reach_smem_limits(), "reach shared-memory limits");
    if (comp && !ctx->reach_side) {   // first call: the search path's side stream
        PV_TRY_CUDA(ctx, cudaStreamCreateWithFlags(&ctx->reach_side, cudaStreamNonBlocking), "reach side stream");
        PV_TRY_CUDA(ctx, cudaEventCreateWithFlags(&ctx->reach_fork, cudaEventDisableTiming), "reach fork event");
        PV_TRY_CUDA(ctx, cudaEventCreateWithFlags(&ctx->reach_join, cudaEventDisableTiming), "reach join event");
    }
    ctx->last_reach_comp = comp;
    uint32_t *flags = ctx->d_reach_flags;
    const uint32_t sms = (uint32_t)ctx->num_sms;
    const uint32_t egrid = std::min<uint32_t>((V * kEdgeLanes + kGridThreads - 1) / kGridThreads, sms * 8);
    const int pr = pv_prof_start(ctx, st, PV_K_REACH);
    reach_clear_kernel<<<(V + 255) / 256, 256, 0, st>>>(V, indeg, flags);
    if (!comp) {
        // the counts, and the flag at flags[kBadOffs], as the no-allocation call
        const uint32_t wgrid = std::min<uint32_t>((V + kGridThreads / 32 - 1) / (kGridThreads / 32), sms * 8);
        reach_check_kernel<<<wgrid, kGridThreads, 0, st>>>(V, num_edges, d_offs, d_cols, d_region, indeg, flags, pairs,
                                                           ctx->d_status, wgrid, ClearArgs{});
        reach_scan_kernel<<<1, 1024, 0, st>>>(V, indeg, in_offs, cursor, nullptr, flags + kBadOffs);
        reach_fill_kernel<<<egrid, kGridThreads, 0, st>>>(V, num_edges, d_offs, d_cols, cursor, in_cols, nullptr,
                                                          flags + kBadOffs);
        const size_t smem = (size_t)V * 8;
        const int per_sm = std::max(1, pv_blocks_per_sm(ctx, (const void *)reach_msbfs_kernel, kReachThreads, smem));
        const uint64_t items = (uint64_t)((num_src + 63) / 64) * num_masks;
        reach_msbfs_kernel<<<(uint32_t)std::min<uint64_t>(items, (uint64_t)per_sm * sms), kReachThreads, smem, st>>>(
            V, in_offs, in_cols, d_region, num_src, d_src, num_masks, d_masks, d_reach, words_per_row, nullptr);
        pv_prof_stop(ctx, st, pr, 5);
        return pv_check_launch(ctx, "reach kernels");
    }
    const uint32_t wgrid = std::min<uint32_t>((V + kGridThreads / 32 - 1) / (kGridThreads / 32), sms * 8);
    // the empty rows: a third beside the check, the rest beside the labels,
    // about as their times are
    const uint64_t all_rows = (uint64_t)num_masks * num_src;
    ClearArgs clear = {d_masks, d_src, num_src, words_per_row, d_reach, 0, all_rows / 96 * 32};
    reach_check_kernel<<<wgrid + 2 * sms, kGridThreads, 0, st>>>(V, num_edges, d_offs, d_cols, d_region, indeg, flags,
                                                                 pairs, ctx->d_status, wgrid, clear);
    clear.lo = clear.hi;
    clear.hi = all_rows;
    // Both paths are launched and the flags pick the one that works: the
    // search path's kernels go to the side stream, so on a symmetric graph
    // their launches overlap the labels and rows kernels instead of queueing
    // behind them; the caller's stream joins it at the end.
    PV_TRY_CUDA(ctx, cudaEventRecord(ctx->reach_fork, st), "reach fork");
    PV_TRY_CUDA(ctx, cudaStreamWaitEvent(ctx->reach_side, ctx->reach_fork, 0), "reach fork");
    cudaStream_t sw = ctx->reach_side;
    reach_scan_kernel<<<1, 1024, 0, sw>>>(V, indeg, in_offs, cursor, flags, flags + kBadOffs);
    reach_fill_kernel<<<egrid, kGridThreads, 0, sw>>>(V, num_edges, d_offs, d_cols, cursor, in_cols, flags,
                                                      flags + kBadOffs);
    // A hub and its two sets take some 10 to 25 us before the first row: more than
    // sweeps while every (mask, 64 sources) item has a block of its own, and on
    // small graphs (sweeps / hub, us; 64 masks: 700 vertices of 1.5 random edges each
    // 76/98, of 6 82/61; 1,000: 96/116, 116/64; 2,000: 260/237, 318/91; without cycles
    // and one edge each 43/53, 53/60, 111/110).
    const uint64_t items = (uint64_t)((num_src + 63) / 64) * num_masks;
    const bool by_hub = items > 4ull * sms && V >= kHubMinV;
    if (by_hub) {
        reach_hub_kernel<<<num_masks, kHubThreads, HubSmem(V).total, sw>>>(V, d_offs, d_cols, in_offs, in_cols, d_region,
                                                                          d_masks, sets, num_src, d_src, rest, rest_n,
                                                                          flags);
        // at most eight blocks an SM: on a symmetric graph they all start and return
        // (the 4,096-vertex WAN 57.4 us with sixteen, 55.4 with eight).  A block's items
        // lie a grid apart: neighbours are of one mask, and a mask with long searches
        // would keep its few blocks for twice as long (8,000 vertices of three edges
        // each, 24 masks: 945 us, 627 a grid apart)
        reach_hub_rows_kernel<<<(uint32_t)std::min<uint64_t>(items, 8ull * sms), kReachThreads, HubRowSmem(V).total, sw>>>(
            V, d_offs, d_cols, in_offs, in_cols, d_region, num_src, d_src, num_masks, d_masks, sets, rest, rest_n,
            d_reach, words_per_row, flags);
    } else {
        reach_msbfs_kernel<<<(uint32_t)std::min<uint64_t>(items, 0x7FFFFFFFull), kReachThreads, (size_t)V * 8, sw>>>(
            V, in_offs, in_cols, d_region, num_src, d_src, num_masks, d_masks, d_reach, words_per_row, flags);
    }
    // a part for every 1,024 vertices of large graphs while most SMs are idle (a
    // second one costs 2 us of 25 at 300 vertices, of 58 on the 4,096-vertex WAN with
    // 64 masks)
    const uint32_t parts = num_masks * 4 <= sms && V >= 4096 ? std::min({kLabelParts, sms / num_masks, V / 1024}) : 1u;
    reach_labels_kernel<<<num_masks * parts + sms, kLabelThreads, LabelSmem(V).total, st>>>(
        V, pairs, d_region, d_masks, lab, slots, table, cap, words_per_row, flags, ctx->d_status, num_masks * parts, parts,
        clear);
    {
        // rows a warp: 32, fewer while that leaves SMs idle (300 vertices, one
        // mask: the call takes 28.4 us with 32, 22 with one), but not more than two
        // blocks an SM: on other graphs the sweeps' blocks are placed around these
        // (1,000 vertices, 16 masks, six edges each: 57 us, with four blocks 75)
        const uint64_t rows = (uint64_t)num_masks * num_src;
        const uint32_t per_warp = (uint32_t)std::min<uint64_t>(32, std::max<uint64_t>(1, rows / (sms * 16)));
        const uint64_t warps = (rows + per_warp - 1) / per_warp;
        const uint32_t rgrid = (uint32_t)std::min<uint64_t>((warps + kRowThreads / 32 - 1) / (kRowThreads / 32), sms * 8);
        reach_rows_kernel<<<rgrid, kRowThreads, 0, st>>>(V, lab, slots, table, cap, num_masks, num_src, d_src, d_reach,
                                                         words_per_row, per_warp, flags);
    }
    PV_TRY_CUDA(ctx, cudaEventRecord(ctx->reach_join, sw), "reach join");
    PV_TRY_CUDA(ctx, cudaStreamWaitEvent(st, ctx->reach_join, 0), "reach join");
    pv_prof_stop(ctx, st, pr, by_hub ? 8 : 7);
    return pv_check_launch(ctx, "reach kernels");
}

// -----------------------------------------------------------------------------
// Compliant reach that allocates nothing.
//
// For callers that must not allocate device memory themselves or through this
// library: a host program whose device memory is owned by another framework's
// pool or held to a fixed budget, or a latency-critical caller that cannot
// afford the device-wide synchronisation cudaMalloc / cudaFree may imply.
// The in-edge CSR this path builds lives in one static device array below;
// every GPU that loads the library holds it until the process exits.
// -----------------------------------------------------------------------------
namespace {

constexpr size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

constexpr uint32_t kNoAllocMaxEdges = 1u << 18;   // directed edges accepted by the no-allocation call
constexpr size_t kNoAllocIndeg = 256;              // [0, 256): status word
constexpr size_t kNoAllocInOffs = kNoAllocIndeg + up256((size_t)(kReachMaxV + 1) * 4);
constexpr size_t kNoAllocCursor = kNoAllocInOffs + up256((size_t)(kReachMaxV + 1) * 4);
constexpr size_t kNoAllocCols = kNoAllocCursor + up256((size_t)kReachMaxV * 4);
constexpr size_t kNoAllocBytes = kNoAllocCols + up256((size_t)kNoAllocMaxEdges * 4);   // about 1.2 MB

__device__ __align__(256) uint8_t g_reach_noalloc_scratch[kNoAllocBytes];

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mutex;
uint8_t *g_noalloc_base[kNoAllocMaxDevices] = {};

// Device address of the static array on the current device, looked up once
// per device (in host code the array's name is not a device address) and
// kept for the life of the process: after a cudaDeviceReset the module is
// loaded again and the kept address would be stale, so the library is not
// to be used on a device after a reset.
int noalloc_scratch(uint8_t **out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return PV_ECUDA;
    if (dev < 0 || dev >= kNoAllocMaxDevices) return PV_EINVAL;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_base[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_reach_noalloc_scratch) != cudaSuccess || !p) return PV_ECUDA;
        g_noalloc_base[dev] = static_cast<uint8_t *>(p);
    }
    *out = g_noalloc_base[dev];
    return PV_OK;
}

}  // namespace

extern "C" int pv_compliant_reach_noalloc(uint32_t V, const uint32_t *d_offs, uint32_t num_edges,
                                          const uint32_t *d_cols, const uint8_t *d_region, uint32_t num_src,
                                          const uint32_t *d_src, uint32_t num_masks, const uint32_t *d_masks,
                                          uint32_t *d_reach, uint32_t words_per_row, pv_stream stream) {
    if (V == 0 || V > kReachMaxV) return PV_EINVAL;
    if (num_edges > kNoAllocMaxEdges) return PV_EINVAL;
    if (words_per_row % 4 != 0 || words_per_row < (V + 31) / 32) return PV_EINVAL;
    if (num_src == 0 || num_masks == 0) return PV_OK;
    if (!d_offs || !d_region || !d_src || !d_masks || !d_reach || (num_edges && !d_cols)) return PV_EINVAL;
    if (((uintptr_t)d_reach & 15) != 0 || num_masks > 65535) return PV_EINVAL;
    uint8_t *base = nullptr;
    const int rc = noalloc_scratch(&base);
    if (rc != PV_OK) return rc;
    int32_t *status = reinterpret_cast<int32_t *>(base);
    uint32_t *indeg = reinterpret_cast<uint32_t *>(base + kNoAllocIndeg);
    uint32_t *in_offs = reinterpret_cast<uint32_t *>(base + kNoAllocInOffs);
    uint32_t *cursor = reinterpret_cast<uint32_t *>(base + kNoAllocCursor);
    uint32_t *in_cols = reinterpret_cast<uint32_t *>(base + kNoAllocCols);
    cudaStream_t st = (cudaStream_t)stream;
    // the array keeps the previous call's contents: clear what must start at zero
    if (cudaMemsetAsync(base, 0, kNoAllocIndeg + (size_t)(V + 1) * 4, st) != cudaSuccess) return PV_ECUDA;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return PV_ECUDA;
    const uint32_t grid = std::min<uint32_t>((V * kEdgeLanes + kGridThreads - 1) / kGridThreads, (uint32_t)sms * 8);
    reach_indeg_kernel<<<grid, kGridThreads, 0, st>>>(V, num_edges, d_offs, d_cols, d_region, indeg, status);
    reach_scan_kernel<<<1, 1024, 0, st>>>(V, indeg, in_offs, cursor, nullptr, indeg + V);
    reach_fill_kernel<<<grid, kGridThreads, 0, st>>>(V, num_edges, d_offs, d_cols, cursor, in_cols, nullptr,
                                                     indeg + V);
    const size_t smem = (size_t)V * 8;
    if (reach_smem_limits() != cudaSuccess) return PV_ECUDA;
    const uint64_t items = (uint64_t)((num_src + 63) / 64) * num_masks;
    const uint32_t g2 = (uint32_t)std::min<uint64_t>(items, (uint64_t)sms * 4);
    reach_msbfs_kernel<<<g2, kReachThreads, smem, st>>>(V, in_offs, in_cols, d_region, num_src, d_src, num_masks,
                                                       d_masks, d_reach, words_per_row, nullptr);
    return cudaGetLastError() == cudaSuccess ? PV_OK : PV_ECUDA;
}
