// Path scheduling (Sec. 4.2: the flow scheduling module computes paths that
// respect the constraint object -- weighted Dijkstra, breadth-first when no
// weights are given -- and turns each path into per-hop flow rules).
//
// A request asks for a path from a source host to a destination host over
// the switches its jurisdiction mask permits and its policy does not forbid,
// through the policy's waypoints in order.  The path is the concatenation of
// shortest segments, each made canonical: walking back from the segment's
// end, every switch takes the predecessor link with the smallest (source
// switch, source port) among those on a shortest path.  Any exact shortest-
// path algorithm therefore yields the same path.  A warp per segment searches
// from the frontier of switches whose distance fell, bounded by the target's
// (sched_segments_kernel); networks whose state does not fit, and the options,
// run one block per request with in-place Bellman-Ford pull sweeps over the
// links into each switch (every sweep only lowers upper bounds, so the fixpoint
// is exact), all in shared memory, and one thread walks the predecessors back
// (sched_paths_kernel).
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "pv_internal.cuh"

namespace {

constexpr int kSchedThreads = 256;
constexpr uint32_t kSchedMaxSwitches = 16384;
constexpr uint32_t kInf = 0xFFFFFFFFu;

struct SchedArgs {
    uint32_t S, H;
    const uint8_t *region;
    const uint32_t *port_offs;
    const uint16_t *host_switch, *host_port;
    const uint32_t *in_offs, *in_links;
    const uint16_t *weights;       // [ports] or null (unit weights)
    const uint4 *pol_hdr;          // path policies (null: none loaded)
    const uint16_t *pol_sw;
    uint32_t num_pol;
    const pv_path_req *req;
    uint32_t R, max_len;
    uint32_t *visits;              // [R][max_len]: switch << 16 | in_port << 8 | out_port
    uint8_t *len, *status;
};

__device__ __forceinline__ uint32_t link_weight(const SchedArgs &a, uint32_t u, uint32_t p) {
    if (!a.weights) return 1u;
    const uint32_t w = a.weights[a.port_offs[u] + p];
    return w ? w : 1u;   // a weight of 0 counts as 1
}

// With kStaged the block first copies the links into each switch, with their
// weights resolved, to shared memory, where every sweep and the predecessor
// pass read them.
template <bool kStaged>
__global__ void __launch_bounds__(kSchedThreads) sched_paths_kernel(SchedArgs a) {
    extern __shared__ uint32_t s_mem[];
    const uint32_t S = a.S, okw = (S + 31) / 32;
    volatile uint32_t *dist = s_mem;                 // [S]
    uint32_t *ok = s_mem + S;                        // [okw] permitted switches
    uint32_t *vis = ok + okw;                        // [max_len] visits
    uint32_t *back = vis + a.max_len;                // [max_len] links of a segment, last first
    uint32_t *pred = back + a.max_len;               // [S] canonical predecessor link (kStaged)
    uint32_t *g_offs = pred + (kStaged ? S : 0u);    // [S + 1]
    const uint32_t L = a.in_offs[S];
    uint32_t *g_links = g_offs + (kStaged ? S + 1 : 0u);   // [L]
    uint16_t *g_w = reinterpret_cast<uint16_t *>(g_links + (kStaged ? L : 0u));   // [L] link weights
    __shared__ uint32_t s_st, s_n;
    const uint32_t t = threadIdx.x, nt = blockDim.x;
    auto allowed = [&](uint32_t s) { return (ok[s >> 5] >> (s & 31)) & 1u; };
    const uint32_t *in_offs = a.in_offs, *in_links = a.in_links;
    if (kStaged) {
        for (uint32_t v = t; v <= S; v += nt) g_offs[v] = a.in_offs[v];
        for (uint32_t l = t; l < L; l += nt) {
            const uint32_t x = a.in_links[l];
            g_links[l] = x;
            g_w[l] = (uint16_t)link_weight(a, x >> 16, (x >> 8) & 0xFFu);
        }
        __syncthreads();
        in_offs = g_offs;
        in_links = g_links;
    }
    // weight of in-link l = (u, p) of switch v
    auto lw = [&](uint32_t l, uint32_t x) -> uint32_t {
        return kStaged ? (uint32_t)g_w[l] : link_weight(a, x >> 16, (x >> 8) & 0xFFu);
    };
    for (uint32_t r = blockIdx.x; r < a.R; r += gridDim.x) {
        const pv_path_req q = a.req[r];
        if (q.src_host >= a.H || q.dst_host >= a.H) {
            if (t == 0) {
                a.status[r] = PV_PATH_NOSRC;
                a.len[r] = 0;
            }
            continue;
        }
        uint4 ph = make_uint4(0, 0, 0, 0);
        if (a.pol_hdr && q.policy < a.num_pol) ph = a.pol_hdr[q.policy];
        for (uint32_t w = t; w < okw; w += nt) {
            uint32_t bits = 0;
            for (uint32_t b = 0; b < 32; ++b) {
                const uint32_t s = w * 32 + b;
                if (s >= S) break;
                const uint32_t reg = a.region[s];
                bool fine = reg < 32 && ((q.allowed_mask >> reg) & 1u);
                for (uint32_t i = 0; i < ph.y && fine; ++i) fine = a.pol_sw[ph.x + i] != s;
                if (fine) bits |= 1u << b;
            }
            ok[w] = bits;
        }
        __syncthreads();
        const uint32_t src_sw = a.host_switch[q.src_host], dst_sw = a.host_switch[q.dst_host];
        uint32_t st = (allowed(src_sw) && allowed(dst_sw)) ? PV_PATH_OK : PV_PATH_BLOCKED;
        for (uint32_t i = 0; i < ph.w && st == PV_PATH_OK; ++i) {
            const uint32_t w = a.pol_sw[ph.z + i];   // of policies loaded for other tables: maybe no switch of these
            if (w >= S || !allowed(w)) st = PV_PATH_BLOCKED;
        }
        uint32_t n = 1, cur = src_sw;
        if (t == 0) vis[0] = src_sw << 16 | (uint32_t)a.host_port[q.src_host] << 8;
        for (uint32_t i = 0; i <= ph.w && st == PV_PATH_OK; ++i) {
            const uint32_t tgt = i < ph.w ? a.pol_sw[ph.z + i] : dst_sw;
            if (tgt == cur) continue;
            for (uint32_t v = t; v < S; v += nt) dist[v] = v == cur ? 0u : kInf;
            __syncthreads();
            // pull sweeps until nothing changes (at most S are needed)
            for (uint32_t round = 0; round <= S; ++round) {
                int changed = 0;
                for (uint32_t v = t; v < S; v += nt) {
                    if (v == cur || !allowed(v)) continue;
                    uint32_t best = dist[v];
                    for (uint32_t l = in_offs[v]; l < in_offs[v + 1]; ++l) {
                        const uint32_t x = in_links[l], u = x >> 16;
                        if (!allowed(u)) continue;
                        const uint32_t du = dist[u];
                        if (du == kInf) continue;
                        const uint32_t c = du + lw(l, x);
                        if (c < best) best = c;
                    }
                    if (best < dist[v]) {
                        dist[v] = best;
                        changed = 1;
                    }
                }
                if (!__syncthreads_or(changed)) break;
            }
            if (dist[tgt] == kInf) {
                st = PV_PATH_BLOCKED;
                break;
            }
            if (kStaged) {
                // every switch's canonical predecessor at once: the first link
                // (smallest (u, p)) on a shortest path into it
                for (uint32_t v = t; v < S; v += nt) {
                    uint32_t pick = kInf;
                    if (v != cur && dist[v] != kInf)
                        for (uint32_t l = in_offs[v]; l < in_offs[v + 1] && pick == kInf; ++l) {
                            const uint32_t x = in_links[l], u = x >> 16;
                            if (allowed(u) && dist[u] != kInf && dist[u] + lw(l, x) == dist[v]) pick = x;
                        }
                    pred[v] = pick;
                }
                __syncthreads();
            }
            if (t == 0) {
                // canonical walk back from tgt: smallest (u, p) on a shortest path
                const uint32_t room = a.max_len - n;
                uint32_t k = 0, v = tgt, s_status = PV_PATH_OK;
                while (v != cur) {
                    uint32_t pick = kInf;
                    if (kStaged) {
                        pick = pred[v];
                    } else {
                        for (uint32_t l = in_offs[v]; l < in_offs[v + 1] && pick == kInf; ++l) {
                            const uint32_t x = in_links[l], u = x >> 16;
                            if (!allowed(u) || dist[u] == kInf) continue;
                            if (dist[u] + lw(l, x) == dist[v]) pick = x;
                        }
                    }
                    if (pick == kInf) {   // cannot happen once the distances are exact
                        s_status = PV_PATH_BLOCKED;
                        break;
                    }
                    if (k >= room) {
                        s_status = PV_PATH_TOO_LONG;
                        break;
                    }
                    // {source port, switch v, its in_port}
                    back[k++] = ((pick >> 8) & 0xFFu) << 24 | v << 8 | (pick & 0xFFu);
                    v = pick >> 16;
                }
                if (s_status == PV_PATH_OK)
                    while (k > 0) {
                        const uint32_t b = back[--k];
                        vis[n - 1] |= b >> 24;                              // out port toward the next switch
                        vis[n++] = ((b >> 8) & 0xFFFFu) << 16 | (b & 0xFFu) << 8;
                    }
                s_st = s_status;
                s_n = n;
            }
            __syncthreads();
            st = s_st;
            n = s_n;
            cur = tgt;
        }
        if (st == PV_PATH_OK) {
            if (t == 0) vis[n - 1] |= a.host_port[q.dst_host];
            if (t == 0) s_st = PV_PATH_OK;
            __syncthreads();
            // a recurring (switch, in_port) cannot be realised by header rules
            for (uint32_t i = t; i < n; i += nt)
                for (uint32_t j = i + 1; j < n; ++j)
                    if ((vis[i] >> 8) == (vis[j] >> 8)) s_st = PV_PATH_REPEAT;
            __syncthreads();
            st = s_st;
        }
        for (uint32_t i = t; i < n && st == PV_PATH_OK; i += nt) a.visits[(size_t)r * a.max_len + i] = vis[i];
        if (t == 0) {
            a.status[r] = (uint8_t)st;
            a.len[r] = (uint8_t)(st == PV_PATH_OK ? n : 0);
        }
        __syncthreads();   // shared state is rebuilt for the next request
    }
}

// The same paths with a warp per path segment.  A request's segments (source
// to first waypoint, and so on) do not depend on one another, so a block
// takes a range of requests, its warps draw segments until none is left, and
// a warp per request then joins the pieces.  A segment is searched from a
// frontier: the switches lowered in one step are listed, and the next step
// relaxes only their outgoing links (four lanes to a switch, atomicMin in
// shared memory).  Labels count from 1; a switch that is not permitted holds
// 0, which no label undercuts.  A label that does not stay below the target's
// is dropped: every switch on a shortest path to the target lies nearer than
// it, so those are exact at the end, and no other label can satisfy the
// canonical walk back's equality.
// A block per request swept every switch until a sweep changed nothing, and
// waited at a block barrier each time: 10,000 weighted requests on 512
// switches took 1,098 us with their rules, 165 us this way.  Bound by the
// shared-memory latency of a segment's steps (about 3,900 warp instructions a
// segment, 53% of issue slots) and, at a group's end, by its longest segments.
// Tried: 32 segments
// to a warp, one per lane (386 us: the union of their frontiers is every
// switch), and a warp per whole request (375 us: as long as the requests with
// the most waypoints).
constexpr uint32_t kSegReqs = 128;               // most requests of a block's group
constexpr uint32_t kSegTasks = 512;              // most segments of a group
constexpr size_t kPieceBytes = 42 * 1024;        // pieces of a group's segments, max_len words each

struct SegmentSmem {
    uint32_t in_offs, in, out, in_w, region, pieces, tasks, warps, marks, list, per_warp, okw;
    __host__ __device__ SegmentSmem(uint32_t S, uint32_t L, uint32_t max_len) {
        // out_offs[S + 1] first
        in_offs = (S + 1) * 4;
        in = in_offs + (S + 1) * 4;              // in[L]: u << 16 | p << 8 | q, links into each switch
        out = in + L * 4;                        // out[L]: v << 16 | weight, links out of each switch
        pieces = out + L * 4;                    // pieces[tasks][max_len]: links of a segment, last first
        tasks = kPieceBytes / 4 / max_len;       // at least the 33 segments of one request
        tasks = tasks < kSegTasks ? tasks : kSegTasks;
        in_w = pieces + tasks * max_len * 4;     // in_w[L]: weights of in[]
        region = in_w + L * 2;                   // region[S]
        warps = (region + S + 15) & ~15u;
        // each warp: dist[S] first (the joined visits, max_len of them, later)
        okw = (S + 31) / 32;
        marks = ((S > max_len ? S : max_len) + 3) / 4 * 16;   // marks[okw]: switches listed for the next step
        list = marks + okw * 4;                  // list[2][S]: the frontier and the next one
        per_warp = (list + 2 * S * 2 + 15) & ~15u;
    }
    __host__ __device__ size_t total(uint32_t n) const { return (size_t)warps + (size_t)n * per_warp; }
};
static_assert(kPieceBytes / 4 / PV_MAX_HOP_CAP >= 33, "a request's segments fit one group");

__global__ void __launch_bounds__(1024, 1) sched_segments_kernel(SchedArgs a) {
    extern __shared__ __align__(16) uint8_t s_raw[];
    __shared__ pv_path_req s_req[kSegReqs];
    __shared__ uint4 s_pol[kSegReqs];
    __shared__ uint32_t s_first[kSegReqs + 1], s_st[kSegReqs];
    __shared__ uint8_t s_seg_st[kSegTasks], s_seg_len[kSegTasks];
    __shared__ uint32_t s_next, s_group;
    const uint32_t S = a.S, L = a.in_offs[S];
    const SegmentSmem M(S, L, a.max_len);
    uint32_t *out_offs = reinterpret_cast<uint32_t *>(s_raw), *in_offs = reinterpret_cast<uint32_t *>(s_raw + M.in_offs);
    uint32_t *in = reinterpret_cast<uint32_t *>(s_raw + M.in), *out = reinterpret_cast<uint32_t *>(s_raw + M.out);
    uint16_t *in_w = reinterpret_cast<uint16_t *>(s_raw + M.in_w);
    uint8_t *region = s_raw + M.region;
    const uint32_t t = threadIdx.x, nt = blockDim.x, lane = t & 31, warp = t >> 5, lt = (1u << lane) - 1u;
    uint8_t *mine = s_raw + M.warps + warp * M.per_warp;
    uint32_t *dist = reinterpret_cast<uint32_t *>(mine), *marks = reinterpret_cast<uint32_t *>(mine + M.marks);
    uint16_t *list = reinterpret_cast<uint16_t *>(mine + M.list);
    // the block's links: in-links as loaded, with weights, then out-links
    // counted and placed by source (their order within a switch is free)
    uint32_t *cursor = reinterpret_cast<uint32_t *>(s_raw + M.warps);   // warp 0's distances, free until the barrier below
    for (uint32_t v = t; v <= S; v += nt) in_offs[v] = a.in_offs[v];
    for (uint32_t v = t; v < S; v += nt) {
        cursor[v] = 0;
        region[v] = a.region[v];
    }
    __syncthreads();
    for (uint32_t l = t; l < L; l += nt) {
        const uint32_t x = a.in_links[l];
        in[l] = x;
        in_w[l] = (uint16_t)link_weight(a, x >> 16, (x >> 8) & 0xFFu);
        atomicAdd(&cursor[x >> 16], 1u);
    }
    __syncthreads();
    if (warp == 0) {
        uint32_t run = 0;
        for (uint32_t v0 = 0; v0 < S; v0 += 32) {
            const uint32_t c = v0 + lane < S ? cursor[v0 + lane] : 0u;
            uint32_t incl = c;
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(PV_FULL_MASK, incl, d);
                if (lane >= (uint32_t)d) incl += y;
            }
            if (v0 + lane < S) {
                out_offs[v0 + lane] = run + incl - c;
                cursor[v0 + lane] = run + incl - c;
            }
            run += __shfl_sync(PV_FULL_MASK, incl, 31);
        }
        if (lane == 0) out_offs[S] = run;
    }
    __syncthreads();
    for (uint32_t v = t; v < S; v += nt)
        for (uint32_t l = in_offs[v]; l < in_offs[v + 1]; ++l) out[atomicAdd(&cursor[in[l] >> 16], 1u)] = v << 16 | in_w[l];
    const uint32_t r_end = (uint32_t)(((uint64_t)a.R * (blockIdx.x + 1)) / gridDim.x);
    for (uint32_t r0 = (uint32_t)(((uint64_t)a.R * blockIdx.x) / gridDim.x); r0 < r_end;) {
        __syncthreads();   // the links are placed; the group before is done with the shared state
        // the group: requests from r0 while their segments fit; refused ones have none
        const uint32_t nreq = min(r_end - r0, kSegReqs);
        if (t < nreq) {
            const pv_path_req q = a.req[r0 + t];
            uint4 ph = make_uint4(0, 0, 0, 0);
            if (a.pol_hdr && q.policy < a.num_pol) ph = a.pol_hdr[q.policy];
            auto permitted = [&](uint32_t s) {
                if (s >= S) return false;   // a waypoint of policies loaded for other tables
                bool fine = region[s] < 32 && ((q.allowed_mask >> region[s]) & 1u);
                for (uint32_t i = 0; i < ph.y && fine; ++i) fine = a.pol_sw[ph.x + i] != s;
                return fine;
            };
            uint32_t st = PV_PATH_NOSRC;
            if (q.src_host < a.H && q.dst_host < a.H) {
                bool fine = permitted(a.host_switch[q.src_host]) && permitted(a.host_switch[q.dst_host]);
                for (uint32_t i = 0; i < ph.w && fine; ++i) fine = permitted(a.pol_sw[ph.z + i]);
                st = fine ? PV_PATH_OK : PV_PATH_BLOCKED;
            }
            s_req[t] = q;
            s_pol[t] = ph;
            s_st[t] = st;
            s_first[t + 1] = st == PV_PATH_OK ? ph.w + 1 : 0u;
        }
        __syncthreads();
        if (t == 0) {
            uint32_t g = 0, sum = 0;
            s_first[0] = 0;
            while (g < nreq && sum + s_first[g + 1] <= M.tasks) {
                sum += s_first[g + 1];
                s_first[++g] = sum;
            }
            s_group = g;
            s_next = 0;
        }
        __syncthreads();
        const uint32_t group = s_group, tasks = s_first[group];
        while (true) {
            uint32_t task = 0;
            if (lane == 0) task = atomicAdd(&s_next, 1u);
            task = __shfl_sync(PV_FULL_MASK, task, 0);
            if (task >= tasks) break;
            uint32_t slot = 0, len = group;   // the request with first[slot] <= task < first[slot + 1]
            while (len > 1) {
                const uint32_t half = len >> 1;
                if (s_first[slot + half] <= task) slot += half;
                len -= half;
            }
            const pv_path_req q = s_req[slot];
            const uint4 ph = s_pol[slot];
            const uint32_t i = task - s_first[slot];
            const uint32_t cur = i == 0 ? a.host_switch[q.src_host] : a.pol_sw[ph.z + i - 1];
            const uint32_t tgt = i < ph.w ? a.pol_sw[ph.z + i] : a.host_switch[q.dst_host];
            uint32_t *piece = reinterpret_cast<uint32_t *>(s_raw + M.pieces) + (size_t)task * a.max_len;
            uint32_t st = PV_PATH_OK, k = 0;
            if (tgt != cur) {
                for (uint32_t v = lane; v < S; v += 32) {
                    const uint32_t reg = region[v];
                    dist[v] = reg < 32 && ((q.allowed_mask >> reg) & 1u) ? kInf : 0u;
                }
                __syncwarp();
                for (uint32_t f = lane; f < ph.y; f += 32) {
                    const uint32_t v = a.pol_sw[ph.x + f];
                    if (v < S) dist[v] = 0;
                }
                if (lane == 0) {
                    dist[cur] = 1;
                    list[0] = (uint16_t)cur;
                }
                uint16_t *from = list, *to = list + S;
                for (uint32_t nf = 1; nf;) {
                    for (uint32_t w = lane; w < M.okw; w += 32) marks[w] = 0;
                    __syncwarp();
                    uint32_t nn = 0;
                    for (uint32_t b = 0; b < nf; b += 8) {
                        const uint32_t bound = *(volatile uint32_t *)(dist + tgt);
                        uint32_t du = 0, l = 0, l1 = 0;
                        if (b + (lane >> 2) < nf) {
                            const uint32_t u = from[b + (lane >> 2)];
                            du = *(volatile uint32_t *)(dist + u);
                            l = out_offs[u] + (lane & 3u);
                            l1 = du < bound ? out_offs[u + 1] : 0u;
                        }
                        while (__any_sync(PV_FULL_MASK, l < l1)) {
                            bool push = false;
                            uint32_t v = 0;
                            if (l < l1) {
                                const uint32_t x = out[l], d = du + (x & 0xFFFFu);
                                v = x >> 16;
                                if (d < bound && d < atomicMin(dist + v, d)) {
                                    const uint32_t bit = 1u << (v & 31u);
                                    push = !(atomicOr(&marks[v >> 5], bit) & bit);
                                }
                                l += 4;
                            }
                            const uint32_t m = __ballot_sync(PV_FULL_MASK, push);
                            if (push) to[nn + __popc(m & lt)] = (uint16_t)v;
                            nn += __popc(m);
                        }
                    }
                    __syncwarp();
                    nf = nn;
                    uint16_t *x = from;
                    from = to;
                    to = x;
                }
                if (dist[tgt] == kInf) st = PV_PATH_BLOCKED;
                // canonical walk back from tgt: smallest (u, p) on a shortest path
                for (uint32_t v = tgt; v != cur && st == PV_PATH_OK;) {
                    const uint32_t dv = dist[v], l1 = in_offs[v + 1];
                    uint32_t pick = kInf;
                    for (uint32_t l0 = in_offs[v]; l0 < l1 && pick == kInf; l0 += 32) {
                        const uint32_t l = min(l0 + lane, l1 - 1), x = in[l], du = dist[x >> 16];
                        const uint32_t m = __ballot_sync(PV_FULL_MASK, l0 + lane < l1 && du - 1u < kInf - 1u && du + in_w[l] == dv);
                        if (m) pick = __shfl_sync(PV_FULL_MASK, x, __ffs(m) - 1);
                    }
                    if (pick == kInf) {   // cannot happen once the distances are exact
                        st = PV_PATH_BLOCKED;
                    } else if (k + 1 >= a.max_len) {   // the source's visit and k + 1 more
                        st = PV_PATH_TOO_LONG;
                    } else {
                        // {source port, switch v, its in_port}
                        if (lane == 0) piece[k] = ((pick >> 8) & 0xFFu) << 24 | v << 8 | (pick & 0xFFu);
                        ++k;
                        v = pick >> 16;
                    }
                }
                __syncwarp();   // the distances are rebuilt for the next segment
            }
            if (lane == 0) {
                s_seg_st[task] = (uint8_t)st;
                s_seg_len[task] = (uint8_t)k;
            }
        }
        __syncthreads();
        // a warp per request: its first failing segment decides, else the
        // pieces in order are its visits
        for (uint32_t g = warp; g < group; g += nt >> 5) {
            const uint32_t r = r0 + g, r_tasks = s_first[g + 1] - s_first[g];
            uint32_t *vis = dist, st = s_st[g], n = 1;
            const pv_path_req q = s_req[g];
            if (st == PV_PATH_OK && lane == 0)
                vis[0] = (uint32_t)a.host_switch[q.src_host] << 16 | (uint32_t)a.host_port[q.src_host] << 8;
            for (uint32_t i = 0; i < r_tasks && st == PV_PATH_OK; ++i) {
                const uint32_t task = s_first[g] + i, k = s_seg_len[task];
                st = s_seg_st[task];
                if (st == PV_PATH_OK && n + k > a.max_len) st = PV_PATH_TOO_LONG;
                if (st != PV_PATH_OK) break;
                const uint32_t *piece = reinterpret_cast<const uint32_t *>(s_raw + M.pieces) + (size_t)task * a.max_len;
                for (uint32_t j = lane; j < k; j += 32) {
                    const uint32_t x = piece[k - 1 - j];
                    vis[n + j] = ((x >> 8) & 0xFFFFu) << 16 | (x & 0xFFu) << 8;
                }
                __syncwarp();
                for (uint32_t j = lane; j < k; j += 32) vis[n - 1 + j] |= piece[k - 1 - j] >> 24;   // out port toward the next switch
                __syncwarp();
                n += k;
            }
            __syncwarp();
            if (st == PV_PATH_OK) {
                if (lane == 0) vis[n - 1] |= a.host_port[q.dst_host];
                __syncwarp();
                // a recurring (switch, in_port) cannot be realised by header
                // rules (a single segment is a simple path)
                bool again = false;
                if (r_tasks > 1)
                    for (uint32_t x = lane; x < n; x += 32)
                        for (uint32_t y = x + 1; y < n; ++y) again = again || (vis[x] >> 8) == (vis[y] >> 8);
                if (__any_sync(PV_FULL_MASK, again)) st = PV_PATH_REPEAT;
            }
            for (uint32_t x = lane; x < n && st == PV_PATH_OK; x += 32) a.visits[(size_t)r * a.max_len + x] = vis[x];
            if (lane == 0) {
                a.status[r] = (uint8_t)st;
                a.len[r] = (uint8_t)(st == PV_PATH_OK ? n : 0);
            }
            __syncwarp();
        }
        r0 += group;
    }
}

// Visit i of an OK request becomes, at its switch, the rule {priority,
// in_port, src /32, dst /32, any destination port, output port}, in slot
// r * max_len + i; unused slots get rule_switch 0xFFFF.
__global__ void compile_path_rules_kernel(uint32_t R, const pv_path_req *__restrict__ req,
                                          const uint32_t *__restrict__ host_ip, uint32_t H, uint32_t max_len,
                                          const uint32_t *__restrict__ visits, const uint8_t *__restrict__ len,
                                          const uint8_t *__restrict__ status, uint16_t priority,
                                          pv_rule *__restrict__ rules, uint16_t *__restrict__ rule_switch) {
    const size_t total = (size_t)R * max_len;
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < total; k += (size_t)gridDim.x * blockDim.x) {
        const uint32_t r = (uint32_t)(k / max_len), i = (uint32_t)(k % max_len);
        pv_rule x;
        x.priority = priority;
        x.in_port = 0;
        x.src_ip = x.dst_ip = 0;
        x.src_len = x.dst_len = 0;
        x.dport_lo = 0;
        x.dport_hi = 0xFFFF;
        x.action = PV_DROP;
        uint16_t sw = 0xFFFF;
        const pv_path_req q = req[r];
        if (status[r] == PV_PATH_OK && i < len[r] && q.src_host < H && q.dst_host < H) {
            const uint32_t h = visits[k];
            x.in_port = (uint16_t)((h >> 8) & 0xFFu);
            x.src_ip = host_ip[q.src_host];
            x.src_len = 32;
            x.dst_ip = host_ip[q.dst_host];
            x.dst_len = 32;
            x.action = (uint16_t)(h & 0xFFu);
            sw = (uint16_t)(h >> 16);
        } else {
            x.priority = 0;
        }
        rules[k] = x;
        rule_switch[k] = sw;
    }
}

}  // namespace

extern "C" int pv_schedule_paths(pv_ctx *ctx, uint32_t num_requests, const pv_path_req *d_requests,
                                 const uint16_t *d_link_weights, uint32_t max_len, uint32_t *d_visits,
                                 uint8_t *d_len, uint8_t *d_status, pv_stream stream) {
    if (!ctx) return PV_EINVAL;
    const pv_table_state &t = ctx->tb;
    if (!t.loaded) return pv_fail(ctx, PV_ESTATE, "pv_schedule_paths: no flow tables loaded");
    if (max_len == 0 || max_len > PV_MAX_HOP_CAP) return pv_fail(ctx, PV_EINVAL, "max_len must be 1..255");
    if (t.num_switches > kSchedMaxSwitches)
        return pv_fail(ctx, PV_EINVAL, "pv_schedule_paths: more than %u switches", kSchedMaxSwitches);
    if (num_requests == 0) return PV_OK;
    if (!d_requests || !d_visits || !d_len || !d_status)
        return pv_fail(ctx, PV_EINVAL, "pv_schedule_paths: NULL device pointer");
    SchedArgs a;
    a.S = t.num_switches;
    a.H = t.num_hosts;
    a.region = t.d_region;
    a.port_offs = t.d_port_offs;
    a.host_switch = t.d_host_switch;
    a.host_port = t.d_host_port;
    a.in_offs = t.d_in_offs;
    a.in_links = t.d_in_links;
    a.weights = d_link_weights;
    a.pol_hdr = ctx->pol.loaded ? ctx->pol.d_hdr : nullptr;
    a.pol_sw = ctx->pol.loaded ? ctx->pol.d_sw : nullptr;
    a.num_pol = ctx->pol.loaded ? ctx->pol.num : 0;
    a.req = d_requests;
    a.R = num_requests;
    a.max_len = max_len;
    a.visits = d_visits;
    a.len = d_len;
    a.status = d_status;
    const size_t base_smem = ((size_t)a.S + (a.S + 31) / 32 + 2 * (size_t)max_len) * 4;
    // the links (with weights) and the predecessors staged when they fit
    const uint32_t L = t.num_links;
    const size_t staged_smem = base_smem + ((size_t)a.S + (size_t)a.S + 1 + L) * 4 + ((size_t)L * 2 + 15) / 16 * 16;
    // 0 automatic: a warp per segment when at least four warps' state fits,
    // else a block per request; 1 block per request, links from global memory;
    // 2 staged
    const int force = ctx->opt_sched_kernel;
    const SegmentSmem W(a.S, L, max_len);
    const size_t smem_cap = ctx->max_smem_optin - 8 * 1024;   // less the kernel's static arrays
    const uint32_t warps = W.warps < smem_cap ? (uint32_t)std::min<size_t>(32, (smem_cap - W.warps) / W.per_warp) : 0u;
    const bool by_warp = force == 0 && warps >= 4;
    const bool staged_fits = staged_smem <= std::min<size_t>(96 * 1024, ctx->max_smem_optin - 1024);
    if (force == 2 && !staged_fits)
        return pv_fail(ctx, PV_EINVAL, "pv_schedule_paths: the staged links do not fit shared memory");
    const bool staged = force == 2 || (force == 0 && staged_fits);
    const size_t smem = by_warp ? W.total(warps) : staged ? staged_smem : base_smem;
    const void *fn = by_warp  ? (const void *)sched_segments_kernel
                     : staged ? (const void *)sched_paths_kernel<true>
                              : (const void *)sched_paths_kernel<false>;
    if (int rc = pv_smem_limit(ctx, fn, "path scheduler shared memory")) return rc;
    const int threads = by_warp ? (int)warps * 32 : kSchedThreads;
    const uint32_t resident = (uint32_t)std::max(pv_blocks_per_sm(ctx, fn, threads, smem), 1) * ctx->num_sms;
    const uint32_t grid = std::min<uint32_t>(num_requests, resident);
    pv_use_begin(ctx, (cudaStream_t)stream);
    const int pr = pv_prof_start(ctx, (cudaStream_t)stream, PV_K_SCHEDULE);
    if (by_warp)
        sched_segments_kernel<<<grid, threads, smem, (cudaStream_t)stream>>>(a);
    else if (staged)
        sched_paths_kernel<true><<<grid, threads, smem, (cudaStream_t)stream>>>(a);
    else
        sched_paths_kernel<false><<<grid, threads, smem, (cudaStream_t)stream>>>(a);
    pv_prof_stop(ctx, (cudaStream_t)stream, pr, 1);
    pv_mark_use(ctx, (cudaStream_t)stream);
    return pv_check_launch(ctx, "path scheduler kernel");
}

extern "C" int pv_compile_path_rules(pv_ctx *ctx, uint32_t num_requests, const pv_path_req *d_requests,
                                     uint32_t max_len, const uint32_t *d_visits, const uint8_t *d_len,
                                     const uint8_t *d_status, uint16_t priority, pv_rule *d_rules,
                                     uint16_t *d_rule_switch, pv_stream stream) {
    if (!ctx) return PV_EINVAL;
    const pv_table_state &t = ctx->tb;
    if (!t.loaded) return pv_fail(ctx, PV_ESTATE, "pv_compile_path_rules: no flow tables loaded");
    if (max_len == 0 || max_len > PV_MAX_HOP_CAP) return pv_fail(ctx, PV_EINVAL, "max_len must be 1..255");
    if (num_requests == 0) return PV_OK;
    if (!d_requests || !d_visits || !d_len || !d_status || !d_rules || !d_rule_switch)
        return pv_fail(ctx, PV_EINVAL, "pv_compile_path_rules: NULL device pointer");
    const size_t total = (size_t)num_requests * max_len;
    const uint32_t grid = (uint32_t)std::min<size_t>((total + 255) / 256, (size_t)ctx->num_sms * 8);
    pv_use_begin(ctx, (cudaStream_t)stream);
    const int pr = pv_prof_start(ctx, (cudaStream_t)stream, PV_K_SCHEDULE);
    compile_path_rules_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(num_requests, d_requests, t.d_host_ip,
                                                                      t.num_hosts, max_len, d_visits, d_len,
                                                                      d_status, priority, d_rules, d_rule_switch);
    pv_prof_stop(ctx, (cudaStream_t)stream, pr, 1);
    pv_mark_use(ctx, (cudaStream_t)stream);
    return pv_check_launch(ctx, "compile_path_rules_kernel");
}

extern "C" int pv_install_path_rules(pv_ctx *ctx, uint32_t num_slots, const pv_rule *d_rules,
                                     const uint16_t *d_rule_switch) {
    if (!ctx) return PV_EINVAL;
    if (!ctx->tb.loaded) return pv_fail(ctx, PV_ESTATE, "pv_install_path_rules: no flow tables loaded");
    if (num_slots == 0) return PV_OK;
    if (!d_rules || !d_rule_switch) return pv_fail(ctx, PV_EINVAL, "pv_install_path_rules: NULL device pointer");
    std::vector<pv_rule> add(num_slots);
    std::vector<uint16_t> sw(num_slots);
    // the compiled rules come from an evaluation call: the load stream waits
    // for it, then reads them and the loaded rules
    if (int rc0 = pv_load_begin(ctx)) return rc0;
    cudaStream_t ls = ctx->load_stream;
    PV_TRY_CUDA(ctx, cudaStreamWaitEvent(ls, ctx->last_use, 0), "pv_install_path_rules");
    const pv_table_host h = ctx->tbh;   // copy: the reload below replaces ctx->tbh
    const uint32_t S = (uint32_t)h.region.size();
    std::vector<pv_rule> base(h.rule_offs[S]);
    PV_TRY_CUDA(ctx, cudaMemcpyAsync(add.data(), d_rules, (size_t)num_slots * sizeof(pv_rule),
                                     cudaMemcpyDeviceToHost, ls),
                "path rules download");
    PV_TRY_CUDA(ctx, cudaMemcpyAsync(sw.data(), d_rule_switch, (size_t)num_slots * 2, cudaMemcpyDeviceToHost, ls),
                "path rule switches download");
    if (!base.empty())
        PV_TRY_CUDA(ctx, cudaMemcpyAsync(base.data(), ctx->tb.d_raw, base.size() * sizeof(pv_rule),
                                         cudaMemcpyDeviceToHost, ls),
                    "loaded rules download");
    PV_TRY_CUDA(ctx, cudaStreamSynchronize(ls), "pv_install_path_rules");
    std::vector<uint32_t> count(S, 0);
    for (uint32_t k = 0; k < num_slots; ++k)
        if (sw[k] < S) ++count[sw[k]];
    std::vector<uint32_t> offs(S + 1, 0);
    for (uint32_t s = 0; s < S; ++s) offs[s + 1] = offs[s] + count[s] + (h.rule_offs[s + 1] - h.rule_offs[s]);
    std::vector<pv_rule> rules(offs[S]);
    std::vector<uint32_t> cur(offs.begin(), offs.end() - 1);
    for (uint32_t k = 0; k < num_slots; ++k)   // new rules first, in slot order: they win priority ties
        if (sw[k] < S) rules[cur[sw[k]]++] = add[k];
    for (uint32_t s = 0; s < S; ++s)
        for (uint32_t i = h.rule_offs[s]; i < h.rule_offs[s + 1]; ++i) rules[cur[s]++] = base[i];
    return pv_load_flow_tables(ctx, S, offs.data(), rules.data(), h.region.data(), h.port_offs.data(),
                               h.port_peer.data(), (uint32_t)h.host_ip.size(), h.host_switch.data(),
                               h.host_port.data(), h.host_ip.data());
}
