// dm_ring.cu -- dual consistent-hash rings with virtual nodes (Sec. 3.4,
// App. A.1.3; d rings for the d-candidate path of App. A.8).  Each live id
// owns V nodes per ring at
//   vpos_f(id, v) = fmix64(splitmix_step((id << 32) | v) ^ S_vf),
// kept sorted by (position, id, v).  Adding an id inserts its V nodes,
// removing it deletes them; all other nodes keep their relative order, so
// only keys on the changed arcs remap.
//
// An update is two kernels: the id's V nodes are generated and sorted (a CTA
// per ring, beside one that sets the instance's state and the next-live
// list), then every surviving old node moves by the number of id nodes before
// it and every new node lands at (its rank among the new nodes + number of
// old nodes before it), each node writing the search-tree entries it becomes
// in passing.  Adding an id first resets its index and logs in a kernel that
// also takes the pointers, so nothing is copied from the host.
// Latency-bound.  256 ids x 1,024 virtual nodes, a removal, an addition and a
// lookup, GB300: 196 us before, 64 us so (sorting in global memory,
// a binary search per node, separate kernels for tree, state and next-live
// list, seven pointer copies and two waits per addition).
#include <algorithm>

#include "dm_internal.cuh"

namespace dm {

__device__ __forceinline__ bool vless(uint64_t pa, uint32_t ia, uint32_t va, uint64_t pb, uint32_t ib,
                                      uint32_t vb) {
    if (pa != pb) return pa < pb;
    if (ia != ib) return ia < ib;
    return va < vb;
}

// Vnode seed of ring f.
__device__ __forceinline__ uint64_t ring_seed(const DevState &d, int f) {
    return f == 0 ? d.Sv1 : f == 1 ? d.Sv2 : d.Svx[f - 2];
}

// A new state of instance id, and next_live[i] = the next live id after i in
// ascending order, cyclically (i itself when there is no other).  One CTA.
__device__ void state_role(const DevState &d, uint32_t id, uint8_t state) {
    __shared__ uint32_t s_live[kMaxInstances / 32];
    const uint32_t words = (d.M + 31) / 32;
    for (uint32_t w = threadIdx.x >> 5; w < words; w += blockDim.x >> 5) {
        const uint32_t i = w * 32 + (threadIdx.x & 31);
        const bool live = i == id ? state == 1 : i < d.M && d.inst_state[i] == 1;
        const uint32_t b = __ballot_sync(0xffffffffu, live);
        if ((threadIdx.x & 31) == 0) s_live[w] = b;
    }
    if (threadIdx.x == 0 && id < d.M) d.inst_state[id] = state;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < d.M; i += blockDim.x) {
        uint32_t nx = i, w = i / 32;
        uint32_t b = s_live[w] & ~((2u << (i & 31)) - 1u);   // ids above i in its word
        for (uint32_t k = 0;; ) {
            if (b) {
                nx = w * 32 + __ffs(b) - 1;
                break;
            }
            if (++k > words) break;   // its own word again, once, for the ids below it
            w = w + 1 == words ? 0 : w + 1;
            b = s_live[w];
        }
        d.next_live[i] = nx;
    }
}

// Sort the P = 2^k entries by (position, vidx): all belong to one id.
__device__ __forceinline__ void sort_nodes(uint64_t *pos, uint32_t *vi, uint32_t P) {
    for (uint32_t k = 2; k <= P; k <<= 1) {
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t q = threadIdx.x; q < P / 2; q += blockDim.x) {
                const uint32_t x = 2 * q - (q & (j - 1)), y = x + j;
                const uint64_t px = pos[x], py = pos[y];
                const uint32_t vx = vi[x], vy = vi[y];
                const bool gt = py < px || (py == px && vy < vx);   // x > y
                if (gt == ((x & k) == 0)) {
                    pos[x] = py;
                    pos[y] = px;
                    vi[x] = vy;
                    vi[y] = vx;
                }
            }
            __syncthreads();
        }
    }
}

// Generate and sort the V nodes of `id` for every ring (one CTA per ring, in
// shared memory when P entries fit it), and one CTA for the state.
constexpr uint32_t kSortSmem = 8192;   // entries sorted in shared memory (96 KB)
__global__ void __launch_bounds__(1024) k_gen_sort(DevState d, uint32_t id, uint64_t *spos, uint32_t *svidx,
                                                   uint32_t P, uint8_t state) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem[];
    if (blockIdx.x == d.nrings) {
        state_role(d, id, state);
        return;
    }
    const int f = blockIdx.x;
    const uint64_t Sv = ring_seed(d, f);
    uint64_t *const gpos = spos + uint64_t(f) * P;
    uint32_t *const gvi = svidx + uint64_t(f) * P;
    const bool in_smem = P <= kSortSmem;
    uint64_t *const pos = in_smem ? reinterpret_cast<uint64_t *>(smem) : gpos;
    uint32_t *const vi = in_smem ? reinterpret_cast<uint32_t *>(smem + size_t(P) * 8) : gvi;
    for (uint32_t v = threadIdx.x; v < P; v += blockDim.x) {
        pos[v] = v < d.V ? vnode_pos(Sv, id, v) : ~0ull;
        vi[v] = v < d.V ? v : 0xFFFFFFFFu;
    }
    __syncthreads();
    sort_nodes(pos, vi, P);
    if (in_smem)
        for (uint32_t v = threadIdx.x; v < d.V; v += blockDim.x) {
            gpos[v] = pos[v];
            gvi[v] = vi[v];
        }
}

// Entries of a sorted node list that precede (p, o, v): a 32-way search, the
// whole warp (owner null: every entry belongs to `id`).
__device__ __forceinline__ uint32_t count_before(const uint64_t *pos, const uint32_t *owner, const uint32_t *vidx,
                                                 uint32_t n, uint32_t id, uint64_t p, uint32_t o, uint32_t v,
                                                 int lane) {
    uint32_t lo = 0, len = n;   // the count lies in [lo, lo + len]
    while (len > 0) {
        const uint32_t step = (len + 31) / 32, x = lo + lane * step;
        const bool in = lane * step < len;
        bool less = false;
        if (in) {
            const uint64_t q = pos[x];
            less = q != p ? q < p : vless(q, owner ? owner[x] : id, vidx[x], p, o, v);
        }
        const uint32_t c = __popc(__ballot_sync(0xffffffffu, less));   // a prefix of the lanes
        if (c == 0) return lo;
        const uint32_t skip = (c - 1) * step + 1;   // entry lo + (c - 1) step precedes it
        len = min(step - 1, len - skip);
        lo += skip;
    }
    return lo;
}

// Destination buffers of every ring, and the search-tree levels of the new
// length.
struct RingSet {
    Ring r[kMaxD];
    uint32_t nlev;
    uint64_t lev_off[kMaxLevels];
};

// Entry k of a new ring: the node, and the tree entries with its position
// (level l entry i = vpos[i * 32^l]).
__device__ __forceinline__ void put_node(const Ring &dst, const RingSet &rs, uint32_t k, uint64_t p, uint32_t o,
                                         uint32_t v) {
    dst.vpos[k] = p;
    dst.owner[k] = o;
    dst.vidx[k] = v;
    uint32_t x = k;
    for (uint32_t l = 1; l < rs.nlev && (x & 31) == 0; ++l) {
        x >>= 5;
        dst.tree[rs.lev_off[l] + x] = p;
    }
}

// Every ring (blockIdx.y): a warp per 32 old nodes, and (kAdd) per new node.
// The id nodes before a warp's first old node are counted by a search, those
// before the others by going on from there (V of R nodes are the id's: a few
// steps at most).
template <bool kAdd>
__global__ void __launch_bounds__(256) k_merge(DevState d, uint32_t id, const uint64_t *spos, const uint32_t *svidx,
                                               uint32_t P, const __grid_constant__ RingSet rs) {
    pdl_enter();
    const int f = blockIdx.y, lane = threadIdx.x & 31;
    const Ring src = d.ring[f];
    const Ring dst = rs.r[f];
    const uint64_t *npos = spos + uint64_t(f) * P;
    const uint32_t *nvi = svidx + uint64_t(f) * P;
    const uint32_t R = d.R, V = d.V, old_warps = (R + 31) / 32;
    const uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w < old_warps) {
        const uint32_t t = w * 32 + lane;
        const bool valid = t < R;
        const uint64_t p = valid ? src.vpos[t] : 0;
        const uint32_t o = valid ? src.owner[t] : 0, v = valid ? src.vidx[t] : 0;
        uint32_t c = count_before(npos, nullptr, nvi, V, id, shfl_u64(p, 0), __shfl_sync(0xffffffffu, o, 0),
                                  __shfl_sync(0xffffffffu, v, 0), lane);
        if (!valid || (!kAdd && o == id)) return;
        while (c < V && vless(npos[c], id, nvi[c], p, o, v)) ++c;
        put_node(dst, rs, kAdd ? t + c : t - c, p, o, v);
    } else if (kAdd && w < old_warps + V) {
        const uint32_t j = w - old_warps;
        const uint64_t p = npos[j];
        const uint32_t v = nvi[j];
        const uint32_t k = j + count_before(src.vpos, src.owner, src.vidx, R, id, p, id, v, lane);
        if (lane == 0) put_node(dst, rs, k, p, id, v);
    }
}

cudaError_t launch_ring_update(DevState &d, const DevState &next, uint32_t id, bool add, uint64_t *scratch_pos,
                               uint32_t *scratch_vidx, cudaStream_t st) {
    uint32_t P = 1;
    while (P < d.V) P <<= 1;
    const size_t smem = P <= kSortSmem ? size_t(P) * 12 : 0;
    static SmemOptIn opt;
    DM_TRY(opt_in_smem(opt, smem, k_gen_sort));   // (state_role's words come on top: past 48 KB from 4,096 entries on)
    DM_TRY(launch_pdl(k_gen_sort, d.nrings + 1, 1024, smem, st, d, id, scratch_pos, scratch_vidx, P,
                      uint8_t(add ? 1 : 2)));
    RingSet rs{};
    for (uint32_t f = 0; f < d.nrings; ++f) rs.r[f] = next.ring[f];
    rs.nlev = next.nlev;
    std::copy(next.lev_off, next.lev_off + kMaxLevels, rs.lev_off);
    const uint32_t warps = (d.R + 31) / 32 + (add ? d.V : 0);
    if (warps > 0)
        DM_TRY(launch_pdl(add ? k_merge<true> : k_merge<false>, dim3((warps + 7) / 8, d.nrings), 256, 0, st, d, id,
                          static_cast<const uint64_t *>(scratch_pos), static_cast<const uint32_t *>(scratch_vidx), P,
                          rs));
    return cudaGetLastError();
}

// next_live of a handle without instances.
__global__ void k_next_live(DevState d) {
    pdl_enter();
    state_role(d, 0xFFFFFFFFu, 0);
}

cudaError_t launch_next_live(const DevState &d, cudaStream_t st) { return launch_pdl(k_next_live, 1, 256, 0, st, d); }

// A (re-)added instance starts with an empty index, logs and queue.  first:
// its buffers, and the spare index buffer that joins the pool with it (or
// null); a re-added id keeps whichever index buffer it holds now and its logs
// start in the buffers first allocated.
__global__ void __launch_bounds__(256) k_reset_instance(DevState d, uint32_t id, InstanceBuffers b) {
    pdl_enter();
    Slot *const t = b.table ? b.table : d.table[id];
    const uint64_t tid = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x, nt = uint64_t(gridDim.x) * blockDim.x;
    const uint4 zero = make_uint4(0, 0, 0, 0);
    for (uint64_t x = tid; x < d.S; x += nt) reinterpret_cast<uint4 *>(t)[x] = zero;
    for (uint64_t x = tid; x < d.logcap / 16; x += nt) {   // logcap is a power of two >= 1,024
        reinterpret_cast<uint4 *>(b.stale[0])[x] = zero;
        reinterpret_cast<uint4 *>(b.stale[1])[x] = zero;
    }
    if (tid == 0) {
        if (b.table) d.table[id] = b.table;
        if (b.spare) d.pool[d.pool_n] = b.spare;
        d.logbuf[id] = b.log[0];
        d.logbuf_alt[id] = b.log[1];
        d.stale[id] = b.stale[0];
        d.stale_alt[id] = b.stale[1];
        d.loghome[id] = b.home[0];
        d.loghome_alt[id] = b.home[1];
        d.log_front[id] = 0;
        d.log_tail[id] = 0;
        d.live[id] = 0;
        d.used[id] = 0;
        d.W[id] = 0;
        d.q_head[id] = 0;
        d.q_tail[id] = 0;
    }
}

cudaError_t launch_reset_instance(const DevState &d, uint32_t id, const InstanceBuffers &b, cudaStream_t st) {
    const uint64_t want = (d.S + d.logcap / 16 + 255) / 256;
    const unsigned grid = (unsigned)std::min<uint64_t>(want, 8ull * sm_count());
    return launch_pdl(k_reset_instance, grid, 256, 0, st, d, id, b);
}

}  // namespace dm
