// Front end of the k-clique pipeline on the device: input validation,
// Pre-Core (Algorithm 3), Pre-List (Algorithm 4), the two orientations
// (degree ordering of Section VI-B, degeneracy ordering of Algorithm 6) and
// the out-neighbour CSR of the DAG, plus the root list the listing kernels
// consume.  Most passes stream the CSR once with warp-per-vertex row scans and
// coalesced loads; the peel is a chain of rounds, bound by the latency of each.
#include <algorithm>
#include <mutex>

#include "kcl_internal.cuh"

namespace kcl {

namespace {

constexpr int kBlock = 256;

inline int grid_for(uint64_t items, int per_block, int num_sms, int per_sm = 16) {
    uint64_t g = (items + per_block - 1) / per_block;
    uint64_t cap = (uint64_t)num_sms * per_sm;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

__device__ __forceinline__ uint32_t warp_global() {
    return (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
}
__device__ __forceinline__ uint32_t warps_total() { return (gridDim.x * blockDim.x) >> 5; }

__device__ __forceinline__ uint32_t block_excl_scan(uint32_t x, uint32_t *smem, uint32_t *total) {
    const unsigned lane = lane_id(), wid = threadIdx.x >> 5;
    uint32_t v = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= (unsigned)o) v += y;
    }
    if (lane == 31) smem[wid] = v;
    __syncthreads();
    if (wid == 0) {
        uint32_t s = lane < (blockDim.x >> 5) ? smem[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= (unsigned)o) s += y;
        }
        smem[lane] = s;
    }
    __syncthreads();
    uint32_t warp_prefix = wid ? smem[wid - 1] : 0;
    *total = smem[(blockDim.x >> 5) - 1];
    __syncthreads();
    return warp_prefix + v - x;
}

// ----------------------------------------------------------- validation
// Row u: strictly ascending, ids < n, no self-loop, and every v in row u has
// u in row v (binary search).  Also records the maximum degree.  A warp takes a
// row; the rest of a row beyond kLongRow entries is left to the whole block, and
// a warp keeps its findings to itself until the end (500k-vertex R-MAT graph:
// 3.28 -> 0.85 ms; a 10,000-vertex graph with a hub 61 -> 45 us).
constexpr uint32_t kLongRow = 512, kLongRows = 64;

__device__ __forceinline__ bool bad_entry(uint32_t n, uint64_t nnz, const uint64_t *__restrict__ rp,
                                          const uint32_t *__restrict__ col, uint32_t u, uint64_t b, uint64_t i) {
    const uint32_t v = col[i];
    if (v >= n || v == u) return true;
    const bool bad = i > b && col[i - 1] >= v;
    uint64_t lo = rp[v], hi = rp[v + 1];  // symmetric: u must be in row v
    if (hi < lo || hi > nnz) return true;
    while (lo < hi) {
        const uint64_t mid = lo + ((hi - lo) >> 1);
        const uint32_t x = col[mid];
        if (x == u) return bad;
        if (x < u) lo = mid + 1; else hi = mid;
    }
    return true;
}

__global__ void k_validate(uint32_t n, uint64_t nnz, const uint64_t *__restrict__ rp,
                           const uint32_t *__restrict__ col, DevResult *res) {
    __shared__ uint32_t rows[kLongRows];
    __shared__ unsigned nlong;
    if (threadIdx.x == 0) nlong = 0;
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (rp[0] != 0 || rp[n] != nnz) atomicOr(&res->status, DEV_ERR_INVALID_GRAPH);
    }
    const unsigned lane = lane_id();
    bool bad = false;
    uint32_t most = 0;
    for (uint32_t u = warp_global(); u < n; u += warps_total()) {
        uint64_t b = rp[u], e = rp[u + 1];
        if (e < b || e > nnz || e - b > 0xFFFFFFFFull) {
            bad = true;
            continue;
        }
        most = max(most, (uint32_t)(e - b));
        uint64_t stop = e;
        if (e - b > 2 * kLongRow) {
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&nlong, 1u);
            at = __shfl_sync(0xffffffffu, at, 0);
            if (at < kLongRows) {
                if (lane == 0) rows[at] = u;
                stop = b + kLongRow;
            }
        }
        for (uint64_t i = b + lane; i < stop; i += 32) bad |= bad_entry(n, nnz, rp, col, u, b, i);
    }
    __syncthreads();
    const unsigned k = min(nlong, kLongRows);
    for (unsigned j = 0; j < k; j++) {
        const uint32_t u = rows[j];
        const uint64_t b = rp[u], e = rp[u + 1];
        for (uint64_t i = b + kLongRow + threadIdx.x; i < e; i += blockDim.x) bad |= bad_entry(n, nnz, rp, col, u, b, i);
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&res->status, DEV_ERR_INVALID_GRAPH);
    if (lane == 0 && most) atomicMax(&res->max_outdeg, most);
}

// ------------------------------------------------------------- Pre-Core
// One warp's lanes append to a list: the position of this lane's entry.
__device__ __forceinline__ uint32_t warp_append(unsigned m, unsigned *count) {
    const unsigned lane = lane_id();
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(count, (unsigned)__popc(m));
    return __shfl_sync(0xffffffffu, base, 0) + __popc(m & ((1u << lane) - 1u));
}

// Algorithm 3, frontier form: the first frontier is every vertex of degree
// < k-1; each round, every vertex of the frontier lowers the degree of its
// neighbours, and a neighbour whose degree falls from k-1 to k-2 joins the next
// one (exactly one thread sees that transition; a vertex that left has fallen
// below its threshold, so nobody sees it again).  Vertices leave through one list,
// a round's frontier being a range of it.
// thr = k-1, or per vertex kmap[v] - 1 when a k map is given (batches of
// graphs with different k).
// Launches are ordinary ones and no block waits for another.  In one cooperative
// launch of co-resident blocks Pre-Core had to wait for room on every SM at once:
// beside a k = 9 call on another stream a k = 5 degree count of the 131k-vertex R-MAT
// graph took as long as that call (2.2 s), and takes 4.2 ms this way.  Short rounds
// would cost a launch each; instead a launch's last block to finish runs the rounds
// that follow while they have at most kPreTail vertices, and leaves wider ones to
// the next launch (k = 5 count of a 2,000-vertex graph: 214 -> 206 us; 100,000
// rounds along a path 202 -> 60 ms; 200 rounds of 1,600 vertices 1.9 ms as launches,
// 6.2 when the last block took up to 2,048, 1.8 in the cooperative launch).
constexpr uint32_t kPreTail = 512;
constexpr int kPreThreads = 1024;

__global__ void k_precore_init(uint32_t n, const uint64_t *__restrict__ rp, uint32_t thr,
                               const uint8_t *__restrict__ kmap, uint8_t *alive, uint32_t *cdeg,
                               uint32_t *list, DevResult *res) {
    const unsigned lane = lane_id();
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    for (uint32_t v0 = tid - lane; v0 < n; v0 += nth) {  // warp-uniform trip count
        const uint32_t v = v0 + lane;
        bool out = false;
        if (v < n) {
            const uint32_t d = (uint32_t)(rp[v + 1] - rp[v]);
            cdeg[v] = d;
            out = d < (kmap ? kmap[v] - 1u : thr);
            alive[v] = out ? 0 : 1;
        }
        const unsigned m = __ballot_sync(0xffffffffu, out);
        if (m) {
            const uint32_t at = warp_append(m, &res->pre_nin);
            if (out) list[at] = v;
        }
    }
}

struct PreArgs {
    const uint64_t *rp;
    const uint32_t *col;
    uint32_t thr;
    const uint8_t *kmap;
    uint8_t *alive;
    uint32_t *cdeg;
    uint32_t *list;  // every vertex that left, in the order of the rounds
    DevResult *res;
};

// Z entries a lane (x, x + 32, ... below e): their vertices lose a degree and may
// leave.
template <int Z>
__device__ __forceinline__ void precore_entries(const PreArgs &a, uint64_t x, uint64_t e, uint32_t at,
                                                unsigned *next) {
    uint32_t w[Z];
    bool out[Z];
#pragma unroll
    for (int z = 0; z < Z; z++) w[z] = x + 32 * z < e ? a.col[x + 32 * z] : 0xFFFFFFFFu;
#pragma unroll
    for (int z = 0; z < Z; z++) {
        const uint32_t t = w[z] == 0xFFFFFFFFu ? 0u : a.kmap ? a.kmap[w[z]] - 1u : a.thr;
        out[z] = t > 0 && atomicSub(&a.cdeg[w[z]], 1u) == t;  // fell from k-1 to k-2
    }
#pragma unroll
    for (int z = 0; z < Z; z++) {
        const unsigned m = __ballot_sync(0xffffffffu, out[z]);
        if (m) {
            const uint32_t i = warp_append(m, next);
            if (out[z]) {
                a.alive[w[z]] = 0;
                a.list[at + i] = w[z];
            }
        }
    }
}

// The round of list[lo, lo + nin) by W warps, this one being number gw; the next
// round is appended behind it.  Most rows are shorter than k: 8 lanes a row, and
// the warp together, four entries a lane, for rows beyond 64 entries (a hub's
// 1M entries 17 -> 13 ms).
__device__ void precore_round(const PreArgs &a, uint32_t lo, uint32_t nin, unsigned *next, uint32_t gw, uint32_t W) {
    const unsigned lane = lane_id();
    const uint32_t at = lo + nin;
    for (uint32_t i0 = gw * 4; i0 < nin; i0 += W * 4) {
        const uint32_t i = i0 + (lane >> 3);
        uint64_t b = 0, e = 0;
        if (i < nin) {
            const uint32_t v = __ldcg(&a.list[lo + i]);
            b = a.rp[v];
            e = a.rp[v + 1];
        }
        const bool big = e - b > 64;
        const uint32_t most = __reduce_max_sync(0xffffffffu, big ? 0u : (uint32_t)(e - b));
        for (uint32_t x = lane & 7u; x - (lane & 7u) < most; x += 8)
            precore_entries<1>(a, b + x, big ? 0ull : e, at, next);
        for (unsigned todo = __ballot_sync(0xffffffffu, big && (lane & 7u) == 0); todo; todo &= todo - 1) {
            const int j = __ffs(todo) - 1;
            const uint64_t rb = __shfl_sync(0xffffffffu, b, j), re = __shfl_sync(0xffffffffu, e, j);
            for (uint64_t x = rb; x < re; x += 128) precore_entries<4>(a, x + lane, re, at, next);
        }
    }
}

__global__ void __launch_bounds__(kPreThreads, 2) k_precore_round(const PreArgs a) {
    __shared__ unsigned next_s, last_s;
    // changed only by the last block, when every block has read them
    uint32_t lo = *(volatile unsigned *)&a.res->pre_lo, nin = *(volatile unsigned *)&a.res->pre_nin;
    if (nin == 0) return;
    const uint32_t W = blockDim.x >> 5, warp = threadIdx.x >> 5;
    precore_round(a, lo, nin, &a.res->pre_next, blockIdx.x * W + warp, gridDim.x * W);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last_s = atomicAdd(&a.res->pre_finished, 1u) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last_s) return;
    lo += nin;
    nin = *(volatile unsigned *)&a.res->pre_next;
    while (nin && nin <= kPreTail) {
        __syncthreads();
        if (threadIdx.x == 0) next_s = 0;
        __syncthreads();
        precore_round(a, lo, nin, &next_s, warp, W);
        __syncthreads();
        lo += nin;
        nin = next_s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a.res->pre_lo = lo;
        a.res->pre_nin = nin;
        a.res->pre_next = 0;
        a.res->pre_finished = 0;
    }
}

// ------------------------------------------------------------- Pre-List
// Clique components of the alive subgraph without forming all components.
// Let r(v) be the smallest id in v's closed alive neighbourhood N[v].  v passes
// when every x in N[v] has r(x) = r(v) and the same alive degree as v.  The
// component of r is a clique iff r(r) = r and all of N[r] pass: then everything
// next to N[r] is next to r (no vertex outside N[r] is reachable), and each of
// the d + 1 vertices of N[r] has degree d.  Conversely the members of a clique
// component all pass.  Almost every vertex fails at once, at the degree of r(v)
// or in the first 32 entries of its row, where union-find over all edges read
// the whole graph with random parent chases (5.1 ms on the 1M-vertex R-MAT
// graph, 0.05 ms here).  parent[v] = r(v).
__global__ void k_pl_min(uint32_t n, const uint64_t *__restrict__ rp, const uint32_t *__restrict__ col,
                         const uint8_t *__restrict__ alive, uint32_t *parent, uint32_t *comp_n,
                         uint32_t *comp_flag, uint32_t per_warp) {
    const unsigned lane = lane_id();
    for (uint32_t v0 = warp_global() * per_warp; v0 < n; v0 += warps_total() * per_warp) {
        const uint32_t v = v0 + lane;
        const bool mine = lane < per_warp && v < n;
        uint32_t r = v;
        bool more = false;
        uint64_t x = 0, e = 0;
        if (mine) {
            comp_n[v] = 0;
            comp_flag[v] = 0;
            if (alive[v]) {
                x = rp[v];
                e = rp[v + 1];
                more = x < e;
                for (int i = 0; i < 4 && more; i++, x++) {  // rows ascend: the first alive id decides
                    const uint32_t w = x < e ? col[x] : 0xFFFFFFFFu;
                    if (w >= v) more = false;
                    else if (alive[w]) { r = w; more = false; }
                }
                more = more && x < e;
            }
        }
        // rows with a long dead prefix: the whole warp, 32 entries at a time
        for (unsigned todo = __ballot_sync(0xffffffffu, more); todo; todo &= todo - 1) {
            const int j = __ffs(todo) - 1;
            const uint32_t u = v0 + j;
            uint64_t y = __shfl_sync(0xffffffffu, x, j);
            const uint64_t ye = __shfl_sync(0xffffffffu, e, j);
            uint32_t got = u;
            for (; y < ye; y += 32) {
                const uint32_t w = y + lane < ye ? col[y + lane] : 0xFFFFFFFFu;
                const unsigned m = __ballot_sync(0xffffffffu, w < u && alive[w]);
                if (m) {
                    got = __shfl_sync(0xffffffffu, w, __ffs(m) - 1);
                    break;
                }
                if (__any_sync(0xffffffffu, w >= u)) break;
            }
            if ((int)lane == j) r = got;
        }
        if (mine) parent[v] = r;
    }
}

// Passing vertices, counted at r(v): a thread settles most vertices at r(v)'s
// own degree and minimum, its warp walks the rows of the others.
__global__ void k_pl_pass(uint32_t n, const uint64_t *__restrict__ rp, const uint32_t *__restrict__ col,
                          const uint8_t *__restrict__ alive, const uint32_t *__restrict__ cdeg,
                          const uint32_t *__restrict__ parent, uint32_t *comp_n, uint32_t per_warp) {
    const unsigned lane = lane_id();
    for (uint32_t v0 = warp_global() * per_warp; v0 < n; v0 += warps_total() * per_warp) {
        const uint32_t v = v0 + lane;
        bool may = false;
        uint32_t r = 0, d = 0;
        if (lane < per_warp && v < n && alive[v]) {
            r = parent[v];
            d = cdeg[v];
            may = cdeg[r] == d && parent[r] == r;
        }
        for (unsigned todo = __ballot_sync(0xffffffffu, may); todo; todo &= todo - 1) {
            const int j = __ffs(todo) - 1;
            const uint32_t u = v0 + j;
            const uint32_t ru = __shfl_sync(0xffffffffu, r, j), du = __shfl_sync(0xffffffffu, d, j);
            bool ok = true;
            for (uint64_t x = rp[u]; x < rp[u + 1] && ok; x += 32) {
                bool bad = false;
                if (x + lane < rp[u + 1]) {
                    const uint32_t w = col[x + lane];
                    bad = alive[w] && (parent[w] != ru || cdeg[w] != du);
                }
                ok = !__any_sync(0xffffffffu, bad);
            }
            if (ok && lane == 0) atomicAdd(&comp_n[ru], 1u);
        }
    }
}

// C(n, k) in 64 bits; sets *ovf when it does not fit.
__device__ unsigned long long binom64(unsigned long long n, unsigned k, bool *ovf) {
    if (k > n) return 0;
    if (k > n - k) k = (unsigned)(n - k);
    unsigned long long r = 1;
    for (unsigned i = 1; i <= k; i++) {
        unsigned long long f = n - k + i;
        unsigned long long hi = __umul64hi(r, f);
        unsigned long long lo = r * f;
        if (hi >= i) { *ovf = true; return 0; }
        // exact division of the 128-bit product (hi:lo) by i, hi < i
        unsigned long long q = 0, rem = hi;
        for (int bit = 63; bit >= 0; bit--) {
            unsigned long long top = rem >> 63;
            rem = (rem << 1) | ((lo >> bit) & 1ull);
            if (top || rem >= i) { rem -= i; q |= 1ull << bit; }
        }
        r = q;
    }
    return r;
}

__global__ void k_pl_check(uint32_t n, uint32_t k, const uint8_t *__restrict__ kmap,
                           const uint8_t *__restrict__ alive,
                           const uint32_t *__restrict__ parent, const uint32_t *__restrict__ comp_n,
                           const uint32_t *__restrict__ cdeg, uint32_t *comp_flag,
                           uint32_t *comp_slot, unsigned long long *vcount, DevResult *res) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        if (!alive[v] || parent[v] != v) continue;
        if (res->pre_nin) continue;  // Pre-Core has rounds left: the call comes back here after them
        const unsigned long long nc = comp_n[v];
        if (nc != (unsigned long long)cdeg[v] + 1) continue;  // not all of N[v] passed
        bool ovf = false;
        unsigned long long c = binom64(nc, kmap ? kmap[v] : k, &ovf);  // a component lies in one graph
        if (ovf) atomicOr(&res->status, DEV_ERR_OVERFLOW);
        add_count(&res->pre_count, &res->count_carry, c);
        if (vcount && c) atomicAdd(&vcount[v], c);  // attributed to the component's root
        uint32_t slot = atomicAdd(&res->n_clique_comps, 1u);
        comp_flag[v] = 1;
        if (comp_slot) comp_slot[v] = slot;
    }
}

__global__ void k_pl_remove(uint32_t n, uint8_t *alive, const uint32_t *__restrict__ parent,
                            const uint32_t *__restrict__ comp_flag) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
        if (alive[v] && comp_flag[parent[v]]) alive[v] = 0;
}

// Listing of Pre-List cliques: gather each clique component's members,
// sort them, then enumerate every k-subset by unranking (combinatorial
// number system) so each k-clique of the component is reported once.
__global__ void k_comp_gather(uint32_t n, const uint32_t *__restrict__ parent,
                              const uint32_t *__restrict__ comp_flag, const uint32_t *__restrict__ comp_slot,
                              const uint8_t *__restrict__ alive_core, const uint32_t *__restrict__ offs,
                              uint32_t *fill, uint32_t *members) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        if (!alive_core[v]) continue;
        uint32_t r = parent[v];
        if (!comp_flag[r]) continue;
        uint32_t s = comp_slot[r];
        members[offs[s] + atomicAdd(&fill[s], 1u)] = v;
    }
}

__global__ void k_comp_sizes(uint32_t n, const uint32_t *__restrict__ comp_flag,
                             const uint32_t *__restrict__ comp_slot, const uint32_t *__restrict__ comp_n,
                             uint32_t *sizes, uint32_t *roots) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        if (!comp_flag[v]) continue;
        sizes[comp_slot[v]] = comp_n[v];
        roots[comp_slot[v]] = v;
    }
}

// One block per component: odd-even transposition sort of its members.
__global__ void k_comp_sort(const uint32_t *__restrict__ offs, const uint32_t *__restrict__ sizes,
                            uint32_t *members) {
    uint32_t s = blockIdx.x;
    uint32_t *m = members + offs[s];
    uint32_t len = sizes[s];
    for (uint32_t phase = 0; phase < len; phase++) {
        for (uint32_t i = 2 * threadIdx.x + (phase & 1); i + 1 < len; i += 2 * blockDim.x) {
            uint32_t a = m[i], b = m[i + 1];
            if (a > b) { m[i] = b; m[i + 1] = a; }
        }
        __syncthreads();
    }
}

// C(n, k) saturated at 2^64 - 1 (used for comparisons while unranking).
__device__ unsigned long long binom_small(unsigned long long n, unsigned k) {
    bool ovf = false;
    unsigned long long r = binom64(n, k, &ovf);
    return ovf ? ~0ull : r;
}

__global__ void k_comp_emit(uint32_t kk, const uint8_t *__restrict__ kmap, const uint32_t *__restrict__ offs,
                            const uint32_t *__restrict__ sizes, const uint32_t *__restrict__ members,
                            uint32_t *ring, unsigned long long capacity, int wrap,
                            const uint32_t *__restrict__ croots, unsigned long long *vcks,
                            const uint32_t *__restrict__ idmap, DevResult *res) {
    uint32_t s = blockIdx.x;
    const uint32_t k = kmap ? kmap[croots[s]] : kk;
    const uint32_t *m = members + offs[s];
    uint32_t nc = sizes[s];
    if (nc < k) return;
    unsigned long long total = binom_small(nc, k);
    unsigned long long local_sum = 0;
    uint32_t ids[KCL_MAX_K];
    for (unsigned long long r = threadIdx.x; r < total; r += blockDim.x) {
        // unrank r: largest c_i with C(c_i, i) <= remaining, i = k..1
        unsigned long long rem = r;
        uint32_t hi = nc;
        for (uint32_t i = k; i >= 1; i--) {
            uint32_t c = i - 1;
            // linear scan upward is fine for the small components this handles
            uint32_t lo = i - 1, up = hi;  // C(c, i) <= rem, c in [i-1, hi-1]
            while (lo + 1 < up) {
                uint32_t mid = (lo + up) >> 1;
                if (binom_small(mid, i) <= rem) lo = mid; else up = mid;
            }
            c = lo;
            rem -= binom_small(c, i);
            ids[i - 1] = idmap ? idmap[m[c]] : m[c];
            hi = c;
        }
        uint64_t h = hash_seed(k);
        for (uint32_t i = 0; i < k; i++) h = mix64(h ^ (uint64_t)ids[i]);
        local_sum += h;
        if (ring) {
            unsigned long long slot = atomicAdd(&res->emitted, 1ull);
            if (wrap) slot %= capacity;
            if (slot < capacity)
                for (uint32_t i = 0; i < k; i++) ring[slot * k + i] = ids[i];
        }
    }
    atomicAdd(&res->pre_checksum, local_sum);
    if (vcks && local_sum) atomicAdd(&vcks[croots[s]], local_sum);
}

// -------------------------------------------------------- orientations
__global__ void k_degree_key(uint32_t n, const uint8_t *__restrict__ alive,
                             const uint32_t *__restrict__ cdeg, uint32_t *key) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
        key[v] = alive[v] ? cdeg[v] : 0xFFFFFFFFu;
}

// Degeneracy ordering by bulk peel rounds: each round removes every remaining
// vertex whose current degree is <= t; when none qualifies t rises to the
// minimum remaining degree.  key[v] = the round v leaves in (UINT_MAX while
// it remains).
__global__ void k_peel_init(uint32_t n, const uint8_t *__restrict__ alive,
                            const uint32_t *__restrict__ cdeg, uint32_t *pdeg, uint32_t *key,
                            DevResult *res) {
    uint32_t cnt = 0;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        pdeg[v] = cdeg[v];
        key[v] = 0xFFFFFFFFu;
        cnt += alive[v] ? 1 : 0;
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane_id() == 0 && cnt) atomicAdd(&res->remaining, cnt);
}

__global__ void k_peel_min(uint32_t n, const uint8_t *__restrict__ alive,
                           const uint32_t *__restrict__ pdeg, const uint32_t *__restrict__ key,
                           DevResult *res) {
    uint32_t mn = 0xFFFFFFFFu;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
        if (alive[v] && key[v] == 0xFFFFFFFFu && pdeg[v] < mn) mn = pdeg[v];
    mn = __reduce_min_sync(0xffffffffu, mn);
    if (lane_id() == 0 && mn != 0xFFFFFFFFu) atomicMin(&res->min_deg, mn);
}

__global__ void k_peel_select_all(uint32_t n, const uint8_t *__restrict__ alive,
                                  const uint32_t *__restrict__ pdeg, uint32_t *key, uint32_t t,
                                  uint32_t round, uint32_t *fout, unsigned *fcount) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        if (alive[v] && key[v] == 0xFFFFFFFFu && pdeg[v] <= t) {
            key[v] = round;
            fout[atomicAdd(fcount, 1u)] = v;
        }
    }
}

__global__ void k_peel_update(const uint64_t *__restrict__ rp, const uint32_t *__restrict__ col,
                              const uint8_t *__restrict__ alive, uint32_t *pdeg, uint32_t *key,
                              const uint32_t *__restrict__ fin, uint32_t nin, uint32_t t,
                              uint32_t next_round, uint32_t *fout, unsigned *fcount) {
    const unsigned lane = lane_id();
    for (uint32_t i = warp_global(); i < nin; i += warps_total()) {
        uint32_t v = fin[i];
        for (uint64_t e = rp[v] + lane; e < rp[v + 1]; e += 32) {
            uint32_t w = col[e];
            if (!alive[w] || key[w] != 0xFFFFFFFFu) continue;
            uint32_t nd = atomicSub(&pdeg[w], 1u) - 1u;
            if (nd <= t && atomicCAS(&key[w], 0xFFFFFFFFu, next_round) == 0xFFFFFFFFu)
                fout[atomicAdd(fcount, 1u)] = w;
        }
    }
}

constexpr unsigned long long kSpinLimit = 1ull << 25;

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned atom_add_acq_rel(unsigned *p, unsigned x) {
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(x) : "memory");
    return old;
}

// Generation barrier: thread 0 of each block arrives with an acquire-release
// add (publishing the block's writes, which __syncthreads has ordered before
// it); the last arrival clears the count and bumps the generation with a
// release, and the others poll the generation with acquire loads.
__device__ bool grid_barrier(PeelCtl *c, unsigned nblocks) {
    __shared__ int ok_s;
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned g = ld_acquire(&c->bar_gen);
        const unsigned arrived = atom_add_acq_rel(&c->bar_count, 1u);
        int ok = 1;
        if (arrived == nblocks - 1) {
            atomicExch(&c->bar_count, 0u);
            atom_add_acq_rel(&c->bar_gen, 1u);
        } else {
            unsigned long long spins = 0;
            while (ld_acquire(&c->bar_gen) == g) {
                if (ld_acquire(&c->error)) { ok = 0; break; }
                if (++spins > kSpinLimit) { atomicExch(&c->error, 1u); ok = 0; break; }
            }
        }
        ok_s = ok && ld_acquire(&c->error) == 0;
    }
    __syncthreads();
    return ok_s != 0;
}

// The same peel in one launch of co-resident blocks: rounds are separated by
// a barrier instead of a kernel boundary and a host round trip.  A graph has
// hundreds of rounds with little work each (660 on R-MAT 20, most of them one
// threshold step with a few vertices), so a round's chain of dependent memory
// accesses and barriers is what bounds the peel:
//   - a vertex is gone once its degree is at or below t, so relaxing an edge
//     is one atomic on the neighbour's degree, with no look at its key or alive
//     flag (vertices that are not alive hold a degree far below zero); the
//     thread that sees t + 1 -> t, and only that one, puts it in the next round;
//   - a threshold step looks only at the near list, the vertices whose degree
//     lies in (t, B]; a relaxation that sees B + 1 -> B adds to it, and a pass
//     over all vertices starts a new one every kNear thresholds;
//   - a round with few vertices spreads each row over several warps;
//   - the whole grid runs the wide first rounds (grid barrier, about 2 us), one
//     cluster of at most 16 CTAs the long tail, with its hardware barrier and the
//     counters in the first CTA's shared memory.
// On the 1M-vertex R-MAT graph (678 rounds) this took the peel from 17.5 to 6.3
// ms, about 7 us a round in the cluster, 3.1 us on 65k vertices.
// Every thread follows the same control flow, derived from counters read after
// a barrier; frontier and big-row counters rotate over three rounds (round r
// reads slot r % 3, appends to (r + 1) % 3 and clears (r + 2) % 3, which
// everybody read two barriers earlier).  Arrays written during the launch are
// read with ld.global.cg (L2) so no stale L1 line is used.  Every grid-barrier
// wait is bounded: past kSpinLimit polls the block records an error, all blocks
// leave, and the host reports KCL_ETIMEOUT.
constexpr int kNear = 32;                 // thresholds a near list covers
constexpr uint32_t kBigRow = 4096;        // longer rows are walked by all warps
constexpr int kGone = -(1 << 30);         // degree of a vertex that is not alive
// 768 threads of 40 registers, two loads a lane: the co-resident CTAs and clusters
// have to find room beside the kernels of other streams, and 1,024 threads of 52
// (four loads a lane) fitted only into almost empty SMs: beside a k = 7 listing a
// colour count of the 262k-vertex R-MAT graph waited 2.2 s for that call's end,
// now 0.28 s.  Alone: 262k vertices 2.62 ms both, 60k 1.42 -> 1.35, 2,000 vertices
// in one CTA 0.141 -> 0.125; 1,024 threads capped at 32 registers spilled (2.87).
constexpr int kPeelThreads = 768;
constexpr int kPeelLoads = 2;
constexpr uint64_t kFetchEntries = 1ull << 25;  // 128 MB of ids

struct PeelArgs {
    uint32_t n;
    const uint64_t *rp;
    const uint32_t *col;
    const uint8_t *alive;
    const uint32_t *cdeg;
    int *deg;          // degrees during the peel
    uint32_t *key;     // round a vertex leaves in
    uint32_t *order;   // vertices in the order they leave: round r's frontier is a range
    uint32_t *near;    // near list
    PeelCtl *ctl;
    uint32_t handover; // grid: leave the rest to the cluster at this many vertices
};

struct GridSync {
    PeelCtl *ctl;
    unsigned nblocks;
    __device__ __forceinline__ bool operator()() const { return grid_barrier(ctl, nblocks); }
};
struct BlockSync {
    __device__ __forceinline__ bool operator()() const {
        __syncthreads();
        return true;
    }
};
struct ClusterSync {
    __device__ __forceinline__ bool operator()() const {
        asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
        return true;
    }
};

// Words other threads of the group write: from L2, or from shared memory (SH).
template <bool SH, typename T>
__device__ __forceinline__ T peel_load(const T *p) {
    if constexpr (SH) return *reinterpret_cast<const volatile T *>(p);
    else return __ldcg(p);
}

// Degrees, keys and the number of vertices to peel.
__device__ void peel_setup(const PeelArgs &a, uint32_t tid, uint32_t nth, unsigned *total) {
    uint32_t cnt = 0;
    for (uint32_t v0 = tid - lane_id(); v0 < a.n; v0 += nth) {  // warp-uniform trip count
        const uint32_t v = v0 + lane_id();
        if (v < a.n) {
            const bool on = a.alive[v] != 0;
            a.deg[v] = on ? (int)a.cdeg[v] : kGone;
            a.key[v] = 0xFFFFFFFFu;
            cnt += on ? 1 : 0;
        }
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane_id() == 0 && cnt) atomicAdd(total, cnt);
}

// A graph's rows: in global memory, or copied to shared memory (small graphs; ids
// below 2^16).
struct GlobalRows {
    const uint64_t *rp;
    const uint32_t *col;
    using Pos = uint64_t;
    __device__ __forceinline__ Pos begin(uint32_t v) const { return rp[v]; }
    __device__ __forceinline__ Pos end(uint32_t v) const { return rp[v + 1]; }
    __device__ __forceinline__ uint32_t entry(Pos x) const { return col[x]; }
};
struct LocalRows {
    const uint32_t *rp;
    const uint16_t *col;
    using Pos = uint32_t;
    __device__ __forceinline__ Pos begin(uint32_t v) const { return rp[v]; }
    __device__ __forceinline__ Pos end(uint32_t v) const { return rp[v + 1]; }
    __device__ __forceinline__ uint32_t entry(Pos x) const { return col[x]; }
};

// Lowers the degrees of up to kPeelLoads neighbours a lane (n of them valid, stride
// `step` from x) and appends those that reach t or B.
template <typename R>
__device__ __forceinline__ void peel_relax(const PeelArgs &a, const R &rows, PeelCounters *c, unsigned *next,
                                           uint32_t next0, typename R::Pos x, typename R::Pos e,
                                           typename R::Pos step, int t, int B, uint32_t round) {
    uint32_t w[kPeelLoads];
    int old[kPeelLoads];
#pragma unroll
    for (int z = 0; z < kPeelLoads; z++) w[z] = x + z * step < e ? rows.entry(x + z * step) : 0xFFFFFFFFu;
#pragma unroll
    for (int z = 0; z < kPeelLoads; z++) old[z] = w[z] != 0xFFFFFFFFu ? atomicSub(&a.deg[w[z]], 1) : kGone;
#pragma unroll
    for (int z = 0; z < kPeelLoads; z++) {
        const bool join = old[z] == t + 1;
        const unsigned m = __ballot_sync(0xffffffffu, join);
        if (m) {
            const uint32_t at = warp_append(m, next);
            if (join) {
                a.order[next0 + at] = w[z];
                a.key[w[z]] = round + 1;
            }
        }
        const bool close = old[z] == B + 1 && B > t;
        const unsigned mc = __ballot_sync(0xffffffffu, close);
        if (mc) {
            const uint32_t at = warp_append(mc, &c->near);
            if (close) a.near[at] = w[z];
        }
    }
}

// The rounds from state `st` on; every thread of the group calls it with the
// same state.  Returns when at most `stop` vertices remain (0: all peeled),
// with the state to resume from; false when a barrier gave up.
template <bool SH, typename R, typename Sync>
__device__ __forceinline__ bool peel_rounds(const PeelArgs &a, const R &rows, PeelCounters *c, PeelState &st,
                                            uint32_t stop, uint32_t tid, uint32_t nth, const Sync &sync) {
    using Pos = typename R::Pos;
    volatile PeelCounters *vc = c;
    const unsigned lane = lane_id();
    const uint32_t gw = tid >> 5, W = nth >> 5;
    uint32_t q = 0;  // threshold passes so far (minimum slots rotate over four)
    while (st.done < st.total && st.total - st.done > stop) {
        const uint32_t fi = st.round % 3u;
        if (st.nin == 0) {
            // every remaining degree is above t: raise t to their minimum
            for (;;) {
                const uint32_t slot = q++ & 3u;
                if (tid == 0) c->top[(slot + 2) & 3u] = c->sel[(slot + 2) & 3u] = 0;
                const bool fresh = st.t + 1 > st.B;  // no near list for t + 1: start one
                uint32_t best = 0;  // of 0x80000000 - degree: the maximum marks the minimum degree
                if (fresh) {
                    if (tid == 0) c->near = 0;
                    if (!sync()) return false;
                    const int B = st.t + kNear;
                    for (uint32_t v0 = tid - lane; v0 < a.n; v0 += nth) {
                        const uint32_t v = v0 + lane;
                        const int d = v < a.n ? peel_load<SH>(&a.deg[v]) : kGone;
                        const bool rest = d > st.t, in = rest && d <= B;
                        if (rest) best = max(best, 0x80000000u - (uint32_t)d);
                        const unsigned m = __ballot_sync(0xffffffffu, in);
                        if (m) {
                            const uint32_t at = warp_append(m, &c->near);
                            if (in) a.near[at] = v;
                        }
                    }
                } else {
                    const uint32_t nn = vc->near;
                    for (uint32_t i0 = tid - lane; i0 < nn; i0 += nth) {
                        const uint32_t i = i0 + lane;
                        uint32_t v = 0;
                        int d = kGone;
                        if (i < nn) {
                            v = peel_load<SH>(&a.near[i]);
                            d = peel_load<SH>(&a.deg[v]);
                        }
                        if (d > st.t) best = max(best, 0x80000000u - (uint32_t)d);
                        const bool sel = d == st.t + 1;
                        const unsigned m = __ballot_sync(0xffffffffu, sel);
                        if (m) {
                            const uint32_t at = warp_append(m, &c->sel[slot]);
                            if (sel) {
                                a.order[st.done + at] = v;
                                a.key[v] = st.round;
                            }
                        }
                    }
                }
                best = __reduce_max_sync(0xffffffffu, best);
                if (lane == 0 && best) atomicMax(&c->top[slot], best);
                if (!sync()) return false;
                const uint32_t top = vc->top[slot];
                const int mn = top ? (int)(0x80000000u - top) : 0;
                if (fresh) {
                    if (!top) {  // cannot happen while vertices remain
                        if (tid == 0) atomicExch(&a.ctl->error, 2u);
                        return false;
                    }
                    const int B = st.t + kNear;
                    st.t = mn - 1;
                    st.B = mn <= B ? B : st.t;  // nothing up to B: start over from the minimum
                    continue;
                }
                st.nin = vc->sel[slot];
                if (st.nin) {
                    st.t++;
                    break;
                }
                if (top) st.t = mn - 1;  // the near list's minimum is higher
                else st.B = st.t;        // the near list is used up
            }
        }
        if (tid == 0) {
            c->fcnt[(st.round + 2u) % 3u] = 0;
            c->bcnt[(st.round + 1u) % 3u] = 0;
        }
        // remove this round's vertices
        unsigned *next = &c->fcnt[(st.round + 1u) % 3u];
        unsigned *bcnt = &c->bcnt[fi];
        uint32_t *big = a.ctl->big[fi];
        const uint32_t next0 = st.done + st.nin;
        uint32_t ls = 0;  // log2 of the warps per row
        while ((st.nin << (ls + 1)) <= W) ls++;
        for (uint32_t unit = gw; unit < st.nin << ls; unit += W) {
            const uint32_t v = peel_load<SH>(&a.order[st.done + (unit >> ls)]);
            const Pos b = rows.begin(v), e = rows.end(v);
            if (ls == 0 && e - b > kBigRow) {
                uint32_t at = 0;
                if (lane == 0) at = atomicAdd(bcnt, 1u);
                at = __shfl_sync(0xffffffffu, at, 0);
                if (at < kPeelBig) {
                    if (lane == 0) big[at] = v;
                    continue;
                }
            }
            const Pos step = (Pos)32 << ls;
            for (Pos x = b + 32 * (unit & ((1u << ls) - 1u)); x < e; x += kPeelLoads * step)
                peel_relax(a, rows, c, next, next0, x + lane, e, step, st.t, st.B, st.round);
        }
        if (!sync()) return false;
        const uint32_t nb = min(vc->bcnt[fi], (unsigned)kPeelBig);
        if (nb) {
            for (uint32_t i = 0; i < nb; i++) {
                const uint32_t v = __ldcg(&big[i]);
                const Pos b = rows.begin(v), e = rows.end(v);
                for (Pos x = b + (Pos)gw * 32; x < e; x += (Pos)kPeelLoads * nth)
                    peel_relax(a, rows, c, next, next0, x + lane, e, nth, st.t, st.B, st.round);
            }
            if (!sync()) return false;
        }
        st.done = next0;
        st.round++;
        st.nin = vc->fcnt[st.round % 3u];
    }
    return true;
}

// The wide rounds, all SMs.
__global__ void __launch_bounds__(kPeelThreads, 2) k_peel_grid(const PeelArgs a) {
    PeelCounters *c = &a.ctl->cnt;
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    const GridSync sync{a.ctl, gridDim.x};
    peel_setup(a, tid, nth, &a.ctl->total);
    if (!sync()) return;
    PeelState st{0, 0, 0, -1, -1, *(volatile unsigned *)&a.ctl->total};
    if (!peel_rounds<false>(a, GlobalRows{a.rp, a.col}, c, st, a.handover, tid, nth, sync)) return;
    if (tid == 0) a.ctl->st = st;
    // The cluster reads the remaining rows on 16 SMs, most of them for the first
    // time: all SMs fetch them into L2 before they leave (262k vertices 2.90 -> 2.74
    // ms with nothing in L2 before, 65k 1.54 -> 1.45), if they fit there.
    if (st.done == st.total || a.rp[a.n] > kFetchEntries) return;
    const unsigned lane = lane_id();
    for (uint32_t v0 = tid - lane; v0 < a.n; v0 += nth) {
        const bool rest = v0 + lane < a.n && __ldcg(&a.deg[v0 + lane]) > st.t;
        for (unsigned todo = __ballot_sync(0xffffffffu, rest); todo; todo &= todo - 1) {
            const uint32_t v = v0 + __ffs(todo) - 1;
            for (uint64_t x = a.rp[v] + 32 * lane; x < a.rp[v + 1]; x += 1024)
                asm volatile("prefetch.global.L2 [%0];" :: "l"(a.col + x));
        }
    }
}

// The rest (or, for small graphs, all of it: resume = 0) in one cluster.
__global__ void __launch_bounds__(kPeelThreads, 2) k_peel_cluster(const PeelArgs a, int resume) {
    __shared__ PeelCounters own;
    __shared__ unsigned total;
    uint32_t rank, csize;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(csize));
    const uint32_t tid = rank * blockDim.x + threadIdx.x, nth = csize * blockDim.x;
    const ClusterSync sync;
    if (resume && a.ctl->error) return;  // the grid's rounds gave up: every thread leaves
    if (threadIdx.x == 0) {
        own = PeelCounters{};
        total = 0;
        if (resume) {
            own = a.ctl->cnt;
            for (int i = 0; i < 4; i++) own.top[i] = own.sel[i] = 0;  // threshold passes start over
        }
    }
    // the first CTA's counters, by their address in the cluster's shared memory
    PeelCounters *c;
    unsigned *tot;
    {
        uint64_t p = reinterpret_cast<uint64_t>(&own), r;
        asm("mapa.u64 %0, %1, 0;" : "=l"(r) : "l"(p));
        c = reinterpret_cast<PeelCounters *>(r);
        p = reinterpret_cast<uint64_t>(&total);
        asm("mapa.u64 %0, %1, 0;" : "=l"(r) : "l"(p));
        tot = reinterpret_cast<unsigned *>(r);
    }
    sync();
    PeelState st;
    if (resume) {
        st = a.ctl->st;
    } else {
        peel_setup(a, tid, nth, tot);
        sync();
        st = PeelState{0, 0, 0, -1, -1, *(volatile unsigned *)tot};
    }
    peel_rounds<false>(a, GlobalRows{a.rp, a.col}, c, st, 0, tid, nth, sync);
    sync();  // the first CTA's shared memory outlives the others' last access
}

// Small graphs in one CTA, with the degrees, the removal order and the near
// list in shared memory, and the rows too when they fit (LOCAL), so a round makes
// no L2 round trip.  Orientation stage of a 2,000-vertex graph of 67 rounds: 0.20
// ms in the cluster, 0.14 with the rows in global memory, 0.13 with all of it here.
template <bool LOCAL>
__global__ void __launch_bounds__(kPeelThreads, 2) k_peel_block(PeelArgs a, uint32_t nnz) {
    extern __shared__ int peel_smem[];
    __shared__ PeelCounters own;
    __shared__ unsigned total;
    a.deg = peel_smem;
    a.order = reinterpret_cast<uint32_t *>(peel_smem + a.n);
    a.near = a.order + a.n;
    uint32_t *rp = a.near + a.n;
    uint16_t *col = reinterpret_cast<uint16_t *>(rp + a.n + 1);
    if (threadIdx.x == 0) {
        own = PeelCounters{};
        total = 0;
    }
    if (LOCAL) {
        for (uint32_t v = threadIdx.x; v <= a.n; v += blockDim.x) rp[v] = (uint32_t)a.rp[v];
        for (uint32_t x = threadIdx.x; x < nnz; x += blockDim.x) col[x] = (uint16_t)a.col[x];
    }
    const BlockSync sync;
    sync();
    peel_setup(a, threadIdx.x, blockDim.x, &total);
    sync();
    PeelState st{0, 0, 0, -1, -1, total};
    if (LOCAL) peel_rounds<true>(a, LocalRows{rp, col}, &own, st, 0, threadIdx.x, blockDim.x, sync);
    else peel_rounds<true>(a, GlobalRows{a.rp, a.col}, &own, st, 0, threadIdx.x, blockDim.x, sync);
}

// Out-degree in the DAG u -> w iff (key[u], u) < (key[w], w), both alive.
__device__ __forceinline__ bool eta_less(uint32_t ku, uint32_t u, uint32_t kw, uint32_t w) {
    return ku < kw || (ku == kw && u < w);
}

// Out-degrees.  key is UINT_MAX for vertices that are not alive, so one random
// read per entry decides it; up to four chunks of a row are read together, and
// a warp keeps its largest out-degree to itself until the end.  The decisions
// on a row's first 64 entries are kept for k_outfill, which then reads no keys
// for them.  Orientation stage of the 1M-vertex R-MAT graph, degree ordering:
// 3.0 -> 1.1 ms with the roots' sort (the rows' 268 MB take 0.04 ms at the
// copy bandwidth; the random key reads bound it).
__global__ void k_outdeg(uint32_t n, const uint64_t *__restrict__ rp, const uint32_t *__restrict__ col,
                         const uint32_t *__restrict__ key, uint32_t *outdeg, unsigned long long *take,
                         DevResult *res) {
    const unsigned lane = lane_id();
    uint32_t most = 0;
    for (uint32_t u = warp_global(); u < n; u += warps_total()) {
        const uint32_t ku = key[u];
        uint32_t c = 0;
        if (ku != 0xFFFFFFFFu) {
            const uint64_t b = rp[u], e = rp[u + 1];
            unsigned long long kept = 0;
            for (uint64_t x = b; x < e; x += 128) {
                uint32_t w[4], kw[4];
#pragma unroll
                for (int z = 0; z < 4; z++) w[z] = x + z * 32 + lane < e ? col[x + z * 32 + lane] : 0u;
#pragma unroll
                for (int z = 0; z < 4; z++) kw[z] = x + z * 32 + lane < e ? key[w[z]] : 0xFFFFFFFFu;
#pragma unroll
                for (int z = 0; z < 4; z++) {
                    const bool out = kw[z] != 0xFFFFFFFFu && eta_less(ku, u, kw[z], w[z]);
                    const unsigned m = __ballot_sync(0xffffffffu, out);
                    c += __popc(m);
                    if (x == b && z < 2) kept |= (unsigned long long)m << (32 * z);
                }
            }
            if (lane == 0) take[u] = kept;
        }
        if (lane == 0) outdeg[u] = c;
        most = max(most, c);
    }
    if (lane == 0 && most) atomicMax(&res->max_outdeg, most);
}

__global__ void k_outfill(uint32_t n, const uint64_t *__restrict__ rp, const uint32_t *__restrict__ col,
                          const uint32_t *__restrict__ key, const unsigned long long *__restrict__ take,
                          const uint32_t *__restrict__ optr, uint32_t *oadj) {
    const unsigned lane = lane_id(), lt = (1u << lane) - 1u;
    for (uint32_t u = warp_global(); u < n; u += warps_total()) {
        uint32_t base = optr[u];
        const uint32_t end = optr[u + 1];
        if (base == end) continue;
        const uint64_t b = rp[u], e = rp[u + 1];
        const unsigned long long kept = take[u];
        const uint32_t ku = key[u];
        for (uint64_t x = b; x < e && base < end; x += 128) {
            uint32_t w[4], kw[4];
#pragma unroll
            for (int z = 0; z < 4; z++) w[z] = x + z * 32 + lane < e ? col[x + z * 32 + lane] : 0u;
#pragma unroll
            for (int z = 0; z < 4; z++)
                kw[z] = (x > b || z > 1) && x + z * 32 + lane < e ? key[w[z]] : 0xFFFFFFFFu;
#pragma unroll
            for (int z = 0; z < 4; z++) {
                unsigned m;
                if (x == b && z < 2) m = (unsigned)(kept >> (32 * z));
                else m = __ballot_sync(0xffffffffu, kw[z] != 0xFFFFFFFFu && eta_less(ku, u, kw[z], w[z]));
                if ((m >> lane) & 1u) oadj[base + __popc(m & lt)] = w[z];
                base += __popc(m);
            }
        }
    }
}

// Roots (alive, d+ >= k-1) counted by out-degree, then placed in descending
// out-degree order by a counting sort: hist index = top - d+ (top is at least
// every out-degree, except that those above the largest class share index 0).
// Most roots share a few small out-degrees: lanes with the same one add once.
__device__ __forceinline__ bool root_bin(uint32_t v, uint32_t n, uint32_t k, const uint32_t *outdeg, uint32_t top,
                                         const uint8_t *mask, const uint8_t *kmap, uint32_t *bin) {
    if (v >= n) return false;
    const uint32_t d = outdeg[v];  // 0 unless alive
    *bin = top > d ? top - d : 0u;
    return d > 0 && d + 1 >= (kmap ? kmap[v] : k) && (!mask || mask[v]);
}

__global__ void k_root_hist(uint32_t n, uint32_t k, const uint32_t *__restrict__ outdeg, uint32_t top,
                            uint32_t *hist, const uint8_t *__restrict__ mask, const uint8_t *__restrict__ kmap,
                            DevResult *res) {
    const unsigned lane = lane_id();
    uint32_t cnt = 0;
    for (uint32_t v0 = blockIdx.x * blockDim.x + threadIdx.x - lane; v0 < n; v0 += gridDim.x * blockDim.x) {
        uint32_t h = 0;
        const bool root = root_bin(v0 + lane, n, k, outdeg, top, mask, kmap, &h);
        const unsigned same = __match_any_sync(0xffffffffu, root ? h : 0xFFFFFFFFu);
        if (root) {
            cnt++;
            if (lane == __ffs(same) - 1) atomicAdd(&hist[h], (unsigned)__popc(same));
        }
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0 && cnt) atomicAdd(&res->n_roots, cnt);
}

__global__ void k_root_scatter(uint32_t n, uint32_t k, const uint32_t *__restrict__ outdeg, uint32_t top,
                               const uint32_t *__restrict__ offs, uint32_t *fill,
                               const uint8_t *__restrict__ mask, const uint8_t *__restrict__ kmap,
                               uint32_t *roots) {
    const unsigned lane = lane_id();
    for (uint32_t v0 = blockIdx.x * blockDim.x + threadIdx.x - lane; v0 < n; v0 += gridDim.x * blockDim.x) {
        const uint32_t v = v0 + lane;
        uint32_t h = 0;
        const bool root = root_bin(v, n, k, outdeg, top, mask, kmap, &h);
        const unsigned same = __match_any_sync(0xffffffffu, root ? h : 0xFFFFFFFFu);
        const int lead = __ffs(same) - 1;
        uint32_t at = 0;
        if (root && (int)lane == lead) at = offs[h] + atomicAdd(&fill[h], (unsigned)__popc(same));
        at = __shfl_sync(0xffffffffu, at, lead);
        if (root) roots[at + __popc(same & ((1u << lane) - 1u))] = v;
    }
}

// res->class_begin[c] = first root position whose d+ <= limits[c] (roots are
// in descending d+), i.e. the number of roots with d+ > limits[c]; the last
// entry is the number of roots.  Also the peel's error word (peel null: no co-resident peel).
__global__ void k_class_bounds(const uint32_t *__restrict__ offs, uint32_t top, const ClassLimits limits,
                               int n_classes, const PeelCtl *peel, DevResult *res) {
    const int c = threadIdx.x;
    if (c < n_classes) {
        const uint32_t lim = limits.d[c];
        // hist index h = top - d; d > lim  <=>  h < top - lim
        res->class_begin[c] = lim >= top ? 0u : offs[top - lim];
    }
    if (c == 0) {
        res->class_begin[n_classes] = res->n_roots;
        res->peel_error = peel ? peel->error : 0u;
    }
}

// --------------------------------------------------------------- scans
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

__global__ void k_scan_tiles(const uint32_t *__restrict__ in, uint32_t *out, uint32_t n,
                             uint32_t *tile_sums) {
    __shared__ uint32_t smem[32];
    uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        v[i] = base + i < n ? in[base + i] : 0;
        s += v[i];
    }
    uint32_t total;
    uint32_t p = block_excl_scan(s, smem, &total);
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        if (base + i < n) out[base + i] = p;
        p += v[i];
    }
    if (threadIdx.x == 0 && tile_sums) tile_sums[blockIdx.x] = total;
}

__global__ void k_scan_add(uint32_t *out, uint32_t n, const uint32_t *__restrict__ tile_offs) {
    uint64_t base = (uint64_t)blockIdx.x * kScanTile;
    uint32_t add = tile_offs[blockIdx.x];
    for (uint32_t i = threadIdx.x; i < kScanTile; i += blockDim.x)
        if (base + i < n) out[base + i] += add;
}

}  // namespace

// ====================================================== host launchers
// ---------------------------------------------------------- batching
// Disjoint union of a batch of graphs: the blocks (b, *) copy graph b's rows and
// columns with its vertex offset voff[b] and edge offset eoff[b].  With one
// block a graph a batch of 64 waited for its largest graph (the whole batched
// call 4.18 ms, 3.75 with the stripes and wider sums).
__global__ void k_union_build(const BatchSrc *__restrict__ src, uint32_t n_total, uint64_t *urp,
                              uint32_t *ucol, uint32_t *graph_of, uint32_t *idmap, uint8_t *kmap) {
    const BatchSrc b = src[blockIdx.x];
    const uint32_t tid = blockIdx.y * blockDim.x + threadIdx.x, nth = gridDim.y * blockDim.x;
    for (uint32_t v = tid; v < b.n; v += nth) {
        urp[b.voff + v] = b.rp[v] + b.eoff;
        graph_of[b.voff + v] = blockIdx.x;
        idmap[b.voff + v] = v;
        kmap[b.voff + v] = (uint8_t)b.k;
    }
    for (uint64_t e = tid; e < b.nnz; e += nth) ucol[b.eoff + e] = b.col[e] + b.voff;
    if (blockIdx.x == gridDim.x - 1 && tid == 0) urp[n_total] = b.eoff + b.nnz;
}

// Per-graph sums of per-vertex attributions (one block per graph).
__global__ void k_graph_sums(const BatchSrc *__restrict__ src, const unsigned long long *__restrict__ vcount,
                             const unsigned long long *__restrict__ vcks, unsigned long long *out_count,
                             unsigned long long *out_cks) {
    __shared__ unsigned long long sc[32], sk[32];
    const BatchSrc b = src[blockIdx.x];
    unsigned long long c = 0, h = 0;
    for (uint32_t v = threadIdx.x; v < b.n; v += blockDim.x) {
        c += vcount[b.voff + v];
        if (vcks) h += vcks[b.voff + v];
    }
    for (int o = 16; o > 0; o >>= 1) {
        c += __shfl_down_sync(0xffffffffu, c, o);
        h += __shfl_down_sync(0xffffffffu, h, o);
    }
    if (lane_id() == 0) { sc[threadIdx.x >> 5] = c; sk[threadIdx.x >> 5] = h; }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long tc = 0, th = 0;
        for (uint32_t i = 0; i < (blockDim.x >> 5); i++) { tc += sc[i]; th += sk[i]; }
        out_count[blockIdx.x] = tc;
        if (out_cks) out_cks[blockIdx.x] = th;
    }
}

int launch_union_build(const BatchSrc *src, uint32_t G, uint32_t n_total, uint64_t *urp,
                       uint32_t *ucol, uint32_t *graph_of, uint32_t *idmap, uint8_t *kmap,
                       cudaStream_t s) {
    if (G == 0) return 0;
    const uint32_t stripes = G < 2048 ? 2048 / G : 1;  // about 13 blocks an SM
    k_union_build<<<dim3(G, stripes), 256, 0, s>>>(src, n_total, urp, ucol, graph_of, idmap, kmap);
    return 1;
}

int launch_graph_sums(const BatchSrc *src, uint32_t G, const unsigned long long *vcount,
                      const unsigned long long *vcks, unsigned long long *out_count,
                      unsigned long long *out_cks, cudaStream_t s) {
    if (G == 0) return 0;
    k_graph_sums<<<G, 1024, 0, s>>>(src, vcount, vcks, out_count, out_cks);
    return 1;
}

int launch_exclusive_scan(const uint32_t *in, uint32_t *out, uint32_t n, uint32_t *block_tmp,
                          cudaStream_t s) {
    // exclusive scan; out may alias in.  block_tmp needs ceil(n/2048) +
    // ceil(n/2048^2) + ... words.
    if (n == 0) return 0;
    uint32_t tiles = (n + kScanTile - 1) / kScanTile;
    if (tiles == 1) {
        k_scan_tiles<<<1, kScanThreads, 0, s>>>(in, out, n, nullptr);
        return 1;
    }
    k_scan_tiles<<<tiles, kScanThreads, 0, s>>>(in, out, n, block_tmp);
    int l = 1 + launch_exclusive_scan(block_tmp, block_tmp, tiles, block_tmp + tiles, s);
    k_scan_add<<<tiles, kScanThreads, 0, s>>>(out, n, block_tmp);
    return l + 1;
}

__global__ void k_set_deadline(DevResult *res, unsigned long long limit_ns) {
    res->deadline_ns = limit_ns ? global_ns() + limit_ns : 0ull;
}

int launch_set_deadline(DevResult *res, uint64_t limit_ms, cudaStream_t s) {
    k_set_deadline<<<1, 1, 0, s>>>(res, (unsigned long long)limit_ms * 1000000ull);
    return 1;
}

int launch_validate(const kcl_graph *g, DevResult *res, cudaStream_t s) {
    int grid = grid_for((uint64_t)g->n * 32, kBlock, g->num_sms, 32);
    k_validate<<<grid, kBlock, 0, s>>>(g->n, g->nnz, g->rp, g->col, res);
    return 1;
}

// The arrays and the threshold of a call's Pre-Core.  A threshold of 0 (k = 1:
// Pre-Core switched off) keeps every vertex, whatever the k map says.  The list is
// in an array that the stages up to the first host read leave alone.
static PreArgs precore_args(const kcl_graph *g, uint32_t k, Workspace &w) {
    return PreArgs{g->rp, g->col, k - 1, k > 1 ? w.kmap : nullptr, w.alive, w.cdeg, w.members, w.res};
}

int launch_precore_rounds(const kcl_graph *g, uint32_t k, Workspace &w, int rounds, uint32_t rows, cudaStream_t s) {
    const PreArgs a = precore_args(g, k, w);
    const int grid = grid_for((uint64_t)rows * 8, kPreThreads, g->num_sms, 2);  // 8 lanes a row
    for (int i = 0; i < rounds; i++) k_precore_round<<<grid, kPreThreads, 0, s>>>(a);
    return rounds;
}

int launch_precore(const kcl_graph *g, uint32_t k, Workspace &w, cudaStream_t s) {
    const PreArgs a = precore_args(g, k, w);
    k_precore_init<<<grid_for(g->n, kBlock, g->num_sms), kBlock, 0, s>>>(g->n, a.rp, a.thr, a.kmap, a.alive, a.cdeg,
                                                                        a.list, a.res);
    // wide rounds by size: 400,000 vertices at k = 10 have four of more than
    // kPreTail vertices, R-MAT graphs up to 2^20 vertices one or two
    return 1 + launch_precore_rounds(g, k, w, g->n <= 2048 ? 1 : g->n <= (1u << 16) ? 2 : 4, g->n, s);
}

int launch_prelist(const kcl_graph *g, uint32_t k, Workspace &w, int listing, cudaStream_t s) {
    int grid = grid_for(g->n, kBlock, g->num_sms);
    // a warp takes 32 vertices, fewer while that leaves warps idle (their rows are walked one by one)
    const uint32_t warps = (uint32_t)g->num_sms * 64;
    uint32_t per_warp = 32;
    while (per_warp > 1 && g->n / per_warp < warps) per_warp >>= 1;
    const int wgrid = grid_for(((uint64_t)g->n + per_warp - 1) / per_warp * 32, kBlock, g->num_sms);
    k_pl_min<<<wgrid, kBlock, 0, s>>>(g->n, g->rp, g->col, w.alive, w.parent, w.comp_n, w.comp_flag, per_warp);
    k_pl_pass<<<wgrid, kBlock, 0, s>>>(g->n, g->rp, g->col, w.alive, w.cdeg, w.parent, w.comp_n, per_warp);
    k_pl_check<<<grid, kBlock, 0, s>>>(g->n, k, w.kmap, w.alive, w.parent, w.comp_n, w.cdeg,
                                       w.comp_flag, listing ? w.comp_slot : nullptr, w.vcount_pre,
                                       w.res);
    k_pl_remove<<<grid, kBlock, 0, s>>>(g->n, w.alive, w.parent, w.comp_flag);
    return 4;
}

int launch_prelist_emit(const kcl_graph *g, uint32_t k, Workspace &w, uint32_t n_comps,
                        const kcl_ring *ring, cudaStream_t s) {
    if (n_comps == 0) return 0;
    int grid = grid_for(g->n, kBlock, g->num_sms);
    // sizes and offsets of the clique components (by slot)
    uint32_t *sizes = w.hist, *offs = w.hist + n_comps, *fill = w.hist + 2 * n_comps;
    uint32_t *croots = w.frontier_b;
    cudaMemsetAsync(fill, 0, n_comps * sizeof(uint32_t), s);
    k_comp_sizes<<<grid, kBlock, 0, s>>>(g->n, w.comp_flag, w.comp_slot, w.comp_n, sizes, croots);
    int l = 2 + launch_exclusive_scan(sizes, offs, n_comps, w.scan_tmp, s);
    k_comp_gather<<<grid, kBlock, 0, s>>>(g->n, w.parent, w.comp_flag, w.comp_slot, w.alive_core,
                                          offs, fill, w.members);
    k_comp_sort<<<n_comps, 256, 0, s>>>(offs, sizes, w.members);
    const bool to_ring = ring && ring->ids && ring->capacity;
    k_comp_emit<<<n_comps, 256, 0, s>>>(k, w.kmap, offs, sizes, w.members, to_ring ? ring->ids : nullptr,
                                        to_ring ? ring->capacity : 0, to_ring ? ring->wrap : 0,
                                        croots, w.vcks_pre, w.idmap, w.res);
    return l + 3;
}

int launch_degree_key(const kcl_graph *g, Workspace &w, cudaStream_t s) {
    int grid = grid_for(g->n, kBlock, g->num_sms);
    k_degree_key<<<grid, kBlock, 0, s>>>(g->n, w.alive, w.cdeg, w.key);
    return 1;
}

int launch_peel_init(const kcl_graph *g, Workspace &w, cudaStream_t s) {
    int grid = grid_for(g->n, kBlock, g->num_sms);
    k_peel_init<<<grid, kBlock, 0, s>>>(g->n, w.alive, w.cdeg, w.peel_deg, w.key, w.res);
    return 1;
}

int launch_peel_min(const kcl_graph *g, Workspace &w, cudaStream_t s) {
    int grid = grid_for(g->n, kBlock, g->num_sms);
    k_peel_min<<<grid, kBlock, 0, s>>>(g->n, w.alive, w.peel_deg, w.key, w.res);
    return 1;
}

int launch_peel_select_all(const kcl_graph *g, Workspace &w, uint32_t t, uint32_t round,
                           uint32_t *fout, cudaStream_t s) {
    int grid = grid_for(g->n, kBlock, g->num_sms);
    k_peel_select_all<<<grid, kBlock, 0, s>>>(g->n, w.alive, w.peel_deg, w.key, t, round, fout,
                                              &w.res->frontier);
    return 1;
}

int launch_peel_update(const kcl_graph *g, Workspace &w, const uint32_t *fin, uint32_t nin,
                       uint32_t t, uint32_t round, uint32_t *fout, cudaStream_t s) {
    int grid = grid_for((uint64_t)nin * 32, kBlock, g->num_sms, 32);
    k_peel_update<<<grid, kBlock, 0, s>>>(g->rp, g->col, w.alive, w.peel_deg, w.key, fin, nin, t,
                                          round + 1, fout, &w.res->frontier);
    return 1;
}

// Up to kClusterVertices vertices and kClusterEntries entries one cluster does the
// whole peel.  Of larger graphs the grid does the wide rounds, leaves the last
// kHandover vertices to the cluster and fetches their rows for it; a graph of fewer
// vertices but more entries it only sets up and fetches (65k vertices of 8M entries:
// 2.75 -> 2.62 ms; of 2M entries 1.59 either way).  Orientation stage of the 262k- and
// the 1M-vertex R-MAT graph in ms: handover at 8k vertices 4.14 / 8.74, 32k 3.02 / 8.28,
// 128k 2.82 / 7.48, 400k (262k vertices: all cluster) 2.86 / 7.93, the grid to the
// end 4.37 / 7.71.
// Up to kBlockVertices (whose arrays fit in shared memory) and kBlockEntries one
// CTA takes the whole peel: 5,000 vertices of 38k entries 0.22 ms against 0.29 in the
// cluster, 8,000 of 61k 0.37 both, 16,000 of 62k 0.41 against 0.31.
constexpr uint32_t kBlockVertices = 1u << 13;
constexpr uint64_t kBlockEntries = 1ull << 16;
constexpr size_t kBlockShared = 220 * 1024;
constexpr uint32_t kClusterVertices = 1u << 17;
constexpr uint64_t kClusterEntries = 1ull << 22;
constexpr uint32_t kHandover = 1u << 17;

// Blocks of the grid's peel for n vertices: one per SM (fewer arrivals per
// grid barrier), none beyond what n needs; -1 if it cannot be resident.
int peel_blocks(int num_sms, uint32_t n) {
    static PerDevice resident;
    const int per_sm = resident.get([](int) {
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_peel_grid, kPeelThreads, 0) != cudaSuccess) {
            (void)cudaGetLastError();
            b = 0;
        }
        return b;
    });
    if (per_sm <= 0) return -1;
    int blocks = num_sms;
    const uint64_t need = ((uint64_t)n + kPeelThreads - 1) / kPeelThreads;
    if (need < (uint64_t)blocks) blocks = need ? (int)need : 1;
    return blocks;
}

static void cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &attr, int size, cudaStream_t s) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)size);
    cfg.blockDim = dim3(kPeelThreads);
    cfg.stream = s;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)size;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
}

// Largest cluster of the peel the current device can place (16 CTAs need the
// non-portable size, which is allowed on each device separately), 0 if none.
static int peel_cluster_size() {
    static PerDevice largest;
    return largest.get([](int) {
        (void)cudaFuncSetAttribute(k_peel_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        for (int size = 16; size >= 1; size >>= 1) {
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute attr;
            cluster_config(cfg, attr, size, nullptr);
            int fit = 0;
            if (cudaOccupancyMaxActiveClusters(&fit, k_peel_cluster, &cfg) == cudaSuccess && fit > 0) return size;
            (void)cudaGetLastError();
        }
        return 0;
    });
}

// The whole peel: wide rounds on the grid, the tail on one cluster.  nnz: the
// entries, or (known = false) a stand-in for them.  The control block is cleared
// first.  Returns the launches, -1 if it cannot run.
static int peel_launches(PeelArgs a, int blocks, uint64_t nnz, bool known, cudaStream_t s) {
    if (cudaMemsetAsync(a.ctl, 0, sizeof(PeelCtl), s) != cudaSuccess) return -1;
    if (a.n <= kBlockVertices && nnz <= kBlockEntries) {
        const size_t lists = 3 * sizeof(uint32_t) * (size_t)a.n;
        const size_t all = lists + sizeof(uint32_t) * ((size_t)a.n + 1) + sizeof(uint16_t) * (size_t)nnz;
        if (known && all <= kBlockShared && allow_max_smem(k_peel_block<true>)) {
            k_peel_block<true><<<1, kPeelThreads, all, s>>>(a, (uint32_t)nnz);
            return 1;
        }
        if (allow_max_smem(k_peel_block<false>)) {
            k_peel_block<false><<<1, kPeelThreads, lists, s>>>(a, 0);
            return 1;
        }
    }
    int size = peel_cluster_size();
    const bool small = size && a.n <= kClusterVertices && nnz <= kClusterEntries;
    int launches = 0;
    if (!small) {
        a.handover = size ? kHandover : 0;
        void *args[] = {&a};
        if (blocks <= 0 || cudaLaunchCooperativeKernel((const void *)k_peel_grid, blocks, kPeelThreads, args, 0, s) !=
                               cudaSuccess)
            return -1;
        launches++;
        if (!size) return launches;
    } else {  // no more CTAs than 8 entries or one vertex a thread
        const uint64_t work = std::max<uint64_t>(a.n, nnz / 8);
        while (size > 1 && (uint64_t)(size / 2) * kPeelThreads >= work) size >>= 1;
    }
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    cluster_config(cfg, attr, size, s);
    if (cudaLaunchKernelEx(&cfg, k_peel_cluster, a, small ? 0 : 1) != cudaSuccess) return -1;
    return launches + 1;
}

int launch_peel(const kcl_graph *g, Workspace &w, cudaStream_t s) {
    const PeelArgs a{g->n, g->rp, g->col, w.alive, w.cdeg, reinterpret_cast<int *>(w.peel_deg), w.key,
                     w.frontier_a, w.frontier_b, w.peel, 0};
    return peel_launches(a, peel_blocks(g->num_sms, g->n), g->nnz, true, s);
}

int launch_orient(const kcl_graph *g, uint32_t k, Workspace &w, cudaStream_t s) {
    (void)k;
    int wgrid = grid_for((uint64_t)g->n * 32, kBlock, g->num_sms, 32);
    k_outdeg<<<wgrid, kBlock, 0, s>>>(g->n, g->rp, g->col, w.key, w.outdeg, w.take, w.res);
    // optr = exclusive scan of outdeg (n + 1 entries; outdeg[n] = 0)
    int l = 1 + launch_exclusive_scan(w.outdeg, w.optr, g->n + 1, w.scan_tmp, s);
    k_outfill<<<wgrid, kBlock, 0, s>>>(g->n, g->rp, g->col, w.key, w.take, w.optr, w.oadj);
    return l + 1;
}

int launch_roots(const kcl_graph *g, uint32_t k, Workspace &w, const uint32_t *class_limits, int n_classes,
                 const PeelCtl *peel, cudaStream_t s) {
    int grid = grid_for(g->n, kBlock, g->num_sms);
    // out-degrees are below n; those above the largest class need no order
    const uint32_t top = std::min<uint32_t>(g->n, KCL_MAX_OUTDEG + 2);
    const uint32_t H = top + 1;
    uint32_t *hist = w.hist, *offs = w.hist + H, *fill = w.hist + 2 * H;
    ClassLimits limits{};
    for (int c = 0; c < n_classes; c++) limits.d[c] = class_limits[c];
    cudaMemsetAsync(w.hist, 0, 3 * H * sizeof(uint32_t), s);
    k_root_hist<<<grid, kBlock, 0, s>>>(g->n, k, w.outdeg, top, hist, w.root_mask, w.kmap, w.res);
    int l = 1 + launch_exclusive_scan(hist, offs, H, w.scan_tmp, s);
    k_root_scatter<<<grid, kBlock, 0, s>>>(g->n, k, w.outdeg, top, offs, fill, w.root_mask, w.kmap, w.roots);
    k_class_bounds<<<1, 32, 0, s>>>(offs, top, limits, n_classes, peel, w.res);
    return l + 2;
}

}  // namespace kcl

// ======================================= allocation-free degeneracy ordering
// Scratch of kcl_degeneracy_order_noalloc: peel degrees, the removal order, the
// near list and the control block of the peel for up to KCL_NOALLOC_MAX_VERTICES vertices.
// It is a fixed device array, so the call never allocates; in host code the
// array's name is only a stand-in, and its device address is looked up with
// cudaGetSymbolAddress once per device.
static constexpr size_t kNoAllocWords =
    3 * (size_t)KCL_NOALLOC_MAX_VERTICES + sizeof(kcl::PeelCtl) / sizeof(uint32_t);
static __device__ __align__(256) uint32_t kcl_noalloc_scratch[kNoAllocWords];

namespace {
constexpr int kNoAllocMaxDevices = 64;
std::mutex noalloc_mu;
uint32_t *noalloc_ptr[kNoAllocMaxDevices];
int noalloc_blocks[kNoAllocMaxDevices];

// Device address of the scratch array and the cooperative grid size for the
// current device, set up on the first call on that device.
kcl_status noalloc_setup(uint32_t **ptr, int *blocks) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) {
        (void)cudaGetLastError();
        return KCL_ECUDA;
    }
    std::lock_guard<std::mutex> lock(noalloc_mu);
    if (!noalloc_ptr[dev]) {
        uint32_t *p = nullptr;
        if (cudaGetSymbolAddress((void **)&p, kcl_noalloc_scratch) != cudaSuccess || !p) {
            (void)cudaGetLastError();
            return KCL_ECUDA;
        }
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) {
            (void)cudaGetLastError();
            return KCL_ECUDA;
        }
        const int blocks = kcl::peel_blocks(sms, KCL_NOALLOC_MAX_VERTICES);
        if (blocks <= 0) return KCL_ECUDA;
        noalloc_blocks[dev] = blocks;
        noalloc_ptr[dev] = p;
    }
    *ptr = noalloc_ptr[dev];
    *blocks = noalloc_blocks[dev];
    return KCL_OK;
}
}  // namespace

extern "C" kcl_status kcl_degeneracy_order_noalloc(uint32_t n, const uint64_t *row_ptr,
                                                   const uint32_t *col, const uint8_t *alive,
                                                   const uint32_t *degree, uint32_t *round_out,
                                                   void *stream) {
    if (n > KCL_NOALLOC_MAX_VERTICES) return KCL_ESIZE;
    if (n == 0) return KCL_OK;
    if (!row_ptr || !col || !alive || !degree || !round_out) return KCL_EINVAL;
    uint32_t *S = nullptr;
    int blocks = 0;
    kcl_status st = noalloc_setup(&S, &blocks);
    if (st != KCL_OK) return st;
    uint64_t need = ((uint64_t)n + kcl::kPeelThreads - 1) / kcl::kPeelThreads;
    if (need < (uint64_t)blocks) blocks = (int)need;
    cudaStream_t s = (cudaStream_t)stream;
    kcl::PeelCtl *ctl = reinterpret_cast<kcl::PeelCtl *>(S + 3 * (size_t)KCL_NOALLOC_MAX_VERTICES);
    const kcl::PeelArgs a{n, row_ptr, col, alive, degree, reinterpret_cast<int *>(S), round_out,
                          S + KCL_NOALLOC_MAX_VERTICES, S + 2 * (size_t)KCL_NOALLOC_MAX_VERTICES, ctl, 0};
    // the entry count is on the device: only small n goes to one CTA (at most
    // n^2 entries) or to the cluster alone
    const uint64_t nnz = n <= 512 ? 0 : n <= 1u << 15 ? kcl::kBlockEntries + 1 : ~0ull;
    if (kcl::peel_launches(a, blocks, nnz, false, s) < 0) {
        (void)cudaGetLastError();
        return KCL_ECUDA;
    }
    unsigned err = 0;
    if (cudaMemcpyAsync(&err, &ctl->error, sizeof(err), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        (void)cudaGetLastError();
        return KCL_ECUDA;
    }
    return err ? KCL_ETIMEOUT : KCL_OK;
}
