// Id-ordered subproblems: counting and listing for k <= 6 and d+_u <= 1024,
// shared by both orderings.  The ordering fixes the DAG outside (degree or
// degeneracy, Algorithms 5 and 6); inside N+_u any acyclic orientation finds
// every clique once (Theorem 1 applied to the subgraph G_u), and these
// kernels orient G_u by vertex id, which is the index order N+_u already has:
// no ranks, no colouring, no re-indexing.  For small k the prunes those buy
// change little (switching the colour prune off moved the listing time of R-MAT
// 20 by under 2 %) while they took most of a root's build: on the 1M-vertex
// R-MAT graph the colour path's k = 3 count, which is all build, took 42.6 ms
// of listing kernels, here 11.8 ms.
//
// Candidate sets on skewed graphs are near-cliques (edge density 0.8-0.9 at
// 40-300 vertices on R-MAT 20), so the last levels work on dense matrices:
// the candidate set C of a node is compacted to its own |C| x |C| bit matrix
// (rows gathered by a parallel bit extract with masks shared by all rows) and
//   counting at level 3 is triangle counting on that matrix, every lane one
//     row q, every step one row p read as a broadcast: |row(q) & row(p)| for
//     the lanes with q in row(p), no queue and no bank conflicts;
//   listing at level 2 walks the matrix with the lanes on the smaller id a
//     and the row b uniform: the checksum's chain over R + {a} is computed
//     once per (node, a) and a clique costs one SplitMix64 round (two when
//     the root's own id is the largest) instead of k and a merge.
// Listing kernels of the 1M-vertex R-MAT graph (16 edges a vertex), before and
// now: k = 5 colour count 179.3 -> 42.4 ms, k = 4 colour listing 201.2 -> 97.0
// ms (2.06e10 records, 3.4 TB/s of stores; the stores alone would take 43 ms at
// the 7.7 TB/s that a fill writes here, the hashes alone 83).  Counting is bound by the ALU pipe, listing by
// issue slots around the hash round.  A kernel per k: with all of k = 3..6 in
// one, 45.0 and 106.0 ms (registers, instruction cache).
#include "kcl_internal.cuh"

namespace kcl {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// ------------------------------------------------------------- layouts
// Words of a row over D vertices (multiple of 4: rows are read as 128-bit
// vectors) and the row stride: an odd number of 16-byte chunks, so 8 lanes
// reading 8 consecutive rows hit 8 different bank quads.
__host__ __device__ inline uint32_t row_words4(uint32_t D) { return (((D + 31) >> 5) + 3) & ~3u; }
__host__ __device__ inline uint32_t row_stride(uint32_t W) { return ((W >> 2) & 1) ? W : W + 4; }

// Compact lower-triangular matrix in groups of G words: row i holds
// G (i / 32 G + 1) words, so rows are G-word aligned and most words above the
// diagonal take no room.  Counting reads rows as 128-bit vectors (G = 4), listing
// single words (G = 2, a third less room at 160 rows).
template <int G>
__host__ __device__ inline uint32_t tri_off(uint32_t i) {
    const uint32_t R = i / (32 * G);
    return 16 * G * G * R * (R + 1) + i % (32 * G) * G * (R + 1);
}
template <int G>
__host__ __device__ inline uint32_t tri_words(uint32_t c) { return tri_off<G>((c + 31) & ~31u); }

// Words a candidate set of c members takes in a warp's room: its ids (listing),
// its matrix, and its index list (u16) at the end.
__host__ __device__ inline uint32_t ids_words(uint32_t c, bool list) { return list ? (c + 3) & ~3u : 0u; }
__host__ __device__ inline uint32_t idx_words(uint32_t c) { return ((c + 7) >> 3) << 2; }
__host__ __device__ inline uint32_t set_room(uint32_t c, bool list) {
    return ids_words(c, list) + (((list ? tri_words<2>(c) : tri_words<4>(c)) + 3) & ~3u) + idx_words(c);
}

// Shared memory of one subproblem (words).  RS, LEN, HK, HV, BM and the queues
// belong to the build and are dead afterwards: the warps' scratch (X) overlays
// them.  Per warp: kBitmaps candidate bitmaps of W words, the extract masks
// (8 W) and the room of the compacted set.
constexpr uint32_t kBitmaps = 3;  // candidate sets of the path (k <= 6)
constexpr uint32_t kMetaDeadline = 2;  // META: unit, children taken, deadline (2 words)
constexpr uint32_t kQueue = 64;   // build: members found in a warp's out-lists, waiting for lookup
struct Lay {
    uint32_t D, W, WP, NBR, META, A, X, RS, LEN, HK, HV, BM, Q, per_warp, room, total;
};

__host__ __device__ inline uint32_t scratch_fixed(uint32_t W) { return (kBitmaps + 8) * W; }

__host__ __device__ inline Lay make_lay(uint32_t D, uint32_t nw, uint32_t room) {
    Lay L;
    const uint32_t T = hash_cap(D);
    L.D = D;
    L.W = row_words4(D);
    L.WP = row_stride(L.W);
    L.NBR = 0;
    L.META = D;                 // 8 words
    L.A = (L.META + 8 + 3) & ~3u;
    L.X = L.A + D * L.WP;
    L.RS = L.X;                 // starts of the members' out-lists
    L.LEN = L.RS + D;           // their lengths
    L.HK = L.LEN + D;           // hash keys
    L.HV = L.HK + T;            // hash values, u16
    L.BM = L.HV + T / 2;        // 16 T filter bits
    L.Q = L.BM + T / 2;         // per warp: kQueue ids, kQueue u16 rows
    L.room = room;
    L.per_warp = scratch_fixed(L.W) + room;
    const uint32_t build = 2 * D + 2 * T + nw * (kQueue + kQueue / 2);
    const uint32_t walk = nw * L.per_warp;
    L.total = L.X + (((build > walk ? build : walk) + 3) & ~3u);
    return L;
}

struct SubArgs {
    const uint32_t *optr, *oadj, *roots;
    uint32_t begin, end;   // root positions of the class
    uint32_t parts;        // CTA form: a root's children are shared by this many units
    unsigned *queue;
    uint32_t *gscratch;    // per-warp room in global memory (larger candidate sets), gwords each
    uint32_t gwords;
    uint32_t D, room, dfs_warps;
    uint32_t *ring;
    unsigned long long capacity;
    int wrap;
    const uint32_t *idmap;
    const uint8_t *kmap;
    unsigned long long *per_root, *root_cks;
    DevResult *res;
};

// A group working on one subproblem: one warp, or the whole CTA.
template <bool CTA>
struct Group {
    static __device__ __forceinline__ uint32_t size() { return CTA ? blockDim.x : 32u; }
    static __device__ __forceinline__ uint32_t tid() { return CTA ? threadIdx.x : lane_id(); }
    static __device__ __forceinline__ uint32_t warp() { return CTA ? threadIdx.x >> 5 : 0u; }
    static __device__ __forceinline__ void sync() {
        if (CTA) __syncthreads();
        else __syncwarp();
    }
};

// --------------------------------------------------------------- build
// A batch of nb <= 32 queued (id, row) pairs: looks the id up in the table of
// N+_u and records the edge.
enum Rows { kNoRows, kLower, kBoth };  // count only; row max(i, j) gets bit min(i, j); both bits
__device__ __forceinline__ uint32_t link(const uint32_t *qid, const uint16_t *qrow, uint32_t nb,
                                         const uint32_t *hk, const uint16_t *hv, uint32_t T, uint32_t shift,
                                         uint32_t *A, uint32_t WP, Rows rows) {
    const unsigned lane = lane_id();
    uint32_t hit = 0;
    if (lane < nb) {
        const int x = hash_find(hk, hv, T, shift, qid[lane]);
        if (x >= 0) {
            hit = 1;
            if (rows != kNoRows) {
                const uint32_t i = qrow[lane], j = (uint32_t)x;
                if (rows == kBoth) {
                    atomicOr(&A[i * WP + (j >> 5)], 1u << (j & 31));
                    atomicOr(&A[j * WP + (i >> 5)], 1u << (i & 31));
                } else {
                    const uint32_t hi = max(i, j), lo = min(i, j);
                    atomicOr(&A[hi * WP + (lo >> 5)], 1u << (lo & 31));
                }
            }
        }
    }
    return hit;
}

// Members N+_u (ascending ids) and the bit-rows of G_u over their indices.
// Each edge of G_u lies in exactly one of the members' DAG out-lists, of which
// about one entry in ten is a member (R-MAT 20): every entry is first tested
// against a bitmap of 16 bits per table slot (at most 1 in 32 set), one shared
// load, and only the survivors are queued and looked up in the hash table, 32
// at a time.  A warp reads its members' lists with 32 lanes a list, or 8 when
// they are short.  Testing every entry in the table itself, with the lists
// flattened over the lanes by a search in their prefix sums, took 2.9x as long
// (the k = 3 count of R-MAT 20: 27.6 ms).
template <bool CTA>
__device__ uint32_t build(uint32_t d, uint32_t base, const SubArgs &a, const Lay &L, uint32_t *S,
                          Rows rows) {
    using G = Group<CTA>;
    const uint32_t tid = G::tid(), lane = lane_id(), warp = G::warp(), nw = G::size() >> 5;
    uint32_t *nbr = S + L.NBR, *rs = S + L.RS, *len = S + L.LEN, *hk = S + L.HK, *bm = S + L.BM, *A = S + L.A;
    uint16_t *hv = reinterpret_cast<uint16_t *>(S + L.HV);
    uint32_t *qid = S + L.Q + warp * (kQueue + kQueue / 2);
    uint16_t *qrow = reinterpret_cast<uint16_t *>(qid + kQueue);
    uint32_t T, hshift;
    hash_size(d, &T, &hshift);
    for (uint32_t i = tid; i < T; i += G::size()) hk[i] = kHashEmpty;
    for (uint32_t i = tid; i < T / 2; i += G::size()) bm[i] = 0;
    if (rows != kNoRows) {
        uint4 *A4 = reinterpret_cast<uint4 *>(A);
        for (uint32_t i = tid; i < (d * L.WP) >> 2; i += G::size()) A4[i] = make_uint4(0, 0, 0, 0);
    }
    G::sync();
    for (uint32_t i = tid; i < d; i += G::size()) {
        const uint32_t v = a.oadj[base + i];
        nbr[i] = v;
        const uint32_t r0 = a.optr[v];
        rs[i] = r0;
        len[i] = a.optr[v + 1] - r0;
        const uint32_t b = hash_slot(v, hshift - 4);  // T >= 2, so 16 T bits fit 32
        atomicOr(&bm[b >> 5], 1u << (b & 31));
        uint32_t h = b >> 4;
        while (atomicCAS(&hk[h], kHashEmpty, v) != kHashEmpty) h = (h + 1) & (T - 1);
        hv[h] = (uint16_t)i;
    }
    G::sync();
    // this warp's members [m0, m1), and the lanes per list
    const uint32_t per = (d + nw - 1) / nw;
    const uint32_t m0 = min(warp * per, d), m1 = min(m0 + per, d);
    uint32_t sum = 0;
    for (uint32_t i = m0 + lane; i < m1; i += 32) sum += len[i];
    sum = __reduce_add_sync(kFull, sum);
    const uint32_t lg = sum >= 24 * (m1 - m0) ? 5 : 3;
    const uint32_t gl = lane & ((1u << lg) - 1u), step = 1u << lg;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t hits = 0, pend = 0;
    for (uint32_t i0 = m0; i0 < m1; i0 += 32 >> lg) {
        const uint32_t i = i0 + (lane >> lg);
        const uint32_t n = i < m1 ? len[i] : 0u;
        const uint32_t *list = a.oadj + (i < m1 ? rs[i] : 0u);
        const uint32_t most = lg == 5 ? n : __reduce_max_sync(kFull, n);
        for (uint32_t e0 = 0; e0 < most; e0 += 4 * step) {
            uint32_t w[4];
            bool in[4];
#pragma unroll
            for (int z = 0; z < 4; z++) {
                const uint32_t e = e0 + z * step + gl;
                in[z] = e < n;
                w[z] = in[z] ? list[e] : 0u;
            }
#pragma unroll
            for (int z = 0; z < 4; z++) {
                const uint32_t b = hash_slot(w[z], hshift - 4);
                const bool on = in[z] && ((bm[b >> 5] >> (b & 31)) & 1u);
                const unsigned bal = __ballot_sync(kFull, on);
                if (!bal) continue;
                if (on) {
                    const uint32_t at = pend + __popc(bal & lt);
                    qid[at] = w[z];
                    qrow[at] = (uint16_t)i;
                }
                pend += __popc(bal);
                if (pend >= 32) {
                    __syncwarp();
                    hits += link(qid, qrow, 32, hk, hv, T, hshift, A, L.WP, rows);
                    __syncwarp();
                    pend -= 32;
                    if (lane < pend) {
                        qid[lane] = qid[32 + lane];
                        qrow[lane] = qrow[32 + lane];
                    }
                    __syncwarp();
                }
            }
        }
    }
    __syncwarp();
    hits += link(qid, qrow, pend, hk, hv, T, hshift, A, L.WP, rows);
    G::sync();
    return hits;
}

// ---------------------------------------------------------- compaction
// A warp's scratch.
struct Scratch {
    uint32_t *cb;      // kBitmaps candidate bitmaps, W words each
    uint32_t *masks;   // extract masks, 8 words per bitmap word
    uint32_t *mem;     // room of the compacted set: ids, matrix, index list at the end
    uint32_t room;
    uint32_t *gmem;    // ids and matrix of larger sets, in global memory
    __device__ __forceinline__ uint16_t *idx(uint32_t c, bool fits) const {
        return reinterpret_cast<uint16_t *>(fits ? mem + room - idx_words(c) : mem);
    }
};

// Members of the bitmap C (words w0 .. nw - 1) in ascending order.
__device__ __forceinline__ void index_list(const uint32_t *C, uint32_t w0, uint32_t nw, uint16_t *idx) {
    const unsigned lane = lane_id(), lt = (1u << lane) - 1u;
    uint32_t base = 0;
    for (uint32_t t = w0; t < nw; t++) {
        const uint32_t m = C[t];
        if ((m >> lane) & 1u) idx[base + __popc(m & lt)] = (uint16_t)(t * 32 + lane);
        base += __popc(m);
    }
    __syncwarp();
}

// Extract masks of each word of C: moving the bits of a word selected by m to
// its low end in five steps of 1, 2, 4, 8, 16 places (the compress of Warren,
// Hacker's Delight 7-4).  A step needs only the destination bits of the moves,
// x = dest ? x >> s : x, because bits outside the selected set are never
// looked at again.  The masks depend on C alone and serve every row.
__device__ __forceinline__ void extract_masks(const uint32_t *C, uint32_t nw, uint32_t *masks) {
    const unsigned lane = lane_id();
    if (lane < nw) {
        uint32_t m = C[lane], mv[5];
        const uint32_t cnt = __popc(m);
        uint32_t mk = ~m << 1;
#pragma unroll
        for (int i = 0; i < 5; i++) {
            uint32_t mp = mk ^ (mk << 1);
            mp ^= mp << 2;
            mp ^= mp << 4;
            mp ^= mp << 8;
            mp ^= mp << 16;
            const uint32_t mm = mp & m;
            mv[i] = mm >> (1 << i);
            m = (m ^ mm) | mv[i];
            mk &= ~mp;
        }
        uint4 *M = reinterpret_cast<uint4 *>(masks) + 2 * lane;
        M[0] = make_uint4(mv[0], mv[1], mv[2], mv[3]);
        M[1] = make_uint4(mv[4], cnt, cnt ? kFull >> (32 - cnt) : 0u, 0u);
    }
    __syncwarp();
}

__device__ __forceinline__ uint32_t pick(uint32_t sel, uint32_t a, uint32_t b) { return (sel & a) | (~sel & b); }

// The rows of C's members restricted to C, as a lower-triangular bit matrix
// over C's own indices (bits below the diagonal).  32 rows at a time, a lane per
// row: the row's words are read as 128-bit vectors, each is extracted by C's
// masks and appended to the lane's output; all lanes append the same number of
// bits, so the bookkeeping is uniform.  Returns the lane's number of set bits.
template <int G>
__device__ uint32_t compact(const uint32_t *A, uint32_t WP, uint32_t c, const uint32_t *masks,
                            const uint16_t *idx, uint32_t *out) {
    const unsigned lane = lane_id(), lt = (1u << lane) - 1u;
    const uint32_t tbeg = (idx[0] >> 7) << 2;
    uint32_t sum = 0;
    for (uint32_t r = 0; r * 32 < c; r++) {
        const uint32_t i = r * 32 + lane;
        const bool act = i < c;
        const uint4 *row = reinterpret_cast<const uint4 *>(A + (uint32_t)idx[act ? i : c - 1] * WP);
        const uint32_t tend = (idx[min(r * 32 + 31, c - 1)] >> 5) + 1;
        uint32_t *o = out + tri_off<G>(i);
        uint32_t lo = 0, ow = 0, sh = 0;
        auto put = [&]() {  // the next output word; words above the diagonal are dropped
            if (ow <= r) {
                uint32_t w = act ? lo : 0u;
                if (ow == r) w &= lt;
                o[ow] = w;
                sum += __popc(w);
            }
            ow++;
        };
        for (uint32_t t0 = tbeg; t0 < tend; t0 += 4) {
            const uint4 v = row[t0 >> 2];
#pragma unroll
            for (uint32_t z = 0; z < 4; z++) {
                if (t0 + z >= tend) break;
                const uint4 *M = reinterpret_cast<const uint4 *>(masks) + 2 * (t0 + z);
                const uint4 m1 = M[1];
                if (m1.y == 0) continue;
                const uint4 m0 = M[0];
                uint32_t x = z == 0 ? v.x : z == 1 ? v.y : z == 2 ? v.z : v.w;
                x = pick(m0.x, x >> 1, x);
                x = pick(m0.y, x >> 2, x);
                x = pick(m0.z, x >> 4, x);
                x = pick(m0.w, x >> 8, x);
                x = pick(m1.x, x >> 16, x) & m1.z;
                lo |= x << sh;
                sh += m1.y;
                if (sh >= 32) {
                    sh -= 32;
                    put();
                    lo = __funnelshift_rc(x, 0u, m1.y - sh);  // the m1.y - sh bits already stored leave
                }
            }
        }
        if (ow <= r) put();
    }
    __syncwarp();
    return sum;
}

// ---------------------------------------------------- triangle counting
__device__ __forceinline__ uint32_t lop_and3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0x80;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}
__device__ __forceinline__ uint32_t lop_xor3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0x96;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}
__device__ __forceinline__ uint32_t lop_maj(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xE8;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}
// Rows p0..p1 (both even) against the lanes' rows (words 4 g .. 4 g + NWD - 1
// of row q in qv): lane q adds |row(q) & row(p)| over those words when bit q
// of row p is set (word b of row p; LAST: b is the group's last word).  Bits
// are summed through a carry-save adder, two rows at a time: POPC runs at a
// quarter of LOP3's rate and is needed only for the carries (weight 2).
template <int NWD, bool LAST, int UNROLL>
__device__ __forceinline__ void tri_rows(const uint32_t *M, uint32_t b, uint32_t g, uint32_t p0, uint32_t p1,
                                         const uint4 &qv, uint32_t &ones, uint32_t &twos) {
    // 2^(31 - lane), opaque to the compiler: moving bit `lane` to the sign is
    // then a multiply, off the ALU pipe that bounds this loop
    uint32_t up;
    asm("shl.b32 %0, %1, %2;" : "=r"(up) : "r"(1u), "r"(31u - lane_id()));
    const uint32_t q[4] = {qv.x, qv.y, qv.z, qv.w};
    for (uint32_t p = p0; p < p1;) {
        const uint32_t R = p >> 7, stride = 4 * (R + 1);
        const uint32_t end = min(p1, (R + 1) << 7);
        const uint32_t *rp = M + tri_off<4>(p) + 4 * g;
#pragma unroll UNROLL
        for (; p < end; p += 2, rp += 2 * stride) {
            const uint4 av = *reinterpret_cast<const uint4 *>(rp);
            const uint4 bv = *reinterpret_cast<const uint4 *>(rp + stride);
            const uint32_t x[4] = {av.x, av.y, av.z, av.w}, y[4] = {bv.x, bv.y, bv.z, bv.w};
            const uint32_t ea = LAST ? x[NWD - 1] : rp[b - 4 * g];
            const uint32_t eb = LAST ? y[NWD - 1] : rp[stride + b - 4 * g];
            const uint32_t ma = (uint32_t)((int32_t)(ea * up) >> 31);
            const uint32_t mb = (uint32_t)((int32_t)(eb * up) >> 31);
#pragma unroll
            for (int w = 0; w < NWD; w++) {
                const uint32_t s = lop_and3(q[w], x[w], ma), t = lop_and3(q[w], y[w], mb);
                twos += __popc(lop_maj(ones, s, t));
                ones = lop_xor3(ones, s, t);
            }
        }
    }
}

// Triangles of the compact matrix M over c vertices (lane's share).
template <int UNROLL>
__device__ uint32_t tri_matrix(const uint32_t *M, uint32_t c) {
    const unsigned lane = lane_id();
    const uint32_t nb = (c + 31) >> 5, rows = (c + 1) & ~1u;
    uint32_t ones = 0, twos = 0;
    for (uint32_t b = 0; b < nb; b++) {
        const uint32_t *rq = M + tri_off<4>(b * 32 + lane);
        const uint32_t last = b >> 2;
        for (uint32_t g = 0; g < last; g++)
            tri_rows<4, false, UNROLL>(M, b, g, b * 32, rows, *reinterpret_cast<const uint4 *>(rq + 4 * g), ones, twos);
        const uint4 qv = *reinterpret_cast<const uint4 *>(rq + 4 * last);
        switch (b & 3) {
            case 0: tri_rows<1, true, UNROLL>(M, b, last, b * 32, rows, qv, ones, twos); break;
            case 1: tri_rows<2, true, UNROLL>(M, b, last, b * 32, rows, qv, ones, twos); break;
            case 2: tri_rows<3, true, UNROLL>(M, b, last, b * 32, rows, qv, ones, twos); break;
            default: tri_rows<4, true, UNROLL>(M, b, last, b * 32, rows, qv, ones, twos);
        }
    }
    return 2 * twos + __popc(ones);
}

// Triangles of G_u within the candidate set C (nw words, c members; A holds
// the bits below the diagonal).  Up to 32 members the rows fit one word: each
// row is gathered by a ballot (lane j tests bit idx[j]) and met at once with
// the rows before it, which the lanes hold.  The sum stays 32-bit: c <= 1024.
__device__ uint32_t tri_count(const uint32_t *A, uint32_t WP, const uint32_t *C, uint32_t nw, uint32_t c,
                              const Scratch &sc) {
    const unsigned lane = lane_id();
    if (c < 3) return 0;
    const bool fits = set_room(c, false) <= sc.room;
    uint16_t *idx = sc.idx(c, fits);
    index_list(C, 0, nw, idx);
    if (c <= 32) {
        // lanes beyond c look at the last member's bit, zero in every row
        const uint32_t me = idx[min(lane, c - 1)];
        const uint32_t *col = A + (me >> 5);
        const uint32_t sh = me & 31u;
        uint32_t mine = 0, acc = 0;
#pragma unroll 4
        for (uint32_t i = 1; i < c; i++) {
            const uint32_t p = __shfl_sync(kFull, me, i);
            const uint32_t w = col[p * WP] >> sh;
            const uint32_t row = __ballot_sync(kFull, w & 1u);
            if (w & 1u) acc += __popc(row & mine);
            if (lane == i) mine = row;
        }
        __syncwarp();
        return acc;
    }
    extract_masks(C, nw, sc.masks);
    uint32_t acc;
    if (fits) {
        compact<4>(A, WP, c, sc.masks, idx, sc.mem);
        acc = tri_matrix<2>(sc.mem, c);
    } else {
        compact<4>(A, WP, c, sc.masks, idx, sc.gmem);
        acc = tri_matrix<2>(sc.gmem, c);
    }
    __syncwarp();
    return acc;
}

// k = 4 counting: sum over p in row v of |row(p) & row(v)|, 32 candidates to
// a batch; rows hold only lower bits, so a batch reads words up to its
// largest p.
__device__ uint32_t pair_count(const uint32_t *A, uint32_t WP, const uint32_t *C, uint32_t nw, uint32_t c,
                               const Scratch &sc) {
    const unsigned lane = lane_id();
    if (c < 2) return 0;
    uint16_t *idx = sc.idx(c, false);
    index_list(C, 0, nw, idx);
    uint32_t acc = 0;
    const uint4 *c4 = reinterpret_cast<const uint4 *>(C);
    for (uint32_t i0 = 0; i0 < c; i0 += 32) {
        const uint32_t i = i0 + lane;
        const uint32_t p = idx[min(i, c - 1)];
        const uint32_t nc = ((uint32_t)idx[min(i0 + 31, c - 1)] >> 7) + 1;
        const uint4 *row = reinterpret_cast<const uint4 *>(A + p * WP);
        uint32_t x = 0;
        for (uint32_t t = 0; t < nc; t++) {
            const uint4 r = row[t], m = c4[t];
            x += __popc(r.x & m.x) + __popc(r.y & m.y) + __popc(r.z & m.z) + __popc(r.w & m.w);
        }
        acc += i < c ? x : 0u;
    }
    __syncwarp();
    return acc;
}

// -------------------------------------------------------------- listing
// Where a node's records go: `total` consecutive record indices from pos.
// NONE: no ring (checksum only); FAST: every record lands below the ring's
// end and its vector stores are aligned; SLOW: each record is placed by itself.
enum class Ring { NONE, FAST, SLOW };
struct Slots {
    unsigned long long pos;  // first record index (mod capacity when the ring wraps)
    Ring mode;
};

// Claims `total` records and says where they go.
template <int K>
__device__ __forceinline__ Slots claim(uint32_t total, const SubArgs &a) {
    Slots s{0ull, Ring::NONE};
    if (!a.ring) return s;
    if (lane_id() == 0) s.pos = atomicAdd(&a.res->emitted, (unsigned long long)total);
    s.pos = __shfl_sync(kFull, s.pos, 0);
    if (a.wrap) s.pos %= a.capacity;
    constexpr uintptr_t align = K == 4 ? 16u : K == 6 ? 8u : 4u;  // put_record's vector stores
    const bool aligned = (reinterpret_cast<uintptr_t>(a.ring) & (align - 1)) == 0;
    s.mode = aligned && s.pos + total <= a.capacity ? Ring::FAST : Ring::SLOW;
    return s;
}

// Writes a record where `on` holds: predicated stores, so the lanes of a row
// need no branch.
template <int K>
__device__ __forceinline__ void put_record(uint32_t *out, const uint32_t (&x)[K], bool on) {
    const uint32_t p = on;
    if constexpr (K == 4) {
        asm volatile("{.reg .pred p; setp.ne.u32 p, %5, 0; @p st.global.v4.u32 [%0], {%1, %2, %3, %4};}"
                     :: "l"(out), "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(p) : "memory");
    } else if constexpr (K == 6) {
        asm volatile("{.reg .pred p; setp.ne.u32 p, %7, 0; @p st.global.v2.u32 [%0], {%1, %2};"
                     " @p st.global.v2.u32 [%0+8], {%3, %4}; @p st.global.v2.u32 [%0+16], {%5, %6};}"
                     :: "l"(out), "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(p)
                     : "memory");
    } else {
#pragma unroll
        for (int z = 0; z < K; z++)
            asm volatile("{.reg .pred p; setp.ne.u32 p, %2, 0; @p st.global.u32 [%0], %1;}"
                         :: "l"(out + z), "r"(x[z]), "r"(p) : "memory");
    }
}

// Rows b0, b0 + bstep, ... below bend of matrix word t: lane a's cliques with
// each row b that holds a.  x: the clique's ids but id(b), which goes to x[AT];
// h: the chain over the ids before it; TAIL: u follows it (one more round).
// 32 rows' words and ids are loaded at once, a lane each, and handed out by
// shuffles, so the row loop waits for no load (larger sets' matrices are in
// global memory).  pos / wp: the node's next record index and its address.
template <int K, bool DIRECT, Ring MODE, bool TAIL>
__device__ __forceinline__ void list_rows(const uint32_t *M, uint32_t WP, uint32_t t, uint32_t b0, uint32_t bend,
                                          uint32_t bstep, const uint32_t *cid, uint64_t h, uint32_t (&x)[K],
                                          uint32_t u, const SubArgs &a, unsigned long long &pos,
                                          uint32_t *&wp, unsigned long long &cks) {
    constexpr int AT = TAIL ? K - 2 : K - 1;
    const unsigned lane = lane_id(), me = 1u << lane, lt = me - 1u;
    for (; b0 < bend; b0 += 32 * bstep) {
        const uint32_t bl = b0 + lane * bstep;
        uint32_t mw = 0, idw = 0;
        if (bl < bend) {
            mw = M[(DIRECT ? bl * WP : tri_off<2>(bl)) + t];
            if (DIRECT && (bl >> 5) == t) mw &= (1u << (bl & 31)) - 1u;
            idw = cid[bl];
        }
        const uint32_t nrow = min(32u, (bend - b0 + bstep - 1) / bstep);
#pragma unroll 1
        for (uint32_t j = 0; j < nrow; j++) {
            const uint32_t m = __shfl_sync(kFull, mw, j), idb = __shfl_sync(kFull, idw, j);
            uint64_t hb = mix64(h ^ (uint64_t)idb);
            if (TAIL) hb = mix64(hb ^ (uint64_t)u);
            const bool on = (m & me) != 0;
            cks += on ? hb : 0ull;
            if (MODE != Ring::NONE) {
                const uint32_t rank = __popc(m & lt);
                x[AT] = idb;
                if (MODE == Ring::FAST) {
                    put_record<K>(wp + rank * K, x, on);
                    wp += __popc(m) * K;
                } else {
                    unsigned long long s = pos + rank;
                    if (a.wrap) s %= a.capacity;
                    if (on && s < a.capacity) {
#pragma unroll
                        for (int z = 0; z < K; z++) a.ring[s * K + z] = x[z];
                    }
                    pos += __popc(m);
                }
            }
        }
    }
}

// The cliques {u} + path + {a, b}: a < b members of the candidate set (ids
// cid[0..c), ascending, all above the path's ids), row(b) of the matrix
// holding the a's.  Rows b = b0, b0 + bstep, ... are taken by this warp.
// The lanes hold 32 a's; b is uniform, and so is the place of u against b:
//   b > u: the chain over path + {u, a} is ready, one round closes the clique;
//   b < u: the chain over path + {a}, then rounds b and u.
// cu: number of members with an id below u.  DIRECT: M is the subproblem's
// own symmetric rows (stride WP), else a compact lower-triangular matrix.
template <int K, bool DIRECT, Ring MODE>
__device__ void list_matrix(const uint32_t *M, uint32_t WP, uint32_t c, const uint32_t *cid, uint32_t cu,
                            const uint32_t *path, uint32_t u, uint32_t b0, uint32_t bstep,
                            const SubArgs &a, unsigned long long pos, unsigned long long &cks) {
    constexpr int NP = K - 3;
    const unsigned lane = lane_id();
    uint32_t pv[NP + 1], qv[NP + 1];  // path; path with u inserted
    uint64_t hp = hash_seed(K), hq = hp;
    uint32_t pend = u;  // u moves up until it meets a larger id
#pragma unroll
    for (int i = 0; i < NP; i++) {
        pv[i] = path[i];
        qv[i] = min(pv[i], pend);
        pend = max(pv[i], pend);
        hp = mix64(hp ^ (uint64_t)pv[i]);
        hq = mix64(hq ^ (uint64_t)qv[i]);
    }
    qv[NP] = pend;
    hq = mix64(hq ^ (uint64_t)pend);
    uint32_t *wp = MODE == Ring::FAST ? a.ring + pos * K : nullptr;
    for (uint32_t t = 0; t * 32 + 1 < c; t++) {
        const uint32_t ai = t * 32 + lane;
        const uint32_t ida = cid[min(ai, c - 1)];
        uint32_t b = b0;  // first row of this warp above the block's first a
        if (b < t * 32) b += (t * 32 - b + bstep - 1) / bstep * bstep;
        uint32_t x[K];
        uint64_t h = mix64(hp ^ (uint64_t)ida);
#pragma unroll
        for (int i = 0; i < NP; i++) x[i] = pv[i];
        x[NP] = ida;
        if (b < cu) {
            x[K - 1] = u;
            list_rows<K, DIRECT, MODE, true>(M, WP, t, b, min(cu, c), bstep, cid, h, x, u, a, pos, wp, cks);
            b += (cu - b + bstep - 1) / bstep * bstep;
        }
        if (ai < cu) {  // a < u
            h = mix64(h ^ (uint64_t)u);
            x[NP + 1] = u;
        } else {
            h = mix64(hq ^ (uint64_t)ida);
#pragma unroll
            for (int i = 0; i <= NP; i++) x[i] = qv[i];
            x[NP + 1] = ida;
        }
        list_rows<K, DIRECT, MODE, false>(M, WP, t, b, c, bstep, cid, h, x, u, a, pos, wp, cks);
    }
}

template <int K, bool DIRECT>
__device__ __forceinline__ void list_by_mode(const uint32_t *M, uint32_t WP, uint32_t c, const uint32_t *cid,
                                             uint32_t cu, const uint32_t *path, uint32_t u, uint32_t b0,
                                             uint32_t bstep, const SubArgs &a, uint32_t total,
                                             unsigned long long &cks) {
    const Slots sl = claim<K>(total, a);
    if (sl.mode == Ring::FAST)
        list_matrix<K, DIRECT, Ring::FAST>(M, WP, c, cid, cu, path, u, b0, bstep, a, sl.pos, cks);
    else if (sl.mode == Ring::NONE)
        list_matrix<K, DIRECT, Ring::NONE>(M, WP, c, cid, cu, path, u, b0, bstep, a, sl.pos, cks);
    else
        list_matrix<K, DIRECT, Ring::SLOW>(M, WP, c, cid, cu, path, u, b0, bstep, a, sl.pos, cks);
}

// Level-2 node: lists the cliques closed by the edges of G_u within C.
template <int K>
__device__ void list_node(const uint32_t *A, uint32_t WP, const uint32_t *C, uint32_t w0, uint32_t nw, uint32_t c,
                          const uint32_t *nbr, uint32_t ru, const uint32_t *path, uint32_t u,
                          const Scratch &sc, const SubArgs &a, unsigned long long &cnt,
                          unsigned long long &cks) {
    const unsigned lane = lane_id();
    const bool fits = set_room(c, true) <= sc.room;
    uint16_t *idx = sc.idx(c, fits);
    index_list(C, w0, nw, idx);
    extract_masks(C, nw, sc.masks);
    uint32_t *ids = fits ? sc.mem : sc.gmem;
    uint32_t *M = ids + ids_words(c, true);
    uint32_t cu = 0;  // members with an id below u: those with an index below ru
    for (uint32_t i = lane; i < c; i += 32) {
        const uint32_t x = idx[i];
        cu += x < ru ? 1u : 0u;
        ids[i] = nbr[x];
    }
    cu = __reduce_add_sync(kFull, cu);
    const uint32_t mine = compact<2>(A, WP, c, sc.masks, idx, M);
    cnt += mine;
    const uint32_t total = __reduce_add_sync(kFull, mine);
    if (total) list_by_mode<K, false>(M, 0, c, ids, cu, path, u, 1, 1, a, total, cks);
    __syncwarp();
}

// ------------------------------------------------------------------ walk
// Where paths are two and more vertices long (k = 6 counting, k >= 5 listing) a
// first-level child is a big unit: in the classes of few, large roots its own
// children are dealt out in kSlices shares (d+ 257..354 of the 131k-vertex R-MAT
// graph at k = 6: 16.0 -> 12.7 ms; in the smaller classes it cost 4 to 16 %).
constexpr uint32_t kSlices = 4;
struct Sub {
    const uint32_t *A, *nbr;
    uint32_t WP, W, d, u, ru;
    uint32_t slice, slices;  // the share of a first-level child's own children this walk takes
};

// The call's time limit, checked at every node that is walked (a first-level child
// alone can take 50 ms: near-complete graph of 600 vertices, k = 6 listing).  The
// deadline lies behind the members in shared memory, where it takes no registers,
// and without a limit one uniform branch is all that is done.
__device__ __forceinline__ bool late(const Sub &s, const SubArgs &a) {
    const unsigned long long d = *reinterpret_cast<const unsigned long long *>(s.nbr + a.D + kMetaDeadline);
    return d && warp_past_deadline(d, a.res);
}

// Candidate set of path vertex w below C (C null: all of N+_u): row(w) & C,
// restricted to indices above w when rows are symmetric (UP).  Returns its size.
template <bool UP>
__device__ __forceinline__ uint32_t next_set(const Sub &s, const uint32_t *C, uint32_t w, uint32_t *out) {
    const unsigned lane = lane_id();
    uint32_t x = 0;
    if (lane < s.W) {
        x = s.A[w * s.WP + lane];
        if (C) x &= C[lane];
        if (UP) {
            if (lane < (w >> 5)) x = 0;
            else if (lane == (w >> 5)) x &= ~((2u << (w & 31)) - 1u);
        }
        out[lane] = x;
    }
    __syncwarp();
    return __reduce_add_sync(kFull, __popc(x));
}

// The subtree of a node with J path vertices below the root, the last one
// `last`, and candidate set C (bitmap J - 1, c members).  Counting ends in
// tri_count at level 3 (J = K - 4) or pair_count (K = 4), listing in list_node at
// level 2 (J = K - 3).
template <int K, int J, bool LIST>
__device__ void walk(const Sub &s, uint32_t last, uint32_t c, uint32_t *path, const Scratch &sc,
                     const SubArgs &a, unsigned long long &cnt, unsigned long long &cks) {
    const uint32_t *C = sc.cb + (J - 1) * s.W;
    // words that can be non-zero: rows hold bits below the diagonal (counting),
    // or both sides and a path ascends (listing)
    const uint32_t w0 = LIST ? last >> 5 : 0u;
    const uint32_t nw = LIST ? (s.d + 31) >> 5 : (last >> 5) + 1;
    if constexpr (LIST && J == K - 3) {
        list_node<K>(s.A, s.WP, C, w0, nw, c, s.nbr, s.ru, path, s.u, sc, a, cnt, cks);
    } else if constexpr (!LIST && K == 4) {
        cnt += pair_count(s.A, s.WP, C, nw, c, sc);
    } else if constexpr (!LIST && J == K - 4) {
        cnt += tri_count(s.A, s.WP, C, nw, c, sc);
    } else {
        uint32_t *Cn = sc.cb + J * s.W;
        uint32_t at = 0;
        for (uint32_t t = w0; t < nw; t++) {
            uint32_t m = C[t];
            while (m) {
                const uint32_t w = t * 32 + (__ffs(m) - 1);
                m &= m - 1;
                if (J == 1 && at++ % s.slices != s.slice) continue;
                const uint32_t n = next_set<LIST>(s, C, w, Cn);
                if (n + J + 2 >= K) {  // K - J - 2 more vertices needed
                    if (late(s, a)) return;
                    if (LIST) path[J] = s.nbr[w];
                    walk<K, J + 1, LIST>(s, w, n, path, sc, a, cnt, cks);
                }
                __syncwarp();
            }
        }
    }
}

// First-level child v of the root.
template <int K, bool LIST>
__device__ void child(const Sub &s, uint32_t v, const Scratch &sc, const SubArgs &a, unsigned long long &cnt,
                      unsigned long long &cks) {
    const uint32_t n = next_set<LIST>(s, nullptr, v, sc.cb);
    if (n + 2 >= K) {
        uint32_t path[4];
        path[0] = LIST ? s.nbr[v] : 0u;
        walk<K, 1, LIST>(s, v, n, path, sc, a, cnt, cks);
    }
    __syncwarp();
}

// k = 3 listing: the edges of G_u, rows shared out to nw warps.
__device__ void list_edges(const Sub &s, uint32_t warp, uint32_t nw, const SubArgs &a,
                           unsigned long long &cnt, unsigned long long &cks) {
    const unsigned lane = lane_id();
    uint32_t mine = 0;
    for (uint32_t b = warp; b < s.d; b += nw) {
        uint32_t x = lane <= (b >> 5) ? s.A[b * s.WP + lane] : 0u;
        if (lane == (b >> 5)) x &= (1u << (b & 31)) - 1u;
        mine += __popc(x);
    }
    cnt += mine;
    const uint32_t total = __reduce_add_sync(kFull, mine);
    if (total) list_by_mode<3, true>(s.A, s.WP, s.d, s.nbr, s.ru, nullptr, s.u, warp, nw, a, total, cks);
}

__device__ __forceinline__ void attribute(unsigned long long mine, unsigned long long *dst) {
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(kFull, mine, o);
    if (lane_id() == 0 && mine) atomicAdd(dst, mine);
}

// ---------------------------------------------------------------- kernel
// CTA: one root (or one of `parts` shares of its children) per CTA, built by
// all warps, first-level children handed out to the warps, the ones with the
// most candidates first.  Else one root per warp.
// KK: the launch's k, or 0 for a batch whose roots have their own (a kernel per
// k keeps each one's code, and its share of the instruction cache, to its leaf).
template <bool CTA, bool LIST, int KK>
__device__ __forceinline__ void run(const SubArgs &a) {
    extern __shared__ __align__(16) uint32_t smem[];
    using G = Group<CTA>;
    const unsigned lane = lane_id();
    const uint32_t wib = threadIdx.x >> 5, nwarps = CTA ? blockDim.x >> 5 : 1u;
    const Lay L = make_lay(a.D, nwarps, a.room);
    uint32_t *S = CTA ? smem : smem + wib * L.total;
    uint32_t *meta = S + L.META;
    uint32_t *x = S + L.X + (CTA ? wib * L.per_warp : 0u);
    Scratch sc;
    sc.cb = x;
    sc.masks = x + kBitmaps * L.W;
    sc.mem = x + scratch_fixed(L.W);
    sc.room = L.room;
    sc.gmem = a.gscratch + (size_t)(blockIdx.x * (blockDim.x >> 5) + wib) * a.gwords;
    const uint32_t units = (a.end - a.begin) * a.parts;
    const uint32_t nd = CTA && a.dfs_warps && a.dfs_warps < nwarps ? a.dfs_warps : nwarps;
    unsigned long long &deadline = *reinterpret_cast<unsigned long long *>(meta + kMetaDeadline);
    if (G::tid() == 0) deadline = __ldcg(&a.res->deadline_ns);
    G::sync();
    unsigned long long cnt = 0, cks = 0;
    for (;;) {
        uint32_t unit;
        if (CTA) {
            if (threadIdx.x == 0) meta[0] = past_deadline(deadline, a.res) ? units : atomicAdd(a.queue, 1u);
            __syncthreads();
            unit = meta[0];
            if (threadIdx.x == 0) meta[1] = 0;  // children taken; published by the build's barriers
        } else {
            if (warp_past_deadline(deadline, a.res)) break;
            unit = 0;
            if (lane == 0) unit = atomicAdd(a.queue, 1u);
            unit = __shfl_sync(kFull, unit, 0);
        }
        if (unit >= units) break;
        const uint32_t part = unit % a.parts;
        const uint32_t u = a.roots[a.begin + unit / a.parts];
        const uint32_t k = KK ? (uint32_t)KK : (uint32_t)a.kmap[u];
        const uint32_t base = a.optr[u], d = a.optr[u + 1] - base;
        const unsigned long long before = cnt, before_cks = cks;
        // a k = 3 root has no children to share: its first unit does all of it
        const bool skip = k == 3 && part > 0;
        if (!skip) {
            const Rows rows = LIST ? kBoth : k > 3 ? kLower : kNoRows;
            const uint32_t hits = build<CTA>(d, base, a, L, S, rows);
            Sub s{S + L.A, S + L.NBR, L.WP, L.W, d, u, 0u, 0u, 1u};
            if (LIST) {
                uint32_t below = 0;  // members with an id below u
                for (uint32_t i = lane; i < d; i += 32) below += s.nbr[i] < u ? 1u : 0u;
                s.ru = __reduce_add_sync(kFull, below);
                if (a.idmap) {  // output ids of a batch's union: monotone within a graph
                    G::sync();
                    for (uint32_t i = G::tid(); i < d; i += G::size()) S[L.NBR + i] = a.idmap[S[L.NBR + i]];
                    s.u = a.idmap[u];
                    G::sync();
                }
            }
            if (k == 3) {
                if (LIST) list_edges(s, G::warp(), nwarps, a, cnt, cks);
                else cnt += hits;
            } else if (G::warp() < nd) {
                // the part's children, the ones with the most candidates first
                const uint32_t nch = part < d ? (d - 1 - part) / a.parts + 1 : 0u;
                if (CTA && a.D > 256 && (LIST ? k > 4 : k > 5)) s.slices = kSlices;
                uint32_t i = 0;
                for (;; i++) {
                    if (CTA) {
                        if (lane == 0) i = atomicAdd(&meta[1], 1u);
                        i = __shfl_sync(kFull, i, 0);
                    }
                    if (i >= nch * s.slices || late(s, a)) break;
                    const uint32_t v = LIST ? part + i / s.slices * a.parts : d - 1 - part - i / s.slices * a.parts;
                    s.slice = i % s.slices;
                    if (k == 4) child<4, LIST>(s, v, sc, a, cnt, cks);
                    else if (k == 5) child<5, LIST>(s, v, sc, a, cnt, cks);
                    else child<6, LIST>(s, v, sc, a, cnt, cks);
                }
            }
            if (a.per_root) attribute(cnt - before, &a.per_root[u]);
            if (LIST && a.root_cks) attribute(cks - before_cks, &a.root_cks[u]);
        }
        G::sync();
    }
    for (int o = 16; o > 0; o >>= 1) {
        cnt += __shfl_down_sync(kFull, cnt, o);
        cks += __shfl_down_sync(kFull, cks, o);
    }
    if (lane == 0) {
        add_count(&a.res->count, &a.res->count_carry, cnt);
        if (LIST && cks) atomicAdd(&a.res->checksum, cks);
    }
}

template <bool LIST, int KK>
__global__ void __launch_bounds__(512, 2) k_sub_cta(const __grid_constant__ SubArgs a) {
    run<true, LIST, KK>(a);
}
template <int KK>
__global__ void __launch_bounds__(128, 8) k_sub_warp(const __grid_constant__ SubArgs a) {
    run<false, false, KK>(a);
}

// -------------------------------------------------------------- host side
constexpr uint32_t kLimits[] = {32, 64, 128, 256, 512, 1024};  // the classes of both orderings
constexpr int kSubClasses = 6;
constexpr int kWarpClasses = 3;
constexpr size_t kHalfSM = 112 * 1024;  // two CTAs per SM
constexpr size_t kFullSM = 220 * 1024;

struct Cfg {
    uint32_t D, warps, room, gwords;
    size_t smem;
    uint32_t per_sm;  // CTAs per SM the global room is sized for
};

// Whether class c runs a CTA per root.  Listing hashes every clique, and at k = 6
// a root's cost grows with the square of its near-cliques: one warp on the
// heaviest root then outlasts the launch (d+ 65..128 of the 131k-vertex R-MAT
// graph: a warp per root 19.6 ms, a CTA 3.7; d+ 33..64 2.1 and 0.75).  Up to k =
// 5 the warp form is the faster one up to d+ = 128 (3.5 against 3.6 ms on 1M
// vertices), and up to d+ = 32 always (the community graph's 292,000 roots at k =
// 6: 0.9 against 1.5 ms).
bool cta_form(int c, uint32_t k, bool listing) { return listing || c >= kWarpClasses || (k > 5 && c > 0); }

// Launch shape of class c for a largest out-degree maxd.
Cfg config(int c, uint32_t k, uint32_t maxd, bool listing) {
    Cfg f;
    uint32_t d = maxd < kLimits[c] ? maxd : kLimits[c];
    f.D = (d + 31) & ~31u;
    if (f.D < 32) f.D = 32;
    const bool cta = cta_form(c, k, listing);
    const uint32_t full = set_room(f.D, listing);
    const uint32_t least = idx_words(f.D), fixed = scratch_fixed(row_words4(f.D));
    if (!cta) {
        f.warps = 4;  // warps per block, one root each
        f.room = full;
        f.smem = 4 * (size_t)make_lay(f.D, 1, full).total * 4;
        f.gwords = 0;
        f.per_sm = 0;
        return f;
    }
    f.warps = f.D <= 128 ? 4 : f.D <= 256 ? 8 : 16;
    f.per_sm = 32 / f.warps;  // 64 registers a thread: 1024 threads per SM
    const uint32_t head = make_lay(f.D, 0, 0).X;
    auto room_in = [&](size_t cap) {
        const uint32_t words = (uint32_t)(cap / 4);
        const uint32_t each = words > head ? (words - head) / f.warps : 0u;
        uint32_t b = each > fixed ? (each - fixed) & ~3u : 0u;
        if (b < least) b = least;
        return b < full ? b : full;
    };
    f.room = room_in(f.D <= 256 ? kFullSM / f.per_sm - 1024 : kHalfSM);
    if (f.D > 256 && ((f.room < 512 && f.room < full) || make_lay(f.D, f.warps, f.room).total * 4 > kHalfSM)) {
        f.per_sm = 1;  // large rows: one CTA with room for its matrices
        f.room = room_in(kFullSM);
    }
    f.smem = (size_t)make_lay(f.D, f.warps, f.room).total * 4;
    f.gwords = f.room < full ? full : 0;
    return f;
}

}  // namespace

bool sub_handles(const kcl_graph *g, uint32_t k, int c, kcl_ordering ord) {
    if (c >= kSubClasses || k > 6) return false;
    if (ord == KCL_ORDER_DEGREE) return g->tuning.sdegree_bitmap[c] != 0xFFFFFFFFu;  // lists asked for
    return !(g->options & KCL_OPT_NO_COLOR_PRUNE);  // the ablation runs the colour path without its prune
}

size_t sub_arena_words(uint32_t k, int num_sms, uint32_t max_outdeg, bool listing) {
    size_t need = 0;
    for (int c = 0; c < kSubClasses; c++) {
        if (c > 0 && kLimits[c - 1] >= max_outdeg) break;
        const Cfg f = config(c, k, max_outdeg, listing);
        const size_t words = (size_t)f.gwords * f.warps * f.per_sm * (size_t)num_sms;
        if (words > need) need = words;
    }
    return need;
}

int launch_sub(const kcl_graph *g, uint32_t k, Workspace &w, int c, uint32_t begin, uint32_t end, unsigned *queue,
               const ListArgs &la, uint32_t dfs_warps, cudaStream_t s) {
    const Cfg f = config(c, k, la.max_outdeg, la.listing);
    SubArgs a;
    a.optr = w.optr;
    a.oadj = w.oadj;
    a.roots = w.roots;
    a.begin = begin;
    a.end = end;
    a.parts = 1;
    a.queue = queue;
    a.gscratch = w.arena;
    a.gwords = f.gwords;
    a.D = f.D;
    a.room = f.room;
    a.dfs_warps = dfs_warps;
    a.ring = la.ring;
    a.capacity = la.capacity;
    a.wrap = la.wrap;
    a.idmap = la.idmap;
    a.kmap = w.kmap;
    a.per_root = la.per_root;
    a.root_cks = la.per_root_cks;
    a.res = w.res;
    const bool cta = cta_form(c, k, la.listing);
    int occ = 0;
    uint32_t n = end - begin;
    using Kernel = void (*)(const SubArgs);
    static const Kernel warp_kernels[] = {k_sub_warp<0>, k_sub_warp<3>, k_sub_warp<4>, k_sub_warp<5>, k_sub_warp<6>};
    static const Kernel cta_kernels[2][5] = {
        {k_sub_cta<false, 0>, k_sub_cta<false, 3>, k_sub_cta<false, 4>, k_sub_cta<false, 5>, k_sub_cta<false, 6>},
        {k_sub_cta<true, 0>, k_sub_cta<true, 3>, k_sub_cta<true, 4>, k_sub_cta<true, 5>, k_sub_cta<true, 6>}};
    const uint32_t ki = w.kmap ? 0u : k - 2;
    const Kernel kern = cta ? cta_kernels[la.listing ? 1 : 0][ki] : warp_kernels[ki];
    if (!cta) {
        if (!allow_max_smem(kern) ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, f.warps * 32, f.smem) != cudaSuccess)
            (void)cudaGetLastError();
        if (occ < 1) occ = 1;
        uint32_t blocks = (uint32_t)g->num_sms * occ;
        const uint32_t need = (n + f.warps - 1) / f.warps;
        if (blocks > need) blocks = need;
        kern<<<blocks, f.warps * 32, f.smem, s>>>(a);
        return 1;
    }
    if (!allow_max_smem(kern) ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, f.warps * 32, f.smem) != cudaSuccess)
        (void)cudaGetLastError();
    if (occ < 1) occ = 1;
    if (occ > (int)f.per_sm) occ = (int)f.per_sm;  // global room per SM
    uint32_t blocks = (uint32_t)g->num_sms * occ;
    // a class with few roots shares each root's children over several CTAs, which
    // all build it: up to 8 units per CTA of the launch (with up to 32, building
    // took over: 131k k = 6 count 41.7 -> 60.6 ms; with up to 4, the tail: 43.1).
    // dfs_warps = 1 asks for one warp per root (NodeParallel), so for no shares.
    if (dfs_warps != 1 && (k >= 5 || (la.listing && k >= 4 && c >= kWarpClasses))) {
        while (a.parts < 8 && n * a.parts < 8 * blocks) a.parts *= 2;
    }
    if (blocks > n * a.parts) blocks = n * a.parts;
    kern<<<blocks, f.warps * 32, f.smem, s>>>(a);
    return 1;
}

}  // namespace kcl
