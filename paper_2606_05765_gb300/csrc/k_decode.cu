// Decode side: plan, ANS pass, rank directories and the bottom-up merge
// (Sec. 3; Sec. 5.2 for ANS-coded bitmaps).
//
//   plan       one CTA per record, or one warp per record in large batches:
//              validates the header and body layout, sizes the ANS scratch,
//              builds the block's node table (bitmap source and children of
//              every internal node, from the canonical or the regrouped tree
//              of the code lengths) and splits the block into root tiles whose
//              levels fit a CTA's level buffers; per-block offsets come from
//              two single-pass scans with decoupled look-back.
//   ans        one warp per unit of ANS segments: decodes the bitmap bytes
//              into the workspace scratch.
//   directory  for blocks with several tiles: per-node rank directories
//              (popcount per superblock, by shares) and, from them, every
//              node's bitmap cursor at every tile boundary (the root cursor is
//              the position; a child's cursor is the parent's rank0 / rank1).
//   tiles      one CTA per tile, independent of the other tiles.  With both
//              boundary cursors known, every node's bit range in the tile is
//              known.  Bottom-up, level by level, every node rebuilds its
//              symbol sequence
//                  out_v[k] = bit ? R[rank1(k)] : L[k - rank1(k)]
//              from its children's sequences or leaf constants (the MVV /
//              MCV / MVC / MCC cases of Sec. 3.2), a flat node from its
//              packed indices.  Ranks come from popcounts of 32-bit bitmap
//              words, a warp scan and the windows' counts; 4 output symbols
//              are one byte permute of a left and a right 4-byte window.  The
//              root writes the output.  A tile whose levels do not fit is
//              decoded in shorter chunks whose bit ranges are found top-down
//              from popcounts.
#include "ans_dev.cuh"
#include "levels.cuh"
#include "lookback.cuh"

namespace pv {

constexpr int kDecThreads = 256;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kLvlFit = 24576;               // the plan's measure of a level (plan_tiles)
constexpr int kLvlBuf = 23360;               // one level buffer of a tile (bytes; what is left of the shared memory)
static_assert(4 * (kLvlFit - 4 * 128 - 32) / 5 + 15 * 128 <= kLvlBuf, "a tile of even statistics fits");
constexpr int kWSlack = 80;                  // over-read room of the byte windows (64 symbols and 11 bytes)
constexpr int kTileCtas = 4;                 // tile CTAs per SM the kernels are built for
constexpr uint32_t kNtabHdr = 32;            // node table header (see plan_block)

// bytes of a block's node table: header, then per node u32 bitmap source,
// u32 children and u32 first rank-directory entry, then the block's 256
// symbols in (length, symbol) order (the tables of its flat nodes)
__host__ __device__ inline uint32_t ntab_bytes(uint32_t V) { return (kNtabHdr + 12u * V + 256u + 15u) & ~15u; }

// rank-directory granularity, and whether every coded block gets a directory
// (random access) rather than only those split into several tiles: header
// word 7, the flag in bit 31
__device__ inline uint32_t dec_dir_bits(const uint8_t *ws) { return reinterpret_cast<const uint32_t *>(ws)[7] & 0xFFFFu; }
__device__ inline bool dec_all_dirs(const uint8_t *ws) { return (reinterpret_cast<const uint32_t *>(ws)[7] >> 31) != 0; }

__host__ __device__ inline uint32_t scratch_stride(uint32_t raw) { return ((raw + 15u) & ~15u) + 16u; }
// scratch of a block's ANS-coded nodes at most (with the last one's 16 bytes of padding: bit addresses stay below
// 2^31; a corrupt record's counts could ask for more than 2^32 bytes, and get a place over its neighbours')
constexpr uint64_t kScratchMax = (1ull << 28) + 16;
// and a node's bits in the record end below that too (bitmaps that are not ANS-coded; nothing later could tell
// their addresses from the scratch's); only in a record of kRecFar bytes can they not
constexpr uint32_t kRecFar = 1u << 28;

// The dynamic shared memory of every kernel here: the merge's selector table
// (1 KiB), then what the item at hand needs.  The big steps are functions of
// their own (their registers are allocated apart, so the tile's loops do not
// spill for the plan's sake), and reach shared memory through these instead
// of pointer arguments, which would make every access a generic one.
constexpr uint32_t kSelBytes = 1024;
template <typename T>
__device__ inline T &smem_item() {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    return *reinterpret_cast<T *>(smem_raw + kSelBytes);
}
__device__ inline uint32_t *smem_sel() {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    return reinterpret_cast<uint32_t *>(smem_raw);
}

__device__ inline int find_node_d(const uint32_t *key, int lo, int hi, uint32_t g) {
    while (hi - lo > 1) {
        const int m = (lo + hi) >> 1;
        if (key[m] <= g) lo = m; else hi = m;
    }
    return lo;
}

// largest b in [0, n) with key[b] <= g (key non-decreasing, key[0] <= g), by
// a whole warp (all lanes, same arguments): 32 probes per
// step, the first around `guess` (where g would sit if the items were spread
// evenly), then 32-way splits of what is left.  key[0] <= g.
__device__ inline int find_block_warp(const uint32_t *key, int n, uint32_t g, int guess) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = n;   // the answer is in [lo, hi); key[lo] <= g
    {
        const int s = max(0, min(guess - 15, n - 32));
        const int b = s + lane;
        const uint32_t m = __ballot_sync(0xffffffffu, b < n && key[b] <= g);   // a prefix of the lanes
        const int c = __popc(m), nv = min(32, n - s);
        if (c > 0) lo = s + c - 1;
        if (c < nv) hi = s + c;
    }
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) >> 5;
        const int b = lo + lane * step;
        const uint32_t m = __ballot_sync(0xffffffffu, lane == 0 || (b < hi && key[b] <= g));
        const int c = __popc(m);
        lo += (c - 1) * step;
        hi = min(hi, lo + step);
    }
    return lo;
}

// bytes of a record staged in shared memory by the parse: the header, the
// length nibbles, n_v, the markers and the alen table of any record
constexpr uint32_t kStage = 2448;
static_assert(kStage >= kNvOff + 5 * 255 + 3 + 4 * 255 && kStage % 16 == 0, "the stage holds a record's tables");

// ---------------------------------------------------------------------------
// Plan: one CTA per record (ticket order), two look-back chains over blocks
//   A: (ANS scratch bytes << 22) | ANS segments
//   B: (node table + directory + cursor bytes << 22) | tiles
// Tuning (from the workspace header): the longest tile and the rank
// directory granularity; neither changes the decoded bytes.
//
// Node table of a coded block (start of its directory region):
//    0 u8 first[17]   first node of each depth (breadth-first node order)
//   17 u8 maxd        depth of the deepest leaf
//   20 u32 ent        rank-directory entries (blocks with several tiles)
//   24 u32 T          root symbols per tile
//   32 per node, three u32 together (random access reads them in one go):
//      src            bit address of the node's bitmap: 8 x record byte offset,
//                     or 8 x block scratch offset | 2^31 for ANS-coded nodes
//      ch             children: child c in bits [16c, 16c + 16), 0x8000 |
//                     symbol for a leaf, else the child's node index; a
//                     flat node's word is ch_flat(D, base)
//      u              the node's first rank-directory entry (blocks with one)
//      u8 sym[256]    the symbols in (length, symbol) order: flat node
//                     symbol x is sym[base + x]
//
// What bounds it: latency, a chain of about twelve short steps per record.
// A whole CTA takes a record (thread t is node t and symbol t) so that a
// step is one instruction sequence and a barrier instead of a warp's loop
// over 256 items: one record alone is planned in 8 us against 25 us by one
// warp.
// ---------------------------------------------------------------------------
struct PlanTree {
    int32_t cnt[17], start[17]; // symbols of each length, index of the first one in (length, symbol) order
    int32_t a[18], first[18];   // leaf-covered prefixes, first node of each depth
    int32_t good, maxd, K;
};

// The canonical tree of the code lengths (c: symbols of length `lane`, lanes
// 1..15; one warp): a[d] prefixes of depth d are leaves or under leaves, the
// others are internal nodes (Sec. 1.1).  Ends with a __syncwarp.
__device__ inline void plan_tree(uint32_t c, bool flat, uint32_t V, PlanTree &P) {
    const int lane = threadIdx.x & 31;
    uint32_t s = c;   // symbols of length <= lane
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
    }
    const int K = (int)__shfl_sync(0xffffffffu, s, 31);
    const uint32_t used = __ballot_sync(0xffffffffu, c != 0);
    const int m = used ? 31 - __clz(used) : 0;
    int32_t a = 0;   // (at most 256 symbols: below 2^24)
#pragma unroll 1
    for (int j = 1; j <= 16; j++) {
        const int32_t cj = (int32_t)__shfl_sync(0xffffffffu, c, j & 15);
        if (j <= lane && lane <= 16) a = 2 * a + (j < 16 ? cj : 0);
    }
    const int32_t open = lane <= 16 ? (1 << lane) - a : 0;
    bool okd = true;
    if (lane <= 16 && (open < 0 || (lane < m && open <= 0) || (lane == m && open != 0))) okd = false;   // (Kraft: full)
    const int32_t mine = lane < m && open > 0 ? open : 0;
    int32_t f = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, f, o);
        if (lane >= o) f += y;
    }
    const int32_t tot = __shfl_sync(0xffffffffu, f, 31);
    // (a regrouped tree has its own node count, checked by the caller)
    const bool good = __all_sync(0xffffffffu, okd) && K >= 2 && tot == K - 1 && (flat || tot == (int32_t)V);
    if (lane <= 16) {
        P.a[lane] = a;
        P.first[lane] = f - mine;
        P.cnt[lane] = lane < 16 ? (int32_t)c : 0;
        P.start[lane] = (int32_t)(s - c);
    }
    if (lane == 0) { P.first[17] = tot; P.good = good; P.maxd = m; P.K = K; }
    __syncwarp();
}

// Children word of node v of the canonical tree at depth d (sorted: the
// symbols in (length, symbol) order); false when it leaves the tree.
__device__ inline bool plan_children(const PlanTree &P, const uint8_t *sorted, uint32_t V, int v, int d, uint32_t &chv) {
    const int32_t p = P.a[d] + (v - P.first[d]);
    bool ok = true;
    chv = 0;
    for (int c = 0; c < 2; c++) {
        const int32_t cp = 2 * p + c;
        uint32_t code = 0;
        if (cp < P.a[d + 1]) {             // a leaf of length d + 1
            const int32_t i = cp - 2 * P.a[d];
            if (d + 1 > 15 || i < 0 || i >= P.cnt[d + 1]) ok = false;
            else code = 0x8000u | sorted[P.start[d + 1] + i];
        } else {
            const int32_t nd = P.first[d + 1] + (cp - P.a[d + 1]);
            if (nd <= v || nd >= (int32_t)V) ok = false;
            else code = (uint32_t)nd;
        }
        chv |= code << (16 * c);
    }
    return ok;
}

// Root symbols per tile and tiles of a block of n symbols (one warp; lvl[d]:
// symbols of level d): a tile's average share of every level is at most 4/5 of
// kLvlFit - 32 bytes, less 4 bytes a node.  With the spans' 15 bytes of rounding
// a node at most, that leaves 16 % of the level buffer free for a level of few
// nodes, 10 % for one of 128; a tile that needs more (the block's statistics
// drift) is decoded in chunks.
__device__ inline void plan_tiles(const PlanTree &P, const uint32_t *lvl, uint32_t n, uint32_t tile_max, uint32_t &T,
                                  uint32_t &ntile) {
    const int lane = threadIdx.x & 31;
    uint64_t tf = ~0ull;
    if (lane >= 1 && lane < 16 && lvl[lane]) {
        const uint32_t nodes = (uint32_t)(P.first[lane + 1] - P.first[lane]);
        const uint64_t room = (uint64_t)kLvlFit > 4ull * nodes + 32 ? kLvlFit - 4ull * nodes - 32 : 0;
        tf = room * n / lvl[lane] / 5 * 4;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) tf = umin64(tf, __shfl_xor_sync(0xffffffffu, tf, o));
    T = n;
    ntile = 1;
    if (!(n <= tile_max && tf >= n)) {
        uint64_t t2 = (tf < (uint64_t)tile_max ? tf : (uint64_t)tile_max) & ~127ull;
        if (t2 < 128) t2 = 128;
        const uint64_t tmin = ((uint64_t)n + (1u << 21) - 1) >> 21;   // at most 2^21 tiles
        if (t2 < tmin) t2 = (tmin + 127) & ~127ull;
        T = (uint32_t)t2;
        ntile = (n + T - 1) / T;
    }
}

// The regrouped tree of the lengths in P (one warp): P.first and P.maxd
// become its own; P.good: it has V nodes.
__device__ inline void plan_flat(PlanTree &P, const uint8_t *sorted, uint32_t V, FlatTree &F) {
    const int lane = threadIdx.x & 31;
    flat_tree_build(P.cnt, P.start, sorted, F);
    const bool ok = F.ok && F.n_nodes == (int32_t)V;
    if (ok && lane < 18) P.first[lane] = lane < F.maxd ? F.first[lane] : F.n_nodes;
    __syncwarp();
    if (lane == 0) { P.good = ok; if (ok) P.maxd = F.maxd; }
    __syncwarp();
}

struct __align__(16) PlanSm {
    uint8_t stg[kStage];        // the record's tables
    uint32_t body_off[256];
    uint32_t nv[256];
    uint32_t ch[256];
    uint32_t u[256];            // first rank-directory entry of node v
    uint32_t soff[256];         // scratch offset of an ANS node within its block
    uint32_t lcnt[kDecWarps][16];   // symbols of each length, by warp
    uint32_t wsum[kDecWarps];   // scan_cta's warp totals
    uint64_t wsum64[2][kDecWarps];
    uint32_t lvl[17];           // symbols of each level
    PlanTree tree;
    uint32_t ntile, T;
    uint8_t marker[256];
    uint8_t sorted[256];
    FlatTree F;
    // CTA look-back
    uint32_t mins[kDecWarps][4];
    uint64_t sums[kDecWarps][2];
};

// what a plan found (the same in every thread)
struct PlanRes {
    int32_t st;                 // PIVCO_OK, PIVCO_ERR_CORRUPT, PIVCO_ERR_INVALID_ARG
    uint32_t kind, V, n, rb, ntile, T, ent, scratch, nsegs;
    uint64_t dir_bytes;
};

// exclusive scan of x over the CTA's threads (every thread calls it); total: the sum
__device__ inline uint32_t scan_cta(uint32_t x, uint32_t *wsum, uint32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    uint32_t base = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < kDecWarps; w++) {
        const uint32_t s = wsum[w];
        if (w < warp) base += s;
        total += s;
    }
    __syncthreads();
    return base + inc - x;
}
__device__ inline uint64_t scan_cta64(uint64_t x, uint64_t *wsum, uint64_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    uint64_t base = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < kDecWarps; w++) {
        const uint64_t s = wsum[w];
        if (w < warp) base += s;
        total += s;
    }
    __syncthreads();
    return base + inc - x;
}

// Whether a bitmap of a record of kRecFar bytes or more (staged at g) ends past
// the bit addresses (every thread the same; out of the way of the others).
__device__ __noinline__ bool plan_far(const uint8_t *g, uint32_t V, uint32_t nsel) {
    const uint8_t *mks = g + kNvOff + 4 * V;
    const uint32_t alen_off = (kNvOff + 5 * V + 3) & ~3u;
    uint64_t off = alen_off + 4 * nsel;
    bool far = false;
    uint32_t k = 0;
    for (int pass = 0; pass < 2; pass++)   // the raw and flat nodes' bodies, then the listed ones'
        for (uint32_t v = 0; v < V; v++) {
            const uint32_t mk = mks[v];
            if (mark_listed(mk) != (pass == 1)) continue;
            const uint64_t bits = (uint64_t)ld_le32(g + kNvOff + 4 * v) * max(1u, (uint32_t)mark_flat_d(mk));
            if (!mark_ans(mk) && 8 * off + bits >= 1ull << 31) far = true;
            off += pass ? ld_le32(g + alen_off + 4 * k++) : (bits + 7) / 8;
        }
    return far;
}

// Parses record b, checks its layout and builds its node table in Q (the
// whole CTA, kDecThreads threads; nothing global is written).
__device__ __noinline__ PlanRes plan_cta(const uint8_t *__restrict__ rec, uint64_t avail, uint32_t dir_bits,
                                         uint32_t tile_max, bool all_dirs) {
    PlanSm &Q = smem_item<PlanSm>();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    PlanRes R{};
    R.ntile = 1;
    // a record starts on a 16-byte boundary (its words are read as words)
    const bool misal = (reinterpret_cast<uintptr_t>(rec) & 15) != 0;
    R.st = misal ? PIVCO_ERR_INVALID_ARG : PIVCO_ERR_CORRUPT;   // unless the checks below pass
    if (misal) return R;
    // one coalesced pass stages the tables; everything below reads shared memory
    {
        const uint32_t ns = (uint32_t)(avail < kStage ? avail : kStage);
        for (uint32_t i = 16 * t; i < kStage; i += 16 * kDecThreads) {
            if (i + 16 <= ns) {
                *reinterpret_cast<uint4 *>(Q.stg + i) = __ldg(reinterpret_cast<const uint4 *>(rec + i));
            } else {
                for (uint32_t j = i; j < i + 16; j++) Q.stg[j] = j < ns ? rec[j] : 0;
            }
        }
        if (t < kDecWarps * 16) (&Q.lcnt[0][0])[t] = 0;
        if (t < 17) Q.lvl[t] = 0;
    }
    __syncthreads();
    const uint8_t *g = Q.stg;
    if (avail < kHdr) return R;
    const uint32_t rb = ld_le32(g), n = ld_le32(g + 4), V = (uint32_t)g[8] | ((uint32_t)g[9] << 8), kind = g[10];
    if (!(g[12] == 'P' && g[13] == 'V' && g[14] == 'C' && (g[15] == '1' || g[15] == '2') && rb >= kHdr && !(rb & 15u) &&
          rb <= avail))
        return R;
    const bool flat = g[15] == '2';
    R.kind = kind;
    R.rb = rb;
    if (kind != 2) {
        const bool ok = kind == 0 ? (n == 0 && V == 0 && g[11] == 0 && rb == kHdr)
                                  : (kind == 1 && n != 0 && V == 0 && rb == kHdr);
        if (ok) { R.st = PIVCO_OK; R.n = n; R.T = n; }
        return R;
    }
    if (V < 1 || V > 255 || n == 0 || g[11] != 0 || rb < kNvOff + 5 * V) return R;
    // ---- thread t: node t's count, marker and body size; symbol t's length ----
    const bool node = (uint32_t)t < V;
    bool bad = false;
    const uint32_t nv = node ? *reinterpret_cast<const uint32_t *>(g + kNvOff + 4 * t) : 0u;
    const uint32_t mk = node ? g[kNvOff + 4 * V + t] : 0u, fd = mark_flat_d(mk);
    const bool listed = mark_listed(mk), ans = mark_ans(mk);
    if (node) {
        // flat markers (0xF0 + D) only in records of the regrouped tree
        if (fd ? !flat : (mk && mk != kMarkRawSel && ((mk & 0x7F) < 1 || (mk & 0x7F) > 50))) bad = true;
        // every symbol under a node occurs at least once
        if (nv < (2u << (fd ? fd - 1 : 0)) || nv > n) bad = true;
        if (fd && (uint64_t)nv * fd > 0xFFFFFFFFull) bad = true;
        if (t == 0 && nv != n) bad = true;
    }
    Q.nv[t] = nv;
    Q.marker[t] = (uint8_t)mk;
    const uint32_t len = (g[kLensOff + (t >> 1)] >> (4 * (t & 1))) & 15u;
    const uint32_t peers = __match_any_sync(0xffffffffu, len);
    const uint32_t lrank = __popc(peers & ((1u << lane) - 1u));   // among the warp's symbols of that length
    if (lrank == 0) Q.lcnt[warp][len] = __popc(peers);
    const uint32_t nsel = (uint32_t)__syncthreads_count(listed);
    const uint32_t alen_off = (kNvOff + 5 * V + 3) & ~3u;
    if (alen_off + 4 * nsel > rb) return R;
    // raw body bytes: ceil(n_v / 8), ceil(n_v D / 8) for a flat node
    const uint32_t raw = (uint32_t)(((uint64_t)nv * (fd ? fd : 1u) + 7) / 8);
    uint32_t al = raw;
    if (nsel) {
        uint32_t tot;
        const uint32_t p = scan_cta(listed, Q.wsum, tot);
        if (listed) al = ld_le32(g + alen_off + 4 * p);
        if (mk == kMarkRawSel && al != raw) bad = true;
    }
    const uint32_t base1 = alen_off + 4 * nsel;
    uint64_t raw_tot, sel_tot = 0;
    const uint64_t ro = scan_cta64(node && !listed ? al : 0u, Q.wsum64[0], raw_tot);
    uint64_t off = base1 + ro;
    if (nsel) {   // (64-bit: corrupt alen values could wrap 32 bits)
        const uint64_t so = scan_cta64(listed ? al : 0u, Q.wsum64[1], sel_tot);
        if (listed) off = base1 + raw_tot + so;
    }
    if (((base1 + raw_tot + sel_tot + 15) & ~15ull) != rb) bad = true;
    if (rb >= kRecFar && plan_far(g, V, nsel)) bad = true;
    Q.body_off[t] = (uint32_t)off;
    uint32_t scratch = 0, nsegs = 0;
    if (nsel) {
        const uint32_t rawb = (nv + 7) / 8;
        uint64_t tot;
        Q.soff[t] = (uint32_t)scan_cta64(ans ? scratch_stride(rawb) : 0u, Q.wsum64[0], tot);
        if (tot > kScratchMax) bad = true;
        scratch = (uint32_t)tot;
        uint32_t full, lanes;
        scan_cta(ans ? ans_full_segs(rawb) : 0u, Q.wsum, full);
        scan_cta(ans ? ans_tail_lanes(rawb) : 0u, Q.wsum, lanes);
        nsegs = ans_units(full, lanes);
    }
    if (warp == 0) {
        uint32_t c = 0;
        if (lane >= 1 && lane < 16)
            for (int w = 0; w < kDecWarps; w++) c += Q.lcnt[w][lane];
        plan_tree(c, flat, V, Q.tree);
    }
    __syncthreads();
    if (!Q.tree.good) return R;
    if (len) {   // symbols in canonical order (length, then value)
        uint32_t r = (uint32_t)Q.tree.start[len] + lrank;
        for (int w = 0; w < warp; w++) r += Q.lcnt[w][len];
        Q.sorted[r & 255u] = (uint8_t)t;
    }
    __syncthreads();
    if (flat) {
        // the regrouped tree with flat subtrees (Sec. 2.2.3-2.2.4); its
        // flat nodes must be the record's (markers 0xF0 + D)
        if (warp == 0) plan_flat(Q.tree, Q.sorted, V, Q.F);
        __syncthreads();
        if (!Q.tree.good) return R;
    }
    // ---- children of every node and the symbols of each depth ----
    if (node) {
        int d = 0;
        uint32_t chv = 0;
        if (flat) {
            if (!flat_node(Q.F, Q.sorted, t, d, chv)) bad = true;
            const uint32_t D = ch_flat_d(chv);
            if (D != fd || (D && (chv & 0xFFu) + (1u << D) > (uint32_t)Q.tree.K)) bad = true;
        } else {
            while (d < 15 && Q.tree.first[d + 1] <= t) d++;
            if (!plan_children(Q.tree, Q.sorted, V, t, d, chv)) bad = true;
        }
        if (d >= 1) atomicAdd(&Q.lvl[d], nv);
        Q.ch[t] = chv;
    }
    if (__syncthreads_or(bad)) return R;
    if (warp == 0) {
        uint32_t T, ntile;
        plan_tiles(Q.tree, Q.lvl, n, tile_max, T, ntile);
        if (lane == 0) { Q.T = T; Q.ntile = ntile; }
    }
    __syncthreads();
    R.T = Q.T;
    R.ntile = Q.ntile;
    R.scratch = scratch;
    R.nsegs = nsegs;
    if (R.ntile > 1 || all_dirs) Q.u[t] = scan_cta((nv + dir_bits - 1) / dir_bits, Q.wsum, R.ent);
    R.dir_bytes = ntab_bytes(V) + (R.ent ? ((4ull * R.ent + 4ull * (R.ntile + 1) * V + 15) & ~15ull) : 0ull);
    R.V = V;
    R.n = n;
    R.st = PIVCO_OK;
    __syncthreads();
    return R;
}

// bit address of node v's bitmap (node table format)
__device__ inline uint32_t plan_src(const PlanSm &Q, uint32_t v) {
    return mark_ans(Q.marker[v]) ? (8u * Q.soff[v]) | 0x80000000u : 8u * Q.body_off[v];
}

// publishes block b's sizes (one thread, right after its plan: successors
// need no more than these to go on)
__device__ inline void plan_publish(const DecWs &W, int b, const PlanRes &R) {
    lb2_publish(W.states_a, W.states_b, b, ((uint64_t)R.scratch << 22) | R.nsegs, (R.dir_bytes << 22) | R.ntile);
}

// Places block b: its offsets from the look-back, its status, and its node
// table when `table` (only where the workspace holds it: a sizing run may
// not; and never from a partial prefix, which would place it over another
// block's table).  The whole CTA; false when the look-back gave up.
__device__ inline bool plan_place(int b, int nblk, uint8_t *__restrict__ ws, uint64_t ws_bytes, const PlanRes &R,
                                  bool table, uint64_t &nbase) {
    PlanSm &Q = smem_item<PlanSm>();
    const int t = threadIdx.x;
    uint32_t *hdr32 = reinterpret_cast<uint32_t *>(ws);
    uint64_t *hdr64 = reinterpret_cast<uint64_t *>(ws);
    const DecWs W = dec_ws(ws, nblk);
    uint64_t ea = 0, eb = 0;
    const uint64_t agg_a = ((uint64_t)R.scratch << 22) | R.nsegs, agg_b = (R.dir_bytes << 22) | R.ntile;
    const bool to = lookback2_cta(W.states_a, W.states_b, b, agg_a, agg_b, ea, eb, hdr64[7], Q.mins, Q.sums);
    if (t == 0) {
        W.blk_scratch[b] = ea >> 22;
        W.blk_seg[b] = (uint32_t)(ea & ((1u << 22) - 1));
        W.blk_dir[b] = eb >> 22;
        W.blk_tile[b] = (uint32_t)(eb & ((1u << 22) - 1));
        W.blk_T[b] = R.T;
        W.blk_ntile[b] = R.ntile;
        if (b == nblk - 1) {
            hdr64[0] = (ea >> 22) + R.scratch;
            hdr32[2] = (uint32_t)((ea & ((1u << 22) - 1)) + R.nsegs);
            hdr64[2] = (eb >> 22) + R.dir_bytes;
            hdr32[6] = (uint32_t)((eb & ((1u << 22) - 1)) + R.ntile);
            // totals from a partial prefix are unusable: every later pass
            // gives the whole batch up (abandoned_batch)
            if (to) atomicExch(&hdr32[13], 1u);
        }
    }
    nbase = decode_ws_fixed_bytes(nblk) + (eb >> 22);
    if (table && R.st == PIVCO_OK && R.kind == 2 && !to && nbase + ntab_bytes(R.V) <= ws_bytes) {
        uint8_t *nt = ws + nbase;
        if (t < 17) nt[t] = (uint8_t)Q.tree.first[t];
        if (t == 17) nt[17] = (uint8_t)Q.tree.maxd;
        if (t == 0) {
            *reinterpret_cast<uint32_t *>(nt + 20) = R.ent;
            *reinterpret_cast<uint32_t *>(nt + 24) = R.T;
        }
        uint32_t *src = reinterpret_cast<uint32_t *>(nt + kNtabHdr);
        if ((uint32_t)t < R.V) {
            src[3 * t] = plan_src(Q, t);
            src[3 * t + 1] = Q.ch[t];
            src[3 * t + 2] = R.ent ? Q.u[t] : 0u;
        }
        nt[kNtabHdr + 12 * R.V + t] = Q.sorted[t];
    }
    return !to;
}

// ---------------------------------------------------------------------------
// The same plan, one warp per record and eight records per CTA: a third of
// the instructions per record (no step is repeated by eight warps), so it is
// the one for batches of many records, where the chip is full either way; one
// record's latency is three times the CTA plan's.
// ---------------------------------------------------------------------------
struct __align__(16) PlanWarpSm {
    uint8_t stg[kStage];
    uint32_t src[256];          // node v's bitmap (node table format)
    uint32_t run[16], lvl[17];
    PlanTree tree;
    uint8_t sorted[256];
    FlatTree F;
};
struct PlanItemSm {
    PlanWarpSm w[kDecWarps];
    uint64_t agg[kDecWarps][2];
    uint32_t mins[kDecWarps][4];
    uint64_t sums[kDecWarps][2];
};

__device__ inline PlanRes plan_warp(const uint8_t *__restrict__ rec, uint64_t avail, uint32_t dir_bits,
                                    uint32_t tile_max, bool all_dirs, PlanWarpSm &Q) {
    const int lane = threadIdx.x & 31;
    PlanRes R{};
    R.ntile = 1;
    const bool misal = (reinterpret_cast<uintptr_t>(rec) & 15) != 0;
    R.st = misal ? PIVCO_ERR_INVALID_ARG : PIVCO_ERR_CORRUPT;   // unless the checks below pass
    if (misal) return R;
    {
        const uint32_t ns = (uint32_t)(avail < kStage ? avail : kStage);
#pragma unroll
        for (uint32_t i = 16 * lane; i < kStage; i += 512) {
            if (i + 16 <= ns) {
                *reinterpret_cast<uint4 *>(Q.stg + i) = __ldg(reinterpret_cast<const uint4 *>(rec + i));
            } else {
                for (uint32_t j = i; j < i + 16; j++) Q.stg[j] = j < ns ? rec[j] : 0;
            }
        }
        if (lane < 16) Q.run[lane] = 0;
        if (lane < 17) Q.lvl[lane] = 0;
        __syncwarp();
    }
    const uint8_t *g = Q.stg;
    if (avail < kHdr) return R;
    const uint32_t rb = ld_le32(g), n = ld_le32(g + 4), V = (uint32_t)g[8] | ((uint32_t)g[9] << 8), kind = g[10];
    if (!(g[12] == 'P' && g[13] == 'V' && g[14] == 'C' && (g[15] == '1' || g[15] == '2') && rb >= kHdr && !(rb & 15u) &&
          rb <= avail))
        return R;
    const bool flat = g[15] == '2';
    R.kind = kind;
    R.rb = rb;
    if (kind != 2) {
        const bool ok = kind == 0 ? (n == 0 && V == 0 && g[11] == 0 && rb == kHdr)
                                  : (kind == 1 && n != 0 && V == 0 && rb == kHdr);
        if (ok) { R.st = PIVCO_OK; R.n = n; R.T = n; }
        return R;
    }
    if (V < 1 || V > 255 || n == 0 || g[11] != 0 || rb < kNvOff + 5 * V) return R;
    const uint32_t *nvs = reinterpret_cast<const uint32_t *>(g + kNvOff);
    const uint8_t *mks = g + kNvOff + 4 * V;
    // ---- nodes: counts, markers, body sizes and places ----
    bool bad = false;
    uint32_t nsel = 0;
    for (uint32_t v0 = 0; v0 < V; v0 += 32)
        nsel += __popc(__ballot_sync(0xffffffffu, v0 + lane < V && mark_listed(mks[min(v0 + lane, V - 1)])));
    const uint32_t alen_off = (kNvOff + 5 * V + 3) & ~3u, base1 = alen_off + 4 * nsel;
    if (base1 > rb) return R;
    uint64_t raw_tot = 0, sel_tot = 0, scratch_tot = 0;
    uint32_t scratch = 0, full = 0, lanes = 0, ent = 0, np = 0;
    for (uint32_t v0 = 0; v0 < V; v0 += 32) {
        const uint32_t v = v0 + lane;
        const bool node = v < V;
        const uint32_t nv = node ? nvs[v] : 0u, mk = node ? mks[v] : 0u, fd = mark_flat_d(mk);
        const bool listed = mark_listed(mk), ans = mark_ans(mk);
        if (node) {
            // flat markers (0xF0 + D) only in records of the regrouped tree
            if (fd ? !flat : (mk && mk != kMarkRawSel && ((mk & 0x7F) < 1 || (mk & 0x7F) > 50))) bad = true;
            // every symbol under a node occurs at least once
            if (nv < (2u << (fd ? fd - 1 : 0)) || nv > n || (v == 0 && nv != n)) bad = true;
            if (fd && (uint64_t)nv * fd > 0xFFFFFFFFull) bad = true;
        }
        const uint32_t raw = (uint32_t)(((uint64_t)nv * (fd ? fd : 1u) + 7) / 8);
        uint32_t al = raw;
        const uint32_t lm = __ballot_sync(0xffffffffu, listed);
        if (listed) al = ld_le32(g + alen_off + 4 * (np + __popc(lm & ((1u << lane) - 1u))));
        np += __popc(lm);
        if (mk == kMarkRawSel && al != raw) bad = true;
        // (64-bit: corrupt sizes could wrap 32 bits)
        uint64_t x = node && !listed ? al : 0u, inc = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (node && !listed) Q.src[v] = 8u * (uint32_t)(base1 + raw_tot + inc - x);
        raw_tot += __shfl_sync(0xffffffffu, inc, 31);
        if (lm) {
            x = listed ? al : 0u;
            inc = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            // (a selected node kept raw: its place among the selected bodies, which follow all others, below)
            const uint32_t st = ans ? scratch_stride((nv + 7) / 8) : 0u, si = warp_inclusive(st);
            if (listed) Q.src[v] = ans ? (8u * (scratch + si - st)) | 0x80000000u : (uint32_t)(sel_tot + inc - x);
            scratch += __shfl_sync(0xffffffffu, si, 31);
            scratch_tot += 16ull * __reduce_add_sync(0xffffffffu, st / 16);   // (32 strides of 2^29 bytes at most: 2^30)
            full += __reduce_add_sync(0xffffffffu, ans ? ans_full_segs((nv + 7) / 8) : 0u);
            lanes += __reduce_add_sync(0xffffffffu, ans ? ans_tail_lanes((nv + 7) / 8) : 0u);
            sel_tot += __shfl_sync(0xffffffffu, inc, 31);
        }
    }
    if (((base1 + raw_tot + sel_tot + 15) & ~15ull) != rb || scratch_tot > kScratchMax) bad = true;
    __syncwarp();
    if (nsel)
        for (uint32_t v = lane; v < V; v += 32)
            if (mks[v] == kMarkRawSel) Q.src[v] = 8u * (uint32_t)(base1 + raw_tot + Q.src[v]);
    if (rb >= kRecFar && plan_far(g, V, nsel)) bad = true;
    // ---- symbols: their number within their length (rounds of 32), the tree, their order ----
    uint32_t rank[8];
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const int sym = 32 * j + lane;
        const uint32_t l = (g[kLensOff + (sym >> 1)] >> (4 * (sym & 1))) & 15u;
        const uint32_t peers = __match_any_sync(0xffffffffu, l), before = Q.run[l];
        const uint32_t r = __popc(peers & ((1u << lane) - 1u));
        rank[j] = (l << 16) | (before + r);
        __syncwarp();
        if (r == 0) Q.run[l] = before + __popc(peers);
        __syncwarp();
    }
    plan_tree(lane >= 1 && lane < 16 ? Q.run[lane] : 0u, flat, V, Q.tree);
    if (!Q.tree.good) return R;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const uint32_t l = rank[j] >> 16;
        if (l) Q.sorted[(Q.tree.start[l] + (rank[j] & 0xFFFFu)) & 255u] = (uint8_t)(32 * j + lane);
    }
    __syncwarp();
    if (flat) {
        plan_flat(Q.tree, Q.sorted, V, Q.F);
        if (!Q.tree.good) return R;
    }
    // ---- children of every node and the symbols of each depth ----
    int d = 0;   // depth of node v (v grows, so the search goes on from the last one)
    for (uint32_t v = lane; v < V; v += 32) {
        uint32_t chv = 0;
        if (flat) {
            if (!flat_node(Q.F, Q.sorted, (int)v, d, chv)) bad = true;
            const uint32_t D = ch_flat_d(chv);
            if (D != mark_flat_d(mks[v]) || (D && (chv & 0xFFu) + (1u << D) > (uint32_t)Q.tree.K)) bad = true;
        } else {
            while (d < 15 && Q.tree.first[d + 1] <= (int)v) d++;
            if (!plan_children(Q.tree, Q.sorted, V, (int)v, d, chv)) bad = true;
        }
        if (d >= 1) atomicAdd(&Q.lvl[d], nvs[v]);
    }
    __syncwarp();
    if (__any_sync(0xffffffffu, bad)) return R;
    plan_tiles(Q.tree, Q.lvl, n, tile_max, R.T, R.ntile);
    if (R.ntile > 1 || all_dirs) {
        for (uint32_t v = lane; v < V; v += 32) ent += (nvs[v] + dir_bits - 1) / dir_bits;
        ent = __reduce_add_sync(0xffffffffu, ent);
    }
    R.ent = ent;
    R.dir_bytes = ntab_bytes(V) + (ent ? ((4ull * ent + 4ull * (R.ntile + 1) * V + 15) & ~15ull) : 0ull);
    R.scratch = scratch;
    R.nsegs = ans_units(full, lanes);
    R.V = V;
    R.n = n;
    R.st = PIVCO_OK;
    __syncwarp();
    return R;
}

// Plans blocks 8 item .. 8 item + 7 (the whole CTA, one warp each) and writes
// their offsets, statuses, node tables and plan_done flags.  Returns the
// number of this item's blocks whose tiles wait for ANS segments or a
// directory (thread 0).
__device__ __noinline__ void plan_item(int item, const uint8_t *__restrict__ comp,
                                       const uint64_t *__restrict__ comp_off, int nblk, uint8_t *__restrict__ ws,
                                       uint64_t ws_bytes, int32_t *__restrict__ status) {
    PlanItemSm &I = smem_item<PlanItemSm>();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = item * kDecWarps + warp;
    uint32_t *hdr32 = reinterpret_cast<uint32_t *>(ws);
    uint64_t *hdr64 = reinterpret_cast<uint64_t *>(ws);
    const DecWs W = dec_ws(ws, nblk);
    const uint32_t dir_bits = dec_dir_bits(ws);
    const bool all_dirs = dec_all_dirs(ws), have = b < nblk;
    PlanWarpSm &Q = I.w[warp];
    PlanRes R{};
    if (have) R = plan_warp(comp + comp_off[b], comp_off[b + 1] - comp_off[b], dir_bits, hdr32[8], all_dirs, Q);
    if (lane == 0) {
        I.agg[warp][0] = ((uint64_t)R.scratch << 22) | R.nsegs;
        I.agg[warp][1] = have ? (R.dir_bytes << 22) | R.ntile : 0ull;
    }
    __syncthreads();
    uint64_t ta = 0, tb = 0, pa = 0, pb = 0;   // the item's sums, and those before this warp's block
#pragma unroll
    for (int w = 0; w < kDecWarps; w++) {
        const uint64_t xa = I.agg[w][0], xb = I.agg[w][1];
        if (w < warp) { pa += xa; pb += xb; }
        ta += xa;
        tb += xb;
    }
    if (threadIdx.x == 0) lb2_publish(W.states_a, W.states_b, item, ta, tb);
    uint64_t ea, eb;
    const bool to = lookback2_cta(W.states_a, W.states_b, item, ta, tb, ea, eb, hdr64[7], I.mins, I.sums);
    ea += pa;
    eb += pb;
    if (have) {
        const bool ok = R.st == PIVCO_OK;
        if (lane == 0) {
            W.blk_scratch[b] = ea >> 22;
            W.blk_seg[b] = (uint32_t)(ea & ((1u << 22) - 1));
            W.blk_dir[b] = eb >> 22;
            W.blk_tile[b] = (uint32_t)(eb & ((1u << 22) - 1));
            W.blk_T[b] = R.T;
            W.blk_ntile[b] = R.ntile;
            status[b] = !ok ? R.st : (to ? PIVCO_ERR_TIMEOUT : PIVCO_OK);
            if (b == nblk - 1) {
                hdr64[0] = (ea >> 22) + R.scratch;
                hdr32[2] = (uint32_t)((ea & ((1u << 22) - 1)) + R.nsegs);
                hdr64[2] = (eb >> 22) + R.dir_bytes;
                hdr32[6] = (uint32_t)((eb & ((1u << 22) - 1)) + R.ntile);
                // totals from a partial prefix are unusable: every later pass
                // gives the whole batch up (abandoned_batch)
                if (to) atomicExch(&hdr32[13], 1u);
            }
        }
        // the node table (only where the workspace holds it: a sizing run may
        // not; and never from a partial prefix, which would place it over
        // another block's table)
        const uint64_t nbase = decode_ws_fixed_bytes(nblk) + (eb >> 22);
        if (ok && R.kind == 2 && !to && nbase + ntab_bytes(R.V) <= ws_bytes) {
            uint8_t *nt = ws + nbase;
            if (lane < 17) nt[lane] = (uint8_t)Q.tree.first[lane];
            if (lane == 17) nt[17] = (uint8_t)Q.tree.maxd;
            if (lane == 0) {
                *reinterpret_cast<uint32_t *>(nt + 20) = R.ent;
                *reinterpret_cast<uint32_t *>(nt + 24) = R.T;
            }
            uint32_t *src = reinterpret_cast<uint32_t *>(nt + kNtabHdr);
            const uint32_t *nvs = reinterpret_cast<const uint32_t *>(Q.stg + kNvOff);
            uint32_t u = 0;
            int d = 0;
            for (uint32_t v0 = 0; v0 < R.V; v0 += 32) {
                const uint32_t v = v0 + lane;
                uint32_t ui = 0, chv = 0;
                if (v < R.V) {   // (again: eight warps' children words would not fit beside their stages)
                    if (Q.stg[15] == '2') {
                        flat_node(Q.F, Q.sorted, (int)v, d, chv);
                    } else {
                        while (d < 15 && Q.tree.first[d + 1] <= (int)v) d++;
                        plan_children(Q.tree, Q.sorted, R.V, (int)v, d, chv);
                    }
                }
                if (R.ent) {
                    const uint32_t x = v < R.V ? (nvs[v] + dir_bits - 1) / dir_bits : 0u, inc = warp_inclusive(x);
                    ui = u + inc - x;
                    u += __shfl_sync(0xffffffffu, inc, 31);
                }
                if (v < R.V) {
                    src[3 * v] = Q.src[v];
                    src[3 * v + 1] = chv;
                    src[3 * v + 2] = ui;
                }
            }
            uint32_t *sym = src + 3 * R.V;
            for (int i = lane; i < 64; i += 32) sym[i] = reinterpret_cast<const uint32_t *>(Q.sorted)[i];
        }
        __syncwarp();
        // the plan is complete (status, offsets, node table); a block of one tile
        // with no ANS segment and no directory can be decoded from here on
        if (lane == 0) {
            const bool simple = ok && !to && R.ntile == 1 && R.nsegs == 0 && !all_dirs;
            __threadfence();
            // (4: the block's item has given up waiting for this plan, and will not come again)
            if ((atomicOr(&W.plan_done[b], simple ? 3u : 1u) & 4u) && ok) status[b] = PIVCO_ERR_TIMEOUT;
        }
    }
}

// Batches of more records than this many per SM are planned by warps
constexpr int kPlanCtaPerSm = 4;

__global__ void __launch_bounds__(kDecThreads) decode_plan_kernel(const uint8_t *__restrict__ comp,
                                                                  const uint64_t *__restrict__ comp_off, int nblk,
                                                                  uint8_t *__restrict__ ws, uint64_t ws_bytes,
                                                                  int32_t *__restrict__ status) {
    __shared__ int s_tile;
    if (threadIdx.x == 0) s_tile = (int)atomicAdd(&reinterpret_cast<uint32_t *>(ws)[3], 1u);
    __syncthreads();
    const int b = s_tile;
    const DecWs W = dec_ws(ws, nblk);
    const PlanRes R = plan_cta(comp + comp_off[b], comp_off[b + 1] - comp_off[b], dec_dir_bits(ws),
                               reinterpret_cast<const uint32_t *>(ws)[8], dec_all_dirs(ws));
    if (threadIdx.x == 0) plan_publish(W, b, R);
    uint64_t nbase;
    const bool ok = plan_place(b, nblk, ws, ws_bytes, R, true, nbase);
    if (threadIdx.x == 0) status[b] = R.st != PIVCO_OK ? R.st : (ok ? PIVCO_OK : PIVCO_ERR_TIMEOUT);
}

__global__ void __launch_bounds__(kDecThreads) decode_plan_items_kernel(const uint8_t *__restrict__ comp,
                                                                        const uint64_t *__restrict__ comp_off, int nblk,
                                                                        uint8_t *__restrict__ ws, uint64_t ws_bytes,
                                                                        int32_t *__restrict__ status) {
    __shared__ int s_item;
    if (threadIdx.x == 0) s_item = (int)atomicAdd(&reinterpret_cast<uint32_t *>(ws)[3], 1u);
    __syncthreads();
    plan_item(s_item, comp, comp_off, nblk, ws, ws_bytes, status);
}

// zero the header, the look-back states and the batch counters; set the
// tuning and the wait bound
__global__ void dec_ws_init_kernel(uint8_t *ws, int nblk, uint32_t dir_bits, uint32_t tile_max, uint64_t limit_ns) {
    const DecWs W = dec_ws(ws, nblk);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nblk; i += gridDim.x * blockDim.x) {
        W.states_a[i] = 0;
        W.states_b[i] = 0;
        W.segs_done[i] = 0;
        W.dir_done[i] = 0;
        W.plan_done[i] = 0;
    }
    if (blockIdx.x == 0 && threadIdx.x < 16) {
        uint32_t *h = reinterpret_cast<uint32_t *>(ws);
        h[threadIdx.x] = threadIdx.x == 7 ? dir_bits : (threadIdx.x == 8 ? tile_max : 0u);
        if (threadIdx.x == 14) h[14] = (uint32_t)limit_ns;
        if (threadIdx.x == 15) h[15] = (uint32_t)(limit_ns >> 32);
    }
}

// True when the plan could not place the batch (a look-back wait ran out
// before the last block's prefix was known) or a CTA of the batched queue
// gave up: the workspace totals and offsets are not to be used.  The caller
// marks every block that still reads OK as timed out (grid-stride, all CTAs
// of a pass may do it) and leaves.  A uniform decision: the flag is set
// before the pass starts, or (batched) before all plans are counted done.
__device__ inline bool abandoned_batch(const uint8_t *ws, int32_t *status, int nblk) {
    if (!*reinterpret_cast<const volatile uint32_t *>(ws + 52)) return false;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nblk; b += gridDim.x * blockDim.x)
        if (*reinterpret_cast<volatile int32_t *>(&status[b]) == PIVCO_OK) status[b] = PIVCO_ERR_TIMEOUT;
    return true;
}

cudaError_t launch_decode_plan(const uint8_t *comp, const uint64_t *comp_off, int nblk, uint8_t *ws, size_t ws_bytes,
                               int32_t *status, cudaStream_t st, bool all_dirs) {
    if (nblk <= 0) return cudaSuccess;
    const DecTuning tu = current_tuning();
    dec_ws_init_kernel<<<min(1024, div_up(nblk, 256)), 256, 0, st>>>(ws, nblk, tu.dir_bits | (all_dirs ? 1u << 31 : 0u),
                                                                      tu.tile_max, wait_limit_ns());
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (nblk <= kPlanCtaPerSm * sms) {
        decode_plan_kernel<<<nblk, kDecThreads, (int)(kSelBytes + sizeof(PlanSm)), st>>>(comp, comp_off, nblk, ws, ws_bytes, status);
    } else {
        const int smem = (int)(kSelBytes + sizeof(PlanItemSm));
        const cudaError_t e = cudaFuncSetAttribute(decode_plan_items_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        decode_plan_items_kernel<<<div_up(nblk, kDecWarps), kDecThreads, smem, st>>>(comp, comp_off, nblk, ws, ws_bytes,
                                                                                     status);
    }
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t read_decode_ws_need(const uint8_t *ws, int nblk, size_t *need, cudaStream_t st) {
    uint8_t h[32];
    cudaError_t e = cudaMemcpyAsync(h, ws, 32, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return e;
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    *need = dec_regions(nblk, h).need;
    return cudaSuccess;
}

// ---------------------------------------------------------------------------
// ANS pass: one warp per unit (ans_dev.cuh): a whole 16 KiB segment, or as
// many of a block's shorter segments as fit 32 lanes.
// What bounds it: the latency of a round's chain (state, class, table entry,
// word), about 380 cycles, 512 rounds a unit whatever its lanes.  2048 blocks
// of 128 KiB, P(0) = 0.95: 147 us before (one warp per segment, 73
// instructions a round), 102 us now (48, no branches in a round).  18 blocks of
// 67842 symbols, a root bitmap of 8.5 KB each: 138 us before, 101 now (153 with
// the words of a unit that does not fit the shared memory read from the record).
// ---------------------------------------------------------------------------
constexpr int kAnsWarps = kDecWarps;
struct AnsGroup {               // a segment of a unit
    uint32_t body, blen;        // its bitmap's ANS body in the record
    uint32_t raw, soff;         // bitmap bytes; where it goes in the block's scratch
    uint32_t s;                 // segment of the bitmap
    uint32_t lane0;             // its first lane
    uint32_t mk;                // marker
    uint32_t before;            // bytes of the body's segments before s
};
struct __align__(16) AnsWarpSm {
    union {
        // per group and class: frequency, start, ceil(2^31 / frequency), class
        // base; then windows of the groups' words
        uint4 tab[36][9];
        struct {
            uint4 tab0[9];
            uint16_t words[kAnsWordWin + 64];   // (a round past the last word reads on)
        } full;
    };
    AnsGroup grp[32];
    uint8_t of_lane[32];        // group of a lane (0xFF: none)
};
struct AnsItemSm {
    AnsWarpSm w[kAnsWarps];
    uint8_t member[256];        // bytes by (popcount, value)
};

// class tables of table id tid into tab (lane-strided)
__device__ inline void ans_tab(uint4 *tab, const AnsTables &A, uint32_t tid, uint32_t i0, uint32_t step) {
    for (uint32_t k = i0; k < 9; k += step)
        tab[k] = make_uint4(A.q[tid][k], A.start[tid][k], (0x80000000u + A.q[tid][k] - 1) / A.q[tid][k], A.class_base[k]);
}

// The classes' starts, two to a word, for ans_class.
struct AnsStarts {
    uint32_t p[4];              // starts of classes 2i + 1 (low half) and 2i + 2
};
// class of a slot: the number of starts at or below it.  Both halves of a
// word compare at once: with bit 15 set, slot - start keeps it exactly when
// slot >= start (slots below 2^15, starts up to 2^15).
__device__ inline uint32_t ans_class(const AnsStarts &s, uint32_t slot) {
    const uint32_t v = slot * 0x00010001u | 0x80008000u;
    const uint32_t m = ((v - s.p[0]) & 0x80008000u) | (((v - s.p[1]) & 0x80008000u) >> 1) |
                       (((v - s.p[2]) & 0x80008000u) >> 2) | (((v - s.p[3]) & 0x80008000u) >> 3);
    return __popc(m);
}
// One step of a state: the coded byte's place in `member`, the state before
// renormalisation.  The index rel / q is exact: q rel < 2^30 (a class holds at
// most 2^15 slots), so the error of the multiplier stays below one.
__device__ inline uint32_t ans_step(const uint4 *tab, const AnsStarts &s, uint32_t &x) {
    const uint32_t slot = x & (kAnsM - 1);
    const uint4 e = tab[ans_class(s, slot)];
    const uint32_t rel = slot - e.y, idx = __umulhi(2 * rel, e.z);
    x = e.x * (x >> kAnsScale) + (rel - idx * e.x);
    return e.w + idx;
}

__device__ inline void ans_members(AnsItemSm &I, const AnsTables &A) {
    for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x) I.member[i] = A.class_member[i];
}

// Decodes unit g (global numbering) into the scratch; returns its block.
// AnsItemSm::member must be loaded.
__device__ __noinline__ int ans_item(uint32_t g, const uint8_t *__restrict__ comp,
                                     const uint64_t *__restrict__ comp_off, int nblk, uint8_t *__restrict__ ws,
                                     uint64_t ws_bytes, int32_t *__restrict__ status, const AnsTables &A) {
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    AnsItemSm &I = smem_item<AnsItemSm>();
    AnsWarpSm &M = I.w[threadIdx.x >> 5];
    const DecWs W = dec_ws(ws, nblk);
    const DecRegions G = dec_regions(nblk, ws);
    const uint64_t scratch_cap = ws_bytes > G.scratch ? ws_bytes - G.scratch : 0;
    uint8_t *scratch = ws + G.scratch;
    const uint32_t total = reinterpret_cast<const uint32_t *>(ws)[2];
    const int b = find_block_warp(W.blk_seg, nblk, g, (int)((uint64_t)g * (uint32_t)nblk / max(total, 1u)));
    if (*reinterpret_cast<volatile int32_t *>(&status[b]) != PIVCO_OK) return b;
    const uint8_t *rec = comp + comp_off[b];   // (the plan has validated it)
    const uint32_t V = (uint32_t)rec[8] | ((uint32_t)rec[9] << 8), unit = g - W.blk_seg[b];
    const uint32_t *nvs = reinterpret_cast<const uint32_t *>(rec + kNvOff);
    const uint8_t *mks = rec + kNvOff + 4 * V;
    // ---- the block's whole segments and its last segments by size ----
    uint32_t full = 0, cnt[6] = {0u, 0u, 0u, 0u, 0u, 0u}, nsel = 0;
    uint64_t raw_tot = 0;
    for (uint32_t v0 = 0; v0 < V; v0 += 32) {
        const uint32_t v = v0 + lane, mk = v < V ? mks[v] : 0u, nv = v < V ? __ldg(nvs + v) : 0u, fd = mark_flat_d(mk);
        const bool ans = mark_ans(mk);
        const uint32_t raw = (nv + 7) / 8, tl = ans ? ans_tail_lanes(raw) : 0u;
        full += __reduce_add_sync(0xffffffffu, ans ? ans_full_segs(raw) : 0u);
#pragma unroll
        for (int c = 0; c < 6; c++) cnt[c] += __popc(__ballot_sync(0xffffffffu, tl == (1u << c)));
        nsel += __popc(__ballot_sync(0xffffffffu, mark_listed(mk)));
        // (bodies lie inside the record: their sizes add up below 2^32)
        raw_tot += __reduce_add_sync(0xffffffffu, mark_listed(mk) ? 0u : (uint32_t)(((uint64_t)nv * (fd ? fd : 1u) + 7) / 8));
    }
    uint32_t off[6];   // first lane of each size, largest first
    off[5] = 0;
#pragma unroll
    for (int c = 4; c >= 0; c--) off[c] = off[c + 1] + (cnt[c + 1] << (c + 1));
    const bool whole = unit < full;
    const uint32_t lanes0 = whole ? 0u : 32u * (unit - full);   // the unit's first lane
    // ---- this unit's segments ----
    const uint32_t alen_off = (kNvOff + 5 * V + 3) & ~3u, base2 = alen_off + 4 * nsel + (uint32_t)raw_tot;
    if (lane < 32) M.of_lane[lane] = 0xFF;
    __syncwarp();
    uint32_t ng = 0, np = 0, soff = 0, sel = 0, fl = 0;
    for (uint32_t v0 = 0; v0 < V; v0 += 32) {
        const uint32_t v = v0 + lane, mk = v < V ? mks[v] : 0u, nv = v < V ? __ldg(nvs + v) : 0u;
        const bool ans = mark_ans(mk), listed = mark_listed(mk);
        const uint32_t lm = __ballot_sync(0xffffffffu, listed);
        if (!lm) continue;
        const uint32_t raw = (nv + 7) / 8, tl = ans ? ans_tail_lanes(raw) : 0u;
        const uint32_t al = listed ? __ldg(reinterpret_cast<const uint32_t *>(rec + alen_off) + np + __popc(lm & lt)) : 0u;
        np += __popc(lm);
        const uint32_t ai = warp_inclusive(al), st = ans ? scratch_stride(raw) : 0u, si = warp_inclusive(st);
        const uint32_t fs = ans ? ans_full_segs(raw) : 0u, fi = warp_inclusive(fs);
        AnsGroup X;
        X.body = base2 + sel + ai - al;
        X.blen = al;
        X.raw = raw;
        X.soff = soff + si - st;
        X.mk = mk;
        X.lane0 = 0;
        X.s = 0;
        X.before = 0;
        bool mine = false;
        if (whole) {
            const uint32_t f0 = fl + fi - fs;
            mine = unit >= f0 && unit < f0 + fs;
            X.s = unit - f0;
        } else if (tl) {
            X.s = ans_full_segs(raw);
        }
        uint32_t l0 = 0;
#pragma unroll
        for (int c = 0; c < 6; c++) {
            const uint32_t m = __ballot_sync(0xffffffffu, tl == (1u << c));
            if (tl == (1u << c)) l0 = off[c] + (__popc(m & lt) << c);
            off[c] += __popc(m) << c;
        }
        if (!whole && tl && l0 >= lanes0 && l0 < lanes0 + 32) { mine = true; X.lane0 = l0 - lanes0; }
        const uint32_t mm = __ballot_sync(0xffffffffu, mine);
        if (mine) {
            const uint32_t gi = ng + __popc(mm & lt);
            M.grp[gi] = X;
            const uint32_t w = whole ? 32u : ans_seg_lanes(raw - X.s * kAnsSeg);
            for (uint32_t i = 0; i < w; i++) M.of_lane[X.lane0 + i] = (uint8_t)gi;
        }
        ng += __popc(mm);
        sel += __shfl_sync(0xffffffffu, ai, 31);
        soff += __shfl_sync(0xffffffffu, si, 31);
        fl += __shfl_sync(0xffffffffu, fi, 31);
    }
    __syncwarp();
    bool ok = ng > 0, room = true;
    for (uint32_t i = 0; i < ng; i++) {   // (bitmaps of several segments only)
        const AnsGroup X = M.grp[i];
        if (!X.s || 4ull * X.s > X.blen) continue;
        uint64_t acc = 0;
        for (uint32_t j = lane; j < X.s; j += 32) acc += 4ull * 32 + 2ull * ld_le32(rec + X.body + 4 * j);
        for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (acc > X.blen) ok = false;
        else if (lane == 0) M.grp[i].before = (uint32_t)acc;
    }
    __syncwarp();
    // ---- the lane's segment: its states and words ----
    const uint32_t gi = M.of_lane[lane];
    const bool on = gi != 0xFF;
    uint32_t sb = 0, nl = 1, li = 0, nw = 0, x = kAnsL;
    const uint8_t *words = rec;
    uint8_t *dst = scratch;
    uint8_t xr = 0;
    if (on) {
        const AnsGroup X = M.grp[gi];
        const uint64_t sdst = W.blk_scratch[b] + X.soff;
        const uint8_t *body = rec + X.body;
        const uint32_t S = ans_seg_count(X.raw);
        room = sdst + scratch_stride(X.raw) <= scratch_cap;
        sb = min(kAnsSeg, X.raw - X.s * kAnsSeg);
        nl = ans_seg_lanes(sb);
        li = lane - X.lane0;
        xr = (X.mk & 0x80) ? 0xFF : 0;
        if (4ull * S > X.blen) {
            ok = false;
        } else {
            const uint64_t sp = 4ull * S + X.before;
            nw = ld_le32(body + 4 * X.s);
            const uint64_t end = sp + 4ull * nl + 2ull * nw;
            if (end > X.blen || (X.s + 1 == S && end != X.blen)) {
                ok = false;
            } else {
                x = ld_le32(body + sp + 4 * li);
                words = body + sp + 4 * nl;
                if (x < kAnsL) ok = false;
            }
        }
        dst = scratch + sdst + (size_t)X.s * kAnsSeg;
    }
    if (__any_sync(0xffffffffu, !room)) {
        if (lane == 0) status[b] = PIVCO_ERR_CAPACITY;
        __syncwarp();
        return b;
    }
    if (__any_sync(0xffffffffu, !ok)) {
        if (lane == 0) status[b] = PIVCO_ERR_CORRUPT;
        __syncwarp();
        return b;
    }
    // (16 bytes after each bitmap read as zeros)
    if (on && sb + M.grp[gi].s * kAnsSeg == M.grp[gi].raw)
        for (uint32_t i = li; i < 16; i += nl) dst[sb + i] = 0;
    const uint32_t tid = on ? (M.grp[gi].mk & 0x7F) - 1 : 0u;
    uint32_t rd = 0;
    if (whole) {
        ans_tab(M.full.tab0, A, tid, lane, 32);
        __syncwarp();
        AnsStarts st;
#pragma unroll
        for (int i = 0; i < 4; i++) st.p[i] = M.full.tab0[2 * i + 1].y | (M.full.tab0[2 * i + 2].y << 16);
        // windows of kAnsWordWin words, copied as whole words of memory under a
        // funnel (the body starts at any byte); refilled between batches of
        // eight rounds, so that a round has no check and no branch
        constexpr uint32_t kBatch = 8;
        uint32_t wbase = 0, wlim = 0;   // words wbase .. wlim - 1 are staged
        const uint32_t *rend = reinterpret_cast<const uint32_t *>(rec + ld_le32(rec));   // (a multiple of 16 bytes)
        uint8_t *o = dst + lane;
        for (uint32_t r = 0; r < kAnsSeg / 32; r += kBatch) {
            if (rd + 32 * kBatch > wlim && wlim < nw) {   // (warp-uniform)
                __syncwarp();
                const uint8_t *p = words + 2ull * rd;
                const uint32_t sh = 8u * (uint32_t)(reinterpret_cast<uintptr_t>(p) & 3), n = min(kAnsWordWin, nw - rd);
                const uint32_t *q = reinterpret_cast<const uint32_t *>(p - sh / 8);
                uint32_t *d = reinterpret_cast<uint32_t *>(M.full.words);
#pragma unroll 8
                for (uint32_t i = lane; i < (n + 1) / 2; i += 32)
                    d[i] = __funnelshift_r(q + i < rend ? __ldg(q + i) : 0u, q + i + 1 < rend ? __ldg(q + i + 1) : 0u, sh);
                wbase = rd;
                wlim = rd + n;
                __syncwarp();
            }
            if (rd > wlim) { ok = false; break; }   // (a corrupt stream: more words than there are)
            const uint16_t *win = M.full.words - wbase;
#pragma unroll
            for (uint32_t j = 0; j < kBatch; j++) {
                const uint32_t by = I.member[ans_step(M.full.tab0, st, x)];
                const bool need = x < kAnsL;
                const uint32_t m = __ballot_sync(0xffffffffu, need);
                // (read by every lane; past the last word the count below is off and the stream refused)
                const uint32_t pos = min(rd + __popc(m & lt), wlim + 31u);
                const uint32_t y = (x << 16) | win[pos];
                x = need ? y : x;
                rd += __popc(m);
                o[32 * j] = (uint8_t)(by ^ xr);
            }
            o += 32 * kBatch;
        }
    } else {
        // the lane's group: its lanes and class tables
        const uint32_t gm = __match_any_sync(0xffffffffu, gi);
        if (on) ans_tab(M.tab[gi], A, tid, li, nl);
        __syncwarp();
        const uint4 *tab = M.tab[on ? gi : 0];
        AnsStarts st;
#pragma unroll
        for (int i = 0; i < 4; i++) st.p[i] = tab[2 * i + 1].y | (tab[2 * i + 2].y << 16);
        // the groups' words go through shared memory: each lane has q4 words of
        // memory of the space beside the tables (4 at least, 8 stream words),
        // a group its lanes' together; they are refilled between batches of
        // four rounds, all groups at once, so that a round has no check and no
        // branch: every lane takes the step and keeps it while its segment lasts
        constexpr uint32_t kBatch = 4;
        static_assert((sizeof(M.tab) - 32 * sizeof(M.tab[0])) / 4 / 32 * 2 >= kBatch, "a batch's words fit");
        const uint32_t q4 = (uint32_t)(sizeof(M.tab) - sizeof(M.tab[0]) * ng) / 4 / 32;
        uint32_t *area = reinterpret_cast<uint32_t *>(M.tab[ng]) + q4 * (on ? M.grp[gi].lane0 : 0u);
        const uint16_t *win = reinterpret_cast<const uint16_t *>(area);
        const uint32_t *rend = reinterpret_cast<const uint32_t *>(rec + ld_le32(rec));   // (a multiple of 16 bytes)
        const uint32_t rounds = __reduce_max_sync(0xffffffffu, (sb + nl - 1) / nl);
        const uint32_t mine_r = li < sb ? (sb - li + nl - 1) / nl : 0u;   // this lane's rounds
        uint32_t wbase = 0, wlim = 0;   // the group's words wbase .. wlim - 1 are staged
        uint8_t *o = dst + li;
        for (uint32_t r0 = 0; r0 < rounds; r0 += kBatch, o += kBatch * nl) {
            if (__any_sync(0xffffffffu, rd + kBatch * nl > wlim && wlim < nw)) {
                __syncwarp();
                // (here rd <= wlim <= nw: a batch takes kBatch nl words at most)
                const uint8_t *p = words + 2ull * rd;
                const uint32_t sh = 8u * (uint32_t)(reinterpret_cast<uintptr_t>(p) & 3), n = min(2 * q4 * nl, nw - min(rd, nw));
                const uint32_t *q = reinterpret_cast<const uint32_t *>(p - sh / 8);
                if (rd <= nw) {
#pragma unroll 8
                    for (uint32_t i = li; i < (n + 1) / 2; i += nl)
                        area[i] = __funnelshift_r(q + i < rend ? __ldg(q + i) : 0u, q + i + 1 < rend ? __ldg(q + i + 1) : 0u, sh);
                    wbase = rd;
                    wlim = rd + n;
                }
                __syncwarp();
            }
            uint32_t at[kBatch];
#pragma unroll
            for (uint32_t j = 0; j < kBatch; j++) {
                const bool active = r0 + j < mine_r;
                uint32_t xn = x;
                at[j] = ans_step(tab, st, xn);
                const bool need = active && xn < kAnsL;
                const uint32_t m = __ballot_sync(0xffffffffu, need) & gm;
                // (past the last word the count below is off and the stream refused)
                const uint32_t y = (xn << 16) | win[min(rd + __popc(m & lt), wlim) - wbase];
                x = active ? (need ? y : xn) : x;
                rd += __popc(m);
            }
            uint32_t by[kBatch];
#pragma unroll
            for (uint32_t j = 0; j < kBatch; j++) by[j] = I.member[at[j]] ^ xr;
            // a single lane's bytes follow one another: whole words (past the end: the zeros)
            if (nl == 1) {
                uint32_t acc = 0;
#pragma unroll
                for (uint32_t j = 0; j < kBatch; j++) acc |= r0 + j < mine_r ? by[j] << (8 * j) : 0u;
                if (r0 < mine_r) *reinterpret_cast<uint32_t *>(dst + r0) = acc;
            } else {
#pragma unroll
                for (uint32_t j = 0; j < kBatch; j++)
                    if (r0 + j < mine_r) o[j * nl] = (uint8_t)by[j];
            }
        }
    }
    if (on && (x != kAnsL || rd != nw)) ok = false;
    if (__any_sync(0xffffffffu, !ok) && lane == 0) status[b] = PIVCO_ERR_CORRUPT;
    __syncwarp();
    return b;
}

__global__ void __launch_bounds__(32 * kAnsWarps) ans_decode_planned_kernel(const uint8_t *__restrict__ comp,
                                                                            const uint64_t *__restrict__ comp_off,
                                                                            int nblk, uint8_t *__restrict__ ws,
                                                                            uint64_t ws_bytes,
                                                                            int32_t *__restrict__ status,
                                                                            const __grid_constant__ AnsTables A) {
    if (abandoned_batch(ws, status, nblk)) return;
    const int w = threadIdx.x >> 5;
    const uint32_t total = reinterpret_cast<const uint32_t *>(ws)[2];
    if (blockIdx.x * kAnsWarps >= total) return;
    ans_members(smem_item<AnsItemSm>(), A);
    __syncthreads();
    for (uint32_t g = blockIdx.x * kAnsWarps + w; g < total; g += gridDim.x * kAnsWarps)
        ans_item(g, comp, comp_off, nblk, ws, ws_bytes, status, A);
}

cudaError_t launch_ans_decode_planned(const uint8_t *comp, const uint64_t *comp_off, int nblk, uint8_t *ws,
                                      size_t ws_bytes, int32_t *status, cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int smem = (int)(kSelBytes + sizeof(AnsItemSm));
    const cudaError_t e = cudaFuncSetAttribute(ans_decode_planned_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    ans_decode_planned_kernel<<<sms * 4, 32 * kAnsWarps, smem, st>>>(
        comp, comp_off, nblk, ws, ws_bytes, status, host_ans_tables());
    count_launches(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// CTA tiles (the bottom-up merge, Sec. 3)
//
// A tile is decoded by one CTA.  Its levels live in two shared-memory level
// buffers; bottom-up, each level is split into windows of 32 groups (a group
// is 32 consecutive symbols of one node: one lane's bitmap word).  The ordinary nodes
// of a level share its windows; a flat node has windows of its own, so that
// all lanes of a window unpack the same index width.  The warps take a
// level's windows in rounds of eight: each warp counts the ones of its
// window's bitmap words; after one barrier every warp has the prefix of the
// round's window counts, from which a group's rank is its window's prefix
// plus the in-window scan, less the same sum at its node's start.  The barrier that publishes a round's counts also orders the
// level below's symbols before their reads, so a level costs one barrier per
// eight windows and no more.  The root, one node with most of the windows, is
// counted first and then merged without any barrier.  The symbols of a window are merged in four
// steps of 256: in a step a lane makes 8 consecutive symbols, the word and
// the child positions coming from the lane that owns the group by shuffle.
// Neighbouring lanes then read neighbouring bytes of the children and write
// neighbouring bytes, so a shared-memory access is one or two wavefronts; with
// 32 symbols to a lane the lanes were 16 bytes apart on each side and every
// access took four (134 wavefronts for 1024 symbols, now about 50).
//
// What bounds it: instruction issue (65 % of the slots used on text-like
// blocks, about 400 instructions for 1024 symbols of a level); on small
// trees with many short levels also the barriers between them.  509 blocks of
// 20-300 KB, 60-120 symbols, canonical tree: 377 us before, 220 us now.
// ---------------------------------------------------------------------------
constexpr int kTileWarps = kDecWarps;
static_assert(kTileWarps == kLvlWarps, "the level tables are laid out by all warps");
constexpr int kStripMax = 256;                 // strips of root windows (a window each up to 2^18 symbols)

struct TileSrc {
    const uint8_t *rec;
    const uint8_t *scr;
    uint64_t scr_bytes;
    uint32_t rec_bytes;
};

// The tile at hand: filled by tile_open or block_open, decoded by ct_decode
// (one inlined copy in each kernel), ended by tile_close or block_close.
struct TileJob {
    TileSrc src;
    uint8_t *dst;
    uint32_t V, P0, P1, k;
    int32_t b;
};

struct __align__(16) CtaTile {
    static constexpr int kBuf = kLvlBuf;
    uint8_t buf[2][kLvlBuf + kWSlack];         // level buffers: depth d writes buf[d & 1]
    uint32_t pos[256];                         // bit address of node v's next bit (bit 31: in the ANS scratch)
    uint32_t dem[256];                         // bits of node v in the current chunk
    uint32_t ch[256];                          // children (node table format)
    uint32_t end[256];                         // bit address of the end of node v's bits in the tile
    uint32_t strip[kStripMax];                 // ones of the root before each strip of windows
    uint32_t wtot[2][kTileWarps];              // ones of a round's ordinary windows, two rounds deep
    uint16_t sp[256];                          // byte offset of node v's sequence in its level buffer
    uint16_t gs[256];                          // first group of the level's i-th ordinary node (at first[d] + i);
    uint16_t fw[256];                          // flat node: its first window among the level's flat windows;
                                               // ordinary node: ones between its window's start and its first group
    uint16_t wpre[kWinMax];                    // prefixes of earlier rounds (levels of more than 8 windows)
    uint16_t lg[16], no[16];                   // groups and number of ordinary nodes of each level
    uint16_t nwo[16], nw[16];                  // ordinary windows, windows of each level
    uint16_t wn_off[16];                       // first window entry of each level
    uint8_t onode[256];                        // the level's i-th ordinary node (at first[d] + i)
    uint8_t wnode[kWinMax];                    // ordinary window: index of the node holding its first group; flat: node
    uint8_t ftab[256];                         // the block's symbols in (length, symbol) order (flat nodes)
    uint8_t first[17];
    uint8_t maxd;
    uint8_t pad[2];
    int32_t blk, flag;
    uint32_t rtot;                             // ones of the root in the chunk
    TileJob job;
};
static_assert(offsetof(CtaTile, pos) % 16 == 0, "level buffers of whole vectors");

// Byte-permute selectors of a bitmap byte (low 16 bits: its low nibble,
// high 16 bits: its high nibble): a one takes the next byte of the right
// window (bytes 4..7), a zero the next byte of the left window (bytes 0..3).
// A leaf side's window is its symbol in all four bytes, so one table serves
// every kind of children.
__device__ inline void sel_init(uint32_t *sel) {
    const int t = threadIdx.x;
    for (int b8 = t; b8 < 256; b8 += blockDim.x) {
        uint32_t pair = 0;
        for (int h = 0; h < 2; h++) {
            const uint32_t nib = (b8 >> (4 * h)) & 15u;
            uint32_t s = 0, ones = 0, zeros = 0;
            for (int j = 0; j < 4; j++) {
                const uint32_t bit = (nib >> j) & 1u;
                s |= (bit ? 4 + ones : zeros) << (4 * j);
                ones += bit;
                zeros += 1 - bit;
            }
            pair |= s << (16 * h);
        }
        sel[b8] = pair;
    }
}

// The two words under 32 bits of a node bitmap from bit address pos + k (bit
// 31 of pos: scratch), loaded ahead of their use.  The bits lie inside the
// node's body (the plan has checked the bodies against the record, the tile
// its cursors against the bodies, and ct_demand the demands of a shorter
// chunk against the tile's end cursors before anything of it is read), so
// only the second word can run past the end; bit addresses stay below 2^31.
struct BitLd {
    uint32_t lo, hi, sh;
};
__device__ inline BitLd tile_ld(const TileSrc &s, uint32_t pos, uint32_t k) {
    const uint32_t e = (pos & 0x7FFFFFFFu) + k, wi = e >> 5;
    BitLd b;
    b.sh = e & 31u;
    b.lo = b.hi = 0;
    if (pos >> 31) {   // written during this launch by other CTAs: through L2
        const uint32_t *w = reinterpret_cast<const uint32_t *>(s.scr) + wi;
        if (4ull * wi + 4 <= s.scr_bytes) b.lo = __ldcg(w);
        if (b.sh && 4ull * wi + 8 <= s.scr_bytes) b.hi = __ldcg(w + 1);
    } else {
        const uint32_t *w = reinterpret_cast<const uint32_t *>(s.rec) + wi;
        b.lo = __ldca(w);
        if (wi + 1 < s.rec_bytes >> 2) b.hi = __ldca(w + 1);
    }
    return b;
}
__device__ inline uint32_t tile_word(const BitLd &b) { return __funnelshift_r(b.lo, b.hi, b.sh); }
__device__ inline uint32_t tile_bits(const TileSrc &s, uint32_t pos, uint32_t k) { return tile_word(tile_ld(s, pos, k)); }

// popcount of bits [e, e + len) (len <= 32 (kW - 1)) of the bitmap at bit
// address pos: the covering words are loaded together, then counted
template <int kW>
__device__ inline uint32_t tile_popc_w(const TileSrc &s, uint32_t pos, uint32_t e, uint32_t len) {
    const bool sc = (pos >> 31) != 0;
    const uint64_t a = (uint64_t)(pos & 0x7FFFFFFFu) + e;
    const uint64_t w0 = a >> 5;
    const uint32_t sh = (uint32_t)a & 31u;
    const uint32_t *w = reinterpret_cast<const uint32_t *>(sc ? s.scr : s.rec);
    const uint64_t lim = sc ? s.scr_bytes : (uint64_t)s.rec_bytes;
    const uint32_t nw = (sh + len + 31) >> 5;   // words holding the range (<= kW)
    uint32_t x[kW];
#pragma unroll
    for (int i = 0; i < kW; i++) x[i] = ((uint32_t)i < nw && 4 * (w0 + i) + 4 <= lim) ? __ldcg(w + w0 + i) : 0u;
    // all bits of the loaded words, less those before sh in the first and
    // those from sh + len on in the last
    uint32_t c = 0, xl = 0;
#pragma unroll
    for (int i = 0; i < kW; i++) {
        c += __popc(x[i]);
        xl = (uint32_t)i + 1 == nw ? x[i] : xl;
    }
    c -= __popc(x[0] & ((1u << sh) - 1u));
    const uint32_t eb = (sh + len) & 31u;
    if (eb) c -= __popc(xl >> eb);
    return c;
}
// (len <= 256; directories are built and used with fewer bits than that, as a rule 128)
__device__ inline uint32_t tile_popc(const TileSrc &s, uint32_t pos, uint32_t e, uint32_t len) {
    return tile_popc_w<9>(s, pos, e, len);
}

// 8 bytes of a level buffer from byte a (reads up to 11 bytes past a)
__device__ inline void win8(const uint8_t *buf, uint32_t a, uint32_t &x0, uint32_t &x1) {
    const uint32_t *w = reinterpret_cast<const uint32_t *>(buf + (a & ~3u));
    const uint32_t sh = a * 8u;   // (the funnel takes it modulo 32)
    const uint32_t w0 = w[0], w1 = w[1], w2 = w[2];
    x0 = __funnelshift_r(w0, w1, sh);
    x1 = __funnelshift_r(w1, w2, sh);
}

// 8 output symbols of a node from bitmap byte b8: la / ra the left / right
// child's next byte in the level below, unless that child is a leaf (its
// symbol then fills kl / kr).  HL / HR: some lane of the warp has an internal
// left / right child.
template <bool HL, bool HR>
__device__ inline uint2 merge8(const uint8_t *bin, uint32_t la, uint32_t ra, bool i0, bool i1, uint32_t kl, uint32_t kr,
                               uint32_t b8, const uint32_t *sel) {
    const uint32_t p0 = __popc(b8 & 15u);
    uint32_t L0 = kl, R0 = kr, Lh = kl, Rh = kr;
    if (HL) {
        uint32_t x0, x1;
        win8(bin, la, x0, x1);
        L0 = i0 ? x0 : kl;
        Lh = i0 ? __funnelshift_rc(x0, x1, 32u - 8u * p0) : kl;
    }
    if (HR) {
        uint32_t x0, x1;
        win8(bin, ra, x0, x1);
        R0 = i1 ? x0 : kr;
        Rh = i1 ? __funnelshift_rc(x0, x1, 8u * p0) : kr;
    }
    const uint32_t sp = sel[b8];
    return make_uint2(__byte_perm(L0, R0, sp), __byte_perm(Lh, Rh, sp >> 16));
}

// The symbols of a window's groups: lane l owns a group of nsym symbols
// (0..32) of bitmap word w with its children's next bytes (or leaf symbols)
// a = left | right << 16 and flags i0 / i1; put(owner lane, byte, 8 symbols)
// takes the symbols 8 byte .. 8 byte + 7 of the owner's group.
template <bool HL, bool HR, typename F>
__device__ inline void merge_window(const uint8_t *bin, uint32_t w, uint32_t a, uint32_t b, const uint32_t *sel, F put) {
    const int lane = threadIdx.x & 31;
    const uint32_t sub = lane & 3, below = (1u << (8 * sub)) - 1u;
#pragma unroll
    for (int s = 0; s < 4; s++) {
        const int own = 8 * s + (lane >> 2);
        const uint32_t ws = __shfl_sync(0xffffffffu, w, own), as = __shfl_sync(0xffffffffu, a, own),
                       bs = __shfl_sync(0xffffffffu, b, own);
        const uint32_t r = __popc(ws & below), x0 = as & 0xFFFFu, x1 = as >> 16;
        const bool i0 = HL && (bs & (1u << 22)), i1 = HR && (bs & (1u << 23));
        const uint2 o = merge8<HL, HR>(bin, i0 ? x0 + 8 * sub - r : 0u, i1 ? x1 + r : 0u, i0, i1, x0 * 0x01010101u,
                                       x1 * 0x01010101u, (ws >> (8 * sub)) & 0xFFu, sel);
        put(s, bs, o);
    }
}

// 8 output symbols of a flat node (Sec. 2.2.3, merge_flat_D): the D-bit
// indices at bit address pos (a raw body in the record; the first index lies
// inside it, as for tile_ld), each mapped through the node's symbols
// tab[0 .. 2^D).  Neighbouring lanes read neighbouring bytes.
__device__ inline uint2 flat8(const TileSrc &s, uint32_t D, uint32_t pos, const uint8_t *tab) {
    const uint32_t e = pos & 0x7FFFFFFFu, wi = e >> 5, lim = s.rec_bytes >> 2;
    const uint32_t *w = reinterpret_cast<const uint32_t *>(s.rec) + wi;
    const uint32_t x0 = __ldca(w), x1 = wi + 1 < lim ? __ldca(w + 1) : 0u, x2 = wi + 2 < lim ? __ldca(w + 2) : 0u;
    const uint32_t b0 = __funnelshift_r(x0, x1, e), b1 = __funnelshift_r(x1, x2, e);   // (modulo 32)
    const uint32_t m = (1u << D) - 1u;
    const uint32_t c0 = b0, c1 = D == 8 ? b1 : __funnelshift_r(b0, b1, 4 * D);   // symbols 0..3, 4..7
    uint2 o;
    o.x = (uint32_t)tab[c0 & m] | ((uint32_t)tab[(c0 >> D) & m] << 8) | ((uint32_t)tab[(c0 >> (2 * D)) & m] << 16) |
          ((uint32_t)tab[(c0 >> (3 * D)) & m] << 24);
    o.y = (uint32_t)tab[c1 & m] | ((uint32_t)tab[(c1 >> D) & m] << 8) | ((uint32_t)tab[(c1 >> (2 * D)) & m] << 16) |
          ((uint32_t)tab[(c1 >> (3 * D)) & m] << 24);
    return o;
}

// the children's demands must be the node's zeros and ones
__device__ inline bool children_ok(const CtaTile &S, uint32_t chv, uint32_t dv, uint32_t ones) {
    const uint32_t c0 = chv & 0xFFFFu, c1 = chv >> 16;
    bool ok = true;
    if (!(c0 & 0x8000u)) ok = ok && S.dem[c0] == dv - ones;
    if (!(c1 & 0x8000u)) ok = ok && S.dem[c1] == ones;
    return ok;
}

// bytes j0 .. j1 - 1 of x at p + j0 ..
__device__ inline void st_bytes(uint8_t *p, uint64_t x, int j0, int j1) {
    for (int j = j0; j < j1; j++) p[j] = (uint8_t)(x >> (8 * j));
}

// The symbols of one step of a window (8 to a lane, 256 in all) at dst: lane
// l's belong at dst + 256 s + 8 l, the first nb bytes of the window exist.
// dst is `mis` bytes past an 8-byte boundary; when it is not 0 every lane
// stores the aligned word that its symbols begin in, completed with the lane
// before it (lane 0 with lane 31 of the step before, kept in `last`).
template <bool kMis>
__device__ inline void put_step(uint8_t *dst, int s, uint2 o, uint32_t nb, uint32_t mis, uint64_t &last) {
    const int lane = threadIdx.x & 31;
    const uint32_t c = 256u * s + 8u * lane;
    const uint64_t cur = o.x | ((uint64_t)o.y << 32);
    if (!kMis) {
        if (c + 8 <= nb) *reinterpret_cast<uint2 *>(dst + c) = o;
        else if (c < nb) st_bytes(dst + c, cur, 0, (int)(nb - c));
        return;
    }
    uint64_t prev = __shfl_up_sync(0xffffffffu, cur, 1);
    if (lane == 0) prev = last;
    last = __shfl_sync(0xffffffffu, cur, 31);
    // bytes c - mis .. c - mis + 7 of the window
    const uint64_t x = (prev >> (64 - 8 * mis)) | (cur << (8 * mis));
    const bool head = c == 0;
    if (!head && c - mis + 8 <= nb) *reinterpret_cast<uint64_t *>(dst + c - mis) = x;
    else if (c < nb + mis) st_bytes(dst + c - mis, x, head ? (int)mis : 0, (int)min(8u, nb + mis - c));
    // the window's last bytes
    if (s == 3 && lane == 31 && nb + mis > 1024) st_bytes(dst + 1016, cur, 8 - (int)mis, (int)nb - 1016);
}

// Demands of a chunk of C root symbols from the current cursors, top-down:
// a node's popcount over its range splits its demand between its children
// (one warp).  False when a node's demand runs past its bits in the tile (the
// bitmaps above it are corrupt): it is found before the node is read, here
// or by the levels.
__device__ inline bool ct_demand(CtaTile &S, const TileSrc &src, uint32_t V, uint32_t C) {
    const int lane = threadIdx.x & 31;
    for (uint32_t v = lane; v < V; v += 32) S.dem[v] = 0;
    __syncwarp();
    if (lane == 0) S.dem[0] = C;
    __syncwarp();
    for (uint32_t v = 0; v < V; v++) {   // breadth-first: parents before children
        const uint32_t dv = S.dem[v], fD = ch_flat_d(S.ch[v]);
        if ((uint64_t)dv * max(1u, fD) > S.end[v] - S.pos[v]) return false;   // (the same in all lanes)
        if (fD) continue;   // a flat node has no children to split for
        uint32_t ones = 0;
        for (uint32_t e = 32 * lane; e < dv; e += 1024) {
            uint32_t w = tile_bits(src, S.pos[v], e);
            if (dv - e < 32) w &= (1u << (dv - e)) - 1u;
            ones += __popc(w);
        }
        ones = __reduce_add_sync(0xffffffffu, ones);
        if (lane == 0) {
            const uint32_t chv = S.ch[v];
            const uint32_t c0 = chv & 0xFFFFu, c1 = chv >> 16;
            if (!(c0 & 0x8000u)) S.dem[c0] = dv - ones;
            if (!(c1 & 0x8000u)) S.dem[c1] = ones;
        }
        __syncwarp();
    }
    return true;
}

// windows per strip of the root (so that there are at most kStripMax strips)
__device__ inline uint32_t strip_len(uint32_t nwin) { return (nwin + kStripMax - 1) / kStripMax; }

// the bitmap word of this lane's group in root window i (dv symbols in all)
__device__ inline uint32_t root_mask(uint32_t w, uint32_t kk, uint32_t dv) {
    if (kk >= dv) return 0u;
    return dv - kk < 32 ? w & ((1u << (dv - kk)) - 1u) : w;
}

// Ones of every strip of the root, turned into prefixes (the whole CTA; ends
// with a barrier).
__device__ inline void ct_count_root(CtaTile &S, const TileSrc &src) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t dv = S.dem[0], pos = S.pos[0];
    const uint32_t nwin = (dv + kWin - 1) / kWin, m = strip_len(nwin), nstrip = (nwin + m - 1) / m;
    // (m is 1 but for tiles above 2^18 symbols)
    for (uint32_t s = warp; s < nstrip; s += 4 * kTileWarps) {
        uint32_t c[4] = {0u, 0u, 0u, 0u};
        for (uint32_t j = 0; j < m; j++) {
            uint32_t k[4];
            BitLd b[4];
#pragma unroll
            for (int r = 0; r < 4; r++) {   // four strips' loads in flight
                const uint32_t win = (s + r * kTileWarps) * m + j;
                k[r] = kWin * win + kGrp * lane;
                b[r] = BitLd{0u, 0u, 0u};
                if (k[r] < dv) b[r] = tile_ld(src, pos, k[r]);
            }
#pragma unroll
            for (int r = 0; r < 4; r++) c[r] += __popc(root_mask(tile_word(b[r]), k[r], dv));
        }
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const uint32_t x = __reduce_add_sync(0xffffffffu, c[r]);
            if (lane == 0 && s + r * kTileWarps < nstrip) S.strip[s + r * kTileWarps] = x;
        }
    }
    __syncthreads();
    if (warp == 0) {   // 8 strips to a lane
        uint32_t x[kStripMax / 32], sum = 0;
#pragma unroll
        for (int j = 0; j < kStripMax / 32; j++) {
            const uint32_t i = kStripMax / 32 * lane + j;
            x[j] = i < nstrip ? S.strip[i] : 0u;
            sum += x[j];
        }
        const uint32_t inc = warp_inclusive(sum);
        uint32_t run = inc - sum;
#pragma unroll
        for (int j = 0; j < kStripMax / 32; j++) {
            const uint32_t i = kStripMax / 32 * lane + j;
            if (i < nstrip) S.strip[i] = run;
            run += x[j];
        }
        if (lane == 31) S.rtot = inc;
    }
    __syncthreads();
}

// The root level of the current chunk into the output: the warps take its
// strips in turn, no barriers.  HL / HR: the left / right child is internal.
template <bool HL, bool HR, bool kMis>
__device__ __forceinline__ void ct_root(CtaTile &S, const TileSrc &src, uint8_t *out, const uint32_t *sel) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint8_t *bin = S.buf[1];
    const uint32_t dv = S.dem[0], chv = S.ch[0], pos = S.pos[0];
    const uint32_t nwin = (dv + kWin - 1) / kWin, m = strip_len(nwin);
    const uint32_t c0 = chv & 0xFFFFu, c1 = chv >> 16, kl = (c0 & 0xFFu) * 0x01010101u, kr = (c1 & 0xFFu) * 0x01010101u;
    const uint32_t s0 = HL ? (uint32_t)S.sp[c0 & 0xFFu] : 0u, s1 = HR ? (uint32_t)S.sp[c1 & 0xFFu] : 0u;
    const uint32_t sub = lane & 3, below = (1u << (8 * sub)) - 1u;
    const uint32_t mis = kMis ? (uint32_t)(reinterpret_cast<uintptr_t>(out) & 7) : 0u;
    BitLd nx{0u, 0u, 0u};
    if (kWin * m * warp + kGrp * lane < dv) nx = tile_ld(src, pos, kWin * m * warp + kGrp * lane);
    for (uint32_t s = warp; s * m < nwin; s += kTileWarps) {
        uint32_t carry = HL || HR ? S.strip[s] : 0u;
        const uint32_t iend = min(nwin, (s + 1) * m);
        for (uint32_t i = s * m; i < iend; i++) {
            const uint32_t w = root_mask(tile_word(nx), kWin * i + kGrp * lane, dv);
            const uint32_t kn = kWin * (i + 1 < iend ? i + 1 : (s + kTileWarps) * m) + kGrp * lane;
            if (kn < dv) nx = tile_ld(src, pos, kn);
            const uint32_t pc = __popc(w), inc = warp_inclusive(pc), r1 = carry + inc - pc;
            if (m > 1) carry += __shfl_sync(0xffffffffu, inc, 31);
            const uint32_t nb = min(kWin, dv - kWin * i);
            uint64_t last = 0;
#pragma unroll
            for (int st = 0; st < 4; st++) {
                const int own = 8 * st + (lane >> 2);
                const uint32_t ws = __shfl_sync(0xffffffffu, w, own);
                const uint32_t rs = __shfl_sync(0xffffffffu, r1, own) + __popc(ws & below);
                // (clamped: a corrupt bitmap must not send the reads past the buffer)
                const uint32_t la = HL ? min(s0 + kWin * i + 256u * st + 8u * lane - rs, (uint32_t)kLvlBuf) : 0u;
                const uint32_t ra = HR ? min(s1 + rs, (uint32_t)kLvlBuf) : 0u;
                const uint2 o = merge8<HL, HR>(bin, la, ra, HL, HR, kl, kr, (ws >> (8 * sub)) & 0xFFu, sel);
                put_step<kMis>(out + kWin * i, st, o, nb, mis, last);
            }
        }
    }
}
template <bool kMis>
__device__ __forceinline__ void ct_root_any(CtaTile &S, const TileSrc &src, uint8_t *out, const uint32_t *sel) {
    const uint32_t chv = S.ch[0], fD = ch_flat_d(chv);
    if (fD) {
        // the whole alphabet one group: indices straight to the output
        const uint32_t dv = S.dem[0], mis = (uint32_t)(reinterpret_cast<uintptr_t>(out) & 7);
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        for (uint32_t i = warp; kWin * i < dv; i += kTileWarps) {
            uint64_t last = 0;
            const uint32_t nb = min(kWin, dv - kWin * i);
#pragma unroll 1
            for (int st = 0; st < 4; st++) {
                const uint32_t kk = kWin * i + 256u * st + 8u * lane;
                uint2 o = make_uint2(0u, 0u);
                if (kk < dv) o = flat8(src, fD, S.pos[0] + kk * fD, S.ftab + (chv & 0xFFu));
                put_step<kMis>(out + kWin * i, st, o, nb, mis, last);
            }
        }
        return;
    }
    // one side is often a leaf (the most frequent symbol): it is not read at all
    const bool i0 = !(chv & 0x8000u), i1 = !(chv >> 31);
    if (i0 && i1) ct_root<true, true, kMis>(S, src, out, sel);
    else if (i1) ct_root<false, true, kMis>(S, src, out, sel);
    else if (i0) ct_root<true, false, kMis>(S, src, out, sel);
    else ct_root<false, false, kMis>(S, src, out, sel);
}

// One level (depth d >= 1) of the current chunk into its buffer.  par
// alternates the count slots.  Returns false when this thread found the
// level corrupt (the caller combines).
__device__ __forceinline__ bool ct_level(CtaTile &S, const TileSrc &src, int d, const uint32_t *sel, uint32_t &par) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint8_t *bin = S.buf[(d + 1) & 1];
    const uint32_t nw = S.nw[d], nwo = S.nwo[d], wn = S.wn_off[d], f0 = S.first[d];
    uint32_t carry = 0;   // ones of the rounds before
    bool bad = false;
    for (uint32_t base = 0; base < nw; base += kTileWarps) {
        const uint32_t i = base + warp;
        uint32_t v = 0, q = 0, w = 0, inc = 0, left = 0;   // left: symbols of the node from this group on (0: none)
        if (i < nwo) {
            left = lvl_locate(S, d, wn, f0, i, v, q);
            if (left) {
                w = tile_bits(src, S.pos[v], kGrp * q);
                if (left < 32) w &= (1u << left) - 1u;
            }
            const uint32_t pc = __popc(w);
            inc = warp_inclusive(pc);
            if (lane == 31) S.wtot[par][warp] = inc;
            inc -= pc;
            // a node's first group: the ones of the window before it
            if (q == 0) S.fw[v] = (uint16_t)inc;
        }
        __syncthreads();
        par ^= 1u;
        if (i < nwo) {
            // ones of the level before each window of the round (lane: window)
            uint32_t ex = 0, ps = 0;
            if (nwo > 1) {
                const uint32_t x = lane < kTileWarps && base + lane < nwo ? S.wtot[par ^ 1u][lane] : 0u;
                uint32_t in = x;
#pragma unroll
                for (int o = 1; o < kTileWarps; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, in, o);
                    if (lane >= o) in += y;
                }
                ex = carry + in - x;
                if (nwo > kTileWarps) {
                    carry += __shfl_sync(0xffffffffu, in, kTileWarps - 1);
                    if (warp == 0 && lane < kTileWarps && base + lane < nwo) S.wpre[wn + base + lane] = (uint16_t)ex;
                }
                // at the node's first group
                const uint32_t gw = (32u * i + lane - q) >> 5;   // its window
                ps = __shfl_sync(0xffffffffu, ex, gw - base);
                if (gw < base) ps = S.wpre[wn + gw];
                ex = __shfl_sync(0xffffffffu, ex, warp);
            }
            const uint32_t r1 = (ex + inc - ps - S.fw[v]) & 0xFFFFu;
            const uint32_t chv = S.ch[v], c0 = chv & 0xFFFFu, c1 = chv >> 16;
            const bool act = left != 0, i0 = act && !(c0 & 0x8000u), i1 = act && !(c1 & 0x8000u);
            if (act && left <= kGrp && !children_ok(S, chv, S.dem[v], r1 + __popc(w))) bad = true;
            const uint32_t la = i0 ? min((uint32_t)S.sp[c0 & 0xFFu] + kGrp * q - r1, (uint32_t)kLvlBuf) : c0 & 0xFFu;
            const uint32_t ra = i1 ? min((uint32_t)S.sp[c1 & 0xFFu] + r1, (uint32_t)kLvlBuf) : c1 & 0xFFu;
            const uint32_t a = la | (ra << 16);
            // bits 0..15: the group's place in its level buffer, 16..21: its symbols, 22 / 23: internal children
            const uint32_t b = (uint32_t)(S.sp[v] + (act ? kGrp * q : 0u)) | (min(left, kGrp) << 16) |
                               (i0 ? 1u << 22 : 0u) | (i1 ? 1u << 23 : 0u);
            // (spans are 16-byte aligned and a multiple of 16 bytes long)
            const uint32_t sub8 = 8u * (lane & 3);
            uint8_t *bout = S.buf[d & 1] + sub8;
            auto put = [&](int, uint32_t bs, uint2 o) {
                if (sub8 < ((bs >> 16) & 63u)) *reinterpret_cast<uint2 *>(bout + (bs & 0xFFFFu)) = o;
            };
            if (__any_sync(0xffffffffu, i0)) merge_window<true, true>(bin, w, a, b, sel, put);
            else if (__any_sync(0xffffffffu, i1)) merge_window<false, true>(bin, w, a, b, sel, put);
            else merge_window<false, false>(bin, w, a, b, sel, put);
        } else if (i < nw) {
            // a flat node's window: 8 symbols of a lane in each of four steps
            const uint32_t v2 = S.wnode[wn + i], chv = S.ch[v2], fD = ch_flat_d(chv), pos = S.pos[v2];
            const uint32_t k0 = (i - nwo - S.fw[v2]) * kWin, k1 = min(S.dem[v2], k0 + kWin);
            const uint8_t *tab = S.ftab + (chv & 0xFFu);
            uint8_t *bout = S.buf[d & 1] + S.sp[v2];
#pragma unroll 2
            for (uint32_t kk = k0 + 8u * lane; kk < k1; kk += 256)
                *reinterpret_cast<uint2 *>(bout + kk) = flat8(src, fD, pos + kk * fD, tab);
        }
    }
    return !bad;
}

// fills n bytes at p with x (whole CTA)
__device__ inline void cta_fill(uint8_t *p, uint32_t n, uint8_t x) {
    const int t = threadIdx.x;
    const uint32_t head = min(n, (uint32_t)((16 - (reinterpret_cast<uintptr_t>(p) & 15)) & 15));
    if (t < (int)head) p[t] = x;
    const uint32_t body = (n - head) / 16;
    const uint32_t x4 = x * 0x01010101u;
    uint4 *q = reinterpret_cast<uint4 *>(p + head);
    for (uint32_t i = t; i < body; i += blockDim.x) q[i] = make_uint4(x4, x4, x4, x4);
    for (uint32_t i = head + 16 * body + t; i < n; i += blockDim.x) p[i] = x;
}

// Decodes root symbols [P0, P1) into dst + P0 with the whole CTA: the tables
// (first, maxd, ftab, pos, end, dem, ch; the demands of the whole tile) are in
// S and checked.  kTileBad when the bitmaps are corrupt; kTileChunked when the
// tile went in several chunks, whose end the caller checks.
enum : int { kTileBad = 0, kTileOk = 1, kTileChunked = 2 };
__device__ __forceinline__ int ct_decode() {
    CtaTile &S = smem_item<CtaTile>();
    const uint32_t *sel = smem_sel();
    const TileSrc src = S.job.src;
    const uint32_t V = S.job.V, P0 = S.job.P0, P1 = S.job.P1;
    uint8_t *dst = S.job.dst;
    const int t = threadIdx.x, warp = t >> 5;
    uint32_t P = P0, C = P1 - P0, par = 0;
    bool chunked = false;
    // the whole tile at once when its levels fit, else chunks found top-down
    while (P < P1) {
        if (chunked) {
            const bool over = warp == 0 && !ct_demand(S, src, V, C);
            if (__syncthreads_or(over)) return kTileBad;
        }
        if (!lvl_layout(S)) {
            chunked = true;
            C = max(32u, (C / 2) & ~31u);
            continue;
        }
        bool ok = true;
        for (int d = S.maxd - 1; d >= 1; d--) ok = ct_level(S, src, d, sel, par) && ok;
        // (a flat root, or one of two leaves, needs no ranks and has no level below, which the barriers here also end)
        const bool ranked = (S.ch[0] & 0x80008000u) != 0x80008000u;
        if (ranked) ct_count_root(S, src);
        if (reinterpret_cast<uintptr_t>(dst + P) & 7) ct_root_any<true>(S, src, dst + P, sel);
        else ct_root_any<false>(S, src, dst + P, sel);
        if (ranked) ok = children_ok(S, S.ch[0], S.dem[0], S.rtot) && ok;
        if (__syncthreads_or(!ok)) return kTileBad;
        if ((uint32_t)t < V) S.pos[t] += S.dem[t] * max(1u, ch_flat_d(S.ch[t]));
        __syncthreads();
        P += C;
        C = min(C, P1 - P);
    }
    return chunked ? kTileChunked : kTileOk;
}

// pad bits of node v's body (nb bits from bit address s0) must be zero
__device__ inline bool pad_bad(const TileSrc &src, uint32_t s0, uint32_t nb) {
    return (nb & 7) && (tile_bits(src, s0, nb & ~7u) & 0xFFu) >> (nb & 7);
}

// A child never has more symbols than its parent, and the node table's
// levels are at most 16, first nodes non-decreasing up to V (thread t checks
// node t; true when something is wrong)
__device__ inline bool ct_tables_bad(const CtaTile &S, uint32_t V) {
    const int t = threadIdx.x;
    bool bad = false;
    if ((uint32_t)t < V) {
        const uint32_t chv = S.ch[t], c0 = chv & 0xFFFFu, c1 = chv >> 16;
        const uint32_t dc = ((c0 & 0x8000u) ? 0u : S.dem[c0 & 0xFFu]) + ((c1 & 0x8000u) ? 0u : S.dem[c1 & 0xFFu]);
        if (dc > S.dem[t]) bad = true;
    }
    if (t == 0 && (S.maxd < 1 || S.maxd > 16 || S.first[0] != 0 || S.first[S.maxd] != V)) bad = true;
    if (t >= 1 && t <= 16 && t <= S.maxd && S.first[t] < S.first[t - 1]) bad = true;
    return bad;
}

// where a tile's tables come from (nt: the block's node table)
struct TileTabs {
    const uint8_t *nt;
    const uint32_t *nsrc, *nv, *cursors;
};
__device__ inline TileTabs tile_tabs(const uint8_t *ws, int nblk, int b, const uint8_t *rec, uint32_t V) {
    const DecWs W = dec_ws(const_cast<uint8_t *>(ws), nblk);
    TileTabs T;
    T.nt = ws + dec_regions(nblk, ws).dir + W.blk_dir[b];
    T.nsrc = reinterpret_cast<const uint32_t *>(T.nt + kNtabHdr);
    T.nv = reinterpret_cast<const uint32_t *>(rec + kNvOff);
    T.cursors = reinterpret_cast<const uint32_t *>(T.nt + ntab_bytes(V)) + *reinterpret_cast<const uint32_t *>(T.nt + 20);
    return T;
}
// node v's cursors at the start and the end of tile k: boundary 0 and the
// block's end need no table; the root's is the position
__device__ inline uint32_t tile_cursor(const TileTabs &T, uint32_t V, uint32_t k, uint32_t ntile, uint32_t v, uint32_t pos,
                                       uint32_t nvv) {
    return k == 0 ? 0u : (k == ntile ? nvv : (v == 0 ? pos : T.cursors[(size_t)k * V + v]));
}

// Sets tile gt of the queue up (the whole CTA, every thread with the same
// arguments; b: the tile's block when the caller knows it).  False when there
// is nothing for ct_decode to do.
__device__ __noinline__ bool tile_open(uint32_t gt, const uint8_t *__restrict__ comp, const uint64_t *__restrict__ comp_off,
                                int nblk, uint8_t *__restrict__ out, const uint64_t *__restrict__ out_off,
                                const uint8_t *__restrict__ ws, uint64_t ws_bytes, int32_t *__restrict__ status,
                                int b = -1) {
    CtaTile &S = smem_item<CtaTile>();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const DecWs W = dec_ws(const_cast<uint8_t *>(ws), nblk);
    const DecRegions G = dec_regions(nblk, ws);
    // one block and one status for the whole CTA (every decision below that
    // chooses a path with barriers is the same in every thread)
    if (warp == 0) {
        if (b < 0) {
            const uint32_t ttot = reinterpret_cast<const uint32_t *>(ws)[6];
            b = find_block_warp(W.blk_tile, nblk, gt, (int)((uint64_t)gt * (uint32_t)nblk / max(ttot, 1u)));
        }
        if (lane == 0) { S.blk = b; S.flag = *reinterpret_cast<volatile int32_t *>(&status[b]); }
    }
    __syncthreads();
    b = S.blk;
    const int32_t st0 = S.flag;   // (nothing in the tile writes blk or flag again)
    if (st0 != PIVCO_OK) return false;
    const uint32_t k = gt - W.blk_tile[b], ntile = W.blk_ntile[b], T = W.blk_T[b];
    const uint8_t *rec = comp + comp_off[b];
    uint8_t *dst = out + out_off[b];
    const uint64_t ocap = out_off[b + 1] - out_off[b];
    const uint32_t rb = ld_le32(rec), n = ld_le32(rec + 4);
    const uint32_t V = (uint32_t)rec[8] | ((uint32_t)rec[9] << 8), kind = rec[10], aux = rec[11];
    if (n != ocap) {                     // the plan validated magic / size / layout
        if (t == 0) status[b] = PIVCO_ERR_CAPACITY;
        return false;
    }
    if (kind == 0) return false;
    const uint32_t P0 = k * T, P1 = min(n, P0 + T);
    if (kind == 1) {
        cta_fill(dst + P0, P1 - P0, (uint8_t)aux);
        return false;
    }
    const uint64_t nbase = G.dir + W.blk_dir[b], ntb = ntab_bytes(V);
    const uint32_t ent = nbase + ntb <= ws_bytes ? *reinterpret_cast<const uint32_t *>(ws + nbase + 20) : 0u;
    if (nbase + ntb > ws_bytes ||
        (ntile > 1 && nbase + ntb + 4ull * ent + 4ull * (ntile + 1) * V > ws_bytes)) {
        if (t == 0) status[b] = PIVCO_ERR_CAPACITY;
        return false;
    }
    const TileTabs TT = tile_tabs(ws, nblk, b, rec, V);
    const uint8_t *nt = TT.nt;
    if (t < 17) S.first[t] = nt[t];
    if (t == 17) S.maxd = nt[17];
    if (t < 64) reinterpret_cast<uint32_t *>(S.ftab)[t] = reinterpret_cast<const uint32_t *>(nt + kNtabHdr + 12 * V)[t];
    const uint64_t sbase = G.scratch + W.blk_scratch[b];
    TileSrc src;
    src.rec = rec;
    src.rec_bytes = rb;
    src.scr = ws + sbase;
    src.scr_bytes = ws_bytes > sbase ? ws_bytes - sbase : 0;
    int bad = V > 255;   // the plan has checked it
    if ((uint32_t)t < V) {
        const uint32_t v = t;
        const uint32_t nvv = __ldg(TT.nv + v);
        const uint32_t cs = tile_cursor(TT, V, k, ntile, v, P0, nvv), ce = tile_cursor(TT, V, k + 1, ntile, v, P1, nvv);
        const uint32_t s0 = TT.nsrc[3 * v], chv = TT.nsrc[3 * v + 1];
        const uint32_t bpe = max(1u, ch_flat_d(chv));   // bits per symbol of the node's body
        if (ce < cs || ce > nvv || bpe > 8 || (uint64_t)(s0 & 0x7FFFFFFFu) + (uint64_t)nvv * bpe >= 0x80000000ull ||
            (bpe > 1 && ((s0 >> 31) || (chv & 0xFFu) + (1u << bpe) > 256u)))
            bad = 1;
        S.pos[v] = s0 + cs * bpe;
        S.end[v] = s0 + ce * bpe;
        S.dem[v] = ce - cs;
        S.ch[v] = chv;
    }
    __syncthreads();
    if (t == 0 && S.dem[0] != P1 - P0) bad = 1;
    if (ct_tables_bad(S, V)) bad = 1;
    if (__syncthreads_or(bad)) {
        if (t == 0) status[b] = PIVCO_ERR_CORRUPT;
        return false;
    }
    // ask L2 for the nodes' bits of the tile, all lines at once
    if ((uint32_t)t < V && !(S.pos[t] >> 31) && S.dem[t]) {
        const uint32_t p0 = S.pos[t], nb = S.dem[t] * max(1u, ch_flat_d(S.ch[t]));
        for (uint32_t a = (p0 >> 3) & ~127u; a < (p0 + nb + 7) >> 3; a += 128)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(rec + a));
    }
    if (t == 0) {
        S.job.src = src;
        S.job.dst = dst;
        S.job.V = V;
        S.job.P0 = P0;
        S.job.P1 = P1;
        S.job.k = k;
        S.job.b = b;
    }
    __syncthreads();
    return true;
}

// Checks a decoded tile's end (the whole CTA): `how` is ct_decode's.
__device__ __noinline__ void tile_close(int how, int nblk, const uint8_t *__restrict__ ws, int32_t *__restrict__ status) {
    CtaTile &S = smem_item<CtaTile>();
    const int t = threadIdx.x, b = S.job.b;
    const uint32_t V = S.job.V, k = S.job.k, ntile = dec_ws(const_cast<uint8_t *>(ws), nblk).blk_ntile[b];
    bool bad = how == kTileBad;
    if (!bad && (uint32_t)t < V) {
        // the chunks must end exactly at the tile's end cursors
        if (how == kTileChunked && S.pos[t] != S.end[t]) bad = true;
        // the last tile checks the pad bits of every body (its end cursors are the bodies' ends)
        if (k + 1 == ntile) {
            const uint32_t nb = __ldg(reinterpret_cast<const uint32_t *>(S.job.src.rec + kNvOff) + t) * max(1u, ch_flat_d(S.ch[t]));
            if (pad_bad(S.job.src, S.end[t] - nb, nb)) bad = true;
        }
    }
    if (__syncthreads_or(bad) && t == 0) status[b] = PIVCO_ERR_CORRUPT;
}

// ---------------------------------------------------------------------------
// Rank directory and tile-boundary cursors of the blocks with several tiles
// (or, for random access, of every coded block).  They follow the block's
// node table in its directory region:
//   dir[u_v + i]   ones of node v before its superblock i (dir_bits bits
//                  each), counted from the node's start or the start of the
//                  share the entry lies in, whichever is later
//   cur[k V + v]   node v's bitmap cursor at tile boundary k (k = 1 ..
//                  ntile - 1, v >= 1); the other places (k = 0, k = ntile,
//                  v = 0) hold the shares' tails: the ones of a share's last
//                  node within it
// The superblocks of a block are cut into at most 128 shares of 2^s entries,
// `ways` times as many as the block has tiles at most (1 in batches of many
// tiles, where the chip is full either way), in two steps:
//   shares    a warp counts the superblocks of one share
//   cursors   a warp takes one tile boundary: the root's cursor is k T;
//             top-down, a child's cursor is the parent's rank0 / rank1 there
//             (Sec. 3.2's running counts, made random-access); the ones of a
//             node before a superblock are its entry plus the tails of the
//             shares between the node's start and the entry
// What bounds them: the latency of dependent reads (a share's windows one
// after another, a boundary's levels one after another).  One CTA per block
// took 242 us for a block of 2^20 symbols alone; as many shares as tiles at
// most, and their cursors, 43 + 29 us; eight times as many 30 + 33.
// ---------------------------------------------------------------------------
constexpr uint32_t kDirShares = 128;   // shares of a block at most
constexpr uint32_t kDirShareMin = 10;  // log2 of the fewest entries of a share (but for the block's last) ...
constexpr uint32_t kDirShareFew = 7;   // ... in batches of few tiles: one step of dir_share_count (300 blocks of two
                                       // tiles and 860 entries: 36 us by one share each, 18 by seven)
constexpr uint32_t kDirTarget = 4864;  // about as many shares as warps of the pass run at once (four CTAs an SM)
constexpr uint32_t kDirWays = 8;

// Shares for each of the batch's tiles (a function of the tiles alone: the
// items of a served request are numbered by it).
__device__ inline uint32_t dir_ways(uint32_t tiles) { return max(1u, min(kDirWays, kDirTarget / max(1u, tiles))); }

__device__ inline uint32_t dir_share_log(uint32_t ent, uint32_t V, uint32_t ntile, uint32_t ways) {
    const uint32_t most = ways == 1 ? min(ntile, kDirShares) : min(min(ntile * ways, kDirShares), 2 * V + ntile - 1);
    uint32_t s = ways == 1 ? kDirShareMin : kDirShareFew;
    while (s < 31 && (ent >> s) + ((ent & ((1u << s) - 1u)) != 0) > most) s++;
    return s;
}

struct DirWarpSm {
    uint32_t u[256], nv[256], src[256], ch[256], cur[256];
    uint32_t base[kDirShares];
    uint8_t first[17];
    uint8_t maxd;
    uint8_t pad[14];
};

// where a block's directory lives (one warp; false: nothing to do)
struct DirRef {
    const uint8_t *rec;
    uint32_t V, ent, ntile, T, slog, shares;
    uint32_t *dirp, *cur;
    TileSrc src;
    // where share s's tail is kept: boundary 0's places, the end's, the root's (fewer than 2 V + ntile)
    __device__ uint32_t *tail(uint32_t s) const {
        return cur + (s < V ? s : s < 2 * V ? (size_t)ntile * V + (s - V) : (size_t)(s - 2 * V + 1) * V);
    }
};
// (share: k is a share, and there is nothing to do past the last one)
__device__ inline bool dir_ref(int b, uint32_t k, bool share, const uint8_t *__restrict__ comp, const uint64_t *__restrict__ comp_off,
                               int nblk, uint8_t *__restrict__ ws, uint64_t ws_bytes, int32_t *__restrict__ status,
                               DirWarpSm &M, DirRef &D) {
    const int lane = threadIdx.x & 31;
    const DecWs W = dec_ws(ws, nblk);
    const DecRegions G = dec_regions(nblk, ws);
    D.ntile = W.blk_ntile[b];
    D.T = W.blk_T[b];
    if ((D.ntile <= 1 && !dec_all_dirs(ws)) || *reinterpret_cast<volatile int32_t *>(&status[b]) != PIVCO_OK) return false;
    // a block that is not coded has an empty region, and its record is not read
    const uint64_t d0 = W.blk_dir[b];
    const uint64_t d1 = b + 1 < nblk ? W.blk_dir[b + 1] : reinterpret_cast<const uint64_t *>(ws)[2];
    if (d1 <= d0) return false;
    const uint8_t *rec = comp + comp_off[b];
    D.rec = rec;
    D.V = (uint32_t)rec[8] | ((uint32_t)rec[9] << 8);
    const uint64_t nbase = G.dir + d0, ntb = ntab_bytes(D.V);
    const uint8_t *nt = ws + nbase;
    D.ent = nbase + ntb <= ws_bytes ? *reinterpret_cast<const uint32_t *>(nt + 20) : 0u;
    if (nbase + ntb + 4ull * D.ent + 4ull * (D.ntile + 1) * D.V > ws_bytes) {
        if (lane == 0 && k == 0) status[b] = PIVCO_ERR_CAPACITY;
        return false;
    }
    D.dirp = reinterpret_cast<uint32_t *>(ws + nbase + ntb);
    D.cur = D.dirp + D.ent;
    D.slog = dir_share_log(D.ent, D.V, D.ntile, dir_ways(reinterpret_cast<const uint32_t *>(ws)[6]));
    D.shares = (D.ent + (1u << D.slog) - 1) >> D.slog;
    if (share && k >= D.shares) return false;
    const uint64_t sbase = G.scratch + W.blk_scratch[b];
    D.src.rec = rec;
    D.src.rec_bytes = ld_le32(rec);
    D.src.scr = ws + sbase;
    D.src.scr_bytes = ws_bytes > sbase ? ws_bytes - sbase : 0;
    const uint32_t *nsrc = reinterpret_cast<const uint32_t *>(nt + kNtabHdr);
    const uint32_t *nv = reinterpret_cast<const uint32_t *>(rec + kNvOff);
    __syncwarp();
#pragma unroll 4
    for (uint32_t v = lane; v < D.V; v += 32) {
        M.nv[v] = __ldg(nv + v);
        M.src[v] = nsrc[3 * v];
        M.ch[v] = nsrc[3 * v + 1];
        M.u[v] = nsrc[3 * v + 2];
    }
    if (lane < 17) M.first[lane] = nt[lane];
    if (lane == 17) M.maxd = nt[17];
    __syncwarp();
    return true;
}

// Share k of block b's directory (one warp): superblocks of dir_bits, whose
// bits lie in kW words at most (five for the 128 bits of the default: 509
// text-like blocks 52 us with nine, 47 with five).
template <int kW>
__device__ inline void dir_share_count(const DirRef &D, const DirWarpSm &M, uint32_t k, uint32_t dir_bits) {
    const int lane = threadIdx.x & 31;
    const uint32_t V = D.V;
    uint32_t *const tail = D.tail(k);
    const uint32_t g0 = k << D.slog, g1 = min(D.ent, g0 + (1u << D.slog));
    const uint32_t le = 0xFFFFFFFFu >> (31 - lane);
    uint32_t vcur = (uint32_t)find_node_d(M.u, 0, (int)V, g0), carry = 0;
    // four windows of 32 superblocks per step: their nodes first (shared
    // memory only), then all their bitmap loads, then the scans
    constexpr int kU = 4;
    for (uint32_t base = g0; base < g1; base += 32 * kU) {
        uint32_t vv[kU], st[kU], pc[kU];
#pragma unroll
        for (int r = 0; r < kU; r++) {
            const uint32_t cand = vcur + 1 + lane, bb = base + 32 * r;
            uint32_t bit = 0;
            if (cand < V) {
                const uint32_t sd = M.u[cand] - bb;
                if (sd < 32) bit = 1u << sd;
            }
            st[r] = __reduce_or_sync(0xffffffffu, bit);
            vv[r] = vcur + __popc(st[r] & le);
            vcur = __shfl_sync(0xffffffffu, vv[r], 31);
        }
#pragma unroll
        for (int r = 0; r < kU; r++) {
            const uint32_t g = base + 32 * r + lane;
            pc[r] = 0;
            if (g < g1) {
                const uint32_t v = vv[r], e0 = (g - M.u[v]) * dir_bits;
                // (a flat node's body is indices: its superblocks are not read)
                if (e0 < M.nv[v] && !ch_flat_d(M.ch[v])) pc[r] = tile_popc_w<kW>(D.src, M.src[v], e0, min(dir_bits, M.nv[v] - e0));
            }
        }
#pragma unroll
        for (int r = 0; r < kU; r++) {
            const uint32_t g = base + 32 * r + lane;
            const uint32_t inc = warp_inclusive(pc[r]), sl = st[r] & le;
            const int sa = sl ? 31 - __clz(sl) : -1;   // where the entry's node starts in the window
            const uint32_t before = __shfl_sync(0xffffffffu, inc, sa > 0 ? sa - 1 : 0);
            const uint32_t ex = inc - pc[r] - (sa > 0 ? before : 0u) + (sa < 0 ? carry : 0u);
            if (g < g1) D.dirp[g] = ex;
            if (base + 32 * r < g1)   // (warp-uniform)
                carry = __shfl_sync(0xffffffffu, ex + pc[r], (int)min(31u, g1 - 1 - (base + 32 * r)));
        }
    }
    if (lane == 0) *tail = carry;
}
__device__ __noinline__ void dir_share(int b, uint32_t k, const uint8_t *__restrict__ comp,
                                       const uint64_t *__restrict__ comp_off, int nblk, uint8_t *__restrict__ ws,
                                       uint64_t ws_bytes, int32_t *__restrict__ status) {
    DirWarpSm &M = (&smem_item<DirWarpSm>())[threadIdx.x >> 5];
    DirRef D;
    if (!dir_ref(b, k, true, comp, comp_off, nblk, ws, ws_bytes, status, M, D)) return;
    const uint32_t dir_bits = dec_dir_bits(ws);
    if (dir_bits <= 128) dir_share_count<5>(D, M, k, dir_bits);
    else dir_share_count<9>(D, M, k, dir_bits);
}

// Cursors of block b at tile boundary k (1 <= k < ntile), after all the
// block's shares (one warp).
__device__ __noinline__ void dir_cursors(int b, uint32_t k, const uint8_t *__restrict__ comp,
                                         const uint64_t *__restrict__ comp_off, int nblk, uint8_t *__restrict__ ws,
                                         uint64_t ws_bytes, int32_t *__restrict__ status) {
    const int lane = threadIdx.x & 31;
    DirWarpSm &M = (&smem_item<DirWarpSm>())[threadIdx.x >> 5];
    DirRef D;
    if (k == 0 || !dir_ref(b, k, false, comp, comp_off, nblk, ws, ws_bytes, status, M, D) || k >= D.ntile) return;
    const uint32_t dir_bits = dec_dir_bits(ws), V = D.V;
    uint32_t carry = 0;   // tails of the shares before each share
    for (uint32_t s = 0; s < D.shares; s += 32) {
        const uint32_t x = s + lane < D.shares ? __ldcg(D.tail(s + lane)) : 0u;
        const uint32_t inc = warp_inclusive(x);
        if (s + lane < D.shares) M.base[s + lane] = carry + inc - x;
        carry += __shfl_sync(0xffffffffu, inc, 31);
    }
    for (uint32_t v = lane; v < V; v += 32) M.cur[v] = 0;
    __syncwarp();
    if (lane == 0) M.cur[0] = k * D.T;
    __syncwarp();
    bool bad = false;
    uint32_t *out = D.cur + (size_t)k * V;
    for (int d = 0; d < (int)M.maxd; d++) {
        const uint32_t f0 = M.first[d], f1 = M.first[d + 1];
        for (uint32_t v = f0 + lane; v < f1; v += 32) {
            const uint32_t c = M.cur[v], nvv = M.nv[v];
            if (v) out[v] = c;
            if (c > nvv) { bad = true; continue; }
            const uint32_t chv = M.ch[v];
            if (ch_flat_d(chv)) continue;   // no children below a flat node
            const uint32_t nsb = (nvv + dir_bits - 1) / dir_bits;
            uint32_t sb = c / dir_bits;
            if (sb >= nsb) sb = nsb - 1;
            const uint32_t g0 = M.u[v], g = g0 + sb;
            const uint32_t ones = __ldcg(D.dirp + g) + M.base[g >> D.slog] - M.base[g0 >> D.slog] +
                                  tile_popc(D.src, M.src[v], sb * dir_bits, c - sb * dir_bits);
            const uint32_t c0 = chv & 0xFFFFu, c1 = chv >> 16;
            if (!(c0 & 0x8000u)) M.cur[c0 & 0xFFu] = c - ones;
            if (!(c1 & 0x8000u)) M.cur[c1 & 0xFFu] = ones;
        }
        __syncwarp();
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) status[b] = PIVCO_ERR_CORRUPT;
    __syncwarp();
}

// The tails of the shares before it into share k's entries of the node that
// runs into it (random access): afterwards dir[u_v + i] is counted from node
// v's start (one warp).
__device__ inline void dir_rebase(int b, uint32_t k, const uint8_t *__restrict__ comp,
                                  const uint64_t *__restrict__ comp_off, int nblk, uint8_t *__restrict__ ws,
                                  uint64_t ws_bytes, int32_t *__restrict__ status) {
    const int lane = threadIdx.x & 31;
    DirWarpSm &M = (&smem_item<DirWarpSm>())[threadIdx.x >> 5];
    DirRef D;
    if (k == 0 || !dir_ref(b, k, true, comp, comp_off, nblk, ws, ws_bytes, status, M, D)) return;
    const uint32_t g0 = k << D.slog, g1 = min(D.ent, g0 + (1u << D.slog));
    const uint32_t v = (uint32_t)find_node_d(M.u, 0, (int)D.V, g0);
    uint32_t x = 0;
    for (uint32_t s = (M.u[v] >> D.slog) + lane; s < k; s += 32) x += __ldcg(D.tail(s));
    x = __reduce_add_sync(0xffffffffu, x);
    const uint32_t ge = min(g1, v + 1 < D.V ? M.u[v + 1] : D.ent);
    if (x)
        for (uint32_t g = g0 + lane; g < ge; g += 32) D.dirp[g] += x;
}

constexpr int kDirSmem = (int)(kSelBytes + sizeof(DirWarpSm) * kDecWarps);   // (below 48 KiB)
static_assert(kDirSmem <= 48 * 1024, "no opt-in needed");
enum : int { kDirShare = 0, kDirCursors = 1, kDirRebase = 2 };

// One step of the directory pass over every tile's shares or boundary, one
// warp each.
template <int kStep>
__global__ void __launch_bounds__(kDecThreads) decode_dir_kernel(const uint8_t *__restrict__ comp,
                                                                 const uint64_t *__restrict__ comp_off, int nblk,
                                                                 uint8_t *__restrict__ ws, uint64_t ws_bytes,
                                                                 int32_t *__restrict__ status) {
    if (abandoned_batch(ws, status, nblk)) return;
    const uint32_t tiles = reinterpret_cast<const uint32_t *>(ws)[6];
    if (tiles == (uint32_t)nblk && (kStep == kDirCursors || !dec_all_dirs(ws))) return;   // one tile each
    const DecWs W = dec_ws(ws, nblk);
    const int warp = threadIdx.x >> 5;
    const uint32_t ways = kStep == kDirCursors ? 1u : dir_ways(tiles);   // (items of a tile)
    for (uint32_t g = blockIdx.x * kDecWarps + warp; g < tiles * ways; g += gridDim.x * kDecWarps) {
        const uint32_t gt = g / ways;
        const int b = find_block_warp(W.blk_tile, nblk, gt, (int)((uint64_t)gt * (uint32_t)nblk / tiles));
        const uint32_t k = g - W.blk_tile[b] * ways;
        if (kStep == kDirShare) dir_share(b, k, comp, comp_off, nblk, ws, ws_bytes, status);
        else if (kStep == kDirCursors) dir_cursors(b, k, comp, comp_off, nblk, ws, ws_bytes, status);
        else dir_rebase(b, k, comp, comp_off, nblk, ws, ws_bytes, status);
    }
}

struct TileSmem {
    uint32_t sel[256];
    CtaTile tile;
};

// Plain tile pass: every CTA takes tiles by ticket (workspace header word 12).
__global__ void __launch_bounds__(kDecThreads, kTileCtas) decode_kernel(const uint8_t *__restrict__ comp,
                                                                        const uint64_t *__restrict__ comp_off,
                                                                        int nblk, uint8_t *__restrict__ out,
                                                                        const uint64_t *__restrict__ out_off,
                                                                        uint8_t *__restrict__ ws, uint64_t ws_bytes,
                                                                        int32_t *__restrict__ status) {
    __shared__ uint32_t s_it;
    if (abandoned_batch(ws, status, nblk)) return;
    sel_init(smem_sel());
    uint32_t *hdr = reinterpret_cast<uint32_t *>(ws);
    const uint32_t total_tiles = hdr[6];
    for (;;) {
        if (threadIdx.x == 0) s_it = atomicAdd(&hdr[12], 1u);
        __syncthreads();
        const uint32_t it = s_it;
        __syncthreads();
        if (it >= total_tiles) break;
        if (tile_open(it, comp, comp_off, nblk, out, out_off, ws, ws_bytes, status))
            tile_close(ct_decode(), nblk, ws, status);
    }
}

// ---------------------------------------------------------------------------
// Batched decode: one persistent launch over a work queue keyed by
// (block, stage).  Every item is taken by a whole CTA, in queue order:
//   plans      (batches of more blocks than CTAs) 8 blocks per item, one warp
//              each, then one item per block: its decode as soon as its own
//              plan is complete, when the block is one tile with no ANS
//              segment and no directory
//   blocks     (smaller batches) one block per item: its plan and, when the
//              block is one tile
//              with no ANS segment and no directory, its decode, straight
//              from the plan's tables in shared memory
//              (plans are in ticket order, as their look-back needs)
//   ANS        8 units per item, one warp each
//   shares     8 directory shares per item (`ways` to a tile), one warp each
//   cursors    8 tile boundaries per item, one warp each
//   tiles      one tile per item (cta_tile)
// An item only waits (bounded) on items earlier in the queue: the ANS and
// later items on all plans; a share on its block's ANS segments; a boundary
// on its block's shares; a tile on its block's ANS segments and cursors.  The
// CTAs that took those items are running, so every wait ends.
// ---------------------------------------------------------------------------
__device__ inline bool wait_geq(const uint32_t *p, uint32_t want, uint64_t limit_ns) {
    if (*reinterpret_cast<const volatile uint32_t *>(p) >= want) { __threadfence(); return true; }
    const uint64_t t0 = globaltimer_ns();
    unsigned ns = 64;
    while (*reinterpret_cast<const volatile uint32_t *>(p) < want) {
        if (globaltimer_ns() - t0 > limit_ns) return false;
        __nanosleep(ns);
        if (ns < 2048) ns <<= 1;
    }
    __threadfence();
    return true;
}

// what a block's plan and its tile's tables do not share: the plan lies over
// the tile's level buffers, which the decode fills after the tables are taken
union BatchUnion {
    AnsItemSm ans;
    DirWarpSm dw[kDecWarps];
    PlanSm plan;
    PlanItemSm plans;
    CtaTile tile;
};
struct BatchSmem {
    uint32_t sel[256];
    BatchUnion u;
    int32_t blk, ok;
    uint32_t pad[2];
};
static_assert(sizeof(AnsItemSm) <= sizeof(CtaTile) && sizeof(DirWarpSm) * kDecWarps <= sizeof(CtaTile) &&
                  sizeof(PlanItemSm) <= sizeof(CtaTile),
              "every item fits the tiles' shared memory");
static_assert(sizeof(PlanSm) <= offsetof(CtaTile, pos), "a plan fits the level buffers");
static_assert(offsetof(BatchSmem, u) == kSelBytes && offsetof(TileSmem, tile) == kSelBytes, "smem_item finds the item");
// kTileCtas CTAs per SM: dynamic + static shared memory + 1 KiB reserved each, of 228 KiB
static_assert(kTileCtas * (sizeof(BatchSmem) + 128 + 1024) <= 228 * 1024, "tile CTAs per SM");

// One request's (batch's) queue: where its records, output and workspace are.
struct BatchQueue {
    const uint8_t *comp;
    const uint64_t *comp_off;
    uint8_t *out;
    const uint64_t *out_off;
    uint8_t *ws;
    uint64_t ws_bytes;
    int32_t *status;
    int nblk;
    bool wide;                  // the form of its queue (wide_batch)
};

// the wait bound of a batch's queue (workspace header)
__device__ inline uint64_t wait_bound(const BatchQueue &q) { return reinterpret_cast<const uint64_t *>(q.ws)[7]; }

// Plans by warps, then the blocks' own items (a wide batch): for more blocks than
// the launch has CTAs, where the plans' instructions count (4096 blocks of
// 64 KiB: 150 us of CTA plans, 50 us of warp plans; the line stands where the
// second wave begins: 862 blocks of 1 to 16 KB decode in 73 to 96 us by warp
// plans, 78 to 99 by CTA plans, 640 in 68 to 87 and 64 to 84); else one item plans
// and decodes a block, its decode starting 6 us after the item (a warp plan takes
// 25 us).  Decided once per batch: the items of
// a served request are taken by several launches, which need not have the same
// number of CTAs (the tuning may change between them), so its form goes with
// the request.
__host__ __device__ inline bool wide_batch(int nblk, int ctas) { return nblk > ctas; }
__device__ inline uint32_t batch_nplan(const BatchQueue &q) {
    return q.wide ? (uint32_t)((q.nblk + kDecWarps - 1) / kDecWarps) : 0u;
}
__device__ inline uint32_t batch_items_blocks(const BatchQueue &q) { return batch_nplan(q) + (uint32_t)q.nblk; }
// plans to wait for (header word 10 counts them)
__device__ inline uint32_t batch_plans(const BatchQueue &q) { return q.wide ? batch_nplan(q) : (uint32_t)q.nblk; }

// Items of each stage once all plans are done (header written by the last
// plan; word 12 counts the blocks whose tiles are still to be decoded).
struct BatchStages {
    uint32_t ans, ways, shares, cursors, tiles;   // ANS items; shares of a tile, share items; cursor items; tile items
};
__device__ inline BatchStages batch_stages(const BatchQueue &q) {
    const uint32_t *hdr = reinterpret_cast<const uint32_t *>(q.ws);
    BatchStages s;
    const uint32_t left = *reinterpret_cast<const volatile uint32_t *>(&hdr[12]);
    s.ans = (hdr[2] + kAnsWarps - 1) / kAnsWarps;
    s.ways = dir_ways(hdr[6]);
    const bool dir = hdr[6] != (uint32_t)q.nblk;   // (one tile each: no directory)
    s.shares = dir ? (hdr[6] * s.ways + kDecWarps - 1) / kDecWarps : 0u;
    s.cursors = dir ? (hdr[6] + kDecWarps - 1) / kDecWarps : 0u;
    s.tiles = left ? hdr[6] : 0u;
    return s;
}
__device__ inline uint32_t batch_items_total(const BatchQueue &q) {
    const BatchStages s = batch_stages(q);
    return batch_items_blocks(q) + s.ans + s.shares + s.cursors + s.tiles;
}

// Block b's item: its plan and, when it needs nothing else, its decode.
// First half: the plan, complete when it returns; true when ct_decode and
// block_close are to follow.
__device__ __noinline__ bool block_open(const BatchQueue &q, int b) {
    const int t = threadIdx.x;
    uint32_t *hdr = reinterpret_cast<uint32_t *>(q.ws);
    const DecWs W = dec_ws(q.ws, q.nblk);
    PlanSm &Q = smem_item<PlanSm>();
    CtaTile &S = smem_item<CtaTile>();
    const uint8_t *rec = q.comp + q.comp_off[b];
    const uint64_t avail = q.comp_off[b + 1] - q.comp_off[b], o0 = q.out_off[b], ocap = q.out_off[b + 1] - o0;
    // ask L2 for the record while its tables are parsed
    for (uint64_t i = 128ull * t; i < avail && i < 128ull * kDecThreads * 2; i += 128ull * kDecThreads)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(rec + i));
    const PlanRes R = plan_cta(rec, avail, dec_dir_bits(q.ws), hdr[8], dec_all_dirs(q.ws));
    if (t == 0) plan_publish(W, b, R);
    const bool simple = R.st == PIVCO_OK && R.ntile == 1 && R.nsegs == 0 && !dec_all_dirs(q.ws);
    uint64_t nbase;
    const bool placed = plan_place(b, q.nblk, q.ws, q.ws_bytes, R, !simple, nbase);
    int32_t st = R.st;
    if (!placed && R.st == PIVCO_OK) st = PIVCO_ERR_TIMEOUT;
    else if (simple && R.n != ocap) st = PIVCO_ERR_CAPACITY;
    // (the workspace must hold a coded block's node table, also where the decode does not need it)
    else if (simple && R.kind == 2 && nbase + ntab_bytes(R.V) > q.ws_bytes) st = PIVCO_ERR_CAPACITY;
    bool go = simple && st == PIVCO_OK && R.kind == 2, bad = false;
    const uint32_t V = R.V;
    if (go) {
        // the tile's tables from the plan's, which the level buffers then overwrite
        if (t < 17) S.first[t] = (uint8_t)Q.tree.first[t];
        if (t == 17) S.maxd = (uint8_t)Q.tree.maxd;
        S.ftab[t] = Q.sorted[t];
        if ((uint32_t)t < V) {
            const uint32_t chv = Q.ch[t], bpe = max(1u, ch_flat_d(chv)), nvv = Q.nv[t], s0 = plan_src(Q, t);
            if (bpe > 8 || (uint64_t)(s0 & 0x7FFFFFFFu) + (uint64_t)nvv * bpe >= 0x80000000ull ||
                (bpe > 1 && (chv & 0xFFu) + (1u << bpe) > 256u))
                bad = true;
            S.pos[t] = s0;
            S.end[t] = s0 + nvv * bpe;
            S.dem[t] = nvv;
            S.ch[t] = chv;
        }
        if (t == 0) {
            S.job.src.rec = rec;
            S.job.src.rec_bytes = R.rb;
            S.job.src.scr = nullptr;
            S.job.src.scr_bytes = 0;
            S.job.dst = q.out + o0;
            S.job.V = V;
            S.job.P0 = 0;
            S.job.P1 = R.n;
        }
    }
    __syncthreads();   // (every thread's writes of the plan, then its flag and count; the tables)
    if (go && ct_tables_bad(S, V)) bad = true;
    if (t == 0) {
        // a CTA that has given up on the queue (below) may have marked the
        // blocks before this plan wrote its status: re-mark it, so a block
        // whose later items may never run does not read as done
        q.status[b] = st;
        if (!simple && R.st == PIVCO_OK) atomicAdd(&hdr[12], 1u);
        __threadfence();
        atomicExch(&W.plan_done[b], simple || R.st != PIVCO_OK ? 3u : 1u);
        if (!simple && *reinterpret_cast<volatile uint32_t *>(&hdr[13]) &&
            *reinterpret_cast<volatile int32_t *>(&q.status[b]) == PIVCO_OK)
            q.status[b] = PIVCO_ERR_TIMEOUT;
        __threadfence();
        atomicAdd(&hdr[10], 1u);
    }
    if (simple && st == PIVCO_OK && R.kind == 1) cta_fill(q.out + o0, R.n, rec[11]);
    if (__syncthreads_or(bad)) {
        if (t == 0) q.status[b] = PIVCO_ERR_CORRUPT;
        go = false;
    }
    return go;
}

// Second half: checks the decoded block's end and writes its status.
__device__ __noinline__ void block_close(const BatchQueue &q, int b, int how) {
    const int t = threadIdx.x;
    CtaTile &S = smem_item<CtaTile>();
    bool bad = how == kTileBad;
    if (!bad && (uint32_t)t < S.job.V) {
        // the chunks must end exactly at the bodies' ends; pad bits are zero
        const uint32_t nb = __ldg(reinterpret_cast<const uint32_t *>(S.job.src.rec + kNvOff) + t) *
                            max(1u, ch_flat_d(S.ch[t]));
        bad = pad_bad(S.job.src, S.end[t] - nb, nb) || (how == kTileChunked && S.pos[t] != S.end[t]);
    }
    // (decoded: whatever another CTA that gave up has marked in the meantime)
    if (__syncthreads_or(bad)) {
        if (t == 0) q.status[b] = PIVCO_ERR_CORRUPT;
    } else if (t == 0) {
        q.status[b] = PIVCO_OK;
    }
}

enum : int { kItemDone = 0, kItemNone = 1, kItemStop = 2, kItemTile = 3, kItemBlock = 4 };

// Runs item `item` of the queue with the whole CTA up to a tile's decode.
// kItemDone: processed; kItemTile / kItemBlock: a tile is set up, the caller
// decodes it and calls tile_close / block_close; kItemNone: past the last item; kItemStop: the wait for the plans expired
// or the plans could not place the batch (every block is marked), the CTA
// must stop.
__device__ __noinline__ int batch_item(const BatchQueue &q, uint32_t item, const AnsTables &A) {
    BatchSmem &B = reinterpret_cast<BatchSmem &>(*smem_sel());
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int nblk = q.nblk;
    uint32_t *hdr = reinterpret_cast<uint32_t *>(q.ws);
    const DecWs W = dec_ws(q.ws, nblk);
    if (!q.wide) {
        if (item < (uint32_t)nblk) {
            return block_open(q, (int)item) ? kItemBlock : kItemDone;
        }
    } else {
        const uint32_t nplan = batch_nplan(q);
        if (item < nplan) {
            plan_item((int)item, q.comp, q.comp_off, nblk, q.ws, q.ws_bytes, q.status);
            if (lane == 0) {
                const int b = (int)item * kDecWarps + warp;
                if (b < nblk) {
                    // blocks whose tiles come after the directories
                    if (q.status[b] == PIVCO_OK && !(W.plan_done[b] & 2u)) atomicAdd(&hdr[12], 1u);
                    // a CTA that has given up on the queue (below) may have marked
                    // the blocks before this plan wrote its status: re-mark it, so a
                    // block whose later items may never run does not read as done
                    __threadfence();
                    if (*reinterpret_cast<volatile uint32_t *>(&hdr[13]) &&
                        *reinterpret_cast<volatile int32_t *>(&q.status[b]) == PIVCO_OK)
                        q.status[b] = PIVCO_ERR_TIMEOUT;
                }
                __threadfence();
            }
            __syncthreads();
            if (t == 0) { __threadfence(); atomicAdd(&hdr[10], 1u); }
            return kItemDone;
        }
        if (item < nplan + (uint32_t)nblk) {
            const int b = (int)(item - nplan);
            if (t == 0) {
                // a wait that runs out leaves its mark in the same word as the plan: the one that comes second sees
                // the other's, so the block does not read OK when the plan is merely late
                uint32_t pd = 0;
                if (wait_geq(&W.plan_done[b], 1u, wait_bound(q))) pd = *reinterpret_cast<volatile uint32_t *>(&W.plan_done[b]);
                else if ((pd = atomicOr(&W.plan_done[b], 4u)) != 0) __threadfence();
                else q.status[b] = PIVCO_ERR_TIMEOUT;
                B.ok = (int)pd;
            }
            __syncthreads();
            const int pd = B.ok;
            __syncthreads();
            if ((pd & 2) && tile_open(W.blk_tile[b], q.comp, q.comp_off, nblk, q.out, q.out_off, q.ws, q.ws_bytes,
                                      q.status, b))
                return kItemTile;
            __syncthreads();
            return kItemDone;
        }
    }
    // everything after the blocks' items needs all plans
    int ok = 1;
    if (t == 0) {
        ok = wait_geq(&hdr[10], batch_plans(q), wait_bound(q));
        // the last plan could not place the batch: nothing after the plans runs
        if (ok && *reinterpret_cast<volatile uint32_t *>(&hdr[13])) ok = 0;
    }
    if (__syncthreads_or(!ok)) {
        // this CTA leaves the queue: every block not yet failed is marked, as
        // its items may now never run (the flag makes plans still running
        // mark theirs, the fences order the flag against their status writes)
        if (t == 0) {
            atomicExch(&hdr[13], 1u);
            __threadfence();
            for (int b = 0; b < nblk; b++)
                if (*reinterpret_cast<volatile int32_t *>(&q.status[b]) == PIVCO_OK) q.status[b] = PIVCO_ERR_TIMEOUT;
        }
        __syncthreads();
        return kItemStop;
    }
    const BatchStages stg = batch_stages(q);
    const uint32_t total_segs = hdr[2], total_tiles = hdr[6];
    uint32_t it = item - batch_items_blocks(q);
    if (it < stg.ans) {
        // ---- ANS segments ----
        ans_members(B.u.ans, A);
        __syncthreads();
        const uint32_t g = it * kAnsWarps + warp;
        if (g < total_segs) {
            const int b = ans_item(g, q.comp, q.comp_off, nblk, q.ws, q.ws_bytes, q.status, A);
            if (lane == 0) { __threadfence(); atomicAdd(&W.segs_done[b], 1u); }
        }
        __syncthreads();
        return kItemDone;
    }
    it -= stg.ans;
    if (it < stg.shares + stg.cursors) {
        // ---- directory shares, then cursors: one per warp ----
        const bool cursors = it >= stg.shares;
        const uint32_t ways = cursors ? 1u : stg.ways, g = (cursors ? it - stg.shares : it) * kDecWarps + warp, gt = g / ways;
        if (gt < total_tiles) {
            const int b = find_block_warp(W.blk_tile, nblk, gt, (int)((uint64_t)gt * (uint32_t)nblk / total_tiles));
            const uint32_t ntile = W.blk_ntile[b], k = g - W.blk_tile[b] * ways;
            if (ntile > 1) {
                int okw = 1;
                if (lane == 0) {
                    const uint32_t nsegs = (b + 1 < nblk ? W.blk_seg[b + 1] : total_segs) - W.blk_seg[b];
                    okw = cursors ? wait_geq(&W.dir_done[b], ntile * stg.ways, wait_bound(q))
                                  : wait_geq(&W.segs_done[b], nsegs, wait_bound(q));
                    if (!okw) q.status[b] = PIVCO_ERR_TIMEOUT;
                }
                okw = __shfl_sync(0xffffffffu, okw, 0);
                if (okw && !cursors) dir_share(b, k, q.comp, q.comp_off, nblk, q.ws, q.ws_bytes, q.status);
                if (okw && cursors) dir_cursors(b, k, q.comp, q.comp_off, nblk, q.ws, q.ws_bytes, q.status);
                __syncwarp();
                if (lane == 0) { __threadfence(); atomicAdd(&W.dir_done[b], 1u); }
            }
        }
        __syncthreads();
        return kItemDone;
    }
    it -= stg.shares + stg.cursors;
    if (it >= stg.tiles) return kItemNone;
    // ---- tile it: after its block's ANS segments and cursors (a block
    // decoded by its own item is skipped) ----
    if (warp == 0) {
        const int b = find_block_warp(W.blk_tile, nblk, it, (int)((uint64_t)it * (uint32_t)nblk / max(total_tiles, 1u)));
        if (lane == 0) {
            int okw = 1;
            if (W.plan_done[b] & 2u) {
                okw = 0;
            } else {
                const uint32_t nsegs = (b + 1 < nblk ? W.blk_seg[b + 1] : total_segs) - W.blk_seg[b];
                okw = wait_geq(&W.segs_done[b], nsegs, wait_bound(q));
                if (okw && W.blk_ntile[b] > 1) okw = wait_geq(&W.dir_done[b], (stg.ways + 1) * W.blk_ntile[b], wait_bound(q));
                if (!okw) q.status[b] = PIVCO_ERR_TIMEOUT;
            }
            B.blk = b;
            B.ok = okw;
        }
    }
    __syncthreads();
    const int b = B.blk, okw = B.ok;
    __syncthreads();
    if (okw && tile_open(it, q.comp, q.comp_off, nblk, q.out, q.out_off, q.ws, q.ws_bytes, q.status, b)) return kItemTile;
    __syncthreads();
    return kItemDone;
}

__global__ void __launch_bounds__(kDecThreads, kTileCtas) decode_batch_kernel(const uint8_t *__restrict__ comp,
                                                                              const uint64_t *__restrict__ comp_off,
                                                                              int nblk, uint8_t *__restrict__ out,
                                                                              const uint64_t *__restrict__ out_off,
                                                                              uint8_t *__restrict__ ws, uint64_t ws_bytes,
                                                                              int32_t *__restrict__ status,
                                                                              const __grid_constant__ AnsTables A) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    BatchSmem &B = *reinterpret_cast<BatchSmem *>(smem_raw);
    __shared__ uint32_t s_item;
    const BatchQueue q{comp, comp_off, out, out_off, ws, ws_bytes, status, nblk, wide_batch(nblk, (int)gridDim.x)};
    uint32_t *hdr = reinterpret_cast<uint32_t *>(ws);
    sel_init(B.sel);
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(&hdr[9], 1u);
        __syncthreads();
        const uint32_t item = s_item;
        __syncthreads();
        const int r = batch_item(q, item, A);
        if (r == kItemTile || r == kItemBlock) {
            const int how = ct_decode();
            if (r == kItemTile) tile_close(how, nblk, q.ws, q.status);
            else block_close(q, (int)item, how);
            __syncthreads();
        } else if (r != kItemDone) {
            return;
        }
    }
}

// ---------------------------------------------------------------------------
// Serving: a device-resident request loop over the batch queue items.
// Requests are published by the host in sequence order into a ring (entry r
// at ring[r % kServeRing], the count in flags->tail, host memory mapped into
// the device).  Every CTA repeatedly takes the next item of request ctl->cur;
// when that request has no items left it moves ctl->cur on, so the items of
// consecutive requests overlap on the device and a request published while
// others run is picked up by the first CTA that frees up.  The CTA that
// finishes a request's last item writes its worst block status and then its
// done flag into mapped host memory.  A CTA leaves when it has found nothing
// to do for idle_ns, when its launch has lived life_ns (checked between
// items), or on flags->stop; the host then launches the loop again if work
// remains.  A request's ring entry and memory are reused only after a launch
// that started later has ended with ctl->cur past it, so no CTA can still
// touch them.
// ---------------------------------------------------------------------------
__device__ inline uint32_t ld_acquire_sys_u32(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ inline void st_release_sys_u32(uint32_t *p, uint32_t v) {
    asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Counts one finished item of request r; the item that completes the
// request's queue writes its worst block status, then its done flag.
__device__ inline void serve_item_done(const BatchQueue &q, uint32_t r, ServeFlags *flags) {
    uint32_t *hdr = reinterpret_cast<uint32_t *>(q.ws);
    __threadfence();
    const uint32_t n = atomicAdd(&hdr[11], 1u) + 1;
    if (*reinterpret_cast<volatile uint32_t *>(&hdr[10]) < batch_plans(q)) return;   // totals not known yet
    __threadfence();
    if (n != batch_items_total(q)) return;
    int32_t worst = PIVCO_OK;
    for (int b = 0; b < q.nblk && worst == PIVCO_OK; b++) worst = *reinterpret_cast<volatile int32_t *>(&q.status[b]);
    flags->worst[r % kServeRing] = worst;
    __threadfence_system();
    st_release_sys_u32(&flags->done[r % kServeRing], r + 1);
}

__global__ void __launch_bounds__(kDecThreads, kTileCtas) serve_loop_kernel(ServeCtl *__restrict__ ctl,
                                                                            const ServeDesc *__restrict__ ring,
                                                                            ServeFlags *flags, uint64_t idle_ns,
                                                                            uint64_t life_ns,
                                                                            const __grid_constant__ AnsTables A) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    BatchSmem &B = *reinterpret_cast<BatchSmem *>(smem_raw);
    __shared__ ServeDesc D;
    __shared__ uint32_t s_cmd, s_item, s_r;
    const int t = threadIdx.x;
    sel_init(B.sel);
    uint32_t have = 0xFFFFFFFFu;   // request whose ring entry is in D (thread 0's view)
    const uint64_t t0 = globaltimer_ns();
    uint64_t idle_since = 0;
    for (;;) {
        if (t == 0) {
            uint32_t cmd = 0;   // 0 work, 1 nothing yet, 2 leave
            const uint64_t now = globaltimer_ns();
            const uint32_t r = *reinterpret_cast<volatile uint32_t *>(&ctl->cur);
            const uint32_t tail = ld_acquire_sys_u32(&flags->tail);
            if (ld_acquire_sys_u32(&flags->stop) || now - t0 > life_ns) {
                cmd = 2;
            } else if (r >= tail) {
                if (!idle_since) idle_since = now;
                cmd = now - idle_since > idle_ns ? 2u : 1u;
            } else {
                idle_since = 0;
                if (r != have) {
                    D = ring[r % kServeRing];
                    if (D.seq != r) cmd = 1;   // not written yet (cannot happen once published)
                    else have = r;
                }
                if (cmd == 0) {
                    s_item = atomicAdd(&reinterpret_cast<uint32_t *>(D.ws)[9], 1u);
                    s_r = r;
                }
            }
            s_cmd = cmd;
        }
        __syncthreads();
        const uint32_t cmd = s_cmd, item = s_item, r = s_r;
        __syncthreads();
        if (cmd == 2) return;
        if (cmd == 1) {
            if (t == 0) __nanosleep(1000);
            continue;
        }
        const BatchQueue q{D.comp, D.comp_off, D.out, D.out_off, D.ws, D.ws_bytes, D.status, (int)D.nblk, D.wide != 0};
        int res = batch_item(q, item, A);
        if (res == kItemTile || res == kItemBlock) {
            const int how = ct_decode();
            if (res == kItemTile) tile_close(how, q.nblk, q.ws, q.status);
            else block_close(q, (int)item, how);
            __syncthreads();
            res = kItemDone;
        }
        if (res != kItemNone) {
            if (t == 0) serve_item_done(q, r, flags);
            if (res == kItemStop) return;
            __syncthreads();
            continue;
        }
        // the request has no items left: move on to the next one
        if (t == 0) atomicCAS(&ctl->cur, r, r + 1);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Random access (NEXT to the bottom-up merge): the symbol at one position of
// one block by a top-down walk, Sec. 2.1's traversal made random-access the
// way a wavelet tree answers access (Sec. 7.2): at node v the position's bit
// picks the child, and the position becomes its rank among the positions of
// that bit, rank1(B_v, x) = the directory's ones before x's superblock plus
// the popcount of the superblock's bits before x.  The workspace comes from
// the plan with a directory for every coded block, the ANS pass and the
// directory pass (pivco_access_prepare).  One thread per query.
// ---------------------------------------------------------------------------
// Ones among bits [e, e + len) (len < 256) of the bitmap at bit address pos,
// and bit e + len itself, from the words that hold them (inside the bitmap:
// e + len is one of its positions).
__device__ inline uint32_t access_rank(const TileSrc &s, uint32_t pos, uint32_t e, uint32_t len, uint32_t &bit) {
    const uint32_t a = (pos & 0x7FFFFFFFu) + e, sh = a & 31u, end = sh + len;
    const uint32_t *w = reinterpret_cast<const uint32_t *>((pos >> 31) ? s.scr : s.rec) + (a >> 5);
    const uint32_t lw = end >> 5;   // word of the last bit
    uint32_t x[5];
#pragma unroll
    for (int i = 0; i < 5; i++) x[i] = (uint32_t)i <= lw ? __ldg(w + i) : 0u;
    uint32_t c = 0, last = x[0];
#pragma unroll
    for (int i = 0; i < 5; i++) {
        if ((uint32_t)i < lw) c += __popc(x[i]);
        if ((uint32_t)i == lw) last = x[i];
    }
    for (uint32_t i = 5; i <= lw; i++) {   // (superblocks of more than 128 bits)
        last = __ldg(w + i);
        if (i < lw) c += __popc(last);
    }
    bit = (last >> (end & 31u)) & 1u;
    return c + __popc(last & ((1u << (end & 31u)) - 1u)) - __popc(x[0] & ((1u << sh) - 1u));
}

__global__ void __launch_bounds__(256) access_kernel(const uint8_t *__restrict__ comp,
                                                     const uint64_t *__restrict__ comp_off, int nblk,
                                                     const uint32_t *__restrict__ qblk, const uint32_t *__restrict__ qpos,
                                                     int nq, uint8_t *__restrict__ sym, int32_t *__restrict__ qstatus,
                                                     const uint8_t *__restrict__ ws, uint64_t ws_bytes,
                                                     const int32_t *__restrict__ status) {
    const DecWs W = dec_ws(const_cast<uint8_t *>(ws), nblk);
    const DecRegions G = dec_regions(nblk, ws);
    const uint32_t dir_bits = dec_dir_bits(ws);
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += gridDim.x * blockDim.x) {
        const uint32_t b = qblk[q], x0 = qpos[q];
        uint8_t out = 0;
        int32_t st = PIVCO_OK;
        if (b >= (uint32_t)nblk) {
            st = PIVCO_ERR_INVALID_ARG;
        } else if ((st = status[b]) == PIVCO_OK) {
            const uint8_t *rec = comp + comp_off[b];   // validated by the plan
            const uint4 h = __ldg(reinterpret_cast<const uint4 *>(rec));   // rb, n, V | kind << 16 | aux << 24, tag
            if (x0 >= h.y) {
                st = PIVCO_ERR_INVALID_ARG;
            } else if (((h.z >> 16) & 0xFFu) == 1) {
                out = (uint8_t)(h.z >> 24);
            } else {
                const uint32_t rb = h.x, V = h.z & 0xFFFFu;
                const uint64_t nbase = G.dir + W.blk_dir[b], ntb = ntab_bytes(V);
                const uint8_t *nt = ws + nbase;
                const uint32_t ent = nbase + ntb <= ws_bytes ? *reinterpret_cast<const uint32_t *>(nt + 20) : 0u;
                if (!ent || nbase + ntb + 4ull * ent > ws_bytes) {
                    st = PIVCO_ERR_INVALID_ARG;   // no directory: the workspace was not prepared for access
                } else {
                    const uint32_t *nsrc = reinterpret_cast<const uint32_t *>(nt + kNtabHdr);
                    const uint32_t *dirp = reinterpret_cast<const uint32_t *>(nt + ntb);
                    const uint32_t *nv = reinterpret_cast<const uint32_t *>(rec + kNvOff);
                    const uint64_t sbase = G.scratch + W.blk_scratch[b];
                    TileSrc src;
                    src.rec = rec;
                    src.rec_bytes = rb;
                    src.scr = ws + sbase;
                    src.scr_bytes = ws_bytes > sbase ? ws_bytes - sbase : 0;
                    uint32_t v = 0, x = x0;
                    st = PIVCO_ERR_CORRUPT;   // unless a leaf is reached within the code-length limit
                    for (int d = 0; d <= (int)kMaxLen && v < V; d++) {
                        const uint32_t nvv = __ldg(nv + v);
                        if (x >= nvv) break;
                        const uint32_t ns = nsrc[3 * v], nc = nsrc[3 * v + 1], nu = nsrc[3 * v + 2];
                        if (const uint32_t D = ch_flat_d(nc)) {
                            // a flat node: the D-bit index of the position, then its symbol
                            const uint32_t xi = tile_bits(src, ns, x * D) & ((1u << D) - 1u);
                            out = nt[kNtabHdr + 12 * V + (nc & 0xFFu) + xi];
                            st = PIVCO_OK;
                            break;
                        }
                        const uint32_t sb = x / dir_bits;
                        uint32_t bit;
                        const uint32_t ones = dirp[nu + sb] + access_rank(src, ns, sb * dir_bits, x - sb * dir_bits, bit);
                        const uint32_t c = (nc >> (16 * bit)) & 0xFFFFu;
                        x = bit ? ones : x - ones;
                        if (c & 0x8000u) {
                            out = (uint8_t)c;
                            st = PIVCO_OK;
                            break;
                        }
                        v = c;
                    }
                }
            }
        }
        sym[q] = out;
        if (qstatus) qstatus[q] = st;
    }
}

cudaError_t launch_access_prepare(const uint8_t *comp, const uint64_t *comp_off, int nblk, uint8_t *ws, size_t ws_bytes,
                                  int32_t *status, cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    cudaError_t e = launch_decode_plan(comp, comp_off, nblk, ws, ws_bytes, status, st, true);
    if (e == cudaSuccess) e = launch_ans_decode_planned(comp, comp_off, nblk, ws, ws_bytes, status, st);
    if (e == cudaSuccess) e = launch_decode_dir(comp, comp_off, nblk, ws, ws_bytes, status, st, true);
    return e;
}

cudaError_t launch_access(const uint8_t *comp, const uint64_t *comp_off, int nblk, const uint32_t *qblk,
                          const uint32_t *qpos, int nq, uint8_t *sym, int32_t *qstatus, const uint8_t *ws,
                          size_t ws_bytes, const int32_t *status, cudaStream_t st) {
    if (nq <= 0) return cudaSuccess;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = min(div_up(nq, 256), sms * 8);
    access_kernel<<<grid, 256, 0, st>>>(comp, comp_off, nblk, qblk, qpos, nq, sym, qstatus, ws, ws_bytes, status);
    count_launches(1);
    return cudaGetLastError();
}

// Host: an upper bound, from host copies of the records, of the workspace the
// decode of these blocks needs under tuning `tu` (never below what the plan
// computes for valid records): the scratch of every ANS-coded node exactly,
// and rank directories plus tile cursors for the most tiles the plan can
// choose (a level of a valid record holds at most n symbols).
size_t decode_ws_bound(const uint8_t *comp, const uint64_t *comp_off, int nblk, const DecTuning &tu) {
    uint64_t dir = 0, scratch = 0;
    // the shortest tile the plan can choose: a level of at most 128 nodes and
    // at most n symbols in a buffer, 20 % headroom, a multiple of 128
    const uint64_t t_fit = ((uint64_t)(kLvlFit - 4 * 128 - 32) / 5 * 4) & ~127ull;
    uint64_t t_min = tu.tile_max < t_fit ? tu.tile_max : t_fit;
    if (t_min < 128) t_min = 128;
    for (int b = 0; b < nblk; b++) {
        const uint8_t *rec = comp + comp_off[b];
        const uint64_t avail = comp_off[b + 1] > comp_off[b] ? comp_off[b + 1] - comp_off[b] : 0;
        if (avail < kNvOff || rec[10] != 2) continue;
        const uint32_t n = (uint32_t)rec[4] | ((uint32_t)rec[5] << 8) | ((uint32_t)rec[6] << 16) | ((uint32_t)rec[7] << 24);
        const uint32_t V = (uint32_t)rec[8] | ((uint32_t)rec[9] << 8);
        if (V < 1 || V > 255 || kNvOff + 5 * V > avail) continue;
        uint64_t ent = 0;
        for (uint32_t v = 0; v < V; v++) {
            const uint8_t *p = rec + kNvOff + 4 * v;
            const uint32_t nv = (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) | ((uint32_t)p[3] << 24);
            const uint8_t m = rec[kNvOff + 4 * V + v];
            ent += (nv + (uint64_t)tu.dir_bits - 1) / tu.dir_bits;
            if (mark_ans(m)) scratch += scratch_stride((nv + 7) / 8);
        }
        uint64_t ntile = ((uint64_t)n + t_min - 1) / t_min;
        if (ntile > (1u << 21)) ntile = 1u << 21;
        dir += ntab_bytes(V) + ((4 * ent + 4 * (ntile + 1) * V + 15) & ~(uint64_t)15);
    }
    return ((decode_ws_fixed_bytes(nblk) + dir + 255) & ~(size_t)255) + scratch + 256;
}

// Host: an upper bound of the same workspace from the blocks' sizes alone
// (no record is read): every block taken as 255 nodes carrying at most 15
// bits per symbol, all of them ANS-coded.  For callers that place records
// they have not seen yet.
size_t decode_ws_size_bound(const uint64_t *blk_off, int nblk, const DecTuning &tu) {
    const uint64_t t_fit = ((uint64_t)(kLvlFit - 4 * 128 - 32) / 5 * 4) & ~127ull;
    uint64_t t_min = tu.tile_max < t_fit ? tu.tile_max : t_fit;
    if (t_min < 128) t_min = 128;
    uint64_t dir = 0, scratch = 0;
    for (int b = 0; b < nblk; b++) {
        const uint64_t n = blk_off[b + 1] - blk_off[b];
        if (n < 2) continue;   // empty and one-symbol blocks have no nodes
        const uint64_t ent = 15 * n / tu.dir_bits + 255;
        uint64_t ntile = (n + t_min - 1) / t_min;
        if (ntile > (1u << 21)) ntile = 1u << 21;
        dir += ntab_bytes(255) + ((4 * ent + 4 * (ntile + 1) * 255 + 15) & ~(uint64_t)15);
        scratch += 15 * n / 8 + 255ull * 48;
    }
    return ((decode_ws_fixed_bytes(nblk) + dir + 255) & ~(size_t)255) + scratch + 256;
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
static int merge_grid(const void *fn, int smem) {
    int dev = 0, sms = 148, occ = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kDecThreads, smem);
    const uint32_t want = current_tuning().ctas_per_sm;
    if (want && (int)want < occ) occ = (int)want;
    if (occ < 1) occ = 1;
    return sms * occ;
}

// The directory pass: shares, then (access = false) the tile boundaries'
// cursors or (access = true, after a plan with a directory for every coded
// block) the entries counted from their block's start.
cudaError_t launch_decode_dir(const uint8_t *comp, const uint64_t *comp_off, int nblk, uint8_t *ws, size_t ws_bytes,
                              int32_t *status, cudaStream_t st, bool access) {
    if (nblk <= 0) return cudaSuccess;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = sms * 4;
    decode_dir_kernel<kDirShare><<<grid, kDecThreads, kDirSmem, st>>>(comp, comp_off, nblk, ws, ws_bytes, status);
    if (access) decode_dir_kernel<kDirRebase><<<grid, kDecThreads, kDirSmem, st>>>(comp, comp_off, nblk, ws, ws_bytes, status);
    else decode_dir_kernel<kDirCursors><<<grid, kDecThreads, kDirSmem, st>>>(comp, comp_off, nblk, ws, ws_bytes, status);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_decode(const uint8_t *comp, const uint64_t *comp_off, int nblk, uint8_t *out,
                          const uint64_t *out_off, uint8_t *ws, size_t ws_bytes, int32_t *status, cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    cudaError_t e = launch_decode_plan(comp, comp_off, nblk, ws, ws_bytes, status, st);
    if (e != cudaSuccess) return e;
    e = launch_ans_decode_planned(comp, comp_off, nblk, ws, ws_bytes, status, st);
    if (e != cudaSuccess) return e;
    return launch_decode_merge(comp, comp_off, nblk, out, out_off, ws, ws_bytes, status, st);
}

cudaError_t launch_decode_merge(const uint8_t *comp, const uint64_t *comp_off, int nblk, uint8_t *out,
                                const uint64_t *out_off, uint8_t *ws, size_t ws_bytes, int32_t *status,
                                cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    cudaError_t e = launch_decode_dir(comp, comp_off, nblk, ws, ws_bytes, status, st, false);
    if (e != cudaSuccess) return e;
    const int smem = (int)sizeof(TileSmem);
    e = cudaFuncSetAttribute(decode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    decode_kernel<<<merge_grid((const void *)decode_kernel, smem), kDecThreads, smem, st>>>(
        comp, comp_off, nblk, out, out_off, ws, ws_bytes, status);
    count_launches(1);
    return cudaGetLastError();
}

bool serve_wide(int nblk) {
    return wide_batch(nblk, merge_grid((const void *)serve_loop_kernel, (int)sizeof(BatchSmem)));
}

cudaError_t launch_serve_loop(ServeCtl *ctl, const ServeDesc *ring, ServeFlags *flags, uint64_t idle_ns,
                              uint64_t life_ns, cudaStream_t st) {
    const int smem = (int)sizeof(BatchSmem);
    cudaError_t e = cudaFuncSetAttribute(serve_loop_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    serve_loop_kernel<<<merge_grid((const void *)serve_loop_kernel, smem), kDecThreads, smem, st>>>(
        ctl, ring, flags, idle_ns, life_ns, host_ans_tables());
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_decode_batch(const uint8_t *comp, const uint64_t *comp_off, int nblk, uint8_t *out,
                                const uint64_t *out_off, uint8_t *ws, size_t ws_bytes, int32_t *status,
                                cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    const DecTuning tu = current_tuning();
    dec_ws_init_kernel<<<min(1024, div_up(nblk, 256)), 256, 0, st>>>(ws, nblk, tu.dir_bits, tu.tile_max,
                                                                      wait_limit_ns());
    const int smem = (int)sizeof(BatchSmem);
    cudaError_t e = cudaFuncSetAttribute(decode_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    decode_batch_kernel<<<merge_grid((const void *)decode_batch_kernel, smem), kDecThreads, smem, st>>>(
        comp, comp_off, nblk, out, out_off, ws, ws_bytes, status, host_ans_tables());
    count_launches(2);
    return cudaGetLastError();
}

}  // namespace pv

namespace pv {
// dynamic shared-memory limits of the decode kernels (set before any capture)
cudaError_t prepare_decode_kernels() {
    cudaError_t e = cudaFuncSetAttribute(decode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TileSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(ans_decode_planned_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kSelBytes + sizeof(AnsItemSm)));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(decode_plan_items_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kSelBytes + sizeof(PlanItemSm)));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(decode_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BatchSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(serve_loop_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BatchSmem));
    return e;
}
}  // namespace pv
