// Encode kernel: per-node bitmap emission by stable partition (Sec. 4, Sec. 2.4.1).
//
// One CTA encodes one block, top-down, level by level; its warps share two
// level buffers.  A block whose levels fit them is coded in one part (the
// planning pass's chunk histograms give every node's symbol count); a big
// block (one whose levels do not fit, or one of a small batch) is coded in
// parts of a length the plan has chosen, by several CTAs (one planning chunk,
// or a share of one, each), a part's counts taken from the input.  A node's bitmap holds, in block order, the code bit of every
// symbol passing through it, so a part's bits of node v start at the symbols
// under v in the parts before it: the cursors advance by each part's counts.
//
// Below the root a symbol travels as its code index, its place in the order
// of codes, in one byte: the leaves under a node are consecutive there, so
// its code bit at node v is (index >= split of v), one byte compare, and the
// index in a flat node's group (Sec. 2.2.3) a subtraction.  Per level, the
// symbols of every node are cut into groups of 32 (one bitmap word) and
// windows of 32 groups, which the warps take in rounds of eight.  In a window
// a lane takes 8 consecutive symbols at a time, so that neighbouring lanes
// read and write neighbouring bytes: the compare gives the lane a byte of the
// bitmap, the window's 128 bytes become one word per lane (written to the
// record at the node's cursor; words shared with a neighbour are ORed into
// the zeroed body), and the symbols are stably partitioned into the internal
// children's spans (EPF / EPL / EPR / EPN of Sec. 2.4.1) at the zeros / ones of
// the node before the group: a warp scan within the window, the windows'
// counts across a round (one barrier), a carry across rounds.
//
// What bounds it: instruction issue and shared-memory wavefronts.  (With 32
// symbols of 16 bits to a lane, a window took about 800 instructions and 200
// wavefronts.)  Before and now: 2048 blocks of 128 KiB, 350 -> 283 us; the
// chunks of one block of 1 MiB, 330 -> 52 us, and of 509 text-like blocks, 564
// -> 361 us; 4096 blocks of 64 KiB, whose root has a leaf child, 439 -> 403 us.

#include "levels.cuh"

namespace pv {

constexpr int kEncThreads = 256;
constexpr int kEncWarps = kEncThreads / 32;
static_assert(kEncWarps == kLvlWarps, "the level tables are laid out by all warps");

struct __align__(16) EncSmem {
    static constexpr int kBuf = kEBuf;      // symbols per level buffer
    uint8_t buf[2][kEBuf + 16];             // depth d >= 1 reads buf[d & 1], writes its children to the other
    uint32_t pos[256];                      // bit address of node v's first bit of the current part
    uint32_t dem[256];                      // symbols of node v in the current part
    uint32_t ch[256];                       // children word (node-table format; ch_flat for a flat node)
    uint32_t end[256];                      // bit address of the end of node v's body (of the item's part of it)
    uint32_t strip[kEncWarps][72];          // a window's bitmap bytes, or a flat step's packed indices
    uint32_t wtot[2][kEncWarps];            // ones of a round's ordinary windows, two rounds deep
    uint16_t sp[256], gs[256], fw[256];     // (levels.cuh; fw of an ordinary node: ones before its first group in
                                            // that group's window)
    uint16_t wpre[kWinMax];                 // prefixes of earlier rounds (levels of more than 8 windows)
    uint16_t lg[16], no[16], nwo[16], nw[16], wn_off[16];
    uint8_t onode[256];
    uint8_t wnode[kWinMax];
    uint8_t split[256];                     // first code index of node v's right child; a flat node's first index
    uint8_t ci[256];                        // code index of symbol s; 255 for a symbol without a code
    uint8_t nlo[256];                       // node v's leaves are code indices nlo[v] .. nhi1[v]
    uint8_t nhi1[256];
    uint32_t lut[256];                      // byte selectors that bring the symbols of a bitmap byte's zeros to the
                                            // front (first four in the low half)
    uint32_t pmask[8];                      // symbols that have a code
    uint32_t bad;                           // the part's symbols do not match its counts
    uint8_t first[17];
    uint8_t maxd;
    uint8_t pad[2];
};
static_assert(kEncCtasPerSm * (sizeof(EncSmem) + 64 + 1024) <= 228 * 1024, "encoder CTAs per SM");
static_assert(offsetof(BlockLayout, ci) <= sizeof(EncSmem::buf[1]) && offsetof(BlockLayout, ci) % 16 == 0,
              "the staged part of the layout fits a level buffer");
static_assert(sizeof(EncSmem::buf[0]) >= 4 * (256 + 256 + 257), "a level buffer holds the counting scratch");

template <typename F, typename G>
__device__ inline uint32_t warp_scan_loop(int n, F f, G out) {
    const int lane = threadIdx.x & 31;
    uint32_t carry = 0;
    for (int base = 0; base < n; base += 32) {
        const int i = base + lane;
        const uint32_t x = i < n ? f(i) : 0;
        uint32_t inc = x;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (i < n) out(i, carry + inc - x);
        carry += __shfl_sync(0xffffffffu, inc, 31);
    }
    return carry;
}

// Node symbol counts of a histogram h by prefix sums in canonical order: the
// leaves under a node are the contiguous canonical range nlo .. nhi1, so its
// count is a difference of two prefix sums.  One warp; hc (256) and ps (257)
// are scratch.
__device__ inline void enc_counts(const EncSmem &S, const uint32_t *h, uint32_t *cnt, uint32_t *hc, uint32_t *ps) {
    const int lane = threadIdx.x & 31;
    const int V = S.first[S.maxd];
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const int s = lane + 32 * i;
        if ((S.pmask[i] >> lane) & 1u) hc[S.ci[s]] = h[s];
    }
    __syncwarp();
    uint32_t x[8], sum = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) { x[j] = hc[8 * lane + j]; sum += x[j]; }
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    uint32_t run = inc - sum;
    if (lane == 0) ps[0] = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) { run += x[j]; ps[8 * lane + j + 1] = run; }
    __syncwarp();
    for (int v = lane; v < V; v += 32) cnt[v] = ps[S.nhi1[v] + 1] - ps[S.nlo[v]];
    __syncwarp();
}

// Writes bits bw (vl of them valid) of one node at bit address a of the
// record.  Lanes of the same node hold consecutive 32-bit runs; a lane
// stores the aligned word its run starts in, completed with the previous
// lane's spill; words shared with another run (or another node) are ORed.
__device__ inline void enc_put_bits(uint32_t *rec32, bool act, uint32_t v, uint32_t a, uint32_t bw, uint32_t vl) {
    const int lane = threadIdx.x & 31;
    const uint32_t sh = a & 31u, wi = a >> 5;
    const uint32_t lo = bw << sh;
    const uint32_t hi = sh ? bw >> (32 - sh) : 0u;
    const uint32_t key = act ? v : 0xFFFFFFFFu;
    const uint32_t pkey = __shfl_up_sync(0xffffffffu, key, 1), nkey = __shfl_down_sync(0xffffffffu, key, 1);
    const uint32_t phi = __shfl_up_sync(0xffffffffu, hi, 1);
    const bool prev_same = lane > 0 && act && pkey == v;
    const bool next_same = lane < 31 && act && nkey == v;
    if (!act) return;
    const uint32_t word = lo | (prev_same ? phi : 0u);
    const bool full = (sh == 0 || prev_same) && vl >= 32 - sh;
    if (full) rec32[wi] = word;
    else if (word) atomicOr(&rec32[wi], word);
    if (hi && !next_same) atomicOr(&rec32[wi + 1], hi);
}

// ---- bytes ----
// bit j: whether byte j of the 8 in x0, x1 is marked in bit 7 of m0, m1 (the
// dot product weighs bits 3 and 7 of byte j by 2^j)
__device__ inline uint32_t gather8(uint32_t m0, uint32_t m1) {
    return __dp4a(((m0 >> 4) & 0x08080808u) | (m1 & 0x80808080u), 0x08040201u, 0u) >> 3;
}
// bytes of x not below those of s, marked in bit 7
__device__ inline uint32_t ge4(uint32_t x, uint32_t s) {
    const uint32_t t = (x | 0x80808080u) - (s & 0x7F7F7F7Fu);
    return (x & ~s) | (~(x ^ s) & t);
}
// bytes of x that are zero, marked in bit 7
__device__ inline uint32_t eq4(uint32_t x) { return ~(((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x); }
// the first n bytes (0..4) of a word
__device__ inline uint32_t mask4(int n) { return n >= 4 ? 0xFFFFFFFFu : (n <= 0 ? 0u : (1u << (8 * n)) - 1u); }

__device__ inline uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
template <int K>
__device__ inline void sts8(uint32_t a, uint32_t v) {
    asm volatile("st.shared.u8 [%0+%2], %1;" ::"r"(a), "r"(v), "n"(K) : "memory");
}

// 8 input bytes at p, `mis` bytes past a 4-byte boundary (bytes at or past
// `end` are not read; at least one byte is before it)
__device__ inline uint2 ldg8(const uint8_t *p, uint32_t mis, const uint8_t *end) {
    const uint32_t *w = reinterpret_cast<const uint32_t *>(p - mis);
    const uint8_t *q = p - mis;
    if (mis == 0) {
        if (!(reinterpret_cast<uintptr_t>(p) & 7) && p + 8 <= end) return __ldg(reinterpret_cast<const uint2 *>(p));
        return make_uint2(__ldg(w), q + 4 < end ? __ldg(w + 1) : 0u);
    }
    const uint32_t a = __ldg(w), b = q + 4 < end ? __ldg(w + 1) : 0u, c = q + 8 < end ? __ldg(w + 2) : 0u;
    return make_uint2(__funnelshift_r(a, b, 8 * mis), __funnelshift_r(b, c, 8 * mis));
}

// What a window's groups carry to their lanes' steps: the bitmap word, the
// children's next places in the level below (of the group's first symbol,
// left | right << 16) and bits 0..5 its symbols, 6 / 7: internal left / right
// child.
struct EncGrp {
    uint32_t w, a, b;
};

// Partitions a window: y[2 s], y[2 s + 1] are the lane's 8 symbols of step s.
// A byte permute by the bitmap byte brings the symbols of its zeros to the
// front; the k-th then goes to the k-th place of the left span or, past the
// zeros, of the right one.
__device__ inline void enc_partition(const EncSmem &S, uint32_t base, const EncGrp &G, const uint32_t (&y)[8]) {
    const int lane = threadIdx.x & 31;
    const uint32_t sub = lane & 3, below = (1u << (8 * sub)) - 1u;
    const bool two = __all_sync(0xffffffffu, (G.b & 0xFFu) == (32u | 0xC0u));   // full groups, both children internal
    if (!__any_sync(0xffffffffu, (G.b & 0xC0u) != 0)) return;
#pragma unroll
    for (int s = 0; s < 4; s++) {
        const int own = 8 * s + (lane >> 2);
        const uint32_t ws = __shfl_sync(0xffffffffu, G.w, own), as = __shfl_sync(0xffffffffu, G.a, own);
        const uint32_t r = __popc(ws & below);
        const uint32_t la = base + (as & 0xFFFFu) + 8 * sub - r;
        uint32_t b8 = (ws >> (8 * sub)) & 0xFFu;
        uint32_t st = 0xFFu;   // sorted symbols stored
        if (!two) {
            const uint32_t bs = __shfl_sync(0xffffffffu, G.b, own);
            const int nv = max(0, min(8, (int)(bs & 63u) - 8 * (int)sub));   // valid symbols of the lane's 8
            b8 |= (0xFFu << nv) & 0xFFu;                                      // (the others sort behind the ones)
            const uint32_t zm = (1u << (8u - __popc(b8))) - 1u;              // the zeros
            st = (bs & 0x40u ? zm : 0u) | (bs & 0x80u ? ((1u << nv) - 1u) & ~zm : 0u);
        }
        const uint32_t z = 8u - __popc(b8), e = S.lut[b8], rb = base + (as >> 16) + r - z;
        const uint32_t s0 = __byte_perm(y[2 * s], y[2 * s + 1], e), s1 = __byte_perm(y[2 * s], y[2 * s + 1], e >> 16);
        if (two) {
            sts8<0>(z > 0 ? la : rb, s0);
            sts8<1>(z > 1 ? la : rb, s0 >> 8);
            sts8<2>(z > 2 ? la : rb, s0 >> 16);
            sts8<3>(z > 3 ? la : rb, s0 >> 24);
            sts8<4>(z > 4 ? la : rb, s1);
            sts8<5>(z > 5 ? la : rb, s1 >> 8);
            sts8<6>(z > 6 ? la : rb, s1 >> 16);
            sts8<7>(z > 7 ? la : rb, s1 >> 24);
        } else {
            if (st & 1u) sts8<0>(z > 0 ? la : rb, s0);
            if (st & 2u) sts8<1>(z > 1 ? la : rb, s0 >> 8);
            if (st & 4u) sts8<2>(z > 2 ? la : rb, s0 >> 16);
            if (st & 8u) sts8<3>(z > 3 ? la : rb, s0 >> 24);
            if (st & 16u) sts8<4>(z > 4 ? la : rb, s1);
            if (st & 32u) sts8<5>(z > 5 ? la : rb, s1 >> 8);
            if (st & 64u) sts8<6>(z > 6 ? la : rb, s1 >> 16);
            if (st & 128u) sts8<7>(z > 7 ? la : rb, s1 >> 24);
        }
    }
}

// One side of a root window (its other child is a leaf): keep: the symbols
// kept, one bit each; at: the place of the group's first kept symbol.
__device__ inline void enc_keep(const EncSmem &S, uint32_t base, uint32_t keep, uint32_t at, const uint32_t (&y)[8]) {
    const int lane = threadIdx.x & 31;
    const uint32_t sub = lane & 3, below = (1u << (8 * sub)) - 1u;
#pragma unroll
    for (int s = 0; s < 4; s++) {
        const int own = 8 * s + (lane >> 2);
        const uint32_t ws = __shfl_sync(0xffffffffu, keep, own), as = __shfl_sync(0xffffffffu, at, own);
        const uint32_t p = base + as + __popc(ws & below), b8 = (ws >> (8 * sub)) & 0xFFu, c = __popc(b8);
        const uint32_t e = S.lut[b8 ^ 0xFFu];
        const uint32_t s0 = __byte_perm(y[2 * s], y[2 * s + 1], e);
        if (c > 0) sts8<0>(p, s0);
        if (c > 1) sts8<1>(p, s0 >> 8);
        if (c > 2) sts8<2>(p, s0 >> 16);
        if (c > 3) sts8<3>(p, s0 >> 24);
        if (__any_sync(0xffffffffu, c > 4)) {   // (rare on the skewed roots that keep one side)
            const uint32_t s1 = __byte_perm(y[2 * s], y[2 * s + 1], e >> 16);
            if (c > 4) sts8<4>(p, s1);
            if (c > 5) sts8<5>(p, s1 >> 8);
            if (c > 6) sts8<6>(p, s1 >> 16);
            if (c > 7) sts8<7>(p, s1 >> 24);
        }
    }
}

// code indices of four symbols; none: a byte of 255 among them
__device__ inline uint32_t enc_codes4(const EncSmem &S, uint32_t x) {
    return (uint32_t)S.ci[x & 0xFFu] | ((uint32_t)S.ci[(x >> 8) & 0xFFu] << 8) | ((uint32_t)S.ci[(x >> 16) & 0xFFu] << 16) |
           ((uint32_t)S.ci[x >> 24] << 24);
}
__device__ inline uint32_t any255(uint32_t c) { return (~c - 0x01010101u) & c & 0x80808080u; }
// 255 is a symbol's index only when all 256 have codes
__device__ inline bool enc_all_codes(const EncSmem &S) {
    return (S.pmask[0] & S.pmask[1] & S.pmask[2] & S.pmask[3] & S.pmask[4] & S.pmask[5] & S.pmask[6] & S.pmask[7]) ==
           0xFFFFFFFFu;
}

// A warp packs 256 symbols of a flat node D bits each (the lane's 8 code
// indices y0, y1, their first nv valid; lo4: the node's first code index in
// all bytes) and writes the nbits packed bits at bit address a of the record:
// words inside the run are stored, the two it shares with its neighbours are
// ORed into the zeroed body.
__device__ inline void enc_flat_step(uint32_t *strip, uint32_t *rec32, uint32_t D, uint32_t lo4, uint32_t y0, uint32_t y1,
                                     int nv, uint32_t a, uint32_t nbits) {
    const int lane = threadIdx.x & 31;
    const uint32_t m = (1u << D) - 1u;
    auto pack = [&](uint32_t y, int n) {
        const uint32_t x = (y - lo4) & mask4(n);   // (every valid byte is at least lo4's)
        return (x & m) | ((x >> (8 - D)) & (m << D)) | ((x >> (16 - 2 * D)) & (m << (2 * D))) |
               (D == 8 ? x & 0xFF000000u : (x >> (24 - 3 * D)) & (m << (3 * D)));
    };
    const uint64_t bits = (uint64_t)pack(y0, nv) | ((uint64_t)pack(y1, nv - 4) << (4 * D));
    uint8_t *sb = reinterpret_cast<uint8_t *>(strip) + D * lane;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 8; k++)
        if ((uint32_t)k < D) sb[k] = (uint8_t)(bits >> (8 * k));
    __syncwarp();
    const uint32_t sh = a & 31u, wi = a >> 5, end = sh + nbits;   // bits sh .. end - 1 of the words from wi on
    for (uint32_t i = lane; 32 * i < end; i += 32) {
        const uint32_t cur = 32 * i < nbits ? strip[i] : 0u, prev = i ? strip[i - 1] : 0u;
        uint32_t o = sh ? (cur << sh) | (prev >> (32 - sh)) : cur;
        if (32 * i + 32 > end) o &= (1u << (end - 32 * i)) - 1u;
        if (32 * i >= sh && 32 * i + 32 <= end) rec32[wi + i] = o;
        else if (o) atomicOr(&rec32[wi + i], o);
    }
}

// One part of a block whose demands and cursors are in S: symbols [src, src +
// C), every level; the whole CTA.  Ends with a barrier.
__device__ inline void enc_part(EncSmem &S, const uint8_t *src, uint32_t C, const uint8_t *src_end, uint32_t *rec32) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t sub = lane & 3;
    uint32_t *strip = S.strip[warp];
    uint8_t *stripb = reinterpret_cast<uint8_t *>(strip);
    uint32_t par = 0;
    // ---- the root: input bytes -> bits, code indices; children ----
    {
        const uint32_t chv = S.ch[0], rD = ch_flat_d(chv);
        const uint32_t c0 = chv & 0xFFFFu, c1 = chv >> 16;
        const bool i0 = !rD && !(c0 & 0x8000u), i1 = !rD && !(c1 & 0x8000u);
        const uint32_t nwin = (C + kWin - 1) / kWin, mis = (uint32_t)(reinterpret_cast<uintptr_t>(src) & 3);
        // a leaf child decides the bit by its symbol alone; two internal ones (or a flat root) by the code index
        const bool code = !rD && !(i0 && i1);
        const uint32_t leaf4 = (i0 ? c1 & 0xFFu : c0 & 0xFFu) * 0x01010101u, flip = i0 ? 0u : 0xFFFFFFFFu;
        const uint32_t split4v = S.split[0] * 0x01010101u;
        const uint32_t base = smem_addr(S.buf[1]);
        const uint32_t sp0 = i0 ? S.sp[c0 & 0xFFu] : 0u, sp1 = i1 ? S.sp[c1 & 0xFFu] : 0u;
        const uint32_t dem0 = i0 ? S.dem[c0 & 0xFFu] : 0xFFFFFFFFu, dem1 = i1 ? S.dem[c1 & 0xFFu] : 0xFFFFFFFFu, pos0 = S.pos[0];
        const bool al8 = !(reinterpret_cast<uintptr_t>(src) & 7);
        uint32_t carry = 0;
        bool bad = false;
        for (uint32_t b0 = 0; b0 < nwin; b0 += kEncWarps) {
            const uint32_t i = b0 + warp, k0 = kWin * i;
            const bool full = k0 + kWin <= C;
            uint32_t y[8], w = 0, inc = 0, pc = 0;
            if (i < nwin) {
                if (full && al8) {
                    const uint2 *p = reinterpret_cast<const uint2 *>(src + k0) + lane;
#pragma unroll
                    for (int s = 0; s < 4; s++) {
                        const uint2 x = __ldg(p + 32 * s);
                        y[2 * s] = x.x;
                        y[2 * s + 1] = x.y;
                    }
                } else {
#pragma unroll
                    for (int s = 0; s < 4; s++) {
                        const uint32_t k = k0 + 256 * s + 8 * lane;
                        uint2 x = make_uint2(0u, 0u);
                        if (k < C) x = ldg8(src + k, mis, src_end);
                        y[2 * s] = x.x;
                        y[2 * s + 1] = x.y;
                    }
                }
                if (!code) {
                    uint32_t none = 0;
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        uint32_t c = enc_codes4(S, y[j]);
                        if (!full) c &= mask4((int)C - (int)(k0 + 256 * (j >> 1) + 8 * lane + 4 * (j & 1)));
                        none |= any255(c);
                        y[j] = c;
                    }
                    if (none && !enc_all_codes(S)) bad = true;
                } else if (!i0 && !i1) {   // two symbols in all: nothing else may occur
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        const uint32_t ok = eq4(y[j] ^ leaf4) | eq4(y[j] ^ ((c1 & 0xFFu) * 0x01010101u));
                        if (~ok & 0x80808080u & mask4((int)C - (int)(k0 + 256 * (j >> 1) + 8 * lane + 4 * (j & 1)))) bad = true;
                    }
                }
                if (rD) {
                    const uint32_t lo4 = split4v;
#pragma unroll
                    for (int s = 0; s < 4; s++) {
                        const uint32_t k = k0 + 256 * s;
                        if (k < C)
                            enc_flat_step(strip, rec32, rD, lo4, y[2 * s], y[2 * s + 1],
                                          max(0, min(8, (int)C - (int)(k + 8 * lane))), pos0 + k * rD, min(256u, C - k) * rD);
                    }
                } else {
                    __syncwarp();
#pragma unroll
                    for (int s = 0; s < 4; s++) {
                        uint32_t m0, m1;
                        if (code) { m0 = eq4(y[2 * s] ^ leaf4) ^ flip; m1 = eq4(y[2 * s + 1] ^ leaf4) ^ flip; }
                        else { m0 = ge4(y[2 * s], split4v); m1 = ge4(y[2 * s + 1], split4v); }
                        stripb[32 * s + lane] = (uint8_t)gather8(m0, m1);
                    }
                    __syncwarp();
                    const uint32_t kk = k0 + kGrp * lane, vl = full ? 32u : (kk < C ? min(32u, C - kk) : 0u);
                    w = strip[lane];
                    if (vl < 32) w &= (1u << vl) - 1u;
                    pc = __popc(w);
                    inc = warp_inclusive(pc);
                    if (lane == 31) S.wtot[par][warp] = inc;
                    inc -= pc;
                    enc_put_bits(rec32, vl != 0, 0u, pos0 + kk, w, vl);
                }
            }
            __syncthreads();
            if (!rD) {
                // ones before each window of the round (lane: window)
                const uint32_t x = lane < kEncWarps && b0 + lane < nwin ? S.wtot[par][lane] : 0u;
                uint32_t in = x;
#pragma unroll
                for (int o = 1; o < kEncWarps; o <<= 1) {
                    const uint32_t z = __shfl_up_sync(0xffffffffu, in, o);
                    if (lane >= o) in += z;
                }
                const uint32_t r1 = carry + __shfl_sync(0xffffffffu, in - x, warp) + inc;
                carry += __shfl_sync(0xffffffffu, in, kEncWarps - 1);
                if (i < nwin) {
                    const uint32_t kk = k0 + kGrp * lane, vl = full ? 32u : (kk < C ? min(32u, C - kk) : 0u);
                    // a part whose symbols do not match its counts must not write past the spans
                    const bool over = vl && (r1 + pc > dem1 || kk + vl - r1 - pc > dem0);
                    if (over) bad = true;
                    if (code) {
                        const uint32_t vm = vl >= 32 ? 0xFFFFFFFFu : (1u << vl) - 1u;
                        if (i0 || i1) enc_keep(S, base, over ? 0u : (i0 ? ~w : w) & vm, i0 ? sp0 + kk - r1 : sp1 + r1, y);
                    } else {
                        EncGrp G;
                        G.w = w;
                        G.a = over ? 0u : (sp0 + kk - r1) | ((sp1 + r1) << 16);
                        G.b = (over ? 0u : vl) | 0xC0u;
                        enc_partition(S, base, G, y);
                    }
                }
            }
            par ^= 1u;
        }
        // (carry: all the root's ones; too few symbols for a child would leave its span as the buffer was)
        if ((i1 && carry != dem1) || (i0 && C - carry != dem0)) bad = true;
        if (code && (i0 || i1)) {
            // the kept symbols are input bytes still: their code indices
            __syncthreads();
            const uint32_t n1 = S.dem[i0 ? c0 & 0xFFu : c1 & 0xFFu];
            uint2 *p = reinterpret_cast<uint2 *>(S.buf[1] + (i0 ? sp0 : sp1));
            uint32_t none = 0;
            for (uint32_t k = 8 * t; k < n1; k += 8 * kEncThreads) {
                uint2 x = p[k >> 3];
                x.x = enc_codes4(S, x.x);
                x.y = enc_codes4(S, x.y);
                p[k >> 3] = x;
                none |= any255(x.x & mask4((int)(n1 - k))) | any255(x.y & mask4((int)(n1 - k) - 4));
            }
            if (none && !enc_all_codes(S)) bad = true;
        }
        if (bad) S.bad = 1;
    }
    __syncthreads();
    // ---- depths 1.. : node spans of buf[d & 1] into the children's spans ----
    for (int d = 1; d < (int)S.maxd; d++) {
        const uint8_t *bin = S.buf[d & 1];
        const uint32_t base = smem_addr(S.buf[(d + 1) & 1]);
        const uint32_t nw = S.nw[d], nwo = S.nwo[d], wn = S.wn_off[d], f0 = S.first[d];
        uint32_t carry = 0;
        bool bad = false;
        for (uint32_t b0 = 0; b0 < nw; b0 += kEncWarps) {
            const uint32_t i = b0 + warp;
            uint32_t v = 0, q = 0, left = 0, y[8], w = 0, inc = 0, pc = 0;
            if (i < nwo) {
                left = lvl_locate(S, d, wn, f0, i, v, q);
                // bits 0..15: the group's place in the level buffer, 16..23: the node's split
                const uint32_t pk = (left ? (uint32_t)S.sp[v] + kGrp * q : 0u) | ((uint32_t)S.split[v] << 16);
                __syncwarp();
#pragma unroll
                for (int s = 0; s < 4; s++) {
                    const uint32_t ps = __shfl_sync(0xffffffffu, pk, 8 * s + (lane >> 2));
                    const uint2 x = *reinterpret_cast<const uint2 *>(bin + (ps & 0xFFFFu) + 8 * sub);
                    const uint32_t sv = (ps >> 16) * 0x01010101u;
                    y[2 * s] = x.x;
                    y[2 * s + 1] = x.y;
                    stripb[32 * s + lane] = (uint8_t)gather8(ge4(x.x, sv), ge4(x.y, sv));
                }
                __syncwarp();
                w = left ? strip[lane] : 0u;
                if (left < 32) w &= (1u << left) - 1u;
                pc = __popc(w);
                inc = warp_inclusive(pc);
                if (lane == 31) S.wtot[par][warp] = inc;
                inc -= pc;
                // a node's first group: the ones of the window before it
                if (q == 0) S.fw[v] = (uint16_t)inc;
                enc_put_bits(rec32, left != 0, v, S.pos[v] + kGrp * q, w, min(32u, left));
            }
            __syncthreads();
            par ^= 1u;
            if (i < nwo) {
                uint32_t ex = 0, ps = 0;
                if (nwo > 1) {
                    // ones of the level before each window of the round (lane: window)
                    const uint32_t x = lane < kEncWarps && b0 + lane < nwo ? S.wtot[par ^ 1u][lane] : 0u;
                    uint32_t in = x;
#pragma unroll
                    for (int o = 1; o < kEncWarps; o <<= 1) {
                        const uint32_t z = __shfl_up_sync(0xffffffffu, in, o);
                        if (lane >= o) in += z;
                    }
                    ex = carry + in - x;
                    if (nwo > kEncWarps) {
                        carry += __shfl_sync(0xffffffffu, in, kEncWarps - 1);
                        if (warp == 0 && lane < kEncWarps && b0 + lane < nwo) S.wpre[wn + b0 + lane] = (uint16_t)ex;
                    }
                    // at the node's first group
                    const uint32_t gw = (32u * i + lane - q) >> 5;   // its window
                    ps = __shfl_sync(0xffffffffu, ex, gw - b0);
                    if (gw < b0) ps = S.wpre[wn + gw];
                    ex = __shfl_sync(0xffffffffu, ex, warp);
                }
                const uint32_t r1 = (ex + inc - ps - S.fw[v]) & 0xFFFFu, kk = kGrp * q, vl = min(32u, left);
                const uint32_t chv = S.ch[v], c0 = chv & 0xFFFFu, c1 = chv >> 16;
                const bool i0 = left && !(c0 & 0x8000u), i1 = left && !(c1 & 0x8000u);
                const uint32_t n0 = kk + vl - r1 - pc, n1 = r1 + pc;
                const uint32_t d0 = i0 ? S.dem[c0 & 0xFFu] : n0, d1 = i1 ? S.dem[c1 & 0xFFu] : n1;
                const bool over = n0 > d0 || n1 > d1;
                // the node's last group: its children have got exactly what they count
                if (over || (left <= 32 && (n0 != d0 || n1 != d1))) bad = true;
                EncGrp G;
                G.w = w;
                G.a = over ? 0u : (((i0 ? (uint32_t)S.sp[c0 & 0xFFu] : 0u) + kk - r1) & 0xFFFFu) |
                                      (((i1 ? (uint32_t)S.sp[c1 & 0xFFu] : 0u) + r1) << 16);
                G.b = (over ? 0u : vl) | (i0 ? 0x40u : 0u) | (i1 ? 0x80u : 0u);
                enc_partition(S, base, G, y);
            } else if (i < nw) {
                // a flat node's window: its packed indices
                const uint32_t v2 = S.wnode[wn + i], fD = ch_flat_d(S.ch[v2]), dv = S.dem[v2], lo4 = S.split[v2] * 0x01010101u;
                const uint32_t k0 = (i - nwo - S.fw[v2]) * kWin, k1 = min(dv, k0 + kWin);
#pragma unroll 1
                for (uint32_t k = k0; k < k1; k += 256) {
                    const uint32_t kl = k + 8 * lane;
                    uint2 x = make_uint2(0u, 0u);
                    if (kl < dv) x = *reinterpret_cast<const uint2 *>(bin + S.sp[v2] + kl);
                    enc_flat_step(strip, rec32, fD, lo4, x.x, x.y, max(0, min(8, (int)dv - (int)kl)), S.pos[v2] + k * fD,
                                  min(256u, dv - k) * fD);
                }
            }
        }
        if (bad) S.bad = 1;
        __syncthreads();
    }
}

// Counts input bytes [lo, hi) of the block at src into hist (256 zeroed bins;
// the whole CTA, no barrier): one shared add per byte, by aligned vectors (the
// order does not matter; equal bytes of a warp's add do not serialise).
__device__ inline void enc_count(const uint8_t *src, uint32_t lo, uint32_t hi, uint32_t *hist) {
    const uint32_t t = threadIdx.x, n = hi - lo;
    const uint8_t *p = src + lo;
    const uint32_t head = min(n, (uint32_t)(-reinterpret_cast<intptr_t>(p) & 15)), vecs = (n - head) / 16;
    if (t < head) atomicAdd(&hist[p[t]], 1u);
    const uint32_t rest = head + 16 * vecs;
    if (t < n - rest) atomicAdd(&hist[p[rest + t]], 1u);
    const uint4 *v = reinterpret_cast<const uint4 *>(p + head);
#pragma unroll 2
    for (uint32_t i = t; i < vecs; i += kEncThreads) {
        const uint4 q = __ldg(v + i);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 4; k++)
#pragma unroll
            for (int c = 0; c < 4; c++) atomicAdd(&hist[__byte_perm(w[k], 0u, 0x4440u + c)], 1u);
    }
}

// Codes block b with the whole CTA (every thread calls it with the same
// arguments).  whole: the block entire, its header written, its body zeroed
// here and its status written; else share `share` of `shares` of plan chunk
// cA of a big block: the reset pass has checked the block, zeroed its body
// and set its status, the share starts at the node cursors the counts of the
// chunks before it (and of the chunk's symbols before the share, counted
// here) give, the first item writes the header and tables, and the status
// only ever turns to an error.
template <bool whole>
__device__ inline void encode_item(int b, uint32_t cA, uint32_t share, uint32_t shares, const uint8_t *__restrict__ in,
                                   const uint64_t *__restrict__ blk_off, const BlockLayout *__restrict__ layout,
                                   const uint32_t *__restrict__ chunk_hist, uint8_t *__restrict__ out,
                                   const uint64_t *__restrict__ out_off, uint64_t *__restrict__ rec_bytes,
                                   int32_t *__restrict__ status, EncSmem &S) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint64_t i0 = blk_off[b], i1 = blk_off[b + 1], o0 = out_off[b], o1 = out_off[b + 1];
    const uint64_t n = i1 - i0;
    const uint32_t nw = enc_nchunks(n);
    // the item's symbols: whole multiples of 32 but for the block's end
    const uint32_t ch0 = whole ? 0u : enc_chunk_start(n, cA, nw), ch1 = whole ? (uint32_t)n : enc_chunk_start(n, cA + 1, nw);
    const uint32_t P0 = ch0 + (uint32_t)((uint64_t)(ch1 - ch0) * share / shares & ~31ull);
    const uint32_t P1 = share + 1 == shares ? ch1 : ch0 + (uint32_t)((uint64_t)(ch1 - ch0) * (share + 1) / shares & ~31ull);
    // the item's input is read by the root pass: ask L2 for it now, so
    // those reads find it there
    {
        const uint8_t *p0 = in + i0 + P0;
        for (uint64_t i = 128ull * t; i < P1 - P0; i += 128ull * kEncThreads)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p0 + i));
    }
    // the block's layout, staged into shared memory once (coalesced); it
    // borrows the second level buffer, unused until the levels start
    {
        const uint4 *g = reinterpret_cast<const uint4 *>(reinterpret_cast<const uint8_t *>(layout) +
                                                          (size_t)b * kLayoutBytes);
        uint4 *d = reinterpret_cast<uint4 *>(S.buf[1]);
        constexpr int kStaged = (int)(offsetof(BlockLayout, ci) / 16), kTab = 768 / 16;
        for (int i = t; i < kStaged; i += kEncThreads) d[i] = __ldg(g + i);
        // the canonical order and the nodes' leaf ranges, straight into their tables
        if (t < kTab) reinterpret_cast<uint4 *>(S.ci)[t] = __ldg(g + kStaged + t);
    }
    __syncthreads();
    const BlockLayout &L = *reinterpret_cast<const BlockLayout *>(S.buf[1]);
    uint8_t *rec = out + o0;
    const uint64_t cap = o1 - o0;
    const uint32_t kind = L.kind;
    int st = PIVCO_OK;
    if (L.status != 0) st = L.status;
    else if (L.n != n || (reinterpret_cast<uintptr_t>(rec) & 15)) st = PIVCO_ERR_INVALID_ARG;
    else if (cap < L.rec_bound) st = PIVCO_ERR_CAPACITY;
    if (st != PIVCO_OK || (!whole && kind != 2)) {   // (the reset pass has reported a big block's)
        if (t == 0 && whole) { status[b] = st; rec_bytes[b] = 0; }
        return;
    }
    const int V = L.n_int;
    const uint32_t rec_bound = L.rec_bound;   // the staged layout is overwritten once the levels start
    const bool head = whole || (cA == 0 && share == 0);   // this item writes the header and tables
    // ---- record header (App. D, adapted) ----
    if (t < 16 && head) {
        uint8_t v = 0;
        const uint32_t rb = L.rec_bound;
        if (t < 4) v = (uint8_t)(rb >> (8 * t));
        else if (t < 8) v = (uint8_t)((uint32_t)n >> (8 * (t - 4)));
        else if (t == 8) v = (uint8_t)V;
        else if (t == 9) v = (uint8_t)(V >> 8);
        else if (t == 10) v = (uint8_t)kind;
        else if (t == 11) v = kind == 1 ? L.csym : 0;
        else v = t == 15 ? (L.flat ? '2' : '1') : (uint8_t)"PVC"[t - 12];
        rec[t] = v;
    }
    if (kind != 2) {
        if (t == 0) { status[b] = PIVCO_OK; rec_bytes[b] = kHdr; }
        return;
    }
    // the record start is 16-byte aligned: the length nibbles and n_v as words
    if (t < 32 && head) {
        uint32_t x = 0;
#pragma unroll
        for (int j = 0; j < 8; j++) x |= (uint32_t)(L.len[8 * t + j] & 15u) << (4 * j);
        reinterpret_cast<uint32_t *>(rec + kLensOff)[t] = x;
    }
    if (t < V && head) reinterpret_cast<uint32_t *>(rec + kNvOff)[t] = L.nv[t];
    if (t < V && head) rec[kNvOff + 4 * V + t] = L.fd[t] ? (uint8_t)(kMarkFlat + L.fd[t]) : (L.sel[t] ? kMarkRawSel : 0);
    if (head) {
        const uint32_t pad_lo = kNvOff + 5 * V, alen_off = (pad_lo + 3) & ~3u;
        if (pad_lo + t < alen_off) rec[pad_lo + t] = 0;
        if (warp == 0 && L.n_sel) {
            // the alen table: raw sizes of the selected nodes, in node order
            warp_scan_loop(V, [&](int v) { return (uint32_t)(L.sel[v] != 0); }, [&](int v, uint32_t p) {
                if (L.sel[v]) {
                    const uint32_t raw = (L.nv[v] + 7) / 8;
                    for (int j = 0; j < 4; j++) rec[alen_off + 4 * p + j] = (uint8_t)(raw >> (8 * j));
                }
            });
        }
        if (whole)
            for (uint32_t i = L.body_end + t; i < L.rec_bound; i += kEncThreads) rec[i] = 0;
    }
    // ---- the bitmaps are ORed into a zeroed body ----
    if (whole) {
        const uint32_t b0 = L.body0, b1 = L.body_end;
        const uint32_t h0 = min(b1, (b0 + 15u) & ~15u), h1 = max(h0, b1 & ~15u);
        for (uint32_t i = b0 + t; i < h0; i += kEncThreads) rec[i] = 0;
        for (uint32_t i = h0 + 16 * t; i < h1; i += 16 * kEncThreads)
            *reinterpret_cast<uint4 *>(rec + i) = make_uint4(0u, 0u, 0u, 0u);
        for (uint32_t i = h1 + t; i < b1; i += kEncThreads) rec[i] = 0;
    }
    // ---- per-block tables ----
    {
        const uint32_t l = L.len[t];
        if (!l) S.ci[t] = 255;
        if (t < V) {
            uint32_t code2 = 0;
            for (int c = 0; c < 2; c++) {
                const int ch = L.child[t][c];
                code2 |= (ch >= 0 ? (uint32_t)ch : (0x8000u | (uint32_t)(-ch - 1))) << (16 * c);
            }
            const uint32_t fd = L.fd[t];
            S.ch[t] = fd ? ch_flat(fd, L.fbase[t]) : code2;
            S.pos[t] = 8u * L.body_off[t];
            S.end[t] = 8u * L.body_off[t] + L.nv[t] * max(1u, fd);
        }
        if (t < 17) S.first[t] = L.depth_first[t];
        if (t == 0) { S.maxd = L.max_depth; S.bad = 0; }
        {   // byte t: zeros to the front, both sides in order
            uint32_t e = 0, z = 0, o = 8u - __popc((uint32_t)t);
            for (uint32_t j = 0; j < 8; j++) {
                const uint32_t k = ((uint32_t)t >> j) & 1u ? o++ : z++;
                e |= j << (4 * k);
            }
            S.lut[t] = e;
        }
    }
    __syncthreads();
    const uint32_t part = max(1024u, L.part);
    const bool big = L.big != 0;
    {
        const uint32_t l = L.len[t];
        const uint32_t pm = __ballot_sync(0xffffffffu, l != 0);
        if (lane == 0) S.pmask[warp] = pm;
        // a node's bit is one from its right child's first code index on
        if (t < V) {
            const uint32_t chv = S.ch[t], c1 = chv >> 16;
            S.split[t] = ch_flat_d(chv) ? S.nlo[t] : (c1 & 0x8000u ? S.ci[c1 & 0xFFu] : S.nlo[c1 & 0xFFu]);
        }
    }
    __syncthreads();   // (the staged layout is dead from here on)
    const uint8_t *src = in + i0;
    const uint8_t *src_end = in + i1;
    uint32_t *rec32 = reinterpret_cast<uint32_t *>(rec);
    // counting scratch in the second level buffer (free between parts)
    uint32_t *hist = reinterpret_cast<uint32_t *>(S.buf[1]);
    uint32_t *hc = hist + 256, *ps = hist + 512;
    uint32_t acc = 0;              // count of symbol t in the plan chunk's symbols counted so far
    // an item inside a block starts every node's cursor after the symbols before it
    if (!whole && (cA > 0 || share > 0)) {
        hist[t] = 0;
        __syncthreads();
        enc_count(src, ch0, P0, hist);
        __syncthreads();
        uint32_t h = hist[t];
        acc = h;
        for (uint32_t c = 0; c < cA; c++) h += __ldg(chunk_hist + ((size_t)b * kEncChunks + c) * 256 + t);
        __syncthreads();
        hist[t] = h;
        __syncthreads();
        if (warp == 0) enc_counts(S, hist, S.dem, hc, ps);
        __syncthreads();
        if (t < V) S.pos[t] += S.dem[t] * max(1u, ch_flat_d(S.ch[t]));
        __syncthreads();
    }
    // ---- parts ----
    uint32_t P = P0, len = whole && !(big && !chunk_hist) ? P1 - P0 : part;
    while (P < P1) {
        const uint32_t C = min(len, P1 - P);
        // the part's histogram: the planning pass's chunk counts, or counted here
        hist[t] = 0;
        __syncthreads();
        const bool given = whole && chunk_hist && C == P1 - P0;
        if (given) {
            uint32_t h = 0;
            for (uint32_t c = 0; c < nw; c++) h += __ldg(chunk_hist + ((size_t)b * kEncChunks + c) * 256 + t);
            hist[t] = h;
        } else {
            enc_count(src, P, P + C, hist);
        }
        __syncthreads();
        const uint32_t hcount = hist[t];
        if (warp == 0) {
            // the counts must total the part, with no symbol the code lacks
            uint32_t tot = 0, nocode = 0;
            for (int s = lane; s < 256; s += 32) {
                tot += hist[s];
                if (hist[s] && !((S.pmask[s >> 5] >> (s & 31)) & 1u)) nocode = 1;
            }
            tot = __reduce_add_sync(0xffffffffu, tot);
            if (__any_sync(0xffffffffu, nocode) || tot != C) { if (lane == 0) S.bad = 1; }
            else enc_counts(S, hist, S.dem, hc, ps);
        }
        __syncthreads();
        if (S.bad) break;
        // no node's bits of this part may run past its body (counts that do
        // not describe the input could otherwise carry a cursor beyond it)
        if (__syncthreads_or(t < V && (uint64_t)S.pos[t] + (uint64_t)S.dem[t] * max(1u, ch_flat_d(S.ch[t])) > S.end[t])) {
            if (t == 0) S.bad = 1;
            break;
        }
        if (!lvl_layout(S)) {
            // a shorter part (32 symbols always fit: a level then holds at
            // most 32 symbols in 160 groups)
            if (C <= 32u) {
                if (t == 0) S.bad = 1;
                break;
            }
            len = max(32u, (len > part ? part : len / 2) & ~31u);
            continue;
        }
        enc_part(S, src + P, C, src_end, rec32);
        if (t < V) S.pos[t] += S.dem[t] * max(1u, ch_flat_d(S.ch[t]));
        __syncthreads();
        if (S.bad) break;
        P += C;
        acc += hcount;
        if (len < part) len = min(part, 2 * len);
    }
    __syncthreads();
    if (!whole && !S.bad) {
        // the chunk's given counts must be the ones counted; an item inside
        // the block ends where the next one starts
        const bool last = share + 1 == shares;
        if (__syncthreads_or(last && acc != __ldg(chunk_hist + ((size_t)b * kEncChunks + cA) * 256 + t))) {
            if (t == 0) S.bad = 1;
        }
        __syncthreads();
    }
    // every node's cursor ends exactly at the end of its body (where the
    // item is the block's last)
    const bool ends = whole || (cA + 1 == nw && share + 1 == shares);
    const bool bad = __syncthreads_or(S.bad || (ends && t < V && S.pos[t] != S.end[t]));
    if (t == 0) {
        if (whole) {
            status[b] = bad ? PIVCO_ERR_INVALID_ARG : PIVCO_OK;
            rec_bytes[b] = bad ? 0 : rec_bound;
        } else if (bad) {
            atomicExch(&status[b], PIVCO_ERR_INVALID_ARG);
            rec_bytes[b] = 0;
        }
    }
    __syncthreads();
}

// The big blocks of a chunked encode (BlockLayout::big): checked, their bodies
// zeroed and their status set OK, and listed; then every chunk of theirs, or
// every share of one, is an item of the chunk kernel's work list.  gridDim.y
// CTAs zero a block.
__global__ void __launch_bounds__(kEncThreads) encode_reset_kernel(const uint64_t *__restrict__ blk_off,
                                                                   BlockLayout *__restrict__ layout,
                                                                   uint8_t *__restrict__ out,
                                                                   const uint64_t *__restrict__ out_off,
                                                                   uint64_t *__restrict__ rec_bytes,
                                                                   int32_t *__restrict__ status) {
    const int b = blockIdx.x, t = threadIdx.x;
    const BlockLayout &L = *layout_of(layout, b);
    if (!L.big || L.kind != 2) return;
    const uint64_t n = blk_off[b + 1] - blk_off[b];
    uint8_t *rec = out + out_off[b];
    const uint64_t cap = out_off[b + 1] - out_off[b];
    int st = PIVCO_OK;
    if (L.status != 0) st = L.status;
    else if (L.n != n || (reinterpret_cast<uintptr_t>(rec) & 15)) st = PIVCO_ERR_INVALID_ARG;
    else if (cap < L.rec_bound) st = PIVCO_ERR_CAPACITY;
    if (st != PIVCO_OK) {
        if (t == 0 && blockIdx.y == 0) { status[b] = st; rec_bytes[b] = 0; }
        return;
    }
    // the body and the record's tail, zeroed (the chunks OR their bits in)
    const uint32_t b0 = L.body0, b1 = L.rec_bound;
    const uint32_t h0 = min(b1, (b0 + 15u) & ~15u);
    const uint32_t tt = blockIdx.y * kEncThreads + t, nt = gridDim.y * kEncThreads;
    for (uint32_t i = b0 + tt; i < h0; i += nt) rec[i] = 0;
    for (uint32_t i = h0 + 16 * tt; i < b1; i += 16 * nt)
        *reinterpret_cast<uint4 *>(rec + i) = make_uint4(0u, 0u, 0u, 0u);
    if (tt == 0) {
        status[b] = PIVCO_OK;
        rec_bytes[b] = L.rec_bound;
        const uint32_t i = atomicAdd(&layout->list_len, 1u);
        layout_of(layout, (int)i)->list_entry = (uint32_t)b;
    }
}

// Lists of at most this many blocks are worked off largest first: the last
// chunks to be taken are the small ones, and the CTAs end together.  (1024
// blocks of 4 KiB to 1 MiB: 1090 us in list order, 890 by size; 509 text-like
// blocks 436 and 386.  With many more blocks than CTAs the order matters less
// and finding each entry's place, quadratic in the list, costs more.)
constexpr uint32_t kEncSortMax = 2048;

// Entry i of the list goes to its place by size (whole CTA); counted in
// list_placed, whose release the chunk kernel acquires.
__device__ inline void enc_list_place(uint32_t i, uint32_t len, const uint64_t *__restrict__ blk_off,
                                      BlockLayout *layout) {
    auto size_of = [&](uint32_t j) {
        const uint32_t b = layout_of(layout, (int)j)->list_entry;
        return blk_off[b + 1] - blk_off[b];
    };
    const uint64_t n = size_of(i);
    int place = 0;
    for (uint32_t j0 = 0; j0 < len; j0 += kEncThreads) {
        const uint32_t j = j0 + threadIdx.x;
        bool before = false;
        if (j < len) {
            const uint64_t m = size_of(j);
            before = m > n || (m == n && j < i);
        }
        place += __syncthreads_count(before);
    }
    if (threadIdx.x == 0) {
        __stcg(&layout_of(layout, place)->list_sorted, layout_of(layout, (int)i)->list_entry);
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&layout->list_placed) : "memory");
    }
    __syncthreads();
}

// One CTA per block (a big block of a chunked encode is left to the chunk
// kernel).
__global__ void __launch_bounds__(kEncThreads, kEncCtasPerSm) encode_kernel(const uint8_t *__restrict__ in,
                                                                            const uint64_t *__restrict__ blk_off,
                                                                            BlockLayout *layout,
                                                                            const uint32_t *__restrict__ chunk_hist,
                                                                            uint8_t *__restrict__ out,
                                                                            const uint64_t *__restrict__ out_off,
                                                                            uint64_t *__restrict__ rec_bytes,
                                                                            int32_t *__restrict__ status) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    EncSmem &S = *reinterpret_cast<EncSmem *>(smem_raw);
    if (chunk_hist) {
        const uint32_t len = layout->list_len;
        if (blockIdx.x < len && len <= kEncSortMax) enc_list_place(blockIdx.x, len, blk_off, layout);
        // (the chunk kernel may start from here on)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        if (layout_of(layout, (int)blockIdx.x)->big) return;
    }
    encode_item<true>((int)blockIdx.x, 0, 0, 1, in, blk_off, layout, chunk_hist, out, out_off, rec_bytes, status, S);
}

// The work list of big blocks' chunks, (block, chunk) by (block, chunk), or
// by shares of a chunk when the chunks alone would leave CTAs without work (a
// share counts the chunk's symbols before it again, so only then): persistent
// CTAs take tickets until the list is done.
__global__ void __launch_bounds__(kEncThreads, kEncCtasPerSm) encode_chunks_kernel(const uint8_t *__restrict__ in,
                                                                              const uint64_t *__restrict__ blk_off,
                                                                              BlockLayout *__restrict__ layout,
                                                                              const uint32_t *__restrict__ chunk_hist,
                                                                              uint8_t *__restrict__ out,
                                                                              const uint64_t *__restrict__ out_off,
                                                                              uint64_t *__restrict__ rec_bytes,
                                                                              int32_t *__restrict__ status, bool early,
                                                                              uint64_t limit_ns) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    EncSmem &S = *reinterpret_cast<EncSmem *>(smem_raw);
    __shared__ uint32_t s_tk;
    // Of what encode_kernel writes, only the list's order is read here.  Started early, this kernel runs once all
    // of its CTAs are past the trigger, which they reach after placing their entries; the trigger does not order
    // those writes, their count does.  (The list itself and all else was there before encode_kernel started.)
    const uint32_t len = __ldcg(&layout->list_len);
    if (early && len && len <= kEncSortMax) {
        if (threadIdx.x == 0) {
            const uint64_t t0 = globaltimer_ns();
            uint32_t v;
            for (;;) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&layout->list_placed) : "memory");
                if (v >= len || globaltimer_ns() - t0 > limit_ns) break;
                __nanosleep(64);
            }
            s_tk = v;
        }
        __syncthreads();
        if (s_tk < len) {   // the wait ran out: the list's blocks are given up
            for (uint32_t i = threadIdx.x; i < len; i += kEncThreads) {
                const uint32_t b = __ldcg(&layout_of(layout, (int)i)->list_entry);
                atomicExch(&status[b], PIVCO_ERR_TIMEOUT);
                rec_bytes[b] = 0;
            }
            if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
            return;
        }
    }
    const uint32_t chunks = len * kEncChunks;
    const uint32_t shares = min(kEncShares, max(1u, gridDim.x / max(1u, chunks))), items = chunks * shares;
    // an item each: by the CTA's number, which the launch deals out over the SMs (tickets taken in the order
    // of arrival put four of the 64 shares of one block on some SMs and none on others: 85 us, 52 spread).
    // More items: by ticket, the largest first to whoever comes first.
    const bool each = items <= gridDim.x;
    uint32_t tk = blockIdx.x;
    while (chunks) {
        if (!each) {
            __syncthreads();
            if (threadIdx.x == 0) s_tk = atomicAdd(&layout->list_ticket, 1u);
            __syncthreads();
            tk = s_tk;
        }
        if (tk >= items) break;
        const BlockLayout *E = layout_of(layout, (int)(tk / (kEncChunks * shares)));
        const int bb = (int)__ldcg(len <= kEncSortMax ? &E->list_sorted : &E->list_entry);
        const uint32_t c = tk / shares % kEncChunks;
        if (c < enc_nchunks(blk_off[bb + 1] - blk_off[bb]))
            encode_item<false>(bb, c, tk % shares, shares, in, blk_off, layout, chunk_hist, out, out_off, rec_bytes,
                               status, S);
        if (each) break;
    }
    // what follows in the stream follows encode_kernel too (one CTA waits, the others leave their slots)
    if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

cudaError_t launch_encode(const uint8_t *in, const uint64_t *blk_off, int nblk, BlockLayout *layout,
                          const uint32_t *chunk_hist, uint8_t *out, const uint64_t *out_off, uint64_t *rec_bytes,
                          int32_t *status, cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    const int smem = (int)sizeof(EncSmem);
    cudaError_t e = cudaFuncSetAttribute(encode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // the work list of big blocks: emptied, then filled by the reset pass
    e = cudaMemsetAsync(&layout->list_len, 0, 3 * sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    if (chunk_hist) {
        // (several CTAs per block when the blocks alone do not fill the chip: one block of 1 MiB 17 us by one CTA,
        // 4 by 16; 1024 mixed blocks 31 us by one each, 24 by two)
        const int per = max(1, min(16, div_up(8 * sms, nblk)));
        encode_reset_kernel<<<dim3(nblk, per), kEncThreads, 0, st>>>(blk_off, layout, out, out_off, rec_bytes, status);
        count_launches(1);
    }
    encode_kernel<<<nblk, kEncThreads, smem, st>>>(in, blk_off, layout, chunk_hist, out, out_off, rec_bytes, status);
    count_launches(1);
    if (chunk_hist) {
        const int smem_big = (int)sizeof(EncSmem);
        e = cudaFuncSetAttribute(encode_chunks_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_big);
        if (e != cudaSuccess) return e;
        // started while encode_kernel's last blocks run: its CTAs take the slots that fall free (509 text-like
        // blocks both ways 807 -> 760 us, 1024 mixed blocks 1297 -> 1205); with a block per SM at most there
        // is nothing to overlap
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(sms * kEncCtasPerSm);
        cfg.blockDim = dim3(kEncThreads);
        cfg.dynamicSmemBytes = (size_t)smem_big;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        const bool early = nblk > sms;
        cfg.numAttrs = early ? 1 : 0;
        e = cudaLaunchKernelEx(&cfg, encode_chunks_kernel, in, blk_off, layout, chunk_hist, out, out_off, rec_bytes, status,
                               early, wait_limit_ns());
        if (e != cudaSuccess) return e;
        count_launches(1);
    }
    return cudaGetLastError();
}

}  // namespace pv

namespace pv {
cudaError_t prepare_encode_kernels() {
    cudaError_t e = cudaFuncSetAttribute(encode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(EncSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(encode_chunks_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(EncSmem));
    return e;
}
}  // namespace pv
