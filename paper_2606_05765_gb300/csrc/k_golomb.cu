// PivCo-Golomb (App. G): pivoted coding applied to Golomb coding with a list
// of bitmaps in place of a tree.  The Golomb parameter is 1 (the unary
// code): value v is v continue bits then one stop bit (1); bitmap j holds,
// in sequence order, the j-th code bit of every value v >= j (1: v == j,
// 0: v > j).  The record layout is in include/pivco.h.
//
// One CTA of eight warps codes a block.  A warp has an eighth of the sequence
// and its part of every level, the values >= j of that eighth, to itself: where
// its part of bitmap j lies is known before the first level, so the levels need
// no barrier.
//   plan    the values' histogram gives m (largest value + 1) and n_j (values
//           >= j, a suffix sum), hence the exact record size.
//   encode  a histogram per warp: the values >= j of the warps before it are
//           the bit its part of bitmap j starts at.  Top-down, 32 values at a
//           time: the stop bits are one ballot (the bitmap word), the
//           continuing values close up in place, towards the start of the
//           warp's list.  32 words are then shifted to the bit the part starts
//           at and written together, ORed where a word is shared.
//   decode  every bitmap's ones are checked against the counts; then each warp
//           follows its start through the levels (the next level's start is
//           this one's less the ones before it), and merges bottom-up (App. G's
//           merge_vec_cst_plus1 with cst 0xFF): out_j[i] = B_j[i] ? 0x00 :
//           out_{j+1}[rank0(B_j, i)] + 1, from the list's end to its start and
//           in place (an index never lies before its child's).
// What bounds it: instruction issue, about a dozen per 32 values and level (the
// last 32 values of a warp stay in its lanes).
// With the whole CTA on a level, two barriers a level and two level buffers
// (three CTAs per SM), 2048 blocks of 9 to 32 Ki values of average 2 took 205 +
// 359 + 217 us (plan, encode, decode); now 35 + 102 + 97.
#include <type_traits>

#include "pivco_dev.cuh"

namespace pv {

constexpr int kGThreads = 256;
constexpr int kGWarps = kGThreads / 32;
constexpr uint32_t kGMaxBlock = PIVCO_GOLOMB_MAX_BLOCK;   // values per block
constexpr uint32_t kGKind = 4;
static_assert(kGMaxBlock % (32 * kGWarps) == 0, "a warp's part is whole groups of 32");

struct __align__(16) GolombSmem {
    uint8_t buf[kGMaxBlock + 16];      // warp w's list starts at its first value's place
    union {
        uint32_t cnt[kGWarps][256];    // encode: the warp's counts, then the values >= j of the warps before it
        uint32_t cur[kGWarps][256];    // decode: the values >= j of the warps before it
    };
    uint32_t nj[257];                  // values >= j
    uint32_t start[256];               // byte offset of bitmap j in the record
    uint32_t wsum[kGWarps];
};

// values per warp (whole groups of 32)
__device__ inline uint32_t g_per(uint32_t n) { return (n + 32u * kGWarps - 1) / (32u * kGWarps) * 32u; }

// The warp's len values from src counted into cnt (zeroed), and stored at dst
// (16-byte aligned) where kStore: words of src, each from the one or two
// aligned words that hold its bytes.
template <bool kStore>
__device__ inline void g_load(const uint8_t *__restrict__ src, uint32_t len, uint8_t *dst, uint32_t *cnt) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t off = (uint32_t)(reinterpret_cast<uintptr_t>(src) & 3), sh = 8 * off;
    const uint32_t *w = reinterpret_cast<const uint32_t *>(src - off);
    const uint32_t words = (off + len + 3) / 4;   // aligned words that hold a value
#pragma unroll 4
    for (uint32_t i = lane; 4 * i < len; i += 32) {
        const uint32_t a = __ldg(w + i), b = sh && i + 1 < words ? __ldg(w + i + 1) : 0u;
        const uint32_t x = __funnelshift_r(a, b, sh);
        if (kStore) reinterpret_cast<uint32_t *>(dst)[i] = x;
        const uint32_t k = len - 4 * i;
        atomicAdd(&cnt[x & 0xFF], 1u);
        if (k > 1) atomicAdd(&cnt[(x >> 8) & 0xFF], 1u);
        if (k > 2) atomicAdd(&cnt[(x >> 16) & 0xFF], 1u);
        if (k > 3) atomicAdd(&cnt[x >> 24], 1u);
    }
}

// Exclusive sum of x over the CTA's threads; total: over all of them.
__device__ inline uint32_t g_scan(uint32_t x, uint32_t *wsum, uint32_t &total) {
    const int t = threadIdx.x, lane = t & 31;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    __syncthreads();
    if (lane == 31) wsum[t >> 5] = inc;
    __syncthreads();
    uint32_t before = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < kGWarps; w++) {
        if (w < (t >> 5)) before += wsum[w];
        total += wsum[w];
    }
    return before + inc - x;
}

// The record size and m from thread t's n_t (0 past the largest value);
// at: where bitmap t starts.
__device__ inline uint32_t g_layout(uint32_t nt, uint32_t *wsum, uint32_t &m, uint32_t &at) {
    m = (uint32_t)__syncthreads_count(nt != 0);   // (n_j never grows with j)
    uint32_t total;
    at = 16 + 4 * m + g_scan((nt + 7) / 8, wsum, total);
    return (16 + 4 * m + total + 15u) & ~15u;
}

struct GolombPlanSmem {
    uint32_t cnt[kGWarps][256];
    uint32_t wsum[kGWarps];
};

__global__ void __launch_bounds__(kGThreads) golomb_plan_kernel(const uint8_t *__restrict__ in,
                                                                const uint64_t *__restrict__ blk_off,
                                                                uint64_t *__restrict__ rec_size,
                                                                int32_t *__restrict__ status) {
    __shared__ GolombPlanSmem S;
    const int b = blockIdx.x, t = threadIdx.x, warp = t >> 5;
    const uint64_t n64 = blk_off[b + 1] - blk_off[b];
    if (n64 > kGMaxBlock) {
        if (t == 0) { rec_size[b] = 16; status[b] = PIVCO_ERR_INVALID_ARG; }
        return;
    }
    const uint32_t n = (uint32_t)n64, per = g_per(n), w0 = min(n, per * warp), w1 = min(n, w0 + per);
#pragma unroll
    for (int w = 0; w < kGWarps; w++) S.cnt[w][t] = 0;
    __syncthreads();
    g_load<false>(in + blk_off[b] + w0, w1 - w0, nullptr, S.cnt[warp]);
    __syncthreads();
    uint32_t c = 0;
#pragma unroll
    for (int w = 0; w < kGWarps; w++) c += S.cnt[w][t];
    uint32_t total, m, at;
    const uint32_t nt = n - g_scan(c, S.wsum, total);   // values >= t
    const uint32_t size = g_layout(nt, S.wsum, m, at);
    if (t == 0) {
        rec_size[b] = size;
        status[b] = PIVCO_OK;
    }
}

// 32 bits from bit a of w, of which the words below lim hold something
__device__ inline uint32_t g_bits(const uint32_t *__restrict__ w, uint32_t a, uint32_t lim) {
    const uint32_t i = a >> 5, sh = a & 31u;
    return __funnelshift_r(__ldg(w + i), sh && i + 1 < lim ? __ldg(w + i + 1) : 0u, sh);
}

__global__ void __launch_bounds__(kGThreads) golomb_encode_kernel(const uint8_t *__restrict__ in,
                                                                  const uint64_t *__restrict__ blk_off,
                                                                  uint8_t *__restrict__ out,
                                                                  const uint64_t *__restrict__ out_off,
                                                                  uint64_t *__restrict__ rec_bytes,
                                                                  int32_t *__restrict__ status) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    GolombSmem &S = *reinterpret_cast<GolombSmem *>(smem_raw);
    const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint64_t n64 = blk_off[b + 1] - blk_off[b];
    uint8_t *rec = out + out_off[b];
    const uint64_t cap = out_off[b + 1] - out_off[b];
    if (n64 > kGMaxBlock) {
        if (t == 0) { rec_bytes[b] = 0; status[b] = PIVCO_ERR_INVALID_ARG; }
        return;
    }
    const uint32_t n = (uint32_t)n64, per = g_per(n), w0 = min(n, per * warp), w1 = min(n, w0 + per);
#pragma unroll
    for (int w = 0; w < kGWarps; w++) S.cnt[w][t] = 0;
    __syncthreads();
    uint8_t *list = S.buf + w0;
    g_load<true>(in + blk_off[b] + w0, w1 - w0, list, S.cnt[warp]);
    __syncwarp();
    {
        // the warp's values >= j: lane l has values 8 l .. 8 l + 7
        uint32_t *c = S.cnt[warp] + 8 * lane;
        uint4 x = reinterpret_cast<const uint4 *>(c)[0], y = reinterpret_cast<const uint4 *>(c)[1];
        y.z += y.w, y.y += y.z, y.x += y.y, x.w += y.x, x.z += x.w, x.y += x.z, x.x += x.y;
        uint32_t inc = x.x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_down_sync(0xffffffffu, inc, o);
            if (lane + o < 32) inc += v;
        }
        const uint32_t above = inc - x.x;
        x.x += above, x.y += above, x.z += above, x.w += above, y.x += above, y.y += above, y.z += above, y.w += above;
        reinterpret_cast<uint4 *>(c)[0] = x;
        reinterpret_cast<uint4 *>(c)[1] = y;
    }
    __syncthreads();
    uint32_t nt = 0;
#pragma unroll
    for (int w = 0; w < kGWarps; w++) {
        const uint32_t x = S.cnt[w][t];
        S.cnt[w][t] = nt;
        nt += x;
    }
    uint32_t m, at;
    const uint32_t size = g_layout(nt, S.wsum, m, at);
    if (cap < size) {
        if (t == 0) { rec_bytes[b] = 0; status[b] = PIVCO_ERR_CAPACITY; }
        return;
    }
    S.start[t] = at;
    // the record zeroed (shared words are ORed in, pad bits stay 0), then header and counts
    {
        const uint32_t head = (uint32_t)(-reinterpret_cast<intptr_t>(rec) & 3), words = (size - head) / 4;
        if (t < (int)head) rec[t] = 0;
        if (t < (int)(size - head - 4 * words)) rec[head + 4 * words + t] = 0;
        uint32_t *z = reinterpret_cast<uint32_t *>(rec + head);
        for (uint32_t i = t; i < words; i += kGThreads) z[i] = 0;
    }
    __syncthreads();
    if (t < 16) {
        uint8_t v = 0;
        if (t < 4) v = (uint8_t)(size >> (8 * t));
        else if (t < 8) v = (uint8_t)(n >> (8 * (t - 4)));
        else if (t == 8) v = (uint8_t)m;
        else if (t == 9) v = (uint8_t)(m >> 8);
        else if (t == 10) v = (uint8_t)kGKind;
        else if (t >= 12) v = (uint8_t)"PVG1"[t - 12];
        rec[t] = v;
    }
    if (t < (int)m) st_le32(rec + 16 + 4 * t, nt);
    // ---- the levels, by the warp ----
    // (an aligned word at a record's edge may hold bytes of its neighbours: it
    // is only ever ORed, with zeros there)
    const uint32_t ro = (uint32_t)(reinterpret_cast<uintptr_t>(rec) & 3);
    uint32_t *ow = reinterpret_cast<uint32_t *>(rec - ro);
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t len = w1 - w0, j = 0;
    __syncwarp();
    for (; len > 32; j++) {
        const uint32_t a0 = 8 * (ro + S.start[j]) + S.cnt[warp][j], sh = a0 & 31u;
        uint32_t next = 0;
        for (uint32_t base = 0; base < len; base += 1024) {
            const uint32_t nb = min(1024u, len - base);
            uint32_t mine = 0;   // lane g: the bits of group g
            // four groups from group g: all whole, or cut at nb
            auto groups = [&](uint32_t g, auto whole_t) {
                uint32_t v[4];
                const uint8_t *p = list + base + 32 * g + lane;
#pragma unroll
                for (int q = 0; q < 4; q++) v[q] = p[32 * q];   // (past the end: not used, within the buffer)
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    uint32_t act = 0xFFFFFFFFu;
                    if (!decltype(whole_t)::value) {
                        const int left = (int)nb - 32 * (int)(g + q);
                        if (left < 32) act = left > 0 ? (1u << left) - 1u : 0u;
                    }
                    const uint32_t stop = __ballot_sync(0xffffffffu, v[q] == j) & act, go = act & ~stop;
                    if ((go >> lane) & 1u) list[next + __popc(go & lt)] = (uint8_t)v[q];
                    next += __popc(go);
                    if (lane == (int)(g + q)) mine = stop;
                }
                __syncwarp();
            };
            uint32_t g = 0;
            for (; 32 * g + 128 <= nb; g += 4) groups(g, std::true_type{});
            if (32 * g < nb) groups(g, std::false_type{});
            // word l of the window: bits 32 l - sh .. 32 l - sh + 31
            const uint32_t lo = __shfl_up_sync(0xffffffffu, mine, 1);
            const uint32_t word = __funnelshift_l(lane ? lo : 0u, mine, sh);
            uint32_t *o = ow + ((a0 + base) >> 5);
            const uint32_t end = sh + nb;
            if (32u * lane < end) {
                if ((lane || !sh) && 32u * (lane + 1) <= end) o[lane] = word;
                else if (word) atomicOr(o + lane, word);
            }
            if (lane == 31 && end > 1024) {
                const uint32_t last = mine >> (32 - sh);
                if (last) atomicOr(o + 32, last);
            }
        }
        len = next;
    }
    // the last 32 values stay in the lanes: a level's bits are gathered from those that have got that far
    const uint32_t v = lane < (int)len ? list[lane] : 0u;
    uint32_t alive = (1ull << len) - 1u;
    for (; alive; j++) {
        const bool stops = ((alive >> lane) & 1u) && v == j;
        const uint32_t bits = __reduce_or_sync(0xffffffffu, stops ? 1u << __popc(alive & lt) : 0u);
        alive &= ~__ballot_sync(0xffffffffu, stops);
        if (bits) {
            const uint32_t a0 = 8 * (ro + S.start[j]) + S.cnt[warp][j], sh = a0 & 31u;
            const uint32_t word = lane ? __funnelshift_l(bits, 0u, sh) : bits << sh;
            if (lane < 2 && word) atomicOr(ow + (a0 >> 5) + lane, word);
        }
    }
    if (t == 0) { rec_bytes[b] = size; status[b] = PIVCO_OK; }
}

// ones among bits a .. a + len - 1 of w (warp)
__device__ inline uint32_t g_ones(const uint32_t *__restrict__ w, uint32_t a, uint32_t len) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t c = 0;
    if (len) {
        const uint32_t i0 = a >> 5, i1 = (a + len - 1) >> 5;
#pragma unroll 8
        for (uint32_t i = i0 + lane; i <= i1; i += 32) {
            uint32_t x = __ldg(w + i);
            if (i == i0) x &= 0xFFFFFFFFu << (a & 31u);
            if (i == i1) x &= 0xFFFFFFFFu >> (31u - ((a + len - 1) & 31u));
            c += __popc(x);
        }
    }
    return __reduce_add_sync(0xffffffffu, c);
}

__global__ void __launch_bounds__(kGThreads) golomb_decode_kernel(const uint8_t *__restrict__ comp,
                                                                  const uint64_t *__restrict__ comp_off,
                                                                  uint8_t *__restrict__ out,
                                                                  const uint64_t *__restrict__ out_off,
                                                                  int32_t *__restrict__ status) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    GolombSmem &S = *reinterpret_cast<GolombSmem *>(smem_raw);
    const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint8_t *rec = comp + comp_off[b];
    const uint64_t avail = comp_off[b + 1] - comp_off[b];
    const uint64_t ocap = out_off[b + 1] - out_off[b];
    uint8_t *dst = out + out_off[b];
    // header checks (every thread the same)
    bool bad = avail < 16;
    uint32_t size = 0, n = 0, m = 0;
    if (!bad) {
        size = ld_le32(rec);
        n = ld_le32(rec + 4);
        m = (uint32_t)rec[8] | ((uint32_t)rec[9] << 8);
        bad = rec[12] != 'P' || rec[13] != 'V' || rec[14] != 'G' || rec[15] != '1' || rec[10] != kGKind ||
              rec[11] != 0 || (size & 15) || size > avail || size < 16 || m > 256 || (n == 0) != (m == 0) ||
              16ull + 4ull * m > size || n > kGMaxBlock;
    }
    // thread j's count
    uint32_t nt = 0;
    bool badn = false;
    if (!bad && t < (int)m) {
        nt = ld_le32(rec + 16 + 4 * t);
        badn = nt == 0 || nt > (t ? ld_le32(rec + 16 + 4 * (t - 1)) : n) || (t == 0 && nt != n) || nt > kGMaxBlock;
        if (badn) nt = 0;
    }
    uint32_t total;
    const uint32_t at = 16 + 4 * m + g_scan((nt + 7) / 8, S.wsum, total);
    S.nj[t] = nt;
    S.start[t] = at;
    if (t == 0) S.nj[256] = 0;
    badn = badn || bad || ((16 + 4 * m + total + 15u) & ~15u) != size;
    if (__syncthreads_or(badn)) {
        if (t == 0) status[b] = PIVCO_ERR_CORRUPT;
        return;
    }
    if (n != ocap) {
        if (t == 0) status[b] = PIVCO_ERR_CAPACITY;
        return;
    }
    const uint32_t ro = (uint32_t)(reinterpret_cast<uintptr_t>(rec) & 3);
    const uint32_t *w = reinterpret_cast<const uint32_t *>(rec - ro);
    // ---- every bitmap: its stops are the values that do not continue, its pad bits are zero ----
    for (uint32_t j = warp; j < m; j += kGWarps) {
        const uint32_t len = S.nj[j], a = 8 * (ro + S.start[j]);
        if (g_ones(w, a, (len + 7) & ~7u) != len - S.nj[j + 1]) bad = true;
        if ((len & 7) && (rec[S.start[j] + (len >> 3)] >> (len & 7))) bad = true;
    }
    if (__syncthreads_or(bad)) {
        if (t == 0) status[b] = PIVCO_ERR_CORRUPT;
        return;
    }
    // ---- where the warp's part of each level starts ----
    const uint32_t per = g_per(n), w0 = min(n, per * warp);
    {
        uint32_t c = w0;
        for (uint32_t j = 0; j < m; j++) {
            if (lane == 0) S.cur[warp][j] = c;
            if (c) c -= g_ones(w, 8 * (ro + S.start[j]), c);
        }
    }
    __syncthreads();
    // ---- merge bottom-up, the warp's list from its end to its start ----
    uint8_t *list = S.buf + w0;
    const uint32_t lim = (ro + size + 3) / 4;
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t clen = 0;
    int j = (int)m - 1;
    {
        // up to 32 values: in the lanes
        uint32_t v = 0, len = 0;
        for (; j >= 0; j--) {
            const uint32_t c0 = S.cur[warp][j], c1 = warp + 1 < kGWarps ? S.cur[warp + 1][j] : S.nj[j];
            len = c1 - c0;
            if (len > 32) break;
            clen = len;
            if (!len) continue;
            const uint32_t zm = ~g_bits(w, 8 * (ro + S.start[j]) + c0, lim) & (len < 32 ? (1u << len) - 1u : 0xFFFFFFFFu);
            const uint32_t c = __shfl_sync(0xffffffffu, v, __popc(zm & lt));
            v = (zm >> lane) & 1u ? c + 1u : 0u;
        }
        if (lane < (int)clen) list[lane] = (uint8_t)v;
        __syncwarp();
    }
    for (; j >= 0; j--) {
        const uint32_t c0 = S.cur[warp][j], c1 = warp + 1 < kGWarps ? S.cur[warp + 1][j] : S.nj[j], len = c1 - c0;
        if (!len) continue;
        const uint32_t a0 = 8 * (ro + S.start[j]) + c0;
        uint32_t z = clen;   // the children from here on are taken
        for (int base = (int)((len - 1) & ~1023u); base >= 0; base -= 1024) {
            const uint32_t nb = min(1024u, len - base);
            uint32_t mine = 0;   // lane g: the zeros of group g
            if (32u * lane < nb) {
                mine = ~g_bits(w, a0 + base + 32 * lane, lim);
                if (nb - 32u * lane < 32) mine &= (1u << (nb - 32u * lane)) - 1u;
            }
            for (int g = (int)((nb - 1) / 128) * 4; g >= 0; g -= 4) {
                uint32_t v[4];
#pragma unroll
                for (int q = 3; q >= 0; q--) {
                    const uint32_t zm = __shfl_sync(0xffffffffu, mine, g + q);
                    z -= __popc(zm);
                    v[q] = 0;
                    if ((zm >> lane) & 1u) v[q] = list[z + __popc(zm & lt)] + 1u;
                }
                __syncwarp();
                uint8_t *p = list + base + 32 * g + lane;
                const int left = (int)nb - 32 * g - lane;
#pragma unroll
                for (int q = 3; q >= 0; q--)
                    if (32 * q < left) p[32 * q] = (uint8_t)v[q];
                __syncwarp();
            }
        }
        clen = len;
    }
    __syncthreads();
    {
        const uint32_t head = min(n, (uint32_t)(-reinterpret_cast<intptr_t>(dst) & 3)), words = (n - head) / 4;
        if (t < (int)head) dst[t] = S.buf[t];
        if (t < (int)(n - head - 4 * words)) dst[head + 4 * words + t] = S.buf[head + 4 * words + t];
        const uint32_t *s = reinterpret_cast<const uint32_t *>(S.buf);
        uint32_t *d = reinterpret_cast<uint32_t *>(dst + head);
        for (uint32_t i = t; i < words; i += kGThreads) d[i] = __funnelshift_r(s[i], s[i + 1], 8 * head);
    }
    if (t == 0) status[b] = PIVCO_OK;
}

static cudaError_t g_attr(const void *fn) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GolombSmem));
}

cudaError_t launch_golomb_plan(const uint8_t *in, const uint64_t *blk_off, int nblk, uint64_t *rec_size,
                               int32_t *status, cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    golomb_plan_kernel<<<nblk, kGThreads, 0, st>>>(in, blk_off, rec_size, status);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_golomb_encode(const uint8_t *in, const uint64_t *blk_off, int nblk, uint8_t *out,
                                 const uint64_t *out_off, uint64_t *rec_bytes, int32_t *status, cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    cudaError_t e = g_attr((const void *)golomb_encode_kernel);
    if (e != cudaSuccess) return e;
    golomb_encode_kernel<<<nblk, kGThreads, sizeof(GolombSmem), st>>>(in, blk_off, out, out_off, rec_bytes, status);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_golomb_decode(const uint8_t *comp, const uint64_t *comp_off, int nblk, uint8_t *out,
                                 const uint64_t *out_off, int32_t *status, cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    cudaError_t e = g_attr((const void *)golomb_decode_kernel);
    if (e != cudaSuccess) return e;
    golomb_decode_kernel<<<nblk, kGThreads, sizeof(GolombSmem), st>>>(comp, comp_off, out, out_off, status);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t prepare_golomb_kernels() {
    cudaError_t e = g_attr((const void *)golomb_encode_kernel);
    if (e == cudaSuccess) e = g_attr((const void *)golomb_decode_kernel);
    return e;
}

}  // namespace pv
