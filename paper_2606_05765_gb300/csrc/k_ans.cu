// Selective ANS of node bitmaps (Sec. 5.2): the standalone bitmap coder /
// decoder and the in-record ANS pass of the encoder.
#include <type_traits>
#include "ans_dev.cuh"

namespace pv {
// ---------------------------------------------------------------------------
// Standalone bitmap ANS (one warp per bitmap; segments sequential).
// ---------------------------------------------------------------------------
constexpr int kAnsStageWords = 4096;      // words staged in shared memory (the rest of a segment's go to global memory)

// The words of a coded segment in decoder order at dst (one warp): word k is
// emission nw - 1 - k.  Emissions cap .. nw - 1 were written at dst in
// emission order (ans_encode_segment's ovf): reversed in place, they become
// words 0 .. nw - cap - 1; the staged emissions 0 .. cap - 1 are the rest.
__device__ inline void ans_place_words(const uint16_t *stage, uint32_t cap, uint32_t nw, uint8_t *dst) {
    const int lane = threadIdx.x & 31;
    if (nw > cap) {
        const uint32_t L = nw - cap;
        for (uint32_t i0 = 0; i0 < L / 2; i0 += 32) {
            const uint32_t i = i0 + lane, j = L - 1 - i;
            uint8_t a0 = 0, a1 = 0, b0 = 0, b1 = 0;
            if (i < L / 2) { a0 = dst[2 * i]; a1 = dst[2 * i + 1]; b0 = dst[2 * j]; b1 = dst[2 * j + 1]; }
            __syncwarp();
            if (i < L / 2) { dst[2 * i] = b0; dst[2 * i + 1] = b1; dst[2 * j] = a0; dst[2 * j + 1] = a1; }
            __syncwarp();
        }
    }
    const uint32_t ns = nw < cap ? nw : cap;
    for (uint32_t k = nw - ns + lane; k < nw; k += 32) {
        const uint16_t w = stage[cap - nw + k];
        dst[2 * k] = (uint8_t)w;
        dst[2 * k + 1] = (uint8_t)(w >> 8);
    }
}

__global__ void __launch_bounds__(32) ans_encode_kernel(const uint8_t *__restrict__ bm, const uint64_t *__restrict__ bm_off,
                                                        const uint8_t *__restrict__ table, uint8_t *__restrict__ bodies,
                                                        const uint64_t *__restrict__ body_off,
                                                        uint64_t *__restrict__ body_bytes, int32_t *__restrict__ status,
                                                        const __grid_constant__ AnsTables A) {
    extern __shared__ __align__(16) uint8_t sm[];
    AnsSm &T = *reinterpret_cast<AnsSm *>(sm);
    uint16_t *stage = reinterpret_cast<uint16_t *>(sm + ((sizeof(AnsSm) + 15) & ~15));
    const int i = blockIdx.x, lane = threadIdx.x;
    const uint32_t nbytes = (uint32_t)(bm_off[i + 1] - bm_off[i]);
    const uint8_t tb = table[i];
    const int tid = (tb & 0x7F) - 1;
    const uint64_t cap = body_off[i + 1] - body_off[i];
    if (tid < 0 || tid >= 50 || nbytes == 0) {
        if (lane == 0) { status[i] = PIVCO_ERR_INVALID_ARG; body_bytes[i] = 0; }
        return;
    }
    load_ans_table(T, A, tid, lane, 32, true);
    __syncwarp();
    const uint8_t xr = (tb & 0x80) ? 0xFF : 0;
    const uint8_t *src = bm + bm_off[i];
    uint8_t *dst = bodies + body_off[i];
    const uint32_t S = ans_seg_count(nbytes);
    uint64_t pos = 4ull * S;
    bool ok = pos <= cap;
    for (uint32_t s = 0; s < S && ok; s++) {
        const uint32_t sb = min(kAnsSeg, nbytes - s * kAnsSeg), W = ans_seg_lanes(sb);
        uint32_t x;
        const uint8_t *ss = src + (size_t)s * kAnsSeg;
        // words past the stage go where the segment's words will be (after its states)
        const uint64_t wo = pos + 4ull * W;
        const uint32_t room = wo < cap ? (uint32_t)min((cap - wo) / 2, (uint64_t)0xFFFFFFFFu) : 0u;
        const uint32_t nw = ans_encode_segment(ss, sb, T, xr, stage, kAnsStageWords, dst + wo, room, x);
        __syncwarp();
        if (pos + 4ull * W + 2ull * nw > cap) { ok = false; break; }
        if (lane == 0) st_le32(dst + 4 * s, nw);
        if (lane < (int)W) st_le32(dst + pos + 4 * lane, x);
        pos += 4ull * W;
        __syncwarp();
        ans_place_words(stage, kAnsStageWords, nw, dst + pos);
        pos += 2ull * nw;
        __syncwarp();
    }
    if (lane == 0) { status[i] = ok ? PIVCO_OK : PIVCO_ERR_CAPACITY; body_bytes[i] = ok ? pos : 0; }
}

// locate segment s of an ANS body: returns byte offset of its states, its word count
__global__ void __launch_bounds__(32) ans_decode_kernel(const uint8_t *__restrict__ bodies, const uint64_t *__restrict__ body_off,
                                                        const uint8_t *__restrict__ table, uint8_t *__restrict__ bm,
                                                        const uint64_t *__restrict__ bm_off, int32_t *__restrict__ status,
                                                        const __grid_constant__ AnsTables A) {
    __shared__ AnsSm T;
    __shared__ uint8_t wst[2 * kAnsWordWin];
    const int i = blockIdx.x, lane = threadIdx.x;
    const uint32_t nbytes = (uint32_t)(bm_off[i + 1] - bm_off[i]);
    const uint8_t tb = table[i];
    const int tid = (tb & 0x7F) - 1;
    const uint64_t blen = body_off[i + 1] - body_off[i];
    if (tid < 0 || tid >= 50 || nbytes == 0) {
        if (lane == 0) status[i] = PIVCO_ERR_INVALID_ARG;
        return;
    }
    load_ans_table(T, A, tid, lane, 32);
    __syncwarp();
    const uint8_t *body = bodies + body_off[i];
    const uint32_t S = ans_seg_count(nbytes);
    bool ok = true;
    uint64_t total = 4ull * S;
    for (uint32_t s = 0; s < S && ok; s++) {
        uint64_t sp; uint32_t nw;
        if (!ans_segment_at(body, blen, nbytes, s, sp, nw)) { ok = false; break; }
        const uint32_t sb = min(kAnsSeg, nbytes - s * kAnsSeg), W = ans_seg_lanes(sb);
        ok = ans_decode_segment(body + sp, body + sp + 4 * W, nw, sb, T, (tb & 0x80) ? 0xFF : 0,
                                bm + bm_off[i] + (size_t)s * kAnsSeg, wst);
        total += 4ull * W + 2ull * nw;
    }
    if (ok && total != blen) ok = false;
    if (lane == 0) status[i] = ok ? PIVCO_OK : PIVCO_ERR_CORRUPT;
}

cudaError_t launch_ans_encode(const uint8_t *bm, const uint64_t *bm_off, const uint8_t *table, int nbm, uint8_t *bodies,
                              const uint64_t *body_off, uint64_t *body_bytes, int32_t *status, cudaStream_t st) {
    if (nbm <= 0) return cudaSuccess;
    const int smem = (int)(((sizeof(AnsSm) + 15) & ~15) + 2 * kAnsStageWords);
    cudaError_t e = cudaFuncSetAttribute(ans_encode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    ans_encode_kernel<<<nbm, 32, smem, st>>>(bm, bm_off, table, bodies, body_off, body_bytes, status, host_ans_tables());
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_ans_decode(const uint8_t *bodies, const uint64_t *body_off, const uint8_t *table, int nbm, uint8_t *bm,
                              const uint64_t *bm_off, int32_t *status, cudaStream_t st) {
    if (nbm <= 0) return cudaSuccess;
    ans_decode_kernel<<<nbm, 32, 0, st>>>(bodies, body_off, table, bm, bm_off, status, host_ans_tables());
    count_launches(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// In-record ANS pass (encode side): every node written with marker 0xFF
// (selected, raw) is coded; bodies not smaller than the raw bitmap are dropped
// (the node stays raw, marker 0xFF).  Then the selected region is rewritten in
// breadth-first order; each final body starts no later than its raw copy and
// ends before the next raw copy, so the in-place rewrite never overwrites
// unread bytes.
//   units   one warp per unit (ans_dev.cuh: a whole segment, or the bitmaps'
//           last segments sharing 32 lanes): a segment of sb bytes is coded into
//           the sb bytes of the workspace that mirror its place in the record:
//           its word count and states at the start, its words at the end (they
//           are emitted backwards, so they come out in the decoder's order).
//           A segment that does not fit there is marked, with its word count.
//   place   one CTA per block: sizes, the choice per node, the rewrite.  The
//           marked segments of a node that is coded all the same, and last
//           segments too short for a mirror, are coded here, a warp each; a
//           block of many, or with no room for the mirror, by one warp, node
//           after node.
// What bounds it: the latency of a round's chain, 512 rounds a unit: the bytes
// and table entries of 8 rounds are loaded before the chain needs them.  One
// warp per block coded its nodes one after another: 236 us for 2048 bitmaps of
// 16 KiB (one unit each), now 85 + 30 us; 445 us for 1024 blocks of many nodes,
// now 57 + 31 us.  Where half of each block is noise, whole encode calls: 1 MiB
// 1909 us before, 2171 with every marked segment left to the one warp, 482 now;
// 64 blocks of 256 KiB 536, 609 and 328.
// ---------------------------------------------------------------------------
// One block by one warp (no room for its mirror, or too many marked segments).
__device__ __noinline__ void ans_encode_block_serial(int b, const BlockLayout *__restrict__ layout, uint8_t *__restrict__ out,
                                                     const uint64_t *__restrict__ out_off,
                                                     uint64_t *__restrict__ rec_bytes, uint8_t *__restrict__ ws,
                                                     uint64_t ws_bytes, const AnsTables &A) {
    extern __shared__ __align__(16) uint8_t sm[];
    AnsSm &T = *reinterpret_cast<AnsSm *>(sm);
    uint16_t *stage = reinterpret_cast<uint16_t *>(sm + ((sizeof(AnsSm) + 15) & ~15));
    __shared__ uint32_t s_body[256];     // ANS body bytes per node (0 = keep raw)
    const int lane = threadIdx.x & 31;
    const BlockLayout &L = *reinterpret_cast<const BlockLayout *>(reinterpret_cast<const uint8_t *>(layout) +
                                                                   (size_t)b * kLayoutBytes);
    uint8_t *rec = out + out_off[b];
    uint8_t *wslot = ws + out_off[b];
    const uint64_t wcap = (out_off[b] < ws_bytes) ? umin64(ws_bytes - out_off[b], out_off[b + 1] - out_off[b]) : 0;
    const int V = L.n_int;
    uint64_t wpos = 0;
    for (int v = 0; v < V; v++) {
        if (!L.sel[v]) continue;
        if (lane == 0) s_body[v] = 0;
        const uint8_t tb = L.sel[v];
        const int tid = (tb & 0x7F) - 1;
        const uint32_t raw = (L.nv[v] + 7) / 8;
        __syncwarp();
        load_ans_table(T, A, tid, lane, 32, true);
        __syncwarp();
        const uint8_t xr = (tb & 0x80) ? 0xFF : 0;
        const uint8_t *src = rec + L.body_off[v];
        const uint32_t S = ans_seg_count(raw);
        uint64_t pos = 4ull * S;
        bool ok = wpos + pos <= wcap && pos < raw;
        for (uint32_t s = 0; s < S && ok; s++) {
            const uint32_t sb = min(kAnsSeg, raw - s * kAnsSeg), W = ans_seg_lanes(sb);
            uint32_t x;
            const uint8_t *ss = src + (size_t)s * kAnsSeg;
            uint8_t *dst = wslot + wpos;
            // words past the stage go where the segment's words will be
            const uint64_t wo = wpos + pos + 4ull * W;
            const uint32_t room = wo < wcap ? (uint32_t)min((wcap - wo) / 2, (uint64_t)0xFFFFFFFFu) : 0u;
            const uint32_t nw = ans_encode_segment(ss, sb, T, xr, stage, kAnsStageWords, dst + pos + 4ull * W, room, x);
            __syncwarp();
            const uint64_t np = pos + 4ull * W + 2ull * nw;
            if (np >= raw || wpos + np > wcap) { ok = false; break; }
            if (lane == 0) st_le32(dst + 4 * s, nw);
            if (lane < (int)W) st_le32(dst + pos + 4 * lane, x);
            pos += 4ull * W;
            __syncwarp();
            ans_place_words(stage, kAnsStageWords, nw, dst + pos);
            pos += 2ull * nw;
            __syncwarp();
        }
        if (ok && lane == 0) s_body[v] = (uint32_t)pos;
        if (ok) wpos += pos;
        __syncwarp();
    }
    // rewrite the selected region in breadth-first order
    __threadfence_block();
    uint32_t q = 0xFFFFFFFFu;
    for (int v = 0; v < V; v++)
        if (L.sel[v]) { q = L.body_off[v]; break; }
    const uint32_t alen_off = (kNvOff + 5u * V + 3u) & ~3u;
    uint64_t wread = 0;
    int k = 0;
    for (int v = 0; v < V; v++) {
        if (!L.sel[v]) continue;
        const uint32_t raw = (L.nv[v] + 7) / 8;
        const uint32_t bl = s_body[v];
        uint32_t len;
        if (bl) {
            for (uint32_t i = lane; i < bl; i += 32) rec[q + i] = wslot[wread + i];
            wread += bl;
            len = bl;
            if (lane == 0) rec[kNvOff + 4 * V + v] = L.sel[v];
        } else {
            const uint8_t *src = rec + L.body_off[v];
            if (q != L.body_off[v])
                for (uint32_t base = 0; base < raw; base += 32) {
                    const uint32_t i = base + lane;
                    const uint8_t c = i < raw ? src[i] : 0;
                    __syncwarp();
                    if (i < raw) rec[q + i] = c;
                    __syncwarp();
                }
            len = raw;
        }
        if (lane == 0) st_le32(rec + alen_off + 4 * k, len);
        k++;
        q += len;
        __syncwarp();
    }
    const uint32_t total = (q + 15u) & ~15u;
    for (uint32_t i = q + lane; i < total; i += 32) rec[i] = 0;
    if (lane == 0) {
        st_le32(rec, total);
        rec_bytes[b] = total;
    }
}


constexpr uint32_t kAnsMirrorMin = 16;    // shorter segments have no room for their header: coded by the place kernel
constexpr uint32_t kAnsMarked = 0x80000000u;   // with the word count of a segment that does not fit its mirror
constexpr uint32_t kAnsMarks = 64;        // marked segments of a block the place kernel codes itself

struct AnsEncGroup {            // a segment of a unit
    uint32_t at, sb;            // its bytes in the record
    uint32_t lane0, mk;         // its first lane, the node's table and XOR flag
};
struct __align__(16) AnsEncSm {
    uint4 tab[32][9];           // per group and class: frequency, start, and ceil(2^48 / frequency) in two words
    AnsEncGroup grp[32];
    uint8_t of_lane[32];        // group of a lane (0xFF: none)
};

// x / q for x < 2^32 from m48 = ceil(2^48 / q) = mh 2^32 + ml (div_q's product
// without its low words)
__device__ inline uint32_t div_q2(uint32_t x, uint32_t ml, uint32_t mh) {
    return (uint32_t)(((uint64_t)x * mh + __umulhi(x, ml)) >> 16);
}

__global__ void __launch_bounds__(32) ans_encode_units_kernel(const BlockLayout *__restrict__ layout,
                                                                             const uint8_t *__restrict__ out,
                                                                             const uint64_t *__restrict__ out_off,
                                                                             uint8_t *__restrict__ ws, uint64_t ws_bytes,
                                                                             const int32_t *__restrict__ status,
                                                                             const __grid_constant__ AnsTables A) {
    __shared__ AnsEncSm M;
    __shared__ uint8_t s_rank[256];
    const int b = blockIdx.x, lane = threadIdx.x;
    const uint32_t lt = (1u << lane) - 1u, gt = ~((2u << lane) - 1u);
    const BlockLayout &L = *layout_of(layout, b);
    if (status[b] != PIVCO_OK || L.kind != 2 || L.n_sel == 0) return;
    if (out_off[b + 1] > ws_bytes) return;   // (the mirror does not fit: the block is coded serially)
    for (int i = lane; i < 256; i += 32) s_rank[i] = A.rank_in_class[i];
    const uint8_t *rec = out + out_off[b];
    uint8_t *mir = ws + out_off[b];
    const uint32_t V = L.n_int;
    // ---- the block's whole segments and its last segments by size ----
    uint32_t full = 0, cnt[6] = {0u, 0u, 0u, 0u, 0u, 0u};
    for (uint32_t v0 = 0; v0 < V; v0 += 32) {
        const uint32_t v = v0 + lane;
        const bool sel = v < V && L.sel[v];
        const uint32_t raw = sel ? (L.nv[v] + 7) / 8 : 0u, tl = ans_tail_lanes(raw);
        full += __reduce_add_sync(0xffffffffu, ans_full_segs(raw));
#pragma unroll
        for (int c = 0; c < 6; c++) cnt[c] += __popc(__ballot_sync(0xffffffffu, tl == (1u << c)));
    }
    uint32_t off0[6];   // first lane of each size, largest first
    off0[5] = 0;
#pragma unroll
    for (int c = 4; c >= 0; c--) off0[c] = off0[c + 1] + (cnt[c + 1] << (c + 1));
    const uint32_t units = ans_units(full, off0[0] + cnt[0]);
    for (uint32_t unit = blockIdx.y; unit < units; unit += gridDim.y) {
        const bool whole = unit < full;
        const uint32_t lanes0 = whole ? 0u : 32u * (unit - full);
        uint32_t off[6];
#pragma unroll
        for (int c = 0; c < 6; c++) off[c] = off0[c];
        __syncwarp();
        M.of_lane[lane] = 0xFF;
        __syncwarp();
        uint32_t ng = 0, fl = 0;
        for (uint32_t v0 = 0; v0 < V; v0 += 32) {
            const uint32_t v = v0 + lane;
            const bool sel = v < V && L.sel[v];
            if (!__any_sync(0xffffffffu, sel)) continue;
            const uint32_t raw = sel ? (L.nv[v] + 7) / 8 : 0u, tl = ans_tail_lanes(raw), fs = ans_full_segs(raw);
            uint32_t fi = fs;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, fi, o);
                if (lane >= o) fi += y;
            }
            const uint32_t f0 = fl + fi - fs;
            fl += __shfl_sync(0xffffffffu, fi, 31);
            uint32_t l0 = 0;
#pragma unroll
            for (int c = 0; c < 6; c++) {
                const uint32_t m = __ballot_sync(0xffffffffu, tl == (1u << c));
                if (tl == (1u << c)) l0 = off[c] + (__popc(m & lt) << c);
                off[c] += __popc(m) << c;
            }
            AnsEncGroup X{0u, 0u, 0u, 0u};
            bool mine;
            if (whole) {
                mine = unit >= f0 && unit < f0 + fs;
                X.at = mine ? L.body_off[v] + (unit - f0) * kAnsSeg : 0u;
                X.sb = kAnsSeg;
            } else {
                mine = tl && l0 >= lanes0 && l0 < lanes0 + 32;
                X.at = mine ? L.body_off[v] + fs * kAnsSeg : 0u;
                X.sb = raw - fs * kAnsSeg;
                X.lane0 = l0 - lanes0;
            }
            if (mine) X.mk = L.sel[v];
            const uint32_t mm = __ballot_sync(0xffffffffu, mine);
            if (mine) {
                const uint32_t gi = ng + __popc(mm & lt);
                M.grp[gi] = X;
                const uint32_t w = ans_seg_lanes(X.sb);
                for (uint32_t i = 0; i < w; i++) M.of_lane[X.lane0 + i] = (uint8_t)gi;
            }
            ng += __popc(mm);
        }
        __syncwarp();
        const uint32_t gi = M.of_lane[lane];
        const bool on = gi != 0xFF && M.grp[gi].sb >= kAnsMirrorMin;
        const uint32_t gm = __match_any_sync(0xffffffffu, gi);
        uint32_t sb = 0, nl = 1, li = 0, at = 0;
        uint8_t xr = 0;
        if (on) {
            const AnsEncGroup X = M.grp[gi];
            sb = X.sb;
            nl = ans_seg_lanes(sb);
            li = lane - X.lane0;
            at = X.at;
            xr = (X.mk & 0x80) ? 0xFF : 0;
            const uint32_t tid = (X.mk & 0x7F) - 1;
            for (uint32_t k = li; k < 9; k += nl) {
                const uint32_t q = A.q[tid][k];
                const uint64_t m48 = ((1ull << 48) + q - 1) / q;
                M.tab[gi][k] = make_uint4(q, A.start[tid][k], (uint32_t)m48, (uint32_t)(m48 >> 32));
            }
        }
        __syncwarp();
        const uint4 *tab = M.tab[on ? gi : 0];
        const uint8_t *__restrict__ src = rec + at + li;
        // the words end at an even address at or below the mirror's end
        uint8_t *lo = mir + at;
        uint16_t *we = reinterpret_cast<uint16_t *>((reinterpret_cast<uintptr_t>(lo) + sb) & ~(uintptr_t)1);
        const uint32_t bytes = (uint32_t)(reinterpret_cast<uint8_t *>(we) - lo);
        const uint32_t cap = on && bytes > 4 + 4 * nl ? (bytes - 4 - 4 * nl) / 2 : 0u;   // words it holds
        const uint32_t mine_r = li < sb ? (sb - li + nl - 1) / nl : 0u;
        const uint32_t rounds = __reduce_max_sync(0xffffffffu, mine_r);
        uint32_t x = kAnsL, nw = 0;
        // the lane's bytes of 8 rounds at a time, the next ones' while these are coded
        auto load8 = [&](int w, uint32_t (&p)[8]) {
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const uint32_t r = 8u * (uint32_t)w + i;
                p[i] = w >= 0 && r < mine_r ? (uint32_t)src[r * nl] : 0u;
            }
        };
        uint32_t cur[8], nxt[8];
        int w = (int)(rounds + 7) / 8 - 1;
        load8(w, cur);
        auto code = [&](auto whole_t) {
            constexpr bool kWhole = decltype(whole_t)::value;   // 32 lanes, active in every round
            for (; w >= 0; w--) {
                load8(w - 1, nxt);
                uint4 e[8];
                uint32_t c[8];
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    const uint32_t by = cur[i] ^ xr;
                    e[i] = tab[__popc(by)];
                    c[i] = e[i].y + s_rank[by] * e[i].x;
                }
#pragma unroll
                for (int i = 7; i >= 0; i--) {
                    const bool active = kWhole || 8u * (uint32_t)w + i < mine_r;
                    const bool emit = active && (x >> 17) >= e[i].x;
                    const uint32_t m = __ballot_sync(0xffffffffu, emit) & (kWhole ? 0xffffffffu : gm);
                    const uint32_t pos = nw + __popc(m & gt);
                    if (emit && pos < cap) we[-1 - (int)pos] = (uint16_t)x;
                    const uint32_t xs = emit ? x >> 16 : x;
                    const uint32_t xn = xs + div_q2(xs, e[i].z, e[i].w) * (kAnsM - e[i].x) + c[i];
                    x = active ? xn : x;
                    nw += __popc(m);
                }
#pragma unroll
                for (int i = 0; i < 8; i++) cur[i] = nxt[i];
            }
        };
        if (whole) code(std::true_type{});
        else code(std::false_type{});
        // word count and states at the mirror's start (any byte)
        if (on) {
            if (li == 0) st_le32(lo, nw <= cap ? nw : kAnsMarked | nw);
            if (nw <= cap) st_le32(lo + 4 + 4 * li, x);
        }
    }
}

constexpr int kAnsPlaceThreads = 128;
constexpr uint32_t kAnsPlaceWarps = kAnsPlaceThreads / 32;

// n bytes to dst by threads t of nt: whole words of dst, each from the one or
// two source words that hold its bytes
__device__ inline void copy_words(uint8_t *__restrict__ dst, const uint8_t *__restrict__ src, uint32_t n, uint32_t t, uint32_t nt) {
    const uint32_t head = min(n, (uint32_t)(-reinterpret_cast<intptr_t>(dst) & 3));
    const uint32_t nwrd = (n - head) / 4, rest = head + 4 * nwrd;
    if (t < head) dst[t] = src[t];
    if (t < n - rest) dst[rest + t] = src[rest + t];
    const uint8_t *s0 = src + head;
    const uint32_t sh = 8 * (uint32_t)(reinterpret_cast<uintptr_t>(s0) & 3);
    const uint32_t *s = reinterpret_cast<const uint32_t *>(reinterpret_cast<uintptr_t>(s0) & ~(uintptr_t)3);
    uint32_t *d = reinterpret_cast<uint32_t *>(dst + head);
#pragma unroll 8
    for (uint32_t i = t; i < nwrd; i += nt) d[i] = __funnelshift_r(s[i], sh ? s[i + 1] : 0u, sh);
}

__global__ void __launch_bounds__(kAnsPlaceThreads, 8) ans_encode_place_kernel(const BlockLayout *__restrict__ layout,
                                                                            uint8_t *__restrict__ out,
                                                                            const uint64_t *__restrict__ out_off,
                                                                            uint64_t *__restrict__ rec_bytes,
                                                                            uint8_t *__restrict__ ws, uint64_t ws_bytes,
                                                                            const int32_t *__restrict__ status,
                                                                            const __grid_constant__ AnsTables A) {
    __shared__ uint32_t s_len[256];      // coded bytes of a node (0: kept raw)
    __shared__ uint32_t s_node[256];     // the selected nodes, in order
    __shared__ uint32_t s_n, s_nw, s_x[32];
    __shared__ bool s_tail[256];         // the node's last segment, without a mirror, is coded here
    __shared__ uint32_t s_nmark, s_mark[kAnsMarks][3];   // marked segments of coded nodes: k, segment, words
    __shared__ AnsSm s_T[kAnsPlaceThreads / 32];
    extern __shared__ __align__(16) uint8_t sm[];
    uint16_t *stage = reinterpret_cast<uint16_t *>(sm + ((sizeof(AnsSm) + 15) & ~15));
    const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const BlockLayout &L = *layout_of(layout, b);
    if (status[b] != PIVCO_OK || L.kind != 2 || L.n_sel == 0) return;
    const uint32_t V = L.n_int;
    uint8_t *rec = out + out_off[b];
    const uint8_t *mir = ws + out_off[b];
    if (warp == 0) {
        uint32_t n = 0;
        for (uint32_t v0 = 0; v0 < V; v0 += 32) {
            const uint32_t v = v0 + lane;
            const bool sel = v < V && L.sel[v];
            const uint32_t m = __ballot_sync(0xffffffffu, sel);
            if (sel) s_node[n + __popc(m & ((1u << lane) - 1u))] = v;
            n += __popc(m);
        }
        if (lane == 0) { s_n = n; s_nmark = 0; }
    }
    __syncthreads();
    const uint32_t nsel = s_n;
    bool serial = out_off[b + 1] > ws_bytes;   // (the same in every thread)
    // ---- sizes: a warp takes a node, its lanes the segments ----
    if (!serial)
        for (uint32_t k = warp; k < nsel; k += kAnsPlaceThreads / 32) {
            const uint32_t v = s_node[k], raw = (L.nv[v] + 7) / 8, S = ans_seg_count(raw), at = L.body_off[v];
            uint64_t sum = 0;
            bool tail = false, marks = false;
            for (uint32_t s = lane; s < S; s += 32) {
                const uint32_t sb = min(kAnsSeg, raw - s * kAnsSeg);
                if (sb < kAnsMirrorMin) { tail = true; continue; }
                const uint32_t nw = ld_le32(mir + at + s * kAnsSeg);
                sum += 4 + 4 * ans_seg_lanes(sb) + 2ull * (nw & ~kAnsMarked);
                if (nw & kAnsMarked) marks = true;
            }
            tail = __any_sync(0xffffffffu, tail);
#pragma unroll
            for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (tail) {   // the last segment's word count
                const uint32_t sb = raw % kAnsSeg, mk = L.sel[v];
                uint32_t x;
                __syncwarp();
                load_ans_table(s_T[warp], A, (mk & 0x7F) - 1, lane, 32, true);
                __syncwarp();
                const uint32_t nw = ans_encode_segment(rec + at + raw - sb, sb, s_T[warp], (mk & 0x80) ? 0xFF : 0, stage, 0u,
                                                       nullptr, 0u, x);
                sum += 4 + 4 * ans_seg_lanes(sb) + 2ull * nw;
            }
            if (marks && sum < raw)
                for (uint32_t s = lane; s < S; s += 32) {
                    if (min(kAnsSeg, raw - s * kAnsSeg) < kAnsMirrorMin) continue;
                    const uint32_t nw = ld_le32(mir + at + s * kAnsSeg);
                    if (!(nw & kAnsMarked)) continue;
                    const uint32_t i = atomicAdd(&s_nmark, 1u);
                    if (i < kAnsMarks) { s_mark[i][0] = k; s_mark[i][1] = s; s_mark[i][2] = nw & ~kAnsMarked; }
                }
            if (lane == 0) { s_len[k] = sum < raw ? (uint32_t)sum : 0u; s_tail[k] = tail; }
        }
    __syncthreads();
    const uint32_t nmark = s_nmark;
    if (serial || nmark > kAnsMarks) {
        if (warp == 0) ans_encode_block_serial(b, layout, out, out_off, rec_bytes, ws, ws_bytes, A);
        return;
    }
    // the marked segments' bytes into their mirrors, where the rewrite leaves them alone
    for (uint32_t i = 0; i < nmark; i++) {
        const uint32_t v = s_node[s_mark[i][0]], raw = (L.nv[v] + 7) / 8, o = s_mark[i][1] * kAnsSeg;
        copy_words(ws + out_off[b] + L.body_off[v] + o, rec + L.body_off[v] + o, min(kAnsSeg, raw - o), t, kAnsPlaceThreads);
    }
    if (nmark) __syncthreads();
    // ---- rewrite the selected region in breadth-first order ----
    // A node with a last segment without a mirror, and one kept raw, reads the record:
    // all the nodes up to it are in place before the next is begun.  The others
    // read the mirror, and end before the next node's raw copy: the warps take
    // their pieces in turn, and run ahead as far as no such node stands between.
    const uint32_t alen_off = (kNvOff + 5u * V + 3u) & ~3u;
    uint32_t q = L.body_off[s_node[0]];
    for (uint32_t k = 0, turn = 0; k < nsel; k++) {
        const uint32_t v = s_node[k], raw = (L.nv[v] + 7) / 8, bl = s_len[k], at = L.body_off[v];
        const bool tail = bl && s_tail[k];
        if (bl) {
            const uint32_t S = ans_seg_count(raw);
            if (tail) {   // before anything of the node is written
                __syncthreads();
                if (warp == 0) {
                    const uint32_t sb = raw % kAnsSeg, mk = L.sel[v];
                    uint32_t x;
                    load_ans_table(s_T[0], A, (mk & 0x7F) - 1, lane, 32, true);
                    __syncwarp();
                    const uint32_t nw = ans_encode_segment(rec + at + raw - sb, sb, s_T[0], (mk & 0x80) ? 0xFF : 0, stage,
                                                           kAnsStageWords, nullptr, 0u, x);
                    s_x[lane] = x;
                    if (lane == 0) s_nw = nw;
                }
                __syncthreads();
            }
            // segments and their words in turn by the warps (p: where the segment's states go)
            uint32_t p = q + 4 * S;
            for (uint32_t s = 0; s < S; s++) {
                const uint32_t sb = min(kAnsSeg, raw - s * kAnsSeg), W = ans_seg_lanes(sb);
                const uint8_t *lo = mir + at + s * kAnsSeg;
                const bool staged = tail && s == S - 1;
                uint32_t mark = kAnsMarks;
                for (uint32_t i = 0; i < nmark; i++)
                    if (s_mark[i][0] == k && s_mark[i][1] == s) mark = i;
                const uint32_t nw = mark < kAnsMarks ? s_mark[mark][2] : (staged ? s_nw : ld_le32(lo));
                if (mark < kAnsMarks) {   // by one warp, its words straight to their place
                    if (turn++ % kAnsPlaceWarps == (uint32_t)warp) {
                        const uint32_t mk = L.sel[v];
                        uint32_t x;
                        __syncwarp();
                        load_ans_table(s_T[warp], A, (mk & 0x7F) - 1, lane, 32, true);
                        __syncwarp();
                        ans_encode_segment(lo, sb, s_T[warp], (mk & 0x80) ? 0xFF : 0, stage, 0u, rec + p + 4 * W, nw, x);
                        __syncwarp();
                        ans_place_words(stage, 0u, nw, rec + p + 4 * W);
                        if (lane < 4) rec[q + 4 * s + lane] = (uint8_t)(nw >> (8 * lane));
                        if (lane < (int)W) st_le32(rec + p + 4 * lane, x);
                    }
                    p += 4 * W + 2 * nw;
                    continue;
                }
                if (turn++ % kAnsPlaceWarps == (uint32_t)warp) {
                    if (lane < 4) rec[q + 4 * s + lane] = (uint8_t)(nw >> (8 * lane));
                    if (lane < (int)W) st_le32(rec + p + 4 * lane, staged ? s_x[lane] : ld_le32(lo + 4 + 4 * lane));
                    if (staged) {
                        const uint16_t *wb = stage + kAnsStageWords - nw;
                        for (uint32_t i = lane; i < nw; i += 32) {
                            rec[p + 4 * W + 2 * i] = (uint8_t)wb[i];
                            rec[p + 4 * W + 2 * i + 1] = (uint8_t)(wb[i] >> 8);
                        }
                    }
                }
                if (!staged) {   // 1 KiB at a time to a warp
                    const uint8_t *wb = reinterpret_cast<const uint8_t *>((reinterpret_cast<uintptr_t>(lo) + sb) & ~(uintptr_t)1) - 2 * nw;
                    for (uint32_t i = 0; i < 2 * nw; i += 1024)
                        if (turn++ % kAnsPlaceWarps == (uint32_t)warp)
                            copy_words(rec + p + 4 * W + i, wb + i, min(1024u, 2 * nw - i), lane, 32);
                }
                p += 4 * W + 2 * nw;
            }
            if (t == 0) rec[kNvOff + 4 * V + v] = L.sel[v];
            if (tail) __syncthreads();   // (the stage)
        } else if (q != at) {
            __syncthreads();
            for (uint32_t base = 0; base < raw; base += kAnsPlaceThreads) {   // down, in order
                const uint32_t i = base + t;
                const uint8_t c = i < raw ? rec[at + i] : 0;
                __syncthreads();
                if (i < raw) rec[q + i] = c;
                __syncthreads();
            }
        }
        const uint32_t len = bl ? bl : raw;
        if (t < 4) rec[alen_off + 4 * k + t] = (uint8_t)(len >> (8 * t));
        q += len;
    }
    const uint32_t total = (q + 15u) & ~15u;
    for (uint32_t i = q + t; i < total; i += kAnsPlaceThreads) rec[i] = 0;
    if (t < 4) rec[t] = (uint8_t)(total >> (8 * t));
    if (t == 0) rec_bytes[b] = total;
}

cudaError_t launch_ans_encode_blocks(const BlockLayout *layout, int nblk, uint8_t *out, const uint64_t *out_off,
                                     uint64_t *rec_bytes, uint8_t *ws, size_t ws_bytes, int32_t *status, cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    const int smem = (int)(((sizeof(AnsSm) + 15) & ~15) + 2 * kAnsStageWords);
    cudaError_t e = cudaFuncSetAttribute(ans_encode_place_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    // warps per block: up to 32, about 32 per SM in all
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int per = max(1, min(32, 32 * sms / nblk));
    ans_encode_units_kernel<<<dim3(nblk, per), 32, 0, st>>>(layout, out, out_off, ws, ws_bytes, status,
                                                                           host_ans_tables());
    ans_encode_place_kernel<<<nblk, kAnsPlaceThreads, smem, st>>>(layout, out, out_off, rec_bytes, ws, ws_bytes, status,
                                                                  host_ans_tables());
    count_launches(2);
    return cudaGetLastError();
}


}  // namespace pv

namespace pv {
cudaError_t prepare_ans_kernels() {
    const int smem = (int)(((sizeof(AnsSm) + 15) & ~15) + 2 * kAnsStageWords);
    cudaError_t e = cudaFuncSetAttribute(ans_encode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ans_encode_place_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e;
}
}  // namespace pv
