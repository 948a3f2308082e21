// The levels of a tile (decoder) or part (encoder) in shared memory: the
// symbols of every node of a level, node after node, in the level's buffer.
// Bottom-up or top-down, a level is worked on in windows of 32 groups, a group
// being 32 consecutive symbols of one node (one bitmap word); the ordinary
// nodes of a level share its windows, a flat node has windows of its own.
//
// The tables are members of the tile's or part's structure T:
//   dem[v], ch[v]      symbols of node v here, its children word
//   first[d], maxd     first node of each depth
//   sp[v]              byte offset of node v's sequence in its level buffer
//   gs[first[d] + i], onode[first[d] + i]
//                      first group of the level's i-th ordinary node, and the node
//   fw[v]              flat node: its first window among the level's flat windows
//   lg[d], no[d]       groups and number of ordinary nodes of the level
//   nwo[d], nw[d]      ordinary windows, windows (the ordinary ones first)
//   wn_off[d]          first entry of the level in wnode
//   wnode[]            ordinary window: index (among the level's ordinary
//                      nodes) of the node holding its first group; flat
//                      window: its node
#pragma once
#include "pivco_dev.cuh"

namespace pv {

constexpr int kLvlWarps = 8;
constexpr int kWinMax = 512;                   // windows of all levels below the root
constexpr uint32_t kGrp = 32;                  // symbols of a group
constexpr uint32_t kWin = 32 * kGrp;           // symbols of a full window

__device__ inline uint32_t warp_inclusive(uint32_t x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Spans, groups and windows of every level for the current demands, by the
// whole CTA: warp w lays out levels w, w + 8, ... (a level's spans, groups
// and flat windows are one packed scan over its own nodes); the levels'
// window tables then follow one another in depth order.  Spans start on
// 16-byte boundaries, so a lane stores its 32 symbols in two vectors (eight
// 4-byte stores 32 bytes apart were 64 wavefronts a window).  False (in
// every thread) when a level (depth >= 1) does not fit a buffer or the
// windows do not fit their table.
template <typename T>
__device__ inline bool lvl_layout(T &S) {
    constexpr uint32_t kBuf = (uint32_t)T::kBuf;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int maxd = S.maxd;
    bool fits = true;
    for (int d = warp; d < maxd; d += kLvlWarps) {
        if (d == 0) continue;   // the root has no span; its windows are strips
        const int f0 = S.first[d], f1 = S.first[d + 1];
        // bytes << 40 | groups of ordinary nodes << 20 | flat windows << 10 | ordinary nodes
        uint64_t carry = 0;
        for (int base = f0; base < f1; base += 32) {
            const int v = base + lane;
            uint64_t x = 0;
            bool flat = false;
            uint32_t dv = 0;
            if (v < f1) {
                dv = S.dem[v];
                flat = ch_flat_d(S.ch[v]) != 0;
                if (dv > kBuf) { fits = false; dv = kBuf; }
                const uint32_t by = (dv + 15u) & ~15u;
                x = ((uint64_t)by << 40) |
                    (flat ? (uint64_t)((dv + kWin - 1) / kWin) << 10 : ((uint64_t)max(1u, (dv + kGrp - 1) / kGrp) << 20) | 1u);
            }
            uint64_t inc = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            const uint64_t ex = carry + inc - x;
            if (v < f1) {
                S.sp[v] = (uint16_t)min((uint64_t)kBuf, ex >> 40);
                if (flat) {
                    S.fw[v] = (uint16_t)((ex >> 10) & 1023u);
                } else {
                    const uint32_t i = (uint32_t)f0 + ((uint32_t)ex & 1023u);
                    S.onode[i] = (uint8_t)v;
                    S.gs[i] = (uint16_t)((ex >> 20) & 0xFFFFFu);
                }
            }
            carry += __shfl_sync(0xffffffffu, inc, 31);
        }
        if ((carry >> 40) > (uint64_t)kBuf) fits = false;
        const uint32_t G = (uint32_t)(carry >> 20) & 0xFFFFFu, nwo = (G + 31) >> 5;
        if (G > 0xFFFFu) fits = false;
        if (lane == 0) {
            S.lg[d] = (uint16_t)G;
            S.no[d] = (uint16_t)(carry & 1023u);
            S.nwo[d] = (uint16_t)nwo;
            S.nw[d] = (uint16_t)(nwo + ((uint32_t)(carry >> 10) & 1023u));
        }
    }
    __syncthreads();
    // window table offsets: lane d holds level d's windows (none at the root)
    const uint32_t nwin_l = lane >= 1 && lane < maxd ? (uint32_t)S.nw[lane] : 0u;
    uint32_t wi = nwin_l;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
        if (lane >= o) wi += y;
    }
    if (__shfl_sync(0xffffffffu, wi, 31) > (uint32_t)kWinMax) fits = false;
    const uint32_t wn_l = wi - nwin_l;
    for (int d = warp; d < maxd; d += kLvlWarps) {
        const uint32_t wn = __shfl_sync(0xffffffffu, wn_l, d);
        if (d == 0) continue;
        if (lane == 0) S.wn_off[d] = (uint16_t)min(wn, (uint32_t)kWinMax);
        // ordinary windows: the last ordinary node whose first group is at or before the window's first
        const uint32_t nwo = S.nwo[d], no = S.no[d];
        const int f0 = S.first[d], f1 = S.first[d + 1];
        for (uint32_t i = lane; i < nwo && wn + i < (uint32_t)kWinMax; i += 32) {
            int lo = 0, hi = (int)no;
            while (hi - lo > 1) {
                const int m = (lo + hi) >> 1;
                if ((uint32_t)S.gs[f0 + m] <= 32u * i) lo = m; else hi = m;
            }
            S.wnode[wn + i] = (uint8_t)lo;
        }
        // flat windows: their node
        if (no != (uint32_t)(f1 - f0))
            for (int v = f0 + lane; v < f1; v += 32)
                if (ch_flat_d(S.ch[v])) {
                    const uint32_t w0 = wn + nwo + S.fw[v], nf = (min(S.dem[v], kBuf) + kWin - 1) / kWin;
                    for (uint32_t i = 0; i < nf && w0 + i < (uint32_t)kWinMax; i++) S.wnode[w0 + i] = (uint8_t)v;
                }
    }
    return !__syncthreads_or(!fits);
}

// This lane's group in ordinary window i of level d (wn, f0: wn_off[d],
// first[d]; the whole warp): its node v and number q within the node.  Returns
// the node's symbols from the group on, 0 when there are none.
template <typename T>
__device__ inline uint32_t lvl_locate(const T &S, int d, uint32_t wn, uint32_t f0, uint32_t i, uint32_t &v, uint32_t &q) {
    const int lane = threadIdx.x & 31;
    const uint32_t g = 32u * i + lane, u = S.wnode[wn + i];
    // the nodes after u that start in the window (every node has a group)
    const uint32_t cand = u + 1 + lane;
    uint32_t bit = 0;
    if (cand < S.no[d]) {
        const uint32_t s = (uint32_t)S.gs[f0 + cand] - 32u * i;
        if (s < 32) bit = 1u << s;
    }
    const uint32_t idx = f0 + u + __popc(__reduce_or_sync(0xffffffffu, bit) & (0xFFFFFFFFu >> (31 - lane)));
    v = S.onode[idx];
    q = g - S.gs[idx];
    const uint32_t dv = S.dem[v];
    return g < S.lg[d] && kGrp * q < dv ? dv - kGrp * q : 0u;
}

}  // namespace pv
