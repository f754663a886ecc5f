// first_pass.cuh -- the first pass of Eq. hll-union as a scatter of the nodes'
// keys, for a group of nodes at once.
#pragma once

#include "hb_device.cuh"

namespace vga {
namespace {

constexpr int kGroupScatterWarps = 4;

// Register j of next[v] is the largest rho among the keys of v and its
// neighbours whose register index is j (first_pass_item).  Neighbouring nodes
// see almost the same ids, so one CTA scatters for the kCodeNodes nodes of a
// group: each of its rows (range lookups by class, the nodes that see the ids)
// is read once, and one atomic OR puts an id's level, min(rho, 16) - 1, into
// the cells of all nodes of the class.  A register's cell holds a bit for every
// level and node, node j's bit of level l being 4 (l % 8) + j of word l / 8: a
// register is its node's highest bit.  Level 15 stands for every rho from 16
// on; the register is then the index's largest rho (gmax), unless several
// lie there (gbig), when the node's ids are searched.
// Bound: shared-memory atomics and the instructions around them, one visit an
// id and group where the per-node scatter has one an id and node: 7,350 ids a
// node against 21,100 on the city graph, 8.5 -> 4.4 ms.
// All threads of a CTA of kGroupScatterWarps warps take part; `cells`: 2 x m
// words of its shared memory.
struct GroupScatterShared {
    uint2 stage[kGroupScatterWarps][32];
    uint32_t mask[1 << kCodeNodes], end[1 << kCodeNodes], own[kCodeNodes];
};

template <bool NIB, class K>
__device__ __forceinline__ void first_pass_group(const GroupItem &gi, const uint32_t *__restrict__ rows,
                                                 const uint2 *__restrict__ cls, const K *__restrict__ keys, uint32_t n,
                                                 int p, int scheme, int s_log2, const uint32_t *__restrict__ gmax,
                                                 const uint32_t *__restrict__ gbig, uint64_t seed,
                                                 uint8_t *__restrict__ nxt, uint32_t *__restrict__ flag,
                                                 uint8_t *__restrict__ chg, uint32_t *s_cells, GroupScatterShared &sh) {
    uint32_t *s_mask = sh.mask, *s_end = sh.end, *s_own = sh.own;
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const uint32_t m = 1u << p, cnt = gi.cnt, nc = gi.nc;
    const uint32_t *src = rows + gi.b;
    for (uint32_t k = threadIdx.x; k < m / 2u; k += blockDim.x)
        reinterpret_cast<uint4 *>(s_cells)[k] = make_uint4(0, 0, 0, 0);
    if (wib == 0) {  // the classes' masks and ends
        const uint2 c = lane < (int)nc ? cls[gi.cls + lane] : make_uint2(0, 0);
        uint32_t end = c.y;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += y;
        }
        if (lane < (int)nc) {
            s_mask[lane] = c.x;
            s_end[lane] = end;
        }
    }
    __syncthreads();
    if (threadIdx.x < kCodeNodes) {  // the nodes' own keys
        const uint32_t v = gi.node[threadIdx.x];
        const uint32_t own = v == 0xffffffffu ? 0xffffff00u : node_key(v, p, seed, NIB);
        s_own[threadIdx.x] = own;
        if (v != 0xffffffffu) {
            const uint32_t level = min(own & 0xffu, 16u) - 1u;
            atomicOr(s_cells + (level >> 3) * m + (own >> 8), 1u << (4u * (level & 7u) + threadIdx.x));
        }
    }
    const int slots = table_rows(scheme);
    uint2 *stage = sh.stage[wib];
    uint32_t c = 0;
    uint32_t r_next = wib * 32u + lane < cnt ? __ldcs(src + wib * 32u + lane) : 0u;
    for (uint32_t base = wib * 32u; base < cnt; base += kGroupScatterWarps * 32u) {
        const uint32_t idx = base + lane;
        const bool valid = idx < cnt;
        const uint32_t r = r_next;
        if (idx + kGroupScatterWarps * 32u < cnt) r_next = __ldcs(src + idx + kGroupScatterWarps * 32u);
        while (s_end[c] <= base) c++;
        uint32_t mask = s_mask[c];
        for (uint32_t d = c; d + 1u < nc && s_end[d] < base + 32u; d++) mask = idx >= s_end[d] ? s_mask[d + 1u] : mask;
        uint32_t slot = 0;
        for (int s = 1; s < slots; s++) slot += r >= (uint32_t)s * n ? 1u : 0u;
        const uint32_t level = scheme == 0 ? slot : 2u * slot;
        const uint32_t packed = (r - slot * n) | (level << 29);  // i < 2^29 (kRunMaxNodes)
#pragma unroll
        for (int grp = 0; grp < 2; grp++) {
            const int G = grp == 0 ? 4 : 16;  // lanes per row: windows of 1..4, of 8..16 ids
            const int per = 32 / G;
            const uint32_t take = __ballot_sync(0xffffffffu, valid && ((level <= 2u) == (grp == 0)));
            if (!take) continue;
            if ((take >> lane) & 1u) stage[__popc(take & ((1u << lane) - 1u))] = make_uint2(packed, mask);
            __syncwarp();
            const int rows_here = __popc(take);
            const int my = lane / G;
            const uint32_t off = (uint32_t)(lane % G);
            for (int q = 0; q < rows_here; q += 4 * per) {
                uint32_t key[4], bits[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int x = q + u * per + my;
                    key[u] = bits[u] = 0u;
                    if (x < rows_here) {
                        const uint2 e = stage[x];
                        if (off < (1u << (e.x >> 29))) {
                            key[u] = __ldg(keys + (e.x & 0x1fffffffu) + off);
                            bits[u] = e.y;
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if (bits[u])
                        atomicOr(s_cells + ((key[u] >> 3) & 1u) * m + (key[u] >> 4), bits[u] << (4u * (key[u] & 7u)));
            }
            __syncwarp();
        }
    }
    __syncthreads();
    // the registers, a word of every node at a time
    constexpr uint32_t F = NIB ? 8u : 4u, WIDTH = NIB ? 4u : 8u;
    const uint32_t words = m / F;
    bool changed = false;
    for (uint32_t k0 = 0; k0 < words; k0 += blockDim.x) {  // a uniform loop
        const uint32_t k = k0 + threadIdx.x;
        const bool in = k < words;
        uint32_t w[kCodeNodes] = {};
#pragma unroll
        for (uint32_t i = 0; i < F; i++) {
            const uint32_t j = k * F + i;
            const uint32_t lo = in ? s_cells[j] : 0u, hi = in ? s_cells[m + j] : 0u;
#pragma unroll
            for (int a = 0; a < kCodeNodes; a++) {
                const uint32_t x = (hi >> a) & 0x11111111u, y = (lo >> a) & 0x11111111u;
                uint32_t rho = x ? 9u + ((31u - __clz(x)) >> 2) : y ? 1u + ((31u - __clz(y)) >> 2) : 0u;
                if (!NIB && __any_sync(0xffffffffu, rho == 16u)) {
                    bool search = false;
                    if (rho == 16u) {
                        rho = __ldg(gmax + j);
                        const uint32_t big = __ldg(gbig + j);
                        search = (big & (big - 1u)) != 0u || (big >> 31) != 0u;
                    }
                    uint32_t todo = __ballot_sync(0xffffffffu, search);
                    while (todo) {  // practically never: the ids of node a with register index j and level 15
                        const int who = __ffs(todo) - 1;
                        todo &= todo - 1u;
                        const uint32_t want = (__shfl_sync(0xffffffffu, j, who) << 4) | 15u;
                        uint32_t best = (s_own[a] >> 8) == want >> 4 ? s_own[a] & 0xffu : 0u;
                        for (uint32_t d = 0; d < nc; d++) {
                            if (!((s_mask[d] >> a) & 1u)) continue;
                            for (uint32_t e = (d ? s_end[d - 1u] : 0u) + lane; e < s_end[d]; e += 32u) {
                                const uint32_t r = src[e];
                                uint32_t slot = 0;
                                for (int s = 1; s < slots; s++) slot += r >= (uint32_t)s * n ? 1u : 0u;
                                const uint32_t id = r - slot * n, len = 1u << (scheme == 0 ? slot : 2u * slot);
                                for (uint32_t o = 0; o < len; o++)
                                    if (keys[id + o] == want) best = max(best, node_key(id + o, p, seed, NIB) & 0xffu);
                            }
                        }
                        best = __reduce_max_sync(0xffffffffu, best);
                        if (lane == who) rho = best;
                    }
                }
                w[a] |= rho << (WIDTH * i);
            }
        }
        if (!in) continue;
        const uint32_t byte = 4u * k, sl = byte >> s_log2;
#pragma unroll
        for (int a = 0; a < kCodeNodes; a++) {
            const uint32_t v = gi.node[a];
            if (v == 0xffffffffu) continue;
            const uint32_t own_j = s_own[a] >> 8;
            const uint32_t mine = own_j / F == k ? (s_own[a] & 0xffu) << (WIDTH * (own_j % F)) : 0u;
            changed |= w[a] != mine;
            if (chg && w[a] != mine) chg[(uint64_t)sl * n + v] = 1u;  // threads of one slice store the same byte
            *reinterpret_cast<uint32_t *>(nxt + (((uint64_t)sl * n + v) << s_log2) + (byte & ((1u << s_log2) - 1u))) = w[a];
        }
    }
    if (__any_sync(0xffffffffu, changed) && lane == 0) {
        if (*reinterpret_cast<volatile uint32_t *>(flag) == 0u) atomicOr(flag, 1u);
    }
}

}  // namespace
}  // namespace vga
