// codes.cuh -- bit-plane codes of the registers, the form in which the grouped
// union gathers them from the second pass on.
//
// No register j of any node ever exceeds G[j], the largest rho inserted with
// index j (kept from Alg. 1's initialisation).  A pass therefore needs only
// the top of each register's range:
//   K = 4  code = max(0, R - B[j]) with B[j] = max(0, G[j] - 15): 4 bits, exact
//          for every value above B[j];
//   K = 1  one bit, R == G[j] (the register has reached its final value).
// A register whose gathered code is 0 while its own value lies below B[j]
// (K = 4) or G[j] (K = 1) is left open: its (node, slice) pair is marked in the
// need masks and recomputed from the bytes, so every result is exact.
//
// Why: the union is bound by the L2 bytes of its row gathers.  A K = 4 row
// holds twice the registers of a byte row and a K = 1 row eight times.  After
// pass 1 practically no register lies 15 below G (measured on the city and
// medium graphs); after pass 2, 82-99 % of the registers equal G, and after
// pass 3 all but 1e-5 of the city's.
//
// Measured (GB300): the city graph's pass 2 takes four launches of 128-byte
// K = 4 rows at 3.16 ms, table included, and pass 3 one of K = 1 rows at 0.73 ms (2.8
// before a class was cut short once all its bits were set, code_group), where the
// byte union takes eight at 2.8 ms each; the d = 3 analysis (with pass 1 by
// groups, first_pass.cuh) 57.4 -> 19.6 ms, the unlimited one at p = 12 343 -> 70
// ms, medium d = 3 3.1 -> 1.5-1.7 ms.  Graphs of small views have to be told apart
// (run_impl, code_rows_pay): there many registers stay below the window, and rows
// are too few to save on.
//
// Layout: a 16-byte unit holds 32 registers as four bit planes (K = 4; word k =
// bit k of the codes, bit i = register i) or 128 registers as one plane
// (K = 1).  In planes the maximum of 32 codes takes 8 three-input logic
// operations (a borrow chain, then a select), 2.5 times fewer per register
// than byte maxima on 16-bit lanes, and the maximum of one-bit codes is OR.
#pragma once

#include "hb_device.cuh"

namespace vga {
namespace {

// Registers per 16-byte unit.
template <int K>
constexpr int kUnitRegs = K == 4 ? 32 : 128;

// Lane-wise maximum of two units.
template <int K>
__device__ __forceinline__ uint4 code_max(uint4 a, uint4 b) {
    if (K == 1) return make_uint4(a.x | b.x, a.y | b.y, a.z | b.z, a.w | b.w);
    uint32_t t = a.x & ~b.x;                 // a > b on bit 0, then up the planes
    t = (a.y & ~b.y) | (t & (a.y | ~b.y));
    t = (a.z & ~b.z) | (t & (a.z | ~b.z));
    t = (a.w & ~b.w) | (t & (a.w | ~b.w));
    return make_uint4((a.x & t) | (b.x & ~t), (a.y & t) | (b.y & ~t), (a.z & t) | (b.z & ~t),
                      (a.w & t) | (b.w & ~t));
}

// Bit 0 of a word's 4 bytes (or 8 nibbles) gathered into its low bits, and back.
__device__ __forceinline__ uint32_t gather_bytes(uint32_t w) { return ((w & 0x01010101u) * 0x01020408u) >> 24; }
__device__ __forceinline__ uint32_t spread_bytes(uint32_t b) { return (b * 0x00204081u) & 0x01010101u; }
__device__ __forceinline__ uint32_t gather_nibbles(uint32_t w) {
    w &= 0x11111111u;
    w = (w | w >> 3) & 0x03030303u;
    w = (w | w >> 6) & 0x000F000Fu;
    return (w | w >> 12) & 0xFFu;
}
__device__ __forceinline__ uint32_t spread_nibbles(uint32_t b) {
    b = (b | b << 12) & 0x000F000Fu;
    b = (b | b << 6) & 0x03030303u;
    return (b | b << 3) & 0x11111111u;
}

// The register window of a run, one word array each in the registers' own
// format (bytes, or nibbles): top[j] = G[j] and low[j] = B[j].
struct CodeWindow {
    const uint32_t *top, *low;
};

// Address of byte `byte` of node v's registers (slice-major, slices of
// 2^s_log2 bytes).
__device__ __forceinline__ uint64_t reg_at(uint32_t n, int s_log2, uint32_t v, uint32_t byte) {
    return (((uint64_t)(byte >> s_log2) * n + v) << s_log2) + (byte & ((1u << s_log2) - 1u));
}

// Codes of unit u of node v, from its registers.
template <int K, bool NIB>
__device__ __forceinline__ uint4 code_pack(const uint8_t *__restrict__ cur, uint32_t n, int s_log2, uint32_t v,
                                           uint32_t u, const CodeWindow &win) {
    constexpr int F = NIB ? 8 : 4;                  // registers per word
    constexpr int BYTES = kUnitRegs<K> * 4 / F;     // register bytes of a unit
    uint32_t p[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int h = 0; h < BYTES / 16; h++) {
        const uint32_t byte = u * BYTES + 16u * h;
        const uint4 x = __ldg(reinterpret_cast<const uint4 *>(cur + reg_at(n, s_log2, v, byte)));
        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int r = (4 * h + i) * F;          // first register of the word, within the unit
            if (K == 4) {
                const uint32_t c = NIB ? w[i] : __vsubus4(w[i], __ldg(win.low + byte / 4u + i));
#pragma unroll
                for (int k = 0; k < 4; k++)
                    p[k] |= (NIB ? gather_nibbles(c >> k) : gather_bytes(c >> k)) << r;
            } else {
                const uint32_t e = equal_bits<NIB>(w[i], __ldg(win.top + byte / 4u + i));
                p[r / 32] |= (NIB ? gather_nibbles(e) : gather_bytes(e)) << (r % 32);
            }
        }
    }
    return make_uint4(p[0], p[1], p[2], p[3]);
}

// next[v] for the registers of unit u, from the unit's gathered codes and the
// node's own registers; returns whether a register changed (bit 0) per 16
// register bytes h in `chg16` and left open in `open16` (bit h each).
template <int K, bool NIB>
__device__ __forceinline__ void code_store(uint4 code, const uint8_t *__restrict__ cur, uint8_t *__restrict__ nxt,
                                           uint32_t n, int s_log2, uint32_t v, uint32_t u, const CodeWindow &win,
                                           uint32_t &chg16, uint32_t &open16) {
    constexpr int F = NIB ? 8 : 4;
    constexpr int BYTES = kUnitRegs<K> * 4 / F;
    const uint32_t p[4] = {code.x, code.y, code.z, code.w};
    chg16 = open16 = 0;
#pragma unroll
    for (int h = 0; h < BYTES / 16; h++) {
        const uint32_t byte = u * BYTES + 16u * h;
        const uint64_t at = reg_at(n, s_log2, v, byte);
        const uint4 x = __ldg(reinterpret_cast<const uint4 *>(cur + at));
        const uint32_t own[4] = {x.x, x.y, x.z, x.w};
        uint32_t res[4], diff = 0, open = 0;
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int r = (4 * h + i) * F;
            if (K == 4) {
                uint32_t c = 0;
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const uint32_t b = (p[k] >> r) & (NIB ? 0xFFu : 0xFu);
                    c |= (NIB ? spread_nibbles(b) : spread_bytes(b)) << k;
                }
                if (NIB) {
                    res[i] = RegFmt<NIB>::max_word(own[i], c);
                } else {
                    const uint32_t low = __ldg(win.low + byte / 4u + i);
                    const uint32_t zero = __vcmpeq4(c, 0u);       // 0xFF where the code is 0
                    res[i] = __vmaxu4(own[i], (c + low) & ~zero);  // c + low <= 15 + B: no carry between bytes
                    open |= zero & __vcmpltu4(own[i], low);
                }
            } else {
                const uint32_t b = (p[r / 32] >> (r % 32)) & (NIB ? 0xFFu : 0xFu);
                const uint32_t set = (NIB ? spread_nibbles(b) * 0xFu : spread_bytes(b) * 0xFFu);
                const uint32_t top = __ldg(win.top + byte / 4u + i);
                res[i] = (own[i] & ~set) | (top & set);
                open |= res[i] ^ top;
            }
            diff |= res[i] ^ own[i];
        }
        *reinterpret_cast<uint4 *>(nxt + at) = make_uint4(res[0], res[1], res[2], res[3]);
        chg16 |= diff ? 1u << h : 0u;
        open16 |= open ? 1u << h : 0u;
    }
}

// Open pieces of unit u of node v (open16: bit per 16 register bytes) to the
// list, as far as it holds them; *count counts them all.  With JOIN the lanes
// that get here together raise it once: on graphs of small views every node has
// some.  (Not in the engine: its kernel for 512-byte rows then took 25 % longer,
// 5.0 ms against 4.0 in the second pass of 64 sites.)
template <int K, bool NIB, bool JOIN>
__device__ __forceinline__ void code_push_open(uint32_t open16, uint32_t v, uint32_t u, uint2 *__restrict__ list,
                                               uint32_t list_cap, uint32_t *count) {
    constexpr uint32_t PIECES = kUnitRegs<K> / (NIB ? 2 : 1) / 16;
    const uint32_t mine = (uint32_t)__popc(open16), here = JOIN ? __activemask() : 0u;
    uint32_t at;
    if (JOIN && __all_sync(here, mine == 1u)) {
        const int lead = __ffs(here) - 1;
        const uint32_t lane = threadIdx.x & 31u;
        if ((int)lane == lead) at = atomicAdd(count, (uint32_t)__popc(here));
        at = __shfl_sync(here, at, lead) + __popc(here & ((1u << lane) - 1u));
    } else {
        at = atomicAdd(count, mine);
    }
    for (uint32_t b = open16; b && at < list_cap; b &= b - 1u)
        list[at++] = make_uint2(v, u * PIECES + (uint32_t)__ffs(b) - 1u);
}

// Maximum of the 16 register bytes at `base` + node * 2^s_log2 over the range
// lookups lk[b .. e), lookups b + first, b + first + step, ... by this lane;
// every lane of its group of G ends with the group's.
template <bool NIB, int G>
__device__ __forceinline__ uint4 code_open_fold(const uint8_t *__restrict__ base, const uint32_t *__restrict__ lk,
                                                uint64_t b, uint64_t e, uint32_t first, uint32_t step, uint32_t n,
                                                int s_log2, int scheme) {
    const int rows = table_rows(scheme);
    uint4 acc = make_uint4(0, 0, 0, 0);
    for (uint64_t k = b + first; k < e; k += step) {
        const uint32_t r = __ldg(lk + k);
        uint32_t slot = 0;
        for (int s = 1; s < rows; s++) slot += r >= (uint32_t)s * n ? 1u : 0u;
        const uint32_t i = r - slot * n, w = 1u << (scheme == 0 ? slot : 2u * slot);
#pragma unroll 4
        for (uint32_t j = 0; j < w; j++)
            acc = RegFmt<NIB>::max4(acc, __ldg(reinterpret_cast<const uint4 *>(base + ((uint64_t)(i + j) << s_log2))));
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        uint4 y;
        y.x = __shfl_xor_sync(0xffffffffu, acc.x, o);
        y.y = __shfl_xor_sync(0xffffffffu, acc.y, o);
        y.z = __shfl_xor_sync(0xffffffffu, acc.z, o);
        y.w = __shfl_xor_sync(0xffffffffu, acc.w, o);
        acc = RegFmt<NIB>::max4(acc, y);
    }
    return acc;
}

// The larger of the folded registers and the node's own into nxt; whether that
// changed them.
template <bool NIB>
__device__ __forceinline__ bool code_open_store(uint4 acc, const uint8_t *__restrict__ cur, uint8_t *__restrict__ nxt,
                                                uint64_t at) {
    const uint4 own = *reinterpret_cast<const uint4 *>(cur + at);
    acc = RegFmt<NIB>::max4(acc, own);
    *reinterpret_cast<uint4 *>(nxt + at) = acc;
    return ((acc.x ^ own.x) | (acc.y ^ own.y) | (acc.z ^ own.z) | (acc.w ^ own.w)) != 0u;
}

struct OpenShared {
    uint4 max[8];
    uint32_t piece[32];
};

// next[v] for the open pieces list[0 .. count) ({node, 16-byte piece}), straight
// from the registers of the nodes' neighbours: the lookups lk[b .. e) that
// range(v, b, e) gives.  This CTA (of 256 threads) is `cta` of `ctas`.  G lanes
// settle a piece whose node has up to MOST lookups and a warp one of up to
// BY_WARP; the CTA does the others one after another, a thread a lookup.
// done(v, byte) is called by one thread for every piece that changed.
template <bool NIB, int G, int MOST, int BY_WARP, class Range, class Done>
__device__ __forceinline__ void code_open_pieces(const uint2 *__restrict__ list, uint32_t count, uint32_t cta,
                                                 uint32_t ctas, const Range &range, const uint32_t *__restrict__ lk,
                                                 const uint8_t *__restrict__ cur, uint8_t *__restrict__ nxt,
                                                 uint32_t n, int s_log2, int scheme, OpenShared &sh,
                                                 const Done &done) {
    constexpr uint32_t GROUPS = 256 / G;
    const uint32_t sub = threadIdx.x % G, group = threadIdx.x / G;
    auto base_of = [&](uint32_t byte) {
        return cur + ((uint64_t)(byte >> s_log2) * n << s_log2) + (byte & ((1u << s_log2) - 1u));
    };
    for (uint64_t first = cta; first < count; first += (uint64_t)GROUPS * ctas) {
        const uint64_t x = first + (uint64_t)group * ctas;
        uint32_t v = 0, byte = 0;
        uint64_t b = 0, e = 0;
        if (x < count) {
            v = list[x].x;
            byte = 16u * list[x].y;
            range(v, b, e);
        }
        const bool whole = e - b > (uint64_t)MOST, mine = x < count && !whole;
        const uint4 acc = code_open_fold<NIB, G>(base_of(byte), lk, b, whole ? b : e, sub, G, n, s_log2, scheme);
        if (mine && sub == 0 && code_open_store<NIB>(acc, cur, nxt, reg_at(n, s_log2, v, byte))) done(v, byte);
        if (sub == 0) sh.piece[group] = whole ? (uint32_t)x : 0xffffffffu;
        __syncthreads();
        if (BY_WARP > MOST) {
            for (uint32_t q = threadIdx.x / 32u; q < GROUPS; q += 8u) {
                const uint32_t y = sh.piece[q];
                if (y == 0xffffffffu) continue;
                v = list[y].x;
                byte = 16u * list[y].y;
                range(v, b, e);
                if (e - b > (uint64_t)BY_WARP) continue;
                const uint4 w = code_open_fold<NIB, 32>(base_of(byte), lk, b, e, threadIdx.x % 32u, 32u, n, s_log2,
                                                        scheme);
                if (threadIdx.x % 32u == 0) {
                    if (code_open_store<NIB>(w, cur, nxt, reg_at(n, s_log2, v, byte))) done(v, byte);
                    sh.piece[q] = 0xffffffffu;
                }
                __syncwarp();
            }
            __syncthreads();
        }
        for (uint32_t q = 0; q < GROUPS; q++) {
            const uint32_t y = sh.piece[q];
            if (y == 0xffffffffu) continue;
            v = list[y].x;
            byte = 16u * list[y].y;
            range(v, b, e);
            uint4 all = code_open_fold<NIB, 32>(base_of(byte), lk, b, e, threadIdx.x, 256u, n, s_log2, scheme);
            if (threadIdx.x % 32u == 0) sh.max[threadIdx.x / 32u] = all;
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int w = 1; w < 8; w++) all = RegFmt<NIB>::max4(all, sh.max[w]);
                if (code_open_store<NIB>(all, cur, nxt, reg_at(n, s_log2, v, byte))) done(v, byte);
            }
            __syncthreads();
        }
        __syncthreads();
    }
}

// Where nodes see little, most have a piece open: with 8 lanes a piece a CTA
// takes 32 at a time (a CTA a piece: 160 us a pass for the 100,000 of a maze
// of as many cells).  Few pieces, up to two a CTA, go faster by a warp or the
// CTA each (12,000 cells, 400 lookups a node, at p = 12: 1.00 ms, by warps 1.08).
template <bool NIB, class Range, class Done>
__device__ __forceinline__ void code_open_settle(const uint2 *__restrict__ list, uint32_t count, uint32_t cta,
                                                 uint32_t ctas, const Range &range, const uint32_t *__restrict__ lk,
                                                 const uint8_t *__restrict__ cur, uint8_t *__restrict__ nxt,
                                                 uint32_t n, int s_log2, int scheme, OpenShared &sh,
                                                 const Done &done) {
    if (count > 2u * ctas)
        code_open_pieces<NIB, 8, 32, 128>(list, count, cta, ctas, range, lk, cur, nxt, n, s_log2, scheme, sh, done);
    else
        code_open_pieces<NIB, 32, 32, 0>(list, count, cta, ctas, range, lk, cur, nxt, n, s_log2, scheme, sh, done);
}

// Word k of the window of a run (CodeWindow) from the largest rho inserted per
// register index.
__device__ __forceinline__ void window_word(const uint32_t *__restrict__ gmax, uint32_t k, bool nib,
                                            uint32_t *__restrict__ top, uint32_t *__restrict__ low) {
    const int f = nib ? 8 : 4, w = nib ? 4 : 8;
    uint32_t t = 0, l = 0;
    for (int i = 0; i < f; i++) {
        const uint32_t g = gmax[k * f + i];
        t |= g << (w * i);
        l |= (g > 15u ? g - 15u : 0u) << (w * i);  // 0 with 4-bit registers
    }
    top[k] = t;
    low[k] = l;
}

// Fold the code rows of entries buf[lo .. hi) of a staged chunk into acc: the
// lane mapping and the steps of lean_fold.
template <int S, int K>
__device__ __forceinline__ void code_fold(const uint8_t *__restrict__ base, const uint32_t *buf, int lo, int hi, int g,
                                          uint4 (&acc)[LeanShape<S>::V4]) {
    using Sh = LeanShape<S>;
    constexpr int STEP = Sh::P * Sh::U;
    auto step = [&](int kb, bool check) {
        uint32_t r[Sh::U];
        if constexpr (Sh::U == 4) {
            const uint4 t = *reinterpret_cast<const uint4 *>(buf + kb);
            r[0] = t.x;
            r[1] = t.y;
            r[2] = t.z;
            r[3] = t.w;
        } else {
            const uint2 t = *reinterpret_cast<const uint2 *>(buf + kb);
            r[0] = t.x;
            r[1] = t.y;
        }
        uint4 x[Sh::U][Sh::V4];
#pragma unroll
        for (int u = 0; u < Sh::U; u++) {
            if (!check || (kb + u >= lo && kb + u < hi)) {
                load_row_chunk<Sh::V4>(base + (uint64_t)r[u] * S, x[u]);
            } else {
#pragma unroll
                for (int q = 0; q < Sh::V4; q++) x[u][q] = make_uint4(0, 0, 0, 0);
            }
        }
#pragma unroll
        for (int q = 0; q < Sh::V4; q++) {
            uint4 t = code_max<K>(x[0][q], x[1][q]);
            if constexpr (Sh::U == 4) t = code_max<K>(t, code_max<K>(x[2][q], x[3][q]));
            acc[q] = code_max<K>(acc[q], t);
        }
    };
    int k0 = lo & ~(Sh::U - 1);
    if (k0 < lo) {
        const int kb = k0 + g * Sh::U;
        if (kb < hi) step(kb, true);
        k0 += STEP;
    }
    for (; k0 + STEP <= hi; k0 += STEP) step(k0 + g * Sh::U, false);
    if (k0 < hi) {
        const int kb = k0 + g * Sh::U;
        if (kb < hi) step(kb, true);
    }
}

// Fold the warp's P lane groups together (every lane ends with the maximum of
// its part of the row).
template <int S, int K>
__device__ __forceinline__ void code_finish(uint4 (&acc)[LeanShape<S>::V4]) {
    using Sh = LeanShape<S>;
#pragma unroll
    for (int o = Sh::G; o < 32; o <<= 1)
#pragma unroll
        for (int q = 0; q < Sh::V4; q++) {
            uint4 y;
            y.x = __shfl_xor_sync(0xffffffffu, acc[q].x, o);
            y.y = __shfl_xor_sync(0xffffffffu, acc[q].y, o);
            y.z = __shfl_xor_sync(0xffffffffu, acc[q].z, o);
            y.w = __shfl_xor_sync(0xffffffffu, acc[q].w, o);
            acc[q] = code_max<K>(acc[q], y);
        }
}

// Whether every one-bit code of this lane's accumulator is set.
template <int V4>
__device__ __forceinline__ bool code_all_set(const uint4 (&acc)[V4]) {
    uint32_t all = 0xffffffffu;
#pragma unroll
    for (int q = 0; q < V4; q++) all &= acc[q].x & acc[q].y & acc[q].z & acc[q].w;
    return all == 0xffffffffu;
}

// One warp's share of the code maxima of a group's nodes, into part[NODES][S /
// 16]: the group's distinct rows in pieces of `len` entries (a multiple of 4,
// at most kLkChunk) through the warp's TMA stage, this warp taking pieces w, w
// + split, ...  Within a piece the rows of a class fold into one accumulator,
// merged into the class's nodes when the class or the piece ends.  `phase`: the
// stage's barrier phases, kept from one group of the warp to the next.
//
// K = 1: once every bit of a class's accumulator is set, its other rows change
// nothing.  Every kCheck rows the warp looks; a class that is there is cut
// short, one whose nodes are all there is passed over, and the walk ends once
// all nodes are.  The classes come in decreasing mask order, so the rows that
// all nodes share are first.  (K = 4 does not look: after pass 2 only 4 % of
// the city's 256-register rows are at the top throughout, and looking cost
// more than that.)
template <int S, int K, int NODES>
__device__ __forceinline__ void code_group(const GroupItem &gi, const uint32_t *__restrict__ rows,
                                           const uint2 *__restrict__ cls, const uint8_t *__restrict__ tab, uint4 *part,
                                           LkStage &st, uint32_t &phase, int lane, int *err, uint32_t w,
                                           uint32_t split, uint32_t len) {
    using Sh = LeanShape<S>;
    constexpr int W16 = S / 16;
    constexpr int STEP = Sh::P * Sh::U;
    constexpr uint32_t kCheck = STEP > 32 ? STEP : 32;  // rows between two looks at the accumulator
    const uint32_t cnt = gi.cnt;
    const uint32_t pieces = (cnt + len - 1) / len;
    if (w >= pieces) return;
    const uint32_t *src = rows + gi.b;  // 16-byte aligned; readable up to a multiple of 4 entries
    auto load = [&](uint32_t k) {
        const uint32_t s0 = (w + k * split) * len;
        if (s0 < cnt) lk_bulk_load(st, (int)(k & 1u), src + s0, ((min(cnt - s0, len) + 3u) & ~3u) * 4u);
    };
    if (lane == 0) {
        load(0);
        load(1);
    }
    uint4 acc[Sh::V4] = {};
    const int g = lane / Sh::G, sub = lane % Sh::G;
    const uint8_t *base = tab + sub * Sh::CH;
    const uint2 *cp = cls + gi.cls;
    uint2 cd = *cp;         // {node mask, rows} of the current class
    uint32_t cend = cd.y;   // group entry where the current class ends
    uint32_t left = 0;      // nodes of the group not yet at the top (bit j: node j)
#pragma unroll
    for (int j = 0; j < NODES; j++) left |= gi.node[j] != 0xffffffffu ? 1u << j : 0u;
    bool at_top = false;    // K = 1: every bit of the current class's accumulator is set
    auto merge = [&]() {
        if (K != 1 || (cd.x & left)) {
            code_finish<S, K>(acc);
#pragma unroll
            for (int j = 0; j < NODES; j++)
                if ((cd.x >> j) & 1u) {
                    if (g == 0) {
#pragma unroll
                        for (int q = 0; q < Sh::V4; q++) {
                            uint4 &pp = part[j * W16 + sub * Sh::V4 + q];
                            pp = code_max<K>(pp, acc[q]);
                        }
                    }
                }
            if (K == 1 && at_top) left &= ~cd.x;
        }
#pragma unroll
        for (int q = 0; q < Sh::V4; q++) acc[q] = make_uint4(0, 0, 0, 0);
    };
    auto wait = [&](uint32_t k) {
        const int slot = (int)(k & 1u);
        if (!__all_sync(0xffffffffu, lk_wait(st, slot, (phase >> slot) & 1u))) {
            if (lane == 0) atomicExch(err, 1);
            lk_wait(st, slot, (phase >> slot) & 1u);  // give an in-flight copy a last chance
        }
        phase ^= 1u << slot;
    };
    for (uint32_t k = 0;; k++) {
        const uint32_t s0 = (w + k * split) * len;
        if (s0 >= cnt) break;
        wait(k);
        if (K == 1 && !left) break;  // the copy of this piece was the last one in flight
        const uint32_t *buf = st.buf[k & 1u];
        uint32_t lo = s0;
        const uint32_t hi = min(cnt, s0 + len);
        while (cend <= lo) {  // the piece starts in a later class
            cd = *++cp;
            cend += cd.y;
            at_top = false;
        }
        while (lo < hi) {  // warp-uniform: split the piece at class ends
            uint32_t seg = min(hi, cend);
            if (K != 1 || (!at_top && (cd.x & left))) {
                if (K == 1) seg = min(seg, s0 + ((lo - s0) & ~(Sh::U - 1u)) + kCheck);
                code_fold<S, K>(base, buf, (int)(lo - s0), (int)(seg - s0), g, acc);
                if (K == 1) at_top = __all_sync(0xffffffffu, code_all_set<Sh::V4>(acc));
            }
            lo = seg;
            if (lo == cend) {
                merge();
                at_top = false;
                if (lo < cnt) {
                    cd = *++cp;
                    cend += cd.y;
                }
            }
        }
        if (hi < cend && (split > 1u || at_top)) merge();  // goes on in another warp's piece, or is all set
        __syncwarp();
        if (left && lane == 0) load(k + 2u);
    }
}

// Rows [r0, r0 + B) of a code slice's table region (units c0 .. c0 + S / 16 of
// every node) straight from the registers: the rows and their halo are packed
// into `buf` once, then each thread folds the window of one output unit, as in
// table_item.  All threads of the CTA take part.
template <int S, int K, bool NIB>
__device__ void code_table_item(const uint8_t *__restrict__ cur, uint8_t *__restrict__ tab, uint32_t n, int s_log2,
                                uint32_t c0, uint32_t r0, uint8_t *buf, int scheme, const CodeWindow &win) {
    using T = TableShape<S>;
    uint4 *b4 = reinterpret_cast<uint4 *>(buf);
    const uint32_t avail = (n - r0 < (uint32_t)T::R) ? n - r0 : (uint32_t)T::R;
    for (int x = threadIdx.x; x < T::R * T::C16; x += blockDim.x) {
        const uint32_t row = x / T::C16, c = x % T::C16;
        b4[x] = row < avail ? code_pack<K, NIB>(cur, n, s_log2, r0 + row, c0 + c, win) : make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
    for (int x = threadIdx.x; x < T::B * T::C16; x += blockDim.x) {
        const uint32_t row = x / T::C16, c = x % T::C16;
        const uint64_t i = (uint64_t)r0 + row;
        uint4 acc = b4[x];
        if (i < n) reinterpret_cast<uint4 *>(tab + i * S)[c] = acc;
#pragma unroll
        for (int j = 1; j < 16; j++) {
            acc = code_max<K>(acc, b4[x + j * T::C16]);
            if ((j & (j + 1)) == 0) {
                const int k = 31 - __clz(j + 1);
                const bool kept = scheme == 0 || (k & 1) == 0;
                const int slot = scheme == 0 ? k : k / 2;
                if (kept && i + (1u << k) <= n)
                    reinterpret_cast<uint4 *>(tab + ((uint64_t)slot * n + i) * S)[c] = acc;
            }
        }
    }
}

}  // namespace
}  // namespace vga
