// codes.cu -- the grouped union over register codes (codes.cuh): per code
// slice, the table of range maxima packed straight from the registers, then
// one warp per group gathering the group's distinct rows.
#include <algorithm>

#include "codes.cuh"

namespace vga {
namespace {

template <int S, int K, bool NIB>
__global__ void __launch_bounds__(256) hb_code_table_kernel(const uint8_t *__restrict__ cur, uint8_t *__restrict__ tab,
                                                            uint32_t n, int s_log2, uint32_t c0, int scheme,
                                                            CodeWindow win) {
    __shared__ __align__(16) uint8_t buf[TableShape<S>::R * S];
    code_table_item<S, K, NIB>(cur, tab, n, s_log2, c0, blockIdx.x * (uint32_t)TableShape<S>::B, buf, scheme, win);
}

// The code union of one slice: `split` warps per group of kCodeNodes nodes
// (CTAs of `split` warps, or of several one-warp groups) gather the code
// maxima of its nodes (code_group), then all their lanes settle next[v] for
// the slice's registers, unit by unit (code_store).  A group whose nodes have
// all their registers at G (full[v], K = 1) has nothing to gather.  Open
// 16-byte register pieces go to the list (the first list_cap of them) and, by
// register slice, to the need masks; flags: [0] a register changed, [2] a
// bounded wait ran out, [8] slices with open pieces, [9] open pieces.
// Bound: the L2 bytes of the rows and the ALU pipe (K = 4: 3.1 ms a city launch
// beside 0.05 of its table, 8 logic operations a 16-byte unit; K = 1: 0.55 ms beside
// 0.17, 2.8 with every row).  One warp
// per group until the groups fill the GPU twice; below that several, which
// took 42,680 cells from 2.19 to 1.85 ms and 4,997 cells at p = 12 from 0.86 to
// 0.74 ms an analysis.  56 registers: measured 25.4 ms on the city against 25.9
// (40 or 64) and 27.7 (48).
template <int S, int K, bool NIB>
__global__ void __maxnreg__(56) hb_code_groups_kernel(
    const GroupItem *__restrict__ items, uint64_t n_items, const uint32_t *__restrict__ rows,
    const uint2 *__restrict__ cls, const uint8_t *__restrict__ cur, const uint8_t *__restrict__ tab,
    uint8_t *__restrict__ nxt, uint32_t n, int s_log2, uint32_t c0, CodeWindow win, uint32_t *__restrict__ flags,
    const uint8_t *__restrict__ full, uint32_t *__restrict__ need, uint8_t *__restrict__ chg,
    uint2 *__restrict__ list, uint32_t list_cap, uint32_t split, uint32_t len) {
    constexpr int W16 = S / 16;
    constexpr int UNIT_BYTES = kUnitRegs<K> / (NIB ? 2 : 1);
    extern __shared__ __align__(128) unsigned char s_dyn[];
    const uint32_t nw = blockDim.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t wib = threadIdx.x >> 5;
    LkStage &st = reinterpret_cast<LkStage *>(s_dyn)[wib];
    uint4 *parts = reinterpret_cast<uint4 *>(s_dyn + (size_t)nw * sizeof(LkStage));
    uint4 *part = parts + (size_t)wib * kCodeNodes * W16;
    const uint64_t item = split > 1u ? blockIdx.x : (uint64_t)blockIdx.x * nw + wib;
    if (item >= n_items) return;  // whole CTAs only when split > 1
    const GroupItem &gi = items[item];
    for (int q = lane; q < kCodeNodes * W16; q += 32) part[q] = make_uint4(0, 0, 0, 0);
    bool gather = true;
    if (K == 1 && full) {
        bool open = false;
#pragma unroll
        for (int j = 0; j < kCodeNodes; j++) {
            const uint32_t v = gi.node[j];
            open |= v != 0xffffffffu && !full[v];
        }
        gather = open;
    }
    __syncwarp();
    if (gather) {
        lk_stage_init(st, lane);
        uint32_t phase = 0;
        code_group<S, K, kCodeNodes>(gi, rows, cls, tab, part, st, phase, lane, reinterpret_cast<int *>(flags + 2),
                                     split > 1u ? wib : 0u, split, len);
    }
    if (split > 1u) __syncthreads();
    else __syncwarp();
    bool changed = false;
    uint32_t open_slices = 0;
    const uint32_t q0 = split > 1u ? threadIdx.x : lane, dq = split > 1u ? blockDim.x : 32u;
    for (uint32_t q = q0; q < (uint32_t)kCodeNodes * W16; q += dq) {
        const uint32_t v = gi.node[q / W16];
        if (v == 0xffffffffu) continue;
        const uint32_t u = c0 + q % W16;
        uint4 code = part[q];
        if (split > 1u) {
            code = parts[q];
            for (uint32_t w = 1; w < split; w++) code = code_max<K>(code, parts[(size_t)w * kCodeNodes * W16 + q]);
        }
        uint32_t chg16, open16;
        code_store<K, NIB>(code, cur, nxt, n, s_log2, v, u, win, chg16, open16);
        changed |= chg16 != 0u;
        uint32_t mine = 0;
#pragma unroll
        for (int h = 0; h < UNIT_BYTES / 16; h++) {
            const uint32_t s = (u * UNIT_BYTES + 16u * h) >> s_log2;
            if (chg && ((chg16 >> h) & 1u)) chg[(uint64_t)s * n + v] = 1u;
            mine |= ((open16 >> h) & 1u) << s;
        }
        if (mine) {
            atomicOr(need + v, mine);
            code_push_open<K, NIB, true>(open16, v, u, list, list_cap, flags + 9);
        }
        open_slices |= mine;
    }
    if (__any_sync(0xffffffffu, changed) && lane == 0) {
        if (*reinterpret_cast<volatile uint32_t *>(flags) == 0u) atomicOr(flags, 1u);
    }
    open_slices = __reduce_or_sync(0xffffffffu, open_slices);
    if (open_slices && lane == 0 &&
        (*reinterpret_cast<volatile uint32_t *>(flags + 8) & open_slices) != open_slices)
        atomicOr(flags + 8, open_slices);
}

// The open pieces of a pass (node, 16-byte register piece), when there are at
// most list_cap: the maximum over the node's neighbours straight from their
// registers (code_open_settle).
// Reading deg(v) pieces costs a 32-byte sector each, far more per register
// than the table's rows, but a handful of open pieces in every slice would
// otherwise cost each slice a table and the whole walk of their groups'
// rows by single warps (city pass 3: 2.4 ms for 0.28 % of the pairs, now 0.1).
template <bool NIB>
__global__ void __launch_bounds__(256, 8) hb_code_open_kernel(const uint2 *__restrict__ list, uint32_t list_cap,
                                                           const uint64_t *__restrict__ lk_off,
                                                           const uint32_t *__restrict__ lk,
                                                           const uint8_t *__restrict__ cur, uint8_t *__restrict__ nxt,
                                                           uint32_t n, int s_log2, int scheme,
                                                           uint32_t *__restrict__ flags, uint8_t *__restrict__ chg) {
    __shared__ OpenShared sh;
    const uint32_t count = flags[9];
    if (count > list_cap) return;
    code_open_settle<NIB>(
        list, count, blockIdx.x, gridDim.x,
        [&](uint32_t v, uint64_t &b, uint64_t &e) {
            b = lk_off[v];
            e = lk_off[v + 1];
        },
        lk, cur, nxt, n, s_log2, scheme, sh,
        [&](uint32_t v, uint32_t byte) {
            if (*reinterpret_cast<volatile uint32_t *>(flags) == 0u) atomicOr(flags, 1u);
            if (chg) chg[(uint64_t)(byte >> s_log2) * n + v] = 1u;
        });
}

// Codes of every node, code slices of 2^cs_log2 bytes a node one after another.
template <int K, bool NIB>
__global__ void __launch_bounds__(256) hb_code_pack_kernel(const uint8_t *__restrict__ cur, uint4 *__restrict__ codes,
                                                           uint32_t n, int s_log2, uint32_t units, int cs_log2,
                                                           CodeWindow win) {
    const uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= (uint64_t)n * units) return;
    const uint32_t v = (uint32_t)(x / units), u = (uint32_t)(x % units);
    codes[reg_at(n, cs_log2, v, 16u * u) / 16u] = code_pack<K, NIB>(cur, n, s_log2, v, u, win);
}

// Ids decoded before their rows are gathered (up to 32 come with a window).
constexpr int kCsrIds = 128;

// The code union of one slice over the neighbour lists, one warp per node: the
// list is decoded 32 bytes at a time (decode_window) into up to kCsrIds ids,
// whose code rows are then folded (code_fold).  K = 1: a node that is at the
// top, or gets there on the way, has nothing more to gather.
// Bound: the L2 bytes of the rows, one per neighbour: half (K = 4) or an eighth
// (K = 1) of what the byte union (hb_union_kernel) reads.  20,011 cells, p = 10,
// d = 5: 4.6 ms an analysis against 21.4 over the bytes.
template <int S, int K, bool NIB>
__global__ void __launch_bounds__(256) hb_code_csr_kernel(const uint64_t *__restrict__ off,
                                                          const uint8_t *__restrict__ bytes,
                                                          const uint8_t *__restrict__ cur,
                                                          const uint8_t *__restrict__ codes, uint8_t *__restrict__ nxt,
                                                          uint32_t n, int s_log2, uint32_t c0, CodeWindow win,
                                                          uint32_t *__restrict__ flags,
                                                          const uint8_t *__restrict__ full, uint8_t *__restrict__ chg,
                                                          uint2 *__restrict__ list, uint32_t list_cap) {
    using Sh = LeanShape<S>;
    constexpr int UNIT_BYTES = kUnitRegs<K> / (NIB ? 2 : 1);
    __shared__ __align__(16) uint32_t s_ids[8][kCsrIds];
    const int lane = threadIdx.x & 31;
    uint32_t *ids = s_ids[threadIdx.x >> 5];
    const uint64_t warp = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (warp >= n) return;
    const uint32_t v = (uint32_t)warp;
    const int g = lane / Sh::G, sub = lane % Sh::G;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const uint8_t *base = codes + sub * Sh::CH;
    uint4 acc[Sh::V4] = {};
    uint64_t pos = off[v];
    const uint64_t end = K == 1 && full[v] ? pos : off[v + 1];
    uint32_t id_base = 0;
    bool at_top = K == 1 && full[v];
    while (pos < end && !at_top) {
        int cnt = 0;
        while (pos < end && cnt <= kCsrIds - 32) {
            const WindowDecode<uint32_t> r = decode_window<uint32_t>(bytes, pos, end, id_base, lane);
            if (r.term_mask == 0) {  // cannot happen on a validated graph; guarantees progress
                pos = end;
                break;
            }
            if ((r.term_mask >> lane) & 1u) ids[cnt + __popc(r.term_mask & lt_mask)] = r.id;
            cnt += __popc(r.term_mask);
            id_base = r.next_base;
            pos += (uint64_t)r.advance;
        }
        __syncwarp();
        code_fold<S, K>(base, ids, 0, cnt, g, acc);
        __syncwarp();
        if (K == 1) at_top = __all_sync(0xffffffffu, code_all_set<Sh::V4>(acc));
    }
    if (K == 1 && full[v]) {  // keeps its registers
#pragma unroll
        for (int q = 0; q < Sh::V4; q++) acc[q] = make_uint4(~0u, ~0u, ~0u, ~0u);
    }
    code_finish<S, K>(acc);
    bool changed = false;
    if (g == 0) {
#pragma unroll
        for (int q = 0; q < Sh::V4; q++) {
            const uint32_t u = c0 + (uint32_t)(sub * Sh::V4 + q);
            uint32_t chg16, open16;
            code_store<K, NIB>(acc[q], cur, nxt, n, s_log2, v, u, win, chg16, open16);
            changed |= chg16 != 0u;
            if (chg) {
#pragma unroll
                for (int h = 0; h < UNIT_BYTES / 16; h++)
                    if ((chg16 >> h) & 1u) chg[(uint64_t)((u * UNIT_BYTES + 16u * h) >> s_log2) * n + v] = 1u;
            }
            if (open16) code_push_open<K, NIB, true>(open16, v, u, list, list_cap, flags + 9);
        }
    }
    if (__any_sync(0xffffffffu, changed) && lane == 0) {
        if (*reinterpret_cast<volatile uint32_t *>(flags) == 0u) atomicOr(flags, 1u);
    }
}

// The open pieces of such a pass, when there are at most list_cap: one warp per
// piece decodes the node's list, a lane per neighbour.
template <bool NIB>
__global__ void __launch_bounds__(256) hb_code_open_csr_kernel(const uint2 *__restrict__ list, uint32_t list_cap,
                                                               const uint64_t *__restrict__ off,
                                                               const uint8_t *__restrict__ bytes,
                                                               const uint8_t *__restrict__ cur,
                                                               uint8_t *__restrict__ nxt, uint32_t n, int s_log2,
                                                               uint32_t *__restrict__ flags,
                                                               uint8_t *__restrict__ chg) {
    const int lane = threadIdx.x & 31;
    const uint32_t count = flags[9];
    if (count > list_cap) return;
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    for (uint32_t e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); e < count; e += warps) {
        const uint32_t v = list[e].x, byte = 16u * list[e].y;
        const uint8_t *base = cur + ((uint64_t)(byte >> s_log2) * n << s_log2) + (byte & ((1u << s_log2) - 1u));
        uint4 acc = make_uint4(0, 0, 0, 0);
        uint64_t pos = off[v];
        const uint64_t end = off[v + 1];
        uint32_t id_base = 0;
        while (pos < end) {
            const WindowDecode<uint32_t> r = decode_window<uint32_t>(bytes, pos, end, id_base, lane);
            if (r.term_mask == 0) break;  // cannot happen on a validated graph; guarantees progress
            if ((r.term_mask >> lane) & 1u)
                acc = RegFmt<NIB>::max4(acc, __ldg(reinterpret_cast<const uint4 *>(base + ((uint64_t)r.id << s_log2))));
            id_base = r.next_base;
            pos += (uint64_t)r.advance;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            uint4 y;
            y.x = __shfl_xor_sync(0xffffffffu, acc.x, o);
            y.y = __shfl_xor_sync(0xffffffffu, acc.y, o);
            y.z = __shfl_xor_sync(0xffffffffu, acc.z, o);
            y.w = __shfl_xor_sync(0xffffffffu, acc.w, o);
            acc = RegFmt<NIB>::max4(acc, y);
        }
        if (lane == 0) {
            const uint64_t at = reg_at(n, s_log2, v, byte);
            const uint4 own = *reinterpret_cast<const uint4 *>(cur + at);
            acc = RegFmt<NIB>::max4(acc, own);
            *reinterpret_cast<uint4 *>(nxt + at) = acc;
            if ((acc.x ^ own.x) | (acc.y ^ own.y) | (acc.z ^ own.z) | (acc.w ^ own.w)) {
                if (*reinterpret_cast<volatile uint32_t *>(flags) == 0u) atomicOr(flags, 1u);
                if (chg) chg[(uint64_t)(byte >> s_log2) * n + v] = 1u;
            }
        }
        __syncwarp();
    }
}

// The window of a run from the largest rho inserted per register index, and its
// counts (launch_code_window): one word of registers a thread.
__global__ void hb_window_kernel(const uint32_t *__restrict__ gmax, uint32_t words, int nib, int s_log2,
                                 uint32_t *__restrict__ top, uint32_t *__restrict__ low,
                                 uint32_t *__restrict__ flags) {
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31u;
    uint32_t idle = 0;
    bool above = false;
    if (k < words) {
        window_word(gmax, k, nib != 0, top, low);
        idle = __popc(nib ? equal_bits<true>(top[k], 0u) : equal_bits<false>(top[k], 0u));
        above = low[k] != 0u;
    }
    const uint32_t any = __ballot_sync(0xffffffffu, above);
    if (lane % 4u == 0u && ((any >> lane) & 0xFu)) {
        atomicAdd(flags + 12, 1u);
        atomicOr(flags + 13, 1u << (((4u * k) >> s_log2) & 31u));
    }
    idle = __reduce_add_sync(0xffffffffu, idle);
    if (lane == 0u && idle) atomicAdd(flags + 14, idle);
}

template <int S, int K, bool NIB>
int launch_slice(const CodePass &C, int slice) {
    const uint32_t c0 = (uint32_t)slice * (S / 16);
    const CodeWindow win{C.top, C.low};
    const unsigned table_blocks = (unsigned)(((uint64_t)C.n + TableShape<S>::B - 1) / TableShape<S>::B);
    hb_code_table_kernel<S, K, NIB><<<table_blocks, 256, 0, C.stream>>>(C.cur, C.tab, C.n, C.s_log2, c0, C.scheme, win);
    count_launch();
    const int warps = C.split > 1 ? C.split : C.warps;
    const size_t smem = (size_t)warps * (sizeof(LkStage) + (size_t)kCodeNodes * S);
    const unsigned blocks = (unsigned)(C.split > 1 ? C.groups->count : (C.groups->count + warps - 1) / warps);
    if (blocks) {
        hb_code_groups_kernel<S, K, NIB><<<blocks, warps * 32, smem, C.stream>>>(
            C.groups->items, C.groups->count, C.groups->rows, C.groups->cls, C.cur, C.tab, C.nxt, C.n, C.s_log2, c0,
            win, C.flags, C.full, C.need, C.chg, C.list, C.list_cap, (uint32_t)C.split, (uint32_t)C.len);
        count_launch();
    }
    VGA_CHECK_CUDA(cudaGetLastError());
    return VGA_OK;
}

template <int S, int K, bool NIB>
void launch_csr_slices(const CodePass &C, uint32_t units, const uint64_t *off, const uint8_t *bytes) {
    const CodeWindow win{C.top, C.low};
    const uint64_t x = (uint64_t)C.n * units;
    hb_code_pack_kernel<K, NIB><<<(unsigned)((x + 255) / 256), 256, 0, C.stream>>>(
        C.cur, reinterpret_cast<uint4 *>(C.tab), C.n, C.s_log2, units, __builtin_ctz((unsigned)S), win);
    count_launch();
    for (uint32_t c0 = 0; c0 < units; c0 += S / 16) {
        hb_code_csr_kernel<S, K, NIB><<<(C.n + 7) / 8, 256, 0, C.stream>>>(
            off, bytes, C.cur, C.tab + (uint64_t)(c0 / (S / 16)) * C.n * S, C.nxt, C.n, C.s_log2, c0, win, C.flags,
            C.full, C.chg, C.list, C.list_cap);
        count_launch();
    }
}

}  // namespace

int launch_code_csr(const CodePass &C, uint32_t m, const uint64_t *off, const uint8_t *bytes, int sms) {
    const uint32_t units = m * (uint32_t)C.K / 128u;
    switch (C.S) {
#define VGA_C(SS)                                                                                              \
    case SS:                                                                                                   \
        if (C.K == 1) C.nib ? launch_csr_slices<SS, 1, true>(C, units, off, bytes) : launch_csr_slices<SS, 1, false>(C, units, off, bytes); \
        else C.nib ? launch_csr_slices<SS, 4, true>(C, units, off, bytes) : launch_csr_slices<SS, 4, false>(C, units, off, bytes);  \
        break;
        VGA_C(16) VGA_C(32) VGA_C(64) VGA_C(128) VGA_C(256) VGA_C(512) VGA_C(1024)
#undef VGA_C
        default:
            set_error("internal: code slice width %d", C.S);
            return VGA_EINVAL;
    }
    const unsigned blocks = (unsigned)std::min<uint32_t>(std::max<uint32_t>(C.list_cap / 8u, 1u), (uint32_t)sms * 8u);
    if (C.nib)
        hb_code_open_csr_kernel<true><<<blocks, 256, 0, C.stream>>>(C.list, C.list_cap, off, bytes, C.cur, C.nxt, C.n,
                                                                   C.s_log2, C.flags, C.chg);
    else
        hb_code_open_csr_kernel<false><<<blocks, 256, 0, C.stream>>>(C.list, C.list_cap, off, bytes, C.cur, C.nxt, C.n,
                                                                    C.s_log2, C.flags, C.chg);
    count_launch();
    VGA_CHECK_CUDA(cudaGetLastError());
    return VGA_OK;
}

int launch_code_slice(const CodePass &C, int slice) {
    switch (C.S) {
#define VGA_C(SS)                                                                              \
    case SS:                                                                                   \
        if (C.K == 1) return C.nib ? launch_slice<SS, 1, true>(C, slice) : launch_slice<SS, 1, false>(C, slice); \
        return C.nib ? launch_slice<SS, 4, true>(C, slice) : launch_slice<SS, 4, false>(C, slice);
        VGA_C(16) VGA_C(32) VGA_C(64) VGA_C(128) VGA_C(256) VGA_C(512) VGA_C(1024)
#undef VGA_C
    }
    set_error("internal: code slice width %d", C.S);
    return VGA_EINVAL;
}

int launch_code_open(const CodePass &C, const uint64_t *lk_off, const uint32_t *lk, int sms) {
    const unsigned blocks = (unsigned)std::min<uint32_t>(std::max<uint32_t>(C.list_cap, 1u), (uint32_t)sms * 8u);
    if (C.nib)
        hb_code_open_kernel<true><<<blocks, 256, 0, C.stream>>>(C.list, C.list_cap, lk_off, lk, C.cur, C.nxt, C.n,
                                                               C.s_log2, C.scheme, C.flags, C.chg);
    else
        hb_code_open_kernel<false><<<blocks, 256, 0, C.stream>>>(C.list, C.list_cap, lk_off, lk, C.cur, C.nxt, C.n,
                                                                C.s_log2, C.scheme, C.flags, C.chg);
    count_launch();
    VGA_CHECK_CUDA(cudaGetLastError());
    return VGA_OK;
}

int launch_code_window(const uint32_t *gmax, uint32_t words, int nib, int s_log2, uint32_t *top, uint32_t *low,
                       uint32_t *flags, cudaStream_t stream) {
    hb_window_kernel<<<(words + 255) / 256, 256, 0, stream>>>(gmax, words, nib, s_log2, top, low, flags);
    count_launch();
    VGA_CHECK_CUDA(cudaGetLastError());
    return VGA_OK;
}

}  // namespace vga
