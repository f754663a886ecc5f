// codes.cu -- the grouped union over register codes (codes.cuh): per code
// slice, the table of range maxima packed straight from the registers, then
// one warp per group gathering the group's distinct rows.
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

// One warp per group of kCodeNodes nodes: the code maxima of its nodes over
// one code slice (code_group), then next[v] for the slice's registers
// (code_store), all lanes on the group's (node, unit) pairs.  A group whose
// nodes have all their registers at G (full[v], K = 1) has nothing to gather.
// Open pairs go to the need masks; flags: [0] a register changed, [2] a
// bounded wait ran out, [8] slices with open pairs, [9] open (group, slice)
// pairs.
template <int S, int K, bool NIB>
__global__ void __launch_bounds__(128) hb_code_groups_kernel(
    const GroupItem *__restrict__ items, uint64_t n_items, const uint32_t *__restrict__ rows,
    const uint2 *__restrict__ cls, const uint8_t *__restrict__ cur, const uint8_t *__restrict__ tab,
    uint8_t *__restrict__ nxt, uint32_t n, int s_log2, uint32_t c0, CodeWindow win, uint32_t *__restrict__ flags,
    const uint8_t *__restrict__ full, uint32_t *__restrict__ need, uint8_t *__restrict__ chg) {
    constexpr int W16 = S / 16;
    constexpr int UNIT_BYTES = kUnitRegs<K> / (NIB ? 2 : 1);
    extern __shared__ __align__(128) unsigned char s_dyn[];
    const int nw = blockDim.x >> 5;
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    LkStage &st = reinterpret_cast<LkStage *>(s_dyn)[wib];
    uint4 *part = reinterpret_cast<uint4 *>(s_dyn + (size_t)nw * sizeof(LkStage)) + (size_t)wib * kCodeNodes * W16;
    const uint64_t warp = (uint64_t)blockIdx.x * nw + wib;
    if (warp >= n_items) return;
    const GroupItem &gi = items[warp];
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
        code_group<S, K, kCodeNodes>(gi, rows, cls, tab, part, st, phase, lane, reinterpret_cast<int *>(flags + 2));
        __syncwarp();
    }
    bool changed = false;
    uint32_t open_slices = 0;
    for (int q = lane; q < kCodeNodes * W16; q += 32) {
        const uint32_t v = gi.node[q / W16];
        if (v == 0xffffffffu) continue;
        const uint32_t u = c0 + (uint32_t)(q % W16);
        uint32_t chg16, open16;
        code_store<K, NIB>(part[q], cur, nxt, n, s_log2, v, u, win, chg16, open16);
        changed |= chg16 != 0u;
        uint32_t mine = 0;
#pragma unroll
        for (int h = 0; h < UNIT_BYTES / 16; h++) {
            const uint32_t s = (u * UNIT_BYTES + 16u * h) >> s_log2;
            if (chg && ((chg16 >> h) & 1u)) chg[(uint64_t)s * n + v] = 1u;
            mine |= ((open16 >> h) & 1u) << s;
        }
        if (mine) atomicOr(need + v, mine);
        open_slices |= mine;
    }
    if (__any_sync(0xffffffffu, changed) && lane == 0) {
        if (*reinterpret_cast<volatile uint32_t *>(flags) == 0u) atomicOr(flags, 1u);
    }
    open_slices = __reduce_or_sync(0xffffffffu, open_slices);
    if (open_slices && lane == 0) {
        if ((*reinterpret_cast<volatile uint32_t *>(flags + 8) & open_slices) != open_slices)
            atomicOr(flags + 8, open_slices);
        atomicAdd(flags + 9, (uint32_t)__popc(open_slices));
    }
}

// The window of a run from the largest rho inserted per register index: one
// word of registers a thread.
__global__ void hb_window_kernel(const uint32_t *__restrict__ gmax, uint32_t words, int nib, uint32_t *__restrict__ top,
                                 uint32_t *__restrict__ low) {
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= words) return;
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

template <int S, int K, bool NIB>
int launch_slice(const CodePass &C, int slice) {
    const uint32_t c0 = (uint32_t)slice * (S / 16);
    const CodeWindow win{C.top, C.low};
    const unsigned table_blocks = (unsigned)(((uint64_t)C.n + TableShape<S>::B - 1) / TableShape<S>::B);
    hb_code_table_kernel<S, K, NIB><<<table_blocks, 256, 0, C.stream>>>(C.cur, C.tab, C.n, C.s_log2, c0, C.scheme, win);
    count_launch();
    const size_t smem = (size_t)C.warps * (sizeof(LkStage) + (size_t)kCodeNodes * S);
    auto kernel = hb_code_groups_kernel<S, K, NIB>;
    const unsigned blocks = (unsigned)((C.groups->count + C.warps - 1) / C.warps);
    if (blocks) {
        kernel<<<blocks, C.warps * 32, smem, C.stream>>>(C.groups->items, C.groups->count, C.groups->rows,
                                                         C.groups->cls, C.cur, C.tab, C.nxt, C.n, C.s_log2, c0, win,
                                                         C.flags, C.full, C.need, C.chg);
        count_launch();
    }
    VGA_CHECK_CUDA(cudaGetLastError());
    return VGA_OK;
}

}  // namespace

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

int launch_code_window(const uint32_t *gmax, uint32_t words, int nib, uint32_t *top, uint32_t *low,
                       cudaStream_t stream) {
    hb_window_kernel<<<(words + 255) / 256, 256, 0, stream>>>(gmax, words, nib, top, low);
    count_launch();
    VGA_CHECK_CUDA(cudaGetLastError());
    return VGA_OK;
}

}  // namespace vga
