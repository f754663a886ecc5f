// first_pass.cu -- the grouped scatter of one analysis (first_pass.cuh), one
// CTA per group.
#include "first_pass.cuh"

namespace vga {
namespace {

template <bool NIB, class K>
__global__ void __launch_bounds__(kGroupScatterWarps * 32) hb_first_pass_groups_kernel(
    const GroupItem *__restrict__ items, const uint32_t *__restrict__ rows, const uint2 *__restrict__ cls,
    const K *__restrict__ keys, uint32_t n, int p, int scheme, int s_log2, const uint32_t *__restrict__ gmax,
    const uint32_t *__restrict__ gbig, uint64_t seed, uint8_t *__restrict__ nxt, uint32_t *__restrict__ flags,
    uint8_t *__restrict__ chg) {
    extern __shared__ __align__(16) uint32_t s_cells[];
    __shared__ GroupScatterShared sh;
    first_pass_group<NIB, K>(items[blockIdx.x], rows, cls, keys, n, p, scheme, s_log2, gmax, gbig, seed, nxt, flags,
                             chg, s_cells, sh);
}

template <bool NIB, class K>
int launch(const FirstPassGroups &F) {
    const size_t smem = 8ull << F.p;
    auto kernel = hb_first_pass_groups_kernel<NIB, K>;
    if (smem > (32u << 10)) VGA_CHECK_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kernel<<<(unsigned)F.groups->count, kGroupScatterWarps * 32, smem, F.stream>>>(
        F.groups->items, F.groups->rows, F.groups->cls, static_cast<const K *>(F.keys), F.n, F.p, F.scheme, F.s_log2,
        F.gmax, F.gbig, F.seed, F.nxt, F.flags, F.chg);
    count_launch();
    VGA_CHECK_CUDA(cudaGetLastError());
    return VGA_OK;
}

}  // namespace

int launch_first_pass_groups(const FirstPassGroups &F) {
    if (F.groups->count == 0) return VGA_OK;
    if (F.p <= kGroupKey16MaxP) return F.nib ? launch<true, uint16_t>(F) : launch<false, uint16_t>(F);
    return F.nib ? launch<true, uint32_t>(F) : launch<false, uint32_t>(F);
}

}  // namespace vga
