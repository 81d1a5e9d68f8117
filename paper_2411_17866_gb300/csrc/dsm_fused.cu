// Host side of the fused round (DSM_FLAG_FUSED_ROUND): which kernel, how much
// shared memory, the launch.  The kernel is in dsm_fused.cuh.

#include <algorithm>

#include "dsm_fused.cuh"

namespace dsm {
namespace {

int fused_global_for(const Problem& p) {
    return p.global_mode == 0 ? kGlobalSign : (p.global_mode == 4 ? kGlobalAdamW : kGlobalRuntime);
}

FusedKernel fused_kernel_for(const Problem& p, bool adamw) {
    switch (fused_global_for(p)) {
        case kGlobalSign: return fused_kernel_sign(p, adamw);
        case kGlobalAdamW: return fused_kernel_adamw(p, adamw);
        default: return fused_kernel_variants(p, adamw);
    }
}

size_t fused_smem_for(const Problem& p, bool adamw) {
    return fused_smem(adamw, p.grad_bf16 != 0, int(p.n), fused_global_for(p));
}

}  // namespace

bool fused_round_available(const Problem& p) {
    // every global step, up to 8 workers (the differences x - x_i of all workers stay in registers)
    return p.global_mode >= 0 && p.global_mode <= 4 && p.n >= 1 && p.n <= kMaxUnrolledWorkers;
}

cudaError_t query_fused_shape(const Problem& p, const TensorDesc* tensors, LaunchShape* out) {
    if (!fused_round_available(p)) return cudaSuccess;
    const FusedKernel fk = fused_kernel_for(p, p.opt_v != nullptr);
    const size_t smem = fused_smem_for(p, p.opt_v != nullptr);
    cudaError_t e = cudaFuncSetAttribute(fk, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    out->grid_fused = grid_for(fk, out->sms, smem);
    // AdamW with 2 to 4 workers on more than L2 holds streams better with 2 CTAs per SM (rounds of two steps, us, 2 / 3
    // CTAs: 184 M parameters, fp32, n = 2 3152 / 3256, n = 3 4434 / 4558, n = 4 5769 / 5862, slower with any number in
    // between; n = 4, 1.6 M 49.3 / 46.6, 1.9 M 63.7 / 61.4, 2.2 M 76.0 / 76.0, 3 M 102 / 104; n = 2, 3 M 49.1 / 46.8,
    // 3.7 M 67.7 / 69.0).  Not so n = 1, n >= 5, SGD-momentum and the global AdamW step.
    // Nor where more than a third of the tiles end a CTA's run of one tensor, each with a reduction of its statistics
    // that the other CTAs of the SM run on through.  Models of equal tensors, by the share of such tiles, 2 / 3 CTAs:
    // n = 2, 60 M, bf16 gradients 0.6 1047 / 1005, 0.34 993 / 978, 0.25 978 / 987, 0.15 959 / 987; n = 4, 30 M, bf16
    // 0.6 889 / 875, 0.34 873 / 877, 0.25 882 / 890; n = 4, 120 M, bf16 0.5 3555 / 3554, 0.34 3518 / 3560; n = 4, 30
    // M, fp32 1.0 985 / 967, 0.6 927 / 942.
    // (The line in bytes lies a little above L2, 129 MB, between the sizes above.)
    const uint64_t bytes = p.d_stride * (uint64_t(p.n) * (12 + (p.grad_bf16 ? 2 : 4)) + 8);
    if (p.opt_v && p.n >= 2 && p.n <= 4 && p.global_mode != 4 && bytes > 150000000ull) {
        const uint32_t two = 2 * static_cast<uint32_t>(out->sms);
        uint64_t runs = 0;
        for (uint32_t t = 0; t < p.num_tensors; ++t) runs += std::min(tensors[t].tile_end - tensors[t].tile_begin, two);
        if (3 * runs <= p.num_tiles) out->grid_fused = std::min(out->grid_fused, static_cast<int>(two));
    }
    return cudaSuccess;
}

cudaError_t launch_fused_last_global(const Problem& p, const LaunchShape& ls, const AdamScalars& a,
                                     const SgdmScalars& sa, const GlobalScalars& g, int opts, cudaStream_t s,
                                     uint32_t* grid_used) {
    if (!fused_round_available(p)) return cudaErrorInvalidValue;
    const int grid = clamp_grid(ls.grid_fused, p.num_tiles);
    *grid_used = static_cast<uint32_t>(grid);
    if (grid == 0) return cudaSuccess;
    const bool adamw = p.opt_v != nullptr;
    return launch(fused_kernel_for(p, adamw), grid, kThreads, fused_smem_for(p, adamw), s, p.early, p, a, sa, g, opts);
}

}  // namespace dsm
