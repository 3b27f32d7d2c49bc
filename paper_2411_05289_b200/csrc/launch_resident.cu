// Verification with the exponentials resident on chip.
#include "spechub_launch.h"
#include "spechub_resident.cuh"
#include "spechub_resident_kary.cuh"

namespace spechub {

// A row is spread over `cs` CTAs of 8 warps; every lane keeps `nb` batches of four 16-byte vectors of the row
// pair as fp32 exponentials (tensor memory, shared memory, registers).  The smallest cluster that holds the
// row with at most four batches per lane is taken.
bool resident_fits(int vocab, ResShape *out) {
    const int nvec = vocab / 8;
    for (int cs = 1; cs <= 8; cs *= 2) {
        const int parts = cs * kResWarps;
        const int seg = (((nvec + parts - 1) / parts) + 7) & ~7;   // vectors per warp, as the kernel cuts them
        const int nb = (seg + 127) / 128;
        if (nb <= kResMaxBatches) { out->cs = cs; out->nb = nb; return true; }
    }
    return false;
}

template <int MASK, int CS>
static int launch_resident_one(int nb, const FusedArgs &f, unsigned rows, cudaStream_t s) {
    auto kern = resident_verify_kernel<MASK, CS>;
    // tensor-memory columns of a CTA: two warps share each lane quarter, 32 columns per batch each
    const uint32_t cols = nb == 1 ? 64u : nb == 2 ? 128u : 256u;
    // Shared memory: e_q of all batches but the last.  A CTA that takes 256 columns asks for at least a
    // third of an SM's shared memory, so that no more than two such CTAs share the SM's 512 columns.
    int smem = (nb - 1) * 4 * 2 * kResThreads * 16;
    if (cols == 256u && smem < 76 * 1024) smem = 76 * 1024;
    constexpr int smem_max = (kResMaxBatches - 1) * 4 * 2 * kResThreads * 16;
    static bool configured[kMaxDevices] = {};
    const int rc = allow_smem(reinterpret_cast<const void *>(kern), smem_max, configured);
    if (rc != SPECHUB_OK) return rc;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = CS > 1 ? 1 : 0;
    cfg.gridDim = dim3(rows * CS); cfg.blockDim = dim3(kResThreads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    return launch_status(cudaLaunchKernelEx(&cfg, kern, f, nb, cols));
}

template <int MASK>
static int launch_resident_mask(ResShape sh, const FusedArgs &f, unsigned rows, cudaStream_t s) {
    if (sh.cs == 1) return launch_resident_one<MASK, 1>(sh.nb, f, rows, s);
    if (sh.cs == 2) return launch_resident_one<MASK, 2>(sh.nb, f, rows, s);
    if (sh.cs == 4) return launch_resident_one<MASK, 4>(sh.nb, f, rows, s);
    return launch_resident_one<MASK, 8>(sh.nb, f, rows, s);
}

// Algorithm 1 with k > 2 drafts: the stages run over the exponentials kept on chip
template <int CS>
static int launch_resident_kary_one(int nb, const KaryArgs &ka, unsigned rows, cudaStream_t s) {
    auto kern = resident_kary_kernel<CS>;
    const uint32_t cols = nb == 1 ? 64u : nb == 2 ? 128u : 256u;
    int smem = (nb - 1) * 4 * 2 * kResThreads * 16;
    if (cols == 256u && smem < 76 * 1024) smem = 76 * 1024;   // at most two CTAs of 256 columns per SM
    constexpr int smem_max = (kResMaxBatches - 1) * 4 * 2 * kResThreads * 16;
    static bool configured[kMaxDevices] = {};
    const int rc = allow_smem(reinterpret_cast<const void *>(kern), smem_max, configured);
    if (rc != SPECHUB_OK) return rc;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = CS > 1 ? 1 : 0;
    cfg.gridDim = dim3(rows * CS); cfg.blockDim = dim3(kResThreads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    return launch_status(cudaLaunchKernelEx(&cfg, kern, ka, nb, cols));
}

int launch_resident_kary(ResShape sh, const KaryArgs &ka, unsigned rows, cudaStream_t s) {
    if (sh.cs == 1) return launch_resident_kary_one<1>(sh.nb, ka, rows, s);
    if (sh.cs == 2) return launch_resident_kary_one<2>(sh.nb, ka, rows, s);
    if (sh.cs == 4) return launch_resident_kary_one<4>(sh.nb, ka, rows, s);
    return launch_resident_kary_one<8>(sh.nb, ka, rows, s);
}

// mask: bit m set = method m (0 SpecHub, 1 RRS, 2 RRSw) is verified; leaf rows go to lean_leaf_kernel
int launch_resident(int mask, ResShape sh, const FusedArgs &f, unsigned rows, cudaStream_t s) {
    if (f.r.node_kind) {
        NodeOutPtrs outs[3];
        int n_out = 0;
        for (int m = 0; m < 3; ++m)
            if (mask & (1 << m)) outs[n_out++] = f.out[m];
        const int lrc = launch_lean_leaf(kBf16, f.r, 2, outs, n_out, rows, s);
        if (lrc != SPECHUB_OK) return lrc;
    }
    if (mask == kMaskSpecHub) return launch_resident_mask<kMaskSpecHub>(sh, f, rows, s);
    if (mask == kMaskRRS) return launch_resident_mask<kMaskRRS>(sh, f, rows, s);
    if (mask == kMaskRRSw) return launch_resident_mask<kMaskRRSw>(sh, f, rows, s);
    return launch_resident_mask<7>(sh, f, rows, s);
}

}  // namespace spechub
