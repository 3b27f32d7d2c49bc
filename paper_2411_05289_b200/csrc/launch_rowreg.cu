// Rows held in registers: calls whose rows do not fill the GPU.
#include "spechub_launch.h"
#include "spechub_rowreg.cuh"

namespace spechub {

// Warps of the whole call up to which these kernels are the faster ones, on rows of several warps (V = 2056 .. 128256,
// both types).  Draft step: one wave, 16 per SM (7 x batch rows of 32000 bf16 ids: 56 rows 8.7 us, streaming 9.7; 112
// rows 10.9, 9.3).  Verification: 20 per SM (32000 fp32 ids, 56 rows 12.3 us, streaming 14.3; 112 rows 18.3, 14.3), and
// 25 while the streaming kernels, one CTA per row, leave half of the SMs without a row (128256 bf16 ids, 56 rows: SpecHub
// 22.6 us, streaming 27.7; RRSw 24.6, 35.3); 24 with more than two drafts, whose streaming kernels read the rows more
// often (k = 3, 208 rows of 32000 bf16 ids: RRSw 27.9 us, streaming 35.7).
constexpr long long max_warps(bool verify, int k, long long rows) {
    return 148 * (!verify ? 16 : rows <= 148 / 2 ? 25 : k > 2 ? 24 : 20);
}

bool reg_plan(bool verify, int dtype, int k, int vocab, long long rows, RegPlan *out) {
    const int nvec = (vocab + 7) / 8, max_nv = dtype == SPECHUB_BF16 ? 8 : 4;
    RegPlan p = {};
    // as many warps per row as one wave holds (16 per SM): the fewest vectors per lane that allow it, or that give the
    // row to one warp (longer vectors take registers, so warps, for nothing: 7168 rows of 1000 bf16 ids, verification
    // with 8 / 4 vectors per lane 33.4 / 26.9 us, draft step 21.5 / 18.9)
    for (p.nv = 1;; p.nv *= 2) {
        const int parts = (nvec + 32 * p.nv - 1) / (32 * p.nv);
        if (parts > kRegMaxParts && p.nv == max_nv) return false;
        if (parts > 64 && p.nv < max_nv) continue;   // (fewer records to merge)
        p.cs = 1;
        while (p.cs * 8 < parts && p.cs < 8) p.cs *= 2;   // CTAs of up to 8 warps measured as good as 4 and better than 16
        p.w = (parts + p.cs - 1) / p.cs;
        if (p.w == 3) p.w = 4;
        if (p.nv == max_nv || parts == 1 || rows * p.w * p.cs <= 16 * 148) break;
    }
    p.rows_per_cta = p.w <= 2 ? 4 / p.w : 1;
    p.seg = (nvec + p.w * p.cs - 1) / (p.w * p.cs);
    *out = p;
    // rows of one warp (verification of bf16 rows: of two) are the faster ones here however many they are (7168 rows,
    // bf16 V = 2056, verification: SpecHub 65.9 us, streaming 85.8; V = 4096: 86.9, 99.3)
    const int few = verify && dtype == SPECHUB_BF16 ? 2 : 1, warps = p.w * p.cs;
    return warps <= few || rows * warps <= max_warps(verify, k, rows);
}

template <class K, class... Args>
static int launch(const RegPlan &pl, K kern, unsigned rows, cudaStream_t s, Args... args) {
    const RegGeo geo = {pl.w, pl.cs, pl.rows_per_cta, pl.seg};
    return launch_grid(kern, pl.cs > 1 ? rows * pl.cs : (rows + pl.rows_per_cta - 1) / pl.rows_per_cta,
                       pl.w * pl.rows_per_cta * 32, 0, pl.cs, s, args..., rows, geo);
}

template <typename LT, int NV>
static int draft(const RegPlan &pl, const KaryArgs &a, int method, unsigned rows, cudaStream_t s) {
    if (a.k == 2) return launch(pl, reg_draft_kernel<LT, NV, 2>, rows, s, a, method);
    return launch(pl, reg_draft_kernel<LT, NV, 0>, rows, s, a, method);
}
template <typename LT, int NV>
static int verify(const RegPlan &pl, const KaryArgs &a, int method, unsigned rows, cudaStream_t s) {
    if (method == kSpecHub) return launch(pl, reg_verify_spechub_kernel<LT, NV>, rows, s, a.r);
    if (a.k == 2) return launch(pl, reg_verify_rrs_kernel<LT, NV, 2>, rows, s, a);
    if (a.k == 3) return launch(pl, reg_verify_rrs_kernel<LT, NV, 3>, rows, s, a);
    if (a.k == 4) return launch(pl, reg_verify_rrs_kernel<LT, NV, 4>, rows, s, a);
    return launch(pl, reg_verify_rrs_kernel<LT, NV, 0>, rows, s, a);
}

template <typename LT>
static int draft_nv(const RegPlan &pl, const KaryArgs &a, int method, unsigned rows, cudaStream_t s) {
    if (pl.nv == 1) return draft<LT, 1>(pl, a, method, rows, s);
    if (pl.nv == 2) return draft<LT, 2>(pl, a, method, rows, s);
    if (pl.nv == 4) return draft<LT, 4>(pl, a, method, rows, s);
    return draft<LT, sizeof(LT) == 2 ? 8 : 4>(pl, a, method, rows, s);
}
template <typename LT>
static int verify_nv(const RegPlan &pl, const KaryArgs &a, int method, unsigned rows, cudaStream_t s) {
    if (pl.nv == 1) return verify<LT, 1>(pl, a, method, rows, s);
    if (pl.nv == 2) return verify<LT, 2>(pl, a, method, rows, s);
    if (pl.nv == 4) return verify<LT, 4>(pl, a, method, rows, s);
    return verify<LT, sizeof(LT) == 2 ? 8 : 4>(pl, a, method, rows, s);
}

int launch_reg_draft(const RegPlan &pl, int dtype, const KaryArgs &a, int method, unsigned rows, cudaStream_t s) {
    return dtype == SPECHUB_BF16 ? draft_nv<__nv_bfloat16>(pl, a, method, rows, s) : draft_nv<float>(pl, a, method, rows, s);
}
int launch_reg_verify(const RegPlan &pl, int dtype, const KaryArgs &a, int method, unsigned rows, cudaStream_t s) {
    return dtype == SPECHUB_BF16 ? verify_nv<__nv_bfloat16>(pl, a, method, rows, s) : verify_nv<float>(pl, a, method, rows, s);
}

}  // namespace spechub
