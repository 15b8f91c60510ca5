// dfv_gas_f32_k.cu -- launchers of the single-gas FP32 stage kernels: 2-D
// (dfv_gasw.cuh) and 3-D (dfv_gas3.cuh), and the TMA tensor maps the 3-D
// kernel reads its plane boxes through.  Built with the fast single-precision
// divide and square root and flush-to-zero, like the other FP32 kernels.
#include <algorithm>
#include <cstring>

#include <cudaTypedefs.h>

#include "dfv_gas3.cuh"
#include "dfv_gasw.cuh"

namespace dfv {

namespace {

// cuTensorMapEncodeTiled through the runtime's driver entry point (the
// library links the runtime only)
PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            (void)cudaGetLastError();
    }
    return fn;
}

}  // namespace

int gasw_max_ctas_per_sm()
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gasw_stage<3, unsigned>, GaswT::THREADS, 0) != cudaSuccess) {
        (void)cudaGetLastError();
        return 1;
    }
    return n < 1 ? 1 : n;
}

cudaError_t gasw_stage(int stage, const GaswArgs &a, int grid, cudaStream_t st)
{
    const dim3 g(grid < 1 ? 1 : grid), b(GaswT::THREADS);
    if (a.wide) {
        if (stage == 1) return launch_pdl(k_gasw_stage<1, unsigned long long>, g, b, 0, st, a);
        if (stage == 2) return launch_pdl(k_gasw_stage<2, unsigned long long>, g, b, 0, st, a);
        return launch_pdl(k_gasw_stage<3, unsigned long long>, g, b, 0, st, a);
    }
    if (stage == 1) return launch_pdl(k_gasw_stage<1, unsigned>, g, b, 0, st, a);
    if (stage == 2) return launch_pdl(k_gasw_stage<2, unsigned>, g, b, 0, st, a);
    return launch_pdl(k_gasw_stage<3, unsigned>, g, b, 0, st, a);
}

int gasw_rows(long long cells)
{
    // 4-row chunks below 2^19 cells, then 8, growing to at most 32 while at
    // least four items remain per resident warp (152 SMs x 20 warps); 64-row
    // chunks were 2 % slower than 32 on the 256-ellipse batch.  The estimate for
    // one grid below gained 4 % on some batches and lost 5 % on others: grids of
    // several sizes do not end their waves together.
    const long long target = 4LL * 152 * GaswT::MIN_CTAS * GaswT::WARPS;
    int rows = cells < (1LL << 19) ? 4 : 8;
    while (rows < 32 && cells / ((long long)GaswT::OWN * rows * 2) >= target) rows *= 2;
    return rows;
}

int gasw_rows(int n0, int n1)
{
    // The length of the least estimated time l (rows + 2): two rows for a
    // chunk's prologue, l a row's time with the CTAs of the SM that has the most.
    // In one wave (five are resident) l is about the same from three CTAs on and
    // less when one or two leave each warp waiting by itself; every whole wave
    // adds its time, and a last one that begins costs two CTAs more than it has
    // (half a percent over a whole wave is lost in the spread of its ends).
    // Fitted to lengths 1 .. 64 on 22 grids of 64^2 .. 3000 x 2000 cells: within
    // 4 % of the best length's time on each.  us a step with the lengths by the
    // number of cells alone and with these: 64^2 22.6, 16.4; 320^2 28.6, 24.7;
    // 640^2 42.6, 38.3; 1200 x 800 70.0, 67.4; 2048^2 248, 231.
    double least = 1e300;
    int best = 1;
    for (int r = 1; r <= 64; r++) {
        const long long items = (long long)gasw_strips(n0) * ((n1 + r - 1) / r);
        const long long ctas = (items + GaswT::WARPS - 1) / GaswT::WARPS;
        long long per = (ctas + 151) / 152;
        double l;
        if (per <= GaswT::MIN_CTAS) {
            l = std::min((double)per + 3.5, 6.0);
        } else {
            per = std::max<long long>(GaswT::MIN_CTAS + 1, (ctas * 199 / 200 + 151) / 152);
            const long long rest = per % GaswT::MIN_CTAS;
            l = 6.0 * (double)(per / GaswT::MIN_CTAS) + (rest ? (double)rest + 2.0 : 0.0);
        }
        if (l * (r + 2) < least) {
            least = l * (r + 2);
            best = r;
        }
    }
    return best;
}

cudaError_t gas3_prepare()
{
    const int bytes = (int)sizeof(Gas3Smem);
    cudaError_t e = cudaSuccess;
    const void *k[6] = {(const void *)k_gas3_stage<1, true>,  (const void *)k_gas3_stage<2, true>,
                        (const void *)k_gas3_stage<3, true>,  (const void *)k_gas3_stage<1, false>,
                        (const void *)k_gas3_stage<2, false>, (const void *)k_gas3_stage<3, false>};
    for (int i = 0; i < 6 && e == cudaSuccess; i++)
        e = cudaFuncSetAttribute(k[i], cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return e;
}

int gas3_planes(int n0, int n1, int n2)
{
    // The number of the least estimated time l (planes + 2), two planes for a
    // chunk's prologue, l a plane's time with the CTAs of the SM that has the
    // most: nearly the same for one to the three that are resident, a whole
    // wave's for each wave, and one CTA more than it has for a last one that
    // begins.  Large grids keep ZCHUNK, as does a grid that would gain less than
    // 10 % (the estimate's own spread).  Fitted to 2 .. 256 planes on 17 grids:
    // us a step at 24 planes and at these, 40^3 167, 49; 64^3 173, 61;
    // 58 x 155 x 86 289, 135; 97 x 90 x 101 452, 266; 128^3 312, 260.
    const long long cols = (long long)((n0 + Gas3T::TX - 1) / Gas3T::TX) * ((n1 + Gas3T::TY - 1) / Gas3T::TY);
    auto time = [&](int z) {
        const long long per = (cols * ((n2 + z - 1) / z) + 151) / 152;
        const long long full = per / Gas3T::CTAS, rest = per % Gas3T::CTAS;
        const double l = per == 1 ? 2.4 : per == 2 ? 2.8 : 3.0 * (double)full + (rest ? (double)rest + 1.0 : 0.0);
        return l * (z + 2);
    };
    int best = Gas3T::ZCHUNK;
    double least = time(best) / 1.1;
    for (int z = n2 < 2 ? 1 : 2; z <= n2 && z <= 64; z++)
        if (time(z) < least) {
            least = time(z);
            best = z;
        }
    return best;
}

bool gas3_encode_map(CUtensorMap *map, const void *base, int n0, int n1, int n2, long long pitch)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn || n0 % 4 != 0 || pitch % 4 != 0 || ((uintptr_t)base & 15u) != 0) return false;
    using T = Gas3T;
    const cuuint64_t dims[4] = {(cuuint64_t)n0, (cuuint64_t)n1, (cuuint64_t)n2, (cuuint64_t)T::BV};
    const cuuint64_t strides[3] = {(cuuint64_t)n0 * 4u, (cuuint64_t)n0 * (cuuint64_t)n1 * 4u, (cuuint64_t)pitch * 4u};
    const cuuint32_t box[4] = {(cuuint32_t)T::BX, (cuuint32_t)T::BY, 1u, (cuuint32_t)T::BV};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void *>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

cudaError_t gas3_stage(int stage, const Gas3Args &a, const CUtensorMap *map, cudaStream_t st)
{
    const dim3 g((a.n0 + Gas3T::TX - 1) / Gas3T::TX, (a.n1 + Gas3T::TY - 1) / Gas3T::TY, (a.n2 + a.zc - 1) / a.zc);
    const dim3 b(Gas3T::THREADS);
    const size_t sm = sizeof(Gas3Smem);
    if (map) {
        const CUtensorMap m = *map;
        if (stage == 1) return launch_pdl(k_gas3_stage<1, true>, g, b, sm, st, a, m);
        if (stage == 2) return launch_pdl(k_gas3_stage<2, true>, g, b, sm, st, a, m);
        return launch_pdl(k_gas3_stage<3, true>, g, b, sm, st, a, m);
    }
    CUtensorMap none;
    memset(&none, 0, sizeof(none));
    if (stage == 1) return launch_pdl(k_gas3_stage<1, false>, g, b, sm, st, a, none);
    if (stage == 2) return launch_pdl(k_gas3_stage<2, false>, g, b, sm, st, a, none);
    return launch_pdl(k_gas3_stage<3, false>, g, b, sm, st, a, none);
}

}  // namespace dfv
