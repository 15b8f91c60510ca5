// dfv_inst.cuh -- builds the launcher table of one precision; included by
// dfv_inst_f64.cu and dfv_inst_f32.cu with R set to the storage type.
#pragma once

#include "dfv_kernels.cuh"
#include "dfv_kernels_z.cuh"
#include "dfv_ops.h"

namespace dfv {

template <class R, int DIM, int NMAT, int SOLID>
struct Impl {
    using L = Lay<DIM, NMAT, SOLID>;
    // tile sizes that are built: in 2-D FP32 the large one only (a CTA's time is
    // then a chain of dependent work, not the SM's FP64 pipe, and the order of
    // the pressure-force sum, which goes by tiles, stays)
    static constexpr int NV = DIM == 1 || (DIM == 2 && sizeof(R) == 8) ? 2 : 1;

    template <int V>
    static dim3 tile_grid(const GridP &g)
    {
        using TL = Tile<DIM, V>;
        return dim3((g.n[0] + TL::TX - 1) / TL::TX, (g.n[1] + TL::TY - 1) / TL::TY, (g.n[2] + TL::TZ - 1) / TL::TZ);
    }
    template <int V>
    static long long tiles(const GridP &g)
    {
        const dim3 t = tile_grid<V>(g);
        return (long long)t.x * t.y * t.z;
    }

    // Whether the stages run on the small tiles.  A stage takes about as long
    // as the SM with the most tiles, ceil(tiles/SMs) of them; a small tile
    // costs more per cell (halo cells, closing faces), in warps' work 2/9 of
    // the large one in 1-D and 9/16 in 2-D.
    static bool small_tiles(const GridP &g)
    {
        if constexpr (NV == 1) {
            return false;
        } else {
            const long long sms = 152, big = (tiles<0>(g) + sms - 1) / sms, sml = (tiles<1>(g) + sms - 1) / sms;
            return DIM == 1 ? 2 * sml < 9 * big : 9 * sml < 16 * big;
        }
    }

    static dim3 stage_grid(const GridP &g)
    {
        if constexpr (NV == 2)
            if (small_tiles(g)) return tile_grid<1>(g);
        return tile_grid<0>(g);
    }

    template <int V>
    static constexpr size_t smem = StageSmem<R, DIM, NMAT, SOLID, V>::bytes;

    // 3-D single-material fluids march along z (k_stage_z); stage 1 with the
    // pressure force keeps the tiled kernel, whose tiles own the force partials
    static constexpr bool ZM = DIM == 3 && SOLID == 0 && NMAT == 1;
    static constexpr size_t zsmem = ZSmem<R, NMAT>::bytes;

    // Planes per CTA: the chunk count that gives the SM with the most CTAs the
    // least time, a chunk's prologue (two more planes of conversions, one more z
    // slope and face) counted as a plane and a half; among equals the fewest.
    // tail: the time of a last wave that has fewer CTAs than are resident, in
    // full waves' CTAs: an FP64 CTA by itself leaves the pipe a third of its
    // slots, an FP32 one waits most of the time (and a launch of about one CTA
    // an SM may come two to an SM, as it starts while the one before it ends).
    // us over two steps (FP64, at rest) and three (FP32, moving) with every CTA
    // counted alike and with tails: 96^3 9928, 5218 and 1778, 917; 64^3 3561,
    // 1984 and 746, 475; 97 x 90 x 101 6404, 6401 and 2378, 1181.
    static int zchunk(const GridP &g, bool rest)
    {
        using Z = ZGeo<R>;
        const int res = sizeof(R) == 8 ? (rest ? 2 : 1) : 3;
        const double tail[3] = {0.0, sizeof(R) == 8 ? 1.35 : 2.4, 2.8};
        const long long cols = (long long)((g.n[0] + Z::TX - 1) / Z::TX) * ((g.n[1] + Z::TY - 1) / Z::TY);
        double best = -1.0;
        int zbest = g.n[2];
        for (int k = 1; k <= g.n[2] && k <= 64; k++) {
            const int zc = (g.n[2] + k - 1) / k;
            const long long ctas = cols * ((g.n[2] + zc - 1) / zc), per = (ctas + 151) / 152;
            const double cost = ((double)(per / res * res) + tail[per % res]) * (2 * zc + 3);
            if (best < 0.0 || cost < best) {
                best = cost;
                zbest = zc;
            }
        }
        return zbest;
    }

    static dim3 zgrid(const GridP &g, int zc)
    {
        using Z = ZGeo<R>;
        return dim3((g.n[0] + Z::TX - 1) / Z::TX, (g.n[1] + Z::TY - 1) / Z::TY, (g.n[2] + zc - 1) / zc);
    }

    // Opt the stage kernels in to their dynamic shared memory on the current
    // device (called at grid creation, outside any stream capture).
    template <class K>
    static cudaError_t opt_in(K *k, size_t bytes)
    {
        return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    }
    template <int V>
    static cudaError_t prepare_v()
    {
        cudaError_t e = opt_in(k_stage<R, DIM, NMAT, SOLID, 1, V>, smem<V>);
        if constexpr (!ZM) {
            if (e == cudaSuccess) e = opt_in(k_stage<R, DIM, NMAT, SOLID, 2, V>, smem<V>);
            if (e == cudaSuccess) e = opt_in(k_stage<R, DIM, NMAT, SOLID, 3, V>, smem<V>);
        }
        // the first-wave size is looked up here, outside any stream capture
        if (e == cudaSuccess) (void)first_wave<V>();
        return e;
    }
    static cudaError_t prepare()
    {
        cudaError_t e = prepare_v<0>();
        if constexpr (NV == 2)
            if (e == cudaSuccess) e = prepare_v<1>();
        if constexpr (ZM) {
            if (e == cudaSuccess) e = opt_in(k_stage_z<R, NMAT, 1, false>, zsmem);
            if (e == cudaSuccess) e = opt_in(k_stage_z<R, NMAT, 2, false>, zsmem);
            if (e == cudaSuccess) e = opt_in(k_stage_z<R, NMAT, 3, false>, zsmem);
            if (e == cudaSuccess) e = opt_in(k_stage_z<R, NMAT, 1, true>, zsmem);
            if (e == cudaSuccess) e = opt_in(k_stage_z<R, NMAT, 2, true>, zsmem);
            if (e == cudaSuccess) e = opt_in(k_stage_z<R, NMAT, 3, true>, zsmem);
        }
        return e;
    }

    template <int S, int V>
    static cudaError_t stage_v(const GridP &g, StageArgs a, cudaStream_t st)
    {
        a.early = S == 1 ? first_wave<V>() : 0;
        a.late = late<V>(g);
        return launch_pdl(k_stage<R, DIM, NMAT, SOLID, S, V>, tile_grid<V>(g), dim3(Tile<DIM, V>::THREADS), smem<V>, st,
                          a, g);
    }

    template <int S>
    static cudaError_t march(const GridP &g, const StageArgs &a, cudaStream_t st)
    {
        const int zc = zchunk(g, a.rest);
        const dim3 b(ZGeo<R>::THREADS);
        return a.rest ? launch_pdl(k_stage_z<R, NMAT, S, true>, zgrid(g, zc), b, zsmem, st, a, g, zc)
                      : launch_pdl(k_stage_z<R, NMAT, S, false>, zgrid(g, zc), b, zsmem, st, a, g, zc);
    }

    template <int S>
    static cudaError_t stage_s(const GridP &g, const StageArgs &a, cudaStream_t st)
    {
        if constexpr (ZM && S != 1) {
            return march<S>(g, a, st);
        } else {
            if constexpr (ZM)
                if (!a.want_force) return march<S>(g, a, st);
            if constexpr (NV == 2)
                if (small_tiles(g)) return stage_v<S, 1>(g, a, st);
            return stage_v<S, 0>(g, a, st);
        }
    }

    // CTAs of the stage-1 kernel resident at once on the device (the first
    // wave), looked up once
    template <int V>
    static int first_wave()
    {
        static int n = -1;
        if (n < 0) {
            int dev = 0, sms = 0, per = 0;
            if (cudaGetDevice(&dev) != cudaSuccess ||
                cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_stage<R, DIM, NMAT, SOLID, 1, V>,
                                                              Tile<DIM, V>::THREADS, smem<V>) != cudaSuccess) {
                (void)cudaGetLastError();
                return 0;
            }
            n = sms * per;
        }
        return n;
    }

    // Whether the next launch has to wait for the end of this one.  Started at
    // once, its CTAs take the slots that are free while this one's still run:
    // two to an SM that this one left empty, none to others.  That doubles a
    // stage's time where few CTAs share an SM, not where half of the SMs hold
    // them all or most slots are taken anyway, nor in FP32 1-D, whose stages
    // are shorter than the start that is then waited for.  us of five steps with
    // the next launch at once and late: cylinder 150 x 140 FP64 832, 636; 200 x
    // 190 953, 817; two-fluid 220 x 120 FP64 (four) 1466, 1197, 300 x 170 FP32
    // 394, 374; 260 x 250 (567 tiles of 608 slots) 904, 912 without the bound.
    template <int V>
    static bool late(const GridP &g)
    {
        const long long t = tiles<V>(g);
        return (DIM > 1 || sizeof(R) == 8) && 2 * t > 152 && 4 * t <= 3LL * first_wave<V>();
    }

    // next: the seeding before stage 1 reads its box from ctl->rnext;
    // flags: bit 0 the pressure force is wanted, bit 1 the body is at rest
    static cudaError_t stage(int s, const GridP &g, const void *in, const void *un, void *out, Ctl *ctl,
                             double *partials, int flags, int next, cudaStream_t st)
    {
        StageArgs a;
        a.in = in;
        a.un = un;
        a.out = out;
        a.ctl = ctl;
        a.partials = partials;
        a.want_force = flags & 1;
        a.rest = flags >> 1 & 1;
        a.early = 0;   // set with the tile size
        a.next = next;
        a.late = 0;    // likewise
        if (s == 1) return stage_s<1>(g, a, st);
        if (s == 2) return stage_s<2>(g, a, st);
        return stage_s<3>(g, a, st);
    }

    template <int OPT>
    static cudaError_t seed_opt_k(const GridP &g, void *U, void *scratch, Ctl *ctl, int fin_mode, cudaStream_t st)
    {
        dim3 block, grid;
        seed_grid(g, block, grid);
        if (g.probe_mode == 1) {
            cudaError_t e = launch_pdl(k_seed<R, DIM, NMAT, SOLID, OPT, 1>, grid, block, 0, st, U, scratch, ctl, g, 0);
            if (e != cudaSuccess) return e;
            return launch_pdl(k_seed<R, DIM, NMAT, SOLID, 0, 2>, grid, block, 0, st, U, scratch, ctl, g, 0);
        }
        if (fin_mode) grid.x += 1;   // the block that runs the deferred finalize
        return launch_pdl(k_seed<R, DIM, NMAT, SOLID, OPT, 0>, grid, block, 0, st, U, scratch, ctl, g, fin_mode);
    }

    // seeding; scratch: planes of the grid's layout free until stage 1;
    // fin_mode: the deferred finalize of the previous step (stepped probe
    // only), 0 for none
    static cudaError_t seed(const GridP &g, void *U, void *scratch, Ctl *ctl, int fin_mode, cudaStream_t st)
    {
        switch (seed_opt(g)) {
        case 0: return seed_opt_k<0>(g, U, scratch, ctl, fin_mode, st);
        case 1: return seed_opt_k<1>(g, U, scratch, ctl, fin_mode, st);
        case 2: return seed_opt_k<2>(g, U, scratch, ctl, fin_mode, st);
        default: return seed_opt_k<3>(g, U, scratch, ctl, fin_mode, st);
        }
    }

    static cudaError_t cfl(const GridP &g, const void *U, double *partials, int nblocks, cudaStream_t st)
    {
        k_cfl<R, DIM, NMAT, SOLID><<<nblocks, 256, 0, st>>>(U, partials, g);
        return cudaGetLastError();
    }

    static cudaError_t p2c(const GridP &g, const double *prim, long long pp, void *U, cudaStream_t st)
    {
        k_prim_to_cons<R, DIM, NMAT, SOLID><<<gs_blocks(g.ncell), 256, 0, st>>>(prim, pp, U, g);
        return cudaGetLastError();
    }

    static cudaError_t c2p(const GridP &g, const void *U, double *prim, long long pp, cudaStream_t st)
    {
        k_cons_to_prim<R, DIM, NMAT, SOLID><<<gs_blocks(g.ncell), 256, 0, st>>>(U, prim, pp, g);
        return cudaGetLastError();
    }

    static cudaError_t c2f(const GridP &g, const void *U, double *o, long long pp, int nvar, cudaStream_t st)
    {
        k_cons_to_f64<R><<<gs_blocks(g.ncell), 256, 0, st>>>(U, o, pp, nvar, g);
        return cudaGetLastError();
    }

    static const Ops *ops()
    {
        static const Ops o = {L::NVAR, Tile<DIM, 0>::THREADS, (int)sizeof(R), &prepare, &stage_grid, &seed, &stage, &cfl,
                              &p2c, &c2p, &c2f};
        return &o;
    }
};

// Tables of one (precision, dimension, materials): fluids, solids and solids
// with plastic-strain planes.  Not built are 3-D solids and the 3-D FP64
// three-material fluid, whose tile exceeds a CTA's shared memory; every other
// form is, and a tile that grows beyond it fails the build.
template <class R, int DIM, int NMAT>
const Ops *select_ops_nmat(int solid)
{
    if constexpr (!(sizeof(R) == 8 && DIM == 3 && NMAT == 3)) {
        static_assert(StageSmem<R, DIM, NMAT, 0, 0>::bytes <= SMEM_CTA, "a fluid's tile fits a CTA");
        if (!solid) return Impl<R, DIM, NMAT, 0>::ops();
    }
    if constexpr (DIM <= 2) {
        static_assert(StageSmem<R, DIM, NMAT, 1, 0>::bytes <= SMEM_CTA, "a solid's tile fits a CTA");
        static_assert(StageSmem<R, DIM, NMAT, 2, 0>::bytes <= SMEM_CTA, "a tile with plastic strains fits a CTA");
        if (solid == 1) return Impl<R, DIM, NMAT, 1>::ops();
        if (solid == 2) return Impl<R, DIM, NMAT, 2>::ops();
    }
    return nullptr;
}

}  // namespace dfv
