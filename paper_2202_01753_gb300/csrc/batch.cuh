// batch.cuh -- the persistent batched sampling kernels: one launch per class
// of integrals (integrand family x dimension) samples one
// iteration of every live integral of that class.  The host lays the class's
// live integrals' samples end to end and cuts that line into one equal,
// cube-aligned chunk per block; a block therefore samples a few segments
// (runs of cubes of one integral each), in order.  Per segment it stages that
// integral's grid and family constants in shared memory, samples with the
// same per-sample code as the single-integral kernel (vsample.cuh), and
// writes the segment's partial sums and, in adjusting iterations, its
// partial histogram.  The refinement launch (batch.cu) reduces an integral's
// segments in their fixed order.  One kernel per class keeps each one fully
// inlined with the register budget of the single-integral kernel.
#pragma once

#include "vsample.cuh"

namespace mc {

// A value that every lane of the warp holds, moved to a uniform register (the
// result of a warp reduction is one): operands and round keys that are launch
// constants in the single-integral kernels are segment constants here (64
// integrals of 2e6 calls: corner d = 8 6.60 -> 6.39, osc d = 10 8.22 -> 7.97
// cycles per SM and sample against reading them from shared memory).
__device__ __forceinline__ uint32_t uni(uint32_t v) { return __reduce_or_sync(0xffffffffu, v); }
__device__ __forceinline__ float uni(float v) { return __uint_as_float(uni(__float_as_uint(v))); }

// One kernel per (family, dimension D): every segment it samples belongs to
// an integral of that dimension.  Registers are bounded as for the
// single-integral kernel of the same family and axis count (3 or 4 resident
// blocks per SM), so that more blocks of the concurrently running classes
// fit on an SM.
template <int FAM, bool MIXED, int D>
__global__ void __launch_bounds__(kVsThreads, vsample_min_blocks<FAM, MIXED, (D + 3) / 4>())
vsample_batch_kernel(const __grid_constant__ BatchArgs a)
{
    constexpr int NB4 = (D + 3) / 4;
    if constexpr (FAM == MCUBES_F_COSMO6 && D != 6) {
        return;  // six axes only: never launched
    } else {
    using Cell = typename Prec<MIXED>::Cell;
    using HT = typename Prec<MIXED>::H;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double red[3][kVsThreads / 32];
    __shared__ __align__(16) BatchSample sd;
    __shared__ uint4 philox_tab[kPhiloxTab * NB4];
    __shared__ uint32_t cube_step[2 * kDMax];

    const uint32_t s_begin = a.blk_seg[blockIdx.x], s_end = a.blk_seg[blockIdx.x + 1];
    for (uint32_t si = s_begin; si < s_end; ++si) {
        const BatchSeg seg = a.segs[si];
        __syncthreads();  // the previous segment is done with sd, cells and hist
        // the integral's state, descriptor and map cells together (their places
        // follow from the slot): one trip to memory
        const BatchState& B = a.st[seg.slot];
        const int2 now = ld_volatile_int2(&B.it);
        {
            const uint32_t* src = reinterpret_cast<const uint32_t*>(static_cast<const BatchSample*>(a.desc + seg.slot));
            uint32_t* dst = reinterpret_cast<uint32_t*>(&sd);
            for (uint32_t i = threadIdx.x; i < sizeof(BatchSample) / 4; i += blockDim.x) dst[i] = src[i];
        }
        HT* hist = reinterpret_cast<HT*>(smem + (MIXED ? 0u : cell_bytes(false) * D * a.nb));
        Cell* cells = reinterpret_cast<Cell*>(smem + (MIXED ? hist_smem_bytes(true, D * a.nb) : 0u));
        if (seg.adjust) clear_hist(hist, D * a.nb);
        stage_cells<MIXED>(cells, static_cast<const unsigned char*>(a.cells) + a.cell_stride * seg.slot, D, a.nb);
        __syncthreads();
        // an integral that finished in an earlier iteration of this step (a
        // step may run several) is skipped; only the refinement changes the state.
        // This iteration adjusts while it < ita (a step's iterations may cross
        // ita).  The refinement reads both flags back.
        const bool run = !now.y && now.x < sd.itmax;
        const bool adjust = run && seg.adjust && now.x < sd.ita;
        if (threadIdx.x == 0) {
            a.segs[si].ran = run ? 1u : 0u;
            a.segs[si].adjust = adjust ? 1u : 0u;
        }
        if (!run) continue;
        constexpr uint32_t d = D;
        const uint32_t nb = a.nb;
        FamConsts uf;  // single precision: the integrand's constants (those it reads)
        if constexpr (MIXED) {
#pragma unroll
            for (int i = 0; i < kParMax; ++i) uf.cf[i] = uni(sd.fam.cf[i]);
        }
        const BatchView v{d,        nb,           uni(sd.g), uni(sd.gmagic),   uni(sd.key0),     uni(sd.key1), d,
                          sd.jac0,  uni(sd.phi_scale_f), sd.inv_p, sd.inv_var_den, sd.inv_p_f, sd.inv_var_den_f, 0u,
                          cube_step, MIXED ? uf : sd.fam};
        const uint32_t it = (uint32_t)now.x;
        fill_philox_table<NB4>(philox_tab, v, it);
        const SampleRng<NB4> rng{it, philox_tab};
        if (threadIdx.x == blockDim.x - 1) {
            const uint64_t n = seg.c1 - seg.c0;
            const uint64_t step = mod_by(mod_by(blockDim.x / sd.lanes, n, seg.perm_inv) * seg.perm_k, n, seg.perm_inv);
            cube_step_digits32((uint32_t)step, (uint32_t)n, (uint32_t)sd.m, D, v, cube_step);
        }
        __syncthreads();

        CubeSums acc;
        auto sample = [&](auto adj_c, auto fix_c) {
            sample_cubes<FAM, MIXED, decltype(adj_c)::value, NB4, D, decltype(fix_c)::value>(
                v, cells, hist, seg.c0, seg.c1 - seg.c0, seg.perm_k, seg.perm_inv, 0, 1, rng, sd.lanes, sd.p, acc);
        };
        bool done = false;
        if constexpr (!MIXED && FixFamily<FAM>::kHas) {
            if (sd.fam.fix) {  // the fixed-point form: uniform over the segment
                if (adjust) sample(std::true_type{}, std::true_type{});
                else sample(std::false_type{}, std::true_type{});
                done = true;
            }
        }
        if (!done) {
            if (adjust) sample(std::true_type{}, std::false_type{});
            else sample(std::false_type{}, std::false_type{});
        }
        block_write_sums<MIXED>(acc, false, red, a.seg_part + 3 * (size_t)si);
        if (adjust) {
            __syncthreads();
            HT* out = reinterpret_cast<HT*>(a.seg_hist) + seg.hist_off;
            for (uint32_t i = threadIdx.x; i < d * nb; i += blockDim.x) out[i] = hist[i];
        }
    }
    }
}

template <int FAM, bool MIXED>
inline auto vsample_batch_kernel_ptr(int d)
{
    using K = void (*)(BatchArgs);
    switch (d) {
    case 1: return (K)vsample_batch_kernel<FAM, MIXED, 1>;
    case 2: return (K)vsample_batch_kernel<FAM, MIXED, 2>;
    case 3: return (K)vsample_batch_kernel<FAM, MIXED, 3>;
    case 4: return (K)vsample_batch_kernel<FAM, MIXED, 4>;
    case 5: return (K)vsample_batch_kernel<FAM, MIXED, 5>;
    case 6: return (K)vsample_batch_kernel<FAM, MIXED, 6>;
    case 7: return (K)vsample_batch_kernel<FAM, MIXED, 7>;
    case 8: return (K)vsample_batch_kernel<FAM, MIXED, 8>;
    case 9: return (K)vsample_batch_kernel<FAM, MIXED, 9>;
    case 10: return (K)vsample_batch_kernel<FAM, MIXED, 10>;
    case 11: return (K)vsample_batch_kernel<FAM, MIXED, 11>;
    default: return (K)vsample_batch_kernel<FAM, MIXED, 12>;
    }
}

template <int FAM>
cudaError_t launch_vsample_batch_family(bool mixed, int d, const BatchArgs& a, int grid, size_t smem,
                                        cudaStream_t s)
{
    auto k = mixed ? vsample_batch_kernel_ptr<FAM, true>(d) : vsample_batch_kernel_ptr<FAM, false>(d);
    cudaError_t e = raise_smem_limit((const void*)k, smem);
    if (e != cudaSuccess) return e;
    k<<<grid, kVsThreads, smem, s>>>(a);
    return cudaGetLastError();
}

template <int FAM>
cudaError_t vsample_batch_occupancy_family(bool mixed, int d, size_t smem, int* blocks)
{
    auto k = mixed ? vsample_batch_kernel_ptr<FAM, true>(d) : vsample_batch_kernel_ptr<FAM, false>(d);
    cudaError_t e = raise_smem_limit((const void*)k, smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, k, kVsThreads, smem);
}

}  // namespace mc

// Instantiates a family's batched kernels and their launchers
// (launch_vsample_batch_<name>, vsample_batch_occupancy_<name>).
#define MC_INSTANTIATE_BATCH_FAMILY(FAM, NAME)                                                        \
    namespace mc {                                                                                    \
    cudaError_t launch_vsample_batch_##NAME(bool mixed, int d, const BatchArgs& a, int grid,          \
                                            size_t smem, cudaStream_t s)                              \
    {                                                                                                 \
        return launch_vsample_batch_family<FAM>(mixed, d, a, grid, smem, s);                          \
    }                                                                                                 \
    cudaError_t vsample_batch_occupancy_##NAME(bool mixed, int d, size_t smem, int* blocks)           \
    {                                                                                                 \
        return vsample_batch_occupancy_family<FAM>(mixed, d, smem, blocks);                           \
    }                                                                                                 \
    }
