// refine.cu -- per-iteration finalisation of a single integral on the
// device: the fixed-order reduction of the sampling launch's block partials,
// Adjust-Bin-Bounds (Alg. 2) as one block per axis (reading and clearing the
// pass's histogram, then rebuilding that axis's map cells), and
// Weighted-Estimates plus Check-Convergence (Alg. 2) as one more block.
// Keeping these on the GPU lets a whole iteration run without the host.
#include "refine_dev.cuh"

namespace mc {

namespace {

using namespace refine_detail;

// Adjust-Bin-Bounds of axis ax (rebin_block): the row of the pass's histogram
// is read and cleared, the new edges and map cells written (in m-Cubes1D for
// every axis).  The tables and edges are read before the sampling pass has
// ended: nothing writes them between two refinements.  (Sharing an axis's
// edges and cells among a cluster of two or four blocks measured no faster,
// f5 d = 8 at 1e5 calls 8% slower: the cluster's blocks have to find room
// beside the sampling blocks.)
static __device__ __forceinline__ void rebin_axis(const RefineArgs& a, int ax)
{
    __shared__ RebinShared s;
    const int nb = a.nb;
    const size_t off = (size_t)ax * nb;
    const int rows = a.hist_d == a.d ? 1 : a.d;  // m-Cubes1D: axis 0's edges go to every axis
    load_log_tables(s);
    for (int k = threadIdx.x; k < nb; k += kRefineThreads) {
        s.B[k] = a.grid[off + k];
        s.Blo[k] = a.grid_lo[off + k];
    }
    grid_dependency_wait();
    if (!*(volatile const int*)&a.st->active) return;  // iteration skipped after convergence: the whole grid
    for (int k = threadIdx.x; k < nb; k += kRefineThreads) {
        const double c = a.hist_acc[off + k];
        s.C[k] = c;
        a.hist[off + k] = c;
        a.hist_acc[off + k] = 0.0;  // for the next pass
    }
    if (!rebin_block(s, nb, a.alpha, &a.st->error, &a.st->done)) return;
    for (int k = threadIdx.x; k < nb; k += kRefineThreads) {
        const DD right = edge_right(s.B, s.Blo, k), left = edge_left(s.B, s.Blo, k);
        for (int r = 0; r < rows; ++r) {
            const size_t i = off + (size_t)r * nb + k;
            const int j = ax + r;
            a.grid[i] = right.hi;
            a.grid_lo[i] = right.lo;
            if (!a.cells_g) continue;
            if (a.mixed) static_cast<float2*>(a.cells_g)[i] = map_cell_f32(left, right, a.lo[j], a.scale[j], nb);
            else if (a.cm.on) static_cast<double2*>(a.cells_g)[i] = map_cell_fix(left, right, a.cm, j);
            else static_cast<double2*>(a.cells_g)[i] = map_cell_f64(left, right, a.lo[j], a.scale[j], a.inv_g);
        }
    }
}

// One iteration's finalisation: block c < nrebin rebins axis c, the last one
// reduces the partials, records the iteration and weighs all of them.
// Bounded by latency: with 500 bins an axis takes 8.2 us (13.3 us as FP64 code
// on a cluster of four blocks), of which 2 us wait for the sampling pass to
// end (the launch overlaps it), weights 1.7, edges 1.8, cells 0.9; the last
// block 5-6 us (9.9 before).  Whole iterations: gauss4 at 1e4 calls 44.6 ->
// 25.5 us, f5 at 1e5 59 -> 37 us, the launch overlap, the smaller grids and the
// cheaper block sums of the sampling pass included.
__global__ void __launch_bounds__(kRefineThreads) refine_kernel(const __grid_constant__ RefineArgs a)
{
    grid_dependents_launch();  // the next sampling pass may set itself up
    const int nrebin = a.adjust ? a.hist_d : 0;
    if ((int)blockIdx.x == nrebin) {
        DevState* st = a.st;
        grid_dependency_wait();
        if (!*(volatile const int*)&st->active) return;
        const IterRecord r{&st->it, &st->done, &st->error, &st->n, &st->converged, &st->estimate, &st->sigma,
                           &st->chi2_dof, st->hist_I, st->hist_V, kItMax, st->rel_tol, st->abs_tol};
        finalize_iteration(a.part, a.nblocks, a.m, r, a.split, a.p);
        return;
    }
    rebin_axis(a, (int)blockIdx.x);
}

// Sums of one sampling pass over a cube range (no state change): block
// d (or 0) adds the partial sums, blocks 0..d-1 copy the histogram rows out
// of the accumulator and clear them (d is the number of axes with a
// histogram).
__global__ void __launch_bounds__(kRefineThreads)
reduce_range_kernel(const double* part, double* hist_acc, int nblocks, int d, int nb, int adjust,
                    double* out_sums, double* out_hist)
{
    __shared__ double scratch[33];
    const int nrebin = adjust ? d : 0;
    if ((int)blockIdx.x == nrebin) {
        double s[3] = {0.0, 0.0, 0.0};
        for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
            for (int q = 0; q < 3; ++q) s[q] += part[3 * (size_t)b + q];
        for (int q = 0; q < 3; ++q) {
            const double t = block_sum(s[q], scratch);
            if (threadIdx.x == 0) out_sums[q] = t;
        }
        return;
    }
    const int ax = blockIdx.x;
    for (int k = threadIdx.x; k < nb; k += blockDim.x) {
        const size_t i = (size_t)ax * nb + k;
        out_hist[i] = hist_acc[i];
        hist_acc[i] = 0.0;
    }
}

// Rank-order sum of gathered shard partials (mcubes_shard_finish): one
// thread per element, the ranks added in order 0, 1, ... so that every rank
// that combines the same gathered array gets the same bits.
__global__ void combine_shards_kernel(const double* gathered, int nranks, int len, double* part, double* hist)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= len) return;
    double s = gathered[i];
    for (int r = 1; r < nranks; ++r) s += gathered[(size_t)r * len + i];
    if (i < MCUBES_SHARD_HEAD) part[i] = s;
    else hist[i - MCUBES_SHARD_HEAD] = s;
}

// Map cell i (axis j) of a context's grid.
__device__ __forceinline__ void write_cell(const CellBox& box, int j, int i, DD left, DD right, int nb, void* out)
{
    if (box.mixed) static_cast<float2*>(out)[i] = map_cell_f32(left, right, box.lo[j], box.scale[j], nb);
    else if (box.cm.on) static_cast<double2*>(out)[i] = map_cell_fix(left, right, box.cm, j);
    else static_cast<double2*>(out)[i] = map_cell_f64(left, right, box.lo[j], box.scale[j], 1.0 / (double)box.g);
}

// Map cells of the whole grid (after the grid is replaced).
__global__ void cells_kernel(const double* grid, const double* grid_lo, const __grid_constant__ CellBox box, int d, int nb, void* out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= d * nb) return;
    const int j = i / nb, k = i - j * nb;
    const DD right = edge_right(grid + (size_t)j * nb, grid_lo + (size_t)j * nb, k);
    const DD left = edge_left(grid + (size_t)j * nb, grid_lo + (size_t)j * nb, k);
    write_cell(box, j, i, left, right, nb, out);
}

// Right edge k of Init-Bins (Alg. 2): nb equal bins, (k+1)/nb held as
// double-double (rounded value + rounded remainder), last edge exactly 1.
__device__ __forceinline__ DD uniform_edge(int k, int nb)
{
    if (k == nb - 1) return DD{1.0, 0.0};
    const double hi = __ddiv_rn((double)(k + 1), (double)nb);
    const double rem = __fma_rn(-hi, (double)nb, (double)(k + 1));  // exact
    return DD{hi, __ddiv_rn(rem, (double)nb)};
}

// A problem's initial state in one launch: the uniform grid and its map cells,
// empty histograms and iteration state (the arguments carry the tolerances,
// so that nothing on the host has to outlive the call).
__global__ void setup_kernel(const __grid_constant__ SetupArgs a)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        DevState* st = a.st;
        st->it = 0;
        st->done = st->active = st->error = st->n = st->converged = 0;
        st->estimate = st->sigma = st->chi2_dof = 0.0;
        st->rel_tol = a.rel_tol;
        st->abs_tol = a.abs_tol;
    }
    if (i >= a.d * a.nb) return;
    const int j = i / a.nb, k = i - j * a.nb;
    const DD right = uniform_edge(k, a.nb), left = k ? uniform_edge(k - 1, a.nb) : DD{0.0, 0.0};
    a.grid[i] = right.hi;
    a.grid_lo[i] = right.lo;
    a.hist[i] = 0.0;
    if (i < a.hist_d * a.nb) a.hist_acc[i] = 0.0;
    write_cell(a.box, j, i, left, right, a.nb, a.cells);
}

}  // namespace

cudaError_t launch_refine(const RefineArgs& a, cudaStream_t s)
{
    return launch_dependent(refine_kernel, (a.adjust ? a.hist_d : 0) + 1, kRefineThreads, 0, s, a);
}

cudaError_t launch_reduce_range(const double* part, double* hist_acc, int nblocks, int d, int nb, int adjust,
                                double* out_sums, double* out_hist, cudaStream_t s)
{
    const int blocks = (adjust ? d : 0) + 1;
    reduce_range_kernel<<<blocks, kRefineThreads, 0, s>>>(part, hist_acc, nblocks, d, nb, adjust, out_sums,
                                                          out_hist);
    return cudaGetLastError();
}

cudaError_t launch_combine_shards(const double* gathered, int nranks, int len, double* part, double* hist,
                                  cudaStream_t s)
{
    combine_shards_kernel<<<(len + 255) / 256, 256, 0, s>>>(gathered, nranks, len, part, hist);
    return cudaGetLastError();
}

cudaError_t launch_cells(const double* grid, const double* grid_lo, const CellBox& box, int d, int nb, void* out,
                         cudaStream_t s)
{
    const int n = d * nb;
    cells_kernel<<<(n + 255) / 256, 256, 0, s>>>(grid, grid_lo, box, d, nb, out);
    return cudaGetLastError();
}

cudaError_t launch_setup(const SetupArgs& a, cudaStream_t s)
{
    const int n = a.d * a.nb;
    setup_kernel<<<(n + 127) / 128, 128, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace mc
