// FP64 fused step kernels (lb_step64.cuh) and their launchers.
#include "lb_step64.cuh"

namespace lbfe {

namespace {

template <bool MRT>
cudaError_t launch_t(const DomDesc& d, const DomDesc* d_descs, const WorkItem* d_items, int n_items,
                     int n_dom, int parity, int bx, int rows, int grid_p, int* sched, cudaStream_t s)
{
    const size_t smem = Layout64(bx / 32).total();
    const int threads = bx + 32;
    if (n_dom == 1 && d_items == nullptr) {
        const dim3 grid((d.nx + bx - 1) / bx, (d.ny + rows - 1) / rows);
        step_single64_kernel<MRT><<<grid, threads, smem, s>>>(d, parity, rows);
    } else {
        const int grid = grid_p > 0 ? grid_p : n_items;
        step_batch64_kernel<MRT><<<grid, threads, smem, s>>>(d_descs, d_items, n_items, parity,
                                                             sched, d.err);
    }
    return cudaGetLastError();
}

template <bool MRT>
int occupancy_t(int bx, bool single)
{
    int n = 0;
    const size_t smem = Layout64(bx / 32).total();
    const cudaError_t e = single ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                       &n, step_single64_kernel<MRT>, bx + 32, smem)
                                 : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                       &n, step_batch64_kernel<MRT>, bx + 32, smem);
    return e == cudaSuccess ? n : 0;
}

template <bool MRT>
cudaError_t allow_large_smem()
{
    const int bytes = 200 * 1024;
    const cudaError_t e = cudaFuncSetAttribute(step_single64_kernel<MRT>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(step_batch64_kernel<MRT>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

}  // namespace

int launch_step_f64(int coll, const DomDesc& d, const DomDesc* d_descs, const WorkItem* d_items,
                    int n_items, int n_dom, int parity, int bx, int rows, int grid_p, int* sched,
                    void* stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return int(coll ? launch_t<true>(d, d_descs, d_items, n_items, n_dom, parity, bx, rows, grid_p,
                                     sched, s)
                    : launch_t<false>(d, d_descs, d_items, n_items, n_dom, parity, bx, rows, grid_p,
                                      sched, s));
}

int batch_occupancy_f64(int coll, int bx, int single)
{
    return coll ? occupancy_t<true>(bx, single != 0) : occupancy_t<false>(bx, single != 0);
}

size_t step_smem_f64(int bx) { return Layout64(bx / 32).total(); }

int prepare_step_f64()
{
    const cudaError_t e = allow_large_smem<true>();
    return int(e != cudaSuccess ? e : allow_large_smem<false>());
}

}  // namespace lbfe
