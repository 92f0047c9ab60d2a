// Two-step compact kernels (lb_step_compact2.cuh), their launchers and the
// four-wide ghost columns they read.
#include "lb_step_compact2.cuh"

namespace lbfe {

namespace {

template <bool MRT, int NWC>
cudaError_t launch_t(const DomDesc& d, int parity, int rows, int band_mul, cudaStream_t s)
{
    const int w = two_step_strip(32 * NWC);
    const dim3 grid((d.nx + w - 1) / w, (d.ny + rows - 1) / rows);
    step_two_compact_kernel<MRT, NWC>
        <<<grid, 64 * NWC + 32, TwoStepLayout(NWC, kStagesTwo).total(), s>>>(d, parity, rows, band_mul);
    return cudaGetLastError();
}

template <bool MRT, int NWC>
cudaError_t prepare_t()
{
    return cudaFuncSetAttribute(step_two_compact_kernel<MRT, NWC>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(TwoStepLayout(NWC, kStagesTwo).total()));
}

template <bool MRT, int NWC>
int occupancy_t()
{
    int n = 0;
    if (prepare_t<MRT, NWC>() != cudaSuccess) return 0;  // else none fits
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &n, step_two_compact_kernel<MRT, NWC>, 64 * NWC + 32, TwoStepLayout(NWC, kStagesTwo).total());
    return e == cudaSuccess ? n : 0;
}

template <bool MRT>
cudaError_t launch_w(const DomDesc& d, int parity, int bx, int rows, int band_mul, cudaStream_t s)
{
    switch (bx) {
        case 64: return launch_t<MRT, 2>(d, parity, rows, band_mul, s);
        case 96: return launch_t<MRT, 3>(d, parity, rows, band_mul, s);
        case 128: return launch_t<MRT, 4>(d, parity, rows, band_mul, s);
        default: return cudaErrorInvalidValue;
    }
}

__global__ void wide_ghosts_kernel(DomDesc D, int parity, bool clear)
{
    float* f = static_cast<float*>(parity ? D.f[1] : D.f[0]);
    float* c = static_cast<float*>(parity ? D.g[1] : D.g[0]);
    const long long n = 13LL * D.ny * 4;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const int which = int(k & 3);  // column -4, -3, nx + 2, nx + 3
        const long long r = k >> 2;    // plane * ny + row
        float* row = (r < 9LL * D.ny ? f + r * D.pitch : c + (r - 9LL * D.ny) * D.pitch) + kXOff;
        const int dst = which < 2 ? which - 4 : D.nx + which;
        const int src = which < 2 ? D.nx + which - 4 : which;
        row[dst] = clear ? 0.f : row[src];
    }
}

}  // namespace

int launch_two_step(int coll, const DomDesc& d, int parity, int bx, int rows, int band_mul,
                    void* stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return int(coll ? launch_w<true>(d, parity, bx, rows, band_mul, s)
                    : launch_w<false>(d, parity, bx, rows, band_mul, s));
}

int two_step_occupancy(int coll, int bx)
{
    switch (bx) {
        case 64: return coll ? occupancy_t<true, 2>() : occupancy_t<false, 2>();
        case 96: return coll ? occupancy_t<true, 3>() : occupancy_t<false, 3>();
        case 128: return coll ? occupancy_t<true, 4>() : occupancy_t<false, 4>();
        default: return 0;
    }
}

int prepare_two_step()
{
    const cudaError_t r[] = {prepare_t<false, 2>(), prepare_t<false, 3>(), prepare_t<false, 4>(),
                             prepare_t<true, 2>(),  prepare_t<true, 3>(),  prepare_t<true, 4>()};
    for (cudaError_t v : r)
        if (v != cudaSuccess) return int(v);
    return 0;
}

int launch_wide_ghosts(const DomDesc& d, int parity, bool clear, void* stream)
{
    wide_ghosts_kernel<<<304, 256, 0, static_cast<cudaStream_t>(stream)>>>(d, parity, clear);
    return int(cudaGetLastError());
}

}  // namespace lbfe
