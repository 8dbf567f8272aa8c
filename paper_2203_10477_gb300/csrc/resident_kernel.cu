// resident_kernel.cu -- launch entry points of the resident warp-window kernel
// (resident.cuh).

#include "resident.cuh"

namespace rswr {

namespace {

using namespace resident;

struct Entry {
    int dtype, form, P;
    const void* fn;        // at most two probes to a window, or few points with more
    const void* fn_dense;
};

template <typename Real, int FORM, int P>
Entry entry()
{
    return Entry{sizeof(Real) == 8 ? kF64 : kF32, FORM, P,
                 reinterpret_cast<const void*>(&resident_kernel<Real, FORM, P, false>),
                 res_dense_kernel(sizeof(Real) == 8 ? kF64 : kF32, P)};
}

const Entry* find(int dtype, int form, int P)
{
    static const Entry entries[] = {
        entry<float, kIncrement, 4>(),   entry<float, kIncrement, 8>(),   entry<float, kIncrement, 16>(),
        entry<float, kIncrement, 32>(),  entry<double, kCanonical, 1>(),  entry<double, kCanonical, 2>(),
        entry<double, kCanonical, 4>(),  entry<double, kCanonical, 8>(),  entry<double, kCanonical, 12>(),
        entry<double, kCanonical, 16>(),
    };
    for (const Entry& e : entries)
        if (e.dtype == dtype && e.form == form && e.P == P) return &e;
    return nullptr;
}

}  // namespace

size_t res_smem_bytes(int dtype, int P, int H, int warps_per_cta, int probe_rows, int* values)
{
    const size_t v = dtype == kF64 ? warp_values<double>(H, P, probe_rows)
                                   : warp_values<float>(H, P, probe_rows);
    *values = (int)v;
    return v * warps_per_cta * (dtype == kF64 ? 8 : 4);
}

int res_max_warps(int dtype, int P) { return dtype == kF64 ? max_warps<double>(P) : max_warps<float>(P); }

size_t res_slot_bytes(int dtype, int H)
{
    return sizeof(ulonglong2) * 4 * (size_t)H * (dtype == kF64 ? slot_words<double> : slot_words<float>);
}

cudaError_t res_occupancy(int dtype, int form, int P, bool dense, int threads, size_t smem, int* ctas_per_sm)
{
    *ctas_per_sm = 0;
    const Entry* e = find(dtype, form, P);
    if (!e) return cudaSuccess;
    const void* const fn = dense ? e->fn_dense : e->fn;
    int dev = 0, per_block = 0;
    cudaError_t st = cudaGetDevice(&dev);
    if (st == cudaSuccess) st = cudaDeviceGetAttribute(&per_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (st != cudaSuccess) return st;
    per_block -= 2048;  // (room for the static part)
    if (smem > (size_t)per_block) return cudaSuccess;
    st = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, per_block);
    if (st != cudaSuccess) return st;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, fn, threads, smem);
}

namespace {

// One launch configuration: a cooperative grid (every warp waits on its
// neighbours, so all CTAs must be resident at once) or one cluster, whose CTAs
// the hardware places together.
void configure(cudaLaunchConfig_t* c, cudaLaunchAttribute* at, int grid, int threads, size_t smem, bool cluster,
               cudaStream_t s)
{
    *c = cudaLaunchConfig_t{};
    c->gridDim = dim3(grid);
    c->blockDim = dim3(threads);
    c->dynamicSmemBytes = smem;
    c->stream = s;
    c->attrs = at;
    c->numAttrs = 1;
    if (cluster) {
        at->id = cudaLaunchAttributeClusterDimension;
        at->val.clusterDim.x = (unsigned)grid;
        at->val.clusterDim.y = at->val.clusterDim.z = 1;
    } else {
        at->id = cudaLaunchAttributeCooperative;
        at->val.cooperative = 1;
    }
}

}  // namespace

cudaError_t res_kernel_clusters(const void* fn, int grid, int threads, size_t smem, int* clusters)
{
    *clusters = 0;
    cudaError_t st = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (st != cudaSuccess) return st;
    cudaLaunchConfig_t c;
    cudaLaunchAttribute at;
    configure(&c, &at, grid, threads, smem, true, nullptr);
    return cudaOccupancyMaxActiveClusters(clusters, fn, &c);
}

cudaError_t res_launch_kernel(const void* fn, const void* params, int grid, int threads, size_t smem, bool cluster,
                              cudaStream_t s)
{
    void* args[] = {const_cast<void*>(params)};
    cudaLaunchConfig_t c;
    cudaLaunchAttribute at;
    configure(&c, &at, grid, threads, smem, cluster, s);
    return cudaLaunchKernelExC(&c, fn, args);
}

cudaError_t res_clusters(int dtype, int form, int P, bool dense, int grid, int threads, size_t smem, int* clusters)
{
    *clusters = 0;
    const Entry* e = find(dtype, form, P);
    return e ? res_kernel_clusters(dense ? e->fn_dense : e->fn, grid, threads, smem, clusters) : cudaSuccess;
}

cudaError_t res_launch(int dtype, int form, int P, bool dense, const void* params, int grid, int threads, size_t smem,
                       bool cluster, cudaStream_t s)
{
    const Entry* e = find(dtype, form, P);
    return e ? res_launch_kernel(dense ? e->fn_dense : e->fn, params, grid, threads, smem, cluster, s) : cudaErrorInvalidValue;
}

}  // namespace rswr
