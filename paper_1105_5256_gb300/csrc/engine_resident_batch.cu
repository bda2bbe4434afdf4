// Resident engine for batches: one launch per kind and cluster size over many instances.
#include "engine_resident.cuh"

namespace ld {

__global__ void k_resident_batch_prep(const Solve *solves) {
    const Solve &s = solves[blockIdx.x];
    __shared__ int cnt;
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    for (int c = threadIdx.x; c < s.ncols; c += blockDim.x) {
        s.pi0[c] = 0.0;
        s.terms[c] = 0.0;
        s.col_iters[c] = 0;
        if (s.class_size[c] > 0.0) atomicAdd(&cnt, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        *s.remaining = cnt;
        *s.status = 0;
    }
}

int engine_resident_batch_prep(const Solve *solves_dev, int count, void *stream) {
    k_resident_batch_prep<<<count, 128, 0, static_cast<cudaStream_t>(stream)>>>(solves_dev);
    return (int)cudaGetLastError();
}

template <typename V>
static const void *batch_fn(int kind) {
    if (kind == KIND_2D5) return reinterpret_cast<const void *>(&k_resident_batch<V, KIND_2D5, RES_BATCH_NT>);
    if (kind == KIND_3D7) return reinterpret_cast<const void *>(&k_resident_batch<V, KIND_3D7, RES_BATCH_NT>);
    return reinterpret_cast<const void *>(&k_resident_batch<V, KIND_2D13_SQ, RES_BATCH_NT>);
}

int engine_resident_batch(int precision, int kind, int M, size_t smem, const Solve *solves_dev, const ResPlan *plans_dev,
                          const int2 *items_dev, int nitems, int cap, void *stream) {
    const void *fn = precision == 0 ? batch_fn<double>(kind) : batch_fn<float>(kind);
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
        return (int)e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(nitems * M));
    cfg.blockDim = dim3(RES_BATCH_NT + 64);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)M;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    void *args[] = {&solves_dev, &plans_dev, &items_dev, &M, &cap};
    e = cudaLaunchKernelExC(&cfg, fn, args);
    if (e != cudaSuccess) cudaGetLastError();
    return (int)e;
}

}  // namespace ld
