// Contraction kernels for sm_103a, in five translation units that compile in parallel:
//
//  * kernels_contract.cu    k_leaf_convert: complex128 leaves -> storage type, with each leaf's
//                           max-abs (one thread per small leaf; blocks per slice of a large leaf);
//                           k_scatter_updates, k_finish_leaf
//  * kernels_step.cu        k_step: one step of one job, one block per work tile (graph mode)
//  * kernels_local.cu       k_warp: warp programs (subtrees of small steps, one warp each);
//                           k_local: one block per CTA-resident subtree program (all operands in
//                           shared memory), block programs and large programs in two launches
//  * kernels_persist_*.cu   k_persist: the persistent dataflow kernel (complex64, complex128)
// Dense tensor-core steps run in their own pack and GEMM launches (kernels_tc.cu).
#include "contract_common.cuh"

namespace tn {

namespace {

// One thread per leaf: the leaf's complex128 entries are read in bursts of 8 independent loads,
// converted to the storage type, and reduced to the leaf's max-abs (gate tensors have at most 16
// entries, so a leaf costs one or two memory latencies).
template <typename T>
__global__ void __launch_bounds__(128) k_leaf_convert(const JobPtrs *__restrict__ jobs) {
    using C = cx_t<T>;
    const JobPtrs &j = jobs[blockIdx.y];
    const int32_t leaf = blockIdx.x * blockDim.x + threadIdx.x;
    if (leaf >= j.n_leaves) return;
    const int64_t b = j.leaf_off[leaf], e = j.leaf_off[leaf + 1];
    C *dst = static_cast<C *>(const_cast<void *>(j.leaf));
    float mx = 0.f;
    constexpr int U = 8;
    for (int64_t i0 = b; i0 < e; i0 += U) {
        double2 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u < e) v[u] = j.leaf64[i0 + u];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u < e) {
                const C w = cmake((T)v[u].x, (T)v[u].y);
                dst[i0 + u] = w;
                mx = fmaxf(mx, absmax2(w));
            }
    }
    j.maxbits[leaf] = __float_as_uint(mx);
    j.exp2[leaf] = 0;
}

// Leaves of more than kLeafSmall entries (dense operands): blocks (leaf, job, slice) stream the
// leaf, slice z taking every gridDim.z-th run of kLeafRun entries, and merge their max-abs into the
// leaf's (zeroed) slot with an atomic max on the float bits.  Bound by HBM (24 bytes an entry in
// complex64): a thread has kLeafRun / 256 16-byte loads in flight and stores pairs of entries (14.7 M
// entries: 58 us, 73 us with one load in flight).
constexpr int64_t kLeafSmall = 64;
constexpr int kLeafRun = 2048;

template <typename T>
__global__ void __launch_bounds__(256) k_leaf_convert_wide(const JobPtrs *__restrict__ jobs) {
    using C = cx_t<T>;
    __shared__ float red[32];
    const JobPtrs &j = jobs[blockIdx.y];
    const int32_t leaf = blockIdx.x;
    if (leaf >= j.n_leaves) return;   // block-uniform
    const int64_t b = j.leaf_off[leaf], e = j.leaf_off[leaf + 1];
    const double2 *__restrict__ src = j.leaf64;
    C *dst = static_cast<C *>(const_cast<void *>(j.leaf));
    float mx = 0.f;
    constexpr int P = kLeafRun / 512;   // pairs of entries per thread
    // pairs start where the destination is 16-byte aligned: at the leaf's first entry or one before it (a
    // job's leaves start at any multiple of the entry size)
    const int64_t first = b - (int64_t)(sizeof(T) == 4 && (reinterpret_cast<uintptr_t>(dst + b) & 15) != 0);
    for (int64_t i0 = first + (int64_t)blockIdx.z * kLeafRun; i0 < e; i0 += (int64_t)gridDim.z * kLeafRun) {
        double2 v[P][2];
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t i = i0 + 2 * (p * 256 + (int)threadIdx.x) + h;
                v[p][h] = i >= b && i < e ? __ldcs(src + i) : make_double2(0, 0);
            }
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int64_t i = i0 + 2 * (p * 256 + (int)threadIdx.x);
            const C w0 = cmake((T)v[p][0].x, (T)v[p][0].y), w1 = cmake((T)v[p][1].x, (T)v[p][1].y);
            if (sizeof(T) == 4 && i >= b && i + 1 < e) {
                *reinterpret_cast<float4 *>(dst + i) = make_float4((float)w0.x, (float)w0.y, (float)w1.x, (float)w1.y);
            } else {
                if (i >= b && i < e) dst[i] = w0;
                if (i + 1 < e) dst[i + 1] = w1;
            }
            mx = fmaxf(mx, fmaxf(absmax2(w0), absmax2(w1)));
        }
    }
    mx = warp_max(mx);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) mx = fmaxf(mx, red[w]);
        if (mx > 0.f) atomicMax(j.maxbits + leaf, __float_as_uint(mx));
        if (blockIdx.z == 0) j.exp2[leaf] = 0;
    }
}

// Scatter staged tensor updates {dst offset, count, src offset} into the complex128 leaves.
__global__ void __launch_bounds__(128) k_scatter_updates(const int64_t *__restrict__ hdr,
                                                         const double2 *__restrict__ vals,
                                                         int64_t n_upd, double2 *__restrict__ leaf64) {
    for (int64_t u = blockIdx.x * 4 + (threadIdx.x >> 5); u < n_upd; u += (int64_t)gridDim.x * 4) {
        const int64_t dst = hdr[3 * u], cnt = hdr[3 * u + 1], src = hdr[3 * u + 2];
        for (int64_t i = threadIdx.x & 31; i < cnt; i += 32) leaf64[dst + i] = vals[src + i];
    }
}

template <typename T>
__global__ void k_finish_leaf(JobPtrs j) {
    const cx_t<T> v = static_cast<const cx_t<T> *>(j.leaf)[0];
    DeviceResult *r = static_cast<DeviceResult *>(j.result);
    r->re = (double)v.x;
    r->im = (double)v.y;
    r->exp2 = 0;
}

}  // namespace

cudaError_t launch_leaf_convert(bool c128, const JobPtrs *jobs_dev, int32_t n_jobs,
                                int32_t max_leaves, int64_t max_leaf_elems, cudaStream_t stream) {
    if (n_jobs <= 0 || max_leaves <= 0) return cudaSuccess;
    if (max_leaf_elems > kLeafSmall) {
        // two runs per slice for the largest leaf, at most 2048 slices
        const int64_t z = std::min<int64_t>(2048, (max_leaf_elems + 2 * kLeafRun - 1) / (2 * kLeafRun));
        const dim3 grid((unsigned)max_leaves, (unsigned)n_jobs, (unsigned)z);
        if (c128) k_leaf_convert_wide<double><<<grid, 256, 0, stream>>>(jobs_dev);
        else k_leaf_convert_wide<float><<<grid, 256, 0, stream>>>(jobs_dev);
        return cudaGetLastError();
    }
    dim3 grid((unsigned)((max_leaves + 127) / 128), (unsigned)n_jobs);
    if (c128) k_leaf_convert<double><<<grid, 128, 0, stream>>>(jobs_dev);
    else k_leaf_convert<float><<<grid, 128, 0, stream>>>(jobs_dev);
    return cudaGetLastError();
}

cudaError_t launch_finish_leaf(bool c128, const JobPtrs &job, cudaStream_t stream) {
    if (c128) k_finish_leaf<double><<<1, 1, 0, stream>>>(job);
    else k_finish_leaf<float><<<1, 1, 0, stream>>>(job);
    return cudaGetLastError();
}

cudaError_t launch_scatter_updates(const int64_t *hdr, const double2 *vals, int64_t n_upd,
                                   double2 *leaf64, cudaStream_t stream) {
    if (n_upd <= 0) return cudaSuccess;
    int64_t blocks = (n_upd + 3) / 4;
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_scatter_updates<<<(unsigned)blocks, 128, 0, stream>>>(hdr, vals, n_upd, leaf64);
    return cudaGetLastError();
}

}  // namespace tn
