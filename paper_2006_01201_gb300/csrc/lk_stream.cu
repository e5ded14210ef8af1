// lk_stream.cu -- the streamed LK kernel (lk_stream_impl.cuh) for float32
// pyramid planes, and the dispatch over storage types. The bfloat16 and
// binary16 instantiations live in lk_stream_bf16.cu and lk_stream_f16.cu so
// that the three compile in parallel.
#include "lk_stream_impl.cuh"

namespace pano {

namespace lks {
PANO_LKS_INSTANTIATE(float)
PANO_LKS_EXTERN(__nv_bfloat16)
PANO_LKS_EXTERN(__half)
}  // namespace lks

PANO_BOUNDS_READER(bounds_read_lk_stream)
PANO_LKS_LOST_READER(lost_read_lk_stream)

cudaError_t lk_stream_lost(unsigned* n) {
    *n = 0;
    cudaError_t e = lost_read_lk_stream(n);
    if (e == cudaSuccess) e = lost_read_lk_stream_bf16(n);
    return e == cudaSuccess ? lost_read_lk_stream_f16(n) : e;
}

#ifdef PANO_BOUNDS_CHECK
namespace {
// a warp that waits for 16 bytes that nobody sends
__global__ void lost_halo_kernel() {
    __shared__ __align__(8) unsigned long long s_bar;
    const unsigned bar = (unsigned)__cvta_generic_to_shared(&s_bar);
    if (threadIdx.x == 0) {
        lks::bar_init(bar);
        lks::bar_expect(bar, 16);
    }
    __syncwarp();
    if (!lks::bar_wait(bar, 0)) atomicAdd(&g_lost_halos, 1u);
}
}  // namespace
cudaError_t launch_lost_halo(cudaStream_t s) {
    lost_halo_kernel<<<1, 32, 0, s>>>();
    return cudaGetLastError();
}
#endif

bool lk_stream_supports(int iters, int radius) { return iters >= 1 && iters <= 5 && radius >= 1 && radius <= 3; }

int lk_stream_cluster(int w, int h, int iters, int radius, int seg_rows) {
    switch (radius) {
        case 1: return lks::stream_plan<1>(w, h, iters, seg_rows).csize;
        case 2: return lks::stream_plan<2>(w, h, iters, seg_rows).csize;
        default: return lks::stream_plan<3>(w, h, iters, seg_rows).csize;
    }
}

int lk_stream_seg_rows(int w, int h, int iters, int radius, int csize) {
    switch (radius) {
        case 1: return lks::stream_seg_rows<1>(w, h, iters, csize);
        case 2: return lks::stream_seg_rows<2>(w, h, iters, csize);
        default: return lks::stream_seg_rows<3>(w, h, iters, csize);
    }
}

cudaError_t lk_stream_prepare(int max_smem_bytes) {
    cudaError_t e;
    if ((e = lks::stream_prepare<float>(max_smem_bytes)) != cudaSuccess) return e;
    if ((e = lks::stream_prepare<__nv_bfloat16>(max_smem_bytes)) != cudaSuccess) return e;
    return lks::stream_prepare<__half>(max_smem_bytes);
}

cudaError_t launch_lk_stream_batch(const LkBatch& b, cudaStream_t s, int* kernels) {
    if (b.n < 1 || b.n > kMaxBatch) return cudaErrorInvalidValue;
    for (int p = 1; p < b.n; ++p)
        if (b.pair[p].pyr != b.pair[0].pyr || b.pair[p].iters != b.pair[0].iters ||
            b.pair[p].radius != b.pair[0].radius)
            return cudaErrorInvalidValue;
    switch (b.pair[0].pyr) {
        case kPyrF32: return lks::stream_launch_batch<float>(b, s, kernels);
        case kPyrBF16: return lks::stream_launch_batch<__nv_bfloat16>(b, s, kernels);
        case kPyrF16: return lks::stream_launch_batch<__half>(b, s, kernels);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_lk_stream(const LkArgs& a, int ndirs, cudaStream_t s) {
    switch (a.pyr) {
        case kPyrF32: return lks::stream_launch<float>(a, ndirs, s);
        case kPyrBF16: return lks::stream_launch<__nv_bfloat16>(a, ndirs, s);
        case kPyrF16: return lks::stream_launch<__half>(a, ndirs, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace pano
