// Row-wise decode attention: one CTA per (beam slot, head), every beam reads its
// own rows through the beam-index table, fp32 ALU arithmetic.  This is the
// direct transcription of the paper's per-beam formulation (Section 3.3): loop
// over the prompt rows, then over the index-selected response rows, one online
// softmax across both (segkv_rowwise.cuh).  It re-reads the prompt once per beam, so it is not the
// fast path: the library uses it for shapes that the tiled kernel does not take while
// the keys are few, and exposes it as a cross-check.
#include "segkv_rowwise.cuh"

namespace segkv_impl {

namespace {

template <typename T, int D>
__global__ void __launch_bounds__(rowwise::kWarps * 32) sdpa_rowwise_kernel(const __grid_constant__ rowwise::Args a) {
    __shared__ float s[rowwise::kScratch<D>];
    rowwise::attend<T, D>(a, blockIdx.y, blockIdx.x, threadIdx.x >> 5, threadIdx.x & 31, s, [] { __syncthreads(); });
}

template <typename T>
cudaError_t dispatch(const Dims& d, const SdpaArgs& a, cudaStream_t st) {
    const dim3 grid(d.heads, d.rows), block(rowwise::kWarps * 32);
    const rowwise::Args r = rowwise::make_args(d, a);
    switch (d.head_dim) {
        case 64: sdpa_rowwise_kernel<T, 64><<<grid, block, 0, st>>>(r); break;
        case 128: sdpa_rowwise_kernel<T, 128><<<grid, block, 0, st>>>(r); break;
        case 256: sdpa_rowwise_kernel<T, 256><<<grid, block, 0, st>>>(r); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sdpa_rowwise(const Dims& d, const SdpaArgs& a, cudaStream_t st) {
    return d.dtype == SEGKV_BF16 ? dispatch<__nv_bfloat16>(d, a, st) : dispatch<__half>(d, a, st);
}

}  // namespace segkv_impl
