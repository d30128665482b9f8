// split_reduce.cu -- the second half of a contraction whose every tile was
// cut into K pieces (EPI_F32_PART, tc_gemm.cuh): sums the pieces' fp32
// partials in piece order and applies the epilogue that a whole tile would
// have applied.  Bound: L2 (the partials were just written; pieces x M x N x
// 4 bytes, at most 40 MB).  One thread per four columns of a row, so partials
// and outputs move as 16-byte vectors of whole rows, and every SM takes part;
// the alternative, the piece that arrives last summing the others from one
// CTA (the tail split), reads up to 128 KB per piece through one SM.  At 93
// rows, d 3,584, 10 pieces (13 MB) it takes 5 us, launch included.
#include "gemm_launch.cuh"

namespace attt {

constexpr int kReduceThreads = 256;

template <bool OUT16>
__global__ void __launch_bounds__(kReduceThreads) split_reduce_kernel(const SplitReduceArgs a) {
    griddep_launch_dependents();
    griddep_wait();  // the pieces, and the row terms of an earlier kernel
    const int64_t i = (int64_t)blockIdx.x * kReduceThreads + threadIdx.x;
    const int n4 = a.N / 4;
    if (i >= (int64_t)a.M * n4) return;
    const int row = (int)(i / n4), col = (int)(i - (int64_t)row * n4) * 4;
    const int tn = col / a.BN;
    // piece p of the tile: `rows` rows of BN columns from part_row(.., p, ..)
    const int64_t y = part_row(row / a.rows, tn, a.tiles_m, 0, a.pieces, a.rows) + row % a.rows;
    const float4 *src = reinterpret_cast<const float4 *>(a.part + y * a.BN + (col - tn * a.BN));
    const int64_t step = (int64_t)a.rows * a.BN / 4;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int p = 0; p < a.pieces; ++p) {
        const float4 v = __ldcg(src + p * step);
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    if constexpr (OUT16) {
        __nv_bfloat162 o[2] = {__floats2bfloat162_rn(a.alpha * s.x, a.alpha * s.y),
                               __floats2bfloat162_rn(a.alpha * s.z, a.alpha * s.w)};
        *reinterpret_cast<uint2 *>(a.out16 + (int64_t)row * a.ld + col) = *reinterpret_cast<uint2 *>(o);
        return;
    }
    const float rb = a.row_beta ? __ldcg(a.row_beta + row) : 1.f;
    float4 o = make_float4(rb * s.x, rb * s.y, rb * s.z, rb * s.w);
    float4 *dst = reinterpret_cast<float4 *>(a.out + (int64_t)row * a.ld + col);
    if (a.accumulate) {
        const float ra = a.row_alpha ? __ldcg(a.row_alpha + row) : 1.f;
        const float4 p = __ldcg(dst);
        o.x = fmaf(ra, p.x, o.x); o.y = fmaf(ra, p.y, o.y);
        o.z = fmaf(ra, p.z, o.z); o.w = fmaf(ra, p.w, o.w);
    }
    if (a.row_gamma) {
        const float gam = __ldcg(a.row_gamma + row);
        int t = __ldg(a.fix_tgt + row);
        if (t < 0 || t >= a.fix_V) t = 0;
        const uint2 u = __ldg(reinterpret_cast<const uint2 *>(a.fix_W + (int64_t)t * a.fix_ld + col));
        const float2 w0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x));
        const float2 w1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
        o.x = fmaf(-gam, w0.x, o.x); o.y = fmaf(-gam, w0.y, o.y);
        o.z = fmaf(-gam, w1.x, o.z); o.w = fmaf(-gam, w1.y, o.w);
    }
    *dst = o;
}

attt_status launch_split_reduce(const SplitReduceArgs &a, cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cdiv((int64_t)a.M * (a.N / 4), kReduceThreads));
    cfg.blockDim = dim3(kReduceThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = a.out16 ? cudaLaunchKernelEx(&cfg, split_reduce_kernel<true>, a)
                                  : cudaLaunchKernelEx(&cfg, split_reduce_kernel<false>, a);
    if (e != cudaSuccess) return ATTT_ERR_CUDA;
    count_launch();
    return cudaGetLastError() == cudaSuccess ? ATTT_OK : ATTT_ERR_CUDA;
}

}  // namespace attt
