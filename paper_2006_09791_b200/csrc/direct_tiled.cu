// Variant DIRECT_TILED: FP32 FFMA kernels for 3x3 layers (and depthwise 5x5) with dilation 1: depthwise layers go to the stream
// and plane kernels (direct_dw.cu, direct_dw_plane.cu), groups of at most 8 filters to the row kernel (direct_rows.cu), the
// rest -- wide or odd groups on planes the tensor-core variant does not take -- to the staged kernel of direct_conv.cu.
#include "gconv_internal.h"

namespace gconv {

namespace {

__global__ void group_pack_kernel(Shape s, const float* __restrict__ w, uint32_t* __restrict__ packed, uint32_t tag, bool mark) {
    const int taps = s.KH * s.KW;
    const size_t n = (size_t)s.C_out * s.Cg * taps;
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) atomicXor(packed, tag);                     // (the header is zeros; any block may add the mark)
    float* dst = reinterpret_cast<float*>(packed + kHeaderBytes / 4);
    for (; i < n; i += (size_t)gridDim.x * blockDim.x) {
        // destination index i = (((g*Cg + c)*taps + rs)*Kg + k)
        const int k = (int)(i % s.Kg);
        size_t t = i / s.Kg;
        const int rs = (int)(t % taps);
        t /= taps;
        const int c = (int)(t % s.Cg);
        const int g = (int)(t / s.Cg);
        const float v = w[(((size_t)g * s.Kg + k) * s.Cg + c) * taps + rs];
        dst[i] = v;
        if (mark && !isfinite(v) && atomicExch(packed + 1, 1u) == 0u) atomicXor(packed, kNonFiniteMark);
    }
}

}  // namespace

// Weights as [g][c][r][s][Kg] behind the header (the filters of one tap are one vector load).  `mark`: weights that are infinite or not a
// number are marked in the tag (the staged kernel leaves its main path for them; the depthwise and row kernels take them as they are).
cudaError_t group_pack(const Shape& s, const float* w, void* packed, uint32_t tag, bool mark, cudaStream_t st) {
    const size_t n = (size_t)s.C_out * s.Cg * s.KH * s.KW;
    const int blocks = (int)((n + 255) / 256 < 1184 ? (n + 255) / 256 : 1184);
    const cudaError_t e = cudaMemsetAsync(packed, 0, kHeaderBytes, st);
    if (e != cudaSuccess) return e;
    group_pack_kernel<<<blocks, 256, 0, st>>>(s, w, reinterpret_cast<uint32_t*>(packed), tag, mark);
    return cudaGetLastError();
}

bool tiled_supported(const Shape& s) {
    if (!s.square()) return false;   // one stride, padding and dilation for both axes
    if (s.KH == 5 && s.KW == 5) return dw_supported(s);   // 5x5: only the depthwise stream kernel
    return s.KH == 3 && s.KW == 3 && s.dilation == 1 && (s.stride == 1 || s.stride == 2) && s.N <= 65535;
}

bool tiled_takes_conv(const Shape& s) { return !dw_supported(s) && !rows_supported(s); }

size_t tiled_packed_bytes(const Shape& s) { return kHeaderBytes + sizeof(float) * (size_t)s.C_out * s.Cg * s.KH * s.KW; }

cudaError_t tiled_pack(const Shape& s, const float* w, void* packed, cudaStream_t st) {
    return group_pack(s, w, packed, pack_tag(s, GCONV_VARIANT_DIRECT_TILED), tiled_takes_conv(s), st);
}

cudaError_t tiled_forward(const Shape& s, const ConvCfg* conv, const DwPlan& dw, const float* x, const void* packed, float* y, Status* status,
                          int sm_count, const Launch& st) {
    if (dw_supported(s)) return dw_forward(s, dw, x, packed, y, status, st);
    if (rows_supported(s)) return rows_forward(s, x, packed, y, status, st);
    return generic_forward(s, conv, x, packed, y, status, sm_count, pack_tag(s, GCONV_VARIANT_DIRECT_TILED), st);
}

}  // namespace gconv
