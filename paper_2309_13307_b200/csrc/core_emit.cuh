// Where a reconstructed block of four coordinates goes: the estimate itself, or the optimiser's update made from it
// (ReconstructEpilogue).  Shared by the kernels that reconstruct; Args has out, k_end, vec_ok and epi.
#pragma once

#include "core_internal.h"

namespace core {

// The estimate r of block q goes out (or the update built from it, with an epilogue): one 16-byte
// store where alignment allows, element by element on the ragged last block.
template <typename Args>
__device__ __forceinline__ void emit_block(const Args &a, uint64_t q, uint64_t q_begin, float4 r) {
    const int64_t off = (int64_t)((q - q_begin) << 2);        // offset into out
    const int64_t k = (int64_t)(q << 2);
    const float step = a.epi.base ? (a.epi.step_dev ? a.epi.step_scale * __ldcg(a.epi.step_dev) : a.epi.step) : 0.f;
    if (a.vec_ok && k + 4 <= a.k_end) {
        float4 v = r;
        if (a.epi.base) {
            float4 b = *reinterpret_cast<const float4 *>(a.epi.base + off);
            if (a.epi.shift_dst) {
                const float4 s = *reinterpret_cast<const float4 *>(a.epi.shift_src + off);
                if (a.epi.lookahead) {
                    const float4 o = *reinterpret_cast<const float4 *>(a.epi.shift_dst + off);
                    b = make_float4(fmaf(a.epi.gamma, s.x - o.x, s.x), fmaf(a.epi.gamma, s.y - o.y, s.y),
                                    fmaf(a.epi.gamma, s.z - o.z, s.z), fmaf(a.epi.gamma, s.w - o.w, s.w));
                }
                *reinterpret_cast<float4 *>(a.epi.shift_dst + off) = s;
            }
            v = make_float4(fmaf(-step, r.x, b.x), fmaf(-step, r.y, b.y),
                            fmaf(-step, r.z, b.z), fmaf(-step, r.w, b.w));
        }
        *reinterpret_cast<float4 *>(a.out + off) = v;
    } else {
        const float vals[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            if (k + l >= a.k_end) continue;
            float v = vals[l];
            if (a.epi.base) {
                float b = a.epi.base[off + l];
                if (a.epi.shift_dst) {
                    const float s = a.epi.shift_src[off + l];
                    if (a.epi.lookahead) b = fmaf(a.epi.gamma, s - a.epi.shift_dst[off + l], s);
                    a.epi.shift_dst[off + l] = s;
                }
                v = fmaf(-step, v, b);
            }
            a.out[off + l] = v;
        }
    }
}

}  // namespace core
