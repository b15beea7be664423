// Device code shared by the kernels of one context and of a batch: strips of four adjacent pixels of a row (packing,
// depth maps), the least-cost label of a segment and the block-wide scan.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <climits>

#include "ftv_internal.h"

namespace ftv {

// Four samples of a plane's row, n of them in the view; vec: in one load (p is aligned to four samples).
template <int SB>
__device__ __forceinline__ void load4(const char* p, int n, bool vec, uint32_t* out) {
    if (vec) {  // four samples in one load
        if (SB == 1) {
            const uint32_t t = __ldg(reinterpret_cast<const uint32_t*>(p));
#pragma unroll
            for (int k = 0; k < 4; ++k) out[k] = (t >> (8 * k)) & 0xff;
        } else {
            const uint2 t = __ldg(reinterpret_cast<const uint2*>(p));
            out[0] = t.x & 0xffff;
            out[1] = t.x >> 16;
            out[2] = t.y & 0xffff;
            out[3] = t.y >> 16;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            out[k] = k >= n ? 0u : SB == 1 ? reinterpret_cast<const uint8_t*>(p)[k] : reinterpret_cast<const uint16_t*>(p)[k];
    }
}

// Clamps samples above max_value, so that they cannot spill into a neighbouring packed field; whether there were any.
__device__ __forceinline__ bool clamp4(uint32_t (&s)[3][4], uint32_t max_value) {
    bool bad = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        bad = bad || s[0][k] > max_value || s[1][k] > max_value || s[2][k] > max_value;
#pragma unroll
        for (int c = 0; c < 3; ++c) s[c][k] = min(s[c][k], max_value);
    }
    return bad;
}

// Stores the texels i .. i + n - 1; vec: n is 4 and the texels are aligned to 16 bytes.
template <int FMT>
__device__ __forceinline__ void store4(void* base, int64_t i, int n, bool vec, const uint32_t (&s)[3][4]) {
    if (FMT == FMT_U8X4 || FMT == FMT_P10) {
        constexpr int sh = FMT == FMT_U8X4 ? 8 : 10;
        uint32_t t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) t[k] = s[0][k] | (s[1][k] << sh) | (s[2][k] << (2 * sh));
        uint32_t* out = static_cast<uint32_t*>(base) + i;
        if (vec) {
            *reinterpret_cast<uint4*>(out) = make_uint4(t[0], t[1], t[2], t[3]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k < n) out[k] = t[k];
        }
    } else {
        uint2 t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            t[k] = make_uint2(s[0][k] | (s[1][k] << 16),
                              FMT == FMT_U16S ? s[2][k] | ((s[0][k] + s[1][k] + s[2][k]) << 16) : s[2][k]);
        uint2* out = static_cast<uint2*>(base) + i;
        if (vec) {
            reinterpret_cast<uint4*>(out)[0] = make_uint4(t[0].x, t[0].y, t[1].x, t[1].y);
            reinterpret_cast<uint4*>(out)[1] = make_uint4(t[2].x, t[2].y, t[3].x, t[3].y);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k < n) out[k] = t[k];
        }
    }
}

// The depth of pixels p .. p + n - 1 from their segments' labels; 0 and ST_BAD_LABEL where there is none.
// vec: n is 4 and both maps are aligned to 16 bytes at p. The pixels' chains of three dependent loads run side by side.
__device__ __forceinline__ void depth4(const int32_t* labels, int64_t p, int n, bool vec, int S, const uint16_t* seg_label,
                                       const float* label_z, int L, float* depth, uint32_t* status) {
    int s[4];
    if (vec) {
        const int4 t = __ldg(reinterpret_cast<const int4*>(labels + p));
        s[0] = t.x;
        s[1] = t.y;
        s[2] = t.z;
        s[3] = t.w;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] = __ldg(labels + p + min(k, n - 1));
    }
    int d[4];
    float z[4];
    bool bad = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        d[k] = (unsigned)s[k] < (unsigned)S ? seg_label[s[k]] : INT_MAX;
        bad = bad || d[k] >= L;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) z[k] = d[k] < L ? label_z[d[k]] : 0.0f;
    if (bad) atomicOr(status, ST_BAD_LABEL);
    if (vec) {
        *reinterpret_cast<float4*>(depth + p) = make_float4(z[0], z[1], z[2], z[3]);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < n) depth[p + k] = z[k];
    }
}

// The label of least cost in a row of L >= 1, the smallest on ties (a whole warp, converged): each lane's first least
// one, then two warp reductions, in place of five exchanges of a 64-bit key (62,000 rows of 64: 24 -> 15 us with twice
// the warps resident).
__device__ __forceinline__ int least_label(const int32_t* row, int L, int lane) {
    int v = lane < L ? row[lane] : INT_MAX, at = lane;  // a lane past the row loses every tie to a label
    for (int d = lane + 32; d < L; d += 32) {
        const int c = row[d];
        if (c < v) {
            v = c;
            at = d;
        }
    }
    const int least = __reduce_min_sync(0xffffffffu, v);
    return __reduce_min_sync(0xffffffffu, v == least ? at : INT_MAX);
}

// Block-wide exclusive scan of one int per thread (whole warps). Returns the exclusive prefix;
// *total receives the block sum.
__device__ inline int block_exclusive_scan(int v, int* total) {
    __shared__ int warp_sums[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        int s = lane < nw ? warp_sums[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += t;
        }
        warp_sums[lane] = s;  // inclusive prefix of warp sums
    }
    __syncthreads();
    const int base = warp > 0 ? warp_sums[warp - 1] : 0;
    *total = warp_sums[(blockDim.x >> 5) - 1];
    __syncthreads();
    return base + incl - v;
}

}  // namespace ftv
