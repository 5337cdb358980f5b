// Full accumulation (K = 0), forward and backward: how a warp's lanes share
// the products of its 32 pixels with the surfels' feature rows.
#pragma once

#include "fss_internal.cuh"
#include "kernels.cuh"
#include "render_common.cuh"

#include <climits>

namespace fss {

constexpr int FULL_THREADS = 128;  // threads per CTA (64 for 8 x 8 tiles): parts of a tile
template <int TS>
constexpr int full_threads() {
    return TS * TS < FULL_THREADS ? TS * TS : FULL_THREADS;
}

// CL lanes share a row's channels, 32 / CL groups of them the pixels: lane l has
// pixels PX (l / CL) on, and of the row the NQ quads of channels 4 (l % CL + CL q).
// With PX = CL a sum over the channels' lanes that leaves one pixel per lane
// leaves each lane its own.  Shared-memory reads per surfel fall from the row's
// C x 4 bytes per lane to (PX + 4 NQ) x 4 (64 channels: 64 cycles of the SM's
// load path to 16).
template <int CMAX>
struct FullLanes {
    static constexpr int CL = CMAX >= 32 ? 8 : 4, PX = CL, NQ = CMAX / (4 * CL);

    static __device__ __forceinline__ float4 load4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
    static __device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
        return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                           __uint_as_float(v.y & 0xffff0000u));
    }
    // the lane's quads of a row (zeros past C)
    template <typename FT>
    static __device__ __forceinline__ void load_row(const FT* row, int cg, int C, float4 (&f)[NQ]) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int c = 4 * (cg + CL * q);
            f[q] = c < C ? load4(row + c) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
    }
    // ... of a row in shared memory, whose channels past C are zeros or unused
    template <typename FT>
    static __device__ __forceinline__ void lds_row(const FT* row, int cg, float4 (&f)[NQ]) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) f[q] = lds4(row + 4 * (cg + CL * q));
    }
    static __device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }
    static __device__ __forceinline__ float4 lds4(const __nv_bfloat16* p) {
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                           __uint_as_float(v.y & 0xffff0000u));
    }
    // PX consecutive pixels' weights in shared memory
    static __device__ __forceinline__ void load_weights(const float* s, float (&w)[PX]) {
#pragma unroll
        for (int i = 0; i < PX / 4; ++i) {
            const float4 v = reinterpret_cast<const float4*>(s)[i];
            w[4 * i] = v.x;
            w[4 * i + 1] = v.y;
            w[4 * i + 2] = v.z;
            w[4 * i + 3] = v.w;
        }
    }
    // Argmax over a pixel's channels, the lowest among equals, NaN only where it is
    // channel 0 (no comparison moves away from it); -1 without contributors.  Called by whole warps.
    static __device__ __forceinline__ void label(const float2 (&acc)[NQ][2], int cg, int C, bool any, int32_t* out) {
        float bv = -INFINITY;
        int bc = INT_MAX;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float v[4] = {acc[q][0].x, acc[q][0].y, acc[q][1].x, acc[q][1].y};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int c = 4 * (cg + CL * q) + e;
                if (c < C && (v[e] > bv || (v[e] == bv && c < bc))) {
                    bv = v[e];
                    bc = c;
                }
            }
        }
        if (cg == 0 && acc[0][0].x != acc[0][0].x) {
            bv = INFINITY;
            bc = -1;
        }
#pragma unroll
        for (int o = 1; o < CL; o <<= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oc = __shfl_xor_sync(0xffffffffu, bc, o);
            if (ov > bv || (ov == bv && oc < bc)) {
                bv = ov;
                bc = oc;
            }
        }
        if (out && cg == 0) *out = any ? max(bc, 0) : -1;
    }
};

}  // namespace fss
