// The passes that come before an NVFP4 reconstruction of a tensor (which needs
// the tensor's absmax before any block is processed): the absmax of w, or one
// AdamW step that also takes the absmax of the updated weights.  The arithmetic
// is the integer kernel's fused step, element for element: packed fp32, the root
// as v' rsqrt(v'), the quotient by the fast reciprocal, and w' = w + (-(w lr wd)
// - step m'/den) rounded once.
#pragma once

#include <cuda_bf16.h>

#include <cstdint>

#include "device_common.cuh"
#include "params.h"

namespace quasar {

// The step's constants, packed, and the step on four elements: w, m and v are
// replaced, amax takes the largest |w'|.
struct AdamwStep {
    float2 beta1, c1b, beta2, c1, nlrwd, nstep, isbc2, eps;
    __device__ __forceinline__ explicit AdamwStep(const AdamwHp& hp)
        : beta1(make_float2(hp.beta1, hp.beta1)),
          c1b(make_float2(hp.c1b, hp.c1b)),
          beta2(make_float2(hp.beta2, hp.beta2)),
          c1(make_float2(hp.c1, hp.c1)),
          nlrwd(make_float2(-hp.lr_wd, -hp.lr_wd)),
          nstep(make_float2(-hp.step_size, -hp.step_size)),
          isbc2(make_float2(hp.isbc2, hp.isbc2)),
          eps(make_float2(hp.eps, hp.eps))
    {
    }
    __device__ __forceinline__ void operator()(float4& w, float4& m, float4& v, const float4& g, float& amax) const
    {
        const float2 gv[2] = {make_float2(g.x, g.y), make_float2(g.z, g.w)};
        float2 wv[2] = {make_float2(w.x, w.y), make_float2(w.z, w.w)};
        float2 mv[2] = {make_float2(m.x, m.y), make_float2(m.z, m.w)};
        float2 hv[2] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
#pragma unroll
        for (int pr = 0; pr < 2; ++pr) {
            mv[pr] = __ffma2_rn(mv[pr], beta1, __fmul2_rn(c1b, gv[pr]));
            hv[pr] = __ffma2_rn(hv[pr], beta2, __fmul2_rn(c1, __fmul2_rn(gv[pr], gv[pr])));
            float2 sq = __fmul2_rn(hv[pr], make_float2(rsqrtf(hv[pr].x), rsqrtf(hv[pr].y)));
            sq.x = hv[pr].x > 0.0f ? sq.x : 0.0f;
            sq.y = hv[pr].y > 0.0f ? sq.y : 0.0f;
            const float2 den = __ffma2_rn(sq, isbc2, eps);
            const float2 upd = make_float2(__fdividef(mv[pr].x, den.x), __fdividef(mv[pr].y, den.y));
            const float2 t = __ffma2_rn(wv[pr], nlrwd, __fmul2_rn(nstep, upd));
            wv[pr] = __fadd2_rn(wv[pr], t);
            amax = fmax3(amax, fabsf(wv[pr].x), fabsf(wv[pr].y));
        }
        w = make_float4(wv[0].x, wv[0].y, wv[1].x, wv[1].y);
        m = make_float4(mv[0].x, mv[0].y, mv[1].x, mv[1].y);
        v = make_float4(hv[0].x, hv[0].y, hv[1].x, hv[1].y);
    }
};

// The largest |w| of float4 groups i, i + stride, ... of n elements, UN of them
// in flight at a time, and of the last n % 4 elements.
template <int UN>
__device__ __forceinline__ float amax_span(const float* w, int64_t n, int64_t i, int64_t stride)
{
    float m = 0.0f;
    const int64_t n4 = n / 4;
    if (i < n - n4 * 4) m = fabsf(w[n4 * 4 + i]);
    const float4* w4 = reinterpret_cast<const float4*>(w);
    for (; i < n4; i += UN * stride) {
        float4 x[UN];
#pragma unroll
        for (int j = 0; j < UN; ++j)
            x[j] = i + j * stride < n4 ? __ldcs(w4 + i + j * stride) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int j = 0; j < UN; ++j)
            m = fmax3(fmax3(m, fabsf(x[j].x), fabsf(x[j].y)), fabsf(x[j].z), fabsf(x[j].w));
    }
    return m;
}

// A warp's largest value into *slot, as the bit pattern of a non-negative
// float (such patterns order like uints).
__device__ __forceinline__ void amax_to_slot(float m, float* slot)
{
    m = lanes_max(m, 0xffffffffu);
    if ((threadIdx.x & 31) == 0 && m > 0.0f) atomicMax(reinterpret_cast<unsigned int*>(slot), __float_as_uint(m));
}

// The same over a whole block of 8 warps: one atomic a block.
__device__ __forceinline__ void block_amax_to_slot(float m, float* slot)
{
    __shared__ float red[8];
    m = lanes_max(m, 0xffffffffu);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) amax_to_slot(red[threadIdx.x & 7], slot);
}

// The step alone: blockIdx.y picks the tensor; each thread takes 4 consecutive
// elements at a time (n is a multiple of 16).  *slot must start at 0.
template <int MAXT>
__global__ void __launch_bounds__(256) k_adamw_amax(const __grid_constant__ AdamwBatch<MAXT> B)
{
    const AdamwItem& it = B.t[blockIdx.y];
    if (it.n == 0) return;
    const AdamwStep step(B.hp);
    float amax = 0.0f;
    const int64_t n4 = it.n / 4;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
        float4 w = __ldcs(reinterpret_cast<const float4*>(it.w) + i);
        float4 m = __ldcs(reinterpret_cast<const float4*>(it.m) + i);
        float4 v = __ldcs(reinterpret_cast<const float4*>(it.v) + i);
        float4 g;
        if (B.hp.g_kind == 2) {
            const uint2 gb = __ldcs(reinterpret_cast<const uint2*>(it.g) + i);
            g = make_float4(bf16lo(gb.x), bf16hi(gb.x), bf16lo(gb.y), bf16hi(gb.y));
        } else {
            g = __ldcs(reinterpret_cast<const float4*>(it.g) + i);
        }
        step(w, m, v, g, amax);
        __stcs(reinterpret_cast<float4*>(it.w) + i, w);
        __stcs(reinterpret_cast<float4*>(it.m) + i, m);
        __stcs(reinterpret_cast<float4*>(it.v) + i, v);
    }
    block_amax_to_slot(amax, it.slot);
}

// The step beside another kernel's work, by few warps: warp `first` of `stride`
// takes units first, first + stride, ... (kAheadUnit weights of one tensor)
// through a ring of tiles filled by bulk copies.  (With plain loads, two float4
// groups a thread in flight, eight warps an SM reached 3.7 TB/s.)  False: a copy
// did not land in time.
template <int MAXT>
__device__ __forceinline__ bool adamw_ring(const AdamwBatch<MAXT>& B, unsigned char* ring, int64_t first,
                                           int64_t stride, uint64_t timeout_ns, unsigned int* status)
{
    constexpr int S = kAheadTiles;
    constexpr uint32_t kMOff = kAheadUnit * 4, kVOff = kAheadUnit * 8, kGOff = kAheadUnit * 12;
    const int lane = threadIdx.x & 31;
    const uint32_t gbytes = B.hp.g_kind == 2 ? 2u : 4u;
    const uint32_t tile = kAheadUnit * (12u + gbytes);
    uint64_t* bars = reinterpret_cast<uint64_t*>(ring + S * tile);
    const int64_t n_units = B.n_units;
    auto tensor_of = [&](int64_t u, int& ti) {
        while (ti + 1 < B.n_t && u >= B.t[ti + 1].unit0) ++ti;
    };
    int ti = 0;
    auto issue = [&](int64_t u, int s) {
        int tj = ti;
        tensor_of(u, tj);
        const AdamwItem& T = B.t[tj];
        const int64_t e0 = (u - T.unit0) * kAheadUnit;
        const uint32_t elems = (uint32_t)min((int64_t)kAheadUnit, T.n - e0);
        unsigned char* st = ring + s * tile;
        mbar_arrive_expect_tx(&bars[s], elems * (12u + gbytes));
        bulk_g2s(st, T.w + e0, elems * 4u, &bars[s]);
        bulk_g2s(st + kMOff, T.m + e0, elems * 4u, &bars[s]);
        bulk_g2s(st + kVOff, T.v + e0, elems * 4u, &bars[s]);
        bulk_g2s(st + kGOff, static_cast<const unsigned char*>(T.g) + e0 * gbytes, elems * gbytes, &bars[s]);
    };
    if (lane == 0) {
        for (int s = 0; s < S; ++s) mbar_init(&bars[s], 1);
        mbar_init_fence();
        for (int s = 0; s < S; ++s)
            if (first + s * stride < n_units) issue(first + s * stride, s);
    }
    __syncwarp();
    const AdamwStep step(B.hp);
    float amax = 0.0f;
    int s_cur = 0, ti_max = 0;
    uint32_t parity = 0;
    for (int64_t u = first; u < n_units; u += stride) {
        if (!warp_wait_bounded(&bars[s_cur], parity, timeout_ns)) {
            // record it, and wait (bounded) for the copies in flight
            if (lane == 0) record_timeout(status);
            for (int j = 0; j < S; ++j)
                if (u + j * stride < n_units)
                    mbar_wait_bounded(&bars[(s_cur + j) % S], parity ^ (s_cur + j >= S ? 1u : 0u), timeout_ns);
            return false;
        }
        tensor_of(u, ti);
        const AdamwItem& T = B.t[ti];
        if (ti != ti_max) {  // a new tensor: hand in the last one's
            amax_to_slot(amax, B.t[ti_max].slot);
            amax = 0.0f;
            ti_max = ti;
        }
        const unsigned char* st = ring + s_cur * tile;
        const int64_t e0 = (u - T.unit0) * kAheadUnit;
        const int elems = (int)min((int64_t)kAheadUnit, T.n - e0);
#pragma unroll 2
        for (int e = lane * 4; e < elems; e += 128) {
            float4 w = lds128(st + e * 4), m = lds128(st + kMOff + e * 4), v = lds128(st + kVOff + e * 4), g;
            if (gbytes == 2) {
                const uint2 gb = lds64(st + kGOff + e * 2);
                g = make_float4(bf16lo(gb.x), bf16hi(gb.x), bf16lo(gb.y), bf16hi(gb.y));
            } else {
                g = lds128(st + kGOff + e * 4);
            }
            step(w, m, v, g, amax);
            stg_cs(reinterpret_cast<float4*>(T.w + e0 + e), w);
            stg_cs(reinterpret_cast<float4*>(T.m + e0 + e), m);
            stg_cs(reinterpret_cast<float4*>(T.v + e0 + e), v);
        }
        __syncwarp();
        if (lane == 0 && u + S * stride < n_units) issue(u + S * stride, s_cur);
        if (++s_cur == S) {
            s_cur = 0;
            parity ^= 1u;
        }
    }
    amax_to_slot(amax, B.t[ti_max].slot);
    return true;
}

// Tensor absmax of a batch: blockIdx.y picks the tensor; max |w| over its n
// elements into *slot, which must start at 0.  Tensors whose amax is supplied
// are skipped.
template <int MAXT>
__global__ void __launch_bounds__(256) k_amax(const __grid_constant__ AmaxBatch<MAXT> B)
{
    const AmaxItem& it = B.t[blockIdx.y];
    if (it.amax_in || it.n == 0) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    block_amax_to_slot(amax_span<4>(it.w, it.n, i, (int64_t)gridDim.x * blockDim.x), it.slot);
}

}  // namespace quasar
