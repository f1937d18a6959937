// QUASAR with symmetric integer codes: the offset-free closed form of
// Sec. 4.1.2.  For each group and clip factor f: step s_f = f amax / Q
// (amax = max |w| of the group, Q = 2^(bits-1) - 1), codes
// q = clamp(round_half_even(w / s_f), -Q, Q), fit s* = sum h q w / sum h q^2,
// and the candidate whose error sum h (s* q - w)^2 = sum h w^2 - S3^2 / S2
// is lowest is kept (S2 = sum h q^2, S3 = sum h q w).
//
// Layout as the asymmetric kernel: a warp takes 8 groups a unit, 4 lanes a
// group, from a ring of tiles shared by the CTA's warps; the candidates' sums
// go to a table in the tile's gradient region.  (With 4 groups a unit, 8 lanes
// a group and a transpose of the sums through shared memory, the work that is
// not per weight and factor was half of all instructions: 91 a weight and
// lane.)  Codes come from magnitudes, min(rne(|w| P), Q), with the clamp taken
// once per set of candidates: for a set whose factors satisfy (Q - 1/2) f_max
// < tau < (Q + 1/2) f_min (with a margin the host checks), |w| capped at tau
// amax / Q rounds to Q for every factor of the set, and below the cap no code
// exceeds Q.
//
// Both sums are over non-negative terms (h |q|^2 and h |q| |w|), so each
// carries a small relative error and S3^2 / S2 a bound of a few ulps:
// candidates within the bound of the best are compared exactly (float-float
// direct errors, whole warp), and the kept fit needs no refinement.  Candidates
// of the best's very sums are settled by their codes.
//
// What bounds it: instruction issue and the FP32 pipe (5 packed operations a
// pair and candidate).  One Llama layer at INT4, group 128, 8 factors (clamp
// sets 3-3-2): 785 -> 566 us, 6.19 TB/s of algorithmic traffic (626 with two
// CTAs an SM and a fixed share of the tiles a warp; 20 warps at 96 registers 576).
#pragma once

#include <cuda_bf16.h>

#include <cstdint>
#include <type_traits>

#include "device_common.cuh"
#include "params.h"

namespace quasar {
namespace sym {

constexpr float kMagic = 8388608.0f;  // 2^23: adding it rounds to an integer (nearest even)
constexpr float kU = 5.9604645e-8f;
// Sums of saliencies beyond this are scaled by 2^-64: S2 and S3^2 stay finite.
constexpr float kLargeSaliency = 1073741824.0f;  // 2^30

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e)
{
    p = __fmul_rn(a, b);
    e = fmaf(a, b, -p);
}

__device__ __forceinline__ void ff_acc(float& hi, float& lo, float xh, float xl)
{
    float s, e;
    two_sum(hi, xh, s, e);
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(e, xl));
}

__device__ __forceinline__ void ff_norm(float& hi, float& lo)
{
    const float s = __fadd_rn(hi, lo);
    lo = __fsub_rn(lo, __fsub_rn(s, hi));
    hi = s;
}

__device__ __forceinline__ void ff_reduce32(float& hi, float& lo)
{
    ff_norm(hi, lo);
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, hi, o);
        const float ol = __shfl_xor_sync(0xffffffffu, lo, o);
        ff_acc(hi, lo, oh, ol);
        ff_norm(hi, lo);
    }
    // the float-pair sum is not symmetric in its operands, so lanes can end
    // one rounding apart: every lane takes lane 0's pair, so that decisions
    // taken from it are the same across the warp
    hi = __shfl_sync(0xffffffffu, hi, 0);
    lo = __shfl_sync(0xffffffffu, lo, 0);
}

// |q| = min(round_half_even(|w| P), Q) as a float
__device__ __forceinline__ float code_n(float aw, float P, float Q)
{
    return __fsub_rn(fminf(__fmaf_rn(aw, P, kMagic), kMagic + Q), kMagic);
}

}  // namespace sym


template <int EPL, int MAXT, int SS>
__global__ void __launch_bounds__(int_max_warps(EPL) * 32, 1) k_recon_sym(const __grid_constant__ IntLaunch<MAXT> Lp)
{
    using namespace sym;
    static_assert(SS == 1 || SS == 2 || SS == 3 || SS == 4 || SS == 8, "clamp sets of 1, 2, 4 or 8, or 3-3-2");
    // clamp sets a sweep of 8 candidates, and the set of the sweep's candidate
    // kk (its first slot is kq + set * SS)
    constexpr int NSETS = SS == 3 ? 3 : 8 / SS;
    auto set_of = [](int kk) { return SS == 3 ? (kk < 3 ? 0 : (kk < 6 ? 1 : 2)) : kk / SS; };
    const IntParams& p = Lp.p;
    constexpr int G = EPL * kIntLanes;
    constexpr int UNIT = kIntGroups * G;
    constexpr int NCHK = EPL / 4;  // 16-byte chunks per lane and group
    // chunk i of a lane is the group's chunk i ^ (gs & SWZ): the two (or
    // four) groups a shared-memory access phase covers then hit different
    // banks
    constexpr int SWZ = NCHK >= 4 ? 3 : (NCHK >= 2 ? 1 : 0);
    extern __shared__ __align__(128) unsigned char smem[];

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    const int gs = lane >> 2;
    const int sl = lane & 3;
    const int swz = gs & SWZ;

    // the CTA's ring: S tile slots, a full barrier each (and one spare for
    // the failure hook), and the sequence number of the tile each slot is
    // loading or holding
    const int S = p.stages;
    unsigned char* ring = smem;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)S * p.stage_bytes);
    volatile int* seq = reinterpret_cast<volatile int*>(bars + S + 1);
    int* next = const_cast<int*>(seq) + S;  // the first tile no warp has taken

    const int gbytes = p.g_kind == 2 ? 2 : (p.g_kind == 1 ? 4 : 0);
    // stage: w | v | g, then the candidates' table
    constexpr uint32_t kVOff = UNIT * 4;
    constexpr uint32_t kGOff = UNIT * 8;

    // tiles: the CTA takes units blockIdx.x + t * gridDim.x, t = 0 .. nt-1, its
    // warps the next tile that none has taken; tile t goes to slot t % S
    const int64_t n_units = Lp.n_units;
    const int nt = n_units > (int64_t)blockIdx.x
                       ? (int)((n_units - 1 - (int64_t)blockIdx.x) / gridDim.x + 1)
                       : 0;
    auto unit_of = [&](int t) { return (int64_t)blockIdx.x + (int64_t)t * gridDim.x; };
    // the tensor of a unit: units are numbered consecutively across the
    // launch's tensors, and each warp meets them in increasing order
    auto tensor_of = [&](int64_t u, int& ti) {
        while (ti + 1 < Lp.n_t && u >= Lp.t[ti + 1].unit0) ++ti;
    };
    int ti = 0;

    // (the unit issued is after the one being processed, or the first ones:
    // its tensor index is found from ti onwards)
    auto issue = [&](int t, int s) {
        const int64_t u = unit_of(t);
        int tj = ti;
        tensor_of(u, tj);
        const IntTensor& T = Lp.t[tj];
        const int64_t g0 = (u - T.unit0) * kIntGroups;
        const int64_t ng = min((int64_t)kIntGroups, T.n_groups - g0);
        const uint32_t elems = (uint32_t)(ng * G);
        unsigned char* st = ring + (size_t)s * p.stage_bytes;
        seq[s] = t;
        mbar_arrive_expect_tx(&bars[s], elems * (8u + (uint32_t)gbytes));
        bulk_g2s(st, T.w + g0 * G, elems * 4u, &bars[s]);
        bulk_g2s(st + kVOff, T.v + g0 * G, elems * 4u, &bars[s]);
        if (gbytes)
            bulk_g2s(st + kGOff, static_cast<const unsigned char*>(T.g) + g0 * G * gbytes,
                     elems * (uint32_t)gbytes, &bars[s]);
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s <= S; ++s) mbar_init(&bars[s], 1);
        for (int s = 0; s < S; ++s) seq[s] = -1;
        *next = nwarps;
        mbar_init_fence();
        for (int s = 0; s < S && s < nt; ++s) issue(s, s);
    }
    __syncthreads();

    // Record the failure and wait (bounded) until every tile issued into
    // the ring has landed, then leave.  (A copy that never lands is given up
    // on, and the CTA then exits with it still in flight.)
    auto fail = [&]() {
        if (lane == 0) record_timeout(p.status);
        for (int s = 0; s < S; ++s) {
            const int ts = seq[s];
            if (ts >= 0) mbar_wait_bounded(&bars[s], (uint32_t)((ts / S) & 1), p.timeout_ns);
        }
    };

    if (p.force_timeout_ns && blockIdx.x == 0 && warp == 0) {
        // Failure-path hook: a barrier nothing ever arrives on.
        if (!warp_wait_bounded(&bars[S], 0, p.force_timeout_ns)) {
            fail();
            return;
        }
    }

    const int Qi = (p.qmax - 1) >> 1;  // qmax = 2Q + 1 levels
    const float Q = (float)Qi;
    const int nch = (p.n_clip + 7) >> 3;  // chunks of 8 candidates
    const float2 beta22 = make_float2(p.beta2, p.beta2);
    const float2 c12 = make_float2(p.c1, p.c1);
    const float2 M2 = make_float2(kMagic, kMagic), nM2 = make_float2(-kMagic, -kMagic);
    const float gam = kU * p.tie_kappa;

    int slot = warp;  // t % S (warps < S)
    uint32_t parity = 0;  // (t / S) & 1
    for (int t = warp; t < nt;) {
        if (!warp_wait_seq(seq + slot, t, p.timeout_ns) ||
            !warp_wait_bounded(&bars[slot], parity, p.timeout_ns)) {
            fail();
            return;
        }
        const int64_t u = unit_of(t);
        unsigned char* st = ring + (size_t)slot * p.stage_bytes;
        float* ws = reinterpret_cast<float*>(st);
        float* hs = reinterpret_cast<float*>(st + kVOff);
        const unsigned char* gsm = st + kGOff;
        // candidates' table (the gradient region, free once pass A is done)
        float* red = reinterpret_cast<float*>(st + kGOff);

        tensor_of(u, ti);
        const IntTensor& T = Lp.t[ti];
        const int64_t grp = (u - T.unit0) * kIntGroups + gs;
        const bool valid = grp < T.n_groups;
        const int64_t gbase = grp * (int64_t)G;
        const float* gws = ws + gs * G;  // this lane's group in the tile
        float* ghs = hs + gs * G;
        auto eoff = [&](int i) { return 16 * (i ^ swz) + 4 * sl; };  // chunk i of this lane


        // ---- pass A: EMA (v' out), the fit's saliency h into the tile, amax
        // and the saliency mass of the group
        float amax = 0.0f, ss = 0.0f;
        {
            float* vout = T.v + gbase;
            auto pass_a = [&](auto gk) {
                constexpr int GK = decltype(gk)::value;
                float2 SS2 = make_float2(0.0f, 0.0f);
#pragma unroll 2
                for (int i = 0; i < NCHK; ++i) {
                    const int eo = eoff(i);
                    const int e = gs * G + eo;
                    const float4 w4 = lds128(ws + e);
                    float4 h4 = lds128(hs + e);
                    if constexpr (GK != 0) {
                        float2 gA, gB;
                        if constexpr (GK == 2) {
                            const uint2 gb = lds64(gsm + e * 2);
                            gA = make_float2(bf16lo(gb.x), bf16hi(gb.x));
                            gB = make_float2(bf16lo(gb.y), bf16hi(gb.y));
                        } else {
                            const float4 g4 = lds128(gsm + e * 4);
                            gA = make_float2(g4.x, g4.y);
                            gB = make_float2(g4.z, g4.w);
                        }
                        const float2 hA = __ffma2_rn(make_float2(h4.x, h4.y), beta22,
                                                     __fmul2_rn(c12, __fmul2_rn(gA, gA)));
                        const float2 hB = __ffma2_rn(make_float2(h4.z, h4.w), beta22,
                                                     __fmul2_rn(c12, __fmul2_rn(gB, gB)));
                        h4 = make_float4(hA.x, hA.y, hB.x, hB.y);
                        *reinterpret_cast<float4*>(hs + e) = h4;
                        if (valid) stg_cs(reinterpret_cast<float4*>(vout + eo), h4);
                    }
                    amax = fmax3(fmax3(amax, fabsf(w4.x), fabsf(w4.y)), fabsf(w4.z), fabsf(w4.w));
                    SS2 = __fadd2_rn(SS2, __fadd2_rn(make_float2(h4.x, h4.y), make_float2(h4.z, h4.w)));
                }
                ss = SS2.x + SS2.y;
            };
            if (p.g_kind == 2) pass_a(std::integral_constant<int, 2>{});
            else if (p.g_kind == 1) pass_a(std::integral_constant<int, 1>{});
            else pass_a(std::integral_constant<int, 0>{});
            if (p.h_mode != kSalEma) {
                // the fit's saliency is v'^2 or 1: rewrite h in the tile (v'
                // went out already) and take its sum again
                ss = 0.0f;
#pragma unroll 1
                for (int i = 0; i < NCHK; ++i) {
                    float4* hp = reinterpret_cast<float4*>(hs + gs * G + eoff(i));
                    float4 h4 = *hp;
                    h4 = p.h_mode == kSalEmaSquared
                             ? make_float4(h4.x * h4.x, h4.y * h4.y, h4.z * h4.z, h4.w * h4.w)
                             : make_float4(1.0f, 1.0f, 1.0f, 1.0f);
                    *hp = h4;
                    ss += (h4.x + h4.y) + (h4.z + h4.w);
                }
            }
        }
#pragma unroll
        for (int o = 2; o; o >>= 1) {
            amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            ss += __shfl_xor_sync(0xffffffffu, ss, o);
        }
        // all saliencies zero: h = 1; a sum of saliencies, or weights, near the
        // bottom of the fp32 range, or saliencies whose sums' square could leave
        // it at the top: scaled by a power of two in the tile
        float unscale = 1.0f;  // of the fit
        const bool h_out = ss < kTinySaliency || ss > kLargeSaliency, w_out = amax < kTinyWeights;  // (zeros stay zeros)
        if (__any_sync(0xffffffffu, h_out || w_out)) {
            if (h_out || w_out) {
                float s1 = 1.0f, s2 = 1.0f, t1 = 1.0f, t2 = 1.0f;
                if (ss > kLargeSaliency) s1 = 5.421011e-20f;  // 2^-64
                else if (h_out && ss > 0.0f) tiny_scale(ss, s1, s2);
                if (w_out) tiny_scale(amax, t1, t2);
#pragma unroll 1
                for (int i = 0; i < NCHK; ++i) {
                    float4* hp = reinterpret_cast<float4*>(hs + gs * G + eoff(i));
                    float4* wp = reinterpret_cast<float4*>(ws + gs * G + eoff(i));
                    const float4 h4 = *hp, w4 = *wp;
                    *hp = ss > 0.0f ? make_float4(h4.x * s1 * s2, h4.y * s1 * s2, h4.z * s1 * s2, h4.w * s1 * s2)
                                    : make_float4(1.0f, 1.0f, 1.0f, 1.0f);
                    *wp = make_float4(w4.x * t1 * t2, w4.y * t1 * t2, w4.z * t1 * t2, w4.w * t1 * t2);
                }
                amax = amax * t1 * t2;
                unscale = (1.0f / t2) * (1.0f / t1);  // a power of two from 2^-149 on: exact
            }
        }
        // the gradient region becomes the candidates' table: every lane is past
        // pass A, and the h rewrites above are visible to all lanes
        __syncwarp();
        const bool flat = !(amax > 0.0f);
        const float R = flat ? 0.0f : __fdividef(Q, amax);  // P = R / f

        // ---- candidates, a chunk of 8 a sweep over the tile: S2 and S3.  Lane
        // sl owns candidates 8 ch + sl and 8 ch + 4 + sl; row k of the group's
        // table: S2, S3, and the upper end of E's error interval.
        float4* tab = reinterpret_cast<float4*>(red) + gs;  // row k at tab[8 k]
        float Eb = -INFINITY;
        int kb = 0x7fff;
        const float rel = 3.0f * gam + 4.0f * kU;  // E's relative error
#pragma unroll 1
        for (int ch = 0; ch < nch; ++ch) {
            const int kq = ch * 8;
            float2 P2[8], A2[8], A3[8];
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                const float P = R * p.invf[kq + kk];
                P2[kk] = make_float2(P, P);
                A2[kk] = A3[kk] = make_float2(0.0f, 0.0f);
            }
            float cp[NSETS];
#pragma unroll
            for (int s = 0; s < NSETS; ++s) cp[s] = p.cap[kq + s * SS] * amax;
#pragma unroll 1
            for (int i = 0; i < NCHK; ++i) {
                const int e = eoff(i);
                const float4 w4 = lds128(gws + e);
                const float4 h4 = lds128(ghs + e);
#pragma unroll
                for (int pr = 0; pr < 2; ++pr) {
                    const float2 aw = pr ? make_float2(fabsf(w4.z), fabsf(w4.w)) : make_float2(fabsf(w4.x), fabsf(w4.y));
                    const float2 h = pr ? make_float2(h4.z, h4.w) : make_float2(h4.x, h4.y);
                    float2 wc[NSETS];
#pragma unroll
                    for (int s = 0; s < NSETS; ++s) wc[s] = make_float2(fminf(aw.x, cp[s]), fminf(aw.y, cp[s]));
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {
                        const float2 n = __fadd2_rn(__ffma2_rn(wc[set_of(kk)], P2[kk], M2), nM2);
                        const float2 t2 = __fmul2_rn(h, n);
                        A2[kk] = __ffma2_rn(t2, n, A2[kk]);
                        A3[kk] = __ffma2_rn(t2, aw, A3[kk]);
                    }
                }
            }
            // the group's 4 lanes scatter the sums while they add them (a step
            // exchanges the candidates the two lanes do not keep)
            float S[2][2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                float x[8], y[4];
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    const float2 a = c == 0 ? A2[kk] : A3[kk];
                    x[kk] = a.x + a.y;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {  // the pair 2 j, 2 j + 1: bit 0 of sl picks
                    const float keep = sl & 1 ? x[2 * j + 1] : x[2 * j], give = sl & 1 ? x[2 * j] : x[2 * j + 1];
                    y[j] = keep + __shfl_xor_sync(0xffffffffu, give, 1);
                }
#pragma unroll
                for (int qd = 0; qd < 2; ++qd) {
                    const float keep = sl & 2 ? y[2 * qd + 1] : y[2 * qd];
                    const float give = sl & 2 ? y[2 * qd] : y[2 * qd + 1];
                    S[qd][c] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
                }
            }
#pragma unroll
            for (int qd = 0; qd < 2; ++qd) {
                const int k = kq + qd * 4 + sl;
                const float S2 = S[qd][0], S3 = S[qd][1];
                float E = S3 * S3 * rcp_ftz(S2);
                if (!(S2 >= kMinNormal)) E = S2 > 0.0f ? __fdividef(S3 * S3, S2) : 0.0f;
                const bool real = k < p.n_clip;
                if (real && E > Eb) {  // strict: keeps the lower k of this lane
                    Eb = E;
                    kb = k;
                }
                tab[8 * k] = make_float4(S2, S3, 0.0f, real ? E + rel * E : -INFINITY);
            }
        }
        __syncwarp();

        // ---- argmax of E (ties: lowest index), contenders
#pragma unroll
        for (int o = 2; o; o >>= 1) {
            const float Eo = __shfl_xor_sync(0xffffffffu, Eb, o);
            const int ko = __shfl_xor_sync(0xffffffffu, kb, o);
            if (Eo > Eb || (Eo == Eb && ko < kb)) {
                Eb = Eo;
                kb = ko;
            }
        }
        if (kb > 0x7ff) kb = 0;
        const float4 tb = tab[8 * kb];
        const float S2b = tb.x, S3b = tb.y;
        // A candidate with the winner's sums bit for bit (a twin) almost always has
        // its codes too, and then its error: the winner, the lowest of them, is
        // kept.  But an element of tiny saliency can change its code without
        // moving the sums.  A code that changes moves S2 by its h at least, so
        // twins are certain where the group's smallest h exceeds twice S2's error
        // (their sums have it each); elsewhere their codes are compared.  Codes
        // move monotonically with 1/f, so (with the factors in order) a twin with
        // the winner's codes shares them with every candidate between the two, and
        // the twins, all above the winner, are taken from the highest down.  (INT4
        // g128 layer 568 -> 570 us, INT3 g32 without gradient 125 -> 129; 578 and
        // 138 with every twin's codes compared; a twin compared exactly, as the
        // contenders, 574 and 132.)
        unsigned set = 0, twins = 0;
        {
            const float lo = Eb - rel * Eb;
#pragma unroll 1
            for (int k = sl; k < p.n_clip; k += 4) {
                const float4 tk = tab[8 * k];
                const bool twin = tk.x == S2b && tk.y == S3b;
                if (k != kb && tk.w >= lo) {
                    if (twin) twins |= 1u << k;
                    else set |= 1u << k;
                }
            }
            if (__any_sync(0xffffffffu, twins != 0u)) {
                float hmn = INFINITY;
#pragma unroll (EPL <= 16 ? NCHK : 1)
                for (int i = 0; i < NCHK; ++i) {
                    const float4 h4 = lds128(ghs + eoff(i));
                    hmn = fmin3(fmin3(hmn, h4.x, h4.y), h4.z, h4.w);
                }
                const unsigned low = __ballot_sync(0xffffffffu, !(hmn > 2.001f * (gam + 2.0f * kU) * S2b));
                if (((low >> (gs * kIntLanes)) & 0xFu) == 0u) twins = 0u;
#pragma unroll 1
                while (__any_sync(0xffffffffu, twins != 0u)) {
                    // the group's highest (none left: the winner itself)
                    unsigned top = twins;
#pragma unroll
                    for (int o = 2; o; o >>= 1) top |= __shfl_xor_sync(0xffffffffu, top, o);
                    const int k = top ? 31 - __clz(top) : kb;
                    const float Pt = R * p.invf[k], Pw = R * p.invf[kb];
                    const float ct = p.cap[k] * amax, cw = p.cap[kb] * amax;
                    const float2 Pt2 = make_float2(Pt, Pt), Pw2 = make_float2(Pw, Pw);
                    uint32_t diff = 0;
#pragma unroll 1
                    for (int i = 0; i < NCHK; ++i) {
                        const float4 w4 = lds128(gws + eoff(i));
#pragma unroll
                        for (int pr = 0; pr < 2; ++pr) {
                            const float x = fabsf(pr ? w4.z : w4.x), y = fabsf(pr ? w4.w : w4.y);
                            const float2 nt = __ffma2_rn(make_float2(fminf(x, ct), fminf(y, ct)), Pt2, M2);
                            const float2 nw = __ffma2_rn(make_float2(fminf(x, cw), fminf(y, cw)), Pw2, M2);
                            diff |= __float_as_uint(nt.x) ^ __float_as_uint(nw.x);
                            diff |= __float_as_uint(nt.y) ^ __float_as_uint(nw.y);
                        }
                    }
                    const bool all = ((__ballot_sync(0xffffffffu, diff == 0u) >> (gs * kIntLanes)) & 0xFu) == 0xFu;
                    if (all && p.monotone) twins = 0u;
                    else twins &= ~(1u << k);
                    if (!all) set |= 1u << k;
                }
            }
            __syncwarp();
#pragma unroll
            for (int o = 2; o; o >>= 1) set |= __shfl_xor_sync(0xffffffffu, set, o);
        }
        if (set) set |= 1u << kb;

        // the fit; with sum h q^2 = 0 it is the candidate's step s_f
        float a_sel = S2b > 0.0f ? S3b / S2b : 0.0f;
        if (!flat && !(S2b > 0.0f)) a_sel = p.f[kb] * amax / Q;

        // ---- exact comparison: float-float direct errors, whole warp per group
        unsigned todo = __ballot_sync(0xffffffffu, valid && !flat && set != 0 && sl == 0);
        while (todo) {
            const int g = (__ffs(todo) - 1) >> 2;
            todo &= todo - 1;
            const int src = g * 4;
            const float gR = __shfl_sync(0xffffffffu, R, src);
            const float gamax = __shfl_sync(0xffffffffu, amax, src);
            unsigned gset = __shfl_sync(0xffffffffu, set, src);
            if (p.stats && lane == 0) atomicAdd(&p.stats[0], 1u);
            const float* tws = ws + g * G;
            const float* ths = hs + g * G;
            float best_h = 0.0f, best_l = 0.0f, best_a = 0.0f;
            int best_k = -1;
            while (gset) {
                const int k = __ffs(gset) - 1;
                gset &= gset - 1;
                const float P = gR * p.invf[k];
                float s2h = 0.0f, s2l = 0.0f, s3h = 0.0f, s3l = 0.0f;
#pragma unroll
                for (int m = 0; m < G / 32; ++m) {
                    const int e = lane + 32 * m;
                    const float w = tws[e], h = ths[e];
                    const float n = code_n(fabsf(w), P, Q);
                    float ph, pl;
                    two_prod(h, n * n, ph, pl);  // n^2 is exact (|n| <= 127)
                    ff_acc(s2h, s2l, ph, pl);
                    two_prod(h * n, fabsf(w), ph, pl);
                    pl = fmaf(fmaf(h, n, -h * n), fabsf(w), pl);
                    ff_acc(s3h, s3l, ph, pl);
                }
                ff_reduce32(s2h, s2l);
                ff_reduce32(s3h, s3l);
                float ah, al;
                if (s2h > 0.0f) {
                    ah = s3h / s2h;
                    float qh, ql;
                    two_prod(ah, s2h, qh, ql);
                    const float rr = __fsub_rn(__fsub_rn(__fadd_rn(__fsub_rn(s3h, qh), s3l), ql), ah * s2l);
                    al = rr / s2h;
                } else {
                    ah = p.f[k] * gamax / Q;
                    al = 0.0f;
                }
                float eh = 0.0f, el = 0.0f;
#pragma unroll
                for (int m = 0; m < G / 32; ++m) {
                    const int e = lane + 32 * m;
                    const float w = tws[e], h = ths[e];
                    const float q = copysignf(code_n(fabsf(w), P, Q), w);
                    // d = a q - w in float-float
                    float dh, dl, ph, pl;
                    two_prod(ah, q, ph, pl);
                    pl = fmaf(al, q, pl);
                    two_sum(ph, -w, dh, dl);
                    dl = __fadd_rn(dl, pl);
                    ff_norm(dh, dl);
                    float sh, sl2;
                    two_prod(dh, dh, sh, sl2);
                    sl2 = fmaf(2.0f * dh, dl, sl2);
                    float th, tl;
                    two_prod(h, sh, th, tl);
                    tl = fmaf(h, sl2, tl);
                    ff_acc(eh, el, th, tl);
                }
                ff_reduce32(eh, el);
                if (best_k < 0 || eh < best_h || (eh == best_h && el < best_l)) {
                    best_h = eh;
                    best_l = el;
                    best_k = k;
                    best_a = ah;
                }
            }
            if (gs == g) {
                kb = best_k;
                a_sel = best_a;
            }
        }

        // ---- outputs: r = a q, codes q + Q, a, b = -a Q, index
        a_sel *= unscale;
        const float Pk = R * p.invf[kb];
        const float capk = p.cap[kb] * amax;
        {
            const float2 a2 = make_float2(a_sel, a_sel), Pk2 = make_float2(Pk, Pk);
            auto outputs = [&](auto bf16, auto with_codes) {
#pragma unroll 2
                for (int i = 0; i < NCHK; ++i) {
                    const int eo = eoff(i);
                    const float4 w4 = lds128(gws + eo);
                    const float2 wc0 = make_float2(fminf(fabsf(w4.x), capk), fminf(fabsf(w4.y), capk));
                    const float2 wc1 = make_float2(fminf(fabsf(w4.z), capk), fminf(fabsf(w4.w), capk));
                    const float2 n0 = __fadd2_rn(__ffma2_rn(wc0, Pk2, M2), nM2);
                    const float2 n1 = __fadd2_rn(__ffma2_rn(wc1, Pk2, M2), nM2);
                    const float2 q0 = make_float2(copysignf(n0.x, w4.x), copysignf(n0.y, w4.y));
                    const float2 q1 = make_float2(copysignf(n1.x, w4.z), copysignf(n1.y, w4.w));
                    float2 r0 = __fmul2_rn(a2, q0), r1 = __fmul2_rn(a2, q1);
                    if (flat) r0 = r1 = make_float2(0.0f, 0.0f);
                    const int64_t ge = gbase + eo;
                    if (!valid) {
                    } else if constexpr (decltype(bf16)::value) {
                        stg_cs(reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(T.r) + ge),
                               make_uint2(pack_bf16x2(r0.x, r0.y), pack_bf16x2(r1.x, r1.y)));
                    } else {
                        stg_cs(reinterpret_cast<float4*>(static_cast<float*>(T.r) + ge),
                               make_float4(r0.x, r0.y, r1.x, r1.y));
                    }
                    if constexpr (decltype(with_codes)::value) {
                        const uint32_t c0 = (uint32_t)(int)(q0.x + Q) | ((uint32_t)(int)(q0.y + Q) << 8);
                        const uint32_t c1 = (uint32_t)(int)(q1.x + Q) | ((uint32_t)(int)(q1.y + Q) << 8);
                        const uint32_t cw = flat ? (uint32_t)Qi * 0x01010101u : c0 | (c1 << 16);
                        if (valid) stg_cs(reinterpret_cast<uint32_t*>(T.codes + ge), cw);
                    }
                }
            };
            const bool u8 = T.codes != nullptr && !p.codes_packed;
            if (p.r_bf16 && !u8) outputs(std::true_type{}, std::false_type{});
            else if (p.r_bf16) outputs(std::true_type{}, std::true_type{});
            else if (!u8) outputs(std::false_type{}, std::false_type{});
            else outputs(std::false_type{}, std::true_type{});
        }
        if (T.codes && p.codes_packed) {
            // the packed format of the asymmetric kernel: each 32-code span fills
            // `bits` words; in two steps, each of the 4 lanes ORs a 4-code field
            // into them in the table's place, and lanes sl and sl + 4 of the
            // span's words are stored
            uint32_t* wsc = reinterpret_cast<uint32_t*>(red) + gs * 8;
#pragma unroll 1
            for (int m = 0; m < G / 32; ++m) {
                __syncwarp();
                wsc[sl] = 0u;
                wsc[sl + 4] = 0u;
                __syncwarp();
#pragma unroll
                for (int j2 = 0; j2 < 2; ++j2) {
                    const int c0 = 16 * j2 + 4 * sl;  // first code of the field
                    uint32_t pk = 0;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float wv = gws[32 * m + c0 + j];
                        const float q = flat ? 0.0f : copysignf(code_n(fabsf(wv), Pk, Q), wv);
                        pk |= (uint32_t)(int)(q + Q) << (j * p.bits);
                    }
                    const uint32_t o = (uint32_t)c0 * (uint32_t)p.bits;
                    const uint64_t f = (uint64_t)pk << (o & 31u);
                    atomicOr(&wsc[o >> 5], (uint32_t)f);
                    if ((uint32_t)(f >> 32)) atomicOr(&wsc[(o >> 5) + 1], (uint32_t)(f >> 32));
                }
                __syncwarp();
                uint32_t* dst = reinterpret_cast<uint32_t*>(T.codes) + grp * (int64_t)(G / 32) * p.bits + m * p.bits;
                if (valid && sl < p.bits) stg_cs(dst + sl, wsc[sl]);
                if (valid && sl + 4 < p.bits) stg_cs(dst + sl + 4, wsc[sl + 4]);
            }
            __syncwarp();
        }
        if (valid && sl == 0) {
            T.a[grp] = flat ? 0.0f : a_sel;
            T.b[grp] = flat ? 0.0f : -a_sel * Q;
            if (T.idx) T.idx[grp] = flat ? 0 : (uint8_t)kb;
        }

        // release the tile: all lanes are done with it; order our generic
        // writes to it before the async-proxy copy that refills it with the
        // slot's next tile
        __syncwarp();
        if (lane == 0 && t + S < nt) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue(t + S, slot);
        }
        int tn = 0;
        if (lane == 0) tn = atomicAdd(next, 1);
        tn = __shfl_sync(0xffffffffu, tn, 0);
        for (slot += tn - t; slot >= S; slot -= S) parity ^= 1u;
        t = tn;
    }
}

}  // namespace quasar
