// Seeded Poisson noise for simulated counts (include/osscir.h,
// osscir_poisson_noise): c ~ Poisson(c^) elementwise, the way the paper's
// simulated data are made noisy (Sec. 3), on the device.
//
// Uniform numbers come from Philox4x32-10 (Salmon, Moraes, Dror, Shaw,
// "Parallel random numbers: as easy as 1, 2, 3", SC 2011): per round the two
// 32x32-bit products of words 0 and 2 with 0xD2511F53 and 0xCD9E8D57 are mixed
// with words 1 and 3 and the key, and the key advances by 0x9E3779B9 and
// 0xBB67AE85.  Sample i takes its t-th draw from counter (i, t, 0, 0) under key
// (seed mod 2^32, seed / 2^32), two output words making one uniform with 53
// random bits.  Means below 10 are sampled by inverting the distribution
// function; larger ones by the transformed rejection with squeeze of Hormann
// (1993).  A count is what the FP64 statement of these draws (poisson_draw, every
// operation spelled as an _rn intrinsic, so no FMA contraction changes it) gives;
// poisson_fast finds the same count on the FP32 pipe wherever its error bounds
// allow no doubt.
#include <cstdint>

#include "../../include/osscir.h"
#include "osscir_dfl.cuh"

using namespace osscir;

namespace {

__device__ __forceinline__ uint4 philox10(uint4 x, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t lo0 = 0xD2511F53u * x.x, hi0 = __umulhi(0xD2511F53u, x.x);
        const uint32_t lo1 = 0xCD9E8D57u * x.z, hi1 = __umulhi(0xCD9E8D57u, x.z);
        x = make_uint4(hi1 ^ x.y ^ k0, lo1, hi0 ^ x.w ^ k1, lo0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return x;
}

// [0, 1) from the top 27 + 26 bits of two words
__device__ __forceinline__ double uniform53(uint32_t hi, uint32_t lo) {
    return __dmul_rn(__dadd_rn(__dmul_rn((double)(hi >> 5), 67108864.0), (double)(lo >> 6)),
                     1.0 / 9007199254740992.0);
}

// log k! : the log of the exact product up to 18! (< 2^53), else the Stirling
// series of log Gamma(k + 1) to its x^-7 term.
__device__ double log_kfact(double k) {
    if (k <= 18.0) {
        double p = 1.0;
        for (double i = 2.0; i <= k; i = __dadd_rn(i, 1.0)) p = __dmul_rn(p, i);
        return log(p);
    }
    const double x = __dadd_rn(k, 1.0), ix = __ddiv_rn(1.0, x), ix2 = __dmul_rn(ix, ix);
    double t = __dsub_rn(1.0 / 1260.0, __dmul_rn(ix2, 1.0 / 1680.0));
    t = __dsub_rn(1.0 / 360.0, __dmul_rn(ix2, t));
    t = __dsub_rn(1.0 / 12.0, __dmul_rn(ix2, t));
    const double series = __dmul_rn(ix, t);
    const double main = __dsub_rn(__dmul_rn(__dsub_rn(x, 0.5), log(x)), x);
    return __dadd_rn(__dadd_rn(main, 0.91893853320467274178), series);
}

__device__ double poisson_draw(double lam, uint32_t i, uint32_t k0, uint32_t k1) {
    if (!(lam > 0.0)) return 0.0;
    if (lam < 10.0) {
        const uint4 r = philox10(make_uint4(i, 0u, 0u, 0u), k0, k1);
        const double u = uniform53(r.x, r.y);
        double p = exp(-lam), F = p, k = 0.0;
        while (u > F && k < 1000.0) {
            k = __dadd_rn(k, 1.0);
            p = __ddiv_rn(__dmul_rn(p, lam), k);
            F = __dadd_rn(F, p);
        }
        return k;
    }
    const double slam = sqrt(lam), loglam = log(lam);
    const double b = __dadd_rn(0.931, __dmul_rn(2.53, slam));
    const double a = __dadd_rn(-0.059, __dmul_rn(0.02483, b));
    const double invalpha = __dadd_rn(1.1239, __ddiv_rn(1.1328, __dsub_rn(b, 3.4)));
    const double vr = __dsub_rn(0.9277, __ddiv_rn(3.6224, __dsub_rn(b, 2.0)));
    for (uint32_t t = 0; t < 64u; ++t) {   // a trial is accepted with probability > 0.9
        const uint4 r = philox10(make_uint4(i, t, 0u, 0u), k0, k1);
        const double U = __dsub_rn(uniform53(r.x, r.y), 0.5), V = uniform53(r.z, r.w);
        const double us = __dsub_rn(0.5, fabs(U));
        const double slope = __dadd_rn(__ddiv_rn(__dmul_rn(2.0, a), us), b);
        const double k = floor(__dadd_rn(__dadd_rn(__dmul_rn(slope, U), lam), 0.43));
        if (us >= 0.07 && V <= vr) return k;
        if (k < 0.0 || (us < 0.013 && V > us)) continue;
        const double lhs =
            __dsub_rn(__dadd_rn(log(V), log(invalpha)), log(__dadd_rn(__ddiv_rn(a, __dmul_rn(us, us)), b)));
        const double rhs = __dsub_rn(__dadd_rn(-lam, __dmul_rn(k, loglam)), log_kfact(k));
        if (lhs <= rhs) return k;
    }
    return floor(lam);
}

constexpr dfl dconst(double v) { return dfl{(float)v, (float)(v - (double)(float)v)}; }

// [0, 1) from the same 53 bits as uniform53, rounded to FP32.
__device__ __forceinline__ float uniform_f(uint32_t hi, uint32_t lo) {
    return ((float)(hi >> 5) + (float)(lo >> 6) * 0x1p-26f) * 0x1p-27f;
}

// (n + frac) 2^-27 for an integer 0 <= n < 2^26 and 0 <= frac <= 1.
__device__ __forceinline__ dfl fixed27(int n, float frac) {
    const float hi = (float)n;
    const dfl v = df_fast2sum(hi, (float)(n - (int)hi) + frac);
    return dfl{v.hi * 0x1p-27f, v.lo * 0x1p-27f};
}

// poisson_draw's count without FP64: every comparison (and the floor) is made in
// FP32 or double-float, and wherever the two sides are closer than a bound on the
// error of that arithmetic the draw is given up (returns false).  The bounds:
//   inversion: expf within 2 ulp and at most 1.2e-7 per later factor, so F is within
//     6e-6 of its FP64 value up to k = 60 (bound 1.6e-5);
//   the floor's argument: the double-float products and sums are within 2^-44 of
//     their size, and the position of us in [0, 1/2] is known to 2^-25 of its unit
//     2^-27 (a relative 3e-8 / n at position n);
//   the log test: rhs = -lam + k log lam - log k! by Stirling's series is
//     k (log1p(x) - x) - log(2 pi k) / 2 - 1/(12 k) + 1/(360 k^3) - 1/(1260 k^5) with
//     x = (lam - k) / k, all terms but the last two of one sign, so nothing cancels:
//     within 5e-6 of its size; the logs of lhs within 5e-6 (bound 1e-3 + 1e-5 |rhs|).
// What bounds it: instruction issue (about 400 instructions a trial, two to three
// trials until every lane of a warp has accepted).  4 x 1024 x 1024 counts take
// 57 us at a mean of 3, 511 us at 30 (the log test's log1pf branch), 217 us at 1000
// and above; the FP64 form alone, bound by the FP64 pipe (1/64 of the FP32 rate),
// took 3302 us for the counts of a 512 x 512 study.
__device__ __forceinline__ bool poisson_fast(float lam, uint32_t i, uint32_t k0, uint32_t k1, float& out) {
    if (!(lam > 0.0f)) {
        out = 0.0f;
        return true;
    }
    if (lam < 10.0f) {
        const uint4 r = philox10(make_uint4(i, 0u, 0u, 0u), k0, k1);
        const float u = uniform_f(r.x, r.y);
        float p = expf(-lam), F = p;
        for (float k = 0.0f; k < 60.0f;) {
            const float d = u - F;
            if (fabsf(d) < 1.6e-5f) return false;
            if (d < 0.0f) {
                out = k;
                return true;
            }
            k += 1.0f;
            p = p * lam / k;
            F += p;
        }
        return false;
    }
    if (!(lam < 16777216.0f)) return false;
    const dfl b = df_add(dconst(0.931), df_mul(dconst(2.53), df_sqrt(dfl{lam, 0.0f})));
    const dfl a = df_add(dconst(-0.059), df_mul(dconst(0.02483), b));
    const float vr = 0.9277f - 3.6224f / (b.hi - 2.0f);
    const float li = floorf(lam), lf = lam - li;
    for (uint32_t t = 0; t < 32u; ++t) {
        const uint4 r = philox10(make_uint4(i, t, 0u, 0u), k0, k1);
        // |U| = (m + f) 2^-27 and us = 1/2 - |U| = (n + 1 - f) 2^-27
        const int s = (int)(r.x >> 5) - (1 << 26);
        const bool neg = s < 0;
        const int m = neg ? -s - 1 : s, n = (1 << 26) - 1 - m;
        const float bits = (float)(r.y >> 6) * 0x1p-26f, f = neg ? 1.0f - bits : bits;
        if (n < 1024) return false;
        const dfl us = fixed27(n, 1.0f - f);
        const dfl slope = df_add(df_mul(dfl{2.0f * a.hi, 2.0f * a.lo}, df_rcp_fma(us)), b);
        const dfl su = df_mul(slope, fixed27(m, f));
        const dfl v = df_add(df_add(neg ? df_neg(su) : su, dconst(0.43)), dfl{lf, 0.0f});
        const float fl = floorf(v.hi), fr = (v.hi - fl) + v.lo;
        const float gap = 2e-6f + fabsf(v.hi) * (1e-12f + 6e-8f / (float)n);
        const float k = li + fl;
        if (!(fabsf(v.hi) < 4e6f) || !(fr > gap) || !(fr < 1.0f - gap) || !(k < 16777216.0f)) return false;
        const float V = uniform_f(r.z, r.w);
        if (fabsf(us.hi - 0.07f) < 1e-7f || fabsf(us.hi - 0.013f) < 1e-7f) return false;
        if (us.hi > 0.07f) {
            if (fabsf(V - vr) < 4e-6f) return false;
            if (V < vr) {
                out = k;
                return true;
            }
        }
        if (k < 0.0f) continue;
        if (us.hi < 0.013f) {
            if (fabsf(V - us.hi) < 1e-6f * us.hi) return false;
            if (V > us.hi) continue;
        }
        if (k < 4.0f || V < 1e-6f) return false;
        const float invalpha = 1.1239f + 1.1328f / (b.hi - 3.4f);
        const float lhs = logf(V * invalpha / (a.hi / (us.hi * us.hi) + b.hi));
        const float x = (lam - k) / k, ik = 1.0f / k, ik2 = ik * ik;
        float h;   // log1p(x) - x
        if (fabsf(x) < 0.125f)
            h = -x * x *
                (0.5f - x * (1.0f / 3.0f - x * (0.25f - x * (0.2f - x * (1.0f / 6.0f - x * (1.0f / 7.0f - x * (0.125f - x * (1.0f / 9.0f))))))));
        else
            h = log1pf(x) - x;
        const float tail = ik * (1.0f / 12.0f - ik2 * (1.0f / 360.0f - ik2 * (1.0f / 1260.0f)));
        const float rhs = k * h - 0.5f * logf(6.28318531f * k) - tail;
        const float diff = rhs - lhs;
        if (!(fabsf(diff) >= 1e-3f + 1e-5f * fabsf(rhs))) return false;
        if (diff > 0.0f) {
            out = k;
            return true;
        }
    }
    return false;
}

__device__ __noinline__ float poisson_exact(float lam, uint32_t i, uint32_t k0, uint32_t k1) {
    return (float)poisson_draw((double)lam, i, k0, k1);
}

__global__ void k_poisson_noise(const float* __restrict__ chat, int n, uint32_t k0, uint32_t k1,
                                float* __restrict__ c) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float lam = chat[i];
        float k;
        if (!poisson_fast(lam, (uint32_t)i, k0, k1, k)) k = poisson_exact(lam, (uint32_t)i, k0, k1);
        c[i] = k;
    }
}

}  // namespace

extern "C" osscir_status osscir_poisson_noise(const float* chat, int n, uint64_t seed, float* c, void* stream) {
    if (n < 0 || (n > 0 && (!chat || !c))) return OSSCIR_E_INVALID;
    if (n == 0) return OSSCIR_OK;
    // a grid-stride loop over at most 64 blocks per SM of the current device
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        return OSSCIR_E_CUDA;
    const int threads = 256, need = (n + threads - 1) / threads, blocks = need < sms * 64 ? need : sms * 64;
    k_poisson_noise<<<blocks, threads, 0, static_cast<cudaStream_t>(stream)>>>(
        chat, n, (uint32_t)seed, (uint32_t)(seed >> 32), c);
    return cudaGetLastError() == cudaSuccess ? OSSCIR_OK : OSSCIR_E_CUDA;
}
