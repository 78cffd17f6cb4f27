// Device helpers of the binary64 fixed-point H*v (hv_phases.cu): the
// binary64 <-> fixed-point conversions, the epilogue parameters, and the fused
// Lanczos reductions.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "internal.h"

namespace hub {

// ---------------------------------------------------------------------------
// binary64 <-> fixed point
__device__ __forceinline__ void fx_split(double x, int emax, int& lo, int& hi) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FF);
    unsigned long long mant = b & ((1ull << 52) - 1);
    if (e != 0) mant |= (1ull << 52);
    const int ee = e > 0 ? e : 1;
    const int rs = max(emax - ee + 5, 1);             // >= 5 whenever |x| < 2^(emax-1022)
    long long X = (rs >= 60) ? 0 : (long long)((mant + (1ull << (rs - 1))) >> rs);
    if (b >> 63) X = -X;
    lo = (int)(X & 0xFFFFFF);
    hi = (int)(X >> 24);
}

__device__ __forceinline__ long long fx_join(int lo, int hi) { return ((long long)hi << 24) + (long long)lo; }

struct I128 {
    unsigned long long lo;
    long long hi;
};

__device__ __forceinline__ void mac128(I128& acc, long long a, long long b) {
    const unsigned long long plo = (unsigned long long)a * (unsigned long long)b;
    const long long phi = __mul64hi(a, b);
    const unsigned long long nlo = acc.lo + plo;
    acc.hi += phi + (nlo < plo ? 1 : 0);
    acc.lo = nlo;
}

// acc + a * 2^s, 0 <= s < 62 (a product with a power of two)
__device__ __forceinline__ void addshift128(I128& acc, long long a, int s) {
    const unsigned long long plo = (unsigned long long)a << s;
    const long long phi = s == 0 ? a >> 63 : a >> (64 - s);
    const unsigned long long nlo = acc.lo + plo;
    acc.hi += phi + (nlo < plo ? 1 : 0);
    acc.lo = nlo;
}

// (hi * 2^64 + lo) * 2^e2, rounded to nearest (ties to even)
__device__ __forceinline__ double i128_to_double(I128 v, int e2) {
    unsigned long long lo = v.lo;
    unsigned long long hi = (unsigned long long)v.hi;
    const bool neg = v.hi < 0;
    if (neg) {
        lo = ~lo + 1ull;
        hi = ~hi + (lo == 0 ? 1ull : 0ull);
    }
    if (hi == 0 && lo == 0) return 0.0;
    const int lz = hi ? __clzll((long long)hi) : 64 + __clzll((long long)lo);
    unsigned long long nh, nl;
    if (lz == 0) {
        nh = hi;
        nl = lo;
    } else if (lz < 64) {
        nh = (hi << lz) | (lo >> (64 - lz));
        nl = lo << lz;
    } else {
        nh = lo << (lz - 64);
        nl = 0;
    }
    unsigned long long mant = nh >> 11;               // 53 bits, leading one at bit 52
    const unsigned long long rem = nh & 0x7FFull;
    const bool up = (rem > 0x400ull) || (rem == 0x400ull && (nl != 0 || (mant & 1ull)));
    mant += up ? 1ull : 0ull;
    int ex = 127 - lz + e2;
    if (mant == (1ull << 53)) {
        mant >>= 1;
        ++ex;
    }
    const int be = ex + 1023;
    if (be <= 0 || be >= 2047) {
        const double m = (double)mant;                // exact
        return ldexp(neg ? -m : m, ex - 52);
    }
    unsigned long long bits = ((unsigned long long)be << 52) | (mant & ((1ull << 52) - 1));
    if (neg) bits |= (1ull << 63);
    return __longlong_as_double((long long)bits);
}

// P * 2^e2, correctly rounded (ties to even), by integer operations: the 64-bit
// integer -> binary64 conversion costs five slots of the FP64 pipe (two lanes a
// clock on this part), which kept that pipe busy for 1.4 ms of the 2.1 ms up
// phase of a 1.7e8-element product; about 20 integer operations give the same
// bits.  The rounded mantissa (leading one at bit 52) is added to the exponent
// field, so a carry out of it raises the exponent; results off the normal
// range go through ldexp.
__device__ __forceinline__ double i64_scaled_to_double(long long P, int e2) {
    if (P == 0) return 0.0;
    const unsigned long long m = P < 0 ? 0ull - (unsigned long long)P : (unsigned long long)P;
    const int lz = __clzll((long long)m);
    const int be = 1086 - lz + e2;                    // biased exponent of 2^(63 - lz) * 2^e2
    if (be <= 0 || be >= 2046) return ldexp(__ll2double_rn(P), e2);
    const unsigned long long n = m << lz;
    unsigned long long mant = n >> 11;
    mant += ((unsigned)n & 0x7FFu) + ((unsigned)mant & 1u) > 0x400u ? 1ull : 0ull;
    const unsigned long long bits = (mant + ((unsigned long long)(be - 1) << 52)) | ((unsigned long long)P & (1ull << 63));
    return __longlong_as_double((long long)bits);
}


struct EpiParams {
    long long A;          // round(-t * 2^m)
    long long Bbeta;      // round(-beta * 2^m)
    long long B[33];      // round(U * n * 2^m), n = 0..32
    int m;
    int nB;
    // exact int64 path, valid when t = +-2^et and U * 2^ju is a small integer:
    //   value = (sgn_t * T * 2^(et+ju) + Uint * n * X) * 2^-(k+ju)
    int fast;
    int tshift;           // et + ju >= 0
    int tneg;             // t < 0
    int ju;
    long long Uint;       // U * 2^ju
    double mbeta;         // -beta, applied after the exact part in the int64 path
    int apow;             // A = +-2^apow exactly (t a power of two), or -1
};

// The int64 epilogue of one element (EpiParams::fast), exact: T the hop sum, xo the
// own element's words, n the doubly occupied sites; |T| < 2^55, |X| <= 2^48,
// |Uint n| < 2^14 and tshift <= 6.  The own element's words are multiplied apart
// (32 x 32 -> 64 bits) and joined once.
__device__ __forceinline__ long long fast_sum(long long T, int2 xo, int n, const EpiParams& ep) {
    const int c = (int)ep.Uint * n;
    const long long t = T << ep.tshift;
    return (ep.tneg ? t : -t) + (((long long)c * xo.y) << 24) + (long long)c * xo.x;
}

// acc += A T: a shift where t is a power of two (the same 128-bit value)
__device__ __forceinline__ void mac_t(I128& acc, long long T, const EpiParams& ep) {
    if (ep.apow >= 0) addshift128(acc, ep.A < 0 ? -T : T, ep.apow);
    else mac128(acc, T, ep.A);
}

__device__ __forceinline__ void add4(int4& A, int4 a, int4 b, int4 c, int4 d) {
    A.x += a.x + b.x + c.x + d.x;
    A.y += a.y + b.y + c.y + d.y;
    A.z += a.z + b.z + c.z + d.z;
    A.w += a.w + b.w + c.w + d.w;
}
__device__ __forceinline__ void add4(int4& A, int4 a) {
    A.x += a.x; A.y += a.y; A.z += a.z; A.w += a.w;
}
__device__ __forceinline__ void add4(int2& A, int2 a, int2 b, int2 c, int2 d) {
    A.x += a.x + b.x + c.x + d.x;
    A.y += a.y + b.y + c.y + d.y;
}
__device__ __forceinline__ void add4(int2& A, int2 a) { A.x += a.x; A.y += a.y; }
__device__ __forceinline__ void sub4(int4& A, int4 a, int4 b, int4 c, int4 d) {
    A.x -= a.x + b.x + c.x + d.x;
    A.y -= a.y + b.y + c.y + d.y;
    A.z -= a.z + b.z + c.z + d.z;
    A.w -= a.w + b.w + c.w + d.w;
}
__device__ __forceinline__ void sub4(int4& A, int4 a) {
    A.x -= a.x; A.y -= a.y; A.z -= a.z; A.w -= a.w;
}
__device__ __forceinline__ void sub4(int2& A, int2 a, int2 b, int2 c, int2 d) {
    A.x -= a.x + b.x + c.x + d.x;
    A.y -= a.y + b.y + c.y + d.y;
}
__device__ __forceinline__ void sub4(int2& A, int2 a) { A.x -= a.x; A.y -= a.y; }


// Lanczos reductions fused into the up-phase epilogue (Algorithm 1): each
// thread accumulates <w, f>, <w, w> and <f, f> over its outputs in a fixed
// order, the CTA sums its threads, and the last CTA the per-CTA partials
// (part[b], part[kPartStride + b], part[2 kPartStride + b]), in fixed trees, so
// the result is deterministic.  binary32 outputs, like the stand-alone dot
// kernels, use a float-float accumulator: each product is split exactly (p + e
// with e = fma(x, y, -p)) and added with Knuth's TwoSum, so the FP32 pipe carries
// some 48 bits and the binary64 pipe (two lanes a clock) is touched once per
// thread, not per element.
struct FFAcc {
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add_product(float x, float y) {
        const float p = x * y;
        const float e = fmaf(x, y, -p);
        const float t = hi + p;
        const float bb = t - hi;
        lo += ((hi - (t - bb)) + (p - bb)) + e;
        hi = t;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// The three sums of a step in one order, whatever forms them: 256 threads a CTA
// (vt = 0 .. 255), a warp's 32 values by the tree of partners 16, 8, 4, 2, 1
// apart, the warps' sums by the same tree, and the CTAs' partials (close_sums3)
// as the 256 threads' were.  a_j and b_{j+1} depend on it in their last bits, and
// with them everything a long run makes of rounding: the step it stops at, the
// small components of a Ritz vector and its sign.
constexpr int kSumPad = 33, kSumSlots = 3 * 32 * 9;

// One warp takes the trees of all eight warps, lane (q, w) those of warp w's sum
// q: 34 FP64 instructions a CTA where shuffles in every warp took 135, a quarter
// of that pipe's work in a ring 12 step.  Threads with vt < 0 only synchronise.
__device__ __forceinline__ void block_sum3_store(double a, double b, double c, double* part, double* red, int vt) {
    if (vt >= 0) {
        const int o = (vt >> 5) * kSumPad + (vt & 31);
        red[o] = a;
        red[8 * kSumPad + o] = b;
        red[16 * kSumPad + o] = c;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x, q = lane >> 3;
        const double* x = red + min(lane, 23) * kSumPad;
        double t[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) t[i] = x[i] + x[i + 16];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < o; ++i) t[i] += t[i + o];
        double s = t[0];
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((lane & 7) == 0 && q < 3) {
            part[q * kPartStride + blockIdx.x] = s;
            __threadfence();                              // before the CTA is counted (close_sums3)
        }
    }
}

// Device-resident Lanczos step control (Algorithm 1): the step in progress is
// closed with beta_{j+1}; the next step's H*v then reads beta = beta_{j+1} and
// completes f_{j+1} = (g + ua f_j) * uinv while staging its rows: ua = -a_j
// when g still holds H f_j - beta_j f_{j-1} (fused sums), 0 when the explicit
// branch already subtracted a_j f_j.  The roundings are those of the host-driven
// step (sqrt and the division are correctly rounded on both sides).
__device__ __forceinline__ void lz_close_step(LzDev* dv, double* hist, double bn, bool fused) {
    const int j = dv->j;
    hist[2 * j + 1] = bn;
    dv->stall = 0;
    dv->ua = fused ? -dv->a : 0.0;
    dv->uinv = 1.0 / bn;
    dv->beta = bn;
    dv->j = j + 1;
}

// Closes a fused reduction inside the kernel that made its partials: the CTA
// that stores its partials last (done counts the nb CTAs and returns to 0) sums
// them all in the order above into part[kRedSlots-1 .. kRedSlots-3] and, for a
// device-resident step, forms a_j and, unless the difference
// <w,w> - 2a^2 + a^2 <f,f> cancels more than six digits, beta_{j+1}.  (When it
// does, the step stalls: kernels enqueued behind it return at once and the host,
// which finds the mark in the history, runs the explicit branch.)  A kernel
// of its own for this took 8-9 us of a 40-70 us step on the small sectors.
__device__ __forceinline__ void close_sums3(double* part, int nb, unsigned* done, LzDev* dv, double* hist, double* red) {
    __shared__ int last;
    __syncthreads();                                      // this CTA's partials are stored
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicInc(done, (unsigned)nb - 1u) == (unsigned)nb - 1u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // 32 groups of 32 partials (nb <= kPartStride): partners 16 and 8 apart by
    // the threads that load them, the rest of a group by one lane, then the groups
    for (int t = threadIdx.x; t < 3 * 32 * 8; t += blockDim.x) {
        const int q = t >> 8, g = (t >> 3) & 31, i = t & 7;
        double x[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int k = 32 * g + i + 8 * c;
            x[c] = k < nb ? __ldcg(part + q * kPartStride + k) : 0.0;
        }
        red[(q * 32 + g) * 9 + i] = 32 * g < nb ? (x[0] + x[2]) + (x[1] + x[3]) : 0.0;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __shared__ double fin[3];
    if (wid < 3) {
        const double* x = red + (wid * 32 + lane) * 9;
        double t = 0.0;
        if (32 * lane < nb) t = ((x[0] + x[4]) + (x[2] + x[6])) + ((x[1] + x[5]) + (x[3] + x[7]));
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) fin[wid] = t;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double s[3] = {fin[0], fin[1], fin[2]};
#pragma unroll
    for (int q = 0; q < 3; ++q) part[kRedSlots - 1 - q] = s[q];
    if (dv == nullptr) return;
    const double a = s[0], b2 = s[1] - 2.0 * a * a + a * a * s[2];
    const int fused = b2 > 1e-6 * s[1];
    dv->a = a;
    dv->fused = fused;
    hist[2 * dv->j] = a;
    if (fused) {
        lz_close_step(dv, hist, sqrt(fmax(b2, 0.0)), true);
    } else {
        hist[2 * dv->j + 1] = -1.0;                       // no beta is negative: the host runs the explicit branch
        dv->stall = 1;
    }
}


// m such that M * 2^m <= 2^61, M = max(|t|, |U| Ns, |beta|, 2 (W |t| + |U| Ns)):
// the last term bounds every Lanczos beta (beta_{j+1} <= |H| <= W |t| + |U| Ns
// by Gershgorin, W = W_up + W_dn), so m does not depend on beta and a device-
// resident step can form round(-beta 2^m) itself with the host's m
inline EpiParams make_epilogue(double t, double U, int ns, double beta, int W) {
    EpiParams p{};
    const double gersh = 2.0 * ((double)W * std::fabs(t) + std::fabs(U) * ns);
    double M = std::max(std::max(std::fabs(t), std::fabs(U) * ns), std::max(std::fabs(beta), gersh));
    int m = 0;
    if (M > 0) {
        int ex = 0;
        std::frexp(M, &ex);                           // M < 2^ex
        m = 61 - ex;
    }
    p.m = m;
    p.A = (long long)std::llround(std::ldexp(-t, m));
    p.Bbeta = (long long)std::llround(std::ldexp(-beta, m));
    p.nB = std::min(ns, 32) + 1;
    for (int n = 0; n < 33; ++n) p.B[n] = n < p.nB ? (long long)std::llround(std::ldexp(U * n, m)) : 0;
    // int64 path: t = +-2^et and U * 2^ju an integer with |U 2^ju| Ns < 2^14 for some ju in [0, 8],
    // et + ju in [0, 6].  Then |T 2^(et+ju)| < 2^55 * 2^6 and |U 2^ju n X| < 2^14 * 2^48, so
    // H v is formed exactly in int64 and rounded once; a -beta w_old term is then added with
    // one fused multiply-add (a second rounding)
    p.fast = 0;
    p.apow = -1;
    p.mbeta = -beta;
    if (t != 0.0) {
        int et = 0;
        const double mt = std::frexp(std::fabs(t), &et);   // |t| = mt * 2^et, mt in [0.5, 1)
        if (mt == 0.5) {
            et -= 1;                                        // |t| = 2^et
            if (et + m >= 0 && et + m < 62) p.apow = et + m;
            for (int ju = 0; ju <= 8; ++ju) {
                const double us = std::ldexp(U, ju);
                if (us == std::floor(us) && std::fabs(us) * ns < 16384.0 && et + ju >= 0 && et + ju <= 6) {
                    p.fast = 1;
                    p.tshift = et + ju;
                    p.tneg = t < 0 ? 1 : 0;
                    p.ju = ju;
                    p.Uint = (long long)us;
                    break;
                }
            }
        }
    }
    return p;
}


}  // namespace hub
