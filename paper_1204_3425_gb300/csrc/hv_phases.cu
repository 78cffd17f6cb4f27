// Two-phase H*v with shared-memory staging (Sec. 4.3 restated for sm_103a).
//
// V is the row-major D_up x D_dn matrix of Fig. 2.  The Kronecker sum of
// Eq. (H-Kroneckersum) splits H*v into
//   row phase  Y[u, :] = sum over down-hops inside row u          (Algorithm 3)
//   up phase   W[u, :] = sum over up-hops u -> u' of rows V[u', :] + Y[u, :]
//                        + U * popcount(s_up & s_dn) * V[u, :]     (Algorithms 2, 4)
// The row phase stages VEC whole rows of V in shared memory and gathers with a
// warp-sliced, bank-coloured hop table (one 16-byte shared load feeds VEC
// outputs).  The up phase combines whole row segments: a warp-uniform hop
// list, lanes over columns, coalesced loads of a column chunk that stays
// resident in L2 while every row of it is formed.
//
// Binary64 path: every element is rounded once to the fixed-point grid 2^-k
// (k = 1070 - emax, emax = biased exponent bound of max|v|) and held as
// (lo, hi) int32 words, X = hi * 2^24 + lo; hop sums are exact integer sums.
// The up phase forms, exactly in 128-bit integers,
//   T*A + X_own*B[n] + G*Bbeta,   A = -t 2^m, B[n] = U n 2^m, Bbeta = -beta 2^m
// (T = hop sum, G = fixed-point w_old) and rounds it once to binary64: the
// FP64 pipe (1.7 op/clk/SM on this part) is not used per element.  When t is
// a power of two and U a small dyadic number (the usual t = 1, integer U),
// the H v part fits int64 exactly and is rounded once; a Lanczos -beta w_old
// term is then one fused multiply-add.
#include <cstdint>
#include <cmath>
#include <type_traits>
#include <cuda_runtime.h>

#include "internal.h"
#include "row_blocks.cuh"
#include "hv_epilogue.cuh"
#include "up_grid.h"

namespace hub {

namespace {

template <int VEC> struct FxVec;
template <> struct FxVec<1> { using T = int2; };
template <> struct FxVec<2> { using T = int4; };

template <int VEC> struct F32Vec;
template <> struct F32Vec<1> { using T = float; };
template <> struct F32Vec<2> { using T = float2; };
template <> struct F32Vec<4> { using T = float4; };

__device__ __forceinline__ float comp(float x, int) { return x; }
__device__ __forceinline__ float comp(float2 x, int i) { return i == 0 ? x.x : x.y; }
__device__ __forceinline__ float comp(float4 x, int i) { return i == 0 ? x.x : (i == 1 ? x.y : (i == 2 ? x.z : x.w)); }

// The exponent bound of a product, found by every CTA of its row phase: the
// largest exponent of v itself (scan: at most kScanElems elements), or of the
// per-CTA maxima an exponent pass left in slots[0 .. nslots).  CTA 0 hands it on to
// the up phase in *emax_p.  Every word is written before it is read within the
// product, so nothing has to be set back between products.
__device__ __forceinline__ int cta_exponent(const double* v, int n, const int* slots, int nslots, int* emax_p) {
    __shared__ int emax_s;
    if (threadIdx.x == 0) emax_s = 1;
    __syncthreads();
    int m = 1;
    if (slots != nullptr) {
        for (int i = threadIdx.x; i < nslots; i += blockDim.x) m = max(m, slots[i]);
    } else {
#pragma unroll 8
        for (int i = threadIdx.x; i < n; i += blockDim.x)
            m = max(m, (int)(((unsigned long long)__double_as_longlong(v[i]) >> 52) & 0x7FF));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(&emax_s, m);
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) *emax_p = emax_s;
    return emax_s;
}

// Row phase, binary64 fixed point: Y[u, d] = sum_{(d', s) in hops_dn(d)} s X[u, d'];
// also writes the fixed-point copy of V to Xg for the up phase.
// UPD: the previous Lanczos step's update is applied on the way in,
// v <- (v + ua fo) * uinv, rounded as k_axpy_scale_f64, and written back to v.
template <int VEC, typename EntT, bool UPD>
__global__ void __launch_bounds__(1024, 1) k_rows_f64x(std::conditional_t<UPD, double*, const double*> v,
                                                     long long* __restrict__ Y,
                                                     int2* __restrict__ Xg, int64_t Dup, int64_t Ddn,
                                                     const int64_t* __restrict__ boff,
                                                     const int32_t* __restrict__ bcnt,
                                                     const EntT* __restrict__ ent,
                                                     int* emax_p, int fixed_emax, int scan,
                                                     const int* slots, int nslots,
                                                     const double* fo, double ua, double uinv,
                                                     const LzDev* dv) {
    using S = typename FxVec<VEC>::T;
    grid_dep_wait();
    if constexpr (UPD) {
        if (dv != nullptr) {                              // device-resident step: the update's scalars
            if (dv->stall) return;
            ua = dv->ua;
            uinv = dv->uinv;
        }
    }
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S* X = reinterpret_cast<S*>(smem_raw);
    int emax = fixed_emax;
    if (!UPD && (scan || slots != nullptr)) emax = cta_exponent(v, (int)(Dup * Ddn), slots, nslots, emax_p);
    else if (fixed_emax <= 0) emax = max(*emax_p, 1);
    const int lane = threadIdx.x & 31;
    const int64_t nblk = (Dup + VEC - 1) / VEC;
    const int64_t step = blockDim.x;
    constexpr int NL = UPD ? 2 : 4;                       // row elements per thread in flight
    {
        const int64_t z0 = staged_slots(Ddn) - 32;
        for (int i = threadIdx.x; i < 32; i += blockDim.x) {
            if constexpr (VEC == 1) X[z0 + i] = make_int2(0, 0);
            else X[z0 + i] = make_int4(0, 0, 0, 0);
        }
    }
    for (int64_t b = blockIdx.x; b < nblk; b += gridDim.x) {
        const int64_t u0 = b * VEC;
        const int nrow = (int)((Dup - u0) < VEC ? (Dup - u0) : VEC);
        // stage rows u0 .. u0+nrow-1 as fixed point, NL loads per row in flight
        // (with UPD every load of a group is issued before the first store)
        for (int64_t d0 = threadIdx.x; d0 < Ddn; d0 += NL * step) {
            double xv[NL][VEC];
            [[maybe_unused]] double fv[NL][VEC];
#pragma unroll
            for (int i = 0; i < NL; ++i)
#pragma unroll
                for (int r = 0; r < VEC; ++r) {
                    const int64_t d = d0 + i * step;
                    const bool in = d < Ddn && r < nrow;
                    xv[i][r] = in ? v[(u0 + r) * Ddn + d] : 0.0;
                    if constexpr (UPD) fv[i][r] = in ? fo[(u0 + r) * Ddn + d] : 0.0;
                }
            if constexpr (UPD) {
#pragma unroll
                for (int i = 0; i < NL; ++i)
#pragma unroll
                    for (int r = 0; r < VEC; ++r) {
                        const int64_t d = d0 + i * step;
                        if (d < Ddn && r < nrow) {
                            xv[i][r] = fma(ua, fv[i][r], xv[i][r]) * uinv;
                            __stcs(v + (u0 + r) * Ddn + d, xv[i][r]);
                        }
                    }
            }
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int64_t d = d0 + i * step;
                if (d >= Ddn) break;
                int w[2 * VEC];
#pragma unroll
                for (int r = 0; r < VEC; ++r) {
                    fx_split(xv[i][r], emax, w[2 * r], w[2 * r + 1]);
                    if (r < nrow) __stcg(Xg + (u0 + r) * Ddn + d, make_int2(w[2 * r], w[2 * r + 1]));
                }
                if constexpr (VEC == 1) X[d] = make_int2(w[0], w[1]);
                else X[d] = make_int4(w[0], w[1], w[2], w[3]);
            }
        }
        __syncthreads();
        for (int64_t d0 = threadIdx.x & ~31; d0 < Ddn; d0 += step) {
            const int64_t g = d0 >> 5;
            const int64_t d = d0 + lane;
            int a0 = 0, a1 = 0, a2 = 0, a3 = 0;
            for_each_hop<EntT>(ent + boff[g], bcnt[g], lane, [&](uint32_t e) {
                const int s = RowEnt<EntT>::sgn(e);           // padding reads a zero slot
                const S x = X[RowEnt<EntT>::idx(e)];
                a0 += s * x.x;
                a1 += s * x.y;
                if constexpr (VEC == 2) {
                    a2 += s * x.z;
                    a3 += s * x.w;
                }
            });
            if (d < Ddn) {
                Y[u0 * Ddn + d] = fx_join(a0, a1);
                if (VEC == 2 && nrow > 1) Y[(u0 + 1) * Ddn + d] = fx_join(a2, a3);
            }
        }
        __syncthreads();
    }
}

// Row phase for binary64 rows of which only one 4-byte word per element fits in
// shared memory (29024 < D_dn <= 58080 with 227 KB to a CTA), of vectors that stay
// in L2: the (lo, hi) words are staged and summed apart.  A plane is one word of one row; the 2 Dup planes, split into groups of
// 32 columns, are dealt to the CTAs in equal contiguous ranges, so a few long
// rows still fill the device evenly (153 rows of 48620 elements are two waves of
// one row per SM).  A gather from L2 fetched a 32-byte sector at L2 latency for
// eight bytes; here it is two conflict-free shared loads (153 x 48620 elements:
// product 304 -> 236 us).  The CTA that begins a row's lo plane also writes its
// fixed-point copy X.  Ys holds the two word sums of an element side by side and
// the up phase joins them: joined here, each CTA would stage both words of two
// rows instead of three planes (259 us).  On HBM-sized vectors one CTA an SM stages
// and sums in turn and the gathers of k_rows_global_f64x overlap better (816 x 43758
// elements: product 0.89 ms with planes, 0.85 without; 1140 x 38760: 1.23, 0.98).
template <typename EntT>
__global__ void __launch_bounds__(1024, 1) k_rows_planes_f64x(const double* v, int* __restrict__ Ys,
                                                            int2* __restrict__ Xg, int64_t Dup, int64_t Ddn,
                                                            const int64_t* __restrict__ boff,
                                                            const int32_t* __restrict__ bcnt,
                                                            const EntT* __restrict__ ent,
                                                            int* emax_p, int fixed_emax, const int* slots,
                                                            int nslots) {
    grid_dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int* Xs = reinterpret_cast<int*>(smem_raw);
    const int emax = fixed_emax > 0     ? fixed_emax
                     : slots != nullptr ? cta_exponent(v, 0, slots, nslots, emax_p)
                                        : max(*emax_p, 1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int n = (int)Ddn, z0 = (int)staged_slots(Ddn) - 32;
    if (threadIdx.x < 32) Xs[z0 + threadIdx.x] = 0;
    const int64_t G = (Ddn + 31) >> 5, T = 2 * Dup * G;
    const int64_t t1 = T * (blockIdx.x + 1) / gridDim.x;
    for (int64_t t = T * blockIdx.x / gridDim.x; t < t1;) {
        const int64_t q = t / G, u = q >> 1;
        const int plane = (int)(q & 1);
        const int g0 = (int)(t - q * G), g1 = (int)min(G, t1 - q * G);
        const double* row = v + u * Ddn;
        int2* xrow = plane == 0 && g0 == 0 ? Xg + u * Ddn : nullptr;
        constexpr int NL = 8;
        for (int d0 = threadIdx.x; d0 < n; d0 += NL * blockDim.x) {
            double x[NL];
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int d = d0 + i * blockDim.x;
                x[i] = d < n ? row[d] : 0.0;
            }
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int d = d0 + i * blockDim.x;
                if (d >= n) break;
                int lo, hi;
                fx_split(x[i], emax, lo, hi);
                Xs[d] = plane ? hi : lo;
                if (xrow != nullptr) xrow[d] = make_int2(lo, hi);
            }
        }
        __syncthreads();
        for (int g = g0 + warp; g < g1; g += nw) {
            int a = 0;
            for_each_hop<EntT>(ent + boff[g], bcnt[g], lane, [&](uint32_t e) {
                a += RowEnt<EntT>::sgn(e) * Xs[RowEnt<EntT>::idx(e)];
            });
            const int d = g * 32 + lane;
            if (d < n) Ys[2 * (u * Ddn + d) + plane] = a;
        }
        __syncthreads();
        t = q * G + g1;
    }
}

// Row phase for binary64 rows too long for shared memory (by the word, or whole on
// HBM-sized vectors): the fixed-point
// copy X is already in global memory (k_to_fixed) and the down-hop gathers
// read row u of it through L1/L2.
template <typename EntT>
__global__ void __launch_bounds__(512) k_rows_global_f64x(const int2* __restrict__ Xg, long long* __restrict__ Y,
                                                           int64_t Dup, int64_t Ddn,
                                                           const int64_t* __restrict__ boff,
                                                           const int32_t* __restrict__ bcnt,
                                                           const EntT* __restrict__ ent) {
    const int lane = threadIdx.x & 31;
    for (int64_t u = blockIdx.x; u < Dup; u += gridDim.x) {
        const int2* X = Xg + u * Ddn;
        for (int64_t d0 = threadIdx.x & ~31; d0 < Ddn; d0 += blockDim.x) {
            const int64_t g = d0 >> 5;
            const int64_t d = d0 + lane;
            int a0 = 0, a1 = 0;
            for_each_hop<EntT>(ent + boff[g], bcnt[g], lane, [&](uint32_t e) {
                const uint32_t i = RowEnt<EntT>::idx(e);
                if (i < Ddn) {                                // padding: no zero slots in global rows
                    const int s = RowEnt<EntT>::sgn(e);
                    const int2 x = __ldg(X + i);
                    a0 += s * x.x;
                    a1 += s * x.y;
                }
            });
            if (d < Ddn) Y[u * Ddn + d] = fx_join(a0, a1);
        }
    }
}


// An item of 16 rows is two per warp; where that leaves fewer items than CTAs
// that fit on the device, 8 rows (one per warp) spread the sector wider.
inline int up_rows(int64_t nchunk, int64_t Dup, int ctas) { return nchunk * ((Dup + 15) / 16) < ctas ? 8 : 16; }

// Signed sum over the warp-uniform hop list of row u: targets t in
// list[kb .. kb+n), the first np with sign +1.  load(t) returns this lane's
// operand from row t; the operands of a group of four of one sign are requested
// together, then add(sign, a, b, c, d) or add(sign, a) takes them.  Loop bounds
// are warp-uniform, so the sign split costs no divergence.
// TAIL: what is left of a sign after the groups of four is requested together,
// zeros in place of the missing operands, and added one by one as without it.
template <typename Val, bool TAIL, typename Load, typename Add>
__device__ __forceinline__ void uniform_hops(const uint32_t* __restrict__ list, int32_t kb, int n, int np, int lane,
                                             Load&& load, Add&& add) {
    for (int k0 = 0; k0 < n; k0 += 32) {
        const int nk = min(32, n - k0);
        const uint32_t mine = lane < nk ? __ldg(list + kb + k0 + lane) : 0u;
        const int pend = max(0, min(nk, np - k0));
        auto span = [&](auto sign, int q, int end) {
            for (; q + 4 <= end; q += 4) {
                const Val a = load(__shfl_sync(0xffffffffu, mine, q));
                const Val b = load(__shfl_sync(0xffffffffu, mine, q + 1));
                const Val c = load(__shfl_sync(0xffffffffu, mine, q + 2));
                const Val d = load(__shfl_sync(0xffffffffu, mine, q + 3));
                add(sign, a, b, c, d);
            }
            if constexpr (TAIL) {
                if (q < end) {
                    const Val a = load(__shfl_sync(0xffffffffu, mine, q));
                    Val b{}, c{};
                    const uint32_t t1 = __shfl_sync(0xffffffffu, mine, q + 1), t2 = __shfl_sync(0xffffffffu, mine, q + 2);
                    if (q + 1 < end) b = load(t1);
                    if (q + 2 < end) c = load(t2);
                    add(sign, a);
                    add(sign, b);
                    add(sign, c);
                }
            } else {
                for (; q < end; ++q) add(sign, load(__shfl_sync(0xffffffffu, mine, q)));
            }
        };
        span(std::integral_constant<int, 1>{}, 0, pend);
        span(std::integral_constant<int, -1>{}, pend, nk);
    }
}

__device__ __forceinline__ void addf(float& A, float a, float b, float c, float d) { A += (a + b) + (c + d); }
__device__ __forceinline__ void addf(float& A, float a) { A += a; }
__device__ __forceinline__ void addf(float2& A, float2 a, float2 b, float2 c, float2 d) {
    A.x += (a.x + b.x) + (c.x + d.x);
    A.y += (a.y + b.y) + (c.y + d.y);
}
__device__ __forceinline__ void addf(float2& A, float2 a) { A.x += a.x; A.y += a.y; }
__device__ __forceinline__ void addf(float4& A, float4 a, float4 b, float4 c, float4 d) {
    A.x += (a.x + b.x) + (c.x + d.x);
    A.y += (a.y + b.y) + (c.y + d.y);
    A.z += (a.z + b.z) + (c.z + d.z);
    A.w += (a.w + b.w) + (c.w + d.w);
}
__device__ __forceinline__ void addf(float4& A, float4 a) { A.x += a.x; A.y += a.y; A.z += a.z; A.w += a.w; }

// the binary32 accumulation: the two signs apart, in list order
template <typename V> struct AddFloat {
    V& P;
    V& N;
    template <typename Sign, typename... Vs>
    __device__ __forceinline__ void operator()(Sign, Vs... xs) const {
        if constexpr (Sign::value > 0) addf(P, xs...);
        else addf(N, xs...);
    }
};

// the binary64 accumulation: exact integers, so one accumulator takes both signs
template <typename IV> struct AddFixed {
    IV& A;
    template <typename Sign, typename... Vs>
    __device__ __forceinline__ void operator()(Sign, Vs... xs) const {
        if constexpr (Sign::value > 0) add4(A, xs...);
        else sub4(A, xs...);
    }
};

// Up phase, binary64 fixed point (Algorithms 2 and 4):
//   W[u, c] = -t (sum_{(u', s) in hops_up(u)} s X[u', c] + Y[u, c]) + U n(u, c) X[u, c]  [- beta w_old]
// Row u of W is a signed combination of whole rows u' of X (Eq. H-Kroneckersum),
// so a warp builds one row segment of CC = 64 columns, two per lane (rows of even
// length), with lanes over columns: the hop list is warp-uniform and every access
// is coalesced.  Work items are (column chunk, block of rbr rows); consecutive items share a
// chunk, which keeps that chunk of X resident in L2 while all rows are
// combined, and consecutive rows share part of their neighbours (L1 reuse).
// PRE: the epilogue's own element and Y are requested before the gathers (their
// HBM latency then overlaps the hop sum); CT: CTAs per SM the launch bounds keep
template <bool FAST, bool TAIL, bool PRE = false, int CT = 4>
__global__ void __launch_bounds__(256, CT) k_up_f64x(const int2* X, const long long* Y,
                                                     double* w, const double* w_old, int64_t Dup, int64_t Ddn,
                                                     int rbr, const int32_t* __restrict__ ptr,
                                                     const int32_t* __restrict__ npos,
                                                     const uint32_t* __restrict__ list,
                                                     const uint32_t* __restrict__ su,
                                                     const uint32_t* __restrict__ sd,
                                                     const __grid_constant__ EpiParams ep,
                                                     const int* emax_p, int fixed_emax) {
    constexpr int VPL = 2;
    using IV = int4;
    __shared__ long long Bs[33];
    for (int i = threadIdx.x; i < 33; i += blockDim.x) Bs[i] = i < ep.nB ? ep.B[i] : 0;
    __syncthreads();
    grid_dep_wait();
    const int emax = fixed_emax > 0 ? fixed_emax : max(*emax_p, 1);
    const int k = 1070 - emax;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    constexpr int CC = 32 * VPL;
    const uint32_t rowb = (uint32_t)Ddn * 8u;             // bytes of a row (Ddn <= kMaxRow)
    const int64_t nchunk = (Ddn + CC - 1) / CC;
    const int64_t nrb = (Dup + rbr - 1) / rbr;
    // item = chunk * nrb + rb, advanced by gridDim.x without division
    int64_t chunk = blockIdx.x / nrb, rb = blockIdx.x % nrb;
    const int64_t dch = gridDim.x / nrb, drb = gridDim.x % nrb;
    for (; chunk < nchunk; chunk += dch, rb += drb) {
        if (rb >= nrb) {
            rb -= nrb;
            ++chunk;
            if (chunk >= nchunk) break;
        }
        const int64_t c_raw = chunk * CC + (int64_t)lane * VPL;
        const bool act = c_raw < Ddn;
        const int64_t c = act ? c_raw : Ddn - VPL;     // tail lanes read a valid column, store nothing
        uint32_t sdc[VPL];
#pragma unroll
        for (int j = 0; j < VPL; ++j) sdc[j] = sd[c + j];
        const char* base = reinterpret_cast<const char*>(X + c);
        const int64_t uend = min(rb * rbr + rbr, Dup);
        for (int64_t u = rb * rbr + warp; u < uend; u += nw) {
            const int32_t kb = ptr[u];
            [[maybe_unused]] int4 t4p;
            [[maybe_unused]] longlong2 y2p;
            if constexpr (PRE) {
                const int64_t J = u * Ddn + c;
                t4p = *(reinterpret_cast<const int4*>(X + J));
                y2p = ld_stream(reinterpret_cast<const longlong2*>(Y + J));
            }
            IV A{};
            uniform_hops<IV, TAIL>(list, kb, ptr[u + 1] - kb, npos[u], lane,
                [&](uint32_t t) { return *(reinterpret_cast<const IV*>(base + (uint64_t)t * rowb)); },
                AddFixed<IV>{A});
            if (act) {
                const uint32_t su_u = su[u];
                const int64_t J = u * Ddn + c;
                int lo[VPL], hi[VPL];
                int2 xo[VPL];
                long long yv[VPL];
                lo[0] = A.x; hi[0] = A.y; lo[1] = A.z; hi[1] = A.w;
                int4 t4;
                longlong2 y2;
                if constexpr (PRE) {
                    t4 = t4p;
                    y2 = y2p;
                } else {
                    t4 = *(reinterpret_cast<const int4*>(X + J));
                    y2 = ld_stream(reinterpret_cast<const longlong2*>(Y + J));
                }
                xo[0] = make_int2(t4.x, t4.y);
                xo[1] = make_int2(t4.z, t4.w);
                yv[0] = y2.x;
                yv[1] = y2.y;
                double r[VPL];
#pragma unroll
                for (int j = 0; j < VPL; ++j) {
                    if constexpr (FAST) {
                        // exact: |T| < 2^55, |X| <= 2^48, |Uint * n| < 2^14 and tshift <= 6
                        const long long Pv = fast_sum(fx_join(lo[j], hi[j]) + yv[j], xo[j], __popc(su_u & sdc[j]), ep);
                        r[j] = i64_scaled_to_double(Pv, -(k + ep.ju));
                        if (w_old != nullptr) r[j] = fma(ep.mbeta, w_old[J + j], r[j]);
                    } else {
                        I128 acc{0ull, 0ll};
                        mac_t(acc, fx_join(lo[j], hi[j]) + yv[j], ep);
                        mac128(acc, fx_join(xo[j].x, xo[j].y), Bs[__popc(su_u & sdc[j])]);
                        if (w_old != nullptr) {
                            int glo, ghi;
                            fx_split(w_old[J + j], emax, glo, ghi);
                            mac128(acc, fx_join(glo, ghi), ep.Bbeta);
                        }
                        r[j] = i128_to_double(acc, -(k + ep.m));
                    }
                }
                __stcs(reinterpret_cast<double2*>(w + J), make_double2(r[0], r[1]));
            }
        }
    }
}

// Work of the Lanczos step kernels: items of 32 * VPL columns by kUpRows rows,
// dealt to the CTAs in turn, thread (warp, lane) of a CTA taking rows warp and
// warp + 8 of an item and columns lane * VPL + j.  The step's sums are over a
// thread's elements in that order (then block_sum3_store), so this division is
// part of the result, in the last bits of a_j and b_{j+1}: it follows the row
// length, the SMs and a vec_cols that the caller sets, and nothing else.
constexpr int kUpRows = 16;
// CTAs an SM of the step kernels: their grids, and with them the partials, are at
// most so many times the SMs
constexpr int kStepCtas64 = 3, kStepCtas32 = 4;
constexpr int up32_ctas(int vpl, bool red) { return red || vpl == 4 ? kStepCtas32 : 5; }

// Lanczos-step variant of k_up_f64x (Algorithm 1 fused with Algorithms 2, 4):
// W = H f - beta w_old and, per CTA, the partials of <W, f>, <W, W> and
// <f, f>, closed by the last CTA.  Its epilogue streams four arrays (own element,
// Y, w_old, f), whose loads are issued before the gathers; the extra live
// registers cost one CTA per SM (3 instead of 4).  Items, rows and the row pitch
// are 32-bit, and T A is always the 128-bit multiply: with 64-bit ones and mac_t's
// two forms the 128-bit epilogue spilled (4x4 (8,8), U = 7.3: step 6.18 -> 5.28 ms,
// U = 8: 5.01 -> 5.00).  YS: Y holds word pairs
// (k_rows_planes_f64x).
// NT = 512: a sector of no more items than SMs, one item a CTA and one row a
// warp; warps 8-15 continue the sums of warps 0-7, in the order above, so a CTA
// has two rows' memory rounds in flight instead of one after the other (3x3 (4,4)
// ground state with its vector 2.04 -> 1.92 ms).
template <int VPL, bool FAST, bool TAIL, bool YS, int NT>
__global__ void __launch_bounds__(NT, NT == 512 ? 1 : kStepCtas64) k_up_step_f64x(
        const int2* X, const long long* Y, double* w, const double* w_old, int64_t Dup,
        int64_t Ddn, const int32_t* __restrict__ ptr, const int32_t* __restrict__ npos,
        const uint32_t* __restrict__ list, const uint32_t* __restrict__ su, const uint32_t* __restrict__ sd,
        const __grid_constant__ EpiParams ep, const int* emax_p, int fixed_emax,
        const double* fv, double* part, unsigned* done, LzDev* dv, double* hist) {
    grid_dep_wait();
    if (dv != nullptr && dv->stall) return;
    using IV = typename FxVec<VPL>::T;
    __shared__ long long Bs[33];
    __shared__ long long sh_bb;
    __shared__ double red[kSumSlots];
    for (int i = threadIdx.x; i < 33; i += blockDim.x) Bs[i] = i < ep.nB ? ep.B[i] : 0;
    double mbeta = ep.mbeta;
    if (dv != nullptr) mbeta = -dv->beta;                 // device-resident step: beta_j on the device
    if (!FAST && threadIdx.x == 0) sh_bb = dv != nullptr ? llround(ldexp(mbeta, ep.m)) : ep.Bbeta;
    __syncthreads();
    const long long Bbeta = FAST ? 0 : sh_bb;
    const int emax = fixed_emax > 0 ? fixed_emax : max(*emax_p, 1);
    const int k = 1070 - emax;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int nw = NT / 32, CC = 32 * VPL;
    const int nchunk = (int)((Ddn + CC - 1) / CC), nrb = (int)((Dup + kUpRows - 1) / kUpRows);
    const uint32_t rowb = (uint32_t)Ddn * 8u;             // bytes of a row (Ddn <= kMaxRow)
    double s1 = 0.0, s2 = 0.0, s3 = 0.0;
    double r[VPL], fj[VPL];                               // this thread's elements of a row
    bool have = false;                                    // NT = 512: r, fj hold its only row
    auto add_row = [&] {
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            s1 = fma(r[j], fj[j], s1);
            s2 = fma(r[j], r[j], s2);
            s3 = fma(fj[j], fj[j], s3);
        }
    };
    // item = chunk * nrb + rb, advanced by gridDim.x without division
    int chunk = (int)blockIdx.x / nrb, rb = (int)blockIdx.x % nrb;
    const int dch = (int)gridDim.x / nrb, drb = (int)gridDim.x % nrb;
    for (; chunk < nchunk; chunk += dch, rb += drb) {
        if (rb >= nrb) {
            rb -= nrb;
            ++chunk;
            if (chunk >= nchunk) break;
        }
        const int c_raw = chunk * CC + lane * VPL;
        const bool act = c_raw < (int)Ddn;
        const int c = act ? c_raw : (int)Ddn - VPL;     // tail lanes read a valid column, store nothing
        uint32_t sdc[VPL];
#pragma unroll
        for (int j = 0; j < VPL; ++j) sdc[j] = sd[c + j];
        const char* base = reinterpret_cast<const char*>(X + c);
        const int uend = min(rb * kUpRows + kUpRows, (int)Dup);
        for (int u = rb * kUpRows + warp; u < uend; u += nw) {
            const int32_t kb = ptr[u];
            const int64_t J = (int64_t)u * (int)Ddn + c;
            // streamed operands of the epilogue, requested before the gathers
            double wv[VPL];
            long long yv[VPL];
            const IV xo4 = *(reinterpret_cast<const IV*>(X + J));
            if constexpr (VPL == 2) {
                const longlong2 y2 = ld_stream(reinterpret_cast<const longlong2*>(Y + J));
                yv[0] = y2.x; yv[1] = y2.y;
                if (w_old != nullptr) {
                    const double2 q = ld_stream(reinterpret_cast<const double2*>(w_old + J));
                    wv[0] = q.x; wv[1] = q.y;
                }
                const double2 q = ld_stream(reinterpret_cast<const double2*>(fv + J));
                fj[0] = q.x; fj[1] = q.y;
            } else {
                yv[0] = ld_stream(Y + J);
                if (w_old != nullptr) wv[0] = ld_stream(w_old + J);
                fj[0] = ld_stream(fv + J);
            }
            IV A{};
            uniform_hops<IV, TAIL>(list, kb, ptr[u + 1] - kb, npos[u], lane,
                [&](uint32_t t) { return *(reinterpret_cast<const IV*>(base + (uint64_t)t * rowb)); },
                AddFixed<IV>{A});
            if (!act) continue;
            const uint32_t su_u = su[u];
#pragma unroll
            for (int j = 0; j < VPL; ++j) {
                long long T;
                int2 xo;
                if constexpr (VPL == 2) {
                    T = j == 0 ? fx_join(A.x, A.y) : fx_join(A.z, A.w);
                    xo = j == 0 ? make_int2(xo4.x, xo4.y) : make_int2(xo4.z, xo4.w);
                } else {
                    T = fx_join(A.x, A.y);
                    xo = xo4;
                }
                if constexpr (YS) T += fx_join((int)yv[j], (int)(yv[j] >> 32));
                else T += yv[j];
                const int nd = __popc(su_u & sdc[j]);
                if constexpr (FAST) {
                    r[j] = i64_scaled_to_double(fast_sum(T, xo, nd, ep), -(k + ep.ju));
                    if (w_old != nullptr) r[j] = fma(mbeta, wv[j], r[j]);
                } else {
                    I128 acc{0ull, 0ll};
                    mac128(acc, T, ep.A);
                    mac128(acc, fx_join(xo.x, xo.y), Bs[nd]);
                    if (w_old != nullptr) {
                        int glo, ghi;
                        fx_split(wv[j], emax, glo, ghi);
                        mac128(acc, fx_join(glo, ghi), Bbeta);
                    }
                    r[j] = i128_to_double(acc, -(k + ep.m));
                }
            }
            if constexpr (VPL == 2) __stcs(reinterpret_cast<double2*>(w + J), make_double2(r[0], r[1]));
            else __stcs(w + J, r[0]);
            if constexpr (NT == 512) have = true;
            else add_row();
        }
    }
    if constexpr (NT == 512) {
        __shared__ double car[3][256];
        const int t = threadIdx.x & 255;
        if (warp < 8) {
            if (have) add_row();
            car[0][t] = s1;
            car[1][t] = s2;
            car[2][t] = s3;
        }
        __syncthreads();
        if (warp >= 8) {
            s1 = car[0][t];
            s2 = car[1][t];
            s3 = car[2][t];
            if (have) add_row();
        }
    }
    block_sum3_store(s1, s2, s3, part, red, (int)threadIdx.x - (NT - 256));
    close_sums3(part, gridDim.x, done, dv, hist, red);
}

// Lanczos-step variant of the binary32 up phase, items and sums as above.  What is
// left of a hop list is requested at once on every size (4x4 (8,8) step 2.75 ->
// 2.62 ms, ring 14 (7,7) 162 -> 146 us).
// RED false: a product or a replayed step that does not take resident rows
// (up_items32).
template <int VPL, bool RED>
__global__ void __launch_bounds__(256, up32_ctas(VPL, RED)) k_up_step_f32(const float* v, const float* Y, float* w,
                                                        const float* w_old, int64_t Dup, int64_t Ddn,
                                                        const int32_t* __restrict__ ptr,
                                                        const int32_t* __restrict__ npos,
                                                        const uint32_t* __restrict__ list,
                                                        const uint32_t* __restrict__ su,
                                                        const uint32_t* __restrict__ sd, float mt, float U, float mbeta,
                                                        double* part, unsigned* done, LzDev* dv, double* hist) {
    grid_dep_wait();
    if (dv != nullptr && dv->stall) return;
    FFAcc s1, s2, s3;
    if (dv != nullptr) mbeta = (float)-dv->beta;          // device-resident step: beta_j on the device
    using V = typename F32Vec<VPL>::T;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    constexpr int CC = 32 * VPL;
    const int64_t nchunk = (Ddn + CC - 1) / CC;
    const int64_t nrb = (Dup + kUpRows - 1) / kUpRows;
    int64_t chunk = blockIdx.x / nrb, rb = blockIdx.x % nrb;
    const int64_t dch = gridDim.x / nrb, drb = gridDim.x % nrb;
    for (; chunk < nchunk; chunk += dch, rb += drb) {
        if (rb >= nrb) {
            rb -= nrb;
            ++chunk;
            if (chunk >= nchunk) break;
        }
        const int64_t c_raw = chunk * CC + (int64_t)lane * VPL;
        const bool act = c_raw < Ddn;
        const int64_t c = act ? c_raw : Ddn - VPL;
        uint32_t sdc[VPL];
#pragma unroll
        for (int j = 0; j < VPL; ++j) sdc[j] = sd[c + j];
        const float* base = v + c;
        const int64_t uend = min(rb * kUpRows + kUpRows, Dup);
        for (int64_t u = rb * kUpRows + warp; u < uend; u += nw) {
            const int32_t kb = ptr[u];
            const int64_t J = u * Ddn + c;
            // epilogue operands, requested before the gathers
            const V xo = *(reinterpret_cast<const V*>(v + J));
            const V yv = ld_stream(reinterpret_cast<const V*>(Y + J));
            V wv{};
            if (w_old != nullptr) wv = ld_stream(reinterpret_cast<const V*>(w_old + J));
            V P{}, N{};
            uniform_hops<V, true>(list, kb, ptr[u + 1] - kb, npos[u], lane,
                [&](uint32_t t) { return *(reinterpret_cast<const V*>(base + (int64_t)t * Ddn)); },
                AddFloat<V>{P, N});
            if (!act) continue;
            const uint32_t su_u = su[u];
            float r[VPL];
#pragma unroll
            for (int j = 0; j < VPL; ++j) {
                const float nd = (float)__popc(su_u & sdc[j]);
                r[j] = fmaf(mt, (comp(P, j) - comp(N, j)) + comp(yv, j), U * nd * comp(xo, j));
                if (w_old != nullptr) r[j] = fmaf(mbeta, comp(wv, j), r[j]);
            }
            if constexpr (VPL == 4) __stcs(reinterpret_cast<float4*>(w + J), make_float4(r[0], r[1], r[2], r[3]));
            else if constexpr (VPL == 2) __stcs(reinterpret_cast<float2*>(w + J), make_float2(r[0], r[1]));
            else __stcs(w + J, r[0]);
            if constexpr (RED) {
#pragma unroll
                for (int j = 0; j < VPL; ++j) {
                    s1.add_product(r[j], comp(xo, j));
                    s2.add_product(r[j], r[j]);
                    s3.add_product(comp(xo, j), comp(xo, j));
                }
            }
        }
    }
    if constexpr (RED) {
        __shared__ double red[kSumSlots];
        block_sum3_store(s1.value(), s2.value(), s3.value(), part, red, threadIdx.x);
        close_sums3(part, gridDim.x, done, dv, hist, red);
    }
}

// Binary32 product or replayed step of the largest vectors (up_lean32): items as
// above, with as few requests in flight as a row takes -- the rest of a hop list
// one by one, epilogue operands after the sum.  On gigabytes the CTAs of faster
// forms drift apart and their chunks no longer share L2 (18 sites (8,9), 8.5 GB a
// vector: 24.4 ms, 27.3 with resident rows, 29.2 with items that request the rest
// at once; (9,7) 17.9, 18.9, 21.6).  Launched alone, behind the row phase: loads
// take the read-only path.
__global__ void __launch_bounds__(256, kStepCtas32) k_up_lean_f32(const float* __restrict__ v, const float* __restrict__ Y,
                                                                float* w, const float* w_old, int64_t Dup, int64_t Ddn,
                                                                const int32_t* __restrict__ ptr,
                                                                const int32_t* __restrict__ npos,
                                                                const uint32_t* __restrict__ list,
                                                                const uint32_t* __restrict__ su,
                                                                const uint32_t* __restrict__ sd, float mt, float U,
                                                                float mbeta) {
    constexpr int VPL = 4, CC = 32 * VPL;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t nchunk = (Ddn + CC - 1) / CC;
    const int64_t nrb = (Dup + kUpRows - 1) / kUpRows;
    int64_t chunk = blockIdx.x / nrb, rb = blockIdx.x % nrb;
    const int64_t dch = gridDim.x / nrb, drb = gridDim.x % nrb;
    for (; chunk < nchunk; chunk += dch, rb += drb) {
        if (rb >= nrb) {
            rb -= nrb;
            ++chunk;
            if (chunk >= nchunk) break;
        }
        const int64_t c_raw = chunk * CC + (int64_t)lane * VPL;
        const bool act = c_raw < Ddn;
        const int64_t c = act ? c_raw : Ddn - VPL;
        uint32_t sdc[VPL];
#pragma unroll
        for (int j = 0; j < VPL; ++j) sdc[j] = sd[c + j];
        const float* base = v + c;
        const int64_t uend = min(rb * kUpRows + kUpRows, Dup);
        for (int64_t u = rb * kUpRows + warp; u < uend; u += nw) {
            const int32_t kb = ptr[u];
            const int n = ptr[u + 1] - kb, np = npos[u];
            const int64_t J = u * Ddn + c;
            float4 P{}, N{};
            for (int k0 = 0; k0 < n; k0 += 32) {          // the order of uniform_hops
                const int nk = min(32, n - k0), pend = max(0, min(nk, np - k0));
                const uint32_t mine = lane < nk ? __ldg(list + kb + k0 + lane) : 0u;
                auto load = [&](int q) {
                    const uint32_t t = __shfl_sync(0xffffffffu, mine, q);
                    return __ldg(reinterpret_cast<const float4*>(base + (int64_t)t * Ddn));
                };
                auto four = [&](float4& A, int q) {
                    const float4 a = load(q), b = load(q + 1), x = load(q + 2), y = load(q + 3);
                    addf(A, a, b, x, y);
                };
                int q = 0;
                for (; q + 4 <= pend; q += 4) four(P, q);
                for (; q < pend; ++q) addf(P, load(q));
                for (; q + 4 <= nk; q += 4) four(N, q);
                for (; q < nk; ++q) addf(N, load(q));
            }
            if (!act) continue;
            const uint32_t su_u = su[u];
            const float4 xo = __ldg(reinterpret_cast<const float4*>(v + J));
            const float4 yv = __ldcs(reinterpret_cast<const float4*>(Y + J));
            float r[VPL];
#pragma unroll
            for (int j = 0; j < VPL; ++j) {
                const float nd = (float)__popc(su_u & sdc[j]);
                r[j] = fmaf(mt, (comp(P, j) - comp(N, j)) + comp(yv, j), U * nd * comp(xo, j));
                if (w_old != nullptr) r[j] = fmaf(mbeta, w_old[J + j], r[j]);
            }
            __stcs(reinterpret_cast<float4*>(w + J), make_float4(r[0], r[1], r[2], r[3]));
        }
    }
}

// Up phase with resident rows: a warp builds one row segment of 32 * VPL * NV
// columns with lanes over columns, as above, but the rows belong to the CTA.
//
// CTA (i, j) of the grid owns row range i and the column chunks j, j + gy, ...;
// its rows' hop lists are staged in shared memory once and serve every chunk
// (a range whose lists do not fit goes in blocks).
// All CTAs sweep the chunks in the same order, so the chunk of X that the rows
// of every CTA gather from stays in L2.  A segment is then one dependent step:
// its gathers and its epilogue operands (own element, Y, w_old, f) are all
// requested at once.  Read per segment, the row pointer, the list and the
// epilogue operands each added an L2 or HBM latency to the chain, and with
// registers for 24-32 warps per SM the phase ran at that chain's pace.
__device__ __forceinline__ void stage_up_lists(unsigned char* smem, int cap, int W, int64_t r0, int nr,
                                               const int32_t* __restrict__ ptr, const int32_t* __restrict__ npos,
                                               const uint32_t* __restrict__ list, const uint32_t* __restrict__ su) {
    int2* cnt = reinterpret_cast<int2*>(smem);
    uint32_t* st = reinterpret_cast<uint32_t*>(cnt + cap);
    uint32_t* L = st + cap;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int r = warp; r < nr; r += nw) {
        const int32_t kb = ptr[r0 + r];
        const int n = ptr[r0 + r + 1] - kb;
        for (int k = lane; k < n; k += 32) L[r * W + k] = list[kb + k];
        if (lane == 0) {
            cnt[r] = make_int2(npos[r0 + r], n);
            st[r] = su[r0 + r];
        }
    }
}

// Sums over a staged hop list, +1 targets then -1 targets: add(neg, entries, k)
// sees groups of four, then what is left of the sign as one group of k < 4, so that
// the loads of a group are always requested together (a rest taken one by one is a
// memory latency for each of its entries).  WINDOWS: in windows of 32 entries, the
// order of uniform_hops, for sums that round.
template <bool WINDOWS, typename Add>
__device__ __forceinline__ void list_hops(const uint32_t* L, int np, int n, Add&& add) {
    int q = 0, end = n;
    do {
        if constexpr (WINDOWS) end = min(q + 32, n);
        const int pend = WINDOWS ? max(q, min(end, np)) : np;
        for (; q + 4 <= pend; q += 4) add(false, L + q, std::integral_constant<int, 4>{}, 4);
        if (q < pend) add(false, L + q, std::integral_constant<int, 0>{}, pend - q);
        for (q = pend; q + 4 <= end; q += 4) add(true, L + q, std::integral_constant<int, 4>{}, 4);
        if (q < end) add(true, L + q, std::integral_constant<int, 0>{}, end - q);
        q = end;
    } while (WINDOWS && end < n);
}

// First row of range i of gx: ranges of equal cost, sum of (hops + kUpRowCost).
// The hop counts of neighbouring rows are alike (they share their upper sites),
// so ranges of equally many rows differed enough to leave the SMs idle for a
// third of the phase.  One warp, 32 probes a round.
__device__ __forceinline__ int64_t up_range_start(const int32_t* __restrict__ ptr, int64_t Dup, int i, int gx) {
    const int lane = threadIdx.x & 31;
    const int64_t total = (int64_t)__ldg(ptr + Dup) + kUpRowCost * Dup;
    const int64_t want = (total * i + gx - 1) / gx;
    int64_t lo = 0, hi = Dup;                             // the answer is in [lo, hi]
    while (hi > lo) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t r = min(lo + step * lane, hi);
        const bool below = (int64_t)__ldg(ptr + r) + kUpRowCost * r < want;
        const int nb = __popc(__ballot_sync(0xffffffffu, below));   // probes below: a prefix of the lanes
        if (nb == 0) return lo;
        const int64_t last = min(lo + step * (nb - 1), hi);         // below
        const int64_t next = nb == 32 ? hi : min(lo + step * nb, hi);
        lo = min(last + 1, hi);
        hi = max(next, lo);
    }
    return lo;
}

// the segments of one CTA, seg(row in the staged block, chunk) for every one
template <typename Seg>
__device__ __forceinline__ void up_segments(unsigned char* smem, int64_t Dup, int64_t nchunk, const UpGrid& g,
                                            const int32_t* __restrict__ ptr, const int32_t* __restrict__ npos,
                                            const uint32_t* __restrict__ list, const uint32_t* __restrict__ su,
                                            Seg&& seg) {
    const int i = blockIdx.x % g.gx, j = blockIdx.x / g.gx;
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __shared__ int64_t range[2];
    if (warp < 2) {
        const int64_t r = up_range_start(ptr, Dup, i + warp, g.gx);
        if ((threadIdx.x & 31) == 0) range[warp] = r;
    }
    __syncthreads();
    const int64_t r0 = range[0];
    const int nr = (int)(range[1] - r0);
    if (nr == 0) return;
    if (nr <= g.cap) {
        stage_up_lists(smem, g.cap, g.W, r0, nr, ptr, npos, list, su);
        __syncthreads();
        // segments in (chunk, row) order, dealt to the warps in turn
        int64_t chunk = j;
        int r = warp;
        while (r >= nr && chunk < nchunk) { r -= nr; chunk += g.gy; }
        while (chunk < nchunk) {
            seg(r0, r, chunk);
            r += nw;
            while (r >= nr && chunk < nchunk) { r -= nr; chunk += g.gy; }
        }
        return;
    }
    // so many rows that a chunk of them does not stay in L2 anyway: block by block,
    // each staged once (22 sites (11,2) binary64 product 6.16 -> 5.68 ms)
    for (int b = 0; b < nr; b += g.cap) {
        const int nb = min(g.cap, nr - b);
        __syncthreads();
        stage_up_lists(smem, g.cap, g.W, r0 + b, nb, ptr, npos, list, su);
        __syncthreads();
        for (int64_t chunk = j; chunk < nchunk; chunk += g.gy)
            for (int r = warp; r < nb; r += nw) seg(r0 + b, r, chunk);
    }
}

// Binary64 fixed point, resident rows.  OLD: a replayed Lanczos step, W = H f -
// beta w_old.  CT: CTAs per SM the launch bounds keep.  YS: Y holds word pairs
// (k_rows_planes_f64x).
template <int VPL, bool FAST, bool OLD, bool YS, int CT>
__global__ void __launch_bounds__(256, CT) k_upr_f64x(const int2* X, const long long* Y,
                                                     double* w, const double* w_old, int64_t Dup, int64_t Ddn,
                                                     UpGrid g, const int32_t* __restrict__ ptr,
                                                     const int32_t* __restrict__ npos,
                                                     const uint32_t* __restrict__ list,
                                                     const uint32_t* __restrict__ su,
                                                     const uint32_t* __restrict__ sd,
                                                     const __grid_constant__ EpiParams ep,
                                                     const int* emax_p, int fixed_emax) {
    grid_dep_wait();
    using IV = typename FxVec<VPL>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ long long Bs[33];
    if constexpr (!FAST)
        for (int i = threadIdx.x; i < 33; i += blockDim.x) Bs[i] = i < ep.nB ? ep.B[i] : 0;
    const int emax = fixed_emax > 0 ? fixed_emax : max(*emax_p, 1);
    const int k = 1070 - emax;
    const int lane = threadIdx.x & 31;
    constexpr int CC = 32 * VPL;
    const int2* cnt = reinterpret_cast<const int2*>(smem_raw);
    const uint32_t* st = reinterpret_cast<const uint32_t*>(cnt + g.cap);
    const uint32_t* L = st + g.cap;
    const uint32_t rowb = (uint32_t)Ddn * 8u;             // bytes of a row (Ddn <= kMaxRow)
    up_segments(smem_raw, Dup, (Ddn + CC - 1) / CC, g, ptr, npos, list, su, [&](int64_t r0, int r, int64_t chunk) {
        const int64_t c_raw = chunk * CC + (int64_t)lane * VPL;
        const bool act = c_raw < Ddn;
        const int64_t c = act ? c_raw : Ddn - VPL;     // tail lanes read a valid column, store nothing
        const int64_t J = (r0 + r) * Ddn + c;
        const char* base = reinterpret_cast<const char*>(X + c);
        auto load = [&](uint32_t t) { return *(reinterpret_cast<const IV*>(base + (uint64_t)t * rowb)); };
        // epilogue operands, requested with the gathers
        const IV xo4 = *(reinterpret_cast<const IV*>(X + J));
        long long yv[VPL];
        double wv[VPL];
        uint32_t sdc[VPL];
        if constexpr (VPL == 2) {
            const longlong2 y2 = ld_stream(reinterpret_cast<const longlong2*>(Y + J));
            yv[0] = y2.x;
            yv[1] = y2.y;
            if constexpr (OLD) {
                const double2 q = ld_stream(reinterpret_cast<const double2*>(w_old + J));
                wv[0] = q.x;
                wv[1] = q.y;
            }
        } else {
            yv[0] = ld_stream(Y + J);
            if constexpr (OLD) wv[0] = ld_stream(w_old + J);
        }
        IV A{};
        const int2 np = cnt[r];
        list_hops<false>(L + r * g.W, np.x, np.y, [&](bool neg, const uint32_t* t, auto full, int m) {
            IV x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                x[q] = IV{};
                if (full.value == 4 || q < m) x[q] = load(t[q]);
            }
            if (neg) sub4(A, x[0], x[1], x[2], x[3]);
            else add4(A, x[0], x[1], x[2], x[3]);
        });
        if (!act) return;
#pragma unroll
        for (int j = 0; j < VPL; ++j) sdc[j] = __ldg(sd + c + j);
        const uint32_t su_u = st[r];
        double res[VPL];
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            long long T;
            int2 xo;
            if constexpr (VPL == 2) {
                T = j == 0 ? fx_join(A.x, A.y) : fx_join(A.z, A.w);
                xo = j == 0 ? make_int2(xo4.x, xo4.y) : make_int2(xo4.z, xo4.w);
            } else {
                T = fx_join(A.x, A.y);
                xo = xo4;
            }
            if constexpr (YS) T += fx_join((int)yv[j], (int)(yv[j] >> 32));
            else T += yv[j];
            const int nd = __popc(su_u & sdc[j]);
            if constexpr (FAST) {
                // exact: |T| < 2^55, |X| <= 2^48, |Uint * n| < 2^14 and tshift <= 6
                const long long Pv = fast_sum(T, xo, nd, ep);
                res[j] = i64_scaled_to_double(Pv, -(k + ep.ju));
                if constexpr (OLD) res[j] = fma(ep.mbeta, wv[j], res[j]);
            } else {
                I128 acc{0ull, 0ll};
                mac_t(acc, T, ep);
                mac128(acc, fx_join(xo.x, xo.y), Bs[nd]);
                if constexpr (OLD) {
                    int glo, ghi;
                    fx_split(wv[j], emax, glo, ghi);
                    mac128(acc, fx_join(glo, ghi), ep.Bbeta);
                }
                res[j] = i128_to_double(acc, -(k + ep.m));
            }
        }
        if constexpr (VPL == 2) __stcs(reinterpret_cast<double2*>(w + J), make_double2(res[0], res[1]));
        else __stcs(w + J, res[0]);
    });
}

// Binary32: same decomposition, float arithmetic.  NV vectors of VPL columns
// per lane, 32 * VPL columns apart, so rows whose length only allows narrow
// vectors still keep as many bytes in flight.
template <int VPL, int NV>
__global__ void __launch_bounds__(256, 4) k_up_f32(const float* v, const float* Y, float* w,
                                                   const float* w_old, int64_t Dup, int64_t Ddn, UpGrid g,
                                                   const int32_t* __restrict__ ptr, const int32_t* __restrict__ npos,
                                                   const uint32_t* __restrict__ list, const uint32_t* __restrict__ su,
                                                   const uint32_t* __restrict__ sd, float mt, float U, float mbeta) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_dep_wait();
    using V = typename F32Vec<VPL>::T;
    const int lane = threadIdx.x & 31;
    constexpr int CC = 32 * VPL * NV;
    const int2* cnt = reinterpret_cast<const int2*>(smem_raw);
    const uint32_t* st = reinterpret_cast<const uint32_t*>(cnt + g.cap);
    const uint32_t* L = st + g.cap;
    const uint32_t rowb = (uint32_t)Ddn * 4u;
    up_segments(smem_raw, Dup, (Ddn + CC - 1) / CC, g, ptr, npos, list, su, [&](int64_t r0, int r, int64_t chunk) {
        int64_t c[NV];
        bool act[NV];
        V xo[NV], yv[NV], wv[NV], P[NV], N[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int64_t c_raw = chunk * CC + (int64_t)(i * 32 + lane) * VPL;
            act[i] = c_raw < Ddn;
            c[i] = act[i] ? c_raw : Ddn - VPL;
            const int64_t J = (r0 + r) * Ddn + c[i];
            xo[i] = *(reinterpret_cast<const V*>(v + J));
            yv[i] = ld_stream(reinterpret_cast<const V*>(Y + J));
            if (w_old != nullptr) wv[i] = ld_stream(reinterpret_cast<const V*>(w_old + J));
            P[i] = V{};
            N[i] = V{};
        }
        auto load = [&](uint32_t t, int i) {
            return *(reinterpret_cast<const V*>(reinterpret_cast<const char*>(v + c[i]) + (uint64_t)t * rowb));
        };
        const int2 np = cnt[r];
        list_hops<true>(L + r * g.W, np.x, np.y, [&](bool neg, const uint32_t* t, auto full, int m) {
            V x[NV][4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    x[i][q] = V{};
                    if (full.value == 4 || q < m) x[i][q] = load(t[q], i);
                }
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                V& A = neg ? N[i] : P[i];
                if constexpr (full.value == 4) {
                    addf(A, x[i][0], x[i][1], x[i][2], x[i][3]);
                } else {
                    addf(A, x[i][0]);
                    addf(A, x[i][1]);
                    addf(A, x[i][2]);
                }
            }
        });
        const uint32_t su_u = st[r];
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            if (!act[i]) continue;
            const int64_t J = (r0 + r) * Ddn + c[i];
            float res[VPL];
#pragma unroll
            for (int j = 0; j < VPL; ++j) {
                const float nd = (float)__popc(su_u & __ldg(sd + c[i] + j));
                res[j] = fmaf(mt, (comp(P[i], j) - comp(N[i], j)) + comp(yv[i], j), U * nd * comp(xo[i], j));
                if (w_old != nullptr) res[j] = fmaf(mbeta, comp(wv[i], j), res[j]);
            }
            if constexpr (VPL == 4) __stcs(reinterpret_cast<float4*>(w + J), make_float4(res[0], res[1], res[2], res[3]));
            else if constexpr (VPL == 2) __stcs(reinterpret_cast<float2*>(w + J), make_float2(res[0], res[1]));
            else __stcs(w + J, res[0]);
        }
    });
}

// ---------------------------------------------------------------------------
// binary32 variants: same structure, float arithmetic (UPD: the deferred
// Lanczos update, rounded as k_axpy_scale_f32)
template <int VEC, typename EntT, bool UPD>
__global__ void __launch_bounds__(1024, 1) k_rows_f32(std::conditional_t<UPD, float*, const float*> v,
                                                    float* __restrict__ Y, int64_t Dup,
                                                    int64_t Ddn, const int64_t* __restrict__ boff,
                                                    const int32_t* __restrict__ bcnt,
                                                    const EntT* __restrict__ ent,
                                                    const float* fo, float ua, float uinv,
                                                    const LzDev* dv) {
    using S = typename F32Vec<VEC>::T;
    grid_dep_wait();
    if constexpr (UPD) {
        if (dv != nullptr) {
            if (dv->stall) return;
            ua = (float)dv->ua;
            uinv = (float)dv->uinv;
        }
    }
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S* X = reinterpret_cast<S*>(smem_raw);
    float* Xf = reinterpret_cast<float*>(smem_raw);
    const int lane = threadIdx.x & 31;
    const int64_t nblk = (Dup + VEC - 1) / VEC;
    const int64_t step = blockDim.x;
    constexpr int NL = UPD ? 2 : 4;                       // row elements per thread in flight
    {
        const int64_t z0 = staged_slots(Ddn) - 32;
        for (int i = threadIdx.x; i < 32 * VEC; i += blockDim.x) Xf[z0 * VEC + i] = 0.0f;
    }
    for (int64_t b = blockIdx.x; b < nblk; b += gridDim.x) {
        const int64_t u0 = b * VEC;
        const int nrow = (int)((Dup - u0) < VEC ? (Dup - u0) : VEC);
        // NL loads per row in flight (with UPD all issued before the first store)
        for (int64_t d0 = threadIdx.x; d0 < Ddn; d0 += NL * step) {
            float xv[NL][VEC];
            [[maybe_unused]] float fv[NL][VEC];
#pragma unroll
            for (int i = 0; i < NL; ++i)
#pragma unroll
                for (int r = 0; r < VEC; ++r) {
                    const int64_t d = d0 + i * step;
                    const bool in = d < Ddn && r < nrow;
                    xv[i][r] = in ? v[(u0 + r) * Ddn + d] : 0.0f;
                    if constexpr (UPD) fv[i][r] = in ? fo[(u0 + r) * Ddn + d] : 0.0f;
                }
            if constexpr (UPD) {
#pragma unroll
                for (int i = 0; i < NL; ++i)
#pragma unroll
                    for (int r = 0; r < VEC; ++r) {
                        const int64_t d = d0 + i * step;
                        if (d < Ddn && r < nrow) {
                            xv[i][r] = fmaf(ua, fv[i][r], xv[i][r]) * uinv;
                            __stcs(v + (u0 + r) * Ddn + d, xv[i][r]);
                        }
                    }
            }
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int64_t d = d0 + i * step;
                if (d >= Ddn) break;
#pragma unroll
                for (int r = 0; r < VEC; ++r) Xf[d * VEC + r] = xv[i][r];
            }
        }
        __syncthreads();
        for (int64_t d0 = threadIdx.x & ~31; d0 < Ddn; d0 += step) {
            const int64_t g = d0 >> 5;
            const int64_t d = d0 + lane;
            float acc[VEC];
#pragma unroll
            for (int r = 0; r < VEC; ++r) acc[r] = 0.0f;
            for_each_hop<EntT>(ent + boff[g], bcnt[g], lane, [&](uint32_t e) {
                const float s = (float)RowEnt<EntT>::sgn(e);  // padding reads a zero slot
                const S x = X[RowEnt<EntT>::idx(e)];
#pragma unroll
                for (int r = 0; r < VEC; ++r) acc[r] = fmaf(s, comp(x, r), acc[r]);
            });
            if (d < Ddn) {
#pragma unroll
                for (int r = 0; r < VEC; ++r)
                    if (r < nrow) Y[(u0 + r) * Ddn + d] = acc[r];
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// thread-safe (static initialisation runs once; callers on other threads wait)
int smem_optin() {
    static const int v = [] {
        int dev = 0, x = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&x, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        return x > 0 ? x : 48 * 1024;
    }();
    return v;
}

int sms() {
    static const int n = [] {
        int dev = 0, x = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&x, cudaDevAttrMultiProcessorCount, dev);
        return x > 0 ? x : 1;
    }();
    return n;
}

// static shared memory of the binary64 row kernels (cta_exponent)
constexpr int kRowStatic = 16;

// largest VEC in {4,2,1} (capped by vmax) whose staging buffer (with the
// zero slots) fits
int pick_vec(int64_t len, int elem_bytes, int vmax, int reserve) {
    for (int v = vmax; v >= 1; v >>= 1)
        if (staged_slots(len) * elem_bytes * v + reserve <= smem_optin()) return v;
    return 0;
}

struct Launch {
    int blocks, threads;
    size_t smem;
};

// ctas = 0: two CTAs per SM when both fit, else one
Launch shape(size_t smem, int ctas) {
    const size_t per_sm = 228 * 1024;
    const int fit = (int)std::max<size_t>(1, std::min<size_t>(2, per_sm / (smem + 2048)));
    if (ctas <= 0 || ctas > fit) ctas = fit;
    Launch L;
    L.smem = smem;
    L.threads = ctas == 1 ? 1024 : 512;
    L.blocks = sms() * ctas;
    return L;
}

// The dynamic shared-memory limit is a per-kernel attribute shared by every
// host thread: raise it once per kernel (the template parameter is the kernel
// itself, so each instantiation has its own flag), to the device maximum, so
// that a concurrent launch of the same kernel can never see a lower limit.
// The limit is what the opt-in maximum leaves next to the kernel's static
// shared memory.
template <auto Kern>
void allow_smem() {
    static const bool once = [] {
        cudaFuncAttributes fa{};
        if (cudaFuncGetAttributes(&fa, Kern) != cudaSuccess) return false;
        const int dyn = smem_optin() - (int)fa.sharedSizeBytes;
        return cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) == cudaSuccess;
    }();
    (void)once;
}

// Which binary64 up phase forms a product or a replayed step of a sector with rows
// of even length (odd ones always take the resident-row kernel):
//   up to kUpSmall elements: work items dealt over all CTAs -- a CTA has one or
//     two, and staging lists would only lengthen its chain;
//   above: resident rows (4x4 (5,5) product 414 -> 376 us), except
//   standalone products of more than kUpHbm bytes a vector (4x4 (8,8) 3.80 ms
//     with items, 4.11 with resident rows; 4x4 (7,7) 2.87, 2.95; ring 16 (6,6),
//     513 MB: 1.10, 1.05).
// A Lanczos step has items of one shape at every size (kUpRows).  On more than
// kUpSmall elements its kernel and the item product take the rest of a hop list
// one by one (4x4 (8,8) product 3.80 ms, 4.49 with padded groups).
constexpr int64_t kUpSmall = 2500000, kUpHbm = 600ll << 20;
// Kernels of a sector start while the one before drains (launch_on) when its
// vectors stay in L2 (ring 12 product 29.9 -> 26.1 us, step 55.9 -> 44.3 us); on
// HBM-sized ones CTAs that take their places early disturb the sweep (4x4 (8,8)
// product 3.80 -> 4.10 ms).
constexpr int64_t kPdlBytes = 100ll << 20;
// up to this many elements every row-phase CTA scans v for its largest exponent
// (ring 8 (4,4) product: two kernels instead of a memset and three)
constexpr int64_t kScanElems = 16384;
constexpr int64_t kMaxRow = (1ll << 29) - 1;       // row pitch in bytes held in 32 bits

// items of a Lanczos step's up phase (k_up_step_f64x, k_up_step_f32)
int64_t up_step_items(int vpl, int64_t Dup, int64_t Ddn) {
    return (Ddn + 32 * vpl - 1) / (32 * vpl) * ((Dup + kUpRows - 1) / kUpRows);
}

// a grid of at most `full` CTAs and no more than the work items
int grid_cap(int full, int64_t items) { return (int)std::max<int64_t>(1, std::min<int64_t>(full, items)); }

// requested vec (0 = largest that fits), capped to what fits
int choose_vec(int req, int64_t len, int elem_bytes, int vmax, int reserve) {
    const int fit = pick_vec(len, elem_bytes, vmax, reserve);
    if (req <= 0 || req > fit) return fit;
    return req;
}

// Whether a binary32 product or replayed step takes items: where a range's lists
// do not fit in shared memory at a time, or serve one chunk of many rows, staging
// them gains nothing (24 sites (8,2), 276 columns: 2.97 ms with resident rows, 2.51
// with items; (12,0): 2.90, 2.71; 18 sites (9,1): 59, 55 us, but 16 sites (8,1),
// 21 rows a range: 19, 21 us).  Rows of odd length keep the resident kernel's two
// segments a lane (22 sites (11,2): 2.86, 3.61 ms).
bool up_items32(const UpGrid& g, int vpl, int64_t nchunk) {
    if (nchunk == 1) return g.rows > 48;
    return vpl > 1 && g.rows > g.cap;
}

// Whether a binary32 product or replayed step takes k_up_lean_f32: 16-byte columns
// and vectors of more than 2 GiB (18 sites (5,9), 1.7 GB: 4.59 ms, 4.38 with resident
// rows; (6,9), 3.6 GB: 10.16, 10.78; narrower columns gain with resident rows at any
// size, (9,8), 8.5 GB: 28.7 ms, 32.2 with items).
bool up_lean32(int64_t D, int vpl) { return vpl == 4 && D * 4 > (2ll << 30); }

UpGrid up_grid_for(const hubbard_sector* H, int64_t nchunk, int ctas) {
    return make_up_grid(H->Dup, (int64_t)H->host[0].tgt.size(), H->host[0].W, nchunk, ctas);
}

}  // namespace

// Returns HUB_OK and launches, or returns -1 when the staging buffers do not fit
// (the caller then uses the single-pass gather kernel).
bool hv_phases_fuse(const hubbard_sector* H, int dtype) {
    if (H->Ddn > kMaxRow) return false;
    if (sms() * kStepCtas32 > kPartStride) return false;   // one partial per CTA
    return dtype == HUB_F64 || choose_vec(H->vec_rows, H->Ddn, 4, 4, 0) != 0;
}

int launch_hv_phases(hubbard_sector* H, const void* v, void* w, int dtype, double beta, const void* w_old,
                     void* ybuf, int fixed_emax, cudaStream_t s, double* part, int* nparts,
                     const RowUpdate* upd, LzDev* dv, double* hist) {
    if (nparts != nullptr) *nparts = 0;
    if (H->Ddn > kMaxRow) return -1;
    if (sms() * kStepCtas32 > kPartStride) part = nullptr;   // partial arrays too short: no fused reduction
    const DevSpin& up = H->dev[0];
    const DevSpin& dn = H->dev[1];
    const int64_t Dup = H->Dup, Ddn = H->Ddn;
    const bool dn16 = dn.ent16 != nullptr;
    unsigned* done = reinterpret_cast<unsigned*>(H->status + 2);   // of the step kernels alone
    const bool pdl = H->D * (dtype == HUB_F64 ? 8 : 4) <= kPdlBytes;
    // up-phase CTAs: as many as the launch bounds keep resident (the phase is
    // bound by L2 latency, so occupancy is what counts): 4 per SM at <= 64
    // registers, 3 where binary64 requests its epilogue's operands before the
    // gathers (the Lanczos step, replayed steps, pre below)
    if (dtype == HUB_F64) {
        const int va = choose_vec(H->vec_rows, Ddn, 8, 2, kRowStatic);
        // exponent bound: found by the row phase itself on the smallest sectors, by a
        // pass of its own otherwise.  On sectors that launch overlapped that pass
        // leaves one maximum per CTA, which the row phase reduces: no memset of a
        // word that all CTAs raise breaks the chain of kernels.
        const bool ysplit = va == 0 && H->D * 8 <= kPdlBytes && staged_slots(Ddn) * 4 + kRowStatic <= smem_optin();
        const int scan = fixed_emax <= 0 && w_old == nullptr && va > 0 && H->D <= kScanElems;
        const bool by_slots = fixed_emax <= 0 && w_old == nullptr && pdl && !scan && (va > 0 || ysplit);
        int* emax = H->status;
        const int* slots = by_slots ? H->status + kStatusWords : nullptr;
        int nslots = 0;
        // the deferred update goes into the row phase when it stages rows in
        // shared memory with a fixed exponent bound; otherwise it is one pass first
        if (upd != nullptr && (va == 0 || fixed_emax <= 0)) {
            if (int rc = launch_axpy_scale(upd->a, upd->inv, upd->fo, const_cast<void*>(v), H->D, dtype, s, upd->dv))
                return rc;
            upd = nullptr;
        }
        if (fixed_emax <= 0 && !scan) {
            if (by_slots) {
                nslots = launch_max_exponent_slots((const double*)v, H->D, H->status + kStatusWords, s);
            } else {
                HUB_CUDA(cudaMemsetAsync(emax, 0, sizeof(int), s));
                launch_max_exponent((const double*)v, H->D, emax, s);
                if (w_old != nullptr) launch_max_exponent((const double*)w_old, H->D, emax, s);
            }
        }
        Launch LA = shape((size_t)staged_slots(Ddn) * 8 * std::max(va, 1), H->ctas_rows);
        LA.blocks = grid_cap(LA.blocks, (Dup + std::max(va, 1) - 1) / std::max(va, 1));   // no idle CTAs
        long long* Y = (long long*)ybuf;
        int2* Xg = (int2*)((char*)ybuf + (size_t)H->D * 8);
        int extra = 0;
        if (ysplit) {
            // rows of which one word per element fits in shared memory
            const size_t sm = (size_t)staged_slots(Ddn) * 4;
            const int64_t groups = 2 * Dup * ((Ddn + 31) / 32);
            const int blocks = grid_cap(sms(), (groups + 31) / 32);
            extra = 1;
#define PLANES64(E, P)                                                                                      \
    allow_smem<k_rows_planes_f64x<E>>();                                                                    \
    launch_on(pdl, k_rows_planes_f64x<E>, blocks, 1024, sm, s, (const double*)v, (int*)Y, Xg, Dup, Ddn, \
        dn.blk_off, dn.blk_cnt, P, emax, fixed_emax, slots, nslots)
            if (dn16) { PLANES64(uint16_t, dn.ent16); } else { PLANES64(uint32_t, dn.ent32); }
#undef PLANES64
        } else if (va == 0) {
            // fixed-point copy first, then gathers through L1/L2
            int* em = emax;
            int* fixed_word = H->status + 1;
            if (fixed_emax > 0) {
                H->fixed_emax_host = fixed_emax;
                HUB_CUDA(cudaMemcpyAsync(fixed_word, &H->fixed_emax_host, sizeof(int), cudaMemcpyHostToDevice, s));
                em = fixed_word;
            }
            launch_to_fixed((const double*)v, H->D, Xg, em, s);
            if (dn16) {
                k_rows_global_f64x<uint16_t><<<grid_cap(sms() * 4, Dup), 512, 0, s>>>(Xg, Y, Dup, Ddn, dn.blk_off,
                                                                                         dn.blk_cnt, dn.ent16);
            } else {
                k_rows_global_f64x<uint32_t><<<grid_cap(sms() * 4, Dup), 512, 0, s>>>(Xg, Y, Dup, Ddn, dn.blk_off,
                                                                                         dn.blk_cnt, dn.ent32);
            }
            extra = 2;
        } else {
#define ROWS64_U(V, E, P, U)                                                                                \
    allow_smem<k_rows_f64x<V, E, U>>();                                                                      \
    launch_on(pdl, k_rows_f64x<V, E, U>, LA.blocks, LA.threads, LA.smem, s, (double*)const_cast<void*>(v), Y, Xg, Dup,   \
        Ddn, dn.blk_off, dn.blk_cnt, P, emax, fixed_emax, scan, slots, nslots, upd ? (const double*)upd->fo : nullptr,            \
        upd ? upd->a : 0.0, upd ? upd->inv : 1.0, upd ? upd->dv : nullptr)
#define ROWS64(V, E, P) if (upd) { ROWS64_U(V, E, P, true); } else { ROWS64_U(V, E, P, false); }
        if (va == 2) {
            if (dn16) { ROWS64(2, uint16_t, dn.ent16); } else { ROWS64(2, uint32_t, dn.ent32); }
        } else {
            if (dn16) { ROWS64(1, uint16_t, dn.ent16); } else { ROWS64(1, uint32_t, dn.ent32); }
        }
        extra = 1;
        }
#undef ROWS64
#undef ROWS64_U
        const EpiParams ep = make_epilogue(H->t, H->U, H->ns, w_old ? beta : 0.0, H->host[0].W + H->host[1].W);
        // columns per lane in the up phase: 2 when Ddn is even (16-byte loads)
        const int vpl = ((Ddn & 1) == 0 && H->vec_cols != 1) ? 2 : 1;
        const bool tail = H->D <= kUpSmall;
        int up_grid = 0;
        if (part != nullptr) {                            // a Lanczos step
            const int64_t items = up_step_items(vpl, Dup, Ddn);
            up_grid = grid_cap(sms() * kStepCtas64, items);
#define UPS64(V, F, T, YS, NT)                                                                              \
    launch_on(pdl, k_up_step_f64x<V, F, T, YS, NT>, up_grid, NT, 0, s, Xg, Y, (double*)w, (const double*)w_old, Dup, \
        Ddn, up.pn_ptr, up.pn_npos, up.pn_list, up.states, dn.states, ep, emax, fixed_emax, (const double*)v, part, \
        done, dv, hist)
#define UPS64_T(V, F)                                                                                      \
    if (ysplit) { if (tail) { UPS64(V, F, true, true, 256); } else { UPS64(V, F, false, true, 256); } }    \
    else if (items <= sms()) { UPS64(V, F, true, false, 512); }                                            \
    else if (tail) { UPS64(V, F, true, false, 256); }                                                      \
    else { UPS64(V, F, false, false, 256); }
            if (vpl == 2) {
                if (ep.fast) { UPS64_T(2, true) } else { UPS64_T(2, false) }
            } else {
                if (ep.fast) { UPS64_T(1, true) } else { UPS64_T(1, false) }
            }
#undef UPS64_T
#undef UPS64
        } else if (vpl == 1 || ysplit || (H->D > kUpSmall && (w_old != nullptr || H->D * 8 <= kUpHbm))) {
            const bool three = w_old != nullptr || (H->ctas_cols == 2 && !ysplit);
            const UpGrid g = up_grid_for(H, (Ddn + 32 * vpl - 1) / (32 * vpl), sms() * (three ? 3 : 4));
#define UPR64(V, F, OLD, YS, CT)                                                                            \
    launch_on(pdl, k_upr_f64x<V, F, OLD, YS, CT>, g.gx * g.gy, 256, g.smem, s, Xg, Y, (double*)w,              \
        (const double*)w_old, Dup, Ddn, g, up.pn_ptr, up.pn_npos, up.pn_list, up.states, dn.states, ep, emax,  \
        fixed_emax)
#define UPR64_S(V, F)                                                                                      \
    if (ysplit) { if (three) { UPR64(V, F, true, true, 3); } else { UPR64(V, F, false, true, 4); } }       \
    else if (w_old != nullptr) { UPR64(V, F, true, false, 3); }                                            \
    else if (three) { UPR64(V, F, false, false, 3); }                                                      \
    else { UPR64(V, F, false, false, 4); }
            if (vpl == 2) {
                if (ep.fast) { UPR64_S(2, true) } else { UPR64_S(2, false) }
            } else {
                if (ep.fast) { UPR64_S(1, true) } else { UPR64_S(1, false) }
            }
#undef UPR64_S
#undef UPR64
        } else {
            const int64_t up_chunks = (Ddn + 63) / 64;
            const int rbr = up_rows(up_chunks, Dup, sms() * 4);
            const int64_t up_items = up_chunks * ((Dup + rbr - 1) / rbr);
            // standalone: request the epilogue's own element and Y before the
            // gathers (at 3 CTAs/SM for the registers) where that measured faster --
            // the 128-bit epilogue and rows staged from global memory -- unless the
            // schedule fixes it (ctas_cols 1: no, 2: yes)
            const bool pre = H->ctas_cols == 2 || (H->ctas_cols == 0 && (!ep.fast || va == 0));
#define UP64(CT, ...)                                                                                       \
    launch_on(pdl, k_up_f64x<__VA_ARGS__>, grid_cap(sms() * CT, up_items), 256, 0, s, Xg, Y, (double*)w,       \
        (const double*)w_old, Dup, Ddn, rbr, up.pn_ptr, up.pn_npos, up.pn_list, up.states, dn.states, ep,  \
        emax, fixed_emax)
#define UP64_T(F, T)                                                                                        \
    if (pre) { UP64(3, F, T, true, 3); } else { UP64(4, F, T); }
            if (tail) {
                if (ep.fast) { UP64_T(true, true) } else { UP64_T(false, true) }
            } else {
                if (ep.fast) { UP64_T(true, false) } else { UP64_T(false, false) }
            }
#undef UP64_T
#undef UP64
        }
        if (part != nullptr && nparts != nullptr) *nparts = up_grid;
        HUB_CUDA(cudaGetLastError());
        count_launches(1 + extra + (fixed_emax <= 0 && !scan ? (w_old ? 2 : 1) : 0));
        return HUB_OK;
    }
    // binary32
    const int va = choose_vec(H->vec_rows, Ddn, 4, 4, 0);
    if (va == 0) return -1;
    Launch LA = shape((size_t)staged_slots(Ddn) * 4 * va, H->ctas_rows);
    LA.blocks = grid_cap(LA.blocks, (Dup + va - 1) / va);
    float* Y = (float*)ybuf;
    // columns per lane in the up phase: the widest aligned vector load, capped by vec_cols
    int vpl = (Ddn & 3) == 0 ? 4 : ((Ddn & 1) == 0 ? 2 : 1);
    if (H->vec_cols > 0 && H->vec_cols < vpl) vpl = H->vec_cols;
#define ROWS32_U(V, E, P, U)                                                                               \
    allow_smem<k_rows_f32<V, E, U>>();                                                                      \
    launch_on(pdl, k_rows_f32<V, E, U>, LA.blocks, LA.threads, LA.smem, s, (float*)const_cast<void*>(v), Y, Dup, Ddn,   \
        dn.blk_off, dn.blk_cnt, P, upd ? (const float*)upd->fo : nullptr, upd ? (float)upd->a : 0.0f,       \
        upd ? (float)upd->inv : 1.0f, upd ? upd->dv : nullptr)
#define ROWS32(V, E, P) if (upd) { ROWS32_U(V, E, P, true); } else { ROWS32_U(V, E, P, false); }
#define BOTH32(M, V, F, P16, P32) if (F) { M(V, uint16_t, P16); } else { M(V, uint32_t, P32); }
    if (va == 4) { BOTH32(ROWS32, 4, dn16, dn.ent16, dn.ent32) }
    else if (va == 2) { BOTH32(ROWS32, 2, dn16, dn.ent16, dn.ent32) }
    else { BOTH32(ROWS32, 1, dn16, dn.ent16, dn.ent32) }
#undef BOTH32
#undef ROWS32
#undef ROWS32_U
    int up_grid = 0;
    const int cols = vpl == 1 ? 64 : 128;                 // of a resident-row segment
    const int64_t nchunk = (Ddn + cols - 1) / cols;
    const UpGrid g = up_grid_for(H, nchunk, sms() * 4);
    if (part == nullptr && up_lean32(H->D, vpl)) {
        up_grid = grid_cap(sms() * kStepCtas32, up_step_items(vpl, Dup, Ddn));
        k_up_lean_f32<<<up_grid, 256, 0, s>>>((const float*)v, Y, (float*)w, (const float*)w_old, Dup, Ddn, up.pn_ptr,
            up.pn_npos, up.pn_list, up.states, dn.states, (float)-H->t, (float)H->U, (float)-beta);
    } else if (part != nullptr || up_items32(g, vpl, nchunk)) {
        up_grid = grid_cap(sms() * up32_ctas(vpl, part != nullptr), up_step_items(vpl, Dup, Ddn));
#define UPS32(V, RED)                                                                                      \
    launch_on(pdl, k_up_step_f32<V, RED>, up_grid, 256, 0, s, (const float*)v, Y, (float*)w, (const float*)w_old, \
        Dup, Ddn, up.pn_ptr, up.pn_npos, up.pn_list, up.states, dn.states, (float)-H->t, (float)H->U,       \
        (float)-beta, part, done, dv, hist)
#define UPS32_R(V) if (part != nullptr) { UPS32(V, true); } else { UPS32(V, false); }
        if (vpl == 4) { UPS32_R(4) } else if (vpl == 2) { UPS32_R(2) } else { UPS32_R(1) }
#undef UPS32_R
#undef UPS32
    } else {
#define UP32(V, NV)                                                                                        \
    {                                                                                                      \
        launch_on(pdl, k_up_f32<V, NV>, g.gx * g.gy, 256, g.smem, s, (const float*)v, Y, (float*)w,         \
            (const float*)w_old, Dup, Ddn, g, up.pn_ptr, up.pn_npos, up.pn_list, up.states, dn.states,      \
            (float)-H->t, (float)H->U, (float)-beta);                                                      \
    }
        if (vpl == 4) { UP32(4, 1) } else if (vpl == 2) { UP32(2, 2) } else { UP32(1, 2) }
#undef UP32
    }
    if (part != nullptr && nparts != nullptr) *nparts = up_grid;
    HUB_CUDA(cudaGetLastError());
    count_launches(2);
    return HUB_OK;
}

}  // namespace hub
