// k_reduce.cu -- readout reductions over the state vector (one read pass each).
//
//  * norm2:  sum |a_x|^2
//  * probs:  marginal probabilities over a set of physical bit positions
//  * expect: sum_t c_t <psi|P_t|psi> for Pauli strings, grouped by X mask so that one pass
//            serves every term with the same X mask: P|x> = i^{#Y} (-1)^{popcount(x&z)} |x^xm>.
//            Groups of four or more terms go through 1024-amplitude Walsh-Hadamard tiles, so
//            the pass costs the same whatever the number of terms; smaller groups loop over
//            their terms per amplitude.
//
// Accumulation: per-thread partial sums (FP64 for complex128; for complex64 at most 32 FP32
// terms are summed before conversion to FP64), warp-shuffle and shared-memory tree per block,
// then a second single-block kernel sums the per-block partials in a fixed order, so results
// are deterministic for a given launch shape.  The per-block partials live in device scratch
// memory owned by the state.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <type_traits>
#include <unordered_map>
#include <vector>

#include "qs_internal.h"
#include "staging.h"

namespace qs {
namespace {

constexpr int kRedThreads = 256;
constexpr int kRedBlocksMax = 4096;
constexpr int kMaxTermsPerGroup = 256;

template <typename R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide sum of two doubles; result valid in thread 0.
__device__ __forceinline__ void block_sum2(double &a, double &b)
{
    __shared__ double sa[32], sb[32];
    a = warp_sum(a);
    b = warp_sum(b);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) { sa[w] = a; sb[w] = b; }
    __syncthreads();
    if (w == 0) {
        const int nw = blockDim.x >> 5;
        a = lane < nw ? sa[lane] : 0.0;
        b = lane < nw ? sb[lane] : 0.0;
        a = warp_sum(a);
        b = warp_sum(b);
    }
}

// Each block handles a contiguous range of amplitudes; thread t of the block reads elements
// t, t + T, ... of that range (coalesced), kUnroll independent loads at a time.
constexpr int kUnroll = 8;
template <typename R>
__global__ void __launch_bounds__(kRedThreads) norm2_kernel(const typename Cx<R>::T *__restrict__ a,
                                                            uint64_t N, double *__restrict__ part)
{
    using T = typename Cx<R>::T;
    const uint64_t per = (N + gridDim.x - 1) / gridDim.x;
    const uint64_t lo = per * blockIdx.x;
    const uint64_t hi = lo + per < N ? lo + per : N;
    double acc = 0.0;
    for (uint64_t x0 = lo + threadIdx.x; x0 < hi; x0 += uint64_t(kUnroll) * blockDim.x) {
        T v[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const uint64_t x = x0 + uint64_t(u) * blockDim.x;
            v[u] = x < hi ? a[x] : T{};
        }
        // complex64: the kUnroll squares are summed in FP32, then added in FP64
        R f = 0;
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            f = fma(v[u].x, v[u].x, f);
            f = fma(v[u].y, v[u].y, f);
        }
        acc += (double)f;
    }
    double dummy = 0.0;
    block_sum2(acc, dummy);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// Sum `count` pairs (re, im) laid out as part[i], part[stride + i]; writes out[0], out[1], or adds to them.
__global__ void __launch_bounds__(kRedThreads) finish_kernel(const double *__restrict__ part, int count,
                                                             int stride, double *__restrict__ out, bool add)
{
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < count; i += blockDim.x) {
        a += part[i];
        if (stride) b += part[stride + i];
    }
    block_sum2(a, b);
    if (threadIdx.x == 0) {
        out[0] = add ? out[0] + a : a;
        out[1] = add ? out[1] + b : b;
    }
}

struct TermGroup {
    uint64_t xm;
    int nterms;
    uint64_t zm[kMaxTermsPerGroup];
    double cre[kMaxTermsPerGroup];  // coeff * Re(i^{#Y})
    double cim[kMaxTermsPerGroup];  // coeff * Im(i^{#Y})
};

// sum_x conj(a[x^xm]) a[x] sum_j c_j i^{ny_j} (-1)^{popc(x & zm_j)}
template <typename R>
__global__ void __launch_bounds__(kRedThreads) expect_kernel(const typename Cx<R>::T *__restrict__ a,
                                                             uint64_t N, const TermGroup *__restrict__ grp,
                                                             double *__restrict__ part)
{
    __shared__ uint64_t zm[kMaxTermsPerGroup];
    __shared__ R cre[kMaxTermsPerGroup], cim[kMaxTermsPerGroup];
    const int nt = grp->nterms;
    const uint64_t xm = grp->xm;
    for (int j = threadIdx.x; j < nt; j += blockDim.x) {
        zm[j] = grp->zm[j];
        cre[j] = (R)grp->cre[j];
        cim[j] = (R)grp->cim[j];
    }
    __syncthreads();
    const uint64_t per = (N + gridDim.x - 1) / gridDim.x;
    const uint64_t lo = per * blockIdx.x;
    const uint64_t hi = lo + per < N ? lo + per : N;
    double accr = 0.0, acci = 0.0;
    R fr = 0, fi = 0;
    int cnt = 0;
    for (uint64_t x = lo + threadIdx.x; x < hi; x += blockDim.x) {
        const auto ax = a[x];
        const auto ay = a[x ^ xm];
        // v = conj(ay) * ax
        const R vr = (R)ay.x * (R)ax.x + (R)ay.y * (R)ax.y;
        const R vi = (R)ay.x * (R)ax.y - (R)ay.y * (R)ax.x;
        R er = 0, ei = 0;
        for (int j = 0; j < nt; ++j) {
            const R s = (__popcll(x & zm[j]) & 1) ? R(-1) : R(1);
            er = fma(s, cre[j], er);
            ei = fma(s, cim[j], ei);
        }
        // (er + i ei) * (vr + i vi)
        fr += er * vr - ei * vi;
        fi += er * vi + ei * vr;
        if (sizeof(R) == 4 && ++cnt == 32) {
            accr += (double)fr;
            acci += (double)fi;
            fr = fi = 0;
            cnt = 0;
        }
    }
    accr += (double)fr;
    acci += (double)fi;
    block_sum2(accr, acci);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = accr;
        part[gridDim.x + blockIdx.x] = acci;
    }
}

// Walsh-Hadamard form of one X-mask group.  Write an index as x = (H, L) with L its low 10 bits
// and split each Z mask the same way, z_t = (zh_t, zl_t).  With v(x) = conj(a[x^xm]) a[x],
//   sum_x v(x) sum_t C_t (-1)^{popc(x & z_t)} = sum_H sum_t C_t s_t(H) Vhat_H(zl_t),
// where s_t(H) = (-1)^{popc(H & zh_t)} and Vhat_H is the Walsh-Hadamard transform of v(H, .)
// over the 1024 values of L.  One warp transforms one tile (10 butterfly stages: the bits held
// in a lane's 32 registers, then the five lane bits through shuffles), writes Vhat to shared
// memory and then spends one lookup per term, so the per-amplitude work no longer grows with
// the number of terms.
//   When xm has a bit p >= 10, the tiles with bit p of the index clear are paired with their
// partners H ^ (xm >> 10): the partner's v is conj(v) and its term signs are those of x times
// (-1)^{popc(xm & z_t)}, so one tile pass covers both and every amplitude is read once.  The
// host folds both into four real coefficients per term: re += A Vr + B Vi, im += C Vi + D Vr.
constexpr int kWhtTileLog = 10;
struct WhtTerms {
    uint64_t xm;
    int nterms;
    int pair;
    uint64_t zh[kMaxTermsPerGroup];
    uint32_t zl[kMaxTermsPerGroup];
    double q[4][kMaxTermsPerGroup];
};

// Asks the L2 to fetch [p, p + bytes) (p 16-byte aligned, bytes a multiple of 16); nothing is
// written to the SM and nothing waits for it.
__device__ __forceinline__ void prefetch_l2_bulk(const void *p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(bytes)
                 : "memory");
}

template <typename R, bool CPLX>
__global__ void __launch_bounds__(kRedThreads) expect_wht_kernel(const typename Cx<R>::T *__restrict__ a, int n,
                                                                 const WhtTerms *__restrict__ wt,
                                                                 double *__restrict__ part)
{
    using T = typename Cx<R>::T;
    constexpr int VL = sizeof(T) == 8 ? 1 : 0;  // complex64: two amplitudes per 16-byte load
    constexpr int NV = 32 >> VL;                // vector loads per lane per tile
    extern __shared__ __align__(16) unsigned char dyn[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    R *wr = reinterpret_cast<R *>(dyn) + (warp << kWhtTileLog) * (CPLX ? 2 : 1);
    R *wi = wr + (1 << kWhtTileLog);
    __shared__ uint64_t zh[kMaxTermsPerGroup];
    __shared__ uint32_t zl[kMaxTermsPerGroup];
    __shared__ R q[4][kMaxTermsPerGroup];
    const int nt = wt->nterms;
    for (int j = threadIdx.x; j < nt; j += blockDim.x) {
        zh[j] = wt->zh[j];
        zl[j] = wt->zl[j];
#pragma unroll
        for (int k = 0; k < 4; ++k) q[k][j] = (R)wt->q[k][j];
    }
    __syncthreads();
    const uint64_t xm = wt->xm, xmh = xm >> kWhtTileLog;
    const uint32_t xml = uint32_t(xm) & ((1u << kWhtTileLog) - 1);
    const bool pair = wt->pair != 0;
    const int p = pair ? 63 - __clzll((long long)xmh) : 0;
    const uint64_t ntiles = 1ull << (n - kWhtTileLog - (pair ? 1 : 0));
    const uint64_t nwarps = uint64_t(gridDim.x) * (blockDim.x >> 5);
    double accr = 0.0, acci = 0.0;
    R fr = 0, fi = 0;
    int cnt = 0;
    for (uint64_t tile = uint64_t(blockIdx.x) * (blockDim.x >> 5) + warp; tile < ntiles; tile += nwarps) {
        const uint64_t H = pair ? ((tile >> p) << (p + 1)) | (tile & ((1ull << p) - 1)) : tile;
        const T *at = a + (H << kWhtTileLog);
        const T *ap = a + ((H ^ xmh) << kWhtTileLog);
        // the warp's next tile moves into L2 while this one is transformed (paired tiles already
        // keep two tiles of loads in flight and ran slower with it: 1.34 -> 1.69 ms at 30 qubits)
        if (!pair && lane == 0 && tile + nwarps < ntiles)
            prefetch_l2_bulk(a + ((tile + nwarps) << kWhtTileLog), uint32_t(sizeof(T)) << kWhtTileLog);
        // element j of the lane sits at L = (j & VL) | lane << VL | (j >> VL) << (5 + VL)
        R vr[32], vi[32];
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const uint32_t L0 = (uint32_t(lane) << VL) | (uint32_t(k) << (5 + VL));
            if constexpr (VL != 0) {
                const float4 x = *reinterpret_cast<const float4 *>(at + L0);
                if constexpr (CPLX) {
                    const uint32_t Lp = (L0 ^ xml) & ~1u;
                    float4 y = *reinterpret_cast<const float4 *>(ap + Lp);
                    if (xml & 1u) y = make_float4(y.z, y.w, y.x, y.y);
                    vr[2 * k] = (R)(y.x * x.x + y.y * x.y);
                    vi[2 * k] = (R)(y.x * x.y - y.y * x.x);
                    vr[2 * k + 1] = (R)(y.z * x.z + y.w * x.w);
                    vi[2 * k + 1] = (R)(y.z * x.w - y.w * x.z);
                } else {
                    vr[2 * k] = (R)(x.x * x.x + x.y * x.y);
                    vr[2 * k + 1] = (R)(x.z * x.z + x.w * x.w);
                }
            } else {
                const T x = at[L0];
                if (CPLX) {
                    const T y = ap[L0 ^ xml];
                    vr[k] = (R)(y.x * x.x + y.y * x.y);
                    vi[k] = (R)(y.x * x.y - y.y * x.x);
                } else {
                    vr[k] = (R)(x.x * x.x + x.y * x.y);
                }
            }
        }
        // butterflies over the five register bits ...
#pragma unroll
        for (int s = 0; s < 5; ++s)
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (!(j >> s & 1)) {
                    const int k = j | (1 << s);
                    const R r0 = vr[j], r1 = vr[k];
                    vr[j] = r0 + r1;
                    vr[k] = r0 - r1;
                    if (CPLX) {
                        const R i0 = vi[j], i1 = vi[k];
                        vi[j] = i0 + i1;
                        vi[k] = i0 - i1;
                    }
                }
        // ... and over the five lane bits (the lane with the bit set keeps the difference)
#pragma unroll
        for (int s = 0; s < 5; ++s) {
            const R sg = (lane >> s & 1) ? R(-1) : R(1);
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                vr[j] = fma(sg, vr[j], __shfl_xor_sync(0xffffffffu, vr[j], 1 << s));
                if (CPLX) vi[j] = fma(sg, vi[j], __shfl_xor_sync(0xffffffffu, vi[j], 1 << s));
            }
        }
        // Vhat(m) sits where v(L = m) was
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const uint32_t L0 = (uint32_t(lane) << VL) | (uint32_t(k) << (5 + VL));
            if constexpr (VL != 0) {
                *reinterpret_cast<float2 *>(wr + L0) = make_float2((float)vr[2 * k], (float)vr[2 * k + 1]);
                if (CPLX) *reinterpret_cast<float2 *>(wi + L0) = make_float2((float)vi[2 * k], (float)vi[2 * k + 1]);
            } else {
                wr[L0] = vr[k];
                if (CPLX) wi[L0] = vi[k];
            }
        }
        __syncwarp();
        for (int t = lane; t < nt; t += 32) {
            const uint32_t m = zl[t];
            const R s = (__popcll(H & zh[t]) & 1) ? R(-1) : R(1);
            const R Vr = wr[m];
            if (CPLX) {
                const R Vi = wi[m];
                fr = fma(s, fma(q[0][t], Vr, q[1][t] * Vi), fr);
                fi = fma(s, fma(q[2][t], Vi, q[3][t] * Vr), fi);
            } else {
                fr = fma(s * q[0][t], Vr, fr);
            }
        }
        __syncwarp();
        if (sizeof(R) == 4 && ++cnt == 8) {
            accr += (double)fr;
            acci += (double)fi;
            fr = fi = 0;
            cnt = 0;
        }
    }
    accr += (double)fr;
    acci += (double)fi;
    block_sum2(accr, acci);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = accr;
        part[gridDim.x + blockIdx.x] = acci;
    }
}

// Marginal probabilities: hist[m] = sum of |a_x|^2 over the x whose bits pos[0..nq) read m.
//
// The index bits fall into three parts: the low ones, which the 32 lanes (and the two amplitudes of a
// 16-byte complex64 load) cover; the selected bits above them, fixed for a warp; and the other bits
// above, which the warp runs over.  Each lane so adds into one or two sums that belong to one bin
// whatever nq is; at the end lanes of the same bin are added with shuffles, the eight warps of a CTA in
// shared memory where they share their bins, and the rest with one FP64 atomic per CTA or warp and bin
// (none where a bin belongs to one warp or CTA).  Bound by HBM (complex64) or the FP64 pipe (complex128,
// two FMAs per amplitude).  The kernels before added each amplitude into a shared-memory histogram with an
// FP64 atomic (10 qubits of 27, complex64: 4.73 ms, now 0.19) or kept every bin in registers with one
// select and add per bin and amplitude (3 qubits of 28, complex64: 0.62 ms, now 0.36).  Masks and offsets
// come from the host: small states wait for the chain of dependent instructions, not for memory.
struct ProbsPlan {
    uint64_t hs;          // selected bits above the low ones
    uint64_t chunk, rest; // other bits above: told apart by warps that share hs; run over, eight loads a step
    uint64_t off[8];      // offsets of the loads of one step
    int ns, nn, logc;     // number of selected / other bits above; log2 of the warps that share one setting of hs
    int gb;               // log2 of the settings of hs in one step (probs_bins_kernel)
    int low, nq;          // number of low bits; of selected ones
    uint32_t keep;        // selected low bits
    uint32_t mhalf;       // index bit of the selection's index bit 0 (complex64), 0 if it is not selected
    uint8_t pos[32];
    uint8_t hpos[24], hidx[24];  // selected bits above: position, and place in the bin's number
};

// the i-th (bit-wise) subset of mask
__host__ __device__ inline uint64_t deposit(uint64_t i, uint64_t mask)
{
    uint64_t r = 0;
    for (; i != 0; i >>= 1, mask &= mask - 1)
        if (i & 1) r |= mask & (~mask + 1);
    return r;
}

// Sum of squares in float-float form, eight amplitudes at a time: squares exact (two-product), sums by two-sum,
// about 48 bits.  Bins of 2^14 to 2^27 amplitudes are within 9e-15 of their exact sums (histograms of FP64
// atomics: 1.7e-14; FP32 sums of 32 amplitudes: 6e-8, and no faster).  Exact
// products need 2^-50 <= |x| (or 0), sums |x| < 2^60; amplitudes outside take FP64, which has 2 FMAs per SM and
// clock for what these instructions do at 128.
struct SquareSum {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void add(float x, float y)
    {
        const float px = __fmul_rn(x, x), py = __fmul_rn(y, y);
        const float ex = __fmaf_rn(x, x, -px), ey = __fmaf_rn(y, y, -py);
        const float s = __fadd_rn(px, py), b = __fsub_rn(s, px);
        const float e = __fadd_rn(__fsub_rn(px, __fsub_rn(s, b)), __fsub_rn(py, b));
        join(s, __fadd_rn(__fadd_rn(ex, ey), e));
    }
    // adds another sum
    __device__ __forceinline__ void join(float s, float r)
    {
        const float t = __fadd_rn(h, s), c = __fsub_rn(t, h);
        const float g = __fadd_rn(__fsub_rn(h, __fsub_rn(t, c)), __fsub_rn(s, c));
        h = t;
        l = __fadd_rn(l, __fadd_rn(r, g));
    }
    __device__ __forceinline__ void join_lane(int mask)
    {
        join(__shfl_xor_sync(0xffffffffu, h, mask), __shfl_xor_sync(0xffffffffu, l, mask));
    }
    __device__ __forceinline__ double value() const { return (double)h + (double)l; }
    __device__ __forceinline__ void flush(double &acc)
    {
        acc += value();
        h = l = 0.f;
    }
};
struct Square64 {  // the same in FP64
    double s = 0.0;
    template <typename F> __device__ __forceinline__ void add(F x, F y)
    {
        s = fma((double)x, (double)x, s);
        s = fma((double)y, (double)y, s);
    }
    __device__ __forceinline__ void join_lane(int mask) { s += __shfl_xor_sync(0xffffffffu, s, mask); }
    __device__ __forceinline__ double value() const { return s; }
};

template <typename R> struct ProbsLoad;
template <> struct ProbsLoad<float> {
    using V = float4;
    static constexpr int VL = 1;  // low bit inside a 16-byte load
    // amplitudes whose squares and sums float-float numbers hold
    template <int U> static __device__ __forceinline__ bool fits(const V (&v)[U])
    {
        uint32_t least = ~0u;
        float most = 0.f;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                least = min(least, 2u * __float_as_uint(w[k]) - 1u);  // (zeros are the largest)
                most = fmaxf(most, fabsf(w[k]));
            }
        }
        return least >= 2u * __float_as_uint(0x1p-50f) - 1u && most < 0x1p60f;
    }
};
template <> struct ProbsLoad<double> {
    using V = double2;
    static constexpr int VL = 0;
};

// lanes of one bin (selected low bits keep them apart)
template <int VL, typename A> __device__ __forceinline__ void join_lanes(A &a, uint32_t keep)
{
#pragma unroll
    for (int l = 0; l < 5; ++l)
        if (!(keep >> (l + VL) & 1u)) a.join_lane(1 << l);
}

// Eight loads a step, and at least one step, per warp and setting of the selected bits above.
template <typename R>
__global__ void __launch_bounds__(kRedThreads) probs_kernel(const typename Cx<R>::T *__restrict__ a,
                                                            const __grid_constant__ ProbsPlan p, double *__restrict__ hist)
{
    using V = typename ProbsLoad<R>::V;
    constexpr int VL = ProbsLoad<R>::VL, U = 8, H = 1 << VL, W = kRedThreads / 32;
    static_assert(W == 8, "eight threads add a bin's eight warps");
    __shared__ double sh[32 * H][W + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t units = 1ull << (p.ns + p.logc);
    const uint64_t mine = uint64_t(lane) << VL;
    const uint64_t iters = 1ull << (p.nn - p.logc - 3);
    const bool joint = p.logc >= 3;  // the CTA's warps share hs
    for (uint64_t u0 = uint64_t(blockIdx.x) * W; u0 < units; u0 += uint64_t(gridDim.x) * W) {
        const uint64_t unit = u0 + warp;
        const bool has = unit < units;
        const uint64_t sel = deposit(unit >> p.logc, p.hs);
        const auto *at = a + (sel | deposit(unit & ((1ull << p.logc) - 1), p.chunk) | mine);
        Square64 acc[H];
        if (has) {
            uint64_t x = 0;
            for (uint64_t it = 0; it < iters; ++it) {
                V v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = __ldcs(reinterpret_cast<const V *>(at + (x | p.off[u])));
                if constexpr (VL == 1) {
                    if (ProbsLoad<R>::fits(v)) {
                        SquareSum f[H];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            f[0].add(v[u].x, v[u].y);
                            f[VL].add(v[u].z, v[u].w);
                        }
                        f[0].flush(acc[0].s);
                        f[VL].flush(acc[VL].s);
                    } else {
#pragma unroll 1
                        for (int u = 0; u < U; ++u) {
                            V t = v[0];
#pragma unroll
                            for (int k = 1; k < U; ++k) t = u == k ? v[k] : t;
                            acc[0].add(t.x, t.y);
                            acc[VL].add(t.z, t.w);
                        }
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < U; ++u) acc[0].add(v[u].x, v[u].y);
                }
                x = ((x | ~p.rest) + 1) & p.rest;  // the next subset of rest
            }
        }
        if (VL == 1 && !(p.keep & 1u)) {
            acc[0].s += acc[VL].s;
            acc[VL].s = acc[0].s;
        }
#pragma unroll
        for (int k = 0; k < H; ++k) join_lanes<VL>(acc[k], p.keep);
        auto store = [&](uint32_t lk, double v) {  // bin of low index lk
            const uint64_t y = sel | lk;
            uint32_t m = 0;
            for (int j = 0; j < p.nq; ++j) m |= uint32_t((y >> p.pos[j]) & 1) << j;
            if (p.logc == 0 || p.logc == 3) hist[m] = v;
            else atomicAdd(&hist[m], v);
        };
        // (of the lanes and halves of a bin, the one whose other low bits are 0 stores it)
        if (joint) {
#pragma unroll
            for (int k = 0; k < H; ++k) sh[(lane << VL) | k][warp] = acc[k].s;
            __syncthreads();
            // eight threads a sum; (32 H) of them, 32 at a time
            for (uint32_t lk = threadIdx.x >> 3; lk < 32u * H; lk += kRedThreads / 8) {
                double v = sh[lk][threadIdx.x & 7];
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                v += __shfl_xor_sync(0xffffffffu, v, 4);
                if ((threadIdx.x & 7) == 0 && (lk & ~p.keep) == 0) store(lk, v);
            }
            __syncthreads();
        } else if (has) {
#pragma unroll
            for (int k = 0; k < H; ++k)
                if (((uint32_t(mine) | k) & ~p.keep) == 0) store(uint32_t(mine) | k, acc[k].s);
        }
    }
}

// Nearly all bits above the low ones selected (NN = 0, 1 or 2 are not), and states smaller than a few loads per
// lane: a step's eight loads belong to 2^(3-NN) settings of the selected bits.  (One setting at a time left
// one to four loads in flight and spent a loop over the bits on each: the upper 20 of 27 qubits 1.91 -> 0.44 ms
// in complex64, of 26 qubits in complex128 1.40 -> 0.67; atomics into device memory took 1.41 and 0.70.)  With
// fewer settings than resident warps, each has a warp of its own.
template <typename R, int NN>
__global__ void __launch_bounds__(kRedThreads) probs_bins_kernel(const typename Cx<R>::T *__restrict__ a,
                                                                 const __grid_constant__ ProbsPlan p, double *__restrict__ hist)
{
    using V = typename ProbsLoad<R>::V;
    constexpr int VL = ProbsLoad<R>::VL, U = 8, H = 1 << VL, W = kRedThreads / 32, G = U >> NN;
    const int lane = threadIdx.x & 31;
    const int gb = p.gb;
    const uint64_t units = 1ull << (p.ns - gb);
    const uint64_t mine = uint64_t(lane) << VL;
    const bool live = (mine >> p.low) == 0;  // states smaller than one load per lane
    const bool writer = live && (uint32_t(mine) & ~(p.keep | (H - 1u))) == 0;
    uint32_t ml = 0, mg[G];
    for (int j = 0; j < p.nq; ++j)
        if (p.pos[j] < p.low) ml |= uint32_t((mine >> p.pos[j]) & 1) << j;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        mg[g] = 0;
#pragma unroll
        for (int j = 0; j < 3 - NN; ++j)
            if (j < gb && (g >> j & 1)) mg[g] |= 1u << p.hidx[j];
    }
    for (uint64_t unit = uint64_t(blockIdx.x) * W + (threadIdx.x >> 5); unit < units; unit += uint64_t(gridDim.x) * W) {
        uint64_t x = mine;
        uint32_t m = ml;
        for (int j = gb; j < p.ns; ++j) {
            const uint64_t bit = (unit >> (j - gb)) & 1;
            x |= bit << p.hpos[j];
            m |= uint32_t(bit) << p.hidx[j];
        }
        V v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            v[u] = V{};
            if (live && (u >> NN) < (1 << gb)) v[u] = __ldcs(reinterpret_cast<const V *>(a + (x | p.off[u])));
        }
        auto bins = [&](auto zero) {
            using A = decltype(zero);
            A s[G][H];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                if (g && g >= (1 << gb)) continue;
#pragma unroll
                for (int i = 0; i < (1 << NN); ++i) {
                    const V t = v[(g << NN) | i];
                    s[g][0].add(t.x, t.y);
                    if constexpr (VL == 1) {
                        if (p.mhalf) s[g][VL].add(t.z, t.w);
                        else s[g][0].add(t.z, t.w);
                    }
                }
            }
            // lane bits outside, bins inside: each exchange of one bin hides behind those of the others
#pragma unroll
            for (int l = 0; l < 5; ++l) {
                if (p.keep >> (l + VL) & 1u) continue;
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    if (g && g >= (1 << gb)) continue;
                    s[g][0].join_lane(1 << l);
                    if (VL == 1 && p.mhalf) s[g][VL].join_lane(1 << l);
                }
            }
            if (!writer) return;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                if (g && g >= (1 << gb)) continue;
                hist[m | mg[g]] = s[g][0].value();
                if (VL == 1 && p.mhalf) hist[m | mg[g] | p.mhalf] = s[g][VL].value();
            }
        };
        if constexpr (VL == 1) {
            if (__all_sync(0xffffffffu, ProbsLoad<R>::fits(v))) bins(SquareSum{});
            else bins(Square64{});
        } else {
            bins(Square64{});
        }
    }
}

ProbsPlan probs_plan(int n, qs_dtype dt, const int *pos, int nq)
{
    ProbsPlan p{};
    p.low = std::min(n, dt == QS_C64 ? 6 : 5);
    p.nq = nq;
    uint64_t sel = 0;
    for (int j = 0; j < nq; ++j) {
        p.pos[j] = uint8_t(pos[j]);
        sel |= 1ull << pos[j];
        if (dt == QS_C64 && pos[j] == 0) p.mhalf = 1u << j;
    }
    const uint64_t lowm = (1ull << p.low) - 1, above = ((1ull << n) - 1) & ~lowm;
    p.keep = uint32_t(sel & lowm);
    p.hs = sel & above;
    for (int q = 0; q < n; ++q)
        if (p.hs >> q & 1) {
            p.hpos[p.ns] = uint8_t(q);
            p.hidx[p.ns++] = uint8_t(std::find(pos, pos + nq, q) - pos);
        }
    const uint64_t other = above & ~sel;
    p.nn = __builtin_popcountll(other);
    if (p.nn < 3) {  // loads of a step: the other bits, then the lowest selected ones
        p.gb = std::max(0, std::min(3 - p.nn, p.ns - 11));  // (2^11 warps are resident at once)
        for (uint32_t u = 0; u < 8; ++u)
            p.off[u] = deposit(u & ((1u << p.nn) - 1), other) | deposit((u >> p.nn) & ((1u << p.gb) - 1), p.hs);
        return p;
    }
    // 2^13 warps fill the GPU (6.7 CTAs of eight per SM).  One warp or one CTA per bin stores without a clear
    // and atomics (3 and 10 qubits of 27: 0.21 -> 0.19 ms, with the masks from the host): two or four warps per
    // bin are rounded to one of them, and small states use one CTA while it has 32 loads a warp at most (12
    // qubits, 29 -> 22 us a call; at 14 qubits a launch less for 2 us more of it).
    p.logc = std::max(0, std::min(13 - p.ns, p.nn - 3));
    if (p.logc > 3 && p.nn <= 8) p.logc = 3;
    if (p.logc == 1 || p.logc == 2) p.logc = p.nn >= 6 ? 3 : 0;
    p.chunk = deposit(((1ull << p.logc) - 1) << (p.nn - p.logc), other);
    const uint64_t run = other & ~p.chunk, inner = deposit(7, run);
    p.rest = run & ~inner;
    for (uint32_t u = 0; u < 8; ++u) p.off[u] = deposit(u, inner);
    return p;
}

int g_sms = 0;
int reduce_blocks(uint64_t N)
{
    if (!g_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_sms <= 0) g_sms = 1;
    }
    uint64_t b = uint64_t(g_sms) * 8;
    if (b > kRedBlocksMax) b = kRedBlocksMax;
    const uint64_t need = (N + kRedThreads - 1) / kRedThreads;
    if (b > need) b = need;
    return b < 1 ? 1 : (int)b;
}

int cuda_fail(const char *what, char *err, size_t errlen)
{
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) return QS_OK;
    snprintf(err, errlen, "%s: %s", what, cudaGetErrorString(e));
    return QS_ECUDA;
}

}  // namespace

size_t reduce_scratch_bytes()
{
    // partials (2 x blocks) + 2 results + one term group + its Walsh-Hadamard term table + one tile's groups
    return sizeof(double) * (2 * kRedBlocksMax + 8) + sizeof(TermGroup) + 256 + sizeof(WhtTerms) + 256 +
           pauli_tile_bytes() + 256;
}

int launch_norm2(const LaunchCtx &c, double *d_scratch, double *h_out, char *err, size_t errlen)
{
    const uint64_t N = 1ull << c.n;
    const int blocks = reduce_blocks(N);
    cudaStream_t st = (cudaStream_t)c.stream;
    double *part = d_scratch, *res = d_scratch + 2 * kRedBlocksMax;
    if (c.dt == QS_C64)
        norm2_kernel<float><<<blocks, kRedThreads, 0, st>>>((const float2 *)c.amp, N, part);
    else
        norm2_kernel<double><<<blocks, kRedThreads, 0, st>>>((const double2 *)c.amp, N, part);
    finish_kernel<<<1, kRedThreads, 0, st>>>(part, blocks, 0, res, false);
    int rc = cuda_fail("norm2 launch", err, errlen);
    if (rc) return rc;
    double r[2];
    if (cudaMemcpyAsync(r, res, sizeof(r), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return cuda_fail("norm2 readback", err, errlen);
    *h_out = r[0];
    return QS_OK;
}

namespace {

int enqueue_probs(const LaunchCtx &c, const int *phys_q, int nq, double *hist, char *err, size_t errlen)
{
    cudaStream_t st = (cudaStream_t)c.stream;
    const ProbsPlan p = probs_plan(c.n, c.dt, phys_q, nq);
    reduce_blocks(1);  // reads the SM count once
    auto blocks = [](uint64_t warps) { return int(std::min<uint64_t>((warps + kRedThreads / 32 - 1) / (kRedThreads / 32), uint64_t(g_sms) * 8)); };
    auto launch = [&](auto R, const auto *a) {
        using T = decltype(R);
        if (p.nn >= 3) return probs_kernel<T><<<blocks(1ull << (p.ns + p.logc)), kRedThreads, 0, st>>>(a, p, hist);
        const int b = blocks(1ull << (p.ns - p.gb));
        if (p.nn == 0) probs_bins_kernel<T, 0><<<b, kRedThreads, 0, st>>>(a, p, hist);
        else if (p.nn == 1) probs_bins_kernel<T, 1><<<b, kRedThreads, 0, st>>>(a, p, hist);
        else probs_bins_kernel<T, 2><<<b, kRedThreads, 0, st>>>(a, p, hist);
    };
    // bins that several CTAs add to start at 0
    if (p.nn >= 3 && p.logc > 3 && cudaMemsetAsync(hist, 0, (size_t(1) << nq) * sizeof(double), st) != cudaSuccess)
        return cuda_fail("probs memset", err, errlen);
    if (c.dt == QS_C64) launch(float{}, (const float2 *)c.amp);
    else launch(double{}, (const double2 *)c.amp);
    return cuda_fail("probs launch", err, errlen);
}

}  // namespace

int launch_probs(const LaunchCtx &c, const int *phys_q, int nq, double *d_scratch,
                 size_t scratch_bytes, double *h_out, char *err, size_t errlen)
{
    const size_t M = size_t(1) << nq;
    if (M * sizeof(double) > scratch_bytes) {
        snprintf(err, errlen, "probs: scratch too small");
        return QS_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)c.stream;
    int rc = enqueue_probs(c, phys_q, nq, d_scratch, err, errlen);
    if (rc) return rc;
    if (cudaMemcpyAsync(h_out, d_scratch, M * sizeof(double), cudaMemcpyDeviceToHost, st) !=
            cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return cuda_fail("probs readback", err, errlen);
    return QS_OK;
}

namespace {

template <typename R, bool CPLX>
int launch_wht_t(const typename Cx<R>::T *a, int n, const WhtTerms *wt, uint64_t ntiles, double *part,
                 cudaStream_t st)
{
    const size_t dsm = (size_t(kRedThreads / 32) << kWhtTileLog) * sizeof(R) * (CPLX ? 2 : 1);
    static int attr_dev = -1, per_sm = 1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (attr_dev != dev) {
        cudaFuncSetAttribute(expect_wht_kernel<R, CPLX>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(dsm));
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, expect_wht_kernel<R, CPLX>, kRedThreads, dsm) !=
                cudaSuccess ||
            per_sm < 1)
            per_sm = 1;
        attr_dev = dev;
    }
    reduce_blocks(1);  // reads the SM count once
    uint64_t nb = uint64_t(g_sms) * uint64_t(per_sm);
    const uint64_t need = std::max<uint64_t>(1, ntiles / (kRedThreads / 32));
    nb = std::min<uint64_t>(std::min<uint64_t>(nb, need), kRedBlocksMax);
    expect_wht_kernel<R, CPLX><<<int(nb), kRedThreads, dsm, st>>>(a, n, wt, part);
    return int(nb);
}

template <typename R>
int launch_wht(const typename Cx<R>::T *a, int n, const WhtTerms *wt, bool cplx, uint64_t ntiles, double *part,
               cudaStream_t st)
{
    return cplx ? launch_wht_t<R, true>(a, n, wt, ntiles, part, st)
                : launch_wht_t<R, false>(a, n, wt, ntiles, part, st);
}

}  // namespace

int launch_expect(const LaunchCtx &c, const uint64_t *xm, const uint64_t *zm, const double *coeff,
                  size_t nterms, double *d_scratch, size_t scratch_bytes, double *h_out, char *err,
                  size_t errlen)
{
    (void)scratch_bytes;
    const uint64_t N = 1ull << c.n;
    cudaStream_t st = (cudaStream_t)c.stream;
    double *part = d_scratch, *res = d_scratch + 2 * kRedBlocksMax;
    TermGroup *dgrp = reinterpret_cast<TermGroup *>(d_scratch + 2 * kRedBlocksMax + 8);
    const int blocks = reduce_blocks(N);
    auto aligned = [](void *p) { return (reinterpret_cast<uintptr_t>(p) + 255) & ~uintptr_t(255); };
    WhtTerms *dpt = reinterpret_cast<WhtTerms *>(aligned(dgrp + 1));
    void *dtile = reinterpret_cast<void *>(aligned(dpt + 1));
    // Terms by X mask, in order of first appearance, at most kMaxTermsPerGroup each.
    std::vector<PauliXGroup> groups;
    {
        std::unordered_map<uint64_t, int> open;  // X mask -> the group that still takes terms
        for (size_t i = 0; i < nterms; ++i) {
            auto it = open.find(xm[i]);
            if (it == open.end() || groups[it->second].zm.size() == size_t(kMaxTermsPerGroup)) {
                open[xm[i]] = int(groups.size());
                groups.push_back(PauliXGroup{xm[i], {}, {}});
                it = open.find(xm[i]);
            }
            groups[it->second].zm.push_back(zm[i]);
            groups[it->second].c.push_back(coeff[i]);
        }
    }
    // One host image per launch, 32 launches between waits (at most 360 KiB).
    auto wait = [st] { cudaStreamSynchronize(st); };
    StagingRing<decltype(wait)> staging(std::max({pauli_tile_bytes(), sizeof(TermGroup), sizeof(WhtTerms)}), 32, wait);
    if (groups.empty()) {
        h_out[0] = h_out[1] = 0.0;
        return QS_OK;
    }
    bool first = true;  // the first launch's sums are stored, the others' added
    // X masks with few terms share reads of the state (k_pauli.cu).  A term costs a tile pass about 2
    // operations per pair of amplitudes, so up to 8 terms per mask are well below a pass of their own.
    // Whether a tile pass is taken depends on what it replaces.  One mask alone: from 18 qubits on it is read
    // once and not twice (complex64, 27 qubits, 1 term: 1054 -> 403 us; below, 40 us either way).  Masks that
    // all have Walsh-Hadamard tiles of their own (4 terms, 16 qubits): in complex64 those run at HBM rate (27
    // qubits 227 us, against 451 for a tile pass and about 130 for each further mask), so from four masks on;
    // in complex128 the transform is FP64 work and the tile pass is ahead (26 qubits, 8 terms: 1488 -> 1230
    // us).  Small complex128 states: up to 16 CTAs, each bound by FP64 issue, 2.5 us a term against 6 us for
    // a launch (14 qubits, 8 terms: 57 us, 41 on its own).
    auto worthwhile = [&](const std::vector<int> &take) {
        size_t nt = 0, light = 0;
        for (int g : take) {
            nt += groups[g].zm.size();
            light += groups[g].zm.size() < 4 || c.n < 16;
        }
        const bool c64 = c.dt == QS_C64;
        if (take.size() == 1 && light) return c.n >= 18;
        if (!c64) return c.n >= 17 || 2 * nt <= 5 * take.size();
        return light > 0 || take.size() >= 4;
    };
    std::vector<int> tiles;
    std::vector<char> done(groups.size(), 0);
    for (size_t g = 0; g < groups.size(); ++g)
        if (groups[g].xm != 0 && groups[g].zm.size() <= 8) tiles.push_back(int(g));
    while (!tiles.empty()) {
        std::vector<int> take;
        void *const htile = staging.next();
        const int b = pauli_tile_plan(c, groups, tiles, take, htile);
        if (b == 0) break;  // more X bits than a tile holds, all of them: passes of their own below
        if (!worthwhile(take)) continue;
        for (int g : take) done[g] = 1;
        if (cudaMemcpyAsync(dtile, htile, pauli_tile_bytes(), cudaMemcpyHostToDevice, st) != cudaSuccess)
            return cuda_fail("expect upload", err, errlen);
        const int nblk = launch_pauli_tile(c, dtile, htile, b, part, kRedBlocksMax);
        finish_kernel<<<1, kRedThreads, 0, st>>>(part, nblk, nblk, res, !first);
        first = false;
        int rc = cuda_fail("expect launch", err, errlen);
        if (rc) return rc;
    }
    for (size_t gi = 0; gi < groups.size(); ++gi) {
        if (done[gi]) continue;
        const PauliXGroup &G = groups[gi];
        TermGroup &hg = *new (staging.next()) TermGroup;
        hg.xm = G.xm;
        hg.nterms = int(G.zm.size());
        for (int j = 0; j < hg.nterms; ++j) {
            const int ny = __builtin_popcountll(G.xm & G.zm[j]) & 3;
            static const double pr[4] = {1, 0, -1, 0}, pi[4] = {0, 1, 0, -1};
            hg.zm[j] = G.zm[j];
            hg.cre[j] = G.c[j] * pr[ny];
            hg.cim[j] = G.c[j] * pi[ny];
        }
        int nblk = blocks;
        if (hg.nterms >= 4 && c.n >= 16) {
            // Walsh-Hadamard tiles; coefficients folded on the host in FP64
            WhtTerms &w = *new (staging.next()) WhtTerms;
            w.xm = hg.xm;
            w.nterms = hg.nterms;
            w.pair = (hg.xm >> kWhtTileLog) != 0;
            for (int t = 0; t < hg.nterms; ++t) {
                w.zh[t] = hg.zm[t] >> kWhtTileLog;
                w.zl[t] = uint32_t(hg.zm[t]) & ((1u << kWhtTileLog) - 1);
                const double cr = hg.cre[t], ci = hg.cim[t];
                // partner tile: coefficient times (-1)^{popc(xm & z)}; none without pairing
                const double sg = (__builtin_popcountll(hg.xm & hg.zm[t]) & 1) ? -1.0 : 1.0;
                const double pr = w.pair ? sg * cr : 0.0, pi = w.pair ? sg * ci : 0.0;
                w.q[0][t] = cr + pr;
                w.q[1][t] = pi - ci;
                w.q[2][t] = cr - pr;
                w.q[3][t] = ci + pi;
            }
            if (cudaMemcpyAsync(dpt, &w, sizeof w, cudaMemcpyHostToDevice, st) != cudaSuccess)
                return cuda_fail("expect upload", err, errlen);
            const WhtTerms *dw = dpt;
            const uint64_t ntiles = 1ull << (c.n - kWhtTileLog - w.pair);
            const bool cplx = hg.xm != 0;
            if (c.dt == QS_C64)
                nblk = launch_wht<float>((const float2 *)c.amp, c.n, dw, cplx, ntiles, part, st);
            else
                nblk = launch_wht<double>((const double2 *)c.amp, c.n, dw, cplx, ntiles, part, st);
        } else {
            if (cudaMemcpyAsync(dgrp, &hg, sizeof(TermGroup), cudaMemcpyHostToDevice, st) != cudaSuccess)
                return cuda_fail("expect upload", err, errlen);
            if (c.dt == QS_C64)
                expect_kernel<float><<<blocks, kRedThreads, 0, st>>>((const float2 *)c.amp, N, dgrp, part);
            else
                expect_kernel<double><<<blocks, kRedThreads, 0, st>>>((const double2 *)c.amp, N, dgrp,
                                                                      part);
        }
        finish_kernel<<<1, kRedThreads, 0, st>>>(part, nblk, nblk, res, !first);
        first = false;
        int rc = cuda_fail("expect launch", err, errlen);
        if (rc) return rc;
    }
    if (cudaMemcpyAsync(h_out, res, 2 * sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return cuda_fail("expect readback", err, errlen);
    staging.idle();
    return QS_OK;
}

// ------------------------------------------------------------------ allocation-free probs
// Fixed scratch for qs_probs_noalloc: one histogram of at most 2^kStaticProbsMaxQubits doubles
// (128 KiB).  It is a file-scope device array, so every GPU that loads the library holds it
// until the process exits.  Host code must not pass `g_static_probs_hist` itself to a kernel:
// on the host that name is only a stand-in symbol, not a device address.  Its device address
// is looked up once per device with cudaGetSymbolAddress (static_probs_scratch below).
namespace {

__device__ __align__(256) double g_static_probs_hist[1 << kStaticProbsMaxQubits];

constexpr int kMaxDevices = 64;
double *g_static_probs_ptr[kMaxDevices] = {nullptr};
std::mutex g_static_probs_mu;

// Device address of the fixed histogram on the current device (set up on first use).
int static_probs_scratch(double **out, char *err, size_t errlen)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        snprintf(err, errlen, "probs_noalloc: no usable current device (%s)",
                 e != cudaSuccess ? cudaGetErrorString(e) : "device index out of range");
        return QS_ECUDA;
    }
    std::lock_guard<std::mutex> lock(g_static_probs_mu);
    if (!g_static_probs_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_probs_hist);
        if (e != cudaSuccess || !p) {
            snprintf(err, errlen, "probs_noalloc: cudaGetSymbolAddress failed: %s",
                     cudaGetErrorString(e));
            cudaGetLastError();
            return QS_ECUDA;
        }
        g_static_probs_ptr[dev] = static_cast<double *>(p);
    }
    *out = g_static_probs_ptr[dev];
    return QS_OK;
}

}  // namespace

int launch_probs_static(const LaunchCtx &c, const int *phys_q, int nq, double *h_out, char *err,
                        size_t errlen)
{
    if (nq < 0 || nq > kStaticProbsMaxQubits) {
        snprintf(err, errlen, "probs_noalloc: nq = %d exceeds the fixed scratch of 2^%d bins", nq,
                 kStaticProbsMaxQubits);
        return QS_EINVAL;
    }
    double *hist = nullptr;
    int rc = static_probs_scratch(&hist, err, errlen);
    if (rc) return rc;
    const size_t M = size_t(1) << nq;
    cudaStream_t st = (cudaStream_t)c.stream;
    rc = enqueue_probs(c, phys_q, nq, hist, err, errlen);
    if (rc) return rc;
    if (cudaMemcpyAsync(h_out, hist, M * sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return cuda_fail("probs_noalloc readback", err, errlen);
    return QS_OK;
}

__global__ void set_one_kernel(void *amp, uint64_t x, int is64)
{
    if (is64) reinterpret_cast<float2 *>(amp)[x] = make_float2(1.f, 0.f);
    else reinterpret_cast<double2 *>(amp)[x] = make_double2(1.0, 0.0);
}

int launch_set_basis(const LaunchCtx &c, uint64_t x, char *err, size_t errlen)
{
    cudaStream_t st = (cudaStream_t)c.stream;
    const size_t bytes = (size_t(1) << c.n) * (c.dt == QS_C64 ? 8 : 16);
    if (cudaMemsetAsync(c.amp, 0, bytes, st) != cudaSuccess)
        return cuda_fail("set_basis memset", err, errlen);
    set_one_kernel<<<1, 1, 0, st>>>(c.amp, x, c.dt == QS_C64 ? 1 : 0);
    return cuda_fail("set_basis launch", err, errlen);
}

}  // namespace qs
