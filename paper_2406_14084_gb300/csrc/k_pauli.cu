// k_pauli.cu -- expectation of Pauli strings whose X masks are many and Z masks per X mask few (chain
// Hamiltonians XX + YY + ZZ, transverse fields), several X masks per read of the state.
//
// sum_x conj(a[x ^ xm]) a[x] C_t (-1)^{popc(x & z_t)}, C_t = c_t i^{#Y}, joins x and x ^ xm: with x0 the
// one whose highest xm bit is clear and v = conj(a[x0 ^ xm]) a[x0], the two contribute
//   #Y even:  2 Re(C_t) (-1)^{popc(x0 & z_t)} Re v        #Y odd:  -2 Im(C_t) (-1)^{popc(x0 & z_t)} Im v.
// A CTA loads a tile of 2^b amplitudes (the low bits plus up to b - lo gathered ones, as the slab
// passes do) into shared memory and evaluates every X mask that lies within the tile's bits, so the
// state is read once per tile choice and not once or twice per X mask.  Per mask a thread forms v for its
// pairs in registers; a term then costs one sign and one addition per pair: pair j = thread + 256 k, and
// the parity of j & z splits into a part of the thread and a part of k that the whole grid shares.
// Bound by shared-memory reads (one amplitude pair per mask) and FP32 / FP64 issue, no longer by HBM:
// a Heisenberg chain of 26 qubits (25 bond masks, 75 terms, and the field) took 14.6 ms with one pass
// per mask and takes 1.33 ms (24 qubits in complex128: 2.03).  Three CTAs fit an SM (64 KiB of tile each,
// terms and offsets behind it as many as there are: two CTAs 1.76 ms, three 1.37); terms whose sign is the
// same for all pairs of a thread, most of a chain's, share one sum (1.37 -> 1.27 ms, complex128 2.99 -> 2.03).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include "dev_common.cuh"

namespace qs {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxGroups = 64, kMaxTerms = 256;  // per launch

struct PauliTerm {
    double c;        // factor of Re v or Im v
    uint64_t zout;   // Z bits outside the tile (physical)
    uint32_t zthr;   // Z bits of the thread's part of the pair index
    uint32_t kpat;   // bit k: sign of the k-th pair of every thread
};
struct PauliGroup {
    uint32_t xm;     // tile-local
    uint8_t piv;     // its highest bit
    uint8_t flush;   // the FP32 sums go to FP64 after this mask
    uint16_t t0, tmid, t1;  // terms [t0, tmid) use Re v, [tmid, t1) Im v
};
struct PauliTile {
    int lo, nhi, ngroups, nterms;
    uint8_t hipos[16];
    PauliGroup g[kMaxGroups];
    PauliTerm t[kMaxTerms];
};

template <typename R> constexpr int tile_bits() { return sizeof(R) == 4 ? 13 : 12; }  // 64 KiB

__device__ __forceinline__ float with_sign(float v, uint32_t s) { return __uint_as_float(__float_as_uint(v) ^ s); }
__device__ __forceinline__ double with_sign(double v, uint32_t s)
{
    return __longlong_as_double(__double_as_longlong(v) ^ (long long)((unsigned long long)s << 32));
}

template <typename R>
__global__ void __launch_bounds__(kThreads, 3) pauli_tile_kernel(const typename Cx<R>::T *__restrict__ a, int b,
                                                              const PauliTile *__restrict__ d, uint64_t ntiles,
                                                              double *__restrict__ part)
{
    using C = typename Cx<R>::T;
    constexpr int K = 1 << (tile_bits<R>() - 9);  // pairs per thread of a full tile
    extern __shared__ __align__(16) unsigned char dyn[];
    C *const sm = reinterpret_cast<C *>(dyn);
    __shared__ double red[kThreads / 32];
    const uint32_t tid = threadIdx.x;
    const int lo = d->lo, nhi = d->nhi, ng = d->ngroups, nt = d->nterms;
    // [tile][segment offsets][terms][groups]
    uint64_t *const seg = reinterpret_cast<uint64_t *>(sm + (size_t(1) << b));
    PauliTerm *const T = reinterpret_cast<PauliTerm *>(seg + (size_t(1) << nhi));
    PauliGroup *const G = reinterpret_cast<PauliGroup *>(T + nt);
    for (uint32_t s = tid; s < (1u << nhi); s += kThreads) {
        uint64_t o = 0;
        for (int m = 0; m < nhi; ++m)
            if (s >> m & 1) o |= 1ull << d->hipos[m];
        seg[s] = o;
    }
    for (int i = int(tid); i < ng; i += kThreads) G[i] = d->g[i];
    for (int i = int(tid); i < nt; i += kThreads) T[i] = d->t[i];
    __syncthreads();
    const uint32_t size = 1u << b, pairs = size >> 1;
    double acc = 0.0;
    for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        uint64_t base = tile << lo;
        for (int m = 0; m < nhi; ++m) {
            const uint64_t lowm = (1ull << d->hipos[m]) - 1;
            base = ((base & ~lowm) << 1) | (base & lowm);
        }
        if (sizeof(C) == 8 && lo > 0) {  // two amplitudes per 16-byte load
#pragma unroll 8
            for (uint32_t i = 2 * tid; i < size; i += 2 * kThreads)
                *reinterpret_cast<float4 *>(sm + i) =
                    __ldcs(reinterpret_cast<const float4 *>(a + base + seg[i >> lo] + (i & ((1u << lo) - 1))));
        } else {
#pragma unroll 8
            for (uint32_t i = tid; i < size; i += kThreads) sm[i] = a[base + seg[i >> lo] + (i & ((1u << lo) - 1))];
        }
        __syncthreads();
        R facc = 0;
        for (int g = 0; g < ng; ++g) {
            const PauliGroup q = G[g];
            const uint32_t low = (1u << q.piv) - 1;
            R v[K];
            auto terms = [&](int from, int to) {
                // (terms without a sign inside a thread share the plain sum)
                R p0 = 0, p1 = 0;
#pragma unroll
                for (int k = 0; k < K; k += 2) {
                    p0 += v[k];
                    p1 += v[k + 1];
                }
                for (int t = from; t < to; ++t) {
                    const uint32_t odd = (__popcll(base & T[t].zout) + __popc(tid & T[t].zthr)) & 1u;
                    const uint32_t kp = T[t].kpat;
                    R s = p0 + p1;
                    if (kp) {
                        R s0 = 0, s1 = 0;
#pragma unroll
                        for (int k = 0; k < K; k += 2) {
                            s0 += with_sign(v[k], (kp << (31 - k)) & 0x80000000u);
                            s1 += with_sign(v[k + 1], (kp << (30 - k)) & 0x80000000u);
                        }
                        s = s0 + s1;
                    }
                    const R c = (R)T[t].c;
                    facc = fma(odd ? -c : c, s, facc);
                }
            };
            auto values = [&](bool imag) {
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const uint32_t j = tid + uint32_t(k) * kThreads;
                    v[k] = R(0);
                    if (j < pairs) {
                        const uint32_t i0 = ((j & ~low) << 1) | (j & low);
                        const C x = sm[i0], y = sm[i0 ^ q.xm];
                        v[k] = imag ? y.x * x.y - y.y * x.x : y.x * x.x + y.y * x.y;
                    }
                }
            };
            if (q.t0 < q.tmid) {
                values(false);
                terms(q.t0, q.tmid);
            }
            if (q.tmid < q.t1) {
                values(true);
                terms(q.tmid, q.t1);
            }
            if (sizeof(R) == 4 && q.flush) {
                acc += (double)facc;
                facc = 0;
            }
        }
        acc += (double)facc;
        __syncthreads();  // the tile is overwritten by the next load
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((tid & 31) == 0) red[tid >> 5] = acc;
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) s += red[w];
        part[blockIdx.x] = s;
        part[gridDim.x + blockIdx.x] = 0.0;  // the sum is real
    }
}

template <typename R>
int launch_t(const LaunchCtx &c, const PauliTile *d, const PauliTile &h, int b, double *part, int max_blocks)
{
    using C = typename Cx<R>::T;
    const size_t smem = (sizeof(C) << b) + (sizeof(uint64_t) << h.nhi) + h.nterms * sizeof(PauliTerm) +
                        h.ngroups * sizeof(PauliGroup);
    static int attr_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (attr_dev != dev) {
        cudaFuncSetAttribute(pauli_tile_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             int((64 << 10) + (8 << 9) + kMaxTerms * sizeof(PauliTerm) + kMaxGroups * sizeof(PauliGroup)));
        attr_dev = dev;
    }
    const uint64_t ntiles = 1ull << (c.n - b);
    const uint64_t per_sm = 3 * (smem + 1088) <= 228 * 1024 ? 3 : 2;  // (with the block's own shared memory and reserve)
    const int blocks = int(std::min<uint64_t>({ntiles, uint64_t(num_sms()) * per_sm, uint64_t(max_blocks)}));
    pauli_tile_kernel<R><<<blocks, kThreads, smem, (cudaStream_t)c.stream>>>(reinterpret_cast<const C *>(c.amp), b, d, ntiles,
                                                                             part);
    return blocks;
}

}  // namespace

size_t pauli_tile_bytes() { return sizeof(PauliTile); }

// Moves the groups listed in `todo` (indices into groups; each has an X mask) that fit the next tile to `take`,
// fills h and returns the tile's bits; 0 if none of them fits a tile.
int pauli_tile_plan(const LaunchCtx &c, const std::vector<PauliXGroup> &groups, std::vector<int> &todo,
                    std::vector<int> &take, void *h)
{
    PauliTile &p = *static_cast<PauliTile *>(h);
    std::memset(&p, 0, sizeof p);
    const int bmax = std::min(c.dt == QS_C64 ? tile_bits<float>() : tile_bits<double>(), c.n);
    const int lo = std::min(c.dt == QS_C64 ? 4 : 3, bmax);
    uint64_t bits = (1ull << lo) - 1;
    std::vector<int> left;
    take.clear();
    size_t nterms = 0;
    for (int gi : todo) {
        const PauliXGroup &g = groups[gi];
        if (take.size() < size_t(kMaxGroups) && nterms + g.zm.size() <= size_t(kMaxTerms) &&
            __builtin_popcountll(bits | g.xm) <= bmax) {
            bits |= g.xm;
            nterms += g.zm.size();
            take.push_back(gi);
        } else {
            left.push_back(gi);
        }
    }
    if (take.empty()) return 0;
    for (int q = 0; __builtin_popcountll(bits) < bmax; ++q) bits |= 1ull << q;
    const int b = __builtin_popcountll(bits);
    p.lo = lo;
    int local_of[64];
    int nl = 0;
    for (int q = 0; q < 64; ++q) {
        local_of[q] = -1;
        if (!(bits >> q & 1)) continue;
        if (nl >= lo) p.hipos[p.nhi++] = (uint8_t)q;
        local_of[q] = nl++;
    }
    auto local = [&](uint64_t m) {
        uint32_t r = 0;
        for (int q = 0; q < 64; ++q)
            if ((m >> q & 1) && local_of[q] >= 0) r |= 1u << local_of[q];
        return r;
    };
    int since = 0;
    for (int gi : take) {
        const PauliXGroup &g = groups[gi];
        PauliGroup &G = p.g[p.ngroups++];
        G.xm = local(g.xm);
        G.piv = uint8_t(31 - __builtin_clz(G.xm));
        G.t0 = uint16_t(p.nterms);
        for (int odd = 0; odd < 2; ++odd) {
            for (size_t t = 0; t < g.zm.size(); ++t) {
                const int ny = __builtin_popcountll(g.xm & g.zm[t]);
                if ((ny & 1) != odd) continue;
                PauliTerm &P = p.t[p.nterms++];
                // 2 Re(i^ny) or -2 Im(i^ny)
                P.c = g.c[t] * (odd ? ((ny & 3) == 1 ? -2.0 : 2.0) : ((ny & 3) == 0 ? 2.0 : -2.0));
                P.zout = g.zm[t] & ~bits;
                // the pair index is the tile index without the pivot bit (which is 0 in x0)
                const uint32_t z = local(g.zm[t]), below = (1u << G.piv) - 1;
                const uint32_t zj = (z & below) | ((z >> (G.piv + 1)) << G.piv);
                P.zthr = zj & (kThreads - 1);
                for (int k = 0; k < 32; ++k)
                    if (__builtin_popcount((zj / kThreads) & k) & 1) P.kpat |= 1u << k;
            }
            if (!odd) G.tmid = uint16_t(p.nterms);
        }
        G.t1 = uint16_t(p.nterms);
        // FP32 sums of at most 8 terms or 4 masks, each of 16 pairs (a pass per mask adds 32 pairs in FP32; the chain
        // takes 1.27 ms without, 1.33 so)
        since += std::max(2, G.t1 - G.t0);
        if (since >= 8) {
            G.flush = 1;
            since = 0;
        }
    }
    todo = std::move(left);
    return b;
}

int launch_pauli_tile(const LaunchCtx &c, const void *d_tile, const void *h_tile, int b, double *part, int max_blocks)
{
    const PauliTile *d = static_cast<const PauliTile *>(d_tile);
    const PauliTile &h = *static_cast<const PauliTile *>(h_tile);
    return c.dt == QS_C64 ? launch_t<float>(c, d, h, b, part, max_blocks) : launch_t<double>(c, d, h, b, part, max_blocks);
}

}  // namespace qs
