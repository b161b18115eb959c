// k_batch_lean.cu -- the batched launch for circuits whose passes all lower to the in-place stage engine
// (variational circuits do; k_batch.cu takes the others and explains the queue and its dependency order).
//
// What bounds a batch is the latency of the stages' shared-memory round trips and dependent FMAs: one CTA of
// eight warps per SM leaves the FP32 pipes idle most of the time (64 circuits of 10-20 qubits, 3.37 ms on
// the general engine; the FMAs alone take 0.4).  Two CTAs per SM, one slab each: while one gathers, stores, waits for the queue or for the last pass
// of its circuit, the other computes.  One warp reads the next item's descriptors, gather tables and
// pass program into the second slot while the slab of this one is under way, so the queue's latency
// (an atomic and three dependent reads) is off the path.  64 circuits of 10-20 qubits: 1.32 ms (one CTA
// with two slabs and a producer warp: 1.99); 300 of 10-15: 750 -> 377 us; 8 of 14-20: 1160 -> 558 us.
// complex64 only: FP64 work gains nothing from a second CTA on the SM, so complex128 stays on the general
// engine (59 circuits of 10-15 qubits: 991 us there, in place 1063 us with one CTA per SM and 1328 with two).
//
// A CTA looks at the next item only after this one is stored, and an item waits only for items before
// it in the queue: the earliest unfinished item can always run.  The wait is bounded.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>

#include "lean_stage.cuh"

namespace qs {
namespace {

constexpr uint32_t kSpinLimit = 1u << 23;
constexpr int kMaxBits = 13;  // 64 KiB of slab

struct __align__(16) LeanSlot {
    uint64_t seg_lo[64], seg_hi[64];  // gather tables of the item's pass, in 16-byte vectors
    DevPass pass;
    BatchItem item;
    BatchCirc circ;
    BatchProg prog;
    uint64_t base;                    // slab base index in the circuit's state
    int st;                           // 0: the queue is empty
    int follows;                      // the next slab of the same run: its dependency holds
};
struct __align__(16) LeanShared {
    LeanSlot slot[2];
    double red[32];
    int late;                         // the dependency wait ran out: skip the work
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// A pass program in shared memory, or in device memory if it is too long.
struct NearWords {
    const ulonglong2 *p;
    __device__ __forceinline__ ulonglong2 operator()(uint32_t i) const { return p[i]; }
    __device__ __forceinline__ ulonglong2 bulk(uint32_t i) const { return p[i]; }
};

// 16-byte chunk of shared memory that holds amplitudes 2 v and 2 v + 1 of the slab
__device__ __forceinline__ uint32_t chunk_of(uint32_t v) { return swz<1>(v << 1) >> 1; }

// One warp: the next slab (of the same run, or the first of the next queue item) into slot Z.
__device__ __forceinline__ void fetch(LeanSlot &Z, const LeanSlot *prev, const BatchArgs &a, ulonglong2 *wbuf, uint32_t wcap, uint32_t lane)
{
    if (lane == 0) {
        Z.st = 1;
        Z.follows = prev != nullptr && prev->item.count > 1;
        if (Z.follows) {
            Z.item = prev->item;
            Z.item.slab += 1;
            Z.item.count -= 1;
        } else {
            const unsigned it = atomicAdd(a.head, 1u);
            if (it >= a.nitems) Z.st = 0;
            else Z.item = a.items[it];
        }
        if (Z.st) {
            Z.circ = a.circs[Z.item.circ];
            const int p = Z.circ.pass0 + Z.item.pass;
            Z.pass = a.passes[p];
            Z.prog = a.progs[p];
        }
    }
    __syncwarp();
    if (!Z.st) return;
    if (Z.prog.nwords <= wcap) {
        const ulonglong2 *w = static_cast<const ulonglong2 *>(a.words) + Z.prog.begin;
        for (uint32_t i = lane; i < Z.prog.nwords; i += 32) cp_async16(smem_addr(wbuf + i), w + i);
    }
    const int lo = Z.pass.lo, nhi = Z.pass.nhi;
    for (uint32_t j = lane; j < 128; j += 32) {
        const uint32_t x = j & 63, sh = (j < 64) ? 0 : 6;
        uint64_t o = 0;
        for (int m = 0; m < 6; ++m)
            if ((x >> m & 1) && int(m + sh) < nhi) o |= 1ull << Z.pass.hipos[m + sh];
        if (j < 64) Z.seg_lo[x] = o >> 1; else Z.seg_hi[x] = o >> 1;
    }
    if (lane == 0) {
        uint64_t base = uint64_t(Z.item.slab) << lo;
        for (int m = 0; m < nhi; ++m) {
            const uint64_t lowm = (1ull << Z.pass.hipos[m]) - 1;
            base = ((base & ~lowm) << 1) | (base & lowm);
        }
        Z.base = base;
    }
}

// <psi| sum_t c_t Z_t |psi> over the slab.  With x = base | deposit(i) (base: the bits outside the slab),
// (-1)^{popcount(x & z_t)} = s_t(base) (-1)^{popcount(i & zl_t)} where zl_t is z_t on the slab's local
// bits, so the slab contributes
//   sum_t c_t s_t(base) P^(zl_t),   P^(z) = sum_i |a_i|^2 (-1)^{popcount(i & z)},
// the Walsh-Hadamard transform of the slab's probabilities (in FP32).  Element i = tid + NT k: the
// levels over k run in registers, the lane bits by shuffles, the warp bits after one exchange.
template <int NT>
__device__ __forceinline__ double slab_energy(float2 *sm, int b, const LeanSlot &Z, const BatchTerm *T, uint32_t tid)
{
    constexpr int TB = NT == 512 ? 9 : 8, KB = kMaxBits - TB, K = 1 << KB;
    const uint32_t nsl = 1u << b, lane = tid & 31;
    float p[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t i = tid + uint32_t(k) * NT;
        p[k] = 0.f;
        if (i < nsl) {
            const float2 v = sm[swz<1>(i)];
            p[k] = v.x * v.x + v.y * v.y;
        }
    }
#pragma unroll
    for (int m = 0; m < KB; ++m)
        if (TB + m < b) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (!(k >> m & 1)) {
                    const float u = p[k], w = p[k | 1 << m];
                    p[k] = u + w;
                    p[k | 1 << m] = u - w;
                }
        }
#pragma unroll
    for (int j = 0; j < 5; ++j)
        if (j < b) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const float o = __shfl_xor_sync(0xffffffffu, p[k], 1 << j);
                p[k] = (lane >> j & 1) ? o - p[k] : p[k] + o;
            }
        }
    float *pr = reinterpret_cast<float *>(sm);
    __syncthreads();  // every amplitude has been read: the buffer now holds the transform
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t i = tid + uint32_t(k) * NT;
        if (i < nsl) pr[i] = p[k];
    }
    __syncthreads();
    if (b > 5) {
        constexpr int WB = TB - 5, W = 1 << WB;  // warp bits
        for (uint32_t q = tid; q < 32u * K; q += NT) {
            const uint32_t i0 = (q & 31) + (q >> 5) * NT;
            if (i0 >= nsl) break;
            float w[W];
#pragma unroll
            for (int x = 0; x < W; ++x) w[x] = i0 + 32u * x < nsl ? pr[i0 + 32u * x] : 0.f;
#pragma unroll
            for (int m = 0; m < WB; ++m)
                if (5 + m < b) {
#pragma unroll
                    for (int x = 0; x < W; ++x)
                        if (!(x >> m & 1)) {
                            const float u = w[x], v = w[x | 1 << m];
                            w[x] = u + v;
                            w[x | 1 << m] = u - v;
                        }
                }
#pragma unroll
            for (int x = 0; x < W; ++x)
                if (i0 + 32u * x < nsl) pr[i0 + 32u * x] = w[x];
        }
        __syncthreads();
    }
    double acc = 0.0;
    for (int t = int(tid); t < Z.circ.nterm; t += NT) {
        const uint64_t zm = T[t].zm;
        uint32_t zl = uint32_t(zm) & ((1u << Z.pass.lo) - 1u);
        for (int m = 0; m < Z.pass.nhi; ++m) zl |= uint32_t((zm >> Z.pass.hipos[m]) & 1u) << (Z.pass.lo + m);
        const double sg = (__popcll(Z.base & zm) & 1) ? -T[t].c : T[t].c;
        acc += sg * double(pr[zl]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    return acc;
}

template <int RB, int NT, int PER_SM>
__global__ void __launch_bounds__(NT, PER_SM)
    batch_lean_kernel(float2 *__restrict__ states, const __grid_constant__ BatchArgs a, uint32_t wcap)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    LeanShared &S = *reinterpret_cast<LeanShared *>(smem_raw);
    ulonglong2 *const wbufs = reinterpret_cast<ulonglong2 *>(smem_raw + ((sizeof(LeanShared) + 127) & ~size_t(127)));
    float2 *const sm = reinterpret_cast<float2 *>(wbufs + 2 * size_t(wcap));
    const uint32_t tid = threadIdx.x;

    if (tid < 32) fetch(S.slot[0], nullptr, a, wbufs, wcap, tid);
    __syncthreads();
    for (uint32_t k = 0;; k ^= 1u) {
        const LeanSlot &Z = S.slot[k];
        if (Z.st == 0) break;
        if (tid == 0) {
            int late = 0;
            if (Z.item.pass > 0 && !Z.follows) {
                // the circuit's previous pass, all of it stored (bounded)
                const unsigned need = 1u << Z.circ.nslab_log;
                const unsigned *cnt = a.done + Z.circ.done0 + Z.item.pass - 1;
                uint32_t n = 0;
                while (ld_acquire(cnt) < need && ++n < kSpinLimit) __nanosleep(128);
                if (n >= kSpinLimit) {
                    atomicExch(a.status, QS_ETIMEOUT);  // the host reports it
                    late = 1;
                }
                __threadfence();
            }
            S.late = late;
        }
        __syncthreads();
        const bool work = S.late == 0;
        {
            const int vps_log = Z.pass.lo - 1;
            const uint32_t nvec = 1u << (Z.pass.b - 1);
            if (Z.item.pass == 0) {
                for (uint32_t e = tid; e < (1u << Z.pass.b); e += NT) {
                    sm[swz<1>(e)] = make_float2(Z.base == 0 && e == 0 ? 1.f : 0.f, 0.f);
                }
            } else if (work) {
                const uint4 *g = reinterpret_cast<const uint4 *>(states + Z.circ.amp_off + Z.base);
                const uint32_t dst = smem_addr(sm);
#pragma unroll 4
                for (uint32_t v = tid; v < nvec; v += NT) {
                    const uint32_t seg = v >> vps_log, w = v & ((1u << vps_log) - 1);
                    cp_async16(dst + 16u * chunk_of(v), g + ((Z.seg_lo[seg & 63] | Z.seg_hi[(seg >> 6) & 63]) + w));
                }
            }
        }
        if (tid < 32) fetch(S.slot[k ^ 1u], &Z, a, wbufs + size_t(k ^ 1u) * wcap, wcap, tid);
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        if (work) {
            const NearWords words{Z.prog.nwords <= wcap ? wbufs + size_t(k) * wcap
                                                        : static_cast<const ulonglong2 *>(a.words) + Z.prog.begin};
            uint32_t at = 0;
#pragma unroll 1
            for (uint32_t o = 0; o < Z.prog.nstages; ++o) {
                at = run_lean_stage<float2, RB>(sm, words, at, static_cast<const float2 *>(a.pool), Z.base, tid);
                __syncthreads();
            }
            if (Z.item.pass == Z.circ.npass - 1) {
                // the final states are not kept (the batch returns expectation values only)
                const double part = slab_energy<NT>(sm, Z.pass.b, Z, a.terms + Z.circ.term0, tid);
                if ((tid & 31) == 0) S.red[tid >> 5] = part;
                __syncthreads();
                if (tid < 32) {
                    double v = tid < NT / 32 ? S.red[tid] : 0.0;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
                    if (tid == 0) atomicAdd(a.results + Z.item.circ, v);
                }
            } else {
                const int vps_log = Z.pass.lo - 1;
                const uint32_t nvec = 1u << (Z.pass.b - 1);
                uint4 *g = reinterpret_cast<uint4 *>(states + Z.circ.amp_off + Z.base);
#pragma unroll 4
                for (uint32_t v = tid; v < nvec; v += NT) {
                    const uint32_t seg = v >> vps_log, w = v & ((1u << vps_log) - 1);
                    st_stream(g + ((Z.seg_lo[seg & 63] | Z.seg_hi[(seg >> 6) & 63]) + w),
                              reinterpret_cast<const uint4 *>(sm)[chunk_of(v)]);
                }
            }
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) atomicAdd(a.done + Z.circ.done0 + Z.item.pass, 1u);
    }
}

template <int RB, int NT, int PER_SM>
int launch_t(void *states, const BatchArgs &a, int b_max, void *stream, char *err, size_t errlen)
{
    // longest pass program that is kept in shared memory (longer ones are read from L2)
    const uint32_t wcap = std::min(a.max_words, 1400u);
    const size_t smem = ((sizeof(LeanShared) + 127) & ~size_t(127)) + 2 * size_t(wcap) * 16 + (sizeof(float2) << b_max);
    auto *const kern = batch_lean_kernel<RB, NT, PER_SM>;
    static int attr_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (attr_dev != dev) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        attr_dev = dev;
    }
    // a second CTA per SM where a round has slabs for it (else it would take work from idle SMs)
    const unsigned sms = unsigned(num_sms()), ctas = a.width > sms ? sms * PER_SM : sms;
    const unsigned grid = std::max(1u, std::min(ctas, unsigned(a.nitems)));
    if (b_max > kMaxBits || smem > 227 * 1024) {
        snprintf(err, errlen, "batch slab of %d bits does not fit in shared memory", b_max);
        return QS_EINVAL;
    }
    kern<<<grid, NT, smem, (cudaStream_t)stream>>>(static_cast<float2 *>(states), a, wcap);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        snprintf(err, errlen, "batch launch failed: %s", cudaGetErrorString(e));
        return QS_ECUDA;
    }
    return QS_OK;
}

}  // namespace

int launch_batch_lean(int stage_bits, void *states, const BatchArgs &a, int b_max, void *stream, char *err, size_t errlen)
{
    if (stage_bits == kStageBitsC64 - 1) return launch_t<kStageBitsC64 - 1, 512, 1>(states, a, b_max, stream, err, errlen);
    return launch_t<kStageBitsC64, 256, 2>(states, a, b_max, stream, err, errlen);
}

}  // namespace qs
