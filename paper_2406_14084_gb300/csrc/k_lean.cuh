// k_lean.cuh -- slab passes whose register stages all run on the in-place engine (lean_stage.cuh).
//
// Same pass as k_slab.cu (load a slab, run its stages, store it), laid out for occupancy instead of
// a per-CTA pipeline: 256 threads at 128 registers and one slab buffer (64 KiB), so two CTAs share
// an SM and one computes while the other loads or stores.  Measured with the stage engine, whole
// circuits, general engine -> now: layered-28 complex64 (20 layers, 14 passes) 89.2 -> 37.9 ms, complete-graph
// QAOA-23 complex64 2.94 -> 0.53 ms, QFT-28 complex128 110.6 -> 72.1 ms (FP64 pipe 89 % busy), layered-25
// complex128 104.2 -> 94.7 ms, layered-26 in double-float form 60.9 -> 37.7 ms.
//
// Each arithmetic has a source file of its own (k_lean.cu complex64, k_lean_c128.cu, k_lean_df.cu): a module is
// loaded whole by the first launch from it, and one with all fifteen kernels grew past the size up to which
// nvcc leaves modules uncompressed (first launch of a process 10 ms, with 11 kernels 1.0).
#pragma once

#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>

#include "lean_stage.cuh"

namespace qs {
namespace {

constexpr uint32_t kMaxVec = 4096;  // 16-byte chunks of the largest slab

// A pass program.  NW > 0: its words travel in the kernel's parameters, i.e. in constant memory, whose
// loads are uniform and short (a stage's fixed part: 570 against 640 ns per slab and SM); NW = 0: in
// device memory, for longer programs (4 KiB of parameters cost less than 32 KiB, hence two sizes).
// Table factors come from device memory in both: through constant memory a table took 374 ns, not 292,
// since f32x2 operands there have to be copied to registers.
template <int NW> struct LeanProgram {
    DevPass pass;
    int nstages;
    const ulonglong2 *g;
    ulonglong2 w[NW];
    __device__ __forceinline__ ulonglong2 bulk(uint32_t i) const { return load_word(g + i); }
    __device__ __forceinline__ ulonglong2 operator()(uint32_t i) const { return w[i]; }
};
template <> struct LeanProgram<0> {
    DevPass pass;
    int nstages;
    const ulonglong2 *g;
    __device__ __forceinline__ ulonglong2 bulk(uint32_t i) const { return load_word(g + i); }
    __device__ __forceinline__ ulonglong2 operator()(uint32_t i) const { return __ldg(g + i); }
};

// SMALL: slabs with fewer groups than threads (states and slab options below the default slab), where whole warps
// have none.  A variant of its own: the test costs full slabs 1 to 6 % in registers.
template <typename R, int RB, int NT, int PER_SM, bool DF, int NW, bool FULL, bool SMALL>
__global__ void __launch_bounds__(NT, PER_SM)
    lean_pass_kernel(typename Cx<R>::T *__restrict__ state, const __grid_constant__ LeanProgram<NW> prog,
                     const void *__restrict__ pool, uint64_t nslabs)
{
    using C = typename Cx<R>::T;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const uint32_t tid = threadIdx.x;
    const int b = prog.pass.b, lo = prog.pass.lo, nhi = prog.pass.nhi;
    const uint32_t nsl = 1u << b, nseg = 1u << nhi;
    // [slab][segment offsets: 16-byte offset of segment s from the slab's base]
    C *const sm = reinterpret_cast<C *>(smem_raw);
    uint64_t *const seg = reinterpret_cast<uint64_t *>(smem_raw + (sizeof(C) << b));
    constexpr int kLog16 = (sizeof(C) == 8) ? 1 : 0;
    for (uint32_t s = tid; s < nseg; s += NT) {
        uint64_t o = 0;
        for (int m = 0; m < nhi; ++m)
            if (s >> m & 1) o |= 1ull << prog.pass.hipos[m];
        seg[s] = o >> kLog16;
    }
    __syncthreads();
    const int vps_log = lo - kLog16;
    const uint32_t nvec = 1u << (b - kLog16);
    auto chunk_of = [](uint32_t v) -> uint32_t { return sizeof(C) == 8 ? (swz<1>(v << 1) >> 1) : swz<2>(v); };
    const uint32_t ct = chunk_of(tid);
    const uint32_t dst = smem_addr(sm);

    for (uint64_t slab = blockIdx.x; slab < nslabs; slab += gridDim.x) {
        uint64_t base = slab << lo;
        for (int m = 0; m < nhi; ++m) {
            const uint64_t lowm = (1ull << prog.pass.hipos[m]) - 1;
            base = ((base & ~lowm) << 1) | (base & lowm);
        }
        uint4 *const g = reinterpret_cast<uint4 *>(state + base);
#pragma unroll 8
        for (uint32_t j = 0; j < kMaxVec / NT; ++j) {
            const uint32_t v = tid + j * NT;
            if (v >= nvec) break;
            cp_async16(dst + 16u * (ct ^ chunk_of(j * NT)), g + (seg[v >> vps_log] + (v & ((1u << vps_log) - 1))));
        }
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        if constexpr (DF) {
            dfp *sd = reinterpret_cast<dfp *>(sm);
            for (uint32_t e = tid; e < nsl; e += NT) {
                const C a = sm[e];
                const df x = d2df(a.x), y = d2df(a.y);
                sd[e] = dfp{pack2(x.h, y.h), pack2(x.l, y.l)};
            }
            __syncthreads();
        }
        uint32_t at = 0;
#pragma unroll 1
        for (int o = 0; o < prog.nstages; ++o) {
            if (SMALL && !with_groups(tid, b - RB)) {
            } else if constexpr (DF)
                at = run_lean_stage<dfp, RB, FULL>(reinterpret_cast<dfp *>(sm), prog, at, static_cast<const dfp *>(pool), base, tid);
            else
                at = run_lean_stage<C, RB, FULL>(sm, prog, at, static_cast<const C *>(pool), base, tid);
            __syncthreads();
        }
#pragma unroll 8
        for (uint32_t j = 0; j < kMaxVec / NT; ++j) {
            const uint32_t v = tid + j * NT;
            if (v >= nvec) break;
            uint4 q = reinterpret_cast<const uint4 *>(sm)[ct ^ chunk_of(j * NT)];
            if constexpr (DF) {
                const df x(__uint_as_float(q.x), __uint_as_float(q.z)), y(__uint_as_float(q.y), __uint_as_float(q.w));
                const double2 d = make_double2(df2d(x), df2d(y));
                q = *reinterpret_cast<const uint4 *>(&d);
            }
            st_stream(g + (seg[v >> vps_log] + (v & ((1u << vps_log) - 1))), q);
        }
        __syncthreads();  // the slab is overwritten by the next load
    }
}

template <typename R, int RB, int NT, int PER_SM, bool DF, int NW, bool FULL, bool SMALL = false>
int launch_lean_t(const LaunchCtx &c, const LeanPassArgs &a, const DevPass &h, char *err, size_t errlen)
{
    using C = typename Cx<R>::T;
    const size_t smem = (sizeof(C) << h.b) + (sizeof(uint64_t) << h.nhi);
    auto *const kern = lean_pass_kernel<R, RB, NT, PER_SM, DF, NW, FULL, SMALL>;
    static int attr_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (attr_dev != dev) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
        attr_dev = dev;
    }
    const uint64_t nslabs = 1ull << (c.n - h.b);
    uint64_t grid = uint64_t(num_sms()) * (smem <= 112 * 1024 ? PER_SM : 1);
    if (grid > nslabs) grid = nslabs;
    LeanProgram<NW> prog;
    prog.pass = h;
    prog.nstages = a.nstages;
    prog.g = static_cast<const ulonglong2 *>(a.d_words);
    if constexpr (NW > 0) std::memcpy(prog.w, a.h_words, size_t(a.nwords) * 16);
    kern<<<(unsigned)grid, NT, smem, (cudaStream_t)c.stream>>>(reinterpret_cast<C *>(c.amp), prog, a.pool, nslabs);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        snprintf(err, errlen, "slab pass launch failed: %s", cudaGetErrorString(e));
        return QS_ECUDA;
    }
    return QS_OK;
}

}  // namespace

// complex128 passes in FP64 and in double-float form (LeanPassArgs::df)
int launch_lean_c128(const LaunchCtx &c, const LeanPassArgs &a, const DevPass &h, char *err, size_t errlen);
int launch_lean_df(const LaunchCtx &c, const LeanPassArgs &a, const DevPass &h, char *err, size_t errlen);

// Fewer groups than threads: warps without one stay out of the arithmetic in complex128 (FP64, 10 qubits, 4
// layers: 188 -> 125 us, 22 qubits with slabs of 8 bits 33.0 -> 10.4 ms; double-float, the same slabs 9.7 -> 5.8
// ms).  complex64 has FP32 issue slots to spare (2.8 -> 1.7 ms there, but 1 % on 10 qubits and 6 % on full slabs
// if tested always) and keeps one kernel.
inline bool small_slab(const LeanPassArgs &a, const DevPass &h, int threads) { return 1 << (h.b - a.stage_bits) < threads; }

}  // namespace qs
