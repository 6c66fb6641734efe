// Shared host/device helpers of the GKA library: work decomposition of the chunked
// forward, workspace layout, I/O type conversion, waits.  No method arithmetic lives here.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/gka.h"

namespace gka {

constexpr int kChunk = 64;            // tokens per chunk (C)
constexpr int kMaxDevices = 64;       // device ordinals for which per-device values are cached
constexpr int kMaxWorkItems = 296;    // upper bound on persistent work items (2 per SM on 148 SMs)
// Division of an index below 2^31 by a divisor fixed for a launch, as a multiplication: with l = ceil(log2 d),
// k = 31 + l and M = floor(2^k / d) + 1, floor(n M / 2^k) = floor(n / d) for every n < 2^31 (the excess
// M d - 2^k is at most d, so the error n (M d - 2^k) / (d 2^k) stays below 1 / d).
struct FastDiv {
    unsigned mul, shift, d;
    __host__ __device__ void set(unsigned div) {
        d = div;
        unsigned l = 0;
        while ((1ull << l) < div) ++l;
        shift = 31 + l;
        mul = (unsigned)((1ull << shift) / div + 1ull);
    }
    __host__ __device__ unsigned div(unsigned n) const { return (unsigned)(((unsigned long long)n * mul) >> shift); }
};

// chunks per sequence: the last one holds the T mod C remaining tokens when T is not a multiple of C
__host__ __device__ constexpr int chunks_of(int T) { return (T + kChunk - 1) / kChunk; }

// ---------------------------------------------------------------------------------------------
// Work decomposition of the state pass on the tensor-core path.  The B*heads sequences of N = ceil(T/128) tiles each form one
// flat list of NC = B*heads*N tiles; work item i of G owns the contiguous range [lo(i), lo(i+1)).  A range may cover several
// sequences and may cut a sequence in the middle.  Where an item's range ends inside a sequence the item's last run is
// summarised (decay product, delta-H, delta-U) by the summary kernel; the summaries of the items that hold the earlier part of a
// sequence are folded into the start state of the next item, by the state kernel itself or, where many items share a sequence,
// by a scan kernel before it.  The state kernel then processes all items independently, carrying (H, U) on chip inside each
// run.  (The fp32 kernels split sequences by rules of their own: gka_recur.cu, gka_fwd_small.cu.)
// ---------------------------------------------------------------------------------------------
struct WorkPlan {
    int N;         // tiles per sequence
    long long NC;  // total tiles
    int G;         // work items
    FastDiv divN;  // flat tile index -> sequence
    __host__ __device__ long long lo(int i) const { return ((long long)i * NC) / G; }
    __host__ __device__ void set(int bh, int n, int g) {
        N = n;
        NC = (long long)bh * n;
        G = g;
        divN.set((unsigned)n);
    }
    // start of the last run of item i (flat tile index)
    __host__ __device__ long long last_run_start(int i) const {
        long long l = lo(i), h = lo(i + 1);
        long long s = ((h - 1) / N) * N;
        return s > l ? s : l;
    }
    __host__ __device__ bool cut_out(int i) const { return (lo(i + 1) % N) != 0; }
    __host__ __device__ bool cut_in(int i) const { return (lo(i) % N) != 0; }
};

// State scan of the tensor-core path (floats): start states [G][st], summaries [G][st], decay products [G].
struct Workspace {
    float *start;
    float *delta;
    float *decay;
};

__host__ __device__ inline size_t state_floats(int dk, int dv) {
    return (size_t)dk * dk + (size_t)dv * dk;
}

// fp32 path, head dimensions 64 and 128: room for 3 G segment states and G floats more (gka_recur.cu lays it out)
inline size_t workspace_bytes_for(int G, int dk, int dv) {
    size_t st = state_floats(dk, dv);
    size_t fl = 3 * (size_t)G * st + (size_t)G;
    return ((fl * sizeof(float) + 255) / 256) * 256;
}

// Head dimensions 16 and 32: one state per 32-token chunk of every sequence, and the chunks' decays.
constexpr int kSmallChunk = 32;
__host__ __device__ constexpr int small_chunks_of(int T) { return (T + kSmallChunk - 1) / kSmallChunk; }
inline size_t small_workspace_bytes_for(long long pairs, int T, int d) {
    return (((size_t)pairs * small_chunks_of(T) * (state_floats(d, d) + 1) * sizeof(float) + 255) / 256) * 256;
}

// ---------------------------------------------------------------------------------------------
// Tensor-core path (bf16 I/O, d = 128 or 64).  Its unit of work is a tile of 128 consecutive tokens of one sequence.  A state
// kernel walks the plan's items, carries the fp32 (H, U) on chip and stores, for every tile,
// the bf16 operand copies of the tile-initial H_0 and U_0 and ||H_0||_F^2; the solve kernel then treats the
// tiles as independent problems.  Workspace: start states [G][st], summaries [G][st], decay products [G],
// ||H_0||_F^2 [tiles], bf16 copies [tiles][H, U][column / 8][row][8 columns], 128 x 128 or 64 x 64 (room for the former either way).
// The solve alone writes and reads nothing of U: half of each copy, summary and start state stays as it was.
// ---------------------------------------------------------------------------------------------
constexpr int kTile = 128;
__host__ __device__ constexpr int tiles_of(int T) { return (T + kTile - 1) / kTile; }
constexpr size_t kTileStateBytes = 2 * 128 * 128 * 2;   // bf16 H_0 and U_0 of one tile
constexpr size_t kTileStateBytes64 = 2 * 64 * 64 * 2;   // the same at head dimension 64

struct TcWorkspace {
    float *start, *delta, *decay, *hh;
    unsigned char *hu;
};
inline size_t tc_workspace_bytes_for(int G, long long ntiles) {
    const size_t st = state_floats(128, 128);
    auto up = [](size_t n) { return (n + 255) / 256 * 256; };
    return 2 * up((size_t)G * st * sizeof(float)) + up((size_t)G * sizeof(float)) + up((size_t)ntiles * sizeof(float)) +
           (size_t)ntiles * kTileStateBytes;
}
inline TcWorkspace carve_tc_workspace(void *base, int G, long long ntiles) {
    const size_t st = state_floats(128, 128);
    auto up = [](size_t n) { return (n + 255) / 256 * 256; };
    unsigned char *p = reinterpret_cast<unsigned char *>(base);
    TcWorkspace w;
    w.start = reinterpret_cast<float *>(p); p += up((size_t)G * st * sizeof(float));
    w.delta = reinterpret_cast<float *>(p); p += up((size_t)G * st * sizeof(float));
    w.decay = reinterpret_cast<float *>(p); p += up((size_t)G * sizeof(float));
    w.hh = reinterpret_cast<float *>(p); p += up((size_t)ntiles * sizeof(float));
    w.hu = p;
    return w;
}

// ---------------------------------------------------------------------------------------------
// I/O element access: T is float or __nv_bfloat16; arithmetic always sees float.
// ---------------------------------------------------------------------------------------------
template <typename T> struct Io;
template <> struct Io<float> {
    static __device__ __forceinline__ float4 load4(const float *p) {
        return *reinterpret_cast<const float4 *>(p);
    }
    static __device__ __forceinline__ void store4(float *p, float4 v) {
        *reinterpret_cast<float4 *>(p) = v;
    }
    static __device__ __forceinline__ float load1(const float *p) { return *p; }
    static __device__ __forceinline__ void store1(float *p, float v) { *p = v; }
};
template <> struct Io<__nv_bfloat16> {
    static __device__ __forceinline__ float4 load4(const __nv_bfloat16 *p) {
        uint2 u = *reinterpret_cast<const uint2 *>(p);
        __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162 *>(&u.x);
        __nv_bfloat162 b = *reinterpret_cast<__nv_bfloat162 *>(&u.y);
        float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
        return make_float4(fa.x, fa.y, fb.x, fb.y);
    }
    static __device__ __forceinline__ void store4(__nv_bfloat16 *p, float4 v) {
        __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y);
        __nv_bfloat162 b = __floats2bfloat162_rn(v.z, v.w);
        uint2 u;
        u.x = *reinterpret_cast<uint32_t *>(&a);
        u.y = *reinterpret_cast<uint32_t *>(&b);
        *reinterpret_cast<uint2 *>(p) = u;
    }
    static __device__ __forceinline__ float load1(const __nv_bfloat16 *p) {
        return __bfloat162float(*p);
    }
    static __device__ __forceinline__ void store1(__nv_bfloat16 *p, float v) {
        *p = __float2bfloat16_rn(v);
    }
};

// Programmatic launches.  Every kernel of a call but the validation pass is launched with programmatic stream serialization: its
// blocks may start while the kernel before it still runs.
//   - The first kernel of a call waits (griddepcontrol.wait: the kernel before is complete and its writes visible) before its first
//     access to global memory.
//   - A call of several kernels: the first one releases its dependents (griddepcontrol.launch_dependents) only behind that wait.
//     Every later kernel of the call therefore exists only since all work before the call is complete, and may read the call's
//     inputs ahead of its own wait (fwd_tc_state_kernel behind a summary, fwd_tc_solve_kernel, small_solve), even where the kernel
//     between them (fwd_scan, small_scan) releases it before it has waited itself.  What the call computes is read behind the wait,
//     which is also where it is first written over.
//   - Memory that an earlier kernel may still be writing when this one starts is not read-only for the life of the kernel.  So
//     it is read by ordinary loads: no ld.global.nc or __ldg, and no __restrict__ on a kernel's pointers, which would let the
//     compiler use them and move loads ahead of the wait.
#ifdef __CUDACC__
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// 1 / x for x well inside the normal range (the weight schedule of Algorithm 1 divides by 4 - rho^2 omega, between 2 and 4):
// the hardware's approximation (relative error at most 2^-23) and one Newton step, whose own error is below 2^-46, so that the last
// rounding decides: within one unit in the last place.  Unlike a division it has no rare branch, so the compiler schedules the
// code around it as one block.
__device__ __forceinline__ float recip(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(r, fmaf(-x, r, 1.f), r);
}

// Wait for an mbarrier phase with a time limit (about a second).  The wait sleeps in hardware
// (try_wait with a suspend-time hint), so a waiting warp leaves the issue slots to working warps.
// Returns false if the phase did not complete in time; the caller records GKA_ERR_TIMEOUT and
// leaves cleanly.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar_addr, uint32_t parity) {
    for (int tries = 0; tries < 200000; ++tries) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar_addr), "r"(parity), "r"(5000u)
            : "memory");
        if (done) return true;
    }
    return false;
}
#endif

// Arguments shared by the chunked-forward kernels.
struct FwdArgs {
    const void *q, *k, *v;
    const float *gate, *lam;
    void *out;
    float *state_out;
    const float *state_in;
    float *fro_out;
    const float *beta;     // optional write strengths [B, T, heads]; nullptr = 1
    const float *alpha;    // optional alpha-connection weights [B, T, heads]; nullptr = 1
    int *device_status;
    int B, T, heads;
    int d;                 // head dimension of the caller's tensors (the tensor path works on 128 channels on chip: 64 is zero-extended)
    FastDiv divH;          // sequence index -> batch entry (divisor: heads)
    int n_iter;
    unsigned flags;
    int sms;               // of the current device
    int after_summary;     // tensor path: the main kernel is launched as a programmatic dependent of the summary kernel
    int start_from_scan;   // tensor path: start states were materialised by the scan kernel (long chains of summaries)
    int solve_only;        // write the solve x_t = CH(H_t + lambda_t I, q_t, r) itself instead of U_t x_t (v unused)
    WorkPlan plan;
    Workspace ws;
    float *tile_hh;        // tensor path: ||H_0||_F^2 of every 128-token tile
    float *tile_hh2;       // its second term, where two blocks keep H (or nullptr)
    unsigned char *tile_hu; // tensor path: bf16 H_0, U_0 of every 128-token tile
    cudaEvent_t ev_start, ev_stop;   // optional, recorded around the main kernel (host side only)
};

// Raises a kernel's dynamic shared-memory limit (by default to the most a block can have), once per device (a driver call of about half a
// microsecond otherwise).  One object per kernel, of static storage; safe from several threads.
struct SmemLimit {
    std::atomic<bool> done[kMaxDevices];
    template <typename Kernel> cudaError_t raise(Kernel *kernel, int bytes = 227 * 1024) {
        int dev = 0;
        cudaError_t err = cudaGetDevice(&dev);
        if (err != cudaSuccess || (dev < kMaxDevices && done[dev].load(std::memory_order_relaxed))) return err;
        err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (err == cudaSuccess && dev < kMaxDevices) done[dev].store(true, std::memory_order_relaxed);
        return err;
    }
};

// Shared memory to ask for so that no SM holds more blocks of a grid than its even share.  A programmatic launch places a
// grid's blocks while the grid before still holds its SMs: without the limit they pile up on the SMs that happen to be free
// (128 decode blocks, d = 128, 30 iterations: 17.0 us per step instead of 10.7).
inline size_t spread_smem(size_t natural, long long blocks, int sms) {
    constexpr size_t kPerSm = 228 * 1024, kReserved = 1024;      // per SM; per resident block
    const long long share = sms > 0 ? (blocks + sms - 1) / sms : 17;
    if (share > 16) return natural;
    const size_t most = kPerSm / (size_t)share - kReserved;
    return most > natural ? most / 16 * 16 : natural;
}

// Launchers implemented in the kernel translation units.  Each returns a cudaError_t.
cudaError_t launch_fwd_recur(const FwdArgs &a, int io_dtype, void *ws, size_t ws_bytes, cudaStream_t stream);
cudaError_t launch_fwd_small(const FwdArgs &a, int io_dtype, void *ws, cudaStream_t stream);
cudaError_t launch_decode(float *state, const void *q, const void *k, const void *v,
                          const float *gate, const float *lam, int n_iter, void *out, int nseq,
                          int heads, int d, int io_dtype, unsigned flags, const float *beta, const float *alpha, int *device_status,
                          int sms, cudaEvent_t ev_start, cudaEvent_t ev_stop, cudaStream_t stream);
// head dimensions 16 and 32, T >= 1 tokens per sequence: one warp per (sequence, head) pair
cudaError_t launch_decode_small(float *state, const void *q, const void *k, const void *v, const float *gate,
                                const float *lam, int n_iter, void *out, int nseq, int T, int heads, int d, int io_dtype,
                                unsigned flags, const float *beta, const float *alpha, cudaEvent_t ev_start,
                                cudaEvent_t ev_stop, cudaStream_t stream);
// the same step over T consecutive tokens per sequence, the state read and written once
cudaError_t launch_decode_multi(float *state, const void *q, const void *k, const void *v, const float *gate,
                                const float *lam, int n_iter, void *out, int nseq, int T, int heads, int d, int io_dtype,
                                unsigned flags, const float *beta, const float *alpha, int *device_status, int sms,
                                cudaEvent_t ev_start, cudaEvent_t ev_stop, cudaStream_t stream);

}  // namespace gka
