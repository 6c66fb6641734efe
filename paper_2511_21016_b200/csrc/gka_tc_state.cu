// tcgen05 path of the chunked GKA forward (bf16 operands, fp32 accumulation) for sm_100a: launcher, the
// segment-summary kernel and the state kernel.  The solve kernel (Algorithm 1 on 128-token tiles) is in
// gka_tc_solve.cu.
//
// The path works on tiles of 128 consecutive tokens of one sequence (two of the paper's chunks: the chunk-wise
// form of Section 4.2.1 is exact for any chunk size).  The state recurrences of eq. (CH),
//     H_t = gamma_t H_{t-1} + beta_t k_t k_t^T,     U_t = gamma_t U_{t-1} + beta_t v_t k_t^T,
// advance tile by tile:  H <- zeta H + K^T diag(w) K,  U <- zeta U + V^T diag(w) K  with zeta the decay of the whole
// tile and w_j the decay from token j to the tile's end (times beta_j).  The state kernel keeps fp32 masters of H
// and U on chip for a whole run of tiles and stores, for every tile, the bf16 operand copies of the
// tile-initial H_0, U_0 and ||H_0||_F^2 (the paper stores the chunk-initial states as well); the solve kernel
// then processes the tiles as independent problems.
//
// Work decomposition (gka_common.cuh): the flat list of tiles is cut into one contiguous range per thread block.
// Where a range ends inside a sequence the summary kernel first computes the decay product and (delta-H,
// delta-U) of its last run, i.e. the run's final state for a zero start state; the state kernel folds the
// summaries of the blocks that hold the earlier part of a sequence into its start state (long chains are
// materialised once by the scan kernel instead).
#include <cuda.h>

#include "gka_common.cuh"
#include "gka_tc_mma.cuh"

namespace gka {
cudaError_t launch_fwd_solve(const FwdArgs &a, cudaStream_t stream);   // gka_tc_solve.cu
namespace {

using namespace tcu;

constexpr int D = 128;
constexpr int NT = kTile;                                // tokens per tile
constexpr int CT = 512;                                  // compute threads; + one warp that issues the products
constexpr int kThreadsState = CT + 32;

// ------------------------------------------------------------------------------------------------------------
// Both kernels advance a state by whole tiles with the products K~^T K~ and V~^T K~ on rows scaled in place,
// K~_j = sqrt(w_j) k_j and V~_j = sqrt(w_j) v_j (w_j includes the write strength beta_j), so that no weighted copy of
// the keys is needed and three TMA stages of K and V tiles fit: the loads run two tiles ahead.
// ------------------------------------------------------------------------------------------------------------
constexpr int NS = 3;                                    // TMA stages
constexpr uint32_t STAGE = 65536;                        // K tile + V tile
constexpr uint32_t KV_SMEM = NS * STAGE + 1024;          // + slack for the 1024-byte alignment of the base
constexpr uint32_t ST_SMEM = KV_SMEM;

// The first N * THREADS 16-byte groups of BOXES operand boxes (64 channels of 128 tokens each) times f[row]
template <int N, int THREADS, int BOXES>
__device__ __forceinline__ void scale_rows(unsigned char *box, const uint2 *f, int t) {
    uint4 v[BOXES][N];
    uint2 fj[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        fj[i] = f[(t + THREADS * i) >> 3];         // 8 groups of 16 bytes in a row
#pragma unroll
        for (int x = 0; x < BOXES; ++x) v[x][i] = *reinterpret_cast<const uint4 *>(box + 16384 * x + (t + THREADS * i) * 16);
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
#pragma unroll
        for (int x = 0; x < BOXES; ++x) *reinterpret_cast<uint4 *>(box + 16384 * x + (t + THREADS * i) * 16) = times_factor(v[x][i], fj[i]);
    }
}

// A wait of the block has given up, so products and copies may still be in flight: the products end (a commit by the thread that
// issued them on a barrier of its own, awaited with a limit) and the copies get time to, before the block gives back its tensor
// and shared memory.  At the kernels' end, off the path of a call that goes well.
__device__ __forceinline__ void drain(uint32_t bar, int issuer) {
    if ((int)threadIdx.x == issuer) {
        mma_commit(bar);
        mbar_spin_bounded(bar, 0u);
    }
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    __syncthreads();
}

// ------------------------------------------------------------------------------------------------------------
// Segment summaries.  The weights are formed in log2 space from the run's total log-decay (one pre-pass over the
// gates) and a running prefix, so every tile is a pure accumulation into TMEM: no rescaling pass.  The kernel
// streams K and V once.  A summarised run never holds the last tile of its sequence, so all its tiles are full.
// ------------------------------------------------------------------------------------------------------------
enum { SB_KV0 = 0, SB_MMA = NS, SB_DRAIN, SB_COUNT };

__global__ void __launch_bounds__(kThreadsState, 1)
fwd_tc_summary_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, FwdArgs a) {
    const WorkPlan &P = a.plan;
    const int item = blockIdx.x;
    // Programmatic launch in stream order: wait for whatever wrote the inputs, then let the state kernel's blocks take the SMs
    // that this grid leaves and run their prologue; they wait for this grid's completion before they read a summary.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (!P.cut_out(item)) return;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t s_bars[SB_COUNT];
    __shared__ uint32_t s_tmem_base;
    __shared__ __align__(16) uint2 s_w[NT];
    __shared__ float s_ca[4], s_red[16];
    __shared__ int s_req, s_abort;
    unsigned char *smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    const uint32_t sb = smem_u32(smem), bars = smem_u32(&s_bars[0]);
    const int t = threadIdx.x, l = t & 31;

    if (t == 0) {
        s_abort = 0;
        for (int i = 0; i < SB_COUNT; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bars + 8 * i));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (t < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(&s_tmem_base))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem_base, tm_H = tmem, tm_U = tmem + 128;

    const long long f0 = P.last_run_start(item), f1 = P.lo(item + 1);
    const int ntiles = (int)(f1 - f0);
    const uint32_t base14 = (sb >> 4) & 0x3FFF;
    auto aborted = [&]() { return *reinterpret_cast<volatile int *>(&s_abort) != 0; };
    auto wait = [&](int which, uint32_t parity) {     // once a wait has given up the later ones return at once
        if (!aborted() && !mbar_spin_bounded(bars + 8 * which, parity)) *reinterpret_cast<volatile int *>(&s_abort) = 1;
    };

    if (t >= CT) {
        // ================================ MMA issuing warp ================================
        for (;;) {
            asm volatile("bar.sync 3, 544;" ::: "memory");         // the compute threads hand over a tile
            const int n = *reinterpret_cast<const volatile int *>(&s_req);
            if (n < 0) break;
            if (l == 0) {
                fence_after();
                const uint32_t kb = base14 + (uint32_t)(n % NS) * (STAGE >> 4), vb = kb + (32768u >> 4);
                if (n == 0) {
                    mma8_mm<0>(tm_H, kb, kb, kIdescMM);
                    if (!a.solve_only) mma8_mm<0>(tm_U, vb, kb, kIdescMM);
                } else {
                    mma8_mm<1>(tm_H, kb, kb, kIdescMM);
                    if (!a.solve_only) mma8_mm<1>(tm_U, vb, kb, kIdescMM);
                }
                mma_commit(bars + 8 * SB_MMA);
            }
            __syncwarp();
        }
    } else {
        // ================================= compute threads =================================
        const int seq = (int)((unsigned)f0 / (unsigned)P.N), b = seq / a.heads, h = seq % a.heads;
        const int n0 = (int)((unsigned)f0 - (unsigned)seq * (unsigned)P.N);   // first tile of the run in its sequence
        const float *grun = a.gate + ((size_t)b * a.T + (size_t)n0 * NT) * a.heads + h;   // token stride: heads
        const float *brun = a.beta ? a.beta + ((size_t)b * a.T + (size_t)n0 * NT) * a.heads + h : nullptr;
        const int ntok_run = ntiles * NT;
        auto issue_tma = [&](int n) {
            const uint32_t dst = sb + (uint32_t)(n % NS) * STAGE;
            const uint32_t bar = bars + 8 * (SB_KV0 + n % NS);
            mbar_expect_tx(bar, a.solve_only ? 32768u : 65536u);
            tma_load_tile3(&tmK, dst, bar, h * a.d, tile_x_hi(h, a.d, a.heads), (n0 + n) * NT, b);
            if (!a.solve_only) tma_load_tile3(&tmV, dst + 32768, bar, h * a.d, tile_x_hi(h, a.d, a.heads), (n0 + n) * NT, b);
        };
        if (t == 0)
            for (int n = 0; n < ntiles && n < NS; ++n) issue_tma(n);

        // ---- pre-pass: total log2 decay of the run
        float total = 0.f;
        {
            float s = 0.f;
            for (int i0 = t; i0 < ntok_run; i0 += 4 * CT) {     // four independent loads in flight per thread
                float g[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = i0 + u * CT;
                    g[u] = (i < ntok_run) ? grun[(size_t)i * a.heads] : 1.f;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) s += fmaxf(log2f(g[u]), -115.f);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (l == 0) s_red[t >> 5] = s;
            asm volatile("bar.sync 1, 512;" ::: "memory");
#pragma unroll
            for (int i = 0; i < 16; ++i) total += s_red[i];
        }

        // threads 0..127: gate of token t of tile n; fetched one tile ahead, the logarithm is taken when the
        // value is used so that nothing waits for the load
        auto load_gate = [&](int n) -> float {
            const int i = n * NT + t;
            return (t < NT && i < ntok_run) ? ld_stream_f32(grun + (size_t)i * a.heads) : 1.f;
        };
        float g_cur = load_gate(0);
        float prefix = 0.f;                    // log2 decay of the tiles before the current one
        for (int n = 0; n < ntiles; ++n) {
            const float g_next = load_gate(n + 1);
            if (t < NT) {
                float incl = fmaxf(log2f(g_cur), -115.f);
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float up = __shfl_up_sync(0xffffffffu, incl, o);
                    if (l >= o) incl += up;
                }
                if (l == 31) s_ca[t >> 5] = incl;
                asm volatile("bar.sync 2, 128;" ::: "memory");
                float before = 0.f, tile_total = 0.f;
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    if (w < (t >> 5)) before += s_ca[w];
                    tile_total += s_ca[w];
                }
                incl += before;
                // w_j = 2^(decay from token j to the end of the run) = 2^((total - prefix) - incl_j); its root scales the rows
                float wt = exp2f(0.5f * ((total - prefix) - incl));
                if (brun) wt *= sqrtf(fmaxf(brun[(size_t)(n * NT + t) * a.heads], 0.f));   // write strength
                s_w[t] = split_factor(wt);
                prefix += tile_total;
            }
            wait(SB_KV0 + n % NS, (uint32_t)((n / NS) & 1));
            asm volatile("bar.sync 1, 512;" ::: "memory");       // weights are published (and the scan scratch is free)
            unsigned char *const stage = smem + (size_t)(n % NS) * STAGE;
            scale_rows<2, CT, 2>(stage, s_w, t);
            if (!a.solve_only) scale_rows<2, CT, 2>(stage + 32768, s_w, t);
            fence_async_smem();
            if (t == 0) *reinterpret_cast<volatile int *>(&s_req) = n;
            asm volatile("bar.sync 3, 544;" ::: "memory");       // hand the tile to the issuing warp
            // the previous tile's products are done: its stage takes the tile after the next
            if (n >= 1) {
                wait(SB_MMA, (uint32_t)((n - 1) & 1));
                if (t == 0 && n + 2 < ntiles && !aborted()) issue_tma(n + 2);
            }
            g_cur = g_next;
        }
        if (ntiles > 0) wait(SB_MMA, (uint32_t)((ntiles - 1) & 1));
        if (t == 0) *reinterpret_cast<volatile int *>(&s_req) = -1;
        asm volatile("bar.sync 3, 544;" ::: "memory");           // releases the issuing warp
        fence_after();
        if (s_abort != 0) {
            if (t == 0 && a.device_status) atomicExch(a.device_status, (int)GKA_ERR_TIMEOUT);
        } else {
            // thread = (row c of dH and of dU, 32 columns)
            const int c = 32 * ((t >> 5) & 3) + l, cq = t >> 7;
            const uint32_t lane_addr = (uint32_t)(32 * ((t >> 5) & 3)) << 16;
            const size_t st = state_floats(D, D);
            float *dst = a.ws.delta + (size_t)item * st + (size_t)c * D + 32 * cq;
#pragma unroll
            for (int which = 0; which < 2; ++which) {
                if (which == 1 && a.solve_only) continue;        // the solve alone reads no U
                uint32_t r[32];
                TMEM_LD32(tmem + 128 * which + lane_addr + 32 * cq, r);
                tmem_wait_ld();
                float *p = dst + which * (size_t)D * D;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    *reinterpret_cast<float4 *>(p + 4 * i) = make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]),
                                                                         __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3]));
            }
            if (t == 0) a.ws.decay[item] = exp2f(total);
        }
    }
    fence_before();
    __syncthreads();
    if (s_abort != 0) drain(bars + 8 * SB_DRAIN, CT);
    if (t < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
}

// ------------------------------------------------------------------------------------------------------------
// State kernel.  A block walks the tiles of a work item in order.  Thread = (state row c, CW columns) of a master, which it keeps in
// registers in fp32 for a whole run.  The tensor cores compute only each tile's increments (dH = K~^T K~, dU = V~^T K~) into
// one of two TMEM buffers, one tile ahead of their use; per tile a thread stores the bf16 copies of its part of the tile-initial
// state (and adds up ||H_0||_F^2), then advances its master: H <- zeta H + dH.
//
// Who waits for whom.  One thread loads (TMA), factor warps turn the gates into row factors and a tile's decay several tiles ahead,
// scaling warps apply them to the rows in shared memory, one thread issues the products, the master warps copy and advance.  Every
// hand-over is an mbarrier per tile; nothing in the loop meets at a block barrier.
//
// What bounds it: device memory where a block has 64 KB of K and V per tile (268 MB at 64 x 4096 tokens), else how long the steps of a
// tile take one after another, so as many tiles as possible are worked on at once.  Every access to shared memory (a shuffle, a barrier, a
// load) waits 100 to 250 cycles behind the scaling warps' traffic, so accesses in a chain count more than instructions:
//   - a row factor is two bf16 terms and a product two instructions per pair of elements (scale_rows);
//   - the copies go straight from registers to global memory: in the workspace eight consecutive columns of a matrix's rows lie
//     together, so a warp's store is 512 consecutive bytes, and the solve kernel reads those bytes as a tensor-core operand without a
//     swizzle.  (Staged in shared memory over the tile's own K and V for a TMA store, a stage could not be loaded again before the
//     copies had been read from it);
//   - what a thread contributes to ||H_0||_F^2 is left in shared memory, and a factor warp adds it up tiles later;
//   - gates and write strengths are loaded a whole turn of the factor warps ahead and looked at only then.
// us per call of this kernel, before (one block-wide step after another, copies staged, head dimension 64 on 128 x 128 masters) and with
// this: 64 sequences x 4096 tokens 80 -> 60; 32 x 2048, solve alone (H only) 36 -> 18; 24 x 1999 with write strengths 61 -> 25 (their
// loads used to be waited for in the issuing warp); 64 x 2048, d = 64: 42 -> 20.
//
// KIND: what a block keeps.
//   kBoth     H and U (128 channels), where sequences are cut or the items alone fill the device
//   kOne      H or U: two blocks per item
//   kQuarter  64 columns of H or of U: four blocks per item
//   kD64      head dimension 64: H over U as one 128 x 64 master, [K V]^T K one product per k-step
//   kD64H     the same for the solve alone: H only.  The product keeps its 128 rows, the upper 64 of them made of zeros that lie behind the
//             stages (its A operand's second 64 columns are at a distance that the descriptor gives), and their master warps have nothing to do.
//             Whole call, before (as kD64 with K in V's place, its copies of U included) and with it: 32 x 2048, r = 30: 137.2 -> 134.7 us,
//             r = 0: 30.5 -> 28.0; 64 x 4096, r = 10: 196.4 -> 191.6; 256 x 1024: 191.7 -> 189.6
// H and U are made from the same rounded keys, whichever block makes them.  (The whole weight on K, and V as it is, halves the scaling of a
// block of U and brings U itself closer, 1.4e-3 against 2.0e-3, but the read U x meets an H of other keys: 4.9e-3 -> 5.7e-3 at 3 heads x
// 1999 tokens, 30 iterations.)  The solve alone keeps no U: no block of U is launched, kBoth skips it, kD64H has no room for it.
// ------------------------------------------------------------------------------------------------------------
enum { kBoth = 0, kOne = 1, kQuarter = 2, kD64 = 3, kD64H = 4 };
// Warps: those that keep the masters; groups that scale rows and take the tiles in turn; helpers (row factors, products, loads).  With 32 KB
// of K (and V) per tile six stages fit, and what counts is how many tiles are worked on at once: two groups of four warps.  With 64 KB
// (kBoth, kOne's blocks of U) three fit, so that a stage has to be given back soon: all sixteen warps scale a tile together, a tile ahead,
// and then keep its masters.  (With V left unscaled in the blocks of U: 64 x 4096 tokens, kOne: 54 us, 58 with a group of eight warps, 60
// with two of four; 32 x 4096, kQuarter: 42 us in one group of all warps, 35.4 with two.)
// Registers of a thread at launch (what its share of 65,536 allows) and after the split.
template <int KIND> struct StateKind {
    static constexpr bool kIs64 = KIND == kD64 || KIND == kD64H, kGroups = KIND == kQuarter || kIs64;
    static constexpr int kColumns = KIND == kBoth ? 256 : KIND == kOne ? 128 : 64;      // of all masters: TMEM columns of a buffer of increments
    static constexpr int kMasters = KIND == kBoth ? 2 : 1, kMasterWarps = kGroups ? 8 : 16;
    static constexpr int kKeepers = KIND == kD64H ? kMasterWarps / 2 : kMasterWarps;    // master warps that have rows to keep
    static constexpr int kCols = kColumns / kMasters / (kMasterWarps / 4);              // columns of a thread, of each master
    static constexpr int kGroupWarps = kGroups ? 4 : 16, kScaleGroups = kGroups ? 2 : 1;
    static constexpr int kFactorWarps = kGroups ? 4 : 2, kHelperWarps = kGroups ? 8 : 4;  // (whole warpgroups)
    static constexpr int kOtherWarps = (kGroups ? kGroupWarps * kScaleGroups : 0) + kHelperWarps, kThreads = 32 * (kMasterWarps + kOtherWarps);
    static constexpr int kRegsLaunch = kGroups ? 80 : 96, kRegsMaster = kGroups ? 112 : 104, kRegsOther = 64;
    static_assert(kHelperWarps >= kFactorWarps + 2 && kThreads * kRegsLaunch <= 65536 &&
                      32 * (kMasterWarps * kRegsMaster + kOtherWarps * kRegsOther) <= kThreads * kRegsLaunch,
                  "register split exceeds the launch allocation");
};
constexpr int kMaxStages = 6;
constexpr uint32_t kZeros = kMaxStages * 16384;          // kD64H: 16 KB of zeros behind the stages of 16 KB
static_assert(kZeros + 16384 + 1024 <= ST_SMEM, "shared memory of kD64H");
constexpr int kSets = kMaxStages + 2;      // sets of row factors, decays and norm terms
// A barrier of a kind for each of kRing consecutive tiles, whatever the number of stages: at least as many as stages, so that none is
// a phase ahead of a waiter; and even, so that the phases of one all belong to the same of two scaling groups.  (With three, a group met
// a barrier whose phase before had been the other group's: where that was not complete yet, the one before it had the same parity.)
constexpr int kRing = 6;
static_assert(kRing >= kMaxStages && kRing % 2 == 0, "ring of barriers");
enum {                            // mbarriers
    TB_KV = 0,                    // + tile % kRing: K and V have landed (TMA) and the tile's row factors and decay are ready (factor warp)
    TB_SC = TB_KV + kRing,        // + tile % kRing: rows scaled (one arrival per scaling warp)
    TB_D = TB_SC + kRing,         // + tile % kRing: the products are complete: increments for the masters, and the stage is free
    TB_AD = TB_D + kRing,         // + buffer: increments read (one arrival per master warp)
    TB_DRAIN = TB_AD + 2,
    TB_COUNT
};

template <int KIND>
__global__ void __launch_bounds__(StateKind<KIND>::kThreads, 1)
fwd_tc_state_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, FwdArgs a) {
    using SK = StateKind<KIND>;
    constexpr int CW = SK::kCols, NM = SK::kMasters;
    constexpr uint32_t DW = SK::kColumns;
    constexpr int MT = 32 * SK::kMasterWarps, CT = 32 * (SK::kMasterWarps + SK::kOtherWarps - SK::kHelperWarps);    // threads that keep masters; those that scale; the helpers
    constexpr int FT = CT + 32 * SK::kFactorWarps;                                 // helpers: factor warps, a warp for the products, one for the loads
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t s_bars[TB_COUNT];
    __shared__ __align__(16) uint2 s_f[kSets][NT];
    __shared__ __align__(16) float s_in[SK::kFactorWarps][2][NT];         // gates and write strengths on their way to their lanes
    __shared__ uint32_t s_tmem_base;
    __shared__ __align__(16) float s_sq[kSets][MT];          // the threads' terms of ||H_0||_F^2
    __shared__ float s_decay[kSets];
    __shared__ int s_abort;
    unsigned char *smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    const uint32_t sb = smem_u32(smem), bars = smem_u32(&s_bars[0]);
    const int t = threadIdx.x, l = t & 31;
    // The call's first kernel waits for whatever wrote its inputs (behind a summary or scan kernel only the summaries are
    // waited for, further down); the solve kernel is launched as a programmatic dependent of this one and reads inputs
    // before it waits, hence this order.
    if (!a.after_summary) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (t == 0) {
        s_abort = 0;
        for (int i = 0; i < TB_COUNT; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bars + 8 * i), "r"(i < TB_SC ? 2 : i < TB_D ? SK::kGroupWarps : i >= TB_AD && i < TB_DRAIN ? SK::kKeepers : 1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (t < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "n"(2 * DW)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if constexpr (KIND == kD64H) {
        for (int i = t; i < 1024; i += SK::kThreads) *reinterpret_cast<uint4 *>(smem + kZeros + 16 * i) = make_uint4(0u, 0u, 0u, 0u);
        for (int i = t; i < kSets * MT; i += SK::kThreads) (&s_sq[0][0])[i] = 0.f;         // (the terms of the warps without rows stay 0)
        fence_async_smem();
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem_base;
    const WorkPlan &P = a.plan;
    const int per_item = KIND == kOne || KIND == kQuarter ? (KIND == kQuarter ? 2 : 1) << (a.solve_only ? 0 : 1) : 1;
    const int item = (int)blockIdx.x / per_item, part = (int)blockIdx.x % per_item;
    const int half = KIND == kQuarter ? part & 1 : 0;                    // columns 64 half .. of the master
    const bool u_only = KIND == kQuarter ? part >> 1 : KIND == kOne ? part != 0 : false;
    const bool both = KIND == kBoth && !a.solve_only;
    // a stage: K (the part of it that is needed), then V
    const uint32_t v_off = KIND == kQuarter || KIND == kD64 ? 16384u : 32768u;
    const uint32_t stage_bytes = KIND == kD64H ? 16384u : KIND == kD64 ? 32768u : (both || u_only) ? v_off + 32768u : 32768u;
    const int ns = stage_bytes <= 32768u ? kMaxStages : stage_bytes == 49152u ? 4 : 3;
    const long long f_lo = P.lo(item);
    const int n_mine = (int)(P.lo(item + 1) - f_lo);
    float *const hh_out = u_only ? nullptr : half ? a.tile_hh2 : a.tile_hh;

    // position of tile m of this block
    struct Pos { int seq, n, b, h, ntok; size_t tok0; };
    auto pos_of = [&](int m) {
        Pos p;
        const unsigned fu = (unsigned)(f_lo + m);
        p.seq = (int)P.divN.div(fu);
        p.n = (int)(fu - (unsigned)p.seq * (unsigned)P.N);
        p.b = (int)a.divH.div((unsigned)p.seq);
        p.h = p.seq - p.b * a.heads;
        p.ntok = min(NT, a.T - p.n * NT);
        p.tok0 = ((size_t)p.b * a.T + (size_t)p.n * NT) * a.heads + p.h;
        return p;
    };
    auto aborted = [&]() { return *reinterpret_cast<volatile int *>(&s_abort) != 0; };
    auto give_up = [&]() { *reinterpret_cast<volatile int *>(&s_abort) = 1; };
    // Once a wait has given up the later ones return at once.  (A look at the flag takes as long as one at the barrier, so it comes
    // second: most of the compute warps' waits find their phase complete.)
    auto wait = [&](int which, uint32_t parity) {
        if (mbar_test(bars + 8 * which, parity) || aborted()) return;
        if (!(SK::kGroups ? mbar_wait_bounded(bars + 8 * which, parity) : mbar_spin_bounded(bars + 8 * which, parity))) give_up();
    };
    auto wait_asleep = [&](int which, uint32_t parity) {     // the same for waits that are long and have time
        if (!aborted() && !mbar_wait_bounded(bars + 8 * which, parity)) give_up();
    };
    // Barrier of tile n among the kRing of a kind, and the parity of its phase
    auto bar_of = [](int n) { return n % kRing; };
    auto phase_of = [](int n) { return (uint32_t)(n / kRing) & 1u; };

    // Rows of tile m, in stage `at`, scaled by the GT threads of a group
    constexpr int GT = 32 * SK::kGroupWarps;
    auto scale = [&](int m, int at, int ts) {
        wait(TB_KV + bar_of(m), phase_of(m));
        unsigned char *const stage = smem + (size_t)at * stage_bytes;
        const uint2 *const f = s_f[m % kSets];
        if constexpr (KIND == kD64H) {
#pragma unroll
            for (int i = 0; i < 2; ++i) scale_rows<4, GT, 1>(stage, f, ts + 4 * GT * i);
        } else if constexpr (SK::kGroups) {
#pragma unroll 2
            for (int i = 0; i < 4; ++i) {
                if (KIND == kQuarter && u_only) scale_rows<2, GT, 3>(stage, f, ts + 2 * GT * i);
                else scale_rows<2, GT, 2>(stage, f, ts + 2 * GT * i);
            }
        } else {
            scale_rows<2, GT, 2>(stage, f, ts);
            if (both || u_only) scale_rows<2, GT, 2>(stage + 32768, f, ts);
        }
        fence_async_smem();
        fence_before();
        __syncwarp();
        if (l == 0) mbar_arrive(bars + 8 * (TB_SC + bar_of(m)));
    };

    // (one instruction for all of a warpgroup, ahead of the roles)
    if (t >= MT) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(SK::kRegsOther));
        if (t >= FT + 32) {
            // ================================ TMA thread: loads of K and V ================================
            if (t == FT + 32) {
                for (int m = 0, stage = 0; m < n_mine; ++m, stage = stage + 1 == ns ? 0 : stage + 1) {
                    if (m >= ns) wait(TB_D + bar_of(m - ns), phase_of(m - ns));
                    if (aborted()) break;                // (a barrier whose copy never landed takes no second announcement)
                    const Pos p = pos_of(m);
                    const uint32_t dst = sb + (uint32_t)stage * stage_bytes, bar = bars + 8 * (TB_KV + bar_of(m));
                    const int x = p.h * a.d, y = p.n * NT;
                    mbar_expect_tx(bar, stage_bytes);
                    if constexpr (SK::kIs64) {
                        tma_load_box3(&tmK, dst, bar, x, y, p.b);
                        if (KIND == kD64) tma_load_box3(&tmV, dst + v_off, bar, x, y, p.b);
                    } else {
                        if (KIND == kQuarter && u_only) tma_load_box3(&tmK, dst, bar, x + 64 * half, y, p.b);
                        else tma_load_tile3(&tmK, dst, bar, x, x + 64, y, p.b);
                        if (both || u_only) tma_load_tile3(&tmV, dst + v_off, bar, x, x + 64, y, p.b);
                    }
                }
            }
        } else if (t >= CT && t < FT) {
            // ================ factor warps: row factors and decays, and the sums of ||H_0||_F^2 ================
            // Row factor of token j of a tile: the root of w_j = beta_j 2^(G_last - G_j); 0 past the sequence.  As two bf16 terms, for scale_rows.
            // The warps take the tiles in turn: a tile's scan, logarithms and sums are a chain of some 4000 cycles beside the warps that scale,
            // several times as long as a tile.  Before it publishes, tile f waits until the products of tile f - ns are complete: the phase
            // before its own of the barrier is then complete, and the masters are past tile f - ns - 2 (the products of a
            // tile are issued when the increments of the tile two before have been read), so with kSets >= ns + 2 sets none is written
            // over that is still to be read.
            struct Scalars { float g[4], b[4]; };
            auto load_scalars = [&](int m, Scalars &x) {         // (taken as they are: nothing here may wait for a load)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    x.g[i] = 1.f;
                    x.b[i] = 0.f;
                }
                if (m >= n_mine) return;
                const Pos p = pos_of(m);
                const size_t at = p.tok0 + (size_t)l * a.heads;
                const float *const gp = a.gate + at, *const bp = a.beta ? a.beta + at : nullptr;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (32 * i + l < p.ntok) {
                        x.g[i] = ld_stream_f32(gp + 32 * i * a.heads);
                        x.b[i] = bp ? ld_stream_f32(bp + 32 * i * a.heads) : 1.f;
                    }
            };
            const int f0 = (t - CT) >> 5;
            auto factors = [&](int f, Scalars &x) {
                // Loaded with lane l at tokens l, 32 + l, 64 + l, 96 + l (with four consecutive tokens per lane a load touches four times as
                // wide a piece of memory: 64 x 4096 tokens 54 -> 60 us), used with tokens 4 l .. 4 l + 3.
                float factor[4], incl[4], run = 0.f;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    s_in[f0][0][32 * i + l] = x.g[i];
                    s_in[f0][1][32 * i + l] = x.b[i];
                }
                __syncwarp();
                const float4 g4 = *reinterpret_cast<const float4 *>(&s_in[f0][0][4 * l]), b4 = *reinterpret_cast<const float4 *>(&s_in[f0][1][4 * l]);
                __syncwarp();
                x = Scalars{{g4.x, g4.y, g4.z, g4.w}, {b4.x, b4.y, b4.z, b4.w}};
#pragma unroll
                for (int i = 0; i < 4; ++i) incl[i] = run += fmaxf(log2f(x.g[i]), -115.f);
                float before = run;                              // of the lanes up to this one, then of those before it
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float up = __shfl_up_sync(0xffffffffu, before, o);
                    before += l >= o ? up : 0.f;
                }
                const float total = __shfl_sync(0xffffffffu, before, 31);
                before = total - (before - run);                 // decay from the start of this lane's tokens to the tile's end
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float e = before - incl[i];
                    factor[i] = exp2f(0.5f * e);
                }
                if (a.beta) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float w = fmaxf(x.b[i], 0.f);
                        factor[i] *= sqrtf(w);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) factor[i] *= x.b[i];      // 1, or 0 past the sequence
                }
                load_scalars(f + SK::kFactorWarps, x);
                if (f >= ns) {
                    wait_asleep(TB_D + bar_of(f - ns), phase_of(f - ns));
                    if (f < 2 * kSets) asm volatile("griddepcontrol.wait;" ::: "memory");
                    if (f >= kSets && hh_out) {                  // tile f - kSets
                        const float4 *p = reinterpret_cast<const float4 *>(s_sq[f % kSets]) + l;
                        float hh = 0.f;
#pragma unroll
                        for (int i = 0; i < MT / 128; ++i) hh += (p[32 * i].x + p[32 * i].y) + (p[32 * i].z + p[32 * i].w);
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) hh += __shfl_xor_sync(0xffffffffu, hh, o);
                        if (l == 0) hh_out[f_lo + f - kSets] = hh;
                    }
                }
                const uint2 w0 = split_factor(factor[0]), w1 = split_factor(factor[1]), w2 = split_factor(factor[2]), w3 = split_factor(factor[3]);
                uint4 *const set = reinterpret_cast<uint4 *>(&s_f[f % kSets][4 * l]);
                set[0] = make_uint4(w0.x, w0.y, w1.x, w1.y);
                set[1] = make_uint4(w2.x, w2.y, w3.x, w3.y);
                if (l == 0) s_decay[f % kSets] = exp2f(total);
                __syncwarp();
                if (l == 0) mbar_arrive(bars + 8 * (TB_KV + bar_of(f)));
            };
            Scalars x;                                           // (of the warp's next tile, in flight)
            load_scalars(f0, x);
            for (int f = f0; f < n_mine; f += SK::kFactorWarps) factors(f, x);
        } else if (t >= FT) {
            // ================================ MMA issuing thread ================================
            if (l == 0) {
                constexpr uint32_t idesc = DW == 64 ? make_idesc(128, 64, 1, 1) : kIdescMM;
                const uint32_t base14 = (sb >> 4) & 0x3FFF;
                for (int m = 0, stage = 0; m < n_mine; ++m, stage = stage + 1 == ns ? 0 : stage + 1) {
                    const uint32_t ph = phase_of(m), ph_ad = ((uint32_t)(m >> 1) & 1u) ^ 1u;      // of tile m - 2's (the phase before a barrier's first one counts as complete)
                    const bool sc = mbar_test(bars + 8 * (TB_SC + bar_of(m)), ph), ad = !SK::kGroups || mbar_test(bars + 8 * (TB_AD + (m & 1)), ph_ad);
                    if (!sc) wait(TB_SC + bar_of(m), ph);
                    if (!ad) wait(TB_AD + (m & 1), ph_ad);
                    if (!(sc && ad) && aborted()) break;
                    fence_after();
                    const uint32_t kb = base14 + (uint32_t)stage * (stage_bytes >> 4), vb = kb + (v_off >> 4);
                    const uint32_t tm_d = tmem + DW * (uint32_t)(m & 1);
                    // (kD64H: the second half of A's columns from the zeros instead of 16384 bytes on; the distance stands in bits 16 to 29)
                    const uint32_t ka = KIND == kD64H ? kb + (((kZeros - 16384u - (uint32_t)stage * stage_bytes) >> 4) << 16) : kb;
                    if (!u_only) mma8_mm<0>(tm_d, ka, kb + (16384u >> 4) * half, idesc);           // dH = K~^T K~ (kD64: [K~ V~]^T K~)
                    if (both || u_only) mma8_mm<0>(tm_d + (NM - 1) * 128, vb, kb, idesc);          // dU = V~^T K~
                    mma_commit(bars + 8 * (TB_D + bar_of(m)));
                }
            }
        } else if constexpr (SK::kGroups) {
            // ================================ scaling groups ================================
            const int ts = (t - MT) % GT;
            for (int m = (t - MT) / GT, at = m; m < n_mine; m += SK::kScaleGroups) {
                scale(m, at, ts);
                at += SK::kScaleGroups;
                if (at >= ns) at -= ns;
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(SK::kRegsMaster));
        // ================================ masters ================================
        const int q = (t >> 5) & 3, cq = t >> 7, c = 32 * q + l, col0 = 64 * half + CW * cq;     // row, first column
        const uint32_t tm_c = tmem + ((uint32_t)(32 * q) << 16) + CW * cq;
        const int which0 = SK::kIs64 ? c >> 6 : u_only ? 1 : 0;              // matrix of the (first) master, and the row in it
        const int row = SK::kIs64 ? c & 63 : c;
        constexpr int DD = SK::kIs64 ? 64 : D;                               // head dimension of the caller's states
        const int n_keep = KIND == kD64H && q >= 2 ? 0 : n_mine;             // tiles that this warp has rows of
        const size_t ext = (size_t)2 * DD * DD;                              // floats of a caller's state
        const size_t e_ext = (size_t)which0 * DD * DD + (size_t)row * DD + col0;
        const size_t st = state_floats(D, D), e_ws = (size_t)which0 * D * D + (size_t)row * D + col0;    // the workspace's states are 128 x 128
        const bool sums = SK::kIs64 ? q < 2 : !u_only;                       // this warp's rows belong to H
        // the copies: [H, U][column / 8][row][8 columns], 64 KB per tile, 16 KB at head dimension 64
        unsigned char *copy = a.tile_hu + (size_t)f_lo * (SK::kIs64 ? kTileStateBytes64 : kTileStateBytes) +
                              which0 * (2 * DD * DD) + (col0 / 8) * (16 * DD) + row * 16;
        // first item of the chain of summaries behind this block's start state
        int chain_j0 = item;
        if ((KIND == kBoth || SK::kIs64) && P.cut_in(item)) {
            const long long seq_start = (f_lo / P.N) * P.N;
            chain_j0 = item - 1;
            while (P.lo(chain_j0) > seq_start) --chain_j0;
        }
        uint64_t mst[NM][CW / 2];
        int seq, n;
        {
            const Pos p0 = pos_of(0);
            seq = p0.seq;
            n = p0.n;
        }
        if (!SK::kGroups && n_mine > 0) scale(0, 0, t);
        // summaries and start states are read, and copies written, after this point only
        asm volatile("griddepcontrol.wait;" ::: "memory");

        for (int m = 0, at = 1; m < n_keep; ++m) {
            if constexpr (!SK::kGroups) {                        // the next tile's rows: its products run under this tile's passes
                if (m + 1 < n_mine) scale(m + 1, at, t);
                if (++at == ns) at = 0;
            }
            if (m == 0 || n == 0) {
                // start of a run: the caller's initial state of the sequence (or zero), carried through the summaries
                // of the blocks that hold the earlier part of the sequence: state <- decay_j * state + delta_j
                const bool chained = (KIND == kBoth || SK::kIs64) && n != 0;
                const bool scanned = chained && a.start_from_scan;
                const float *const s0 = scanned ? a.ws.start + (size_t)item * st + e_ws : a.state_in ? a.state_in + (size_t)seq * ext + e_ext : nullptr;
                const int j0 = chained && !scanned ? chain_j0 : 0, j1 = chained && !scanned ? item : 0;
#pragma unroll
                for (int w = 0; w < NM; ++w) {
#pragma unroll
                    for (int i = 0; i < CW / 4; ++i) {
                        ulonglong2 v = make_ulonglong2(0ull, 0ull);
                        if (s0 && (w == 0 || both)) v = *reinterpret_cast<const ulonglong2 *>(s0 + w * D * D + 4 * i);      // (the solve alone: nobody has written U's)
                        mst[w][2 * i] = v.x;
                        mst[w][2 * i + 1] = v.y;
                    }
                    for (int j = j0; j < j1 && (w == 0 || both); ++j) {
                        // summaries come from the kernel this one may overlap with as its programmatic dependent: ordinary loads
                        const float dj = *reinterpret_cast<const volatile float *>(a.ws.decay + j);
                        const uint64_t dj2 = f2_pack(dj, dj);
                        const float *const dd = a.ws.delta + (size_t)j * st + e_ws + w * D * D;
#pragma unroll
                        for (int i = 0; i < CW / 4; ++i) {
                            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(dd + 4 * i);
                            mst[w][2 * i] = f2_fma(dj2, mst[w][2 * i], v.x);
                            mst[w][2 * i + 1] = f2_fma(dj2, mst[w][2 * i + 1], v.y);
                        }
                    }
                }
            }
            // ---- the increments on their way (their products ran under the tile before), the bf16 copies of the tile-initial state
            // and the thread's term of ||H_0||_F^2, then the masters advanced: zeta m + increment
            wait(TB_D + bar_of(m), phase_of(m));
            fence_after();
            const float decay = s_decay[m % kSets];
            const uint64_t decay2 = f2_pack(decay, decay);
            uint64_t sq = 0ull;
            constexpr int PW = NM == 1 ? 32 : 16;                // columns at a time
#pragma unroll
            for (int w = 0; w < NM; ++w) {
                if (w == 1 && !both) continue;
#pragma unroll
                for (int c0 = 0; c0 < CW; c0 += PW) {
                    uint32_t x[PW];
                    if constexpr (PW == 32) TMEM_LD32(tm_c + DW * (m & 1) + c0, x);
                    else TMEM_LD16(tm_c + DW * (m & 1) + 128 * w + c0, x);
#pragma unroll
                    for (int i = 0; i < PW / 8; ++i) {
                        uint32_t pk[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const uint64_t v = mst[w][c0 / 2 + 4 * i + u];
                            float v0, v1;
                            f2_unpack(v, v0, v1);
                            pk[u] = pack_bf16(v0, v1);
                            if (w == 0) sq = f2_fma(v, v, sq);
                        }
                        *reinterpret_cast<uint4 *>(copy + w * 32768 + 16 * DD * (c0 / 8 + i)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    }
                    if (w == 0 && c0 + PW == CW) {
                        float a0, a1;
                        f2_unpack(sq, a0, a1);
                        s_sq[m % kSets][t] = sums ? a0 + a1 : 0.f;
                    }
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < PW / 2; ++i)
                        mst[w][c0 / 2 + i] = f2_fma(decay2, mst[w][c0 / 2 + i], f2_pack(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1])));
                }
            }
            if constexpr (SK::kGroups) {                         // (else the warp's next arrival with scaled rows says the same)
                fence_before();
                __syncwarp();
                if (l == 0) mbar_arrive(bars + 8 * (TB_AD + (m & 1)));
            }
            copy += SK::kIs64 ? kTileStateBytes64 : kTileStateBytes;
            // ---- final state of the sequence, in the caller's layout
            if (++n == P.N) {
                if (a.state_out) {
                    float *const so = a.state_out + (size_t)seq * ext + e_ext;
#pragma unroll
                    for (int w = 0; w < NM; ++w)
#pragma unroll
                        for (int i = 0; i < CW / 4; ++i)
                            *reinterpret_cast<ulonglong2 *>(so + w * D * D + 4 * i) = make_ulonglong2(mst[w][2 * i], mst[w][2 * i + 1]);
                }
                n = 0;
                ++seq;
            }
        }
    }
    fence_before();
    __syncthreads();
    if (t < 32 * kSets && hh_out) {
        const int m = n_mine - kSets + (t >> 5);             // (tiles before the last ones: the factor warps)
        if (m >= 0) {
            float hh = 0.f;
#pragma unroll
            for (int i = 0; i < MT / 32; ++i) hh += s_sq[m % kSets][32 * i + l];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) hh += __shfl_xor_sync(0xffffffffu, hh, o);
            if (l == 0) hh_out[f_lo + m] = hh;
        }
    }
    if (t == 0) {
        if (s_abort != 0 && a.device_status) atomicExch(a.device_status, (int)GKA_ERR_TIMEOUT);
    }
    if (s_abort != 0) drain(bars + 8 * TB_DRAIN, FT);
    if (t < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(2 * DW) : "memory");
}

// (cfg: all but the block size and the shared memory, which belong to the kind)
template <int KIND>
cudaError_t launch_state(cudaLaunchConfig_t cfg, const CUtensorMap &tmK, const CUtensorMap &tmV, const FwdArgs &a) {
    static SmemLimit limit;
    const cudaError_t err = limit.raise(fwd_tc_state_kernel<KIND>, (int)ST_SMEM);
    if (err != cudaSuccess) return err;
    cfg.blockDim = dim3(StateKind<KIND>::kThreads);
    cfg.dynamicSmemBytes = ST_SMEM;
    return cudaLaunchKernelEx(&cfg, fwd_tc_state_kernel<KIND>, tmK, tmV, a);
}

// Scan over work items: the start state of item i (when its range starts inside a sequence) is the
// fold  state <- decay_j * state + delta_j  over the items j < i that hold the earlier part of the
// same sequence, starting from the sequence's initial state.  A sequence spans few items, so every
// item folds its own short chain independently: blockIdx.y = item, four state elements per thread.
__global__ void fwd_scan(FwdArgs a) {
    // programmatic dependent of the summary kernel, and the state kernel one of this kernel: both may be scheduled early,
    // and each waits here for its producer
    constexpr int st = 2 * D * D;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const WorkPlan &P = a.plan;
    const int i = blockIdx.y + 1;
    __shared__ int s_j0, s_seq;           // the chain is found once per block (64-bit divisions are slow)
    if (threadIdx.x == 0) {
        int j0 = -1;
        if (P.cut_in(i)) {
            // first item of the chain: the one whose range holds the start of this sequence (its last run
            // begins there, whatever sequence the item itself started in)
            const long long seq_start = (P.lo(i) / P.N) * P.N;
            j0 = i - 1;
            while (P.lo(j0) > seq_start) --j0;
        }
        s_j0 = j0;
        s_seq = (int)(P.lo(i) / P.N);
    }
    __syncthreads();
    const int j0 = s_j0, seq = s_seq;
    if (j0 < 0) return;
    const int e = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (e >= st) return;
    float4 carry = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.state_in) {
        const int dd = 2 * a.d * a.d;
        if (dd == st) {
            carry = *reinterpret_cast<const float4 *>(a.state_in + (size_t)seq * st + e);
        } else {
            // the workspace holds states zero-extended to the on-chip head dimension
            const int which = e / (D * D), row = (e / D) % D, col = e % D;
            if (row < a.d && col < a.d) carry = *reinterpret_cast<const float4 *>(a.state_in + (size_t)seq * dd + (size_t)which * a.d * a.d + (size_t)row * a.d + col);
        }
    }
    for (int j = j0; j < i; ++j) {
        const float dcy = a.ws.decay[j];
        const float4 d = *reinterpret_cast<const float4 *>(a.ws.delta + (size_t)j * st + e);
        carry.x = fmaf(dcy, carry.x, d.x);
        carry.y = fmaf(dcy, carry.y, d.y);
        carry.z = fmaf(dcy, carry.z, d.z);
        carry.w = fmaf(dcy, carry.w, d.w);
    }
    *reinterpret_cast<float4 *>(a.ws.start + (size_t)i * st + e) = carry;
}

}  // namespace

bool fwd_tc_available() { return get_encode_fn() != nullptr; }

cudaError_t launch_fwd_tc(const FwdArgs &a_in, cudaStream_t stream) {
    FwdArgs a = a_in;
    cudaError_t err = cudaSuccess;
    bool any_cut = false;
    int longest = 0;                   // most summaries behind any item's start state
    for (int i = 0; i + 1 < a.plan.G; ++i) any_cut |= a.plan.cut_out(i);
    for (int i = 1; i < a.plan.G && any_cut; ++i) {
        if (!a.plan.cut_in(i)) continue;
        const long long seq_start = (a.plan.lo(i) / a.plan.N) * a.plan.N;
        int j0 = i - 1;
        while (a.plan.lo(j0) > seq_start) --j0;
        longest = (i - j0) > longest ? (i - j0) : longest;
    }
    // Short chains are folded by the state kernel's blocks themselves; long ones (a sequence spread over many
    // work items) would make every block re-read its whole chain, so the scan kernel materialises the start
    // states once instead.
    a.start_from_scan = longest > 4 ? 1 : 0;
    // Blocks per work item (the kernel's KIND): one with both masters where a sequence is cut, else one per master, or one per 64
    // columns of a master, as long as those fit one per SM.  The solve alone has no blocks for U.
    const int masters = a.solve_only ? 1 : 2;
    int kind = kBoth, per_item = 1;
    if (a.d == 64) {
        kind = a.solve_only ? kD64H : kD64;
    } else if (!any_cut && masters * a.plan.G <= a.sms) {
        kind = kOne;
        per_item = masters;
        // the second half of ||H_0||_F^2 goes to the summaries' place, which nothing else uses when no sequence is cut
        if (2 * masters * a.plan.G <= a.sms && a.plan.NC <= (long long)a.plan.G * (long long)state_floats(D, D)) {
            kind = kQuarter;
            per_item = 2 * masters;
            a.tile_hh2 = a.ws.delta;
        }
    }
    alignas(64) CUtensorMap tmK, tmV;           // boxes of 128 tokens x 64 channels
    const int cols = a.heads * a.d;
    if (!make_tile_map(&tmK, a.k, a.B, a.T, cols, NT) || !make_tile_map(&tmV, a.v, a.B, a.T, cols, NT))
        return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.stream = stream;
    static SmemLimit summary_limit;
    if (any_cut) {
        if ((err = summary_limit.raise(fwd_tc_summary_kernel, (int)KV_SMEM)) != cudaSuccess) return err;
        cfg.gridDim = dim3((unsigned)a.plan.G);
        cfg.blockDim = dim3(kThreadsState);
        cfg.dynamicSmemBytes = KV_SMEM;
        if ((err = cudaLaunchKernelEx(&cfg, fwd_tc_summary_kernel, tmK, tmV, a)) != cudaSuccess) return err;
        if (a.start_from_scan) {
            cfg.gridDim = dim3((a.solve_only ? 1 : 2) * D * D / 4 / 256, (unsigned)(a.plan.G - 1));
            cfg.blockDim = dim3(256);
            cfg.dynamicSmemBytes = 0;
            if ((err = cudaLaunchKernelEx(&cfg, fwd_scan, a)) != cudaSuccess) return err;
        }
        a.after_summary = 1;
    }
    cfg.gridDim = dim3((unsigned)(a.plan.G * per_item));
    err = kind == kD64H ? launch_state<kD64H>(cfg, tmK, tmV, a) : kind == kD64 ? launch_state<kD64>(cfg, tmK, tmV, a) : kind == kQuarter ? launch_state<kQuarter>(cfg, tmK, tmV, a)
          : kind == kOne ? launch_state<kOne>(cfg, tmK, tmV, a) : launch_state<kBoth>(cfg, tmK, tmV, a);
    if (err != cudaSuccess) return err;
    return launch_fwd_solve(a, stream);
}

}  // namespace gka
