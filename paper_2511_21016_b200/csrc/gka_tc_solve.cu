// tcgen05 / TMEM solve kernel of the chunk-wise GKA forward (bf16 operands, fp32 accumulation) for sm_100a.
//
// Input: for every tile of 128 consecutive tokens of a sequence, the bf16 copies of the tile-initial states
// H_0, U_0 and ||H_0||_F^2 (written by the state kernel, gka_tc_state.cu).  Tiles are independent problems.  One
// persistent thread block per SM keeps two tiles ("slots") in flight and runs them in opposite phases: while the
// tensor pipe works on the products of one slot, the CUDA cores run the fp32 update of the other.  A tile puts one
// token on each TMEM lane; every product of the chunk-wise form (Section 4.2.1; Algorithm 1 on the whole tile) is
// an M = 128 tile.
//
// Algorithm 1 in residual form.  With d_i = x_i - x_{i-1} (x_{-1} = 0, d_0 = x_0 = 2 q / (L + mu)) the update
// x_{i+1} = x_i + (omega_{i+1} - 1) d_i + (2 omega_{i+1} / (L + mu)) (q - A x_i) reads
//     r_i = r_{i-1} - A d_i  (r_{-1} = q),     d_{i+1} = beta d_i + sigma r_i,     x_{i+1} = x_i + d_{i+1},
// the same iterates in exact arithmetic.  The matrix is applied to the increment d_i, so the bf16 rounding of the
// tensor-core operand is relative to the (shrinking) increment and the iterate itself stays in fp32; the value
// added to x is the rounded operand, which keeps x and the residual consistent.  Per token c of the tile
//     A d = zeta_c H_0 d + sum_{j<=c} Gamma[c][j] k_j (k_j . d) + lambda_c d,     Gamma[c][j] = 2^(G_c - G_j),
// G the cumulative log2 gate in the tile.  The operand is E = -zt_c d_c in bf16 (zt_c = max(zeta_c, 2^-60)), the
// keys are staged as Khat_j = sqrt(beta_j) 2^(-G_j / 2) k_j, and the accumulator R starts as q:
//     S = E Khat^T,   P = S masked to j <= c (packed bf16, written over S in TMEM),   R += E H_0^T + P Khat
// leaves R = q - (A - lambda) x_i with no factor anywhere in the masked-score epilogue; the lambda term uses the
// fp32 iterate.  Tiles whose decay falls below 2^-60 keep unscaled keys and per-element factors instead.
// The read o_c = zeta_c U_0 x_c + sum_{j<=c} Gamma[c][j] v_j (k_j . x_c) uses the final iterate split into two
// bf16 terms (x is dominated by directions that U barely reads; a single bf16 rounding of x would swamp the rest).
// Chunk-wise Frobenius norms of Section 4.2.1 come from Khat H_0, the Gram matrix Khat Khat^T and an affine scan.
//
// On-chip layout.  Tensor memory (512 columns): one score tile S shared by the two slots (only one slot at a time
// is between its score product and the product that consumes the masked scores: the issuing thread hands S from
// slot to slot, which is also what keeps the slots in opposite phases), and per slot the fp32 accumulator R (128
// columns) and the operand E as packed bf16 (64 columns).  E and P feed the products from tensor memory, so a
// product reads only its B operand (keys, H_0, U_0, values) from shared memory and leaves half of the shared-memory
// bandwidth to everything else.  Shared memory per slot: keys, H_0 (later U_0), q (later V, then the result).
//
// Warp roles: 4 compute warps per slot, a thread owns one token (one TMEM lane) and all 128 channels of its iterate in
// registers, and masks its own scores; one warp prepares the gate scalars one tile ahead; one thread per slot issues that
// slot's TMA stores and the loads that follow them; one thread issues every tcgen05.mma for both slots.  Requests to the
// issuing thread are counters in shared memory (one count per warp), completion comes back through tcgen05.commit mbarriers.
// What bounds the iterations is the turn of a slot on the score tile (score product, epilogue, second product), and in it how
// fast a warp that has been woken gets through its instructions: what the warps of a block execute per iteration does not fit
// the first-level instruction cache, so the number of instructions between two hand-overs counts more than their kind.
// Hence the increment is added to the iterate when it is next unpacked, the diagonal block is masked after the conversion,
// and there are no separate warps for the scores (as a third party they had to be told whose scores come next, started
// cold, and shared every scheduler with two update warps).  B = 4, 16 heads, T = 4096, 10 / 30 iterations, both builds in turn, 20
// calls back to back: 406 / 827 us per call before, 354 / 736 with these (413 and 370 at 10 iterations over seconds of
// calls, where the power cap sets the clock).
//
// Head dimension 64 arrives zero-extended to 128 channels (the upper TMA box reads zeros).  The kernel instantiated
// with HALF leaves out what the zero channels would contribute: contractions over the channels take four k-steps
// instead of eight, products into R have 64 columns, and the passes of the compute warps stop at channel 64.  R and E then
// take half of their columns, which leaves room for a score tile per slot: nothing is handed from slot to slot, so a slot is
// one chain of its four compute warps, and one of their threads issues the slot's products (no issuing thread: a request no
// longer waits for a thread that serves both slots).  B = 4, 16 heads, T = 2048, 10 / 30 iterations: 177 / 351 us per call with
// the shared score tile, 152 / 288 with this (121 at 10 with the present state kernel).  Two threads per token, each with half of the
// channels and every other key block, measured slower (117.4 -> 120.4).
#include <cuda.h>

#include "gka_common.cuh"
#include "gka_tc_mma.cuh"

namespace gka {
namespace {

using namespace tcu;

constexpr int NT = kTile;                  // tokens per tile: one per TMEM lane
constexpr int kSlots = 2;
constexpr int ST = 128;                    // compute threads per slot
constexpr int CT = kSlots * ST;            // compute threads
// Warpgroups: 0 = helpers (gate scalars, TMA: one warp per slot, MMA issue), 1 and 2 = the compute warps of slot 0 and slot 1.
constexpr int kThreadsSolve = 128 + CT;
// register split after setmaxnreg (128 channels): with 216 / 72 the compute threads spilled 32 bytes (64 x 4096 tokens, 10 iterations: 299 -> 295 us)
constexpr int kRegsLaunch = 168, kRegsCompute = 224, kRegsHelper = 56;
static_assert(kThreadsSolve * kRegsLaunch <= 65536, "launch registers");
static_assert(CT * kRegsCompute + 128 * kRegsHelper <= kThreadsSolve * kRegsLaunch, "register split exceeds the launch allocation");

// ---- shared memory map (bytes; operand buffers 1024-byte aligned): three operand tiles per slot, then the scalars
constexpr uint32_t BUF_A = 0;                  // keys (Khat)
constexpr uint32_t BUF_B = kTileBytes;         // bf16 H_0, later U_0
constexpr uint32_t BUF_C = 2 * kTileBytes;     // q, later V, then the result tile
constexpr uint32_t SLOT_BYTES = 3 * kTileBytes;
constexpr uint32_t OFF_SC = kSlots * SLOT_BYTES;

struct GateScalars {       // per token of a tile, from the gates and the other per-token inputs alone
    float lg[NT];          // log2 gamma_c
    float G2[NT];          // cumulative log2 gate
    float ac[NT];          // G2_c - max(G2_c, -60): exponent correction of clamped tokens
    float zt[NT];          // clamped zeta_c
    float iz[NT];          // 1 / zt_c
    float lam[NT];         // lambda_c as given
    float al[NT];          // alpha_c (alpha-connection)
    float ks[NT];          // row factor of the staged keys: sqrt(beta_j) 2^(-G_j / 2), or sqrt(beta_j) alone when the tile decays below 2^-60
};
struct SlotScalars {
    GateScalars g[2];
    float carry[2][4];     // per-warp totals (a, b) of the affine scan
};
constexpr uint32_t SC_BYTES = (sizeof(SlotScalars) + 127) / 128 * 128;
constexpr uint32_t SOLVE_SMEM = OFF_SC + kSlots * SC_BYTES + 1024;   // + slack for the 1024-byte alignment of the base
static_assert(SOLVE_SMEM + 4096 <= 232448, "shared memory budget");

// ---- TMEM columns: shared score accumulator S (P overwrites it in place); per slot the residual / output
// accumulator R and the bf16 operand E
// (128 channels), or, with head dimension 64, where R and E take half of the columns, a score tile per slot
__host__ __device__ constexpr uint32_t tm_s_of(bool half, int s) { return half ? 128u * (uint32_t)s : 0u; }
__host__ __device__ constexpr uint32_t tm_r_of(bool half, int s) { return half ? 256u + 64u * (uint32_t)s : 128u + 128u * (uint32_t)s; }
__host__ __device__ constexpr uint32_t tm_e_of(int s) { return 384u + 64u * (uint32_t)s; }
// products whose result goes to R have as many columns as there are channels
__host__ __device__ constexpr uint32_t idesc_r_kk(bool half) { return make_idesc(128, half ? 64 : 128, 0, 0); }
__host__ __device__ constexpr uint32_t idesc_r_pm(bool half) { return make_idesc(128, half ? 64 : 128, 0, 1); }

enum {                 // per slot
    B_LD_K = 0,        // K tile has landed (TMA)
    B_LD_H,            // H_0 tile
    B_LD_Q,            // q tile
    B_LD_U,            // U_0 tile
    B_LD_V,            // V tile
    B_RDY_ST,          // compute warps -> TMA thread: the result tile is staged
    B_QF,              // compute warps -> TMA thread: q has been read, V may take its buffer
    B_MMA_S,           // tcgen05.commit: the Frobenius batch (Gram matrix, K H_0) is complete
    B_MMA_R,           // tcgen05.commit: accumulator-side batch complete
    B_GS0, B_GS1,      // gate scalars of buffer 0 / 1 are ready
    B_GF0, B_GF1,      // compute warps -> gate helper: buffer 0 / 1 is free
    B_PER_SLOT
};
constexpr int B_DRAIN = kSlots * B_PER_SLOT;   // every product is complete (before the tensor memory is given back)
constexpr int B_SC = B_DRAIN + 1;              // + slot: tcgen05.commit, a score product of the slot is complete
constexpr int B_COUNT = B_SC + kSlots;

// Requests a slot makes to the issuing thread: every warp of the slot adds one to the slot's request counter in
// shared memory (a poll of both counters is one 40-cycle load, where a test of an mbarrier phase takes 100 cycles);
// request n of a slot is ready when its counter has reached 4 (n + 1).  In this order per tile:
// FROB, then n_iter times (ITER1, ITER2), then (unless the solve itself is the result) OUT_S, OUT_O
enum { OP_FROB = 0, OP_ITER1, OP_ITER2, OP_OUT_S, OP_OUT_O };

__device__ __forceinline__ bool aborted(uint32_t abort_addr) {
    int v;
    asm volatile("ld.volatile.shared.b32 %0, [%1];" : "=r"(v) : "r"(abort_addr) : "memory");
    return v != 0;
}
__device__ __forceinline__ void set_abort(uint32_t abort_addr) {
    asm volatile("st.volatile.shared.b32 [%0], %1;" ::"r"(abort_addr), "r"(1) : "memory");
}
// Bounded wait (about a second; the wait suspends in hardware between polls); once any wait of the block has given up
// every later wait returns at once, so the block runs to its end without further delays and reports
// GKA_ERR_TIMEOUT.  One compact loop in a single asm block: the wait is inlined at some thirty places.
__device__ __forceinline__ void wait_bar(uint32_t bar, uint32_t parity, uint32_t abort_addr) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .u32 n, ab;\n\t"
        "mov.u32 n, 0;\n\t"
        "ld.volatile.shared.b32 ab, [%4];\n\t"
        "setp.ne.u32 p, ab, 0;\n\t"
        "@p bra WAIT_DONE;\n"
        "WAIT_LOOP:\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "@p bra WAIT_DONE;\n\t"
        "add.u32 n, n, 1;\n\t"
        "setp.lt.u32 q, n, 200000;\n\t"
        "@q bra WAIT_LOOP;\n"
        "WAIT_DONE:\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(5000u), "r"(abort_addr)
        : "memory");
    if (!ok) set_abort(abort_addr);
}
// one count per warp on a shared-memory counter, after every lane's writes and fences (release)
__device__ __forceinline__ void warp_post(uint32_t addr, int lane) {
    __syncwarp();
    if (lane == 0) asm volatile("red.release.cta.shared::cta.add.u32 [%0], 1;" ::"r"(addr) : "memory");
}
// The same where the warp has written tensor memory only: tcgen05.wait::st and tcgen05.fence::before_thread_sync order that
// for the thread that issues the products, and the count itself need not wait for anything else.
__device__ __forceinline__ void warp_post_tmem(uint32_t addr, int lane) {
    __syncwarp();
    if (lane == 0) asm volatile("red.relaxed.cta.shared::cta.add.u32 [%0], 1;" ::"r"(addr) : "memory");
}
// one arrival per warp, after every lane's writes and fences
__device__ __forceinline__ void warp_arrive(uint32_t bar, int lane) {
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
}

struct TileInfo {
    int seq, n, b, h, ntok;
    size_t tok0;
};
__device__ __forceinline__ TileInfo tile_info(const FwdArgs &a, long long tile) {
    TileInfo t;
    const unsigned fu = (unsigned)tile;
    t.seq = (int)a.plan.divN.div(fu);
    t.n = (int)(fu - (unsigned)t.seq * (unsigned)a.plan.N);
    t.b = (int)a.divH.div((unsigned)t.seq);
    t.h = t.seq - t.b * a.heads;
    t.ntok = min(NT, a.T - t.n * NT);
    t.tok0 = ((size_t)t.b * a.T + (size_t)t.n * NT) * a.heads + t.h;
    return t;
}

// H_0 of a tile; head dimension 64: and U_0 behind it, which nobody has written for the solve alone
template <bool HALF>
__device__ __forceinline__ void load_h0(const FwdArgs &a, long long tile, uint32_t dst, uint32_t bar, bool h_only) {
    const uint32_t bytes = !HALF ? 32768u : h_only ? (uint32_t)kTileStateBytes64 / 2 : (uint32_t)kTileStateBytes64;
    mbar_expect_tx(bar, bytes);
    bulk_load(dst, a.tile_hu + (size_t)tile * (HALF ? kTileStateBytes64 : kTileStateBytes), bytes, bar);
}

// Products of the issuing thread: 8 k-steps of 16 each, unrolled with immediate descriptor offsets: every instruction
// of the issuing thread takes of the order of ten cycles beside the working warps of its scheduler, and the issue then
// keeps up with the tensor pipe (one tcgen05.mma per 64 to 78 cycles).
// D (+)= A x B with A (packed bf16 pairs, 8 columns per k-step of 16) in TMEM and B in shared memory
template <int ACC, uint32_t B_CONST, uint32_t B_HI = kDescHi>
__device__ __forceinline__ void mma_ts_c(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_base, uint32_t idesc) {
    asm volatile(
        "{\n\t.reg .b64 db;\n\t.reg .b32 lb;\n\t"
        "add.u32 lb, %2, %5;\n\tmov.b64 db, {lb, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, %6;\n\t}" ::"r"(d_tmem), "r"(a_tmem), "r"(b_base), "r"(idesc),
        "r"(B_HI), "n"(B_CONST), "n"(ACC)
        : "memory");
}
// A = operand tile in TMEM (64 columns: channels 2 u, 2 u + 1 of a token in column u), B K-major
template <int ACC0, int NK = 8, int KS = 0>
__device__ __forceinline__ void mma8_ek(uint32_t d, uint32_t e_tmem, uint32_t b_base, uint32_t idesc) {
    if constexpr (KS < NK) {
        mma_ts_c<(KS == 0 ? ACC0 : 1), t_kmaj(0) + t_kstep(KS)>(d, e_tmem + 8 * KS, b_base, idesc);
        mma8_ek<ACC0, NK, KS + 1>(d, e_tmem, b_base, idesc);
    }
}
// The same, B a copy of H_0 or U_0
template <int ACC0, int NK = 8, int KS = 0>
__device__ __forceinline__ void mma8_es(uint32_t d, uint32_t e_tmem, uint32_t b_base, uint32_t idesc) {
    if constexpr (KS < NK) {
        mma_ts_c<(KS == 0 ? ACC0 : 1), t_state<NK>(KS), kDescHiState>(d, e_tmem + 8 * KS, b_base, idesc);
        mma8_es<ACC0, NK, KS + 1>(d, e_tmem, b_base, idesc);
    }
}
// The contractions over the channels: with head dimension 64 (zero-extended on chip) the channels 64..127 of every
// operand are zero, and the four k-steps over them are left out.
template <int ACC0>
__device__ __forceinline__ void prod_ek(bool half, uint32_t d, uint32_t e_tmem, uint32_t b_base, uint32_t idesc) {
    if (half) mma8_ek<ACC0, 4>(d, e_tmem, b_base, idesc);
    else mma8_ek<ACC0, 8>(d, e_tmem, b_base, idesc);
}
template <int ACC0>
__device__ __forceinline__ void prod_kk(bool half, uint32_t d, uint32_t a_base, uint32_t b_base, uint32_t idesc) {
    if (half) mma8_kk<ACC0, 4>(d, a_base, b_base, idesc);
    else mma8_kk<ACC0, 8>(d, a_base, b_base, idesc);
}
template <int ACC0>
__device__ __forceinline__ void prod_es(bool half, uint32_t d, uint32_t e_tmem, uint32_t b_base, uint32_t idesc) {
    if (half) mma8_es<ACC0, 4>(d, e_tmem, b_base, idesc);
    else mma8_es<ACC0, 8>(d, e_tmem, b_base, idesc);
}
template <int ACC0>
__device__ __forceinline__ void prod_ks(bool half, uint32_t d, uint32_t a_base, uint32_t b_base, uint32_t idesc) {
    if (half) mma8_ks<ACC0, 4>(d, a_base, b_base, idesc);
    else mma8_ks<ACC0, 8>(d, a_base, b_base, idesc);
}
// The products of one request.  kb, hb, cb: descriptor bases (shared address >> 4) of the slot's buffers.
__device__ __forceinline__ void issue_batch(int op, bool half, uint32_t kb, uint32_t hb, uint32_t cb, uint32_t tm_S, uint32_t tm_R,
                                            uint32_t tm_E, uint32_t bar_s, uint32_t bar_r, uint32_t bar_sc) {
    switch (op) {
        case OP_FROB:    // Gram matrix Khat Khat^T and Khat H_0
            prod_kk<0>(half, tm_S, kb, kb, kIdescKK);
            prod_ks<0>(half, tm_R, kb, hb, idesc_r_kk(half));
            mma_commit(bar_s);
            break;
        case OP_ITER1:   // S = E Khat^T, R += E H_0^T (the second runs under the masked-score epilogue)
            prod_ek<0>(half, tm_S, tm_E, kb, kIdescKK);
            mma_commit(bar_sc);
            prod_es<1>(half, tm_R, tm_E, hb, idesc_r_kk(half));
            break;
        case OP_ITER2:   // R += P Khat
            mma8_pm_rows(tm_R, tm_S, kb, idesc_r_pm(half));
            mma_commit(bar_r);
            break;
        case OP_OUT_S:   // scores of the final iterate: S = X_hi Khat^T + X_lo Khat^T (X_lo sits in the first columns of R)
            prod_ek<0>(half, tm_S, tm_E, kb, kIdescKK);
            prod_ek<1>(half, tm_S, tm_R, kb, kIdescKK);
            mma_commit(bar_sc);
            prod_es<0>(half, tm_R, tm_E, half ? hb + (8192u >> 4) : hb, idesc_r_kk(half));   // O = X_hi U_0^T (64 channels: U_0 follows H_0) (runs under the masked-score epilogue; X_lo has been read)
            break;
        case OP_OUT_O:   // O += P V
            mma8_pm(tm_R, tm_S, cb, idesc_r_pm(half));
            mma_commit(bar_r);
            break;
        default:
            break;
    }
}

struct Ctx {
    int l, q, c;                  // lane, TMEM lane quadrant, token / TMEM lane of the slot's tile
    uint32_t tm_s, tm_r, tm_e;    // TMEM addresses of this thread's lane: scores, accumulator, operand
};

// Masked scores of 16 keys: S (fp32, 16 columns) -> P (packed bf16 pairs in 8 registers).  EXACT: per-element factor
// 2^(ac_c - G_j) (strongly decaying tiles, whose keys are not pre-scaled); KEYF: key j's column times ks[j] (the pass
// whose P meets the unscaled V); DIAG: mk masks the keys i <= l of the 32-key block.
template <bool EXACT, bool KEYF, bool DIAG>
__device__ __forceinline__ void p_half(const uint32_t (&r)[16], uint32_t (&pk)[8], const float *G2h, const float *ksh,
                                       float ac_c, const uint32_t *mk) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        float p0 = __uint_as_float(r[2 * u]), p1 = __uint_as_float(r[2 * u + 1]);
        if (EXACT) {
            p0 *= ex2_fast(fminf(ac_c - G2h[2 * u], 126.f));
            p1 *= ex2_fast(fminf(ac_c - G2h[2 * u + 1], 126.f));
        }
        if (KEYF) {
            const float2 f = *reinterpret_cast<const float2 *>(ksh + 2 * u);
            p0 *= f.x;
            p1 *= f.y;
        }
        pk[u] = pack_bf16(p0, p1);
        if (DIAG) pk[u] &= mk[u];
    }
}
// The keys of the diagonal block that token l of a lane quadrant sees, as masks of the packed pairs 2 u, 2 u + 1: a table in
// shared memory (rows of 20 words: no bank conflict), fetched while the scores are on their way.  Selecting before the
// conversion took four instructions per pair, on a scheduler that the update warps of the other slot keep busy.
struct DiagMasks { uint32_t row[32][20]; };
__device__ __forceinline__ void diag_masks(const DiagMasks &m, int l, uint32_t (&mk)[16]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint4 v = *reinterpret_cast<const uint4 *>(&m.row[l][4 * i]);
        mk[4 * i] = v.x; mk[4 * i + 1] = v.y; mk[4 * i + 2] = v.z; mk[4 * i + 3] = v.w;
    }
}
// Masked-score epilogue of token c = 32 q + l: key blocks below q need no mask, block q is the diagonal block, the
// blocks above it are zero.  P for keys 32 kb + 2 u, 2 u + 1 goes to column 32 kb + u of the score tile.  The epilogue
// is a chain of tensor-memory round trips (loads of a 32-key block, conversion, stores), so the zero blocks are stored
// first.
template <bool EXACT, bool KEYF>
__device__ __forceinline__ void p_convert(const Ctx &cx, const GateScalars *gs, float ac_c, int kb, const uint32_t (&ra)[16],
                                          const uint32_t (&rb)[16], const DiagMasks &dm) {
    uint32_t pa[8], pb[8];
    const float *G2kb = gs->G2 + 32 * kb, *kskb = gs->ks + 32 * kb;
    uint32_t mk[16];
    if (kb == cx.q) {
        diag_masks(dm, cx.l, mk);
        p_half<EXACT, KEYF, true>(ra, pa, G2kb, kskb, ac_c, mk);
        p_half<EXACT, KEYF, true>(rb, pb, G2kb + 16, kskb + 16, ac_c, mk + 8);
    } else {
        p_half<EXACT, KEYF, false>(ra, pa, G2kb, kskb, ac_c, mk);
        p_half<EXACT, KEYF, false>(rb, pb, G2kb + 16, kskb + 16, ac_c, mk + 8);
    }
    TMEM_ST8(cx.tm_s + 32 * kb, pa);
    TMEM_ST8(cx.tm_s + 32 * kb + 8, pb);
}
// The same for all key blocks of lane quadrant Q, as straight-line code.
template <int Q, int KB>
__device__ __forceinline__ void p_block(const Ctx &cx, const DiagMasks &dm, const uint32_t (&r)[32]) {
    uint32_t mk[16];
    if constexpr (KB == Q) diag_masks(dm, cx.l, mk);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t pk[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            pk[u] = pack_bf16(__uint_as_float(r[16 * h + 2 * u]), __uint_as_float(r[16 * h + 2 * u + 1]));
            if constexpr (KB == Q) pk[u] &= mk[8 * h + u];
        }
        TMEM_ST8(cx.tm_s + 32 * KB + 8 * h, pk);
    }
}
// AHEAD (128 channels): the next block's scores are on their way while a block is converted (4 to 5 % of a call; with head
// dimension 64 it measured 1 % slower).
template <int Q, bool AHEAD>
__device__ __forceinline__ void p_blocks(const Ctx &cx, const DiagMasks &dm) {
    uint32_t ra[32], rb[32];
    auto load = [&](int kb, uint32_t(&r)[32]) { TMEM_LD32(cx.tm_s + 32 * kb, r); };
    load(0, ra);
    tmem_wait_ld();
    if constexpr (!AHEAD) {
        p_block<Q, 0>(cx, dm, ra);
        if constexpr (Q > 0) { load(1, ra); tmem_wait_ld(); p_block<Q, 1>(cx, dm, ra); }
        if constexpr (Q > 1) { load(2, ra); tmem_wait_ld(); p_block<Q, 2>(cx, dm, ra); }
        if constexpr (Q > 2) { load(3, ra); tmem_wait_ld(); p_block<Q, 3>(cx, dm, ra); }
    } else {
        if constexpr (Q > 0) load(1, rb);
        p_block<Q, 0>(cx, dm, ra);
        if constexpr (Q > 0) { tmem_wait_ld(); if constexpr (Q > 1) load(2, ra); p_block<Q, 1>(cx, dm, rb); }
        if constexpr (Q > 1) { tmem_wait_ld(); if constexpr (Q > 2) load(3, rb); p_block<Q, 2>(cx, dm, ra); }
        if constexpr (Q > 2) { tmem_wait_ld(); p_block<Q, 3>(cx, dm, rb); }
    }
}
template <bool EXACT, bool KEYF, bool AHEAD>
__device__ __forceinline__ void p_epilogue_t(const Ctx &cx, const GateScalars *gs, float ac_c, const DiagMasks &dm) {
    if (!KEYF && !EXACT) {
        if (cx.q == 0) p_blocks<0, AHEAD>(cx, dm);
        else if (cx.q == 1) p_blocks<1, AHEAD>(cx, dm);
        else if (cx.q == 2) p_blocks<2, AHEAD>(cx, dm);
        else p_blocks<3, AHEAD>(cx, dm);
        tmem_wait_st();
        return;
    }
    if (KEYF) {      // (the product of an iteration leaves out the rows whose key block is above the diagonal instead)
        uint32_t z[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) z[i] = 0u;
#pragma unroll 1
        for (int kb = cx.q + 1; kb < 4; ++kb) {
            TMEM_ST8(cx.tm_s + 32 * kb, z);
            TMEM_ST8(cx.tm_s + 32 * kb + 8, z);
        }
    }
#pragma unroll 1
    for (int kb = 0; kb <= cx.q; ++kb) {
        uint32_t ra[16], rb[16];
        TMEM_LD16(cx.tm_s + 32 * kb, ra);
        TMEM_LD16(cx.tm_s + 32 * kb + 16, rb);
        tmem_wait_ld();
        p_convert<EXACT, KEYF>(cx, gs, ac_c, kb, ra, rb, dm);
    }
    tmem_wait_st();
}
// The epilogues of strongly decaying tiles, which most calls never run, as functions: inlined they lie between the others' code (what
// the warps execute does not fit the first-level instruction cache, and neighbours of it are fetched too).  The read's as a function:
// 64 x 2048 tokens, d = 64: 117.8 -> 116.3 us, nothing else changes; an iteration's too: with beta, alpha or for the solve alone 197.7
// -> 194.0 (24 x 1999, 30 iterations) and 185.5 -> 183.0 (32 x 2048), but in the plain kernel at 128 channels a call there costs spills
// (349 -> 350, 131072 tokens 5700 -> 5740), so there it stays inlined.
// What such tiles cost (gates of mean 1 or less before the sigmoid instead of 2): 64 x 4096 tokens, 10 iterations 330 -> 464 us per call; 24 x
// 1999, 30 iterations 196 -> 272; 32 x 2048, the solve alone 184 -> 287; 64 x 2048, d = 64 117 -> 171.  All inlined they take 460, 272,
// 294 and 170: the functions cost them up to 1 %, and save the solve alone 2.
template <bool KEYF>
__device__ __noinline__ void p_epilogue_exact(uint32_t tm_s, int q, int l, const GateScalars *gs, float ac_c, const DiagMasks *dm) {
    Ctx cx;
    cx.tm_s = tm_s;
    cx.q = q;
    cx.l = l;
    p_epilogue_t<true, KEYF, false>(cx, gs, ac_c, *dm);
}
template <bool KEYF, bool AHEAD, bool CALL>
__device__ __forceinline__ void p_epilogue(const Ctx &cx, const GateScalars *gs, bool exact, float ac_c, const DiagMasks &dm) {
    if (exact) {
        if constexpr (CALL) p_epilogue_exact<KEYF>(cx.tm_s, cx.q, cx.l, gs, ac_c, &dm);
        else p_epilogue_t<true, KEYF, AHEAD>(cx, gs, ac_c, dm);
    } else p_epilogue_t<false, KEYF, AHEAD>(cx, gs, ac_c, dm);
}

// Sum over one 32-key block of the squared Gram entries of the earlier keys (decayed when the keys are not
// pre-scaled) and the key's own squared norm.
template <bool DIAG, bool EXACT>
__device__ __forceinline__ void gram_block(const uint32_t (&r)[32], const float *G2kb, float G2j, int l, float &gsum) {
    float acc[4] = {0.f, 0.f, 0.f, 0.f}, gd = 0.f;      // four partial sums: the additions do not wait for one another
#pragma unroll
    for (int ii = 0; ii < 32; ++ii) {
        const float g = __uint_as_float(r[ii]);
        const float g2 = g * g;
        if (DIAG) gd = ii == l ? g2 : gd;
        float w = EXACT ? ex2_fast(G2j - G2kb[ii]) * g2 : g2;
        if (DIAG) w = ii < l ? w : 0.f;
        acc[ii & 3] += w;
    }
    gsum += 2.f * ((acc[0] + acc[1]) + (acc[2] + acc[3])) + gd;
}

// Inclusive scan over the tile's 128 tokens (the slot's four warps, one token per thread) of the affine maps
// s -> a s + b, composed in token order; returns the map's value at `seed`.
__device__ __forceinline__ float affine_scan(const Ctx &cx, SlotScalars *sc, int slot, float a, float b, float seed) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float pa = __shfl_up_sync(0xffffffffu, a, o), pb = __shfl_up_sync(0xffffffffu, b, o);
        if (cx.l >= o) {
            b = fmaf(a, pb, b);
            a *= pa;
        }
    }
    // (the previous tile's carries have long been read: every warp of the slot has passed several hand-overs since)
    if (cx.l == 31) {
        sc->carry[0][cx.q] = a;
        sc->carry[1][cx.q] = b;
    }
    asm volatile("bar.sync %0, 128;" ::"r"(slot + 1) : "memory");
    float s = seed;
    for (int w = 0; w < cx.q; ++w) s = fmaf(sc->carry[0][w], s, sc->carry[1][w]);
    return fmaf(a, s, b);
}

template <bool EXTRA, bool HALF>
__global__ void __launch_bounds__(kThreadsSolve, 1)
fwd_tc_solve_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                    const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmO, FwdArgs a, long long ntiles) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t s_bars[B_COUNT];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    __shared__ __align__(16) uint32_t s_req[4];     // per slot: requests posted (warps), Gram matrices read (warps)
    __shared__ __align__(16) DiagMasks dm;

    unsigned char *smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    const int tid = threadIdx.x;
    const uint32_t bars = smem_u32(&s_bars[0]);
    const uint32_t abort_addr = smem_u32(&s_abort);

    if (tid == 0) {
        s_abort = 0;
        s_req[0] = s_req[1] = s_req[2] = s_req[3] = 0u;
        for (int i = 0; i < B_COUNT; ++i) {
            const int b = i % B_PER_SLOT;
            const bool per_warp = i < B_DRAIN && (b == B_RDY_ST || b == B_QF || b == B_GF0 || b == B_GF1);
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bars + 8 * i), "r"(per_warp ? ST / 32 : 1));
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < 32 * 16; i += kThreadsSolve) {
        const int ml = i >> 4, u = i & 15;
        dm.row[ml][u] = (2 * u <= ml ? 0x0000FFFFu : 0u) | (2 * u + 1 <= ml ? 0xFFFF0000u : 0u);
    }
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem_base))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem_base;
    const uint32_t sbase = smem_u32(smem);

    // this block's tiles: a contiguous range, dealt to the two slots in turn
    const long long t_lo = (ntiles * blockIdx.x) / gridDim.x, t_hi = (ntiles * (blockIdx.x + 1)) / gridDim.x;
    const int n_mine = (int)(t_hi - t_lo);
    const bool solve_only = EXTRA && a.solve_only != 0;   // the result is the solve itself: no V, no U, no output product
    const float *const beta_p = EXTRA ? a.beta : nullptr;
    const float *const alpha_p = EXTRA ? a.alpha : nullptr;
    const bool mix = alpha_p != nullptr && !solve_only;   // alpha-connection: the read uses alpha x + (1 - alpha) q
    constexpr bool half = HALF;                           // head dimension 64: channels 64..127 are zero, their k-steps are left out

    // The helper warps come first: when a scheduler changes warps it prefers the oldest eligible one, and the thread
    // that issues the products must not wait behind the compute warps of its scheduler.
    if (tid < 128) {
        if constexpr (!HALF) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsHelper));
        const int hw = tid >> 5, lane = tid & 31;
        if (hw == 0) {
            // ================= gate scalars of every tile, one tile ahead of the compute warps =================
            for (int k = 0; k < n_mine; ++k) {
                const int slot = k & 1, j = k >> 1;
                const uint32_t sb = bars + 8 * (slot * B_PER_SLOT);
                if (j >= 2) wait_bar(sb + 8 * (B_GF0 + (j & 1)), (uint32_t)(((j - 2) >> 1) & 1), abort_addr);
                const TileInfo ti = tile_info(a, t_lo + k);
                GateScalars *g = &reinterpret_cast<SlotScalars *>(smem + OFF_SC + slot * SC_BYTES)->g[j & 1];
                float run = 0.f;
                float ks_g[4], ks_s[4];
#pragma unroll
                for (int grp = 0; grp < 4; ++grp) {
                    const int cc = 32 * grp + lane;
                    const bool in = cc < ti.ntok;       // tokens past the sequence: no decay, unit lambda / strengths
                    const size_t idx = ti.tok0 + (size_t)cc * a.heads;
                    const float gv = in ? *(a.gate + idx) : 1.f;
                    const float lamv = in ? *(a.lam + idx) : 1.f;
                    const float bv = (beta_p && in) ? *(beta_p + idx) : 1.f;
                    const float av = (alpha_p && in) ? *(alpha_p + idx) : 1.f;
                    const float lgc = fmaxf(log2f(gv), -115.f);
                    float incl = lgc;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const float up = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += up;
                    }
                    const float G2c = run + incl;
                    run += __shfl_sync(0xffffffffu, incl, 31);
                    const float mc = fmaxf(G2c, -60.f);
                    g->lg[cc] = lgc;
                    g->G2[cc] = G2c;
                    g->ac[cc] = G2c - mc;
                    g->zt[cc] = exp2f(mc);
                    g->iz[cc] = exp2f(-mc);
                    g->lam[cc] = lamv;
                    g->al[cc] = av;
                    ks_g[grp] = G2c;
                    ks_s[grp] = sqrtf(fmaxf(bv, 0.f));
                }
                {
                    // the decay of the whole tile decides how the keys are staged (ti.ntok - 1 is the last token)
                    const float Glast = __shfl_sync(0xffffffffu, ks_g[(ti.ntok - 1) >> 5], (ti.ntok - 1) & 31);
                    const bool exact = Glast < -60.f;
#pragma unroll
                    for (int grp = 0; grp < 4; ++grp)
                        g->ks[32 * grp + lane] = exact ? ks_s[grp] : ks_s[grp] * exp2f(-0.5f * ks_g[grp]);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(sb + 8 * (B_GS0 + (j & 1)));
            }
        } else if (hw == 1 || hw == 3) {
            // ========== TMA thread of a slot: first loads, V once q has been read, result stores, the next q ==========
            const int slot = hw >> 1;
            const int n_slot = (n_mine - slot + 1) >> 1;       // tiles of this slot: k = slot, slot + 2, ...
            if (lane == 0 && n_slot > 0) {
                const uint32_t sb = bars + 8 * (slot * B_PER_SLOT);
                const uint32_t sl = sbase + slot * SLOT_BYTES;
                auto load_q = [&](int k) {
                    const TileInfo ti = tile_info(a, t_lo + k);
                    mbar_expect_tx(sb + 8 * B_LD_Q, 32768u);
                    tma_load_tile3(&tmQ, sl + BUF_C, sb + 8 * B_LD_Q, ti.h * a.d, tile_x_hi(ti.h, a.d, a.heads), ti.n * NT, ti.b);
                };
                // the inputs do not depend on the state kernel; its per-tile states do
                {
                    const TileInfo ti = tile_info(a, t_lo + slot);
                    load_q(slot);
                    mbar_expect_tx(sb + 8 * B_LD_K, 32768u);
                    tma_load_tile3(&tmK, sl + BUF_A, sb + 8 * B_LD_K, ti.h * a.d, tile_x_hi(ti.h, a.d, a.heads), ti.n * NT, ti.b);
                    asm volatile("griddepcontrol.wait;" ::: "memory");
                    load_h0<HALF>(a, t_lo + slot, sl + BUF_B, sb + 8 * B_LD_H, solve_only);
                }
                for (int j = 0; j < n_slot; ++j) {
                    const int k = slot + 2 * j;
                    const TileInfo ti = tile_info(a, t_lo + k);
                    if (!solve_only) {
                        wait_bar(sb + 8 * B_QF, (uint32_t)(j & 1), abort_addr);
                        if (aborted(abort_addr)) break;
                        mbar_expect_tx(sb + 8 * B_LD_V, 32768u);
                        tma_load_tile3(&tmV, sl + BUF_C, sb + 8 * B_LD_V, ti.h * a.d, tile_x_hi(ti.h, a.d, a.heads), ti.n * NT, ti.b);
                    }
                    wait_bar(sb + 8 * B_RDY_ST, (uint32_t)(j & 1), abort_addr);
                    for (int hf = 0; hf < a.d / 64; ++hf)   // rows past the sequence are clipped; channels from a.d on are not stored
                        asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::
                                         "l"(reinterpret_cast<uint64_t>(&tmO)), "r"(ti.h * a.d + 64 * hf), "r"(ti.n * NT),
                                     "r"(ti.b), "r"(sl + BUF_C + 16384 * hf)
                                     : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the staged tile has been read
                    if (j + 1 < n_slot && !aborted(abort_addr)) load_q(k + 2);
                }
                asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // output stores are complete
            }
        } else if constexpr (!HALF) {
            // ================================ MMA issuing thread (128 channels only) ================================
            // Serves the requests of both slots in the order they become ready.  The score tile S is held by a slot
            // from its FROB request until its warps have read the Gram matrix (counted in shared memory), from ITER1 to the issue of
            // ITER2 and from OUT_S to the issue of OUT_O (products run in issue order, so the next owner's score
            // product follows the last read of P).
            if (lane == 0) {
                const uint32_t base14 = (sbase >> 4) & 0x3FFF;
                // Per-slot state in scalars (arrays indexed by the slot would live in local memory).  Every instruction
                // of this thread competes with the compute warps of its scheduler, so the paths between a request and
                // its products are kept as short as possible.
                int op0 = OP_FROB, op1 = OP_FROB, it0 = 0, it1 = 0, left0 = (n_mine + 1) >> 1, left1 = n_mine >> 1;
                uint32_t thr0 = 4u, thr1 = 4u;          // request counter values at which the next request of a slot is complete
                uint32_t gthr0 = 4u, gthr1 = 4u;        // the same for the Gram-read counters
                uint32_t til0 = 0, til1 = 0;            // tiles done (phase of the per-tile TMA barriers)
                const uint32_t req_addr = smem_u32(&s_req[0]);
                int owner = -1;                         // slot that holds S while its warps read the Gram matrix
                int prefer = 0;                         // slot to serve first when both are ready
                bool gave_up = false;
                auto issue = [&](int sl, int o) {
                    const uint32_t sbb = bars + 8 * (sl * B_PER_SLOT);
                    const uint32_t sl14 = base14 + ((sl * SLOT_BYTES) >> 4);
                    fence_after();
                    issue_batch(o, false, sl14 + (BUF_A >> 4), sl14 + (BUF_B >> 4), sl14 + (BUF_C >> 4), tmem + tm_s_of(false, sl),
                                tmem + tm_r_of(false, sl), tmem + tm_e_of(sl), sbb + 8 * B_MMA_S, sbb + 8 * B_MMA_R, bars + 8 * (B_SC + sl));
                };
                // Bookkeeping of a request of slot sl that has just been issued, together with its follow-up (ITER2 after
                // ITER1, OUT_O after OUT_S): the slot's next request, counters and tile count.  Returns the counter value
                // at which the follow-up is posted.
                auto book = [&](int sl, int o) -> uint32_t {
                    bool tile_done = false;
                    int it = sl ? it1 : it0, nop;
                    const uint32_t thr = (sl ? thr1 : thr0) + 4u;
                    if (o == OP_FROB) {
                        owner = sl;                          // until the Gram matrix has been read
                        nop = it < a.n_iter ? OP_ITER1 : OP_OUT_S;
                        if (a.n_iter == 0 && solve_only) tile_done = true;
                    } else if (o == OP_ITER1) {
                        ++it;
                        nop = it < a.n_iter ? OP_ITER1 : OP_OUT_S;
                        if (it >= a.n_iter && solve_only) tile_done = true;
                    } else {
                        nop = OP_FROB;
                        tile_done = true;
                    }
                    if (tile_done) {
                        nop = OP_FROB;
                        it = 0;
                    }
                    if (sl) { op1 = nop; it1 = it; thr1 = thr + (o == OP_FROB ? 0u : 4u); if (tile_done) { --left1; ++til1; } }
                    else { op0 = nop; it0 = it; thr0 = thr + (o == OP_FROB ? 0u : 4u); if (tile_done) { --left0; ++til0; } }
                    return thr;
                };
                int next_s = -1;                        // slot known to have its request posted (no poll needed)
                while ((left0 > 0 || left1 > 0) && !gave_up) {
                    // ---- a slot whose next request (FROB, ITER1 or OUT_S: all need the score tile) is posted and may have S
                    int s = next_s;
                    next_s = -1;
                    for (int polls = 0; s < 0;) {
                        uint32_t c0, c1, g0, g1;
                        asm volatile("ld.volatile.shared::cta.v4.u32 {%0, %1, %2, %3}, [%4];"
                                     : "=r"(c0), "=r"(c1), "=r"(g0), "=r"(g1)
                                     : "r"(req_addr)
                                     : "memory");
                        if (owner == 0 && (int)(g0 - gthr0) >= 0) { gthr0 += 4u; owner = -1; }
                        if (owner == 1 && (int)(g1 - gthr1) >= 0) { gthr1 += 4u; owner = -1; }
                        const bool r0 = left0 > 0 && owner != 1 && (int)(c0 - thr0) >= 0;
                        const bool r1 = left1 > 0 && owner != 0 && (int)(c1 - thr1) >= 0;
                        if (r0 | r1) {
                            s = (r0 && !(r1 && prefer == 1)) ? 0 : 1;
                            break;
                        }
                        if ((++polls & 1023) == 0 && (aborted(abort_addr) || polls > (1 << 24))) {
                            gave_up = true;
                            break;
                        }
                    }
                    if (gave_up) break;
                    prefer = 1 - s;
                    int o = s ? op1 : op0;
                    // a request of the slot that still holds S for its Gram reads implies that those are done
                    if (owner == s) {
                        if (s) gthr1 += 4u; else gthr0 += 4u;
                        owner = -1;
                    }
                    uint32_t til = s ? til1 : til0;
                    if (o == OP_FROB) wait_bar(bars + 8 * (s * B_PER_SLOT + B_LD_H), til & 1u, abort_addr);   // the H_0 tile (TMA)
                    if (o == OP_OUT_S) wait_bar(bars + 8 * (s * B_PER_SLOT + B_LD_U), til & 1u, abort_addr);  // the U_0 tile
                    issue(s, o);
                    uint32_t thr = book(s, o);
                    if (o == OP_FROB) continue;
                    // ---- ITER1 or OUT_S of slot s is running: its follow-up (ITER2, OUT_O) comes next.  In the steady state
                    // of the iterations the other slot's ITER1 follows at once; everything both need is worked out here,
                    // while the products run and the scores are masked, so that a handful of instructions lie between the
                    // posts and the products.
                    for (;;) {
                        const int t = 1 - s;
                        const uint32_t s14 = base14 + ((s * SLOT_BYTES) >> 4), t14 = base14 + ((t * SLOT_BYTES) >> 4);
                        const uint32_t p_kb = s14 + (BUF_A >> 4), p_tmR = tmem + tm_r_of(false, s);
                        const uint32_t p_barR = bars + 8 * (s * B_PER_SLOT + B_MMA_R);
                        const bool t_iter = (t ? left1 : left0) > 0 && (t ? op1 : op0) == OP_ITER1;
                        const uint32_t thr_t = t ? thr1 : thr0;
                        const uint32_t n_kb = t14 + (BUF_A >> 4), n_tmE = tmem + tm_e_of(t);
                        uint32_t c_t = 0u;
                        for (int polls = 0;;) {
                            uint32_t c0, c1;
                            asm volatile("ld.volatile.shared::cta.v2.u32 {%0, %1}, [%2];" : "=r"(c0), "=r"(c1) : "r"(req_addr) : "memory");
                            c_t = s ? c0 : c1;
                            if ((int)((s ? c1 : c0) - thr) >= 0) break;
                            if ((++polls & 1023) == 0 && (aborted(abort_addr) || polls > (1 << 24))) {
                                gave_up = true;
                                break;
                            }
                        }
                        if (gave_up) break;
                        if (o == OP_ITER1) {
                            fence_after();
                            mma8_pm_rows(p_tmR, tmem + tm_s_of(false, s), p_kb, idesc_r_pm(false));  // ITER2: R += P Khat
                            mma_commit(p_barR);
                        } else {                                 // OUT_O: the V tile (TMA)
                            wait_bar(bars + 8 * (s * B_PER_SLOT + B_LD_V), til & 1u, abort_addr);
                            issue(s, OP_OUT_O);
                        }
                        bool t_posted = (int)(c_t - thr_t) >= 0;
                        if (t_iter && !t_posted) {
                            // the other slot is in its iterations and its update is about to end (this slot's own next
                            // request is a whole update away): wait for it here, where its products are prepared
                            for (int polls = 0; polls < 4096 && !t_posted; ++polls) {
                                uint32_t c0, c1;
                                asm volatile("ld.volatile.shared::cta.v2.u32 {%0, %1}, [%2];" : "=r"(c0), "=r"(c1) : "r"(req_addr) : "memory");
                                t_posted = (int)((t ? c1 : c0) - thr_t) >= 0;
                            }
                        }
                        if (!(t_iter && t_posted)) {
                            // the other slot's request, if it was already posted, is served next without a poll
                            if ((t ? left1 : left0) > 0 && t_posted) next_s = t;
                            break;
                        }
                        // ---- ITER1 of the other slot, at once
                        fence_after();
                        prod_ek<0>(false, tmem + tm_s_of(false, t), n_tmE, n_kb, kIdescKK);           // S = E Khat^T
                        mma_commit(bars + 8 * (B_SC + t));
                        prod_es<1>(false, tmem + tm_r_of(false, t), n_tmE, n_kb + ((BUF_B - BUF_A) >> 4), idesc_r_kk(false));   // R += E H_0^T
                        if (owner == t) {                        // (its Gram reads are done: it has asked again)
                            if (t) gthr1 += 4u; else gthr0 += 4u;
                            owner = -1;
                        }
                        prefer = s;
                        til = t ? til1 : til0;
                        thr = book(t, OP_ITER1);
                        o = OP_ITER1;
                        s = t;
                    }
                }
                if (gave_up) set_abort(abort_addr);
                // every product is complete before the block gives its tensor memory back
                mma_commit(bars + 8 * B_DRAIN);
                if (!mbar_spin_bounded(bars + 8 * B_DRAIN, 0u)) set_abort(abort_addr);
            }
        }
    } else {
        // ================================= compute threads =================================
        if constexpr (!HALF) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsCompute));
        const int slot = (tid >> 7) - 1;
        Ctx cx;
        cx.l = tid & 31;
        cx.q = (tid >> 5) & 3;
        cx.c = 32 * cx.q + cx.l;
        const uint32_t lane_addr = (uint32_t)(32 * cx.q) << 16;
        cx.tm_s = tmem + tm_s_of(half, slot) + lane_addr;
        cx.tm_r = tmem + tm_r_of(half, slot) + lane_addr;
        cx.tm_e = tmem + tm_e_of(slot) + lane_addr;
        const int c = cx.c, l = cx.l;
        const bool leader = c == 0;                              // issues the slot's loads that follow a product
        const bool adaptive = (a.flags & GKA_FLAG_ADAPTIVE_LAMBDA) != 0;
        const uint32_t sb = bars + 8 * (slot * B_PER_SLOT);
        const uint32_t sl = sbase + slot * SLOT_BYTES;
        unsigned char *const bufa = smem + slot * SLOT_BYTES + BUF_A, *const bufc = smem + slot * SLOT_BYTES + BUF_C;
        SlotScalars *const sc = reinterpret_cast<SlotScalars *>(smem + OFF_SC + slot * SC_BYTES);
        // the per-tile states and norms come from the state kernel
        asm volatile("griddepcontrol.wait;" ::: "memory");

        // Head dimension 64: the passes over the channels stop at channel 64 (the rest is zero in every operand and stays so)
        constexpr int NG16 = HALF ? 4 : 8;    // groups of 16 channels
        uint64_t xs[64];                      // -zt_c x_c: the token's 128 channels as fp32 pairs
        uint32_t n_s = 0, n_r = 0;            // completed phases of MMA_S, MMA_R
        auto wait_s = [&]() { wait_bar(sb + 8 * B_MMA_S, n_s & 1u, abort_addr); ++n_s; fence_after(); };
        auto wait_r = [&]() { wait_bar(sb + 8 * B_MMA_R, n_r & 1u, abort_addr); ++n_r; fence_after(); };
        const uint32_t req_addr = smem_u32(&s_req[slot]), grd_addr = smem_u32(&s_req[2 + slot]);
        // Requests.  With 128 channels they go to the issuing thread.  HALF: one thread of the slot waits for the slot's other warps
        // and issues the products itself (one thread, so that they run in order; in the warp with the fewest key blocks, which
        // can best afford to wait until the tensor pipe has taken them).
        uint32_t n_req = 0;                   // requests of this slot so far (HALF)
        uint32_t n_sc = 0;                    // completed phases of B_SC
        auto request = [&](int op, uint32_t tile_parity) {
            if constexpr (!HALF) {
                if (op != OP_FROB) warp_post_tmem(req_addr, l);
                else warp_post(req_addr, l);
            } else {
                ++n_req;
                if (cx.q != 0) {
                    if (op != OP_FROB) warp_post_tmem(req_addr, l);
                    else warp_post(req_addr, l);
                } else {
                    __syncwarp();
                    if (l == 0) {
                        uint32_t cnt = 0u;
                        for (int polls = 0;; ++polls) {
                            asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(cnt) : "r"(req_addr) : "memory");
                            if ((int)(cnt - 3u * n_req) >= 0) break;
                            if ((polls & 1023) == 1023 && (aborted(abort_addr) || polls > (1 << 24))) {
                                set_abort(abort_addr);
                                break;
                            }
                        }
                        if (op == OP_FROB) wait_bar(sb + 8 * B_LD_H, tile_parity, abort_addr);    // the H_0 tile (TMA)
                        if (op == OP_OUT_O) wait_bar(sb + 8 * B_LD_V, tile_parity, abort_addr);   // the V tile
                        fence_after();
                        const uint32_t s14 = (sl >> 4) & 0x3FFF;
                        issue_batch(op, true, s14 + (BUF_A >> 4), s14 + (BUF_B >> 4), s14 + (BUF_C >> 4), tmem + tm_s_of(true, slot),
                                    tmem + tm_r_of(true, slot), tmem + tm_e_of(slot), sb + 8 * B_MMA_S, sb + 8 * B_MMA_R, bars + 8 * (B_SC + slot));
                    }
                    __syncwarp();
                }
            }
        };
        auto wait_scores = [&]() { wait_bar(bars + 8 * (B_SC + slot), n_sc & 1u, abort_addr); ++n_sc; fence_after(); };
        // -xs (times `scale`) as packed bf16 pairs of channel group g8 (8 channels): its leading part, or the remainder
        auto pack_x = [&](int g8, bool lo, float scale, uint32_t(&pk)[4]) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float xa, xb;
                f2_unpack(xs[4 * g8 + u], xa, xb);
                xa *= -scale;
                xb *= -scale;
                uint32_t p = pack_bf16(xa, xb);
                if (lo) p = pack_bf16(xa - bf16_lo(p), xb - bf16_hi(p));
                pk[u] = p;
            }
        };

        for (int k = slot, j = 0; k < n_mine; k += kSlots, ++j) {
            const long long tile = t_lo + k;
            const bool more = k + kSlots < n_mine;
            const GateScalars *const gs = &sc->g[j & 1];
            const TileInfo ti = tile_info(a, tile);
            const bool valid = c < ti.ntok;
            // loads of the slot's next tile, issued by the leader as soon as the buffer's last reader is done (none once a wait has
            // given up: a barrier whose copy never landed takes no second announcement)
            auto load_next_k = [&]() {
                if (leader && more && !aborted(abort_addr)) {
                    const TileInfo tn = tile_info(a, tile + kSlots);
                    mbar_expect_tx(sb + 8 * B_LD_K, 32768u);
                    tma_load_tile3(&tmK, sl + BUF_A, sb + 8 * B_LD_K, tn.h * a.d, tile_x_hi(tn.h, a.d, a.heads), tn.n * NT, tn.b);
                }
            };
            auto load_next_h = [&]() {
                if (leader && more && !aborted(abort_addr)) load_h0<HALF>(a, tile + kSlots, sl + BUF_B, sb + 8 * B_LD_H, solve_only);
            };
            auto after_last_h0_product = [&]() {      // H_0 has been read for the last time
                if (solve_only) {
                    load_next_k();
                    load_next_h();
                } else if (!HALF && leader && !aborted(abort_addr)) {
                    mbar_expect_tx(sb + 8 * B_LD_U, 32768u);
                    bulk_load(sl + BUF_B, a.tile_hu + (size_t)tile * kTileStateBytes + 32768, 32768u, sb + 8 * B_LD_U);
                }
            };
            // ||H_0||_F^2 of the tile (state kernel, one or two terms): fetched now, added up and used by the scan (added up here,
            // where the addition waits for the loads: +0.7 %)
            const float hh = ld_stream_f32(a.tile_hh + tile), hh2 = a.tile_hh2 ? ld_stream_f32(a.tile_hh2 + tile) : 0.f;
            // ---- gate scalars (helper warp) and the K tile (TMA) of this tile
            // Khat of tile jj of this slot: gate scalars (helper warp) and K tile (TMA) awaited, the token's key row scaled
            // in place
            auto stage_keys = [&](int jj) {
                wait_bar(sb + 8 * (B_GS0 + (jj & 1)), (uint32_t)((jj >> 1) & 1), abort_addr);
                wait_bar(sb + 8 * B_LD_K, (uint32_t)(jj & 1), abort_addr);
                const uint2 fj = split_factor(sc->g[jj & 1].ks[c]);
#pragma unroll 1
                for (int g = 0; g < 2 * NG16; g += 4) {          // (rolled: code that runs once per tile is kept small)
                    uint4 v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) v[u] = *reinterpret_cast<const uint4 *>(bufa + tile_off(c, g + u));
#pragma unroll
                    for (int u = 0; u < 4; ++u) *reinterpret_cast<uint4 *>(bufa + tile_off(c, g + u)) = times_factor(v[u], fj);
                }
                fence_async_smem();
            };
            if (j == 0 || solve_only) stage_keys(j);             // (otherwise done under the previous tile's read)
            const bool exact = gs->G2[ti.ntok - 1] < -60.f;     // the tile decays below 2^-60: per-element factors
            const float G2c = gs->G2[c];
            if (HALF) fence_before();
            request(OP_FROB, (uint32_t)(j & 1));
            wait_s();
            if (a.n_iter == 0) after_last_h0_product();
            // ---- chunk-wise Frobenius norms: for the token's key, k^T H_0 k and the decayed squared Gram entries of
            // the earlier keys
            float kh = 0.f, gsum = 0.f;
            {
                float khp[4] = {0.f, 0.f, 0.f, 0.f};
                uint32_t ra[32];
                // (the Gram matrix first: it sits in the score tile, which the other slot is waiting for)
#pragma unroll 1
                for (int kb = 0; kb <= cx.q; ++kb) {
                    TMEM_LD32(cx.tm_s + 32 * kb, ra);
                    tmem_wait_ld();
                    if (exact) {
                        if (kb == cx.q) gram_block<true, true>(ra, gs->G2 + 32 * kb, G2c, l, gsum);
                        else gram_block<false, true>(ra, gs->G2 + 32 * kb, G2c, l, gsum);
                    } else {
                        if (kb == cx.q) gram_block<true, false>(ra, gs->G2 + 32 * kb, G2c, l, gsum);
                        else gram_block<false, false>(ra, gs->G2 + 32 * kb, G2c, l, gsum);
                    }
                }
                fence_before();
                if (!HALF) warp_post(grd_addr, l);               // the Gram matrix has been read: S is free again
#pragma unroll 1
                for (int p = 0; p < NG16 / 2; ++p) {
                    TMEM_LD32(cx.tm_r + 32 * p, ra);
                    uint4 kv[4];
#pragma unroll
                    for (int h4 = 0; h4 < 4; ++h4) kv[h4] = *reinterpret_cast<const uint4 *>(bufa + tile_off(c, 4 * p + h4));
                    tmem_wait_ld();
#pragma unroll
                    for (int h4 = 0; h4 < 4; ++h4) {
                        const uint32_t *pk = reinterpret_cast<const uint32_t *>(&kv[h4]);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            khp[h4] = fmaf(__uint_as_float(ra[8 * h4 + 2 * u]), bf16_lo(pk[u]), khp[h4]);
                            khp[h4] = fmaf(__uint_as_float(ra[8 * h4 + 2 * u + 1]), bf16_hi(pk[u]), khp[h4]);
                        }
                    }
                }
                kh = (khp[0] + khp[1]) + (khp[2] + khp[3]);
            }
            // ---- f_c by an affine scan (s_c = gamma_c^2 s_{c-1} + d_c, s_{-1} = ||H_0||^2), Chebyshev set-up
            float rho2, czb, lz;
            {
                // pre-scaled keys: both sums carry 2^(-2 G_c); plain keys: k H_0 k carries zeta_c
                const float dc = exact ? fmaf(2.f * ex2_fast(G2c), kh, gsum) : ex2_fast(2.f * G2c) * fmaf(2.f, kh, gsum);
                const float s = affine_scan(cx, sc, slot, ex2_fast(2.f * gs->lg[c]), dc, hh + hh2);
                const float fc = sqrtf(fmaxf(s, 0.f));
                float lamc = gs->lam[c];
                if (adaptive) lamc *= fc;
                const float Lpm = fc + 2.f * lamc;
                const float iL = 1.f / Lpm;
                const float rho = fc * iL;
                rho2 = rho * rho;
                czb = valid ? -gs->zt[c] * (2.f * iL) : 0.f;
                lz = lamc * gs->iz[c];
                if (a.fro_out && valid) a.fro_out[ti.tok0 + (size_t)c * a.heads] = fc;
            }
            wait_bar(sb + 8 * B_LD_Q, (uint32_t)(j & 1), abort_addr);   // q tile has landed
            // ---- x_0: R = q, E_0 = czb q; xs takes an increment when it is next read from the operand columns
#pragma unroll
            for (int g16 = 0; g16 < NG16; ++g16) {
                uint32_t rr[16], pk[8];
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) {
                    const uint4 qv = *reinterpret_cast<const uint4 *>(bufc + tile_off(c, 2 * g16 + h2));
                    const uint32_t *qq = reinterpret_cast<const uint32_t *>(&qv);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float qa = bf16_lo(qq[u]), qb = bf16_hi(qq[u]);
                        rr[8 * h2 + 2 * u] = __float_as_uint(qa);
                        rr[8 * h2 + 2 * u + 1] = __float_as_uint(qb);
                        pk[4 * h2 + u] = pack_bf16(czb * qa, czb * qb);
                        xs[8 * g16 + 4 * h2 + u] = 0ull;
                    }
                }
                TMEM_ST16(cx.tm_r + 16 * g16, rr);
                TMEM_ST8(cx.tm_e + 8 * g16, pk);
            }
            if (!solve_only && !mix) warp_arrive(sb + 8 * B_QF, l);      // q has been read: V may take its buffer
            tmem_wait_st();
            // ---- Algorithm 1
            float omega = 2.f;
            if (a.n_iter > 0) {
                fence_before();
                request(OP_ITER1, 0u);
            }
            for (int it = 0; it < a.n_iter; ++it) {
                const bool last = it + 1 == a.n_iter;
                omega = 4.f * recip(4.f - rho2 * omega);         // weight schedule
                const float beta = omega - 1.f, cz = czb * omega;
                const uint64_t beta2 = f2_pack(beta, beta), cz2 = f2_pack(cz, cz), lz2 = f2_pack(lz, lz);
                wait_scores();                                   // the masked scores
                p_epilogue<false, !HALF, EXTRA>(cx, gs, exact, exact ? gs->ac[c] : 0.f, dm);
                fence_before();
                request(OP_ITER2, 0u);
                wait_r();
                if (last) after_last_h0_product();
                // xs += e_old (the value the operand held), e_new = beta e_old + cz (R + lz xs) as bf16.  Sixteen channels at
                // a time; the next group's loads are in flight while a group is computed.  (Adding e_new at once would unpack
                // every increment twice: 9 instead of 7 instructions per pair of channels in code that runs once per
                // iteration and does not fit the first-level instruction cache.)
                {
                    uint32_t ra[16], rb[16], ea[8], eb[8];
                    TMEM_LD16(cx.tm_r, ra);
                    TMEM_LD8(cx.tm_e, ea);
                    tmem_wait_ld();
#pragma unroll
                    for (int g = 0; g < NG16; ++g) {
                        uint32_t(&r)[16] = (g & 1) ? rb : ra;
                        uint32_t(&rn)[16] = (g & 1) ? ra : rb;
                        uint32_t(&e)[8] = (g & 1) ? eb : ea;
                        uint32_t(&en_)[8] = (g & 1) ? ea : eb;
                        if (g < NG16 - 1) {
                            TMEM_LD16(cx.tm_r + 16 * (g + 1), rn);
                            TMEM_LD8(cx.tm_e + 8 * (g + 1), en_);
                        }
                        uint32_t pk[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const int i = 8 * g + u;
                            const uint64_t eo = f2_pack(bf16_lo(e[u]), bf16_hi(e[u]));
                            xs[i] = f2_add(xs[i], eo);
                            const uint64_t res = f2_fma(lz2, xs[i], f2_pack(__uint_as_float(r[2 * u]), __uint_as_float(r[2 * u + 1])));
                            float ea_, eb_;
                            f2_unpack(f2_fma(cz2, res, f2_mul(beta2, eo)), ea_, eb_);
                            pk[u] = pack_bf16(ea_, eb_);
                        }
                        TMEM_ST8(cx.tm_e + 8 * g, pk);
                        if (g < NG16 - 1) tmem_wait_ld();
                    }
                    if (!last) {
                        tmem_wait_st();
                        fence_before();
                        request(OP_ITER1, 0u);
                    }
                }
            }
            // ---- final iterate: the last increment
            tmem_wait_st();
#pragma unroll
            for (int g = 0; g < NG16; g += 4) {
                uint32_t e[32];
                TMEM_LD32(cx.tm_e + 8 * g, e);
                tmem_wait_ld();
#pragma unroll
                for (int u = 0; u < 32; ++u) xs[8 * g + u] = f2_add(xs[8 * g + u], f2_pack(bf16_lo(e[u]), bf16_hi(e[u])));
            }
            if (solve_only) {
                // the solve is the result: x_c = -xs / zt_c as bf16, staged in the q buffer and stored by TMA
                const float izc = gs->iz[c];
#pragma unroll
                for (int g8 = 0; g8 < 2 * NG16; ++g8) {
                    uint32_t pk[4];
                    pack_x(g8, false, izc, pk);
                    *reinterpret_cast<uint4 *>(bufc + tile_off(c, g8)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                }
                fence_async_smem();
                warp_arrive(sb + 8 * (B_GF0 + (j & 1)), l);
                warp_arrive(sb + 8 * B_RDY_ST, l);
                continue;
            }
            if (mix) {
                // alpha-connection (Section 4.3): the read uses alpha x + (1 - alpha) q; q is still in its buffer
                const float alc = gs->al[c], nzt = valid ? -gs->zt[c] : 0.f;
#pragma unroll
                for (int g8 = 0; g8 < 2 * NG16; ++g8) {
                    const uint4 qv = *reinterpret_cast<const uint4 *>(bufc + tile_off(c, g8));
                    const uint32_t *qq = reinterpret_cast<const uint32_t *>(&qv);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        float xa, xb;
                        f2_unpack(xs[4 * g8 + u], xa, xb);
                        const float qa = nzt * bf16_lo(qq[u]), qb = nzt * bf16_hi(qq[u]);
                        xs[4 * g8 + u] = f2_pack(fmaf(alc, xa - qa, qa), fmaf(alc, xb - qb, qb));
                    }
                }
                warp_arrive(sb + 8 * B_QF, l);                   // q has been read: V may take its buffer
            }
            // The read uses the final iterate as two bf16 terms in the score product (the recent keys resolve directions
            // of x that one bf16 rounding would lose): the leading term takes the operand columns, the remainder the
            // first columns of the accumulator, whose content is no longer needed.
#pragma unroll
            for (int g8 = 0; g8 < 2 * NG16; g8 += 2) {
                uint32_t hi[8], lo[8];
                pack_x(g8, false, 1.f, *reinterpret_cast<uint32_t(*)[4]>(&hi[0]));
                pack_x(g8 + 1, false, 1.f, *reinterpret_cast<uint32_t(*)[4]>(&hi[4]));
                pack_x(g8, true, 1.f, *reinterpret_cast<uint32_t(*)[4]>(&lo[0]));
                pack_x(g8 + 1, true, 1.f, *reinterpret_cast<uint32_t(*)[4]>(&lo[4]));
                TMEM_ST8(cx.tm_e + 4 * g8, hi);
                TMEM_ST8(cx.tm_r + 4 * g8, lo);
            }
            tmem_wait_st();
            fence_before();
            request(OP_OUT_S, (uint32_t)(j & 1));
            wait_scores();
            load_next_k();                                       // its products were the last readers of the keys
            p_epilogue<true, !HALF, true>(cx, gs, exact, exact ? gs->ac[c] : 0.f, dm);
            fence_before();
            request(OP_OUT_O, (uint32_t)(j & 1));
            // (the values stay as loaded: their row factor sqrt(beta_j) 2^(-G_j / 2) rides on the masked scores)
            if (more) stage_keys(j + 1);                         // the next tile's keys, under the read
            wait_r();
            load_next_h();                                       // every product of the tile is complete
            // O as bf16 into the V buffer (no product reads it any more), stored by TMA
            {
                // (the iterate's registers are free by now: all four loads are in flight at once)
                uint32_t r[4][32];
#pragma unroll
                for (int p = 0; p < NG16 / 2; ++p) TMEM_LD32(cx.tm_r + 32 * p, r[p]);
                tmem_wait_ld();
#pragma unroll
                for (int p = 0; p < NG16 / 2; ++p) {
#pragma unroll
                    for (int h4 = 0; h4 < 4; ++h4) {
                        uint32_t pk[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) pk[u] = pack_bf16(__uint_as_float(r[p][8 * h4 + 2 * u]), __uint_as_float(r[p][8 * h4 + 2 * u + 1]));
                        *reinterpret_cast<uint4 *>(bufc + tile_off(c, 4 * p + h4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    }
                }
            }
            fence_async_smem();
            fence_before();
            warp_arrive(sb + 8 * (B_GF0 + (j & 1)), l);
            warp_arrive(sb + 8 * B_RDY_ST, l);
        }
        if (HALF && cx.q == 0 && l == 0) {                       // every product is complete before the tensor memory is given back
            mma_commit(sb + 8 * B_MMA_R);
            if (!mbar_spin_bounded(sb + 8 * B_MMA_R, n_r & 1u)) set_abort(abort_addr);
        }
    }

    fence_before();
    __syncthreads();
    if (s_abort != 0) {
        // a wait gave up: leave time for copies still in flight before the shared memory is given back
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);
        if (tid == 0 && a.device_status) atomicExch(a.device_status, (int)GKA_ERR_TIMEOUT);
    }
    if (tid < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

}  // namespace

cudaError_t launch_fwd_solve(const FwdArgs &a, cudaStream_t stream) {
    alignas(64) CUtensorMap tmK, tmV, tmQ, tmO;
    const int cols = a.heads * a.d;
    const long long ntiles = a.plan.NC;
    if (!make_tile_map(&tmK, a.k, a.B, a.T, cols, NT) || !make_tile_map(&tmV, a.v, a.B, a.T, cols, NT) ||
        !make_tile_map(&tmQ, a.q, a.B, a.T, cols, NT) || !make_tile_map(&tmO, a.out, a.B, a.T, cols, NT))
        return cudaErrorInvalidValue;
    const bool extra = a.beta != nullptr || a.alpha != nullptr || a.solve_only != 0;
    const bool half = a.d == 64;
    auto kernel = extra ? (half ? fwd_tc_solve_kernel<true, true> : fwd_tc_solve_kernel<true, false>)
                        : (half ? fwd_tc_solve_kernel<false, true> : fwd_tc_solve_kernel<false, false>);
    static SmemLimit limit[2][2];
    cudaError_t err = limit[extra][half].raise(kernel, (int)SOLVE_SMEM);
    if (err != cudaSuccess) return err;
    const long long want = ntiles < a.sms ? ntiles : (long long)a.sms;   // one persistent block per SM, two tiles in flight each
    if (a.ev_start) cudaEventRecord(a.ev_start, stream);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(want < 1 ? 1 : want));
    cfg.blockDim = dim3(kThreadsSolve);
    cfg.dynamicSmemBytes = SOLVE_SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = a.ev_start ? 0 : 1;
    err = cudaLaunchKernelEx(&cfg, kernel, tmK, tmV, tmQ, tmO, a, ntiles);
    if (err != cudaSuccess) return err;
    if (a.ev_stop) cudaEventRecord(a.ev_stop, stream);
    return cudaGetLastError();
}

}  // namespace gka
