// fp32 GKA recurrence on CUDA cores (sm_100a) for head dimensions 64 and 128: several consecutive tokens of a
// (sequence, head) pair per pass over a register-resident H.  Serves gka_decode_tokens and the chunked forward and solve in
// fp32 arithmetic (f32 I/O, GKA_PREC_HIGH, sequences of fewer than 16 tokens).
//
// A block holds H (D x D, fp32) in registers and U in shared memory and walks its tokens in batches of M = 4 (the rest of a
// run in batches of 2 or 1).  Inside a batch, relative to the state (H_0, U_0) before it,
//
//     H_t = zeta_t H_0 + sum_{j <= t} Gamma[t][j] k_j k_j^T,     zeta_t = prod_{i <= t} gamma_i, Gamma[t][j] = prod_{j < i <= t} gamma_i
//     H_t d = zeta_t (H_0 d) + sum_{j <= t} k_j Gamma[t][j] (k_j . d)
//     ||H_t||_F^2 = gamma_t^2 ||H_{t-1}||_F^2 + 2 gamma_t k_t^T H_{t-1} k_t + (k_t . k_t)^2
//
// so the M solves of a batch (Algorithm 1 in residual form, as in the tensor-core path) advance together: every register of
// H meets M operands per iteration, and the shuffles, barriers and latencies of an iteration are shared by M tokens.
//
// Why this form: the fp32 multiply-add pipe bounds it.  A token costs D^2 multiply-adds per iteration plus 2 (t + 1) D for
// the batch's own keys (6 % at M = 4); the chunk-wise form with 64 tokens per chunk costs D^2 + 2 * 64 D (dense masked
// scores), two to three times as much.  Next to that pipe it is the shared-memory path: operands come from there at 128
// bytes per clock whatever is broadcast, and shuffles share it.  A thread therefore holds 8 rows x D / 8 columns of H
// (D = 128: 128 registers), which loads an operand value once per 8 multiply-adds; with 4 x 16 the loads took as long as the
// arithmetic.  Row m of a thread's block is row m ^ lane8 of its group of 8 rows: the transposing sum over the 8 lanes of a
// group then needs no selects, and thread i ends up with row i for every token of the batch.
//
// The forward splits every sequence into P segments of L tokens (and a segment into F parts) so that the blocks fill the
// device; recur_summary computes what a segment adds to the state, recur_scan folds that into the start state of every
// segment, and a block of a later part first folds the tokens of its segment that come before it.
//
// Measured, before (chunk-wise fp32 kernels; one token at a time for decoding) and with these kernels: B=2, 8 heads, T=8192,
// d=128, f32, r=8: 3209 -> 1945 us; 64 x 32 pairs, 8 tokens, d=128, bf16, r=10: 425 -> 267 us; B=1, 2 heads, T=256, d=64, f32,
// r=8: 118.5 -> 25.5 us (there: three dependent launches and the chain of batches).  Tried: scalar instead of two-wide
// multiply-adds +10 %, the batch's constants in shared memory +8 %, rolled loops +3 %, both tokens of a pair updated in two-wide
// registers +5 % (fewer instructions, a longer chain), two-wide multiply-adds in recur_summary 228 -> 260 us.
#include "gka_common.cuh"
#include "gka_tc_util.cuh"

namespace gka {
namespace {

using tcu::f2_add;
using tcu::f2_fma;
using tcu::f2_mul;
using tcu::f2_pack;
using tcu::f2_unpack;

constexpr int kBatch = 4;          // tokens per pass over H
constexpr int kSumTokens = 16;     // tokens of a stage of the summary kernel

struct RecurArgs {
    const void *q, *k, *v;
    const float *gate, *lam, *beta, *alpha;
    void *out;
    const float *state_in;     // [pairs][2 D D] or nullptr (zero)
    float *state_out;          // may be state_in itself (in-place decode)
    float *fro_out;
    float *seg;                // [pairs][P - 1][2 D D]: what segment s adds, then the start state of segment s + 1
    float *seg_decay;          // [pairs][P - 1]
    int *device_status;
    int T, heads, n_iter;
    unsigned flags;
    int solve_only;
    int P, L, F, Lp;           // segments per sequence and their tokens, parts per segment and their tokens (multiples of 4)
};

template <int D> struct Rc {
    static constexpr int NT = D;            // threads: groups of 8 lanes share 8 rows
    static constexpr int NW = NT / 32;
    static constexpr int CG = D / 32;       // float4 column groups of a thread: columns 4 (lane8 + 8 n)
    static constexpr int kMinBlocks = D == 128 ? 2 : 6;
    // floats: state buffer, operands, q, k, v [M][D], raw staging (at most fp32) [3][M][D], small arrays
    static constexpr int kSmall = 64 + 8 * NW + 16 + 16;
    static constexpr size_t kSmem = sizeof(float) * (D * D + 4 * kBatch * D + 3 * kBatch * D + kSmall);
};

__device__ __forceinline__ float4 lds4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ ulonglong2 lds2x2(const float *p) { return *reinterpret_cast<const ulonglong2 *>(p); }
__device__ __forceinline__ float hsum(uint64_t v) {
    float a, b;
    f2_unpack(v, a, b);
    return a + b;
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// v[m][q]: row sums of the thread's block of H against operands q = 0 .. Q - 1 (xs: [Q][D] in shared memory)
template <int D, int Q>
__device__ __forceinline__ void row_sums(const ulonglong2 (&H)[8][Rc<D>::CG], const float *xs, int lane8, float (&v)[8][Q]) {
    uint64_t acc[8][Q];
#pragma unroll
    for (int n = 0; n < Rc<D>::CG; ++n) {
        ulonglong2 x[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) x[q] = lds2x2(xs + q * D + 4 * (lane8 + 8 * n));
#pragma unroll
        for (int m = 0; m < 8; ++m)
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                acc[m][q] = n == 0 ? f2_mul(H[m][n].x, x[q].x) : f2_fma(H[m][n].x, x[q].x, acc[m][q]);
                acc[m][q] = f2_fma(H[m][n].y, x[q].y, acc[m][q]);
            }
    }
#pragma unroll
    for (int m = 0; m < 8; ++m)
#pragma unroll
        for (int q = 0; q < Q; ++q) v[m][q] = hsum(acc[m][q]);
}
// Transposing sum over the 8 lanes of a group: row m of lane l is row m ^ l of the group, so half of the values go to the
// partner in each step and what is left at the end is the lane's own row.
template <int Q>
__device__ __forceinline__ void reduce_rows(float (&v)[8][Q], float (&y)[Q]) {
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1)
#pragma unroll
        for (int m = 0; m < h; ++m)
#pragma unroll
            for (int q = 0; q < Q; ++q) v[m][q] += __shfl_xor_sync(0xffffffffu, v[m + h][q], h);
#pragma unroll
    for (int q = 0; q < Q; ++q) y[q] = v[0][q];
}
// y[t] = (H x_t)[row of this thread]; xs: [M][D] in shared memory
template <int D, int M>
__device__ __forceinline__ void matvec(const ulonglong2 (&H)[8][Rc<D>::CG], const float *xs, int lane8, float (&y)[M]) {
    constexpr int Q = M == 1 ? 1 : 2;       // two tokens at a time: the accumulators of four would not fit beside H
#pragma unroll
    for (int p = 0; p < M / Q; ++p) {
        float v[8][Q], yp[Q];
        row_sums<D, Q>(H, xs + Q * p * D, lane8, v);
        reduce_rows<Q>(v, yp);
#pragma unroll
        for (int q = 0; q < Q; ++q) y[Q * p + q] = yp[q];
    }
}
// Two tokens of the batch, the warp's own (t0 for even warps, t0 + 1 for odd ones) and the other: row sums v[.][0] and v[.][1] of the
// thread's block of H, and S[4 t + j] = Gamma[t][j] (k_j . x_t) of the own token with kj the columns of key lane / 8.  (No branch: the
// arithmetic of the pair before is scheduled into this one's.  No selects: choosing the own token's words of two operands was 16
// instructions per pair; 64 x 32 pairs, 8 tokens 287.6 -> 268.1 us, 2 x 8 pairs, T = 8192 2071 -> 1952.)
template <int D>
__device__ __forceinline__ void pair_sums(const ulonglong2 (&H)[8][Rc<D>::CG], const ulonglong2 (&kj)[Rc<D>::CG], const float *sX,
                                          const float *sGam, float *sS, int t0, float (&v)[8][2]) {
    const int lane = threadIdx.x & 31, lane8 = lane & 7, odd = (threadIdx.x >> 5) & 1;
    const float *const xa_p = sX + (t0 + odd) * D + 4 * lane8, *const xb_p = sX + (t0 + 1 - odd) * D + 4 * lane8;
    uint64_t acc[8][2], dot = 0ull;
#pragma unroll
    for (int n = 0; n < Rc<D>::CG; ++n) {
        const ulonglong2 xa = lds2x2(xa_p + 32 * n), xb = lds2x2(xb_p + 32 * n);
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            acc[m][0] = n == 0 ? f2_mul(H[m][n].x, xa.x) : f2_fma(H[m][n].x, xa.x, acc[m][0]);
            acc[m][1] = n == 0 ? f2_mul(H[m][n].x, xb.x) : f2_fma(H[m][n].x, xb.x, acc[m][1]);
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            acc[m][0] = f2_fma(H[m][n].y, xa.y, acc[m][0]);
            acc[m][1] = f2_fma(H[m][n].y, xb.y, acc[m][1]);
        }
        dot = f2_fma(kj[n].x, xa.x, dot);
        dot = f2_fma(kj[n].y, xa.y, dot);
    }
    float s = hsum(dot);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const int i = 4 * (t0 + odd) + (lane >> 3);
    if (lane8 == 0) sS[i] = sGam[i] * s;
#pragma unroll
    for (int m = 0; m < 8; ++m)
#pragma unroll
        for (int q = 0; q < 2; ++q) v[m][q] = hsum(acc[m][q]);
}
// dst[4 t + j] = w[4 t + j] (k_j . x_t) (w = nullptr: 1), j = 0 .. M - 1: warp t mod NW takes token t, its group j of 8
// lanes key j.  Values with j > t are not used (their weights are zero).
template <int D, int M>
__device__ __forceinline__ void key_dots(const float *sK, const float *xs, const float *w, float *dst, int warp, int lane) {
    constexpr int CG = Rc<D>::CG, NW = Rc<D>::NW;
    const int j = lane >> 3, lane8 = lane & 7;
#pragma unroll
    for (int t0 = 0; t0 < M; t0 += NW) {
        const int t = t0 + warp;
        if (t < M) {
            uint64_t acc = 0ull;
#pragma unroll
            for (int n = 0; n < CG; ++n) {
                const ulonglong2 kk = lds2x2(sK + j * D + 4 * (lane8 + 8 * n)), x = lds2x2(xs + t * D + 4 * (lane8 + 8 * n));
                acc = f2_fma(kk.x, x.x, acc);
                acc = f2_fma(kk.y, x.y, acc);
            }
            float s = hsum(acc);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane8 == 0) dst[4 * t + j] = w ? w[4 * t + j] * s : s;
        }
    }
}

// Pointers into a block's shared memory
template <int D, typename IoT> struct Mem {
    float *U, *X, *Q, *K, *V, *S, *Gram, *Gam, *Sc, *Red;
    IoT *raw;            // [3][M][D] the next batch's q, k, v as they arrive
    float *raw_sc;       // [4][M] its gate, lambda, beta, alpha
    __device__ explicit Mem(float *base) {
        U = base;            // [D][D] U; H passes through it on the way into the registers and out of them
        X = base + D * D;
        Q = X + kBatch * D;
        K = Q + kBatch * D;
        V = K + kBatch * D;
        raw = reinterpret_cast<IoT *>(V + kBatch * D);
        float *p = V + kBatch * D + 3 * kBatch * D;
        S = p;               // [t][j] Gamma[t][j] (k_j . x_t)
        Gram = p + 16;
        Gam = p + 32;
        raw_sc = p + 48;
        Red = p + 64;        // [warp][8]: k_t^T H_0 k_t (4), ||H_0||^2
        Sc = Red + 8 * Rc<D>::NW;   // [4][M] gate, lambda, beta, alpha of this batch
    }
};

// A block's progress through its tokens
struct Run {
    float *state_out;    // final state of the sequence, or nullptr
    uint32_t bar;        // mbarrier of the copies into the state buffer
    bool u_pending;      // the copy of U has not been waited for
};
// Wait (bounded) for the copy of U before its first use, and a block barrier; false: it never landed.
__device__ __forceinline__ bool u_ready(Run &r) {
    bool bad = false;
    if (r.u_pending) {
        r.u_pending = false;
        bad = !mbar_wait_bounded(r.bar, 1u);
    }
    return !__syncthreads_or(bad);
}

// One pass over U: products of the old U with the operands in X (READ), U <- zeta_M U + sum_j Gamma[M][j] v_j k_j^T (update).
template <int D, typename IoT, int M, bool READ>
__device__ __forceinline__ void u_pass(const Mem<D, IoT> &sm, float zM, bool update, float (&y)[M]) {
    constexpr int CG = Rc<D>::CG;
    const int tid = threadIdx.x, lane8 = tid & 7, row8 = tid & ~7;
    const float *const gl = sm.Gam + 4 * (M - 1);
    const uint64_t zM2 = f2_pack(zM, zM);
    float v[8][M];
#pragma unroll
    for (int half = 0; half < 2; ++half) {                   // four rows at a time
        uint64_t acc[4][M];
        float vc[4][M];
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int j = 0; j < M; ++j) {
                acc[e][j] = 0ull;
                vc[e][j] = gl[j] * sm.V[j * D + row8 + ((4 * half + e) ^ lane8)];
            }
#pragma unroll
        for (int n = 0; n < CG; ++n) {
            const int col = 4 * (lane8 + 8 * n);
            ulonglong2 u[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) u[e] = lds2x2(sm.U + (row8 + ((4 * half + e) ^ lane8)) * D + col);
            if constexpr (READ) {
#pragma unroll
                for (int j = 0; j < M; ++j) {
                    const ulonglong2 z = lds2x2(sm.X + j * D + col);
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[e][j] = f2_fma(u[e].y, z.y, f2_fma(u[e].x, z.x, acc[e][j]));
                }
            }
            if (update) {
                ulonglong2 inc[4];
#pragma unroll
                for (int j = 0; j < M; ++j) {
                    const ulonglong2 kc = lds2x2(sm.K + j * D + col);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const uint64_t w2 = f2_pack(vc[e][j], vc[e][j]);
                        inc[e].x = j == 0 ? f2_mul(w2, kc.x) : f2_fma(w2, kc.x, inc[e].x);
                        inc[e].y = j == 0 ? f2_mul(w2, kc.y) : f2_fma(w2, kc.y, inc[e].y);
                    }
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    u[e].x = f2_fma(zM2, u[e].x, inc[e].x);
                    u[e].y = f2_fma(zM2, u[e].y, inc[e].y);
                    *reinterpret_cast<ulonglong2 *>(sm.U + (row8 + ((4 * half + e) ^ lane8)) * D + col) = u[e];
                }
            }
        }
        if constexpr (READ) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int j = 0; j < M; ++j) v[4 * half + e][j] = hsum(acc[e][j]);
        }
    }
    if constexpr (READ) reduce_rows<M>(v, y);
}

// What the tokens of one batch do to the state, and (SOLVE) the solves and reads.  nv <= M tokens exist; the others have
// zero vectors, gate 1, lambda 1.  Thread i holds row i of the iterates.  Returns false if the copy of U never landed.
template <int D, typename IoT, int M, bool SOLVE>
__device__ __forceinline__ bool batch(const RecurArgs &a, const Mem<D, IoT> &sm, ulonglong2 (&H)[8][Rc<D>::CG], float &ss,
                                      size_t tok, int nv, bool last, Run &run) {
    constexpr int CG = Rc<D>::CG, NW = Rc<D>::NW;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lane8 = tid & 7, row8 = tid & ~7;
    const bool update = !last || run.state_out;
    float zts[M];
#pragma unroll
    for (int t = 0; t < M; ++t) zts[t] = t == 0 ? sm.Sc[0] : zts[t - 1] * sm.Sc[t];

    if constexpr (SOLVE) {
        // ---- Frobenius norms: k_t^T H_0 k_t, the Gram matrix of the batch's keys, ||H_0||_F^2
        {
            float w[M];
            key_dots<D, M>(sm.K, sm.K, nullptr, sm.Gram, warp, lane);
            matvec<D, M>(H, sm.K, lane8, w);
#pragma unroll
            for (int t = 0; t < M; ++t) {
                w[t] *= sm.K[t * D + tid];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) w[t] += __shfl_xor_sync(0xffffffffu, w[t], o);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            if (lane == 0) {
#pragma unroll
                for (int t = 0; t < M; ++t) sm.Red[8 * warp + t] = w[t];
                sm.Red[8 * warp + 4] = ss;
            }
        }
        __syncthreads();
        float x[M], d[M], res[M], s0[M], rho2[M], om[M], lam[M];
        {
            float f2 = 0.f, khk[M];
#pragma unroll
            for (int t = 0; t < M; ++t) khk[t] = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
#pragma unroll
                for (int t = 0; t < M; ++t) khk[t] += sm.Red[8 * w + t];
                f2 += sm.Red[8 * w + 4];
            }
#pragma unroll
            for (int t = 0; t < M; ++t) {
                float s = (t == 0 ? 1.f : zts[t > 0 ? t - 1 : 0]) * khk[t];
#pragma unroll
                for (int j = 0; j < t; ++j) s = fmaf(sm.Gam[4 * (t - 1) + j], sm.Gram[4 * t + j] * sm.Gram[4 * t + j], s);
                const float g = sm.Sc[t], kk = sm.Gram[4 * t + t];
                f2 = fmaf(g, fmaf(g, f2, 2.f * s), kk * kk);
                const float f = sqrtf(fmaxf(f2, 0.f));
                if (a.fro_out && tid == t && t < nv) a.fro_out[tok + (size_t)t * a.heads] = f;
                float l = sm.Sc[4 + t];
                if (a.flags & GKA_FLAG_ADAPTIVE_LAMBDA) l *= f;
                const float Lpm = f + 2.f * l;               // L + mu
                const float rho = f / Lpm;
                rho2[t] = rho * rho;
                s0[t] = 2.f / Lpm;
                om[t] = 2.f;
                lam[t] = l;
                res[t] = sm.Q[t * D + tid];
                d[t] = s0[t] * res[t];
                x[t] = 0.f;
                sm.X[t * D + tid] = d[t];
            }
        }
        float kr[M];
#pragma unroll
        for (int j = 0; j < M; ++j) kr[j] = sm.K[j * D + tid];
        __syncthreads();

        // ---- Algorithm 1 in residual form; x: iterate, d: increment (the published operand), res: q - H_t x
        auto advance = [&](int t, float y, float4 s4) {      // s4: S of token t (zero beyond j = t)
            float h = zts[t] * y;
            h = fmaf(kr[0], s4.x, h);
            if (t >= 1) h = fmaf(kr[M > 1 ? 1 : 0], s4.y, h);
            if (t >= 2) h = fmaf(kr[M > 2 ? 2 : 0], s4.z, h);
            if (t >= 3) h = fmaf(kr[M > 2 ? 3 : 0], s4.w, h);
            om[t] = 4.f * recip(4.f - rho2[t] * om[t]);
            x[t] += d[t];
            res[t] -= h;
            d[t] = fmaf(s0[t] * om[t], fmaf(-lam[t], x[t], res[t]), (om[t] - 1.f) * d[t]);
            sm.X[t * D + tid] = d[t];
        };
        if constexpr (M == 4) {
            // Tokens 0, 1 and tokens 2, 3 half an iteration apart: between two barriers the products of one pair run beside
            // the sums over the lanes and the update of the other.
            ulonglong2 kj[CG];                               // key (lane / 8), for the pair's products with the keys
#pragma unroll
            for (int n = 0; n < CG; ++n) kj[n] = lds2x2(sm.K + (lane >> 3) * D + 4 * (lane8 + 8 * n));
            const bool odd = (warp & 1) != 0;                // v[.][0] is the warp's own token
            float v0[8][2], v1[8][2];
            auto finish = [&](int t0, float (&v)[8][2], float4 sa, float4 sb) {
                float y[2];
                reduce_rows<2>(v, y);
                advance(t0, odd ? y[1] : y[0], sa);
                advance(t0 + 1, odd ? y[0] : y[1], sb);
            };
            // products of the tokens t1, t1 + 1 beside the update of the tokens t0, t0 + 1
            auto region = [&](int t1, float (&v1)[8][2], int t0, float (&v0)[8][2]) {
                const float4 sa = lds4(sm.S + 4 * t0), sb = lds4(sm.S + 4 * t0 + 4);
                pair_sums<D>(H, kj, sm.X, sm.Gam, sm.S, t1, v1);
                finish(t0, v0, sa, sb);
                __syncthreads();
            };
            if (a.n_iter > 0) {
                pair_sums<D>(H, kj, sm.X, sm.Gam, sm.S, 0, v0);
                __syncthreads();
                for (int it = 1; it < a.n_iter; ++it) {
                    region(2, v1, 0, v0);
                    region(0, v0, 2, v1);
                }
                region(2, v1, 0, v0);
                finish(2, v1, lds4(sm.S + 8), lds4(sm.S + 12));
            }
        } else {
            for (int it = 0; it < a.n_iter; ++it) {
                float y[M];
                key_dots<D, M>(sm.K, sm.X, sm.Gam, sm.S, warp, lane);
                matvec<D, M>(H, sm.X, lane8, y);
                __syncthreads();                             // every read of X is done, S is complete
#pragma unroll
                for (int t = 0; t < M; ++t) advance(t, y[t], lds4(sm.S + 4 * t));
                __syncthreads();
            }
        }
        IoT *const out = reinterpret_cast<IoT *>(a.out);
#pragma unroll
        for (int t = 0; t < M; ++t) {
            x[t] += d[t];                                    // the final iterate
            if (a.solve_only) {
                if (t < nv) Io<IoT>::store1(out + (tok + (size_t)t * a.heads) * D + tid, x[t]);
            } else {
                // the read takes x or (alpha-connection, Section 4.3) alpha x + (1 - alpha) q
                if (a.alpha) {
                    const float qv = sm.Q[t * D + tid];
                    x[t] = fmaf(sm.Sc[12 + t], x[t] - qv, qv);
                }
                sm.X[t * D + tid] = x[t];
            }
        }
        if (!a.solve_only) {
            // ---- read o_t = zeta_t (U_0 z_t) + sum_j v_j Gamma[t][j] (k_j . z_t), and the update of U
            if (!u_ready(run)) return false;
            key_dots<D, M>(sm.K, sm.X, sm.Gam, sm.S, warp, lane);
            float y[M];
            u_pass<D, IoT, M, true>(sm, zts[M - 1], update, y);
            __syncthreads();                                 // S is complete
#pragma unroll
            for (int t = 0; t < M; ++t) {
                float h = zts[t] * y[t];
#pragma unroll
                for (int j = 0; j <= t; ++j) h = fmaf(sm.V[j * D + tid], sm.S[4 * t + j], h);
                if (t < nv) Io<IoT>::store1(out + (tok + (size_t)t * a.heads) * D + tid, h);
            }
        }
    } else if (!a.solve_only) {
        if (!u_ready(run)) return false;
        float y[M];
        u_pass<D, IoT, M, false>(sm, zts[M - 1], true, y);
    }

    // ---- H <- zeta_M H + sum_j Gamma[M][j] k_j k_j^T (the increments are summed before they meet H: one rounding of H)
    if (update) {
        const uint64_t zM2 = f2_pack(zts[M - 1], zts[M - 1]);
        uint64_t sq = 0ull;
        float wr[M][8];
#pragma unroll
        for (int j = 0; j < M; ++j)
#pragma unroll
            for (int m = 0; m < 8; ++m) wr[j][m] = sm.Gam[4 * (M - 1) + j] * sm.K[j * D + row8 + (m ^ lane8)];
#pragma unroll
        for (int n = 0; n < CG; ++n) {
            ulonglong2 kc[M];
#pragma unroll
            for (int j = 0; j < M; ++j) kc[j] = lds2x2(sm.K + j * D + 4 * (lane8 + 8 * n));
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                ulonglong2 inc;
#pragma unroll
                for (int j = 0; j < M; ++j) {
                    const uint64_t w2 = f2_pack(wr[j][m], wr[j][m]);
                    inc.x = j == 0 ? f2_mul(w2, kc[j].x) : f2_fma(w2, kc[j].x, inc.x);
                    inc.y = j == 0 ? f2_mul(w2, kc[j].y) : f2_fma(w2, kc[j].y, inc.y);
                }
                H[m][n].x = f2_fma(zM2, H[m][n].x, inc.x);
                H[m][n].y = f2_fma(zM2, H[m][n].y, inc.y);
                sq = f2_fma(H[m][n].x, H[m][n].x, sq);
                sq = f2_fma(H[m][n].y, H[m][n].y, sq);
            }
        }
        ss = hsum(sq);
    }
    return true;
}

template <int D, typename IoT>
__global__ void __launch_bounds__(Rc<D>::NT, Rc<D>::kMinBlocks) recur_kernel(RecurArgs a) {
    constexpr int CG = Rc<D>::CG, NT = Rc<D>::NT;
    constexpr uint32_t kMatBytes = D * D * sizeof(float);
    extern __shared__ __align__(128) float smem[];
    const Mem<D, IoT> sm(smem);
    const uint32_t bar = smem_u32(sm.Sc + 16), buf = smem_u32(sm.U);
    const int tid = threadIdx.x, lane8 = tid & 7, row8 = tid & ~7;
    const int pf = a.P * a.F;
    const int pair = blockIdx.x / pf, sp = blockIdx.x % pf, s = sp / a.F, part = sp % a.F;
    const int seq = pair / a.heads, h = pair % a.heads;
    const int t_seg = s * a.L, t_end = min(a.T, t_seg + a.L);
    const int t_lo = t_seg + part * a.Lp, t_hi = min(t_end, t_lo + a.Lp);
    if (t_lo >= t_hi) return;
    Run run;
    run.state_out = (t_hi == a.T && a.state_out) ? a.state_out + (size_t)pair * 2 * D * D : nullptr;
    run.bar = bar;
    run.u_pending = false;
    const size_t tok_base = (size_t)seq * a.T * a.heads + h;     // token t of this pair: tok_base + t heads

    // the tokens t .. t + 3 on their way into the staging buffer
    auto fetch = [&](int t) {
        constexpr int PV = D * (int)sizeof(IoT) / 16;            // 16-byte pieces of a vector
        const int nv = min(kBatch, t_hi - t), nvec = a.solve_only ? 2 : 3;
        for (int i = tid; i < nvec * kBatch * PV; i += NT) {
            const int vec = i / (kBatch * PV), tt = (i / PV) % kBatch, pc = i % PV;
            const void *src = vec == 0 ? a.q : (vec == 1 ? a.k : a.v);
            if (tt < nv)
                cp_async16(smem_u32(sm.raw + (vec * kBatch + tt) * D) + 16 * pc,
                           reinterpret_cast<const unsigned char *>(src) + (tok_base + (size_t)(t + tt) * a.heads) * D * sizeof(IoT) + 16 * pc);
        }
        if (tid < 16 && (tid & 3) < nv) {
            const float *src = tid < 4 ? a.gate : (tid < 8 ? a.lam : (tid < 12 ? a.beta : a.alpha));
            if (src) cp_async4(smem_u32(sm.raw_sc + tid), src + tok_base + (size_t)(t + (tid & 3)) * a.heads);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto bulk_in = [&](const float *src) {                       // one matrix into the state buffer (one thread)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(kMatBytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
                         "r"(buf), "l"(src), "r"(kMatBytes), "r"(bar)
                     : "memory");
    };
    auto bulk_out = [&](float *dst) {                            // and out of it (one thread); returns when it has been read
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(buf), "r"(kMatBytes) : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    };
    auto fail = [&] {                                            // a copy never landed: the same decision in every thread
        if (tid == 0 && a.device_status) atomicExch(a.device_status, (int)GKA_ERR_TIMEOUT);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    };
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 16) sm.S[tid] = 0.f;
    asm volatile("griddepcontrol.wait;" ::: "memory");           // programmatic launch: the scan's start states, or the inputs
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const float *const start = s > 0 ? a.seg + ((size_t)pair * (a.P - 1) + s - 1) * 2 * D * D
                                     : (a.state_in ? a.state_in + (size_t)pair * 2 * D * D : nullptr);
    if (tid == 0 && start) bulk_in(start);
    fetch(t_seg);
    ulonglong2 H[8][CG];
    float ss = 0.f;
    __syncthreads();
    if (start) {
        if (__syncthreads_or(!mbar_wait_bounded(bar, 0u))) return fail();
        uint64_t sq = 0ull;
#pragma unroll
        for (int m = 0; m < 8; ++m)
#pragma unroll
            for (int n = 0; n < CG; ++n) {
                H[m][n] = lds2x2(sm.U + (row8 + (m ^ lane8)) * D + 4 * (lane8 + 8 * n));
                sq = f2_fma(H[m][n].x, H[m][n].x, sq);
                sq = f2_fma(H[m][n].y, H[m][n].y, sq);
            }
        ss = hsum(sq);
        tcu::fence_async_smem();
        __syncthreads();
        if (!a.solve_only) {
            run.u_pending = true;
            if (tid == 0) bulk_in(start + (size_t)D * D);
        }
    } else {
#pragma unroll
        for (int m = 0; m < 8; ++m)
#pragma unroll
            for (int n = 0; n < CG; ++n) H[m][n].x = H[m][n].y = 0ull;
        for (int e = 4 * tid; e < D * D; e += 4 * NT) *reinterpret_cast<float4 *>(sm.U + e) = make_float4(0.f, 0.f, 0.f, 0.f);
    }

    for (int t = t_seg; t < t_hi; t += kBatch) {
        const int nv = min(kBatch, t_hi - t);
        // ---- the batch's vectors and scalars out of the staging buffer
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        for (int i = tid; i < 3 * kBatch * D / 4; i += NT) {
            const int vec = i / (kBatch * D / 4), tt = (i / (D / 4)) % kBatch, c4 = i % (D / 4);
            float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
            if (tt < nv && !(vec == 2 && a.solve_only)) f = Io<IoT>::load4(sm.raw + (vec * kBatch + tt) * D + 4 * c4);
            if (vec > 0 && a.beta && tt < nv) {
                // write strength beta (Remark on the beta-augmented variant, Section 4.1): beta k k^T and beta v k^T are the
                // plain writes of sqrt(beta) k and sqrt(beta) v
                const float sb = sqrtf(fmaxf(sm.raw_sc[8 + tt], 0.f));
                f.x *= sb; f.y *= sb; f.z *= sb; f.w *= sb;
            }
            *reinterpret_cast<float4 *>((vec == 0 ? sm.Q : (vec == 1 ? sm.K : sm.V)) + tt * D + 4 * c4) = f;
        }
        if (tid < 16) {
            sm.Sc[tid] = (tid & 3) < nv ? sm.raw_sc[tid] : 1.f;
            const int tt = tid >> 2, j = tid & 3;                // Gamma[tt][j]
            float g = j <= tt ? 1.f : 0.f;
            for (int i = j + 1; i <= tt; ++i) g *= i < nv ? sm.raw_sc[i] : 1.f;
            sm.Gam[tid] = g;
        }
        __syncthreads();
        if (t + kBatch < t_hi) fetch(t + kBatch);
        const size_t tok = tok_base + (size_t)t * a.heads;
        const bool last = t + kBatch >= t_hi;
        bool ok;
        if (t < t_lo) ok = batch<D, IoT, 4, false>(a, sm, H, ss, tok, nv, last, run);
        else if (nv > 2) ok = batch<D, IoT, 4, true>(a, sm, H, ss, tok, nv, last, run);
        else if (nv == 2) ok = batch<D, IoT, 2, true>(a, sm, H, ss, tok, nv, last, run);
        else ok = batch<D, IoT, 1, true>(a, sm, H, ss, tok, nv, last, run);
        if (!ok) return fail();
    }

    if (run.state_out) {                                         // U, then H, through the state buffer
        tcu::fence_async_smem();
        __syncthreads();
        if (tid == 0) bulk_out(run.state_out + (size_t)D * D);
        __syncthreads();
#pragma unroll
        for (int m = 0; m < 8; ++m)
#pragma unroll
            for (int n = 0; n < CG; ++n)
                *reinterpret_cast<ulonglong2 *>(sm.U + (row8 + (m ^ lane8)) * D + 4 * (lane8 + 8 * n)) = H[m][n];
        tcu::fence_async_smem();
        __syncthreads();
        if (tid == 0) bulk_out(run.state_out);
    }
}

// What a segment adds to the state: decay product and (delta-H, delta-U) relative to a zero start, 256 threads in a 16 x 16
// grid with a (D / 16)^2 block of both matrices each.  Bound by the multiply-add pipe (2 D^2 per token).  The tokens are
// taken from the last to the first, so that the weight of a token (the product of the later gates) is a running product and
// the accumulators are never rescaled; they arrive by asynchronous copies, one stage ahead, in the I/O type.
template <int D, typename IoT>
__global__ void __launch_bounds__(256, 1) recur_summary(RecurArgs a) {
    constexpr int TR = D / 16, G4 = TR / 4, NS = kSumTokens;
    __shared__ __align__(16) IoT sK[2][NS][D], sV[2][NS][D];
    __shared__ float sG[2][NS], sB[2][NS];
    asm volatile("griddepcontrol.wait;" ::: "memory");           // whatever wrote the inputs (programmatic launch)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int pair = blockIdx.x / (a.P - 1), s = blockIdx.x % (a.P - 1);
    const int seq = pair / a.heads, h = pair % a.heads;
    const size_t tok_base = (size_t)seq * a.T * a.heads + h;
    const int t_lo = s * a.L, t_hi = min(a.T, t_lo + a.L), stages = (t_hi - t_lo + NS - 1) / NS;
    auto fetch = [&](int st, int b) {                            // stage st holds tokens t_lo + st NS ..
        constexpr int PV = D * (int)sizeof(IoT) / 16;
        const int t0 = t_lo + st * NS, nv = min(NS, t_hi - t0);
        for (int i = tid; i < (a.solve_only ? 1 : 2) * NS * PV; i += 256) {
            const int which = i / (NS * PV), tt = (i / PV) % NS, pc = i % PV;
            if (tt < nv)
                cp_async16(smem_u32(which ? sV[b][tt] : sK[b][tt]) + 16 * pc,
                           reinterpret_cast<const unsigned char *>(which ? a.v : a.k) + (tok_base + (size_t)(t0 + tt) * a.heads) * D * sizeof(IoT) + 16 * pc);
        }
        if (tid < nv) {
            cp_async4(smem_u32(&sG[b][tid]), a.gate + tok_base + (size_t)(t0 + tid) * a.heads);
            if (a.beta) cp_async4(smem_u32(&sB[b][tid]), a.beta + tok_base + (size_t)(t0 + tid) * a.heads);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float aH[TR][TR], aU[TR][TR];
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int c = 0; c < TR; ++c) aH[i][c] = aU[i][c] = 0.f;
    float decay = 1.f;
    fetch(stages - 1, (stages - 1) & 1);
    for (int st = stages - 1; st >= 0; --st) {
        const int b = st & 1, nv = min(NS, t_hi - t_lo - st * NS);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                                         // this stage is in, and the one before it has been used
        if (st > 0) fetch(st - 1, b ^ 1);
#pragma unroll 2
        for (int t = nv - 1; t >= 0; --t) {
            const float w = a.beta ? decay * fmaxf(sB[b][t], 0.f) : decay;
            float kr[TR], kc[TR], vr[TR];
#pragma unroll
            for (int g4 = 0; g4 < G4; ++g4) {
                const float4 r = Io<IoT>::load4(&sK[b][t][64 * g4 + 4 * ty]), c = Io<IoT>::load4(&sK[b][t][64 * g4 + 4 * tx]);
                const float4 vv = Io<IoT>::load4(&sV[b][t][64 * g4 + 4 * ty]);
                kr[4 * g4 + 0] = r.x; kr[4 * g4 + 1] = r.y; kr[4 * g4 + 2] = r.z; kr[4 * g4 + 3] = r.w;
                kc[4 * g4 + 0] = w * c.x; kc[4 * g4 + 1] = w * c.y; kc[4 * g4 + 2] = w * c.z; kc[4 * g4 + 3] = w * c.w;
                vr[4 * g4 + 0] = vv.x; vr[4 * g4 + 1] = vv.y; vr[4 * g4 + 2] = vv.z; vr[4 * g4 + 3] = vv.w;
            }
            decay *= sG[b][t];
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int c = 0; c < TR; ++c) aH[i][c] = fmaf(kr[i], kc[c], aH[i][c]);
            if (!a.solve_only) {
#pragma unroll
                for (int i = 0; i < TR; ++i)
#pragma unroll
                    for (int c = 0; c < TR; ++c) aU[i][c] = fmaf(vr[i], kc[c], aU[i][c]);
            }
        }
    }
    float *const dst = a.seg + (size_t)blockIdx.x * 2 * D * D;
#pragma unroll
    for (int gi = 0; gi < G4; ++gi)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int gc = 0; gc < G4; ++gc) {
                float *p = dst + (size_t)(64 * gi + 4 * ty + i) * D + 64 * gc + 4 * tx;
                const int r = 4 * gi + i, c = 4 * gc;
                *reinterpret_cast<float4 *>(p) = make_float4(aH[r][c], aH[r][c + 1], aH[r][c + 2], aH[r][c + 3]);
                if (!a.solve_only)
                    *reinterpret_cast<float4 *>(p + (size_t)D * D) = make_float4(aU[r][c], aU[r][c + 1], aU[r][c + 2], aU[r][c + 3]);
            }
    if (tid == 0) a.seg_decay[blockIdx.x] = decay;
}

// Start states: fold the segments of a sequence in order, in place (slot s: addition of segment s -> start of segment s + 1).  Bound
// by latency: eight segments are loaded ahead of their stores, behind which a load of the same array would wait.  B=1, 2 heads,
// T=256, d=64, f32, r=8: 29.2 -> 26.9 us for the call; B=2, 8 heads, T=8192, d=128: 2077 -> 2062.
__global__ void recur_scan(RecurArgs a, int st) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int e = 4 * (blockIdx.x * blockDim.x + threadIdx.x), pair = blockIdx.y;
    if (e >= st) return;
    float4 c = a.state_in ? lds4(a.state_in + (size_t)pair * st + e) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 *p = reinterpret_cast<float4 *>(a.seg + (size_t)pair * (a.P - 1) * st + e);
    const float *dec = a.seg_decay + (size_t)pair * (a.P - 1);
    for (int s0 = 0; s0 < a.P - 1; s0 += 8) {
        float4 d[8];
        float g[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (s0 + i < a.P - 1) {
                d[i] = p[(size_t)(s0 + i) * (st / 4)];
                g[i] = dec[s0 + i];
            }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (s0 + i < a.P - 1) {
                c.x = fmaf(g[i], c.x, d[i].x); c.y = fmaf(g[i], c.y, d[i].y); c.z = fmaf(g[i], c.z, d[i].z); c.w = fmaf(g[i], c.w, d[i].w);
                p[(size_t)(s0 + i) * (st / 4)] = c;
            }
    }
}

// Split of every sequence into P segments and of every segment into F parts (header comment).  Costs in units of one
// iteration of a batch; measured per batch: 5 for its norms, read and state update, 2.5 to fold it without solving, 1.2 in the
// summary kernel, and about 15 for the two launches that a split into segments needs.
struct Split { int P, L, F, Lp; };
Split choose_split(long long pairs, int T, int n_iter, int slots, long long max_states) {
    const long long nb = (T + kBatch - 1) / kBatch;          // batches of a sequence
    const long long seg_cap = max_states / pairs + 1 < nb ? max_states / pairs + 1 : nb;
    const double solve = n_iter + 5.0;
    Split best{1, (int)(nb * kBatch), 1, (int)(nb * kBatch)};
    double best_cost = 1e300;
    auto consider = [&](long long P, long long S) {          // about S parts of a sequence, in P segments
        if (P < 1 || P > seg_cap || S < P) return;
        const long long seg = (nb + P - 1) / P;
        P = (nb + seg - 1) / seg;
        long long F = (S + P - 1) / P;
        const long long part = (seg + F - 1) / F;
        F = (seg + part - 1) / part;
        const long long waves = (pairs * P * F + slots - 1) / slots;
        const double cost = (double)waves * ((double)part * solve + (double)(seg - part) * 2.5) + (P > 1 ? 15.0 + 1.2 * (double)seg : 0.0);
        if (cost < best_cost) {
            best_cost = cost;
            best = {(int)P, (int)(seg * kBatch), (int)F, (int)(part * kBatch)};
        }
    };
    long long parts[6] = {1, 2, 3, slots / pairs, 2LL * slots / pairs, 3LL * slots / pairs};
    for (long long S : parts) {
        if (S < 1) continue;
        if (S > nb) S = nb;
        consider(1, S);
        consider(S < seg_cap ? S : seg_cap, S);
    }
    return best;
}

template <int D, typename IoT>
cudaError_t launch_typed(RecurArgs a, long long pairs, int sms, void *ws, size_t ws_bytes, cudaEvent_t ev_start, cudaEvent_t ev_stop,
                         cudaStream_t stream) {
    const size_t st = state_floats(D, D);
    Split sp{1, (a.T + kBatch - 1) / kBatch * kBatch, 1, 0};
    sp.Lp = sp.L;
    if (ws) {
        const long long max_states = (long long)(ws_bytes / sizeof(float) / (st + 1));
        sp = choose_split(pairs, a.T, a.n_iter, Rc<D>::kMinBlocks * sms, max_states);
        a.seg = reinterpret_cast<float *>(ws);
        a.seg_decay = a.seg + (size_t)pairs * (sp.P - 1) * st;
    }
    a.P = sp.P; a.L = sp.L; a.F = sp.F; a.Lp = sp.Lp;
    cudaError_t err;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.stream = stream;
    if (a.P > 1) {
        cfg.gridDim = dim3((unsigned)(pairs * (a.P - 1)));
        cfg.blockDim = dim3(256);
        if ((err = cudaLaunchKernelEx(&cfg, recur_summary<D, IoT>, a)) != cudaSuccess) return err;
        const int n4 = (int)(st / (a.solve_only ? 2 : 1)) / 4;       // the solve alone needs no U
        cfg.gridDim = dim3((n4 + 127) / 128, (unsigned)pairs);
        cfg.blockDim = dim3(128);
        if ((err = cudaLaunchKernelEx(&cfg, recur_scan, a, (int)st)) != cudaSuccess) return err;
    }
    const size_t smem = spread_smem(Rc<D>::kSmem, pairs * a.P * a.F, sms);
    static SmemLimit limit;
    if ((err = limit.raise(recur_kernel<D, IoT>)) != cudaSuccess) return err;
    if (ev_start) cudaEventRecord(ev_start, stream);
    cfg.gridDim = dim3((unsigned)(pairs * a.P * a.F));
    cfg.blockDim = dim3(Rc<D>::NT);
    cfg.dynamicSmemBytes = smem;
    cfg.numAttrs = ev_start ? 0 : 1;
    err = cudaLaunchKernelEx(&cfg, recur_kernel<D, IoT>, a);
    if (ev_stop) cudaEventRecord(ev_stop, stream);
    return err;
}

cudaError_t launch_any(const RecurArgs &a, int d, int io_dtype, long long pairs, int sms, void *ws, size_t ws_bytes,
                       cudaEvent_t ev_start, cudaEvent_t ev_stop, cudaStream_t stream) {
    if (d == 128)
        return io_dtype == GKA_BF16 ? launch_typed<128, __nv_bfloat16>(a, pairs, sms, ws, ws_bytes, ev_start, ev_stop, stream)
                                    : launch_typed<128, float>(a, pairs, sms, ws, ws_bytes, ev_start, ev_stop, stream);
    return io_dtype == GKA_BF16 ? launch_typed<64, __nv_bfloat16>(a, pairs, sms, ws, ws_bytes, ev_start, ev_stop, stream)
                                : launch_typed<64, float>(a, pairs, sms, ws, ws_bytes, ev_start, ev_stop, stream);
}

}  // namespace

cudaError_t launch_fwd_recur(const FwdArgs &f, int io_dtype, void *ws, size_t ws_bytes, cudaStream_t stream) {
    RecurArgs a = {};
    a.q = f.q; a.k = f.k; a.v = f.v; a.gate = f.gate; a.lam = f.lam; a.beta = f.beta; a.alpha = f.alpha; a.out = f.out;
    a.state_in = f.state_in; a.state_out = f.state_out; a.fro_out = f.fro_out; a.device_status = f.device_status;
    a.T = f.T; a.heads = f.heads; a.n_iter = f.n_iter; a.flags = f.flags; a.solve_only = f.solve_only;
    return launch_any(a, f.d, io_dtype, (long long)f.B * f.heads, f.sms, ws, ws_bytes, f.ev_start, f.ev_stop, stream);
}

cudaError_t launch_decode_multi(float *state, const void *q, const void *k, const void *v, const float *gate,
                                const float *lam, int n_iter, void *out, int nseq, int T, int heads, int d, int io_dtype,
                                unsigned flags, const float *beta, const float *alpha, int *device_status, int sms,
                                cudaEvent_t ev_start, cudaEvent_t ev_stop, cudaStream_t stream) {
    RecurArgs a = {};
    a.q = q; a.k = k; a.v = v; a.gate = gate; a.lam = lam; a.beta = beta; a.alpha = alpha; a.out = out;
    a.state_in = state; a.state_out = state; a.device_status = device_status;
    a.T = T; a.heads = heads; a.n_iter = n_iter; a.flags = flags;
    return launch_any(a, d, io_dtype, (long long)nseq * heads, sms, nullptr, 0, ev_start, ev_stop, stream);
}

}  // namespace gka
