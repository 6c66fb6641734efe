// fp32 chunked forward and solve for the head dimensions 16 and 32 (sm_100a), whatever the I/O type and precision asked for.
//
// At these sizes the explicit H_t of a token fits the registers of a few lanes, so every token is solved against its own
// matrix: d^2 multiply-adds per iteration and nothing else, where the chunk-wise form would add 2 * 64 d for the masked
// scores (nine times d^2 at d = 16).  The unit of work is a chunk of 32 consecutive tokens of a (sequence, head) pair:
//
//   small_summary   one warp per chunk: what the chunk adds to (H, U), and its decay
//   small_scan      per pair and state element, over the chunks: additions -> states at the chunk starts, and the final state
//   small_solve     one warp per chunk: Algorithm 1 (residual form) and the read of its 32 tokens
//
// small_solve, d = 16: two lanes per token (8 rows each), 16 tokens at a time, states every 8 tokens in shared memory.
// d = 32: eight lanes per token (4 rows each), 4 runs of 8 tokens side by side.  Both hold 128 matrix elements per lane as
// 64 two-wide registers; the fp32 multiply-add pipe bounds them.
#include "gka_common.cuh"
#include "gka_tc_util.cuh"

namespace gka {
namespace {

using tcu::f2_add;
using tcu::f2_fma;
using tcu::f2_mul;
using tcu::f2_pack;
using tcu::f2_unpack;

constexpr int kCh = kSmallChunk;       // 32 tokens, one per lane where a token's data are loaded

struct SmallArgs {
    const void *q, *k, *v;
    const float *gate, *lam, *beta, *alpha, *state_in;
    void *out;
    float *state_out, *fro_out;
    float *slot;               // [pairs][chunks][2 d^2]: additions, then start states
    float *decay;              // [pairs][chunks]
    int T, heads, pairs, chunks, n_iter;
    unsigned flags;
    int solve_only;
};

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ ulonglong2 ld2x2(const float *p) { return *reinterpret_cast<const ulonglong2 *>(p); }
__device__ __forceinline__ float hsum(uint64_t v) {
    float a, b;
    f2_unpack(v, a, b);
    return a + b;
}
__device__ __forceinline__ uint64_t dup(float v) { return f2_pack(v, v); }

// A chunk's keys, values and scalars in one warp's shared memory.  Rows of d + 4 floats: 16-byte accesses of the 32 lanes
// to their own rows meet no bank conflict.
template <int D> struct Chunk {
    static constexpr int S = D + 4;
    float k[kCh][S], v[kCh][S];
    float g[kCh], lam[kCh], al[kCh];
};

// Lane l loads token l; tokens past the end have zero vectors, gate 1, lambda 1.  Keys and values are scaled by sqrt(beta_t):
// beta k k^T and beta v k^T are the plain writes of the scaled rows (Remark on the beta-augmented variant, Section 4.1).
template <int D, typename IoT>
__device__ __forceinline__ void load_chunk(const SmallArgs &a, Chunk<D> &c, size_t tok0, int nv, bool values) {
    const int l = threadIdx.x & 31;
    const bool in = l < nv;
    const size_t tok = tok0 + (size_t)(in ? l : 0) * a.heads;
    const float sb = (in && a.beta) ? sqrtf(fmaxf(a.beta[tok], 0.f)) : 1.f;
#pragma unroll
    for (int i = 0; i < D / 4; ++i) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
        if (in) {
            x = Io<IoT>::load4(reinterpret_cast<const IoT *>(a.k) + tok * D + 4 * i);
            if (values) y = Io<IoT>::load4(reinterpret_cast<const IoT *>(a.v) + tok * D + 4 * i);
        }
        st4(&c.k[l][4 * i], make_float4(sb * x.x, sb * x.y, sb * x.z, sb * x.w));
        if (values) st4(&c.v[l][4 * i], make_float4(sb * y.x, sb * y.y, sb * y.z, sb * y.w));
    }
    c.g[l] = in ? a.gate[tok] : 1.f;
    c.lam[l] = in ? a.lam[tok] : 1.f;
    c.al[l] = (in && a.alpha) ? a.alpha[tok] : 1.f;
    __syncwarp();
}

struct Where {
    int pair, chunk, nv;
    size_t tok0;
};
__device__ __forceinline__ Where where(const SmallArgs &a, int pair, int chunk) {
    Where p;
    p.pair = pair;
    p.chunk = chunk;
    const int seq = p.pair / a.heads, h = p.pair % a.heads;
    p.tok0 = ((size_t)seq * a.T + (size_t)p.chunk * kCh) * a.heads + h;
    p.nv = min(kCh, a.T - p.chunk * kCh);
    return p;
}

// ---- additions of a chunk: lane l owns d^2 / 32 consecutive elements of a row of both matrices; tokens from the last to the
// first, so that a token's weight (the product of the later gates) is a running product
constexpr int kSumWarps = 4;
template <int D, typename IoT>
__global__ void __launch_bounds__(32 * kSumWarps) small_summary(SmallArgs a) {
    constexpr int E = D * D / 32;
    __shared__ __align__(16) Chunk<D> sm[kSumWarps];
    asm volatile("griddepcontrol.wait;" ::: "memory");           // whatever wrote the inputs (programmatic launch)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int warp = threadIdx.x >> 5, l = threadIdx.x & 31;
    const long long w = (long long)blockIdx.x * kSumWarps + warp;
    if (w >= (long long)a.pairs * a.chunks) return;
    const Where p = where(a, (int)(w % a.pairs), (int)(w / a.pairs));
    Chunk<D> &c = sm[warp];
    load_chunk<D, IoT>(a, c, p.tok0, p.nv, !a.solve_only);
    const int row = l * E / D, col = l * E % D;
    uint64_t h[E / 2], u[E / 2];
#pragma unroll
    for (int i = 0; i < E / 2; ++i) h[i] = u[i] = 0ull;
    float wt = 1.f;
#pragma unroll 4
    for (int t = p.nv - 1; t >= 0; --t) {
        const uint64_t kr = dup(wt * c.k[t][row]), vr = dup(wt * c.v[t][row]);
        wt *= c.g[t];
#pragma unroll
        for (int i = 0; i < E / 4; ++i) {
            const ulonglong2 kc = ld2x2(&c.k[t][col + 4 * i]);
            h[2 * i] = f2_fma(kr, kc.x, h[2 * i]);
            h[2 * i + 1] = f2_fma(kr, kc.y, h[2 * i + 1]);
            u[2 * i] = f2_fma(vr, kc.x, u[2 * i]);
            u[2 * i + 1] = f2_fma(vr, kc.y, u[2 * i + 1]);
        }
    }
    float *dst = a.slot + ((size_t)p.pair * a.chunks + p.chunk) * 2 * D * D + l * E;
#pragma unroll
    for (int i = 0; i < E / 4; ++i) {
        *reinterpret_cast<ulonglong2 *>(dst + 4 * i) = make_ulonglong2(h[2 * i], h[2 * i + 1]);
        if (!a.solve_only) *reinterpret_cast<ulonglong2 *>(dst + D * D + 4 * i) = make_ulonglong2(u[2 * i], u[2 * i + 1]);
    }
    if (l == 0) a.decay[(size_t)p.pair * a.chunks + p.chunk] = wt;
}

// ---- start states in place and the final state: four state elements per thread, blockIdx.y = pair.  Bound by latency: a load
// behind a store to the same array waits for it, so eight chunks are loaded ahead of their stores (in a loop over the chunks every
// chunk was a round trip to memory).  64 x 8 pairs, T = 196, d = 16, 30 iterations: 91.7 -> 84.6 us for the call.
__global__ void small_scan(SmallArgs a, int st, int elements) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int e = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (e >= elements) return;
    for (int pair = blockIdx.y; pair < a.pairs; pair += gridDim.y) {
        float4 c = a.state_in ? ld4(a.state_in + (size_t)pair * st + e) : make_float4(0.f, 0.f, 0.f, 0.f);
        float4 *p = reinterpret_cast<float4 *>(a.slot + (size_t)pair * a.chunks * st + e);
        const float *dec = a.decay + (size_t)pair * a.chunks;
        for (int n0 = 0; n0 < a.chunks; n0 += 8) {
            float4 d[8];
            float g[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (n0 + i < a.chunks) {
                    d[i] = p[(size_t)(n0 + i) * (st / 4)];
                    g[i] = dec[n0 + i];
                }
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (n0 + i < a.chunks) {
                    p[(size_t)(n0 + i) * (st / 4)] = c;
                    c.x = fmaf(g[i], c.x, d[i].x); c.y = fmaf(g[i], c.y, d[i].y); c.z = fmaf(g[i], c.z, d[i].z); c.w = fmaf(g[i], c.w, d[i].w);
                }
        }
        if (a.state_out) st4(a.state_out + (size_t)pair * st + e, c);
    }
}

// ---- Algorithm 1 in residual form on R rows of a token's system per lane (x: iterate, d: increment, r: q - H_t x), L and mu
// from the norm; EXCHANGE(d2, full) gives every lane the whole increment in the order of its matrix columns.
template <int R, int C, typename Exchange>
__device__ __forceinline__ void chebyshev(const uint64_t (&H)[R][C / 2], uint64_t (&x)[R / 2], uint64_t (&r)[R / 2], float fro,
                                          float lam, int n_iter, Exchange exchange) {
    const float Lpm = fro + 2.f * lam, rho = fro / Lpm, rho2 = rho * rho, s0 = 2.f / Lpm;      // Lpm = L + mu
    const uint64_t nlam = dup(-lam), minus = dup(-1.f);
    uint64_t d[R / 2], f[C / 2];
    float om = 2.f;
#pragma unroll
    for (int i = 0; i < R / 2; ++i) {
        d[i] = f2_mul(dup(s0), r[i]);
        x[i] = 0ull;
    }
#pragma unroll 1
    for (int it = 0; it < n_iter; ++it) {
        exchange(d, f);
        om = 4.f * recip(4.f - rho2 * om);
        const uint64_t step = dup(s0 * om), mom = dup(om - 1.f);
        uint64_t y[R];
#pragma unroll
        for (int m = 0; m < R; ++m) y[m] = f2_mul(H[m][0], f[0]);
#pragma unroll
        for (int c = 1; c < C / 2; ++c)
#pragma unroll
            for (int m = 0; m < R; ++m) y[m] = f2_fma(H[m][c], f[c], y[m]);
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
            x[i] = f2_add(x[i], d[i]);
            r[i] = f2_fma(minus, f2_pack(hsum(y[2 * i]), hsum(y[2 * i + 1])), r[i]);
            d[i] = f2_fma(step, f2_fma(nlam, x[i], r[i]), f2_mul(mom, d[i]));
        }
    }
#pragma unroll
    for (int i = 0; i < R / 2; ++i) x[i] = f2_add(x[i], d[i]);
}

// H <- gam H + k k^T on a lane's R rows and C columns, returns the sum of squares of what it holds
template <int R, int C>
__device__ __forceinline__ float write_key(uint64_t (&H)[R][C / 2], const uint64_t (&kc)[C / 2], const float (&kr)[R], float gam) {
    const uint64_t g2 = dup(gam);
    uint64_t sq[2] = {0ull, 0ull};
#pragma unroll
    for (int m = 0; m < R; ++m) {
        const uint64_t k2 = dup(kr[m]);
#pragma unroll
        for (int i = 0; i < C / 2; ++i) {
            H[m][i] = f2_fma(g2, H[m][i], f2_mul(k2, kc[i]));
            sq[i & 1] = f2_fma(H[m][i], H[m][i], sq[i & 1]);
        }
    }
    return hsum(f2_add(sq[0], sq[1]));
}

template <typename IoT, int R>
__device__ __forceinline__ void store_rows(IoT *dst, const uint64_t (&o)[R / 2]) {
#pragma unroll
    for (int i = 0; i < R / 4; ++i) {
        float4 v;
        f2_unpack(o[2 * i], v.x, v.y);
        f2_unpack(o[2 * i + 1], v.z, v.w);
        Io<IoT>::store4(dst + 4 * i, v);
    }
}

// Blocks of two warps, 8 warps per SM: with 12 (168 registers, some spilled) this kernel took 95 us instead of 80 at 64 x 8 pairs,
// T = 196, d = 16, 30 iterations (multiply-add pipe 69 % of active cycles; the call: 84 us, 3997 us before on the chunk-wise kernel
// zero-extended to 64 channels).
constexpr int kSolveWarps = 2;
constexpr int kSolveBlocks = 4;

template <int D> struct SolveMem;
template <> struct SolveMem<16> {
    Chunk<16> c;
    float q[kCh][20];
    float H[4][16 * 16 + 4], U[4][16 * 16 + 4];   // states before tokens 0, 8, 16, 24; rows 8 .. 15 shifted by 4 floats
};
template <> struct SolveMem<32> {
    Chunk<32> c;
    float q[kCh][36];
    float U[32 * 32 + 32];                        // state at the chunk's start; every four rows shifted by 4 floats
    float x[2][4][36];                            // the four groups' iterates, double-buffered
};

template <typename IoT>
__device__ __forceinline__ void solve_chunk(const SmallArgs &a, const Where &p, SolveMem<16> &sm, const float *start) {
    const int l = threadIdx.x & 31, g = l >> 1, hf = l & 1, row0 = 8 * hf;
    Chunk<16> &c = sm.c;
    {   // ---- states every 8 tokens: lane l carries 8 elements of row l / 2 of both matrices through the chunk
        const int row = l >> 1, col = 8 * (l & 1), at = row * 16 + (row >> 3) * 4 + col;
        uint64_t h[4], u[4];
        const float *s0 = start + row * 16 + col;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const ulonglong2 h4 = ld2x2(s0 + 4 * i);
            ulonglong2 u4 = make_ulonglong2(0ull, 0ull);
            if (!a.solve_only) u4 = ld2x2(s0 + 256 + 4 * i);
            h[2 * i] = h4.x; h[2 * i + 1] = h4.y; u[2 * i] = u4.x; u[2 * i + 1] = u4.y;
        }
#pragma unroll 1
        for (int s = 0; s < 4; ++s) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                *reinterpret_cast<ulonglong2 *>(&sm.H[s][at + 4 * i]) = make_ulonglong2(h[2 * i], h[2 * i + 1]);
                *reinterpret_cast<ulonglong2 *>(&sm.U[s][at + 4 * i]) = make_ulonglong2(u[2 * i], u[2 * i + 1]);
            }
#pragma unroll 4
            for (int t = 8 * s; t < 8 * s + 8; ++t) {
                const uint64_t g2 = dup(c.g[t]), kr = dup(c.k[t][row]), vr = dup(c.v[t][row]);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const ulonglong2 kc = ld2x2(&c.k[t][col + 4 * i]);
                    h[2 * i] = f2_fma(g2, h[2 * i], f2_mul(kr, kc.x));
                    h[2 * i + 1] = f2_fma(g2, h[2 * i + 1], f2_mul(kr, kc.y));
                    u[2 * i] = f2_fma(g2, u[2 * i], f2_mul(vr, kc.x));
                    u[2 * i + 1] = f2_fma(g2, u[2 * i + 1], f2_mul(vr, kc.y));
                }
            }
        }
        __syncwarp();
    }
    // ---- lanes 2 g, 2 g + 1: tokens 2 g and 2 g + 1; H in registers, the columns of the lane's own half first
    const int s = g >> 2, tl = 2 * (g & 3), t8 = 8 * s, own = row0, other = 8 - row0;
    auto columns = [&](const float *rowp, uint64_t (&o)[8]) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const ulonglong2 u4 = ld2x2(rowp + own + 4 * i), w4 = ld2x2(rowp + other + 4 * i);
            o[2 * i] = u4.x; o[2 * i + 1] = u4.y; o[4 + 2 * i] = w4.x; o[5 + 2 * i] = w4.y;
        }
    };
    auto rows = [&](const float *rowp, float (&o)[8]) {
        const float4 r0 = ld4(rowp + row0), r1 = ld4(rowp + row0 + 4);
        o[0] = r0.x; o[1] = r0.y; o[2] = r0.z; o[3] = r0.w; o[4] = r1.x; o[5] = r1.y; o[6] = r1.z; o[7] = r1.w;
    };
    uint64_t H[8][8];
    {
        float w[6], z = 1.f;
#pragma unroll
        for (int j = 5; j >= 0; --j) {
            w[j] = j < tl ? z : 0.f;
            z *= j < tl ? c.g[t8 + j] : 1.f;
        }
        const uint64_t z2 = dup(z);
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            columns(&sm.H[s][(row0 + m) * 16 + 4 * hf], H[m]);
#pragma unroll
            for (int i = 0; i < 8; ++i) H[m][i] = f2_mul(z2, H[m][i]);
        }
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            uint64_t kc[8];
            float kr[8];
            columns(c.k[t8 + j], kc);
            rows(c.k[t8 + j], kr);
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const uint64_t k2 = dup(w[j] * kr[m]);
#pragma unroll
                for (int i = 0; i < 8; ++i) H[m][i] = f2_fma(k2, kc[i], H[m][i]);
            }
        }
    }
    auto exchange = [&](const uint64_t (&d)[4], uint64_t (&f)[8]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f[i] = d[i];
            f[4 + i] = __shfl_xor_sync(0xffffffffu, d[i], 1);
        }
    };
#pragma unroll 1
    for (int e = 0; e < 2; ++e) {
        const int t = 2 * g + e;
        const size_t tok = p.tok0 + (size_t)t * a.heads;
        float ss;
        {
            uint64_t kc[8];
            float kr[8];
            columns(c.k[t], kc);
            rows(c.k[t], kr);
            ss = write_key<8, 16>(H, kc, kr, c.g[t]);
        }
        ss += __shfl_xor_sync(0xffffffffu, ss, 1);
        const float fro = sqrtf(ss);
        if (a.fro_out && hf == 0 && t < p.nv) a.fro_out[tok] = fro;
        const float lam = (a.flags & GKA_FLAG_ADAPTIVE_LAMBDA) ? c.lam[t] * fro : c.lam[t];
        uint64_t x[4], r[4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const ulonglong2 q4 = ld2x2(&sm.q[t][row0 + 4 * i]);
            r[2 * i] = q4.x; r[2 * i + 1] = q4.y;
        }
        chebyshev<8, 16>(H, x, r, fro, lam, a.n_iter, exchange);
        uint64_t o[4] = {x[0], x[1], x[2], x[3]};
        if (!a.solve_only) {
            if (a.alpha) {                       // alpha-connection (Section 4.3): the read takes alpha x + (1 - alpha) q
                const uint64_t al = dup(c.al[t]), minus = dup(-1.f);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const ulonglong2 q4 = ld2x2(&sm.q[t][row0 + 4 * i]);
                    x[2 * i] = f2_fma(al, f2_fma(minus, q4.x, x[2 * i]), q4.x);
                    x[2 * i + 1] = f2_fma(al, f2_fma(minus, q4.y, x[2 * i + 1]), q4.y);
                }
            }
            // ---- o = zeta (U x) + sum_j Gamma[t][j] v_j (k_j . x) over the tokens since the last stored state
            uint64_t z[8], acc[4] = {0ull, 0ull, 0ull, 0ull};
            exchange(x, z);
            float w = 1.f;
#pragma unroll 2
            for (int j = 7; j >= 0; --j) {
                const ulonglong2 k0 = ld2x2(&c.k[t8 + j][own]), k1 = ld2x2(&c.k[t8 + j][own + 4]);
                float dot = hsum(f2_add(f2_fma(k0.x, z[0], f2_mul(k0.y, z[1])), f2_fma(k1.x, z[2], f2_mul(k1.y, z[3]))));
                dot += __shfl_xor_sync(0xffffffffu, dot, 1);
                const bool in = j <= tl + e;
                const uint64_t s2 = dup(in ? w * dot : 0.f);
                const ulonglong2 v0 = ld2x2(&c.v[t8 + j][row0]), v1 = ld2x2(&c.v[t8 + j][row0 + 4]);
                acc[0] = f2_fma(s2, v0.x, acc[0]); acc[1] = f2_fma(s2, v0.y, acc[1]);
                acc[2] = f2_fma(s2, v1.x, acc[2]); acc[3] = f2_fma(s2, v1.y, acc[3]);
                w *= in ? c.g[t8 + j] : 1.f;
            }
            const uint64_t w2 = dup(w);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                float y[2];
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    uint64_t u[8];
                    columns(&sm.U[s][(row0 + 2 * m + b) * 16 + 4 * hf], u);
                    uint64_t sum = f2_mul(u[0], z[0]);
#pragma unroll
                    for (int i = 1; i < 8; ++i) sum = f2_fma(u[i], z[i], sum);
                    y[b] = hsum(sum);
                }
                o[m] = f2_fma(w2, f2_pack(y[0], y[1]), acc[m]);
            }
        }
        if (t < p.nv) store_rows<IoT, 8>(reinterpret_cast<IoT *>(a.out) + tok * 16 + row0, o);
    }
}

template <typename IoT>
__device__ __forceinline__ void solve_chunk(const SmallArgs &a, const Where &p, SolveMem<32> &sm, const float *start) {
    const int l = threadIdx.x & 31, g = l >> 3, li = l & 7, row0 = 4 * li;
    Chunk<32> &c = sm.c;
    if (!a.solve_only) {
        for (int e = 4 * l; e < 32 * 32; e += 128) st4(&sm.U[e + (e >> 7) * 4], ld4(start + 32 * 32 + e));
    }
    // ---- H before token 8 g: the chunk's start state and the tokens before that one
    uint64_t H[4][16];
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int i = 0; i < 16; ++i) H[m][i] = 0ull;
    auto columns = [&](const float *rowp, uint64_t (&o)[16]) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const ulonglong2 u4 = ld2x2(rowp + 4 * i);
            o[2 * i] = u4.x; o[2 * i + 1] = u4.y;
        }
    };
    float w = 1.f;
#pragma unroll 1
    for (int j = 23; j >= 0; --j) {
        uint64_t kc[16];
        columns(c.k[j], kc);
        const float4 k4 = ld4(&c.k[j][row0]);
        const bool in = j < 8 * g;
        const float wj = in ? w : 0.f, kr[4] = {wj * k4.x, wj * k4.y, wj * k4.z, wj * k4.w};
        w *= in ? c.g[j] : 1.f;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const uint64_t k2 = dup(kr[m]);
#pragma unroll
            for (int i = 0; i < 16; ++i) H[m][i] = f2_fma(k2, kc[i], H[m][i]);
        }
    }
    {
        const uint64_t w2 = dup(w);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            uint64_t h[16];
            columns(start + (row0 + m) * 32, h);
#pragma unroll
            for (int i = 0; i < 16; ++i) H[m][i] = f2_fma(w2, h[i], H[m][i]);
        }
    }
    int buf = 0;
    auto exchange = [&](const uint64_t (&d)[2], uint64_t (&f)[16]) {     // one barrier per iteration: the buffers alternate
        *reinterpret_cast<ulonglong2 *>(&sm.x[buf][g][row0]) = make_ulonglong2(d[0], d[1]);
        __syncwarp();
        columns(sm.x[buf][g], f);
        buf ^= 1;
    };
#pragma unroll 1
    for (int e = 0; e < 8; ++e) {
        const int t = 8 * g + e;
        const size_t tok = p.tok0 + (size_t)t * a.heads;
        float ss;
        {
            uint64_t kc[16];
            columns(c.k[t], kc);
            const float4 k4 = ld4(&c.k[t][row0]);
            const float kr[4] = {k4.x, k4.y, k4.z, k4.w};
            ss = write_key<4, 32>(H, kc, kr, c.g[t]);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const float fro = sqrtf(ss);
        if (a.fro_out && li == 0 && t < p.nv) a.fro_out[tok] = fro;
        const float lam = (a.flags & GKA_FLAG_ADAPTIVE_LAMBDA) ? c.lam[t] * fro : c.lam[t];
        const ulonglong2 q4 = ld2x2(&sm.q[t][row0]);
        uint64_t x[2], r[2] = {q4.x, q4.y};
        chebyshev<4, 32>(H, x, r, fro, lam, a.n_iter, exchange);
        uint64_t o[2] = {x[0], x[1]};
        if (!a.solve_only) {
            if (a.alpha) {                       // alpha-connection (Section 4.3): the read takes alpha x + (1 - alpha) q
                const uint64_t al = dup(c.al[t]), minus = dup(-1.f);
                x[0] = f2_fma(al, f2_fma(minus, q4.x, x[0]), q4.x);
                x[1] = f2_fma(al, f2_fma(minus, q4.y, x[1]), q4.y);
            }
            // ---- o = zeta (U_0 x) + sum_j Gamma[t][j] v_j (k_j . x); lane li has the products of keys li, li + 8, ...
            uint64_t z[16], acc[2] = {0ull, 0ull};
            exchange(x, z);
            float wt = 1.f;
#pragma unroll 1
            for (int b = 3; b >= 0; --b) {
                uint64_t dot = 0ull;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const ulonglong2 k4 = ld2x2(&c.k[8 * b + li][4 * i]);
                    dot = f2_fma(k4.x, z[2 * i], f2_fma(k4.y, z[2 * i + 1], dot));
                }
                const float s = hsum(dot);
#pragma unroll
                for (int jj = 7; jj >= 0; --jj) {
                    const int j = 8 * b + jj;
                    const bool in = j <= t;
                    const float sj = __shfl_sync(0xffffffffu, s, jj, 8);
                    const uint64_t s2 = dup(in ? wt * sj : 0.f);
                    const ulonglong2 v4 = ld2x2(&c.v[j][row0]);
                    acc[0] = f2_fma(s2, v4.x, acc[0]);
                    acc[1] = f2_fma(s2, v4.y, acc[1]);
                    wt *= in ? c.g[j] : 1.f;
                }
            }
            const uint64_t w2 = dup(wt);
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                float y[2];
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    uint64_t u[16];
                    columns(&sm.U[(row0 + 2 * m + b) * 32 + li * 4], u);
                    uint64_t sum = f2_mul(u[0], z[0]);
#pragma unroll
                    for (int i = 1; i < 16; ++i) sum = f2_fma(u[i], z[i], sum);
                    y[b] = hsum(sum);
                }
                o[m] = f2_fma(w2, f2_pack(y[0], y[1]), acc[m]);
            }
        }
        if (t < p.nv) store_rows<IoT, 4>(reinterpret_cast<IoT *>(a.out) + tok * 32 + row0, o);
    }
}

template <int D, typename IoT>
__global__ void __launch_bounds__(32 * kSolveWarps, kSolveBlocks) small_solve(SmallArgs a) {
    __shared__ __align__(16) SolveMem<D> sms[kSolveWarps];
    const int warp = threadIdx.x >> 5, l = threadIdx.x & 31;
    const long long w = (long long)blockIdx.x * kSolveWarps + warp;
    if (w >= (long long)a.pairs * a.chunks) return;
    // All pairs' first chunks, then their second ones, ... (as in the summary kernel): neighbouring warps are heads of the same
    // tokens.  16 x 8 pairs, T = 1024, d = 16, 10 iterations: 67.0 -> 65.3 us for the call; 64 x 8, T = 196, 30: 92.8 -> 91.8.  A
    // last chunk of at most 16 tokens with one token per lane pair (half its time): 89.8 there, but +2 % on full chunks.
    const Where p = where(a, (int)(w % a.pairs), (int)(w / a.pairs));
    SolveMem<D> &sm = sms[warp];
    load_chunk<D, IoT>(a, sm.c, p.tok0, p.nv, !a.solve_only);
#pragma unroll
    for (int i = 0; i < D / 4; ++i) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (l < p.nv) x = Io<IoT>::load4(reinterpret_cast<const IoT *>(a.q) + (p.tok0 + (size_t)l * a.heads) * D + 4 * i);
        st4(&sm.q[l][4 * i], x);
    }
    __syncwarp();
    asm volatile("griddepcontrol.wait;" ::: "memory");           // the scan's start states
    solve_chunk<IoT>(a, p, sm, a.slot + ((size_t)p.pair * a.chunks + p.chunk) * 2 * D * D);
}

template <int D, typename IoT>
cudaError_t launch_typed(const SmallArgs &a, cudaEvent_t ev_start, cudaEvent_t ev_stop, cudaStream_t stream) {
    const long long units = (long long)a.pairs * a.chunks;
    const int st = 2 * D * D, elements = a.solve_only ? D * D : st;
    cudaError_t err;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.stream = stream;
    cfg.gridDim = dim3((unsigned)((units + kSumWarps - 1) / kSumWarps));
    cfg.blockDim = dim3(32 * kSumWarps);
    if ((err = cudaLaunchKernelEx(&cfg, small_summary<D, IoT>, a)) != cudaSuccess) return err;
    cfg.gridDim = dim3((unsigned)((elements / 4 + 127) / 128), (unsigned)(a.pairs < 65535 ? a.pairs : 65535));
    cfg.blockDim = dim3(elements / 4 < 128 ? elements / 4 : 128);
    if ((err = cudaLaunchKernelEx(&cfg, small_scan, a, st, elements)) != cudaSuccess) return err;
    if (ev_start) cudaEventRecord(ev_start, stream);
    cfg.numAttrs = ev_start ? 0 : 1;
    cfg.gridDim = dim3((unsigned)((units + kSolveWarps - 1) / kSolveWarps));
    cfg.blockDim = dim3(32 * kSolveWarps);
    err = cudaLaunchKernelEx(&cfg, small_solve<D, IoT>, a);
    if (ev_stop) cudaEventRecord(ev_stop, stream);
    return err;
}

}  // namespace

cudaError_t launch_fwd_small(const FwdArgs &f, int io_dtype, void *ws, cudaStream_t stream) {
    SmallArgs a = {};
    a.q = f.q; a.k = f.k; a.v = f.v; a.gate = f.gate; a.lam = f.lam; a.beta = f.beta; a.alpha = f.alpha; a.out = f.out;
    a.state_in = f.state_in; a.state_out = f.state_out; a.fro_out = f.fro_out;
    a.T = f.T; a.heads = f.heads; a.pairs = f.B * f.heads; a.chunks = small_chunks_of(f.T); a.n_iter = f.n_iter;
    a.flags = f.flags; a.solve_only = f.solve_only;
    a.slot = reinterpret_cast<float *>(ws);
    a.decay = a.slot + (size_t)a.pairs * a.chunks * 2 * f.d * f.d;
    if (f.d == 16)
        return io_dtype == GKA_BF16 ? launch_typed<16, __nv_bfloat16>(a, f.ev_start, f.ev_stop, stream)
                                    : launch_typed<16, float>(a, f.ev_start, f.ev_stop, stream);
    return io_dtype == GKA_BF16 ? launch_typed<32, __nv_bfloat16>(a, f.ev_start, f.ev_stop, stream)
                                : launch_typed<32, float>(a, f.ev_start, f.ev_stop, stream);
}

}  // namespace gka
