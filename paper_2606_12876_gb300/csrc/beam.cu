// aq_beam_search: the code update of Alg. 1 ("update assignments b using beam search"; App. C:
// the search for codeword combinations that minimise the error of the layer's outputs), in
// the reading stated in aq.h: every (row o, group g), with the row's other groups at their
// current codes, chooses its M codes by a beam search of width K over the books in order,
// minimising the row's Drop-by-Drop objective sum_k lambda_k e^(k) S e^(k)^T (Sec. 5, the
// trace form of Sec. 2.2 with S the symmetric part of H). The terms that depend on the
// group's codes are delta_k^T S_gg delta_k + 2 delta_k^T h_k, with
// delta_k = w_g - s_o * (sum_{j<k} C_j[b_j]) and h_k = (S e^(k))_g - S_gg e^(k)_g.
//
// Kernels (all fp32):
//   beam_resid_kernel  E_k[o][i] = W[o][i] - s_o * (sum_{j<k} C_j[b_j])  (current codes)
//   beam_sym_kernel    S = (H + H^T) / 2
//   beam_gemm_kernel   V_k = E_k S (tiled, CUDA cores: the cross terms need fp32)
//   beam_kernel        one warp per (row, group): h_k, then the beam over the books
#include <cfloat>

#include "aq_internal.cuh"

namespace aq {
namespace {

constexpr int kBeamMaxK = 16;
constexpr int kBeamWarps = 8;

// The prefix weights lambda_1..lambda_M, passed by value.
struct Lambdas {
    float v[8];
};

// Workspace: [status 256 B][S: in*in][E: M*out*in][V: M*out*in] (fp32)
inline size_t beam_s_off() { return kWsStatusBytes; }
inline size_t beam_e_off(const Dims& d) { return round_up(beam_s_off() + (size_t)d.in * d.in * 4, 256); }
inline size_t beam_v_off(const Dims& d) {
    return round_up(beam_e_off(d) + (size_t)d.M * d.out * d.in * 4, 256);
}

template <int BDT, int SDT>
__global__ void beam_resid_kernel(const uint16_t* __restrict__ w, const void* __restrict__ codes,
                                  const uint16_t* __restrict__ books,
                                  const uint16_t* __restrict__ scales, float* __restrict__ E,
                                  int out, int in, int ng, int M, int B) {
    pdl_wait();
    pdl_launch_dependents();
    const size_t n = (size_t)out * ng;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (size_t)gridDim.x * blockDim.x) {
        const int o = (int)(t / ng), g = (int)(t % ng);
        const float s = bits_to_f32<SDT>(scales[o]);
        float wv[8], P[8];
        unpack8<BDT>(*(const uint4*)(w + (size_t)o * in + (size_t)g * 8), wv);
#pragma unroll
        for (int e = 0; e < 8; ++e) P[e] = 0.0f;
        for (int k = 0; k < M; ++k) {
            const size_t ci = ((size_t)o * ng + g) * M + k;
            const uint32_t c = B == 16 ? ((const uint16_t*)codes)[ci] : ((const uint8_t*)codes)[ci];
            float cv[8];
            unpack8<BDT>(*(const uint4*)(books + (((size_t)k << B) + c) * 8), cv);
            float* dst = E + ((size_t)k * out + o) * in + (size_t)g * 8;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                P[e] += cv[e];
                dst[e] = wv[e] - s * P[e];
            }
        }
    }
}

__global__ void beam_sym_kernel(const void* __restrict__ h, int h_dt, float* __restrict__ S, int in) {
    pdl_wait();
    pdl_launch_dependents();
    const size_t n = (size_t)in * in;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (size_t)gridDim.x * blockDim.x) {
        const size_t i = t / in, j = t % in;
        float a, b;
        if (h_dt == AQ_F32) {
            a = ((const float*)h)[i * in + j];
            b = ((const float*)h)[j * in + i];
        } else {
            a = bits_to_f32<AQ_BF16>(((const uint16_t*)h)[i * in + j]);
            b = bits_to_f32<AQ_BF16>(((const uint16_t*)h)[j * in + i]);
        }
        S[t] = (a + b) * 0.5f;
    }
}

// C[r][j] = sum_i A[r][i] * S[i][j] for r < rows, j < in (A = E of every prefix, rows = M*out).
// Bound: the fp32 FMA pipe (2 * M * out * in^2 operations on the CUDA cores), with shared memory close
// behind: a 16-byte load of a warp is four wavefronts even where lanes share it, so 8 x 8 outputs per
// thread (16 words for 64 FMAs) cost as many clocks of shared memory as of FMAs. T x T tiles of C; at
// T = 128 a thread has 8 x 16 outputs (24 words for 128 FMAs; 128 threads), in packed fp32 pairs (1024 x
// 4096, M = 4, the call: 6.69 ms with 8 x 8, 6.35 with 8 x 16; with A's elements stored twice, which
// saves the packing moves, 7.24). 16-deep k steps: the next step's tiles travel (A through registers,
// which transposes it, S by cp.async) while the current ones are multiplied, and two shared buffers
// leave one barrier per step. Every output is one chain of fused multiply-adds over i in ascending
// order from +0, so the values do not depend on the tile. T = 128, or 64 where 128 gives fewer tiles
// than SMs.
template <int T>
constexpr int kBeamGemmThreads = T == 128 ? 128 : 256;
template <int T>
__global__ void __launch_bounds__(kBeamGemmThreads<T>, 2) beam_gemm_kernel(const float* __restrict__ A,
                                                                           const float* __restrict__ S,
                                                                           float* __restrict__ C, int rows, int in) {
    constexpr int NT = kBeamGemmThreads<T>, TX = NT / 16;      // thread columns
    constexpr int N = T / 64, NC = T / (4 * TX);               // 4-row and 4-column parts per thread
    constexpr int LD = T * 4 / NT;         // 16-byte loads per thread of a 16-deep tile
    __shared__ __align__(16) float As[2][16][T + 4], Bs[2][16][T];
    pdl_wait();
    pdl_launch_dependents();
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int c0 = blockIdx.x * T, nk = (in + 15) / 16;
    for (int r0 = blockIdx.y * T; r0 < rows; r0 += gridDim.y * T) {
        float4 ra[LD];
        auto load = [&](int k0, int buf) {
#pragma unroll
            for (int l = 0; l < LD; ++l) {
                const int i = tid + l * NT, r = r0 + i / 4, k = k0 + (i & 3) * 4;
                ra[l] = r < rows && k < in ? __ldg((const float4*)(A + (size_t)r * in + k)) : float4{};
                const int kb = k0 + i / (T / 4), cc = c0 + i % (T / 4) * 4;
                float4* dst = (float4*)&Bs[buf][i / (T / 4)][i % (T / 4) * 4];
                if (kb < in && cc < in) cp_async16(dst, S + (size_t)kb * in + cc);
                else *dst = float4{};
            }
            cp_async_commit();
        };
        auto store = [&](int buf) {
#pragma unroll
            for (int l = 0; l < LD; ++l) {
                const int i = tid + l * NT, r = i / 4, k = (i & 3) * 4;
                As[buf][k][r] = ra[l].x;
                As[buf][k + 1][r] = ra[l].y;
                As[buf][k + 2][r] = ra[l].z;
                As[buf][k + 3][r] = ra[l].w;
            }
        };
        float2 acc[4 * N][2 * NC];
#pragma unroll
        for (int u = 0; u < 4 * N; ++u)
#pragma unroll
            for (int v = 0; v < 2 * NC; ++v) acc[u][v] = make_float2(0.0f, 0.0f);
        load(0, 0);
        store(0);
        cp_async_wait<0>();
        __syncthreads();
        for (int kt = 0; kt < nk; ++kt) {
            const int buf = kt & 1;
            if (kt + 1 < nk) load((kt + 1) * 16, buf ^ 1);
#pragma unroll
            for (int kk = 0; kk < 16; ++kk) {
                float4 a4[N], b4[NC];
#pragma unroll
                for (int h = 0; h < N; ++h) a4[h] = *(const float4*)&As[buf][kk][h * 64 + ty * 4];
#pragma unroll
                for (int g = 0; g < NC; ++g) b4[g] = *(const float4*)&Bs[buf][kk][g * 4 * TX + tx * 4];
#pragma unroll
                for (int h = 0; h < N; ++h) {
                    const float av[4] = {a4[h].x, a4[h].y, a4[h].z, a4[h].w};
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int g = 0; g < NC; ++g) {
                            const float2 aa = make_float2(av[u], av[u]);
                            acc[4 * h + u][2 * g] = ffma2(aa, make_float2(b4[g].x, b4[g].y), acc[4 * h + u][2 * g]);
                            acc[4 * h + u][2 * g + 1] =
                                ffma2(aa, make_float2(b4[g].z, b4[g].w), acc[4 * h + u][2 * g + 1]);
                        }
                }
            }
            if (kt + 1 < nk) store(buf ^ 1);
            cp_async_wait<0>();
            __syncthreads();
        }
#pragma unroll
        for (int u = 0; u < 4 * N; ++u)
#pragma unroll
            for (int g = 0; g < NC; ++g) {
                const int r = r0 + (u >> 2) * 64 + ty * 4 + (u & 3), c = c0 + g * 4 * TX + tx * 4;
                if (r < rows && c < in)    // in is a multiple of 8
                    *(float4*)(C + (size_t)r * in + c) = make_float4(acc[u][2 * g].x, acc[u][2 * g].y,
                                                                     acc[u][2 * g + 1].x, acc[u][2 * g + 1].y);
            }
    }
}

// Candidate order: smaller score first, then smaller index (parent rank * 2^B + codeword).
__device__ __forceinline__ bool before(float a, int ia, float b, int ib) {
    return a < b || (a == b && ia < ib);
}

// One warp per (row, group), the rows of one group handled by the warps of a CTA (the group's
// block S_gg and the codebooks are staged once per CTA). Per book t, the candidates are every
// (state, codeword) pair, index j = rank * 2^B + c, and the K first in (score, index) order are
// kept. Bound: issue. Scoring every candidate by its definition costs about 100 operations (the
// 8 x 8 quadratic form); instead
//  1. every candidate gets an estimate of its score from the expanded form
//     A_r + C_t[c] . G_r + lambda s^2 (C_t[c]^T S_gg C_t[c]),  G_r = -2 lambda s (S_gg u_r + h),
//     u_r = w_g - s P_r: about six operations, G_r in registers, the last term tabled per CTA. Each lane
//     keeps its smallest estimate per state and per codeword;
//  2. the keep-th smallest of the 32 lanes' smallest estimates is at least the keep-th smallest
//     estimate; with both forms' rounding errors below eps, every candidate among the K first has an
//     estimate of at most that plus 2 eps. Candidates whose state and codeword minima are in reach
//     (typically about keep + 2 of up to 4096) are listed;
//  3. the listed candidates are scored by the definition, in the fixed order of operations, and
//     the K first of them are the K first of all: the result is the full search's, bit for bit.
// eps: both forms add up products bounded by the terms of T_r = |score_r| + lambda (D^T |S_gg| D +
// 2 D . |h|), D = |w_g| + |s| (|P_r| + max_c |C_t[c]|), each term with at most about 30 roundings of
// 2^-24 and the expanded form with four such sums: eps = 2^-16 max_r T_r covers their sum twice. What products
// lose below fp32's normal range (2^-149 each, times the factors that follow) is at most about
// 2^-140 lambda (1 + |s|)^2 (2 + max |C_t| + max D), and is kept below eps / 4; the estimates are not used where
// that, C_t[c]^T S_gg C_t[c] or lambda s^2 is out of range (codebooks of 2^62 and scales of 2^-68 overflowed the
// table, and only the smallest codewords were found).
// Where the list would overflow (many equal scores) or T_r is out of range, every candidate is scored by the
// definition, once, and the list holds the best so far. (512 x 2048, M = 4, K = 8: equal codewords in every book
// 9.9 ms, half of the rows of zero scale 5.7, half of the inputs without energy in H, which needs no scores,
// 1.2; scored anew for each of the K, 60.3, 30.8 and 35.7; sorted lists per lane 14.4, 18.2 and 19.5.)
// (rows x inputs 1024 x 4096, M = 4, K = 8: scoring every candidate with sorted lists per lane took
// 75 ms, this form 3.9 ms.)
constexpr int kBeamList = 256;     // listed candidates per warp

// A warp's scratch.
struct BeamWarp {
    float h[8][8];                                     // h_k of every prefix
    struct States {
        float P[kBeamMaxK][8];
        float score[kBeamMaxK];
        unsigned long long codes[kBeamMaxK];           // code of book k in byte k
    } st[2];
    float G[kBeamMaxK][8], A[kBeamMaxK];
    float lscore[kBeamList];
    int lidx[kBeamList];
};

// Smallest estimates over this lane's codewords (c = lane + 32 i) for RC states at once: per state in
// mr, per codeword in mc[32 i + lane] (the first RC states, or together with the earlier ones').
template <int RC, bool FIRST>
__device__ __forceinline__ void beam_estimates(const float4* lo, const float4* hi, const float* Q, float F,
                                               const float* G, const float* A, int lane, float* mr,
                                               float* mc) {
    // two states per packed fp32 operation, the codeword's elements doubled
    float2 g2[RC / 2][8], a2[RC / 2];
#pragma unroll
    for (int r = 0; r < RC; r += 2) {
#pragma unroll
        for (int e = 0; e < 8; ++e) g2[r / 2][e] = make_float2(G[r * 8 + e], G[r * 8 + 8 + e]);
        a2[r / 2] = make_float2(A[r], A[r + 1]);
        mr[r] = mr[r + 1] = FLT_MAX;
    }
#pragma unroll 2
    for (int i = 0; i < 8; ++i) {
        const int c = lane + 32 * i;
        const float4 x = lo[c], y = hi[c];
        const float cv[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
        const float fq = F * Q[c];
        float m = FIRST ? FLT_MAX : mc[c];
#pragma unroll
        for (int r = 0; r < RC; r += 2) {
            float2 t = add2(a2[r / 2], make_float2(fq, fq));
#pragma unroll
            for (int e = 0; e < 8; ++e) t = ffma2(make_float2(cv[e], cv[e]), g2[r / 2][e], t);
            mr[r] = fminf(mr[r], t.x);
            mr[r + 1] = fminf(mr[r + 1], t.y);
            m = fminf(fminf(m, t.x), t.y);
        }
        mc[c] = m;
    }
}

// The K-th smallest (0-based rank k) of the 32 lanes' values: a bitonic sort across the lanes.
__device__ __forceinline__ float warp_kth(float v, int k, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const float o = __shfl_xor_sync(0xffffffffu, v, stride);
            const bool up = (lane & size) == 0, low = (lane & stride) == 0;
            v = up == low ? fminf(v, o) : fmaxf(v, o);
        }
    return __shfl_sync(0xffffffffu, v, k);
}

// The candidates in reach: bit r of *rmask, bit i of *cmask where the lane's smallest estimate of
// state r, of codeword lane + 32 i, is within `slack` of the keep-th smallest of the lanes' smallest
// (at most RC * NCH states; mc: 256 floats of scratch, read and written by the same lanes).
template <int RC, int NCH>
__device__ __forceinline__ void beam_reach(const float4* lo, const float4* hi, const float* Q, float F,
                                           const float* G, const float* A, float* mc, int lane, int keep,
                                           float slack, uint32_t* rmask, uint32_t* cmask) {
    float mr[RC * NCH];
    beam_estimates<RC, true>(lo, hi, Q, F, G, A, lane, mr, mc);
    if constexpr (NCH == 2) beam_estimates<RC, false>(lo, hi, Q, F, G + RC * 8, A + RC, lane, mr + RC, mc);
    float m = mr[0];
#pragma unroll
    for (int r = 1; r < RC * NCH; ++r) m = fminf(m, mr[r]);
    const float reach = warp_kth(m, keep - 1, lane) + slack;
    *rmask = *cmask = 0;
#pragma unroll
    for (int r = 0; r < RC * NCH; ++r) *rmask |= (mr[r] <= reach ? 1u : 0u) << r;
#pragma unroll
    for (int i = 0; i < 8; ++i) *cmask |= (mc[lane + 32 * i] <= reach ? 1u : 0u) << i;
}

template <int BDT, int SDT>
__global__ void __launch_bounds__(kBeamWarps * 32, 2)
beam_kernel(const uint16_t* __restrict__ w, const uint16_t* __restrict__ books,
            const uint16_t* __restrict__ scales, const float* __restrict__ S,
            const float* __restrict__ E, const float* __restrict__ V, void* __restrict__ codes_out,
            Lambdas lam, int out, int in, int ng, int M, int B, int K) {
    extern __shared__ __align__(16) float bsm[];
    const int nb = 1 << B;
    float4* lo = (float4*)bsm;                         // [M][nb] codebooks, fp32: elements 0..3
    float4* hi = lo + (size_t)M * nb;                  // elements 4..7
    float* Q = (float*)(hi + (size_t)M * nb);          // [M][nb] C^T S_gg C
    float* Sgg = Q + (size_t)M * nb;                   // [8][8]
    unsigned int* cmax = (unsigned int*)(Sgg + 64);    // [M][8] max |C_t[c]_e| (float bits)
    unsigned int* qmax = cmax + 64;                    // max |Q| (infinities and NaN are the largest)
    float* csum = (float*)(qmax + 1);                  // sum of all of cmax; infinity if Q is out of range
    BeamWarp& bw = ((BeamWarp*)(qmax + 4))[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_wait();
    pdl_launch_dependents();
    const int g = blockIdx.y;
    for (int i = threadIdx.x; i < 64; i += blockDim.x) {
        Sgg[i] = S[(size_t)(g * 8 + i / 8) * in + g * 8 + i % 8];
        cmax[i] = 0u;
        if (i == 0) *qmax = 0u;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < M * nb; i += blockDim.x) {
        float cv[8];
        unpack8<BDT>(*(const uint4*)(books + (size_t)i * 8), cv);
        lo[i] = make_float4(cv[0], cv[1], cv[2], cv[3]);
        hi[i] = make_float4(cv[4], cv[5], cv[6], cv[7]);
        float q = 0.0f;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            float sc = 0.0f;
#pragma unroll
            for (int f = 0; f < 8; ++f) sc = fmaf(Sgg[e * 8 + f], cv[f], sc);
            q = fmaf(cv[e], sc, q);
            atomicMax(&cmax[(i >> B) * 8 + e], __float_as_uint(fabsf(cv[e])));
        }
        Q[i] = q;
        atomicMax(qmax, __float_as_uint(fabsf(q)));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float sum = 0.0f;
        for (int i = 0; i < M * 8; ++i) sum += __uint_as_float(cmax[i]);
        *csum = __uint_as_float(*qmax) < 1.0e37f ? sum : INFINITY;
    }
    __syncthreads();

    for (int o = blockIdx.x * kBeamWarps + warp; o < out; o += gridDim.x * kBeamWarps) {
        const float s = bits_to_f32<SDT>(scales[o]);
        float wg[8];
        unpack8<BDT>(*(const uint4*)(w + (size_t)o * in + (size_t)g * 8), wg);
        // h_k = (S e^(k))_g - S_gg e^(k)_g, lane (k, e) for k < M, e < 8 (M <= 4 here per
        // pass of 32 lanes; two passes for more books)
        for (int idx = lane; idx < M * 8; idx += 32) {
            const int k = idx / 8, e = idx % 8;
            const float* ek = E + ((size_t)k * out + o) * in + (size_t)g * 8;
            float v = V[((size_t)k * out + o) * in + (size_t)g * 8 + e];
#pragma unroll
            for (int f = 0; f < 8; ++f) v = fmaf(-Sgg[e * 8 + f], ek[f], v);
            bw.h[k][e] = v;
        }
        // the single empty state
        if (lane < 8) bw.st[0].P[0][lane] = 0.0f;
        if (lane == 0) {
            bw.st[0].score[0] = 0.0f;
            bw.st[0].codes[0] = 0ull;
        }
        __syncwarp();
        // What the estimates lose by underflow, over lambda, and eps / 4 of it as a bound of T (2^-122)
        float wmax = 0.0f;
#pragma unroll
        for (int e = 0; e < 8; ++e) wmax = fmaxf(wmax, fabsf(wg[e]));
        const float s1 = 1.0f + fabsf(s), tmin = 1.8807909e-37f * s1 * s1 * (2.0f + wmax + s1 * *csum);
        int nstates = 1;
        for (int t = 0; t < M; ++t) {
            const BeamWarp::States& cur = bw.st[t & 1];
            BeamWarp::States& nxt = bw.st[(t + 1) & 1];
            const float lt = lam.v[t];
            const float* ht = bw.h[t];
            const float4 *lot = lo + (size_t)t * nb, *hit = hi + (size_t)t * nb;
            const int ncand = nstates * nb, keep = ncand < K ? ncand : K;
            // the score by its definition (the fixed order of operations)
            auto score = [&](int j) {
                const int r = j >> B, c = j & (nb - 1);
                const float4 p0 = *(const float4*)cur.P[r], p1 = *(const float4*)(cur.P[r] + 4);
                const float4 c0 = lot[c], c1 = hit[c];
                float d[8] = {p0.x + c0.x, p0.y + c0.y, p0.z + c0.z, p0.w + c0.w,
                              p1.x + c1.x, p1.y + c1.y, p1.z + c1.z, p1.w + c1.w};
#pragma unroll
                for (int e = 0; e < 8; ++e) d[e] = fmaf(-s, d[e], wg[e]);
                float q = 0.0f, l = 0.0f;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    float sd = 0.0f;
#pragma unroll
                    for (int f = 0; f < 8; ++f) sd = fmaf(Sgg[e * 8 + f], d[f], sd);
                    q = fmaf(d[e], sd, q);
                    l = fmaf(d[e], ht[e], l);
                }
                const float sc = fmaf(lt, fmaf(2.0f, l, q), cur.score[r]);
                return sc <= FLT_MAX ? sc : FLT_MAX;   // NaN and +inf last: keeps the order total
            };
            // the new state of rank i from candidate j with score sc (one lane)
            auto keep_state = [&](int i, int j, float sc) {
                const int r = j >> B, c = j & (nb - 1);
                const float4 p0 = *(const float4*)cur.P[r], p1 = *(const float4*)(cur.P[r] + 4);
                const float4 c0 = lot[c], c1 = hit[c];
                *(float4*)nxt.P[i] = make_float4(p0.x + c0.x, p0.y + c0.y, p0.z + c0.z, p0.w + c0.w);
                *(float4*)(nxt.P[i] + 4) = make_float4(p1.x + c1.x, p1.y + c1.y, p1.z + c1.z, p1.w + c1.w);
                nxt.score[i] = sc;
                nxt.codes[i] = cur.codes[r] | ((unsigned long long)c << (8 * t));
            };
            // magnitude bound T_r, and the expanded form's G_r and A_r: four lanes per state
            float tot = 0.0f;
            bool differ = false;                       // scores of one state's candidates may differ
            // (eight states, or all sixteen places: the estimates read no further)
            for (int r = lane >> 2; r < (nstates > 8 ? kBeamMaxK : 8); r += 8) {
                float ga[2], au = 0.0f, tr = 0.0f;
                const int rr = r < nstates ? r : 0, e0 = (lane & 3) * 2;
                float u[8], D[8];
#pragma unroll
                for (int f = 0; f < 8; ++f) {
                    u[f] = fmaf(-s, cur.P[rr][f], wg[f]);
                    D[f] = fabsf(wg[f]) + fabsf(s) * (fabsf(cur.P[rr][f]) + __uint_as_float(cmax[t * 8 + f]));
                }
                float ue[2], De[2];                    // elements e0, e0 + 1 (lane & 3 picks)
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if ((e >> 1) == (lane & 3)) {
                        ue[e & 1] = u[e];
                        De[e & 1] = D[e];
                    }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    float su = 0.0f, sD = 0.0f;
#pragma unroll
                    for (int f = 0; f < 8; ++f) {
                        const float sv = Sgg[(e0 + i) * 8 + f];
                        su = fmaf(sv, u[f], su);
                        sD = fmaf(fabsf(sv), D[f], sD);
                    }
                    const float hv = ht[e0 + i];
                    ga[i] = -2.0f * lt * s * (su + hv);
                    au = fmaf(ue[i], fmaf(2.0f, hv, su), au);
                    tr = fmaf(De[i], fmaf(2.0f, fabsf(hv), sD), tr);
                }
                au += __shfl_xor_sync(0xffffffffu, au, 1);
                au += __shfl_xor_sync(0xffffffffu, au, 2);
                tr += __shfl_xor_sync(0xffffffffu, tr, 1);
                tr += __shfl_xor_sync(0xffffffffu, tr, 2);
                bw.G[r][e0] = ga[0];
                bw.G[r][e0 + 1] = ga[1];
                // a state that is not there is never in reach
                if ((lane & 3) == 0) bw.A[r] = r < nstates ? fmaf(lt, au, cur.score[rr]) : FLT_MAX;
                const float T = fmaf(lt, tr, fabsf(cur.score[rr]));
                tot = fmaxf(tot, T < 1.0e36f ? T : FLT_MAX);   // (a NaN counts as too large)
                differ = differ || !(lt * tr == 0.0f);
            }
            differ = __any_sync(0xffffffffu, differ);
#pragma unroll
            for (int sh = 16; sh >= 4; sh >>= 1)
                tot = fmaxf(tot, __shfl_xor_sync(0xffffffffu, tot, sh));
            __syncwarp();
            const float F = lt * s * s;
            const bool fine = tot > fmaxf(1.0e-30f, lt * tmin) && F >= FLT_MIN && lt >= FLT_MIN;
            int n = -1;                                // listed candidates (-1: no list)
            if (tot < 1.0e36f && (!differ || nb < 256 || fine)) {
                if (!differ) {
                    // every candidate has its state's score (a prefix weight of zero; an input that H has no
                    // energy for: the terms of T_r bound the score's): the first `keep` indices are the first
                    if (lane < keep) bw.lidx[lane] = lane;
                    n = keep;
                } else if (nb < 256) {                 // at most 256 candidates: all of them
                    for (int j = lane; j < ncand; j += 32) bw.lidx[j] = j;
                    n = ncand;
                } else {
                    const float slack = 3.0517578125e-5f * tot;   // 2 eps
                    const float* Qt = Q + (size_t)t * nb;
                    uint32_t rmask, cmask;
                    if (nstates <= 2)
                        beam_reach<2, 1>(lot, hit, Qt, F, bw.G[0], bw.A, bw.lscore, lane, keep, slack, &rmask, &cmask);
                    else if (nstates <= 4)
                        beam_reach<4, 1>(lot, hit, Qt, F, bw.G[0], bw.A, bw.lscore, lane, keep, slack, &rmask, &cmask);
                    else if (nstates <= 8)
                        beam_reach<8, 1>(lot, hit, Qt, F, bw.G[0], bw.A, bw.lscore, lane, keep, slack, &rmask, &cmask);
                    else
                        beam_reach<8, 2>(lot, hit, Qt, F, bw.G[0], bw.A, bw.lscore, lane, keep, slack, &rmask, &cmask);
                    rmask &= (1u << nstates) - 1u;
                    const int mine = __popc(rmask) * __popc(cmask);
                    int at = mine;                     // inclusive prefix sum over the lanes
#pragma unroll
                    for (int sh = 1; sh < 32; sh <<= 1) {
                        const int v = __shfl_up_sync(0xffffffffu, at, sh);
                        if (lane >= sh) at += v;
                    }
                    n = __shfl_sync(0xffffffffu, at, 31);
                    if (n > kBeamList) n = -1;
                    else {
                        at -= mine;
                        for (uint32_t rm = rmask; rm; rm &= rm - 1)
                            for (uint32_t cm = cmask; cm; cm &= cm - 1)
                                bw.lidx[at++] = ((__ffs(rm) - 1) << B) | (lane + 32 * (__ffs(cm) - 1));
                    }
                }
                __syncwarp();
            }
            if (n >= 0 && n <= 32) {
                // one listed candidate per lane; its rank is the number of candidates before it
                const int j = lane < n ? bw.lidx[lane] : 0x7fffffff;
                const float sc = lane < n ? score(j) : FLT_MAX;
                int rank = 0;
                for (int i = 0; i < n; ++i) {
                    const float os = __shfl_sync(0xffffffffu, sc, i);
                    const int oj = __shfl_sync(0xffffffffu, j, i);
                    rank += before(os, oj, sc, j) ? 1 : 0;
                }
                if (lane < n && rank < keep) keep_state(rank, j, sc);
            } else {
                // The first `keep` of the list's first n places in order, rank by rank: each round a minimum over the
                // candidates after the last one taken.
                auto in_order = [&](int n, auto take) {
                    float ps = -FLT_MAX;
                    int pj = -1;
                    for (int i = 0; i < keep; ++i) {
                        float bs = FLT_MAX;
                        int bj = 0x7fffffff;
                        for (int q = lane; q < n; q += 32) {
                            const int j = bw.lidx[q];
                            const float sc = bw.lscore[q];
                            if ((i == 0 || before(ps, pj, sc, j)) && before(sc, j, bs, bj)) {
                                bs = sc;
                                bj = j;
                            }
                        }
#pragma unroll
                        for (int sh = 16; sh > 0; sh >>= 1) {
                            const float os = __shfl_xor_sync(0xffffffffu, bs, sh);
                            const int oj = __shfl_xor_sync(0xffffffffu, bj, sh);
                            if (before(os, oj, bs, bj)) {
                                bs = os;
                                bj = oj;
                            }
                        }
                        ps = bs;
                        pj = min(bj, ncand - 1);       // every round finds one; only guards the index
                        take(i, pj, ps);
                    }
                };
                if (n >= 0) {
                    for (int i = lane; i < n; i += 32) bw.lscore[i] = score(bw.lidx[i]);
                } else {
                    // No list: every candidate is scored once, in index order, and listed if it comes before the
                    // keep-th best of those that the list has been cut down to. (Where all tie, nothing after
                    // the first list is.)
                    float ks = FLT_MAX;
                    int kj = 0x7fffffff;
                    n = 0;
                    for (int q = 0; q < ncand; q += 32) {
                        const int j = q + lane;
                        const float sc = j < ncand ? score(j) : FLT_MAX;
                        const bool add = j < ncand && before(sc, j, ks, kj);
                        const uint32_t adds = __ballot_sync(0xffffffffu, add);
                        if (add) {
                            const int at = n + __popc(adds & ((1u << lane) - 1u));
                            bw.lidx[at] = j;
                            bw.lscore[at] = sc;
                        }
                        n += __popc(adds);
                        if (n > kBeamList - 32) {      // no room for 32 more
                            __syncwarp();
                            float ws = 0.0f;           // the candidate of rank `lane`
                            int wj = 0;
                            in_order(n, [&](int i, int j2, float s2) {
                                if (i == lane) {
                                    ws = s2;
                                    wj = j2;
                                }
                                ks = s2;
                                kj = j2;
                            });
                            __syncwarp();
                            if (lane < keep) {
                                bw.lidx[lane] = wj;
                                bw.lscore[lane] = ws;
                            }
                            n = keep;
                        }
                    }
                }
                __syncwarp();
                in_order(n, [&](int i, int j, float sc) {
                    if (lane == 0) keep_state(i, j, sc);
                });
            }
            __syncwarp();
            nstates = keep;
        }
        const unsigned long long best = bw.st[M & 1].codes[0];
        if (lane < M) ((uint8_t*)codes_out)[((size_t)o * ng + g) * M + lane] = (uint8_t)(best >> (8 * lane));
        __syncwarp();
    }
}

inline size_t beam_smem(int M, int B) {
    return ((size_t)M << B) * 9 * 4 + (64 + 64 + 4) * 4 + kBeamWarps * sizeof(BeamWarp);
}

template <int BDT, int SDT>
aq_status run_beam(const Dims& d, const void* w, const void* codes, const void* books,
                   const void* scales, const void* h, int h_dt, const Lambdas& lam, int K,
                   void* codes_out, void* ws, cudaStream_t st) {
    DeviceInfo di;
    if (aq_status e = device_info(&di); e != AQ_OK) return e;
    float* S = (float*)((char*)ws + beam_s_off());
    float* E = (float*)((char*)ws + beam_e_off(d));
    float* V = (float*)((char*)ws + beam_v_off(d));
    const int grid = di.sms * 8;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.stream = st;
    cfg.blockDim = dim3(256);
    cfg.gridDim = dim3(grid);
    if (aq_status e = cuda_ok(cudaLaunchKernelEx(&cfg, beam_resid_kernel<BDT, SDT>, (const uint16_t*)w, codes,
                                                 (const uint16_t*)books, (const uint16_t*)scales, E, d.out,
                                                 d.in, d.ng, d.M, d.B),
                              "cudaLaunchKernelEx (beam residuals)");
        e != AQ_OK)
        return e;
    if (aq_status e = cuda_ok(cudaLaunchKernelEx(&cfg, beam_sym_kernel, h, h_dt, S, d.in),
                              "cudaLaunchKernelEx (beam symmetric part)");
        e != AQ_OK)
        return e;
    const long long rows = (long long)d.M * d.out;
    const bool big = ((rows + 127) / 128) * ((d.in + 127) / 128) >= di.sms;
    const int T = big ? 128 : 64;
    const int row_tiles = (int)((rows + T - 1) / T);
    cfg.gridDim = dim3((d.in + T - 1) / T, row_tiles < 65535 ? row_tiles : 65535);
    cfg.blockDim = dim3(big ? kBeamGemmThreads<128> : kBeamGemmThreads<64>);
    if (aq_status e = cuda_ok(cudaLaunchKernelEx(&cfg, big ? beam_gemm_kernel<128> : beam_gemm_kernel<64>,
                                                 (const float*)E, (const float*)S, V, (int)rows, d.in),
                              "cudaLaunchKernelEx (beam cross terms)");
        e != AQ_OK)
        return e;
    auto kern = beam_kernel<BDT, SDT>;
    const size_t smem = beam_smem(d.M, d.B);
    if (smem > (size_t)di.smem_optin) return AQ_ERR_UNSUPPORTED;
    if (cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        e != cudaSuccess)
        return cuda_fail(e, "cudaFuncSetAttribute");
    // Row blocks per group: enough CTAs for two waves of two per SM, and 16 rows per warp before
    // that (the staging of the books and their quadratic terms costs about one row's search).
    int xb = (d.out + 16 * kBeamWarps - 1) / (16 * kBeamWarps);
    const int want = (di.sms * 4 + d.ng - 1) / d.ng, most = (d.out + kBeamWarps - 1) / kBeamWarps;
    if (xb < want) xb = want < most ? want : most;
    cfg.gridDim = dim3(xb, d.ng);
    cfg.blockDim = dim3(kBeamWarps * 32);
    cfg.dynamicSmemBytes = smem;
    return cuda_ok(cudaLaunchKernelEx(&cfg, kern, (const uint16_t*)w, (const uint16_t*)books,
                                      (const uint16_t*)scales, (const float*)S, (const float*)E,
                                      (const float*)V, codes_out, lam, d.out, d.in, d.ng, d.M,
                                      d.B, K),
                   "cudaLaunchKernelEx (beam search)");
}

}  // namespace

size_t beam_ws_bytes(const Dims& d) { return beam_v_off(d) + (size_t)d.M * d.out * d.in * 4; }

aq_status launch_beam(const Dims& d, const void* w, const void* codes, const void* books,
                      const void* scales, const void* h, int h_dt, const double* lambda, int K,
                      void* codes_out, void* ws, cudaStream_t st) {
    if (d.out == 0) return AQ_OK;
    Lambdas lam = {};
    for (int k = 0; k < d.M; ++k) lam.v[k] = lambda ? (float)lambda[k] : 1.0f;
    const int key = (d.book_dt == AQ_BF16) * 2 + (d.scale_dt == AQ_BF16);
    switch (key) {
        case 0: return run_beam<AQ_F16, AQ_F16>(d, w, codes, books, scales, h, h_dt, lam, K, codes_out, ws, st);
        case 1: return run_beam<AQ_F16, AQ_BF16>(d, w, codes, books, scales, h, h_dt, lam, K, codes_out, ws, st);
        case 2: return run_beam<AQ_BF16, AQ_F16>(d, w, codes, books, scales, h, h_dt, lam, K, codes_out, ws, st);
        default: return run_beam<AQ_BF16, AQ_BF16>(d, w, codes, books, scales, h, h_dt, lam, K, codes_out, ws, st);
    }
}

}  // namespace aq
