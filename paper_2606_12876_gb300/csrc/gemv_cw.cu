// gemv_cw: y = x * W_m^T for 1..16 tokens with 4- and 8-bit codes (the prefix-m reconstruction
// of Sec. 3.2 / Sec. 5; Y = W X of Sec. 2.2), one kernel per call. gemv.cu and gemm.cu say which
// calls come here.
//
// By linearity in the books (Sec. 5), x_g . (sum_k C_k[b_k]) = sum_k x_g . C_k[b_k], and a
// 16-byte codeword is, as it stands, the eight weights of one row and group: it goes straight
// into the A fragment of a 16-bit tensor-core multiply (mma.sync m16n8k16, fp32 accumulation),
// with no sum, no conversion and no rounding of weights on the way. In lane 4g + c (g < 8,
// c < 4) the fragment holds row g (and g + 8), and the four K positions that the lane owns in
// each of two multiplies are bound to the two halves of the codeword of one group; the K order
// of a multiply is free, so in step j (0..7) of a 256-input slice lane c takes group 4j + c, and the B
// fragment of the step is the same group of the lane's token g: one 16-byte load, 64 contiguous
// bytes over the lanes c. (With groups 8c + j a load touched 32 lines instead of 8; every SM reads all
// activations, and at about half an uncoalesced request a clock and SM that took 3.4-5 us a call.)
//
// Bound: shared-memory wavefronts of the codeword gathers (16 bytes per code; one 16-byte load of
// a warp is four wavefronts when no two of the eight lanes of a phase meet in a bank group). Each
// codebook is staged in 2^cshift interleaved copies, lane L reading copy L mod 2^cshift: with
// eight copies there are no conflicts whatever the codes (a single copy costs about 2.6 times the
// wavefronts). At 8 codes per clock and SM the gate projection (14336 x 4096, m = 4) cannot take
// less than 12.6 us for eight tokens; the issue slots (34 %) and the tensor pipe (25 %) have slack.
//
// A CTA holds eight tokens (the N of the multiply); 9..16 tokens are two token tiles along the grid's y,
// which gather every codeword twice. (One tile of 16 tokens spilled registers and kept fewer loads in
// flight: 1024 x 4096, m = 2, 16 tokens 9.0 us, two tiles 5.3.) Larger layers run gemm_ts.cu instead, which
// decodes once for all tokens (ts_clocks against cw_clocks, in gemv.cu).
//
// Work split: a warp's work item is a (32-row block, slice, book); a cluster of kc CTAs (16 warps
// each) owns whole row blocks, its warps share the row block's (slice, book) units evenly in
// slice-major order (so a warp's B fragments, 32 registers, are loaded once per slice), and
// the warps' accumulators are added in a fixed order in shared memory (and over the cluster
// through distributed shared memory). So the kernel writes y itself: no partial planes in the
// workspace and no reduction launch. kc > 1 is for layers with too few row blocks for the SMs.
//
// Operand types: books and activations both fp16, or both bf16, are multiplied as they are. fp16
// books with bf16 activations: every (token, slice) of x is scaled by a power of two that puts
// its largest |x| in [2^14, 2^15) and rounded to fp16, which is exact for values within 2^29 of
// the largest, and the slice's sums are scaled back when they are added to the total. bf16 books
// with fp16 activations: the books are scaled the same way (one power of two for the m books, by their
// largest finite entry).
//
// Measured, 8B block (seven layers; q/k/v and gate/up as groups): 8 tokens, m = 3 83.2 us (the eight-token
// tables and tf32 kernel before: 145.8), 4-bit codes, 4 tokens, m = 4 92.0 us (fp32 kernel before: 229.7).
// 14336 x 4096, 8 tokens: m = 3 17.8 us, m = 4 22.1 us; 4 tokens (fp32 sums): 18.8, 23.5; 1024 x 1024, m = 4, 16
// tokens: 3.8 us.
#include "aq_internal.cuh"
#include "cw_split.h"
#include "launch.cuh"
#include "operand_scale.cuh"
#include "tc_ptx.cuh"

namespace aq {
namespace {

constexpr int kCwWarps = 16;
constexpr int kCwThreads = kCwWarps * 32;
constexpr int kCwPitch = 36;       // floats per token in a warp's sums (4 of padding: no conflicts)
constexpr int kCwTokens = 8;       // tokens of a CTA (more: token tiles along the grid's y)

// One layer of a launch; a launch holds one layer, or several that share the activations and the split
// (aq_gemv_group): cluster c of the layer takes row blocks c, c + nclusters, ...
struct CwLayer {
    const uint8_t* planes;
    const uint16_t *books, *scales;
    void* y;
    int out, rows_pad, RBc;
    int c0, nclusters;             // the layer's clusters of the grid
    size_t plane_bytes;
};
struct CwArgs {
    CwLayer L[4];
    int nlayers;
    const uint16_t* x;
    const void* y_prev;            // added to the product (refinement), or null
    int y_dt, scale_dt, m, batch, in, ng, S;
    int cshift;                    // log2 of the interleaved copies of a codebook
    int kc;                        // CTAs per cluster
    int static_weights;
};

// Shared memory: books [m][2^B][2^cshift] x 16 B, codes 16 warps x 32 rows, the warps' sums (two
// buffers of [16][8][36] floats), the CTA's sums (two buffers of [8][32]; clusters only).
constexpr size_t kCwRedFloats = (size_t)kCwWarps * kCwTokens * kCwPitch;
inline size_t cw_smem_bytes(int B, int m, int cshift) {
    return ((size_t)m * 16 << B << cshift) + (size_t)kCwWarps * 32 * unit_bytes(B) +
           (2 * kCwRedFloats + 2 * 32 * kCwTokens) * 4;
}

template <int DT>
__device__ __forceinline__ void mma16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                      uint32_t b0, uint32_t b1) {
    if constexpr (DT == AQ_F16)
        asm(
            "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
            "{%8, %9}, {%0, %1, %2, %3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
    else
        asm(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
            "{%8, %9}, {%0, %1, %2, %3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Eight 16-bit values of type DT times sc (a power of two), as fp16.
template <int DT>
__device__ __forceinline__ uint4 scaled_to_f16(const uint4& v, float sc) {
    float f[8];
    unpack8<DT>(v, f);
    return make_uint4(round_pack2<AQ_F16>(f[0] * sc, f[1] * sc), round_pack2<AQ_F16>(f[2] * sc, f[3] * sc),
                      round_pack2<AQ_F16>(f[4] * sc, f[5] * sc), round_pack2<AQ_F16>(f[6] * sc, f[7] * sc));
}

template <int DT>
__device__ __forceinline__ float max_abs8(const uint4& v) {
    float f[8], mx = 0.0f;
    unpack8<DT>(v, f);
#pragma unroll
    for (int e = 0; e < 8; ++e) mx = fmaxf(mx, fabsf(f[e]));
    return mx;
}

// The exponent e that puts mx * 2^-e in [2^14, 2^15); 0 for 0. At most 114 (infinity); at least -126,
// so that 2^-e is a float: bf16 values are multiples of 2^-133, which 2^126 makes normal fp16 values.
__device__ __forceinline__ int f16_exponent(float mx) { return mx > 0.0f ? max(-126, exponent_of(mx) - 14) : 0; }

// The codes of a row's slice unit as stored (position p holds group (p + o) mod 32), staged in group
// order (B = 8: the groups 4j + c of each c together).
template <int B>
__device__ __forceinline__ void store_unrotated(unsigned char* buf, int row, const uint4 (&raw)[2]) {
    if constexpr (B == 8) {
        const uint32_t w[8] = {raw[0].x, raw[0].y, raw[0].z, raw[0].w, raw[1].x, raw[1].y, raw[1].z, raw[1].w};
        uint32_t u[8];
        unrotate_codes(w, row, u);
        // byte c of the eight words (groups 4j + c) together at byte 8c: two 4 x 4 byte transposes
        uint32_t o[4][2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t t0 = prmt(u[4 * h], u[4 * h + 1], 0x5140u), t1 = prmt(u[4 * h + 2], u[4 * h + 3], 0x5140u);
            const uint32_t t2 = prmt(u[4 * h], u[4 * h + 1], 0x7362u), t3 = prmt(u[4 * h + 2], u[4 * h + 3], 0x7362u);
            o[0][h] = prmt(t0, t1, 0x5410u);
            o[1][h] = prmt(t0, t1, 0x7632u);
            o[2][h] = prmt(t2, t3, 0x5410u);
            o[3][h] = prmt(t2, t3, 0x7632u);
        }
        // the row's 16-byte halves change places in rows 4..7 of every eight: no bank conflicts
        const int sw = (row >> 2) & 1;
        *(uint4*)(buf + row * 32 + sw * 16) = make_uint4(o[0][0], o[0][1], o[1][0], o[1][1]);
        *(uint4*)(buf + row * 32 + (sw ^ 1) * 16) = make_uint4(o[2][0], o[2][1], o[3][0], o[3][1]);
    } else {
        const uint32_t w[4] = {raw[0].x, raw[0].y, raw[0].z, raw[0].w};
        uint32_t u[4];
        unrotate_nibbles(w, row, u);
        *(uint4*)(buf + row * 16) = make_uint4(u[0], u[1], u[2], u[3]);
    }
}

// The codes of groups 4j + c (j = 0..7) of a staged row: eight bytes (B = 8), or the low nibbles of the
// halves of four words (B = 4).
template <int B>
struct RowCodes {
    uint32_t w[B == 8 ? 2 : 4];
    __device__ __forceinline__ void load(const unsigned char* buf, int row, int c) {
        if constexpr (B == 8) {
            const uint2 v = *(const uint2*)(buf + row * 32 + (((c >> 1) ^ ((row >> 2) & 1)) * 16) + (c & 1) * 8);
            w[0] = v.x;
            w[1] = v.y;
        } else {
            const uint4 v = *(const uint4*)(buf + row * 16);
            w[0] = v.x >> (4 * c);
            w[1] = v.y >> (4 * c);
            w[2] = v.z >> (4 * c);
            w[3] = v.w >> (4 * c);
        }
    }
    __device__ __forceinline__ uint32_t code(int j) const {
        if constexpr (B == 8) return prmt(w[j >> 2], 0u, 0x4440u | (uint32_t)(j & 3));
        else return (w[j >> 1] >> (16 * (j & 1))) & 15u;
    }
};

// CHAIN: multiplies (of 16 inputs) that the tensor pipe accumulates before an fp32 addition takes them over. The
// pipe truncates as it accumulates, so the longer the chain, the larger the error of an fp32 y:
//   1: the two multiplies of a step are added, then the steps of a unit, the units of a warp, and the warps in
//      pairs: as accurate as the table kernel's fp32 sums (0.7 to 1.05 times its error);
//   4: two steps: 0.5 to 0.95 times the error of fp32 sums in input order;
//   0: all units of a warp (4096 x 14336, m = 1 / 4: 1.1e-6 / 4.3e-6).
template <int B, int BDT, int XDT, int CHAIN>
__global__ void __launch_bounds__(kCwThreads, 1) gemv_cw_kernel(const __grid_constant__ CwArgs a) {
    constexpr int UNIT = unit_bytes(B), NC = 1 << B;
    constexpr int MDT = BDT == AQ_BF16 && XDT == AQ_BF16 ? AQ_BF16 : AQ_F16;   // operand type
    constexpr bool kScaleX = XDT != MDT, kScaleB = BDT != MDT;
    constexpr int kTake = CHAIN == 4 ? 2 : 8;           // steps between the additions to the accumulators
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ unsigned int s_bmax;
    uint4* books_s = (uint4*)smem;
    const int nslot = (a.m * NC) << a.cshift;
    unsigned char* codes_s = smem + (size_t)nslot * 16;
    float* red = (float*)(codes_s + kCwWarps * 32 * UNIT);
    float* csum = red + 2 * kCwRedFloats;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = a.kc > 1 ? (int)cluster_rank() : 0;
    int cid = (int)blockIdx.x / a.kc, layer = 0;
    while (layer + 1 < a.nlayers && cid >= a.L[layer + 1].c0) ++layer;
    const CwLayer& L = a.L[layer];
    cid -= L.c0;
    const int tb = (int)blockIdx.y * kCwTokens;               // first token

    // this warp's (slice, book) units u0 .. u1-1 of every row block of the cluster; u = s*m + k
    const long long U = (long long)a.S * a.m;
    const int nwarps = kCwWarps * a.kc, gw = rank * kCwWarps + warp;
    const int u0 = (int)(U * gw / nwarps), u1 = (int)(U * (gw + 1) / nwarps);
    const int sk0 = (u0 / a.m) << 3 | (u0 % a.m);             // slice and book of u0 (m <= 8)
    struct Item {
        int rb, u, s, k;
    };
    auto next_item = [&](Item& it) {
        if (++it.u == u1) {
            // (a division per pass costs 1 % of a call; where the sums take registers, one for it costs as much)
            if constexpr (CHAIN == 0) it = Item{it.rb + L.nclusters, u0, sk0 >> 3, sk0 & 7};
            else it = Item{it.rb + L.nclusters, u0, u0 / a.m, u0 % a.m};
        } else if (++it.k == a.m) {
            it.k = 0;
            ++it.s;
        }
    };
    uint4 raw[2];
    auto load_codes = [&](const Item& it) {
        if (u0 < u1 && it.rb < L.RBc) {
            const uint8_t* src = L.planes + (size_t)it.k * L.plane_bytes +
                                 ((size_t)it.s * L.rows_pad + (size_t)it.rb * 32 + lane) * UNIT;
            raw[0] = ld_stream_v4(src);
            if constexpr (B == 8) raw[1] = ld_stream_v4(src + 16);
        }
    };
    Item nxt{cid, u0, sk0 >> 3, sk0 & 7};
    float bfac = 1.0f;                                   // 2^f of the staged books (kScaleB)
    auto stage_books = [&]() {
        if constexpr (kScaleB) {
            if (tid == 0) s_bmax = 0u;
            __syncthreads();
            float mx = 0.0f;
            for (int i = tid; i < a.m * NC; i += kCwThreads)
                mx = fmaxf(mx, __uint_as_float(codeword_max_bits<BDT>(__ldg((const uint4*)L.books + i))));
            atomicMax(&s_bmax, __float_as_uint(mx));     // non-negative floats order as integers
            __syncthreads();
            const int f = f16_exponent(__uint_as_float(s_bmax));
            bfac = pow2f(f);
            const float sc = pow2f(-f);
            for (int i = tid; i < nslot; i += kCwThreads)
                books_s[i] = scaled_to_f16<BDT>(__ldg((const uint4*)L.books + (i >> a.cshift)), sc);
        } else if constexpr (B == 4) {                  // few codewords: a thread per copy
            for (int i = tid; i < nslot; i += kCwThreads) books_s[i] = __ldg((const uint4*)L.books + (i >> a.cshift));
        } else {
            // each codeword loaded once (two in flight), its copies written from copy `lane` on, so that eight
            // lanes meet no bank group twice
            auto put = [&](int i, const uint4& c) {
                if (a.cshift == 3) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) books_s[i * 8 + ((q + lane) & 7)] = c;
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) books_s[i * 4 + ((q + lane) & 3)] = c;
                }
            };
            const int n = a.m * NC;
            for (int i = tid; i < n; i += 2 * kCwThreads) {
                const int j = i + kCwThreads;
                const uint4 c0 = __ldg((const uint4*)L.books + i);
                const uint4 c1 = j < n ? __ldg((const uint4*)L.books + j) : c0;
                put(i, c0);
                if (j < n) put(j, c1);
            }
        }
    };
    if (a.static_weights) {   // read-only weights: requested before the preceding kernel has finished
        load_codes(nxt);
        stage_books();
    }
    pdl_wait();
    pdl_launch_dependents();
    if (!a.static_weights) {
        load_codes(nxt);
        stage_books();
    }
    __syncthreads();

    const int g = lane >> 2, c = lane & 3;
    unsigned char* buf = codes_s + warp * 32 * UNIT;
    const uint32_t mul = 16u << a.cshift;
    const uint32_t books_u = smem_u32(books_s) + ((uint32_t)(lane & ((1 << a.cshift) - 1)) << 4);
    uint4 bf[8];                                         // B fragments of slice cur_s
    float fac[2] = {1.0f, 1.0f};                         // (kScaleX) 2^e of tokens 2c, 2c+1
    int cur_s = -1;
    auto load_b = [&](int s) {
        const int t = tb + g;
        const uint4* src = (const uint4*)(a.x + (size_t)t * a.in) + s * 32 + c;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            bf[j] = t < a.batch && s * 32 + 4 * j + c < a.ng ? __ldg(src + 4 * j) : make_uint4(0u, 0u, 0u, 0u);
        if constexpr (kScaleX) {
            float mx = 0.0f;
#pragma unroll
            for (int j = 0; j < 8; ++j) mx = fmaxf(mx, max_abs8<XDT>(bf[j]));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const int e = f16_exponent(mx);
            const float sc = pow2f(-e), up = pow2f(e);
#pragma unroll
            for (int j = 0; j < 8; ++j) bf[j] = scaled_to_f16<XDT>(bf[j], sc);
            fac[0] = __shfl_sync(0xffffffffu, up, 8 * c);
            fac[1] = __shfl_sync(0xffffffffu, up, 8 * c + 4);
        }
        cur_s = s;
    };

    int pass = 0;
    for (int rb = cid; rb < L.RBc; rb += L.nclusters, ++pass) {
        float acc[2][4];
        // The warps' sums of a pass, added in warp order or (CHAIN) in pairs. Two buffers: a pass's writes meet the sums
        // that are read two passes earlier, which every thread finished before the last barrier.
        float* rp = red + (pass & 1) * kCwRedFloats;
        float* mine = rp + (size_t)warp * kCwTokens * kCwPitch;
        bool first = true;
        // the row scale of the output this thread finishes, requested before the pass's gathers
        auto my_o = [&]() { return rb * 32 + (tid & 31); };
        const uint16_t my_s = tid < 32 * kCwTokens && my_o() < L.out ? L.scales[my_o()] : (uint16_t)0;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[mt][e] = 0.0f;
        // The accumulators into the warp's sums in shared memory; with kScaleX once per slice, times
        // the slice's 2^e (added to the earlier slices'), else once at the end of the pass.
        auto fold = [&]() {
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float* p = mine + (2 * c + (e & 1)) * kCwPitch + 16 * mt + 8 * (e >> 1) + g;
                    if constexpr (kScaleX) {
                        const float v = acc[mt][e] * fac[e & 1];
                        *p = first ? v : *p + v;
                        acc[mt][e] = 0.0f;
                    } else {
                        *p = acc[mt][e];
                    }
                }
            first = false;
        };
        for (int u = u0; u < u1; ++u) {
            const int s = nxt.s, k = nxt.k;
            store_unrotated<B>(buf, lane, raw);
            __syncwarp();
            next_item(nxt);
            load_codes(nxt);                             // travels while this item is multiplied
            if (s != cur_s) {
                if (kScaleX && u > u0) fold();
                load_b(s);
            }
            RowCodes<B> cw[4];
#pragma unroll
            for (int rr = 0; rr < 4; ++rr) cw[rr].load(buf, g + 8 * rr, c);
            __syncwarp();                                // the buffer may be refilled
            const uint32_t base = books_u + (uint32_t)k * (NC * mul);
            float part[2][4] = {};                       // the unit's sums (CHAIN 1), the current chain (4)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                uint4 w[4];
#pragma unroll
                for (int rr = 0; rr < 4; ++rr) w[rr] = lds128(base + cw[rr].code(j) * mul);
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    const uint4 &p = w[2 * mt], &q = w[2 * mt + 1];
                    if constexpr (CHAIN == 1) {
                        float d[4] = {}, e[4] = {};
                        mma16<MDT>(d, p.x, q.x, p.y, q.y, bf[j].x, bf[j].y);
                        mma16<MDT>(e, p.z, q.z, p.w, q.w, bf[j].z, bf[j].w);
#pragma unroll
                        for (int i = 0; i < 4; ++i) part[mt][i] += d[i] + e[i];
                    } else {
                        float(&d)[4] = CHAIN ? part[mt] : acc[mt];
                        mma16<MDT>(d, p.x, q.x, p.y, q.y, bf[j].x, bf[j].y);
                        mma16<MDT>(d, p.z, q.z, p.w, q.w, bf[j].z, bf[j].w);
                    }
                    if (CHAIN && j % kTake == kTake - 1)
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            acc[mt][i] += part[mt][i];
                            part[mt][i] = 0.0f;
                        }
                }
            }
        }
        fold();
        __syncthreads();
        const int i0 = a.kc > 1 ? rank * (32 * kCwTokens / a.kc) : 0;      // outputs this CTA finishes
        const int i1 = a.kc > 1 ? i0 + 32 * kCwTokens / a.kc : 32 * kCwTokens;
        float* cs = csum + (pass & 1) * 32 * kCwTokens;
        float v = 0.0f;
        if (tid < 32 * kCwTokens) {
            const float* p = rp + (tid >> 5) * kCwPitch + (tid & 31);
            if constexpr (CHAIN == 0) {
#pragma unroll
                for (int w = 0; w < kCwWarps; ++w) v += p[w * kCwTokens * kCwPitch];
            } else {
                float t[kCwWarps];
#pragma unroll
                for (int w = 0; w < kCwWarps; ++w) t[w] = p[w * kCwTokens * kCwPitch];
#pragma unroll
                for (int n = kCwWarps / 2; n > 0; n /= 2)
#pragma unroll
                    for (int w = 0; w < n; ++w) t[w] = t[2 * w] + t[2 * w + 1];
                v = t[0];
            }
            if (a.kc > 1) cs[tid] = v;
        }
        if (a.kc > 1) {
            cluster_sync();
            v = 0.0f;
            if (tid >= i0 && tid < i1)
                for (int r = 0; r < a.kc; ++r) {          // the CTAs' sums, in rank order
                    float p;
                    asm volatile("ld.shared::cluster.f32 %0, [%1];"
                                 : "=f"(p) : "r"(map_to_rank(smem_u32(cs + tid), (uint32_t)r)) : "memory");
                    v += p;
                }
        }
        const int t = tb + (tid >> 5), o = my_o();
        if (tid >= i0 && tid < i1 && t < a.batch && o < L.out) {
            float r = v * bfac * bits_to_f32_rt(my_s, a.scale_dt);
            const size_t yi = (size_t)t * L.out + o;
            if (a.y_prev)
                r = (a.y_dt == AQ_F32 ? ((const float*)a.y_prev)[yi]
                                      : bits_to_f32_rt(((const uint16_t*)a.y_prev)[yi], a.y_dt)) + r;
            if (a.y_dt == AQ_F32) ((float*)L.y)[yi] = r;
            else ((uint16_t*)L.y)[yi] = a.y_dt == AQ_F16 ? f32_to_bits<AQ_F16>(r) : f32_to_bits<AQ_BF16>(r);
        }
    }
    if (a.kc > 1) cluster_sync();   // no CTA leaves while a peer may still read its sums
}

// Copies of a codebook (log2): eight while they fit next to the sums, else four.
inline int cw_cshift(int B, int m) { return B == 4 || m <= 5 ? 3 : 2; }

// CTAs per cluster: the split with the smallest estimated time of the busiest cluster, in clocks: passes over its
// row blocks times
//  * the gathers of a CTA's units: 185 clocks each with 8-bit codes (128 wavefronts, staging, sums), 160 with 4-bit
//    codes, 300 with four copies of a book, at least 2500 for each unit of a warp; where no warp has a second unit
//    1700 and about half of the gathers;
//  * 1500 to 2200 clocks of reduction and start-up (1000 less where one pass and one unit are all);
//  * the activations of a warp's further slices (64 bytes a clock and SM), and 800 clocks a slice if they are scaled;
// plus what a cluster launch and its barriers cost over a plain one: 600, 1000 and 1900 clocks for 2, 4 and 8 CTAs,
// 3000 and 2600 for 2 and 4 where the call's CTAs exceed half of the SMs (its clusters then wait for those of
// the preceding kernel). Within 6 % of most calls measured with the cluster size given; clusters of 1 / 2 / 4 / 8,
// 8-bit codes, 3 tokens, fp16 x: 256 x 8192, m = 1 5.5 / 4.6 / 4.4 / 4.7 us, m = 4 15.1 / 9.5 / 6.4 / 5.3; 1024 x 4096,
// m = 1 3.6 / 4.4 / 5.2 / 11.3, m = 4 8.6 / 6.4 / 6.1 / 14.9; 32 x 32768, m = 1 16.7 / 10.2 / 6.5 / 4.5; 256 x 1024, m = 5
// 5.0 / 4.3 / 3.6 / 4.4.
// Clusters are taken for a gain of 1400 clocks or more only: layers of a group share a launch where their sizes
// agree, and one more launch costs about 3 us (block of hidden 2800, m = 2, 4-bit codes, 5 tokens: 29.0 us with
// the key and value projections in clusters of two, 25.4 without; but 256 x 1024, m = 5 by itself takes 4.9 us
// where clusters of four take 3.6).
// Clusters of 2, 4 and 8 that are resident at once: 76, 36 and (beside the preceding call's) 8 on 152 SMs;
// sixteen clusters of eight took twice the time of eight (512 x 8192, m = 1: 8.8 us). With several token tiles
// each tile has its share of the SMs.
inline int cw_tiles(int batch) { return (batch + kCwTokens - 1) / kCwTokens; }
inline int cw_clusters(int kc, int tiles, int sms) {
    const int n = (kc == 1 ? sms : kc == 2 ? sms / 2 : kc == 4 ? sms * 9 / 38 : sms / 19) / tiles;
    return n < 1 ? 1 : n;
}
inline int cw_cluster(const Dims& d, int m, int batch, int x_dt, int sms, int* nclusters, double* clocks) {
    const int tiles = cw_tiles(batch);
    const bool scaled = d.book_dt == AQ_F16 && x_dt == AQ_BF16;
    int best = 1;
    double best_t = -1.0;
    for (int kc = 1; kc <= 8; kc *= 2) {
        int nc = cw_clusters(kc, tiles, sms);
        if (nc > d.RBc) nc = d.RBc;
        const long long U = (long long)d.S * m;
        const long long units = (U + 16 * kc - 1) / (16 * kc);
        const double gather = cw_cshift(d.B, m) != 3 ? 300.0 : d.B == 8 ? 185.0 : 160.0;
        const double all = (double)((U + kc - 1) / kc) * gather, least = units * 2500.0;
        const double work = units == 1 ? 1700.0 + 0.55 * all : all > least ? all : least;
        const bool wide = 2 * nc * kc * tiles > sms;
        const double cluster = kc == 1 ? (units == 1 ? -1000.0 : 0.0) : kc == 2 ? (wide ? 3000.0 : 600.0)
                               : kc == 4 ? (wide ? 2600.0 : 1000.0) : 1900.0;
        const double slices = units > m ? (double)units / m : 1.0;    // of a warp
        const double x_clk = d.in * 2.0 * (batch < kCwTokens ? batch : kCwTokens) / kc / 64.0 * (1.0 - 1.0 / slices) +
                             (scaled ? 800.0 * slices : 0.0);
        const double t = (double)((d.RBc + nc - 1) / nc) * (work + x_clk + (kc > 1 ? 2200.0 : 1500.0)) + cluster;
        if (best_t < 0.0 || t + (best == 1 ? 1400.0 : 0.0) < best_t) {
            best_t = t;
            best = kc;
            *nclusters = nc;
        }
    }
    *clocks = best_t;
    return best;
}

template <int B, int BDT, int XDT, int CHAIN>
aq_status run_cw(CwArgs a, cudaStream_t st) {
    auto kern = gemv_cw_kernel<B, BDT, XDT, CHAIN>;
    a.cshift = cw_cshift(B, a.m);
    const size_t smem = cw_smem_bytes(B, a.m, a.cshift);
    int occ = 0;
    if (aq_status e = prepare(kern, smem, kCwThreads, a.m, &occ); e != AQ_OK) return e;
    const CwLayer& last = a.L[a.nlayers - 1];
    return launch_pdl_cluster(a.kc, kern, dim3((last.c0 + last.nclusters) * a.kc, cw_tiles(a.batch)), dim3(kCwThreads), smem, st, a);
}

// The chain by what the other forms of the product give. 8-bit codes have fp32 tables up to four tokens. From five,
// sums of several books are rounded to 11 bits in the other forms (2e-4), where any chain will do; one book's
// codewords are exact there, in sums with errors of 3.0e-7 to 6.4e-7: the pipe's chain over one unit stays below that
// (2.4e-7 to 3.5e-7), but not over two. 4-bit codes: fp32 sums over the inputs in order (2 to 3e-7).
template <int B, int BDT, int XDT>
aq_status run_cw_chain(const CwArgs& a, cudaStream_t st) {
    if constexpr (B == 4) return run_cw<B, BDT, XDT, 4>(a, st);
    else if (a.batch <= 4 || (a.m == 1 && a.S > kCwWarps * a.kc)) return run_cw<B, BDT, XDT, 1>(a, st);
    else return run_cw<B, BDT, XDT, 0>(a, st);
}

template <int B>
aq_status run_cw_types(const CwArgs& a, int book_dt, int x_dt, cudaStream_t st) {
    if (book_dt == AQ_BF16)
        return x_dt == AQ_BF16 ? run_cw_chain<B, AQ_BF16, AQ_BF16>(a, st) : run_cw_chain<B, AQ_BF16, AQ_F16>(a, st);
    return x_dt == AQ_BF16 ? run_cw_chain<B, AQ_F16, AQ_BF16>(a, st) : run_cw_chain<B, AQ_F16, AQ_F16>(a, st);
}

}  // namespace

double cw_clocks(const Dims& d, int m, int batch, int x_dt) {
    DeviceInfo di;
    int nc;
    double t = -1.0;
    if (device_info(&di) == AQ_OK) cw_cluster(d, m, batch, x_dt, di.sms, &nc, &t);
    return t;
}

aq_status launch_cw(const Dims* ds, int n, int m, const void* const* planes, const void* const* books,
                    const void* const* scales, const void* x, int x_dt, int batch, void* const* y, int y_dt,
                    const void* y_prev, cudaStream_t st) {
    DeviceInfo di;
    if (aq_status e = device_info(&di); e != AQ_OK) return e;
    const Dims& d = ds[0];
    int kcs[4], own[4];
    const int tiles = cw_tiles(batch);
    double clocks;
    for (int l = 0; l < n; ++l) kcs[l] = cw_cluster(ds[l], m, batch, x_dt, di.sms, &own[l], &clocks);
    bool done[4] = {};
    for (int f = 0; f < n; ++f) {
        if (done[f]) continue;
        // the layers with this one's cluster size: their sums are those of their own calls
        CwArgs a = {};
        a.kc = kcs[f];
        int rbs[4], set[4];
        for (int l = f; l < n; ++l)
            if (!done[l] && kcs[l] == a.kc) {
                done[l] = true;
                rbs[a.nlayers] = ds[l].RBc;
                set[a.nlayers++] = l;
            }
        const int passes = cw_group_passes(rbs, a.nlayers, cw_clusters(a.kc, tiles, di.sms));
        a.static_weights = 1;
        for (int i = 0, c0 = 0; i < a.nlayers; ++i) {
            const int l = set[i];
            CwLayer& L = a.L[i];
            L.planes = (const uint8_t*)planes[l];
            L.books = (const uint16_t*)books[l];
            L.scales = (const uint16_t*)scales[l];
            L.y = y[l];
            L.out = ds[l].out;
            L.rows_pad = ds[l].rows_pad;
            L.RBc = ds[l].RBc;
            L.plane_bytes = ds[l].plane_bytes;
            L.c0 = c0;
            L.nclusters = a.nlayers > 1 ? cw_layer_clusters(ds[l].RBc, passes) : own[l];
            c0 += L.nclusters;
            if (!(ds[l].flags & AQ_LAYOUT_STATIC_WEIGHTS)) a.static_weights = 0;
        }
        a.x = (const uint16_t*)x;
        a.y_prev = y_prev;
        a.y_dt = y_dt;
        a.scale_dt = d.scale_dt;
        a.m = m;
        a.batch = batch;
        a.in = d.in;
        a.ng = d.ng;
        a.S = d.S;
        const aq_status e = d.B == 4 ? run_cw_types<4>(a, d.book_dt, x_dt, st) : run_cw_types<8>(a, d.book_dt, x_dt, st);
        if (e != AQ_OK) return e;
    }
    return AQ_OK;
}

}  // namespace aq
