// gemm_ts: y = x * W_m^T for 9 to about two thousand tokens (the prefix-m reconstruction of Sec. 3.2 /
// Sec. 5; Y = W X of Sec. 2.2) on the tcgen05 tensor cores with the decoded weights in tensor memory.
//
// The weights are the A operand: a CTA owns a tile of 32*qr output rows (qr = 1..4, one warp quarter
// of tensor-memory lanes each) and up to 256 tokens, and its decoder warps write the codewords of
// their rows straight into tensor memory (tcgen05.st), from where tcgen05.mma reads them; the
// activations are the B operand, brought by TMA (128-byte swizzle). So a decoded weight never
// passes through shared memory, the tokens need not be padded beyond a multiple of 16, and the
// tile's height is chosen to spread the rows over the SMs.
//
// Bound at up to about 128 tokens: the codeword gathers from shared memory (16 bytes per code).
// The codebooks are staged in eight interleaved copies (no bank conflicts, 8 codes per
// clock and SM; a single copy gives about 3).
//
// The decoders add the m codewords of a group in fp32, in book order, and round once to fp16 (the
// values of the other prefill kernels).
//
// K is walked in rounds of four 256-input slices: decoder warp set w (four warps, one per quarter)
// takes slice 4*round + w and produces its four 64-input stages; the MMAs take the stages of the round's
// slices in turn. A stage has one barrier for both operands (an arrival per decoder warp, and the
// TMA's bytes) and one commit: every shared-memory operation of the issuing thread queues behind
// the gathers (about 100 clocks each), so at few tokens its barrier operations would be the bound
// (two waits with abort flags and two commits per stage: 0.35 us a stage; one of each: 0.13). A
// cluster of kc CTAs splits the slices of a tile; every CTA stages its sums in shared memory (free
// once its MMAs completed) and each finishes a share of the tokens, adding the CTAs' sums in rank
// order.
// Measured (the call, with the copy of bf16 activations), against the pair kernel: 4096 x 14336, m = 3,
// 100 tokens 26.9 / 213 us; 14336 x 4096, m = 4, 100 tokens 31.0 / 79.4 us, 512 tokens 74.5 / 83 us; 16 tokens,
// m = 4: 27.7 us against 54.9 of the tf32 kernel before and 42.8 of gemv_cw. Five to eight books,
// 14336 x 4096, 16 tokens: 32 / 37 / 56 / 64 us (tf32 kernel: 66 / 77 / 88 / 179).
// Roles: warps 0-15 decoders (warp w: quarter w mod 4, set w / 4; the warps of absent quarters idle)
// and epilogue; one warp for TMA (and L2 prefetch of the codes), one for MMA issue and the
// tensor-memory allocation: with qr = 4 two more warps (96 registers a thread), else two of the idle
// ones (128 registers: with four books the next slice's codes then fit beside the current ones).
// Every mbarrier wait is bounded; a timeout records AQ_ERR_TIMEOUT in the status word and the CTA
// winds down without waiting further.
#include <cuda.h>

#include <cstring>

#include "aq_internal.cuh"
#include "launch.cuh"
#include "operand_scale.cuh"
#include "tc_ptx.cuh"

namespace aq {
namespace {

constexpr int kTsDec = 16;          // decoder warps
constexpr int kTsMaxM = 8;          // prefixes compiled (4-bit codes: 4)
constexpr int kTsRing = 8;          // weight stages in tensor memory (32 columns each, from column 256)
// Log2 of the interleaved copies of a codebook: eight while m books of them fit.
constexpr int ts_copies(int m) { return m <= 6 ? 3 : 2; }
constexpr int kTsBars = 2 * kTsRing + 1;

// One layer of a launch; a launch holds one layer, or several that share the activations and the split
// of K (aq_gemv_group), their tiles one after the other.
struct TsLayer {
    const uint8_t* planes;
    const uint16_t *books, *scales;
    void* y;
    int out, rows_pad, tile0;       // tile0: the layer's first row tile of the grid
    size_t plane_bytes;
};
struct TsArgs {
    TsLayer L[4];
    int nlayers;
    const float* xfac;              // per-token factor of the activations, or null
    unsigned int* status;
    int y_dt, scale_dt, tokens, in, ng, S;
    int qr, kc, n, nsb, spc;   // n: tokens of a tile (multiple of 16); nsb: activation stages;
    int books_off, bar_off;            // spc: slices per CTA; shared-memory offsets
    int static_weights;
};

template <int B, int BDT, int MB, bool Q4>   // Q4: four row quarters
__global__ void __launch_bounds__(Q4 ? 576 : 512, 1)
gemm_ts_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ TsArgs a) {
    constexpr int UNIT = unit_bytes(B), NC = 1 << B, NW = UNIT / 4, m = MB;
    constexpr int kTsThreads = Q4 ? 576 : 512, kTmaWarp = Q4 ? 16 : 3, kMmaWarp = Q4 ? 17 : 7;
    constexpr bool kAhead = MB <= (Q4 ? 3 : 4);         // next slice's codes in registers ahead of use
    constexpr int kCopies = ts_copies(MB);
    extern __shared__ __align__(1024) unsigned char smem[];
    uint4* books_s = (uint4*)(smem + a.books_off);
    uint64_t* full = (uint64_t*)(smem + a.bar_off);     // both operands of a stage are in place
    uint64_t* empty = full + kTsRing;                   // the MMAs reading the stage completed
    uint64_t* acc_full = empty + kTsRing;
    float* scale_s = (float*)(smem + a.bar_off + (kTsBars + 1) * 8);   // [128] row scales times 2^f
    float* xf_s = scale_s + 128;                        // [256] token factors
    __shared__ uint32_t s_tmem;
    __shared__ unsigned int s_wmax[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = a.kc > 1 ? (int)cluster_rank() : 0;
    int tile = (int)blockIdx.x / a.kc, layer = 0;
    while (layer + 1 < a.nlayers && tile >= a.L[layer + 1].tile0) ++layer;
    const TsLayer& L = a.L[layer];
    const int row0 = (tile - L.tile0) * 32 * a.qr;
    const int t0 = (int)blockIdx.y * a.n;
    const int sl0 = rank * a.spc, nsl = max(0, min(a.S - sl0, a.spc));   // this CTA's slices

    if (smem_u32(smem) & 1023u) {   // the same answer in every CTA
        if (tid == 0) record_status(a.status, AQ_ERR_ALIGNMENT);
        return;
    }
    // Everything that the weights give, requested before anything is waited for: a CTA's start is one
    // chain of latencies (codebooks, their largest entry, their copies, the first codes), and a call has the
    // SM to itself, so none of it hides behind other work.
    const int q = warp & 3, ws = warp >> 2;             // decoders: row quarter, slice of a round
    const bool decoder = warp < kTsDec && q < a.qr;
    const int row = row0 + q * 32 + lane;
    const bool row_in = row < L.rows_pad;
    // A row's codes of a slice, in two steps to group order (position p holds group (p + row) mod
    // 32): the loads bring the 8-byte pieces rotated by whole pieces (B = 8), unrotate() does the
    // rest of the rotation, a word and up to three bytes.
    const int rr8 = (row >> 3) & 3;
    auto load_raw = [&](int s, int k, uint32_t (&raw)[NW]) {
#pragma unroll
        for (int i = 0; i < NW; ++i) raw[i] = 0u;
        if (row_in) {
            const uint8_t* src = L.planes + (size_t)k * L.plane_bytes + ((size_t)s * L.rows_pad + row) * UNIT;
            if constexpr (B == 8) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint2 v = __ldg((const uint2*)src + ((i - rr8) & 3));
                    raw[2 * i] = v.x;
                    raw[2 * i + 1] = v.y;
                }
            } else {
                const uint4 v = ld_stream_v4(src);
                raw[0] = v.x;
                raw[1] = v.y;
                raw[2] = v.z;
                raw[3] = v.w;
            }
        }
    };
    uint32_t raw[MB][NW];
    auto load_slice = [&](int s) {
#pragma unroll
        for (int k = 0; k < MB; ++k) load_raw(s, k, raw[k]);
    };
    // the codes of a round's slices, HBM to L2
    const int rows_here = max(0, min(32 * a.qr, L.rows_pad - row0));
    auto prefetch_round = [&](int r) {
        if (rows_here > 0)
            for (int w = 0; w < 4 && 4 * r + w < nsl; ++w)
                for (int k = 0; k < m; ++k)
                    prefetch_l2(L.planes + (size_t)k * L.plane_bytes +
                                    ((size_t)(sl0 + 4 * r + w) * L.rows_pad + row0) * UNIT,
                                (uint32_t)(rows_here * UNIT));
    };
    constexpr int kPer = (MB * NC + kTsThreads - 1) / kTsThreads;
    uint4 bk[kPer];                                     // this thread's codewords
    uint16_t sbits = 0;                                 // the scale of row row0 + tid
    auto fetch = [&]() {
#pragma unroll
        for (int l = 0; l < kPer; ++l) {
            const int i = tid + l * kTsThreads;
            bk[l] = i < m * NC ? __ldg((const uint4*)L.books + i) : make_uint4(0u, 0u, 0u, 0u);
        }
        if (warp == kTmaWarp && elect_one()) {
            prefetch_round(0);
            prefetch_round(1);
        }
        if (kAhead && decoder && ws < nsl) load_slice(sl0 + ws);
        if (tid < 32 * a.qr && row0 + tid < L.out) sbits = L.scales[row0 + tid];
    };
    if (a.static_weights) fetch();   // read-only weights: before the preceding kernel has finished
    if (tid == 0) {
        for (int i = 0; i < kTsRing; ++i) {
            mbar_init(&full[i], a.qr + 1);
            mbar_init(&empty[i], 1);
        }
        mbar_init(acc_full, 1);
        mbar_fence_init();
    }
    if (tid < 8) s_wmax[tid] = 0u;
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    __syncthreads();
    if (!a.static_weights) {
        pdl_wait();
        pdl_launch_dependents();
        fetch();
    }
    // Books staged times 2^-f (fp16 range, operand_scale.cuh): each thread writes the copies of its
    // codewords, starting at copy `lane` so that eight lanes meet no bank group twice.
#pragma unroll
    for (int l = 0; l < kPer; ++l) {
        const int i = tid + l * kTsThreads;
        const unsigned int mx = codeword_max_bits<BDT>(bk[l]);
        if constexpr (B == 8) {                         // the 32 codewords of a warp are of one book
            const unsigned int wm = __reduce_max_sync(0xffffffffu, mx);
            if (lane == 0 && i < m * NC) atomicMax(&s_wmax[i >> B], wm);
        } else if (i < m * NC) {
            atomicMax(&s_wmax[i >> B], mx);
        }
    }
    __syncthreads();
    const int f = book_exponent<BDT>(s_wmax, MB);
    const float bfac = pow2f(f);
#pragma unroll
    for (int l = 0; l < kPer; ++l) {
        const int i = tid + l * kTsThreads;
        const uint4 v = f ? scale_codeword<BDT>(bk[l], pow2f(-f)) : bk[l];
        if (i < m * NC)
#pragma unroll
            for (int c = 0; c < 1 << kCopies; ++c) books_s[(i << kCopies) + ((c + lane) & ((1 << kCopies) - 1))] = v;
    }
    if (tid < 128) scale_s[tid] = bits_to_f32_rt(sbits, a.scale_dt) * bfac;
    if (a.static_weights) {
        pdl_wait();
        pdl_launch_dependents();
    }
    // the token factors of the preceding copy, for the epilogue
    const float xf_r = a.xfac && tid < a.n && t0 + tid < a.tokens ? a.xfac[t0 + tid] : 1.0f;
    tc_fence_before();
    __syncthreads();          // books staged, barriers initialised, tensor memory allocated
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const int nrounds = (nsl + 3) / 4;
    const int stage_b = a.n * 128;

    if (warp == kTmaWarp) {
        // ---------------- activations: stages (j, w) of every round
        if (elect_one()) {
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&xmap) : "memory");
            int issued = 0, slot = 0;
            bool stop = false;
            for (int r = 0; r < nrounds && !stop; ++r) {
                if (r + 2 < nrounds) prefetch_round(r + 2);
                const int ns = min(4, nsl - 4 * r);
                for (int j = 0; j < 4 && !stop; ++j)
                    for (int w = 0; w < ns; ++w) {
                        // the slot's previous stage (a.nsb <= kTsRing stages ago) has been multiplied
                        const int prev = issued - a.nsb;
                        if (prev >= 0 && !mbar_wait(&empty[prev & (kTsRing - 1)], (prev / kTsRing) & 1)) {
                            record_status(a.status, AQ_ERR_TIMEOUT);
                            stop = true;
                            break;
                        }
                        uint64_t* bar = &full[issued & (kTsRing - 1)];
                        mbar_arrive_expect_tx(bar, (uint32_t)stage_b);
                        tma_load_2d(smem + (size_t)slot * stage_b, &xmap, (sl0 + 4 * r + w) * 256 + j * 64, t0, bar);
                        ++issued;
                        if (++slot == a.nsb) slot = 0;
                    }
            }
            // No copy may still be in flight when the CTA reuses the stages or exits: every stage's
            // barrier completes (its decoders arrive too, even after a timeout).
            for (int i = max(0, issued - a.nsb); i < issued; ++i) mbar_wait(&full[i & (kTsRing - 1)], (i / kTsRing) & 1);
        }
        __syncwarp();
    } else if (warp == kMmaWarp) {
        // ---------------- MMA issuer
        if (elect_one()) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(a.n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
            const uint32_t b0 = smem_u32(smem);
            int slot = 0;
            for (int i = 0; i < 4 * nsl; ++i) {
                const int st = i & (kTsRing - 1);
                if (!mbar_wait(&full[st], (i / kTsRing) & 1)) {
                    record_status(a.status, AQ_ERR_TIMEOUT);
                    break;
                }
                tc_fence_after();
                const uint32_t bs = b0 + (uint32_t)slot * stage_b;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    umma_f16_ts(tmem, tmem + 256 + st * 32 + kk * 8, umma_desc_sw128(bs + kk * 32), idesc,
                                (i > 0 || kk > 0) ? 1u : 0u);
                umma_commit(&empty[st]);
                if (++slot == a.nsb) slot = 0;
            }
            umma_commit(acc_full);
            mbar_wait(acc_full, 0);         // every MMA has completed before anything is reused
            tc_fence_after();
            tc_fence_before();
        }
        __syncwarp();
    } else if (decoder) {
        // ---------------- decoders
        constexpr uint32_t mul = 16u << kCopies;
        const uint32_t books_u = smem_u32(books_s) + ((uint32_t)(lane & ((1 << kCopies) - 1)) << 4);
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + 256;
        auto unrotate = [&](const uint32_t (&raw)[NW], uint32_t (&u)[NW]) {
            if constexpr (B == 8) {
                const bool odd = (row >> 2) & 1;
                const int rb = (row & 3) * 8;
                uint32_t t[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) t[i] = odd ? raw[(i + 7) & 7] : raw[i];
#pragma unroll
                for (int i = 0; i < 8; ++i) u[i] = __funnelshift_l(t[(i + 7) & 7], t[i], rb);
            } else {
                unrotate_nibbles(raw, row, u);
            }
        };
        // byte offset of the codeword of group 8j + i in its book's copies
        auto offset = [&](const uint32_t (&u)[NW], int j, int i) {
            if constexpr (B == 8) return prmt(u[2 * j + (i >> 2)], 0u, 0x4440u | (uint32_t)(i & 3)) * mul;
            else return ((u[j] >> (4 * i)) & 15u) * mul;
        };
        // writes one stage (eight groups; group(i) = the eight fp16 weights of group g0 + i)
        bool dead = false;                              // a wait gave up: no more waiting
        auto write_stage = [&](int idx, int g0, auto group) {
            const int st = idx & (kTsRing - 1);
            if (idx >= kTsRing && !dead && !mbar_wait(&empty[st], ((idx / kTsRing) - 1) & 1)) {
                record_status(a.status, AQ_ERR_TIMEOUT);
                dead = true;
            }
            __syncwarp();
            tc_fence_after();
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                uint32_t r[8];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    uint4 c = group(2 * h + i);
                    if (g0 + 2 * h + i >= a.ng) c = make_uint4(0u, 0u, 0u, 0u);   // past the row's end
                    r[4 * i] = c.x;
                    r[4 * i + 1] = c.y;
                    r[4 * i + 2] = c.z;
                    r[4 * i + 3] = c.w;
                }
                tmem_st8(tq + st * 32 + h * 8, r);
            }
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[st]);
        };
        int base = 0;                                   // weight stages of the earlier rounds
        // The next slice's codes are requested before the last stage of a slice (when most of the
        // current ones are used up), so their way from L2 (about 2000 clocks) is not waited for.
        for (int r = 0; r < nrounds; ++r) {
            const int ns = min(4, nsl - 4 * r);
            if (ws < ns) {
                const int s = sl0 + 4 * r + ws;
                if (!kAhead) load_slice(s);
                uint32_t u[MB][NW];
#pragma unroll
                for (int k = 0; k < MB; ++k) unrotate(raw[k], u[k]);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (kAhead && j == 3 && 4 * (r + 1) + ws < nsl) load_slice(s + 4);
                    write_stage(base + j * ns + ws, s * 32 + 8 * j, [&](int i) {
                        const uint4 c0 = lds128(books_u + offset(u[0], j, i));
                        if constexpr (MB == 1 && BDT == AQ_F16) {
                            return c0;              // an fp16 codeword as it is
                        } else {
                            // one mixed-type add per element; -0 + v = v exactly
                            float v[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) v[e] = -0.0f;
                            add_widen2<BDT>(c0.x, v[0], v[1]);
                            add_widen2<BDT>(c0.y, v[2], v[3]);
                            add_widen2<BDT>(c0.z, v[4], v[5]);
                            add_widen2<BDT>(c0.w, v[6], v[7]);
#pragma unroll
                            for (int k = 1; k < MB; ++k) {
                                const uint4 ck = lds128(books_u + (uint32_t)k * (NC * mul) + offset(u[k], j, i));
                                add_widen2<BDT>(ck.x, v[0], v[1]);
                                add_widen2<BDT>(ck.y, v[2], v[3]);
                                add_widen2<BDT>(ck.z, v[4], v[5]);
                                add_widen2<BDT>(ck.w, v[6], v[7]);
                            }
                            return make_uint4(f16x2(make_float2(v[0], v[1])), f16x2(make_float2(v[2], v[3])),
                                              f16x2(make_float2(v[4], v[5])), f16x2(make_float2(v[6], v[7])));
                        }
                    });
                }
            }
            base += 4 * ns;
        }
    }

    // ---------------- epilogue: the CTA's sums [token][row] into shared memory, then y
    __syncthreads();          // (the issuer waited for the last MMA: the operand stages and books are free)
    tc_fence_after();
    const int R = 32 * a.qr, P = R + 4;
    float* cs = (float*)smem;
    if (tid < a.n) xf_s[tid] = xf_r;
    if (decoder) {
        for (int c = ws * 16; c < a.n; c += 64) {
            float v[16];
            if (nsl > 0) tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + c, v);
            else
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = 0.0f;
#pragma unroll
            for (int i = 0; i < 16; ++i) cs[(c + i) * P + q * 32 + lane] = v[i];
        }
    }
    tc_fence_before();
    if (a.kc > 1) cluster_sync();
    else __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
    const int ntok = min(a.n, a.tokens - t0), share = (ntok + a.kc - 1) / a.kc;
    const int ta = rank * share, tb = min(ntok, ta + share);
    const bool vec = (L.out & 7) == 0;
    // A thread finishes four rows (always the same ones) of every nt-th token: 16 bytes of each CTA's sums,
    // contiguous over the lanes (eight rows, 32 bytes apart, took 5400 clocks for 28 tokens of four CTAs).
    const int R4 = 8 * a.qr, nt = kTsThreads / R4, rr = tid % R4 * 4, o = row0 + rr;
    const float4 sc = *(const float4*)(scale_s + rr);
    void* const y = L.y;
    const int out = L.out;
    for (int tl = ta + tid / R4; tl < tb && tid < nt * R4 && o < out; tl += nt) {
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        const uint32_t addr = smem_u32(cs + tl * P + rr);
        for (int r4 = 0; r4 < a.kc; r4 += 4) {         // the CTAs' sums, in rank order; four loads in flight
            float4 p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r4 + i;
                p[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (r == rank) {
                    p[i] = *(const float4*)(cs + tl * P + rr);
                } else if (r < a.kc) {
                    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                                 : "=f"(p[i].x), "=f"(p[i].y), "=f"(p[i].z), "=f"(p[i].w)
                                 : "r"(map_to_rank(addr, (uint32_t)r)) : "memory");
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                v.x += p[i].x;
                v.y += p[i].y;
                v.z += p[i].z;
                v.w += p[i].w;
            }
        }
        const float xf = xf_s[tl];
        const size_t yi = (size_t)(t0 + tl) * out + o;
        auto scaled = [&](float p, float s) { return p * (xf > 1.0f ? s : xf) * (xf > 1.0f ? xf : s); };   // operand_scale.cuh
        const float w[4] = {scaled(v.x, sc.x), scaled(v.y, sc.y), scaled(v.z, sc.z), scaled(v.w, sc.w)};
        if (vec && a.y_dt == AQ_F32) {
            *(float4*)((float*)y + yi) = make_float4(w[0], w[1], w[2], w[3]);
        } else if (vec) {
            *(uint2*)((uint16_t*)y + yi) =
                a.y_dt == AQ_F16 ? make_uint2(round_pack2<AQ_F16>(w[0], w[1]), round_pack2<AQ_F16>(w[2], w[3]))
                                 : make_uint2(round_pack2<AQ_BF16>(w[0], w[1]), round_pack2<AQ_BF16>(w[2], w[3]));
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (o + e < out) {
                    if (a.y_dt == AQ_F32) ((float*)y)[yi + e] = w[e];
                    else ((uint16_t*)y)[yi + e] = a.y_dt == AQ_F16 ? f32_to_bits<AQ_F16>(w[e]) : f32_to_bits<AQ_BF16>(w[e]);
                }
        }
    }
    if (a.kc > 1) cluster_sync();   // no CTA leaves while a peer may still read its sums
}

// ---- host side ------------------------------------------------------------------------------

struct TsPlan {
    int n, ntiles, qr, kc, spc, nsb, books_off, bar_off;   // (kc, spc: of the first layer)
    size_t smem;
    double clocks;                     // estimated time of the call
};

// The split of a call: token tiles of equal height (multiples of 16 up to 256), then the tile height
// in row quarters and the cluster size with the smallest estimated time, in clocks: waves of the
// busiest SM times 64-input stages plus the fixed cost of a CTA (staging the books, filling the
// pipeline, the epilogue) and of a cluster's exchange. A stage takes the longest of (measured): its
// MMAs (268 clocks at 112 tokens, 556 at 256); the issuer's barrier and commit (270); shared memory:
// the gathers of 8 groups per row and book at 60 % of 8 codes a clock, and the activations' way
// through it; a decoder warp's own chain (120 m + 165, a stage in four being its own), which bounds
// one or two quarters and a last round of fewer than four slices. From five books the codes of a slice are
// waited for (their registers leave no room to load them ahead), and from seven the four copies of a book
// cost about twice the gathers; three quarters at most keep 128 registers a thread. Eight clusters of eight are
// resident at once beside the preceding call's (see cw_cluster); sixteen ran in two waves (1024 x 8192, m = 2,
// 16 tokens: 15.3 us where eight of them, 256 rows, took 7.9).
// With a group of layers (nl > 1; the same K and number of books, so the same kc and spc each), the
// tile height is chosen for the tiles of all of them and kc is the given one.
bool ts_plan(const Dims* ds, int nl, int m, int tokens, const DeviceInfo& di, TsPlan* p, int only_kc = 0) {
    const Dims& d = ds[0];
    if ((d.B != 8 && d.B != 4) || m > (d.B == 8 ? kTsMaxM : 4)) return false;
    p->ntiles = (tokens + 255) / 256;
    p->n = ((tokens + p->ntiles - 1) / p->ntiles + 15) / 16 * 16;
    const int books = (m * 16 << d.B) << ts_copies(m), stage = p->n * 128;
    const int tail = (kTsBars + 1) * 8 + (128 + 256) * 4;
    int nsb = (di.smem_optin - books - tail - 1024 - 16) / stage;   // (1 KiB of static shared memory)
    if (nsb > kTsRing) nsb = kTsRing;
    if (nsb < 2) return false;
    p->nsb = nsb;
    double best = -1.0;
    const double gathers = m <= 6 ? m : 1.9 * m;
    for (int qr = 1; qr <= (m <= 4 ? 4 : 3); ++qr)
        for (int kc = 1; kc <= 8; kc *= 2) {
            if (kc > d.S || (only_kc && kc != only_kc)) continue;
            long long tiles = 0;
            for (int l = 0; l < nl; ++l) tiles += (ds[l].out + 32 * qr - 1) / (32 * qr);
            tiles *= p->ntiles;
            const int cap = kc == 1 ? di.sms : kc == 2 ? di.sms / 2 : kc == 4 ? di.sms * 9 / 38 : di.sms / 19;
            const int spc = (d.S + kc - 1) / kc;
            const long long waves = (tiles + cap - 1) / cap;
            const double chain = (m <= 6 ? 120.0 : 180.0) * m + (m <= 4 ? 165.0 : 200.0) + p->n * 0.3;
            double stage_clk = p->n * 2.2 > 270.0 ? p->n * 2.2 : 270.0;
            if (qr * 53.0 * gathers + p->n * 0.45 > stage_clk) stage_clk = qr * 53.0 * gathers + p->n * 0.45;
            if (chain > stage_clk) stage_clk = chain;
            const double t = waves * (spc / 4 * 16 * stage_clk + (spc % 4 ? 16 * chain : 0.0) + 5000.0 +
                                      (kc == 1 ? 0.0 : 1500.0) + p->n * 16.0);
            if (best < 0.0 || t < best) {
                best = t;
                p->qr = qr;
                p->kc = kc;
                p->spc = spc;
            }
        }
    p->clocks = best;
    const size_t ring = (size_t)p->nsb * stage, sums = (size_t)p->n * (32 * p->qr + 4) * 4;
    p->books_off = (int)ring;
    size_t end = ring + books;
    if (end < sums) end = sums;
    p->bar_off = (int)round_up(end, 16);
    p->smem = p->bar_off + tail;
    // One CTA per SM always (each allocates all of tensor memory, and a cluster whose CTAs wait for
    // each other must not wait for tensor memory that another cluster holds).
    if (p->smem < 118 * 1024) p->smem = 118 * 1024;
    return p->smem + 1024 <= (size_t)di.smem_optin;
}

template <int B, int BDT, int MB>
aq_status run_ts(const TsPlan& p, const CUtensorMap& map, const TsArgs& a, int tiles, cudaStream_t st) {
    auto kern = gemm_ts_kernel<B, BDT, MB, false>;
    if constexpr (MB <= 4)
        if (p.qr == 4) kern = gemm_ts_kernel<B, BDT, MB, true>;
    const int threads = p.qr == 4 ? 576 : 512;
    int occ = 0;
    // slot 0: the limit is raised to the most a launch may use; each plan stays below it
    if (aq_status e = prepare(kern, 118 * 1024, threads, 0, &occ); e != AQ_OK) return e;
    return launch_pdl_cluster(p.kc, kern, dim3(tiles * p.kc, p.ntiles), dim3(threads), p.smem, st, map, a);
}

template <int B, int BDT>
aq_status run_ts_m(const TsPlan& p, const CUtensorMap& map, const TsArgs& a, int m, int tiles, cudaStream_t st) {
    switch (m) {
        case 1: return run_ts<B, BDT, 1>(p, map, a, tiles, st);
        case 2: return run_ts<B, BDT, 2>(p, map, a, tiles, st);
        case 3: return run_ts<B, BDT, 3>(p, map, a, tiles, st);
        case 4: return run_ts<B, BDT, 4>(p, map, a, tiles, st);
    }
    if constexpr (B == 8) {
        switch (m) {
            case 5: return run_ts<B, BDT, 5>(p, map, a, tiles, st);
            case 6: return run_ts<B, BDT, 6>(p, map, a, tiles, st);
            case 7: return run_ts<B, BDT, 7>(p, map, a, tiles, st);
            case 8: return run_ts<B, BDT, 8>(p, map, a, tiles, st);
        }
    }
    return AQ_ERR_UNSUPPORTED;
}

// One launch: plan p, the layers of a filled in, `tiles` row tiles.
aq_status launch_ts_set(const Dims& d, int m, const TsPlan& p, TsArgs a, int tiles, const void* x, const float* xfac,
                        int tokens, int y_dt, void* ws, cudaStream_t st) {
    EncodeTiledFn encode;
    if (aq_status e = get_encode_fn(&encode); e != AQ_OK) return e;
    CUtensorMap map;
    std::memset(&map, 0, sizeof(map));
    const cuuint64_t dims[2] = {(cuuint64_t)d.in, (cuuint64_t)tokens};
    const cuuint64_t strides[1] = {(cuuint64_t)d.in * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)p.n};
    const cuuint32_t estr[2] = {1, 1};
    if (encode(&map, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, const_cast<void*>(x), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return AQ_ERR_CUDA;
    a.xfac = xfac;
    a.status = (unsigned int*)ws;
    a.y_dt = y_dt;
    a.scale_dt = d.scale_dt;
    a.tokens = tokens;
    a.in = d.in;
    a.ng = d.ng;
    a.S = d.S;
    a.qr = p.qr;
    a.kc = p.kc;
    a.n = p.n;
    a.nsb = p.nsb;
    a.spc = p.spc;
    a.books_off = p.books_off;
    a.bar_off = p.bar_off;
    if (d.B == 4)
        return d.book_dt == AQ_BF16 ? run_ts_m<4, AQ_BF16>(p, map, a, m, tiles, st)
                                    : run_ts_m<4, AQ_F16>(p, map, a, m, tiles, st);
    return d.book_dt == AQ_BF16 ? run_ts_m<8, AQ_BF16>(p, map, a, m, tiles, st)
                                : run_ts_m<8, AQ_F16>(p, map, a, m, tiles, st);
}

}  // namespace

double ts_clocks(const Dims& d, int m, int tokens) {
    DeviceInfo di;
    TsPlan p;
    return device_info(&di) == AQ_OK && ts_plan(&d, 1, m, tokens, di, &p) ? p.clocks : -1.0;
}

// x: fp16 [tokens][in], 16-byte aligned. n layers that share it: those whose own plans have the same
// cluster size go together (their sums are then those of their own calls), unless launches of their own
// are estimated to be faster.
aq_status launch_ts(const Dims* ds, int n, int m, const void* const* planes, const void* const* books,
                    const void* const* scales, const void* x, const float* xfac, int tokens, void* const* y,
                    int y_dt, void* ws, cudaStream_t st) {
    DeviceInfo di;
    if (aq_status e = device_info(&di); e != AQ_OK) return e;
    TsPlan own[4];
    for (int l = 0; l < n; ++l)
        if (!ts_plan(&ds[l], 1, m, tokens, di, &own[l])) return AQ_ERR_UNSUPPORTED;
    bool done[4] = {};
    for (int f = 0; f < n; ++f) {
        if (done[f]) continue;
        Dims set[4];
        int idx[4], ns = 0;
        TsPlan p = own[f];
        double apart = 0.0;
        for (int l = f; l < n; ++l) {
            if (done[l] || own[l].kc != own[f].kc) continue;
            set[ns] = ds[l];
            idx[ns++] = l;
            apart += own[l].clocks;
            // a launch of its own costs about 3000 clocks more than its tiles
            TsPlan joint;
            if (ns > 1) {
                if (ts_plan(set, ns, m, tokens, di, &joint, own[f].kc) && joint.clocks < apart + 3000.0 * (ns - 1)) p = joint;
                else {
                    apart -= own[l].clocks;
                    --ns;
                }
            }
        }
        TsArgs a = {};
        a.nlayers = ns;
        a.static_weights = 1;
        int tiles = 0;
        for (int i = 0; i < ns; ++i) {
            const int l = idx[i];
            done[l] = true;
            TsLayer& L = a.L[i];
            L.planes = (const uint8_t*)planes[l];
            L.books = (const uint16_t*)books[l];
            L.scales = (const uint16_t*)scales[l];
            L.y = y[l];
            L.out = ds[l].out;
            L.rows_pad = ds[l].rows_pad;
            L.plane_bytes = ds[l].plane_bytes;
            L.tile0 = tiles;
            tiles += (ds[l].out + 32 * p.qr - 1) / (32 * p.qr);
            if (!(ds[l].flags & AQ_LAYOUT_STATIC_WEIGHTS)) a.static_weights = 0;
        }
        if (aq_status e = launch_ts_set(ds[f], m, p, a, tiles, x, xfac, tokens, y_dt, ws, st); e != AQ_OK) return e;
    }
    return AQ_OK;
}

}  // namespace aq
