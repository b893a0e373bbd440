// hcw_small.cu -- whole stacks of narrow layers (d = 64 or 128) over short windows
// (n <= 128), bf16: a CTA keeps 128 tokens, whole samples, on chip through the
// forward and / or the input gradient of every layer.
//
// The stacked launches of hcw_tc.cu hand every layer's rows to the next through
// global memory and counters: at d = 128 a layer step of their chain is about 6 us,
// of which the products are a tenth.  At these sizes a 128-token tile holds every
// partner (links stay inside a sample), so nothing has to leave the SM between layers:
//   - A (128 tokens x d, K-major, 128-byte swizzle) holds the layer's input (in the
//     backward: its dz), and A2 the partner rows, row for row: the thread that owns a
//     token writes its new row into A and into the row of A2 that receives from it;
//   - z = A W_self^T + A2 W_nbr^T is d / 16 MMAs each (tcgen05, M = 128, N = d) into one
//     TMEM accumulator, self part first; a link that not every row takes runs its
//     partner MMAs with the other lanes' output disabled;
//   - eight epilogue warps (a row and half the columns a thread) apply bias, ReLU,
//     residual (kept in registers) and the bf16 rounding, write the ReLU masks, and
//     store the next A and A2;
//   - both weight matrices of the next layer stream into a two-stage ring meanwhile;
//     one copy of a matrix, as 64-feature tiles, serves the forward as a K-major
//     operand and the input gradient as an MN-major one;
//   - A goes to global memory by TMA while the MMAs read it (the stack's acts, and dz).
// The sums and roundings are those of the layer-by-layer launches, in the same order:
// the results are the same bits.
//
// What bounds it: a layer is a chain of the MMAs and the epilogue, 4,700 cycles
// forward and 4,200 backward at d = 128 (16 MMAs 1,500; accumulator to bf16 1,400 with
// bias and ReLU, 500 without, bound by the warps' issue slots; the ReLU mask of dz 500;
// A and A2 written 750, bound by shared-memory bandwidth; barriers 600).  Training
// step of 16,384 tokens (n = 64, d = 128, 6 layers, without the causal rule): the forward
// and input gradient 70.8 -> 37.9 us, the step 101 -> 64 us (55 as programmatic
// dependents); a 20-layer causal forward of 1,216 tokens 107 -> 58 us.
#include "hcw.h"
#include "hcw_internal.h"
#include "hcw_ptx.cuh"

#include <atomic>
#include <type_traits>

namespace hcw {

namespace {

constexpr int kTok = 128;                  // tokens per CTA
constexpr int kEpi = 8;                    // epilogue warps: two per TMEM lane quarter
constexpr int kSmallThreads = 64 + 32 * kEpi;
constexpr int kBiasSlots = 4;              // steps' biases in flight

struct __align__(8) SmallBars {
    uint64_t wfull[2];    // a layer's weights landed
    uint64_t wempty[2];   // its MMAs have read them
    uint64_t aready;      // A and A2 hold a step's operands (the epilogue warps)
    uint64_t wseen;       // the MMA thread has seen the step's weights and bias land
    uint64_t accfull;     // the step's MMAs are complete
    uint64_t astored;     // the step's store of A (if any) has read it
    uint64_t drain;
    uint32_t tmem_base;
    int abort;
    // lanes without a partner part, per direction and layer
    uint32_t skip[2][kMaxSmallLayers][4];
};

template <int D>
constexpr size_t small_smem() {
    return 1024 + (size_t)2 * 2 * D * D * 2 + (size_t)2 * kTok * D * 2 + kBiasSlots * D * 4 +
           sizeof(SmallBars);
}

// link s of position i of a sample of n: as in hcw_simt.cu
__device__ __forceinline__ bool link_receives(int i, int s, unsigned flags) {
    if (s < 0) return i + s >= 0;
    return !(flags & 1u) || ((i >> s) & 1);
}
// the position that takes x_i as its partner input, or -1
__device__ __forceinline__ int link_reader(int i, int s, int n, unsigned flags) {
    if (s < 0) return i - s < n ? i - s : -1;
    const int p = i ^ (1 << s);
    return link_receives(p, s, flags) ? p : -1;
}
__device__ __forceinline__ int link_partner(int i, int s) { return s >= 0 ? i ^ (1 << s) : i + s; }

// `bytes` (a multiple of 16, both addresses 16-byte aligned) from global memory into this
// CTA's shared memory, completing on bar
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// tcgen05.mma with the output lanes of the set bits left as they are
__device__ __forceinline__ void mma_bf16_f32_masked(uint32_t d_tmem, uint64_t adesc,
                                                    uint64_t bdesc, uint32_t idesc,
                                                    const uint32_t (&m)[4]) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.eq.b32 p, 0, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, {%4, %5, %6, %7}, p;\n\t}" ::"r"(
            d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(m[0]), "r"(m[1]), "r"(m[2]), "r"(m[3])
        : "memory");
}

template <int D>
__global__ void __launch_bounds__(kSmallThreads, D == 64 ? 2 : 1)
    hcw_small_kernel(const __grid_constant__ SmallLaunch L) {
    constexpr int KT = D / 64;                        // 64-feature tiles
    constexpr uint32_t kTileA = kTok * 128;           // bytes of a tile of A
    constexpr uint32_t kMat = D * D * 2;              // bytes of a weight matrix
    constexpr int HC = D / 2;                         // columns per epilogue thread
    constexpr int NW = HC / 2;                        // ... as bf16 pairs
    constexpr int NM = HC / 32;                       // ... and mask words
    constexpr int WPR = D / 32;                       // mask words per row
    constexpr uint32_t IDESC_F = idesc_bf16_f32(kTok, D, 0, 0);
    constexpr uint32_t IDESC_B = idesc_bf16_f32(kTok, D, 0, 1);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* wts = smem;                              // [2 stages][W_self, W_nbr]
    uint8_t* A = smem + 4 * kMat;
    uint8_t* A2 = A + kTok * D * 2;
    float* biases = reinterpret_cast<float*>(A2 + kTok * D * 2);   // [kBiasSlots][D]
    SmallBars* bars = reinterpret_cast<SmallBars*>(biases + kBiasSlots * D);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort = &bars->abort;
    const uint64_t tmo = L.timeout_ns;
    const int nL = L.n_layers;
    const int steps = (L.fwd ? nL : 0) + (L.bwd ? nL : 0);   // per block of tokens
    const int blocks = (L.tokens + kTok - 1) / kTok;
    // step -> layer and direction
    auto step_fwd = [&](int t) { return L.fwd && t < nL; };
    auto step_layer = [&](int t) {
        return step_fwd(t) ? t : nL - 1 - (L.fwd ? t - nL : t);
    };

    if (threadIdx.x == 0) {
        tma_prefetch_desc(&L.mWs);
        tma_prefetch_desc(&L.mWn);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars->wfull[i], 1);
            mbar_init(&bars->wempty[i], 1);
        }
        mbar_init(&bars->aready, kEpi);
        mbar_init(&bars->wseen, 1);
        mbar_init(&bars->accfull, 1);
        mbar_init(&bars->astored, 1);
        mbar_init(&bars->drain, 1);
        bars->abort = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(&bars->tmem_base, D);
        tmem_relinquish();
    }
    if (!L.bias)
        for (int i = threadIdx.x; i < kBiasSlots * D; i += kSmallThreads) biases[i] = 0.f;
    if (warp >= 2 && warp < 6) {
        // rows 32 q .. 32 q + 31 (a sample starts on a multiple of n)
        const int q = warp - 2, i = (q * 32 + lane) & (L.n - 1);
        for (int l = 0; l < nL; ++l) {
            const int s = L.link[l];
            const uint32_t f = __ballot_sync(0xffffffffu, !link_receives(i, s, L.flags));
            const uint32_t g = __ballot_sync(0xffffffffu, link_reader(i, s, L.n, L.flags) < 0);
            if (lane == 0) {
                bars->skip[0][l][q] = f;
                bars->skip[1][l][q] = g;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = bars->tmem_base;
    // the prologue above touched no global memory: it overlaps the end of the kernel
    // before it when launched as a programmatic dependent
    pdl_wait();
    pdl_trigger();

    if (warp == 0) {
        // ------------------------------------------------------------ weights
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int b = blockIdx.x; b < blocks && ok; b += gridDim.x)
                for (int t = 0; t < steps; ++t, ++it) {
                    const int st = it & 1;
                    if (it >= 2 && !mbar_wait(&bars->wempty[st], ((it >> 1) - 1) & 1, abort, tmo)) {
                        ok = false;
                        break;
                    }
                    uint8_t* dst = wts + (size_t)st * 2 * kMat;
                    const int row = step_layer(t) * D;
                    const bool bias = L.bias && step_fwd(t);
                    mbar_arrive_expect_tx(&bars->wfull[st], 2 * kMat + (bias ? D * 4 : 0));
                    // (the slot's last reader, step it - 4's epilogue, was done before step
                    // it - 3's MMAs began)
                    if (bias)
                        bulk_load(biases + (it % kBiasSlots) * D, L.bias + row, D * 4,
                                  &bars->wfull[st]);
                    tma_load_3d(dst, &L.mWs, &bars->wfull[st], 0, row, 0);
                    tma_load_3d(dst + kMat, &L.mWn, &bars->wfull[st], 0, row, 0);
                }
            if (!ok)   // let the copies in flight land before the CTA exits
                for (uint32_t j = it > 2 ? it - 2 : 0; j < it; ++j)
                    mbar_wait_drain(&bars->wfull[j & 1], (j >> 1) & 1, tmo);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMAs, stores of A
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int b = blockIdx.x; b < blocks && ok; b += gridDim.x)
                for (int t = 0; t < steps; ++t, ++it) {
                    const int l = step_layer(t);
                    const bool f = step_fwd(t);
                    // lanes whose row has no partner part (bit set: output disabled)
                    uint32_t m[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) m[q] = bars->skip[f ? 0 : 1][l][q];
                    const bool all = (m[0] | m[1] | m[2] | m[3]) == 0u;
                    const int st = it & 1;
                    if (!mbar_wait(&bars->wfull[st], (it >> 1) & 1, abort, tmo) ||
                        !mbar_wait(&bars->aready, it & 1, abort, tmo)) {
                        ok = false;
                        break;
                    }
                    // (after aready: the epilogue has seen the step before)
                    mbar_arrive(&bars->wseen);
                    // A to global memory (the forward's input of layer l > 0, or dz_l), read
                    // while the MMAs run; the epilogue overwrites A after both
                    if (f ? l > 0 : true) {
                        for (int k = 0; k < KT; ++k)
                            tma_store_3d(f ? &L.mActs : &L.mDz, A + k * kTileA, k * 64, b * kTok,
                                         f ? l - 1 : l);
                        bulk_commit();
                    }
                    tc_fence_after();
                    const uint32_t a = smem_u32(A), a2 = smem_u32(A2);
                    const uint32_t ws = smem_u32(wts) + (uint32_t)st * 2 * kMat, wn = ws + kMat;
                    const uint32_t idesc = f ? IDESC_F : IDESC_B;
                    auto adesc = [&](uint32_t base, int kk) {
                        return smem_desc_sw128(base + (kk >> 2) * kTileA + (kk & 3) * 32, 16, 1024);
                    };
                    // forward: rows o of W, K-major; input gradient: columns of W, blocks of
                    // 64 columns D * 128 bytes apart, 16 rows (o) a step
                    auto bdesc = [&](uint32_t base, int kk) {
                        return f ? smem_desc_sw128(base + (kk >> 2) * (D * 128) + (kk & 3) * 32, 16,
                                                   1024)
                                 : smem_desc_sw128(base + kk * 2048, D * 128, 1024);
                    };
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        mma_bf16_f32(tmem_base, adesc(a, kk), bdesc(ws, kk), idesc, kk != 0);
                    if (all) {
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk)
                            mma_bf16_f32(tmem_base, adesc(a2, kk), bdesc(wn, kk), idesc, 1);
                    } else {
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk)
                            mma_bf16_f32_masked(tmem_base, adesc(a2, kk), bdesc(wn, kk), idesc, m);
                    }
                    mma_commit(&bars->wempty[st]);
                    mma_commit(&bars->accfull);
                    bulk_wait_read<0>();
                    mbar_arrive(&bars->astored);
                }
            if (it > 0) {
                // the MMAs have completed before TMEM can be freed
                mma_commit(&bars->drain);
                mbar_wait_drain(&bars->drain, 0, tmo);
            }
            bulk_wait<0>();
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int half = (warp - 2) >> 2, row = (warp & 3) * 32 + lane;
        const int col0 = half * HC;
        const int pos = row & (L.n - 1), smp = row - pos;
        const bool relu = (L.flags & 4u) != 0, resid = (L.flags & 2u) != 0;
        // 16-byte piece m of this thread's columns of row r
        auto piece = [&](uint8_t* base, int r, int m) {
            const int c = col0 / 8 + m;   // piece of the whole row
            return reinterpret_cast<uint4*>(base + (c >> 3) * kTileA + r * 128 +
                                            (((c & 7) ^ (r & 7)) << 4));
        };
        uint32_t res[NW];     // this thread's input (backward: output gradient), bf16 pairs
        uint32_t it = 0;
        bool ok = true;
        // the next step's operands: w into A, and into the row of A2 that takes this row
        auto place = [&](const uint32_t (&w)[NW], int to) {
#pragma unroll
            for (int m = 0; m < NW / 4; ++m) {
                const uint4 q = make_uint4(w[4 * m], w[4 * m + 1], w[4 * m + 2], w[4 * m + 3]);
                *piece(A, row, m) = q;
                if (to >= 0) *piece(A2, smp + to, m) = q;
            }
            fence_proxy_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->aready);
        };
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            const bool r = ok && mbar_wait(bar, parity, abort, tmo);
            ok = __all_sync(0xffffffffu, r) != 0;
        };
        // the row that takes this one at step t
        auto taker = [&](int t) {
            const int s = L.link[step_layer(t)];
            if (step_fwd(t)) return link_reader(pos, s, L.n, L.flags);
            return link_receives(pos, s, L.flags) ? link_partner(pos, s) : -1;
        };
        for (int b = blockIdx.x; b < blocks && ok; b += gridDim.x) {
            const long long tok = (long long)b * kTok + row;
            const bool valid = tok < L.tokens;
            const size_t at = (size_t)tok * D + col0;
            auto load_row = [&](const __nv_bfloat16* p, uint32_t (&w)[NW]) {
#pragma unroll
                for (int m = 0; m < NW / 4; ++m) {
                    uint4 q = make_uint4(0, 0, 0, 0);
                    if (valid) q = reinterpret_cast<const uint4*>(p + at)[m];
                    w[4 * m] = q.x;
                    w[4 * m + 1] = q.y;
                    w[4 * m + 2] = q.z;
                    w[4 * m + 3] = q.w;
                }
            };
            auto store_row = [&](__nv_bfloat16* p, const uint32_t (&w)[NW]) {
                if (valid) {
#pragma unroll
                    for (int m = 0; m < NW / 4; ++m)
                        reinterpret_cast<uint4*>(p + at)[m] =
                            make_uint4(w[4 * m], w[4 * m + 1], w[4 * m + 2], w[4 * m + 3]);
                }
            };
            auto mask_at = [&](int l) {
                return L.masks + ((size_t)l * L.tokens + tok) * WPR + half * NM;
            };
            // w as the next step's residual; without one a zero that leaves every v alone: -0
            // (v + -0 is v), under the ReLU +0 (which turns z * 0 = -0 into +0)
            auto keep_res = [&](const uint32_t (&w)[NW], uint32_t none) {
#pragma unroll
                for (int q = 0; q < NW; ++q) res[q] = resid ? w[q] : none;
            };
            const uint32_t none_f = relu ? 0u : 0x80008000u, none_b = 0x80008000u;
            // dz = g under the ReLU mask words mw
            auto masked = [&](uint32_t (&w)[NW], const uint32_t (&mw)[NM]) {
#pragma unroll
                for (int h = 0; h < NM; ++h) {
                    const PairMasks keep(mw[h]);
#pragma unroll
                    for (int q = 0; q < 16; ++q) w[h * 16 + q] &= keep(q);
                }
            };
            // the first step's operands
            {
                uint32_t w[NW];
                load_row(L.fwd ? L.x : L.dy, w);
                keep_res(w, L.fwd ? none_f : none_b);
                if (!L.fwd && relu) {
                    uint32_t mw[NM];
#pragma unroll
                    for (int h = 0; h < NM; ++h) mw[h] = valid ? mask_at(nL - 1)[h] : 0u;
                    masked(w, mw);
                }
                place(w, taker(0));
            }
            for (int t = 0; t < steps; ++t, ++it) {
                const int l = step_layer(t);
                const bool f = step_fwd(t), last = t + 1 == steps;
                const int to = last ? -1 : taker(t + 1);
                // loaded while the MMAs run: this row's mask words of the layer below, or
                // (the last forward layer of a fused launch) its output gradient
                uint32_t mw[NM], g[NW];
                if (!f && l > 0 && relu) {
#pragma unroll
                    for (int h = 0; h < NM; ++h) mw[h] = valid ? mask_at(l - 1)[h] : 0u;
                }
                const bool turn = f && l == nL - 1 && L.bwd;
                if (turn) load_row(L.dy, g);
                wait(&bars->wseen, it & 1);
                wait(&bars->accfull, it & 1);
                if (!ok) break;
                tc_fence_after();
                uint32_t out[NW];
                // z + bias, ReLU (fwd), + residual, bf16: compiled per direction and
                // activation, with a zero in res where there is no residual
                auto math = [&](auto fwd_tag, auto relu_tag) {
                    constexpr bool FWD = decltype(fwd_tag)::value, RELU = decltype(relu_tag)::value;
                    const float* bias = biases + (it % kBiasSlots) * D + col0;
#pragma unroll
                    for (int h = 0; h < NM; ++h) {
                        uint32_t raw[32];
                        tmem_ld_32x32b_x32(tmem_base + ((uint32_t)((warp & 3) * 32) << 16) +
                                               (uint32_t)(col0 + h * 32),
                                           raw);
                        tmem_ld_wait_regs(raw);
                        // the arithmetic of the stacked launches' epilogue, on the FP32
                        // pipe: b = [z > 0] as 1.0 / 0.0 (z * 2^200 saturated), y = fma(z,
                        // b, res), and the mask word as two 16-bit sums of b_c 2^c on top of
                        // 2^23 (compares and bit ors took 350 cycles more a layer)
                        uint64_t lo = f32x2_pack(0x1p23f, 0.f), hi = lo;
#pragma unroll
                        for (int q4 = 0; q4 < 8; ++q4) {
                            float4 bb = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (FWD) bb = *reinterpret_cast<const float4*>(bias + h * 32 + 4 * q4);
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                const int q = 2 * q4 + i;
                                uint64_t v = f32x2_pack(__uint_as_float(raw[2 * q]),
                                                        __uint_as_float(raw[2 * q + 1]));
                                if (FWD)
                                    v = f32x2_add(v, i ? f32x2_pack(bb.z, bb.w)
                                                       : f32x2_pack(bb.x, bb.y));
                                const uint64_t r = bf16x2_to_f32x2(res[h * 16 + q]);
                                if (RELU) {
                                    const float2 t2 = f32x2_unpack(f32x2_mul(v, kF32x2Pow100));
                                    const uint64_t b2 = f32x2_pack(mul_sat_f32(t2.x, 0x1p100f),
                                                                   mul_sat_f32(t2.y, 0x1p100f));
                                    const uint64_t w2 =
                                        f32x2_pack((float)(1u << ((2 * q) & 15)),
                                                   (float)(1u << ((2 * q + 1) & 15)));
                                    if (q < 8)
                                        lo = f32x2_fma(b2, w2, lo);
                                    else
                                        hi = f32x2_fma(b2, w2, hi);
                                    v = f32x2_fma(v, b2, r);
                                } else {
                                    v = f32x2_add(v, r);
                                }
                                const float2 t = f32x2_unpack(v);
                                out[h * 16 + q] = pack_bf16x2(t.x, t.y);
                            }
                        }
                        uint32_t bits = 0;
                        if (RELU) {
                            const float2 l2 = f32x2_unpack(lo), h2 = f32x2_unpack(hi);
                            bits = __byte_perm(__float_as_uint(l2.x + l2.y),
                                               __float_as_uint(h2.x + h2.y), 0x5410);
                        }
                        if (RELU) {
                            if (L.masks && valid) mask_at(l)[h] = bits;
                            mw[h] = bits;
                        }
                    }
                };
                if (!f)
                    math(std::false_type{}, std::false_type{});
                else if (relu)
                    math(std::true_type{}, std::true_type{});
                else
                    math(std::true_type{}, std::false_type{});
                wait(&bars->astored, it & 1);
                if (!ok) break;
                if (f && l == nL - 1) {
                    store_row(L.y, out);
                    if (turn) {
                        // the turn: g = dy, dz = dy under the mask just made
#pragma unroll
                        for (int q = 0; q < NW; ++q) out[q] = g[q];
                        keep_res(g, none_b);
                        if (relu) masked(out, mw);
                        place(out, to);
                    }
                    continue;
                }
                if (!f && l == 0) {
                    store_row(L.dx, out);
                    continue;
                }
                keep_res(out, f ? none_f : none_b);
                if (!f && relu) masked(out, mw);
                place(out, to);
            }
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, D);
    }
}

template <int D>
cudaError_t launch_small_t(const SmallLaunch& L, int sms, cudaStream_t st) {
    constexpr size_t smem = small_smem<D>();
    static_assert(smem <= 232448, "shared memory budget");
    auto kern = hcw_small_kernel<D>;
    // the shared-memory opt-in is a per-device function attribute: set it once per device
    static std::atomic<uint64_t> configured[4] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = 1ull << (dev & 63);
    std::atomic<uint64_t>& word = configured[(dev >> 6) & 3];
    if (dev >= 256 || !(word.load(std::memory_order_acquire) & bit)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (dev < 256) word.fetch_or(bit, std::memory_order_acq_rel);
    }
    const int blocks = (L.tokens + kTok - 1) / kTok;
    const int ctas = sms * (D == 64 ? 2 : 1);   // (two of the narrow kernel fit an SM)
    return launch_pdl(kern, dim3(blocks < ctas ? blocks : ctas), dim3(kSmallThreads), smem, st, L);
}

}  // namespace

bool small_supported(int d, int n, long long tokens, int L) {
    return (d == 64 || d == 128) && n <= kTok && tokens > 0 && tokens < (1ll << 30) && L >= 1 &&
           L <= kMaxSmallLayers;
}

cudaError_t launch_small(const SmallLaunch& L, int d, int sms, cudaStream_t st) {
    if (!small_supported(d, L.n, L.tokens, L.n_layers) || (!L.fwd && !L.bwd))
        return cudaErrorInvalidValue;
    return d == 128 ? launch_small_t<128>(L, sms, st) : launch_small_t<64>(L, sms, st);
}

cudaError_t small_error_word_read_clear(int* word) {
    const int zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(word, g_error_word, sizeof(int));
    if (e == cudaSuccess && *word) e = cudaMemcpyToSymbol(g_error_word, &zero, sizeof(int));
    return e;
}

}  // namespace hcw
