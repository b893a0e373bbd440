// hcw_decode.cu -- one-token decode of a causal stack (Sec. 6, "Deployability":
// the decode path runs one token at a time, and a sparse layer needs only the
// last k inputs it links to, so its cache does not grow).
//
// B sequences advance together by one position t.  Layer l with link distance
// k_l (2^s for the hypercube link along dimension s, k for a shift layer) keeps
// a ring of k_l + 1 slots; the input of position p sits in slot p mod (k_l + 1).
// Position t receives at layer l when bit s of t is set (hypercube link) or
// t >= k (shift); its partner is position t - k_l, in slot (t + 1) mod
// (k_l + 1), which is never the slot t's own input goes to.  So layer l's
// epilogue writes its output straight into layer l + 1's ring, and nothing is
// read and overwritten within one step.
//
// The sequences never interact inside a layer (Eq. (1) mixes position t with
// one earlier position of the same sequence), so one position of the whole
// stack splits into independent blocks of 16 rows.  A thread-block cluster of
// C CTAs (C <= 16) runs one row block through all L layers; CTA q of the
// cluster owns output columns [q OC, (q + 1) OC), OC = d / C, and contracts the
// partner part first (it does not depend on the previous layer), then the self
// part once the layer input is complete: [16 x d] x [d x OC] twice, fp32
// accumulation.  The epilogue (bias, ReLU, residual, bf16) writes the CTA's 16 x
// OC slice to the next layer's ring slot in global memory and sends it into every
// cluster CTA's input buffer of the next layer (distributed shared memory: bulk
// copies, or in decode_tc_kernel asynchronous remote stores) with its bytes
// counted on that CTA's "input ready" mbarrier: the layer input is complete when
// every slice has landed, with no fence or barrier between the CTAs.  No layer boundary
// goes through global memory or a grid-wide barrier.
//
// Two contractions (hcw_set_decode_kernel):
//   - decode_mma_kernel (the default): eight warps share the K range with the
//     warp-level bf16 MMA (m16n8k16), weights and partner rows straight from
//     global memory into registers;
//   - decode_tc_kernel: one thread issues tcgen05.mma over weights that a
//     producer warp streams into a ring of shared-memory stages by TMA (3-D boxes
//     of 64 features, rows, K tiles, 128-byte swizzle), running ahead of the
//     layers; the partner rows come the same way.  A tile holds 16 rows, below
//     the 64-row minimum, so the MMA runs with M = 64 on the 16 rows (its other
//     48 rows read whatever follows in shared memory; only D's rows 0..15, TMEM
//     lanes 0..15, are used) and N = OC.  Warp 7 issues, warp 0 drains D into the
//     row sums, and a layer's partner part is contracted into the other of two
//     accumulators while the layer before is drained.  Issuing a layer's 32
//     partner-part MMAs (N = OC = 32 at d = 512, K = 16) only after its input
//     arrived costs 0.75 us a layer, so one thread's tcgen05.mma run about 45
//     cycles each in sequence; the commit, the TMEM drain and a proxy fence (the
//     remote stores are generic writes that the MMA reads through the async
//     proxy) add to the chain.  So the tensor-core version is the slower of the
//     two here.
#include <atomic>

#include "hcw_internal.h"
#include "hcw_ptx.cuh"

namespace hcw {

namespace {

constexpr int kRows = 16;          // rows of a row block
constexpr int kMmaWarps = 8;       // warps 0..7: MMA + epilogue (decode_tc_kernel: warp 7
                                   // issues, warps 0..6 run the epilogue; warp 8: producer)
constexpr int kThreads = (kMmaWarps + 1) * 32;
// decode_tc_kernel: accumulators a layer's K tiles alternate over, for each layer parity (64
// columns each); four in turn measured no faster than one
constexpr int kNAcc = 1;
constexpr uint32_t kTmemCols = 2 * kNAcc * 64 < 32 ? 32 : 2 * kNAcc * 64;
constexpr int kMaxStages = 8;

struct DecodeArgs {
    CUtensorMap mWs, mWn;   // [L d][d] bf16, box (64 features, OC rows, kc / 64 tiles)
    CUtensorMap mCache;     // the rings as [rows][d] bf16, box (64, 16, d / 64)
    CUtensorMap mX;         // x_t [B][d] bf16, box (64, 16, d / 64)
    int prow[kMaxDecodeLayers];                 // cache row of the partner slot, or -1
    __nv_bfloat16* out[kMaxDecodeLayers];       // [B][d] next layer's ring slot, or y_t
    const float* bias;     // [L][d] or null
    __nv_bfloat16* ring0;  // layer 0's ring slot of position t
    DecodeGeo g;
    int L, B;
    unsigned flags;
    unsigned long long timeout_ns;
};

// barrier slots of decode_tc_kernel
enum : int {
    B_FULL = 0,                       // [kMaxStages] stage filled (tx bytes)
    B_EMPTY = kMaxStages,             // [kMaxStages] stage consumed (a commit)
    B_XS_READY = 2 * kMaxStages,      // [2] layer input complete (tx bytes from every cluster CTA)
    B_X0 = 2 * kMaxStages + 2,        // x_t rows loaded
    B_XP_FULL = 2 * kMaxStages + 3,   // [2] partner rows loaded
    B_XP_FREE = 2 * kMaxStages + 5,   // [2] partner buffer consumed (a commit)
    B_DFULL = 2 * kMaxStages + 7,     // [2] a layer's accumulator complete (commit)
    B_TFREE = 2 * kMaxStages + 9,     // [2] a layer's accumulator drained by warp 0
    B_DRAIN = 2 * kMaxStages + 11,    // the issuer's last MMAs completed
    B_COUNT = 2 * kMaxStages + 12
};

// Shared memory of decode_tc_kernel (1024-byte aligned): Xs[2] (layer inputs) and Xp[2] (partner
// rows), each d / 64 tiles of 16 rows x 128 bytes; stages[S], each kc / 64
// tiles of OC rows x 128 bytes; all bf16 in the 128-byte swizzle (16-byte
// chunk c of row r at chunk c ^ (r & 7)).  Then red[2][16][OC] fp32 (the
// partial sums of alternate layers), the mbarriers and the abort word.
struct Smem {
    uint8_t* base;
    const DecodeGeo& g;
    __device__ Smem(uint8_t* b, const DecodeGeo& geo) : base(b), g(geo) {}
    __device__ uint8_t* xs(int buf) const { return base + (size_t)buf * kRows * g.d * 2; }
    __device__ uint8_t* xpart(int buf) const { return base + (size_t)(2 + buf) * kRows * g.d * 2; }
    __device__ uint8_t* stage(int s) const {
        return base + (size_t)4 * kRows * g.d * 2 + (size_t)s * g.oc * g.kc * 2;
    }
    __device__ float* red(int buf) const {
        return reinterpret_cast<float*>(stage(g.stages)) + buf * kRows * g.oc;
    }
    __device__ uint64_t* bars() const {
        return reinterpret_cast<uint64_t*>(red(2));
    }
    __device__ int* abort_word() const { return reinterpret_cast<int*>(bars() + B_COUNT); }
    __device__ uint32_t* tmem_slot() const {
        return reinterpret_cast<uint32_t*>(abort_word() + 1);
    }
};

// byte offset of the 16-byte chunk holding features [8 c, 8 c + 8) of row r
// in a swizzled buffer of 64-feature tiles, tile_bytes apart
__device__ __forceinline__ uint32_t sw_off(int r, int col, uint32_t tile_bytes) {
    const int ch = (col >> 3) & 7;
    return (uint32_t)(col >> 6) * tile_bytes + r * 128 + ((ch ^ (r & 7)) << 4);
}

// D (16 x 8, fp32) += A (16 x 16 bf16, row-major) * B (16 x 8 bf16, column-major)
__device__ __forceinline__ void mma_16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, "
        "{%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// 16 bytes into the shared memory of a cluster CTA; the bytes complete on that
// CTA's mbarrier (both given by shared::cluster addresses in the same CTA)
__device__ __forceinline__ void st_async_v4(uint32_t addr, uint4 v, uint32_t bar) {
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, "
        "[%5];" ::"r"(addr),
        "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
        : "memory");
}

// K chunk c of a part: [c kc, min(d, (c + 1) kc))
__device__ __forceinline__ int chunk_len(const DecodeGeo& g, int c) {
    const int k0 = c * g.kc;
    return g.d - k0 < g.kc ? g.d - k0 : g.kc;
}

// The end of a layer for one epilogue thread (8 columns of one row, v =
// the row sums plus bias): ReLU, residual, bf16; the result goes into every
// cluster CTA's next-layer input (remote stores counted on its input barrier)
// and, for a valid row, to the layer's output in global memory.
__device__ __forceinline__ void decode_epilogue(const DecodeArgs& a, const Smem& sm, float (&v)[8],
                                                uint4 xin, int l, int xb, int q, int row0,
                                                int vr, int pr, int pc8, uint32_t poff) {
    const DecodeGeo& g = a.g;
    const int d = g.d, col0 = q * g.oc;
    if (a.flags & 4u) {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = v[e] > 0.f ? v[e] : 0.f;
    }
    if (a.flags & 2u) {
        const uint32_t w[4] = {xin.x, xin.y, xin.z, xin.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 f = unpack_bf16x2(w[e]);
            v[2 * e] += f.x;
            v[2 * e + 1] += f.y;
        }
    }
    uint4 pk;
    pk.x = pack_bf16x2(v[0], v[1]);
    pk.y = pack_bf16x2(v[2], v[3]);
    pk.z = pack_bf16x2(v[4], v[5]);
    pk.w = pack_bf16x2(v[6], v[7]);
    if (l + 1 < a.L) {
        const uint8_t* dst = sm.xs(xb ^ 1) + poff;
        const uint64_t* rb = &sm.bars()[B_XS_READY + (xb ^ 1)];
        for (int cr = 0; cr < g.csize; ++cr)
            st_async_v4(mapa_shared(dst, cr), pk, mapa_shared(rb, cr));
    }
    if (pr < vr) {
        if (l == 0)   // position t's layer-0 input into layer 0's ring
            *reinterpret_cast<uint4*>(a.ring0 + (size_t)(row0 + pr) * d + col0 + pc8) = xin;
        *reinterpret_cast<uint4*>(a.out[l] + (size_t)(row0 + pr) * d + col0 + pc8) = pk;
    }
}

// The MMA and epilogue warps of decode_tc_kernel: warp 7 issues the
// tcgen05 MMAs, warp 0 drains each layer's accumulator into the row sums, and
// warps 0..6 run the epilogue (bias, ReLU, residual, bf16, pushes).
__device__ __forceinline__ void decode_tc_body(const DecodeArgs& a, const Smem& sm, int warp,
                                            int lane, int q, int row0, int vr) {
    const DecodeGeo& g = a.g;
    uint64_t* bars = sm.bars();
    const int d = g.d, oc = g.oc, col0 = q * oc, nch = g.nchunks;
    const uint32_t xtile = kRows * 128, wtile = (uint32_t)oc * 128;
    volatile int* abort = sm.abort_word();
    const uint32_t IDESC = idesc_bf16_f32(64, oc, 0, 0);
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(sm.tmem_slot());
    const int packs = kRows * oc / 8;   // epilogue: a thread per 8 columns of a row
    const int pr = threadIdx.x / (oc / 8), pc8 = (threadIdx.x % (oc / 8)) * 8;
    const uint32_t poff = sw_off(pr, col0 + pc8, xtile);
    bool ok = true;
    if (warp == kMmaWarps - 1) {
        if (lane == 0) {
            // ---------------------------------------------- MMA issuer
            uint32_t it = 0;
            int xp_uses[2] = {0, 0};
            for (int l = 0; l < a.L && ok; ++l) {
                const int xb = l & 1, ab = l & 1;
                const bool recv = a.prow[l] >= 0;
                // the accumulator of this parity has been drained (layer l - 2)
                if (l >= 2)
                    ok = mbar_wait(&bars[B_TFREE + ab], ((l - 2) >> 1) & 1, abort, a.timeout_ns);
                if (!ok) break;
                tc_fence_after();
                // K tile j of the layer goes to accumulator j mod kNAcc: consecutive
                // MMAs do not wait on each other's result
                int tix = 0;
                for (int part = recv ? 1 : 0; part >= 0 && ok; --part) {
                    uint32_t X;
                    if (part) {
                        ok = mbar_wait(&bars[B_XP_FULL + xb], xp_uses[xb]++ & 1, abort,
                                       a.timeout_ns);
                        X = smem_u32(sm.xpart(xb));
                    } else {
                        ok = l == 0 ? mbar_wait(&bars[B_X0], 0, abort, a.timeout_ns)
                                    : mbar_wait_cluster(&bars[B_XS_READY + xb], ((l - 1) >> 1) & 1,
                                                        abort, a.timeout_ns);
                        X = smem_u32(sm.xs(xb));
                        // the input came by remote stores (generic proxy); the MMAs
                        // read it through the async proxy
                        if (ok) fence_proxy_async_smem();
                    }
                    if (!ok) break;
                    tc_fence_after();
                    for (int c = 0; c < nch && ok; ++c, ++it) {
                        const int s = (int)(it % (uint32_t)g.stages);
                        ok = mbar_wait(&bars[B_FULL + s], (it / g.stages) & 1, abort, a.timeout_ns);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t W = smem_u32(sm.stage(s));
                        const int tiles = chunk_len(g, c) / 64, t0 = c * g.kc / 64;
                        for (int t = 0; t < tiles; ++t, ++tix) {
                            const uint32_t d_tmem =
                                tmem_base + (uint32_t)((ab * kNAcc + tix % kNAcc) * 64);
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk) {
                                const uint64_t ad = smem_desc_sw128(
                                    X + (uint32_t)(t0 + t) * xtile + kk * 32, 16, 1024);
                                const uint64_t bd =
                                    smem_desc_sw128(W + (uint32_t)t * wtile + kk * 32, 16, 1024);
                                mma_bf16_f32(d_tmem, ad, bd, IDESC,
                                             (tix < kNAcc && kk == 0) ? 0u : 1u);
                            }
                        }
                        mma_commit(&bars[B_EMPTY + s]);
                    }
                    if (ok && part) mma_commit(&bars[B_XP_FREE + xb]);
                }
                if (ok) mma_commit(&bars[B_DFULL + ab]);
            }
            if (!ok) *abort = 1;
            // the MMAs have completed before the CTA frees TMEM at the end
            if (it > 0) {
                mma_commit(&bars[B_DRAIN]);
                mbar_wait_drain(&bars[B_DRAIN], 0, a.timeout_ns);
            }
        }
        __syncwarp();
        return;
    }
    for (int l = 0; l < a.L; ++l) {
        const int xb = l & 1, ab = l & 1;
        // the next layer's input arrives as 16 x d x 2 bytes from the cluster
        if (threadIdx.x == 0 && l + 1 < a.L)
            mbar_arrive_expect_tx(&bars[B_XS_READY + (xb ^ 1)], (uint32_t)kRows * d * 2);
        // this thread's bias values, loaded while the layer runs
        float4 bv0 = make_float4(0.f, 0.f, 0.f, 0.f), bv1 = bv0;
        if (a.bias && (int)threadIdx.x < packs) {
            const float4* bl = reinterpret_cast<const float4*>(a.bias + (size_t)l * d + col0 + pc8);
            bv0 = __ldg(bl);
            bv1 = __ldg(bl + 1);
        }
        float* red = sm.red(xb);
        if (warp == 0) {
            // D rows 0..15 (TMEM lanes 0..15) into this layer's row sums
            bool r = ok && mbar_wait(&bars[B_DFULL + ab], (l >> 1) & 1, abort, a.timeout_ns);
            ok = __all_sync(0xffffffffu, r);
            if (ok) {
                tc_fence_after();
                // the accumulators the layer's K tiles went to, added in order
                const int ntiles = (a.prow[l] >= 0 ? 2 : 1) * (d / 64);
                const int nacc = ntiles < kNAcc ? ntiles : kNAcc;
                for (int c0 = 0; c0 < oc; c0 += 32) {
                    float sum[32];
#pragma unroll
                    for (int e = 0; e < 32; ++e) sum[e] = 0.f;
                    for (int ac = 0; ac < nacc; ++ac) {
                        uint32_t raw[32];
                        tmem_ld_32x32b_x32(
                            tmem_base + (uint32_t)((ab * kNAcc + ac) * 64 + c0), raw);
                        tmem_ld_wait_regs(raw);
#pragma unroll
                        for (int e = 0; e < 32; ++e) sum[e] += __uint_as_float(raw[e]);
                    }
                    const int nc = oc - c0 < 32 ? oc - c0 : 32;
                    if (lane < kRows) {
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (e < nc) red[lane * oc + c0 + e] = sum[e];
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[B_TFREE + ab]);
            }
        }
        // the layer input (the residual) is complete here: every thread takes
        // the barrier's acquire before it reads it
        {
            bool r = ok && (l == 0 ? mbar_wait(&bars[B_X0], 0, abort, a.timeout_ns)
                                   : mbar_wait_cluster(&bars[B_XS_READY + xb], ((l - 1) >> 1) & 1,
                                                       abort, a.timeout_ns));
            ok = __all_sync(0xffffffffu, r);
        }
        // every thread past this point has finished the previous layer's
        // epilogue, so the other row-sum buffer is free again
        named_bar_sync(1, (kMmaWarps - 1) * 32);
        if (ok && (int)threadIdx.x < packs) {
            const uint4 xin = *reinterpret_cast<const uint4*>(sm.xs(xb) + poff);
            const float* rr = red + pr * oc + pc8;
            const float bvals[8] = {bv0.x, bv0.y, bv0.z, bv0.w, bv1.x, bv1.y, bv1.z, bv1.w};
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = rr[e] + bvals[e];
            decode_epilogue(a, sm, v, xin, l, xb, q, row0, vr, pr, pc8, poff);
        }
    }
}

__global__ void __launch_bounds__(kThreads, 1)
    decode_tc_kernel(const __grid_constant__ DecodeArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const DecodeGeo& g = a.g;
    const Smem sm(base, g);
    uint64_t* bars = sm.bars();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = (int)cluster_ctarank();
    const int row0 = (int)(blockIdx.x / g.csize) * kRows;   // this cluster's row block
    const int vr = a.B - row0 < kRows ? a.B - row0 : kRows;   // valid rows
    const int d = g.d, oc = g.oc, col0 = q * oc;
    const int nch = g.nchunks;
    volatile int* abort = sm.abort_word();

    if (threadIdx.x == 0) {
        *abort = 0;
        for (int s = 0; s < g.stages; ++s) {
            mbar_init(&bars[B_FULL + s], 1);
            mbar_init(&bars[B_EMPTY + s], 1);
        }
        mbar_init(&bars[B_XS_READY + 0], 1);
        mbar_init(&bars[B_XS_READY + 1], 1);
        mbar_init(&bars[B_X0], 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars[B_XP_FULL + b], 1);
            mbar_init(&bars[B_XP_FREE + b], 1);
            mbar_init(&bars[B_DFULL + b], 1);
            mbar_init(&bars[B_TFREE + b], 1);
        }
        mbar_init(&bars[B_DRAIN], 1);
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(sm.tmem_slot(), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();   // barriers initialised in every CTA of the cluster
    tc_fence_after();

    if (warp == kMmaWarps) {
        // ---------------------------------------------------------- producer
        if (lane == 0) {
            tma_prefetch_desc(&a.mWs);
            tma_prefetch_desc(&a.mWn);
            tma_prefetch_desc(&a.mCache);
            uint32_t it = 0;            // weight chunks issued
            int xp_fills[2] = {0, 0};   // partner-buffer fills issued
            bool ok = true;
            mbar_arrive_expect_tx(&bars[B_X0], (uint32_t)kRows * d * 2);
            tma_load_3d(sm.xs(0), &a.mX, &bars[B_X0], 0, row0, 0);
            for (int l = 0; l < a.L && ok; ++l) {
                const int prow = a.prow[l];
                if (prow >= 0) {
                    const int b = l & 1, u = xp_fills[b];
                    if (u > 0)
                        ok = mbar_wait(&bars[B_XP_FREE + b], (u - 1) & 1, abort, a.timeout_ns);
                    if (!ok || *abort) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&bars[B_XP_FULL + b], (uint32_t)kRows * d * 2);
                    tma_load_3d(sm.xpart(b), &a.mCache, &bars[B_XP_FULL + b], 0, prow + row0, 0);
                    xp_fills[b] = u + 1;
                }
                // weight chunks: the partner part (if any), then the self part
                for (int part = prow >= 0 ? 1 : 0; part >= 0 && ok; --part) {
                    const CUtensorMap* mW = part ? &a.mWn : &a.mWs;
                    for (int c = 0; c < nch; ++c) {
                        const int s = (int)(it % (uint32_t)g.stages);
                        const int klen = chunk_len(g, c);
                        if (it >= (uint32_t)g.stages)
                            ok = mbar_wait(&bars[B_EMPTY + s], ((it / g.stages) - 1) & 1, abort,
                                           a.timeout_ns);
                        if (!ok || *abort) {
                            ok = false;
                            break;
                        }
                        // a ragged last chunk is the box's first klen / 64 tiles; the
                        // rest fall past d and arrive as zeros (counted in full)
                        mbar_arrive_expect_tx(&bars[B_FULL + s], (uint32_t)oc * g.kc * 2);
                        tma_load_3d(sm.stage(s), mW, &bars[B_FULL + s], 0, l * d + col0,
                                    c * g.kc / 64);
                        ++it;
                    }
                }
            }
            // after an abort: let every copy this CTA issued land before it exits
            if (!ok) {
                mbar_wait_drain(&bars[B_X0], 0, a.timeout_ns);
                for (uint32_t j = it > (uint32_t)g.stages ? it - g.stages : 0; j < it; ++j)
                    mbar_wait_drain(&bars[B_FULL + j % g.stages], (j / g.stages) & 1,
                                    a.timeout_ns);
                for (int b = 0; b < 2; ++b)
                    if (xp_fills[b] > 0)
                        mbar_wait_drain(&bars[B_XP_FULL + b], (xp_fills[b] - 1) & 1,
                                        a.timeout_ns);
            }
        }
        __syncwarp();
    } else {
        decode_tc_body(a, sm, warp, lane, q, row0, vr);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();   // no CTA leaves while a peer may still write its shared memory
    if (warp == 0) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(*sm.tmem_slot(), kTmemCols);
    }
}

// ------------------------------------------------------------ warp-level MMA
struct DecodeMmaArgs {
    const __nv_bfloat16 *Ws, *Wn;   // [L d][d]
    const __nv_bfloat16* x;         // x_t [B][d]
    const __nv_bfloat16* cache;     // the rings as [rows][d]
    const float* bias;              // [L][d] or null
    __nv_bfloat16* ring0;           // layer 0's ring slot of position t
    int prow[kMaxDecodeLayers];             // cache row of the partner slot, or -1
    __nv_bfloat16* out[kMaxDecodeLayers];   // [B][d] next layer's ring slot, or y_t
    int d, csize, L, B;
    unsigned flags;
    unsigned long long timeout_ns;
};

// A layer-input buffer holds the cluster's slices one after the other, each 16 rows of
// OC features, as a CTA sends its slice: one copy a peer.  Bytes of a row, of a slice as
// copied, and from slice to slice; the odd 16 bytes put the 16-byte reads of a
// fragment's rows on different banks (for OC = 16 on two a bank).
__host__ __device__ constexpr int mma_row_bytes(int oc) { return 2 * oc + (oc == 64 ? 16 : 0); }
__host__ __device__ constexpr int mma_slice_bytes(int oc) { return kRows * mma_row_bytes(oc); }
__host__ __device__ constexpr int mma_slice_step(int oc) {
    return mma_slice_bytes(oc) + (oc == 64 ? 0 : 16);
}
// floats per row of a warp's block of sums (OC + 8: the fragments' rows on different banks)
__host__ __device__ constexpr int mma_sum_row(int oc) { return oc + 8; }

// whether the partner parts have warps of their own (kPWarps), and the threads of a CTA
constexpr int kPWarps = 4;
__host__ __device__ constexpr bool mma_split(int oc) { return oc < 64; }
__host__ __device__ constexpr int mma_threads(int oc) {
    return (kMmaWarps + (mma_split(oc) ? kPWarps : 0)) * 32;
}
constexpr int kMmaBars = 2 + 4 * kPWarps;

// bytes from this CTA's shared memory into a cluster CTA's; they complete on that CTA's
// mbarrier (destination and barrier as shared::cluster addresses)
__device__ __forceinline__ void copy_to_peer(uint32_t dst, uint32_t src, uint32_t bytes,
                                             uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, "
        "[%3];" ::"r"(dst),
        "r"(src), "r"(bytes), "r"(bar)
        : "memory");
}

// takes bytes off a barrier's pending transactions, as if a copy of that size had landed
__device__ __forceinline__ void mbar_complete_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
constexpr uint64_t kDrainNs = 1000000000ull;   // 1 s

// 16 features of a row
struct Feat16 {
    uint32_t r[8];
};
// one 32-byte load of a 32-byte aligned piece (W32), else two of 16 bytes.  (Not the
// read-only path: the kernel before this one, which this one's start overlaps, may
// have written the ring slot.)
template <bool W32>
__device__ __forceinline__ Feat16 ldg_stream(const void* p) {
    Feat16 v;
    if constexpr (W32) {
        asm volatile("ld.global.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(v.r[0]), "=r"(v.r[1]), "=r"(v.r[2]), "=r"(v.r[3]), "=r"(v.r[4]),
                       "=r"(v.r[5]), "=r"(v.r[6]), "=r"(v.r[7])
                     : "l"(p));
    } else {
#pragma unroll
        for (int h = 0; h < 2; ++h)
            asm volatile("ld.global.L1::no_allocate.v4.b32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(v.r[4 * h]), "=r"(v.r[4 * h + 1]), "=r"(v.r[4 * h + 2]),
                           "=r"(v.r[4 * h + 3])
                         : "l"(static_cast<const uint8_t*>(p) + 16 * h));
    }
    return v;
}
__device__ __forceinline__ Feat16 lds16(const uint8_t* p) {
    const uint4 a = *reinterpret_cast<const uint4*>(p), b = *reinterpret_cast<const uint4*>(p + 16);
    return Feat16{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}

// Warp w (of eight) contracts the K groups (64 features) w GP .. w GP + GP - 1 with all OC
// columns.  Inside a group the contraction may take the features in any order, as long
// as both operands do: lane (g = lane / 4, c = lane % 4) takes features 16 c .. 16 c + 15
// of rows g and g + 8 of the input and of weight rows 8 u + g, one 32-byte load each
// (a warp's load: eight whole 128-byte lines), and those are the fragments of the
// group's four MMAs (MMA m takes the pieces' words 2 m and 2 m + 1).  So the weights and the partner rows go from global
// memory (L2) straight into the registers the MMA reads; as a group has been
// contracted, its registers are reloaded for the next part.  The sums of the eight
// warps meet in shared memory in warp order (deterministic).
//
// OC < 64 (SPLIT): warps 8 .. 11 contract the partner parts (a quarter of the K groups
// each), up to two layers ahead of warps 0 .. 7, and hand their accumulators to warps 0
// .. 3 to start the self part with.  Warps 0 .. 7 hold the self weights of two layers:
// a layer's are requested a whole layer before they are needed, between its pushes
// and the next input's arrival, where issuing loads costs the chain nothing.  At OC =
// 64 (d > 512) a part takes 128 registers a lane: eight warps contract both parts in
// turn and reload a group as it has been contracted.
//
// What bounds it: the bytes an SM takes in, and a chain per layer (input landed, self
// MMAs, sums, epilogue, slices sent and landed).  64 KB of weights and 16 KB of slices a
// layer at d = 512 are 2,000 cycles at the 39 bytes a cycle an SM gets from L2; the
// chain alone is about 1,500, of which the MMAs take 260.  So it holds no wait but the
// input's, no address arithmetic that could be set up before, no constant-cache line
// first touched there and no global load (the layer table and the biases are copied to
// shared memory first: a bias load queued behind the weights' took 800 cycles), no
// float atomics in shared memory (a compare-and-swap loop, 110 cycles each), and one
// bulk copy a peer (1,024 remote 16-byte stores waited behind the weight loads, 850).
// Microseconds a position at 64 sequences, 16 layers, d = 512, and cycles a layer:
//   weights staged in shared memory by TMA, atomics, remote stores     52    6,900
//   no atomics, whole parts staged (one wait a part)                   33    4,350
//   weights in registers, eight warps for both parts                   30    4,200
//   partner warps                                                      27    3,300
//   self weights two layers deep, biases in shared memory              25    3,200
//   slices sent as bulk copies (this)                                  23    2,600
template <int OC, int GP, bool W32>
__global__ void __launch_bounds__(mma_threads(OC), 1)
    decode_mma_kernel(const __grid_constant__ DecodeMmaArgs a) {
    constexpr bool SPLIT = mma_split(OC);
    constexpr int NB = OC / 8;                               // n8 blocks
    constexpr int RS = mma_sum_row(OC);
    constexpr int kPacks = kRows * OC / 8;                   // 8-column pieces of the slice
    constexpr int kGroups = kMmaWarps * 8;                   // groups of four threads
    constexpr int kPer = (kPacks + kGroups - 1) / kGroups;   // pieces a group
    extern __shared__ __align__(128) uint8_t smem[];
    const int d = a.d, L = a.L;
    constexpr uint32_t RB = mma_row_bytes(OC), SB = mma_slice_bytes(OC), SS = mma_slice_step(OC);
    const uint32_t xbuf = a.csize * SS;
    uint8_t* xs = smem;                                      // [2][csize] slices
    uint8_t* slice = smem + 2 * xbuf;                        // [2] this CTA's, as sent
    float* sums = reinterpret_cast<float*>(slice + 2 * SB);  // [8 warps][16][RS]
    // SPLIT: the partner warps' accumulators, [2][4 warps][NB][32 lanes]
    float4* pacc = reinterpret_cast<float4*>(sums + kMmaWarps * kRows * RS);
    uint64_t* bars = reinterpret_cast<uint64_t*>(pacc + (SPLIT ? 2 * kPWarps * NB * 32 : 0));
    uint64_t* const xs_bar = bars;                   // [2] layer input complete
    uint64_t* const pfull = bars + 2;                // [2][4] accumulators handed over
    uint64_t* const pfree = pfull + 2 * kPWarps;     // [2][4] ... and taken
    __nv_bfloat16** outp = reinterpret_cast<__nv_bfloat16**>(bars + kMmaBars);
    int* prow = reinterpret_cast<int*>(outp + kMaxDecodeLayers);
    volatile int* abort = prow + kMaxDecodeLayers;
    // after an abort somewhere in the cluster: that there was one, and for every CTA of the
    // cluster how many of its slices it did not send to this one
    volatile int* down = abort + 1;
    volatile int* unsent = abort + 4;   // [16]
    float* bias_s = const_cast<float*>(reinterpret_cast<volatile float*>(unsent + 16));   // [L][OC]
    const bool partner_warp = SPLIT && threadIdx.x >= kMmaWarps * 32;
    const int warp = (threadIdx.x >> 5) - (partner_warp ? kMmaWarps : 0);
    const int lane = threadIdx.x & 31;
    const int q = (int)cluster_ctarank();
    const int row0 = (int)(blockIdx.x / a.csize) * kRows;     // this cluster's row block
    const int vr = a.B - row0 < kRows ? a.B - row0 : kRows;   // valid rows
    const int col0 = q * OC, g = lane >> 2, c = lane & 3;

    if (threadIdx.x < L) {
        outp[threadIdx.x] = a.out[threadIdx.x];
        prow[threadIdx.x] = a.prow[threadIdx.x];
    }
    if (threadIdx.x < 16) unsent[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        *abort = 0;
        *down = 0;
        for (int i = 0; i < kMmaBars; ++i) mbar_init(&bars[i], 1);
        fence_mbar_init();
    }
    __syncthreads();
    cluster_sync_all();   // barriers initialised in every CTA of the cluster
    // nothing above touched global memory: it overlaps the end of the kernel before
    // this one (the position before, in a decode loop)
    pdl_wait();
    pdl_trigger();

    for (int i = threadIdx.x; i < L * OC; i += mma_threads(OC))
        bias_s[i] = a.bias ? a.bias[(size_t)(i / OC) * d + col0 + i % OC] : 0.f;
    // K groups of this warp: [warp gw, warp gw + gw) clipped to d / 64
    const int gw = partner_warp ? GP * kMmaWarps / kPWarps : GP;
    const int k0 = warp * gw * 64 + 16 * c;   // the lane's features of group 0
    const int ng = d / 64 - warp * gw;       // groups of this warp: min(ng, gw)
    const size_t wlane = ((size_t)(col0 + g) * d + k0) * 2, wlayer = (size_t)d * d * 2;
    const size_t ublk = (size_t)16 * d;      // bytes of 8 weight rows
    const uint8_t* const ws = reinterpret_cast<const uint8_t*>(a.Ws) + wlane;
    const uint8_t* const wn = reinterpret_cast<const uint8_t*>(a.Wn) + wlane;
    float acc[NB][4];
    auto load_group = [&](Feat16 (&w)[NB], const uint8_t* p, int i) {
        if (i < ng) {
#pragma unroll
            for (int u = 0; u < NB; ++u) w[u] = ldg_stream<W32>(p + u * ublk + i * 128);
        }
    };
    // partner rows g, g + 8 of layer l, group i
    auto load_partner = [&](Feat16 (&xp)[2], int l, int i) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = g + 8 * h;
            if (i < ng && row < vr)
                xp[h] = ldg_stream<W32>(a.cache + (size_t)(prow[l] + row0 + row) * d + k0 + i * 64);
            else
                xp[h] = Feat16{};
        }
    };
    // group i of a part: rows lo (g) and hi (g + 8) against w
    auto contract = [&](const Feat16& lo, const Feat16& hi, const Feat16 (&w)[NB], int i) {
        if (i < ng) {
#pragma unroll
            for (int m = 0; m < 8; m += 2) {
                const uint32_t af[4] = {lo.r[m], hi.r[m], lo.r[m + 1], hi.r[m + 1]};
#pragma unroll
                for (int u = 0; u < NB; ++u) mma_16816(acc[u], af, w[u].r[m], w[u].r[m + 1]);
            }
        }
    };
    auto clear = [&]() {
#pragma unroll
        for (int u = 0; u < NB; ++u)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[u][e] = 0.f;
    };
    // every lane waits (each gets the acquire); the outcome is made warp-uniform so
    // that the aligned MMAs never run divergent
    bool ok = true;
    int armed = 0, seen = 0;   // last layer whose input this thread has armed, and waited for
    auto wait = [&](uint64_t* bar, uint32_t parity, bool cluster) {
        const bool r = ok && (cluster ? mbar_wait_cluster(bar, parity, abort, a.timeout_ns)
                                      : mbar_wait(bar, parity, abort, a.timeout_ns));
        ok = __all_sync(0xffffffffu, r);
    };
    auto next_recv = [&](int l) {   // the next layer from l on that has a partner part
        while (l < L && prow[l] < 0) ++l;
        return l;
    };

    if (partner_warp) {
        constexpr int GW = GP * kMmaWarps / kPWarps;
        Feat16 w[GW][NB], xp[GW][2];   // weights and rows of the next layer with a partner part
        int l = next_recv(0);
        if (l < L) {
#pragma unroll
            for (int i = 0; i < GW; ++i) {
                load_group(w[i], wn + l * wlayer, i);
                load_partner(xp[i], l, i);
            }
        }
        __syncthreads();   // (x_t and the biases in place)
        for (uint32_t use = 0; l < L; ++use) {
            const int nl = next_recv(l + 1);
            const uint32_t slot = (use & 1) * kPWarps + warp;
            clear();
#pragma unroll
            for (int i = 0; i < GW; ++i) {
                contract(xp[i][0], xp[i][1], w[i], i);
                if (nl < L) {
                    load_group(w[i], wn + nl * wlayer, i);
                    load_partner(xp[i], nl, i);
                }
            }
            if (use >= 2) wait(&pfree[slot], ((use >> 1) - 1) & 1, false);
            float4* dst = pacc + (size_t)slot * NB * 32 + lane;
#pragma unroll
            for (int u = 0; u < NB; ++u)
                dst[u * 32] = make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
            __syncwarp();
            if (lane == 0) mbar_arrive(&pfull[slot]);
            l = nl;
        }
    } else {
        // weights of the part contracted next, and (SPLIT) of the layer after
        Feat16 w[GP][NB], w2[SPLIT ? GP : 1][NB], xp[GP][2];
        // the first part this warp contracts of layer l
        auto first_part = [&](int l) {
            return (!SPLIT && prow[l] >= 0 ? wn : ws) + l * wlayer;
        };
#pragma unroll
        for (int i = 0; i < GP; ++i) {
            if (SPLIT)
                load_group(w2[i], ws, i);
            else
                load_group(w[i], first_part(0), i);
            if (!SPLIT && prow[0] >= 0) load_partner(xp[i], 0, i);
        }
        // x_t, layer 0's input
        for (int p = threadIdx.x; p < kRows * (d / 8); p += kMmaWarps * 32) {
            const int row = p / (d / 8), pc = p - row * (d / 8);
            uint4 v = make_uint4(0, 0, 0, 0);
            if (row < vr)
                v = *reinterpret_cast<const uint4*>(a.x + (size_t)(row0 + row) * d + pc * 8);
            *reinterpret_cast<uint4*>(xs + pc / NB * SS + row * RB + pc % NB * 16) = v;
        }
        // epilogue: thread c of a group of four has columns 2 c, 2 c + 1 of the group's
        // pieces; lanes 0 and 1 of warp w send the slice to CTAs w and w + 8 of the cluster
        const int group = threadIdx.x >> 2;
        const int to = warp + kMmaWarps * lane;
        const bool sends = lane < 2 && to < a.csize;
        // shared::cluster offset from this CTA to that one
        const uint32_t peer = sends ? mapa_shared(smem, to) - smem_u32(smem) : 0u;
        // every piece of a group has the same columns: kGroups is a multiple of NB
        const int ecol = (group % NB) * 8;
        const float* const bias = bias_s + ecol + 2 * c;
        float* const mine = sums + warp * (kRows * RS) + g * RS + 2 * c;
        const uint8_t* const xa = xs + k0 / OC * SS + g * RB + k0 % OC * 2;
        const bool relu = (a.flags & 4u) != 0, residual = (a.flags & 2u) != 0;
        uint32_t use = 0;
        int sent = 0;   // slices that this lane has sent
        __syncthreads();   // x_t and the biases in place

        for (int l = 0; l < L; ++l) {
            const uint32_t xb = l & 1;
            const bool recv = prow[l] >= 0;
            // the next layer's input arrives as a slice from every CTA of the cluster
            if (threadIdx.x == 0 && ok && l + 1 < L) {
                mbar_arrive_expect_tx(&xs_bar[xb ^ 1], a.csize * SB);
                armed = l + 1;
            }
            const float2 bv = *reinterpret_cast<const float2*>(bias + l * OC);
            if (SPLIT) {
#pragma unroll
                for (int i = 0; i < GP; ++i) {
#pragma unroll
                    for (int u = 0; u < NB; ++u) w[i][u] = w2[i][u];
                    if (l + 1 < L) load_group(w2[i], ws + (l + 1) * wlayer, i);
                }
            }
            if (SPLIT && recv && warp < kPWarps) {
                const uint32_t slot = (use & 1) * kPWarps + warp;
                wait(&pfull[slot], (use >> 1) & 1, false);
                const float4* src = pacc + (size_t)slot * NB * 32 + lane;
#pragma unroll
                for (int u = 0; u < NB; ++u) {
                    const float4 t = src[u * 32];
                    acc[u][0] = t.x;
                    acc[u][1] = t.y;
                    acc[u][2] = t.z;
                    acc[u][3] = t.w;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&pfree[slot]);
                ++use;
            } else {
                clear();
            }
            if (!SPLIT) {
                if (recv) {
#pragma unroll
                    for (int i = 0; i < GP; ++i) {
                        contract(xp[i][0], xp[i][1], w[i], i);
                        load_group(w[i], ws + l * wlayer, i);
                    }
                }
                if (l + 1 < L && prow[l + 1] >= 0) {
#pragma unroll
                    for (int i = 0; i < GP; ++i) load_partner(xp[i], l + 1, i);
                }
            }
            const uint8_t* xl = xa + xb * xbuf;
            if (l > 0) wait(&xs_bar[xb], ((l - 1) >> 1) & 1, true);
            if (ok) seen = l;
#pragma unroll
            for (int i = 0; i < GP; ++i)
                if (i < ng) {
                    const uint8_t* xg = xl + i * (64 / OC * SS);
                    contract(lds16(xg), lds16(xg + 8 * RB), w[i], i);
                    if (!SPLIT && l + 1 < L) load_group(w[i], first_part(l + 1), i);
                }
            // A warp writes its block of sums again only once the next layer's input is
            // complete, which this CTA has sent after every thread's reads.
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                *reinterpret_cast<float2*>(mine + u * 8) = make_float2(acc[u][0], acc[u][1]);
                *reinterpret_cast<float2*>(mine + 8 * RS + u * 8) =
                    make_float2(acc[u][2], acc[u][3]);
            }
            named_bar_sync(1, kMmaWarps * 32);
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int pk = group + i * kGroups;
                if (pk >= kPacks) break;   // warp-uniform
                const int row = pk / NB;
                const float* sum = sums + row * RS + ecol + 2 * c;
                float2 p[kMmaWarps];
#pragma unroll
                for (int k = 0; k < kMmaWarps; ++k)
                    p[k] = *reinterpret_cast<const float2*>(sum + k * (kRows * RS));
                const uint32_t off = row * RB + ecol * 2;   // the piece in a slice
                const uint32_t xin =
                    *reinterpret_cast<const uint32_t*>(xs + xb * xbuf + q * SS + off + 4 * c);
                float2 v = p[0];
#pragma unroll
                for (int k = 1; k < kMmaWarps; ++k) {
                    v.x += p[k].x;
                    v.y += p[k].y;
                }
                v.x += bv.x;
                v.y += bv.y;
                if (relu) {
                    v.x = v.x > 0.f ? v.x : 0.f;
                    v.y = v.y > 0.f ? v.y : 0.f;
                }
                if (residual) {
                    const float2 f = unpack_bf16x2(xin);
                    v.x += f.x;
                    v.y += f.y;
                }
                const uint32_t out = pack_bf16x2(v.x, v.y);
                uint4 p4;
                p4.x = __shfl_sync(0xffffffffu, out, 0, 4);
                p4.y = __shfl_sync(0xffffffffu, out, 1, 4);
                p4.z = __shfl_sync(0xffffffffu, out, 2, 4);
                p4.w = __shfl_sync(0xffffffffu, out, 3, 4);
                if (c == 0) *reinterpret_cast<uint4*>(slice + (xb ^ 1) * SB + off) = p4;
                if (row < vr) {
                    const size_t at = (size_t)(row0 + row) * d + col0 + ecol;
                    if (l == 0)   // position t's layer-0 input into layer 0's ring
                        *reinterpret_cast<uint32_t*>(a.ring0 + at + 2 * c) = xin;
                    if (c == 0) *reinterpret_cast<uint4*>(outp[l] + at) = p4;
                }
            }
            if (l + 1 < L) {
                // the slice to every CTA of the cluster, this one included.  (Its buffer is
                // free: the copies of two layers ago were part of inputs since used.)
                fence_proxy_async_smem();
                named_bar_sync(1, kMmaWarps * 32);
                if (ok && sends) {
                    copy_to_peer(smem_u32(xs) + (xb ^ 1) * xbuf + q * SS + peer,
                                 smem_u32(slice) + (xb ^ 1) * SB, SB,
                                 smem_u32(xs_bar) + 8 * (xb ^ 1) + peer);
                    ++sent;
                }
                __syncwarp();
            }
        }
        if (!ok) {   // a warp that gave up: every CTA is told, and what it was not sent
            if (sends) st_remote(mapa_shared(const_cast<int*>(unsent) + q, to), L - 1 - sent);
            if (lane < a.csize) st_remote(mapa_shared(const_cast<int*>(down), lane), 1);
        }
    }
    __syncwarp();
    cluster_sync_all();   // no CTA sends any more
    // Normally every copy has been waited for as part of an input.  After an abort the ones
    // on their way into this CTA are: the bytes of the slices that were not sent are taken
    // off an input's barrier, and it completes when the others have landed.  (At most two
    // inputs are under way, on different barriers: a CTA sends the one after next only with
    // this CTA's slice of the next.)  Then all CTAs leave, with nothing read from them either.
    if (*down) {
        if (threadIdx.x == 0)
            for (int l = seen + 1; l < L; ++l) {
                int n = 0;
                for (int i = 0; i < a.csize; ++i) n += L - 1 - unsent[i] >= l;
                if (n == 0) break;
                uint64_t* bar = &xs_bar[l & 1];
                if (l > armed) mbar_arrive_expect_tx(bar, a.csize * SB);
                if (n < a.csize) mbar_complete_tx(bar, (a.csize - n) * SB);
                if (!mbar_wait_drain(bar, ((l - 1) >> 1) & 1, kDrainNs)) break;
            }
        __syncthreads();
        cluster_sync_all();
    }
}

size_t decode_mma_smem(int d, int oc, int L) {
    return (size_t)2 * (d / oc) * mma_slice_step(oc) + 2 * mma_slice_bytes(oc) +
           (size_t)kMmaWarps * kRows * mma_sum_row(oc) * 4 +
           (mma_split(oc) ? (size_t)2 * kPWarps * kRows * oc * 4 : 0) + kMmaBars * 8 +
           kMaxDecodeLayers * 12 + 16 + 64 + (size_t)L * oc * 4;
}

}  // namespace

bool decode_geometry(int d, DecodeGeo* g) {
    if (d < 64 || d % 64 != 0 || d > 1024) return false;
    int oc = 16;
    while (d / oc > 16) oc *= 2;   // C = d / OC CTAs, at most 16; OC in {16, 32, 64}
    g->d = d;
    g->oc = oc;
    g->csize = d / oc;
    g->kc = oc == 64 ? 128 : 256;
    if (g->kc > d) g->kc = d;
    g->nchunks = (d + g->kc - 1) / g->kc;
    const size_t fixed =
        1024 + (size_t)4 * kRows * d * 2 + (size_t)2 * kRows * oc * 4 + B_COUNT * 8 + 16;
    const size_t stage = (size_t)oc * g->kc * 2;
    const size_t budget = 226 * 1024;
    const int s = (int)((budget - fixed) / stage);
    g->stages = s > kMaxStages ? kMaxStages : s;
    return g->stages >= 2;
}

size_t decode_smem_bytes(const DecodeGeo& g) {
    return 1024 + (size_t)4 * kRows * g.d * 2 + (size_t)g.stages * g.oc * g.kc * 2 +
           (size_t)2 * kRows * g.oc * 4 + B_COUNT * 8 + 16;
}

// Clusters of csize CTAs, one per 16 rows; pdl: as a programmatic dependent.  The
// kernel's attributes are set once per device and a cluster that does not fit is the
// launch's own error: with two attributes and an occupancy query a call, windows of
// short steps were bound by the host (32 positions of 22 layers at d = 64: 614 us, 583
// without; 256 of 16 layers at d = 512: 5,993 us, 5,860).
template <typename Args>
using ClusterKernel = void (*)(Args);
template <typename Args, ClusterKernel<Args> kern>
static cudaError_t launch_clusters(const Args& a, int threads, size_t smem, bool pdl,
                                   cudaStream_t st, int csize) {
    static std::atomic<bool> configured[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    auto configure = [&]() {
        int most = 0;
        cudaError_t r = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (r == cudaSuccess)
            r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (r == cudaSuccess)
            r = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (r == cudaSuccess && dev < 64) configured[dev].store(true, std::memory_order_release);
        return r;
    };
    const bool cached = dev < 64 && configured[dev].load(std::memory_order_acquire);
    if (!cached && (e = configure()) != cudaSuccess) return e;
    const int blocks = (a.B + kRows - 1) / kRows;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(blocks * csize));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)csize;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 2 : 1;
    e = cudaLaunchKernelEx(&cfg, kern, a);
    if (e == cudaSuccess || !cached) return e;
    // the attributes do not outlive a device reset: set them again, once
    cudaGetLastError();
    e = configure();
    return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, kern, a) : e;
}

cudaError_t launch_decode(const DecodeLaunch& p, cudaStream_t st) {
    if (p.L < 1 || p.L > kMaxDecodeLayers) return cudaErrorInvalidValue;
    if (p.tc) {
        DecodeArgs a;
        a.mWs = p.mWs;
        a.mWn = p.mWn;
        a.mCache = p.mCache;
        a.mX = p.mX;
        for (int l = 0; l < p.L; ++l) {
            a.prow[l] = p.prow[l];
            a.out[l] = p.out[l];
        }
        a.bias = p.bias;
        a.ring0 = p.ring0;
        a.g = p.g;
        a.L = p.L;
        a.B = p.B;
        a.flags = p.flags;
        a.timeout_ns = p.timeout_ns;
        return launch_clusters<DecodeArgs, decode_tc_kernel>(a, kThreads, decode_smem_bytes(p.g),
                                                             false, st, p.g.csize);
    }
    DecodeMmaArgs a;
    a.Ws = p.Ws;
    a.Wn = p.Wn;
    a.x = p.x;
    a.cache = p.cache;
    a.bias = p.bias;
    a.ring0 = p.ring0;
    for (int l = 0; l < p.L; ++l) {
        a.prow[l] = p.prow[l];
        a.out[l] = p.out[l];
    }
    a.d = p.g.d;
    a.csize = p.g.csize;
    a.L = p.L;
    a.B = p.B;
    a.flags = p.flags;
    a.timeout_ns = p.timeout_ns;
    // K groups of 64 features a warp: OC = 16 up to d = 256, 32 up to 512, then 64
    const bool w32 = ((reinterpret_cast<uintptr_t>(p.Ws) | reinterpret_cast<uintptr_t>(p.Wn) |
                       reinterpret_cast<uintptr_t>(p.cache)) & 31) == 0;
    auto launch =
        p.g.oc == 16 ? (w32 ? launch_clusters<DecodeMmaArgs, decode_mma_kernel<16, 1, true>>
                            : launch_clusters<DecodeMmaArgs, decode_mma_kernel<16, 1, false>>)
        : p.g.oc == 32 ? (w32 ? launch_clusters<DecodeMmaArgs, decode_mma_kernel<32, 1, true>>
                              : launch_clusters<DecodeMmaArgs, decode_mma_kernel<32, 1, false>>)
                       : (w32 ? launch_clusters<DecodeMmaArgs, decode_mma_kernel<64, 2, true>>
                              : launch_clusters<DecodeMmaArgs, decode_mma_kernel<64, 2, false>>);
    return launch(a, mma_threads(p.g.oc), decode_mma_smem(p.g.d, p.g.oc, p.L), true, st,
                  p.g.csize);
}

cudaError_t decode_error_word_read_clear(int* word) {
    const int zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(word, g_error_word, sizeof(int));
    if (e == cudaSuccess && *word) e = cudaMemcpyToSymbol(g_error_word, &zero, sizeof(int));
    return e;
}

}  // namespace hcw
