// hcw_simt.cu -- CUDA-core kernels of libhcw:
//   * the fp32 path of the layer (forward, input gradient, weight gradient),
//     tiled FFMA with fp32 accumulation, for callers that need fp32 accuracy;
//   * the elementwise / reduction helpers of the bf16 path: ReLU gradient
//     mask, deterministic column sums (dbias), split-K reduction of dW;
//   * the device partner table (same index code as the kernels).
//
// Index rules, per layer link s inside each sample of n positions:
//   s >= 0 (Sec. 3.1): partner p(i) = i XOR 2^s; causal: i receives from p(i)
//          iff bit s of i is set;
//   s < 0  (Eq. (1) with k = -s, "near" of App. A is k = 1): p(i) = i - k, and
//          i receives iff i >= k (a shift always links earlier to later).
#include "hcw_internal.h"

#include <mutex>

namespace hcw {

namespace {

__device__ __forceinline__ int partner_of(int i, int s) { return s >= 0 ? i ^ (1 << s) : i + s; }

__device__ __forceinline__ bool receives(int i, int s, unsigned flags) {
    if (s < 0) return i + s >= 0;
    return !(flags & 1u) || ((i >> s) & 1);
}

// the position that takes x_i as its partner input at link s, or -1
__device__ __forceinline__ int reader_of(int i, int s, int n, unsigned flags) {
    if (s < 0) return i - s < n ? i - s : -1;
    const int p = i ^ (1 << s);
    return receives(p, s, flags) ? p : -1;
}

constexpr int T = 32;   // tile edge of the fp32 kernels

// The fp32 kernels: 32 x 32 output tiles, 32 x 8 threads, 4 outputs per thread,
// the contraction in steps of 32 through shared memory, the next step's operands
// loaded into registers while one is computed.  Their users' sizes are small
// (checks and first experiments, d in the tens): they are bound by launches and by
// the latency of a step, so every launch is a programmatic dependent of the one
// before it, the input gradient writes the layer below's dz itself, and one launch
// computes the weight and bias gradients of a whole stack (seven layers at 3,968 rows of
// d = 91, whose gradient blocks each walked all rows: 2,493 us, now 402).  Narrow layers
// run in one launch a direction (f32_chain_kernel).

// z[r][o] = sum_k Ws[o][k] x[r][k] + m_r sum_k Wn[o][k] x[p(r)][k] + bias[o]
// mout (optional): ReLU mask words [rows][ceil(d/32)], bit o%32 of word o/32 = (z > 0).
__global__ void __launch_bounds__(256)
    f32_fwd_kernel(const float* x, const float* Ws, const float* Wn, const float* bias, int s,
                   int n, int d, long long rows, unsigned flags, float* y, float* z,
                   uint32_t* mout) {
    pdl_wait();   // until the kernel before it in the stream has finished
    pdl_trigger();
    __shared__ float xs[T][T + 1], xp[T][T + 1], ws[T][T + 1], wn[T][T + 1];
    const long long r0 = (long long)blockIdx.y * T;
    const int o0 = blockIdx.x * T;
    const int tx = threadIdx.x, ty = threadIdx.y;
    // this thread's rows ty, ty + 8, ... of the tile: row, partner row (or null)
    const float *xr[4], *pr[4], *wsr[4], *wnr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long r = r0 + ty + 8 * q;
        const int i = (int)(r & (n - 1)), o = o0 + ty + 8 * q;
        xr[q] = r < rows ? x + r * d : nullptr;
        pr[q] = r < rows && receives(i, s, flags) ? x + (r - i + partner_of(i, s)) * d : nullptr;
        wsr[q] = o < d ? Ws + (long long)o * d : nullptr;
        wnr[q] = o < d ? Wn + (long long)o * d : nullptr;
    }
    float a[4], b[4], u[4], v4[4];
    auto load = [&](int k) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            a[q] = xr[q] && k < d ? xr[q][k] : 0.f;
            b[q] = pr[q] && k < d ? pr[q][k] : 0.f;
            u[q] = wsr[q] && k < d ? wsr[q][k] : 0.f;
            v4[q] = wnr[q] && k < d ? wnr[q][k] : 0.f;
        }
    };
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    load(tx);
    for (int k0 = 0; k0 < d; k0 += T) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            xs[ty + 8 * q][tx] = a[q];
            xp[ty + 8 * q][tx] = b[q];
            ws[ty + 8 * q][tx] = u[q];
            wn[ty + 8 * q][tx] = v4[q];
        }
        __syncthreads();
        if (k0 + T < d) load(k0 + T + tx);
#pragma unroll 8
        for (int kk = 0; kk < T; ++kk) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int rr = ty + 8 * q;
                acc[q] = fmaf(xs[rr][kk], ws[tx][kk], acc[q]);
                acc[q] = fmaf(xp[rr][kk], wn[tx][kk], acc[q]);
            }
        }
        __syncthreads();
    }
    const int o = o0 + tx;
    const int wpr = (d + 31) >> 5;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long r = r0 + ty + 8 * q;
        const bool ok = r < rows && o < d;
        float v = ok ? acc[q] + (bias ? bias[o] : 0.f) : 0.f;
        if (mout) {
            // the warp covers the 32 columns of one mask word of row r
            const unsigned bits = __ballot_sync(0xffffffffu, ok && v > 0.f);
            if (tx == 0 && r < rows) mout[r * wpr + (o0 >> 5)] = bits;
        }
        if (!ok) continue;
        if (z) z[r * d + o] = v;
        if (flags & 4u) v = v > 0.f ? v : 0.f;
        if (flags & 2u) v += x[r * d + o];
        y[r * d + o] = v;
    }
}

// dx[r][k] = sum_o dz[r][o] Ws[o][k] + m_{p(r)} sum_o dz[p(r)][o] Wn[o][k] (+ dy[r][k]),
// written to dx (if given) and, where the mask bits mprev of the layer below are set
// (else 0), to dz_prev (if given).
__global__ void __launch_bounds__(256)
    f32_dx_kernel(const float* dz, const float* dy, const float* Ws, const float* Wn, int s, int n,
                  int d, long long rows, unsigned flags, float* dx, const uint32_t* mprev,
                  float* dz_prev) {
    pdl_wait();   // until the kernel before it in the stream has finished
    pdl_trigger();
    __shared__ float gs[T][T + 1], gp[T][T + 1], ws[T][T + 1], wn[T][T + 1];
    const long long r0 = (long long)blockIdx.y * T;
    const int k0 = blockIdx.x * T;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int k = k0 + tx;
    const float *gr[4], *pr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long r = r0 + ty + 8 * q;
        const int i = (int)(r & (n - 1));
        const int j = reader_of(i, s, n, flags);
        gr[q] = r < rows ? dz + r * d : nullptr;
        pr[q] = r < rows && j >= 0 ? dz + (r - i + j) * d : nullptr;
    }
    float a[4], b[4], u[4], v4[4];
    auto load = [&](int o0) {
        const int o = o0 + tx;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int oo = o0 + ty + 8 * q;
            const bool w = oo < d && k < d;
            a[q] = gr[q] && o < d ? gr[q][o] : 0.f;
            b[q] = pr[q] && o < d ? pr[q][o] : 0.f;
            u[q] = w ? Ws[(long long)oo * d + k] : 0.f;
            v4[q] = w ? Wn[(long long)oo * d + k] : 0.f;
        }
    };
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    load(0);
    for (int o0 = 0; o0 < d; o0 += T) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            gs[ty + 8 * q][tx] = a[q];
            gp[ty + 8 * q][tx] = b[q];
            ws[ty + 8 * q][tx] = u[q];
            wn[ty + 8 * q][tx] = v4[q];
        }
        __syncthreads();
        if (o0 + T < d) load(o0 + T);
#pragma unroll 8
        for (int oo = 0; oo < T; ++oo) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int rr = ty + 8 * q;
                acc[q] = fmaf(gs[rr][oo], ws[oo][tx], acc[q]);
                acc[q] = fmaf(gp[rr][oo], wn[oo][tx], acc[q]);
            }
        }
        __syncthreads();
    }
    if (k >= d) return;
    const int wpr = (d + 31) >> 5;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long r = r0 + ty + 8 * q;
        if (r >= rows) continue;
        float v = acc[q];
        if (flags & 2u) v += dy[r * d + k];
        if (dx) dx[r * d + k] = v;
        // (the tile's 32 columns are one mask word)
        if (dz_prev) dz_prev[r * d + k] = (mprev[r * wpr + (k0 >> 5)] >> tx) & 1u ? v : 0.f;
    }
}

// ---- fp32 stacks of narrow layers: all layers in one launch ----
// A block keeps the rows of whole windows on chip and walks the layers over them (every
// partner of a row is in its window), the next layers' weights, biases and masks on their
// way into a ring of shared-memory buffers while one is computed.  Layer by layer these
// stacks are bound by launches, about 4 us each: four layers forward and backward at 64
// rows of d = 32 took 46 us a call of each, now 29 (the host's part), 19 of them on the
// GPU.  One or two output columns a lane, kChainRows rows per warp at a time, and the
// products in the order of the tiled kernels: the same bits.  A layer is bound by
// shared-memory reads (ten 16-byte ones for 32 products a lane, twelve for 64 with two
// columns), 0.7 us at 16 rows of d = 32.
constexpr int kChainRows = 4;
constexpr size_t kChainSmem = 232448;

__device__ __forceinline__ void cp_async_f32(float* dst, const float* src, bool vec) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(dst);
    if (vec)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(a), "l"(src) : "memory");
}

// Row stride in shared memory: whole 16-byte pieces, an odd number of them (a quarter of
// a warp reading one piece of eight rows hits every bank once).
__host__ __device__ inline int chain_ld(int d) { return 4 * (((d + 3) / 4) | 1); }

// One buffer of the ring, in floats: both weights, and the bias or the rows' mask words.
__host__ __device__ inline size_t chain_stage(int d, int rows) {
    const size_t ld = chain_ld(d), d4 = (d + 3) & ~3, mw = (size_t)rows * ((d + 31) / 32);
    return 2 * d4 * ld + (((mw > d4 ? mw : d4) + 3) & ~(size_t)3);
}

// Shared memory, in floats: the ring, three buffers of rows, a row of zeros.
__host__ __device__ inline size_t chain_floats(int d, int rows, int stages) {
    return stages * chain_stage(d, rows) + (3 * (size_t)rows + 1) * chain_ld(d);
}

// BWD false: x through layers 0 .. L-1 to acts, y and the mask words.  BWD true: dy down
// through layers L-1 .. 0 to every layer's dz and dx.
// NC: output columns a lane, 32 apart.
template <bool BWD, int NC>
__global__ void __launch_bounds__(256) f32_chain_kernel(const __grid_constant__ F32ChainArgs A) {
    extern __shared__ float4 chain_smem[];
    float* smem = reinterpret_cast<float*>(chain_smem);
    const int d = A.d, d4 = (d + 3) & ~3, ld = chain_ld(d), n = A.n;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wsz = d4 * ld, xsz = A.block_rows * ld;
    const int stage = (int)chain_stage(d, A.block_rows);
    float* const xbuf = smem + A.stages * stage;
    float* const gbuf = xbuf + 2 * xsz;      // BWD: the unmasked gradient (residual)
    const int zero = (int)(gbuf + xsz - smem);   // the row of zeros
    const int pieces = (int)(chain_floats(d, A.block_rows, A.stages) / 4);
    for (int i = threadIdx.x; i < pieces; i += blockDim.x)
        chain_smem[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    pdl_wait();   // until the kernel before it in the stream has finished
    pdl_trigger();

    const long long r0 = (long long)blockIdx.x * A.block_rows;
    const int rows = A.rows - r0 < A.block_rows ? (int)(A.rows - r0) : A.block_rows;
    const bool vec = A.vec;
    const int wpr = (d + 31) >> 5;
    const bool relu = A.flags & 4u, res = A.flags & 2u;
    // this thread's piece of a row, and the rows a pass of the block takes
    const int prow = threadIdx.x >> A.lanes_log2, prows = 256 >> A.lanes_log2;
    const int pcol = (threadIdx.x & ((1 << A.lanes_log2) - 1)) * (vec ? 4 : 1);
    // the i-th layer of the walk into its buffer (nothing past the last: an empty group)
    auto issue = [&](int i) {
        if (i >= A.L) {
            asm volatile("cp.async.commit_group;" ::: "memory");
            return;
        }
        const int l = BWD ? A.L - 1 - i : i;
        float* const buf = smem + (i & (A.stages - 1)) * stage;
        const float* const src[2] = {A.Ws + (size_t)l * d * d, A.Wn + (size_t)l * d * d};
        for (int o = prow; o < d; o += prows)
            if (pcol < d) {
                cp_async_f32(buf + o * ld + pcol, src[0] + o * d + pcol, vec);
                cp_async_f32(buf + wsz + o * ld + pcol, src[1] + o * d + pcol, vec);
            }
        const float* aux = nullptr;
        int count = 0;
        if (!BWD && A.bias) {
            aux = A.bias + (size_t)l * d;
            count = d;
        } else if (BWD && relu && l > 0) {
            aux = reinterpret_cast<const float*>(A.masks + (size_t)(l - 1) * A.mask_words + r0 * wpr);
            count = rows * wpr;
        }
        for (int t = threadIdx.x; t < count; t += 256)
            cp_async_f32(buf + 2 * wsz + t, aux + t, false);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int top = A.L - 1;
    if (!BWD && pcol < d)   // the rows: part of the first layer's group
        for (int r = prow; r < rows; r += prows)
            cp_async_f32(xbuf + r * ld + pcol, A.in + (r0 + r) * d + pcol, vec);
    for (int i = 0; i + 1 < A.stages; ++i) issue(i);
    if (BWD && pcol < d) {
        // the top layer's dz
        const uint32_t* const mask = A.masks + (size_t)top * A.mask_words + r0 * wpr + (pcol >> 5);
        auto row = [&](int r, auto v) {
            const uint32_t w = (relu ? mask[r * wpr] : ~0u) >> (pcol & 31);
            const size_t at = (r0 + r) * d + pcol;
            *reinterpret_cast<decltype(v)*>(gbuf + r * ld + pcol) = v;
            float* e = reinterpret_cast<float*>(&v);
#pragma unroll
            for (int j = 0; j < (int)(sizeof(v) / 4); ++j) e[j] = (w >> j) & 1u ? e[j] : 0.f;
            *reinterpret_cast<decltype(v)*>(xbuf + r * ld + pcol) = v;
            *reinterpret_cast<decltype(v)*>(A.acts + (size_t)top * A.act_elems + at) = v;
        };
        if (vec)
            for (int r = prow; r < rows; r += prows)
                row(r, *reinterpret_cast<const float4*>(A.in + (r0 + r) * d + pcol));
        else
            for (int r = prow; r < rows; r += prows) row(r, A.in[(r0 + r) * d + pcol]);
    }

    const int cwarps = (wpr + NC - 1) / NC, groups = 8 / cwarps;   // column warps, row groups
    const int cw = (warp % cwarps) * NC, grp = warp / cwarps;      // first mask word, group
    const int c0 = cw * 32 + lane;
    int cc[NC];
#pragma unroll
    for (int h = 0; h < NC; ++h) cc[h] = c0 + 32 * h < d ? c0 + 32 * h : 0;
    for (int i = 0; i < A.L; ++i) {
        const int l = BWD ? A.L - 1 - i : i;
        if (A.stages == 4)
            asm volatile("cp.async.wait_group 2;" ::: "memory");
        else
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();   // this layer's weights and rows are there, the one before is done
        issue(i + A.stages - 1);
        const float* ws = smem + (i & (A.stages - 1)) * stage;
        const float* wn = ws + wsz;
        const float* aux = wn + wsz;
        const float* cur = xbuf + (i & 1) * xsz;
        const int curo = (int)(cur - smem);
        float* next = xbuf + ((i + 1) & 1) * xsz;
        const int s = A.s[l];
        const bool last = i + 1 == A.L;
        float bias[NC];
#pragma unroll
        for (int h = 0; h < NC; ++h) bias[h] = !BWD && A.bias ? aux[cc[h]] : 0.f;
        if (grp < groups)
            for (int rb = grp * kChainRows; rb < rows; rb += groups * kChainRows) {
                int xr[kChainRows], pr[kChainRows];   // rows' offsets in shared memory
                uint32_t mw[NC][kChainRows];
#pragma unroll
                for (int q = 0; q < kChainRows; ++q) {
                    const int rr = rb + q, j = rr & (n - 1);
                    int from = -1;
                    if (rr < rows) {
                        if (BWD)
                            from = reader_of(j, s, n, A.flags);
                        else if (receives(j, s, A.flags))
                            from = partner_of(j, s);
                    }
                    xr[q] = rr < rows ? curo + rr * ld : zero;
                    pr[q] = from >= 0 ? curo + (rr - j + from) * ld : zero;
#pragma unroll
                    for (int h = 0; h < NC; ++h)
                        mw[h][q] = BWD && relu && !last && rr < rows && cw + h < wpr
                                       ? reinterpret_cast<const uint32_t*>(aux)[rr * wpr + cw + h]
                                       : ~0u;
                }
                float acc[NC][kChainRows];
#pragma unroll
                for (int h = 0; h < NC; ++h)
#pragma unroll
                    for (int q = 0; q < kChainRows; ++q) acc[h][q] = 0.f;
#pragma unroll(NC == 1 ? 4 : 2)
                for (int k = 0; k < d4; k += 4) {
                    float u[NC][4], v[NC][4];
                    float4 xv[kChainRows], pv[kChainRows];
#pragma unroll
                    for (int h = 0; h < NC; ++h) {
                        if (BWD) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                u[h][j] = ws[(k + j) * ld + cc[h]];
                                v[h][j] = wn[(k + j) * ld + cc[h]];
                            }
                        } else {
                            const float4 a = *reinterpret_cast<const float4*>(ws + cc[h] * ld + k);
                            const float4 b = *reinterpret_cast<const float4*>(wn + cc[h] * ld + k);
                            u[h][0] = a.x, u[h][1] = a.y, u[h][2] = a.z, u[h][3] = a.w;
                            v[h][0] = b.x, v[h][1] = b.y, v[h][2] = b.z, v[h][3] = b.w;
                        }
                    }
#pragma unroll
                    for (int q = 0; q < kChainRows; ++q) {
                        xv[q] = *reinterpret_cast<const float4*>(smem + xr[q] + k);
                        pv[q] = *reinterpret_cast<const float4*>(smem + pr[q] + k);
                    }
                    auto step = [&](auto at, int j) {
#pragma unroll
                        for (int h = 0; h < NC; ++h)
#pragma unroll
                            for (int q = 0; q < kChainRows; ++q)
                                acc[h][q] = fmaf(at(xv[q]), u[h][j], acc[h][q]);
#pragma unroll
                        for (int h = 0; h < NC; ++h)
#pragma unroll
                            for (int q = 0; q < kChainRows; ++q)
                                acc[h][q] = fmaf(at(pv[q]), v[h][j], acc[h][q]);
                    };
                    step([](const float4& f) { return f.x; }, 0);
                    step([](const float4& f) { return f.y; }, 1);
                    step([](const float4& f) { return f.z; }, 2);
                    step([](const float4& f) { return f.w; }, 3);
                }
#pragma unroll
                for (int q = 0; q < kChainRows; ++q) {
                    const int rr = rb + q;
                    if (rr >= rows) break;   // warp-uniform
#pragma unroll
                    for (int h = 0; h < NC; ++h) {
                        if (cw + h >= wpr) break;   // warp-uniform
                        const int c = c0 + 32 * h;
                        const bool col_ok = c < d;
                        const size_t at = (r0 + rr) * d + c;
                        if (BWD) {
                            float v = acc[h][q];
                            if (!col_ok) continue;
                            if (res) v += gbuf[rr * ld + c];
                            gbuf[rr * ld + c] = v;
                            if (last) {
                                A.out[at] = v;
                            } else {
                                v = (mw[h][q] >> lane) & 1u ? v : 0.f;
                                next[rr * ld + c] = v;
                                A.acts[(size_t)(l - 1) * A.act_elems + at] = v;
                            }
                        } else {
                            float v = col_ok ? acc[h][q] + bias[h] : 0.f;
                            if (A.mask_out) {
                                const unsigned bits = __ballot_sync(0xffffffffu, v > 0.f);
                                if (lane == 0)
                                    A.mask_out[(size_t)l * A.mask_words + (r0 + rr) * wpr + cw + h] =
                                        bits;
                            }
                            if (!col_ok) continue;
                            if (relu) v = v > 0.f ? v : 0.f;
                            if (res) v += cur[rr * ld + c];
                            if (last) {
                                A.out[at] = v;
                            } else {
                                next[rr * ld + c] = v;
                                A.acts[(size_t)l * A.act_elems + at] = v;
                            }
                        }
                    }
                }
            }
    }
}

// A sum kept with its rounding errors (Knuth's two-sum), for the bias gradients: one chain
// over many rows in fp32 alone loses digits with their number (65,536 rows in one split:
// 1.3e-6 relative in eight chains, 1.9e-7 in a tree of 64-row sums, 0.7e-7 so).
struct LongSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = __fadd_rn(s, x), b = __fsub_rn(t, s);
        c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b)));
        s = t;
    }
    // (past an infinity the errors are no numbers, the sum is)
    __device__ __forceinline__ float value() const { return isfinite(s) ? s + c : s; }
};

// Per layer l and split sp of the rows,
//   dWs[o][k] = sum_r dz[r][o] x[r][k];  dWn[o][k] = sum_r m_r dz[r][o] x[p(r)][k];
//   dbias[o] = sum_r dz[r][o]
// A block per 32 o x 32 k and (l, sp) = blockIdx.z; its rows in order.  One split
// writes the gradients, several their partial sums [l][sp][2 d d + d], which
// f32_dw_reduce_kernel adds in split order: the same bits every time.
__global__ void __launch_bounds__(256) f32_dw_kernel(const __grid_constant__ F32DwArgs A) {
    pdl_wait();   // until the kernel before it in the stream has finished
    pdl_trigger();
    __shared__ float gz[T][T + 1], xs[T][T + 1], xp[T][T + 1];
    const int l = blockIdx.z / A.splits, sp = blockIdx.z - l * A.splits;
    const int n = A.n, d = A.d, s = A.s[l];
    const unsigned flags = A.flags;
    const float* x = l == 0 ? A.x : A.acts + (l - 1) * A.act_elems;
    const float* dz = A.dz + l * A.act_elems;
    const long long rb = (long long)sp * A.rows_per_split;
    const long long re = rb + A.rows_per_split < A.rows ? rb + A.rows_per_split : A.rows;
    const int o0 = blockIdx.y * T, k0 = blockIdx.x * T;
    const int tx = threadIdx.x, ty = threadIdx.y;
    float g[4], a[4], b[4];
    auto load = [&](long long r0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const long long r = r0 + ty + 8 * q;
            const int i = (int)(r & (n - 1));
            g[q] = r < re && o0 + tx < d ? dz[r * d + o0 + tx] : 0.f;
            a[q] = r < re && k0 + tx < d ? x[r * d + k0 + tx] : 0.f;
            b[q] = r < re && k0 + tx < d && receives(i, s, flags)
                       ? x[(r - i + partner_of(i, s)) * d + k0 + tx]
                       : 0.f;
        }
    };
    float as[4] = {0.f, 0.f, 0.f, 0.f}, an[4] = {0.f, 0.f, 0.f, 0.f};
    LongSum cs;
    load(rb);
    for (long long r0 = rb; r0 < re; r0 += T) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            gz[ty + 8 * q][tx] = g[q];
            xs[ty + 8 * q][tx] = a[q];
            xp[ty + 8 * q][tx] = b[q];
        }
        cs.add((g[0] + g[1]) + (g[2] + g[3]));
        __syncthreads();
        if (r0 + T < re) load(r0 + T);
#pragma unroll 8
        for (int rr = 0; rr < T; ++rr) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float gv = gz[rr][ty + 8 * q];
                as[q] = fmaf(gv, xs[rr][tx], as[q]);
                an[q] = fmaf(gv, xp[rr][tx], an[q]);
            }
        }
        __syncthreads();
    }
    const size_t dd = (size_t)d * d;
    float* part = A.part + ((size_t)l * A.splits + sp) * (2 * dd + d);
    float* ws = A.splits > 1 ? part : A.dWs + l * dd;
    float* wn = A.splits > 1 ? part + dd : A.dWn + l * dd;
    const int k = k0 + tx;
    if (k < d) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int o = o0 + ty + 8 * q;
            if (o >= d) continue;
            ws[(size_t)o * d + k] = as[q];
            wn[(size_t)o * d + k] = an[q];
        }
    }
    if (blockIdx.x == 0 && A.dbias) {
        // the eight row lanes' column sums, in a fixed order
        gz[ty][tx] = cs.value();
        __syncthreads();
        if (ty == 0 && o0 + tx < d) {
            const float t = ((gz[0][tx] + gz[1][tx]) + (gz[2][tx] + gz[3][tx])) +
                            ((gz[4][tx] + gz[5][tx]) + (gz[6][tx] + gz[7][tx]));
            (A.splits > 1 ? part + 2 * dd : A.dbias + (size_t)l * d)[o0 + tx] = t;
        }
    }
}

// The split sums of f32_dw_kernel, in split order: a thread per output of layer
// blockIdx.y.
__global__ void __launch_bounds__(256) f32_dw_reduce_kernel(const __grid_constant__ F32DwArgs A) {
    pdl_wait();   // until the kernel before it in the stream has finished
    pdl_trigger();
    const int l = blockIdx.y;
    const size_t dd = (size_t)A.d * A.d, tot = 2 * dd + A.d;
    const size_t e = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= tot || (e >= 2 * dd && !A.dbias)) return;
    const float* p = A.part + (size_t)l * A.splits * tot + e;
    if (e >= 2 * dd) {
        LongSum b;
#pragma unroll 8
        for (int sp = 0; sp < A.splits; ++sp) b.add(p[sp * tot]);
        A.dbias[(size_t)l * A.d + e - 2 * dd] = b.value();
        return;
    }
    float t = 0.f;
#pragma unroll 8
    for (int sp = 0; sp < A.splits; ++sp) t += p[sp * tot];
    if (e < dd)
        A.dWs[l * dd + e] = t;
    else
        A.dWn[l * dd + e - dd] = t;
}

template <typename V>
__device__ __forceinline__ float to_f(V v);
template <>
__device__ __forceinline__ float to_f<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) {
    return __bfloat162float(v);
}

// dz = z > 0 ? dy : 0 over count elements, a thread per 16 bytes (all three
// 16-byte aligned), four pieces in flight; the last count % VEC elements one a
// thread.  Bound by memory: at 8.4 M bf16 elements (50 MB) 23.7 us with one
// element a thread and access, 13 us so.
template <typename V>
__global__ void __launch_bounds__(256)
    relu_grad_kernel(const V* dy, const V* z, V* dz, size_t count) {
    pdl_wait();   // until the kernel before it in the stream has finished
    pdl_trigger();
    constexpr int VEC = 16 / sizeof(V), U = 4;
    const size_t pieces = count / VEC, stride = (size_t)gridDim.x * blockDim.x;
    const size_t t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (size_t t = t0; t < pieces; t += U * stride) {
        uint4 g[U], a[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (t + u * stride < pieces) {
                g[u] = reinterpret_cast<const uint4*>(dy)[t + u * stride];
                a[u] = reinterpret_cast<const uint4*>(z)[t + u * stride];
            }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (t + u * stride < pieces) {
                V* gv = reinterpret_cast<V*>(&g[u]);
                const V* av = reinterpret_cast<const V*>(&a[u]);
#pragma unroll
                for (int i = 0; i < VEC; ++i) gv[i] = to_f(av[i]) > 0.f ? gv[i] : V(0.f);
                reinterpret_cast<uint4*>(dz)[t + u * stride] = g[u];
            }
    }
    const size_t rest = pieces * VEC + t0;
    if (rest < count) dz[rest] = to_f(z[rest]) > 0.f ? dy[rest] : V(0.f);
}

// dz[t][o] = mask bit (t, o) ? dy[t][o] : 0, masks as written by the forward
// (any d: rows of ceil(d / 32) mask words).
__global__ void relu_grad_mask_f32_kernel(const float* dy, const uint32_t* mask, float* dz,
                                          long long rows, int d) {
    pdl_wait();   // until the kernel before it in the stream has finished
    pdl_trigger();
    const int wpr = (d + 31) >> 5;
    const size_t count = (size_t)rows * d;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < count;
         t += (size_t)gridDim.x * blockDim.x) {
        const size_t r = t / d;
        const int o = (int)(t - r * d);
        dz[t] = (mask[r * wpr + (o >> 5)] >> (o & 31)) & 1u ? dy[t] : 0.f;
    }
}

// The same for bf16 rows (d a multiple of 64): one thread per 16 bytes of a
// row, so a group never straddles a mask word.
__global__ void relu_grad_mask_kernel(const __nv_bfloat16* __restrict__ dy,
                                      const uint32_t* __restrict__ mask,
                                      __nv_bfloat16* __restrict__ dz, long long rows, int d) {
    constexpr int VEC = 8;
    const int wpr = d >> 5;
    const int gpr = d / VEC;   // groups per row
    const size_t count = (size_t)rows * gpr;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < count;
         t += (size_t)gridDim.x * blockDim.x) {
        const size_t r = t / gpr;
        const int o = (int)(t - r * gpr) * VEC;
        const uint32_t bits = (mask[r * wpr + (o >> 5)] >> (o & 31)) & ((1u << VEC) - 1u);
        uint4 v = reinterpret_cast<const uint4*>(dy)[t];
        uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
            w[i] &= ((bits >> (2 * i)) & 1u ? 0x0000FFFFu : 0u) |
                    ((bits >> (2 * i + 1)) & 1u ? 0xFFFF0000u : 0u);
        reinterpret_cast<uint4*>(dz)[t] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// rows per partial of the column sum: 64 up to 65,536 rows (enough CTAs to
// fill the GPU), 256 above (the partials stay small)
inline long long col_rows(long long rows) { return rows <= 65536 ? 64 : 256; }

// partial[c][o] = sum_{r in chunk c} dz[r][o] for bf16 rows (d a multiple of 64), 16-byte
// loads.  Block: 64 column groups of 16 bytes x 4 row lanes; each thread sums its group over
// every 4th row of the chunk, then the 4 row lanes are added in a fixed order.
__global__ void colsum_partial_kernel(const __nv_bfloat16* __restrict__ dz, long long rows, int d,
                                      int crows, float* __restrict__ partial) {
    constexpr int VEC = 8;
    __shared__ float red[4][64][VEC + 1];
    // blockIdx.z selects one of several equally shaped matrices (layers)
    dz += (size_t)blockIdx.z * rows * d;
    partial += (size_t)blockIdx.z * gridDim.y * d;
    const int gpr = d / VEC;
    const int g = blockIdx.x * 64 + threadIdx.x;
    const long long r0 = (long long)blockIdx.y * crows;
    const long long r1 = min(rows, r0 + crows);
    float acc[VEC];
#pragma unroll
    for (int i = 0; i < VEC; ++i) acc[i] = 0.f;
    if (g < gpr) {
        const uint4* src = reinterpret_cast<const uint4*>(dz) + g;
        for (long long r = r0 + threadIdx.y; r < r1; r += 4) {
            const uint4 q = src[(size_t)r * gpr];
            const __nv_bfloat16* e = reinterpret_cast<const __nv_bfloat16*>(&q);
#pragma unroll
            for (int i = 0; i < VEC; ++i) acc[i] += __bfloat162float(e[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < VEC; ++i) red[threadIdx.y][threadIdx.x][i] = acc[i];
    __syncthreads();
    if (threadIdx.y == 0 && g < gpr) {
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            const float s = ((red[0][threadIdx.x][i] + red[1][threadIdx.x][i]) +
                             red[2][threadIdx.x][i]) + red[3][threadIdx.x][i];
            partial[(long long)blockIdx.y * d + (long long)g * VEC + i] = s;
        }
    }
}

// out[o] = sum over the chunks c of partial[c][o], in chunk order: a CTA of 32
// warps per 32 columns, a column a lane; warp w adds chunks w, w + 32, ...,
// then the warp sums meet in shared memory in warp order.
__global__ void __launch_bounds__(1024) colsum_final_kernel(const float* __restrict__ partial,
                                                            int chunks, int d,
                                                            float* __restrict__ out) {
    __shared__ float red[32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int o = blockIdx.x * 32 + lane;
    partial += (size_t)blockIdx.y * chunks * d;
    out += (size_t)blockIdx.y * d;
    float s = 0.f;
    if (o < d) {
#pragma unroll 4
        for (int c = warp; c < chunks; c += 32) s += partial[(long long)c * d + o];
    }
    red[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && o < d) {
        float t = 0.f;
        for (int w = 0; w < 32; ++w) t += red[w][lane];
        out[o] = t;
    }
}

// out_w[l][o][k] = sum over the splits s of partial[l][w][s][o][k], w in {self,
// partner}; grid.y = 3 adds dbias[l][o] = sum over the self part's splits of
// bpart[l][s][o].  Block: 64 float4 columns x 8 split lanes; lane y adds the
// splits y, y + 8, ... in order, then the 8 lane sums meet in shared memory
// in lane order (deterministic).  grid.y = the part, grid.z = the layer.
__global__ void __launch_bounds__(512) splitk_reduce_kernel(
    const float* partial, int splits_max, int splits_self, int splits_nbr, int d,
    size_t part_stride, float* dWs, float* dWn, size_t out_stride, const float* bpart,
    float* dbias) {
    pdl_wait();   // until the kernel before it in the stream has finished
    pdl_trigger();
    __shared__ float4 red[8][64];
    const int which = blockIdx.y;
    const int S = which == 1 ? splits_nbr : splits_self;
    if (S <= 1) return;   // written directly by the GEMM
    const size_t total4 = which == 2 ? (size_t)d / 4 : (size_t)d * d / 4;
    const size_t e4 = (size_t)blockIdx.x * 64 + threadIdx.x;
    if ((size_t)blockIdx.x * 64 >= total4) return;   // (the dbias rows are short)
    const float4* src = reinterpret_cast<const float4*>(
        which == 2 ? bpart + (size_t)blockIdx.z * splits_self * d
                   : partial + blockIdx.z * part_stride + (size_t)which * splits_max * d * d);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e4 < total4) {
        for (int sp = threadIdx.y; sp < S; sp += 8) {
            const float4 b = src[(size_t)sp * total4 + e4];
            a.x += b.x;
            a.y += b.y;
            a.z += b.z;
            a.w += b.w;
        }
    }
    red[threadIdx.y][threadIdx.x] = a;
    __syncthreads();
    if (threadIdx.y == 0 && e4 < total4) {
#pragma unroll
        for (int y = 1; y < 8; ++y) {
            const float4 b = red[y][threadIdx.x];
            a.x += b.x;
            a.y += b.y;
            a.z += b.z;
            a.w += b.w;
        }
        float* out = which == 2 ? dbias + (size_t)blockIdx.z * d
                                : (which ? dWn : dWs) + blockIdx.z * out_stride;
        reinterpret_cast<float4*>(out)[e4] = a;
    }
}

// out[b][i] = in[b][i - k] for 0 <= i - k < n, else 0 (k of either sign):
// the partner rows of a shift layer (k > 0) or their readers (k < 0), as a
// row-aligned second operand.  One thread per 16-byte piece.
__global__ void shift_rows_kernel(const uint4* __restrict__ in, uint4* __restrict__ out,
                                  long long rows, int n, int pieces, int k) {
    const long long total = rows * pieces;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long r = t / pieces;
        const int c = (int)(t - r * pieces);
        const int i = (int)(r % n);
        const int j = i - k;
        out[t] = (j >= 0 && j < n) ? in[(r - i + j) * pieces + c] : make_uint4(0, 0, 0, 0);
    }
}

__global__ void partner_table_kernel(int s, int n, unsigned flags, int* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = receives(i, s, flags) ? partner_of(i, s) : -1;
}

inline int blocks_for(size_t count, int threads, int cap = 152 * 16) {
    size_t b = (count + threads - 1) / threads;
    return (int)(b < (size_t)cap ? (b == 0 ? 1 : b) : cap);
}

}  // namespace

cudaError_t launch_f32_fwd(const float* x, const float* Ws, const float* Wn, const float* bias,
                           int s, int B, int n, int d, unsigned flags, float* y, float* z,
                           uint32_t* mout, cudaStream_t st) {
    const long long rows = (long long)B * n;
    dim3 grid((d + T - 1) / T, (unsigned)((rows + T - 1) / T));
    return launch_pdl(f32_fwd_kernel, grid, dim3(T, 8), 0, st, x, Ws, Wn, bias, s, n, d, rows,
                      flags, y, z, mout);
}

cudaError_t launch_relu_grad_mask_f32(const float* dy, const uint32_t* mask, float* dz,
                                      long long rows, int d, cudaStream_t st) {
    return launch_pdl(relu_grad_mask_f32_kernel, dim3(blocks_for((size_t)rows * d, 256)), dim3(256),
                      0, st, dy, mask, dz, rows, d);
}

cudaError_t launch_relu_grad_mask_bf16(const __nv_bfloat16* dy, const uint32_t* mask,
                                       __nv_bfloat16* dz, long long rows, int d,
                                       cudaStream_t st) {
    relu_grad_mask_kernel<<<blocks_for((size_t)rows * d / 8, 256), 256, 0, st>>>(dy, mask, dz, rows,
                                                                               d);
    return cudaGetLastError();
}

cudaError_t launch_f32_dx(const float* dz, const float* dy, const float* Ws, const float* Wn,
                          int s, int B, int n, int d, unsigned flags, float* dx,
                          const uint32_t* mprev, float* dz_prev, cudaStream_t st) {
    const long long rows = (long long)B * n;
    dim3 grid((d + T - 1) / T, (unsigned)((rows + T - 1) / T));
    return launch_pdl(f32_dx_kernel, grid, dim3(T, 8), 0, st, dz, dy, Ws, Wn, s, n, d, rows, flags,
                      dx, mprev, dz_prev);
}

// Splits of the rows: enough blocks for two an SM, at least 128 rows (four steps)
// each.  One split at 49 tiles (d = 200) leaves 103 SMs idle and walks all rows in
// one block.
int f32_dw_splits(long long rows, int d, int layers, int sms) {
    const long long tiles = (long long)((d + T - 1) / T) * ((d + T - 1) / T) * layers;
    long long s = (2ll * sms + tiles - 1) / tiles;
    if (s > rows / 128) s = rows / 128;
    return s < 1 ? 1 : (int)s;
}

cudaError_t launch_f32_dw(F32DwArgs& a, int layers, int splits, cudaStream_t st, int* launches) {
    *launches = 0;
    const long long steps = (a.rows + T - 1) / T;
    a.rows_per_split = (steps + splits - 1) / splits * T;
    a.splits = (int)((a.rows + a.rows_per_split - 1) / a.rows_per_split);   // no empty split
    const unsigned t = (unsigned)((a.d + T - 1) / T);
    cudaError_t e = launch_pdl(f32_dw_kernel, dim3(t, t, (unsigned)(layers * a.splits)),
                               dim3(T, 8), 0, st, a);
    if (e != cudaSuccess) return e;
    *launches = 1;
    if (a.splits == 1) return e;
    const size_t tot = 2 * (size_t)a.d * a.d + a.d;
    e = launch_pdl(f32_dw_reduce_kernel, dim3((unsigned)((tot + 255) / 256), (unsigned)layers),
                   dim3(256), 0, st, a);
    if (e == cudaSuccess) *launches = 2;
    return e;
}

// Output columns a lane of the one launch: two, which halves the reads of x a product,
// where one would take the rows in more than one pass (n = 16, 64 rows, graphs of four
// layers forward and backward: d = 112 82 us, two columns 58; 4,096 rows of d = 64 86 and
// 76; but one window of two rows and d = 64 23 and 27).
static int chain_cols(int d, int rows) {
    const int cols = (d + 31) / 32;
    return cols > 1 && rows > kChainRows * (8 / cols) ? 2 : 1;
}

// The windows a block of the one launch takes, one wave of blocks, where a layer costs
// it less than its own launch does.  Both sides in us a layer and direction, fitted to
// four layers forward and backward (graphs; us layer by layer, in one launch): n = 16,
// 64 rows: d = 16 35.6, 16.6; d = 32 36.2, 18.6; d = 64 52.7, 30.5; d = 91 67, 65; d = 96
// 67, 51; 1,024 rows of d = 91 77, 81.  4,096 rows: d = 32 44.4, 35.7; d = 64 128, 76;
// d = 96 235, 160.  n = 64, 64 rows: d = 32 36.1, 34.3; d = 48 52, 56; 4,096 rows of
// d = 64 122, 93.  n = 256: one window is too much for a block from d = 16 on (41, 80)
// unless there are many (64 windows of d = 48: 348, 295).
int f32_chain_rows(long long rows, int n, int d, int L, int sms) {
    if (L < 2 || L > kMaxF32Layers || d > 128) return 0;
    const long long windows = rows / n;
    const long long per = (windows + sms - 1) / sms;   // windows a block, one wave
    if (per * n > 4096) return 0;
    const int R = (int)(per * n);
    if (chain_floats(d, R, 2) * sizeof(float) > kChainSmem) return 0;
    const int cols = (d + 31) / 32, nc = chain_cols(d, R), groups = 8 / ((cols + nc - 1) / nc);
    const int passes = (R + kChainRows * groups - 1) / (kChainRows * groups);
    const double step = nc == 1 ? 0.17 * (cols * groups / 8.0) : 0.2;   // of four k
    double chain = passes * (0.5 + step * ((d + 3) / 4));
    if (d % 4) chain *= 1.5;   // weights copied 4 bytes at a time
    const double steps = (double)((rows + T - 1) / T) * cols * cols;   // of all tiles
    const double one = 1.05 * (1.8 + 1.75 * cols), many = 1.0 + 0.0185 * steps;
    return chain < (one > many ? one : many) ? R : 0;
}

template <bool BWD, int NC>
static cudaError_t launch_chain(const F32ChainArgs& a, cudaStream_t st) {
    static std::once_flag once[64];
    static cudaError_t set_err[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::call_once(once[dev], [&] {
        set_err[dev] = cudaFuncSetAttribute(f32_chain_kernel<BWD, NC>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)kChainSmem);
    });
    if (set_err[dev] != cudaSuccess) return set_err[dev];
    const unsigned grid = (unsigned)((a.rows + a.block_rows - 1) / a.block_rows);
    return launch_pdl(f32_chain_kernel<BWD, NC>, dim3(grid), dim3(256),
                      chain_floats(a.d, a.block_rows, a.stages) * sizeof(float), st, a);
}

cudaError_t launch_f32_chain(F32ChainArgs& a, bool bwd, cudaStream_t st) {
    a.vec = a.d % 4 == 0 && (reinterpret_cast<uintptr_t>(a.Ws) & 15) == 0 &&
            (reinterpret_cast<uintptr_t>(a.Wn) & 15) == 0 &&
            (reinterpret_cast<uintptr_t>(a.in) & 15) == 0 &&
            (reinterpret_cast<uintptr_t>(a.acts) & 15) == 0;
    const int pieces = a.vec ? a.d / 4 : a.d;
    a.lanes_log2 = 0;
    while ((1 << a.lanes_log2) < pieces) ++a.lanes_log2;
    a.stages = a.L > 2 && chain_floats(a.d, a.block_rows, 4) * sizeof(float) <= kChainSmem ? 4 : 2;
    if (chain_cols(a.d, a.block_rows) == 1)
        return bwd ? launch_chain<true, 1>(a, st) : launch_chain<false, 1>(a, st);
    return bwd ? launch_chain<true, 2>(a, st) : launch_chain<false, 2>(a, st);
}

cudaError_t launch_relu_grad_f32(const float* dy, const float* z, float* dz, size_t count,
                                 cudaStream_t st) {
    return launch_pdl(relu_grad_kernel<float>, dim3(blocks_for(count / 4, 256)), dim3(256), 0, st,
                      dy, z, dz, count);
}

cudaError_t launch_relu_grad_bf16(const __nv_bfloat16* dy, const __nv_bfloat16* z,
                                  __nv_bfloat16* dz, size_t count, cudaStream_t st) {
    return launch_pdl(relu_grad_kernel<__nv_bfloat16>, dim3(blocks_for(count / 8, 256)), dim3(256),
                      0, st, dy, z, dz, count);
}

size_t colsum_workspace_bytes(long long rows, int d) {
    const long long chunks = (rows + col_rows(rows) - 1) / col_rows(rows);
    return (size_t)(chunks < 1 ? 1 : chunks) * (size_t)d * sizeof(float);
}

static cudaError_t colsum(const __nv_bfloat16* dz, long long rows, int d, float* partial,
                          float* out, cudaStream_t st, int batch = 1) {
    const int crows = (int)col_rows(rows);
    const long long chunks = (rows + crows - 1) / crows;
    if (chunks == 0) {
        cudaError_t e = cudaMemsetAsync(out, 0, (size_t)batch * d * sizeof(float), st);
        return e;
    }
    dim3 grid((d / 8 + 63) / 64, (unsigned)chunks, (unsigned)batch);
    colsum_partial_kernel<<<grid, dim3(64, 4), 0, st>>>(dz, rows, d, crows, partial);
    colsum_final_kernel<<<dim3((d + 31) / 32, batch), 1024, 0, st>>>(partial, (int)chunks, d, out);
    return cudaGetLastError();
}

cudaError_t launch_colsum_bf16_batched(const __nv_bfloat16* dz, int batch, long long rows, int d,
                                       float* partial, float* out, cudaStream_t st) {
    return colsum(dz, rows, d, partial, out, st, batch);
}

cudaError_t launch_colsum_bf16(const __nv_bfloat16* dz, long long rows, int d, float* partial,
                               float* out, cudaStream_t st) {
    return colsum(dz, rows, d, partial, out, st);
}

cudaError_t launch_splitk_reduce(const float* partial, int splits_max, int splits_self,
                                 int splits_nbr, int d, float* dWs, float* dWn,
                                 cudaStream_t st, int layers, size_t part_stride,
                                 size_t out_stride, const float* bpart, float* dbias) {
    const size_t total4 = (size_t)d * d / 4;
    if (layers < 1) return cudaSuccess;
    const unsigned parts = (bpart && dbias) ? 3 : 2;
    return launch_pdl(splitk_reduce_kernel,
                      dim3((unsigned)((total4 + 63) / 64), parts, (unsigned)layers), dim3(64, 8), 0,
                      st, partial, splits_max, splits_self, splits_nbr, d, part_stride, dWs, dWn,
                      out_stride, bpart, dbias);
}

cudaError_t launch_shift_rows_bf16(const __nv_bfloat16* in, __nv_bfloat16* out, long long rows,
                                   int n, int d, int k, cudaStream_t st) {
    const int pieces = d / 8;   // d % 64 == 0 on the bf16 path
    shift_rows_kernel<<<blocks_for((size_t)rows * pieces, 256), 256, 0, st>>>(
        reinterpret_cast<const uint4*>(in), reinterpret_cast<uint4*>(out), rows, n, pieces, k);
    return cudaGetLastError();
}

cudaError_t launch_partner_table(int s, int n, unsigned flags, int* out, cudaStream_t st) {
    partner_table_kernel<<<(n + 255) / 256, 256, 0, st>>>(s, n, flags, out);
    return cudaGetLastError();
}

}  // namespace hcw
