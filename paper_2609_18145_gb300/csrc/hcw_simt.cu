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
// computes the weight and bias gradients of a whole stack (four layers forward and
// backward at 64 rows of d = 32: 24 launches, 127 us, now 10, 48 us; seven layers
// at 3,968 rows of d = 91, whose gradient blocks each walked all rows: 2,493 us,
// now 402).

// z[r][o] = sum_k Ws[o][k] x[r][k] + m_r sum_k Wn[o][k] x[p(r)][k] + bias[o]
// mout (optional): ReLU mask words [rows][ceil(d/32)], bit o%32 of word o/32 = (z > 0).
__global__ void __launch_bounds__(256)
    f32_fwd_kernel(const float* __restrict__ x, const float* __restrict__ Ws,
                   const float* __restrict__ Wn, const float* __restrict__ bias, int s, int n,
                   int d, long long rows, unsigned flags, float* __restrict__ y,
                   float* __restrict__ z, uint32_t* __restrict__ mout) {
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
    f32_dx_kernel(const float* __restrict__ dz, const float* __restrict__ dy,
                  const float* __restrict__ Ws, const float* __restrict__ Wn, int s, int n, int d,
                  long long rows, unsigned flags, float* __restrict__ dx,
                  const uint32_t* __restrict__ mprev, float* __restrict__ dz_prev) {
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
    const float* __restrict__ x = l == 0 ? A.x : A.acts + (l - 1) * A.act_elems;
    const float* __restrict__ dz = A.dz + l * A.act_elems;
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
    float as[4] = {0.f, 0.f, 0.f, 0.f}, an[4] = {0.f, 0.f, 0.f, 0.f}, cs = 0.f;
    load(rb);
    for (long long r0 = rb; r0 < re; r0 += T) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            gz[ty + 8 * q][tx] = g[q];
            xs[ty + 8 * q][tx] = a[q];
            xp[ty + 8 * q][tx] = b[q];
            cs += g[q];
        }
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
        // the eight row lanes' column sums, in order
        gz[ty][tx] = cs;
        __syncthreads();
        if (ty == 0 && o0 + tx < d) {
            float t = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) t += gz[q][tx];
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
    float t = 0.f;
#pragma unroll 8
    for (int sp = 0; sp < A.splits; ++sp) t += p[sp * tot];
    if (e < dd)
        A.dWs[l * dd + e] = t;
    else if (e < 2 * dd)
        A.dWn[l * dd + e - dd] = t;
    else
        A.dbias[(size_t)l * A.d + e - 2 * dd] = t;
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
    relu_grad_kernel(const V* __restrict__ dy, const V* __restrict__ z, V* __restrict__ dz,
                     size_t count) {
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
__global__ void relu_grad_mask_f32_kernel(const float* __restrict__ dy,
                                          const uint32_t* __restrict__ mask,
                                          float* __restrict__ dz, long long rows, int d) {
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
template <typename V>
__global__ void relu_grad_mask_kernel(const V* __restrict__ dy, const uint32_t* __restrict__ mask,
                                      V* __restrict__ dz, long long rows, int d) {
    constexpr int VEC = 16 / sizeof(V);
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
        if (VEC == 8) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                w[i] &= ((bits >> (2 * i)) & 1u ? 0x0000FFFFu : 0u) |
                        ((bits >> (2 * i + 1)) & 1u ? 0xFFFF0000u : 0u);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) w[i] = (bits >> i) & 1u ? w[i] : 0u;
        }
        reinterpret_cast<uint4*>(dz)[t] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// rows per partial of the column sum: 64 up to 65,536 rows (enough CTAs to
// fill the GPU), 256 above (the partials stay small)
inline long long col_rows(long long rows) { return rows <= 65536 ? 64 : 256; }

// partial[c][o] = sum_{r in chunk c} dz[r][o] for bf16 rows (d a multiple of 64),
// 16-byte loads.  Block: 64
// column groups of 16 bytes x 4 row lanes; each thread sums its group over every 4th row of
// the chunk, then the 4 row lanes are added in a fixed order.
template <typename V>
__global__ void colsum_partial_kernel(const V* __restrict__ dz, long long rows, int d, int crows,
                                      float* __restrict__ partial) {
    constexpr int VEC = 16 / sizeof(V);
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
            const V* e = reinterpret_cast<const V*>(&q);
#pragma unroll
            for (int i = 0; i < VEC; ++i) acc[i] += to_f(e[i]);
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
    const float* __restrict__ partial, int splits_max, int splits_self, int splits_nbr, int d,
    size_t part_stride, float* __restrict__ dWs, float* __restrict__ dWn, size_t out_stride,
    const float* __restrict__ bpart, float* __restrict__ dbias) {
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
    relu_grad_mask_kernel<__nv_bfloat16>
        <<<blocks_for((size_t)rows * d / 8, 256), 256, 0, st>>>(dy, mask, dz, rows, d);
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

template <typename V>
static cudaError_t colsum(const V* dz, long long rows, int d, float* partial, float* out,
                          cudaStream_t st, int batch = 1) {
    const int crows = (int)col_rows(rows);
    const long long chunks = (rows + crows - 1) / crows;
    if (chunks == 0) {
        cudaError_t e = cudaMemsetAsync(out, 0, (size_t)batch * d * sizeof(float), st);
        return e;
    }
    constexpr int VEC = 16 / sizeof(V);
    dim3 grid((d / VEC + 63) / 64, (unsigned)chunks, (unsigned)batch);
    colsum_partial_kernel<V><<<grid, dim3(64, 4), 0, st>>>(dz, rows, d, crows, partial);
    colsum_final_kernel<<<dim3((d + 31) / 32, batch), 1024, 0, st>>>(partial, (int)chunks, d, out);
    return cudaGetLastError();
}

cudaError_t launch_colsum_bf16_batched(const __nv_bfloat16* dz, int batch, long long rows, int d,
                                       float* partial, float* out, cudaStream_t st) {
    return colsum<__nv_bfloat16>(dz, rows, d, partial, out, st, batch);
}

cudaError_t launch_colsum_bf16(const __nv_bfloat16* dz, long long rows, int d, float* partial,
                               float* out, cudaStream_t st) {
    return colsum<__nv_bfloat16>(dz, rows, d, partial, out, st);
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
