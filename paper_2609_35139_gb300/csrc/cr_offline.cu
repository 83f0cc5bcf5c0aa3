// Offline preparation kernels (bandwidth-bound):
//   canon_kernel    chunk-cache canonicalisation, K^c_t = R_M(q_t)^{-1} K_t with
//                   V as stored (Sec. 4.1, "Chunk-cache preparation")
//   sigma_*_kernel  per-coordinate RMS statistics over corpus caches: sigma_stale
//                   from stale caches, sigma_Delta from joint - stale residual
//                   targets (Sec. 4.2, "Normalization and objective")
#include <cuda_bf16.h>

#include "cr_internal.h"
#include "cr_ptx.cuh"

namespace cr {
namespace {

struct Freq {
    float f[64];
};

__device__ __forceinline__ void load8(const uint16_t* p, float* v) {
    const uint4 w = *reinterpret_cast<const uint4*>(p);
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[2 * i] = __uint_as_float(u[i] << 16);
        v[2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
    }
}
__device__ __forceinline__ void load8(const float* p, float* v) {
    const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void store8(uint16_t* p, const float* v) {
    *reinterpret_cast<uint4*>(p) = make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]),
                                              pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
}
__device__ __forceinline__ void store8(float* p, const float* v) {
    reinterpret_cast<float4*>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
}

// One thread per (token, layer range, KV head, group of 8 rotation pairs): the 8 angles
// q_t * f_d are computed once and applied to that group in the head's K segment of each
// of the thread's layers (rotate-half pairs (d, d + d_h/2) inside each d_h-wide segment,
// by -q_t f_d: (a, b) -> (a cos + b sin, b cos - a sin)), one rounding to the cache dtype.
// With dir = -1 the sine changes sign and the rotation is by +q_t f_d, R_M itself (the
// stale cache's re-rotation of K to request positions, Sec. 2.2).  HBM-bound: the groups
// and heads of one layer are neighbouring lanes, so a warp reads and writes whole runs of
// a layer's K, and kSegs layers are loaded before any is rotated.  Measured with the
// assembly before it (3264 tokens of the 8B shape; the rotation reads and writes 0.43
// GB): 234 us with ranges of layers as neighbouring lanes and two segments in flight,
// 221 with four in flight, 211 in this order with four, 206 with eight.
constexpr int kSegs = 8;
template <typename T>
__global__ void __launch_bounds__(256) canon_kernel(T* kv, int64_t n, const int32_t* __restrict__ pos,
                                                    int L, int H, int dh, int parts_log2,
                                                    const __grid_constant__ Freq f, float dir) {
    pdl_launch_dependents();
    pdl_wait();
    const int groups = dh / 16;
    const int lanes = groups * H;   // threads of one (token, layer range)
    const int64_t D = static_cast<int64_t>(2) * L * H * dh;
    const int64_t layer = static_cast<int64_t>(2) * H * dh;
    const int parts = 1 << parts_log2;   // layer ranges
    const int64_t work = n * lanes * parts;
    for (int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; idx < work;
         idx += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t tp = idx / lanes;
        const int gh = static_cast<int>(idx - tp * lanes);
        const int64_t t = tp >> parts_log2;
        const int part = static_cast<int>(tp) & (parts - 1);
        const int h = gh / groups, g = gh - h * groups;
        const float q = static_cast<float>(__ldg(pos + t));
        float c[8], s[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            sincos_prod(q, f.f[g * 8 + i], &s[i], &c[i]);
            s[i] *= dir;
        }
        const int l1 = (part + 1) * L / parts;
        T* const first = kv + t * D + h * dh + g * 8;
        for (int l = part * L / parts; l < l1; l += kSegs) {
            float a[kSegs][8], b[kSegs][8];
#pragma unroll
            for (int u = 0; u < kSegs; ++u) {
                const T* p = first + (l + u < l1 ? l + u : l) * layer;
                load8(p, a[u]);
                load8(p + dh / 2, b[u]);
            }
#pragma unroll
            for (int u = 0; u < kSegs; ++u) {
                if (l + u >= l1) break;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float x = a[u][i], y = b[u][i];
                    a[u][i] = x * c[i] + y * s[i];
                    b[u][i] = y * c[i] - x * s[i];
                }
                T* p = first + (l + u) * layer;
                store8(p, a[u]);
                store8(p + dh / 2, b[u]);
            }
        }
    }
}

// The same where the layers are few: a thread's segments run over the heads, too, so that
// the angles, the larger part of the work there, are worked out once for four segments or
// so.  Lane p of a token's `step` takes every step-th of its L H segments (layer by layer),
// from the p-th.  us, by layer ranges / by segments: 20000 tokens of 1 layer of 8 heads 103 /
// 12, 30000 of 2 layers in fp32 25 / 8, 20000 of 4 layers of 2 heads in fp32 43 / 15; but 128
// tokens of the last 3.2 / 4.0.  Eight layers as one range instead of four: 24 -> 13 us (3000
// tokens, 8 heads).
constexpr int kFew = 4;   // segments in flight
template <typename T>
__global__ void __launch_bounds__(256) canon_few_kernel(T* kv, int64_t n, const int32_t* __restrict__ pos,
                                                        int L, int H, int dh, int step,
                                                        const __grid_constant__ Freq f, float dir) {
    pdl_launch_dependents();
    pdl_wait();
    const int groups = dh / 16;
    const int lanes = groups * step;
    const int layer = 2 * H * dh, all = L * H;
    const int64_t work = n * lanes;
    for (int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; idx < work;
         idx += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t t = idx / lanes;
        const int gp = static_cast<int>(idx - t * lanes);
        const int p = gp / groups, g = gp - p * groups;
        const float q = static_cast<float>(__ldg(pos + t));
        float c[8], s[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            sincos_prod(q, f.f[g * 8 + i], &s[i], &c[i]);
            s[i] *= dir;
        }
        T* const row = kv + t * L * layer + g * 8;
        int l = p / H, h = p - l * H;   // the next segment's layer and head
        for (int k = p; k < all; k += kFew * step) {
            T* seg[kFew];
            float a[kFew][8], b[kFew][8];
#pragma unroll
            for (int u = 0; u < kFew; ++u) {
                seg[u] = u == 0 || k + u * step < all ? row + l * layer + h * dh : seg[0];
                load8(seg[u], a[u]);
                load8(seg[u] + dh / 2, b[u]);
                for (h += step; h >= H; h -= H) ++l;
            }
#pragma unroll
            for (int u = 0; u < kFew; ++u) {
                if (k + u * step >= all) break;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float x = a[u][i], y = b[u][i];
                    a[u][i] = x * c[i] + y * s[i];
                    b[u][i] = y * c[i] - x * s[i];
                }
                store8(seg[u], a[u]);
                store8(seg[u] + dh / 2, b[u]);
            }
        }
    }
}

// Partial sums of squares: block (x, y) covers 8 THREADS coordinates (8 per thread)
// over the 64-token slice y; part[y][j].  With b, the squares of a - b.  HBM-bound:
// blocks of 128 threads leave less of the chip idle in the last round than 256 (5120
// tokens of the 7B shape against another cache, 0.59 GB: the statistic 142 -> 132 us),
// but two bf16 caches with rows of 128 KB or more stream unevenly in them at some lengths, and
// take 192 (the 8B shape, us, 256 / 128 / 192 threads: 4096 tokens 208 / 198 / 202, 5120
// 242 / 274 / 235, 7000 330 / 366 / 324, 12000 566 / 622 / 556).
template <typename T, int THREADS>
__global__ void __launch_bounds__(THREADS) sigma_partial_kernel(const T* __restrict__ a, const T* __restrict__ b,
                                                                int64_t n, int64_t D, float* __restrict__ part) {
    pdl_launch_dependents();
    pdl_wait();
    const int64_t col = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) * 8;
    if (col >= D) return;
    const int64_t t0 = static_cast<int64_t>(blockIdx.y) * kSigmaSlice;
    const int64_t t1 = t0 + kSigmaSlice < n ? t0 + kSigmaSlice : n;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    int64_t t = t0;
    // four rows in flight, added in row order (the sum's order is fixed)
    for (; t + 4 <= t1; t += 4) {
        float x[4][8];
#pragma unroll
        for (int u = 0; u < 4; ++u) load8(a + (t + u) * D + col, x[u]);
        if (b) {
            float y[4][8];
#pragma unroll
            for (int u = 0; u < 4; ++u) load8(b + (t + u) * D + col, y[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int i = 0; i < 8; ++i) x[u][i] -= y[u][i];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = fmaf(x[u][i], x[u][i], acc[i]);
    }
    for (; t < t1; ++t) {
        float x[8];
        load8(a + t * D + col, x);
        if (b) {
            float y[8];
            load8(b + t * D + col, y);
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] -= y[i];
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = fmaf(x[i], x[i], acc[i]);
    }
    store8(part + static_cast<int64_t>(blockIdx.y) * D + col, acc);
}

// sumsq[j] += sum over slices, in slice order (deterministic), in fp64.  A chain of loads:
// sixteen slices in flight and blocks of 64 threads, so that every SM has some (111 ->
// 107 us of the statistic above).
__global__ void __launch_bounds__(256) sigma_reduce_kernel(const float* __restrict__ part, int slices,
                                                           int64_t D, double* sumsq) {
    pdl_launch_dependents();
    pdl_wait();
    for (int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; j < D;
         j += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        // sixteen slices in flight, added in slice order
        double s = 0.0;
        const float* p = part + j;
        int k = 0;
        for (; k + 16 <= slices; k += 16) {
            float v[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) v[u] = p[(k + u) * D];
#pragma unroll
            for (int u = 0; u < 16; ++u) s += static_cast<double>(v[u]);
        }
        for (; k < slices; ++k) s += static_cast<double>(p[k * D]);
        sumsq[j] += s;
    }
}

__global__ void __launch_bounds__(256) sigma_finalize_kernel(const double* __restrict__ sumsq, int64_t D,
                                                             double inv_count, float* __restrict__ sigma) {
    pdl_launch_dependents();
    pdl_wait();
    for (int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; j < D;
         j += static_cast<int64_t>(gridDim.x) * blockDim.x)
        sigma[j] = static_cast<float>(sqrt(sumsq[j] * inv_count));
}

}  // namespace

cr_status launch_canonicalize(void* kv, bool f32, int64_t n, const int32_t* pos, int L, int H, int dh,
                              const float* inv_freq_host, cudaStream_t st, float dir) {
    if (n <= 0) return CR_OK;
    if (dh != 64 && dh != 128) return CR_ERR_UNSUPPORTED;
    Freq f{};
    for (int i = 0; i < dh / 2; ++i) f.f[i] = inv_freq_host[i];
    const int groups = dh / 16;
    const auto grid_of = [](int64_t work) {
        const int64_t blocks = std::min<int64_t>((work + 255) / 256, static_cast<int64_t>(num_sms()) * 16);
        return dim3(static_cast<unsigned>(blocks));
    };
    // Few layers: threads that share the angles over the heads, once they are two warps an SM
    // or more.  Fewer (and the angles' cost does not show) take a layer each.
    const int step = std::max(1, L * H / 4);
    if (L < kSegs && n * groups * step >= static_cast<int64_t>(num_sms()) * 64) {
        const dim3 grid = grid_of(n * groups * step);
        return f32 ? launch_pdl(canon_few_kernel<float>, grid, dim3(256), 0, st, static_cast<float*>(kv), n, pos, L, H,
                                dh, step, f, dir)
                   : launch_pdl(canon_few_kernel<uint16_t>, grid, dim3(256), 0, st, static_cast<uint16_t*>(kv), n, pos,
                                L, H, dh, step, f, dir);
    }
    // else ranges of at most eight layers or so a thread, four ranges at most
    const int parts_log2 = L < kSegs || L >= 20 ? 2 : (L >= 12 ? 1 : 0);
    const dim3 grid = grid_of((n * groups * H) << parts_log2);
    return f32 ? launch_pdl(canon_kernel<float>, grid, dim3(256), 0, st, static_cast<float*>(kv), n, pos, L, H, dh,
                            parts_log2, f, dir)
               : launch_pdl(canon_kernel<uint16_t>, grid, dim3(256), 0, st, static_cast<uint16_t*>(kv), n, pos, L, H,
                            dh, parts_log2, f, dir);
}

cr_status launch_sigma_accumulate(const void* a, const void* b, bool f32, int64_t n, int64_t D,
                                  float* part, double* sumsq, cudaStream_t st) {
    if (n <= 0) return CR_OK;
    const int64_t slices = (n + kSigmaSlice - 1) / kSigmaSlice;
    // (in shorter calls, below 2048 tokens of the 8B shape, latency counts and 128 are faster)
    const bool wide = b && !f32 && D >= 65536 && n * D >= (1 << 27);
    const int threads = wide ? 192 : 128;
    const dim3 grid(static_cast<unsigned>((D / 8 + threads - 1) / threads), static_cast<unsigned>(slices));
    cr_status s;
    if (f32)
        s = launch_pdl(sigma_partial_kernel<float, 128>, grid, dim3(threads), 0, st, static_cast<const float*>(a),
                       static_cast<const float*>(b), n, D, part);
    else
        s = launch_pdl(wide ? sigma_partial_kernel<uint16_t, 192> : sigma_partial_kernel<uint16_t, 128>, grid,
                       dim3(threads), 0, st, static_cast<const uint16_t*>(a), static_cast<const uint16_t*>(b), n, D,
                       part);
    if (s != CR_OK) return s;
    const int64_t blocks = (D + 63) / 64;
    return launch_pdl(sigma_reduce_kernel, dim3(static_cast<unsigned>(blocks)), dim3(64), 0, st,
                      static_cast<const float*>(part), static_cast<int>(slices), D, sumsq);
}

cr_status launch_sigma_finalize(const double* sumsq, int64_t D, int64_t count, float* sigma,
                                cudaStream_t st) {
    int64_t blocks = (D + 255) / 256;
    if (blocks > static_cast<int64_t>(num_sms()) * 8) blocks = static_cast<int64_t>(num_sms()) * 8;
    return launch_pdl(sigma_finalize_kernel, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, st, sumsq,
                      D, 1.0 / static_cast<double>(count), sigma);
}

}  // namespace cr
