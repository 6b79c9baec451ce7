// Shape-generic kernels of the verification step (fp32 or bf16 storage, fp32 arithmetic).
// They serve every shape the specialised sm_100a kernels do not cover (fp32 models, odd head
// sizes) and all the small element-wise steps between the projections.
#include <atomic>
#include <mutex>
#include <algorithm>
#include "trj_internal.h"
#include "timeline.cuh"

namespace trj {
namespace {

// Index checks: a cache row index that a device-held length or path would push outside the cache is never
// dereferenced: the access is skipped (one compare per row; the step's result is then unspecified, since the
// caller's contract seq_len[b] + rows <= max_seq is broken, but no memory outside the cache is touched and nothing
// traps).  The debug build (-DTRJ_DEBUG) also records which check fired in a flag word.
#ifdef TRJ_DEBUG
static __device__ int g_debug_flags;
#define TRJ_DEBUG_CHECK(ok, bit) ((ok) ? true : (atomicOr(&g_debug_flags, (bit)), false))
#else
#define TRJ_DEBUG_CHECK(ok, bit) (ok)
#endif
enum { DBG_ROPE_ROW = 1, DBG_COMPACT_ROW = 2, DBG_ATTENTION_LEN = 4 };

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// Activations that feed a projection keep (almost) fp32 precision in bf16 models: the value is
// stored as a bf16 pair hi + lo (lo = the rounding error of hi), which the projection adds back.
template <typename T>
__device__ __forceinline__ void store_split(T* hi, T* lo, size_t i, float v) {
    const T h = from_f<T>(v);
    hi[i] = h;
    if (lo) lo[i] = from_f<T>(v - to_f(h));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Sum of the split-K pieces of a projection result at flat index i (fixed order).
__device__ __forceinline__ float parts_at(const Parts& p, size_t i) {
    float v = p.ptr[i];
    for (int s = 1; s < p.splits; ++s) v += p.ptr[(size_t)s * p.stride + i];
    return v;
}
__device__ __forceinline__ float4 parts_at4(const Parts& p, size_t i4) {
    float4 v = reinterpret_cast<const float4*>(p.ptr)[i4];
    for (int s = 1; s < p.splits; ++s) {
        const float4 b = reinterpret_cast<const float4*>(p.ptr + (size_t)s * p.stride)[i4];
        v.x += b.x; v.y += b.y; v.z += b.z; v.w += b.w;
    }
    return v;
}

// Same for four consecutive values.  The pieces are requested BATCH at a time before any is added, so the
// loads overlap; the additions keep the order of the pieces.
template <int BATCH>
__device__ __forceinline__ float4 parts_at4_batched(const Parts& p, size_t i4) {
    float4 v = reinterpret_cast<const float4*>(p.ptr)[i4];
    for (int s0 = 1; s0 < p.splits; s0 += BATCH) {
        float4 b[BATCH];
#pragma unroll
        for (int j = 0; j < BATCH; ++j)
            if (s0 + j < p.splits) b[j] = reinterpret_cast<const float4*>(p.ptr + (size_t)(s0 + j) * p.stride)[i4];
#pragma unroll
        for (int j = 0; j < BATCH; ++j)
            if (s0 + j < p.splits) { v.x += b[j].x; v.y += b[j].y; v.z += b[j].z; v.w += b[j].w; }
    }
    return v;
}

// Sequence that owns a global row (B is small: linear scan of the offsets).
__device__ __forceinline__ int seq_of_row(const int32_t* row_off, int B, int row) {
    int b = 0;
    while (b + 1 < B && row >= row_off[b + 1]) ++b;
    return b;
}

// Sine and cosine of a rotary angle: formed in fp64 (positions reach thousands of radians) and reduced to [-pi, pi] there;
// sin/cos of the reduced angle in fp32 are then accurate to ~1e-7.
__device__ __forceinline__ void rotation(double ang, float& sn, float& cs) {
    const double red = ang - 6.283185307179586476925 * rint(ang * 0.15915494309189533577);
    sincosf((float)red, &sn, &cs);
}

// ---------------------------------------------------------------- embedding
// With a table (`rot`) it also works out, once per forward, what the rotary kernel of every layer needs of a row: the cosines
// and sines of its position and where its K/V rows go.
template <typename T>
__global__ void embed_kernel(const T* __restrict__ embed, const int32_t* __restrict__ tokens,
                             float* __restrict__ h, int d, const double* __restrict__ inv_freq, int half,
                             const int32_t* __restrict__ depth, const int32_t* __restrict__ seq_len,
                             const int32_t* __restrict__ row_off, int B, float* __restrict__ rot, int2* __restrict__ row_at) {
    pdl_wait();                                  // the chain's fence: everything enqueued earlier is complete
    pdl_launch_dependents();                     // before any later kernel of the chain may start
    TRJ_TL_DECL; TRJ_TL_BEGIN(TRJ_TL_EMBED);
    const int row = blockIdx.x;
    const T* src = embed + (size_t)tokens[row] * d;
    constexpr int VEC = 16 / (int)sizeof(T);                 // elements per 16-byte load
    if (d % VEC == 0 && ((uintptr_t)embed % 16) == 0 && ((uintptr_t)h % 16) == 0) {
        // the table's rows are cold in HBM: few wide loads per thread, all in flight at once
        for (int c = threadIdx.x * VEC; c < d; c += blockDim.x * VEC) {
            const uint4 raw = *reinterpret_cast<const uint4*>(src + c);
            const T* e = reinterpret_cast<const T*>(&raw);
            float out[VEC];
#pragma unroll
            for (int i = 0; i < VEC; ++i) out[i] = to_f(e[i]);
#pragma unroll
            for (int i = 0; i < VEC; i += 4)
                *reinterpret_cast<float4*>(h + (size_t)row * d + c + i) = make_float4(out[i], out[i + 1], out[i + 2], out[i + 3]);
        }
    } else {
        for (int c = threadIdx.x; c < d; c += blockDim.x) h[(size_t)row * d + c] = to_f(src[c]);
    }
    if (rot) {
        const int b = seq_of_row(row_off, B, row);
        const int len = seq_len[b];
        for (int i = threadIdx.x; i < half; i += blockDim.x) {
            float sn, cs;
            rotation((double)(len + depth[row]) * inv_freq[i], sn, cs);
            rot[(size_t)row * 2 * half + i] = cs;
            rot[(size_t)row * 2 * half + half + i] = sn;
        }
        if (threadIdx.x == 0) row_at[row] = make_int2(b, len + row - row_off[b]);
    }
    TRJ_TL_END(TRJ_TL_EMBED);
}

// ---------------------------------------------------------------- residual add + RMSNorm
// One CTA per row.  h += add (summing the split-K pieces of `add` on the way), x = rmsnorm(h) * gain.
// Fast path: d % 4 == 0 and d <= RMS_MAX_D; the row lives in registers between the two phases.  Up to one row per SM a
// row takes 1024 threads, for many loads in flight (the row and its split-K pieces come from L2); more rows take 256 threads
// each, so that eight CTAs share an SM and one's barriers overlap the others' loads (1024 rows of 4096: 22.5 -> 11.6 us, 64 MB
// from and to L2; 320 rows with two pieces 8.6 -> 7.0 us).
constexpr int RMS_MAX_D = 8192;
constexpr int RMS_FEW_ROWS = 148, RMS_FEW_ROWS_THREADS = 1024;

__device__ __forceinline__ float block_sum(float v, float* red) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        float t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
        t = warp_sum(t);
        if (threadIdx.x == 0) red[0] = t;
    }
    __syncthreads();
    return red[0];
}

template <typename T>
__device__ __forceinline__ void store_split4(T* hi, T* lo, size_t i, float4 v);
template <>
__device__ __forceinline__ void store_split4<float>(float* hi, float*, size_t i, float4 v) {
    *reinterpret_cast<float4*>(hi + i) = v;
}
template <>
__device__ __forceinline__ void store_split4<__nv_bfloat16>(__nv_bfloat16* hi, __nv_bfloat16* lo, size_t i, float4 v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    uint2 pk;
    pk.x = *reinterpret_cast<const uint32_t*>(&a); pk.y = *reinterpret_cast<const uint32_t*>(&b);
    *reinterpret_cast<uint2*>(hi + i) = pk;
    if (lo) {
        const __nv_bfloat162 c = __floats2bfloat162_rn(v.x - __low2float(a), v.y - __high2float(a));
        const __nv_bfloat162 e = __floats2bfloat162_rn(v.z - __low2float(b), v.w - __high2float(b));
        pk.x = *reinterpret_cast<const uint32_t*>(&c); pk.y = *reinterpret_cast<const uint32_t*>(&e);
        *reinterpret_cast<uint2*>(lo + i) = pk;
    }
}

template <typename T, int THREADS, int CHUNKS>
__global__ void __launch_bounds__(THREADS) add_rmsnorm_vec_kernel(float* __restrict__ h, const Parts add,
                                                                 const float* __restrict__ gain, T* __restrict__ x,
                                                                 T* __restrict__ x_lo, int d, float eps) {
    pdl_prologue();
    TRJ_TL_DECL; TRJ_TL_BEGIN(TRJ_TL_RMSNORM);
    __shared__ float red[32];
    const int row = blockIdx.x, n4 = d >> 2;
    float4 v[CHUNKS];
    float ss = 0.f;
    if constexpr (THREADS == RMS_FEW_ROWS_THREADS) {
        // one load after the other: requesting them together makes this kernel faster (4.0 -> 3.7 us) and the step it sits
        // in slower (33 rows 3.13 -> 3.15 ms): the next projection's weight ring is filling at the same time
#pragma unroll
        for (int k = 0; k < CHUNKS; ++k) {
            const int j = threadIdx.x + k * THREADS;
            if (j < n4) {
                v[k] = reinterpret_cast<const float4*>(h + (size_t)row * d)[j];
                if (add.ptr) {
                    const float4 a = parts_at4(add, (size_t)row * n4 + j);
                    v[k].x += a.x; v[k].y += a.y; v[k].z += a.z; v[k].w += a.w;
                    reinterpret_cast<float4*>(h + (size_t)row * d)[j] = v[k];
                }
                ss += v[k].x * v[k].x + v[k].y * v[k].y + v[k].z * v[k].z + v[k].w * v[k].w;
            }
        }
    } else {
        float4 a[CHUNKS];
#pragma unroll
        for (int k = 0; k < CHUNKS; ++k) {
            const int j = threadIdx.x + k * THREADS;
            if (j < n4) v[k] = reinterpret_cast<const float4*>(h + (size_t)row * d)[j];
        }
        if (add.ptr) {
#pragma unroll
            for (int k = 0; k < CHUNKS; ++k) {
                const int j = threadIdx.x + k * THREADS;
                if (j < n4) a[k] = parts_at4(add, (size_t)row * n4 + j);
            }
#pragma unroll
            for (int k = 0; k < CHUNKS; ++k) {
                const int j = threadIdx.x + k * THREADS;
                if (j < n4) {
                    v[k].x += a[k].x; v[k].y += a[k].y; v[k].z += a[k].z; v[k].w += a[k].w;
                    reinterpret_cast<float4*>(h + (size_t)row * d)[j] = v[k];
                }
            }
        }
#pragma unroll
        for (int k = 0; k < CHUNKS; ++k)
            if (threadIdx.x + k * THREADS < n4) ss += v[k].x * v[k].x + v[k].y * v[k].y + v[k].z * v[k].z + v[k].w * v[k].w;
    }
    const float inv = rsqrtf(block_sum(ss, red) / (float)d + eps);
#pragma unroll
    for (int k = 0; k < CHUNKS; ++k) {
        const int j = threadIdx.x + k * THREADS;
        if (j < n4) {
            const float4 g = reinterpret_cast<const float4*>(gain)[j];
            store_split4<T>(x, x_lo, (size_t)row * d + 4 * j,
                            make_float4(v[k].x * inv * g.x, v[k].y * inv * g.y, v[k].z * inv * g.z, v[k].w * inv * g.w));
        }
    }
#ifdef TRJ_TIMELINE
    __syncthreads();
#endif
    TRJ_TL_END(TRJ_TL_RMSNORM);
}

template <typename T>
__global__ void add_rmsnorm_kernel(float* __restrict__ h, const Parts add,
                                   const float* __restrict__ gain, T* __restrict__ x, T* __restrict__ x_lo,
                                   int d, float eps) {
    pdl_prologue();
    __shared__ float red[32];
    const int row = blockIdx.x;
    float* hr = h + (size_t)row * d;
    float ss = 0.f;
    for (int c = threadIdx.x; c < d; c += blockDim.x) {
        float v = hr[c];
        if (add.ptr) { v += parts_at(add, (size_t)row * d + c); hr[c] = v; }
        ss += v * v;
    }
    const float inv = rsqrtf(block_sum(ss, red) / (float)d + eps);
    for (int c = threadIdx.x; c < d; c += blockDim.x) store_split(x, x_lo, (size_t)row * d + c, hr[c] * inv * gain[c]);
}

// ---------------------------------------------------------------- plain tiled GEMM
// y[M][N] = (x + x_lo)[M][K] . w[N][K]^T ; 64x64 tile, 16-deep slices, 4x4 outputs per thread.
template <typename T>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const T* __restrict__ x, const T* __restrict__ x_lo,
                                                        const T* __restrict__ w, float* __restrict__ y,
                                                        int M, int N, int K) {
    constexpr int BM = 64, BN = 64, BK = 16;
    __shared__ float xs[BK][BM + 4];
    __shared__ float ws[BK][BN + 4];
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int lr = tid >> 2, lk = (tid & 3) * 4;          // this thread stages row lr, k-slice lk..lk+3
    float acc[4][4] = {};
    for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = k0 + lk + i;
            const int xm = m0 + lr, wn = n0 + lr;
            float xv = 0.f;
            if (xm < M && k < K) {
                xv = to_f(x[(size_t)xm * K + k]);
                if (x_lo) xv += to_f(x_lo[(size_t)xm * K + k]);
            }
            xs[lk + i][lr] = xv;
            ws[lk + i][lr] = (wn < N && k < K) ? to_f(w[(size_t)wn * K + k]) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { a[i] = xs[kk][ty * 4 + i]; b[i] = ws[kk][tx * 4 + i]; }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tx * 4 + j;
            if (n < N) y[(size_t)m * N + n] = acc[i][j];
        }
    }
}

// ---------------------------------------------------------------- fp32 GEMM of few tiles
// y[M][N] = x[M][K] . w[N][K]^T in fp32 for products so small that their latency is all that counts: a CTA takes 16 rows x 8
// columns, so that even N = 256 gives 32 CTAs (the 64 x 64 tiles above give 4, each a serial loop of K / 16 slices with two
// barriers and a trip to L2 per slice), and its eight warps split K.  The weight rows go to shared memory ahead of the wait
// for the previous kernel, the activations after it, all of them requested at once: one trip to L2 in all.  The warps'
// sums are added in a fixed order.  11 x 1376 x 256: 16.1 -> 3.2 us per launch (back to back in a graph).
constexpr int SF_ROWS = 16, SF_COLS = 8, SF_THREADS = 256, SF_WARPS = SF_THREADS / 32;
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ float4 silu_mul(const float4& g, const float4& u) {
    return make_float4(g.x / (1.f + expf(-g.x)) * u.x, g.y / (1.f + expf(-g.y)) * u.y,
                       g.z / (1.f + expf(-g.z)) * u.z, g.w / (1.f + expf(-g.w)) * u.w);
}
// What precedes a projection of the decoder can be its input: every CTA works the few rows out for itself (residual + RMSNorm,
// or SwiGLU) while they pass into shared memory, which costs less than a kernel of its own in a chain that launches bound:
// a step of the tiny decoder (2 layers of 256, 11 rows) has 7 of 23 launches less, 93.0 -> 83.1 us.  All loads of a thread come
// before their first use; row by row and chunk by chunk they made it 102.7 us.  The CTAs of the first columns keep the
// residual stream, in another buffer, since the rest still read the old one.
enum { SF_PLAIN = SmallF32Input::PLAIN, SF_NORM = SmallF32Input::NORM, SF_SWIGLU = SmallF32Input::SWIGLU };
constexpr int SF_MAX_K = 1024;
template <int IN, int CHUNKS>                // CHUNKS: float4 of a row per lane, K <= 128 CHUNKS
__global__ void __launch_bounds__(SF_THREADS) gemm_small_f32_kernel(const SmallF32Input in, const float* __restrict__ w,
                                                                    float* __restrict__ y, int M, int N, int K) {
    extern __shared__ __align__(16) float sf_smem[];
    __shared__ float red[SF_WARPS][SF_ROWS * SF_COLS];
    const int stride = K + 4, k4 = K >> 2;
    float* ws = sf_smem;                                     // [SF_COLS][stride]
    float* xs = sf_smem + SF_COLS * stride;                  // [SF_ROWS][stride]
    const int n0 = blockIdx.x * SF_COLS, m0 = blockIdx.y * SF_ROWS;
    const int n_cols = min(SF_COLS, N - n0), n_rows = min(SF_ROWS, M - m0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pdl_launch_dependents();
    for (int c = warp; c < n_cols; c += SF_WARPS)
        for (int i = lane; i < k4; i += 32) cp_async16(ws + c * stride + 4 * i, w + (size_t)(n0 + c) * K + 4 * i);
    float4 gain[IN == SF_NORM ? CHUNKS : 1];
    if constexpr (IN == SF_NORM) {
#pragma unroll
        for (int t = 0; t < CHUNKS; ++t)
            if (lane + 32 * t < k4) gain[t] = reinterpret_cast<const float4*>(in.gain)[lane + 32 * t];
    }
    pdl_wait();
    if constexpr (IN == SF_PLAIN) {
        for (int r = warp; r < n_rows; r += SF_WARPS)
            for (int i = lane; i < k4; i += 32) cp_async16(xs + r * stride + 4 * i, in.x + (size_t)(m0 + r) * K + 4 * i);
    } else {
        // rows warp and warp + 8, everything of both requested before any of it is used
        constexpr int ROWS = SF_ROWS / SF_WARPS;
        const float4* src = reinterpret_cast<const float4*>(in.x) + (size_t)m0 * k4 * (IN == SF_SWIGLU ? 2 : 1);
        const float4* add = reinterpret_cast<const float4*>(in.add) + (size_t)m0 * k4;
        float4 v[ROWS][CHUNKS], a[ROWS][CHUNKS];
#pragma unroll
        for (int t = 0; t < CHUNKS; ++t) {
            const int i = lane + 32 * t;
#pragma unroll
            for (int e = 0; e < ROWS; ++e) {
                const int r = warp + SF_WARPS * e;
                v[e][t] = a[e][t] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (i >= k4 || r >= n_rows) continue;
                if constexpr (IN == SF_SWIGLU) {
                    v[e][t] = src[(size_t)r * 2 * k4 + i];
                    a[e][t] = src[(size_t)r * 2 * k4 + k4 + i];
                } else {
                    v[e][t] = src[(size_t)r * k4 + i];
                    if (in.add) a[e][t] = add[(size_t)r * k4 + i];
                }
            }
        }
#pragma unroll
        for (int e = 0; e < ROWS; ++e) {
            const int r = warp + SF_WARPS * e;
            if (r >= n_rows) break;
            float inv = 0.f;
            if constexpr (IN == SF_NORM) {
                float ss = 0.f;
#pragma unroll
                for (int t = 0; t < CHUNKS; ++t) {
                    float4& h = v[e][t];
                    h.x += a[e][t].x; h.y += a[e][t].y; h.z += a[e][t].z; h.w += a[e][t].w;
                    ss += h.x * h.x + h.y * h.y + h.z * h.z + h.w * h.w;
                }
                inv = rsqrtf(warp_sum(ss) / (float)K + in.eps);
            }
#pragma unroll
            for (int t = 0; t < CHUNKS; ++t) {
                const int i = lane + 32 * t;
                if (i >= k4) break;
                const float4 h = v[e][t];
                if constexpr (IN == SF_NORM) {
                    if (in.h_out && blockIdx.x == 0) reinterpret_cast<float4*>(in.h_out)[(size_t)(m0 + r) * k4 + i] = h;
                    *reinterpret_cast<float4*>(xs + r * stride + 4 * i) =
                        make_float4(h.x * inv * gain[t].x, h.y * inv * gain[t].y, h.z * inv * gain[t].z, h.w * inv * gain[t].w);
                } else {
                    *reinterpret_cast<float4*>(xs + r * stride + 4 * i) = silu_mul(h, a[e][t]);
                }
            }
        }
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    // a lane owns rows r, r + 8 and columns c, c + 4; rows and columns past the end read whatever is there and are not stored
    const int r = lane >> 2, c = lane & 3;
    float acc[2][2] = {};
    for (int i = warp; i < k4; i += SF_WARPS) {
        float4 a[2], b[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            a[e] = *reinterpret_cast<const float4*>(xs + (r + 8 * e) * stride + 4 * i);
            b[e] = *reinterpret_cast<const float4*>(ws + (c + 4 * e) * stride + 4 * i);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int f = 0; f < 2; ++f)
                acc[e][f] = fmaf(a[e].w, b[f].w, fmaf(a[e].z, b[f].z, fmaf(a[e].y, b[f].y, fmaf(a[e].x, b[f].x, acc[e][f]))));
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int f = 0; f < 2; ++f) red[warp][(r + 8 * e) * SF_COLS + c + 4 * f] = acc[e][f];
    __syncthreads();
    if (threadIdx.x < SF_ROWS * SF_COLS) {
        const int row = threadIdx.x / SF_COLS, col = threadIdx.x % SF_COLS;
        float v = 0.f;
#pragma unroll
        for (int g = 0; g < SF_WARPS; ++g) v += red[g][threadIdx.x];
        if (row < n_rows && col < n_cols) y[(size_t)(m0 + row) * N + n0 + col] = v;
    }
}

// ---------------------------------------------------------------- rotary embedding + K/V append
// Two kernels, both bound by the chain of loads and not by bytes.  Few rows: a thread takes a head's q, k and v (18 loads of
// split-K pieces in flight) in a few fat CTAs, and works out its rotations ahead of the wait, where they cost nothing.  Many
// rows: each layer and head working out the same rotations again does cost (1024 rows of the 7B shape: 45 us a layer), so the
// embedding kernel leaves them in a table and a thread takes one head of q, k or v (26 us).  At 33 rows the table is the slower
// way: 3.18 against 3.15 ms a step, its loads come after the wait.
constexpr int ROPE_THREADS = 256;           // 16 heads of 128 dimensions
constexpr int ROPE_FEW_ROWS = 148;
// Four consecutive dimensions and the four they are rotated with per thread (head_dim / 2 a multiple of 4): 16-byte loads of
// the projection pieces, 8-byte (bf16) or 16-byte (fp32) stores.  One CTA covers heads_per_cta heads of a row.
template <typename T>
__global__ void __launch_bounds__(ROPE_THREADS) rope_kv_write_few_kernel(const Parts qkv, const double* __restrict__ inv_freq,
                                         const int32_t* __restrict__ depth, const int32_t* __restrict__ seq_len,
                                         const int32_t* __restrict__ row_off, int B, T* __restrict__ q_out,
                                         T* __restrict__ k_slab, T* __restrict__ v_slab, int H, int Hkv, int D, int max_seq,
                                         int heads_per_cta) {
    pdl_launch_dependents();
    // geometry and rotations do not depend on the projection: have them ready before waiting for it
    const int half = D >> 1, HD = H * D, KD = Hkv * D, per_head = half >> 2;
    const int row = blockIdx.x, hh = blockIdx.y * heads_per_cta + (int)threadIdx.x / per_head;
    const int i = ((int)threadIdx.x % per_head) * 4;
    TRJ_TL_DECL;
    if (hh >= H) return;                                     // never thread 0: a CTA's first thread has a head
    const int b = seq_of_row(row_off, B, row);
    const int local = row - row_off[b];
    const int pos = seq_len[b] + depth[row];
    const bool has_kv = hh < Hkv;                            // this thread also handles K/V head hh
    const int n_e = has_kv ? 6 : 2;
    const size_t src = (size_t)row * (HD + 2 * KD) + hh * D + i;    // flat index of query head hh in the projection result
    const size_t cache_at = (((size_t)b * Hkv + hh) * max_seq + seq_len[b] + local) * D + i;
    const size_t q_at = (size_t)row * HD + hh * D + i;
    float sn[4], cs[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        rotation((double)pos * inv_freq[i + e], sn[e], cs[e]);
    }
    pdl_wait();
    TRJ_TL_BEGIN(TRJ_TL_ROPE);
    float4 acc[6];                                           // q, k, v: first and second half of the head
#pragma unroll
    for (int e = 0; e < 6; ++e) acc[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    // the pieces are requested three at a time (18 loads in flight) and added in ascending order
    for (int s0 = 0; s0 < qkv.splits; s0 += 3) {
        float4 t[3][6];
#pragma unroll
        for (int j = 0; j < 3; ++j)
            if (s0 + j < qkv.splits) {
                const float* piece = qkv.ptr + (size_t)(s0 + j) * qkv.stride + src;
#pragma unroll
                for (int e = 0; e < 6; ++e)                  // q at 0, k at HD, v at HD + KD; first and second half of the head
                    if (e < n_e) t[j][e] = *reinterpret_cast<const float4*>(piece + (e >> 1 == 0 ? 0 : e >> 1 == 1 ? HD : HD + KD) + (e & 1) * half);
            }
#pragma unroll
        for (int j = 0; j < 3; ++j)
            if (s0 + j < qkv.splits) {
#pragma unroll
                for (int e = 0; e < 6; ++e)
                    if (e < n_e) { acc[e].x += t[j][e].x; acc[e].y += t[j][e].y; acc[e].z += t[j][e].z; acc[e].w += t[j][e].w; }
            }
    }
    auto rot_lo = [&](const float4& a, const float4& bb) {
        return make_float4(a.x * cs[0] - bb.x * sn[0], a.y * cs[1] - bb.y * sn[1], a.z * cs[2] - bb.z * sn[2], a.w * cs[3] - bb.w * sn[3]);
    };
    auto rot_hi = [&](const float4& a, const float4& bb) {
        return make_float4(bb.x * cs[0] + a.x * sn[0], bb.y * cs[1] + a.y * sn[1], bb.z * cs[2] + a.z * sn[2], bb.w * cs[3] + a.w * sn[3]);
    };
    store_split4<T>(q_out, nullptr, q_at, rot_lo(acc[0], acc[1]));
    store_split4<T>(q_out, nullptr, q_at + half, rot_hi(acc[0], acc[1]));
    if (has_kv && TRJ_DEBUG_CHECK((unsigned)(seq_len[b] + local) < (unsigned)max_seq, DBG_ROPE_ROW)) {
        store_split4<T>(k_slab, nullptr, cache_at, rot_lo(acc[2], acc[3]));
        store_split4<T>(k_slab, nullptr, cache_at + half, rot_hi(acc[2], acc[3]));
        store_split4<T>(v_slab, nullptr, cache_at, acc[4]);
        store_split4<T>(v_slab, nullptr, cache_at + half, acc[5]);
    }
    TRJ_TL_END(TRJ_TL_ROPE);                                 // thread 0's own stores; the others' end within the same few hundred ns
}

// The same with the rows' table: heads are those of the projection result, H of q, Hkv of k, Hkv of v (only moved).
template <typename T, int BATCH>            // BATCH: split-K pieces requested at a time
__global__ void __launch_bounds__(ROPE_THREADS) rope_kv_write_kernel(const Parts qkv, const float* __restrict__ rot, const int2* __restrict__ row_at,
                                         T* __restrict__ q_out, T* __restrict__ k_slab, T* __restrict__ v_slab, int H, int Hkv, int D, int max_seq) {
    pdl_launch_dependents();
    const int half = D >> 1, per_head = half >> 2, heads = H + 2 * Hkv;
    const int row = blockIdx.x, hh = (int)(blockIdx.y * ROPE_THREADS + threadIdx.x) / per_head;
    const int i = ((int)threadIdx.x % per_head) * 4;
    TRJ_TL_DECL;
    if (hh >= heads) return;                                 // never thread 0: a CTA's first thread has a head
    const float* src = qkv.ptr + ((size_t)row * heads + hh) * D + i;
    pdl_wait();
    TRJ_TL_BEGIN(TRJ_TL_ROPE);
    const float4 cs = *reinterpret_cast<const float4*>(rot + (size_t)row * D + i), sn = *reinterpret_cast<const float4*>(rot + (size_t)row * D + half + i);
    const int2 at = row_at[row];
    float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
    for (int s0 = 0; s0 < qkv.splits; s0 += BATCH) {         // added in ascending order
        float4 a[BATCH], b[BATCH];
#pragma unroll
        for (int j = 0; j < BATCH; ++j)
            if (s0 + j < qkv.splits) {
                const float* piece = src + (size_t)(s0 + j) * qkv.stride;
                a[j] = *reinterpret_cast<const float4*>(piece);
                b[j] = *reinterpret_cast<const float4*>(piece + half);
            }
#pragma unroll
        for (int j = 0; j < BATCH; ++j)
            if (s0 + j < qkv.splits) {
                lo.x += a[j].x; lo.y += a[j].y; lo.z += a[j].z; lo.w += a[j].w;
                hi.x += b[j].x; hi.y += b[j].y; hi.z += b[j].z; hi.w += b[j].w;
            }
    }
    if (hh < H + Hkv) {
        const float4 l = lo, h = hi;
        lo = make_float4(l.x * cs.x - h.x * sn.x, l.y * cs.y - h.y * sn.y, l.z * cs.z - h.z * sn.z, l.w * cs.w - h.w * sn.w);
        hi = make_float4(h.x * cs.x + l.x * sn.x, h.y * cs.y + l.y * sn.y, h.z * cs.z + l.z * sn.z, h.w * cs.w + l.w * sn.w);
    }
    T* dst;
    size_t to;
    if (hh < H) {
        dst = q_out; to = ((size_t)row * H + hh) * D + i;
    } else {
        dst = hh < H + Hkv ? k_slab : v_slab;
        to = (((size_t)at.x * Hkv + (hh < H + Hkv ? hh - H : hh - H - Hkv)) * max_seq + at.y) * D + i;
        if (!TRJ_DEBUG_CHECK((unsigned)at.y < (unsigned)max_seq, DBG_ROPE_ROW)) return;
    }
    store_split4<T>(dst, nullptr, to, lo);
    store_split4<T>(dst, nullptr, to + half, hi);
    TRJ_TL_END(TRJ_TL_ROPE);                                 // thread 0's own stores; the others' end within the same few hundred ns
}

// ---------------------------------------------------------------- tree attention, one CTA per (row, head)
// 4 warps split the keys; inside a warp every lane scores one key of a 32-key chunk, the chunk's
// statistics are merged with an online softmax, and P.V is accumulated with lanes spread over D.
template <typename T, int D>
__global__ void __launch_bounds__(128) tree_attention_generic_kernel(
        const T* __restrict__ q, const T* __restrict__ k_slab, const T* __restrict__ v_slab,
        const uint64_t* __restrict__ anc, int anc_words, const int32_t* __restrict__ seq_len,
        const int32_t* __restrict__ row_off, int B, int H, int Hkv, int max_seq, T* __restrict__ out, T* __restrict__ out_lo,
        int shared_cache) {
    constexpr int PER = D / 32;                  // output dims per lane
    constexpr int VEC = 16 / (int)sizeof(T);     // elements per 16-byte load
    pdl_prologue();
    __shared__ float qs[D];
    __shared__ float part_m[4], part_l[4];
    __shared__ float part_acc[4][D];
    const int row = blockIdx.x, hh = blockIdx.y;
    const int b = seq_of_row(row_off, B, row);
    const int S = min(max(seq_len[b], 0), max_seq);      // a length outside the cache reads nothing outside it
    const int rows_b = row_off[b + 1] - row_off[b];
    const int total = TRJ_DEBUG_CHECK(seq_len[b] >= 0 && S + rows_b <= max_seq, DBG_ATTENTION_LEN) ? S + rows_b : min(S + rows_b, max_seq);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kvh = hh / (H / Hkv);              // grouped-query attention: the K/V head of this query head
    const int cb = shared_cache ? 0 : b;         // pieces of one prompt chunk share the cache of sequence 0
    const T* kb = k_slab + ((size_t)cb * Hkv + kvh) * max_seq * D;
    const T* vb = v_slab + ((size_t)cb * Hkv + kvh) * max_seq * D;
    const uint64_t* mask = anc + (size_t)row * anc_words;
    for (int c = threadIdx.x; c < D; c += blockDim.x) qs[c] = to_f(q[((size_t)row * H + hh) * D + c]);
    __syncthreads();
    const float scale = rsqrtf((float)D);
    float m_run = -INFINITY, l_run = 0.f, acc[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) acc[i] = 0.f;
    for (int base = warp * 32; base < total; base += 128) {
        const int j = base + lane;
        bool vis = j < total;
        if (vis && j >= S) { const int t = j - S; vis = (mask[t >> 6] >> (t & 63)) & 1ull; }
        float s = -INFINITY;
        if (vis) {
            // the key's row in 16-byte loads, all in flight at once (a row is a multiple of 128 bytes)
            const uint4* kr = reinterpret_cast<const uint4*>(kb + (size_t)j * D);
            float dot = 0.f;
#pragma unroll
            for (int c0 = 0; c0 < D / VEC; c0 += 16) {
                uint4 raw[16];
#pragma unroll
                for (int c = 0; c < 16; ++c) if (c0 + c < D / VEC) raw[c] = kr[c0 + c];
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    if (c0 + c >= D / VEC) continue;
                    const T* e = reinterpret_cast<const T*>(&raw[c]);
#pragma unroll
                    for (int i = 0; i < VEC; ++i) dot = fmaf(qs[(c0 + c) * VEC + i], to_f(e[i]), dot);
                }
            }
            s = dot * scale;
        }
        const float cmax = warp_max(s);
        if (cmax == -INFINITY) continue;          // whole chunk masked (warp-uniform)
        const float m_new = fmaxf(m_run, cmax);
        const float corr = (m_run == -INFINITY) ? 0.f : expf(m_run - m_new);
        const float p = vis ? expf(s - m_new) : 0.f;
        l_run = l_run * corr + warp_sum(p);
#pragma unroll
        for (int i = 0; i < PER; ++i) acc[i] *= corr;
        const int nk = min(32, total - base);
        for (int j0 = 0; j0 < nk; j0 += 8) {      // eight rows of V in flight; a masked key's row (which may hold anything) is not read
            float v[8][PER], pj[8];
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
                pj[jj] = __shfl_sync(0xffffffffu, p, j0 + jj);        // 0 past nk
                const T* vr = vb + (size_t)(base + j0 + jj) * D + lane * PER;
#pragma unroll
                for (int i = 0; i < PER; ++i) v[jj][i] = pj[jj] != 0.f ? to_f(vr[i]) : 0.f;
            }
#pragma unroll
            for (int jj = 0; jj < 8; ++jj)
#pragma unroll
                for (int i = 0; i < PER; ++i) acc[i] = fmaf(pj[jj], v[jj][i], acc[i]);
        }
        m_run = m_new;
    }
    if (lane == 0) { part_m[warp] = m_run; part_l[warp] = l_run; }
#pragma unroll
    for (int i = 0; i < PER; ++i) part_acc[warp][lane * PER + i] = acc[i];
    __syncthreads();
    const float m_all = fmaxf(fmaxf(part_m[0], part_m[1]), fmaxf(part_m[2], part_m[3]));
    for (int c = threadIdx.x; c < D; c += blockDim.x) {
        float l = 0.f, o = 0.f;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const float f = (part_m[w] == -INFINITY) ? 0.f : expf(part_m[w] - m_all);
            l += part_l[w] * f;
            o += part_acc[w][c] * f;
        }
        store_split(out, out_lo, ((size_t)row * H + hh) * D + c, o / l);
    }
}

// ---------------------------------------------------------------- SwiGLU
template <typename T>
__global__ void swiglu_kernel(const Parts gu, T* __restrict__ act, T* __restrict__ act_lo,
                              int rows, int f) {
    pdl_prologue();
    const size_t n = (size_t)rows * f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / f, c = i % f;
        const float g = parts_at(gu, r * 2 * f + c), u = parts_at(gu, r * 2 * f + f + c);
        store_split(act, act_lo, i, g / (1.f + expf(-g)) * u);
    }
}

// Four columns per thread (f a multiple of 4).
// From split-K pieces.  64 registers, eight CTAs an SM: with 101 the 710 CTAs of 33 rows of the 7B shape take two waves (3.22
// against 3.14 ms a step, measured when that step used this kernel), with 51 or 42 the eight loads of an item no longer fit
// and go one after the other (3.19, 3.26 ms).
constexpr int SWIGLU_THREADS = 128, SWIGLU_MAX_CTAS = 2368;
template <typename T>
__global__ void __launch_bounds__(SWIGLU_THREADS, 8) swiglu_pieces_kernel(const Parts gu, T* __restrict__ act, T* __restrict__ act_lo, int rows, int f) {
    pdl_prologue();
    TRJ_TL_DECL; TRJ_TL_BEGIN(TRJ_TL_SWIGLU);
    const int f4 = f >> 2;
    const size_t n4 = (size_t)rows * f4;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / f4, c4 = i % f4;
        store_split4<T>(act, act_lo, 4 * i, silu_mul(parts_at4_batched<4>(gu, r * 2 * f4 + c4), parts_at4_batched<4>(gu, r * 2 * f4 + f4 + c4)));
    }
#ifdef TRJ_TIMELINE
    __syncthreads();
#endif
    TRJ_TL_END(TRJ_TL_SWIGLU);
}
// From finished sums (many rows): blockIdx.y walks the rows instead of a 64-bit division per item, and without the pieces'
// buffers 16 CTAs fit an SM.  1024 rows x 11008 (135 MB): 47 -> 29 us.
template <typename T>
__global__ void __launch_bounds__(SWIGLU_THREADS) swiglu_rows_kernel(const float4* __restrict__ gu, T* __restrict__ act, T* __restrict__ act_lo, int rows, int f) {
    pdl_prologue();
    TRJ_TL_DECL; TRJ_TL_BEGIN(TRJ_TL_SWIGLU);
    const int f4 = f >> 2, c4 = blockIdx.x * SWIGLU_THREADS + threadIdx.x;
    if (c4 < f4) {
        for (int r = blockIdx.y; r < rows; r += gridDim.y) {
            const size_t at = (size_t)r * 2 * f4 + c4;
            store_split4<T>(act, act_lo, (size_t)r * f + 4 * c4, silu_mul(gu[at], gu[at + f4]));
        }
    }
#ifdef TRJ_TIMELINE
    __syncthreads();
#endif
    TRJ_TL_END(TRJ_TL_SWIGLU);
}

// ---------------------------------------------------------------- arg-max + acceptance
// Candidate of a (partial) row scan: best value/index and the runner-up value.
struct Top { float v1; int i1; float v2; };
__device__ __forceinline__ Top top_merge(const Top& a, const Top& b) {
    const bool a_wins = (a.v1 > b.v1) || (a.v1 == b.v1 && a.i1 < b.i1);
    Top r;
    r.v1 = a_wins ? a.v1 : b.v1;
    r.i1 = a_wins ? a.i1 : b.i1;
    r.v2 = fmaxf(a_wins ? b.v1 : a.v1, fmaxf(a.v2, b.v2));
    return r;
}
__device__ __forceinline__ void top_push(Top& t, float v, int i) {
    if (v > t.v1 || (v == t.v1 && i < t.i1)) { t.v2 = fmaxf(t.v2, t.v1); t.v1 = v; t.i1 = i; }
    else t.v2 = fmaxf(t.v2, v);
}
__device__ __forceinline__ Top top_shfl_xor(const Top& t, int o) {
    Top r;
    r.v1 = __shfl_xor_sync(0xffffffffu, t.v1, o);
    r.i1 = __shfl_xor_sync(0xffffffffu, t.i1, o);
    r.v2 = __shfl_xor_sync(0xffffffffu, t.v2, o);
    return r;
}

constexpr int ARGMAX_THREADS = 256;
constexpr int ARGMAX_CHUNKS = 8;              // vocabulary slices per row (one CTA each)

// The acceptance walk of one sequence, run by one CTA after every prediction of it is known.
__device__ void accept_sequence(const int32_t* tokens, const int32_t* parent, const int32_t* depth,
                                const int32_t* pred, int rows, int32_t* k_acc, int32_t* path, int32_t* bonus) {
    rows = min(rows, TRJ_MAX_ROWS);              // the host refuses larger trees; a bad device-side row_off must not overrun
    __shared__ unsigned char ok[TRJ_MAX_ROWS];
    __shared__ int32_t s_tok[TRJ_MAX_ROWS], s_par[TRJ_MAX_ROWS], s_dep[TRJ_MAX_ROWS], s_pred[TRJ_MAX_ROWS];
    __shared__ int s_best;
    // all threads fetch the tree, then one thread walks it out of shared memory
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
        s_tok[i] = tokens[i]; s_par[i] = parent[i]; s_dep[i] = depth[i];
        s_pred[i] = __ldcg(pred + i);            // possibly written by other CTAs of this launch: read it from L2
    }
    __syncthreads();
    // ok[i] = every row on the path root..i carries the token its parent predicted.  Pointer jumping: after round r a
    // row has folded in the matches of its 2^r nearest ancestors, so ceil(log2(rows)) rounds replace a serial walk
    // over the rows (the walk was the longest single piece of this kernel).
    __shared__ short jump[2][TRJ_MAX_ROWS];
    __shared__ unsigned char okb[2][TRJ_MAX_ROWS];
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
        const int p = s_par[i];
        okb[0][i] = i == 0 || s_tok[i] == s_pred[p];
        jump[0][i] = (short)(i == 0 ? 0 : p);
    }
    __syncthreads();
    int cur = 0;
    for (int span = 1; span < rows; span <<= 1, cur ^= 1) {
        for (int i = threadIdx.x; i < rows; i += blockDim.x) {
            const int j = jump[cur][i];
            okb[cur ^ 1][i] = okb[cur][i] && okb[cur][j];
            jump[cur ^ 1][i] = jump[cur][j];
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < rows; i += blockDim.x) ok[i] = okb[cur][i];
    __syncthreads();
    if (threadIdx.x < 32) {
        // the deepest accepted row, the smallest among equals: the largest depth * 128 + (127 - row)
        unsigned key = TRJ_MAX_ROWS - 1;                     // the root, always accepted
        for (int i = threadIdx.x; i < rows; i += 32)
            if (i > 0 && ok[i] && s_dep[i] > 0) key = max(key, (unsigned)s_dep[i] * TRJ_MAX_ROWS + (TRJ_MAX_ROWS - 1 - i));
        key = __reduce_max_sync(0xffffffffu, key);
        if (threadIdx.x == 0) {
            const int best = TRJ_MAX_ROWS - 1 - (int)(key % TRJ_MAX_ROWS), best_depth = (int)(key / TRJ_MAX_ROWS);
            *k_acc = best_depth;
            *bonus = s_pred[best];
            int node = best;
            for (int j = best_depth; j >= 0; --j) { path[j] = node; node = s_par[node]; }
            s_best = best_depth;
        }
    }
    __syncthreads();
    for (int j = s_best + 1 + (int)threadIdx.x; j < TRJ_PATH_STRIDE; j += blockDim.x) path[j] = -1;
}

template <typename T>
__global__ void __launch_bounds__(ARGMAX_THREADS) argmax_accept_kernel(
        const T* __restrict__ logits, int V, const int32_t* __restrict__ tokens,
        const int32_t* __restrict__ parent, const int32_t* __restrict__ depth,
        const int32_t* __restrict__ row_off, int B, int32_t* node_argmax,
        float* __restrict__ margin, int32_t* __restrict__ k_acc, int32_t* __restrict__ path,
        int32_t* __restrict__ bonus, int do_accept, unsigned int* tickets, Top* partial) {
    pdl_prologue();
    __shared__ Top red[ARGMAX_THREADS / 32];
    __shared__ int last_flag;
    const int row = blockIdx.x, chunk = blockIdx.y;
    const int per = (V + ARGMAX_CHUNKS - 1) / ARGMAX_CHUNKS;
    const int v0 = chunk * per, v1 = min(V, v0 + per);
    const T* lr = logits + (size_t)row * V;
    Top t{-INFINITY, 0x7fffffff, -INFINITY};
    constexpr int VEC = 16 / (int)sizeof(T);                 // elements per 16-byte load
    if (V % VEC == 0 && per % VEC == 0 && ((uintptr_t)logits % 16) == 0) {
        for (int v = v0 + threadIdx.x * VEC; v < v1; v += ARGMAX_THREADS * VEC) {
            const uint4 raw = *reinterpret_cast<const uint4*>(lr + v);
            const T* e = reinterpret_cast<const T*>(&raw);
#pragma unroll
            for (int i = 0; i < VEC; ++i) top_push(t, to_f(e[i]), v + i);
        }
    } else {
        for (int v = v0 + threadIdx.x; v < v1; v += ARGMAX_THREADS) top_push(t, to_f(lr[v]), v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t = top_merge(t, top_shfl_xor(t, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        Top r = red[0];
        for (int w = 1; w < ARGMAX_THREADS / 32; ++w) r = top_merge(r, red[w]);
        partial[(size_t)row * ARGMAX_CHUNKS + chunk] = r;
        __threadfence();
        const int b = seq_of_row(row_off, B, row);
        const unsigned int need = (unsigned int)(row_off[b + 1] - row_off[b]) * ARGMAX_CHUNKS;
        const unsigned int got = atomicAdd(&tickets[b], 1u);
        last_flag = (got + 1 == need) ? b : -1;
    }
    __syncthreads();
    const int b = last_flag;
    if (b < 0) return;
    // this CTA saw the last slice of sequence b: finish its rows, then walk the tree
    __threadfence();
    const int r0 = row_off[b], rows = row_off[b + 1] - r0;
    for (int i = threadIdx.x; i < rows; i += ARGMAX_THREADS) {
        const volatile Top* pp = partial + (size_t)(r0 + i) * ARGMAX_CHUNKS;
        Top r{pp[0].v1, pp[0].i1, pp[0].v2};
        for (int c = 1; c < ARGMAX_CHUNKS; ++c) { Top o{pp[c].v1, pp[c].i1, pp[c].v2}; r = top_merge(r, o); }
        node_argmax[r0 + i] = r.i1;
        if (margin) margin[r0 + i] = r.v1 - r.v2;
    }
    if (threadIdx.x == 0) tickets[b] = 0;       // ready for the next call
    __syncthreads();
    if (do_accept)
        accept_sequence(tokens + r0, parent + r0, depth + r0, node_argmax + r0, rows,
                        k_acc + b, path + (size_t)b * TRJ_PATH_STRIDE, bonus + b);
}

// ---------------------------------------------------------------- per-row top-K (K = 1: arg-max) + acceptance
// One CTA per row.  Every thread keeps the KMAX best of its share of the row as a sorted list in registers (order:
// larger value first, equal values by ascending id); each warp then merges its 32 lists into one by KMAX rounds of a
// warp-wide arg-max over the lists' heads, and the first warp merges the 32 warp lists the same way.  The CTA that
// finishes the last row of a sequence walks that sequence's tree.
constexpr int TOPK_THREADS = 1024;
// Top-K (K <= TRJ_MAX_TOPK) of a row, value first and the smaller id among equals.  The row is taken in chunks of
// 32 x 1024 elements that the CTA's threads hold in registers (element j * 1024 + t of the chunk in thread t).
// Per chunk: (A) the 32 warp maxima; their K-th largest is a value that at least K elements of the chunk reach, so
// together with the K-th value of the row's running list it is a threshold below which nothing can enter the list;
// (B) every element at or above the threshold goes to a candidate buffer in shared memory (slots handed out by an
// atomic counter: the order in the buffer is arbitrary, the selection below is not); (C) the first warp selects the K
// best among the candidates and the running list by K rounds of a scan and a shuffle reduction.  Typically a few
// dozen elements survive the threshold.  If more survive than the buffer holds (many equal values), the chunk is
// done the slow way: K rounds of selection over all its elements, in every warp and then over the warps' lists.
constexpr int TOPK_PER_THREAD = 32;
constexpr int TOPK_CAND = 1024;
__device__ __forceinline__ bool top_better(float v, int i, float w, int j) { return v > w || (v == w && i < j); }
__device__ __forceinline__ void warp_best(float& bv, int& bi) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (top_better(ov, oi, bv, bi)) { bv = ov; bi = oi; }
    }
}
template <typename T>
__global__ void __launch_bounds__(TOPK_THREADS) topk_accept_kernel(
        const T* __restrict__ logits, int V, int K, const int32_t* __restrict__ tokens,
        const int32_t* __restrict__ parent, const int32_t* __restrict__ depth,
        const int32_t* __restrict__ row_off, int B, int32_t* __restrict__ topk, int32_t* node_argmax,
        float* __restrict__ margin, int32_t* __restrict__ k_acc, int32_t* __restrict__ path,
        int32_t* __restrict__ bonus, int do_accept, unsigned int* tickets) {
    pdl_prologue();
    __shared__ float cand_v[TOPK_CAND + TRJ_MAX_TOPK];             // candidates of the chunk, then the running list
    __shared__ int cand_i[TOPK_CAND + TRJ_MAX_TOPK];
    __shared__ float list_v[TOPK_THREADS / 32][TRJ_MAX_TOPK];      // slow path: the warps' sorted lists; [0] also: warp maxima
    __shared__ int list_i[TOPK_THREADS / 32][TRJ_MAX_TOPK];
    __shared__ float best_v[TRJ_MAX_TOPK];                          // the row's running list, sorted
    __shared__ int best_i[TRJ_MAX_TOPK];
    __shared__ float warp_max_v[TOPK_THREADS / 32];
    __shared__ float thr;
    __shared__ int cand_n;
    __shared__ int last_flag;
    const int row = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const T* lr = logits + (size_t)row * V;
    if (tid < TRJ_MAX_TOPK) { best_v[tid] = -INFINITY; best_i[tid] = 0x7fffffff; }
    for (int base = 0; base < V; base += TOPK_PER_THREAD * TOPK_THREADS) {
        float x[TOPK_PER_THREAD];
        float tm = -INFINITY;
#pragma unroll
        for (int j = 0; j < TOPK_PER_THREAD; ++j) {
            const int id = base + j * TOPK_THREADS + tid;
            x[j] = id < V ? to_f(lr[id]) : -INFINITY;
            tm = fmaxf(tm, x[j]);
        }
        // (A) warp maxima, then the K-th largest of them (with multiplicity) in the first warp
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tm = fmaxf(tm, __shfl_xor_sync(0xffffffffu, tm, o));
        if (lane == 0) warp_max_v[warp] = tm;
        __syncthreads();
        if (warp == 0) {
            float mine = warp_max_v[lane], kth = -INFINITY;
            for (int r = 0; r < K; ++r) {
                float m = mine;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                kth = m;
                const unsigned holders = __ballot_sync(0xffffffffu, mine == m);
                if (lane == __ffs(holders) - 1) mine = -INFINITY;      // one holder gives its value up per round
            }
            if (lane == 0) { thr = fmaxf(kth, best_v[K - 1]); cand_n = 0; }
        }
        __syncthreads();
        // (B) candidates
        const float t = thr;
#pragma unroll
        for (int j = 0; j < TOPK_PER_THREAD; ++j) {
            const int id = base + j * TOPK_THREADS + tid;
            if (id < V && x[j] >= t) {
                const int slot = atomicAdd(&cand_n, 1);
                if (slot < TOPK_CAND) { cand_v[slot] = x[j]; cand_i[slot] = id; }
            }
        }
        __syncthreads();
        const int n_cand = cand_n;                           // the same for every thread
        if (n_cand <= TOPK_CAND) {
            // (C) the first warp: K best of the candidates and the running list
            if (warp == 0) {
                if (lane < K) { cand_v[n_cand + lane] = best_v[lane]; cand_i[n_cand + lane] = best_i[lane]; }
                __syncwarp();
                const int n = n_cand + K;
                float mv = -INFINITY;
                int mi = 0x7fffffff;
                for (int r = 0; r < K; ++r) {
                    float bv = -INFINITY;
                    int bi = 0x7fffffff, bs = -1;
                    for (int e = lane; e < n; e += 32) {
                        const float v = cand_v[e];
                        const int i = cand_i[e];
                        if (i != 0x7fffffff && top_better(v, i, bv, bi)) { bv = v; bi = i; bs = e; }
                    }
                    const int mine_i = bi;
                    warp_best(bv, bi);
                    if (bs >= 0 && mine_i == bi) cand_i[bs] = 0x7fffffff;     // taken (ids are unique: one lane owns it)
                    __syncwarp();
                    if (lane == r) { mv = bv; mi = bi; }
                }
                if (lane < K) { best_v[lane] = mv; best_i[lane] = mi; }
            }
        } else {
            // slow path: K rounds over all elements of the chunk in every warp, then over the warps' lists
            uint32_t taken = 0;
            for (int r = 0; r < K; ++r) {
                float bv = -INFINITY;
                int bj = -1;
#pragma unroll
                for (int j = 0; j < TOPK_PER_THREAD; ++j)    // ascending ids: "strictly larger" keeps the smallest id among equals
                    if (!((taken >> j) & 1u) && x[j] > bv) { bv = x[j]; bj = j; }
                int bi = bj >= 0 ? base + bj * TOPK_THREADS + tid : 0x7fffffff;
                const int mine_i = bi;
                warp_best(bv, bi);
                if (bi == mine_i && bj >= 0) taken |= 1u << bj;
                if (lane == 0) { list_v[warp][r] = bv; list_i[warp][r] = bi; }
            }
            __syncthreads();
            if (warp == 0) {
                int head = 0;
                float mv = -INFINITY;
                int mi = 0x7fffffff;
                for (int r = 0; r < K; ++r) {
                    float bv = head < K ? list_v[lane][head] : -INFINITY;
                    int bi = head < K ? list_i[lane][head] : 0x7fffffff;
                    const int mine_i = bi;
                    warp_best(bv, bi);
                    if (bi == mine_i && bi != 0x7fffffff) ++head;
                    if (lane == r) { mv = bv; mi = bi; }
                }
                if (lane < K) { list_v[0][lane] = mv; list_i[0][lane] = mi; }
                __syncwarp();
                if (lane == 0) {                             // two sorted lists of K entries -> the K best
                    float nv[TRJ_MAX_TOPK];
                    int ni[TRJ_MAX_TOPK];
                    int a = 0, c = 0;
                    for (int r = 0; r < K; ++r) {
                        if (top_better(list_v[0][a], list_i[0][a], best_v[c], best_i[c])) { nv[r] = list_v[0][a]; ni[r] = list_i[0][a]; ++a; }
                        else { nv[r] = best_v[c]; ni[r] = best_i[c]; ++c; }
                    }
                    for (int r = 0; r < K; ++r) { best_v[r] = nv[r]; best_i[r] = ni[r]; }
                }
            }
        }
        __syncthreads();                                     // the buffers are rewritten by the next chunk
    }
    if (tid < K && topk) topk[(size_t)row * K + tid] = best_i[tid];
    if (tid == 0) {
        node_argmax[row] = best_i[0];
        if (margin) margin[row] = best_v[0] - best_v[K > 1 ? 1 : 0];
        __threadfence();
        const int b = seq_of_row(row_off, B, row);
        const unsigned int need = (unsigned int)(row_off[b + 1] - row_off[b]);
        const unsigned int got = atomicAdd(&tickets[b], 1u);
        last_flag = (got + 1 == need) ? b : -1;
        if (got + 1 == need) tickets[b] = 0;                 // ready for the next call
    }
    __syncthreads();
    const int b = last_flag;
    if (b < 0 || !do_accept) return;
    __threadfence();                                         // the other rows' predictions were written by other CTAs
    const int r0 = row_off[b], rows = row_off[b + 1] - r0;
    accept_sequence(tokens + r0, parent + r0, depth + r0, node_argmax + r0, rows,
                    k_acc + b, path + (size_t)b * TRJ_PATH_STRIDE, bonus + b);
}

// The arg-max of every verification step (K = 1): one CTA per row, five instructions per element.  A thread scans its
// elements in ascending id order, so "strictly larger" keeps the smallest id among equals; the runner-up value (for
// the margin) is max(v2, min(v1, x)).  Threads, then warps, are merged with the full (value, id) order.
// 1024 threads a row up to one row per SM, 512 up to four, else 256: the rows then run in one wave, and what a row waits for
// (its loads, its reductions, its ticket) is overlapped by the others on its SM.  bf16, us a call with 1024 / 512 / 256 threads: rows x 32000: 64:
// 7.7 / 7.7 / 8.2, 296: 14.9 / 9.6 / 9.8, 592: 22.6 / 12.8 / 12.8, 700: 24.1 / 14.8 / 15.8, 2000: 70.6 / 33.9 / 31.3; x 128256: 64: 11.3 / 12.1 / 14.4, 296: 23.5 /
// 18.4 / 19.2, 592: 47.5 / 31.6 / 33.9, 700: 50.3 / 42.4 / 46.9, 1024: 69.4 / 49.1 / 52.6, 2000: 141 / 89 / 88.  fp32 x 128256: 364: 43.6 / 34.2 / 39.3, 593: 69.5 / 58.9 /
// 52.0, 1500: 154 / 126 / 140.  Where 256 threads are taken 512 are up to 10 % faster for wide vocabularies and 10 - 30 % slower for narrow ones.
template <typename T, int THREADS>
__global__ void __launch_bounds__(THREADS) argmax_row_accept_kernel(
        const T* __restrict__ logits, int V, const int32_t* __restrict__ tokens,
        const int32_t* __restrict__ parent, const int32_t* __restrict__ depth,
        const int32_t* __restrict__ row_off, int B, int32_t* node_argmax,
        float* __restrict__ margin, int32_t* __restrict__ k_acc, int32_t* __restrict__ path,
        int32_t* __restrict__ bonus, int do_accept, unsigned int* tickets) {
    pdl_prologue();
    __shared__ Top red[THREADS / 32];
    __shared__ int last_flag;
    const int row = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const T* lr = logits + (size_t)row * V;
    float v1 = -INFINITY, v2 = -INFINITY;
    int i1 = 0x7fffffff;
    auto look = [&](float x, int i) {
        v2 = fmaxf(v2, fminf(v1, x));
        i1 = x > v1 ? i : i1;
        v1 = fmaxf(v1, x);
    };
    constexpr int VEC = 16 / (int)sizeof(T);
    if (V % VEC == 0 && ((uintptr_t)logits % 16) == 0) {
        constexpr int BATCH = 4;                             // four 16-byte loads in flight per thread
        for (int v0 = threadIdx.x * VEC; v0 < V; v0 += BATCH * THREADS * VEC) {
            uint4 raw[BATCH];
#pragma unroll
            for (int j = 0; j < BATCH; ++j) {
                const int v = v0 + j * THREADS * VEC;
                if (v < V) raw[j] = *reinterpret_cast<const uint4*>(lr + v);
            }
#pragma unroll
            for (int j = 0; j < BATCH; ++j) {
                const int v = v0 + j * THREADS * VEC;
                if (v < V) {
                    const T* e = reinterpret_cast<const T*>(&raw[j]);
#pragma unroll
                    for (int i = 0; i < VEC; ++i) look(to_f(e[i]), v + i);
                }
            }
        }
    } else {
        for (int v = threadIdx.x; v < V; v += THREADS) look(to_f(lr[v]), v);
    }
    Top t{v1, i1, v2};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t = top_merge(t, top_shfl_xor(t, o));
    if (lane == 0) red[warp] = t;
    __syncthreads();
    if (warp == 0) {
        t = lane < THREADS / 32 ? red[lane] : Top{-INFINITY, 0x7fffffff, -INFINITY};
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t = top_merge(t, top_shfl_xor(t, o));
        if (lane == 0) {
            node_argmax[row] = t.i1 == 0x7fffffff ? 0 : t.i1;      // nothing above -inf: still an id of the vocabulary
            if (margin) margin[row] = t.v1 - t.v2;
            __threadfence();
            const int b = seq_of_row(row_off, B, row);
            const unsigned int need = (unsigned int)(row_off[b + 1] - row_off[b]);
            const unsigned int got = atomicAdd(&tickets[b], 1u);
            last_flag = (got + 1 == need) ? b : -1;
            if (got + 1 == need) tickets[b] = 0;             // ready for the next call
        }
    }
    __syncthreads();
    const int b = last_flag;
    if (b < 0 || !do_accept) return;
    __threadfence();                                         // the other rows' predictions were written by other CTAs
    const int r0 = row_off[b], rows = row_off[b + 1] - r0;
    accept_sequence(tokens + r0, parent + r0, depth + r0, node_argmax + r0, rows,
                    k_acc + b, path + (size_t)b * TRJ_PATH_STRIDE, bonus + b);
}

// Arg-max of every row from the candidates a projection's epilogue left (one per 32 outputs), then acceptance as above.
__global__ void __launch_bounds__(128) argmax_table_accept_kernel(
        const TopEntry* __restrict__ table, int per_row, const int32_t* __restrict__ tokens,
        const int32_t* __restrict__ parent, const int32_t* __restrict__ depth,
        const int32_t* __restrict__ row_off, int B, int32_t* node_argmax,
        float* __restrict__ margin, int32_t* __restrict__ k_acc, int32_t* __restrict__ path,
        int32_t* __restrict__ bonus, int do_accept, unsigned int* tickets) {
    pdl_prologue();
    __shared__ Top red[4];
    __shared__ int last_flag;
    const int row = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const TopEntry* tr = table + (size_t)row * per_row;
    Top t{-INFINITY, 0x7fffffff, -INFINITY};
    for (int i = threadIdx.x; i < per_row; i += 128) {
        const TopEntry e = tr[i];
        t = top_merge(t, Top{e.v1, e.i1, e.v2});
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t = top_merge(t, top_shfl_xor(t, o));
    if (lane == 0) red[warp] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        t = top_merge(top_merge(red[0], red[1]), top_merge(red[2], red[3]));
        node_argmax[row] = t.i1;
        if (margin) margin[row] = t.v1 - t.v2;
        __threadfence();
        const int b = seq_of_row(row_off, B, row);
        const unsigned int need = (unsigned int)(row_off[b + 1] - row_off[b]);
        const unsigned int got = atomicAdd(&tickets[b], 1u);
        last_flag = (got + 1 == need) ? b : -1;
        if (got + 1 == need) tickets[b] = 0;                 // ready for the next call
    }
    __syncthreads();
    const int b = last_flag;
    if (b < 0 || !do_accept) return;
    __threadfence();                                         // the other rows' predictions were written by other CTAs
    const int r0 = row_off[b], rows = row_off[b + 1] - r0;
    accept_sequence(tokens + r0, parent + r0, depth + r0, node_argmax + r0, rows,
                    k_acc + b, path + (size_t)b * TRJ_PATH_STRIDE, bonus + b);
}

__global__ void accept_only_kernel(const int32_t* __restrict__ tokens, const int32_t* __restrict__ parent,
                                   const int32_t* __restrict__ depth, const int32_t* __restrict__ row_off,
                                   const int32_t* __restrict__ node_argmax, int32_t* __restrict__ k_acc,
                                   int32_t* __restrict__ path, int32_t* __restrict__ bonus) {
    pdl_prologue();
    const int b = blockIdx.x, r0 = row_off[b], rows = row_off[b + 1] - r0;
    accept_sequence(tokens + r0, parent + r0, depth + r0, node_argmax + r0, rows,
                    k_acc + b, path + (size_t)b * TRJ_PATH_STRIDE, bonus + b);
}

// ---------------------------------------------------------------- KV compaction
// One CTA per (layer, sequence, head, K|V).  Rows are moved in ascending order in batches that are
// fully loaded before they are stored; since path[j] >= j and the path is strictly increasing, a
// destination never overwrites a row that a later batch still has to read.
constexpr int COMPACT_BATCH = 16;
__global__ void __launch_bounds__(256) compact_kernel(uint4* __restrict__ k_cache, uint4* __restrict__ v_cache,
                                                      int B_cache, int B, int H, int max_seq, int row_vec,
                                                      int32_t* seq_len,
                                                      const int32_t* __restrict__ k_acc,
                                                      const int32_t* __restrict__ path, unsigned int* tickets) {
    pdl_prologue();
    extern __shared__ uint4 stage[];             // [COMPACT_BATCH][row_vec]
    int idx = blockIdx.x;
    const int kv = idx & 1; idx >>= 1;
    const int hh = idx % H; idx /= H;
    const int b = idx % B; const int l = idx / B;
    const int k = min(k_acc[b], TRJ_PATH_STRIDE - 1);    // a path holds at most TRJ_PATH_STRIDE rows
    const int S = seq_len[b];
    // With tickets the sequence's length is advanced here as well: every CTA has read it by the time it draws its
    // ticket, so the CTA that draws the last one may write it (and leaves the ticket at zero for the next call).
    auto finish = [&]() {
        if (!tickets) return;
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned int per_seq = gridDim.x / (unsigned int)B;
            if (atomicAdd(&tickets[b], 1u) + 1u == per_seq) { tickets[b] = 0; seq_len[b] = S + k + 1; }
        }
    };
    if (k <= 0) { finish(); return; }
    uint4* slab = (kv ? v_cache : k_cache) + (((size_t)l * B_cache + b) * H + hh) * (size_t)max_seq * row_vec;
    const int32_t* pb = path + (size_t)b * TRJ_PATH_STRIDE;
    for (int j0 = 1; j0 <= k; j0 += COMPACT_BATCH) {
        const int nj = min(COMPACT_BATCH, k - j0 + 1);
        for (int e = threadIdx.x; e < nj * row_vec; e += blockDim.x) {
            const int j = j0 + e / row_vec, c = e % row_vec;
            if (TRJ_DEBUG_CHECK(pb[j] >= 0 && (unsigned)(S + pb[j]) < (unsigned)max_seq, DBG_COMPACT_ROW))
                stage[e] = slab[(size_t)(S + pb[j]) * row_vec + c];
        }
        __syncthreads();
        for (int e = threadIdx.x; e < nj * row_vec; e += blockDim.x) {
            const int j = j0 + e / row_vec, c = e % row_vec;
            if (TRJ_DEBUG_CHECK(pb[j] >= 0 && (unsigned)(S + pb[j]) < (unsigned)max_seq && (unsigned)(S + j) < (unsigned)max_seq, DBG_COMPACT_ROW))
                slab[(size_t)(S + j) * row_vec + c] = stage[e];
        }
        __syncthreads();
    }
    finish();
}

__global__ void advance_len_kernel(int32_t* seq_len, const int32_t* k_acc, int B) {
    pdl_prologue();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) seq_len[b] += k_acc[b] + 1;
}
__global__ void set_chunk_kernel(int32_t* row_off2, int m) { row_off2[0] = 0; row_off2[1] = m; }
__global__ void prefill_geometry_kernel(const int32_t* seq_len_b, int32_t* lens, int n_sub, int sub, int m, int32_t* off_all,
                                        int32_t* off_pieces) {
    for (int j = threadIdx.x; j < n_sub; j += blockDim.x) lens[j] = *seq_len_b + j * sub;
    for (int j = threadIdx.x; j <= n_sub; j += blockDim.x) off_pieces[j] = min(j * sub, m);
    if (threadIdx.x == 0) { off_all[0] = 0; off_all[1] = m; }
}
__global__ void bump_len_kernel(int32_t* seq_len_b, int delta) { *seq_len_b += delta; }

}  // namespace

// ============================================================================ launchers
static std::atomic<bool> g_pdl{true};
bool pdl_enabled() { return g_pdl.load(std::memory_order_relaxed); }
void set_pdl(bool on) { g_pdl.store(on, std::memory_order_relaxed); }
static thread_local int t_chain_depth = 0;
bool chain_active() { return t_chain_depth > 0 && pdl_enabled(); }
ChainScope::ChainScope() { ++t_chain_depth; }
ChainScope::~ChainScope() { --t_chain_depth; }
#ifdef TRJ_DEBUG
cudaError_t debug_flags_read(int* flags) {
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(flags, g_debug_flags, sizeof(int));
    const int zero = 0;
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_debug_flags, &zero, sizeof(int));
    return e;
}
#endif
#ifdef TRJ_TIMELINE
cudaError_t timeline_reset_generic(cudaStream_t st) { return tl::reset(st); }
int timeline_read_generic(int kind, int max_launches, uint64_t* b, uint64_t* e) { return tl::read(kind, max_launches, b, e); }
#endif
static std::atomic<uint64_t> g_launches{0};
void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
uint64_t launches_so_far() { return g_launches.load(std::memory_order_relaxed); }

#define DISPATCH_T(dtype, ...)                                         \
    if ((dtype) == TRJ_BF16) { using T = __nv_bfloat16; __VA_ARGS__; } \
    else { using T = float; __VA_ARGS__; }

cudaError_t launch_embed(const void* embed, int32_t dtype, const int32_t* tokens, float* h, int32_t d, const double* inv_freq, int32_t D,
                         const int32_t* depth, const Batch& bt, const Rotary& rot, cudaStream_t st) {
    count_launch();
    cudaError_t launch_err = cudaSuccess;
    DISPATCH_T(dtype, launch_err = launch_chain(embed_kernel<T>, dim3(bt.rows_total), dim3(256), 0, st, (const T*)embed, tokens, h, d, inv_freq, D / 2,
                                                depth, bt.seq_len, bt.row_off, bt.B, rotary_table_used(bt.rows_total) ? rot.table : nullptr, rot.row_at));
    return launch_err != cudaSuccess ? launch_err : cudaGetLastError();
}

cudaError_t launch_add_rmsnorm(float* h, const Parts& add, const float* gain, void* x, void* x_lo, int32_t dtype,
                               int32_t rows, int32_t d, float eps, cudaStream_t st) {
    count_launch();
    cudaError_t launch_err = cudaSuccess;
    const bool vec = d % 4 == 0 && d <= RMS_MAX_D && add.stride % 4 == 0 &&
                     ((uintptr_t)h | (uintptr_t)add.ptr | (uintptr_t)gain | (uintptr_t)x | (uintptr_t)x_lo) % 16 == 0;
    if (vec) {
#define RMS(THREADS, CHUNKS) \
    DISPATCH_T(dtype, launch_err = launch_chain(add_rmsnorm_vec_kernel<T, THREADS, CHUNKS>, dim3(rows), dim3(THREADS), 0, st, h, add, gain, (T*)x, (T*)x_lo, d, eps))
        if (rows <= RMS_FEW_ROWS) { RMS(RMS_FEW_ROWS_THREADS, 2); }
        else { if (d <= 4096) { RMS(256, 4); } else { RMS(256, 8); } }
#undef RMS
    } else {
        DISPATCH_T(dtype, launch_err = launch_chain(add_rmsnorm_kernel<T>, dim3(rows), dim3(256), 0, st, h, add, gain, (T*)x, (T*)x_lo, d, eps));
    }
    return launch_err != cudaSuccess ? launch_err : cudaGetLastError();
}

// The small kernel against the tiled one, us per launch at K = 256 by 64 x 64 tiles: 4: 2.1 / 15.6, 22: 6.0 / 18.2, 66: 12.3 /
// 18.3, 96: 16.6 / 18.3, 132: 21.7 / 18.4 (it reads its operands again for every 16 rows and 8 columns).  K is bounded by the
// 24 rows of K that a CTA keeps in shared memory.
bool gemm_small_f32_shape(int32_t M, int32_t N, int32_t K) {
    return K % 4 == 0 && K <= SF_MAX_K && (int64_t)((N + 63) / 64) * ((M + 63) / 64) <= SMALL_F32_MAX_TILES;
}
cudaError_t launch_gemm_small_f32(const SmallF32Input& in, const float* w, float* y, int32_t M, int32_t N, int32_t K, cudaStream_t st) {
    static std::once_flag once;
    static cudaError_t attr_err = cudaSuccess;
    const auto smem_of = [](int k) { return (size_t)(SF_ROWS + SF_COLS) * (k + 4) * sizeof(float); };
    std::call_once(once, [&] {
        for (auto kernel : {gemm_small_f32_kernel<SF_PLAIN, 1>, gemm_small_f32_kernel<SF_NORM, 2>, gemm_small_f32_kernel<SF_NORM, 8>,
                            gemm_small_f32_kernel<SF_SWIGLU, 8>})
            if (attr_err == cudaSuccess)
                attr_err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(SF_MAX_K));
    });
    if (attr_err != cudaSuccess) return attr_err;
    count_launch();
    auto kernel = in.kind == SmallF32Input::PLAIN ? gemm_small_f32_kernel<SF_PLAIN, 1> : in.kind == SmallF32Input::SWIGLU ? gemm_small_f32_kernel<SF_SWIGLU, 8>
                  : K <= 256 ? gemm_small_f32_kernel<SF_NORM, 2> : gemm_small_f32_kernel<SF_NORM, 8>;
    const cudaError_t e = launch_chain(kernel, dim3((N + SF_COLS - 1) / SF_COLS, (M + SF_ROWS - 1) / SF_ROWS), dim3(SF_THREADS), smem_of(K), st, in, w, y, M, N, K);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_gemm_simt(const void* x, const void* x_lo, const void* w, float* y, int32_t M, int32_t N,
                             int32_t K, int32_t dtype, cudaStream_t st) {
    // Few 64 x 64 tiles and a K whose rows fit shared memory: latency is what counts.
    if (dtype == TRJ_F32 && gemm_small_f32_shape(M, N, K) && ((uintptr_t)x | (uintptr_t)w) % 16 == 0)
        return launch_gemm_small_f32(SmallF32Input{SmallF32Input::PLAIN, (const float*)x, nullptr, nullptr, nullptr, 0.f}, (const float*)w, y, M, N, K, st);
    count_launch();
    dim3 grid((N + 63) / 64, (M + 63) / 64);
    DISPATCH_T(dtype, gemm_simt_kernel<T><<<grid, 256, 0, st>>>((const T*)x, (const T*)x_lo, (const T*)w, y, M, N, K));
    return cudaGetLastError();
}

bool rotary_table_used(int32_t rows) { return rows > ROPE_FEW_ROWS; }

cudaError_t launch_rope_kv_write(const Parts& qkv, const Rotary& rot, const double* inv_freq, const int32_t* depth, const Batch& bt, void* q_out,
                                 void* k_slab, void* v_slab, int32_t dtype, int32_t H, int32_t Hkv, int32_t D, int32_t max_seq, cudaStream_t st) {
    if (D % 8 != 0 || ROPE_THREADS % (D / 8) != 0 || qkv.stride % 4 != 0 || ((uintptr_t)qkv.ptr % 16) != 0) return cudaErrorInvalidValue;
    count_launch();
    const int per_head = D / 8;                              // threads per head
    cudaError_t launch_err = cudaSuccess;
    if (rotary_table_used(bt.rows_total)) {
        const int heads_per_cta = ROPE_THREADS / per_head;
        DISPATCH_T(dtype, launch_err = launch_chain(qkv.splits > 1 ? rope_kv_write_kernel<T, 4> : rope_kv_write_kernel<T, 1>,
                                                    dim3(bt.rows_total, (H + 2 * Hkv + heads_per_cta - 1) / heads_per_cta), dim3(ROPE_THREADS), 0, st,
                                                    qkv, rot.table, rot.row_at, (T*)q_out, (T*)k_slab, (T*)v_slab, H, Hkv, D, max_seq));
    } else {
        const int hpc = std::max(1, std::min(H, ROPE_THREADS / per_head));
        DISPATCH_T(dtype, launch_err = launch_chain(rope_kv_write_few_kernel<T>, dim3(bt.rows_total, (H + hpc - 1) / hpc), dim3(per_head * hpc), 0, st,
                                                    qkv, inv_freq, depth, bt.seq_len, bt.row_off, bt.B, (T*)q_out, (T*)k_slab, (T*)v_slab, H, Hkv, D,
                                                    max_seq, hpc));
    }
    return launch_err != cudaSuccess ? launch_err : cudaGetLastError();
}

cudaError_t launch_tree_attention_generic(const void* q, const void* k_slab, const void* v_slab,
                                          const uint64_t* anc, int32_t anc_words, const Batch& bt,
                                          int32_t H, int32_t Hkv, int32_t D, int32_t max_seq, int32_t dtype,
                                          void* out, void* out_lo, cudaStream_t st) {
    count_launch();
    dim3 grid(bt.rows_total, H);
    cudaError_t launch_err = cudaSuccess;
#define ATT(DD)                                                                                          \
    DISPATCH_T(dtype, launch_err = launch_chain(tree_attention_generic_kernel<T, DD>, grid, dim3(128), 0, st, \
                          (const T*)q, (const T*)k_slab, (const T*)v_slab, anc, anc_words, bt.seq_len,   \
                          bt.row_off, bt.B, H, Hkv, max_seq, (T*)out, (T*)out_lo, bt.shared_cache))
    if (D == 64) { ATT(64); }
    else if (D == 128) { ATT(128); }
    else return cudaErrorInvalidValue;
#undef ATT
    return launch_err != cudaSuccess ? launch_err : cudaGetLastError();
}

cudaError_t launch_swiglu(const Parts& gu, void* act, void* act_lo, int32_t dtype, int32_t rows, int32_t f,
                          cudaStream_t st) {
    count_launch();
    cudaError_t launch_err = cudaSuccess;
    const bool vec = f % 4 == 0 && gu.stride % 4 == 0 && ((uintptr_t)gu.ptr % 16) == 0;
    const size_t n = (size_t)rows * (vec ? f / 4 : f);
    const int blocks = (int)std::min<size_t>((n + SWIGLU_THREADS - 1) / SWIGLU_THREADS, SWIGLU_MAX_CTAS);
    if (vec && gu.splits > 1) {
        DISPATCH_T(dtype, launch_err = launch_chain(swiglu_pieces_kernel<T>, dim3(blocks), dim3(SWIGLU_THREADS), 0, st, gu, (T*)act, (T*)act_lo, rows, f));
    } else if (vec) {
        const int across = (f / 4 + SWIGLU_THREADS - 1) / SWIGLU_THREADS;
        DISPATCH_T(dtype, launch_err = launch_chain(swiglu_rows_kernel<T>, dim3(across, std::min(rows, std::max(1, SWIGLU_MAX_CTAS / across))),
                                                    dim3(SWIGLU_THREADS), 0, st, (const float4*)gu.ptr, (T*)act, (T*)act_lo, rows, f));
    } else {
        DISPATCH_T(dtype, launch_err = launch_chain(swiglu_kernel<T>, dim3(blocks), dim3(128), 0, st, gu, (T*)act, (T*)act_lo, rows, f));
    }
    return launch_err != cudaSuccess ? launch_err : cudaGetLastError();
}

size_t argmax_workspace_bytes(int32_t rows_total, int32_t B) {
    (void)B;
    return align_up(sizeof(unsigned int) * TRJ_MAX_BATCH, 256) + align_up(sizeof(Top) * ARGMAX_CHUNKS * (size_t)rows_total, 256);
}

cudaError_t launch_argmax_accept(const void* logits, int32_t dtype, int32_t V,
                                 const int32_t* tokens, const int32_t* parent, const int32_t* depth,
                                 const int32_t* row_off, int32_t B, int32_t rows_total,
                                 int32_t* node_argmax, float* margin, int32_t* k_acc, int32_t* path,
                                 int32_t* bonus, bool do_argmax, bool do_accept, void* ws, cudaStream_t st) {
    if (do_argmax || do_accept) count_launch();
    cudaError_t launch_err = cudaSuccess;
    if (do_argmax) {
        unsigned int* tickets = (unsigned int*)ws;
        Top* partial = (Top*)((char*)ws + align_up(sizeof(unsigned int) * TRJ_MAX_BATCH, 256));
        dim3 grid(rows_total, ARGMAX_CHUNKS);
        DISPATCH_T(dtype, launch_err = launch_chain(argmax_accept_kernel<T>, grid, dim3(ARGMAX_THREADS), 0, st,
                                                    (const T*)logits, V, tokens, parent, depth, row_off, B, node_argmax,
                                                    margin, k_acc, path, bonus, do_accept ? 1 : 0, tickets, partial));
    } else if (do_accept) {
        launch_err = launch_chain(accept_only_kernel, dim3(B), dim3(32), 0, st, tokens, parent, depth, row_off,
                                  (const int32_t*)node_argmax, k_acc, path, bonus);
    }
    return launch_err != cudaSuccess ? launch_err : cudaGetLastError();
}

size_t topk_workspace_bytes() { return align_up(sizeof(unsigned int) * TRJ_MAX_BATCH, 256); }

cudaError_t launch_topk_accept(const void* logits, int32_t dtype, int32_t V, int32_t K,
                               const int32_t* tokens, const int32_t* parent, const int32_t* depth,
                               const int32_t* row_off, int32_t B, int32_t rows_total, int32_t* topk,
                               int32_t* node_argmax, float* margin, int32_t* k_acc, int32_t* path,
                               int32_t* bonus, bool do_accept, void* ws, cudaStream_t st) {
    if (K < 1 || K > TRJ_MAX_TOPK) return cudaErrorInvalidValue;
    count_launch();
    cudaError_t launch_err = cudaSuccess;
    unsigned int* tickets = (unsigned int*)ws;
    if (K == 1) {                                            // the step's arg-max: a kernel of its own, five instructions per element
        const int threads = rows_total <= 148 ? 1024 : rows_total <= 4 * 148 ? 512 : 256;
        DISPATCH_T(dtype, launch_err = launch_chain(threads == 1024 ? argmax_row_accept_kernel<T, 1024>
                                                    : threads == 512 ? argmax_row_accept_kernel<T, 512> : argmax_row_accept_kernel<T, 256>,
                                                    dim3(rows_total), dim3(threads), 0, st,
                                                    (const T*)logits, V, tokens, parent, depth, row_off, B, node_argmax,
                                                    margin, k_acc, path, bonus, do_accept ? 1 : 0, tickets));
        if (launch_err == cudaSuccess && topk)
            launch_err = cudaMemcpyAsync(topk, node_argmax, sizeof(int32_t) * (size_t)rows_total, cudaMemcpyDeviceToDevice, st);
    } else {
        DISPATCH_T(dtype, launch_err = launch_chain(topk_accept_kernel<T>, dim3(rows_total), dim3(TOPK_THREADS), 0, st,
                                                    (const T*)logits, V, K, tokens, parent, depth, row_off, B, topk, node_argmax,
                                                    margin, k_acc, path, bonus, do_accept ? 1 : 0, tickets));
    }
    return launch_err != cudaSuccess ? launch_err : cudaGetLastError();
}

cudaError_t launch_argmax_table_accept(const TopEntry* table, int32_t entries_per_row, const int32_t* tokens,
                                       const int32_t* parent, const int32_t* depth, const int32_t* row_off, int32_t B,
                                       int32_t rows_total, int32_t* node_argmax, float* margin, int32_t* k_acc,
                                       int32_t* path, int32_t* bonus, bool do_accept, void* ws, cudaStream_t st) {
    count_launch();
    cudaError_t e = launch_chain(argmax_table_accept_kernel, dim3(rows_total), dim3(128), 0, st, table, entries_per_row, tokens,
                                 parent, depth, row_off, B, node_argmax, margin, k_acc, path, bonus, do_accept ? 1 : 0,
                                 (unsigned int*)ws);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// ---------------------------------------------------------------- arg-max + accept without a caller workspace
// Scratch of the allocation-free entry point: the tickets and the per-slice candidates live in this
// file-scope device array, which every GPU that loads the library holds until the process exits.
constexpr int STATIC_MAX_ROWS = TRJ_STATIC_MAX_ROWS;
constexpr size_t STATIC_TICKET_BYTES = 256;
constexpr size_t STATIC_SCRATCH_BYTES = STATIC_TICKET_BYTES + sizeof(Top) * ARGMAX_CHUNKS * (size_t)STATIC_MAX_ROWS;
static __device__ __align__(256) unsigned char g_static_scratch[STATIC_SCRATCH_BYTES];

// In host code `g_static_scratch` is only a handle for the runtime, not an address a kernel can use: the
// device address is looked up once per device (with that device current) and remembered.
static cudaError_t static_scratch_address(void** out, cudaStream_t st) {
    constexpr int MAX_DEVICES = 64;
    static std::mutex mu;
    static void* addr[MAX_DEVICES] = {};
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        // the lookup may load the module: it must not happen while `st` is being captured
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        e = cudaStreamIsCapturing(st, &cs);
        if (e != cudaSuccess) return e;
        if (cs != cudaStreamCaptureStatusNone) return cudaErrorStreamCaptureUnsupported;
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess) return e;
        addr[dev] = p;
    }
    *out = addr[dev];
    return cudaSuccess;
}

cudaError_t launch_argmax_accept_static(const void* logits, int32_t dtype, int32_t V,
                                        const int32_t* tokens, const int32_t* parent, const int32_t* depth,
                                        const int32_t* row_off, int32_t B, int32_t rows_total,
                                        int32_t* node_argmax, float* margin, int32_t* k_acc, int32_t* path,
                                        int32_t* bonus, cudaStream_t st) {
    void* scratch = nullptr;
    cudaError_t e = static_scratch_address(&scratch, st);
    if (e != cudaSuccess) return e;
    // the array keeps whatever the previous call left: the tickets must start at zero
    e = cudaMemsetAsync(scratch, 0, STATIC_TICKET_BYTES, st);
    if (e != cudaSuccess) return e;
    count_launch();
    unsigned int* tickets = (unsigned int*)scratch;
    Top* partial = (Top*)((char*)scratch + STATIC_TICKET_BYTES);
    dim3 grid(rows_total, ARGMAX_CHUNKS);
    DISPATCH_T(dtype, argmax_accept_kernel<T><<<grid, ARGMAX_THREADS, 0, st>>>(
                          (const T*)logits, V, tokens, parent, depth, row_off, B, node_argmax, margin, k_acc,
                          path, bonus, 1, tickets, partial));
    return cudaGetLastError();
}

cudaError_t launch_compact(void* k_cache, void* v_cache, int32_t L, int32_t B_cache, int32_t B, int32_t H,
                           int32_t max_seq, int32_t D, int32_t dtype, int32_t* seq_len,
                           const int32_t* k_acc, const int32_t* path, cudaStream_t st, unsigned int* tickets) {
    count_launch();
    const int row_vec = (int)(D * dtype_size(dtype) / 16);
    const size_t smem = sizeof(uint4) * COMPACT_BATCH * row_vec;
    cudaError_t e = launch_chain(compact_kernel, dim3(L * B * H * 2), dim3(256), smem, st, (uint4*)k_cache, (uint4*)v_cache,
                                 B_cache, B, H, max_seq, row_vec, seq_len, k_acc, path, tickets);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess || tickets) return e;
    // without a ticket array (the op-level call has no workspace) the lengths are advanced by a second kernel
    count_launch();
    e = launch_chain(advance_len_kernel, dim3((B + 63) / 64), dim3(64), 0, st, seq_len, k_acc, B);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_set_chunk(int32_t* row_off2, int32_t m, cudaStream_t st) {
    count_launch();
    set_chunk_kernel<<<1, 1, 0, st>>>(row_off2, m);
    return cudaGetLastError();
}
cudaError_t launch_prefill_geometry(const int32_t* seq_len_b, int32_t* lens, int32_t n_sub, int32_t sub, int32_t m,
                                    int32_t* off_all, int32_t* off_pieces, cudaStream_t st) {
    count_launch();
    prefill_geometry_kernel<<<1, 32, 0, st>>>(seq_len_b, lens, n_sub, sub, m, off_all, off_pieces);
    return cudaGetLastError();
}
cudaError_t launch_bump_len(int32_t* seq_len_b, int32_t delta, cudaStream_t st) {
    count_launch();
    bump_len_kernel<<<1, 1, 0, st>>>(seq_len_b, delta);
    return cudaGetLastError();
}

}  // namespace trj
