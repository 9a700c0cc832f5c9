// Preparation and finalisation kernels of the Gauss-sum path.
//
//  * common mean of all query and key points (the shift safeguard of
//    Remark 2, Sec. 2: the kernel depends on q - k only, so any common shift
//    is exact and only changes rounding), rounded to the input format's
//    grid so that the shift itself adds no rounding near the mean;
//  * centring, rounding to the MMA operand type and the scaled squared norms
//    A_m = -(c/2)||q^_m||^2, B_n = -(c/2)||k^_n||^2 (c = tau log2 e) taken
//    from the ROUNDED points, so that c q^.k^ + A_m + B_n is exactly
//    -(c/2)||q^_m - k^_n||^2 up to fp32 rounding (the norm factors of Alg. 1,
//    folded into one exponent);
//  * the value operand: per-channel power-of-two scaling of v (or of the
//    gradient values (v_n k_n, v_n) of Sec. 3) rounded to fp16 and stored
//    transposed (channel-major) so that both MMAs read K-major operands;
//  * the fixed-order sum of key-split partials and the final scaling, or
//    the gradient tau (S[:D] - q_m S[D]) of Sec. 3.
#include <algorithm>
#include <type_traits>

#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math_constants.h>

#include "internal.h"
#include "ptx.cuh"

namespace gs {
namespace {

template <typename T> __device__ __forceinline__ float to_f(T x);
template <> __device__ __forceinline__ float to_f<float>(float x) { return x; }
template <> __device__ __forceinline__ float to_f<__half>(__half x) { return __half2float(x); }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 x) {
    return __bfloat162float(x);
}

// a / b for a non-negative a below 2^32 with 32-bit division (much
// cheaper than the 64-bit one), else 64-bit.
__device__ __forceinline__ int64_t div_nonneg(int64_t a, int b) {
    if (a <= 0xffffffffLL)
        return static_cast<int64_t>(static_cast<uint32_t>(a) / static_cast<uint32_t>(b));
    return a / b;
}

template <typename H> __device__ __forceinline__ H from_f(float x);
template <> __device__ __forceinline__ __half from_f<__half>(float x) { return __float2half_rn(x); }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float x) {
    return __float2bfloat16_rn(x);
}

// ---------------------------------------------------------------- mean
// Block (32, 8): 32 consecutive coordinates x 8 row lanes; each block sums
// a contiguous chunk of the stacked rows [q; k] and writes, per coordinate,
// its partial sum (partial[block][d]) and largest magnitude
// (partial[G + block][d]).
template <typename T>
__global__ void mean_partial_kernel(const T* __restrict__ q, const T* __restrict__ k, int64_t M,
                                    int64_t N, int D, int64_t rows_per_block,
                                    float* __restrict__ partial) {
    pdl_trigger();
    pdl_wait();
    __shared__ float red[8][33];
    __shared__ float big[8][33];
    // Problem blockIdx.y of a batch: its own points and partial rows.
    q += static_cast<int64_t>(blockIdx.y) * M * D;
    k += static_cast<int64_t>(blockIdx.y) * N * D;
    partial += static_cast<int64_t>(blockIdx.y) * 2 * gridDim.x * D;
    const int64_t r0 = static_cast<int64_t>(blockIdx.x) * rows_per_block;
    const int64_t r1 = min(r0 + rows_per_block, M + N);
    for (int d0 = 0; d0 < D; d0 += 32) {
        const int d = d0 + threadIdx.x;
        float acc = 0.f, mx = 0.f;
        if (d < D) {
            for (int64_t r = r0 + threadIdx.y; r < r1; r += 8) {
                const float x = to_f(r < M ? q[r * D + d] : k[(r - M) * D + d]);
                acc += x;
                mx = fmaxf(mx, fabsf(x));
            }
        }
        red[threadIdx.y][threadIdx.x] = acc;
        big[threadIdx.y][threadIdx.x] = mx;
        __syncthreads();
        if (threadIdx.y == 0 && d < D) {
            float sum = 0.f, m = 0.f;
#pragma unroll
            for (int y = 0; y < 8; ++y) {
                sum += red[y][threadIdx.x];
                m = fmaxf(m, big[y][threadIdx.x]);
            }
            partial[static_cast<int64_t>(blockIdx.x) * D + d] = sum;
            partial[static_cast<int64_t>(gridDim.x + blockIdx.x) * D + d] = m;
        }
        __syncthreads();
    }
}

// Vectorised variant for 16-bit inputs with D a power of two in [8, 2048]:
// 256 threads read 16-byte vectors (8 coordinates) of a contiguous run of
// rows; a block advances by 2048 elements, a multiple of D, so every thread
// always sees the same 8 coordinates and keeps their sums and maxima in
// registers.  Blocks [0, Gq) cover rows of q, blocks [Gq, G) rows of k
// (none when q and k are the same points).  Same partial layout as above.
// Blocks from G on, when given a record job, write the FMA kernel's key
// records instead (see key_record_kernel): they depend on the values only,
// so they ride along in this first launch of the call rather than taking
// a launch of their own later in the chain.
constexpr int kMeanVecThreads = 256;

// How the rows of [q; k] are split into partial sums (see mean_split).
struct MeanSplit {
    bool vec;            // mean_partial_vec_kernel's split, else mean_partial_rows_kernel's
    int64_t rpb;         // rows per partial
    int Gq, G;           // partials of q (vec), of both
};

template <typename TV>
struct RecordJob {
    const TV* v;         // N x C values per problem (batch-stacked)
    int64_t N, pairs;    // keys and key pairs (Npad / 2) per problem
    int C;
    float* rec;          // pairs x 2C floats per problem
    bool signs;          // sign records (see sign_record) instead of values
};

// Sign records of the FMA kernel with folded value magnitudes (C = 1, the
// magnitudes sit in the key operands): per key tile of kRecTile keys, the
// floats s_n = sign(v_n) 2^16 in key order (0 for v_n = 0 and for padded
// keys), then one word per group of 32 keys: -2^16 if the group's nonzero
// values are all negative, 0 if it has values of both signs, else 2^16.
// One thread per key n < Npad of problem `problem`, whole warps per group.
constexpr int kRecTile = 128;
constexpr int kRecTileFloats = kRecTile + kRecTile / 32;

__device__ __forceinline__ void write_sign_record(const __half* v, int64_t N, float* rec, int64_t n,
                                                  int problem, int64_t npad) {
    const float x = n < N ? __half2float(v[static_cast<int64_t>(problem) * N + n]) : 0.f;
    const float sg = x > 0.f ? 65536.f : x < 0.f ? -65536.f : 0.f;
    float* r = rec + (static_cast<int64_t>(problem) * (npad / kRecTile) + n / kRecTile) * kRecTileFloats;
    const int kn = static_cast<int>(n % kRecTile);
    r[kn] = sg;
    // Zero values and padded keys contribute nothing whatever the group's
    // sign (their folded exponent flushes), so only the signs of the
    // nonzero values decide.
    const bool any_pos = __any_sync(0xffffffffu, x > 0.f);
    const bool any_neg = __any_sync(0xffffffffu, x < 0.f);
    if ((kn & 31) == 0) r[kRecTile + kn / 32] = any_pos && any_neg ? 0.f : any_neg ? -65536.f : 65536.f;
}

// One block per problem b: the AND over its 32-key groups of "values of
// one sign" (group word != 0), into the word after all problems' records.
// Every thread of the block calls this.
__device__ __forceinline__ void write_vf_flag(float* __restrict__ rec, int64_t tiles, int batch, int b) {
    const float* gw = rec + static_cast<int64_t>(b) * tiles * kRecTileFloats + kRecTile;
    bool mixed = false;
    for (int64_t i = threadIdx.x; i < tiles * (kRecTile / 32); i += blockDim.x)
        mixed |= gw[(i / (kRecTile / 32)) * kRecTileFloats + i % (kRecTile / 32)] == 0.f;
    const int any_mixed = __syncthreads_or(mixed ? 1 : 0);
    if (threadIdx.x == 0)
        reinterpret_cast<unsigned*>(rec + static_cast<int64_t>(batch) * tiles * kRecTileFloats)[b] =
            any_mixed ? 0u : 1u;
}

__global__ void __launch_bounds__(256)
vf_flags_kernel(float* __restrict__ rec, int64_t tiles, int batch) {
    pdl_trigger();
    pdl_wait();
    write_vf_flag(rec, tiles, batch, blockIdx.x);
}

__global__ void sign_record_kernel(const __half* __restrict__ v, int64_t N, int64_t npad,
                                   float* __restrict__ rec) {
    pdl_trigger();
    pdl_wait();
    const int64_t n = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (n < npad) write_sign_record(v, N, rec, n, blockIdx.y, npad);
}

template <typename TV>
__device__ __forceinline__ void write_key_record(const RecordJob<TV>& j, int64_t t, int problem) {
    const int64_t n0 = 2 * t, n1 = 2 * t + 1;
    const TV* v = j.v + static_cast<int64_t>(problem) * j.N * j.C;
    float* out = j.rec + (static_cast<int64_t>(problem) * j.pairs + t) * (2 * j.C);
    for (int c = 0; c < j.C; ++c) {
        out[2 * c] = n0 < j.N ? to_f(v[n0 * j.C + c]) : 0.f;
        out[2 * c + 1] = n1 < j.N ? to_f(v[n1 * j.C + c]) : 0.f;
    }
}

// Thread t of the blocks that write records instead of partial sums: key record
// t, or the sign record of key t.
template <typename TV>
__device__ __forceinline__ void write_record(const RecordJob<TV>& rj, int64_t t, int problem) {
    if (rj.signs) {
        if constexpr (std::is_same<TV, __half>::value) {
            if (t < 2 * rj.pairs) write_sign_record(rj.v, rj.N, rj.rec, t, problem, 2 * rj.pairs);
        }
    } else if (t < rj.pairs) {
        write_key_record(rj, t, problem);
    }
}

struct MeanShared {
    float sum[kMeanVecThreads][9];
    float max[kMeanVecThreads][9];
};

// Partial sums and maxima of block `block` of the split, by the whole thread
// block, into D values each.
template <typename T>
__device__ __forceinline__ void mean_vec_block(const T* __restrict__ q, const T* __restrict__ k, int64_t M,
                                               int64_t N, int D, int64_t rows_per_block, int Gq, int block,
                                               MeanShared& sh, float* out_sum, float* out_max) {
    auto& s_sum = sh.sum;
    auto& s_max = sh.max;
    const int t = threadIdx.x;
    const bool on_q = block < Gq;
    const int64_t b = on_q ? block : block - Gq;
    const int64_t rows = on_q ? M : N;
    const T* x = on_q ? q : k;
    const int64_t r0 = b * rows_per_block;
    const int64_t r1 = min(r0 + rows_per_block, rows);
    const int64_t v0 = r0 * D / 8, v1 = r1 * D / 8;      // 8-element vectors
    const uint4* xv = reinterpret_cast<const uint4*>(x);
    float sum[8], mx[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) sum[e] = mx[e] = 0.f;
    // Four vectors in flight per thread, then the remainder one at a time
    // (each thread's vectors are accumulated in index order either way).
    auto add = [&](const uint4 u) {
        const T* h = reinterpret_cast<const T*>(&u);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float f = to_f(h[e]);
            sum[e] += f;
            mx[e] = fmaxf(mx[e], fabsf(f));
        }
    };
    int64_t v = v0 + t;
    for (; v + 3 * kMeanVecThreads < v1; v += 4 * kMeanVecThreads) {
        uint4 u[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) u[r] = xv[v + r * kMeanVecThreads];
#pragma unroll
        for (int r = 0; r < 4; ++r) add(u[r]);
    }
    for (; v < v1; v += kMeanVecThreads) add(xv[v]);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        s_sum[t][e] = sum[e];
        s_max[t][e] = mx[e];
    }
    __syncthreads();
    // Thread t holds coordinates 8 (t mod NG) .. +7, NG = D / 8 groups.
    const int NG = D / 8;
    // (Sums and maxima by different threads: D is often a quarter of the block.)
    for (int i = t; i < 2 * D; i += kMeanVecThreads) {
        const int d = i < D ? i : i - D;
        const int g = d >> 3, e = d & 7;
        float a = 0.f;
        if (i < D) {
#pragma unroll 8
            for (int u = g; u < kMeanVecThreads; u += NG) a += s_sum[u][e];
            out_sum[d] = a;
        } else {
#pragma unroll 8
            for (int u = g; u < kMeanVecThreads; u += NG) a = fmaxf(a, s_max[u][e]);
            out_max[d] = a;
        }
    }
}

template <typename T, typename TV>
__global__ void __launch_bounds__(kMeanVecThreads)
mean_partial_vec_kernel(const T* __restrict__ q, const T* __restrict__ k, int64_t M, int64_t N,
                        int D, int64_t rows_per_block, int Gq, int G, float* __restrict__ partial,
                        const RecordJob<TV> rj) {
    pdl_trigger();
    pdl_wait();
    if (static_cast<int>(blockIdx.x) >= G) {
        write_record(rj, static_cast<int64_t>(blockIdx.x - G) * kMeanVecThreads + threadIdx.x, blockIdx.y);
        return;
    }
    // Problem blockIdx.y of a batch: its own points and partial rows.
    __shared__ MeanShared sh;
    partial += static_cast<int64_t>(blockIdx.y) * 2 * G * D;
    mean_vec_block(q + static_cast<int64_t>(blockIdx.y) * M * D, k + static_cast<int64_t>(blockIdx.y) * N * D,
                   M, N, D, rows_per_block, Gq, static_cast<int>(blockIdx.x), sh,
                   partial + static_cast<int64_t>(blockIdx.x) * D,
                   partial + static_cast<int64_t>(G + blockIdx.x) * D);
}

// Any other width up to 256 (16-bit inputs): the partial sums and maxima of
// mean_partial_kernel, in the same order of additions (bit for bit), read in
// 16-byte vectors.  Eight rows are D vectors, and a block of
// mean_partial_kernel adds up every eighth row, so thread t of the D threads
// of a chunk (one block's rows there) owns vector t of each group of eight
// rows: its eight elements are of fixed (row mod 8, coordinate) all along.
// Chunks that do not start on 16 bytes take narrower loads; groups that
// straddle q and k or end with the chunk are read element by element.  A block holds `chunks` chunks of D
// threads; blocks from mblocks on write key records (see RecordJob).
// Bound: load latency (ncu, with the records: 50021 points of D = 50 6.4 us,
// where mean_partial_kernel took 7.2 us and the records and their flags two
// more launches, 7.5 us).
// Chunks [chunk0, chunk0 + chunks) of the split into G, by the whole thread
// block; put(chunk, d, sum, max) takes the results.
template <typename T, typename Put>
__device__ __forceinline__ void mean_rows_block(const T* __restrict__ q, const T* __restrict__ k, int64_t M,
                                                int64_t N, int D, int64_t rows_per_block, int G, int chunks,
                                                int chunk0, MeanShared& sh, Put put) {
    auto& s_sum = sh.sum;
    auto& s_max = sh.max;
    const int local = static_cast<int>(threadIdx.x) / D;     // chunk of this block
    const int t = static_cast<int>(threadIdx.x) - local * D;
    const int chunk = chunk0 + local;
    float sum[8], mx[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) sum[e] = mx[e] = 0.f;
    if (local < chunks && chunk < G) {
        const int64_t r0 = static_cast<int64_t>(chunk) * rows_per_block;
        const int64_t r1 = min(r0 + rows_per_block, M + N);
        auto add = [&](const uint4 u) {
            const T* h = reinterpret_cast<const T*>(&u);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float f = to_f(h[e]);
                sum[e] += f;
                mx[e] = fmaxf(mx[e], fabsf(f));
            }
        };
        // Whole groups of eight rows from r on: in q up to M, in k after it; in
        // the widest loads that the first row's address allows.
        auto groups = [&](int64_t r, int64_t end) {
            const T* x = (r < M ? q : k - M * D) + r * D + 8 * t;
            const int64_t n = (end - r) / 8;
            const int64_t step = 8 * static_cast<int64_t>(D);
            auto walk = [&](auto tag) {
                using L = decltype(tag);
                constexpr int PER = 16 / static_cast<int>(sizeof(L));
                auto load = [&](const T* p) {
                    uint4 u;
                    L* w = reinterpret_cast<L*>(&u);
#pragma unroll
                    for (int i = 0; i < PER; ++i) w[i] = reinterpret_cast<const L*>(p)[i];
                    return u;
                };
                int64_t g = 0;
                for (; g + 8 <= n; g += 8, x += 8 * step) {
                    uint4 u[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) u[i] = load(x + i * step);
#pragma unroll
                    for (int i = 0; i < 8; ++i) add(u[i]);
                }
                for (; g < n; ++g, x += step) add(load(x));
            };
            const unsigned at = static_cast<unsigned>(reinterpret_cast<uintptr_t>(x)) & 15u;
            if (at == 0) walk(uint4());
            else if ((at & 7u) == 0) walk(uint2());
            else if ((at & 3u) == 0) walk(unsigned());
            else walk(static_cast<unsigned short>(0));
            return r + 8 * n;
        };
        // One group (or what is left of it), element by element.
        auto single = [&](int64_t r) {
            for (int e = 0; e < 8; ++e) {
                const int i = 8 * t + e;
                const int64_t row = r + i / D;
                if (row < r1) {
                    const int d = i % D;
                    const float f = to_f(row < M ? q[row * D + d] : k[(row - M) * D + d]);
                    sum[e] += f;
                    mx[e] = fmaxf(mx[e], fabsf(f));
                }
            }
        };
        int64_t r = r0;
        while (r < r1) {
            const int64_t end = r < M ? min(r1, M) : r1;
            const int64_t next = groups(r, end);
            if (next == r) {
                single(r);
                r += 8;
            } else {
                r = next;
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        s_sum[threadIdx.x][e] = sum[e];
        s_max[threadIdx.x][e] = mx[e];
    }
    __syncthreads();
    if (local >= chunks || chunk >= G) return;
    // Coordinate t of the chunk: rows 0 .. 7 (mod 8) in order.
    float a = 0.f, m = 0.f;
#pragma unroll
    for (int y = 0; y < 8; ++y) {
        const int i = y * D + t, u = local * D + (i >> 3), e = i & 7;
        a += s_sum[u][e];
        m = fmaxf(m, s_max[u][e]);
    }
    put(chunk, t, a, m);
}

template <typename T, typename TV>
__global__ void __launch_bounds__(kMeanVecThreads)
mean_partial_rows_kernel(const T* __restrict__ q, const T* __restrict__ k, int64_t M, int64_t N,
                         int D, int64_t rows_per_block, int G, int chunks, int mblocks,
                         float* __restrict__ partial, const RecordJob<TV> rj) {
    pdl_trigger();
    pdl_wait();
    if (static_cast<int>(blockIdx.x) >= mblocks) {
        write_record(rj, static_cast<int64_t>(blockIdx.x - mblocks) * kMeanVecThreads + threadIdx.x, blockIdx.y);
        return;
    }
    // Problem blockIdx.y of a batch: its own points and partial rows.
    __shared__ MeanShared sh;
    partial += static_cast<int64_t>(blockIdx.y) * 2 * G * D;
    mean_rows_block(q + static_cast<int64_t>(blockIdx.y) * M * D, k + static_cast<int64_t>(blockIdx.y) * N * D,
                    M, N, D, rows_per_block, G, chunks, static_cast<int>(blockIdx.x) * chunks, sh,
                    [&](int chunk, int d, float sum, float mx) {
                        partial[static_cast<int64_t>(chunk) * D + d] = sum;
                        partial[static_cast<int64_t>(G + chunk) * D + d] = mx;
                    });
}

// mu_d = the mean of coordinate d rounded to a multiple of g_d, the spacing
// of the input format at max |x_d| (2^(e - mant_bits) for max |x_d| in
// [2^e, 2^(e+1)), at least the subnormal spacing 2^min_exp).  Every input
// x_d is a multiple of its own spacing, which divides g_d, so x_d - mu_d is
// a multiple of the spacing of x_d: it is exact in the input format
// whenever |x_d - mu_d| stays below 2^(e_x + 1) (x_d in [2^e_x, 2^(e_x+1))),
// i.e. the shift adds no rounding for points near the mean.  Any common
// shift leaves the Gauss sum unchanged.
constexpr int kMeanFinalThreads = 256;

// The grid-rounded mean of the folded sum s and largest magnitude mx.
__device__ __forceinline__ float rounded_mean(float s, float mx, float total, int mant_bits,
                                              int min_exp) {
    // float32 throughout: any shift is exact for the Gauss sum, so the mean
    // needs no more precision than that, and float64 is slow on this GPU.
    float m = s / total;
    if (mx > 0.f) {
        int e;
        frexpf(mx, &e);                                   // mx in [2^(e-1), 2^e)
        const float g = ldexpf(1.f, max(e - 1 - mant_bits, min_exp));
        m = rintf(m / g) * g;
    }
    return m;
}

// Many partials per coordinate (G > kMeanFinalThreadMax): one block per
// (coordinate d, problem blockIdx.y); thread t folds partials t, t + 256,
// ... in order, a fixed butterfly adds the lanes of each warp and thread 0
// the warps in order (deterministic).
constexpr int kMeanFinalThreadMax = 32;

__global__ void __launch_bounds__(kMeanFinalThreads)
mean_final_block_kernel(const float* __restrict__ partial, int G, int D, float total,
                        int mant_bits, int min_exp, float* __restrict__ mu,
                        const ZeroWords zero) {
    pdl_trigger();
    pdl_wait();
    if (blockIdx.x == 0 && blockIdx.y == 0)
        for (int i = threadIdx.x; i < zero.n; i += kMeanFinalThreads) zero.p[i] = 0u;
    constexpr int W = kMeanFinalThreads / 32;
    __shared__ float red_s[W];
    __shared__ float red_m[W];
    const int d = blockIdx.x;
    const int t = threadIdx.x;
    partial += static_cast<int64_t>(blockIdx.y) * 2 * G * D;
    mu += static_cast<int64_t>(blockIdx.y) * D;
    float s = 0.f;
    float mx = 0.f;
    for (int g = t; g < G; g += kMeanFinalThreads) {
        s += partial[static_cast<int64_t>(g) * D + d];
        mx = fmaxf(mx, partial[static_cast<int64_t>(G + g) * D + d]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if ((t & 31) == 0) {
        red_s[t >> 5] = s;
        red_m[t >> 5] = mx;
    }
    __syncthreads();
    if (t == 0) {
        float a = 0.f, m = 0.f;
        for (int w = 0; w < W; ++w) {
            a += red_s[w];
            m = fmaxf(m, red_m[w]);
        }
        mu[d] = rounded_mean(a, m, total, mant_bits, min_exp);
    }
}

// Few partials per coordinate (the small problems of a batch): one thread
// per item = (problem b, coordinate d), folding the G partials in order.
// Bound: the latency of its loads, which a loop over G pays for every few
// partials, so sixteen of each kind are in flight together. Whole calls,
// one GB300, with mean_vec_block's tail split over the block: 64 problems of
// 2000 points (MMD^2) 62.5 -> 60.2 us, 64 x 4096^2, D = 64 243.3 -> 241.9 us.
constexpr int kMeanFinalLoads = 16;

__global__ void __launch_bounds__(kMeanFinalThreads)
mean_final_kernel(const float* __restrict__ partial, int G, int D, int64_t items, float total,
                  int mant_bits, int min_exp, float* __restrict__ mu,
                  const ZeroWords zero) {
    pdl_trigger();
    pdl_wait();
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < zero.n; i += kMeanFinalThreads) zero.p[i] = 0u;
    const int64_t it = static_cast<int64_t>(blockIdx.x) * kMeanFinalThreads + threadIdx.x;
    if (it >= items) return;
    const int64_t b = it / D;
    const int d = static_cast<int>(it - b * D);
    partial += b * 2 * G * D;                      // problem b
    float s = 0.f;
    float mx = 0.f;
    for (int g0 = 0; g0 < G; g0 += kMeanFinalLoads) {
        float a[kMeanFinalLoads], m[kMeanFinalLoads];
#pragma unroll
        for (int i = 0; i < kMeanFinalLoads; ++i) {
            const bool in = g0 + i < G;
            a[i] = in ? partial[static_cast<int64_t>(g0 + i) * D + d] : 0.f;
            m[i] = in ? partial[static_cast<int64_t>(G + g0 + i) * D + d] : 0.f;
        }
        // (Zeros past G change neither: s starts at +0 and maxima are of magnitudes.)
#pragma unroll
        for (int i = 0; i < kMeanFinalLoads; ++i) {
            s += a[i];
            mx = fmaxf(mx, m[i]);
        }
    }
    mu[it] = rounded_mean(s, mx, total, mant_bits, min_exp);
}

// ---------------------------------------------------------------- MMA operands
// Both operand layouts are written by one kernel that stages kRowsPerBlock
// rows through shared memory: the block's input rows are one contiguous
// run of rows x D elements (16-byte vector loads), and its output rows one
// contiguous run of rows x Dp elements (16-byte vector stores).  One warp
// per row inside the block.
//
// Plain layout (AUG = false): centred points rounded to the MMA type,
// x^ = rn(x - mu), zero padded to Dp columns, and the scaled squared norm
// nrm = -(c/2)||x^||^2 (c = tau log2 e) taken from the ROUNDED point, so that
// c q^.k^ + A_m + B_n is exactly -(c/2)||q^_m - k^_n||^2 up to fp32
// rounding (the norm factors of Alg. 1 folded into one exponent).  Rows in
// [rows, rows_pad) become zero rows with norm `pad_value` (-inf for padded
// keys, so their kernel value is 0).
//
// Augmented layout (AUG = true): x^ followed by 2 NT columns that make the
// MMA produce the whole exponent up to the factor c:
//   query rows  [q^, F, 1, .., 1, a_0, a_1, .., a_NT-1, 0 ...]
//   key rows    [k^, b_0, b_1, .., b_NT-1, F, 1, .., 1, 0 ...]
// with a = -||q^||^2 / 2 and b = -||k^||^2 / 2 taken from the rounded
// points in fp32 and written as F t_0 + t_1 + ... + t_NT-1, each t_i a
// rounded remainder, so that
//   q^_aug . k^_aug = q^.k^ + a + b = -||q^ - k^||^2 / 2
// up to the split error (|a| 2^-22 for two fp16 terms, |a| 2^-24 for three
// bf16 terms) and the fp32 accumulation; the kernel value is 2^(c S).  The
// power of two F (1024 for fp16) keeps norms up to 6.7e7 inside the fp16
// range.  Padded key rows get b_0 = -30000 / F (their values are zero as
// well); padded query rows are zero.  `out_q` and/or `out_k` may be given
// (both for q = k).
//
// Folded exponent scale and value magnitudes (cf = c > 0, one fp16 value
// per key in vw): the query rows hold u = rn(c q^), with a = -||u||^2/(2c),
// and the key rows b = -c ||k^||^2 / 2 + log2(|v_n| 2^-16), so that the MMA
// yields S = u.k^ + a + b = -(1/(2c)) ||u - c k^||^2 + log2(|v_n| 2^-16):
// the exponent of Phi |v_n| 2^-16 itself, at the query point u / c (within
// 2^-12 of q^ per coordinate), and never above log2(|v_n| 2^-16) in exact
// arithmetic.  The FMA kernel then needs no multiply by c and only the
// signs of the values (see write_sign_record).  |v_n| < 2^16 for every
// finite fp16 value.  Keys with v_n = 0 get -256: their 2^S flushes to
// zero, so they may sit in a group of either sign (padded keys have
// -30000 already).
constexpr float kZeroWeightLog2 = -256.f;

__device__ __forceinline__ float log_weight(const __half* vw) {
    if (!vw) return 0.f;
    const float a = fabsf(__half2float(*vw));
    return a > 0.f ? log2f(a * (1.f / 65536.f)) : kZeroWeightLog2;
}

constexpr int kRowsPerBlock = 32;
constexpr int kOperandThreads = 128;
constexpr int kOperandMaxCols = 256;

// (The vector path below takes every call but those of D = 0 and of 2^30 rows.)

template <typename T, bool AUG>
__global__ void __launch_bounds__(kOperandThreads)
operand_kernel(const T* __restrict__ x, int64_t rows, int64_t rows_pad, int D, int Dp, int nt, float F,
               const float* __restrict__ mu, float half_c, float pad_value,
               T* __restrict__ out_q, T* __restrict__ out_k, float* __restrict__ nrm,
               const __half* __restrict__ vw, float cf) {
    pdl_trigger();
    pdl_wait();
    constexpr int R = kRowsPerBlock;
    // Dynamic shared memory sized to this call: s_out holds R x Dp
    // elements per written layout (AUG: q rows, then k rows), s_in the R x D
    // input elements (rounded up to 16 bytes), then D floats of mu.
    extern __shared__ __align__(16) uint8_t operand_smem[];
    const bool wq = AUG ? out_q != nullptr : true;
    const bool wk = AUG && out_k != nullptr;
    const int nout = (wq ? 1 : 0) + (wk ? 1 : 0);
    T* s_out = reinterpret_cast<T*>(operand_smem);
    T* s_in = s_out + nout * R * Dp;
    float* s_mu = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(s_in) +
                                           ((R * D * static_cast<int>(sizeof(T)) + 15) & ~15));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // Problem blockIdx.y of a batch: its own rows, mean and outputs.
    {
        const int64_t b = blockIdx.y;
        x += b * rows * D;
        if (mu) mu += b * D;
        if (out_q) out_q += b * rows_pad * Dp;
        if (out_k) out_k += b * rows_pad * Dp;
        if (nrm) nrm += b * rows_pad;
        if (vw) vw += b * rows;
    }
    const int64_t r0 = static_cast<int64_t>(blockIdx.x) * R;
    for (int d = tid; d < D; d += kOperandThreads) s_mu[d] = mu ? mu[d] : 0.f;
    const int64_t left = rows - r0;
    const int rin = left <= 0 ? 0 : left >= R ? R : static_cast<int>(left);
    {
        // The block's rows are one run of rin x D elements.  Within one
        // problem its start (r0 D sizeof(T), r0 a multiple of 32) is 16-byte
        // aligned; a later problem of a batch may start anywhere, so the
        // vector loads are used only when the run is 16-byte aligned.
        const int n_el = rin * D;
        constexpr int PER_VEC = 16 / static_cast<int>(sizeof(T));
        const T* src = x + r0 * D;
        const int nvec = (reinterpret_cast<uintptr_t>(src) & 15u) == 0 ? n_el / PER_VEC : 0;
        for (int i = tid; i < nvec; i += kOperandThreads)
            reinterpret_cast<uint4*>(s_in)[i] = reinterpret_cast<const uint4*>(src)[i];
        for (int i = nvec * PER_VEC + tid; i < n_el; i += kOperandThreads) s_in[i] = src[i];
    }
    __syncthreads();
    T* sq = s_out;
    T* sk = s_out + (wq ? R * Dp : 0);
    const T zero = from_f<T>(0.f);
    for (int row = warp; row < R; row += kOperandThreads / 32) {
        const bool valid = row < rin;
        T* oq = sq + row * Dp;
        T* ok = sk + row * Dp;
        float acc = 0.f, accu = 0.f;
        const bool fold = AUG && cf > 0.f;
        const int dend = AUG ? D : Dp;
        for (int d = lane; d < dend; d += 32) {
            const float val = (valid && d < D) ? to_f(s_in[row * D + d]) - s_mu[d] : 0.f;
            const T h = from_f<T>(val);
            const float hf = to_f(h);
            if (fold) {
                const T hs = from_f<T>(cf * hf);   // folded scale: the query row holds rn(c x^)
                if (wq) oq[d] = hs;
                accu = fmaf(to_f(hs), to_f(hs), accu);
            } else if (wq) {
                oq[d] = h;
            }
            if (wk) ok[d] = h;
            acc = fmaf(hf, hf, acc);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            acc += __shfl_xor_sync(0xffffffffu, acc, o);
            accu += __shfl_xor_sync(0xffffffffu, accu, o);
        }
        if (!AUG) {
            if (lane == 0) nrm[r0 + row] = valid ? -half_c * acc : pad_value;
            continue;
        }
        for (int d = D + 2 * nt + lane; d < Dp; d += 32) {
            if (wq) oq[d] = zero;
            if (wk) ok[d] = zero;
        }
        if (lane < nt) {
            // Lane i writes term i of the split and its partner column (the
            // key side with its log weight, when values are folded).
            auto split_term = [&](float r) {
                T t = from_f<T>(r / F);
                r -= F * to_f(t);
                for (int i = 1; i <= lane; ++i) {
                    t = from_f<T>(r);
                    r -= to_f(t);
                }
                return t;
            };
            T t = zero, tk = zero, one = zero;
            if (valid) {
                if (fold) {
                    t = split_term(-0.5f * accu / cf);
                    tk = split_term(-0.5f * cf * acc + log_weight(vw ? vw + r0 + row : nullptr));
                } else {
                    t = tk = split_term(-0.5f * acc);
                }
                one = from_f<T>(lane == 0 ? F : 1.f);
            } else if (lane == 0) {
                t = tk = from_f<T>(-30000.f / F);
            }
            if (wq) {
                oq[D + lane] = valid ? one : zero;
                oq[D + nt + lane] = valid ? t : zero;
            }
            if (wk) {
                ok[D + lane] = tk;
                ok[D + nt + lane] = one;
            }
        }
    }
    __syncthreads();
    // r0 Dp sizeof(T) is a multiple of 16 (Dp is a multiple of 16).
    const int nvec = R * Dp * static_cast<int>(sizeof(T)) / 16;
    if (wq) {
        uint4* dst = reinterpret_cast<uint4*>(out_q + r0 * Dp);
        for (int i = tid; i < nvec; i += kOperandThreads) dst[i] = reinterpret_cast<const uint4*>(sq)[i];
    }
    if (wk) {
        uint4* dst = reinterpret_cast<uint4*>(out_k + r0 * Dp);
        for (int i = tid; i < nvec; i += kOperandThreads) dst[i] = reinterpret_cast<const uint4*>(sk)[i];
    }
}

// 3xTF32 operands (fp32 inputs on the tensor cores).  Row r of problem b
// becomes 2 Dp floats [hi_0 .. hi_Dp-1, lo_0 .. lo_Dp-1] with
// x^ = x - mu (fp32), hi = x^ rounded to tf32 and lo = (x^ - hi) rounded to
// tf32, zero padded; q^.k^ is then hi.hi + hi.lo + lo.hi up to the dropped
// lo.lo term (2^-22 relative).  nrm = -(c/2) ||x^||^2 from the fp32 x^;
// rows in [rows, rows_pad) are zero with norm pad_value.  Rows of job j0 (all
// problems), then of j1, in one launch; rows_pad is a multiple of 128, so the
// kSplitRows rows of a warp are of one problem and job.  Bound: HBM, but for
// the loads' latency: one row per warp took 303 us for 2^20 rows of D = 32
// (1.3 TB/s), with the job and problem worked out again for each; whole call
// (32 keys) 448 -> 263 us.  The key records ride along.
constexpr int kSplitRows = 8;
constexpr int kSplitThreads = 256;

template <int P>   // Dp = 32 P
__global__ void __launch_bounds__(kSplitThreads)
tf32_split_kernel(const Tf32Job j0, const Tf32Job j1, int64_t total0, int64_t total_rows, int D,
                  const float* __restrict__ mu, float half_c, float pad_value,
                  unsigned* __restrict__ guard, const RecordJob<float> rec) {
    pdl_trigger();
    pdl_wait();
    constexpr int Dp = 32 * P;
    // guard: the largest (c/2) ||x - mu||^2, as the bits of a non-negative
    // float (or of a NaN, above them all), which order like the floats.
    __shared__ unsigned big;
    if (guard) {
        if (threadIdx.x == 0) big = 0u;
        __syncthreads();
    }
    const int64_t w = ((static_cast<int64_t>(blockIdx.x) * kSplitThreads + threadIdx.x) >> 5) * kSplitRows;
    const int lane = threadIdx.x & 31;
    if (w < total_rows) {
        const bool second = w >= total0;
        const float* x = second ? j1.x : j0.x;
        float* out = second ? j1.out : j0.out;
        float* nrm = second ? j1.nrm : j0.nrm;
        const int64_t rows = second ? j1.rows : j0.rows, pad = second ? j1.rows_pad : j0.rows_pad;
        const int64_t i0 = second ? w - total0 : w;        // first batch-stacked output row
        const int64_t b = pad <= 0x7fffffff ? div_nonneg(i0, static_cast<int>(pad)) : i0 / pad;
        const int64_t r0 = i0 - b * pad;
        x += (b * rows + r0) * D + lane;
        out += i0 * 2 * Dp + lane;
        const int left = static_cast<int>(min(static_cast<int64_t>(kSplitRows), rows - r0));
        float m[P], v[kSplitRows][P], acc[kSplitRows];
#pragma unroll
        for (int p = 0; p < P; ++p) m[p] = mu && lane + 32 * p < D ? mu[b * D + lane + 32 * p] : 0.f;
#pragma unroll
        for (int r = 0; r < kSplitRows; ++r)
#pragma unroll
            for (int p = 0; p < P; ++p)
                v[r][p] = r < left && lane + 32 * p < D ? x[r * D + 32 * p] - m[p] : 0.f;
#pragma unroll
        for (int r = 0; r < kSplitRows; ++r) {
            acc[r] = 0.f;
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const float hi = round_tf32(v[r][p]);
                out[r * 2 * Dp + 32 * p] = hi;
                out[r * 2 * Dp + Dp + 32 * p] = round_tf32(v[r][p] - hi);
                acc[r] = fmaf(v[r][p], v[r][p], acc[r]);
            }
        }
#pragma unroll
        for (int s = 16; s > 0; s >>= 1)
#pragma unroll
            for (int r = 0; r < kSplitRows; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], s);
        unsigned most = 0u;
        float norm = 0.f;                                  // of row i0 + lane
#pragma unroll
        for (int r = 0; r < kSplitRows; ++r) {
            if (lane == r) norm = r < left ? -half_c * acc[r] : pad_value;
            if (r < left) most = max(most, __float_as_uint(half_c * acc[r]) & 0x7fffffffu);
        }
        if (lane < kSplitRows) nrm[i0 + lane] = norm;
        if (guard && lane == 0) atomicMax(&big, most);
        if (second || j1.x == nullptr) {
            // Keys: their records (quads, see key_record_kernel), of which B are
            // the norm terms; kSplitRows / 4 quads of 1 + C groups of four floats.
            float* q = rec.rec + (i0 >> 2) * (4 + 4 * rec.C);
            const int items = (1 + rec.C) * kSplitRows;
            for (int t0 = 0; t0 < items; t0 += 32) {
                const int t = t0 + lane;
                const int quad = t / (4 + 4 * rec.C), e = t - quad * (4 + 4 * rec.C);
                const int r = 4 * quad + (e & 3), c = (e >> 2) - 1;
                const float B = __shfl_sync(0xffffffffu, norm, r);
                if (t < items) q[t] = c < 0 ? B : r < left ? rec.v[(b * rows + r0 + r) * rec.C + c] : 0.f;
            }
        }
    }
    if (guard) {
        __syncthreads();
        if (threadIdx.x == 0) atomicMax(guard, big);
    }
}

// Contributor slots of pair of query tiles r of the FMA kernel (see
// launch_finalize_slots in internal.h).
__device__ __forceinline__ int64_t contributor_slots(int64_t r, int fixed_slots, int64_t key_tiles,
                                                     int64_t unit_len, int64_t tri_kt) {
    if (fixed_slots > 0) return fixed_slots;
    if (tri_kt > 0) {
        // Upper-triangle order (folded rows of tri_kt + 2 units: pair s,
        // then pair ppb - 1 - s): pair P of problem b holds tri_kt - 2P units.
        const int64_t ppb = tri_kt / 2;
        const int64_t bb = r / ppb, P = r - bb * ppb;
        const int64_t U = ppb * tri_kt - ppb * (ppb - 1);
        const int64_t s = 2 * P <= ppb - 1 ? P : ppb - 1 - P;
        const int64_t start = bb * U + s * (tri_kt + 2) + (s == P ? 0 : tri_kt - 2 * s);
        return (start + tri_kt - 2 * P - 1) / unit_len - start / unit_len + 1;
    }
    return ((r + 1) * key_tiles - 1) / unit_len - r * key_tiles / unit_len + 1;
}

__global__ void finalize_slots_kernel(const float* __restrict__ part, int64_t Mpad, int64_t M,
                                      int C, int rows_per_unit, int64_t key_tiles,
                                      int64_t unit_len, int64_t batch, int fixed_slots,
                                      int64_t tri_kt, float* __restrict__ out) {
    pdl_trigger();
    pdl_wait();
    // out: batch x M x C; partial rows are batch-stacked with Mpad rows per
    // problem and batch Mpad rows per slot.
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= batch * M * C) return;
    const int64_t bm = div_nonneg(idx, C);
    const int c = static_cast<int>(idx - bm * C);
    const int64_t b = M <= 0x7fffffff ? div_nonneg(bm, static_cast<int>(M)) : bm / M;
    const int64_t m = (bm - b * M) + b * Mpad;
    const int64_t nslots =
        contributor_slots(m / rows_per_unit, fixed_slots, key_tiles, unit_len, tri_kt);
    float acc = 0.f;
    for (int64_t sl = 0; sl < nslots; ++sl) acc += part[(sl * batch * Mpad + m) * C + c];
    out[idx] = acc;
}

// Vectorised variant of operand_kernel for D >= 1: G lanes share a row, each
// converting up to kOperandVecs vectors of 8 coordinates; the squared norm is
// reduced over the G lanes and the group's first lane writes the columns past
// D (norm terms or zeros).  Same outputs as operand_kernel.
constexpr int kOperandVecThreads = 256;

template <typename T> __device__ __forceinline__ T bits_to(unsigned short b);
template <> __device__ __forceinline__ __half bits_to<__half>(unsigned short b) {
    return __ushort_as_half(b);
}
template <> __device__ __forceinline__ __nv_bfloat16 bits_to<__nv_bfloat16>(unsigned short b) {
    return __ushort_as_bfloat16(b);
}
template <typename T> __device__ __forceinline__ unsigned short to_bits(T h);
template <> __device__ __forceinline__ unsigned short to_bits<__half>(__half h) {
    return __half_as_ushort(h);
}
template <> __device__ __forceinline__ unsigned short to_bits<__nv_bfloat16>(__nv_bfloat16 h) {
    return __bfloat16_as_ushort(h);
}

// Packed 16-bit pair arithmetic of the operand conversion.  x - mu of two
// 16-bit inputs and a mean on the input grid (see rounded_mean), rounded
// once to the input format (the MMA operand type), and the pair as floats.
template <typename T> struct Pair;
template <> struct Pair<__half> {
    using P = __half2;
    static __device__ __forceinline__ P sub(P a, P b) { return __hsub2(a, b); }
    static __device__ __forceinline__ float2 to_f2(P a) { return __half22float2(a); }
    static __device__ __forceinline__ P from_f2(float lo, float hi) { return __floats2half2_rn(lo, hi); }
};
template <> struct Pair<__nv_bfloat16> {
    using P = __nv_bfloat162;
    static __device__ __forceinline__ P sub(P a, P b) { return __hsub2(a, b); }
    static __device__ __forceinline__ float2 to_f2(P a) { return __bfloat1622float2(a); }
    static __device__ __forceinline__ P from_f2(float lo, float hi) { return __floats2bfloat162_rn(lo, hi); }
};

// One output row of the operand layouts, converted by the G lanes of a
// row group: lane vi holds the row's 16-byte input vectors vi, vi + G, ...
// (in[e] = vector vi + G e, 8 coordinates each, for vi + G e < D / 8; up to
// kOperandVecs of them) and smean the problem's mean as packed pairs of the
// input format in shared memory (exact: the mean lies on the input grid).
// out_q / out_k: the row in either layout (either may be null; AUG only).
// Every lane of the warp must call this together (the squared norm is
// reduced with shuffles over the G lanes); rows outside the output (in_pad
// false) write nothing.  Returns the norm term written for the row (plain
// layout: -(c/2)||x^||^2, or pad_value) in every lane.
constexpr int kOperandVecs = 8;

template <typename T, bool AUG, int G, bool RAGGED>
__device__ __forceinline__ float operand_row(const uint4 (&in)[kOperandVecs],
                                             const uint4* __restrict__ smean, int vi,
                                             bool in_pad, bool valid, int D, int Dp, int nt,
                                             float F, float half_c, float pad_value,
                                             T* __restrict__ out_q, T* __restrict__ out_k,
                                             float cf, const __half* vw) {
    using PT = Pair<T>;
    const int V = RAGGED ? (D + 7) / 8 : D / 8;   // (coordinates past D are 0 - 0)
    const bool fold = AUG && cf > 0.f;
    float acc = 0.f, accu = 0.f;
    // RAGGED: the squares are added in operand_kernel's order (coordinates of
    // one residue mod 32 in sequence, then a tree over the residues), so that
    // rows of any width keep their norms bit for bit: ps[8 j + e] is residue
    // 8 (vi + G j) + e mod 32 of this lane.
    constexpr int R8 = RAGGED ? 4 / G : 1;            // residue groups of 8 per lane
    float ps[8 * R8], pu[8 * R8];
    if (RAGGED) {
#pragma unroll
        for (int i = 0; i < 8 * R8; ++i) ps[i] = pu[i] = 0.f;
    }
    if (in_pad) {
        uint64_t acc2 = 0ull, accu2 = 0ull;
#pragma unroll
        for (int e = 0; e < kOperandVecs; ++e) {
            const int v = vi + G * e;
            if (v >= V) break;
            uint4 u = make_uint4(0u, 0u, 0u, 0u), us = u;
            if (valid) {
                const uint4 m2 = smean[v];
                const typename PT::P* x2 = reinterpret_cast<const typename PT::P*>(&in[e]);
                const typename PT::P* mm = reinterpret_cast<const typename PT::P*>(&m2);
                typename PT::P h[4], hs[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    h[k] = PT::sub(x2[k], mm[k]);
                    const float2 f = PT::to_f2(h[k]);
                    const uint64_t f2 = f32x2_pack(f.x, f.y);
                    const int i = RAGGED ? 8 * (e % R8) + 2 * k : 0;
                    if (RAGGED) {
                        ps[i] = fmaf(f.x, f.x, ps[i]);
                        ps[i + 1] = fmaf(f.y, f.y, ps[i + 1]);
                    } else {
                        acc2 = f32x2_fma(f2, f2, acc2);
                    }
                    if (fold) {
                        // Folded scale: the query row holds rn(c x^).
                        hs[k] = PT::from_f2(cf * f.x, cf * f.y);
                        const float2 g = PT::to_f2(hs[k]);
                        const uint64_t g2 = f32x2_pack(g.x, g.y);
                        if (RAGGED) {
                            pu[i] = fmaf(g.x, g.x, pu[i]);
                            pu[i + 1] = fmaf(g.y, g.y, pu[i + 1]);
                        } else {
                            accu2 = f32x2_fma(g2, g2, accu2);
                        }
                    }
                }
                u = *reinterpret_cast<const uint4*>(h);
                us = fold ? *reinterpret_cast<const uint4*>(hs) : u;
            }
            if (out_q) *reinterpret_cast<uint4*>(out_q + 8 * v) = fold ? us : u;
            if (out_k) *reinterpret_cast<uint4*>(out_k + 8 * v) = u;
        }
        if (!RAGGED) {
            float lo, hi;
            f32x2_unpack(acc2, lo, hi);
            acc = lo + hi;
            f32x2_unpack(accu2, lo, hi);
            accu = lo + hi;
        }
    }
    if (RAGGED) {
        // The tree over residues: 16 apart, then 8, 4, 2, 1.  G = 1: all in this
        // lane; G = 2: 16 apart in this lane (j, j + 1), 8 apart in the other;
        // G = 4: 16 and 8 apart in other lanes.
        auto tree = [&](float (&p)[8 * R8]) {
            float t[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (G == 1) {
                    t[i] = (p[i] + p[(16 + i) % (8 * R8)]) + (p[(8 + i) % (8 * R8)] + p[(24 + i) % (8 * R8)]);
                } else if (G == 2) {
                    t[i] = p[i] + p[(8 + i) % (8 * R8)];
                    t[i] += __shfl_xor_sync(0xffffffffu, t[i], 1);
                } else {
                    t[i] = p[i] + __shfl_xor_sync(0xffffffffu, p[i], 2);
                    t[i] += __shfl_xor_sync(0xffffffffu, t[i], 1);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) t[i] += t[i + 4];
            t[0] += t[2];
            t[1] += t[3];
            return t[0] + t[1];
        };
        acc = tree(ps);
        if (fold) accu = tree(pu);
    } else {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
            acc += __shfl_xor_sync(0xffffffffu, acc, o, G);
            if (fold) accu += __shfl_xor_sync(0xffffffffu, accu, o, G);
        }
    }
    const float nrm = valid ? -half_c * acc : pad_value;
    if (RAGGED) __syncwarp();   // the last vector's lane has written columns past D
    if (!in_pad || vi != 0) return nrm;
    if (!AUG) {
        for (int c = 8 * V; c < Dp; c += 8)
            *reinterpret_cast<uint4*>(out_q + c) = make_uint4(0u, 0u, 0u, 0u);
        return nrm;
    }
    // Norm terms: a (or b) = -||x^||^2 / 2 = F t_0 + t_1 + ... (rounded
    // remainders, nt <= 3 of them), partners F, 1, 1 on the other side.
    // Built in registers: element e of the query tail is the partner
    // (F, 1, 1) for e < nt and t_(e - nt) for nt <= e < 2 nt; the key tail
    // the other way round; zeros after that.
    unsigned short t0 = 0, t1 = 0, t2 = 0, k0 = 0, k1 = 0, k2 = 0;
    auto split = [&](float r, unsigned short& z0, unsigned short& z1, unsigned short& z2) {
        const T a0 = from_f<T>(r * (1.f / F));   // F is a power of two: exact
        r -= F * to_f(a0);
        const T a1 = from_f<T>(r);
        r -= to_f(a1);
        const T a2 = from_f<T>(r);
        z0 = to_bits(a0);
        z1 = to_bits(a1);
        z2 = nt > 2 ? to_bits(a2) : 0;
    };
    if (valid) {
        if (fold) {
            // Folded: a = -||u||^2 / (2c) from the rounded scaled row, and
            // b = -c ||k^||^2 / 2 + log2(|v| 2^-16) (see log_weight).
            split(-0.5f * accu / cf, t0, t1, t2);
            // (Explicitly one rounding for RAGGED rows, as in operand_kernel, and
            // two for the others: a last bit of b moves signed sums of 65536
            // keys by 2e-5 of their norm, so the choice is not the compiler's.)
            const float lw = log_weight(vw);
            split(RAGGED ? fmaf(-0.5f * cf, acc, lw) : __fadd_rn(__fmul_rn(-0.5f * cf, acc), lw), k0, k1, k2);
        } else {
            split(-0.5f * acc, t0, t1, t2);
            k0 = t0; k1 = t1; k2 = t2;
        }
    }
    const unsigned short oneF = valid ? to_bits(from_f<T>(F)) : 0;
    const unsigned short one1 = valid ? to_bits(from_f<T>(1.f)) : 0;
    const unsigned short pad_b = valid ? k0 : to_bits(from_f<T>(-30000.f / F));
    auto term = [&](int i) { return i == 0 ? pad_b : i == 1 ? k1 : k2; };
    auto qterm = [&](int i) { return i == 0 ? t0 : i == 1 ? t1 : t2; };
    auto partner = [&](int i) { return i == 0 ? oneF : one1; };
    auto tail_q = [&](int e) -> unsigned {
        return e < nt ? partner(e) : e < 2 * nt ? qterm(e - nt) : 0u;
    };
    auto tail_k = [&](int e) -> unsigned {
        return e < nt ? term(e) : e < 2 * nt ? partner(e - nt) : 0u;
    };
    if constexpr (RAGGED) {
        // The columns past D start anywhere: zeros to the end of the row, then
        // the norm terms and their partners one by one.
        for (int c = 8 * V; c < Dp; c += 8) {
            if (out_q) *reinterpret_cast<uint4*>(out_q + c) = make_uint4(0u, 0u, 0u, 0u);
            if (out_k) *reinterpret_cast<uint4*>(out_k + c) = make_uint4(0u, 0u, 0u, 0u);
        }
        for (int e = 0; e < 2 * nt; ++e) {
            if (out_q) out_q[D + e] = bits_to<T>(static_cast<unsigned short>(tail_q(e)));
            if (out_k) out_k[D + e] = bits_to<T>(static_cast<unsigned short>(tail_k(e)));
        }
    } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = D + 8 * h;
            if (c >= Dp) break;
            uint32_t wq[4], wk[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                wq[e] = tail_q(8 * h + 2 * e) | (tail_q(8 * h + 2 * e + 1) << 16);
                wk[e] = tail_k(8 * h + 2 * e) | (tail_k(8 * h + 2 * e + 1) << 16);
            }
            if (out_q) *reinterpret_cast<uint4*>(out_q + c) = make_uint4(wq[0], wq[1], wq[2], wq[3]);
            if (out_k) *reinterpret_cast<uint4*>(out_k + c) = make_uint4(wk[0], wk[1], wk[2], wk[3]);
        }
        for (int c = D + 16; c < Dp; c += 8) {
            if (out_q) *reinterpret_cast<uint4*>(out_q + c) = make_uint4(0u, 0u, 0u, 0u);
            if (out_k) *reinterpret_cast<uint4*>(out_k + c) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    return nrm;
}

// One array's operand rows: x (batch x rows x D) into out_q / out_k
// (batch x rows_pad x Dp; either may be null, AUG only) and, for the plain
// layout, the norm terms nrm (batch x rows_pad).
struct OperandJob {
    const void* x;
    int64_t rows, rows_pad;
    void* out_q;
    void* out_k;
    float* nrm;
    const void* vw;      // fp16 values of the rows written to out_k (folded magnitudes), or null
};

// Vector path of the operand preparation: G lanes per
// row (G = 1 up to D = 64, 2 up to 128, 4 up to 256), each lane converting
// up to eight 16-byte vectors of its row, all loaded before any is
// converted; so every lane of a warp does its own row's work (no lanes idle
// during the norm split) and has up to 128 bytes of loads in flight.  The
// block's output rows are staged in shared memory (a row stride of an odd
// number of 16-byte vectors, so that the lanes' row stores do not share
// banks) and then written as one contiguous run of 16-byte vectors, one per
// thread and step, instead of one row per lane.
// Blocks [0, blocks0) of grid row b convert rows of job j0 of problem b,
// the rest those of j1 (the keys, when they are not the queries), so that
// both arrays of every problem take one launch; a block never straddles
// two problems.  The problem's mean is staged once per block in shared
// memory as packed pairs of the input format.
// RAGGED (D not a multiple of 8, rows that start anywhere): the block's
// input rows, one contiguous run, are copied to shared memory in 16-byte
// vectors first and each lane gathers its row's vectors there.  (One warp per
// row in operand_kernel before: 50021 points, D = 50, both layouts: 26.7 ->
// 10.1 us, 19 MB moved.)
// Rows [blk SLOTS, (blk + 1) SLOTS) of job j, problem b, by the whole block:
// stage_mean() stages the problem's mean in smean (it runs between the row
// loads and their use), staged holds the output rows (and, RAGGED, behind
// them the input rows).
template <typename T, bool AUG, int G, bool RAGGED, typename StageMean>
__device__ __forceinline__ void operand_block(const OperandJob& j, int b, int blk, int D, int Dp, int nt,
                                              float F, float half_c, float pad_value, float cf,
                                              const uint4* smean, uint4* staged, StageMean stage_mean) {
    constexpr int SLOTS = kOperandVecThreads / G;    // rows of a block
    const int vi = threadIdx.x % G;                  // first vector of this lane
    const int slot = threadIdx.x / G;
    const int V = RAGGED ? (D + 7) / 8 : D / 8;
    const int rows_pad = static_cast<int>(j.rows_pad);
    const int rows = static_cast<int>(j.rows);
    const int i = blk * SLOTS + slot;                // row of problem b
    const bool wq = AUG ? j.out_q != nullptr : true;
    const bool wk = AUG && j.out_k != nullptr;
    const int sv = (Dp / 8) | 1;                     // staged row stride (odd) in 16-byte vectors
    uint4 in[kOperandVecs];
    if (RAGGED) {
        // Behind the staged output rows (see operand_typed).
        T* raw = reinterpret_cast<T*>(staged + ((wq ? 1 : 0) + (wk ? 1 : 0)) * SLOTS * sv);
        const int i0 = blk * SLOTS;
        const int n_el = max(0, min(SLOTS, rows - i0)) * D;
        const T* src = static_cast<const T*>(j.x) + (static_cast<int64_t>(b) * rows + i0) * D;
        // (A later problem of a batch may start anywhere.)
        const int nvec = (reinterpret_cast<uintptr_t>(src) & 15u) == 0 ? n_el / 8 : 0;
        for (int u = threadIdx.x; u < nvec; u += kOperandVecThreads)
            reinterpret_cast<uint4*>(raw)[u] = reinterpret_cast<const uint4*>(src)[u];
        for (int u = nvec * 8 + threadIdx.x; u < n_el; u += kOperandVecThreads) raw[u] = src[u];
        __syncthreads();
        const T* row = raw + slot * D;
#pragma unroll
        for (int e = 0; e < kOperandVecs; ++e) {
            const int c = 8 * (vi + G * e);
            uint32_t w[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int c2 = c + 2 * h;
                unsigned lo = 0u, hi = 0u;
                if (i < rows && c2 < D) {
                    if (D & 1) {
                        lo = to_bits(row[c2]);
                        hi = c2 + 1 < D ? to_bits(row[c2 + 1]) : 0u;
                        lo |= hi << 16;
                    } else {
                        lo = *reinterpret_cast<const uint32_t*>(row + c2);   // even row starts
                    }
                }
                w[h] = lo;
            }
            in[e] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    } else {
        const T* xr = static_cast<const T*>(j.x) + (static_cast<int64_t>(b) * rows + i) * D;
#pragma unroll
        for (int e = 0; e < kOperandVecs; ++e) {
            const int v = vi + G * e;
            in[e] = (i < rows && v < V) ? *reinterpret_cast<const uint4*>(xr + 8 * v)
                                        : make_uint4(0u, 0u, 0u, 0u);
        }
    }
    stage_mean();
    __syncthreads();
    const bool in_pad = i < rows_pad;
    const int64_t row = static_cast<int64_t>(b) * rows_pad + i;   // batch-stacked output row
    const __half* vw = (wk && j.vw && i < rows)
                           ? static_cast<const __half*>(j.vw) + static_cast<int64_t>(b) * rows + i
                           : nullptr;
    const int nv = Dp / 8;                           // 16-byte vectors per output row
    uint4* stage_q = staged;
    uint4* stage_k = staged + (wq ? SLOTS * sv : 0);
    const float n = operand_row<T, AUG, G, RAGGED>(
        in, smean, vi, in_pad, i < rows, D, Dp, nt, F, half_c, pad_value,
        wq ? reinterpret_cast<T*>(stage_q + slot * sv) : nullptr,
        wk ? reinterpret_cast<T*>(stage_k + slot * sv) : nullptr, cf, vw);
    if (!AUG && in_pad && vi == 0) j.nrm[row] = n;
    __syncthreads();
    // The block's rows [i0, i0 + nrows) are consecutive output rows.
    const int i0 = blk * SLOTS;
    const int nrows = min(SLOTS, rows_pad - i0);
    const int total = nrows * nv;
    const int64_t base = (static_cast<int64_t>(b) * rows_pad + i0) * Dp;
    uint4* gq = wq ? reinterpret_cast<uint4*>(static_cast<T*>(j.out_q) + base) : nullptr;
    uint4* gk = wk ? reinterpret_cast<uint4*>(static_cast<T*>(j.out_k) + base) : nullptr;
    for (int u = threadIdx.x; u < total; u += kOperandVecThreads) {
        const int r = u / nv;
        const int s = r * sv + (u - r * nv);
        if (wq) gq[u] = stage_q[s];
        if (wk) gk[u] = stage_k[s];
    }
}

template <typename T, bool AUG, int G, bool RAGGED>
__global__ void __launch_bounds__(kOperandVecThreads)
operand_vec_kernel(const OperandJob j0, const OperandJob j1, unsigned blocks0, int D, int Dp,
                   int nt, float F, const float* __restrict__ mu, float half_c, float pad_value,
                   float cf, unsigned op_blocks, float* __restrict__ vf_rec, int64_t vf_tiles) {
    using PT = Pair<T>;
    pdl_trigger();
    pdl_wait();
    if (blockIdx.x >= op_blocks) {
        // Folded values: the per-problem flag of the sign records (written
        // by an earlier launch of the call), one extra block per problem.
        write_vf_flag(vf_rec, vf_tiles, static_cast<int>(gridDim.y), blockIdx.y);
        return;
    }
    __shared__ uint4 smean[kOperandMaxCols / 8];
    extern __shared__ uint4 staged[];                // the block's rows of each output
    const int b = blockIdx.y;                        // problem of the batch
    const bool second = blockIdx.x >= blocks0;
    const OperandJob j = second ? j1 : j0;
    const int blk = static_cast<int>(second ? blockIdx.x - blocks0 : blockIdx.x);
    const int V = RAGGED ? (D + 7) / 8 : D / 8;
    operand_block<T, AUG, G, RAGGED>(j, b, blk, D, Dp, nt, F, half_c, pad_value, cf, smean, staged, [&] {
        const float* mb = mu ? mu + static_cast<int64_t>(b) * D : nullptr;
        typename PT::P* sm = reinterpret_cast<typename PT::P*>(smean);
        for (int c = threadIdx.x; c < 4 * V; c += kOperandVecThreads) {
            const float m0 = mb && 2 * c < D ? mb[2 * c] : 0.f;
            const float m1 = mb && 2 * c + 1 < D ? mb[2 * c + 1] : 0.f;
            sm[c] = PT::from_f2(m0, m1);
        }
    });
}

template <typename T, bool AUG>
cudaError_t operand_typed(const OperandJob& j0, const OperandJob* j1, int D, int Dp, int nt,
                          float F, const float* mu, float half_c, float pad_value, cudaStream_t s,
                          int batch, float cf, float* vf_rec, int64_t vf_tiles, bool* flags_done) {
    const OperandJob none = {nullptr, 0, 0, nullptr, nullptr, nullptr, nullptr};
    for (const OperandJob* j : {&j0, j1}) {
        if (j && (j->rows_pad % kRowsPerBlock != 0)) return cudaErrorInvalidValue;
    }
    if (Dp % 16 != 0 || Dp > kOperandMaxCols || (AUG && 2 * Dp > kOperandMaxCols))
        return cudaErrorInvalidValue;
    // The vector path indexes rows with 32-bit integers.
    const int64_t most_rows = std::max(j0.rows_pad, j1 ? j1->rows_pad : int64_t(0)) * batch;
    if (D >= 1 && (!AUG || Dp - D >= 2 * nt) && most_rows < (int64_t(1) << 30)) {
        // Vector path: G lanes per row (up to kOperandVecs vectors each),
        // both arrays in one launch.
        const bool ragged = D % 8 != 0;
        const int V = (D + 7) / 8;
        const int G = V <= kOperandVecs ? 1 : V <= 2 * kOperandVecs ? 2 : 4;
        const int64_t per_block = kOperandVecThreads / G;
        const int64_t b0 = (j0.rows_pad + per_block - 1) / per_block;
        const int64_t b1 = j1 ? (j1->rows_pad + per_block - 1) / per_block : 0;
        if (b0 + b1 == 0 || batch == 0) return cudaSuccess;
        const unsigned op_blocks = static_cast<unsigned>(b0 + b1);
        // Staged output rows: one or two outputs per job (AUG with q = k
        // writes both layouts of the same rows).
        auto nout = [](const OperandJob* j) {
            return j ? (AUG ? (j->out_q ? 1 : 0) + (j->out_k ? 1 : 0) : 1) : 0;
        };
        const size_t smem = static_cast<size_t>(std::max(nout(&j0), nout(j1))) * per_block *
                                ((Dp / 8) | 1) * 16 +
                            (ragged ? (static_cast<size_t>(per_block) * D * sizeof(T) + 15) / 16 * 16 : 0);
        auto go = [&](auto kern) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 static_cast<int>(smem));
            if (e != cudaSuccess) return e;
            launch_kernel(kern, dim3(op_blocks + (vf_rec ? 1u : 0u), static_cast<unsigned>(batch)),
                          kOperandVecThreads, smem, s, j0, j1 ? *j1 : none, static_cast<unsigned>(b0),
                          D, Dp, nt, F, mu, half_c, pad_value, cf, op_blocks, vf_rec, vf_tiles);
            return cudaSuccess;
        };
        if (flags_done) *flags_done = vf_rec != nullptr;
        cudaError_t e;
        switch (G) {
            case 1: e = ragged ? go(operand_vec_kernel<T, AUG, 1, true>) : go(operand_vec_kernel<T, AUG, 1, false>); break;
            case 2: e = ragged ? go(operand_vec_kernel<T, AUG, 2, true>) : go(operand_vec_kernel<T, AUG, 2, false>); break;
            default: e = ragged ? go(operand_vec_kernel<T, AUG, 4, true>) : go(operand_vec_kernel<T, AUG, 4, false>); break;
        }
        if (e != cudaSuccess) return e;
        note_launches(1);
        return cudaGetLastError();
    }
    for (const OperandJob* j : {&j0, j1}) {
        if (!j) continue;
        const int64_t blocks = j->rows_pad / kRowsPerBlock;
        if (blocks == 0) continue;
        const int nout = AUG ? (j->out_q ? 1 : 0) + (j->out_k ? 1 : 0) : 1;
        const size_t smem = static_cast<size_t>(nout) * kRowsPerBlock * Dp * sizeof(T) +
                            ((static_cast<size_t>(kRowsPerBlock) * D * sizeof(T) + 15) & ~size_t(15)) +
                            static_cast<size_t>(D) * sizeof(float);
        launch_kernel(operand_kernel<T, AUG>, dim3(static_cast<unsigned>(blocks), batch),
                      kOperandThreads, smem, s, static_cast<const T*>(j->x), j->rows, j->rows_pad,
                      D, Dp, nt, F, mu, half_c, pad_value, static_cast<T*>(j->out_q),
                      static_cast<T*>(j->out_k), j->nrm, static_cast<const __half*>(j->vw), cf);
        note_launches(1);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// ---------------------------------------------------------------- values
// Value of channel ch of key n.  Forward (Eq. 1): w[n, ch] (Cw = channels).
// Gradients (Sec. 3, and the vector-Jacobian product of Eq. 1): channel
// ch = c (D + 1) + d holds w[n, c] (x[n, d] - mu_d) for d < D and w[n, c]
// for d = D, one group of D + 1 channels per weight channel c < Cw; a null
// w means unit weights (the weighted vector-Jacobian pass, whose weights
// enter through the kernel values instead).
template <typename T, typename W, bool GRAD>
__device__ __forceinline__ float value_at(const W* __restrict__ w, const T* __restrict__ x,
                                          const float* __restrict__ mu, int64_t n, int ch, int D,
                                          int Cw) {
    if (GRAD) {
        const int c = ch / (D + 1);
        const int d = ch - c * (D + 1);
        const float wn = w ? to_f(w[n * Cw + c]) : 1.f;
        if (d < D) return wn * (to_f(x[n * D + d]) - (mu ? mu[d] : 0.f));
        return wn;
    }
    return to_f(w[n * Cw + ch]);
}

// Per-channel max |value| over the keys for channels ch0 .. ch0 + Cc - 1;
// block (32, 8) as in the mean.
template <typename T, typename W, bool GRAD>
__global__ void value_max_kernel(const W* __restrict__ w, const T* __restrict__ x,
                                 const float* __restrict__ mu, int64_t N, int D, int Cw, int ch0,
                                 int Cc, int64_t rows_per_block, unsigned* __restrict__ vmax_bits) {
    pdl_trigger();
    pdl_wait();
    __shared__ float red[8][33];
    const int64_t r0 = static_cast<int64_t>(blockIdx.x) * rows_per_block;
    const int64_t r1 = min(r0 + rows_per_block, N);
    for (int c0 = 0; c0 < Cc; c0 += 32) {
        const int c = c0 + threadIdx.x;
        float mx = 0.f;
        if (c < Cc)
            for (int64_t n = r0 + threadIdx.y; n < r1; n += 8)
                mx = fmaxf(mx, fabsf(value_at<T, W, GRAD>(w, x, mu, n, ch0 + c, D, Cw)));
        red[threadIdx.y][threadIdx.x] = mx;
        __syncthreads();
        if (threadIdx.y == 0 && c < Cc) {
            float m = 0.f;
#pragma unroll
            for (int y = 0; y < 8; ++y) m = fmaxf(m, red[y][threadIdx.x]);
            // Non-negative floats order like their bit patterns.
            atomicMax(&vmax_bits[c], __float_as_uint(m));
        }
        __syncthreads();
    }
}

// Power-of-two channel scale 2^e with e = -floor(log2 max|value|), so that
// the scaled channel's largest magnitude lies in [1, 2); e is clamped to
// [-126, 126] and is 0 for an all-zero channel.  Exact bit construction.
__device__ __forceinline__ int channel_exponent(unsigned max_bits) {
    if (max_bits == 0u) return 0;
    int E = static_cast<int>((max_bits >> 23) & 0xffu);
    if (E == 0) E = 1;             // subnormal maximum: clamp
    if (E == 0xff) return 0;       // inf / nan: leave unscaled
    int e = 127 - E;               // -floor(log2 max)
    return max(-126, min(126, e));
}

__device__ __forceinline__ float pow2f(int e) { return __uint_as_float(static_cast<unsigned>(e + 127) << 23); }

// Transposed, scaled fp16 value operand vt[j][n] = value of channel ch0 + j
// (Cp x Npad, zero padded), through a 32 x 32 shared-memory tile; block
// (32, 8).
template <typename T, typename W, bool GRAD>
__global__ void value_prep_kernel(const W* __restrict__ w, const T* __restrict__ x,
                                  const float* __restrict__ mu, int64_t N, int64_t Npad, int D,
                                  int Cw, int ch0, int Cc, int Cp,
                                  const unsigned* __restrict__ vmax_bits, __half* __restrict__ vt,
                                  float* __restrict__ inv_scale) {
    pdl_trigger();
    pdl_wait();
    // A block transposes 64 keys x 32 channels; each thread stores two
    // adjacent keys of one channel as a half2 (Npad is a multiple of 128).
    __shared__ float tile[64][33];
    const int64_t n0 = static_cast<int64_t>(blockIdx.x) * 64;
    const int c0 = blockIdx.y * 32;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int64_t n = n0 + threadIdx.y + 8 * i;
        const int c = c0 + threadIdx.x;
        float val = 0.f;
        if (n < N && c < Cc) val = value_at<T, W, GRAD>(w, x, mu, n, ch0 + c, D, Cw);
        tile[threadIdx.y + 8 * i][threadIdx.x] = val;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c = c0 + threadIdx.y + 8 * i;
        const int64_t n = n0 + 2 * threadIdx.x;
        if (c < Cp && n < Npad) {
            const float sc = c < Cc ? pow2f(channel_exponent(vmax_bits[c])) : 0.f;
            const int cl = threadIdx.y + 8 * i;
            *reinterpret_cast<__half2*>(vt + static_cast<int64_t>(c) * Npad + n) =
                __floats2half2_rn(tile[2 * threadIdx.x][cl] * sc, tile[2 * threadIdx.x + 1][cl] * sc);
        }
    }
    if (blockIdx.x == 0 && threadIdx.y == 0) {
        const int c = c0 + threadIdx.x;
        if (c < Cp) inv_scale[c] = c < Cc ? pow2f(-channel_exponent(vmax_bits[c])) : 0.f;
    }
}

// ---------------------------------------------------------------- key records
// One thread per key pair t, values in fp32, zero for padded keys.  Without B
// (augmented operands) the pair's values channel by channel; with B per four
// keys their B and then, channel by channel, their values (see
// tc_gauss_fma.cu).
template <typename T>
__global__ void key_record_kernel(const T* __restrict__ v, const float* __restrict__ B, int64_t N,
                                  int64_t pairs, int C, float* __restrict__ rec) {
    pdl_trigger();
    pdl_wait();
    const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t >= pairs) return;
    const int64_t n0 = 2 * t, n1 = 2 * t + 1;
    // Problem blockIdx.y of a batch (2 pairs keys per problem).
    v += static_cast<int64_t>(blockIdx.y) * N * C;
    if (B) B += static_cast<int64_t>(blockIdx.y) * 2 * pairs;
    rec += static_cast<int64_t>(blockIdx.y) * pairs * ((B ? 2 : 0) + 2 * C);
    // The pair's first float, and the distance between its channels.
    float* out = rec + (B ? (t >> 1) * (4 + 4 * C) + (t & 1) * 2 : t * (2 * C));
    const int step = B ? 4 : 2;
    if (B) {
        out[0] = B[n0];
        out[1] = B[n1];
        out += step;
    }
    for (int c = 0; c < C; ++c, out += step) {
        out[0] = n0 < N ? to_f(v[n0 * C + c]) : 0.f;
        out[1] = n1 < N ? to_f(v[n1 * C + c]) : 0.f;
    }
}

// ---------------------------------------------------------------- pair weights
// Factors of the pair weights w_mn = sum_c r[m, c] k[n, c] of the weighted
// vector-Jacobian pass (row factors r: the rows of the Gauss sum, column
// factors k: its keys; C <= WT channels, zero padded to WT).  Blocks
// [0, rblocks) write the row factors row-major in float32,
// rowf[m WT + c] (Rpad rows, zero past R); the other blocks write the
// column factors per key tile of BN keys, channel-major inside the tile,
// colT[(n / BN) WT BN + c BN + n % BN] (Npad keys, zero past Ncol), so that
// one bulk copy brings a key tile's factors into shared memory.  wmax[c]
// and wmax[WT + c] receive the largest |r[., c]| and |k[., c]| (float bits,
// atomicMax over blocks; the caller zeroes them).  One thread per (row or
// key, channel), 256 threads per block.
constexpr int kWeightThreads = 256;

template <typename TR, typename TC>
__global__ void __launch_bounds__(kWeightThreads)
weight_prep_kernel(const TR* __restrict__ rsrc, int64_t R, int64_t Rpad,
                   const TC* __restrict__ csrc, int64_t Ncol, int64_t Npad, int C, int WT, int BN,
                   unsigned rblocks, float* __restrict__ rowf, float* __restrict__ colT,
                   unsigned* __restrict__ wmax) {
    pdl_trigger();
    pdl_wait();
    __shared__ float red[kWeightThreads];
    const bool on_rows = blockIdx.x < rblocks;
    const int64_t blk = on_rows ? blockIdx.x : blockIdx.x - rblocks;
    const int64_t idx = blk * kWeightThreads + threadIdx.x;
    const int64_t i = idx / WT;                 // row or key
    const int c = static_cast<int>(idx - i * WT);
    float val = 0.f;
    if (on_rows) {
        if (i < Rpad) {
            if (i < R && c < C) val = to_f(rsrc[i * C + c]);
            rowf[idx] = val;
        }
    } else if (i < Npad) {
        if (i < Ncol && c < C) val = to_f(csrc[i * C + c]);
        colT[(i / BN) * WT * BN + static_cast<int64_t>(c) * BN + i % BN] = val;
    }
    // Channel c of this block: threads t with t % WT == c (WT divides 256).
    red[threadIdx.x] = fabsf(val);
    __syncthreads();
    if (threadIdx.x < WT) {
        float m = 0.f;
        for (int t = threadIdx.x; t < kWeightThreads; t += WT) m = fmaxf(m, red[t]);
        // Non-negative floats order like their bit patterns.
        atomicMax(&wmax[(on_rows ? 0 : WT) + threadIdx.x], __float_as_uint(m));
    }
}

// ---------------------------------------------------------------- finalise
// Forward: out[m, c] = inv_scale[c] sum_s part[s][m][c] (splits added in
// order).  part: splits blocks of split_stride_rows rows x part_ld floats.
__global__ void finalize_kernel(const float* __restrict__ part, int splits,
                                int64_t split_stride_rows, int64_t M, int Cv, int part_ld,
                                const float* __restrict__ inv_scale, float* __restrict__ out,
                                int64_t main_rows) {
    pdl_trigger();
    pdl_wait();
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= M * Cv) return;
    const int64_t m = div_nonneg(idx, Cv);
    const int c = static_cast<int>(idx - m * Cv);
    float acc = 0.f;
    const int ns = m < main_rows ? 1 : splits;
    const float* p = part + m * part_ld + c;
    const int64_t step = split_stride_rows * part_ld;
    int s = 0;
    // Eight splits' loads in flight together where there are that many (the
    // sum keeps the split order).
    for (; s + 8 <= ns; s += 8, p += 8 * step) {
        float x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = p[i * step];
#pragma unroll
        for (int i = 0; i < 8; ++i) acc += x[i];
    }
    for (; s < ns; ++s, p += step) acc += *p;
    out[idx] = acc * (inv_scale ? inv_scale[c] : 1.f);
}

// The same for many splits of few rows (the fp32 SIMT path: inv_scale null, one
// contiguous M x Cv block of partials per split): one thread per output walked
// up to 256 splits with most of the chip idle (513 x 8192, D = 16, C = 4: 17 us
// of a 43 us call).  Here kFinalizeLanes threads share an output: thread y adds
// splits y, y + kFinalizeLanes, ... in order, and thread 0 the sums in order.
constexpr int kFinalizeLanes = 8;

// Whether an output's n partial sums are shared by several threads: 16 or more,
// or four or more where one thread per output leaves SMs idle.
__host__ __device__ inline bool many_partials(int n, int64_t outputs) {
    return n >= 16 || (n >= 4 && outputs < 152 * 256);
}

// p[0], p[stride], .. (n of them) added up by the block's column of threads
// threadIdx.x, into the return value of thread y = 0; a few (see many_partials)
// in order by that thread, as finalize_kernel adds them.  Every thread of the
// block calls this (n <= 0: none).
__device__ __forceinline__ float sum_lanes(const float* __restrict__ p, int64_t stride, int n, int64_t outputs) {
    __shared__ float sums[kFinalizeLanes][32];
    const int lanes = many_partials(n, outputs) ? kFinalizeLanes : 1;
    float acc = 0.f;
    int s = static_cast<int>(threadIdx.y);
    if (s < lanes) {
        p += s * stride;
        const int64_t step = lanes * stride;
        for (; s + 7 * lanes < n; s += 8 * lanes, p += 8 * step) {
            float x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = p[i * step];
#pragma unroll
            for (int i = 0; i < 8; ++i) acc += x[i];
        }
        for (; s < n; s += lanes, p += step) acc += *p;
    }
    sums[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.y == 0 && lanes > 1) {
#pragma unroll
        for (int y = 1; y < kFinalizeLanes; ++y) acc += sums[y][threadIdx.x];
    }
    return acc;
}

__global__ void __launch_bounds__(32 * kFinalizeLanes)
finalize_many_kernel(const float* __restrict__ part, int splits, int64_t total, float* __restrict__ out) {
    pdl_trigger();
    pdl_wait();
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * 32 + threadIdx.x;
    const float sum = sum_lanes(part + idx, total, idx < total ? splits : 0, total);
    if (threadIdx.y == 0 && idx < total) out[idx] = sum;
}

// Guarded sums of one problem (see Guard): the SIMT path's splits (simt,
// simt_splits), or the FMA kernel's contributor slots as in
// finalize_slots_kernel.
__global__ void __launch_bounds__(32 * kFinalizeLanes)
finalize_guarded_kernel(const float* __restrict__ part, int64_t Mpad, int64_t M, int C, int rows_per_unit,
                        int64_t key_tiles, int64_t unit_len, int fixed_slots,
                        const float* __restrict__ simt, int simt_splits, float* __restrict__ out,
                        const Guard guard) {
    pdl_trigger();
    pdl_wait();
    const int64_t total = M * C;
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * 32 + threadIdx.x;
    const float* p = simt + idx;
    int64_t stride = total;
    int n = 0;
    if (idx < total) {
        if (guard_simt(guard)) {
            n = simt_splits;
        } else {
            n = static_cast<int>(contributor_slots(div_nonneg(idx, C) / rows_per_unit, fixed_slots, key_tiles,
                                                   unit_len, 0));
            p = part + idx;
            stride = Mpad * C;
        }
    }
    const float sum = sum_lanes(p, stride, n, total);
    if (threadIdx.y == 0 && idx < total) out[idx] = sum;
}

// The same for Cv a multiple of 4 (part_ld is a multiple of 16): one thread
// per quad of channels.  (Bound: HBM and load latency; 65536 rows of 64
// channels, ncu: one thread per channel 26.0 us, quads 10.9.)
constexpr int kFinalizeThreads = 256;

// The sum over ns splits of one quad, added in split order.
__device__ __forceinline__ float4 sum_splits4(const float* __restrict__ p, int64_t step, int ns) {
    float4 a = *reinterpret_cast<const float4*>(p);
    int s = 1;
    for (; s + 8 <= ns; s += 8) {     // (eight loads in flight)
        float4 x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = *reinterpret_cast<const float4*>(p + (s + i) * step);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            a.x += x[i].x;
            a.y += x[i].y;
            a.z += x[i].z;
            a.w += x[i].w;
        }
    }
    for (; s < ns; ++s) {
        const float4 x = *reinterpret_cast<const float4*>(p + s * step);
        a.x += x.x;
        a.y += x.y;
        a.z += x.z;
        a.w += x.w;
    }
    return a;
}

__global__ void __launch_bounds__(kFinalizeThreads)
finalize_quads_kernel(const float* __restrict__ part, int splits, int64_t split_stride_rows,
                      int64_t M, int Cv, int part_ld, const float* __restrict__ inv_scale,
                      float* __restrict__ out, int64_t main_rows) {
    pdl_trigger();
    pdl_wait();
    const int Q = Cv / 4;
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * kFinalizeThreads + threadIdx.x;
    if (idx >= M * Q) return;
    const int64_t m = div_nonneg(idx, Q);
    const int c = 4 * static_cast<int>(idx - m * Q);
    const float4 sc = inv_scale ? *reinterpret_cast<const float4*>(inv_scale + c)
                                : make_float4(1.f, 1.f, 1.f, 1.f);
    float4 a = sum_splits4(part + m * part_ld + c, split_stride_rows * part_ld, m < main_rows ? 1 : splits);
    a.x *= sc.x;
    a.y *= sc.y;
    a.z *= sc.z;
    a.w *= sc.w;
    reinterpret_cast<float4*>(out)[idx] = a;
}

// Gradient contraction for the channels ch0 .. ch0 + Cc - 1 of one launch
// (channel ch = c (D + 1) + d, as in value_at).  With S_j the sum over
// splits of partial channel j (times inv_scale[j] when given):
//   out[m, d] (+)= tau sum_c u[m, c] (S_{c,d} - x^_{m,d} S_{c,D})
//   s_out[m, c]   = S_{c,D}
// where x^ = x - mu is the row's centred point.  DIRECT: the partials
// already hold sum Phi w (k - x) (the fp32 kernel's difference form), so the
// x^ S_{c,D} term is left out.  Terms whose channel lies outside this launch
// are added by the launch that holds it (accumulate = 1 adds to out).  u
// null means u = 1; out may be null when only s_out is wanted.  One thread
// per (m, d) for d < max(D, 1).
template <bool DIRECT, typename T, typename U>
__global__ void finalize_points_kernel(const float* __restrict__ part, int splits,
                                       int64_t split_stride_rows, int64_t M, int part_ld,
                                       const float* __restrict__ inv_scale,
                                       const T* __restrict__ x, const float* __restrict__ mu,
                                       float tau, int D, int Cw, int ch0, int Cc,
                                       const U* __restrict__ u, int accumulate,
                                       float* __restrict__ out, float* __restrict__ s_out,
                                       int64_t main_rows) {
    pdl_trigger();
    pdl_wait();
    const int width = D > 0 ? D : 1;
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= M * width) return;
    const int64_t m = div_nonneg(idx, width);
    const int d = static_cast<int>(idx - m * width);
    const int ns = m < main_rows ? 1 : splits;
    auto S = [&](int j) {
        float acc = 0.f;
        // Unrolled so that the loads of several splits are in flight
        // together (the sum keeps the split order): 71 -> 58 us on the
        // 131072-point gradient with four splits.
#pragma unroll 4
        for (int s = 0; s < ns; ++s)
            acc += part[(static_cast<int64_t>(s) * split_stride_rows + m) * part_ld + j];
        return inv_scale ? acc * inv_scale[j] : acc;
    };
    const int G = D + 1;
    const int c_lo = ch0 / G, c_hi = (ch0 + Cc - 1) / G;
    const float xd = (DIRECT || d >= D) ? 0.f : to_f(x[m * D + d]) - (mu ? mu[d] : 0.f);
    float acc = 0.f;
    for (int c = c_lo; c <= c_hi; ++c) {
        const int jd = c * G + d - ch0;
        const int js = c * G + D - ch0;
        const bool has_d = d < D && jd >= 0 && jd < Cc;
        const bool has_s = js >= 0 && js < Cc;
        if (!has_d && !(has_s && (d == 0 || !DIRECT))) continue;
        const float ss = has_s ? S(js) : 0.f;
        if (d == 0 && has_s && s_out) s_out[m * Cw + c] = ss;
        if (d >= D) continue;
        float t = has_d ? S(jd) : 0.f;
        if (!DIRECT && has_s) t -= xd * ss;
        acc += (u ? to_f(u[m * Cw + c]) : 1.f) * t;
    }
    if (out && d < D) out[m * D + d] = (accumulate ? out[m * D + d] : 0.f) + tau * acc;
}

// finalize_points_kernel for one weight channel whose D + 1 channels are one
// launch's (the q-gradient and the weighted vector-Jacobian passes): one
// thread per quad of coordinates, all its loads issued before any is used.
// The same operations per output, in the same order.  (Bound: HBM and load
// latency, about 4 (D + 16) bytes read and 4 D written per row; 131072 rows,
// D = 32, ncu: one thread per output 56.5 us, quads 14.3.)
// IN_FLIGHT: splits loaded together.  Two cost the fewest registers, and most
// rows have one split; few rows against many keys have up to 64 and wait for
// them (gradient of 78 points against 61876, D = 32: two 72 us, eight 43 per call).
template <typename T, typename U, int IN_FLIGHT>
__global__ void __launch_bounds__(kFinalizeThreads, IN_FLIGHT > 2 ? 2 : 5)
finalize_point_quads_kernel(const float* __restrict__ part, int splits, int64_t split_stride_rows,
                            int64_t M, int part_ld, const float* __restrict__ inv_scale,
                            const T* __restrict__ x, const float* __restrict__ mu, float tau, int D,
                            const U* __restrict__ u, float* __restrict__ out,
                            float* __restrict__ s_out, int64_t main_rows) {
    pdl_trigger();
    pdl_wait();
    const int Q = (D + 3) / 4;
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * kFinalizeThreads + threadIdx.x;
    if (idx >= M * Q) return;
    const int64_t m = div_nonneg(idx, Q);
    const int d = 4 * static_cast<int>(idx - m * Q);
    const int ns = m < main_rows ? 1 : splits;
    const int64_t step = split_stride_rows * part_ld;
    const float* p = part + m * part_ld;
    const bool whole = (D & 3) == 0;    // quads of x and out are aligned
    float xf[4];
    if (whole) {
        T h[4];
        *reinterpret_cast<uint2*>(h) = *reinterpret_cast<const uint2*>(x + m * D + d);
#pragma unroll
        for (int e = 0; e < 4; ++e) xf[e] = to_f(h[e]);
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) xf[e] = d + e < D ? to_f(x[m * D + d + e]) : 0.f;
    }
    const float w = u ? to_f(u[m]) : 1.f;
    // (Channels up to d + 3 < part_ld exist; mu has D values.)
    const float4 is = *reinterpret_cast<const float4*>(inv_scale + d);
    const float isd = inv_scale[D];
    float mf[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) mf[e] = mu && d + e < D ? mu[d + e] : 0.f;
    float4 a = *reinterpret_cast<const float4*>(p + d);
    float ss = p[D];
    int s = 1;
    for (; IN_FLIGHT > 2 && s + IN_FLIGHT <= ns; s += IN_FLIGHT) {
        float4 b[IN_FLIGHT];
        float w1[IN_FLIGHT];
#pragma unroll
        for (int i = 0; i < IN_FLIGHT; ++i) {
            b[i] = *reinterpret_cast<const float4*>(p + (s + i) * step + d);
            w1[i] = p[(s + i) * step + D];
        }
#pragma unroll
        for (int i = 0; i < IN_FLIGHT; ++i) {
            ss += w1[i];
            a.x += b[i].x;
            a.y += b[i].y;
            a.z += b[i].z;
            a.w += b[i].w;
        }
    }
#pragma unroll 2
    for (; s < ns; ++s) {
        const float4 b = *reinterpret_cast<const float4*>(p + s * step + d);
        ss += p[s * step + D];
        a.x += b.x;
        a.y += b.y;
        a.z += b.z;
        a.w += b.w;
    }
    const float sd = ss * isd;
    if (d == 0 && s_out) s_out[m] = sd;
    if (!out) return;
    const float v[4] = {a.x * is.x, a.y * is.y, a.z * is.z, a.w * is.w};
    float o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) o[e] = tau * (w * fmaf(-(xf[e] - mf[e]), sd, v[e]));
    float* dst = out + m * D + d;
    if (whole) {
        *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[3]);
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (d + e < D) dst[e] = o[e];
    }
}

// ---------------------------------------------------------------- values of one weight channel
// value_max_kernel and value_prep_kernel for the D + 1 channels of one weight
// channel (channels w (x - mu) and w).  A block stages kValueRows rows of x,
// one contiguous run, in shared memory with 16-byte loads (any D), then takes
// per-channel maxima, or writes 16 keys of a channel per thread (two 16-byte
// stores, whole sectors).  The element-wise kernels read 2 bytes at a time and
// stored 4: 131072 keys, D = 32, ncu: 19.6 + 24.1 us, these 9.3 + 11.8.  Blocks
// of 128 rows and 128 threads, or of 32 rows and 256 threads where each thread's
// chain of rows is what a call waits for (whole calls, with blocks of 128 rows / of
// 32: gradient of 3000 points, D = 128 57 / 39 us, of 601 points against 44831, D =
// 64 72 / 53; of 300 against 65536, D = 1 52 / 47, D = 12 49 / 44, D = 32 51 / 43, D
// = 64 77 / 54; against 131072, D = 1 57 / 61, D = 12 55 / 57, D = 32 63 / 61, D =
// 64 86 / 80; against 200000, D = 64 100 / 110; vector-Jacobian product of 300
// points, D = 64 78 / 56).
constexpr int kValueRows = 128;
constexpr int kValueThreads = 128;
constexpr int kFewValueRows = 32;
constexpr int kFewValueThreads = 256;
constexpr int64_t kFewValueBlocks = 1280;    // of the larger blocks, 163840 keys,
constexpr int64_t kFewNarrowBlocks = 768;    // or 98304 of fewer than 32 coordinates

// Rows [n0, n0 + ROWS) of x into raw (zeros past N); weights into sw (1
// without weights, 0 past N).  By the whole block.
template <int ROWS, typename T, typename W>
__device__ __forceinline__ void stage_value_rows(const W* __restrict__ w, const T* __restrict__ x,
                                                 int64_t N, int D, int64_t n0, T* raw, float* sw) {
    const int rows = static_cast<int>(max(int64_t(0), min(static_cast<int64_t>(ROWS), N - n0)));
    const int nt = blockDim.x;
    const T* src = x + n0 * D;          // n0 is a multiple of 32: 16-byte aligned
    const int n_el = rows * D, nvec = n_el / 8;
    for (int i = threadIdx.x; i < nvec; i += nt)
        reinterpret_cast<uint4*>(raw)[i] = reinterpret_cast<const uint4*>(src)[i];
    for (int i = nvec * 8 + threadIdx.x; i < n_el; i += nt) raw[i] = src[i];
    for (int i = n_el + threadIdx.x; i < ROWS * D; i += nt) raw[i] = from_f<T>(0.f);
    for (int i = threadIdx.x; i < ROWS; i += nt)
        sw[i] = i < rows ? (w ? to_f(w[n0 + i]) : 1.f) : 0.f;
    __syncthreads();
}

// Largest |value| per channel of the staged rows, into big (float bits; lanes
// take coordinates, warps rows).
template <typename T>
__device__ __forceinline__ void value_rows_max(const T* raw, const float* sw, const float* mu, int rows,
                                               int D, unsigned* big) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    for (int d = lane; d <= D; d += 32) {
        const float m = d < D && mu ? mu[d] : 0.f;
        float mx = 0.f;
        for (int r = warp; r < rows; r += warps)
            mx = fmaxf(mx, fabsf(d < D ? sw[r] * (to_f(raw[r * D + d]) - m) : sw[r]));
        // Non-negative floats order like their bit patterns.
        atomicMax(&big[d], __float_as_uint(mx));
    }
}

// The staged rows' scaled values into vt: item i is channel i mod Cp, keys
// 16 (i / Cp) .. + 15 of the block.  (Npad is a multiple of 128, so the
// block's keys are all inside.)
template <int ROWS, typename T>
__device__ __forceinline__ void value_rows_write(const T* raw, const float* sw, const float* mu, int D, int Cp,
                                                 const unsigned* vmax_bits, int64_t Npad, int64_t n0,
                                                 __half* __restrict__ vt) {
    for (int i = threadIdx.x; i < Cp * (ROWS / 16); i += blockDim.x) {
        const int g = i / Cp, c = i - g * Cp;
        const float sc = c <= D ? pow2f(channel_exponent(vmax_bits[c])) : 0.f;
        const float m = c < D && mu ? mu[c] : 0.f;
        __half2 h[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            float v[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int r = 16 * g + 2 * k + e;
                v[e] = c < D ? sw[r] * (to_f(raw[r * D + c]) - m) : c == D ? sw[r] : 0.f;
            }
            h[k] = __floats2half2_rn(v[0] * sc, v[1] * sc);
        }
        uint4* dst = reinterpret_cast<uint4*>(vt + static_cast<int64_t>(c) * Npad + n0 + 16 * g);
        dst[0] = reinterpret_cast<const uint4*>(h)[0];
        dst[1] = reinterpret_cast<const uint4*>(h)[1];
    }
}

template <int ROWS, int THREADS, typename T, typename W>
__global__ void __launch_bounds__(THREADS)
point_value_max_kernel(const W* __restrict__ w, const T* __restrict__ x,
                       const float* __restrict__ mu, int64_t N, int D,
                       unsigned* __restrict__ vmax_bits) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) uint8_t value_smem[];
    T* raw = reinterpret_cast<T*>(value_smem);
    __shared__ float sw[ROWS];
    __shared__ unsigned big[kOperandMaxCols + 1];
    for (int i = threadIdx.x; i <= D; i += THREADS) big[i] = 0u;
    const int64_t n0 = static_cast<int64_t>(blockIdx.x) * ROWS;
    stage_value_rows<ROWS>(w, x, N, D, n0, raw, sw);
    value_rows_max(raw, sw, mu, static_cast<int>(min(static_cast<int64_t>(ROWS), N - n0)), D, big);
    __syncthreads();
    for (int i = threadIdx.x; i <= D; i += THREADS)
        if (big[i] != 0u) atomicMax(&vmax_bits[i], big[i]);
}

template <int ROWS, int THREADS, typename T, typename W>
__global__ void __launch_bounds__(THREADS)
point_value_prep_kernel(const W* __restrict__ w, const T* __restrict__ x,
                        const float* __restrict__ mu, int64_t N, int64_t Npad, int D, int Cp,
                        const unsigned* __restrict__ vmax_bits, __half* __restrict__ vt,
                        float* __restrict__ inv_scale) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) uint8_t value_smem[];
    T* raw = reinterpret_cast<T*>(value_smem);
    __shared__ float sw[ROWS];
    const int64_t n0 = static_cast<int64_t>(blockIdx.x) * ROWS;
    stage_value_rows<ROWS>(w, x, N, D, n0, raw, sw);
    value_rows_write<ROWS>(raw, sw, mu, D, Cp, vmax_bits, Npad, n0, vt);
    if (blockIdx.x == 0)
        for (int c = threadIdx.x; c < Cp; c += THREADS)
            inv_scale[c] = c <= D ? pow2f(-channel_exponent(vmax_bits[c])) : 0.f;
}

// ---------------------------------------------------------------- small problems in one launch
// The whole preparation of a small problem by one cluster of kPrepCluster
// blocks: the partial sums of the mean (the blocks' shares of the split that
// the separate kernels would use, so that the mean has the same bits), their
// fold through distributed shared memory, the operand rows, and what rides
// along: key or sign records and folded-value flags.  The
// smallest calls wait for the host, about 2 us per launch; this takes two
// launches out.  Its own chain (loads, reduction, two cluster barriers, rows)
// is longer than that of the three kernels it replaces once a block has more
// than one chunk of the mean and one block of rows, hence kPrepMaxRows.
// Measured (whole calls, one GB300, three launches / this one): 1024^2, D = 64
// 25.3 / 21.0 us, 16 problems of 512^2 25.0 / 22.8, of 600 points (MMD^2)
// 29.9 / 26.7; beyond the limit 1500 x 2500, D = 64 24.8 / 27.9, 4000 points,
// D = 50 30.4 / 34.5 us.
constexpr int kPrepCluster = 8;
constexpr int kPrepMaxChunks = 8;            // mean chunks per block of the cluster
constexpr int kPrepMaxParts = 32;            // mean partials folded in sequence (kMeanFinalThreadMax)

template <typename T>
struct PrepArgs {
    const T* q;
    const T* k;
    int64_t M, N;                            // N = 0 for q = k
    MeanSplit split;
    int chunks;                              // chunks per block and step (rows form; 1 otherwise)
    float total;
    int mant_bits, min_exp;
    float* mu;
    // Records (out null: none) and folded-value flags (vf_rec null: none).
    RecordArgs rec;
    float* vf_rec;
    int64_t vf_tiles;
    // Operands: blocks [0, nb0) of j0, then of j1.
    OperandJob j0, j1;
    int nb0, nb;
    int D, Dp, nt;
    float F, half_c, pad_value, cf;
};

template <typename T, bool AUG, int G, bool RAGGED>
__global__ void __cluster_dims__(kPrepCluster, 1, 1) __launch_bounds__(kOperandVecThreads)
prep_cluster_kernel(const PrepArgs<T> a) {
    namespace cg = cooperative_groups;
    using PT = Pair<T>;
    static_assert(kOperandVecThreads == kMeanVecThreads, "one block does both");
    pdl_trigger();
    pdl_wait();
    extern __shared__ uint4 staged[];
    __shared__ float part[2][kPrepMaxChunks][kOperandMaxCols];
    __shared__ float mean[kOperandMaxCols];
    __shared__ uint4 smean[kOperandMaxCols / 8];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = static_cast<int>(cluster.block_rank());
    const int b = blockIdx.y;                // problem of the batch
    const int tid = threadIdx.x;
    const int D = a.D;

    // What depends on the values alone.
    if (a.rec.out) {
        const int64_t pairs = a.rec.Npad / 2;
        const int64_t n = a.rec.signs ? 2 * pairs : pairs;     // signs: whole warps (n % 32 == 0)
        for (int64_t t = rank * kOperandVecThreads + tid; t < n; t += kPrepCluster * kOperandVecThreads) {
            if (a.rec.signs) {
                if constexpr (std::is_same<T, __half>::value)
                    write_sign_record(static_cast<const __half*>(a.rec.v), a.rec.N, a.rec.out, t, b, a.rec.Npad);
            } else if (a.rec.v_f32) {
                write_key_record(RecordJob<float>{static_cast<const float*>(a.rec.v), a.rec.N, pairs, a.rec.C,
                                                  a.rec.out, false}, t, b);
            } else {
                write_key_record(RecordJob<T>{static_cast<const T*>(a.rec.v), a.rec.N, pairs, a.rec.C,
                                              a.rec.out, false}, t, b);
            }
        }
    }

    // Mean: this block's chunks of the split, then the fold over all of them.
    const T* q = a.q + static_cast<int64_t>(b) * a.M * D;
    const T* k = a.k + static_cast<int64_t>(b) * a.N * D;
    const int W = a.chunks, parts = a.split.G;
    MeanShared& sh = *reinterpret_cast<MeanShared*>(staged);
    for (int it = 0;; ++it) {
        const int chunk0 = (it * kPrepCluster + rank) * W;
        if (chunk0 >= parts) break;
        float* ps = part[0][it * W];
        float* pm = part[1][it * W];
        if (a.split.vec)
            mean_vec_block(q, k, a.M, a.N, D, a.split.rpb, a.split.Gq, chunk0, sh, ps, pm);
        else
            mean_rows_block(q, k, a.M, a.N, D, a.split.rpb, parts, W, chunk0, sh,
                            [&](int chunk, int d, float sum, float mx) {
                                ps[(chunk - chunk0) * kOperandMaxCols + d] = sum;
                                pm[(chunk - chunk0) * kOperandMaxCols + d] = mx;
                            });
        __syncthreads();
    }
    cluster.sync();
    // All partials into this block's own shared memory, then the fold in order
    // (one thread per coordinate reading the other blocks' memory partial by
    // partial would wait for each in turn).
    float* all_sum = reinterpret_cast<float*>(staged);
    float* all_max = all_sum + kPrepMaxParts * D;
    for (int g = tid >> 5; g < parts; g += kOperandVecThreads / 32) {
        const int step = g / W, slot = (step / kPrepCluster) * W + (g - step * W);
        const float* rp = cluster.map_shared_rank(&part[0][0][0], step % kPrepCluster) + slot * kOperandMaxCols;
        for (int d = tid & 31; d < D; d += 32) {
            all_sum[g * D + d] = rp[d];
            all_max[g * D + d] = rp[kPrepMaxChunks * kOperandMaxCols + d];
        }
    }
    __syncthreads();
    for (int d = tid; d < D; d += kOperandVecThreads) {
        float s = 0.f, mx = 0.f;
#pragma unroll 8
        for (int g = 0; g < parts; ++g) {
            s += all_sum[g * D + d];
            mx = fmaxf(mx, all_max[g * D + d]);
        }
        const float m = rounded_mean(s, mx, a.total, a.mant_bits, a.min_exp);
        mean[d] = m;
        if (rank == 0) a.mu[static_cast<int64_t>(b) * D + d] = m;
    }
    __syncthreads();
    {
        typename PT::P* sm = reinterpret_cast<typename PT::P*>(smean);
        for (int c = tid; c < 4 * ((D + 7) / 8); c += kOperandVecThreads)
            sm[c] = PT::from_f2(2 * c < D ? mean[2 * c] : 0.f, 2 * c + 1 < D ? mean[2 * c + 1] : 0.f);
    }
    if (a.vf_rec && rank == kPrepCluster - 1)   // (the records are visible since the cluster barrier)
        write_vf_flag(a.vf_rec, a.vf_tiles, static_cast<int>(gridDim.y), b);
    for (int blk = rank; blk < a.nb; blk += kPrepCluster) {
        __syncthreads();                        // staged: the previous use is over
        const bool second = blk >= a.nb0;
        operand_block<T, AUG, G, RAGGED>(second ? a.j1 : a.j0, b, second ? blk - a.nb0 : blk, D, a.Dp, a.nt,
                                         a.F, a.half_c, a.pad_value, a.cf, smean, staged, [] {});
    }
    cluster.sync();     // other blocks may still read this block's shared memory
}

template <typename T, typename W, bool GRAD>
cudaError_t value_prep_typed(const void* w, const void* x, const float* mu, int64_t N,
                             int64_t Npad, int D, int Cw, int ch0, int Cc, int Cp,
                             unsigned* vmax_bits, void* vt, float* inv_scale, cudaStream_t s,
                             bool zeroed) {
    cudaError_t e = cudaSuccess;
    if (!zeroed) {
        e = cudaMemsetAsync(vmax_bits, 0, sizeof(unsigned) * Cp, s);
        if (e != cudaSuccess) return e;
        pdl_reset();   // the next kernel follows a memset
    }
    if (GRAD && Cw == 1 && ch0 == 0 && Cc == D + 1 && D >= 1 && N > 0) {
        auto go = [&](auto kern, int64_t blocks, int rows, int threads, auto... args) {
            const size_t smem = static_cast<size_t>(rows) * D * sizeof(T);
            cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 static_cast<int>(smem));
            if (r != cudaSuccess) return r;
            launch_kernel(kern, static_cast<unsigned>(blocks), threads, smem, s, args...);
            note_launches(1);
            return cudaGetLastError();
        };
        auto both = [&](auto rows_tag, auto threads_tag) {
            constexpr int R = decltype(rows_tag)::value, TH = decltype(threads_tag)::value;
            const cudaError_t r = go(point_value_max_kernel<R, TH, T, W>, (N + R - 1) / R, R, TH,
                                     static_cast<const W*>(w), static_cast<const T*>(x), mu, N, D, vmax_bits);
            if (r != cudaSuccess) return r;
            return go(point_value_prep_kernel<R, TH, T, W>, Npad / R, R, TH, static_cast<const W*>(w),
                      static_cast<const T*>(x), mu, N, Npad, D, Cp, static_cast<const unsigned*>(vmax_bits),
                      static_cast<__half*>(vt), inv_scale);
        };
        if (Npad / kValueRows < (D < 32 ? kFewNarrowBlocks : kFewValueBlocks))
            return both(std::integral_constant<int, kFewValueRows>(), std::integral_constant<int, kFewValueThreads>());
        return both(std::integral_constant<int, kValueRows>(), std::integral_constant<int, kValueThreads>());
    }
    // 64 rows per block: several blocks per SM even for N of a few 10^4.
    const int64_t rows_per_block = 64;
    const int64_t blocks = N > 0 ? (N + rows_per_block - 1) / rows_per_block : 0;
    if (blocks > 0) {
        launch_kernel(value_max_kernel<T, W, GRAD>, static_cast<unsigned>(blocks), dim3(32, 8), 0, s, 
            static_cast<const W*>(w), static_cast<const T*>(x), mu, N, D, Cw, ch0, Cc,
            rows_per_block, vmax_bits);
        note_launches(1);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    dim3 grid(static_cast<unsigned>((Npad + 63) / 64), static_cast<unsigned>((Cp + 31) / 32));
    launch_kernel(value_prep_kernel<T, W, GRAD>, grid, dim3(32, 8), 0, s, 
        static_cast<const W*>(w), static_cast<const T*>(x), mu, N, Npad, D, Cw, ch0, Cc, Cp,
        vmax_bits, static_cast<__half*>(vt), inv_scale);
    note_launches(1);
    return cudaGetLastError();
}

template <bool DIRECT, typename T, typename U>
cudaError_t finalize_points_typed(const float* part, int splits, int64_t stride_rows, int64_t M,
                                  int part_ld, const float* inv_scale, const void* x,
                                  const float* mu, float tau, int D, int Cw, int ch0, int Cc,
                                  const void* u, int accumulate, float* out, float* s_out,
                                  cudaStream_t s, int64_t main_rows) {
    const int64_t total = M * (D > 0 ? D : 1);
    if (total == 0) return cudaSuccess;
    if constexpr (!DIRECT) {
        if (D >= 1 && Cw == 1 && ch0 == 0 && Cc == D + 1 && !accumulate && inv_scale && part_ld % 4 == 0) {
            auto go = [&](auto kern) {
                launch_kernel(kern,
                              static_cast<unsigned>((M * ((D + 3) / 4) + kFinalizeThreads - 1) / kFinalizeThreads),
                              kFinalizeThreads, 0, s, part, splits, stride_rows, M, part_ld, inv_scale,
                              static_cast<const T*>(x), mu, tau, D, static_cast<const U*>(u), out, s_out,
                              main_rows);
                note_launches(1);
                return cudaGetLastError();
            };
            return splits > 8 ? go(finalize_point_quads_kernel<T, U, 8>) : go(finalize_point_quads_kernel<T, U, 2>);
        }
    }
    const int threads = 256;
    const int64_t blocks = (total + threads - 1) / threads;
    launch_kernel(finalize_points_kernel<DIRECT, T, U>, static_cast<unsigned>(blocks), threads, 0, s, 
        part, splits, stride_rows, M, part_ld, inv_scale, static_cast<const T*>(x), mu, tau, D,
        Cw, ch0, Cc, static_cast<const U*>(u), accumulate, out, s_out, main_rows);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace

namespace {

// How the rows of [q; k] (N = 0 for q = k) are split into at most `blocks`
// partial sums.
MeanSplit mean_split(InType t, int64_t M, int64_t N, int D, int blocks) {
    MeanSplit r;
    const int64_t total = M + N;
    r.vec = t != InType::F32 && D >= 8 && D <= 2048 && (D & (D - 1)) == 0 && 2048 % D == 0 && blocks >= 4;
    if (r.vec) {
        // At most `blocks` blocks over both arrays (the partial buffer holds
        // `blocks` rows of 2 D floats).
        r.rpb = std::max<int64_t>(1, (total + blocks - 3) / (blocks - 2));
        r.Gq = static_cast<int>((M + r.rpb - 1) / r.rpb);
        r.G = r.Gq + static_cast<int>((N + r.rpb - 1) / r.rpb);
    } else {
        r.rpb = (total + blocks - 1) / blocks;
        r.Gq = 0;
        r.G = static_cast<int>((total + r.rpb - 1) / r.rpb);
    }
    return r;
}

// Spacing of the input format that the mean is rounded to.
int mean_mant_bits(InType t) { return t == InType::F16 ? 10 : t == InType::BF16 ? 7 : 23; }
int mean_min_exp(InType t) { return t == InType::F16 ? -24 : t == InType::BF16 ? -133 : -149; }

}  // namespace

cudaError_t launch_mean(InType t, const void* q, const void* k, int64_t M, int64_t N, int D,
                        int blocks, float* partial, float* mu, cudaStream_t s, int batch,
                        const RecordArgs* rec, bool* rec_done, ZeroWords zero) {
    if (rec_done) *rec_done = false;
    // q and k the same points: the mean of [q; q] is the mean of q.
    if (q == k && M == N) N = 0;
    const int64_t total = M + N;
    const MeanSplit sp = mean_split(t, M, N, D, blocks);
    const int G = sp.G, Gq = sp.Gq;
    const int64_t rpb = sp.rpb;
    if (sp.vec || (t != InType::F32 && D >= 1 && D <= kMeanVecThreads)) {
        // Key records (see RecordJob) in the blocks behind those of the mean, one
        // thread per key pair, or per key for sign records.
        const int64_t pairs = rec ? rec->Npad / 2 : 0;
        const int64_t rthreads = rec && rec->signs ? 2 * pairs : pairs;
        const int rblocks = static_cast<int>((rthreads + kMeanVecThreads - 1) / kMeanVecThreads);
        // (Rows form: as many chunks per block as leave about 300 blocks.)
        const int chunks = sp.vec ? 1 : static_cast<int>(std::min<int64_t>(
            kMeanVecThreads / D, std::max<int64_t>(1, static_cast<int64_t>(G) * batch / 304)));
        const int mblocks = (G + chunks - 1) / chunks;
        auto go = [&](auto tag, auto vtag) {
            using T = decltype(tag);
            using TV = decltype(vtag);
            const RecordJob<TV> rj = {rec ? static_cast<const TV*>(rec->v) : nullptr, rec ? rec->N : 0,
                                      pairs, rec ? rec->C : 0, rec ? rec->out : nullptr,
                                      rec && rec->signs};
            const T* qt = static_cast<const T*>(q);
            const T* kt = static_cast<const T*>(k);
            const dim3 grid(mblocks + rblocks, batch);
            if (sp.vec)
                launch_kernel(mean_partial_vec_kernel<T, TV>, grid, kMeanVecThreads, 0, s, qt, kt, M, N, D, rpb, Gq,
                              G, partial, rj);
            else
                launch_kernel(mean_partial_rows_kernel<T, TV>, grid, kMeanVecThreads, 0, s, qt, kt, M, N, D, rpb, G,
                              chunks, mblocks, partial, rj);
        };
        const bool vf = rec && rec->v_f32;
        if (t == InType::F16) {
            if (vf) go(__half(), float()); else go(__half(), __half());
        } else {
            if (vf) go(__nv_bfloat16(), float()); else go(__nv_bfloat16(), __nv_bfloat16());
        }
        if (rec_done) *rec_done = rec != nullptr;
        note_launches(1);
    } else {
        // fp32 inputs (16-bit ones have D <= 256).
        launch_kernel(mean_partial_kernel<float>, dim3(G, batch), dim3(32, 8), 0, s,
                      static_cast<const float*>(q), static_cast<const float*>(k), M, N, D, rpb, partial);
        note_launches(1);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int mant_bits = mean_mant_bits(t), min_exp = mean_min_exp(t);
    if (G > kMeanFinalThreadMax) {
        launch_kernel(mean_final_block_kernel, dim3(D, batch), kMeanFinalThreads, 0, s, partial,
                      G, D, static_cast<float>(total), mant_bits, min_exp, mu, zero);
    } else {
        const int64_t items = static_cast<int64_t>(batch) * D;
        launch_kernel(mean_final_kernel,
                      dim3(static_cast<unsigned>((items + kMeanFinalThreads - 1) / kMeanFinalThreads)),
                      kMeanFinalThreads, 0, s, partial, G, D, items, static_cast<float>(total),
                      mant_bits, min_exp, mu, zero);
    }
    note_launches(1);
    return cudaGetLastError();
}

namespace {

// Sec. 3: MMD^2 = v^T s for s = K v (q = k).  Block g of problem b folds
// the products v_n s_n of its chunk of kMmdChunk points (n = chunk start + t,
// + 256, ...) in float64, a fixed tree adds the threads, and
// mmd2_final_kernel adds the chunks of each problem in order
// (deterministic).
constexpr int64_t kMmdChunk = 4096;

template <typename T>
__global__ void __launch_bounds__(256)
mmd2_reduce_kernel(const float* __restrict__ s, const T* __restrict__ v, int64_t N,
                   double* __restrict__ partial) {
    pdl_trigger();
    pdl_wait();
    __shared__ double red[256];
    const int t = threadIdx.x;
    const int64_t b = blockIdx.y;
    const int64_t n0 = static_cast<int64_t>(blockIdx.x) * kMmdChunk;
    const int64_t n1 = min(N, n0 + kMmdChunk);
    double acc = 0.0;
    for (int64_t n = n0 + t; n < n1; n += 256)
        acc += static_cast<double>(to_f(v[b * N + n])) * static_cast<double>(s[b * N + n]);
    red[t] = acc;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (t < w) red[t] += red[t + w];
        __syncthreads();
    }
    if (t == 0) partial[b * gridDim.x + blockIdx.x] = red[0];
}

// The same with s_n added up here from the FMA kernel's contributor slots (in
// slot order, as finalize_slots_kernel does), which saves writing and reading
// s and a launch; with one chunk per problem the result is written at once.
// kMmdChunk points are 16 pairs of 128-row query tiles, whose slot counts are
// worked out once per block; the sums s_n of the chunk are formed by all
// threads, four points each with their loads in flight together (with two
// passes of few blocks the loads' latency is what this costs: one point at a
// time by 256 threads took 10 to 20 us more), and folded in
// mmd2_reduce_kernel's order.  Whole calls, with the overlapped segments
// before and after: 64 problems of 2000 points 70.0 -> 62.5 us, 16 of 4096
// 82 -> 56, 8 of 8000 79.3 -> 73.5, one of 30000 105.3 -> 105.3 us.  (bf16; one
// of 5000 points, D = 64, with two slots' loads in flight 34.9, with six 33.5.)
constexpr int kMmdThreads = 1024;
constexpr int kMmdSlots = 6;

template <typename T>
__global__ void __launch_bounds__(kMmdThreads)
mmd2_slots_kernel(const float* __restrict__ part, int64_t Mpad, int64_t N, int rows_per_unit,
                  int64_t key_tiles, int64_t unit_len, int fixed_slots, int64_t tri_kt,
                  const T* __restrict__ v, double* __restrict__ partial, float* __restrict__ out) {
    pdl_trigger();
    pdl_wait();
    constexpr int PER = static_cast<int>(kMmdChunk) / kMmdThreads;
    __shared__ double red[256];
    __shared__ float sums[kMmdChunk];
    __shared__ int slots[kMmdChunk / 256];
    const int t = threadIdx.x;
    const int64_t b = blockIdx.y, batch = gridDim.y;
    const int64_t n0 = static_cast<int64_t>(blockIdx.x) * kMmdChunk;
    const int64_t n1 = min(N, n0 + kMmdChunk);
    if (t < kMmdChunk / 256)
        slots[t] = n0 + 256 * t < n1
                       ? static_cast<int>(contributor_slots((b * Mpad + n0 + 256 * t) / rows_per_unit,
                                                            fixed_slots, key_tiles, unit_len, tri_kt))
                       : 0;
    __syncthreads();
    const int64_t step = batch * Mpad;
    const float* p = part + b * Mpad + n0 + t;     // (rows up to Mpad exist; those past N are not used)
    int ns[PER], most = 0;
    float s[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        ns[i] = n0 + t + i * kMmdThreads < n1 ? slots[(t + i * kMmdThreads) / 256] : 0;
        most = max(most, ns[i]);
        s[i] = 0.f;
    }
    // (Six slots' loads of the four points in flight together.)
    for (int sl = 0; sl < most; sl += kMmdSlots) {
        float x[kMmdSlots][PER];
#pragma unroll
        for (int u = 0; u < kMmdSlots; ++u)
#pragma unroll
            for (int i = 0; i < PER; ++i)
                x[u][i] = sl + u < ns[i] ? p[(sl + u) * step + i * kMmdThreads] : 0.f;
#pragma unroll
        for (int u = 0; u < kMmdSlots; ++u)
#pragma unroll
            for (int i = 0; i < PER; ++i)
                if (sl + u < ns[i]) s[i] += x[u][i];
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) sums[t + i * kMmdThreads] = s[i];
    __syncthreads();
    if (t < 256) {
        double acc = 0.0;
        for (int64_t n = n0 + t; n < n1; n += 256)
            acc += static_cast<double>(to_f(v[b * N + n])) * static_cast<double>(sums[n - n0]);
        red[t] = acc;
    }
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (t < w) red[t] += red[t + w];
        __syncthreads();
    }
    if (t != 0) return;
    if (gridDim.x == 1) out[b] = static_cast<float>(red[0]);
    else partial[b * gridDim.x + blockIdx.x] = red[0];
}

__global__ void mmd2_final_kernel(const double* __restrict__ partial, int chunks, int64_t B,
                                  float* __restrict__ out) {
    pdl_trigger();
    pdl_wait();
    const int64_t b = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (b >= B) return;
    double acc = 0.0;
    for (int g = 0; g < chunks; ++g) acc += partial[b * chunks + g];
    out[b] = static_cast<float>(acc);
}

}  // namespace

size_t mmd2_partial_bytes(int64_t B, int64_t N) {
    const int64_t chunks = std::max<int64_t>(1, (N + kMmdChunk - 1) / kMmdChunk);
    return static_cast<size_t>(B * chunks) * sizeof(double);
}

cudaError_t launch_mmd2_reduce(InType t, const float* s, const void* v, int64_t B, int64_t N,
                               double* partial, float* out, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    const int64_t chunks = std::max<int64_t>(1, (N + kMmdChunk - 1) / kMmdChunk);
    const dim3 grid(static_cast<unsigned>(chunks), static_cast<unsigned>(B));
    switch (t) {
        case InType::F16:
            launch_kernel(mmd2_reduce_kernel<__half>, grid, 256, 0, st, s, static_cast<const __half*>(v), N,
                                                             partial);
            break;
        case InType::BF16:
            launch_kernel(mmd2_reduce_kernel<__nv_bfloat16>, grid, 256, 0, st, 
                s, static_cast<const __nv_bfloat16*>(v), N, partial);
            break;
        default:
            launch_kernel(mmd2_reduce_kernel<float>, grid, 256, 0, st, s, static_cast<const float*>(v), N,
                                                            partial);
    }
    note_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    launch_kernel(mmd2_final_kernel, static_cast<unsigned>((B + 127) / 128), 128, 0, st, 
        partial, static_cast<int>(chunks), B, out);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_mmd2_slots(InType t, const float* part, int64_t Mpad, int64_t M, int rows_per_unit,
                              int64_t key_tiles, int64_t unit_len, const void* v, double* partial,
                              float* out, cudaStream_t st, int batch, int fixed_slots,
                              int64_t tri_key_tiles) {
    if (rows_per_unit != 256) return cudaErrorInvalidValue;   // (slot counts per 256 rows)
    const int64_t chunks = std::max<int64_t>(1, (M + kMmdChunk - 1) / kMmdChunk);
    const dim3 grid(static_cast<unsigned>(chunks), static_cast<unsigned>(batch));
    if (t == InType::BF16)
        launch_kernel(mmd2_slots_kernel<__nv_bfloat16>, grid, kMmdThreads, 0, st, part, Mpad, M, rows_per_unit,
                      key_tiles, unit_len, fixed_slots, tri_key_tiles,
                      static_cast<const __nv_bfloat16*>(v), partial, out);
    else
        launch_kernel(mmd2_slots_kernel<__half>, grid, kMmdThreads, 0, st, part, Mpad, M, rows_per_unit, key_tiles,
                      unit_len, fixed_slots, tri_key_tiles, static_cast<const __half*>(v), partial, out);
    note_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || chunks == 1) return e;
    launch_kernel(mmd2_final_kernel, static_cast<unsigned>((batch + 127) / 128), 128, 0, st, partial,
                  static_cast<int>(chunks), static_cast<int64_t>(batch), out);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_finalize_slots(const float* part, int64_t Mpad, int64_t M, int C,
                                  int rows_per_unit, int64_t key_tiles, int64_t unit_len,
                                  float* out, cudaStream_t s, int batch, int fixed_slots,
                                  int64_t tri_key_tiles) {
    const int64_t total = static_cast<int64_t>(batch) * M * C;
    if (total == 0) return cudaSuccess;
    const int threads = 256;
    launch_kernel(finalize_slots_kernel, static_cast<unsigned>((total + threads - 1) / threads), threads, 0, s, 
        part, Mpad, M, C, rows_per_unit, key_tiles, unit_len, static_cast<int64_t>(batch),
        fixed_slots, tri_key_tiles, out);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_operands(InType t, bool aug, const void* q, int64_t M, int64_t Mpad,
                            void* qh, void* qh_as_key, float* nrm_q, bool with_k, const void* k,
                            int64_t N, int64_t Npad, void* kh, float* nrm_k, int D, int Dp,
                            const float* mu, float half_c, float pad_value, cudaStream_t s,
                            int batch, const void* vw, float cf, float* vf_rec, bool* flags_done) {
    if (flags_done) *flags_done = false;
    const int64_t vf_tiles = Npad / kRecTile;
    OperandJob jq, jk;
    if (aug) {
        // vw: folded value magnitudes on the key rows (the q job writes the
        // key rows too when q is k).
        jq = {q, M, Mpad, qh, qh_as_key, nullptr, qh_as_key ? vw : nullptr};
        jk = {k, N, Npad, nullptr, kh, nullptr, vw};
    } else {
        jq = {q, M, Mpad, qh, nullptr, nrm_q, nullptr};
        jk = {k, N, Npad, kh, nullptr, nrm_k, nullptr};
    }
    if (!aug) cf = 0.f;
    // (k itself may be null: an empty array when D = 0.)
    const OperandJob* j1 = with_k ? &jk : nullptr;
    const int nt = aug ? aug_norm_terms(t) : 0;
    if (t == InType::BF16) {
        return aug ? operand_typed<__nv_bfloat16, true>(jq, j1, D, Dp, nt, 1.f, mu, 0.f, 0.f, s, batch,
                                                        cf, vf_rec, vf_tiles, flags_done)
                   : operand_typed<__nv_bfloat16, false>(jq, j1, D, Dp, 0, 1.f, mu, half_c,
                                                         pad_value, s, batch, cf, vf_rec,
                                                         vf_tiles, flags_done);
    }
    return aug ? operand_typed<__half, true>(jq, j1, D, Dp, nt, 1024.f, mu, 0.f, 0.f, s, batch,
                                             cf, vf_rec, vf_tiles, flags_done)
               : operand_typed<__half, false>(jq, j1, D, Dp, 0, 1.f, mu, half_c, pad_value, s,
                                              batch, cf, vf_rec, vf_tiles, flags_done);
}

namespace {

template <typename T, bool AUG>
cudaError_t prep_cluster_typed(PrepArgs<T> a, int batch, cudaStream_t s) {
    const bool ragged = a.D % 8 != 0;
    const int V = (a.D + 7) / 8;
    const int G = V <= kOperandVecs ? 1 : V <= 2 * kOperandVecs ? 2 : 4;
    const int64_t slots = kOperandVecThreads / G;
    a.nb0 = static_cast<int>((a.j0.rows_pad + slots - 1) / slots);
    a.nb = a.nb0 + static_cast<int>(a.j1.x ? (a.j1.rows_pad + slots - 1) / slots : 0);
    auto nout = [](const OperandJob& j) { return AUG ? (j.out_q ? 1 : 0) + (j.out_k ? 1 : 0) : 1; };
    size_t smem = static_cast<size_t>(std::max(nout(a.j0), nout(a.j1))) * slots * ((a.Dp / 8) | 1) * 16 +
                  (ragged ? (static_cast<size_t>(slots) * a.D * sizeof(T) + 15) / 16 * 16 : 0);
    smem = std::max(smem, std::max(sizeof(MeanShared), sizeof(float) * 2 * kPrepMaxParts * a.D));
    auto go = [&](auto kern) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   static_cast<int>(smem));
        if (e != cudaSuccess) return e;
        launch_kernel(kern, dim3(kPrepCluster, static_cast<unsigned>(batch)), kOperandVecThreads, smem, s, a);
        note_launches(1);
        return cudaGetLastError();
    };
    switch (G) {
        case 1: return ragged ? go(prep_cluster_kernel<T, AUG, 1, true>) : go(prep_cluster_kernel<T, AUG, 1, false>);
        case 2: return ragged ? go(prep_cluster_kernel<T, AUG, 2, true>) : go(prep_cluster_kernel<T, AUG, 2, false>);
        default: return ragged ? go(prep_cluster_kernel<T, AUG, 4, true>) : go(prep_cluster_kernel<T, AUG, 4, false>);
    }
}

}  // namespace

bool prep_cluster_fits(InType t, const void* q, const void* k, int64_t M, int64_t N, int D, int Dp, int blocks,
                       bool aug, int batch) {
    if (t == InType::F32 || D < 1 || D > kOperandMaxCols || batch > 65535) return false;
    if (aug && (Dp - D < 2 * aug_norm_terms(t) || 2 * Dp > kOperandMaxCols)) return false;
    if (q == k && M == N) N = 0;
    if (M + N > kPrepMaxRows || (M + N) * D > kPrepMaxElements || static_cast<int64_t>(batch) * kPrepCluster > kPrepMaxBlocks) return false;
    return mean_split(t, M, N, D, blocks).G <= kPrepMaxParts;
}

cudaError_t launch_prep_cluster(InType t, bool aug, const void* q, int64_t M, int64_t Mpad, void* qh,
                                void* qh_as_key, float* nrm_q, bool with_k, const void* k, int64_t N,
                                int64_t Npad, void* kh, float* nrm_k, int D, int Dp, int blocks, float* mu,
                                float half_c, float pad_value, cudaStream_t s, int batch, const void* vw,
                                float cf, const RecordArgs* rec, float* vf_rec) {
    auto fill = [&](auto tag) {
        using T = decltype(tag);
        PrepArgs<T> a = {};
        const int64_t kN = q == k && M == N ? 0 : N;
        a.q = static_cast<const T*>(q);
        a.k = static_cast<const T*>(k);
        a.M = M;
        a.N = kN;
        a.split = mean_split(t, M, kN, D, blocks);
        // (Rows form: as many chunks of D threads per step as the cluster has
        // use for; at most kPrepMaxChunks slots per block either way.)
        a.chunks = a.split.vec ? 1 : std::max(1, std::min(kMeanVecThreads / D,
                                                          (a.split.G + kPrepCluster - 1) / kPrepCluster));
        a.total = static_cast<float>(M + kN);
        a.mant_bits = mean_mant_bits(t);
        a.min_exp = mean_min_exp(t);
        a.mu = mu;
        if (rec) a.rec = *rec;
        a.vf_rec = vf_rec;
        a.vf_tiles = Npad / kRecTile;
        a.D = D;
        a.Dp = Dp;
        a.nt = aug ? aug_norm_terms(t) : 0;
        a.F = aug && t == InType::F16 ? 1024.f : 1.f;
        a.half_c = aug ? 0.f : half_c;
        a.pad_value = aug ? 0.f : pad_value;
        a.cf = aug ? cf : 0.f;
        if (aug) {
            a.j0 = {q, M, Mpad, qh, qh_as_key, nullptr, qh_as_key ? vw : nullptr};
            if (with_k) a.j1 = {k, N, Npad, nullptr, kh, nullptr, vw};
        } else {
            a.j0 = {q, M, Mpad, qh, nullptr, nrm_q, nullptr};
            if (with_k) a.j1 = {k, N, Npad, kh, nullptr, nrm_k, nullptr};
        }
        return a;
    };
    if (t == InType::BF16)
        return aug ? prep_cluster_typed<__nv_bfloat16, true>(fill(__nv_bfloat16()), batch, s)
                   : prep_cluster_typed<__nv_bfloat16, false>(fill(__nv_bfloat16()), batch, s);
    return aug ? prep_cluster_typed<__half, true>(fill(__half()), batch, s)
               : prep_cluster_typed<__half, false>(fill(__half()), batch, s);
}

cudaError_t launch_tf32_split(const Tf32Job& q, const Tf32Job* k, int D, int Dp, const float* mu,
                              float half_c, float pad_value, cudaStream_t s, int batch,
                              unsigned* guard, const RecordArgs& rec) {
    const RecordJob<float> rj = {static_cast<const float*>(rec.v), rec.N, rec.Npad / 2, rec.C, rec.out, false};
    const int64_t total0 = q.rows_pad * batch;
    const int64_t total = total0 + (k ? k->rows_pad * batch : 0);
    if (total == 0) return cudaSuccess;
    if ((Dp != 32 && Dp != 64) || q.rows_pad % kSplitRows != 0 || (k && k->rows_pad % kSplitRows != 0))
        return cudaErrorInvalidValue;
    const int64_t warps = total / kSplitRows;
    const unsigned blocks = static_cast<unsigned>((warps * 32 + kSplitThreads - 1) / kSplitThreads);
    const Tf32Job jk = k ? *k : Tf32Job{};
    if (Dp == 32)
        launch_kernel(tf32_split_kernel<1>, blocks, kSplitThreads, 0, s, q, jk, total0, total, D, mu, half_c,
                      pad_value, guard, rj);
    else
        launch_kernel(tf32_split_kernel<2>, blocks, kSplitThreads, 0, s, q, jk, total0, total, D, mu, half_c,
                      pad_value, guard, rj);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_value_prep(InType t, bool grad, bool w_f32, const void* w, const void* x,
                              const float* mu, int64_t N, int64_t Npad, int D, int Cw, int ch0,
                              int Cc, int Cp, unsigned* vmax_bits, void* vt, float* inv_scale,
                              cudaStream_t s, bool zeroed) {
#define GS_VALUE_PREP(T, W, G) \
    value_prep_typed<T, W, G>(w, x, mu, N, Npad, D, Cw, ch0, Cc, Cp, vmax_bits, vt, inv_scale, s, zeroed)
    if (t == InType::BF16) {
        if (!grad)
            return w_f32 ? GS_VALUE_PREP(__nv_bfloat16, float, false)
                         : GS_VALUE_PREP(__nv_bfloat16, __nv_bfloat16, false);
        return w_f32 ? GS_VALUE_PREP(__nv_bfloat16, float, true)
                     : GS_VALUE_PREP(__nv_bfloat16, __nv_bfloat16, true);
    }
    if (!grad) return w_f32 ? GS_VALUE_PREP(__half, float, false) : GS_VALUE_PREP(__half, __half, false);
    return w_f32 ? GS_VALUE_PREP(__half, float, true) : GS_VALUE_PREP(__half, __half, true);
#undef GS_VALUE_PREP
}


cudaError_t launch_key_records(InType t, const void* v, const float* B, int64_t N, int64_t Npad,
                               int C, float* rec, cudaStream_t s, int batch, bool signs) {
    if (signs) {
        // Sign records (fp16 values, C = 1): one thread per key, 256 per block.
        if (t != InType::F16 || C != 1 || B || Npad % kRecTile != 0) return cudaErrorInvalidValue;
        if (Npad == 0) return cudaSuccess;
        launch_kernel(sign_record_kernel, dim3(static_cast<unsigned>((Npad + 255) / 256), batch), 256, 0,
                      s, static_cast<const __half*>(v), N, Npad, rec);
        note_launches(1);
        return cudaGetLastError();
    }
    const int64_t pairs = Npad / 2;
    if (pairs == 0) return cudaSuccess;
    const int threads = 256;
    const unsigned blocks = static_cast<unsigned>((pairs + threads - 1) / threads);
    if (t == InType::BF16)
        launch_kernel(key_record_kernel<__nv_bfloat16>, dim3(blocks, batch), threads, 0, s, 
            static_cast<const __nv_bfloat16*>(v), B, N, pairs, C, rec);
    else if (t == InType::F32)
        launch_kernel(key_record_kernel<float>, dim3(blocks, batch), threads, 0, s, 
            static_cast<const float*>(v), B, N, pairs, C, rec);
    else
        launch_kernel(key_record_kernel<__half>, dim3(blocks, batch), threads, 0, s, static_cast<const __half*>(v), B, N,
                                                             pairs, C, rec);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_vf_flags(float* rec, int64_t Npad, int batch, cudaStream_t s) {
    if (batch <= 0) return cudaSuccess;
    launch_kernel(vf_flags_kernel, dim3(static_cast<unsigned>(batch)), 256, 0, s, rec, Npad / kRecTile,
                  batch);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_weight_prep(InType t, const void* rsrc, bool r_f32, int64_t R, int64_t Rpad,
                               const void* csrc, bool c_f32, int64_t Ncol, int64_t Npad, int C,
                               int WT, int BN, float* rowf, float* colT, unsigned* wmax,
                               cudaStream_t s, bool zeroed) {
    if (WT <= 0 || kWeightThreads % WT != 0 || C > WT) return cudaErrorInvalidValue;
    if (!zeroed) {
        const cudaError_t e = cudaMemsetAsync(wmax, 0, sizeof(unsigned) * 2 * WT, s);
        if (e != cudaSuccess) return e;
        pdl_reset();   // the next kernel follows a memset
    }
    const int64_t rb = (Rpad * WT + kWeightThreads - 1) / kWeightThreads;
    const int64_t cb = (Npad * WT + kWeightThreads - 1) / kWeightThreads;
    if (rb + cb == 0) return cudaSuccess;
    const dim3 grid(static_cast<unsigned>(rb + cb));
    const unsigned rbu = static_cast<unsigned>(rb);
#define GS_WPREP(TR, TC)                                                                        \
    launch_kernel(weight_prep_kernel<TR, TC>, grid, kWeightThreads, 0, s,                      \
                  static_cast<const TR*>(rsrc), R, Rpad, static_cast<const TC*>(csrc), Ncol,   \
                  Npad, C, WT, BN, rbu, rowf, colT, wmax)
    // One side is the float32 upstream gradient, the other the inputs' dtype.
    if (t == InType::BF16) {
        if (r_f32 && !c_f32) GS_WPREP(float, __nv_bfloat16);
        else if (!r_f32 && c_f32) GS_WPREP(__nv_bfloat16, float);
        else return cudaErrorInvalidValue;
    } else if (t == InType::F16) {
        if (r_f32 && !c_f32) GS_WPREP(float, __half);
        else if (!r_f32 && c_f32) GS_WPREP(__half, float);
        else return cudaErrorInvalidValue;
    } else {
        return cudaErrorInvalidValue;
    }
#undef GS_WPREP
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_finalize(const float* part, int splits, int64_t split_stride_rows,
                            int64_t M, int Cv, int part_ld, const float* inv_scale, float* out,
                            cudaStream_t s, int64_t main_rows) {
    const int64_t total = M * Cv;
    if (total == 0) return cudaSuccess;
    if (many_partials(splits, total) && !inv_scale && main_rows == 0 && part_ld == Cv &&
        split_stride_rows == M) {
        launch_kernel(finalize_many_kernel, static_cast<unsigned>((total + 31) / 32), dim3(32, kFinalizeLanes), 0,
                      s, part, splits, total, out);
        note_launches(1);
        return cudaGetLastError();
    }
    if (Cv % 4 == 0 && part_ld % 4 == 0) {
        launch_kernel(finalize_quads_kernel,
                      static_cast<unsigned>((total / 4 + kFinalizeThreads - 1) / kFinalizeThreads),
                      kFinalizeThreads, 0, s, part, splits, split_stride_rows, M, Cv, part_ld, inv_scale, out, main_rows);
        note_launches(1);
        return cudaGetLastError();
    }
    const int threads = 256;
    const int64_t blocks = (total + threads - 1) / threads;
    launch_kernel(finalize_kernel, static_cast<unsigned>(blocks), threads, 0, s, 
        part, splits, split_stride_rows, M, Cv, part_ld, inv_scale, out, main_rows);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_finalize_guarded(const float* part, int64_t Mpad, int64_t M, int C, int rows_per_unit,
                                    int64_t key_tiles, int64_t unit_len, int fixed_slots, const float* simt,
                                    int simt_splits, float* out, cudaStream_t s, const Guard& guard) {
    const int64_t total = M * C;
    if (total == 0) return cudaSuccess;
    launch_kernel(finalize_guarded_kernel, static_cast<unsigned>((total + 31) / 32), dim3(32, kFinalizeLanes), 0, s,
                  part, Mpad, M, C, rows_per_unit, key_tiles, unit_len, fixed_slots, simt, simt_splits, out, guard);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_finalize_points(bool direct, InType t, bool u_f32, const float* part,
                                   int splits, int64_t split_stride_rows, int64_t M, int part_ld,
                                   const float* inv_scale, const void* x, const float* mu,
                                   float tau, int D, int Cw, int ch0, int Cc, const void* u,
                                   int accumulate, float* out, float* s_out, cudaStream_t s,
                                   int64_t main_rows) {
#define GS_FIN(DIR, T, U)                                                                     \
    finalize_points_typed<DIR, T, U>(part, splits, split_stride_rows, M, part_ld, inv_scale, x, \
                                     mu, tau, D, Cw, ch0, Cc, u, accumulate, out, s_out, s,      \
                                     main_rows)
    if (direct) return GS_FIN(true, float, float);
    if (t == InType::BF16)
        return u_f32 ? GS_FIN(false, __nv_bfloat16, float)
                     : GS_FIN(false, __nv_bfloat16, __nv_bfloat16);
    return u_f32 ? GS_FIN(false, __half, float) : GS_FIN(false, __half, __half);
#undef GS_FIN
}

}  // namespace gs
