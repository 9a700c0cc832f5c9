// fp32 SIMT Gauss-sum kernels (the single-precision regime of the paper's
// appendix, where tensor-core attention is not available).
//
// Query rows live in registers, zero padded; keys stream through shared
// memory in tiles (zero padded likewise, so padded coordinates add
// (0 - 0)^2 = 0).  For each pair the squared distance is formed in the
// direct-difference form sum_d (q_d - k_d)^2 (no Gram identity, hence no
// cancellation), the kernel value is 2^(-(c/2) d^2) with c = tau log2 e, and
// the values are accumulated with fp32 FMAs:
//   forward (Eq. 1):     acc[j] += Phi v[n, c0 + j]       for CBLK channels
//   gradient (Sec. 3):   acc[d] += Phi w_n (k_d - q_d),   acc[D] += Phi w_n
//                        with w_n = v[n, c] for one weight channel c
// The key range is split over gridDim.y; partial sums go to a workspace and
// are added in a fixed order by the finalise kernel.  Coordinates are
// handled in pairs with the packed f32x2 subtract / FMA of sm_100+ (the
// squared distance accumulates even and odd coordinates separately and
// adds the two at the end).  Bound: the fp32 lanes, 2 D operations per pair.
#include <algorithm>
#include <cmath>

#include "internal.h"
#include "ptx.cuh"

namespace gs {
namespace {

constexpr int KT = 64;       // keys per shared-memory tile (gradient; forward: key_tile)
constexpr int THREADS = 128; // threads per block (forward: or fewer, see plan_simt)
// Partial sums of more than one split (16 MiB): the scratch of gauss_sum_noalloc
// holds every call that it would hold unsplit.
constexpr int64_t kMaxSplitFloats = int64_t(1) << 22;

// ---------------------------------------------------------------- forward
// Each thread holds ROWS = 4 query rows of up to 32 coordinates, so that one
// broadcast load of four key coordinates serves 16 packed operations: with
// one row per thread the 16-byte loads, not the packed subtracts and FMAs,
// set the pace (in-register rate of the mix by rows per load: 1 row 66 % of
// the fp32 lanes, 2 rows 74 %, 4 rows 80 %, 8 rows 84 %).  Wider points are
// shared by L = 2 or 4 neighbouring lanes: lane l of a group holds the
// coordinate quads l, l + L, .. of the group's four rows, and the lanes
// exchange partial squared distances so that each ends up with 4 / L rows of
// its own for the exponential and the values.  Key tiles are copied with
// cp.async into two buffers, the next one under the arithmetic of the current
// one.  Measured (one GB300, whole calls, C = 1, one row per thread in tiles
// of 16, 32, 64 or 128 coordinates / this kernel): M = N = 16384, D = 4 435 /
// 106 us, D = 16 435 / 281, D = 32 794 / 524, D = 48 1306 / 824, D = 64 1316
// / 1088 (78 % of the lanes), D = 128 2919 / 2291; 4096^2, D = 16 39 / 27 us.
constexpr int ROWS = 4;
__host__ __device__ constexpr int lanes_per_group(int dmax) { return dmax <= 32 ? 1 : dmax <= 64 ? 2 : 4; }
__host__ __device__ constexpr int key_tile(int dmax) { return dmax <= 64 ? 64 : 32; }
// Blocks per SM that the registers are limited to (65536 / (128 x blocks)).
__host__ __device__ constexpr int min_blocks(int dmax, int cblk) {
    return dmax <= 16 ? 4 : dmax == 32 && cblk == 4 ? 2 : 3;
}

__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(valid ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

template <int DMAX, int CBLK>
__global__ void __launch_bounds__(THREADS, min_blocks(DMAX, CBLK))
simt_sum_kernel(const float* __restrict__ q, const float* __restrict__ k,
                const float* __restrict__ v, int64_t M, int64_t N, int D, int Cv, float half_c,
                int64_t keys_per_split, float* __restrict__ part,
                const Guard guard) {
    pdl_trigger();
    pdl_wait();
    if (guard.words && !guard_simt(guard)) return;   // the tensor-core path does the call
    constexpr int L = lanes_per_group(DMAX);
    constexpr int DL = DMAX / L;          // coordinates per lane
    constexpr int OWN = ROWS / L;         // rows whose sums a lane keeps
    constexpr int KTF = key_tile(DMAX);
    static_assert(DL % 4 == 0 && DL <= 32, "coordinate quads of a lane");
    __shared__ __align__(16) float ks[2][KTF][DMAX];
    __shared__ __align__(16) float vs[2][KTF][CBLK];

    const int nthreads = blockDim.x, GROUPS = nthreads / L;
    const int sub = threadIdx.x % L;
    const int64_t m0 = static_cast<int64_t>(blockIdx.x) * (GROUPS * ROWS) + threadIdx.x / L;
    const int split = blockIdx.y;
    const int c0 = blockIdx.z * CBLK;
    const int64_t n_begin = static_cast<int64_t>(split) * keys_per_split;
    const int64_t n_end = min(N, n_begin + keys_per_split);

    // Tile of up to KTF keys from t0 into buffer b; the coordinates and channels
    // past D and Cv are filled with zeros (nothing is read for them; their
    // source address is v, which is never null here, as k may be when D = 0).
    // Rows past n_end are left as they are, and not used.
    auto load_tile = [&](int b, int64_t t0) {
        const int cnt = static_cast<int>(min(static_cast<int64_t>(KTF), n_end - t0));
        const float* kt = k + t0 * D;
        for (int i = threadIdx.x; i < cnt * DMAX; i += nthreads) {
            const int kk = i / DMAX, d = i - kk * DMAX;
            const bool in = d < D;
            cp_async4(&ks[b][kk][d], in ? kt + kk * D + d : v, in);
        }
        const float* vt = v + t0 * Cv + c0;
        for (int i = threadIdx.x; i < cnt * CBLK; i += nthreads) {
            const int kk = i / CBLK, j = i - kk * CBLK;
            const bool in = c0 + j < Cv;
            cp_async4(&vs[b][kk][j], in ? vt + static_cast<int64_t>(kk) * Cv + j : v, in);
        }
        cp_async_commit();
    };
    if (n_begin < n_end) load_tile(0, n_begin);

    uint64_t qr[ROWS][DL / 2];   // coordinate pairs of the query rows
    // Sums of the key tiles, added up tile by tile (two-level summation: the
    // rounding error of a split's sum grows with the keys per tile plus the
    // tiles, not with all its keys).
    float acc[OWN][CBLK];
    // (In the widest loads that every row's alignment allows: each load touches
    // 32 rows, and 4-byte loads of four 32-coordinate rows kept the load path
    // busy for about 8 us per block.)
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const int64_t m = m0 + r * GROUPS;
        const float* qm = q + m * D;
#pragma unroll
        for (int i = 0; i < DL; i += 4) {
            const int d = i * L + 4 * sub;
            float x[4] = {0.f, 0.f, 0.f, 0.f};
            if (m < M && d < D) {
                if ((D & 3) == 0) {
                    *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(qm + d);
                } else if ((D & 1) == 0) {
                    *reinterpret_cast<float2*>(x) = *reinterpret_cast<const float2*>(qm + d);
                    if (d + 2 < D) *reinterpret_cast<float2*>(x + 2) = *reinterpret_cast<const float2*>(qm + d + 2);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (d + e < D) x[e] = qm[d + e];
                }
            }
            qr[r][i / 2] = f32x2_pack(x[0], x[1]);
            qr[r][i / 2 + 1] = f32x2_pack(x[2], x[3]);
        }
    }
#pragma unroll
    for (int r = 0; r < OWN; ++r)
#pragma unroll
        for (int j = 0; j < CBLK; ++j) acc[r][j] = 0.f;

    int b = 0;
    for (int64_t t0 = n_begin; t0 < n_end; t0 += KTF, b ^= 1) {
        const int cnt = static_cast<int>(min(static_cast<int64_t>(KTF), n_end - t0));
        if (t0 + KTF < n_end) {
            load_tile(b ^ 1, t0 + KTF);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        float tile[OWN][CBLK];
#pragma unroll
        for (int r = 0; r < OWN; ++r)
#pragma unroll
            for (int j = 0; j < CBLK; ++j) tile[r][j] = 0.f;
        for (int kk = 0; kk < cnt; ++kk) {
            uint64_t d2p[ROWS];   // (even, odd) partial squared distances
#pragma unroll
            for (int r = 0; r < ROWS; ++r) d2p[r] = 0ull;
#pragma unroll
            for (int i = 0; i < DL; i += 4) {
                const float4 kv = *reinterpret_cast<const float4*>(&ks[b][kk][i * L + 4 * sub]);
                const uint64_t k01 = f32x2_pack(kv.x, kv.y), k23 = f32x2_pack(kv.z, kv.w);
#pragma unroll
                for (int r = 0; r < ROWS; ++r) {
                    const uint64_t t01 = f32x2_sub(qr[r][i / 2], k01);
                    const uint64_t t23 = f32x2_sub(qr[r][i / 2 + 1], k23);
                    d2p[r] = f32x2_fma(t01, t01, d2p[r]);
                    d2p[r] = f32x2_fma(t23, t23, d2p[r]);
                }
            }
            float d2[ROWS];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                float d2e, d2o;
                f32x2_unpack(d2p[r], d2e, d2o);
                d2[r] = d2e + d2o;
            }
            // Halve the rows with the neighbouring lanes: each keeps the
            // half that own_row names and hands over the other.
            if (L >= 2) {
                const bool hi = (threadIdx.x & 1) != 0;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float give = hi ? d2[r] : d2[r + 2], keep = hi ? d2[r + 2] : d2[r];
                    d2[r] = keep + __shfl_xor_sync(0xffffffffu, give, 1);
                }
            }
            if (L >= 4) {
                const bool hi = (threadIdx.x & 2) != 0;
                const float give = hi ? d2[0] : d2[1], keep = hi ? d2[1] : d2[0];
                d2[0] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
            }
#pragma unroll
            for (int r = 0; r < OWN; ++r) {
                const float phi = ex2_approx(-half_c * d2[r]);
#pragma unroll
                for (int j = 0; j < CBLK; ++j) tile[r][j] = fmaf(phi, vs[b][kk][j], tile[r][j]);
            }
        }
#pragma unroll
        for (int r = 0; r < OWN; ++r)
#pragma unroll
            for (int j = 0; j < CBLK; ++j) acc[r][j] += tile[r][j];
        __syncthreads();   // every thread is done with buffer b
    }
#pragma unroll
    for (int r = 0; r < OWN; ++r) {
        const int own_row = L == 1 ? r : L == 2 ? 2 * (sub & 1) + r : 2 * (sub & 1) + (sub >> 1);
        const int64_t m = m0 + own_row * GROUPS;
        if (m >= M) continue;
        float* out = part + (static_cast<int64_t>(split) * M + m) * Cv + c0;
#pragma unroll
        for (int j = 0; j < CBLK; ++j)
            if (c0 + j < Cv) out[j] = acc[r][j];
    }
}

// ---------------------------------------------------------------- gradient
template <int DMAX>
__global__ void __launch_bounds__(THREADS)
simt_grad_kernel(const float* __restrict__ q, const float* __restrict__ k,
                 const float* __restrict__ v, int64_t M, int64_t N, int D, int Cv,
                 int wch, float half_c, int64_t keys_per_split, float* __restrict__ part) {
    pdl_trigger();
    pdl_wait();
    __shared__ __align__(16) float ks[KT][DMAX];
    __shared__ float vs[KT];

    const int64_t m = static_cast<int64_t>(blockIdx.x) * THREADS + threadIdx.x;
    const int split = blockIdx.y;
    const int64_t n_begin = static_cast<int64_t>(split) * keys_per_split;
    const int64_t n_end = min(N, n_begin + keys_per_split);

    uint64_t qr[DMAX / 2];   // coordinate pairs of the query row
#pragma unroll
    for (int d = 0; d < DMAX; d += 2)
        qr[d / 2] = f32x2_pack((m < M && d < D) ? q[m * D + d] : 0.f,
                               (m < M && d + 1 < D) ? q[m * D + d + 1] : 0.f);
    float acc = 0.f;              // sum of Phi w
    uint64_t acc2[DMAX / 2];      // gradient coordinates, in pairs
#pragma unroll
    for (int j = 0; j < DMAX / 2; ++j) acc2[j] = 0ull;

    for (int64_t t0 = n_begin; t0 < n_end; t0 += KT) {
        const int cnt = static_cast<int>(min(static_cast<int64_t>(KT), n_end - t0));
        __syncthreads();
        for (int i = threadIdx.x; i < KT * DMAX; i += THREADS) {
            const int kk = i / DMAX, d = i - kk * DMAX;
            ks[kk][d] = (kk < cnt && d < D) ? k[(t0 + kk) * D + d] : 0.f;
        }
        // v is N x Cv; the weight is its channel wch.
        for (int i = threadIdx.x; i < KT; i += THREADS)
            vs[i] = i < cnt ? v[(t0 + i) * Cv + wch] : 0.f;
        __syncthreads();
        for (int kk = 0; kk < cnt; ++kk) {
            uint64_t d2p = 0ull;   // (even, odd) partial squared distances
#pragma unroll
            for (int d = 0; d < DMAX; d += 4) {
                const float4 kv = *reinterpret_cast<const float4*>(&ks[kk][d]);
                const uint64_t t0 = f32x2_sub(qr[d / 2], f32x2_pack(kv.x, kv.y));
                const uint64_t t1 = f32x2_sub(qr[d / 2 + 1], f32x2_pack(kv.z, kv.w));
                d2p = f32x2_fma(t0, t0, d2p);
                d2p = f32x2_fma(t1, t1, d2p);
            }
            float d2e, d2o;
            f32x2_unpack(d2p, d2e, d2o);
            const float phi = ex2_approx(-half_c * (d2e + d2o));
            const float w = phi * vs[kk];
            const uint64_t w2 = f32x2_pack(w, w);
#pragma unroll
            for (int d = 0; d < DMAX; d += 4) {
                const float4 kv = *reinterpret_cast<const float4*>(&ks[kk][d]);
                acc2[d / 2] = f32x2_fma(w2, f32x2_sub(f32x2_pack(kv.x, kv.y), qr[d / 2]), acc2[d / 2]);
                acc2[d / 2 + 1] =
                    f32x2_fma(w2, f32x2_sub(f32x2_pack(kv.z, kv.w), qr[d / 2 + 1]), acc2[d / 2 + 1]);
            }
            acc += w;
        }
    }
    if (m >= M) return;
    float* out = part + (static_cast<int64_t>(split) * M + m) * (D + 1);
#pragma unroll
    for (int d = 0; d < DMAX; d += 2) {
        float lo, hi;
        f32x2_unpack(acc2[d / 2], lo, hi);
        if (d < D) out[d] = lo;
        if (d + 1 < D) out[d + 1] = hi;
    }
    out[D] = acc;
}

template <int DMAX>
cudaError_t launch_grad(const SimtPlan& p, const float* q, const float* k, const float* v, int Cw,
                        int wch, float half_c, float* part, cudaStream_t s) {
    dim3 grid(static_cast<unsigned>((p.M + THREADS - 1) / THREADS), p.splits);
    launch_kernel(simt_grad_kernel<DMAX>, grid, THREADS, 0, s, q, k, v, p.M, p.N,
                  static_cast<int>(p.D), Cw, wch, half_c, p.keys_per_split, part);
    note_launches(1);
    return cudaGetLastError();
}

template <int DMAX, int CBLK>
cudaError_t launch_cblk(const SimtPlan& p, const float* q, const float* k, const float* v,
                        float half_c, float* part, cudaStream_t s, const Guard& guard) {
    const int rows = p.threads / lanes_per_group(DMAX) * ROWS;
    dim3 grid(static_cast<unsigned>((p.M + rows - 1) / rows), p.splits,
              static_cast<unsigned>((p.Cv + CBLK - 1) / CBLK));
    launch_kernel(simt_sum_kernel<DMAX, CBLK>, grid, p.threads, 0, s, q, k, v, p.M, p.N,
                  static_cast<int>(p.D), static_cast<int>(p.Cv), half_c, p.keys_per_split, part,
                  guard);
    note_launches(1);
    return cudaGetLastError();
}

// Channel blocks of 4, or of 1 or 2 for as few channels (no idle FMAs).
template <int DMAX>
cudaError_t launch_dmax(const SimtPlan& p, const float* q, const float* k, const float* v,
                        float half_c, float* part, cudaStream_t s, const Guard& guard) {
    if (p.cblk == 1) return launch_cblk<DMAX, 1>(p, q, k, v, half_c, part, s, guard);
    if (p.cblk == 2) return launch_cblk<DMAX, 2>(p, q, k, v, half_c, part, s, guard);
    return launch_cblk<DMAX, 4>(p, q, k, v, half_c, part, s, guard);
}

}  // namespace

bool plan_simt(int64_t M, int64_t N, int64_t D, int64_t C, bool grad, int split_override,
               int sms, SimtPlan* p, const char** why) {
    p->M = M;
    p->N = N;
    p->D = D;
    p->Cv = grad ? D + 1 : C;
    const int64_t dlimit = grad ? 64 : 128;
    if (D > dlimit) {
        *why = grad ? "fp32 gradient supports D <= 64" : "fp32 path supports D <= 128";
        return false;
    }
    p->micros = 0.0;
    p->cblk = p->Cv >= 3 ? 4 : static_cast<int>(std::max<int64_t>(1, p->Cv));
    int64_t rows, keys;   // query rows per block, keys per shared-memory tile
    if (grad) {
        p->dmax = D <= 16 ? 16 : D <= 32 ? 32 : 64;
        rows = THREADS;
        keys = KT;
    } else {
        // Register tiles of the query rows: the smallest that holds D.
        p->dmax = D <= 4 ? 4 : D <= 8 ? 8 : D <= 16 ? 16 : D <= 24 ? 24 : D <= 32 ? 32
                : D <= 48 ? 48 : D <= 56 ? 56 : D <= 64 ? 64 : 128;
        rows = THREADS / lanes_per_group(p->dmax) * ROWS;
        keys = key_tile(p->dmax);
    }
    const int64_t chunks = grad ? 1 : std::max<int64_t>(1, (p->Cv + p->cblk - 1) / p->cblk);
    int64_t blocks = (M + rows - 1) / rows * chunks;   // per key split
    p->threads = THREADS;
    const int64_t key_tiles = std::max<int64_t>(1, (N + keys - 1) / keys);
    if (grad || split_override > 0) {
        int64_t splits = split_override > 0 ? split_override : (4LL * sms + blocks - 1) / blocks;
        splits = std::max<int64_t>(1, std::min<int64_t>(splits, key_tiles));
        splits = std::min<int64_t>(splits, 65535);
        p->keys_per_split = grad ? (key_tiles + splits - 1) / splits * keys
                                 : std::max<int64_t>(4, ((N + splits - 1) / splits + 3) / 4 * 4);
    } else {
        // Threads per block and key splits by an estimate of the busiest SM's
        // time, fitted to whole calls (one GB300, 1800 shapes of 1 to 200000
        // rows and keys, 1 to 128 coordinates, 1 to 16 channels, each with 30
        // choices: the estimate's choice is 4 % slower than the best one on
        // average).  A warp takes `key` issue cycles per key of its rows:
        // coordinates, exponentials, values and its share of copying the key
        // tile, which few threads per block make dear; an SMSP with fewer than
        // about two warps waits for latencies instead.  Each block costs a
        // start, each split a partial sum per output to write and add, and the
        // blocks of a single wave wait at their barriers together.  Blocks
        // of 128 threads share the copies best; 64 and 32 (128 query rows up to
        // 32 coordinates) are for few rows, which full blocks would pad: 32 x
        // 65536, D = 64, 256 splits of 64-thread blocks 67 us, 608 of 32
        // threads 41.
        const int L = lanes_per_group(p->dmax);
        const double issue = 2.3 * (p->dmax / L) + 10.0 + 2.0 * p->cblk / L + (L > 1 ? 20.0 : 0.0);
        const double few = L > 1 ? 1.5 : 2.1;                  // warps per SMSP
        const double few4 = few * few * few * few;
        const int64_t smem = 2 * keys * (p->dmax + p->cblk) * 4 + 1024;
        double best = 1e300;
        for (int threads = THREADS; threads >= 32; threads /= 2) {
            const int64_t r = rows * threads / THREADS;
            const double key = issue + 20.0 * (p->dmax + p->cblk) / threads;
            const double warps = threads / 128.0;              // per SMSP and block
            const int64_t fit = std::min<int64_t>(228 * 1024 / smem, min_blocks(p->dmax, p->cblk) * THREADS / threads);
            blocks = (M + r - 1) / r * chunks;
            int64_t tried = 0;
            for (int64_t per : {1, 2, 3, 4, 6, 8, 12, 16, 24, 32}) {
                const int64_t want = std::max<int64_t>(1, per * sms / blocks);
                const int64_t kps = std::max<int64_t>(16, ((N + want - 1) / want + 3) / 4 * 4);
                const int64_t n = (N + kps - 1) / kps;
                if (n == tried) continue;
                tried = n;
                if (n > 1 && n * M * p->Cv > kMaxSplitFloats) break;
                const int64_t per_sm = (blocks * n + sms - 1) / sms;
                const int64_t conc = std::min(per_sm, fit), rounds = per_sm / conc, rem = per_sm - rounds * conc;
                auto time = [&](int64_t nb) {
                    const double w = nb * warps, w2 = w * w;
                    return nb == 0 ? 0.0 : std::sqrt(std::sqrt(w2 * w2 + few4)) * key * kps + 200.0 + 60.0 * w;
                };
                const double cost = (rounds * time(conc) + time(rem)) * (1.0 + 0.07 * conc / per_sm) + 9.0 * n +
                                    (n > 1 ? 0.2 * n * M * p->Cv / sms : 0.0);
                if (cost < best * 0.995) {
                    best = cost;
                    p->keys_per_split = kps;
                    p->threads = threads;
                }
            }
        }
        // (Measured, D = 33 to 64: 640 to 810 of these units in a microsecond.)
        p->micros = best / 700.0 + 5.0;
    }
    p->splits = static_cast<int>((N + p->keys_per_split - 1) / p->keys_per_split);
    if (p->splits < 1) p->splits = 1;
    p->off_part = 0;
    p->total = static_cast<size_t>(p->splits) * M * p->Cv * sizeof(float);
    p->total = (p->total + 1023) & ~static_cast<size_t>(1023);
    return true;
}

cudaError_t launch_simt(const SimtPlan& p, bool grad, const float* q, const float* k,
                        const float* v, int Cw, int wch, float half_c, float* part,
                        cudaStream_t s, const Guard& guard) {
    if (grad) {
        switch (p.dmax) {
            case 16: return launch_grad<16>(p, q, k, v, Cw, wch, half_c, part, s);
            case 32: return launch_grad<32>(p, q, k, v, Cw, wch, half_c, part, s);
            default: return launch_grad<64>(p, q, k, v, Cw, wch, half_c, part, s);
        }
    }
    switch (p.dmax) {
        case 4: return launch_dmax<4>(p, q, k, v, half_c, part, s, guard);
        case 8: return launch_dmax<8>(p, q, k, v, half_c, part, s, guard);
        case 16: return launch_dmax<16>(p, q, k, v, half_c, part, s, guard);
        case 24: return launch_dmax<24>(p, q, k, v, half_c, part, s, guard);
        case 32: return launch_dmax<32>(p, q, k, v, half_c, part, s, guard);
        case 48: return launch_dmax<48>(p, q, k, v, half_c, part, s, guard);
        case 56: return launch_dmax<56>(p, q, k, v, half_c, part, s, guard);
        case 64: return launch_dmax<64>(p, q, k, v, half_c, part, s, guard);
        default: return launch_dmax<128>(p, q, k, v, half_c, part, s, guard);
    }
}

}  // namespace gs
