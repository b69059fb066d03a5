// Batched forward and backward of the learned-bias MLP on the tensor cores.
//
// Backward of sum_i g_i b(x_i) for a tile of 128 rows (arXiv:2206.11234 has no
// learned bias; the objective it serves is described with the training step):
//   h1 = tanh(W1 x + b1), z2 = W2 h1 + b2, h2 = tanh(z2), b = w3 . h2 + b3
//   d2 = g w3 (1 - h2^2)          dw3 += g h2,  db3 += g,  db2 += d2
//   dh1 = W2^T d2  (tensor cores)  d1 = dh1 (1 - h1^2)
//   dW2 += d2^T h1 (tensor cores, K = the 128 rows, accumulated in TMEM over tiles)
//   dW1 += d1 x^T, db1 += d1
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "abi_internal.h"
#include "fpt.h"
#include "mlp.cuh"

namespace fpt {
namespace {

constexpr int kFwdTmemCols = 64;
constexpr int kBwdTmemCols = 128;
// Forward CTAs use 64 TMEM columns each: at most 7 can be resident per SM
// (7 x 64 <= 512) because each requests at least this much shared memory.
constexpr size_t kFwdMinSmem = 30 * 1024;

__global__ void __launch_bounds__(128) mlp_forward_kernel(const fpt_mlp_params* __restrict__ P,
                                                          const float* __restrict__ phi,
                                                          const float* __restrict__ N, long long n,
                                                          float* __restrict__ out_b, unsigned* __restrict__ status) {
    extern __shared__ __align__(1024) unsigned char s_raw[];
    MlpTile& S = *reinterpret_cast<MlpTile*>(s_raw);
    if ((threadIdx.x >> 5) == 0) {
        tc::tmem_alloc(&S.tmem, kFwdTmemCols);
        tc::tmem_relinquish();
        tc::fence_before_sync();
    }
    mlp_tile_load(S, P);  // ends with __syncthreads (also publishes S.tmem)
    tc::fence_after_sync();
    uint32_t phase = 0;
    const long long tiles = (n + 127) / 128;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const long long i = t * 128 + threadIdx.x;
        const float p = i < n ? phi[i] : 0.f;
        const float x = i < n ? N[i] : 0.f;
        const float b = mlp_tile_forward(S, p, x, phase);
        if (i < n) out_b[i] = b;
        __syncthreads();
    }
    __syncthreads();
    if (threadIdx.x == 0 && S.status) atomicOr(status, S.status);
    if ((threadIdx.x >> 5) == 0) {
        if (S.status) tc::mbar_wait(&S.mbar, phase ^ 1u);  // a commit left pending by an expired wait
        tc::tmem_dealloc(S.tmem, kFwdTmemCols);
    }
}

// Column sums.  Every parameter gradient but dW2 is a sum over rows of quantities
// that one thread has for its row.  The rows go to shared memory (h2 in BF16, as the
// network computes it, delta1 in FP32) and are read back by columns: thread t adds
// up four columns (4 (t mod 16) ..) of eight rows (8 (t / 16) ..) in registers
// that live as long as the CTA, and the sixteen row groups meet once, at the end.
constexpr int kH2Row = 144;  // bytes of a row of h2: 64 bf16 and padding against bank conflicts
constexpr int kD1Row = 272;  // bytes of a row of delta1: 64 floats and padding

struct MlpBwdSmem {
    MlpTile f;                                 // A = h1 (rows r, columns k), W2 (rows n, columns k)
    // delta2 (rows r, columns n) as an operand, then h2; once both have been read,
    // delta1 takes the place of the two
    alignas(128) unsigned char D2[kTileBytes64];
    unsigned char H2[128 * kH2Row];
    float x[128][2];                           // normalised inputs of the rows
    float g[128];
    float gw1[kHid][2];
    float gb1[kHid];
    float gb2[kHid];
    float gw3[kHid];
    float gb3;
};
static_assert(kTileBytes64 + 128 * kH2Row >= 128 * kD1Row, "delta1 fits over delta2 and h2");

// 1 - h^2 of two BF16 values
__device__ __forceinline__ tc::f32x2 one_minus_square(uint32_t h) {
    const float lo = tc::bf16_lo(h), hi = tc::bf16_hi(h);
    return tc::fma2(tc::pair(-lo, -hi), tc::pair(lo, hi), tc::pair(1.f, 1.f));
}

constexpr uint32_t kIdescDh1 = tc::idesc_bf16_tn(128, 64, false, true);  // delta2 W2: W2's rows are K
constexpr uint32_t kIdescDW2 = tc::idesc_bf16_tn(128, 64, true, true);   // delta2^T h1: the tile's rows are K

// What bounds it: shared-memory accesses (61 % of their rate, ncu) and their
// latencies around three small products; the tensor pipe idles.  The products read
// the same tiles in both orders (K-major and MN-major descriptors) instead of
// transposed copies; that and the column sums replaced 128 two-byte shared accesses
// and 320 shuffles per row and tile, and 56 KB of copies, so that three CTAs fit
// where two did.  1,000,003 rows: 280 us with them, 150 us without, 139 us with two
// threads per row (24 warps per SM instead of 12).
//
// CTAs.  Each ends with 4489 additions to the one gradient, some 0.1 us that the CTAs
// take in turn: fewer of them are the faster until an SM has enough tiles for two or
// three (calls in us with 1, 2 and 3 per SM: 20,000 rows 58 61 60, 58,368 60 85 101,
// 100,000 64 75 98, 300,000 97 98 111, 600,000 135 123 133, 1,000,000 195 160 161,
// 4,000,000 615 447 408).
constexpr int kBwdThreads = 256;  // two threads per row, 32 of the 64 units each

__global__ void __launch_bounds__(kBwdThreads, 3) mlp_backward_kernel(const fpt_mlp_params* __restrict__ P,
                                                           const float* __restrict__ phi,
                                                           const float* __restrict__ N,
                                                           const float* __restrict__ g, long long n,
                                                           float* __restrict__ grad,
                                                           unsigned* __restrict__ status) {
    extern __shared__ __align__(1024) unsigned char s_raw[];
    MlpBwdSmem& B = *reinterpret_cast<MlpBwdSmem*>(s_raw);
    MlpTile& S = B.f;
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    if (warp == 0) {
        tc::tmem_alloc(&S.tmem, kBwdTmemCols);
        tc::tmem_relinquish();
        tc::fence_before_sync();
    }
    for (int j = tid; j < kHid; j += blockDim.x) {
        B.gw1[j][0] = B.gw1[j][1] = 0.f;
        B.gb1[j] = B.gb2[j] = B.gw3[j] = 0.f;
    }
    if (tid == 0) B.gb3 = 0.f;
    mlp_tile_load(S, P);  // fences the generic writes above and synchronises
    tc::fence_after_sync();
    uint32_t phase = 0;
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    const long long tiles = (n + 127) / 128;
    const int row = tid & 127, half = tid >> 7;           // this thread's row and units 32 half ..
    const int c0 = 4 * (tid & 15), r0 = 8 * (tid >> 4);  // columns and rows of its sums
    // two columns each; 0 is two binary32 zeros
    tc::f32x2 a_w3[2] = {0, 0}, a_b2[2] = {0, 0}, a_b1[2] = {0, 0}, a_x0[2] = {0, 0}, a_x1[2] = {0, 0};
    float a_g = 0.f;
    int done = 0;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x, ++done) {
        const long long i = t * 128 + row;
        const bool valid = i < n;
        const float gi = valid ? g[i] : 0.f;
        const float x0 = ((valid ? phi[i] : 0.f) - S.norm[0]) * S.norm[1];
        const float x1 = ((valid ? N[i] : 0.f) - S.norm[2]) * S.norm[3];
        if (half == 0) {
            B.x[row][0] = x0;
            B.x[row][1] = x1;
            B.g[row] = gi;
            a_g += gi;
        }
        mlp_layer1_to_tile<4, 4>(S, S.A, row, x0, x1, 4 * half);
        tc::fence_proxy_async();
        __syncthreads();
        if (tid == 0) mlp_issue_z2(S);
        if (S.status != 0u || !tc::mbar_wait(&S.mbar, phase)) S.status = 1u;  // one expiry, not one per tile
        phase ^= 1u;
        tc::fence_after_sync();
        // h2 and delta2 = g w3 (1 - h2^2) of the row
        const tc::f32x2 gg = tc::pair(gi, gi);
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
            const int c = 2 * half + cc;
            float z[16];
            tc::tmem_ld16(S.tmem + lane_base + 16 * c, z);
            tc::tmem_wait_ld();
            uint32_t q[8], hh[8];
#pragma unroll
            for (int e = 0; e < 16; e += 4) {
                const int n0 = 16 * c + e;
                tc::f32x2 bb[2], w[2];
                tc::load_pairs(S.b2 + n0, bb[0], bb[1]);
                tc::load_pairs(S.w3 + n0, w[0], w[1]);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const uint32_t h = tc::tanh_bf16x2(
                        tc::pack_bf16(tc::add2(tc::pair(z[e + 2 * k], z[e + 2 * k + 1]), bb[k])));
                    hh[e / 2 + k] = h;
                    q[e / 2 + k] = tc::pack_bf16(tc::mul2(tc::mul2(gg, w[k]), one_minus_square(h)));
                }
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                *reinterpret_cast<uint4*>(B.D2 + tc::kmajor_offset(row, 16 * c + 8 * u, 64)) =
                    make_uint4(q[4 * u], q[4 * u + 1], q[4 * u + 2], q[4 * u + 3]);
                *reinterpret_cast<uint4*>(B.H2 + row * kH2Row + 32 * c + 16 * u) =
                    make_uint4(hh[4 * u], hh[4 * u + 1], hh[4 * u + 2], hh[4 * u + 3]);
            }
        }
        tc::fence_before_sync();
        tc::fence_proxy_async();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after_sync();
            const uint32_t d2 = tc::smem_u32(B.D2), w2 = tc::smem_u32(S.W2), h1 = tc::smem_u32(S.A);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)  // dh1 = delta2 W2 -> columns 0..63, 16 of the n at a time
                tc::mma_bf16(S.tmem, tc::smem_desc(d2 + 256 * kk, 128, 1024),
                             tc::smem_desc(w2 + 2048 * kk, 1024, 128), kIdescDh1, kk > 0 ? 1u : 0u);
            // dW2 += delta2^T h1 -> columns 64..127, 16 rows at a time (of the 128
            // result rows the first 64 are n; the others hold no result)
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
                tc::mma_bf16(S.tmem + 64, tc::smem_desc(d2 + 2048 * kk, 1024, 128),
                             tc::smem_desc(h1 + 2048 * kk, 1024, 128), kIdescDW2, (done > 0 || kk > 0) ? 1u : 0u);
            tc::mma_commit(&S.mbar);
        }
        // meanwhile dw3 = sum g h2 and db2 = w3 sum g (1 - h2^2) (w3 at the end)
#pragma unroll 4
        for (int r = r0; r < r0 + 8; ++r) {
            const uint2 h = *reinterpret_cast<const uint2*>(B.H2 + r * kH2Row + 2 * c0);
            const tc::f32x2 gr = tc::pair(B.g[r], B.g[r]);
            const uint32_t hw[2] = {h.x, h.y};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                a_w3[u] = tc::fma2(gr, tc::pair(tc::bf16_lo(hw[u]), tc::bf16_hi(hw[u])), a_w3[u]);
                a_b2[u] = tc::fma2(gr, one_minus_square(hw[u]), a_b2[u]);
            }
        }
        if (S.status != 0u || !tc::mbar_wait(&S.mbar, phase)) S.status = 1u;  // one expiry, not one per tile
        phase ^= 1u;
        tc::fence_after_sync();
        __syncthreads();  // h2 has been read: delta1 may take its place
        // delta1 = dh1 (1 - h1^2) of the row
        unsigned char* d1 = B.D2;
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
            const int c = 2 * half + cc;
            float dh[16];
            tc::tmem_ld16(S.tmem + lane_base + 16 * c, dh);
            tc::tmem_wait_ld();
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const uint4 hq = *reinterpret_cast<const uint4*>(S.A + tc::kmajor_offset(row, 16 * c + 8 * u, 64));
                const uint32_t hw[4] = {hq.x, hq.y, hq.z, hq.w};
                ulonglong2* o = reinterpret_cast<ulonglong2*>(d1 + row * kD1Row + 64 * c + 32 * u);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int k = 8 * u + 4 * e;
                    o[e] = make_ulonglong2(
                        tc::mul2(tc::pair(dh[k], dh[k + 1]), one_minus_square(hw[2 * e])),
                        tc::mul2(tc::pair(dh[k + 2], dh[k + 3]), one_minus_square(hw[2 * e + 1])));
                }
            }
        }
        tc::fence_before_sync();
        __syncthreads();
        // db1 = sum delta1, dW1 = sum delta1 x^T
#pragma unroll 4
        for (int r = r0; r < r0 + 8; ++r) {
            const ulonglong2 d = *reinterpret_cast<const ulonglong2*>(d1 + r * kD1Row + 4 * c0);
            const float2 xr = *reinterpret_cast<const float2*>(B.x[r]);
            const tc::f32x2 dv[2] = {d.x, d.y}, xx0 = tc::pair(xr.x, xr.x), xx1 = tc::pair(xr.y, xr.y);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                a_b1[u] = tc::add2(a_b1[u], dv[u]);
                a_x0[u] = tc::fma2(dv[u], xx0, a_x0[u]);
                a_x1[u] = tc::fma2(dv[u], xx1, a_x1[u]);
            }
        }
        __syncthreads();  // delta1, the inputs and h1 have been read
    }
    tc::fence_after_sync();
    // dW2 from TMEM rows 0..63 (warps 0 and 1), the other sums through shared memory
    if (done > 0 && warp < 2) {
        const int nn = 32 * warp + lane;
        for (int c = 0; c < 4; ++c) {
            float v[16];
            tc::tmem_ld16(S.tmem + lane_base + 64 + 16 * c, v);
            tc::tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; ++e) atomicAdd(&grad[kW2 + nn * kHid + 16 * c + e], v[e]);
        }
    }
    if (done > 0) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int k = c0 + 2 * u;
            float lo, hi;
            tc::split(a_w3[u], lo, hi);
            atomicAdd(&B.gw3[k], lo);
            atomicAdd(&B.gw3[k + 1], hi);
            tc::split(a_b2[u], lo, hi);
            atomicAdd(&B.gb2[k], S.w3[k] * lo);
            atomicAdd(&B.gb2[k + 1], S.w3[k + 1] * hi);
            tc::split(a_b1[u], lo, hi);
            atomicAdd(&B.gb1[k], lo);
            atomicAdd(&B.gb1[k + 1], hi);
            tc::split(a_x0[u], lo, hi);
            atomicAdd(&B.gw1[k][0], lo);
            atomicAdd(&B.gw1[k + 1][0], hi);
            tc::split(a_x1[u], lo, hi);
            atomicAdd(&B.gw1[k][1], lo);
            atomicAdd(&B.gw1[k + 1][1], hi);
        }
        atomicAdd(&B.gb3, a_g);
        __syncthreads();
        for (int j = tid; j < kHid; j += blockDim.x) {
            atomicAdd(&grad[kW1 + 2 * j], B.gw1[j][0]);
            atomicAdd(&grad[kW1 + 2 * j + 1], B.gw1[j][1]);
            atomicAdd(&grad[kB1 + j], B.gb1[j]);
            atomicAdd(&grad[kB2 + j], B.gb2[j]);
            atomicAdd(&grad[kW3 + j], B.gw3[j]);
        }
        if (tid == 0) atomicAdd(&grad[kB3], B.gb3);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0 && S.status) atomicOr(status, S.status);
    if (warp == 0) {
        if (S.status) tc::mbar_wait(&S.mbar, phase ^ 1u);  // a commit left pending by an expired wait
        tc::tmem_dealloc(S.tmem, kBwdTmemCols);
    }
}

constexpr int kMaxCtas = 32;  // per SM: no limit but the kernel's own

// Grid for a persistent MLP kernel and a check that its resident CTAs cannot
// ask for more TMEM columns than an SM has (an allocation would then wait for
// a CTA that never exits).
int mlp_grid(const void* func, int threads, size_t smem, int tmem_cols, long long tiles, int max_per_sm, int* grid) {
    int n_sm = 0;
    int rc = device_sm_count(&n_sm);
    if (rc) return rc;
    cudaError_t e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "MLP kernel shared memory");
    int per_sm = 0;
    rc = resident_ctas(func, threads, smem, tmem_cols, &per_sm);
    if (rc) return rc;
    if (per_sm < 1) return fail(FPT_EUNSUPPORTED, "MLP kernel does not fit on an SM");
    const long long full = (long long)std::min(per_sm, max_per_sm) * n_sm;
    *grid = (int)(tiles < full ? (tiles < 1 ? 1 : tiles) : full);
    return FPT_OK;
}

int run_status(unsigned* d_status, cudaStream_t st) {
    unsigned h = 0;
    cudaError_t e = cudaMemcpyAsync(&h, d_status, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaError_t ef = cudaFreeAsync(d_status, st);
    if (e != cudaSuccess) return cuda_fail(e, "MLP status readback");
    if (ef != cudaSuccess) return cuda_fail(ef, "MLP status free");
    if (h) return fail(FPT_EDEVICE_STATUS, "MLP kernel: a tensor-core wait expired (status 0x%x)", h);
    return FPT_OK;
}

}  // namespace

size_t mlp_fwd_smem_bytes() {
    return sizeof(MlpTile) > kFwdMinSmem ? sizeof(MlpTile) : kFwdMinSmem;
}

}  // namespace fpt

using namespace fpt;

namespace fpt {
namespace {
// One warp waits, with the library's bounded wait, on an mbarrier that nobody
// arrives at; it records the expiry and then completes the phase itself, so the
// barrier ends in a clean state.
__global__ void wait_selftest_kernel(unsigned* __restrict__ expired) {
    __shared__ __align__(8) uint64_t mbar;
    if (threadIdx.x == 0) tc::mbar_init(&mbar, 1);
    __syncthreads();
    const bool ok = tc::mbar_wait(&mbar, 0u);
    if (!ok) atomicOr(expired, 1u);
    __syncwarp();
    if (threadIdx.x == 0) tc::mbar_arrive(&mbar);
}
}  // namespace
}  // namespace fpt

extern "C" int fpt_wait_selftest(int32_t* expired_out, double* seconds_out, void* stream) {
    if (!expired_out) return fail(FPT_EINVAL, "expired_out is NULL");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    unsigned* d = nullptr;
    cudaError_t e = lib_malloc_retained_async(reinterpret_cast<void**>(&d), sizeof(unsigned), st);
    if (e != cudaSuccess) return cuda_fail(e, "self-test flag");
    cudaMemsetAsync(d, 0, sizeof(unsigned), st);
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    cudaEventRecord(a, st);
    wait_selftest_kernel<<<1, 32, 0, st>>>(d);
    e = cudaGetLastError();
    cudaEventRecord(b, st);
    unsigned h = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    cudaFreeAsync(d, st);
    if (e != cudaSuccess) return cuda_fail(e, "wait self-test");
    *expired_out = (int32_t)h;
    if (seconds_out) *seconds_out = ms / 1e3;
    return FPT_OK;
}

extern "C" int fpt_mlp_forward(const fpt_mlp_params* w, const float* phi, const float* N, int64_t n, float* out_b,
                               void* stream) {
    NvtxRange nvtx_range("fpt_mlp_forward");
    if (n < 0) return fail(FPT_EINVAL, "n %lld < 0", (long long)n);
    if (!w || (n > 0 && (!phi || !N || !out_b))) return fail(FPT_EINVAL, "pointer is NULL");
    if ((reinterpret_cast<uintptr_t>(w) & 15u) != 0) return fail(FPT_EINVAL, "parameters must be 16-byte aligned");
    if (n == 0) return FPT_OK;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const size_t smem = mlp_fwd_smem_bytes();
    int grid = 0;
    int rc = mlp_grid((const void*)mlp_forward_kernel, 128, smem, kFwdTmemCols, (n + 127) / 128, kMaxCtas, &grid);
    if (rc) return rc;
    unsigned* d_status = nullptr;
    cudaError_t e = lib_malloc_retained_async(reinterpret_cast<void**>(&d_status), sizeof(unsigned), st);
    if (e != cudaSuccess) return cuda_fail(e, "MLP status");
    cudaMemsetAsync(d_status, 0, sizeof(unsigned), st);
    mlp_forward_kernel<<<grid, 128, smem, st>>>(w, phi, N, (long long)n, out_b, d_status);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        cudaFreeAsync(d_status, st);
        return cuda_fail(e, "MLP forward launch");
    }
    return run_status(d_status, st);
}

extern "C" int fpt_mlp_backward(const fpt_mlp_params* w, const float* phi, const float* N, const float* g,
                                int64_t n, float* grad, void* stream) {
    NvtxRange nvtx_range("fpt_mlp_backward");
    if (n < 0) return fail(FPT_EINVAL, "n %lld < 0", (long long)n);
    if (!w || !grad || (n > 0 && (!phi || !N || !g))) return fail(FPT_EINVAL, "pointer is NULL");
    if ((reinterpret_cast<uintptr_t>(w) & 15u) != 0) return fail(FPT_EINVAL, "parameters must be 16-byte aligned");
    if (n == 0) return FPT_OK;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const size_t smem = sizeof(MlpBwdSmem);
    int grid = 0;
    const long long tiles = (n + 127) / 128;
    int n_sm = 0;
    int rc = device_sm_count(&n_sm);
    if (rc) return rc;
    rc = mlp_grid((const void*)mlp_backward_kernel, kBwdThreads, smem, kBwdTmemCols, tiles,
                  tiles < 20LL * n_sm ? 1 : tiles < 50LL * n_sm ? 2 : kMaxCtas, &grid);
    if (rc) return rc;
    unsigned* d_status = nullptr;
    cudaError_t e = lib_malloc_retained_async(reinterpret_cast<void**>(&d_status), sizeof(unsigned), st);
    if (e != cudaSuccess) return cuda_fail(e, "MLP status");
    cudaMemsetAsync(d_status, 0, sizeof(unsigned), st);
    mlp_backward_kernel<<<grid, kBwdThreads, smem, st>>>(w, phi, N, g, (long long)n, grad, d_status);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        cudaFreeAsync(d_status, st);
        return cuda_fail(e, "MLP backward launch");
    }
    return run_status(d_status, st);
}
