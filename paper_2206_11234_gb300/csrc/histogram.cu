// Weighted histogram of first-passage times (arXiv:2206.11234 §2.1 Eq. (9),
// §2.2 Eq. (16)), several histograms (one per parameter set) per launch.
//
// Per bin: n_j, max ln w and, with x = ln w - max <= 0, s1 = sum exp(x),
// s2 = sum exp(2 x), l_k = sum x^k for k = 1..4 (the moments of ln w behind the
// lognormal estimator and normality test of §2.4).  Two streaming passes over the
// records.  What bounds them is GB300's binary64 pipe, one warp instruction per SM
// every 16 cycles whatever its active lanes, so both are written to spend few:
//   pass 1: classify each record (16 B read) with one multiply-add, store its bin
//           (2 B), keep the per-bin maximum of ln w as an order-preserving 64-bit
//           key in shared memory (one global atomic per bin and block);
//   pass 2: each block sorts a tile of ln w by bin in shared memory (counting sort,
//           integers only), so that a thread adds up consecutive records of one
//           bin in registers: 8 binary64 instructions per record, and sums leave
//           for global memory once per bin change.
// Bins are right-closed: j = ceil((N - lo)/d) - 1, clamped to [0, n_bins).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

#include "exp_table.inc"  // kExp62[4096] = 2^(62 - j/4096), kExpStep2..0 = ln 2 / 4096 x 2^98, kExpPerStep = 4096 / ln 2 x 2^19
#include "histogram.h"

namespace fpt {
namespace {

__device__ __forceinline__ unsigned long long ord_key(double x) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double ord_value(unsigned long long k) {
    const unsigned long long u = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)u);
}

constexpr unsigned long long kKeyNegInf = 0x000fffffffffffffull;  // ord_key(-inf)
constexpr int kSums = 6;                                          // s1, s2, l1 .. l4 per bin
constexpr unsigned kNoBin = 0xffffu;

// Signed integers in the order of the numbers: NaN above +inf or below -inf by its sign.
__host__ __device__ __forceinline__ long long signed_key(long long u) {
    return u ^ (long long)((unsigned long long)(u >> 63) >> 1);
}
constexpr long long kSignedPosInf = 0x7ff0000000000000ll;
constexpr long long kSignedNegInf = (long long)0x800fffffffffffffull;

// Fixed point of the bin coordinate: N / d - lo / d + kFix has an ulp of 2^-36.
constexpr double kFix = 98304.0;  // 1.5 x 2^16
// Largest |edge| / d for which the multiply-add is within 3 ulp of (N - lo) / d:
// 2^-37 each from its own rounding and fix's (twice that where lo / d = -2^15), 2^-38
// each from 1/d in both products, 2^-39 from the second's rounding.
constexpr double kFastCoord = 32768.0;

// Bin of N within its histogram; the comparisons are on integers and the
// quotient is one multiply-add in fixed point.  Only where that lies within 4 ulp
// of an edge does the division decide, as written.
__device__ __forceinline__ int bin_of(double N, const HistSeg& h, unsigned* status) {
    const double t = __fma_rn(N, h.inv_d, h.fix);
    const unsigned hi = (unsigned)__double2hiint(t), lo4 = (unsigned)__double2loint(t) + 4u;
    int j = (int)((hi >> 4) & 0x7fffu);
    if (((hi + (lo4 < 4u ? 1u : 0u)) & 15u) == 0u && lo4 < 8u) {
        const long long e = (long long)ceil((N - h.lo) / h.d) - 1;
#if FPT_DEBUG
        // rounding at the edges gives -1 or n_bins, which the clamp absorbs; more is a broken segment
        if ((e < -1 || e > h.n_bins) && status) atomicOr(status, kStatusHistBin);
#endif
        j = e < 0 ? 0 : (int)(e < (long long)h.n_bins ? e : (long long)h.n_bins - 1);
    }
#if FPT_DEBUG
    if (j >= h.n_bins && status) atomicOr(status, kStatusHistBin);
#else
    (void)status;
#endif
    return j < h.n_bins ? j : h.n_bins - 1;
}

__global__ void hist_init(const HistSeg* __restrict__ segs, int n_segs, fpt_bin* __restrict__ bins,
                          fpt_hist_counts* __restrict__ counts) {
    const HistSeg h = segs[blockIdx.y];
    const int nb = h.n_bins * h.n_sub;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) {
        fpt_bin* o = bins + h.bin0 + b;
        o->max_lw = __longlong_as_double((long long)kKeyNegInf);  // holds the key until hist_final
        o->s1 = 0.0;
        o->s2 = 0.0;
        o->l1 = 0.0;
        o->l2 = 0.0;
        o->l3 = 0.0;
        o->l4 = 0.0;
        o->count = 0;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        counts[blockIdx.y].under = 0;
        counts[blockIdx.y].over = 0;
        counts[blockIdx.y].censored = 0;
        counts[blockIdx.y].total = h.n;
    }
}

constexpr int kMaxThreads = 512;  // pass 1
constexpr int kMaxUnroll = 4;     // records of a thread in flight

__global__ void __launch_bounds__(kMaxThreads) hist_pass_max(const double* __restrict__ N,
                                                             const double* __restrict__ lw,
                                                             const HistSeg* __restrict__ segs,
                                                             fpt_bin* __restrict__ bins,
                                                             fpt_hist_counts* __restrict__ counts, unsigned* status,
                                                             uint16_t* __restrict__ bin_idx) {
    extern __shared__ unsigned long long s_key[];
    const HistSeg h = segs[blockIdx.y];
    const int nb = h.n_bins * h.n_sub;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) s_key[b] = kKeyNegInf;
    __syncthreads();
    unsigned under = 0, over = 0, cens = 0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    // jackknife subset of the thread's next record: ids advance by the stride
    unsigned sub = 0, sub_step = 0;
    if (h.n_sub > 1) {
        sub = (unsigned)((h.id_offset + (unsigned long long)first) % (unsigned long long)h.n_sub);
        sub_step = (unsigned)(stride % h.n_sub);
    }
    for (long long i = first; i < h.n; i += kMaxUnroll * stride) {
        double x[kMaxUnroll], y[kMaxUnroll];
#pragma unroll
        for (int k = 0; k < kMaxUnroll; ++k)
            if (i + k * stride < h.n) {
                x[k] = N[h.first + i + k * stride];
                y[k] = lw[h.first + i + k * stride];
            }
#pragma unroll
        for (int k = 0; k < kMaxUnroll; ++k) {
            if (i + k * stride >= h.n) break;
            const long long s = signed_key(__double_as_longlong(x[k]));
            unsigned bin = kNoBin;
            if (s > h.key_hi) {
                if (s < kSignedPosInf) ++over; else ++cens;
            } else if (s <= h.key_lo) {
                if (s >= kSignedNegInf) ++under; else ++cens;
            } else {
                bin = sub * (unsigned)h.n_bins + (unsigned)bin_of(x[k], h, status);
                const unsigned long long key = ord_key(y[k]);
                // rarely larger than what is there already
                if (key > *reinterpret_cast<volatile unsigned long long*>(&s_key[bin])) atomicMax(&s_key[bin], key);
            }
            bin_idx[h.first + i + k * stride] = (uint16_t)bin;
            sub += sub_step;
            if (sub >= (unsigned)h.n_sub) sub -= (unsigned)h.n_sub;
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
        if (s_key[b] != kKeyNegInf)
            atomicMax(reinterpret_cast<unsigned long long*>(&bins[h.bin0 + b].max_lw), s_key[b]);
    under = __reduce_add_sync(0xffffffffu, under);
    over = __reduce_add_sync(0xffffffffu, over);
    cens = __reduce_add_sync(0xffffffffu, cens);
    if ((threadIdx.x & 31u) == 0u) {
        if (under) atomicAdd(reinterpret_cast<unsigned long long*>(&counts[blockIdx.y].under), (unsigned long long)under);
        if (over) atomicAdd(reinterpret_cast<unsigned long long*>(&counts[blockIdx.y].over), (unsigned long long)over);
        if (cens) atomicAdd(reinterpret_cast<unsigned long long*>(&counts[blockIdx.y].censored), (unsigned long long)cens);
    }
}

// exp(x) for x <= 0 in integers (table-driven exponential, Tang, ACM TOMS 15 (1989)):
// |x| = k ln 2 / 4096 + r in fixed point, the table's 2^(-k/4096) times the series of
// exp(-r) to r^3, |r| <= 8.5e-5; within 0.77 units in the last place.  Some 50
// integer instructions take about as long as one of the 8 binary64 instructions that
// they replace (64 cycles each of a sub-partition): pass 2 of 2^24 records
// 582 -> 364 us, its binary64 pipe 80 -> 65 % busy, the rest sorting.  From 512 on,
// infinities and NaN: the library's.
__device__ __forceinline__ double exp_neg(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x) & 0x7fffffffu;
    if (hi >= 0x40800000u) return exp(x);
    const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | (uint32_t)__double2loint(x)) << 11;
    const uint64_t z = m >> min(1031 - (int)(hi >> 20), 63);  // |x| 2^55; 0 becomes one unit, too little to matter
    const uint32_t k = (uint32_t)(((z >> 32) * kExpPerStep + (1ull << 41)) >> 42);
    const uint64_t kstep = (uint64_t)k * kExpStep1 + __umulhi(k, kExpStep0) + ((uint64_t)(k * kExpStep2) << 32);
    const int64_t r = (int64_t)((z << 11) - kstep);                   // 2^-66, exact but for the constant, |r| < 2^53
    const int32_t rs = (int32_t)(r >> 22);                            // 2^-44
    const uint32_t r2 = (uint32_t)__mulhi(rs, rs);                    // 2^-56
    const uint32_t w = 0x80000000u - (uint32_t)__mulhi(rs, 174763);   // 1/2 - r/6, 2^-32 (174763 = 2^20 / 6)
    const int64_t p = r - (int64_t)(((uint64_t)r2 * w) >> 22);        // 1 - exp(-r), 2^-66
    const uint64_t T = __ldg(&kExp62[k & 4095u]);
    const int32_t Th = (int32_t)(T >> 32), ph = (int32_t)(p >> 32);
    const int64_t Tp = (int64_t)Th * ph + __umulhi((uint32_t)Th, (uint32_t)p) +
                       2 * __mulhi((int32_t)((uint32_t)T >> 1), ph);  // 2^-64
    uint64_t e = T - (uint64_t)(Tp >> 2);                             // 2^-62, in (1/2, 1 + 1e-4)
    const uint32_t over = (uint32_t)(e >> 62);
    e = (e >> over) + 256u;
    return __longlong_as_double((long long)(((uint64_t)(1021u + over - (k >> 12)) << 52) + (e >> 9)));
}

constexpr int kSumThreads = 256;  // pass 2

// Shared memory of pass 2: R records per thread sorted by bin (one padding element
// per thread, so that threads reading their own runs do not collide), and a counter
// per bin.
template <int R>
constexpr size_t sum_smem_bytes(int max_nb) {
    return (size_t)kSumThreads * (R + 1) * (sizeof(double) + sizeof(uint16_t)) + (size_t)((max_nb + 3) & ~3) * sizeof(int);
}

__device__ __forceinline__ void add_sums(fpt_bin* o, const double v[kSums]) {
    atomicAdd(&o->s1, v[0]);
    atomicAdd(&o->s2, v[1]);
    atomicAdd(&o->l1, v[2]);
    atomicAdd(&o->l2, v[3]);
    atomicAdd(&o->l3, v[4]);
    atomicAdd(&o->l4, v[5]);
}

template <int R>
__global__ void __launch_bounds__(kSumThreads) hist_pass_sum(const double* __restrict__ lw,
                                                             const HistSeg* __restrict__ segs,
                                                             fpt_bin* __restrict__ bins,
                                                             const uint16_t* __restrict__ bin_idx) {
    constexpr int kTile = kSumThreads * R;
    extern __shared__ __align__(16) double s_x[];
    uint16_t* s_bin = reinterpret_cast<uint16_t*>(s_x + kSumThreads * (R + 1));
    int* s_at = reinterpret_cast<int*>(s_bin + kSumThreads * (R + 1));  // count, then first place of a bin
    __shared__ int s_warp[kSumThreads / 32];
    const HistSeg h = segs[blockIdx.y];
    const int nb = h.n_bins * h.n_sub;
    const unsigned FULL = 0xffffffffu;
    const unsigned tid = threadIdx.x, lane = tid & 31u;
    fpt_bin* out = bins + h.bin0;
    for (long long base = (long long)blockIdx.x * kTile; base < h.n; base += (long long)gridDim.x * kTile) {
        for (int b = tid; b < ((nb + 3) & ~3); b += kSumThreads) s_at[b] = 0;
        __syncthreads();
        // count the tile's records per bin; a record's rank among its bin's packed with the bin
        double x[R];
        unsigned at[R];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const long long i = base + k * kSumThreads + tid;
            at[k] = kNoBin;
            if (i < h.n) {
                at[k] = bin_idx[h.first + i];
                x[k] = lw[h.first + i];
            }
        }
#pragma unroll
        for (int k = 0; k < R; ++k)
            if (at[k] != kNoBin) at[k] |= (unsigned)atomicAdd(&s_at[at[k]], 1) << 16;
        __syncthreads();
        // first places (exclusive sums of the counts); the counts go to the output here
        int carry = 0;
        for (int b0 = 0; b0 < nb; b0 += 4 * kSumThreads) {
            const int b = b0 + 4 * (int)tid;  // four bins a thread: 4096 bins in four rounds of barriers
            const int4 c = b < nb ? *reinterpret_cast<const int4*>(s_at + b) : make_int4(0, 0, 0, 0);
            const int sum = c.x + c.y + c.z + c.w;
            int v = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(FULL, v, o);
                if ((int)lane >= o) v += u;
            }
            if (lane == 31u) s_warp[tid >> 5] = v;
            __syncthreads();
            int before = carry;
#pragma unroll
            for (int w = 0; w < kSumThreads / 32; ++w) {
                if (w < (int)(tid >> 5)) before += s_warp[w];
                carry += s_warp[w];
            }
            if (b < nb) {
                const int at0 = before + v - sum;
                const int cs[4] = {c.x, c.y, c.z, c.w};
                *reinterpret_cast<int4*>(s_at + b) = make_int4(at0, at0 + c.x, at0 + c.x + c.y, at0 + c.x + c.y + c.z);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (cs[k]) atomicAdd(reinterpret_cast<unsigned long long*>(&out[b + k].count), (unsigned long long)cs[k]);
            }
            __syncthreads();
        }
        const int total = carry;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const unsigned b = at[k] & 0xffffu;
            if (b != kNoBin) {
                const int p = s_at[b] + (int)(at[k] >> 16);
                s_x[p + p / R] = x[k];
                s_bin[p + p / R] = (uint16_t)b;
            }
        }
        __syncthreads();
        // every thread's R consecutive places: one bin after the other
        double v[kSums] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        unsigned cur = kNoBin;
        double mx = 0.0;
        const int mine = min(R, total - (int)tid * R);
        for (int k = 0; k < mine; ++k) {
            const unsigned b = s_bin[tid * (R + 1) + k];
            if (b != cur) {
                if (cur != kNoBin) add_sums(&out[cur], v);
#pragma unroll
                for (int f = 0; f < kSums; ++f) v[f] = 0.0;
                cur = b;
                mx = ord_value((unsigned long long)__double_as_longlong(out[b].max_lw));
            }
            const double y = __dsub_rn(s_x[tid * (R + 1) + k], mx);
            const double e = exp_neg(y), y2 = __dmul_rn(y, y);
            v[0] = __dadd_rn(v[0], e);
            v[1] = __fma_rn(e, e, v[1]);
            v[2] = __dadd_rn(v[2], y);
            v[3] = __dadd_rn(v[3], y2);
            v[4] = __fma_rn(y2, y, v[4]);
            v[5] = __fma_rn(y2, y2, v[5]);
        }
        // the last bins of a warp's threads: lanes of one bin are neighbours; add
        // up each group towards its highest lane, which writes it
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned cb = __shfl_up_sync(FULL, cur, o);
            const bool same = (int)lane >= o && cb == cur && cur != kNoBin;
            if (!__any_sync(FULL, same)) break;
#pragma unroll
            for (int f = 0; f < kSums; ++f) {
                const double u = __shfl_up_sync(FULL, v[f], o);
                if (same) v[f] = __dadd_rn(v[f], u);
            }
        }
        const unsigned next = __shfl_down_sync(FULL, cur, 1);
        if (cur != kNoBin && (lane == 31u || next != cur)) add_sums(&out[cur], v);
        __syncthreads();
    }
}

__global__ void hist_final(const HistSeg* __restrict__ segs, fpt_bin* __restrict__ bins) {
    const HistSeg h = segs[blockIdx.y];
    const int nb = h.n_bins * h.n_sub;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) {
        fpt_bin* o = bins + h.bin0 + b;
        o->max_lw = ord_value((unsigned long long)__double_as_longlong(o->max_lw));
    }
}

template <int R>
cudaError_t launch_sum(const HistSeg* d_segs, int n_segs, int max_nb, long long max_n, const double* lw, fpt_bin* bins,
                       int n_sm, cudaStream_t stream, const uint16_t* bin_idx) {
    cudaError_t e = cudaFuncSetAttribute(hist_pass_sum<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sum_smem_bytes<R>(FPT_MAX_HIST_BINS));
    if (e != cudaSuccess) return e;
    const size_t smem = sum_smem_bytes<R>(max_nb);
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hist_pass_sum<R>, kSumThreads, smem);
    if (e != cudaSuccess) return e;
    const long long tiles = std::max(1LL, (max_n + kSumThreads * R - 1) / (kSumThreads * R));
    const long long cap = std::max(1LL, ((long long)std::max(per_sm, 1) * n_sm + n_segs - 1) / n_segs);
    hist_pass_sum<R><<<dim3((unsigned)std::min(tiles, cap), n_segs), kSumThreads, smem, stream>>>(lw, d_segs, bins,
                                                                                                 bin_idx);
    return cudaGetLastError();
}

long long host_key(double x) {
    x += 0.0;  // -0 compares like +0
    long long u;
    std::memcpy(&u, &x, sizeof(u));
    return signed_key(u);
}

}  // namespace

HistSeg hist_seg(long long first, long long n, unsigned long long id_offset, double lo, double hi, int n_bins,
                 int n_sub, long long bin0) {
    HistSeg h;
    h.first = first;
    h.n = n;
    h.id_offset = id_offset;
    h.lo = lo;
    h.hi = hi;
    h.d = (hi - lo) / (double)n_bins;
    h.n_bins = n_bins;
    h.n_sub = n_sub;
    h.bin0 = bin0;
    h.key_lo = host_key(lo);
    h.key_hi = host_key(hi);
    // outside the fixed point's range every record takes the division
    h.inv_d = 1.0 / h.d;
    const bool fast = std::isnormal(h.d) && std::isnormal(h.inv_d) && std::fabs(lo) * h.inv_d <= kFastCoord &&
                      std::fabs(hi) * h.inv_d <= kFastCoord;
    if (!fast) h.inv_d = 0.0;
    h.fix = kFix - lo * h.inv_d;
    return h;
}

cudaError_t hist_launch(const HistSeg* d_segs, int n_segs, int max_nb, long long max_n,
                        const double* N, const double* lw, fpt_bin* bins, fpt_hist_counts* counts,
                        int n_sm, cudaStream_t stream, unsigned* status, uint16_t* bin_idx) {
    const size_t smem_max = (size_t)max_nb * sizeof(unsigned long long);
    cudaError_t e;
    const int threads = 256;
    const int init_blocks = (max_nb + threads - 1) / threads;
    hist_init<<<dim3(init_blocks, n_segs), threads, 0, stream>>>(d_segs, n_segs, bins, counts);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // as many blocks as fit at once, at least one per segment
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hist_pass_max, kMaxThreads, smem_max);
    if (e != cudaSuccess) return e;
    const long long want = std::max(1LL, (max_n + kMaxThreads - 1) / kMaxThreads);
    const long long cap = std::max(1LL, ((long long)std::max(per_sm, 1) * n_sm + n_segs - 1) / n_segs);
    hist_pass_max<<<dim3((unsigned)std::min(want, cap), n_segs), kMaxThreads, smem_max, stream>>>(
        N, lw, d_segs, bins, counts, status, bin_idx);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // long runs per thread amortise the sort and the last bins' reduction (2^24 records, 4000 bins: 469 us for
    // the histogram with 32 per thread, 477 with 20 and 547 with 16, three blocks per SM); short ones spread
    // small inputs over the SMs.  Up to one record per thread of a CTA per SM, one it is: no chain of bins
    // (100 records, 4096 bins: a call of 43 us, 50 with 8 per thread; 38,000 records 46 and 56)
    if (max_n * n_segs >= 4LL * n_sm * kSumThreads * 32)
        e = launch_sum<32>(d_segs, n_segs, max_nb, max_n, lw, bins, n_sm, stream, bin_idx);
    else if (max_n * n_segs <= (long long)n_sm * kSumThreads)
        e = launch_sum<1>(d_segs, n_segs, max_nb, max_n, lw, bins, n_sm, stream, bin_idx);
    else
        e = launch_sum<8>(d_segs, n_segs, max_nb, max_n, lw, bins, n_sm, stream, bin_idx);
    if (e != cudaSuccess) return e;
    hist_final<<<dim3(init_blocks, n_segs), threads, 0, stream>>>(d_segs, bins);
    return cudaGetLastError();
}

}  // namespace fpt
