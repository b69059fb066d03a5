// Stepper for few runs: one warp of a CTA steps 32 runs, three compute their noise.
//
// Binary32.  A warp that has its scheduler to itself is not bound by a pipe but by its own
// order: in the persistent stepper (stepper.cuh) it takes 55 to 65 cycles per step,
// of which the run's chain, reciprocal, multiply-add and add, is 28; the noise's
// XU operations queue in front of the chain's reciprocal and share its
// scoreboards.  Here the chain is alone in its warp: the noise warps, on the SM's
// other schedulers, write what a step needs of each Box–Muller pair to shared
// memory, every third 16-step group each, and the chain warp reads it one group
// ahead: 28 cycles per step and some 50 to 90 per group for the hand-over, 31 to 33 cycles
// per step alone on an SM (39 with binary64 sums, 41 to 47 with a wall, 42 to 57 with three
// on an SM).  The numbers, their order and so the records are those of the persistent
// stepper, bit for bit.
// us, persistent -> this, at one and at three chain warps per SM (4864, 14,592 runs):
// power 2423 -> 1783, 2409 -> 2206; wall 3784 -> 2801, 3782 -> 3403; ladder
// 258 -> 183, 256 -> 233; quartic 151 -> 110, 137 -> 119; diffusive 1057 -> 917 at
// three; 512 runs of some 2150 steps 146 -> 109.  With four per SM the noise warps contend with the
// chains (0.93 to 1.19 times as fast), with six they lose (0.71 to 1.0).
// Slots of two groups read without the copy ahead measured 3 to 9 % slower.
//
// Binary64 (quadratic model).  A warp has the binary64 unit of its scheduler, one
// instruction per 64 cycles, 15 per step: 9 of them are noise, which the noise warps
// take to the other schedulers' units; 6 are left to the chain.
// 516 cycles per step alone on an SM, 720 with a wall, 772 and 945 with three.
// us, persistent -> this: 500 runs 2119 -> 1073 (m = 1, to N = 6), 9728 2671 -> 1422,
// 16,384 2994 -> 2253, 19,456 2985 -> 2211; with a wall, m = 0.1, 19,456 2718 -> 2321;
// with a fifth CTA on an SM (24,320) 3153 -> 3076 and 3051 -> 3978.
//
// Runs are handed out once, 32 to a CTA; all of a warp are at the same step, which
// is what lets the noise run ahead of them.
//
// Every wait ends: a noise warp announces each slot that it was given until it finds the
// stop flag, and the chain warp, once its runs have finished (at the latest at their cap),
// takes one more announcement of each slot and gives it back with the flag set.
#pragma once
#include "stepper.cuh"

namespace fpt {

constexpr int kNoiseWarps = 3;
static_assert(kFewThreads == 32 * (1 + kNoiseWarps), "one chain warp and its noise warps");

// what a step pair needs of its noise, [slot][part][pair][lane]
//   binary32: {t0, t1, rho, c + s} with step terms t, or {q c, q s} with the power bias
//   binary64: {t0, t1}, {r, c}, and s in an array of its own behind them, so that four CTAs of
//   64 sets fit on an SM (padded to a third part they were three, and 19,456 runs took a second
//   wave: 2585 -> 2175 us, with a wall 1768 -> 1160; persistent stepper 2960 and 1326)
template <typename Real>
struct FewNoise {
    using Part = float4;
    static constexpr int kParts = 1, kSingles = 0;
};
template <>
struct FewNoise<double> {
    using Part = double2;
    static constexpr int kParts = 2, kSingles = 1;
};
template <typename Real>
constexpr size_t kRingBytes = (size_t)kNoiseWarps * 8 * 32 *
                              (FewNoise<Real>::kParts * sizeof(typename FewNoise<Real>::Part) +
                               FewNoise<Real>::kSingles * sizeof(Real));

// Hand-over of a slot between its noise warp and the chain warp, 64 threads each:
// one side arrives and goes on, the other waits for it.
__device__ __forceinline__ void hand_arrive(int id) {
    __syncwarp();
    asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory");
}
__device__ __forceinline__ void hand_wait(int id) {
    __syncwarp();
    asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}
__device__ __forceinline__ int full_id(int slot) { return 1 + slot; }
__device__ __forceinline__ int empty_id(int slot) { return 1 + kNoiseWarps + slot; }

// dynamic shared memory but for the set table
template <typename Real, int PREC>
constexpr int few_smem_bytes() {
    return (int)(kRingBytes<Real> + 32 * sizeof(Pending<Real, PREC>));
}

template <typename Real, int PREC, int MODEL, bool WALL, int FOLD>
__global__ void __launch_bounds__(kFewThreads) stepper_few_kernel(const StepperParams P) {
    constexpr bool F64 = sizeof(Real) == 8;
    using Entry = Pending<Real, PREC>;
    using Part = typename FewNoise<Real>::Part;
    constexpr int kSlot = FewNoise<Real>::kParts * 8 * 32;
    static_assert(F64 ? MODEL == FPT_MODEL_QUADRATIC && 16 % FOLD == 0 : FOLD % 16 == 0,
                  "folds and 16-step groups are whole numbers of one another");
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ volatile int s_stop[kNoiseWarps];
    const int n_sets = P.n_sets;
    SetConst* s_sets = reinterpret_cast<SetConst*>(s_dyn);
    long long* s_first = reinterpret_cast<long long*>(s_dyn + (size_t)n_sets * sizeof(SetConst));
    Part* ring = reinterpret_cast<Part*>(s_dyn + stepper_table_bytes(n_sets));
    Real* singles = reinterpret_cast<Real*>(ring + kNoiseWarps * kSlot);  // binary64 only
    Entry* q = reinterpret_cast<Entry*>(s_dyn + stepper_table_bytes(n_sets) + kRingBytes<Real>);
    for (int i = threadIdx.x; i < n_sets; i += blockDim.x) {
        s_sets[i] = P.sets[i];
        s_first[i] = P.sets[i].ticket0;
    }
    if (threadIdx.x == 0) s_first[n_sets] = (long long)P.n_total;
    if (threadIdx.x < kNoiseWarps) s_stop[threadIdx.x] = 0;
    __syncthreads();

    const unsigned FULL = 0xffffffffu;
    const unsigned lane = threadIdx.x & 31u;
    const int warp = (int)(threadIdx.x >> 5);
    // the chain warps of the CTAs that share an SM (b, b + n_sm, ...) on different schedulers
    const int chain = (int)((blockIdx.x / (unsigned)P.n_sm) % (1 + kNoiseWarps));

    // this lane's run: ticket 32 blockIdx + lane, the last set s with ticket0[s] <= ticket
    const unsigned long long t = 32ull * blockIdx.x + lane;
    bool have = t < P.n_total;
    int lo = 0, hi = n_sets - 1;
    while (have && lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((long long)t >= s_first[mid]) lo = mid; else hi = mid - 1;
    }
#if FPT_DEBUG
    if (have && ((long long)t < s_first[lo] || (long long)t >= s_first[lo + 1])) {
        atomicOr(&P.scratch->status, kStatusSetIndex);
        have = false;  // as if there were no such run
    }
#endif
    const SetConst& S = s_sets[lo];
    const unsigned long long i = have ? t - (unsigned long long)s_first[lo] : 0ull;
    typename StepOf<Real, MODEL>::type model;
    model.load(S);

    if (warp != chain) {
        // ---- a noise warp: groups slot, slot + 3, ... until told to stop ----
        const int slot = (warp - chain + kNoiseWarps) % (1 + kNoiseWarps);
        const PhiloxLane pl = philox_lane(S.traj_offset + i, S.set_id, P.keys);
        Part* out = ring + slot * kSlot + lane;
        for (uint32_t G = (uint32_t)slot;; G += kNoiseWarps) {
            uint32_t V[12];
            philox_group(pl, G, P.keys, V);
            Part f[kSlot / 32];
            [[maybe_unused]] Real single[8];
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                if constexpr (F64) {
                    const PairF64 np = group_pair_f64(V, p >> 1, p & 1);
                    const double q2 = __dmul_rn(np.r, model.kq);
                    f[p] = make_double2(__fma_rn(q2, np.c, model.tc), __fma_rn(q2, np.s, model.tc));
                    f[8 + p] = make_double2(np.r, np.c);
                    single[p] = np.s;
                } else {
                    const NormalPair np = group_pair_f32(V, p >> 1, p & 1);
                    const float q2 = __fmul_rn(model.kq, np.rho);
                    if constexpr (is_pow_model(MODEL))
                        f[p] = make_float4(__fmul_rn(q2, np.c), __fmul_rn(q2, np.s), 0.f, 0.f);
                    else
                        f[p] = make_float4(__fmaf_rn(q2, np.c, model.tc), __fmaf_rn(q2, np.s, model.tc), np.rho,
                                           np.c + np.s);
                }
            }
            if (G >= (uint32_t)kNoiseWarps) {
                hand_wait(empty_id(slot));
                if (s_stop[slot] != 0) return;
            }
#pragma unroll
            for (int p = 0; p < kSlot / 32; ++p) out[32 * p] = f[p];
            if constexpr (F64) {
#pragma unroll
                for (int p = 0; p < 8; ++p) singles[slot * 256 + 32 * p + lane] = single[p];
            }
            hand_arrive(full_id(slot));
        }
    }

    // ---- the chain warp ----
    bool on = have;
    if (have && S.phi_in <= S.phi_end) {
        // starts at or below the end of inflation: N = 0, w = 1
        P.out_N[S.first + (long long)i] = 0.0;
        P.out_logw[S.first + (long long)i] = 0.0;
        on = false;
    }
    const bool ran = on;
    Real phi = set_phi_in<Real, MODEL>(S);
    const Real phi_end = set_phi_end<Real, MODEL>(S), twouv = set_twouv<Real, MODEL>(S);
    const int m_max = S.m_max;
    // the state at the last fold before the run's end, as the persistent stepper leaves it
    Real phi0 = phi, acc = (Real)0;
    int m0 = 0;
    WSum<PREC> W;
    W.reset();
    unsigned long long my_steps = 0;

    int slot = 0;  // of the next group to take
    auto release = [&]() {
        hand_arrive(empty_id(slot));
        slot = slot + 1 == kNoiseWarps ? 0 : slot + 1;
    };
    int m = 0;  // steps done
    // the end of a fold: runs that have not finished are committed
    auto fold = [&](bool reached) {
        on = on && !reached && m < m_max;
        WSum<PREC> Wn = W;
        Wn.add(acc);
        W.take(Wn, on);
        acc = (Real)0;
        phi0 = on ? phi : phi0;
        m0 = on ? m : m0;
    };
    if constexpr (F64) {
        Reached64<MODEL> low;
        low.reset(phi, phi_end);
        while (__any_sync(FULL, on)) {
            hand_wait(full_id(slot));
            const Part* f = ring + slot * kSlot + lane;
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const double2 t = f[32 * p], rc = f[32 * (8 + p)];
                const double s = singles[slot * 256 + 32 * p + lane];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    phi = model.step(phi, h == 0 ? t.x : t.y);
                    acc = __fma_rn(rc.x, h == 0 ? rc.y : s, acc);
                    if constexpr (WALL) phi = real_min(phi, twouv - phi);
                    low.see(phi);
                }
                m += 2;
                if ((2 * (p + 1)) % FOLD == 0) fold(low.any());
            }
            release();
        }
    } else if (__any_sync(FULL, on)) {
        float mn = phi;
        auto take = [&](float4 f[8]) {
            hand_wait(full_id(slot));
#pragma unroll
            for (int p = 0; p < 8; ++p) f[p] = ring[slot * kSlot + p * 32 + (int)lane];
        };
        // 16 steps; false once every run has finished
        auto group = [&](const float4 f[8]) -> bool {
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                float first;
                if constexpr (is_pow_model(MODEL)) {
                    phi = model.advance_g(phi, f[p].x, acc);
                    if constexpr (WALL) phi = fminf(phi, twouv - phi);
                    first = phi;
                    phi = model.advance_g(phi, f[p].y, acc);
                    if constexpr (WALL) phi = fminf(phi, twouv - phi);
                } else {
                    phi = step1_f32<WALL>(model, phi, f[p].x, twouv);
                    first = phi;
                    phi = step1_f32<WALL>(model, phi, f[p].y, twouv);
                    acc = __fmaf_rn(f[p].z, f[p].w, acc);
                }
                mn = min3f(mn, first, phi);
            }
            m += 16;
            if (m % FOLD != 0) return true;
            fold(mn <= phi_end);
            return __any_sync(FULL, on);
        };
        float4 a[8], b[8];
        take(a);
        release();
        for (;;) {
            take(b);  // one group ahead: the reads return during the steps
            if (!group(a)) break;
            release();
            take(a);
            if (!group(b)) break;
            release();
        }
        release();
    }
    // the three groups that the noise warps have ready, or will have, are not wanted any more
#pragma unroll
    for (int k = 0; k < kNoiseWarps; ++k) {
        hand_wait(full_id(slot));
        s_stop[slot] = 1;
        __syncwarp();
        release();
    }
    const unsigned runs = __ballot_sync(FULL, ran);
    if (ran) {
        Entry& e = q[__popc(runs & ((1u << lane) - 1u))];
        e.rec = (unsigned long long)S.first + i;
        e.m0 = m0;
        e.set = lo;
        e.phi0 = phi0;
        e.W = W;
    }
    __syncwarp();
    replay_batch<Real, PREC, MODEL, WALL, FOLD>(q, __popc(runs), P, s_sets, lane, my_steps);
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) my_steps += __shfl_xor_sync(FULL, my_steps, o);
    if (lane == 0) {
        atomicAdd(&P.scratch->steps, my_steps);
        if (P.steps_out) atomicAdd(P.steps_out, my_steps);
    }
}

}  // namespace fpt
