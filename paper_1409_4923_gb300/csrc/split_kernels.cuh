// split_kernels.cuh -- runs of few paths: each 32 paths' noise is drawn by warps
// of its own, beside the warp that integrates them.
//
// A run of 1024 paths puts one warp on 32 of the 608 schedulers, and its time
// is the latency of a step.  A warp issues in order, so with the draws in line
// (Philox, three-point or Box-Muller increments, jump events: more than half of
// a step's 45 instructions) the loop-carried chain of the coordinate (an SFU
// cosine and seven dependent FP32 operations) was stretched from about 70 cycles
// to 115.  Here the drawing warps run up to two 32-step blocks ahead and leave
// each path's increments of a block in shared memory (together with the
// drive), and the integrating warp's step is the scheme alone with one load.
// The increments and the order of the arithmetic are those of run_steps, so
// the results are the same bit for bit.  Measured: the 1024-path Poisson run
// (50,000 steps) 1.86 ms instead of 2.77 (77 cycles a step), the 1024-path
// piecewise-linear run in ten launches of 4000 steps 2.51 ms instead of 4.17,
// 20,011 paths with Box-Muller over 4850 steps 0.39 ms instead of 0.75.
#pragma once
#include "chi_kernels.cuh"

namespace sde {

constexpr uint32_t kSplitBlock = 32u;      // steps per block, at absolute multiples of 32

// What a step needs from the drawing warp: the Gaussian increment, the
// corrector's jump increment (Poissonian plus dichotomous), and the
// dichotomous drift term; packed into 1, 2 or 4 floats.
template <bool POIS, int DICH, int GAUSS>
struct SplitLayout {
    static constexpr bool gauss = GAUSS != 0, jump = POIS || DICH == 1, drift = DICH == 2;
    static constexpr int planes = (gauss ? 1 : 0) + (jump ? 1 : 0) + (drift ? 1 : 0);
    static constexpr int width = planes <= 2 ? planes : 4;
    static constexpr int i_jump = gauss ? 1 : 0, i_drift = i_jump + (jump ? 1 : 0);
    static constexpr uint32_t slot_floats = kSplitBlock * 32u * width + kSplitBlock;     // increments, drive
    static constexpr uint32_t bytes = 2u * slot_floats * 4u;
};

// Warps: 0 integrates; then either one that draws everything, or, where that
// would be slower than the integration (Box-Muller; both jump processes), one
// for the jumps and one or (Box-Muller) two for the Gaussian increments, which
// hold no state and alternate between the blocks.
template <bool POIS, int DICH, int GAUSS>
struct SplitWarps {
    static constexpr bool merged = GAUSS != kGaussNormal && !(POIS && DICH != 0);
    static constexpr int jumps = !merged && (POIS || DICH != 0) ? 1 : 0;
    static constexpr int gauss = merged ? 0 : GAUSS == kGaussNormal ? 2 : GAUSS != 0 ? 1 : 0;
    static constexpr int threads = 32 * (1 + (merged ? 1 : jumps + gauss));
    static constexpr int meet = 32 * (1 + (merged ? 1 : jumps + (gauss > 0 ? 1 : 0)));   // threads per slot's barriers
};

// Named barriers of the two slots: 1, 2 "drawn", 3, 4 "used".
template <int FIRST, int THREADS>
__device__ __forceinline__ void split_arrive(uint32_t slot)
{
    if (slot == 0u) asm volatile("bar.arrive %0, %1;" :: "n"(FIRST), "n"(THREADS) : "memory");
    else asm volatile("bar.arrive %0, %1;" :: "n"(FIRST + 1), "n"(THREADS) : "memory");
}
template <int FIRST, int THREADS>
__device__ __forceinline__ void split_sync(uint32_t slot)
{
    if (slot == 0u) asm volatile("bar.sync %0, %1;" :: "n"(FIRST), "n"(THREADS) : "memory");
    else asm volatile("bar.sync %0, %1;" :: "n"(FIRST + 1), "n"(THREADS) : "memory");
}

// A drawing warp: its share (the Gaussian increments, the jumps and their event
// state, the drive) of the blocks first, first + every, ... of steps [na, nb).
template <bool POIS, int DICH, int GAUSS, bool DO_GAUSS, bool DO_JUMPS, bool DO_DRIVE>
__device__ __forceinline__ void split_draw(PathState& S, const PointConsts& P, const LaunchConsts& K, uint32_t path,
                                           uint32_t lane, uint32_t na, uint32_t nb, float* ring, uint32_t first,
                                           uint32_t every)
{
    using L = SplitLayout<POIS, DICH, GAUSS>;
    constexpr int kMeet = SplitWarps<POIS, DICH, GAUSS>::meet;
    const uint32_t base = na & ~(kSplitBlock - 1u), blocks = (nb - base + kSplitBlock - 1u) / kSplitBlock;
    uint32_t k = first;
    for (; k < blocks; k += every) {
        const uint32_t slot = k & 1u, n0 = base + kSplitBlock * k;
        if (k >= 2u) split_sync<3, kMeet>(slot);
        float* out = ring + slot * L::slot_floats + lane * L::width;       // step i: out + 32 width i
        if (DO_DRIVE) ring[slot * L::slot_floats + kSplitBlock * 32u * L::width + lane] = drive_at(n0 + 1u + lane, P);
        const uint32_t wend = min(n0 + kSplitBlock, nb);
        if constexpr (DO_GAUSS && GAUSS == kGauss3Point) {
#pragma unroll
            for (uint32_t b = 0; b < 2u; ++b) {
                const uint4 w = stream(K, P.c1_gauss, path, (n0 >> 4) + b);
#pragma unroll
                for (uint32_t i = 0; i < 4u; ++i) {
                    uint32_t r = i == 0u ? w.x : (i == 1u ? w.y : (i == 2u ? w.z : w.w));
#pragma unroll
                    for (uint32_t j = 0; j < 4u; ++j) out[(16u * b + 4u * i + j) * 32u * L::width] = three_point(r, P);
                }
            }
        } else if constexpr (DO_GAUSS && GAUSS == kGaussNormal) {
#pragma unroll 2
            for (uint32_t g = 0; g < kSplitBlock / 4u; ++g) {
                const uint4 w = stream(K, P.c1_gauss, path, (n0 >> 2) + g);
#pragma unroll
                for (uint32_t j = 0; j < 4u; ++j) out[(4u * g + j) * 32u * L::width] = gauss_inc<GAUSS>(w, j, P);
            }
        }
        if constexpr (DO_JUMPS && (POIS || DICH != 0)) {
            uint32_t dm = 0u;                    // bit i: dichotomous state at step n0 + i
            if constexpr (DICH != 0) {
                dm = S.dst ? 0xffffffffu : 0u;
                while (S.eD < wend) {
                    const uint32_t off = S.eD - n0;
                    dich_event(S, P, K, path);
                    dm ^= 0xffffffffu << off;
                }
            }
#pragma unroll
            for (uint32_t i = 0; i < kSplitBlock; ++i) {
                const float dg = (dm >> i) & 1u ? P.Fb_dt : P.mFa_dt;
                if (L::jump) out[i * 32u * L::width + L::i_jump] = POIS ? (DICH == 1 ? -P.aP_dt + dg : -P.aP_dt) : dg;
                if (L::drift) out[i * 32u * L::width + L::i_drift] = dg;
            }
            if constexpr (POIS) {
                while (S.eP < wend) {
                    const uint32_t off = S.eP - n0;
                    const float z = pois_event(S, P, K, path);
                    const float dg = (dm >> off) & 1u ? P.Fb_dt : P.mFa_dt;
                    out[off * 32u * L::width + L::i_jump] = DICH == 1 ? z + dg : z;
                }
            }
        }
        split_arrive<1, kMeet>(slot);
    }
    // the integrating warp's signals after this warp's blocks among the last two
    for (uint32_t j = blocks >= 2u ? blocks - 2u : 0u; j < blocks; ++j)
        if (every == 1u || (j & 1u) == first) split_sync<3, kMeet>(j & 1u);
}

// A path's increments of one step as the drawing warp left them.
template <class L>
struct SplitStep {
    float v[L::width];
    __device__ __forceinline__ void load(const float* p)
    {
        if constexpr (L::width == 1) v[0] = *p;
        else if constexpr (L::width == 2) {
            const float2 t = *(const float2*)p;
            v[0] = t.x; v[1] = t.y;
        } else {
            const float4 t = *(const float4*)p;
            v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
        }
    }
};

template <int MODEL, bool POIS, int DICH, int GAUSS, bool ACC, bool FOLD>
__device__ __forceinline__ void split_step(PathState& S, const PointConsts& P,
                                           const SplitStep<SplitLayout<POIS, DICH, GAUSS>>& s, float d0, float d1)
{
    using L = SplitLayout<POIS, DICH, GAUSS>;
    const float dxi = L::gauss ? s.v[0] : 0.0f;
    // the jump increment enters where pc_step adds its Poissonian one; a drift
    // term where it adds the dichotomous one
    const float j = L::jump ? s.v[L::i_jump] : 0.0f, dg = L::drift ? s.v[L::i_drift] : 0.0f;
    pc_step<MODEL, L::jump, DICH == 2 ? 2 : 0, ACC, FOLD, false, true>(S, P, dxi, j, dg, d0, d1);
}

// One whole block of 32 steps in one phase; the increments of each group of
// four steps are loaded a group ahead.
template <int MODEL, bool POIS, int DICH, int GAUSS, bool ACC>
__device__ __forceinline__ void split_chunk(PathState& S, const PointConsts& P, const float* in, const float* drive,
                                            float& dcur)
{
    using L = SplitLayout<POIS, DICH, GAUSS>;
    SplitStep<L> cur[4], nxt[4];
    float4 dc = *(const float4*)drive, dn = dc;
#pragma unroll
    for (uint32_t j = 0; j < 4u; ++j) cur[j].load(in + j * 32u * L::width);
#pragma unroll 4
    for (uint32_t g = 0; g < kSplitBlock / 4u; ++g) {
        const uint32_t h = min(g + 1u, kSplitBlock / 4u - 1u);
        dn = *(const float4*)(drive + 4u * h);
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j) nxt[j].load(in + (4u * h + j) * 32u * L::width);
        const float d[4] = {dc.x, dc.y, dc.z, dc.w};
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j) {
            split_step<MODEL, POIS, DICH, GAUSS, ACC, FoldPerStep<MODEL>::value>(S, P, cur[j], dcur, d[j]);
            dcur = d[j];
        }
        if (!FoldPerStep<MODEL>::value) fold<MODEL, true>(S);
        dc = dn;
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j) cur[j] = nxt[j];
    }
}

// The integrating warp: steps [na, nb) with run_steps' arithmetic (whole
// 32-step blocks of a phase folded every four steps, the rest step by step).
template <int MODEL, bool POIS, int DICH, int GAUSS>
__device__ __forceinline__ void split_integrate(PathState& S, const PointConsts& P, uint32_t lane, uint32_t na,
                                                uint32_t nb, const float* ring)
{
    using L = SplitLayout<POIS, DICH, GAUSS>;
    constexpr bool kAcc = MODEL == kModelInertial;
    constexpr int kMeet = SplitWarps<POIS, DICH, GAUSS>::meet;
    const uint32_t ntr = P.n_tr;
    const bool starts = na < ntr || (na == 0u && ntr == 0u);     // the averaging window starts in this call
    const auto window = [&]() {
        if (!FoldPerStep<MODEL>::value) fold<MODEL, true>(S);
        S.c_i = S.c;
        S.kf_i = S.kf;
    };
    float dcur = drive_at(na, P);
    uint32_t k = 0u;
    for (uint32_t n0 = na & ~(kSplitBlock - 1u); n0 < nb; n0 += kSplitBlock, ++k) {
        const uint32_t slot = k & 1u;
        split_sync<1, kMeet>(slot);
        const float* in = ring + slot * L::slot_floats + lane * L::width;
        const float* drive = ring + slot * L::slot_floats + kSplitBlock * 32u * L::width;
        const uint32_t lo = max(n0, na), hi = min(n0 + kSplitBlock, nb);
        if (hi - lo == kSplitBlock && (ntr <= n0 || ntr >= hi)) {
            if (n0 == ntr && starts) window();
            if (n0 >= ntr) {
                split_chunk<MODEL, POIS, DICH, GAUSS, kAcc>(S, P, in, drive, dcur);
                if (kAcc && (hi & 255u) == 0u) {
                    S.svd += (double)S.sv;
                    S.sv2d += (double)S.sv2;
                    S.sv = 0.0f;
                    S.sv2 = 0.0f;
                }
            } else {
                split_chunk<MODEL, POIS, DICH, GAUSS, false>(S, P, in, drive, dcur);
            }
        } else {
            for (uint32_t n = lo; n < hi; ++n) {
                if (n == ntr && starts) window();
                SplitStep<L> s;
                s.load(in + (n - n0) * 32u * L::width);
                const float d1 = drive[n - n0];
                if (n >= ntr) split_step<MODEL, POIS, DICH, GAUSS, kAcc, true>(S, P, s, dcur, d1);
                else split_step<MODEL, POIS, DICH, GAUSS, false, true>(S, P, s, dcur, d1);
                dcur = d1;
            }
        }
        split_arrive<3, kMeet>(slot);
    }
    if (nb == ntr && starts) window();
}

// The integrating warp of a step-size probe: steps [0, n_steps) one at a time
// with chi_kernel's arithmetic.
template <int MODEL, bool POIS, int DICH, int GAUSS>
__device__ __forceinline__ void split_chi(PathState& S, const PointConsts& P, uint32_t lane, uint32_t n_steps,
                                          const float* ring, ChiSums& sums)
{
    using L = SplitLayout<POIS, DICH, GAUSS>;
    constexpr int kMeet = SplitWarps<POIS, DICH, GAUSS>::meet;
    float dcur = drive_at(0u, P);
    for (uint32_t n0 = 0u, k = 0u; n0 < n_steps; n0 += kSplitBlock, ++k) {
        const uint32_t slot = k & 1u;
        split_sync<1, kMeet>(slot);
        const float* in = ring + slot * L::slot_floats + lane * L::width;
        const float* drive = ring + slot * L::slot_floats + kSplitBlock * 32u * L::width;
        const uint32_t steps = min(kSplitBlock, n_steps - n0);
#pragma unroll 4
        for (uint32_t i = 0; i < steps; ++i) {
            SplitStep<L> s;
            s.load(in + i * 32u * L::width);
            const float d1 = drive[i];
            float chi[2];
            pc_step<MODEL, L::jump, DICH == 2 ? 2 : 0, false, true, true, true>(
                S, P, L::gauss ? s.v[0] : 0.0f, L::jump ? s.v[L::i_jump] : 0.0f, L::drift ? s.v[L::i_drift] : 0.0f,
                dcur, d1, chi);
            sums.add(chi);
            dcur = d1;
        }
        if ((n0 & 255u) == 224u && steps == kSplitBlock) sums.flush();
        split_arrive<3, kMeet>(slot);
    }
}

// A step-size probe of few paths; block i: paths 32 i .. 32 i + 31.  Measured
// (4096 paths, 100 steps, Poissonian and three-point noise): 27 us a call
// instead of 66, where one warp drew a Philox block for every step.
template <int MODEL, bool POIS, int DICH, int GAUSS>
__global__ void __launch_bounds__(SplitWarps<POIS, DICH, GAUSS>::threads)
split_chi_kernel(const __grid_constant__ PointConsts P, const __grid_constant__ LaunchConsts K, uint32_t n_steps,
                 double* __restrict__ partials)
{
    using W = SplitWarps<POIS, DICH, GAUSS>;
    extern __shared__ __align__(16) float split_ring[];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, path = blockIdx.x * 32u + lane;
    PathState S;
    init_path<MODEL, POIS, DICH>(S, P, K, path);
    if (warp == 0u) {
        ChiSums sums;
        split_chi<MODEL, POIS, DICH, GAUSS>(S, P, lane, n_steps, split_ring, sums);
        sums.store(partials, blockIdx.x, lane, path < P.n_paths);
    } else if (W::merged || (W::jumps && warp == 1u)) {
        split_draw<POIS, DICH, GAUSS, W::merged, true, true>(S, P, K, path, lane, 0u, n_steps, split_ring, 0u, 1u);
    } else {
        split_draw<POIS, DICH, GAUSS, true, false, !W::jumps>(S, P, K, path, lane, 0u, n_steps, split_ring,
                                                             W::gauss == 2 ? warp - 1u - W::jumps : 0u,
                                                             W::gauss == 2 ? 2u : 1u);
    }
}

// Block i: paths 32 i .. 32 i + 31 of the run, steps [na, nb); M.base == NULL:
// a whole run in one launch, else the states are loaded (na > 0) and saved.
template <int MODEL, bool POIS, int DICH, int GAUSS>
__global__ void __launch_bounds__(SplitWarps<POIS, DICH, GAUSS>::threads, 768 / SplitWarps<POIS, DICH, GAUSS>::threads)
split_kernel(const __grid_constant__ PointConsts P, const __grid_constant__ LaunchConsts K, const StatePlanes M, uint32_t na,
             uint32_t nb, double* __restrict__ partials, const PathOutPtrs po)
{
    using W = SplitWarps<POIS, DICH, GAUSS>;
    extern __shared__ __align__(16) float split_ring[];
    const uint32_t lane = threadIdx.x & 31u, item = blockIdx.x;
    const uint32_t local = item * 32u + lane, path = P.path0 + local;
    const bool last = nb == P.n_tr + P.n_avg, valid = local < P.n_paths;
    PathState S;
    if (na == 0u) init_path<MODEL, POIS, DICH>(S, P, K, path);
    else load_state(S, M, local);
    const uint32_t warp = threadIdx.x >> 5;
    if (warp == 0u) {
        split_integrate<MODEL, POIS, DICH, GAUSS>(S, P, lane, na, nb, split_ring);
        if (M.base) store_motion(S, M, local);
        if (last) {
            PathResult R;
            finish_path<MODEL, false, 0>(S, P, R);
            if (valid) {
                if (po.X_f) po.X_f[local] = R.X_f;
                if (po.v_f) po.v_f[local] = R.v_f;
                if (po.vbar) po.vbar[local] = R.vbar;
            }
            store_partial(partials, item, lane, valid, R);
        }
    } else if (W::merged || (W::jumps && warp == 1u)) {
        split_draw<POIS, DICH, GAUSS, W::merged, true, true>(S, P, K, path, lane, na, nb, split_ring, 0u, 1u);
        if (M.base) store_events(S, M, local);
        if (last && valid) {
            if (po.jP) po.jP[local] = POIS ? S.JP - 1u : 0u;
            if (po.jD) po.jD[local] = DICH ? S.JD - 1u : 0u;
        }
    } else {
        split_draw<POIS, DICH, GAUSS, true, false, !W::jumps>(S, P, K, path, lane, na, nb, split_ring,
                                                             W::gauss == 2 ? warp - 1u - W::jumps : 0u,
                                                             W::gauss == 2 ? 2u : 1u);
        if (!W::jumps && warp == 1u) {
            if (M.base) store_events(S, M, local);
            if (last && valid) {
                if (po.jP) po.jP[local] = 0u;
                if (po.jD) po.jD[local] = 0u;
            }
        }
    }
}

template <int MODEL, bool POIS, int DICH, int GAUSS>
cudaError_t launch_split_t(const PointConsts& P, const LaunchConsts& K, const StatePlanes& M, uint32_t na, uint32_t nb,
                           const Workspace& ws, const PathOutPtrs& po, cudaStream_t st)
{
    if constexpr (SplitLayout<POIS, DICH, GAUSS>::planes == 0) {
        return cudaErrorInvalidValue;      // nothing to draw (split_blocks_per_sm is 0)
    } else {
        split_kernel<MODEL, POIS, DICH, GAUSS><<<K.n_items, SplitWarps<POIS, DICH, GAUSS>::threads, SplitLayout<POIS, DICH, GAUSS>::bytes, st>>>(
            P, K, M, na, nb, ws.partials, po);
        return cudaGetLastError();
    }
}

template <int MODEL, bool POIS, int DICH, int GAUSS>
cudaError_t launch_split_chi_t(const PointConsts& P, const LaunchConsts& K, uint32_t n_steps, const Workspace& ws,
                               cudaStream_t st)
{
    if constexpr (SplitLayout<POIS, DICH, GAUSS>::planes == 0) {
        return cudaErrorInvalidValue;
    } else {
        split_chi_kernel<MODEL, POIS, DICH, GAUSS><<<K.n_items, SplitWarps<POIS, DICH, GAUSS>::threads,
                                                     SplitLayout<POIS, DICH, GAUSS>::bytes, st>>>(P, K, n_steps,
                                                                                                  ws.partials);
        return cudaGetLastError();
    }
}

// Instantiation unit of one model.
#define SDE_SPLIT_UNIT(MODEL) \
    cudaError_t launch_split_chi_m##MODEL(bool pois, int dich, int gauss, const PointConsts& P, const LaunchConsts& K, \
                                          uint32_t n_steps, const Workspace& ws, cudaStream_t st) \
    { \
        SDE_FOR_EACH_VARIANT(SDE_SPLIT_CHI_CASE_##MODEL) \
        return cudaErrorInvalidValue; \
    } \
    cudaError_t launch_split_m##MODEL(bool pois, int dich, int gauss, const PointConsts& P, const LaunchConsts& K, \
                                      const StatePlanes& M, uint32_t na, uint32_t nb, const Workspace& ws, \
                                      const PathOutPtrs& po, cudaStream_t st) \
    { \
        SDE_FOR_EACH_VARIANT(SDE_SPLIT_CASE_##MODEL) \
        return cudaErrorInvalidValue; \
    }
#define SDE_SPLIT_CASE(MODEL, PO, DI, GA) \
    if (pois == PO && dich == DI && gauss == GA) return launch_split_t<MODEL, PO, DI, GA>(P, K, M, na, nb, ws, po, st);
#define SDE_SPLIT_CHI_CASE(MODEL, PO, DI, GA) \
    if (pois == PO && dich == DI && gauss == GA) return launch_split_chi_t<MODEL, PO, DI, GA>(P, K, n_steps, ws, st);
#define SDE_SPLIT_CHI_CASE_0(PO, DI, GA) SDE_SPLIT_CHI_CASE(0, PO, DI, GA)
#define SDE_SPLIT_CHI_CASE_1(PO, DI, GA) SDE_SPLIT_CHI_CASE(1, PO, DI, GA)
#define SDE_SPLIT_CHI_CASE_2(PO, DI, GA) SDE_SPLIT_CHI_CASE(2, PO, DI, GA)
#define SDE_SPLIT_CASE_0(PO, DI, GA) SDE_SPLIT_CASE(0, PO, DI, GA)
#define SDE_SPLIT_CASE_1(PO, DI, GA) SDE_SPLIT_CASE(1, PO, DI, GA)
#define SDE_SPLIT_CASE_2(PO, DI, GA) SDE_SPLIT_CASE(2, PO, DI, GA)

}  // namespace sde
