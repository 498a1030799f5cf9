// Compile-time table of Euler sweep kernels for one element type: every
// (dim, layout, scheme, tile variant) combination whose shared memory fits.
#pragma once
#include <type_traits>

#include "euler_sweep_pair.cuh"
#include "euler_sweep_pair3.cuh"
#include "euler_sweep_row3.cuh"
#include "resident.h"
#include "runtime.h"

namespace ripple {

constexpr int kMaxDynSmem = 227 * 1024;

// The kernel behind a table entry: the one-cell kernel, or for the pair
// variant with FP32 fields the packed cell-pair kernel.
template <typename T, int DIM, int LAYOUT, int SCHEME, int V>
struct SweepKernel {
    static constexpr bool pair = V == kPairVariant;
    static constexpr bool row = V == kRowVariant;
    static constexpr int TX = kSweepVariants[V].tx;
    static constexpr int TY = kSweepVariants[V].ty;
    static constexpr bool f32 = std::is_same<T, float>::value;
    // the pair kernels cover every FP32 scheme (the split FORCE step one sweep per
    // launch); the row kernel only the FP32 3D MUSCL-Hancock step
    static constexpr bool exists = row ? (f32 && DIM == 3 && SCHEME == SCHEME_MUSCL) : (!pair || f32);
    // 3D MUSCL-Hancock: the split-barrier schedule (euler_sweep_pair3.cuh)
    static constexpr bool pair3 = pair && DIM == 3 && SCHEME == SCHEME_MUSCL;
    static constexpr int smem()
    {
        if constexpr (row) return Row3Cfg<LAYOUT>::SMEM;
        else if constexpr (pair3) return Pair3Cfg<LAYOUT>::SMEM;
        else if constexpr (pair) return PairCfg<DIM, LAYOUT, SCHEME>::SMEM;
        else return SweepCfg<T, DIM, LAYOUT, SCHEME, TX, TY>::SMEM;
    }
    static constexpr int nt() { return row ? Row3Cfg<LAYOUT>::NT : TX * TY; }
    static auto fn()
    {
        if constexpr (row && exists) return euler_sweep_row3_kernel<LAYOUT>;
        else if constexpr (pair3 && f32) return euler_sweep_pair3_kernel<LAYOUT>;
        else if constexpr (pair && f32) return euler_sweep_pair_kernel<DIM, LAYOUT, SCHEME>;
        else return euler_sweep_kernel<T, DIM, LAYOUT, SCHEME, (row ? 32 : TX), (row ? 8 : TY)>;
    }
};

template <typename T, int DIM, int LAYOUT, int SCHEME, int V>
struct SweepEntry {
    using K = SweepKernel<T, DIM, LAYOUT, SCHEME, V>;
    static constexpr int TX = K::TX;
    static constexpr int TY = K::TY;
    struct SmemOnly {
        static constexpr int SMEM = K::exists ? K::smem() : 0;
        static constexpr int NT = K::nt();
    };
    using C = SmemOnly;
    static constexpr bool fits = K::exists && C::SMEM > 0 && C::SMEM <= kMaxDynSmem;

    static cudaError_t launch(const SweepLaunch& L)
    {
        if constexpr (!fits) {
            return cudaErrorInvalidValue;
        } else {
            auto k = K::fn();
            if (occupancy() == 0) return cudaErrorInvalidValue;  // also opts in to the shared memory
            // Short steps are placed while the last CTAs of the one before run
            // (step_begin): us a step, without / with, MUSCL-Hancock 20^3 11.7 / 9.5,
            // 48^3 15.8 / 13.8, AoS 17.5 / 14.7, 64^3 21.7 / 19.6; Rusanov 96^3 37.1 /
            // 35.9; FP64 2D MUSCL-Hancock 128^2 28.2 / 26.0, FORCE 34.4 / 28.8.  CTAs
            // placed as others leave spread less evenly over the SMs, which costs more
            // than the gap when a step is long or its CTAs take several items: 96^3
            // MUSCL-Hancock (12 planes an item) 43.7 / 45.3, 256^3 517 / 539, AoS 626 /
            // 651, FP64 2D MUSCL-Hancock 300^2 (380 items) 98.5 / 109.
            const bool ahead = L.sg.items <= L.grid && L.sg.zchunk <= (SCHEME == SCHEME_MUSCL ? 8 : 16);
            cudaLaunchAttribute dep{};
            dep.id = cudaLaunchAttributeProgrammaticStreamSerialization;
            dep.val.programmaticStreamSerializationAllowed = 1;
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3(L.grid);
            cfg.blockDim = dim3(C::NT);
            cfg.dynamicSmemBytes = C::SMEM;
            cfg.stream = L.stream;
            cfg.attrs = &dep;
            cfg.numAttrs = ahead ? 1 : 0;
            return cudaLaunchKernelEx(&cfg, k, *L.map_in, *L.map_out, static_cast<T*>(L.out), L.ctl, L.sg, L.prm);
        }
    }
    static int smem() { return fits ? C::SMEM : 0; }
    static int occupancy()
    {
        if constexpr (!fits) {
            return 0;
        } else {
            static ResidentCtas resident;
            return resident.get(K::fn(), C::NT, C::SMEM);
        }
    }
};

template <typename T, int DIM, int LAYOUT, int SCHEME>
struct SweepRow {
    template <int V>
    static cudaError_t launch_v(int v, const SweepLaunch& L)
    {
        if constexpr (V >= kNumSweepVariants) {
            return cudaErrorInvalidValue;
        } else {
            if (v == V) return SweepEntry<T, DIM, LAYOUT, SCHEME, V>::launch(L);
            return launch_v<V + 1>(v, L);
        }
    }
    template <int V>
    static int smem_v(int v)
    {
        if constexpr (V >= kNumSweepVariants) {
            return 0;
        } else {
            if (v == V) return SweepEntry<T, DIM, LAYOUT, SCHEME, V>::smem();
            return smem_v<V + 1>(v);
        }
    }
    template <int V>
    static int occ_v(int v)
    {
        if constexpr (V >= kNumSweepVariants) {
            return 0;
        } else {
            if (v == V) return SweepEntry<T, DIM, LAYOUT, SCHEME, V>::occupancy();
            return occ_v<V + 1>(v);
        }
    }
};

// Dispatch on (layout, scheme) for a fixed dim.
template <typename T, int DIM>
struct SweepDim {
    static cudaError_t launch(int layout, int scheme, int v, const SweepLaunch& L)
    {
        if (layout == LAYOUT_SOA) {
            if (scheme == SCHEME_MUSCL) return SweepRow<T, DIM, LAYOUT_SOA, SCHEME_MUSCL>::template launch_v<0>(v, L);
            if (scheme == SCHEME_FORCE) return SweepRow<T, DIM, LAYOUT_SOA, SCHEME_FORCE>::template launch_v<0>(v, L);
            return SweepRow<T, DIM, LAYOUT_SOA, SCHEME_RUSANOV1>::template launch_v<0>(v, L);
        }
        if (scheme == SCHEME_MUSCL) return SweepRow<T, DIM, LAYOUT_AOS, SCHEME_MUSCL>::template launch_v<0>(v, L);
        if (scheme == SCHEME_FORCE) return SweepRow<T, DIM, LAYOUT_AOS, SCHEME_FORCE>::template launch_v<0>(v, L);
        return SweepRow<T, DIM, LAYOUT_AOS, SCHEME_RUSANOV1>::template launch_v<0>(v, L);
    }
    static int smem(int layout, int scheme, int v)
    {
        if (layout == LAYOUT_SOA) {
            if (scheme == SCHEME_MUSCL) return SweepRow<T, DIM, LAYOUT_SOA, SCHEME_MUSCL>::template smem_v<0>(v);
            if (scheme == SCHEME_FORCE) return SweepRow<T, DIM, LAYOUT_SOA, SCHEME_FORCE>::template smem_v<0>(v);
            return SweepRow<T, DIM, LAYOUT_SOA, SCHEME_RUSANOV1>::template smem_v<0>(v);
        }
        if (scheme == SCHEME_MUSCL) return SweepRow<T, DIM, LAYOUT_AOS, SCHEME_MUSCL>::template smem_v<0>(v);
        if (scheme == SCHEME_FORCE) return SweepRow<T, DIM, LAYOUT_AOS, SCHEME_FORCE>::template smem_v<0>(v);
        return SweepRow<T, DIM, LAYOUT_AOS, SCHEME_RUSANOV1>::template smem_v<0>(v);
    }
    static int occ(int layout, int scheme, int v)
    {
        if (layout == LAYOUT_SOA) {
            if (scheme == SCHEME_MUSCL) return SweepRow<T, DIM, LAYOUT_SOA, SCHEME_MUSCL>::template occ_v<0>(v);
            if (scheme == SCHEME_FORCE) return SweepRow<T, DIM, LAYOUT_SOA, SCHEME_FORCE>::template occ_v<0>(v);
            return SweepRow<T, DIM, LAYOUT_SOA, SCHEME_RUSANOV1>::template occ_v<0>(v);
        }
        if (scheme == SCHEME_MUSCL) return SweepRow<T, DIM, LAYOUT_AOS, SCHEME_MUSCL>::template occ_v<0>(v);
        if (scheme == SCHEME_FORCE) return SweepRow<T, DIM, LAYOUT_AOS, SCHEME_FORCE>::template occ_v<0>(v);
        return SweepRow<T, DIM, LAYOUT_AOS, SCHEME_RUSANOV1>::template occ_v<0>(v);
    }
};

}  // namespace ripple
