// Kernel launchers of one storage precision: dispatch on (dimension, patch
// size) to the template instances of amr_kernels.cuh. Included once by each
// precision unit (amr_f32.cu, amr_f64.cu) with AMR_T set to its type.
#pragma once
#include "amr_kernels.cuh"

namespace amr {

// Chunk (DZ planes in 3D, DY rows in 2D/3D), block size, least resident CTAs
// per SM (the register cap) and CTAs per SM of the grid of the fused RHS:
// candidate V of a precision, dimension and patch size. Several small CTAs per
// SM rather than one of 256 threads: while one stages or waits at a barrier
// the others compute, and the faces of a chunk fill whole rounds of its
// threads. us per launch, one 256-thread CTA per SM and whole patches (2D) or
// two planes (3D) -> these:
//   FP32 2D 16^2, 25600 patches           917 ->  385  (544 faces in 4.25 rounds of 128)
//   FP32 2D 32^2, 4096 patches            408 ->  232  (halves of 16 rows)
//   FP32 2D  8^2, 16384 patches           392 ->   98  (144 faces in 1.5 rounds of 96)
//   FP32 3D  8^3, 854 leaves, hybrid       98 ->   55  (four planes: fewer halo planes and z faces)
// FP64 is bound by the FP64 pipe (one warp instruction per SM in 9.2 ns, one
// per sub-partition in 31 ns): whole groups of four warps, and smaller chunks
// where an SM would otherwise hold one CTA or the last wave be nearly empty:
//   FP64 2D 16^2, 808 leaves             1008 ->  798  (8 rows)
//   FP64 2D  8^2, 1024 patches            352 ->  305
//   FP64 3D 16^3, 120 leaves             4000 -> 3733  (8 rows: two CTAs of 78 KB per SM)
//   FP64 3D  8^3, 24^3 base, 3 levels    1411 -> 1115  (four planes)
// (FP64 2D 32^2 stays: 1545 against 1572 in halves).
// GRID: CTAs per SM of the grid. Wider than the resident CTAs evens out the
// tail of a launch (FP64 2D 16^2, 808 leaves: 892 us at 2, 798 at 8). FP64 3D
// 16^3 stays at two, as a wider grid can put more chunks on one SM's FP64 pipe
// while others idle (64 patches: 2099 us at 2, 2262 at 4). FP32 3D 16^3 takes
// 12 where a launch has at least 8 waves, and 2 below (172 patches: 208 us per
// step at 2, 216 at 12). Any launch of at most two chunks per SM takes two CTAs
// per SM, as the first CTAs of a wider grid fill some SMs with more (FP32 2D
// 32^2, 148 leaves: 17.9 us at 2, 19.9 at 4).
template <typename T, int D, int N, int V = 0> struct RhsCfg {
    static constexpr bool F32 = sizeof(T) == 4;
    static constexpr int DZ = D == 3 ? (F32 || N == 8 ? 4 : 2) : 1;
    static constexpr int DY = D == 2 && F32 && N == 32 ? 16 : (D >= 2 && !F32 && N == 16 ? 8 : N);
    static constexpr int NTH = D == 1 ? (F32 ? 64 : 128)
                               : D == 2 ? (N == 8 ? (F32 ? 96 : 160) : (F32 || N == 16 ? 128 : 256))
                                        : (N == 8 ? 128 : (F32 ? 256 : 128));
    static constexpr int MINB = D == 1 ? 1
                                : D == 2 ? (N == 8 ? (F32 ? 6 : 3) : (F32 || N == 16 ? 4 : 1))
                                         : (N == 8 ? (F32 ? 4 : 3) : 2);
    static constexpr int GRID = D == 1 ? 2 : D == 2 ? (F32 ? MINB : (N == 16 ? 8 : (N == 8 ? 3 : 2)))
                                                    : (F32 ? (N == 16 ? 12 : MINB) : (N == 8 ? 8 : 2));
    static constexpr int SOME = D == 3 && F32 && N == 16 ? 2 : GRID;
    // a hierarchy is small (RHS_FEW) up to SMs / few_k leaves: there the finer
    // chunks below take less time. us per launch, these chunks / the finer ones,
    // uniform meshes, below and above the line:
    //   FP32 2D  8^2  144 leaves   9.9 / 8.1     289   9.9 / 11.9
    //        2D 16^2   72         12.3 / 9.7     144  12.3 / 12.4
    //        2D 32^2   30         15.7 / 13.6     72  15.7 / 19.5
    //        3D  8^3   27         16.5 / 12.0     48  16.2 / 17.7
    //        3D 16^3    9         26.8 / 18.0     27  26.7 / 37.5
    //   FP64 2D  8^2   72           55 / 46      100    57 / 85
    //        2D 16^2   30          112 / 62       72   111 / 115
    //        2D 32^2   72          539 / 404     100   548 / 559
    //        3D  8^3   27          346 / 240      48   341 / 347
    //        3D 16^3    4          340 / 214       8   340 / 417
    // the hybrid flux, whose FP64 cost sits in the chunks at a front, gains from
    // finer chunks for longer (8^3, 128 leaves: 549 / 442; 16^3, 8: 392 / 284)
    static constexpr int few_k(int flux) {
        const bool hyb = flux == AMR_FLUX_HYBRID;
        return D == 1   ? 1
               : D == 2 ? (F32 ? (N == 8 ? 1 : N == 16 ? 2 : 4) : (N == 16 ? 4 : 2))
                        : (F32 ? (N == 8 ? 4 : 8) : (N == 8 ? (hyb ? 1 : 4) : (hyb ? 16 : 32)));
    }
    static constexpr bool TMA = false;
};
// the other candidates of FP32 3D 16^3 patches: two-plane chunks (72 KB) at
// three CTAs of at most 80 registers per SM (more warps to hide the staging
// loads), and eight-plane chunks (195 KB) of 512 threads at one CTA per SM
// (fewer halo planes staged per interior plane); candidates 3 and 4 are 0 and 2
// with the halo planes brought in by tensor copies (TMA) while the threads
// stage the centre planes
template <> struct RhsCfg<float, 3, 16, 1> {
    static constexpr int DZ = 2, DY = 16, NTH = 256, MINB = 3;
    static constexpr bool TMA = false;
};
template <> struct RhsCfg<float, 3, 16, 2> {
    static constexpr int DZ = 8, DY = 16, NTH = 512, MINB = 1;
    static constexpr bool TMA = false;
};
template <> struct RhsCfg<float, 3, 16, 3> {
    static constexpr int DZ = 4, DY = 16, NTH = 256, MINB = 2;
    static constexpr bool TMA = true;
};
template <> struct RhsCfg<float, 3, 16, 4> {
    static constexpr int DZ = 8, DY = 16, NTH = 512, MINB = 1;
    static constexpr bool TMA = true;
};
// The chunks of a small hierarchy (RHS_FEW), whose whole patches would leave
// most of the chip idle: finer, and as many threads as faces, so that a launch
// takes one round of faces per chunk
constexpr int FEW = 9;
template <typename T, int D, int N> struct RhsCfg<T, D, N, FEW> {
    static constexpr bool F32 = sizeof(T) == 4;
    static constexpr int DZ = D == 3 ? 2 : 1;
    static constexpr int DY = D == 1 ? 1 : D == 2 ? (F32 ? 4 : 2) : (F32 ? (N == 8 ? 8 : 4) : 2);
    static constexpr int NTH = D == 1   ? 64
                               : D == 2 ? (F32 ? (N == 8 ? 96 : N == 16 ? 160 : 320) : (N == 8 ? 64 : N == 16 ? 96 : 192))
                                        : (F32 ? (N == 8 ? 288 : 320) : (N == 8 ? 96 : 192));
    static constexpr int MINB = 1, GRID = !F32 && D == 3 ? 8 : 2;
    static constexpr bool TMA = false;
};
template <typename T, int D, int N, int FLUX> struct RhsShapes {
    static constexpr int n = (sizeof(T) == 4 && D == 3 && N == 16 && FLUX == AMR_FLUX_RUSANOV) ? 5 : 1;
};

#define AMR_DISPATCH(g, CALL)                                   \
    switch ((g).dim * 100 + (g).N) {                            \
    case 108: { constexpr int D = 1, N = 8; CALL; } break;      \
    case 116: { constexpr int D = 1, N = 16; CALL; } break;     \
    case 132: { constexpr int D = 1, N = 32; CALL; } break;     \
    case 208: { constexpr int D = 2, N = 8; CALL; } break;      \
    case 216: { constexpr int D = 2, N = 16; CALL; } break;     \
    case 232: { constexpr int D = 2, N = 32; CALL; } break;     \
    case 308: { constexpr int D = 3, N = 8; CALL; } break;      \
    case 316: { constexpr int D = 3, N = 16; CALL; } break;     \
    default: return cudaErrorInvalidValue;                      \
    }

inline double4 d4(const double* v) { return make_double4(v[0], v[1], v[2], v[3]); }

template <typename T, int D, int N, int FLUX, int V>
static cudaError_t rhs_launch_v(const Grid& g, const T* Us, const T* U0, T* Uout, T* faces, int stage, int grid,
                                cudaStream_t s, int one_slot, int flags, const CUtensorMap* tmap) {
    using C = RhsCfg<T, D, N, V>;
    static const CUtensorMap none{};                     // the kernels without tensor copies ignore it
    if (C::TMA && !tmap) return cudaErrorInvalidValue;   // no tensor map of this state array
    k_rhs<T, D, N, C::DZ, C::DY, C::NTH, C::MINB, FLUX, C::TMA>
        <<<grid, C::NTH, rhs_smem_bytes<T, D, N, C::DZ, C::DY, FLUX, C::TMA>(), s>>>(g, Us, U0, Uout, faces, stage,
                                                                          one_slot, flags, tmap ? *tmap : none);
    return cudaSuccess;
}

template <typename T, int D, int N, int FLUX>
static cudaError_t rhs_launch_f(const Grid& g, const T* Us, const T* U0, T* Uout, T* faces, int stage, int grid,
                                cudaStream_t s, int one_slot, int flags, const CUtensorMap* tmap, int cls) {
    if constexpr (D >= 2)
        if (cls == RHS_FEW && g.rhs_shape == 0)
            return rhs_launch_v<T, D, N, FLUX, FEW>(g, Us, U0, Uout, faces, stage, grid, s, one_slot, flags, tmap);
    if constexpr (RhsShapes<T, D, N, FLUX>::n == 5) {
        switch (g.rhs_shape) {
        case 1: return rhs_launch_v<T, D, N, FLUX, 1>(g, Us, U0, Uout, faces, stage, grid, s, one_slot, flags, tmap);
        case 2: return rhs_launch_v<T, D, N, FLUX, 2>(g, Us, U0, Uout, faces, stage, grid, s, one_slot, flags, tmap);
        case 3: return rhs_launch_v<T, D, N, FLUX, 3>(g, Us, U0, Uout, faces, stage, grid, s, one_slot, flags, tmap);
        case 4: return rhs_launch_v<T, D, N, FLUX, 4>(g, Us, U0, Uout, faces, stage, grid, s, one_slot, flags, tmap);
        default: break;
        }
    }
    return rhs_launch_v<T, D, N, FLUX, 0>(g, Us, U0, Uout, faces, stage, grid, s, one_slot, flags, tmap);
}

template <typename T, int D, int N>
static cudaError_t rhs_launch(const Grid& g, const T* Us, const T* U0, T* Uout, T* faces, int stage, int grid,
                              cudaStream_t s, int one_slot, int flags, const CUtensorMap* tmap, int cls) {
    // one instantiation per flux: the Rusanov kernel carries no HLLC code
    cudaError_t e;
    if (g.flux == AMR_FLUX_CENTRAL)
        e = rhs_launch_f<T, D, N, AMR_FLUX_CENTRAL>(g, Us, U0, Uout, faces, stage, grid, s, one_slot, flags, tmap, cls);
    else if (g.flux == AMR_FLUX_HYBRID)
        e = rhs_launch_f<T, D, N, AMR_FLUX_HYBRID>(g, Us, U0, Uout, faces, stage, grid, s, one_slot, flags, tmap, cls);
    else if (g.flux == AMR_FLUX_HLLC)
        e = rhs_launch_f<T, D, N, AMR_FLUX_HLLC>(g, Us, U0, Uout, faces, stage, grid, s, one_slot, flags, tmap, cls);
    else
        e = rhs_launch_f<T, D, N, AMR_FLUX_RUSANOV>(g, Us, U0, Uout, faces, stage, grid, s, one_slot, flags, tmap, cls);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T, int D, int N, int FLUX, int V>
static cudaError_t rhs_prepare_v() {
    using C = RhsCfg<T, D, N, V>;
    return cudaFuncSetAttribute(k_rhs<T, D, N, C::DZ, C::DY, C::NTH, C::MINB, FLUX, C::TMA>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)rhs_smem_bytes<T, D, N, C::DZ, C::DY, FLUX, C::TMA>());
}

template <typename T, int D, int N, int FLUX>
static cudaError_t rhs_prepare_f() {
    cudaError_t e = rhs_prepare_v<T, D, N, FLUX, 0>();
    if constexpr (D >= 2)
        if (e == cudaSuccess) e = rhs_prepare_v<T, D, N, FLUX, FEW>();
    if constexpr (RhsShapes<T, D, N, FLUX>::n == 5) {
        if (e == cudaSuccess) e = rhs_prepare_v<T, D, N, FLUX, 1>();
        if (e == cudaSuccess) e = rhs_prepare_v<T, D, N, FLUX, 2>();
        if (e == cudaSuccess) e = rhs_prepare_v<T, D, N, FLUX, 3>();
        if (e == cudaSuccess) e = rhs_prepare_v<T, D, N, FLUX, 4>();
    }
    return e;
}

template <typename T, int D, int N>
static cudaError_t rhs_prepare() {
    cudaError_t e = rhs_prepare_f<T, D, N, AMR_FLUX_RUSANOV>();
    if (e == cudaSuccess) e = rhs_prepare_f<T, D, N, AMR_FLUX_HLLC>();
    if (e == cudaSuccess) e = rhs_prepare_f<T, D, N, AMR_FLUX_HYBRID>();
    if (e == cudaSuccess) e = rhs_prepare_f<T, D, N, AMR_FLUX_CENTRAL>();
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_flag_plain<T, D, N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)flag_smem_bytes<T, D, N>());
}

template <typename T, int D, int N>
static int rhs_shapes_of(int flux) {
    switch (flux) {
    case AMR_FLUX_RUSANOV: return RhsShapes<T, D, N, AMR_FLUX_RUSANOV>::n;
    case AMR_FLUX_HLLC: return RhsShapes<T, D, N, AMR_FLUX_HLLC>::n;
    case AMR_FLUX_HYBRID: return RhsShapes<T, D, N, AMR_FLUX_HYBRID>::n;
    default: return RhsShapes<T, D, N, AMR_FLUX_CENTRAL>::n;
    }
}

template <typename T>
int Kernels<T>::rhs_shapes(const Grid& g) {
    switch (g.dim * 100 + g.N) {
    case 108: return rhs_shapes_of<T, 1, 8>(g.flux);
    case 116: return rhs_shapes_of<T, 1, 16>(g.flux);
    case 132: return rhs_shapes_of<T, 1, 32>(g.flux);
    case 208: return rhs_shapes_of<T, 2, 8>(g.flux);
    case 216: return rhs_shapes_of<T, 2, 16>(g.flux);
    case 232: return rhs_shapes_of<T, 2, 32>(g.flux);
    case 308: return rhs_shapes_of<T, 3, 8>(g.flux);
    case 316: return rhs_shapes_of<T, 3, 16>(g.flux);
    default: return 1;
    }
}

template <typename T, int D, int N>
static RhsPlan rhs_plan_of(int flux, long long leaves, long long cap, int nsm) {
    using C = RhsCfg<T, D, N>;
    using W = RhsCfg<T, D, N, FEW>;
    constexpr int nch = Chunk<D, N, C::DZ, C::DY>::NCH, nch_few = Chunk<D, N, W::DZ, W::DY>::NCH;
    const long long slots = (long long)nsm * C::MINB;
    RhsPlan p;
    p.cls = D >= 2 && leaves * C::few_k(flux) <= nsm ? RHS_FEW
            : leaves * nch <= 2 * nsm                ? RHS_PAIR
            : leaves * nch < 8 * slots               ? RHS_SOME
                                                     : RHS_MANY;
    const long long most = cap * (p.cls == RHS_FEW ? nch_few : nch);   // items of the fullest pool
    p.per_sm = p.cls == RHS_FEW ? W::GRID : p.cls == RHS_PAIR ? 2 : p.cls == RHS_SOME ? C::SOME : C::GRID;
    const long long grid = (long long)nsm * p.per_sm;
    p.grid = (int)(most < grid ? most : grid);
    return p;
}

template <typename T>
RhsPlan Kernels<T>::rhs_plan(const Grid& g, int leaves, int nsm) {
    switch (g.dim * 100 + g.N) {
    case 108: return rhs_plan_of<T, 1, 8>(g.flux, leaves, g.cap, nsm);
    case 116: return rhs_plan_of<T, 1, 16>(g.flux, leaves, g.cap, nsm);
    case 132: return rhs_plan_of<T, 1, 32>(g.flux, leaves, g.cap, nsm);
    case 208: return rhs_plan_of<T, 2, 8>(g.flux, leaves, g.cap, nsm);
    case 216: return rhs_plan_of<T, 2, 16>(g.flux, leaves, g.cap, nsm);
    case 232: return rhs_plan_of<T, 2, 32>(g.flux, leaves, g.cap, nsm);
    case 308: return rhs_plan_of<T, 3, 8>(g.flux, leaves, g.cap, nsm);
    default: return rhs_plan_of<T, 3, 16>(g.flux, leaves, g.cap, nsm);
    }
}

template <typename T>
cudaError_t Kernels<T>::prepare(const Grid& g) {
    AMR_DISPATCH(g, return (rhs_prepare<T, D, N>()));
    return cudaSuccess;
}

template <typename T>
cudaError_t Kernels<T>::ghost_fill(const Grid& g, T* U, double tfrac, int grid, cudaStream_t s, int one_slot,
                                   int chunk, bool stage_only, bool look) {
    if (chunk < 32) return cudaErrorInvalidValue;
    const int n_cells = stage_only ? g.n_ghost_face : g.n_ghost;
    if (stage_only && look) {
        AMR_DISPATCH(g, (k_ghost<T, D, N, true, D == 2><<<grid, 256, 0, s>>>(g, U, tfrac, one_slot, d4(g.dmr_pre),
                                                                              d4(g.dmr_post), chunk, n_cells)));
    } else if (stage_only) {
        AMR_DISPATCH(g, (k_ghost<T, D, N, true><<<grid, 256, 0, s>>>(g, U, tfrac, one_slot, d4(g.dmr_pre),
                                                                      d4(g.dmr_post), chunk, n_cells)));
    } else {
        AMR_DISPATCH(g, (k_ghost<T, D, N, false><<<grid, 256, 0, s>>>(g, U, tfrac, one_slot, d4(g.dmr_pre),
                                                                       d4(g.dmr_post), chunk, n_cells)));
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::rhs_stage(const Grid& g, const T* Us, const T* U0, T* Uout, T* faces, int stage, int grid,
                                  cudaStream_t s, int one_slot, int flags, const void* tmap, int cls) {
    AMR_DISPATCH(g, return (rhs_launch<T, D, N>(g, Us, U0, Uout, faces, stage, grid, s, one_slot, flags,
                                                static_cast<const CUtensorMap*>(tmap), cls)));
    return cudaSuccess;
}

template <typename T>
cudaError_t Kernels<T>::reflux(const Grid& g, T* Uout, const T* faces, int stage, int grid, cudaStream_t s,
                               int one_item) {
    AMR_DISPATCH(g, (k_reflux<T, D, N><<<grid, 256, 0, s>>>(g, Uout, faces, stage, one_item)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::restrict_level(const Grid& g, T* U, int level, int grid, cudaStream_t s, int one_slot) {
    AMR_DISPATCH(g, (k_restrict<T, D, N><<<grid, 256, 0, s>>>(g, U, level, one_slot)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::begin_step(const Grid& g, T* U, int ncfl, int grid, int chunk, bool look, cudaStream_t s) {
    if (look) {
        AMR_DISPATCH(g, (k_begin<T, D, N, D == 2><<<grid, 256, 0, s>>>(g, U, ncfl, d4(g.dmr_pre), d4(g.dmr_post),
                                                                        chunk, g.n_ghost_face)));
    } else {
        AMR_DISPATCH(g, (k_begin<T, D, N><<<grid, 256, 0, s>>>(g, U, ncfl, d4(g.dmr_pre), d4(g.dmr_post), chunk,
                                                               g.n_ghost_face)));
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::settle(const Grid& g, T* U, const T* faces, int stage, int grid, cudaStream_t s) {
    AMR_DISPATCH(g, (k_settle<T, D, N><<<grid, 256, 0, s>>>(g, U, faces, stage)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::after_stage(const Grid& g, T* U, const T* faces, int stage, bool next, double tfrac, int chunk,
                                    cudaStream_t s) {
    auto go = [&](auto n) {
        k_after<T, 1, decltype(n)::value><<<AFTER_CTAS, 256, 0, s>>>(g, U, faces, stage, next ? 1 : 0, tfrac, d4(g.dmr_pre),
                                                                     d4(g.dmr_post), chunk, g.n_ghost_face);
    };
    if (g.dim != 1) return cudaErrorInvalidValue;
    if (g.N == 8) go(std::integral_constant<int, 8>{});
    else if (g.N == 16) go(std::integral_constant<int, 16>{});
    else if (g.N == 32) go(std::integral_constant<int, 32>{});
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::cfl(const Grid& g, const T* U, int grid, cudaStream_t s, int one_slot, bool finalize) {
    AMR_DISPATCH(g, (k_cfl<T, D, N><<<grid, 256, 0, s>>>(g, U, one_slot, finalize ? 1 : 0)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::init_ic(const Grid& g, T* U, const int* list, int n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int grid = (int)(((long long)n * 4096 + 255) / 256 < 65536 ? ((long long)n * 4096 + 255) / 256 : 65536);
    AMR_DISPATCH(g, (k_init_ic<T, D, N><<<grid, 256, 0, s>>>(g, U, list, n, d4(g.dmr_pre), d4(g.dmr_post))));
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::prolong_new(const Grid& g, T* U, const int* list, int n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int grid = n < 65536 ? n : 65536;
    AMR_DISPATCH(g, (k_prolong_new<T, D, N><<<grid, 256, 0, s>>>(g, U, list, n)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::flag_plain(const Grid& g, const T* U, int* anyflag, int grid, cudaStream_t s) {
    if (g.dim == 3) {                                    // OR over a patch's slabs
        const cudaError_t e = cudaMemsetAsync(anyflag, 0, sizeof(int) * (size_t)g.cap, s);
        if (e != cudaSuccess) return e;
    }
    AMR_DISPATCH(g, (k_flag_plain<T, D, N><<<grid, 256, flag_smem_bytes<T, D, N>(), s>>>(g, U, anyflag)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::cons_sums(const Grid& g, const T* U, double* partial, double* out, cudaStream_t s) {
    AMR_DISPATCH(g, (k_cons_partial<T, D, N><<<1024, 256, 0, s>>>(g, U, partial)));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    switch (g.nv) {
    case 3: k_cons_total<3><<<1, 256, 0, s>>>(g.counts, partial, out); break;
    case 4: k_cons_total<4><<<1, 256, 0, s>>>(g.counts, partial, out); break;
    default: k_cons_total<5><<<1, 256, 0, s>>>(g.counts, partial, out); break;
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::unpack_interiors(const Grid& g, const T* U, const int* slots, int n, double* out,
                                         cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    AMR_DISPATCH(g, (k_unpack<T, D, N><<<1024, 256, 0, s>>>(g, U, slots, n, out)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t Kernels<T>::pack_interiors(const Grid& g, T* U, const int* slots, int n, const double* in,
                                       cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    AMR_DISPATCH(g, (k_pack<T, D, N><<<1024, 256, 0, s>>>(g, U, slots, n, in)));
    return cudaGetLastError();
}

}  // namespace amr
