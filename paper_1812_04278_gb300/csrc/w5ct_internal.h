// w5ct_internal.h -- declarations shared by the translation units of libw5ct.
#pragma once
#include <cuda_runtime.h>

#include "w5ct_kernels.cuh"

namespace w5ct {

// Record the text that w5ct_last_error(NULL) returns (calls without a context).
void set_global_error(const char *text);

// Launch a kernel of a single-patch step so that its blocks may be scheduled
// before the kernel ahead of it in the stream has drained (programmatic
// dependent launch; the kernel waits for it in chain_begin).  A 32^3 step is 13
// kernels of 3 to 10 us, and their launch latencies do not overlap otherwise:
// two 32^3 FP32-bulk steps with their state loaded and read back 250 -> 186 us
// (of that, dt formed by the CFL kernel's last block: two operations a step).
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Launch the FP32 characteristic sweep along `axis` (0, 1, 2) with WENO
// variant `variant` (0 = JS, 1 = Z) over one patch in the default tile
// (SweepTuning), and, in either type, all three sweeps in one launch
// (sweep_all_kernel).  Defined in w5ct_sweep32.cu / w5ct_sweep64.cu.
cudaError_t launch_sweep_f32(int axis, int variant, const SweepArgs<float> &a, cudaStream_t s);
template <typename Real>
cudaError_t launch_sweep_all(int variant, const SweepArgs<Real> (&a)[3], cudaStream_t s);

// The three FP64 single-patch sweeps in one launch with the WENO part of every
// flux in double-word arithmetic, and the shared-memory allowance of its
// kernels.  Defined in w5ct_sweep64dw.cu.
cudaError_t launch_sweep_all_f64dw(int variant, const SweepArgs<double> (&a)[3], cudaStream_t s);
cudaError_t prepare_sweeps_f64dw();

// Sweep tiling per arithmetic type: faces per block in the second tile
// direction (x-sweep: pencils along y; y- and z-sweeps: faces along the
// axis) and the minimum resident blocks per SM the register budget targets.
template <typename Real>
struct SweepTuning;

// Defaults measured on GB300.  FP32: 128-thread blocks, two faces per thread,
// four blocks per SM, 32 x 8 tiles along x and 16 x 16 in the other two sweeps:
// 27.36 ms for two 256^3 WENO-Z steps and 109.8 ms for a 512^3 WENO5 step, against
// 27.95 and 113.1 for 256-thread blocks of 32 x 16 (a barrier stalls half an
// SM's warps there), 27.47 and 110.8 for 8 x 32, 28.17 and 113.9 for one face
// per thread, 28.1 and 112.8 for three, 28.7 and 116.2 for four (26.5 and 108.3 for
// the chosen one with the later forms of the box and the eigenvectors).
#ifndef W5CT_F32_T2X
#define W5CT_F32_T2X 8
#endif
#ifndef W5CT_F32_T2YZ
#define W5CT_F32_T2YZ 16
#endif
#ifndef W5CT_F32_MINB
#define W5CT_F32_MINB 4
#endif
#ifndef W5CT_F32_FPT
#define W5CT_F32_FPT 2
#endif
#ifndef W5CT_F32_BXX
#define W5CT_F32_BXX 32
#endif
#ifndef W5CT_F32_BXYZ
#define W5CT_F32_BXYZ 16
#endif
template <>
struct SweepTuning<float> {
    static constexpr int T2X = W5CT_F32_T2X, T2YZ = W5CT_F32_T2YZ, MINB = W5CT_F32_MINB, FPT = W5CT_F32_FPT,
                         BXX = W5CT_F32_BXX, BXYZ = W5CT_F32_BXYZ;
};
template <int AX, typename Real>
struct SweepCfg {
    static constexpr int T2 = AX == 0 ? SweepTuning<Real>::T2X : SweepTuning<Real>::T2YZ;
    static constexpr int BX = AX == 0 ? SweepTuning<Real>::BXX : SweepTuning<Real>::BXYZ;
    static constexpr int MINB = SweepTuning<Real>::MINB;
    static constexpr int FPT = SweepTuning<Real>::FPT;
    using TT = SweepTile<AX, T2, BX, FPT>;
    static constexpr size_t smem = (size_t)TT::template cells<Real> * box_quantities<Real>() * sizeof(Real);
};

// Single-patch sweep in tiles of BX x T2 faces, FPT per thread (the block
// is BX x T2 / FPT threads).
template <int AX, typename Real, int VAR, int T2, int MINB, int FPT, int BX = 32>
struct SinglePatchSweep {
    using TT = SweepTile<AX, T2, BX, FPT>;
    static constexpr size_t smem = (size_t)TT::template cells<Real> * box_quantities<Real>() * sizeof(Real);
    static cudaError_t prepare() {
        return cudaFuncSetAttribute(sweep_kernel<AX, Real, VAR, T2, MINB, FPT, BX>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    }
    static dim3 grid(int nx, int ny, int nz) {
        if (AX == 0 || AX == 1) return dim3((nx + BX - 1) / BX, (ny + TT::BY - 1) / TT::BY, nz);
        return dim3((nx + BX - 1) / BX, ny, (nz + TT::BZ - 1) / TT::BZ);
    }
    static cudaError_t launch(const SweepArgs<Real> &a, cudaStream_t s) {
        return launch_chained(sweep_kernel<AX, Real, VAR, T2, MINB, FPT, BX>, grid(a.nx, a.ny, a.nz), dim3(BX, TT::ROWS),
                              smem, s, a);
    }
};

// Tile shapes of the batched sweeps (chosen per patch and axis by the
// autotuner).  Variant 0 is 32 x 16; the float path also has narrower tiles
// that waste fewer lanes on patches whose sizes are not multiples of 32 or of
// 16: (BX, T2, faces per thread) = (16, 16, 2), (8, 16, 1), (8, 8, 1).  Every
// variant keeps 128 registers per thread in float: min blocks per SM = 512 /
// threads per block.  One launch per axis and variant computes a float
// or double 32 x 16 tile as two halves, in blocks of 128 threads like the
// single-patch tiles (double, 168 registers: three per SM along x, two along y and
// z, whose boxes of 84 KB fill it, instead of one of 256 threads; 48 patches 50.6 ->
// 48.3 ms per step).
// Step of the 512-patch workload with one variant forced on every patch: 24.1,
// 23.4, 24.0, 23.4 ms, and 22.8 ms with the choice per patch and axis; before
// the halves, whole 32 x 16 tiles in 256-thread blocks took 27.6 ms.
constexpr int kMaxTileVariants = 4;

template <int AX, typename Real, int V>
struct TileV;
template <int AX, typename Real>
struct TileV<AX, Real, 0> {
    static constexpr int T2 = 16, BX = 32, FPT = 2, MINB = sizeof(Real) == 8 ? 1 : 2;
};
template <int AX, typename Real>
struct TileV<AX, Real, 1> {
    static constexpr int T2 = 16, BX = 16, FPT = 2, MINB = 4;
};
template <int AX, typename Real>
struct TileV<AX, Real, 2> {
    static constexpr int T2 = 16, BX = 8, FPT = 1, MINB = 4;
};
template <int AX, typename Real>
struct TileV<AX, Real, 3> {
    static constexpr int T2 = 8, BX = 8, FPT = 1, MINB = 8;
};

template <typename Real>
inline int num_tile_variants() {
    return sizeof(Real) == 4 ? kMaxTileVariants : 1;
}

// (BX, T2) of variant v along axis `axis` (host side, for the tile tables)
template <typename Real>
inline void tile_shape(int axis, int v, int &bx, int &t2) {
    if (v == 0) {
        bx = 32;
        t2 = 16;
    } else {
        bx = v == 1 ? 16 : 8;
        t2 = v == 3 ? 8 : 16;
    }
}

template <int AX, typename Real, int VAR, int V>
struct BatchedSweep {
    using C = TileV<AX, Real, V>;
    static constexpr bool kHalves = V == 0;
    static constexpr int BX = kHalves && AX != 0 ? C::BX / 2 : C::BX, T2 = kHalves && AX == 0 ? C::T2 / 2 : C::T2,
                         MINB = !kHalves ? C::MINB : std::is_same<Real, float>::value ? 2 * C::MINB : 3;
    using TT = SweepTile<AX, T2, BX, C::FPT>;
    static constexpr size_t smem = (size_t)TT::template cells<Real> * box_quantities<Real>() * sizeof(Real);
    static cudaError_t prepare() {
        return cudaFuncSetAttribute(sweep_batched_kernel<AX, Real, VAR, T2, MINB, BX, C::FPT, kHalves>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    }
    static cudaError_t launch(const SweepArgs<Real> &a, const PatchGeom *pgs, const int4 *tiles, int ntiles,
                              cudaStream_t s) {
        sweep_batched_kernel<AX, Real, VAR, T2, MINB, BX, C::FPT, kHalves>
            <<<(unsigned)ntiles * (kHalves ? 2u : 1u), dim3(BX, TT::ROWS), smem, s>>>(a, pgs, tiles);
        return cudaGetLastError();
    }
};

// Persistent sweep of one tile variant over the three axes: a grid of
// resident blocks takes work items (tiles of any axis, the axis in bits 28-29
// of item.x, the patch in bits 0-27) from a device counter with atomicAdd
// until the list is exhausted.  Nothing waits on another block, so the
// queue needs no spin; the counter is zeroed before the launch.  The three
// axes' sweeps of a stage are independent (all read the stage state), so one
// queue covers them and their tails overlap.
template <typename Real, int VAR, int V>
struct PersistentSweep {
    using C0 = TileV<0, Real, V>;
    using C1 = TileV<1, Real, V>;
    using C2 = TileV<2, Real, V>;
    using T0 = SweepTile<0, C0::T2, C0::BX, C0::FPT>;
    using T1 = SweepTile<1, C1::T2, C1::BX, C1::FPT>;
    using T2_ = SweepTile<2, C2::T2, C2::BX, C2::FPT>;
    static_assert(T0::NT == T1::NT && T1::NT == T2_::NT && C0::BX == C1::BX && C1::BX == C2::BX,
                  "one block shape for the three axes");
    static constexpr int NT = T0::NT, BX = C0::BX, ROWS = T0::ROWS, MINB = C0::MINB;
    static constexpr size_t smem0 = (size_t)T0::template cells<Real> * box_quantities<Real>() * sizeof(Real);
    static constexpr size_t smem1 = (size_t)T1::template cells<Real> * box_quantities<Real>() * sizeof(Real);
    static constexpr size_t smem2 = (size_t)T2_::template cells<Real> * box_quantities<Real>() * sizeof(Real);
    static constexpr size_t smem = smem0 > smem1 ? (smem0 > smem2 ? smem0 : smem2) : (smem1 > smem2 ? smem1 : smem2);
};

template <typename Real, int VAR, int V>
__global__ void __launch_bounds__(PersistentSweep<Real, VAR, V>::NT, PersistentSweep<Real, VAR, V>::MINB)
    sweep_persistent_kernel(SweepArgs<Real> a0, SweepArgs<Real> a1, SweepArgs<Real> a2,
                            const PatchGeom *__restrict__ pgs, const int4 *__restrict__ items, int nitems,
                            int *counter) {
    using P = PersistentSweep<Real, VAR, V>;
    extern __shared__ __align__(16) unsigned char w5ct_smem[];
    __shared__ int s_item;
    Real *sm = reinterpret_cast<Real *>(w5ct_smem);
    for (;;) {
        if (threadIdx.x == 0 && threadIdx.y == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= nitems) break;           // the same value in every thread of the block
        const int4 t = items[it];
        const int ax = t.x >> kItemAxisShift;
        const PatchGeom pg = pgs[t.x & kItemPatchMask];
        if (ax == 0)
            sweep_tile<0, Real, VAR, P::C0::T2, P::BX, P::C0::FPT, 1>(a0, pg, t.y, t.z, t.w, sm);
        else if (ax == 1)
            sweep_tile<1, Real, VAR, P::C1::T2, P::BX, P::C1::FPT, 1>(a1, pg, t.y, t.z, t.w, sm);
        else
            sweep_tile<2, Real, VAR, P::C2::T2, P::BX, P::C2::FPT, 1>(a2, pg, t.y, t.z, t.w, sm);
        __syncthreads();                   // shared memory and s_item are reused
    }
}

template <typename Real, int VAR, int V>
struct PersistentLaunch {
    using P = PersistentSweep<Real, VAR, V>;
    static cudaError_t prepare() {
        return cudaFuncSetAttribute(sweep_persistent_kernel<Real, VAR, V>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)P::smem);
    }
    // resident blocks of this kernel on the whole device
    static cudaError_t grid(int &blocks) {
        int dev = 0, sms = 0, per = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, sweep_persistent_kernel<Real, VAR, V>, P::NT, P::smem);
        blocks = sms * (per > 0 ? per : 1);
        return e;
    }
    static cudaError_t launch(const SweepArgs<Real> (&a)[3], const PatchGeom *pgs, const int4 *items, int nitems,
                              int *counter, int blocks, cudaStream_t s) {
        sweep_persistent_kernel<Real, VAR, V><<<blocks, dim3(P::BX, P::ROWS), P::smem, s>>>(a[0], a[1], a[2], pgs, items,
                                                                                         nitems, counter);
        return cudaGetLastError();
    }
};

// The three sweeps of a stage in one launch (sweep_all_kernel).
template <typename Real, int VAR, bool DW = false>
struct AllSweeps {
    template <int AX>
    static constexpr size_t smem_of = (size_t)SweepTile<AX, AllTile<AX>::T2, AllTile<AX>::BX, 1>::template cells<Real> *
                                      box_quantities<Real>() * sizeof(Real);
    static constexpr size_t smem = smem_of<0> > smem_of<1> ? smem_of<0> : smem_of<1>;   // (y and z alike)
    static cudaError_t prepare() {
        return cudaFuncSetAttribute(sweep_all_kernel<Real, VAR, DW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    }
    static cudaError_t launch(const SweepArgs<Real> (&a)[3], cudaStream_t st) {
        SweepAll<Real> s;
        const int n[3] = {a[0].nx, a[0].ny, a[0].nz};
        s.first[0] = 0;
        for (int ax = 0; ax < 3; ++ax) {
            s.a[ax] = a[ax];
            const int bx = ax == 0 ? AllTile<0>::BX : AllTile<1>::BX, t2 = ax == 0 ? AllTile<0>::T2 : AllTile<1>::T2;
            s.nbx[ax] = (n[0] + bx - 1) / bx;
            s.nb2[ax] = (n[ax == 2 ? 2 : 1] + t2 - 1) / t2;
            s.first[ax + 1] = s.first[ax] + s.nbx[ax] * s.nb2[ax] * n[ax == 2 ? 1 : 2];
        }
        return launch_chained(sweep_all_kernel<Real, VAR, DW>, dim3(s.first[3]), dim3(kAllThreads), smem, st, s);
    }
};

// allow the dynamic shared memory of every sweep kernel of this type
template <int AX, typename Real, int VAR>
cudaError_t prepare_sweep_axis() {
    cudaError_t e = cudaSuccess;
    if constexpr (std::is_same<Real, float>::value) {
        using C = SweepCfg<AX, Real>;
        e = SinglePatchSweep<AX, Real, VAR, C::T2, C::MINB, C::FPT, C::BX>::prepare();
        if (e != cudaSuccess) return e;
    }
    if ((e = BatchedSweep<AX, Real, VAR, 0>::prepare()) != cudaSuccess) return e;
    if constexpr (sizeof(Real) == 4) {
        if ((e = BatchedSweep<AX, Real, VAR, 1>::prepare()) != cudaSuccess) return e;
        if ((e = BatchedSweep<AX, Real, VAR, 2>::prepare()) != cudaSuccess) return e;
        if ((e = BatchedSweep<AX, Real, VAR, 3>::prepare()) != cudaSuccess) return e;
    }
    if constexpr (AX == 0) {
        if ((e = AllSweeps<Real, VAR>::prepare()) != cudaSuccess) return e;
        if ((e = PersistentLaunch<Real, VAR, 0>::prepare()) != cudaSuccess) return e;
        if constexpr (sizeof(Real) == 4) {
            if ((e = PersistentLaunch<Real, VAR, 1>::prepare()) != cudaSuccess) return e;
            if ((e = PersistentLaunch<Real, VAR, 2>::prepare()) != cudaSuccess) return e;
            if ((e = PersistentLaunch<Real, VAR, 3>::prepare()) != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

template <typename Real>
cudaError_t prepare_sweeps_impl() {
    cudaError_t e;
    if constexpr (std::is_same<Real, double>::value)
        if ((e = prepare_sweeps_f64dw()) != cudaSuccess) return e;
    if ((e = prepare_sweep_axis<0, Real, 0>()) != cudaSuccess) return e;
    if ((e = prepare_sweep_axis<1, Real, 0>()) != cudaSuccess) return e;
    if ((e = prepare_sweep_axis<2, Real, 0>()) != cudaSuccess) return e;
    if ((e = prepare_sweep_axis<0, Real, 1>()) != cudaSuccess) return e;
    if ((e = prepare_sweep_axis<1, Real, 1>()) != cudaSuccess) return e;
    return prepare_sweep_axis<2, Real, 1>();
}

// Defined in w5ct_sweep32.cu / w5ct_sweep64.cu.
template <typename Real>
cudaError_t prepare_sweeps();
// Tiles `tiles` (all of tile variant tv) of the batched sweep along `axis`.
template <typename Real>
cudaError_t launch_sweep_batched(int axis, int variant, int tv, const SweepArgs<Real> &a, const PatchGeom *pgs,
                                 const int4 *tiles, int ntiles, cudaStream_t s);

// The persistent sweep of tile variant tv over items (three axes, see
// sweep_persistent_kernel) with `blocks` resident blocks; and that block count.
template <typename Real>
cudaError_t launch_sweep_persistent(int variant, int tv, const SweepArgs<Real> (&a)[3], const PatchGeom *pgs,
                                    const int4 *items, int nitems, int *counter, int blocks, cudaStream_t s);
template <typename Real>
cudaError_t persistent_grid(int variant, int tv, int &blocks);

template <typename Real, int VAR>
cudaError_t launch_sweep_persistent_v(int tv, const SweepArgs<Real> (&a)[3], const PatchGeom *pgs, const int4 *items,
                                      int nitems, int *counter, int blocks, cudaStream_t s) {
    if constexpr (sizeof(Real) == 4) {
        if (tv == 1) return PersistentLaunch<Real, VAR, 1>::launch(a, pgs, items, nitems, counter, blocks, s);
        if (tv == 2) return PersistentLaunch<Real, VAR, 2>::launch(a, pgs, items, nitems, counter, blocks, s);
        if (tv == 3) return PersistentLaunch<Real, VAR, 3>::launch(a, pgs, items, nitems, counter, blocks, s);
    }
    if (tv != 0) return cudaErrorInvalidValue;
    return PersistentLaunch<Real, VAR, 0>::launch(a, pgs, items, nitems, counter, blocks, s);
}

template <typename Real, int VAR>
cudaError_t persistent_grid_v(int tv, int &blocks) {
    if constexpr (sizeof(Real) == 4) {
        if (tv == 1) return PersistentLaunch<Real, VAR, 1>::grid(blocks);
        if (tv == 2) return PersistentLaunch<Real, VAR, 2>::grid(blocks);
        if (tv == 3) return PersistentLaunch<Real, VAR, 3>::grid(blocks);
    }
    if (tv != 0) return cudaErrorInvalidValue;
    return PersistentLaunch<Real, VAR, 0>::grid(blocks);
}

template <int AX, typename Real, int VAR>
cudaError_t launch_sweep_batched_axis(int tv, const SweepArgs<Real> &a, const PatchGeom *pgs, const int4 *tiles,
                                      int ntiles, cudaStream_t s) {
    if constexpr (sizeof(Real) == 4) {
        if (tv == 1) return BatchedSweep<AX, Real, VAR, 1>::launch(a, pgs, tiles, ntiles, s);
        if (tv == 2) return BatchedSweep<AX, Real, VAR, 2>::launch(a, pgs, tiles, ntiles, s);
        if (tv == 3) return BatchedSweep<AX, Real, VAR, 3>::launch(a, pgs, tiles, ntiles, s);
    }
    if (tv != 0) return cudaErrorInvalidValue;
    return BatchedSweep<AX, Real, VAR, 0>::launch(a, pgs, tiles, ntiles, s);
}

template <typename Real>
cudaError_t launch_sweep_batched_impl(int axis, int variant, int tv, const SweepArgs<Real> &a, const PatchGeom *pgs,
                                      const int4 *tiles, int ntiles, cudaStream_t s) {
    if (variant == 0) {
        if (axis == 0) return launch_sweep_batched_axis<0, Real, 0>(tv, a, pgs, tiles, ntiles, s);
        if (axis == 1) return launch_sweep_batched_axis<1, Real, 0>(tv, a, pgs, tiles, ntiles, s);
        return launch_sweep_batched_axis<2, Real, 0>(tv, a, pgs, tiles, ntiles, s);
    }
    if (axis == 0) return launch_sweep_batched_axis<0, Real, 1>(tv, a, pgs, tiles, ntiles, s);
    if (axis == 1) return launch_sweep_batched_axis<1, Real, 1>(tv, a, pgs, tiles, ntiles, s);
    return launch_sweep_batched_axis<2, Real, 1>(tv, a, pgs, tiles, ntiles, s);
}

// blocks of the single-patch sweep along `axis` in tiles of bx lanes x t2
inline long long sweep_blocks(int axis, int t2, int bx, int nx, int ny, int nz) {
    const long long nbx = (nx + bx - 1) / bx;
    if (axis == 2) return nbx * ny * ((nz + t2 - 1) / t2);
    return nbx * ((ny + t2 - 1) / t2) * nz;     // x- and y-sweeps: t2 pencils or faces along y
}

// Whether the three FP32 sweeps of a single patch go in one launch
// (sweep_all_kernel; the FP64 ones always do).
// FP64: the small blocks balance the SMs better than they lose by their larger
// boxes: step of 32^3 1.93 -> 1.01 ms against three launches of 32 x 16 and 16 x
// 32 tiles, 64^3 7.68 -> 6.60, 100 x 70 x 50 10.26 -> 9.80 (WENO5), 160^3 101.4 ->
// 100.4, 256^3 413.4 -> 411.4 ms.
// FP32: one launch saves two launches' latency and tail; its blocks are twice as
// many and cost more each, also where an axis is thin and they hold one row of
// faces (512 x 512 x 1).  So it is taken up to 12 waves of its blocks (four per
// SM), and to more where nx leaves lanes of 16-wide tiles empty that its 8-wide
// ones fill (`lanes`: 1 for none, 1/2 for nx <= 8).  us a step, three launches against
// one (waves): 48^3 150, 128 (4.7); 64^3 236, 230 (10); 192 x 192 x 1 141, 128 (8.5);
// 208 x 1 x 208 171, 174 (12); 256 x 256 x 1 185, 194 (15); 80^3 473, 482 (21);
// 512 x 512 x 1 500, 658 (61); 256^2 x 16 845, 897 (40); with lanes 0.9 72^3 387, 379
// (17), 66 x 200 x 200 2615, 2713 (126); 0.83 40 x 200 x 100 878, 857 (39); 0.75 24 x
// 200 x 200 1003, 926 (42), 4 x 512 x 512 (0.5) 4342, 3794 (162).
inline bool sweeps_in_one_f32(int nx, int ny, int nz, int sms) {
    using X = AllTile<0>;
    using YZ = AllTile<1>;
    const double waves = (double)(sweep_blocks(0, X::T2, X::BX, nx, ny, nz) + sweep_blocks(1, YZ::T2, YZ::BX, nx, ny, nz) +
                                  sweep_blocks(2, YZ::T2, YZ::BX, nx, ny, nz)) / (4.0 * sms);
    const double lanes = (double)((nx + 7) / 8) / (2 * ((nx + 15) / 16));
    return waves * (lanes - 0.8) <= 2.4;
}

// Whether W5CT_FP64_DW sweeps a patch in double-word arithmetic: where each
// sweep has at least two blocks of 512 faces (32 x 16 along x, 16 x 32 in the
// others) per SM.
inline bool dw_applies(int nx, int ny, int nz, int sms) {
    const long long least = 2LL * sms;
    return sweep_blocks(0, 16, 32, nx, ny, nz) >= least && sweep_blocks(1, 32, 16, nx, ny, nz) >= least &&
           sweep_blocks(2, 32, 16, nx, ny, nz) >= least;
}

template <int AX, int VAR>
cudaError_t launch_sweep_axis(const SweepArgs<float> &a, cudaStream_t s) {
    using C = SweepCfg<AX, float>;
    // (its shared memory is allowed by prepare_sweeps() at w5ct_init_grid)
    return SinglePatchSweep<AX, float, VAR, C::T2, C::MINB, C::FPT, C::BX>::launch(a, s);
}

}  // namespace w5ct
