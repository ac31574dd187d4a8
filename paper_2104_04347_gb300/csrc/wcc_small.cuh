// wcc_small.cuh -- many half-steps of a small mesh in one launch.
//
// A mesh of a few tiles keeps a few SMs busy for a few microseconds per
// half-step, and launching the next half-step, reading the device state and
// the grid-wide reduction through global memory (an atomic maximum, a fence,
// a counter, the last CTA's bookkeeping) cost as much again.  Here the tiles of
// the mesh are the CTAs of one thread-block cluster that marches up to
// kSmallSteps half-steps: the stages stay in the two stage buffers (in L2), every
// warp posts its largest speed into the shared memory of all CTAs, one
// hardware cluster barrier ends the half-step (it also makes the new stage
// visible), and every CTA derives the next dt for itself while its parents'
// loads are in flight.  At the end one thread writes the device state that the
// single half-steps would have left.
//
// A march to a time (t_stop finite, from an integer stage) ends before a half-step
// that does not fit: a pair of them at an integer stage, one at a half stage
// (wcc_step_until's rule, decided here by every CTA from the same numbers).
//
// Measured per half-step, one launch each in graphs of 32 / one cluster:
// advection P = 2 FP64, 200 cells (2 CTAs) 7.1 / 3.8 us; Euler P = 3 FP32-mixed, 2000
// cells (8 CTAs) 6.3 / 3.2 us; Euler P = 3 FP64, 2001 cells (16 CTAs) 22.7 / 19.5 us
// (its FP64 chain alone takes 15).  The rule takes the cluster wherever one holds
// the mesh, up to 16 tiles (2032 cells in FP64 and 4080 in FP32-mixed), and the
// options do not ask for the tile kernels.
#pragma once

#include "wcc_mixed2.cuh"

namespace wcc {

constexpr int kSmallCtas = 16;    // largest cluster (above 8 it needs the opt-in attribute)
constexpr int kSmallSteps = 256;  // half-steps per launch at most

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_ctas() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// All threads of all CTAs; their earlier writes (shared and global) are
// visible to the cluster afterwards.
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// *p of this CTA's shared memory, in CTA `rank` of the cluster.
__device__ __forceinline__ unsigned remote_address(const void* p, unsigned rank) {
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void store_remote(const unsigned* p, unsigned rank, unsigned v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote_address(p, rank)), "r"(v) : "memory");
}
__device__ __forceinline__ void store_remote(const unsigned long long* p, unsigned rank, unsigned long long v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(remote_address(p, rank)), "l"(v) : "memory");
}

template <int SYS, int P, bool F32>
__global__ void __launch_bounds__(kThreadsMixed) halfstep_small(const StepArgs args, int nsteps,
                                                                double t_stop) {
    static_assert(kThreadsMixed == kThreads, "one block size for both precisions");
    using Key = decltype(speed_key(std::conditional_t<F32, float, double>{}));
    constexpr int kWarps = kThreads / 32;
    constexpr int kTileCells = F32 ? kTileMixed : kTile;
    __shared__ float2 rec32[F32 ? mixed2_smem_float2<SYS, P>() : 1];
    __shared__ double rec64[F32 ? 1 : nvars(SYS) * (P + 3)][kThreads];
    __shared__ Key keys[2][kSmallCtas * kWarps];  // largest speed per warp of the cluster, by half-step parity
    const unsigned rank = cluster_rank(), ctas = cluster_ctas();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x < 2 * kSmallCtas * kWarps) (&keys[0][0])[threadIdx.x] = 0;
    cluster_sync_all();  // no CTA posts before every slot is cleared

    DevState* st = args.st;
    const bool keeper = rank == 0 && threadIdx.x == 0;
    const long long step0 = st->step;
    double t = st->t;
    unsigned err = 0u;
    StepSize z;
    int s = 0;
    // the bound of the stage that half-step s - 1 made
    auto bound_key = [&]() -> Key {
        Key k = keys[(s - 1) & 1][lane];
        const Key k2 = keys[(s - 1) & 1][lane + 32];
        return warp_max_key(k2 > k ? k2 : k);
    };
    auto value = [](Key k) -> double {
        if constexpr (F32) return (double)__uint_as_float(k);
        else return __longlong_as_double((long long)k);
    };
    Key sized_key = ~Key(0);  // the bound that z's quotients were taken from (none at first: no speed has these bits)
    int sized = -1;  // the half-step that z belongs to
    auto step = [&]() -> const StepSize& {
        if (sized == s) return z;
        sized = s;
        if (s == 0) return z = step_size(args);
        const Key k = bound_key();
        if (k == sized_key) return z;  // waves of constant speed keep their half-step
        sized_key = k;
        cfl_quotients(args.cfl, args.dx, args.inv_dx, value(k), z.dt, z.lam);
        if constexpr (F32) split_to_floats(z.lam, z.lam_hi, z.lam_lo);
        return z;
    };
    for (; s < nsteps; ++s) {
        const bool odd = s & 1;
        if (t_stop < INFINITY && !(t_stop - t >= (odd ? 1.0 : 2.0) * step().dt * (1.0 - 1e-12))) break;
        const int parity = args.parity ^ (int)odd;
        const long long n_old = odd ? args.n_new : args.n_old, n_new = odd ? args.n_old : args.n_new;
        Key key;
        if constexpr (F32) {
            const TileIO io{odd ? args.out32 : args.in32, odd ? const_cast<float*>(args.in32) : args.out32, args.pitch,
                            n_old, n_new, (long long)rank * kTileCells, parity, args.bc};
            float speed = 0.f;
            mixed_tile2<SYS, P, true, (P >= 3), true>(io, step, args, rec32, speed, err);
            if (speed != speed) {
                speed = INFINITY;
                err |= ERR_NONFINITE;
            }
            key = warp_max_key(speed_key(speed));
        } else {
            const TileIO64 io{odd ? args.out64 : args.in64, odd ? const_cast<double*>(args.in64) : args.out64, args.pitch,
                              n_old, n_new, (long long)rank * kTileCells, parity};
            double speed = 0.0;
            fp64_tile<SYS, P>(io, step, args, rec64, speed, err);
            if (speed != speed) {
                speed = INFINITY;
                err |= ERR_NONFINITE;
            }
            key = warp_max_key(speed_key(speed));
        }
        if (lane < (int)ctas) store_remote(&keys[odd][rank * kWarps + warp], lane, key);
        if (keeper) {
            if (step0 + s < args.hist_cap) args.hist[step0 + s] = z.dt;
            if (not_finite(z.dt)) err |= ERR_NONFINITE;
        }
        t = t + z.dt;
        cluster_sync_all();
    }
    err = __reduce_or_sync(0xffffffffu, err);
    if (lane == 0 && err) atomicOr(&st->err, err);
    if (s == 0) return;  // nothing fitted: the state is as it was
    const double amax = value(bound_key());
    if (keeper) {
        // what the last single half-step's bookkeeping would leave
        const int now = args.parity ^ (s & 1);
        st->amax_bits[now] = (unsigned long long)__double_as_longlong(amax);
        st->amax_bits[now ^ 1] = 0ull;
        if constexpr (F32) {
            st->amax_f32[now] = __float_as_uint((float)amax);
            st->amax_f32[now ^ 1] = 0u;
        }
        st->step = step0 + s;
        st->t = t;
        double dt, lam;
        cfl_quotients(args.cfl, args.dx, args.inv_dx, amax, dt, lam);
        st->next_dt = dt;
        st->next_lam = lam;
        if constexpr (F32) split_to_floats(lam, st->next_lam_hi, st->next_lam_lo);
        st->next_cfl = args.cfl;
    }
}

// The cluster for n new cells at most (0: too many for one).  Sizes are powers
// of two; CTAs beyond the mesh build nothing.
template <bool F32>
inline int small_ctas(long long n) {
    const long long tiles = (n + (F32 ? kTileMixed : kTile) - 1) / (F32 ? kTileMixed : kTile);
    int c = 1;
    while (c < tiles && c <= kSmallCtas) c *= 2;
    return c <= kSmallCtas ? c : 0;
}

template <int SYS, int P, bool F32>
cudaError_t launch_small_t(const StepArgs& args, int nsteps, double t_stop, int ctas, cudaStream_t stream, int* fits) {
    auto* k = halfstep_small<SYS, P, F32>;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (fits) {  // asked once per solver: can the device hold such a cluster?
        cudaError_t e = cudaSuccess;
        if (ctas > 8) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        int n = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k, &cfg);
        *fits = e == cudaSuccess ? n : 0;
        if (e != cudaSuccess) cudaGetLastError();
        return cudaSuccess;
    }
    return cudaLaunchKernelEx(&cfg, k, args, nsteps, t_stop);
}

}  // namespace wcc
