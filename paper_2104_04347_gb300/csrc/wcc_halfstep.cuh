// wcc_halfstep.cuh -- the fused half-step kernel (FP64 instantiation) and
// the small auxiliary kernels (stage CFL bound, layout conversion).
//
// One launch advances a whole stage by one staggered half-step
// (Sec. 2.1, Fig. 1).  Each CTA:
//   1. loads kThreads parent cells (coalesced: consecutive threads read
//      consecutive cells of each [var][k] plane), runs the Cauchy-Kovalewski
//      procedure once per parent, and keeps the parent record (two flux /
//      half-average contributions and the vertex Taylor coefficients) in
//      shared memory -- each parent is a vertex of two new cells;
//   2. builds kTile new cells from neighbouring records: finite-volume cell
//      average, central-difference derivatives, point value, limiter;
//   3. reduces the new stage's largest characteristic speed (warp shuffles,
//      one atomic per CTA); the last CTA to finish publishes the stage bound,
//      advances t and records dt, so the next launch derives its dt on the
//      device without a host round trip.
#pragma once

#include "wcc_pdl.cuh"
#include "wcc_scheme.cuh"

namespace wcc {

__device__ __forceinline__ long long parent_index(long long p, long long n, int bc) {
    if (bc == BC_PERIODIC) {
        if (p < 0) p += n;
        if (p >= n) p -= n;
        if (p < 0 || p >= n) p = ((p % n) + n) % n;  // tail CTAs reach past one period
        return p;
    }
    // transmissive: ghost staggered cells copy the adjacent cell
    return p < 0 ? 0 : (p >= n ? n - 1 : p);
}

template <class T>
__device__ __forceinline__ T warp_max(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Bit patterns of non-negative numbers, and the largest of a warp's.
__device__ __forceinline__ unsigned speed_key(float s) { return __float_as_uint(s); }
__device__ __forceinline__ unsigned long long speed_key(double s) {
    return (unsigned long long)__double_as_longlong(s);
}
__device__ __forceinline__ unsigned warp_max_key(unsigned k) { return __reduce_max_sync(0xffffffffu, k); }
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long k) {
    const unsigned hi = (unsigned)(k >> 32);
    const unsigned m = __reduce_max_sync(0xffffffffu, hi);
    const unsigned lo = __reduce_max_sync(0xffffffffu, hi == m ? (unsigned)k : 0u);
    return ((unsigned long long)m << 32) | lo;
}

// dt = cfl dx / amax and lam = dt / dx, rounded as the divisions, from reciprocals:
// on the serial path between half-steps a warp's FP64 instruction takes 64 cycles and a
// division nine of them.  Sizes far from 1 take the divisions.
__device__ __forceinline__ void cfl_quotients(double cfl, double dx, double inv_dx, double amax, double& dt,
                                              double& lam) {
    const double x = cfl * dx;
    if (moderate(amax) && moderate(x) && moderate(inv_dx)) {
        const d3 a(amax), t = quotient(d3(x), a, recip(a));
        dt = t.v;
        lam = quotient(t, d3(dx), d3(inv_dx)).v;
    } else {
        dt = x / amax;
        lam = dt / dx;
    }
}

// The size of the next half-step into the state.  (The FP32 kernels of one
// half-step per launch keep the divisions: the form above costs them
// registers, and two half-steps per launch at P = 2 ran 1.3 % slower.)
template <bool F32>
__device__ __forceinline__ void next_step(DevState* st, double cfl, double dx, double inv_dx, double amax) {
    double dt, lam;
    if constexpr (F32) {
        dt = cfl * dx / amax;
        lam = dt / dx;
        split_to_floats(lam, st->next_lam_hi, st->next_lam_lo);
    } else {
        cfl_quotients(cfl, dx, inv_dx, amax, dt, lam);
    }
    st->next_dt = dt;
    st->next_lam = lam;
    st->next_cfl = cfl;
}

// Bookkeeping of a solver state after the last CTA of a half-step finished:
// publish the new stage's bound, clear the slots the next launches
// accumulate into, record dt, advance t and prepare the next CFL step.
// FP32 kernels (F32) accumulate the bound in amax_f32.
template <bool F32>
__device__ __forceinline__ void finalize_state(DevState* st, double dt, double* hist, long long hist_cap,
                                               int parity, int cfl_mode, double cfl, double dx, double inv_dx) {
    if (F32) {
        const float fm = __uint_as_float(st->amax_f32[parity ^ 1]);
        st->amax_bits[parity ^ 1] = (unsigned long long)__double_as_longlong((double)fm);
        st->amax_f32[parity] = 0u;
    }
    // Every CTA of this launch has read amax_bits[parity]; clear it for the
    // launch after next, which accumulates into it.
    st->amax_bits[parity] = 0ull;
    const long long k = st->step;
    if (k < hist_cap) hist[k] = dt;
    st->step = k + 1;
    st->t = st->t + dt;
    st->blocks_done = 0u;
    if (not_finite(dt)) st->err |= ERR_NONFINITE;
    if (cfl_mode) {
        next_step<F32>(st, cfl, dx, inv_dx, __longlong_as_double((long long)st->amax_bits[parity ^ 1]));
    } else {
        st->next_cfl = 0.0;
    }
    __threadfence();
}

// Block-wide max of the speed (in the kernel's compute type T), one atomic
// per CTA into st, then count the CTA as done; the CTA that completes the
// `ctas` of this state does its bookkeeping.  Synchronises the block.
template <class T, int NT = kThreads>
__device__ __forceinline__ void reduce_and_finish(T speed, unsigned err, double dt, DevState* st, long long ctas,
                                                  double* hist, long long hist_cap, int parity, int cfl_mode,
                                                  double cfl, double dx, double inv_dx) {
    // One block barrier: the warps' maxima and error bits meet in shared
    // memory, thread 0 combines them, posts them and counts the CTA; the CTA
    // that counts last finishes the launch's bookkeeping.  The barrier also
    // guarantees that every warp is done with the tile's shared records.
    using Key = decltype(speed_key(speed));
    __shared__ Key s_max[NT / 32];
    __shared__ unsigned s_err[NT / 32];
    // NaN must win the max: map it to +Inf and flag it
    if (speed != speed) {
        speed = (T)INFINITY;
        err |= ERR_NONFINITE;
    }
    // (the bits of non-negative numbers order like the numbers: the maxima are
    // taken on the integer pipe)
    Key key = speed_key(speed);
    key = warp_max_key(key);
    err = __reduce_or_sync(0xffffffffu, err);
    if ((threadIdx.x & 31) == 0) {
        s_max[threadIdx.x >> 5] = key;
        s_err[threadIdx.x >> 5] = err;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        Key m = s_max[0];
        unsigned e = s_err[0];
#pragma unroll
        for (int w = 1; w < NT / 32; ++w) {
            m = s_max[w] > m ? s_max[w] : m;
            e |= s_err[w];
        }
        if constexpr (sizeof(T) == 8) {
            if (m) atomicMax(&st->amax_bits[parity ^ 1], m);
        } else {
            if (m) atomicMax(&st->amax_f32[parity ^ 1], m);
        }
        if (e) atomicOr(&st->err, e);
        __threadfence();
        const unsigned done = atomicAdd(&st->blocks_done, 1u);
        if (done == (unsigned)(ctas - 1)) {
            __threadfence();
            finalize_state<sizeof(T) == 4>(st, dt, hist, hist_cap, parity, cfl_mode, cfl, dx, inv_dx);
        }
    }
}
template <class T, int NT = kThreads>
__device__ __forceinline__ void finish_halfstep(T speed, unsigned err, double dt, const StepArgs& args) {
    reduce_and_finish<T, NT>(speed, err, dt, args.st, (long long)gridDim.x, args.hist, args.hist_cap, args.parity,
                             args.cfl_mode, args.cfl, args.dx, args.inv_dx);
}

// Where one FP64 tile reads and writes.
struct TileIO64 {
    const double* in64;
    double* out64;
    long long pitch;
    long long n_old;
    long long n_new;
    long long first_new;
    int parity;
};

// One tile of the FP64 half-step: kThreads parents (stage index io.first_new +
// t - parity), kTile new cells.  step() gives the half-step's size.  speed
// receives the thread's new cell's speed (unchanged outside the stage); the
// caller synchronises the block before rec is written again.
template <int SYS, int P, class Step>
__device__ __forceinline__ void fp64_tile(const TileIO64& io, Step&& step, const StepArgs& args,
                                          double (*rec)[kThreads], double& speed, unsigned& err) {
    constexpr int NV = nvars(SYS);
    constexpr int K = P + 1;
    const int t = threadIdx.x;

    // ---- phase 1: parent record of parent slot t
    {
        const long long p = parent_index(io.first_new + t - (io.parity ? 1 : 0), io.n_old, args.bc);
        d3 c[NV][K];
        sfor<0, NV>([&](auto V) {
            constexpr int v = decltype(V)::value;
            sfor<0, K>([&](auto Ki) {
                constexpr int k = decltype(Ki)::value;
                c[v][k] = d3::reg(io.in64[(long long)(v * K + k) * io.pitch + p]);
            });
        });
        const StepSize& z = step();  // after the parents' loads have been issued
        ParentRecord<SYS, P, d3> r;
        parent_record<SYS, P>(c, d3(z.lam), args, r);
        sfor<0, NV>([&](auto V) {
            constexpr int v = decltype(V)::value;
            rec[v][t] = r.A[v].v;
            rec[NV + v][t] = r.B[v].v;
            sfor<0, K>([&](auto Ki) {
                constexpr int k = decltype(Ki)::value;
                rec[2 * NV + v * K + k][t] = r.vtx[v][k].v;
            });
        });
    }
    __syncthreads();

    // ---- phase 2: new cell t from parent slots t (left) and t + 1 (right)
    const long long i = io.first_new + t;
    if (t < kTile && i < io.n_new) {
        d3 e[NV][K], ubar[NV], vl[NV], vr[NV];
        sfor<0, NV>([&](auto V) {
            constexpr int v = decltype(V)::value;
            d3 vL[K], vR[K];
            sfor<0, K>([&](auto Ki) {
                constexpr int k = decltype(Ki)::value;
                vL[k] = d3::reg(rec[2 * NV + v * K + k][t]);
                vR[k] = d3::reg(rec[2 * NV + v * K + k][t + 1]);
            });
            ubar[v] = d3::reg(rec[v][t]) + d3::reg(rec[NV + v][t + 1]);
            vl[v] = vL[0];
            vr[v] = vR[0];
            derivatives_and_point_value<P, d3>(ubar[v], vL, vR, e[v]);
        });

        if (args.limiter) {
            if constexpr (NV == 1) {
                limit_scalar<P, SCALAR>(e[0], ubar[0], vl[0], vr[0], args);
            } else {
                // Sec. 4: limit characteristic variables L(ubar) U, map back with R(ubar).
                EulerChar<d3> E;
                if (!euler_char<d3>(ubar, d3(args.gamma), E)) err |= ERR_POSITIVITY;
                d3 ce[3][K], cub[3], cvl[3], cvr[3];
                E.left(ubar[0], ubar[1], ubar[2], cub);
                E.left(vl[0], vl[1], vl[2], cvl);
                E.left(vr[0], vr[1], vr[2], cvr);
                sfor<0, K>([&](auto Ki) {
                    constexpr int k = decltype(Ki)::value;
                    d3 w[3];
                    E.left(e[0][k], e[1][k], e[2][k], w);
                    ce[0][k] = w[0];
                    ce[1][k] = w[1];
                    ce[2][k] = w[2];
                });
                limit_scalar<P, CHARACTERISTIC>(ce[0], cub[0], cvl[0], cvr[0], args);
                limit_scalar<P, CHARACTERISTIC>(ce[1], cub[1], cvl[1], cvr[1], args);
                const d3 w0 = limit_scalar<P, LAST_CHARACTERISTIC>(ce[2], cub[2], cvl[2], cvr[2], args);
                sfor<0, K>([&](auto Ki) {
                    constexpr int k = decltype(Ki)::value;
                    if constexpr (k < 2) E.right(ce[0][k], ce[1][k], ce[2][k], e[0][k], e[1][k], e[2][k]);
                    else E.right_scaled(ce[0][k], ce[1][k], w0, ce[2][k], e[0][k], e[1][k], e[2][k]);
                });
            }
        }

        bool bad = false;
        sfor<0, NV>([&](auto V) {
            constexpr int v = decltype(V)::value;
            sfor<0, K>([&](auto Ki) {
                constexpr int k = decltype(Ki)::value;
                bad |= not_finite(e[v][k]);
                __stcs(io.out64 + (long long)(v * K + k) * io.pitch + i, e[v][k].v);
            });
        });
        if (bad) err |= ERR_NONFINITE;
        d3 u0[NV];
        sfor<0, NV>([&](auto V) { u0[decltype(V)::value] = e[decltype(V)::value][0]; });
        speed = wave_speed<SYS, d3>(u0, args, err).v;
    }
}

template <int SYS, int P>
__global__ void __launch_bounds__(kThreads) halfstep_fp64(const StepArgs args) {
    __shared__ double rec[nvars(SYS) * (P + 3)][kThreads];
    pdl_begin();
    const TileIO64 io{args.in64, args.out64, args.pitch, args.n_old, args.n_new,
                      (long long)blockIdx.x * kTile, args.parity};
    StepSize z;
    double speed = 0.0;
    unsigned err = 0u;
    fp64_tile<SYS, P>(io, [&]() -> const StepSize& { return z = step_size(args); }, args, rec, speed, err);
    finish_halfstep<double>(speed, err, z.dt, args);
}

// Largest characteristic speed of a stage (used once after loading data).
template <int SYS>
__global__ void __launch_bounds__(256) stage_speed(const double* u0planes, long long var_stride, long long n,
                                                    StepArgs args, int slot) {
    constexpr int NV = nvars(SYS);
    double m = 0.0;
    unsigned err = 0u;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        d3 u0[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) u0[v] = d3::reg(u0planes[v * var_stride + i]);
        double s = wave_speed<SYS, d3>(u0, args, err).v;
        if (s != s) {
            s = __longlong_as_double(0x7ff0000000000000ll);
            err |= ERR_NONFINITE;
        }
        m = fmax(m, s);
    }
    m = warp_max<double>(m);
    if ((threadIdx.x & 31) == 0 && m > 0.0)
        atomicMax(&args.st->amax_bits[slot], (unsigned long long)__double_as_longlong(m));
    if (err) atomicOr(&args.st->err, err);
}

}  // namespace wcc
