// wcc2d_kernels.cuh -- kernels of the 2D WCC path: the fused half-step, the
// CFL rate of a loaded stage, and the conversions between the host layout
// [row][col][var][q] (FP64) and the device planes.
//
// Device layout: plane (v, q) holds the Taylor coefficient e_kl = u_{kx,ly} /
// (k! l!) of variable v (q = position of (k, l); FP64: of (3, 0) and (0, 3) the
// derivative itself, see kept) for every cell, row-major with `pitch` elements per
// row; planes are `plane` elements apart.  T is double (FP64 path) or float (FP32
// path).
//
// The half-step kernel runs one CTA of TW threads per strip of TW - 1 new
// columns and `rows_per_cta` new rows.  It marches up the strip: each step
// computes the Cauchy-Kovalewski expansion and Appendix-B terms of one row of
// TW parents (thread t: parent column t of the strip) into a two-row ring
// in shared memory; the new cells between the previous parent row and this
// one then read their four parents from the ring (thread t: new cell between
// parent columns t and t + 1).  Every parent is expanded once per strip; the
// first parent row of a strip is also expanded by the strip below.
#pragma once

#include <algorithm>

#include "wcc2d_scheme.cuh"
#include "wcc_convert.cuh"
#include "wcc_halfstep.cuh"
#include "wcc_pdl.cuh"

namespace wcc2d {

struct DevState2D {
    // rate_bits[s]: max over the stage of parity s of s_x/dx + s_y/dy at
    // the cell centres, as the bit pattern of a non-negative double
    unsigned long long rate_bits[2];
    double t;
    long long step;
    unsigned int blocks_done;
    unsigned int err;  // ERR_* bits, sticky
};

struct Step2D {
    const void* in;
    void* out;
    long long pitch, plane;
    long long rows_alloc;  // rows of a plane
    int nx_old, ny_old, nx_new, ny_new;
    int parity, bc, rows_per_cta;
    double dx, dy;
    double inv_dx, inv_dy;  // 1 / dx, 1 / dy (host)
    double dt_given;  // > 0: the half-step size; otherwise cfl / rate of the old stage
    double cfl;
    Law2D law;
    DevState2D* st;
    double* hist;
    long long hist_cap;
    int strip;      // FP64: threads per CTA, 32 or 0 (the degree's full width, strip_width)
    int* resident;  // host: not null asks for the kernel's resident CTAs per SM instead of a launch
};

__device__ __forceinline__ int parent_index(int j, int n_old, int bc) {
    if (bc == PERIODIC) {
        // one wrap covers every index a strip touches on meshes wider than
        // the strip; the remainder is for the narrow ones
        if (j >= -n_old && j < 2 * n_old) return j < 0 ? j + n_old : (j >= n_old ? j - n_old : j);
        j %= n_old;
        return j < 0 ? j + n_old : j;
    }
    return j < 0 ? 0 : (j > n_old - 1 ? n_old - 1 : j);
}

// Compute type of a stage type, and values between the two.
template <class T>
using compute_t = std::conditional_t<sizeof(T) == 8, d3, float>;
__device__ __forceinline__ float from_memory(float x) { return x; }
__device__ __forceinline__ d3 from_memory(double x) { return d3::reg(x); }
__device__ __forceinline__ float to_memory(float x) { return x; }
__device__ __forceinline__ double to_memory(d3 x) { return x.v; }

// Reads parent records from the ring: vertex r = 0..3 is parent column t
// (r = 0, 3) or t + 1 (r = 1, 2) of the lower (r = 0, 1) or upper row.
template <class T, int TW, int NV, int NQ1>
struct RingReader {
    using R = compute_t<T>;
    const T* lo;
    const T* hi;
    int t;
    __device__ __forceinline__ R get(int r, int f) const {
        return from_memory(r == 0 ? lo[f * TW + t] : r == 1 ? lo[f * TW + t + 1] : r == 2 ? hi[f * TW + t + 1]
                                                                                       : hi[f * TW + t]);
    }
    __device__ __forceinline__ R c(int r, int v) const { return get(r, v * 4 + r); }
    __device__ __forceinline__ R V(int r, int v, int q) const { return get(r, NV * 4 + v * NQ1 + q); }
};

template <int SYS, int P>
__host__ __device__ constexpr int record_fields() {
    return nvars(SYS) * (4 + nq(P - 1));
}

template <class T, int TW>
__host__ __device__ constexpr size_t ring_bytes(int fields) {
    return 2 * (size_t)fields * TW * sizeof(T);
}

// The half-step size: dt_given, or cfl over the rate of the old stage.  One
// thread takes the FP64 division and shares it (block barrier).
__device__ __forceinline__ double step_dt2d(const Step2D& a) {
    __shared__ double s_dt;
    if (threadIdx.x == 0) {
        double dt = a.dt_given;
        if (!(dt > 0.0)) dt = a.cfl / __longlong_as_double((long long)a.st->rate_bits[a.parity]);
        s_dt = dt;
    }
    __syncthreads();
    return s_dt;
}

// Block-wide max of the rate (on the bits of the non-negative numbers) and OR
// of the error bits, one atomic each per CTA; the CTA that finishes last does
// the half-step's bookkeeping.
template <class T, int NT>
__device__ __forceinline__ void finish2d(T rate, unsigned err, double dt, const Step2D& a) {
    using Key = decltype(wcc::speed_key(rate));
    __shared__ Key s_max[NT / 32];
    __shared__ unsigned s_err[NT / 32];
    if (rate != rate) {
        rate = (T)INFINITY;
        err |= ERR_NONFINITE;
    }
    const Key key = wcc::warp_max_key(wcc::speed_key(rate));
    err = __reduce_or_sync(0xffffffffu, err);
    if ((threadIdx.x & 31) == 0) {
        s_max[threadIdx.x >> 5] = key;
        s_err[threadIdx.x >> 5] = err;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        Key mk = s_max[0];
        unsigned e = s_err[0];
#pragma unroll
        for (int w = 1; w < NT / 32; ++w) {
            mk = s_max[w] > mk ? s_max[w] : mk;
            e |= s_err[w];
        }
        double m;
        if constexpr (sizeof(T) == 8) m = __longlong_as_double((long long)mk);
        else m = (double)__uint_as_float(mk);
        DevState2D* st = a.st;
        atomicMax(&st->rate_bits[a.parity ^ 1], (unsigned long long)__double_as_longlong(m));
        if (e) atomicOr(&st->err, e);
        __threadfence();
        const unsigned total = gridDim.x * gridDim.y;
        const unsigned done = atomicAdd(&st->blocks_done, 1u);
        if (done == total - 1) {
            __threadfence();
            // every CTA has read rate_bits[parity]; clear it for the launch after next
            st->rate_bits[a.parity] = 0ull;
            const long long k = st->step;
            if (k < a.hist_cap) a.hist[k] = dt;
            st->step = k + 1;
            st->t = st->t + dt;
            st->blocks_done = 0u;
            if (!(dt > 0.0) || dt == INFINITY) st->err |= ERR_NONFINITE;
            __threadfence();
        }
    }
}

// Resident CTAs the FP32 kernels are compiled for (caps their registers at
// 65536 / (4 x TW)); FP64 kernels are bound by the FP64 pipe and keep their
// registers.
template <class T>
constexpr int min_ctas2d() {
    return sizeof(T) == 4 ? 4 : 1;
}

// The FP64 kernel is bound by the FP64 pipe: Euler P = 3 issues about 2020 FP64
// instructions per cell, all three-register DFMAs (about 3000 of every form in
// the derivative form with the compiler's divisions): 192 x 192 0.42 -> 0.27 ms per
// half-step.  The FP32 kernels are bound by issue and dependency latency at 12 to
// 16 warps per SM.
template <int SYS, int P, class T, int TW>
__global__ void __launch_bounds__(TW, min_ctas2d<T>()) halfstep2d(const Step2D a) {
    constexpr int NV = nvars(SYS), NQ = nq(P), NQ1 = nq(P - 1);
    constexpr int NF = record_fields<SYS, P>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* ring = reinterpret_cast<T*>(smem_raw);  // [2][NF][TW]

    const int t = threadIdx.x;
    const int off = a.parity ? -1 : 0;
    const int i0 = blockIdx.x * (TW - 1);
    const int j0 = blockIdx.y * a.rows_per_cta;
    const int rows = min(a.rows_per_cta, a.ny_new - j0);

    wcc::pdl_begin();
    const double dt = step_dt2d(a);
    using R = compute_t<T>;
    const R lamx = (R)(dt * a.inv_dx), lamy = (R)(dt * a.inv_dy);
    const R idx = (R)a.inv_dx, idy = (R)a.inv_dy;

    const T* in = static_cast<const T*>(a.in);
    T* out = static_cast<T*>(a.out);
    const int pc = parent_index(i0 + t + off, a.nx_old, a.bc);
    T rate_max = 0;
    unsigned err = 0;

    for (int s = 0; s <= rows; ++s) {
        {
            const int pr = parent_index(j0 + off + s, a.ny_old, a.bc);
            long long cell = (long long)pr * a.pitch + pc;
#ifdef WCC2D_BOUNDS_CHECK
            // opt-in checked build: an out-of-range parent is recorded and cell 0 read instead
            if (pr < 0 || pr >= a.rows_alloc || pc < 0 || pc >= a.pitch) {
                atomicOr(&a.st->err, ERR_BOUNDS);
                cell = 0;
            }
#endif
            R q[NV][NQ];
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int qq = 0; qq < NQ; ++qq) q[v][qq] = from_memory(in[(long long)(v * NQ + qq) * a.plane + cell]);
            Parent<SYS, P, R> par;
            parent_terms<SYS, P, R>(q, lamx, lamy, a.law, par);
            T* r = ring + (s & 1) * NF * TW;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
#pragma unroll
                for (int k = 0; k < 4; ++k) r[(v * 4 + k) * TW + t] = to_memory(par.c[v][k]);
#pragma unroll
                for (int qq = 0; qq < NQ1; ++qq) r[(NV * 4 + v * NQ1 + qq) * TW + t] = to_memory(par.V[v][qq]);
            }
        }
        __syncthreads();
        if (s >= 1 && t < TW - 1 && i0 + t < a.nx_new) {
            const RingReader<T, TW, NV, NQ1> rd{ring + ((s - 1) & 1) * NF * TW, ring + (s & 1) * NF * TW, t};
            // FP64 Euler: the first derivatives after the projection (limit_euler)
            constexpr bool kLate = SYS == EULER && sizeof(T) == 8;
            R D[NV][NQ], ub[NV], vv[NV][4];
            linear_cell<SYS, P, kLate ? 2 : 1, R>(rd, D, ub);
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int r = 0; r < 4; ++r) vv[v][r] = rd.V(r, v, 0) - ub[v];
            bool limited = false;
            if (a.law.limiter) {
                if constexpr (SYS == EULER) {
                    limited = limit_euler<P, R>(D, ub, vv, lamx, lamy, a.law);
                    if (!limited) err |= ERR_POSITIVITY;
                } else {
                    limit_scalar<P, R>(D[0], vv[0], a.law, ub[0]);
                }
            }
            if constexpr (kLate) {
                if (!limited) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) first_derivatives<P, R>(D[v], vv[v]);
                }
            }
            // the limiter keeps the cell average (every candidate has mean ubar)
#pragma unroll
            for (int v = 0; v < NV; ++v) D[v][0] = ub[v] - even_correction<P, R>(D[v]);
            const long long cell = (long long)(j0 + s - 1) * a.pitch + (i0 + t);
            bool store = true;
#ifdef WCC2D_BOUNDS_CHECK
            if (j0 + s - 1 >= a.rows_alloc || i0 + t >= a.pitch) {  // recorded, not written
                atomicOr(&a.st->err, ERR_BOUNDS);
                store = false;
            }
#endif
            if (store) {
#pragma unroll
                for (int v = 0; v < NV; ++v)
#pragma unroll
                    for (int qq = 0; qq < NQ; ++qq) out[(long long)(v * NQ + qq) * a.plane + cell] = to_memory(D[v][qq]);
            }
            R centre[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) centre[v] = D[v][0];
            const R rate = cfl_rate<SYS, R>(centre, a.law, idx, idy);
            if (is_nan(rate)) {
                err |= (SYS == EULER && !is_nan(ub[0])) ? ERR_POSITIVITY : ERR_NONFINITE;
                rate_max = (T)INFINITY;
            } else {
                const T r = to_memory(rate);
                rate_max = wcc::speed_key(r) > wcc::speed_key(rate_max) ? r : rate_max;
            }
        }
        __syncthreads();
    }
    finish2d<T, TW>(rate_max, err, dt, a);
}

// A warp's largest CFL rate of a loaded stage into rate_bits[0] (and the error bits).
__device__ __forceinline__ void post_rate(double r, unsigned err, DevState2D* st) {
    const unsigned long long key = wcc::warp_max_key(wcc::speed_key(r));
    err = __reduce_or_sync(0xffffffffu, err);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&st->rate_bits[0], key);
        if (err) atomicOr(&st->err, err);
    }
}

// CFL rate of a loaded stage into rate_bits[0] (and the error bits).
template <int SYS, class T>
__global__ void __launch_bounds__(256) stage_rate2d(const T* planes, long long pitch, long long plane, int nx, int ny,
                                                    int nq_, Law2D law, double dx, double dy, DevState2D* st) {
    constexpr int NV = nvars(SYS);
    using R = compute_t<T>;
    T m = 0;
    unsigned err = 0;
    const long long n = (long long)nx * ny;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
        const long long cell = (c / nx) * pitch + (c % nx);
        R centre[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) centre[v] = from_memory(planes[(long long)(v * nq_) * plane + cell]);
        const R r = cfl_rate<SYS, R>(centre, law, (R)(1.0 / dx), (R)(1.0 / dy));
        if (is_nan(r)) {
            err |= SYS == EULER ? ERR_POSITIVITY : ERR_NONFINITE;
            m = (T)INFINITY;
        } else if (to_memory(r) > m) {
            m = to_memory(r);
        }
    }
    post_rate((double)m, err, st);
}

// Conversions between the host layout [row][col][v][q] (FP64 scaled derivatives,
// in a staging buffer) and the planes.  A CTA takes kConvCells cells of a row:
// its host-layout side is one run of doubles, its plane side a run per plane,
// and the transposition goes through shared memory, so that both sides move
// whole sectors.  (One thread per cell, stepping through its cell's doubles:
// 158 us to the planes and 527 us back at 1024 x 1024, FP32-mixed, P = 3; about
// 110 and 190 us this way.)
// FP32 coefficients are converted on the FP32 and integer pipes (wcc_convert.cuh);
// what joins the FP32-mixed average and the point value is summed in FP64.
constexpr int kConvCells = 64, kConvThreads = 256;

// 1/(k! l!) and k! l! of position q
__host__ __device__ constexpr double fact_q(int q) { return factd(qk_of(q)) * factd(ql_of(q)); }

// One variable of one cell, d its scaled derivatives (bit patterns), put(plane, x):
// FP64 (T = double), FP32 point values, or FP32-mixed (cell average as a
// float-float pair in planes 0 and -1).
template <int P, bool MX, class T, class Put>
__device__ __forceinline__ void variable_to_planes(const unsigned long long* d, Put&& put) {
    if constexpr (sizeof(T) == 8) {
        unroll<nq(P)>([&](auto qc) {
            constexpr double w = kept<d3>(qc) / fact_q(qc);
            const double x = __longlong_as_double((long long)d[qc]);
            put(qc, w == 1.0 ? x : x * w);
        });
    } else {
        ff e[nq(P)];
        unroll<nq(P)>([&](auto qc) {
            constexpr wcc::ffc w = wcc::ffc_of(1.0 / fact_q(qc));
            e[qc] = wcc::split_double_bits(d[qc]);
            if constexpr (fact_q(qc) != 1.0) e[qc] = wcc::ff_mul_c(e[qc], w);
            else e[qc] = wcc::fast_two_sum(e[qc].hi, e[qc].lo);
        });
        if constexpr (MX) {
            double u = __longlong_as_double((long long)d[0]);
            if constexpr (P >= 2) {
                u = ::fma(1.0 / 24.0, __longlong_as_double((long long)d[qidx(0, 2)]), u);
                u = ::fma(1.0 / 24.0, __longlong_as_double((long long)d[qidx(2, 0)]), u);
            }
            float hi, lo;
            wcc::split_double(u, hi, lo);
            put(0, hi);
            put(-1, lo);
        } else {
            put(0, e[0].hi);
        }
        unroll<nq(P) - 1>([&](auto qc) { put(qc + 1, e[qc + 1].hi); });
    }
}

// The way back: get(plane) reads, d receives the scaled derivatives.
template <int P, bool MX, class T, class Get>
__device__ __forceinline__ void planes_to_variable(Get&& get, unsigned long long* d) {
    if constexpr (sizeof(T) == 8) {
        unroll<nq(P)>([&](auto qc) {
            constexpr double w = fact_q(qc) / kept<d3>(qc);
            const double x = get(qc);
            d[qc] = (unsigned long long)__double_as_longlong(w == 1.0 ? x : x * w);
        });
    } else {
        float e[nq(P)];
        unroll<nq(P) - 1>([&](auto qc) {
            constexpr int i = qc + 1;
            e[i] = get(i);
            d[i] = wcc::float_times_exact<(unsigned)fact_q(i)>(e[i]);
        });
        if constexpr (MX) {
            double u = __longlong_as_double((long long)wcc::float_times_exact<1>(get(0))) +
                       __longlong_as_double((long long)wcc::float_times_exact<1>(get(-1)));
            if constexpr (P >= 2) {
                u = ::fma(-1.0 / 24.0, __longlong_as_double((long long)d[qidx(0, 2)]), u);
                u = ::fma(-1.0 / 24.0, __longlong_as_double((long long)d[qidx(2, 0)]), u);
            }
            d[0] = (unsigned long long)__double_as_longlong(u);
        } else {
            d[0] = wcc::float_times_exact<1>(get(0));
        }
    }
}

template <int P, bool MX, class T, bool TO_PLANES>
__global__ void __launch_bounds__(kConvThreads) convert2d(double* aos, T* planes, int nx, int ny, int nv,
                                                          long long pitch, long long plane) {
    constexpr int NQ = nq(P), MAXROW = 4 * NQ;
    __shared__ unsigned long long sm[kConvCells * (MAXROW | 1)];  // odd row length: no bank conflicts
    const int nd = nv * NQ, row = nd | 1;
    const int tiles_x = (nx + kConvCells - 1) / kConvCells;
    const long long tiles = (long long)tiles_x * ny;
    unsigned long long* host = reinterpret_cast<unsigned long long*>(aos);
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int j = (int)(tile / tiles_x), i0 = (int)(tile % tiles_x) * kConvCells;
        const int cnt = min(kConvCells, nx - i0);
        unsigned long long* run = host + ((long long)j * nx + i0) * nd;
        if constexpr (TO_PLANES) {
            for (int i = threadIdx.x; i < cnt * nd; i += kConvThreads) sm[(i / nd) * row + i % nd] = run[i];
            __syncthreads();
        }
        for (int i = threadIdx.x; i < kConvCells * nv; i += kConvThreads) {
            const int c = i % kConvCells, v = i / kConvCells;
            if (c >= cnt) continue;
            T* p = planes + (long long)j * pitch + i0 + c;
            auto at = [&](int qq) -> T& { return p[(long long)(qq < 0 ? nv * NQ + v : v * NQ + qq) * plane]; };
            unsigned long long* d = sm + c * row + v * NQ;
            if constexpr (TO_PLANES) variable_to_planes<P, MX, T>(d, [&](int qq, T x) { at(qq) = x; });
            else planes_to_variable<P, MX, T>([&](int qq) { return at(qq); }, d);
        }
        __syncthreads();
        if constexpr (!TO_PLANES) {
            for (int i = threadIdx.x; i < cnt * nd; i += kConvThreads) run[i] = sm[(i / nd) * row + i % nd];
            __syncthreads();
        }
    }
}

template <int P, bool MX, class T>
cudaError_t launch_convert2d_t(bool to_planes, double* aos, void* planes, int nx, int ny, int nv, long long pitch,
                               long long plane, cudaStream_t stream) {
    const long long tiles = (long long)((nx + kConvCells - 1) / kConvCells) * ny;
    const int grid = (int)std::min<long long>(tiles, 152LL * 8);
    if (to_planes)
        convert2d<P, MX, T, true><<<grid, kConvThreads, 0, stream>>>(aos, static_cast<T*>(planes), nx, ny, nv, pitch, plane);
    else
        convert2d<P, MX, T, false><<<grid, kConvThreads, 0, stream>>>(aos, static_cast<T*>(planes), nx, ny, nv, pitch, plane);
    return cudaGetLastError();
}

// CTA width of the half-step: 64 threads for FP64, 128 for FP32, narrowed
// in steps of one warp until the shared ring fits in the 48 KB a kernel gets
// without the opt-in attribute (Euler at P = 3: 32 for FP64, 96 for FP32).
template <int SYS, int P, class T>
constexpr int strip_width() {
    int tw = sizeof(T) == 8 ? 64 : 128;
    while (tw > 32 && ring_bytes<T, 1>(record_fields<SYS, P>()) * tw > 48 * 1024 - 256) tw -= 32;
    return tw;
}

// Strip height and width (0: full) of a half-step.
struct StripPlan {
    int rows, strip;
};

// Strip height for a mesh, from a model of the time: a CTA marches rows + 1
// parent rows and rows new rows, about equally dear (2 rows + 1 units), and
// the CTAs run in waves of `slots`, so the time goes as
// ceil(CTAs / slots) (2 rows + 1).  The minimum over the heights trades the
// parent row that neighbouring strips both expand against SMs left idle.
// FP32: slots are the resident CTAs.  Measured (FP32-mixed Euler, P = 3):
// 1024 x 1024 0.259 ms at 16 rows (704 CTAs on 608 slots, two waves) against
// 0.200 ms at the 19 rows this picks (594 CTAs, one wave); sweeps of the
// height at 400, 700 and 1024 cells a side found nothing faster than its pick.
// FP64: a warp's FP64 instruction takes its scheduler's share of the pipe for
// 64 cycles whatever else runs, so the slots are the 4 schedulers per SM and
// the unit is the warp; strips of one warp are taken where they shorten the
// longest chain (192 x 192 Euler, P = 3: 48 CTAs of 64 threads and 16 rows
// 1.87 ms, 455 of 32 threads and 3 rows 0.42 ms with the same arithmetic).
inline StripPlan plan_strips(int tw, bool fp64, int resident, int sms, int nx_new, int ny_new) {
    StripPlan best{16, 0};
    double best_cost = 1e300;
    for (int width = tw; width >= 32; width = width > 32 && fp64 ? 32 : 0) {
        const long long strips = (nx_new + width - 2) / (width - 1);
        for (int rows = 48; rows >= 1; --rows) {
            if (rows > ny_new) continue;
            long long units = strips * ((ny_new + rows - 1) / rows);
            if (fp64) units *= width / 32;
            const long long slots = (long long)sms * (fp64 ? 4 : resident);
            const double cost = (double)((units + slots - 1) / slots) * (2 * rows + 1);
            if (cost < best_cost) {
                best_cost = cost;
                best = StripPlan{rows, width == tw ? 0 : width};
            }
        }
    }
    return best;
}

template <int SYS, int P, class T, int TW>
cudaError_t launch_strips2d(const Step2D& a, cudaStream_t stream) {
    constexpr size_t smem = ring_bytes<T, TW>(record_fields<SYS, P>());
    static_assert(smem <= 48 * 1024 - 256, "the shared ring and the static shared words must fit without the opt-in attribute");
    if (a.resident) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(a.resident, halfstep2d<SYS, P, T, TW>, TW, smem);
    const dim3 grid((a.nx_new + TW - 2) / (TW - 1), (a.ny_new + a.rows_per_cta - 1) / a.rows_per_cta);
    return wcc::launch_pdl<Step2D>(halfstep2d<SYS, P, T, TW>, grid, TW, smem, stream, a);
}

// Launch one half-step of system SYS at degree P in type T.
template <int SYS, int P, class T>
cudaError_t launch_halfstep2d_t(const Step2D& a, cudaStream_t stream) {
    if constexpr (sizeof(T) == 8) {
        if (a.strip == 32) return launch_strips2d<SYS, P, T, 32>(a, stream);
    }
    return launch_strips2d<SYS, P, T, strip_width<SYS, P, T>()>(a, stream);
}

template <int SYS, class T>
cudaError_t launch_halfstep2d_sys(int P, const Step2D& a, cudaStream_t stream) {
    switch (P) {
        case 1: return launch_halfstep2d_t<SYS, 1, T>(a, stream);
        case 2: return launch_halfstep2d_t<SYS, 2, T>(a, stream);
        case 3: return launch_halfstep2d_t<SYS, 3, T>(a, stream);
        default: return cudaErrorInvalidValue;
    }
}

template <int SYS>
cudaError_t launch_stage_rate2d_sys(bool fp32, const void* planes, long long pitch, long long plane, int nx, int ny,
                                    int nq_, const Law2D& law, double dx, double dy, DevState2D* st,
                                    cudaStream_t stream) {
    const long long n = (long long)nx * ny;
    const int grid = (int)std::min<long long>((n + 255) / 256, 152 * 8);
    if (fp32)
        stage_rate2d<SYS, float><<<grid, 256, 0, stream>>>(static_cast<const float*>(planes), pitch, plane, nx, ny,
                                                           nq_, law, dx, dy, st);
    else
        stage_rate2d<SYS, double><<<grid, 256, 0, stream>>>(static_cast<const double*>(planes), pitch, plane, nx,
                                                            ny, nq_, law, dx, dy, st);
    return cudaGetLastError();
}

// --------------------------------------------------------- FP32-mixed kernel

// Stage layout of the FP32-mixed path: plane (v, 0) holds the high part of
// the cell average (not the point value), planes (v, q >= 1) the scaled
// derivatives in float, and plane NV * NQ + v the low part of the average.
// A parent record: per variable its four shares of the children's averages
// and its vertex point value at t^{n+1/2}, float-float pairs stored as
// float2 (pair field v * 4 + k for share k, NV * 4 + v for the vertex value),
// then the vertex derivatives q = 1 .. NQ1 - 1 (float, from float offset
// 10 NV of the record).
template <int SYS, int P>
__host__ __device__ constexpr int record_fields_mx() {
    return nvars(SYS) * (10 + nq(P - 1) - 1);
}


template <int SYS, int P>
constexpr int strip_width_mx() {
    int tw = 128;
    while (tw > 32 && ring_bytes<float, 1>(record_fields_mx<SYS, P>()) * tw > 48 * 1024 - 256) tw -= 32;
    return tw;
}

// Threads per CTA of a kernel's full-width strips (host).
inline int strip_threads(int system, int P, bool fp32, bool mixed) {
    auto width = [&](auto sys) {
        constexpr int S = decltype(sys)::value;
        auto at = [&](auto pc) {
            constexpr int Q = decltype(pc)::value;
            return mixed ? strip_width_mx<S, Q>() : fp32 ? strip_width<S, Q, float>() : strip_width<S, Q, double>();
        };
        return P == 1 ? at(std::integral_constant<int, 1>{}) : P == 2 ? at(std::integral_constant<int, 2>{})
                                                                      : at(std::integral_constant<int, 3>{});
    };
    return system == EULER ? width(std::integral_constant<int, EULER>{}) : width(std::integral_constant<int, ADVECTION>{});
}

template <int TW, int NV, int NQ1>
struct RingReaderMx {
    const float* lo;
    const float* hi;
    int t;
    __device__ __forceinline__ float get(int r, int f) const {
        return r == 0 ? lo[f * TW + t] : r == 1 ? lo[f * TW + t + 1] : r == 2 ? hi[f * TW + t + 1] : hi[f * TW + t];
    }
    __device__ __forceinline__ ff get2(int r, int pf) const {
        const float2* l2 = reinterpret_cast<const float2*>(lo);
        const float2* h2 = reinterpret_cast<const float2*>(hi);
        const float2 x = r == 0 ? l2[pf * TW + t] : r == 1 ? l2[pf * TW + t + 1] : r == 2 ? h2[pf * TW + t + 1] : h2[pf * TW + t];
        return ff{x.x, x.y};
    }
    __device__ __forceinline__ ff cf(int r, int v) const { return get2(r, v * 4 + r); }
    __device__ __forceinline__ ff v00(int r, int v) const { return get2(r, NV * 4 + v); }
    __device__ __forceinline__ float V(int r, int v, int q) const {
        return q == 0 ? get2(r, NV * 4 + v).hi : get(r, NV * 10 + v * (NQ1 - 1) + q - 1);
    }
};

// Bound by instruction issue (12 warps per SM: 168 registers and the 46 KB ring);
// Cauchy products without binomial weights, edge fluxes by parity, two
// residuals instead of four and float constants took Euler P = 3 at 1024 x 1024
// from 0.200 to 0.167 ms per half-step.
template <int SYS, int P, int TW>
__global__ void __launch_bounds__(TW, 4) halfstep2d_mx(const Step2D a) {
    constexpr int NV = nvars(SYS), NQ = nq(P), NQ1 = nq(P - 1);
    constexpr int NF = record_fields_mx<SYS, P>();
    static_assert((NF * TW) % 2 == 0, "the second row buffer of the ring must start on an 8-byte boundary");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* ring = reinterpret_cast<float*>(smem_raw);  // [2][NF][TW]

    const int t = threadIdx.x;
    const int off = a.parity ? -1 : 0;
    const int i0 = blockIdx.x * (TW - 1);
    const int j0 = blockIdx.y * a.rows_per_cta;
    const int rows = min(a.rows_per_cta, a.ny_new - j0);

    wcc::pdl_begin();
    const double dt = step_dt2d(a);
    // lam rounded to float in every term, the leading flux terms included:
    // the half-step is one of size fl(lam) dx, the same in all its Taylor
    // terms (a float-float lam for the leading terms alone was measured to
    // move the fine-mesh errors away from FP64's, not towards them)
    const float lamx = (float)(dt * a.inv_dx), lamy = (float)(dt * a.inv_dy);
    const float hx = 0.5f * lamx, hy = 0.5f * lamy;
    const float idx = (float)a.inv_dx, idy = (float)a.inv_dy;

    const float* in = static_cast<const float*>(a.in);
    float* out = static_cast<float*>(a.out);
    const int pc = parent_index(i0 + t + off, a.nx_old, a.bc);
    float rate_max = 0.f;
    unsigned err = 0;

    for (int s = 0; s <= rows; ++s) {
        {
            const int pr = parent_index(j0 + off + s, a.ny_old, a.bc);
            const long long cell = (long long)pr * a.pitch + pc;
            float q[NV][NQ];
            ff ub[NV], u00[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                ub[v] = ff{in[(long long)(v * NQ) * a.plane + cell], in[(long long)(NV * NQ + v) * a.plane + cell]};
                q[v][0] = 0.f;
#pragma unroll
                for (int qq = 1; qq < NQ; ++qq) q[v][qq] = in[(long long)(v * NQ + qq) * a.plane + cell];
                u00[v] = wcc::ff_add(ub[v], -even_correction<P, float>(q[v]));
                q[v][0] = u00[v].hi;
            }
            Parent<SYS, P, float, true> par;
            parent_terms<SYS, P, float, true>(q, lamx, lamy, a.law, par);
            ff F[NV], G[NV];
            lead_flux_ff<SYS>(u00, a.law, F, G);
            float* r = ring + (s & 1) * NF * TW;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                // the shares a +- p +- q +- r with a = ubar/4 and the leading
                // flux terms hx f(u_00) in p, hy g(u_00) in q:
                // the O(1) parts are added exactly, the float parts p, q, r
                // in one sum, the low parts in another.  c3 is taken as
                // ubar - c0 - c1 - c2, so the parent's shares add up to its
                // ubar to float-float rounding.
                const float q4h = 0.25f * ub[v].hi, q4l = 0.25f * ub[v].lo;
                const ff hF = ffm_lazy(F[v], hx), hG = ffm_lazy(G[v], hy);
                const float pr = par.p[v] + par.r[v], mr = par.p[v] - par.r[v];
                ff c[4];
                c[0] = ff_sum4(q4h, hF.hi, hG.hi, par.q[v] + pr, (q4l + hF.lo) + hG.lo);
                c[1] = ff_sum4(q4h, -hF.hi, hG.hi, par.q[v] - pr, (q4l - hF.lo) + hG.lo);
                c[2] = ff_sum4(q4h, -hF.hi, -hG.hi, -(par.q[v] + mr), (q4l - hF.lo) - hG.lo);
                c[3] = ff_rest3(ub[v], c[0], c[1], c[2]);
                float2* r2 = reinterpret_cast<float2*>(r);
#pragma unroll
                for (int k = 0; k < 4; ++k) r2[(v * 4 + k) * TW + t] = make_float2(c[k].hi, c[k].lo);
                const ff v00 = ff_add_u(u00[v], par.V[v][0]);  // read as a pair only
                r2[(NV * 4 + v) * TW + t] = make_float2(v00.hi, v00.lo);
#pragma unroll
                for (int qq = 1; qq < NQ1; ++qq) r[(NV * 10 + v * (NQ1 - 1) + qq - 1) * TW + t] = par.V[v][qq];
            }
        }
        __syncthreads();
        if (s >= 1 && t < TW - 1 && i0 + t < a.nx_new) {
            const RingReaderMx<TW, NV, NQ1> rd{ring + ((s - 1) & 1) * NF * TW, ring + (s & 1) * NF * TW, t};
            float D[NV][NQ];
            ff ub[NV];
            linear_cell_mx<SYS, P>(rd, D, ub);
            if (a.law.limiter) {
                // deviation form: the vertex values less the average, taken
                // from the float-float pairs and rounded, so that the
                // limiter's slopes and residuals near smooth extrema are not
                // float cancellations of O(1) values
                float vv[NV][4];
#pragma unroll
                for (int v = 0; v < NV; ++v)
#pragma unroll
                    for (int k = 0; k < 4; ++k) vv[v][k] = ff_close_diff(rd.v00(k, v), ub[v]);
                if constexpr (SYS == EULER) {
                    const float ubf[4] = {ub[0].hi, ub[1].hi, ub[2].hi, ub[3].hi};
                    if (!limit_euler<P, float>(D, ubf, vv, lamx, lamy, a.law)) err |= ERR_POSITIVITY;
                } else {
                    limit_scalar<P, float>(D[0], vv[0], a.law, 0.f);
                }
            }
            // the limiter keeps the cell average (every candidate has mean ubar)
            const long long cell = (long long)(j0 + s - 1) * a.pitch + (i0 + t);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                out[(long long)(v * NQ) * a.plane + cell] = ub[v].hi;
                out[(long long)(NV * NQ + v) * a.plane + cell] = ub[v].lo;
#pragma unroll
                for (int qq = 1; qq < NQ; ++qq) out[(long long)(v * NQ + qq) * a.plane + cell] = D[v][qq];
            }
            float centre[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) centre[v] = wcc::ff_add(ub[v], -even_correction<P, float>(D[v])).hi;
            const float rate = cfl_rate<SYS, float>(centre, a.law, idx, idy);
            if (rate != rate) {
                err |= (SYS == EULER && ub[0].hi == ub[0].hi) ? ERR_POSITIVITY : ERR_NONFINITE;
                rate_max = INFINITY;
            } else {
                rate_max = rate > rate_max ? rate : rate_max;
            }
        }
        __syncthreads();
    }
    finish2d<float, TW>(rate_max, err, dt, a);
}

// CFL rate of a loaded FP32-mixed stage: the point value from the average
template <int SYS, int P>
__global__ void __launch_bounds__(256) stage_rate2d_mx(const float* planes, long long pitch, long long plane, int nx,
                                                       int ny, Law2D law, double dx, double dy, DevState2D* st) {
    constexpr int NV = nvars(SYS), NQ = nq(P);
    float m = 0.f;
    unsigned err = 0;
    const long long n = (long long)nx * ny;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
        const long long cell = (c / nx) * pitch + (c % nx);
        float centre[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            float d[NQ];
            d[0] = 0.f;
#pragma unroll
            for (int qq = 1; qq < NQ; ++qq) d[qq] = planes[(long long)(v * NQ + qq) * plane + cell];
            const ff ub{planes[(long long)(v * NQ) * plane + cell], planes[(long long)(NV * NQ + v) * plane + cell]};
            centre[v] = wcc::ff_add(ub, -even_correction<P, float>(d)).hi;
        }
        const float r = cfl_rate<SYS, float>(centre, law, (float)(1.0 / dx), (float)(1.0 / dy));
        if (r != r) {
            err |= SYS == EULER ? ERR_POSITIVITY : ERR_NONFINITE;
            m = INFINITY;
        } else if (r > m) {
            m = r;
        }
    }
    post_rate((double)m, err, st);
}

template <int SYS, int P>
cudaError_t launch_halfstep2d_mx_t(const Step2D& a, cudaStream_t stream) {
    constexpr int TW = strip_width_mx<SYS, P>();
    constexpr size_t smem = ring_bytes<float, TW>(record_fields_mx<SYS, P>());
    static_assert(smem <= 48 * 1024 - 256, "the shared ring and the static shared words must fit without the opt-in attribute");
    if (a.resident) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(a.resident, halfstep2d_mx<SYS, P, TW>, TW, smem);
    const dim3 grid((a.nx_new + TW - 2) / (TW - 1), (a.ny_new + a.rows_per_cta - 1) / a.rows_per_cta);
    return wcc::launch_pdl<Step2D>(halfstep2d_mx<SYS, P, TW>, grid, TW, smem, stream, a);
}

}  // namespace wcc2d

namespace wcc2d {
// Instantiated in wcc2d_mixed.cu.
cudaError_t launch_halfstep2d_mx(int system, int P, const Step2D& a, cudaStream_t stream);
cudaError_t launch_stage_rate2d_mx(int system, int P, const float* planes, long long pitch, long long plane, int nx,
                                   int ny, const Law2D& law, double dx, double dy, DevState2D* st, cudaStream_t stream);
// precision: 0 FP64, 1 FP32, 2 FP32-mixed planes
cudaError_t launch_convert2d(int P, int precision, bool to_planes, double* aos, void* planes, int nx, int ny, int nv,
                             long long pitch, long long plane, cudaStream_t stream);
}  // namespace wcc2d

namespace wcc2d {
// Instantiated in wcc2d_scalar.cu, wcc2d_euler_f64.cu, wcc2d_euler_f32.cu.
cudaError_t launch_halfstep2d(int system, int P, bool fp32, const Step2D& a, cudaStream_t stream);
cudaError_t launch_stage_rate2d(int system, bool fp32, const void* planes, long long pitch, long long plane, int nx,
                                int ny, int nq_, const Law2D& law, double dx, double dy, DevState2D* st,
                                cudaStream_t stream);
}  // namespace wcc2d
