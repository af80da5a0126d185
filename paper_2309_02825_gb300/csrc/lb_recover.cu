// Macroscopic recovery (Sec. III.C) with TMA-staged halos.
//
// Each block recovers one row segment of kTile nodes.  For every population
// i it copies the source row segment [x0 - H, x0 + kTile + H) (H = one
// 16-byte vector, clipped to the row) from HBM into shared memory with one
// bulk asynchronous copy (cp.async.bulk, completing on an mbarrier), so the
// one-node x-halo that the pull f_i(x) = P_i(x - e_i) needs arrives with
// the tile; only the two periodic wrap nodes of a row (x = 0 pulling from
// N0 - 1, x = N0 - 1 pulling from 0) read a scalar from global memory.
// Then theta = sum f, J = sum e f (exact integer sums for 64-bit fixed
// point), grad theta = -s1 J / (sigma dx) and u = (2 - s1) c J / theta.
// With mirror walls (MIR) a row or population beyond a wall is read from its
// reflection (pop_source), and the wall nodes of x read x = 1 and N0 - 2 of
// the x-reflected population instead of the periodic wrap.
// The mbarrier wait is bounded: on timeout the block records an error flag,
// waits (again bounded) for its own copies and returns.
#include <math.h>
#include <stdint.h>

#include "lb_device.cuh"

namespace lbk {

constexpr int kTile = 256;                          // nodes per block (one per thread)
constexpr unsigned long long kWaitLimitNs = 1000000000ull;  // 1 s bound on a staging wait

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Test of an mbarrier phase; the hardware may suspend the thread for a short
// time first (polling threads take issue slots from the blocks that compute).
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Poll the phase until it completes or limit_ns of wall time have passed.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity,
                                                  unsigned long long limit_ns = kWaitLimitNs)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity))
        if (global_ns() - t0 > limit_ns) return false;
    return true;
}

template <typename T> struct RecAcc {
    using type = double;
};
template <> struct RecAcc<long long> {
    using type = long long;  // exact integer moment sums
};

// theta, grad theta and u of one node from theta - theta_ref and J (storage units).
template <class L, typename T>
__device__ __forceinline__ void recover_store(double thm, const double (&Jd)[4], const Recov &r, int64_t nodes,
                                              int64_t node, double *__restrict__ theta, double *__restrict__ grad,
                                              double *__restrict__ u, StatusFlag *__restrict__ flag)
{
    const double thd = std::is_same<T, float>::value ? thm + r.theta_ref : thm;
    if (theta) theta[node] = thd;
    {  // theta > 0 and finite, as bit tests on the integer pipes
        const long long tb = __double_as_longlong(thd);
        if (!(tb > 0) || ((tb >> 52) & 0x7ff) == 0x7ff) raise_flag(flag, 1);
    }
    const double cu = quot_int(r.ucoef, thd);  // the storage scale is folded into ucoef and gcoef
#pragma unroll
    for (int a = 0; a < L::D; ++a) {
        const double Ja = Jd[a];
        if (grad) grad[a * nodes + node] = r.gcoef * Ja;
        if (u) u[a * nodes + node] = cu * Ja;
    }
}

// The recovery of one node from its pulled values.
template <class L, typename T>
__device__ __forceinline__ void recover_node(const T (&vals)[L::Q], const Recov &r, double scale, int64_t nodes,
                                             int64_t node, double *__restrict__ theta, double *__restrict__ grad,
                                             double *__restrict__ u, StatusFlag *__restrict__ flag)
{
    double thm, Jd[4];  // theta - theta_ref and J in storage units
    if constexpr (std::is_same<T, float>::value) {
        // FP32 shifted storage: theta and J summed on the integer pipes
        // (f32_align in lb_device.cuh), each rounded once to FP64 by the hardware
        // (one FP64 instruction each, where the integer assembly takes 35)
        constexpr int PB = f32_align_bit<L::Q>();
        unsigned emax = 1;
#pragma unroll
        for (int i = 0; i < L::Q; ++i) emax = max(emax, f32_exp(vals[i]));
        long long thi = 0, Ji[4] = {0, 0, 0, 0};
        static_for<0, L::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            const long long fv = f32_align<PB>(vals[i], emax);
            thi += fv;
            static_for<0, L::D>([&](auto Ad) {
                constexpr int a = decltype(Ad)::value;
                constexpr int ev = L::E[i][a];
                if constexpr (ev == 1) Ji[a] += fv;
                if constexpr (ev == -1) Ji[a] -= fv;
            });
        });
        const int k = f32_unit<PB>(emax);
        thm = emax == 0xffu ? __longlong_as_double(0x7ff8000000000000ll) : i64_to_f64_hw(thi, k);
#pragma unroll
        for (int a = 0; a < L::D; ++a) Jd[a] = i64_to_f64_hw(Ji[a], k);
    } else {
        if constexpr (std::is_same<T, double>::value) {
            // FP64 states: the sums formed exactly on the integer pipes where the
            // node's values allow it (f64_align), each rounded once
            long long v[L::Q];
            unsigned emax;
            if (f64_align<L::Q, f64_align_bit<L>()>(vals, v, emax)) {
                long long th = 0, J[4] = {0, 0, 0, 0};
                static_for<0, L::Q>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    th += v[i];
                    static_for<0, L::D>([&](auto Ad) {
                        constexpr int a = decltype(Ad)::value;
                        constexpr int e = L::E[i][a];
                        if constexpr (e == 1) J[a] += v[i];
                        if constexpr (e == -1) J[a] -= v[i];
                    });
                });
                thm = f64_from_aligned<f64_align_bit<L>()>(th, emax);
#pragma unroll
                for (int a = 0; a < L::D; ++a) Jd[a] = f64_from_aligned<f64_align_bit<L>()>(J[a], emax);
                recover_store<L, T>(thm, Jd, r, nodes, node, theta, grad, u, flag);
                return;
            }
        }
        using A = typename RecAcc<T>::type;
        A th = 0, J[4] = {0, 0, 0, 0};
        static_for<0, L::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            const A fv = (A)vals[i];
            th += fv;
            static_for<0, L::D>([&](auto Ad) {
                constexpr int a = decltype(Ad)::value;
                constexpr int e = L::E[i][a];
                if constexpr (e == 1) J[a] += fv;
                if constexpr (e == -1) J[a] -= fv;
            });
        });
        if constexpr (std::is_same<A, long long>::value) {  // exact integer sums
            thm = (double)th * scale;
#pragma unroll
            for (int a = 0; a < L::D; ++a) Jd[a] = (double)J[a];
        } else {
            thm = th;
#pragma unroll
            for (int a = 0; a < L::D; ++a) Jd[a] = J[a];
        }
    }
    recover_store<L, T>(thm, Jd, r, nodes, node, theta, grad, u, flag);
}

// Rows row0 .. row0 + nrow - 1 of the grid (all rows in a plain recovery);
// the outputs hold those rows only, node (row - row0) * N0 + x.
template <class L, typename T, bool MIR>
__global__ void __launch_bounds__(kTile) recover_kernel(const T *__restrict__ src, Geom g, Recov r, double scale,
                                                       double *__restrict__ theta, double *__restrict__ grad,
                                                       double *__restrict__ u, StatusFlag *__restrict__ flag, int64_t row0,
                                                       int64_t nrow)
{
    constexpr int H = 16 / (int)sizeof(T);  // halo = one 16-byte vector
    constexpr int TW = kTile + 2 * H;        // tile width per population
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *tile = reinterpret_cast<T *>(smem_raw);
    __shared__ __align__(8) unsigned long long bar;

    const int tiles_per_row = (g.N0 + kTile - 1) / kTile;
    const int64_t row = row0 + blockIdx.x / tiles_per_row;
    const int x0 = (int)(blockIdx.x % tiles_per_row) * kTile;
    const RowPos rpos = row_pos<L::D>(g, row);
    // copy window: multiples of H elements, i.e. 16-byte aligned and sized
    const int xs = max(x0 - H, 0);
    const int xe = min(x0 + kTile + H, g.pitch);
    const uint32_t bytes = (uint32_t)((xe - xs) * (int)sizeof(T));
    const uint32_t barp = smem_u32(&bar);

    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(barp), "r"(1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(barp),
                     "r"(bytes * (uint32_t)L::Q)
                     : "memory");
        static_for<0, L::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            const PopSrc ps = pop_source<L, i, MIR>(g, rpos);
            const T *gsrc = src + (int64_t)ps.pop * g.slab + ps.row * g.pitch + xs;
            const uint32_t dst = smem_u32(tile + i * TW + (xs - x0 + H));
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                "l"(gsrc), "r"(bytes), "r"(barp)
                : "memory");
        });
    }
    if (!mbar_wait_bounded(barp, 0)) {
        if (threadIdx.x == 0) raise_flag(flag, 4);
        // Give this block's copies a second bounded interval to land before its
        // shared memory goes away.  If that also runs out the block returns with
        // copies possibly still in flight; the host treats flag bit 2 as fatal
        // for the context's state (lb_macros returns LB_ETIMEOUT and the context
        // needs a new state before it launches again).
        mbar_wait_bounded(barp, 0);
        return;
    }

    const int x = x0 + (int)threadIdx.x;
    if (x >= g.N0) return;
    T vals[L::Q];
    static_for<0, L::Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int ex = L::E[i][0];
        const int sx = x - ex;
        if (sx >= 0 && sx < g.N0) {
            vals[i] = tile[i * TW + (sx - x0 + H)];
        } else {  // across the row end: a scalar from the other end, or the x-reflection
            const PopSrc ps = pop_source<L, i, MIR>(g, rpos);
            if (MIR && (g.mirror & 1u))
                vals[i] = src[(int64_t)ps.popx * g.slab + ps.row * g.pitch + (sx < 0 ? 1 : g.N0 - 2)];
            else
                vals[i] = src[(int64_t)ps.pop * g.slab + ps.row * g.pitch + (sx < 0 ? g.N0 - 1 : 0)];
        }
    });
    recover_node<L, T>(vals, r, scale, (int64_t)g.N0 * nrow, (row - row0) * g.N0 + x, theta, grad, u, flag);
}

// The recovery with the nodes numbered row-major, one per thread, for rows
// that leave much of the staged kernel's 256-node tiles idle (a 50-node row: 80
// %).  Each population is one load at its wrapped or reflected source;
// neighbouring threads read neighbouring elements, so the loads stay coalesced
// across row ends.  50^4 fixed point: 1274 -> 300 us (2.1 GB of state and fields),
// with all 33 loads in flight: without a count of resident blocks the compiler takes
// 68 registers instead of 92 there and adds between the loads, 346 us.
template <class L, typename T, bool MIR>
__device__ __forceinline__ void recover_flat(const T *__restrict__ src, const Geom &g, const Recov &r, double scale,
                                             double *__restrict__ theta, double *__restrict__ grad,
                                             double *__restrict__ u, StatusFlag *__restrict__ flag, int64_t row0, int64_t nrow)
{
    const int64_t nodes = (int64_t)g.N0 * nrow;
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= nodes) return;
    const unsigned nd = (unsigned)n, rw = nd / (unsigned)g.N0;  // nodes <= 2^31
    const int x = (int)(nd - rw * (unsigned)g.N0);
    const RowPos rpos = row_pos<L::D>(g, row0 + rw);
    T vals[L::Q];
    if constexpr (!MIR && L::D < 4) {  // (4D: 53 registers instead of 96, fewer loads in flight, 300 -> 337 us at 50^4)
        const PullOffsets<L::D> from(g, x, rpos);
        static_for<0, L::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            vals[i] = __ldg(src + (int64_t)i * g.slab + from.template at<L, i>());
        });
        recover_node<L, T>(vals, r, scale, nodes, n, theta, grad, u, flag);
        return;
    }
    const bool mx = MIR && (g.mirror & 1u);
    static_for<0, L::Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int ex = L::E[i][0];
        const PopSrc ps = pop_source<L, i, MIR>(g, rpos);
        int sx = x - ex, pop = ps.pop;
        if (ex != 0 && (sx < 0 || sx >= g.N0)) {
            if (mx) {
                pop = ps.popx;
                sx = sx < 0 ? 1 : g.N0 - 2;
            } else {
                sx = sx < 0 ? g.N0 - 1 : 0;
            }
        }
        vals[i] = __ldg(src + (int64_t)pop * g.slab + ps.row * g.pitch + sx);
    });
    recover_node<L, T>(vals, r, scale, nodes, n, theta, grad, u, flag);
}

template <class L, typename T, bool MIR>
__global__ void __launch_bounds__(128) recover_flat_kernel(const T *__restrict__ src, Geom g, Recov r, double scale,
                                                           double *__restrict__ theta, double *__restrict__ grad,
                                                           double *__restrict__ u, StatusFlag *__restrict__ flag, int64_t row0,
                                                           int64_t nrow)
{
    recover_flat<L, T, MIR>(src, g, r, scale, theta, grad, u, flag, row0, nrow);
}
// The same with a register budget for five blocks per SM (4D fixed point).
template <class L, typename T, bool MIR>
__global__ void __launch_bounds__(128, 5) recover_flat5_kernel(const T *__restrict__ src, Geom g, Recov r, double scale,
                                                               double *__restrict__ theta, double *__restrict__ grad,
                                                               double *__restrict__ u, StatusFlag *__restrict__ flag, int64_t row0,
                                                               int64_t nrow)
{
    recover_flat<L, T, MIR>(src, g, r, scale, theta, grad, u, flag, row0, nrow);
}

// All 2D instances of a batch in one launch: the flat recovery of each node's
// own instance.
template <typename T>
__global__ void __launch_bounds__(128) batch_recover_kernel(const int64_t *__restrict__ node_off, int count,
                                                            const BatchInst *__restrict__ inst, const T *__restrict__ src,
                                                            double *__restrict__ theta, double *__restrict__ u,
                                                            StatusFlag *__restrict__ flag)
{
    const int64_t n = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int j = batch_instance(node_off, count, n);
    if (j < 0) return;
    const BatchInst &d = inst[j];
    const Geom &g = d.g;
    const int64_t n0 = node_off[j];
    const unsigned nd = (unsigned)(n - n0), row = nd / (unsigned)g.N0;
    const int x = (int)(nd - row * (unsigned)g.N0);
    const RowPos rpos = row_pos<2>(g, row);
    const T *s = src + d.off;
    const PullOffsets<2> from(g, x, rpos);
    T vals[D2Q9::Q];
    static_for<0, D2Q9::Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        vals[i] = __ldg(s + (int64_t)i * g.slab + from.template at<D2Q9, i>());
    });
    recover_node<D2Q9, T>(vals, d.rec, d.scale, node_off[j + 1] - n0, nd, theta ? theta + n0 : nullptr, nullptr,
                          u ? u + 2 * n0 : nullptr, flag);
}

cudaError_t launch_batch_recover(int precision, const int64_t *node_off, int count, int64_t nodes, const BatchInst *inst,
                                 const void *src, double *theta, double *u, StatusFlag *flag, cudaStream_t s)
{
    const unsigned nb = (unsigned)((nodes + 127) / 128);
    if (precision == LB_FX64)
        batch_recover_kernel<long long><<<nb, 128, 0, s>>>(node_off, count, inst, (const long long *)src, theta, u, flag);
    else if (precision == LB_FP32_SHIFTED)
        batch_recover_kernel<float><<<nb, 128, 0, s>>>(node_off, count, inst, (const float *)src, theta, u, flag);
    else
        batch_recover_kernel<double><<<nb, 128, 0, s>>>(node_off, count, inst, (const double *)src, theta, u, flag);
    return cudaGetLastError();
}

// Recovery constants of a context; *scale: the storage unit.
Recov make_recov(const lb_ctx *c, double *scale)
{
    Recov r;
    *scale = (c->precision == LB_FX64) ? ldexp(1.0, -c->fx_bits) : 1.0;
    // J is summed in storage units: the scale (a power of two, exact) goes into the constants
    r.ucoef = (2.0 - c->s1) * c->c * *scale;
    r.gcoef = -c->s1 / (c->sigma * c->dx) * *scale;
    r.theta_ref = (c->precision == LB_FP32_SHIFTED) ? c->theta_ref : 0.0;
    return r;
}

template <class L, typename T, bool MIR>
static cudaError_t recover_t(lb_ctx *c, const void *src, double *th, double *gr, double *u, StatusFlag *flag, int64_t row0,
                             int64_t nrow)
{
    constexpr int H = 16 / (int)sizeof(T);
    const size_t smem = (size_t)L::Q * (kTile + 2 * H) * sizeof(T);
    // up to 68 KB (D4Q33, 8-byte storage): allow more than the default 48 KB
    cudaError_t e = cudaFuncSetAttribute(recover_kernel<L, T, MIR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    double scale;
    const Recov r = make_recov(c, &scale);
    const int64_t tiles = (c->geom.N0 + kTile - 1) / kTile, blocks = nrow * tiles;
    if (blocks == 0) return cudaSuccess;
    if (c->geom.N0 * 4 < tiles * kTile * 3) {  // under three quarters of the tiles' nodes
        const int64_t nodes = nrow * c->geom.N0;
        const unsigned nb = (unsigned)((nodes + 127) / 128);
        if constexpr (L::D == 4 && std::is_same<T, long long>::value)
            recover_flat5_kernel<L, T, MIR><<<nb, 128, 0, c->stream>>>((const T *)src, c->geom, r, scale, th, gr, u, flag,
                                                                        row0, nrow);
        else
            recover_flat_kernel<L, T, MIR><<<nb, 128, 0, c->stream>>>((const T *)src, c->geom, r, scale, th, gr, u, flag,
                                                                       row0, nrow);
        return cudaGetLastError();
    }
    recover_kernel<L, T, MIR><<<(unsigned)blocks, kTile, smem, c->stream>>>((const T *)src, c->geom, r, scale, th,
                                                                             gr, u, flag, row0, nrow);
    return cudaGetLastError();
}

template <class L, bool MIR>
static cudaError_t recover_m(lb_ctx *c, const void *src, double *th, double *gr, double *u, StatusFlag *flag, int64_t row0,
                             int64_t nrow)
{
    switch (c->precision) {
    case LB_FX64: return recover_t<L, long long, MIR>(c, src, th, gr, u, flag, row0, nrow);
    case LB_FP32_SHIFTED: return recover_t<L, float, MIR>(c, src, th, gr, u, flag, row0, nrow);
    default: return recover_t<L, double, MIR>(c, src, th, gr, u, flag, row0, nrow);
    }
}

template <class L>
static cudaError_t recover_l(lb_ctx *c, const void *src, double *th, double *gr, double *u, StatusFlag *flag, int64_t row0,
                             int64_t nrow)
{
    return c->geom.mirror ? recover_m<L, true>(c, src, th, gr, u, flag, row0, nrow)
                          : recover_m<L, false>(c, src, th, gr, u, flag, row0, nrow);
}

// Self-test of the bounded wait: a barrier that nothing completes.
__global__ void staging_timeout_selftest_kernel(int *flag, unsigned long long limit_ns)
{
    __shared__ __align__(8) unsigned long long bar;
    const uint32_t barp = smem_u32(&bar);
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(barp), "r"(1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (!mbar_wait_bounded(barp, 0, limit_ns) && threadIdx.x == 0) atomicOr(flag, 4);
}

cudaError_t launch_macros_rows(lb_ctx *c, const void *src, double *th, double *gr, double *u, StatusFlag *flag, int64_t row0,
                               int64_t nrow)
{
    switch (c->d) {
    case 1: return recover_l<D1Q3>(c, src, th, gr, u, flag, row0, nrow);
    case 2: return recover_l<D2Q9>(c, src, th, gr, u, flag, row0, nrow);
    case 3: return recover_l<D3Q19>(c, src, th, gr, u, flag, row0, nrow);
    default: return recover_l<D4Q33>(c, src, th, gr, u, flag, row0, nrow);
    }
}

cudaError_t launch_macros(lb_ctx *c, const void *src, double *th, double *gr, double *u, StatusFlag *flag)
{
    return launch_macros_rows(c, src, th, gr, u, flag, 0, c->geom.rows);
}

}  // namespace lbk

extern "C" lb_status lb_selftest_staging_timeout(double limit_s, void *stream, double *waited_s)
{
    if (!(limit_s > 0.0) || limit_s > 10.0) return LB_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int *dflag = nullptr;
    int flag = 0;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaMalloc(&dflag, sizeof(int));
    if (e == cudaSuccess) e = cudaMemsetAsync(dflag, 0, sizeof(int), st);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e == cudaSuccess) e = cudaEventRecord(e0, st);
    if (e == cudaSuccess) {
        lbk::staging_timeout_selftest_kernel<<<1, 32, 0, st>>>(dflag, (unsigned long long)(limit_s * 1e9));
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaEventRecord(e1, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&flag, dflag, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    float ms = 0.0f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (waited_s) *waited_s = ms / 1e3;
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(dflag);
    if (e != cudaSuccess) return LB_ECUDA;
    return (flag & 4) ? LB_ETIMEOUT : LB_OK;
}
