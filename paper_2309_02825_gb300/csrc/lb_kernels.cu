// CUDA kernels of the MRT-LB hot path (sm_103a).
//
// Sweep = pull-stream + MRT collision of Eq. (distribution-f), fused, one
// warp per row segment of 32*V nodes (V = 2 doubles or 4 floats per thread,
// one 16-byte vector per population).  Populations with e_x = 0 are plain
// aligned vector loads; e_x = +-1 shifts by one element, done with an
// aligned vector load plus one warp shuffle, and a scalar load only at the
// warp edge and the periodic wrap.  Every store is an aligned vector.
//
// The collision is written in moment space in closed form (no q x q
// product): from theta, J_a = sum e_a f, P_aa = sum e_a^2 f and
// P_ab = sum e_a e_b f the relaxed moments follow from S; third-order
// moments relax to 0 and fourth-order ones to 4 wd theta (rate 1), so they
// are never formed; M^-1 is applied analytically.
#include <math.h>

#include "lb_device.cuh"

namespace lbk {

// ---------------------------------------------------------------------------
// Initialisation (first two terms of Eq. (f-feq-o5), closed form):
//   f_0 = w0 th,  f(+-e_a) = w1 th -+ iax d_a th,  f(diag e) = wd th - idg (e . grad th),
// stored in P form, P_0(y, i) = f_i(y + e_i, 0).  One thread per node x
// forms all q values of x once and stores f_i(x) at y = x - e_i (periodic
// wrap).  On an axis with mirror walls a destination beyond a wall is not
// stored (the doubled grid's ghost), and a thread next to a wall (x_a = 1
// with e_ia = +1, or x_a = N_a - 2 with e_ia = -1) also stores f_i(x) in
// the wall node's slot of the reflected population: that slot's source lies
// beyond the wall, at the mirror image of x.  Every stored slot has exactly
// one writer.  The wall-normal gradient component is odd across the wall, so
// on a wall node it is taken as zero.
//
// FXI (64-bit fixed point formed in integers): theta and dx * grad theta are
// converted to fixed point once per node, every product with a constant is
// rounded once, and the rest population is theta minus the others, so
// sum_i f_i(x) = round(theta0(x) 2^F) exactly.  FXI = 2 takes the collision's
// split product (mulfx_c, constants of 64 fraction bits), for constants in
// (-1/2, 1/2); FXI = 1 the 128-bit product with 62 fraction bits, about three
// times the instructions, for the rest (1D eps above 0.83).
//
// Otherwise the values are formed in FP64, which issues at 1/64 of the FP32 and
// integer rates and binds the kernel there: each shared term is formed once (a
// plane's four velocities have e . grad = +-(g_a + g_b), +-(g_a - g_b)) and FP32
// values are rounded to float on the integer pipes: 13 (FP64) and 16 (FP32)
// FP64 operations per D2Q9 node instead of 35 and 31.
//
// Each value is stored as soon as it is formed, so that few registers hold a
// node and enough warps are resident to keep the scattered stores in flight.
// ---------------------------------------------------------------------------
// round(v 2^F) to nearest, ties to even, from the fields of the IEEE double
// v in integer arithmetic (v 2^F is exact; only its rounding to an integer is
// done here).  Sets `range` when |v 2^F| >= 2^61, NaN and infinities included.
__device__ __forceinline__ long long fx_round(double v, int F, bool &range)
{
    const long long bits = __double_as_longlong(v);
    const int e = (int)((bits >> 52) & 0x7ff);
    const long long mant = (bits & ((1ll << 52) - 1)) | (e ? (1ll << 52) : 0ll);
    const int sh = (e ? e : 1) - 1075 + F;  // |v| 2^F = mant 2^sh
    if (e == 0x7ff || sh > 8) {             // mant >= 2^52: sh >= 9 means >= 2^61
        range = true;
        return 0;
    }
    long long r;
    if (sh >= 0) {
        r = mant << sh;
    } else if (sh < -53) {
        r = 0;  // below one half
    } else {
        const int k = -sh;
        const long long q = mant >> k, rem = mant & ((1ll << k) - 1), half = 1ll << (k - 1);
        r = q + ((rem > half || (rem == half && (q & 1))) ? 1 : 0);
    }
    return bits < 0 ? -r : r;
}

constexpr int kInitThreads = 128;

// The populations of a node from v = theta and dx grad theta in one fixed-point
// unit, handed to put in the order of the velocities.
template <class L, class Mul, class Put>
__device__ __forceinline__ void init_fx(const long long (&v)[1 + L::D], const InitK &K, Mul mul, Put put)
{
    constexpr int D = L::D, B0 = 1 + 2 * D;
    const long long t = v[0];
    // the velocities of an axis sum to 2 W1, those of a plane to 4 WD
    const long long W1 = mul(t, K.w1k), WD = D > 1 ? mul(t, K.wdk) : 0;
    put(std::integral_constant<int, 0>{}, t - (2 * D * W1 + 2 * D * (D - 1) * WD));
    static_for<0, D>([&](auto Ai) {
        constexpr int a = decltype(Ai)::value;
        const long long A = mul(v[1 + a], K.iak);
        put(std::integral_constant<int, 1 + a>{}, W1 - A);
        put(std::integral_constant<int, 1 + D + a>{}, W1 + A);
    });
    static_for<0, D *(D - 1) / 2>([&](auto Pi) {
        constexpr int p = decltype(Pi)::value;
        constexpr int a = pair_a<D>(p), b = pair_b<D>(p);
        // e . (dx grad) = +-(G_a + G_b) or +-(G_a - G_b); one rounded product per pair and sign
        const long long P = mul(v[1 + a] + v[1 + b], K.wdk), M = mul(v[1 + a] - v[1 + b], K.wdk);
        put(std::integral_constant<int, B0 + 4 * p>{}, WD - P);      // (+1, +1)
        put(std::integral_constant<int, B0 + 4 * p + 1>{}, WD + M);  // (-1, +1)
        put(std::integral_constant<int, B0 + 4 * p + 2>{}, WD + P);  // (-1, -1)
        put(std::integral_constant<int, B0 + 4 * p + 3>{}, WD - M);  // (+1, -1)
    });
}

template <class L, typename T, int FXI, bool MIR>
__device__ __forceinline__ void init_node(T *__restrict__ dst, const Geom &g, const InitK &K, int64_t node, int64_t nodes,
                                          const double *__restrict__ theta0, const double *__restrict__ grad,
                                          StatusFlag *__restrict__ flag)
{
    constexpr int D = L::D, B0 = 1 + 2 * D;
    // coordinates in 32-bit arithmetic (nodes <= 2^31)
    const int n[4] = {g.N0, g.N1, g.N2, g.N3};
    int c[4] = {0, 0, 0, 0};
    unsigned left = (unsigned)node;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const unsigned q = a + 1 < D ? left / (unsigned)n[a] : 0u;
        c[a] = (int)(left - q * (unsigned)n[a]);
        left = q;
    }

    // checks on the bit patterns (integer pipes): theta > 0 and finite, a
    // finite gradient (exponent field not all ones)
    const double th = theta0[node];
    const long long tb = __double_as_longlong(th);
    double gr[D];
    bool bad = !(tb > 0) || ((tb >> 52) & 0x7ff) == 0x7ff;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        gr[a] = grad[a * nodes + node];
        bad |= ((__double_as_longlong(gr[a]) >> 52) & 0x7ff) == 0x7ff;
        if (MIR && ((g.mirror >> a) & 1u) && (c[a] == 0 || c[a] == n[a] - 1)) gr[a] = 0.0;
    }
    if (bad) raise_flag(flag, 1);

    // periodic: destination offset = sum over axes of one of three wrapped
    // offsets (shift -1, 0, +1), formed once per node (a population has at most
    // 2^31 nodes and a row's padding each: below 2^32)
    unsigned off[4][3] = {};
    {
        unsigned stride = 1;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const int dn = c[a] == 0 ? n[a] - 1 : c[a] - 1;  // x_a - 1
            const int up = c[a] == n[a] - 1 ? 0 : c[a] + 1;  // x_a + 1
            off[a][0] = (unsigned)up * stride;               // e = -1 stores at x_a + 1
            off[a][1] = (unsigned)c[a] * stride;
            off[a][2] = (unsigned)dn * stride;               // e = +1 stores at x_a - 1
            stride *= (a == 0) ? (unsigned)g.pitch : (unsigned)n[a];
        }
    }
    const auto put = [&](auto I, T v) {
        constexpr int i = decltype(I)::value;
        constexpr int E0 = L::E[i][0], E1 = L::E[i][1], E2 = L::E[i][2], E3 = L::E[i][3];
        if constexpr (!MIR) {
            const unsigned at = off[0][E0 + 1] + off[1][E1 + 1] + off[2][E2 + 1] + off[3][E3 + 1];
            dst[(int64_t)i * g.slab + at] = v;
        } else {
            const int ev[4] = {E0, E1, E2, E3};
            int y[4];
            bool ghost = false;
            unsigned near = 0;  // axes where x is next to a wall it streams onto
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const int e = ev[a];
                int w = c[a] - e;
                if (e != 0 && ((g.mirror >> a) & 1u)) {
                    if (w < 0 || w >= n[a]) ghost = true;
                    if ((e > 0 && c[a] == 1) || (e < 0 && c[a] == n[a] - 2)) near |= 1u << a;
                } else if (w < 0) {
                    w += n[a];
                } else if (w >= n[a]) {
                    w -= n[a];
                }
                y[a] = w;
            }
            if (ghost) return;
            const int64_t at = (((int64_t)y[3] * g.N2 + y[2]) * g.N1 + y[1]) * g.pitch + y[0];
            dst[(int64_t)i * g.slab + at] = v;
            if (near) {
                constexpr int nzm = (E0 != 0 ? 1 : 0) | (E1 != 0 ? 2 : 0) | (E2 != 0 ? 4 : 0) | (E3 != 0 ? 8 : 0);
                static_for<1, 16>([&](auto Mi) {
                    constexpr int M = decltype(Mi)::value;
                    if constexpr ((M & ~nzm) == 0) {
                        if ((M & ~near) == 0) dst[(int64_t)reflect_pop<L>(i, M) * g.slab + at] = v;
                    }
                });
            }
        }
    };

    bool range = false;
    if constexpr (FXI != 0) {
        const auto mul = [](long long a, long long k) { return FXI == 2 ? mulfx_c(a, k) : mulfx(a, k); };
        unsigned acc = 0u;  // OR of the values' high words + 2^29: |v| < 2^61 exactly when it stays below 2^30
        const auto put_fx = [&](auto I, long long v) {
            // (the rest population lies below wmass max|theta0| <= 2^61)
            if constexpr (decltype(I)::value > 0) acc |= (unsigned)((unsigned long long)v >> 32) + 0x20000000u;
            put(I, v);
        };
        long long v[1 + D];
        v[0] = fx_round(th, K.fx_bits, range);
#pragma unroll
        for (int a = 0; a < D; ++a) v[1 + a] = fx_round(gr[a] * K.gscale, 0, range);
        init_fx<L>(v, K, mul, put_fx);
        if (acc >= 0x40000000u) range = true;
    } else {
        constexpr bool kF32 = std::is_same<T, float>::value;
        const auto put_d = [&](auto I, double v) {
            if constexpr (kF32)
                put(I, f64_to_f32_rn(v));
            else
                put(I, to_store<T>(v, K.fxscale, range));
        };
        const double dth = kF32 ? th - K.theta_ref : th;  // FP32 stores f_i - w_i theta_ref
        if constexpr (kF32) {
            // The fixed-point formation below, on theta - theta_ref and dx grad
            // aligned to the larger exponent (f64_align_round: 60 bits), each
            // population rounded once to FP32: 1 + D FP64 instructions in place of
            // 16 (2D; 85 % of that pipe).  1999 x 1501: 145 -> 66 us, 101 x 90 x 77:
            // 70 -> 33 us.
            double x[1 + D];
            x[0] = dth;
#pragma unroll
            for (int a = 0; a < D; ++a) x[1 + a] = K.dx * gr[a];
            long long v[1 + D];
            unsigned emax;
            constexpr int PB = 7;
            // (a theta so near its reference that bits of its own terms would be lost
            // beside the gradient's, zero included, takes the FP64 form)
            const unsigned e0 = ((unsigned)__double2hiint(dth) >> 20) & 0x7ffu;
            if (K.ints && f64_align_round<1 + D, PB>(x, v, emax) && emax - 983u <= 140u && emax - e0 <= 20u) {
                const int k = (int)emax - 1075 - PB;  // the unit's exponent, -99 .. 41
                init_fx<L>(v, K, [](long long a, long long c) { return mulfx_c(a, c); },
                           [&](auto I, long long f) { put(I, i64_to_f32_rn(f, k)); });
                return;
            }
        }
        const double b1 = K.w1 * dth, bd = K.wd * dth;
        put_d(std::integral_constant<int, 0>{}, K.w0 * dth);
        static_for<0, D>([&](auto Ai) {
            constexpr int a = decltype(Ai)::value;
            const double ga = K.iax * gr[a];
            put_d(std::integral_constant<int, 1 + a>{}, kF32 ? b1 - ga : fma(-K.iax, gr[a], b1));
            put_d(std::integral_constant<int, 1 + D + a>{}, kF32 ? b1 + ga : fma(K.iax, gr[a], b1));
        });
        static_for<0, D *(D - 1) / 2>([&](auto Pi) {
            constexpr int p = decltype(Pi)::value;
            constexpr int a = pair_a<D>(p), b = pair_b<D>(p);
            const double sp = gr[a] + gr[b], sm = gr[a] - gr[b];
            put_d(std::integral_constant<int, B0 + 4 * p>{}, fma(-K.idg, sp, bd));
            put_d(std::integral_constant<int, B0 + 4 * p + 1>{}, fma(K.idg, sm, bd));
            put_d(std::integral_constant<int, B0 + 4 * p + 2>{}, fma(K.idg, sp, bd));
            put_d(std::integral_constant<int, B0 + 4 * p + 3>{}, fma(-K.idg, sm, bd));
        });
    }
    if (range) raise_flag(flag, 2);
}

template <class L, typename T, int FXI, bool MIR>
__global__ void __launch_bounds__(kInitThreads) init_kernel(T *__restrict__ dst, Geom g, InitK K,
                                                            const double *__restrict__ theta0,
                                                            const double *__restrict__ grad, StatusFlag *__restrict__ flag)
{
    const int64_t nodes = (int64_t)g.N0 * g.rows;
    const int64_t node = (int64_t)blockIdx.x * kInitThreads + threadIdx.x;
    if (node < nodes) init_node<L, T, FXI, MIR>(dst, g, K, node, nodes, theta0, grad, flag);
}

// All instances of a batch in one launch (batch_instance finds a node's own).
template <typename T, int FXI>
__global__ void __launch_bounds__(kInitThreads) batch_init_kernel(const int64_t *__restrict__ node_off, int count,
                                                                  const BatchInst *__restrict__ inst, T *__restrict__ dst,
                                                                  const double *__restrict__ theta0,
                                                                  const double *__restrict__ grad, StatusFlag *__restrict__ flag)
{
    const int64_t n = (int64_t)blockIdx.x * kInitThreads + threadIdx.x;
    const int j = batch_instance(node_off, count, n);
    if (j < 0) return;
    const int64_t n0 = node_off[j];
    const BatchInst &d = inst[j];
    init_node<D2Q9, T, FXI, false>(dst + d.off, d.g, d.init, n - n0, node_off[j + 1] - n0, theta0 + n0, grad + 2 * n0, flag);
}

// Fourth-order central difference of theta along each axis: periodic, or,
// on an axis with mirror walls (bit a of mirror), the even reflection of
// theta across the wall nodes (theta(-k) = theta(k)).  An axis of fewer than
// four nodes wraps more than once.
__device__ __forceinline__ int fd4_at(int t, int n, bool mir)
{
    if (mir) return t < 0 ? -t : (t >= n ? 2 * (n - 1) - t : t);
    while (t < 0) t += n;
    while (t >= n) t -= n;
    return t;
}
// -th(2) + 8 th(1) - 8 th(-1) + th(-2) of an axis: exactly in integers, rounded
// once, where the four values' exponents lie within 4 of each other (57 bits, 2 +
// 16 of them below 2^62), which saves three of five FP64 instructions.
// 1999 x 1501: 51 -> 38 us.
template <int D>
__global__ void __launch_bounds__(256) fd4_kernel(const double *__restrict__ th, double *__restrict__ grad, int N0, int N1,
                                                  int N2, int N3, unsigned mirror, double inv12dx)
{
    const int64_t nodes = (int64_t)N0 * N1 * N2 * N3;  // <= 2^31
    const int64_t node = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (node >= nodes) return;
    const int n[4] = {N0, N1, N2, N3};
    unsigned left = (unsigned)node, stride = 1;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const unsigned q = a + 1 < D ? left / (unsigned)n[a] : 0u;
        const int c = (int)(left - q * (unsigned)n[a]);
        left = q;
        const bool mir = (mirror >> a) & 1u;
        const bool inner = c >= 2 && c < n[a] - 2;
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int m = k < 2 ? 2 - k : 1 - k;  // 2, 1, -1, -2
            const int to = inner ? m : fd4_at(c + m, n[a], mir) - c;
            v[k] = __ldg(th + (node + (int64_t)to * stride));
        }
        long long x[4];
        unsigned emax;
        double acc;
        if (f64_align<4, 4>(v, x, emax)) {
            acc = f64_from_aligned<4>((x[3] - x[0]) + 8 * (x[1] - x[2]), emax);
        } else {
            acc = -v[0];
            acc += 8.0 * v[1];
            acc += -8.0 * v[2];
            acc += v[3];
        }
        grad[a * nodes + node] = acc * inv12dx;
        stride *= (unsigned)n[a];
    }
}

// ---------------------------------------------------------------------------
// Deterministic FP64 reductions: per-block partials (warp shuffles, then
// shared memory), then one block folds the partials in a fixed order.
// ---------------------------------------------------------------------------
template <int NS> struct Acc {
    double v[NS];
};

// op[k]: 0 = sum, 1 = max.  The block's values go through shared memory, 16
// threads to a slot: the FP64 pipe takes a whole warp instruction's time for
// every step of a shuffle tree (5 per slot and warp: 16 of the 47 us of a 3D
// norms pass at 7e5 nodes), while each of these adds serves 32 lanes.
template <int NS>
__device__ __forceinline__ void block_reduce_store(Acc<NS> &a, const int (&op)[NS], double *dst)
{
    constexpr int P = 16;  // partial sums per slot
    __shared__ double sh[NS][kRedThreads + 1];
    __shared__ double part[NS][P];
#pragma unroll
    for (int k = 0; k < NS; ++k) sh[k][threadIdx.x] = a.v[k];
    __syncthreads();
    for (int j = threadIdx.x; j < NS * P; j += kRedThreads) {
        const int k = j / P, p = j - k * P;
        bool mx = false;
#pragma unroll
        for (int q = 0; q < NS; ++q) mx = q == k ? op[q] != 0 : mx;
        double s = sh[k][p];
        for (int w = p + P; w < kRedThreads; w += P) s = mx ? fmax(s, sh[k][w]) : s + sh[k][w];
        part[k][p] = s;
    }
    __syncthreads();
    if (threadIdx.x < NS) {
        const int k = threadIdx.x;
        bool mx = false;
#pragma unroll
        for (int q = 0; q < NS; ++q) mx = q == k ? op[q] != 0 : mx;
        double s = part[k][0];
        for (int w = 1; w < P; ++w) s = mx ? fmax(s, part[k][w]) : s + part[k][w];
        dst[k] = s;
    }
}

// Weight of a row of nodes in the conserved total: 1/2 per mirror wall of
// the y, z, w axes the row lies on (the doubled periodic grid holds interior
// nodes twice, wall nodes once); the x walls halve the row's first and last
// node.
__device__ __forceinline__ double row_wall_weight(const Geom &g, int64_t row)
{
    double wt = 1.0;
    const int y = (int)(row % g.N1);
    const int64_t r2 = row / g.N1;
    const int z = (int)(r2 % g.N2);
    const int w = (int)(r2 / g.N2);
    if ((g.mirror & 2u) && (y == 0 || y == g.N1 - 1)) wt *= 0.5;
    if ((g.mirror & 4u) && (z == 0 || z == g.N2 - 1)) wt *= 0.5;
    if ((g.mirror & 8u) && (w == 0 || w == g.N3 - 1)) wt *= 0.5;
    return wt;
}

template <typename T> struct SumAcc {
    using type = double;
};
template <> struct SumAcc<long long> {
    using type = __int128;  // exact: fixed-point values add without rounding
};
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(__int128 v)
{
    const long long hi = (long long)(v >> 64);
    const unsigned long long lo = (unsigned long long)v;
    return (double)hi * 0x1p64 + (double)lo;
}

// Sum of the stored state over populations and nodes of a grid with mirror
// walls, weighted by the wall weights: one warp per row of one population,
// aligned 16-byte vector loads along the row.
template <typename T>
__global__ void __launch_bounds__(kRedThreads) sum_state_kernel(const T *__restrict__ src, Geom g, int q,
                                                                double scale, double *__restrict__ partial)
{
    constexpr int V = Vec<T>::V;
    double accw = 0.0;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // rows of the sum: g.rows per population (a sub-range of the grid's rows
    // when src starts past row 0), populations g.slab values apart
    const int64_t nrows = (int64_t)q * g.rows;
    constexpr int U = 4;  // vectors in flight per lane
    for (int64_t r = warp; r < nrows; r += nwarps) {
        const int64_t pop = r / g.rows, row = r - pop * g.rows;
        const T *rowp = src + pop * g.slab + row * g.pitch;
        const double rw = row_wall_weight(g, row);
        for (int x0 = lane * V; x0 < g.N0; x0 += U * 32 * V) {
            T a[U][V];
#pragma unroll
            for (int j = 0; j < U; ++j)
                if (x0 + j * 32 * V < g.N0) ld_vec(rowp + x0 + j * 32 * V, a[j]);
#pragma unroll
            for (int j = 0; j < U; ++j) {
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    const int x = x0 + j * 32 * V + k;
                    if (x >= g.N0) continue;
                    const double xw = ((g.mirror & 1u) && (x == 0 || x == g.N0 - 1)) ? 0.5 : 1.0;
                    accw += (double)a[j][k] * (rw * xw);
                }
            }
        }
    }
    Acc<1> a{{accw * scale}};
    const int op[1] = {0};
    block_reduce_store<1>(a, op, partial + (int64_t)blockIdx.x * kRedSlots);
}

// The same without walls: the rows of a population lie one after the other, so
// a thread takes 16-byte vectors at a grid-wide stride, whatever the row
// length, U of them in flight; padding is masked to zero.  Fixed point: exact
// 128-bit sums.  FP32: the U vectors' floats in one integer-pipe sum
// (sum_f32_int) and one FP64 addition.  The walled kernel above gives each row
// to a warp: rows of 101 floats kept 26 of 32 lanes busy once per row (101 x 90
// x 77: 274 us for 53 MB).
template <typename T>
__global__ void __launch_bounds__(kRedThreads) sum_flat_kernel(const T *__restrict__ src, Geom g, int q, double scale,
                                                               double *__restrict__ partial)
{
    constexpr int V = Vec<T>::V, U = 4;
    typename SumAcc<T>::type acc = 0;
    const int vr = g.pitch / V;                      // vectors per row
    const int64_t nv = g.rows * vr;                  // per population (populations g.slab values apart)
    const int64_t stride = (int64_t)gridDim.x * kRedThreads;
    int64_t i = (int64_t)blockIdx.x * kRedThreads + threadIdx.x;
    const int dx = (int)(stride % vr);
    int xv = (int)(i % vr), pop = 0;
    const bool pad = g.pitch != g.N0;
    while (i >= nv && pop < q) {
        i -= nv;
        ++pop;
    }
    while (pop < q) {
        T a[U][V];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            if (pop < q)
                ld_vec(src + pop * g.slab + i * V, a[j]);
            else
#pragma unroll
                for (int k = 0; k < V; ++k) a[j][k] = T(0);
            if (pad) {
#pragma unroll
                for (int k = 0; k < V; ++k)
                    if (xv * V + k >= g.N0) a[j][k] = T(0);
                xv += dx;
                if (xv >= vr) xv -= vr;
            }
            i += stride;
            while (i >= nv && pop < q) {
                i -= nv;
                ++pop;
            }
        }
        if constexpr (std::is_same<T, float>::value) {
            float f[U * V];
#pragma unroll
            for (int j = 0; j < U * V; ++j) f[j] = a[j / V][j % V];
            acc += sum_f32_int(f);
        } else {
#pragma unroll
            for (int j = 0; j < U * V; ++j) acc += a[j / V][j % V];
        }
    }
    Acc<1> s{{to_double(acc) * scale}};
    const int op[1] = {0};
    block_reduce_store<1>(s, op, partial + (int64_t)blockIdx.x * kRedSlots);
}

// Error norms: slots 3v+0 sum err^2, 3v+1 max |err|, 3v+2 sum exact^2 for
// v = 0 (theta), 1..d (u); slot 3(d+1) = sum theta.
template <int D>
__global__ void __launch_bounds__(kRedThreads) norms_kernel(const double *__restrict__ th,
                                                            const double *__restrict__ u,
                                                            const double *__restrict__ eth,
                                                            const double *__restrict__ eu, int64_t nodes,
                                                            double *__restrict__ partial)
{
    constexpr int NS = 3 * (D + 1) + 1;
    Acc<NS> a;
#pragma unroll
    for (int k = 0; k < NS; ++k) a.v[k] = 0.0;
    // max |err| on the integer pipes: for non-negative doubles the bit
    // patterns order like the values (a NaN error shows in the RMSE sums)
    long long mx[D + 1];
#pragma unroll
    for (int c = 0; c <= D; ++c) mx[c] = 0;
    constexpr long long kAbs = 0x7fffffffffffffffll;
#pragma unroll 2
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < nodes;
         n += (int64_t)gridDim.x * blockDim.x) {
        const double t = th[n], te = eth[n];
        const double e = t - te;
        a.v[0] = fma(e, e, a.v[0]);
        mx[0] = max(mx[0], __double_as_longlong(e) & kAbs);
        a.v[2] = fma(te, te, a.v[2]);
        a.v[NS - 1] += t;
        if (u) {
#pragma unroll
            for (int c = 0; c < D; ++c) {
                const double uv = u[c * nodes + n], ue = eu[c * nodes + n];
                const double eu2 = uv - ue;
                a.v[3 * (c + 1) + 0] = fma(eu2, eu2, a.v[3 * (c + 1) + 0]);
                mx[c + 1] = max(mx[c + 1], __double_as_longlong(eu2) & kAbs);
                a.v[3 * (c + 1) + 2] = fma(ue, ue, a.v[3 * (c + 1) + 2]);
            }
        }
    }
#pragma unroll
    for (int c = 0; c <= D; ++c) a.v[3 * c + 1] = __longlong_as_double(mx[c]);
    int op[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) op[k] = (k < NS - 1 && k % 3 == 1) ? 1 : 0;
    block_reduce_store<NS>(a, op, partial + (int64_t)blockIdx.x * kRedSlots);
}

// Clears n status flags and their mirrors from mirror on, in stream order.
__global__ void clear_flags_kernel(StatusFlag *flag, int *mirror, int n)
{
    if ((int)threadIdx.x >= n) return;
    flag[threadIdx.x] = {0, 0, mirror + threadIdx.x};
    mirror[threadIdx.x] = 0;
}
cudaError_t launch_clear_flags(StatusFlag *flag, int *mirror, int n, cudaStream_t s)
{
    clear_flags_kernel<<<1, 32, 0, s>>>(flag, mirror, n);
    return cudaGetLastError();
}

// max |x| over n values.
__global__ void __launch_bounds__(kRedThreads) maxabs_kernel(const double *__restrict__ x, int64_t n,
                                                             double *__restrict__ partial)
{
    Acc<1> a{{0.0}};
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        a.v[0] = fmax(a.v[0], fabs(x[t]));
    const int op[1] = {1};
    block_reduce_store<1>(a, op, partial + (int64_t)blockIdx.x * kRedSlots);
}

// Fold nb partial rows of kRedSlots in a fixed order.  opmask bit k = max.  A
// warp per slot, so all slots wait for their loads together.
__global__ void __launch_bounds__(32 * kRedSlots) fold_kernel(const double *__restrict__ partial, int nb, int ns,
                                                              unsigned opmask, double *__restrict__ out)
{
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (k >= ns) return;
    const bool mx = (opmask >> k) & 1u;
    double s = 0.0;
    for (int b0 = lane; b0 < nb; b0 += 32 * 8) {
        double v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = b0 + 32 * j < nb ? partial[(int64_t)(b0 + 32 * j) * kRedSlots + k] : 0.0;
#pragma unroll
        for (int j = 0; j < 8; ++j) s = mx ? fmax(s, v[j]) : s + v[j];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double t = __shfl_xor_sync(0xffffffffu, s, o);
        s = mx ? fmax(s, t) : s + t;
    }
    if (lane == 0) out[k] = s;
}

// ---------------------------------------------------------------------------
// Host-side dispatch.
// ---------------------------------------------------------------------------
template <typename T> Coll<T> make_coll(const lb_ctx &cc)
{
    const lb_ctx *c = &cc;
    const double d = c->d;
    const double s2x = c->s2x, s22 = (c->d > 1) ? c->s22 : 1.0, wd = (c->d > 1) ? c->wd : 0.0;
    Coll<T> k;
    k.k1 = (T)((1.0 - c->s1) / 2.0);
    k.k2 = (T)((1.0 - s2x) / 2.0);
    k.k3 = (T)((1.0 - s22) / 4.0);
    k.c0 = (T)(1.0 - d * s2x * c->sigma + 2.0 * d * (d - 1.0) * wd);
    k.cA = (T)(s2x * c->sigma / 2.0 - 2.0 * (d - 1.0) * wd);
    k.wd = (T)wd;
    return k;
}
template Coll<double> make_coll<double>(const lb_ctx &);
template Coll<float> make_coll<float>(const lb_ctx &);


template <typename T> struct SweepK {
    using type = Coll<T>;
    static type make(const lb_ctx &c) { return make_coll<T>(c); }
};
template <> struct SweepK<double> {
    using type = CollF64;
    static type make(const lb_ctx &c) { return make_coll_f64(c); }
};

template <class L, typename T> static cudaError_t sweep_t(lb_ctx *c, const void *src, void *dst)
{
    using K = typename SweepK<T>::type;
    const K k = SweepK<T>::make(*c);
    constexpr int TH = sweep_threads<T>();
    const bool flat = sweep_flat(c->geom, L::D, (int)sizeof(T));
    const unsigned nb = (unsigned)(((flat ? c->geom.fseg : c->geom.nseg) + TH / 32 - 1) / (TH / 32));
    if constexpr (L::D == 4 && sizeof(T) == 8) {
        if (flat) {
            sweep_flat_kernel<L, T, K><<<nb, TH, 0, c->stream>>>((const T *)src, (T *)dst, c->geom,
                                                                       k);
            return cudaGetLastError();
        }
    }
    if (c->geom.mirror)
        sweep_kernel<L, T, K, true><<<nb, TH, 0, c->stream>>>(
            (const T *)src, (T *)dst, c->geom, k);
    else
        sweep_kernel<L, T, K><<<nb, TH, 0, c->stream>>>(
            (const T *)src, (T *)dst, c->geom, k);
    return cudaGetLastError();
}

cudaError_t launch_sweep(lb_ctx *c, const void *src, void *dst)
{
    if (c->precision == LB_FX64) return launch_sweep_fx(c, src, dst);
    const bool f64 = c->precision == LB_FP64;
    switch (c->d) {
    case 1: return f64 ? sweep_t<D1Q3, double>(c, src, dst) : sweep_t<D1Q3, float>(c, src, dst);
    case 2: return f64 ? sweep_t<D2Q9, double>(c, src, dst) : sweep_t<D2Q9, float>(c, src, dst);
    case 3: return f64 ? sweep_t<D3Q19, double>(c, src, dst) : sweep_t<D3Q19, float>(c, src, dst);
    default: return f64 ? sweep_t<D4Q33, double>(c, src, dst) : sweep_t<D4Q33, float>(c, src, dst);
    }
}

cudaError_t launch_fd4_grad(const lb_ctx *c, const double *theta0, double *grad)
{
    const int64_t nodes = c->nodes;
    const auto go = [&](auto kernel) {
        kernel<<<(unsigned)((nodes + 255) / 256), 256, 0, c->stream>>>(theta0, grad, (int)c->N[0], (int)c->N[1], (int)c->N[2],
                                                                       (int)c->N[3], c->geom.mirror, 1.0 / (12.0 * c->dx));
    };
    switch (c->d) {
    case 1: go(fd4_kernel<1>); break;
    case 2: go(fd4_kernel<2>); break;
    case 3: go(fd4_kernel<3>); break;
    default: go(fd4_kernel<4>);
    }
    return cudaGetLastError();
}

template <class L, typename T, int FXI>
static cudaError_t init_go(lb_ctx *c, const InitK &K, const double *theta0, const double *grad, StatusFlag *flag)
{
    const unsigned nb = (unsigned)((c->nodes + kInitThreads - 1) / kInitThreads);
    if (c->geom.mirror)
        init_kernel<L, T, FXI, true><<<nb, kInitThreads, 0, c->stream>>>((T *)c->f[c->cur], c->geom, K, theta0, grad, flag);
    else
        init_kernel<L, T, FXI, false><<<nb, kInitThreads, 0, c->stream>>>((T *)c->f[c->cur], c->geom, K, theta0, grad, flag);
    return cudaGetLastError();
}

// The constants of a context's initialisation and the formation they admit
// (FXI of init_node; 0 but for fixed point).
static int make_initk(const lb_ctx *c, InitK &K)
{
    const double d = c->d;
    const double wd = (c->d > 1) ? c->wd : 0.0;
    K.w0 = c->w0;
    K.w1 = c->w1;
    K.wd = wd;
    K.iax = 0.5 * c->dx * (c->sigma / c->s1 - 4.0 * (d - 1.0) * wd);
    K.idg = wd * c->dx;
    K.theta_ref = (c->precision == LB_FP32_SHIFTED) ? c->theta_ref : 0.0;
    K.fxscale = ldexp(1.0, c->fx_bits);
    K.gscale = c->dx * K.fxscale;
    K.fx_bits = c->fx_bits;
    K.dx = c->dx;
    K.w1k = K.wdk = K.iak = 0;
    K.ints = 0;
    if (c->precision == LB_FP64) return 0;
    // integer formation needs every constant inside the product's range and a
    // total weight that keeps the rest population's sum below 2^61
    const double ia = K.iax / c->dx;
    const double wmass = fabs(c->w0) + 2.0 * d * fabs(c->w1) + 2.0 * d * (d - 1.0) * fabs(wd);
    if (!(fabs(ia) < 1.5 && fabs(c->w1) < 1.0 && fabs(wd) < 1.0 && wmass <= 4.0)) return 0;
    const double most = 0.5 - 0x1p-30;  // mulfx_c's range
    const bool split = fabs(ia) < most && fabs(c->w1) < most && fabs(wd) < most;
    const int bits = split ? kFxCollBits : kFxCoefBits;
    K.w1k = llrint(ldexp(c->w1, bits));
    K.wdk = llrint(ldexp(wd, bits));
    K.iak = llrint(ldexp(ia, bits));
    K.ints = split;
    if (c->precision == LB_FP32_SHIFTED) return 0;
    return split ? 2 : 1;
}

template <class L, typename T>
static cudaError_t init_t(lb_ctx *c, const double *theta0, const double *grad, StatusFlag *flag)
{
    InitK K;
    const int fxi = make_initk(c, K);
    if constexpr (std::is_same<T, long long>::value) {
        if (fxi == 2) return init_go<L, T, 2>(c, K, theta0, grad, flag);
        if (fxi == 1) return init_go<L, T, 1>(c, K, theta0, grad, flag);
    }
    return init_go<L, T, 0>(c, K, theta0, grad, flag);
}

bool make_batch_inst(const lb_ctx *c, int64_t off, BatchInst *out)
{
    out->g = c->geom;
    out->off = off;
    const int fxi = make_initk(c, out->init);
    out->rec = make_recov(c, &out->scale);
    return c->precision != LB_FX64 || fxi == 2;
}

cudaError_t launch_batch_init(int precision, const int64_t *node_off, int count, int64_t nodes, const BatchInst *inst,
                              void *dst, const double *theta0, const double *grad, StatusFlag *flag, cudaStream_t s)
{
    const unsigned nb = (unsigned)((nodes + kInitThreads - 1) / kInitThreads);
    if (precision == LB_FX64)
        batch_init_kernel<long long, 2><<<nb, kInitThreads, 0, s>>>(node_off, count, inst, (long long *)dst, theta0, grad, flag);
    else if (precision == LB_FP32_SHIFTED)
        batch_init_kernel<float, 0><<<nb, kInitThreads, 0, s>>>(node_off, count, inst, (float *)dst, theta0, grad, flag);
    else
        batch_init_kernel<double, 0><<<nb, kInitThreads, 0, s>>>(node_off, count, inst, (double *)dst, theta0, grad, flag);
    return cudaGetLastError();
}

cudaError_t launch_init(lb_ctx *c, const double *theta0, const double *grad, StatusFlag *flag)
{
    if (c->precision == LB_FX64) {
        switch (c->d) {
        case 1: return init_t<D1Q3, long long>(c, theta0, grad, flag);
        case 2: return init_t<D2Q9, long long>(c, theta0, grad, flag);
        case 3: return init_t<D3Q19, long long>(c, theta0, grad, flag);
        default: return init_t<D4Q33, long long>(c, theta0, grad, flag);
        }
    }
    const bool f64 = c->precision == LB_FP64;
    switch (c->d) {
    case 1: return f64 ? init_t<D1Q3, double>(c, theta0, grad, flag) : init_t<D1Q3, float>(c, theta0, grad, flag);
    case 2: return f64 ? init_t<D2Q9, double>(c, theta0, grad, flag) : init_t<D2Q9, float>(c, theta0, grad, flag);
    case 3: return f64 ? init_t<D3Q19, double>(c, theta0, grad, flag) : init_t<D3Q19, float>(c, theta0, grad, flag);
    default: return f64 ? init_t<D4Q33, double>(c, theta0, grad, flag) : init_t<D4Q33, float>(c, theta0, grad, flag);
    }
}

cudaError_t launch_sum_state_rows(lb_ctx *c, const void *src, double *out_dev, int64_t row0, int64_t nrow)
{
    const int nb = c->scratch_blocks;
    Geom g = c->geom;  // rows row0 .. row0 + nrow - 1 of every population (no walls on a sub-range)
    g.rows = nrow;
    if (row0 != 0 || nrow != c->geom.rows) g.mirror = 0;
    const int64_t off = row0 * g.pitch;
    const double scale = c->precision == LB_FX64 ? ldexp(1.0, -c->fx_bits) : 1.0;
    const auto launch = [&](auto *p) {
        using T = std::remove_pointer_t<decltype(p)>;
        if (g.mirror)
            sum_state_kernel<T><<<nb, kRedThreads, 0, c->stream>>>((const T *)src + off, g, c->q, scale, c->scratch);
        else
            sum_flat_kernel<T><<<nb, kRedThreads, 0, c->stream>>>((const T *)src + off, g, c->q, scale, c->scratch);
    };
    if (c->precision == LB_FP64)
        launch((double *)nullptr);
    else if (c->precision == LB_FX64)
        launch((long long *)nullptr);
    else
        launch((float *)nullptr);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    fold_kernel<<<1, 32 * kRedSlots, 0, c->stream>>>(c->scratch, nb, 1, 0u, out_dev);
    return cudaGetLastError();
}

cudaError_t launch_sum_state(lb_ctx *c, const void *src, double *out_dev)
{
    return launch_sum_state_rows(c, src, out_dev, 0, c->geom.rows);
}

cudaError_t launch_maxabs(lb_ctx *c, const double *x, int64_t n, double *out_dev)
{
    const int nb = c->scratch_blocks;
    maxabs_kernel<<<nb, kRedThreads, 0, c->stream>>>(x, n, c->scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    fold_kernel<<<1, 32 * kRedSlots, 0, c->stream>>>(c->scratch, nb, 1, 1u, out_dev);
    return cudaGetLastError();
}

cudaError_t launch_norms(lb_ctx *c, const double *th, const double *u, const double *eth, const double *eu,
                         double *out_dev)
{
    const int nb = c->scratch_blocks;
    const int ns = 3 * (c->d + 1) + 1;
    unsigned mask = 0;
    for (int k = 0; k < ns - 1; ++k)
        if (k % 3 == 1) mask |= 1u << k;
    switch (c->d) {
    case 1: norms_kernel<1><<<nb, kRedThreads, 0, c->stream>>>(th, u, eth, eu, c->nodes, c->scratch); break;
    case 2: norms_kernel<2><<<nb, kRedThreads, 0, c->stream>>>(th, u, eth, eu, c->nodes, c->scratch); break;
    case 3: norms_kernel<3><<<nb, kRedThreads, 0, c->stream>>>(th, u, eth, eu, c->nodes, c->scratch); break;
    default: norms_kernel<4><<<nb, kRedThreads, 0, c->stream>>>(th, u, eth, eu, c->nodes, c->scratch); break;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    fold_kernel<<<1, 32 * kRedSlots, 0, c->stream>>>(c->scratch, nb, ns, mask, out_dev);
    return cudaGetLastError();
}

// Norm reduction into caller-provided partial rows (nblocks of kRedSlots)
// and one raw-sum row; used by the allocation-free entry point.
cudaError_t launch_norms_into(int d, int64_t nodes, const double *th, const double *u, const double *eth,
                              const double *eu, double *partials, int nb, double *raw_out, cudaStream_t s)
{
    const int ns = 3 * (d + 1) + 1;
    unsigned mask = 0;
    for (int k = 0; k < ns - 1; ++k)
        if (k % 3 == 1) mask |= 1u << k;
    switch (d) {
    case 1: norms_kernel<1><<<nb, kRedThreads, 0, s>>>(th, u, eth, eu, nodes, partials); break;
    case 2: norms_kernel<2><<<nb, kRedThreads, 0, s>>>(th, u, eth, eu, nodes, partials); break;
    default: norms_kernel<3><<<nb, kRedThreads, 0, s>>>(th, u, eth, eu, nodes, partials); break;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    fold_kernel<<<1, 32 * kRedSlots, 0, s>>>(partials, nb, ns, mask, raw_out);
    return cudaGetLastError();
}

}  // namespace lbk
