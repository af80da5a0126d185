// Resident sweeps of short 1D grids: any number of steps in one launch of one
// block, the whole state in registers.
//
// A 1D sweep of a few hundred nodes lasts about as long as its launch: 800
// steps of an 81-node grid took 2.3 us each, replayed from a graph (now 0.34), for nine
// floating-point operations per node.  Here a thread owns V consecutive nodes
// for all steps; a step exchanges only the two values that leave the thread,
// P_1 of its last node and P_2 of its first, through shared memory (two
// buffers in turn, so one barrier per step orders both its writes before the
// reads and the next step's writes after them).  The periodic wrap, or the
// wall's reflection (the node at x = 0 pulls P_2(1), the one at N0 - 1 pulls
// P_1(N0 - 2)), is a ghost slot that the source's owner writes too.  The
// collision is the sweep's own: the results are bit for bit those of one sweep
// per launch.
#include "lb_device.cuh"

namespace lbk {

constexpr int kLineThreads = 1024;

template <typename T, class K, int V>
__global__ void __launch_bounds__(kLineThreads) line_kernel(const T *__restrict__ src, T *__restrict__ dst, Geom g, K k,
                                                            int64_t steps)
{
    __shared__ T right[2][kLineThreads + 2], left[2][kLineThreads + 2];  // [t + 1]: thread t's; the ends are ghosts
    const int t = threadIdx.x, x0 = t * V, N = g.N0;
    const bool mir = g.mirror & 1u;
    T p[V][3];
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int i = 0; i < 3; ++i) p[v][i] = x0 + v < N ? src[(int64_t)i * g.slab + x0 + v] : T(0);
    // what node 0 pulls from the left and node N - 1 from the right: who owns it
    const int lx = mir ? 1 : N - 1, rx = mir ? N - 2 : 0;
    const int lp = mir ? 2 : 1, rp = mir ? 1 : 2;
    unsigned acc = 0u;  // fixed point: OR of the high words + 2^29 (|v| < 2^61 check)
    for (int64_t s = 0; s < steps; ++s) {
        const int b = (int)(s & 1);
        right[b][t + 1] = p[V - 1][1];
        left[b][t + 1] = p[0][2];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if (x0 + v == lx) right[b][0] = lp == 1 ? p[v][1] : p[v][2];
            if (x0 + v == rx) left[b][kLineThreads + 1] = rp == 1 ? p[v][1] : p[v][2];
        }
        __syncthreads();
        T f[V][3];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            f[v][0] = p[v][0];
            f[v][1] = v > 0 ? p[v - 1][1] : right[b][t];
            f[v][2] = v < V - 1 ? p[v + 1][2] : left[b][t + 2];
            if (x0 + v == N - 1) f[v][2] = left[b][kLineThreads + 1];
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            collide_at<T>(D1Q3{}, f[v], k, x0 + v, N);
#pragma unroll
            for (int i = 0; i < 3; ++i) p[v][i] = f[v][i];
            if constexpr (std::is_same<K, CollFxR>::value) {
                if (x0 + v < N) {
#pragma unroll
                    for (int i = 0; i < 3; ++i) acc |= (unsigned)((unsigned long long)f[v][i] >> 32) + 0x20000000u;
                }
            }
        }
    }
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int i = 0; i < 3; ++i)
            if (x0 + v < N) dst[(int64_t)i * g.slab + x0 + v] = p[v][i];
    if constexpr (std::is_same<K, CollFxR>::value) {
        if (acc >= 0x40000000u) raise_flag_call(k.range, 1);
    }
}

template <typename T, class K> static cudaError_t line_t(lb_ctx *c, const void *src, void *dst, int64_t steps, const K &k)
{
    const int n = (int)c->N[0], v = n <= kLineThreads ? 1 : (n <= 2 * kLineThreads ? 2 : 4);
    const int threads = ((n + v - 1) / v + 31) / 32 * 32;
    const T *s = (const T *)src;
    T *d = (T *)dst;
    if (v == 1)
        line_kernel<T, K, 1><<<1, threads, 0, c->stream>>>(s, d, c->geom, k, steps);
    else if (v == 2)
        line_kernel<T, K, 2><<<1, threads, 0, c->stream>>>(s, d, c->geom, k, steps);
    else
        line_kernel<T, K, 4><<<1, threads, 0, c->stream>>>(s, d, c->geom, k, steps);
    return cudaGetLastError();
}

// One SM's throughput against a launch per step (2.4-2.8 us): FP64 up to 2048
// nodes, the others up to 4096.
bool line_fits(const lb_ctx *c)
{
    return c->d == 1 && c->N[0] <= (c->precision == LB_FP64 ? 2 : 4) * kLineThreads;
}

// A call of few steps: the one block's loads and stores are spread over no more
// steps than that.  us per call, resident / one sweep per launch: one step FP64 2048 nodes
// 6.2 / 4.1, FP32 4096 8.2 / 4.1, fixed point 2048 6.2 / 4.1; fixed point 4096 one
// to five steps 12.4, 14.4, 15.5, 16.5, 18.5 / 4.1, 8.2, 12.3, 16.4, 20.5; two
// steps elsewhere no more than two sweeps.
int line_least(const lb_ctx *c) { return c->precision == LB_FX64 && c->N[0] > 2 * kLineThreads ? 5 : 2; }

cudaError_t line_launch(lb_ctx *c, const void *src, void *dst, int64_t steps)
{
    if (c->precision == LB_FP64) return line_t<double>(c, src, dst, steps, make_coll_f64(*c));
    if (c->precision == LB_FP32_SHIFTED) return line_t<float>(c, src, dst, steps, make_coll<float>(*c));
    CollFxR k;
    static_cast<CollFx &>(k) = make_coll_fx(c);
    k.range = c->dflag + kFlagRange;
    return line_t<long long>(c, src, dst, steps, k);
}

}  // namespace lbk
