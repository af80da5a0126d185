// Marching sweeps: several time steps per launch on large periodic 2D and 3D
// grids, with the intermediate states on chip.
//
// A block owns a window of columns (2D: x positions; 3D: an x-y patch), one
// column per thread, and marches along the slowest axis (the rows of 2D, the
// planes of 3D).  KS steps run as a pipeline of KS stages: in iteration t,
// stage 1 pulls row t of the stored state from global memory and collides it;
// stage s + 1 collides, two rows behind stage s, the state that stage s made;
// stage KS stores.  HBM is read and written once per KS steps, rows are never
// recomputed inside a block's march (only at its two ends), and columns only
// over the KS - 1 outermost columns of each window edge.  The square tiles of
// batch_tb_kernel recompute a halo on four sides (23 % more updates at 4
// steps, 28^2), move every value through shared memory once per step and
// separate their load, step and store phases by barriers; here the loads of
// the next row are in flight while all stages of this one compute, the KS
// collisions of an iteration are independent of each other, and one barrier
// per iteration orders them.
//
// Between two stages, a population that moves within the row goes through
// shared memory (another thread's column reads it) and one that keeps its
// column stays in the thread's registers.  A population with velocity component
// em along the march, made for row r in iteration t, is read in iteration
// t + 2 + em, so rings of 3 + em rows (2, 3, 4) let every iteration write one
// slot while the slots still to be read stay untouched: the slot read is always
// the next one to be overwritten.
//
// The arithmetic per node is the sweep's own collision on the same inputs, so
// the results are bit for bit those of one sweep per launch.  Threads whose
// stage lies outside its valid columns or rows compute on whatever the slots
// hold (fixed point, float) or skip the collision (FP64, whose integer form
// would leave its fast path on such values); nothing of theirs is stored,
// checked or read by a valid node.
#include <algorithm>

#include "lb_device.cuh"

namespace lbk {
// Collision constants as the sweeps take them.
template <typename T> struct MarchK {
    using type = Coll<T>;
    static type make(lb_ctx *c) { return make_coll<T>(*c); }
};
template <> struct MarchK<double> {
    using type = CollF64;
    static type make(lb_ctx *c) { return make_coll_f64(*c); }
};
template <> struct MarchK<long long> {
    using type = CollFxR;
    static type make(lb_ctx *c)
    {
        CollFxR k;
        static_cast<CollFx &>(k) = make_coll_fx(c);
        k.range = c->dflag + kFlagRange;
        return k;
    }
};

template <class L> struct MarchL {
    static constexpr int A = L::D - 1;  // the march axis
    // zero velocity within the row: held in registers
    __host__ __device__ static constexpr bool own(int i)
    {
        for (int a = 0; a < A; ++a)
            if (L::E[i][a] != 0) return false;
        return true;
    }
    // ring slots of the shared populations before i
    __host__ __device__ static constexpr int slot0(int i)
    {
        int s = 0;
        for (int j = 0; j < i; ++j)
            if (!own(j)) s += 3 + L::E[j][A];
        return s;
    }
    static constexpr int kSlots = slot0(L::Q);
    __host__ __device__ static constexpr int pick(int em)  // the register population with march component em
    {
        for (int i = 0; i < L::Q; ++i)
            if (own(i) && L::E[i][A] == em) return i;
        return -1;
    }
};

// 3D windows are 32 columns along x, one warp per row of the patch: a warp's
// loads then cover 8-9 sectors per 8-byte population (16 columns: 5-6 sectors
// for half the columns; 256^3 fixed point 27.4 -> 30.6 GLUPS, FP32 51 -> 62),
// and wider windows leave fewer rows in a block, so more recomputed ones.
constexpr int kMarchW = 32;
// Pad columns before and after the rings: the reads of the outermost columns stay inside the allocation.
template <class L> __host__ __device__ constexpr int march_pad() { return L::D == 3 ? kMarchW + 1 : 2; }
template <class L, int KS, int TH> constexpr size_t march_smem(int elem)
{
    return ((size_t)(KS - 1) * MarchL<L>::kSlots * TH + 2 * (size_t)march_pad<L>()) * elem;
}

// SKIP: a stage outside its rows (the pipeline's fill and drain) does nothing.
// The branch is block-uniform, but ends a scheduling region; where the
// collisions are short (3D float) that costs more than the idle work (256^3:
// 75 against 66 GLUPS), elsewhere less (1024^2 fixed point 76 against 66).
template <class L, typename T, class K, int KS, int TH, bool SKIP>
__device__ __forceinline__ void march_body(const T *__restrict__ src, T *__restrict__ dst, const Geom &g, const K &k,
                                           int x0, int nx, int y0, int ny, int r0, int nr)
{
    constexpr int D = L::D, Q = L::Q, A = D - 1, S = MarchL<L>::kSlots;
    constexpr int IM = MarchL<L>::pick(-1), IC = MarchL<L>::pick(0), IP = MarchL<L>::pick(1);
    extern __shared__ __align__(16) unsigned char march_raw[];
    T *const sm = reinterpret_cast<T *>(march_raw);
    const int tid = threadIdx.x;
    const int NR = D == 3 ? g.N2 : g.N1;  // rows of the march
    constexpr int bw = D == 3 ? kMarchW : TH;
    const int cx = D == 3 ? tid % bw : tid, cy = D == 3 ? tid / bw : 0;
    // stage s is valid on columns s - 1 <= cx < nx + 2 KS - 1 - s (cy likewise): its distance to the window's edge
    int edge = min(cx, nx + 2 * (KS - 1) - 1 - cx);
    if (D == 3) edge = min(edge, min(cy, ny + 2 * (KS - 1) - 1 - cy));

    // offsets of this column's sources within a population: x - ex (and y - ey) wrapped
    auto wrapn = [](int v, int n) {
        v %= n;
        return v < 0 ? v + n : v;
    };
    const int gx = wrapn(x0 - (KS - 1) + cx, g.N0);
    const int gxs[3] = {gx + 1 == g.N0 ? 0 : gx + 1, gx, gx == 0 ? g.N0 - 1 : gx - 1};  // by ex + 1
    int gys[3] = {0, 0, 0};
    if (D == 3) {
        const int gy = wrapn(y0 - (KS - 1) + cy, g.N1);
        gys[0] = (gy + 1 == g.N1 ? 0 : gy + 1) * g.pitch;
        gys[1] = gy * g.pitch;
        gys[2] = (gy == 0 ? g.N1 - 1 : gy - 1) * g.pitch;
    }
    const int64_t rstride = D == 3 ? (int64_t)g.N1 * g.pitch : (int64_t)g.pitch;

    // rows r - 1, r, r + 1 of stage 1, wrapped
    int rc = wrapn(r0 - (KS - 1), NR);
    auto load_row = [&](T(&f)[Q], int r) {
        const T *rows[3] = {src + (r + 1 == NR ? 0 : r + 1) * rstride, src + r * rstride,
                            src + (r == 0 ? NR - 1 : r - 1) * rstride};  // by em + 1
        static_for<0, Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            constexpr int ex = L::E[i][0], ey = D == 3 ? L::E[i][1] : 0, em = L::E[i][A];
            const int col = gxs[ex + 1] + (D == 3 ? gys[ey + 1] : 0);
            f[i] = __ldcg(rows[em + 1] + (int64_t)i * g.slab + col);
        });
    };

    // shared rings: [gap][slot of the population][column]
    T *const mine = sm + march_pad<L>() + tid;
    int w2 = 0, w3 = 0, w4 = 0;  // slot written in this iteration, per ring, in elements

    // register populations between stages: made in the last one (m, c, p), two (c, p) and three (p) iterations
    T hm[KS - 1 > 0 ? KS - 1 : 1], hc[KS - 1 > 0 ? KS - 1 : 1][2], hp[KS - 1 > 0 ? KS - 1 : 1][3];
#pragma unroll
    for (int s = 0; s < KS - 1; ++s) {
        hm[s] = T(0);
        hc[s][0] = hc[s][1] = T(0);
        hp[s][0] = hp[s][1] = hp[s][2] = T(0);
    }

    unsigned acc = 0u;  // fixed point: OR of the high words + 2^29 (|v| < 2^61 check of every stage)
    const int last = nr + 3 * (KS - 1);  // iterations
    T f[Q];
    load_row(f, rc);
    for (int t = 0; t < last; ++t) {
        const int r2 = w2 ? 0 : TH, r3 = w3 == 2 * TH ? 0 : w3 + TH, r4 = w4 == 3 * TH ? 0 : w4 + TH;  // slots read
        T nm, nc, np;  // stage s's register populations, entering the history after stage s + 1 has read it
        static_for<1, KS + 1>([&](auto Si) {
            constexpr int s = decltype(Si)::value;
            // stage s's row of this iteration, counted from the chunk's first row, and where it is valid
            const int row = t - (KS - 1) - 2 * (s - 1);
            const bool rok = row >= s - KS && row < nr + KS - s;  // block-uniform
            const bool ok = rok && edge >= s - 1;
            T n[Q];
            if (!SKIP || rok) {
                if constexpr (s == 1) {
#pragma unroll
                    for (int i = 0; i < Q; ++i) n[i] = f[i];
                } else {
                    constexpr int gp = s - 2;
                    const T *const at = mine + gp * S * TH;
                    static_for<0, Q>([&](auto I) {
                        constexpr int i = decltype(I)::value;
                        constexpr int ex = L::E[i][0], ey = D == 3 ? L::E[i][1] : 0, em = L::E[i][A];
                        if constexpr (i == IM)
                            n[i] = hm[gp];
                        else if constexpr (i == IC)
                            n[i] = hc[gp][1];
                        else if constexpr (i == IP)
                            n[i] = hp[gp][2];
                        else
                            n[i] = at[MarchL<L>::slot0(i) * TH - ex - ey * bw + (em < 0 ? r2 : (em > 0 ? r4 : r3))];
                    });
                }
                if constexpr (std::is_same<T, double>::value) {
                    if (ok) collide(L{}, n, k);
                } else {
                    collide(L{}, n, k);
                }
                if constexpr (std::is_same<K, CollFxR>::value) {
                    unsigned a = 0u;
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        if (i < 1 + 2 * D || ((i - 1 - 2 * D) & 3) < 2)  // a diagonal pair's two values are equal
                            a |= (unsigned)((unsigned long long)n[i] >> 32) + 0x20000000u;
                    }
                    if (ok) acc |= a;
                }
                if constexpr (s < KS) {
                    T *const at = mine + (s - 1) * S * TH;
                    static_for<0, Q>([&](auto I) {
                        constexpr int i = decltype(I)::value;
                        constexpr int em = L::E[i][A];
                        if constexpr (!MarchL<L>::own(i))
                            at[MarchL<L>::slot0(i) * TH + (em < 0 ? w2 : (em > 0 ? w4 : w3))] = n[i];
                    });
                } else if (ok) {
                    T *dp = dst + (r0 + row) * rstride + gxs[1] + gys[1];
#pragma unroll
                    for (int i = 0; i < Q; ++i) dp[(int64_t)i * g.slab] = n[i];
                }
            }
            if constexpr (s > 1) {  // stage s - 1's register populations of this iteration
                constexpr int gp = s - 2;
                hm[gp] = nm;
                hc[gp][1] = hc[gp][0];
                hc[gp][0] = nc;
                hp[gp][2] = hp[gp][1];
                hp[gp][1] = hp[gp][0];
                hp[gp][0] = np;
            }
            if constexpr (s < KS) {
                nm = n[IM];
                nc = n[IC];
                np = n[IP];
            }
            if constexpr (s == 1) {  // the next row's loads fly while the other stages compute
                rc = rc + 1 == NR ? 0 : rc + 1;
                if (t + 1 < nr + 2 * (KS - 1)) load_row(f, rc);
            }
        });
        __syncthreads();
        w2 = r2;
        w3 = r3;
        w4 = r4;
    }
    if constexpr (std::is_same<K, CollFxR>::value) {
        if (__any_sync(0xffffffffu, acc >= 0x40000000u) && (tid & 31) == 0) raise_flag_call(k.range, 1);
    }
}

template <class L, typename T, class K, int KS, int TH, int MINB, bool SKIP>
__global__ void __launch_bounds__(TH, MINB) march_kernel(const T *__restrict__ src, T *__restrict__ dst, Geom g, K k,
                                                         MarchPlan p)
{
    unsigned b = blockIdx.x;
    const int x0 = (int)(b % (unsigned)p.nx) * p.bx;
    b /= (unsigned)p.nx;
    const int y0 = L::D == 3 ? (int)(b % (unsigned)p.ny) * p.by : 0;
    const int r0 = (L::D == 3 ? (int)(b / (unsigned)p.ny) : (int)b) * p.chunk;
    const int NR = L::D == 3 ? g.N2 : g.N1;
    march_body<L, T, K, KS, TH, SKIP>(src, dst, g, k, x0, min(p.bx, g.N0 - x0), y0,
                                      L::D == 3 ? min(p.by, g.N1 - y0) : 1, r0, min(p.chunk, NR - r0));
}

// Batched 2D instances: the block's window, chunk and instance from tables.
template <typename T, int KS, int TH, int MINB>
__global__ void __launch_bounds__(TH, MINB) march_batch_kernel(const InstDesc<T> *__restrict__ inst,
                                                               const MarchBlock *__restrict__ blocks,
                                                               const T *__restrict__ src, T *__restrict__ dst)
{
    const MarchBlock b = blocks[blockIdx.x];
    const InstDesc<T> d = inst[b.inst];
    march_body<D2Q9, T, typename CollOf<T>::type, KS, TH, true>(src + d.off, dst + d.off, d.g, d.k, b.x0, b.nx, 0, 1, b.r0,
                                                                b.nr);
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
// Cut `n` into the fewest near-equal parts of at most `most`.
static void cut(int n, int most, int &parts, int &size)
{
    parts = (n + most - 1) / most;
    size = (n + parts - 1) / parts;
    parts = (n + size - 1) / size;
}

// What marching has to offer against one sweep per launch (march_setup).
struct MarchRule {
    int64_t least, nodes;  // at least so many nodes, for short calls and for all
    double use;     // of a launch's thread-iterations at least this share ends in stored nodes
    double full;    // 2D, below 450000 nodes, all calls: the same with as many blocks on every SM as on the fullest
    // 3D: us per step and unit of the plan's model, less than the sweeps' us per 1000
    // nodes, lanes of the rows' warps, and nodes beyond 650000 (no longer in L2), replayed
    // from a graph; launched one by one a sweep takes about 2.5 us more
    double unit, node, lane, far;
};

template <class L, typename T, int KS, int TH, int MINB, bool SKIP> struct March {
    using KT = typename MarchK<T>::type;
    static constexpr int kRing = KS - 1;

    // The cheapest cut by a model of the launch: full waves of the resident
    // blocks, each as long as its iterations (its rows, the pipeline's fill and
    // about 4 rows of latency), an iteration taking the time of the warps at
    // work, or of 0.7 of a full SM's where fewer no longer hide latency (0.85 of the
    // one block per SM in 3D).  In 3D also more, lower windows than the rings have
    // room for, in blocks of fewer warps, where they fill the SMs better
    // (101 x 90 x 77 FP32: 36 windows of 10 rows by 4 chunks on 152 SMs instead of
    // 32 of 12, 50 GLUPS against 44).
    static void plan(const lb_ctx *c, const MarchRule &rule, MarchPlan *out, MarchWorth *worth)
    {
        const Geom &g = c->geom;
        *out = MarchPlan{};
        *worth = kMarchNo;
        if (g.slab >= (1ll << 30)) return;  // offsets within a population are int
        const int NR = L::D == 3 ? g.N2 : g.N1, high = TH / kMarchW;
        MarchPlan p{};
        p.steps = KS;
        cut(g.N0, (L::D == 3 ? kMarchW : TH) - 2 * kRing, p.nx, p.bx);
        const int64_t slots = (int64_t)c->sms * MINB;
        double least = 1e300;
        for (int extra = 0; extra <= (L::D == 3 ? 8 : 0); ++extra) {
            p.ny = p.by = 1;
            if (L::D == 3) {
                cut(g.N1, high - 2 * kRing, p.ny, p.by);
                cut(g.N1, (g.N1 + p.ny + extra - 1) / (p.ny + extra), p.ny, p.by);
            }
            p.threads = L::D == 3 ? kMarchW * (p.by + 2 * kRing) : TH;  // 3D: a warp is a row of the window
            const double rows = L::D == 3 ? (double)(p.by + 2 * kRing) / high : 1.0;  // of the most warps that a block has
            const int64_t win = (int64_t)p.nx * p.ny;
            for (int nc = 1; nc <= NR; ++nc) {
                const int chunk = (NR + nc - 1) / nc;
                if (nc > 1 && chunk < 4 * kRing) break;
                const int64_t blocks = win * ((NR + chunk - 1) / chunk);
                const int64_t waves = (blocks + slots - 1) / slots;
                if (blocks > 0x7fffffff || (out->chunk && waves > 64)) break;
                const double resident = (double)((blocks + waves * c->sms - 1) / (waves * c->sms));
                const double t = (double)waves * (chunk + 3 * kRing + 4) * std::max(resident * rows, (L::D == 3 ? 0.85 : 0.7) * MINB);
                if (t < least) {
                    least = t;
                    p.chunk = chunk;
                    p.nc = (NR + chunk - 1) / chunk;
                    *out = p;
                }
            }
        }
        if (out->chunk == 0) {  // more windows than a launch has blocks
            *out = MarchPlan{};
            return;
        }
        const int64_t blocks = (int64_t)out->nx * out->ny * out->nc, waves = (blocks + slots - 1) / slots;
        const int64_t filled = (blocks + waves * c->sms - 1) / (waves * c->sms) * waves * c->sms;
        const double each = (double)out->threads * (out->chunk + 3 * kRing), nodes = (double)c->nodes;
        if (c->nodes < rule.least || nodes / (blocks * each) < rule.use) return;
        const double lanes = (double)g.nseg * 32 * lane_width<L, T>();
        const double less = L::D == 3 ? 1e-3 * (rule.node * nodes + rule.lane * lanes + rule.far * std::max(0.0, nodes - 650000)) -
                                            rule.unit * least / KS
                                      : 0.0;  // us per step
        const bool full = L::D == 3 || c->nodes >= 450000 || nodes / (filled * each) >= rule.full;
        *worth = c->nodes >= rule.nodes && full && less >= 0.0 ? kMarchYes : (less > -2.5 ? kMarchShort : kMarchNo);
    }
    static const void *kernel() { return (const void *)march_kernel<L, T, KT, KS, TH, MINB, SKIP>; }
    static cudaError_t setup(lb_ctx *c, const MarchRule &rule, MarchPlan *out, MarchWorth *worth)
    {
        plan(c, rule, out, worth);
        return cudaFuncSetAttribute(kernel(), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)march_smem<L, KS, TH>(sizeof(T)));
    }
    static cudaError_t launch(lb_ctx *c, const void *src, void *dst, cudaStream_t s)
    {
        const MarchPlan &p = c->march;
        march_kernel<L, T, KT, KS, TH, MINB, SKIP>
            <<<(unsigned)((int64_t)p.nx * p.ny * p.nc), p.threads, march_smem<L, KS, TH>(sizeof(T)), s>>>(
                (const T *)src, (T *)dst, c->geom, MarchK<T>::make(c), p);
        return cudaGetLastError();
    }
};

// Steps per launch, threads and blocks per SM, as measured at 4096^2 and 256^3
// (GLUPS).  More steps than these need rings that leave too little L1 for the
// rows in flight, or registers that leave too few warps.
//   2D fixed point: 3 steps, 64 threads x 10: 108.5 (2 steps: 88; 4: 96; 256 x 2: 104)
//   2D FP32:        5 steps, 128 x 5: 315 (4 steps: 276; 6: 297; 128 x 7 at 4 steps: 227)
//   2D FP64:        2 steps, 128 x 6: 52 (3 steps: 50.6; 256 x 3: 47)
//   3D fixed point: 2 steps, 416 x 1: 35.5 (512: 32; 384: 33.5)
//   3D FP32:        3 steps, 512 x 1: 75 (2 steps: 62; 448: 71)
// 3D FP64 (19 integer-form collisions' worth of registers) was slower than one
// sweep per launch, and 4D has no room for a window.
using March2Fx = March<D2Q9, long long, 3, 64, 10, true>;
using March2F = March<D2Q9, float, 5, 128, 5, true>;
using March2D = March<D2Q9, double, 2, 128, 6, true>;
using March3Fx = March<D3Q19, long long, 2, 416, 1, true>;
using March3F = March<D3Q19, float, 3, 512, 1, false>;

// Where marching beats one sweep per launch, replayed from graphs (GLUPS, march / sweep):
//   2D fixed point 256^2 16 / 20, 384^2 29 / 31, 526^2 58 / 49, 1024^2 76 / 43, 1999x1501 94 / 44, 4096^2 108 / 47
//   2D FP32        256^2 22 / 23, 384^2 50 / 46, 526^2 84 / 79, 1024^2 194 / 124, 1999x1501 258 / 85, 4096^2 315 / 97
//   2D FP64        768^2 34 / 40, 1024^2 37 / 39, 1999x1501 48 / 42, 4096^2 52 / 47
//   3D fixed point 67^3 22 / 19, 101x90x77 26 / 20, 126^3 30 / 22, 256^3 36 / 23
//   3D FP32        72^3 42 / 48, 87^3 46 / 48, 93^3 51 / 45, 101x90x77 49 / 51, 106^3 53 / 42, 126^3 57 / 43, 256^3 75 / 46
// 2D grids of 0.2M to 0.45M nodes are one wave of few blocks per SM, as long as the
// fullest SM's: us per step, march / sweep, fixed point 526^2 (4 blocks on every SM)
// 4.8 / 5.7, 263 x 1052 (5 on some) 6.15 / 5.6, 448^2 4.8 / 4.7; FP32 427^2 2.9 / 2.7, 6036 x
// 30 4.1 / 2.95, 526^2 3.3 / 3.5 (the smaller ones mostly fit tiles, faster than either).
// In 3D a few planes, or rows that fill the sweep's warps, favour the sweeps: FP32
// 126x31x126 10.3 / 8.0, 234x234x15 20.8 / 16.8, 50x200x50 10.6 / 13.2; fixed point
// 169x169x11 14.3 / 13.6, 27x106x106 12.3 / 19.9.  The 3D costs are fitted to 70 grids of
// 0.3M to 2M nodes; none of them is slower by the rule.  Sweeps of calls shorter than
// a graph cost 2 us more each, and there the windows still pay on many of these (FP32
// 101x90x77 14.2 / 16.4, 79^3 10.3 / 12.3; fixed point 169x169x11 14.3 / 16.4, 263 x 1052 6.15 / 7.7).
cudaError_t march_setup(lb_ctx *c, MarchPlan *plan, MarchWorth *worth)
{
    *plan = MarchPlan{};
    *worth = kMarchNo;
    if (c->geom.mirror) return cudaSuccess;
    if (c->d == 2) {
        if (c->precision == LB_FX64) return March2Fx::setup(c, {200000, 240000, 0.45, 0.47}, plan, worth);
        if (c->precision == LB_FP32_SHIFTED) return March2F::setup(c, {180000, 240000, 0.45}, plan, worth);
        return March2D::setup(c, {1800000, 1800000, 0.8}, plan, worth);
    }
    if (c->d == 3) {
        if (c->precision == LB_FX64) return March3Fx::setup(c, {300000, 300000, 0.4, 0.0, 1.9, 0.026, 0.017}, plan, worth);
        if (c->precision == LB_FP32_SHIFTED) return March3F::setup(c, {350000, 350000, 0.3, 0.0, 1.57, 0.009, 0.0069, 0.014}, plan, worth);
    }
    return cudaSuccess;
}

cudaError_t march_launch(lb_ctx *c, const void *src, void *dst, cudaStream_t s)
{
    if (c->d == 2) {
        if (c->precision == LB_FX64) return March2Fx::launch(c, src, dst, s);
        if (c->precision == LB_FP32_SHIFTED) return March2F::launch(c, src, dst, s);
        return March2D::launch(c, src, dst, s);
    }
    if (c->precision == LB_FX64) return March3Fx::launch(c, src, dst, s);
    return March3F::launch(c, src, dst, s);
}

// ---------------------------------------------------------------------------
// Batched 2D instances.
// ---------------------------------------------------------------------------
template <typename T, int KS, int TH, int MINB> struct MarchB {
    // Chunks of at most c rows, c the cheapest by a model of the launch: the
    // longest block's iterations (latency), and twice the mean block's work per
    // wave of resident blocks (its rows, the recomputed ones and about 6 rows of
    // fill).  Against chunks of 8 to 512 rows measured one by one on 7 batches
    // (8 to 512 instances of 32^2 to 512^2) in each precision, its choice was
    // 1.4 % above the fastest in the mean and 8 % at the most.  The longest blocks
    // start first.
    static void plan(const lb_ctx *inst, int count, int sms, std::vector<MarchBlock> *out, int *steps, int *threads, int *cols,
                     int *resident)
    {
        constexpr int ring = KS - 1;
        *steps = KS;
        *resident = sms * MINB;
        *threads = TH;
        *cols = TH - 2 * ring;
        const double slots = (double)sms * MINB;
        double least = 1e300;
        int best = 16;
        for (int c = 8; c <= 65536; c += std::max(1, c / 8)) {
            double work = 0.0, blocks = 0.0;
            int longest = 0, highest = 0;
            for (int j = 0; j < count; ++j) {
                int nx, bx, nc, ch;
                cut((int)inst[j].N[0], TH - 2 * ring, nx, bx);
                cut((int)inst[j].N[1], c, nc, ch);
                blocks += (double)nx * nc;
                work += (double)nx * nc * (ch + ring + 6);
                longest = std::max(longest, ch + 3 * ring);
                highest = std::max(highest, (int)inst[j].N[1]);
            }
            const double t = longest + 2.0 * ceil(blocks / slots) * work / blocks;
            if (t < least) {
                least = t;
                best = c;
            }
            if (c >= highest) break;
        }
        out->clear();
        for (int j = 0; j < count; ++j) {
            const int n0 = (int)inst[j].N[0], n1 = (int)inst[j].N[1];
            int nx, bx, nc, ch;
            cut(n0, TH - 2 * ring, nx, bx);
            cut(n1, best, nc, ch);
            for (int r = 0; r < n1; r += ch)
                for (int x = 0; x < n0; x += bx) out->push_back({j, x, std::min(bx, n0 - x), r, std::min(ch, n1 - r)});
        }
        std::stable_sort(out->begin(), out->end(), [](const MarchBlock &a, const MarchBlock &b) { return a.nr > b.nr; });
    }
    static cudaError_t launch(const void *desc, const MarchBlock *blocks, int n, const void *src, void *dst, cudaStream_t s)
    {
        constexpr size_t smem = march_smem<D2Q9, KS, TH>(sizeof(T));
        static_assert(smem <= 48 * 1024, "no opt-in needed");
        march_batch_kernel<T, KS, TH, MINB><<<(unsigned)n, TH, smem, s>>>((const InstDesc<T> *)desc, blocks, (const T *)src,
                                                                          (T *)dst);
        return cudaGetLastError();
    }
};

// Variant 0 is a new batch's own choice.  Instances of 32 to 512 columns leave
// fewer of a 64-thread window's columns idle: FP32 21.4M nodes 230 GLUPS
// against 215 with 128 threads, 0.65M 129 against 112; fixed point about equal.
template <class F> static void march_batch_pick(int precision, int variant, F &&f)
{
    if (precision == LB_FX64) {
        if (variant == 0)
            f(MarchB<long long, 3, 64, 10>{});
        else
            f(MarchB<long long, 3, 128, 5>{});
    } else if (precision == LB_FP32_SHIFTED) {
        if (variant == 0)
            f(MarchB<float, 5, 64, 10>{});
        else
            f(MarchB<float, 5, 128, 5>{});
    } else {
        f(MarchB<double, 2, 128, 6>{});
    }
}

int march_batch_variants(int precision) { return precision == LB_FP64 ? 1 : 2; }

void march_batch_plan(const lb_ctx *inst, int count, int precision, int variant, int sms, std::vector<MarchBlock> *blocks,
                      int *steps, int *threads, int *cols, int *resident)
{
    march_batch_pick(precision, variant,
                     [&](auto m) { decltype(m)::plan(inst, count, sms, blocks, steps, threads, cols, resident); });
}

cudaError_t march_batch_launch(int precision, int variant, const void *desc, const MarchBlock *blocks, int n,
                               const void *src, void *dst, cudaStream_t s)
{
    cudaError_t e = cudaSuccess;
    march_batch_pick(precision, variant, [&](auto m) { e = decltype(m)::launch(desc, blocks, n, src, dst, s); });
    return e;
}

}  // namespace lbk
