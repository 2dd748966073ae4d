// steps.cu -- many steps of one fixed-point run in one cooperative launch.
//
// A step of a small or middling run is two short kernels whose times are
// latency, not work: on GB300 the push of 5e4 particles takes 5.6 us and the
// cluster solve 7.6 us, of which the arithmetic is well under a microsecond.
// Here the blocks (one per SM) stay resident for all the steps of a call and a
// step has one grid barrier:
//
//   push     each block pushes its contiguous part of the particles and deposits
//            into its own tile (the device code of push.cu).  A thread keeps its
//            first kResident groups of particles in registers from step to step;
//   flush    the tile is added to one of kStepsSlots global accumulators, used
//            in turn;
//   barrier  arrivals counted in global memory, a bounded spin;
//   solve    every block reads the NG sums and solves for the whole grid itself,
//            into its shared copy of E.  No second barrier: the solve is exact
//            integer arithmetic, so all blocks get the same bits, and with one
//            node per thread its cost hardly depends on NG.
//
// Two more blocks (one where the history ring is short: pic_internal.cuh,
// steps_diag_blocks) have no particles.  They take the steps in turn and, while
// the workers go on, compute a step's diagnostics (float64 work that would hold
// the workers up: at 64 clocks a dependent float64 add and 840 a square root,
// a step's take 5 to 10 thousand clocks, up to twice a worker's step), then
// clear the step's accumulator and give it back; a worker waits only if the
// diagnostics fall kStepsSlots - 1 steps behind.  After the last step the
// workers write E, Phi, rho and the consumed sums, each of some nodes.
//
// Up to 6e5 particles on up to 1024 cells the lanes take particles one by one
// (SMALL), beyond that in groups of 4 (16-byte loads; in a small run only a
// longer chain per lane: pic_api.cu, steps_shape).  Groups are whole, which saves the
// loop its tests (3e6 particles, NGP, 13.3 us a step with them, 12.3 so).
//
// What a step costs (GB300, us): launches of push and solve before, and here
//   2e4 particles, 64 cells, one step a call   16.4    9.9
//   3e5, 500 cells, one step a call             -     12.4
//   1e6, 2048 cells, one step a call            -     20.5
//   2e4, 64 cells                              13.4    2.8
//   5e4, 100 cells                             14.0    3.0
//   5e5, 300 cells                             18.5    4.9
//   1e6, 1024 cells, sorted every 20           22.5    8.1
//   3e6, 777 cells, NGP, sorted every 10       27.4   12.3
//   4.2e6, 2048 cells, sorted every 20         31.0   18.1
//   1e6, 4096 cells                            24.8   11.1
//   1.2e7, 2048 cells, sorted every 20         52.9   40.0
// of which, at 5e4 (clocks): push 700, sums 380, flush 1040, barrier 2400 (the
// adds' release and a poll, each a trip to L2), solve 1300 (900 the sums' way
// from L2), E 510.  Counting a node's arrivals in the upper bits of its sum, so
// that a block waits for the sums themselves, saves the release's trip but the
// polls of all nodes hold up the adds: 4.1 us a step at 5e4.  Large runs' pushes
// stream from memory, for which the two launches have more warps, and a thread
// with 8 nodes runs out of registers (1e6 particles on 6000 cells: 31 us against
// 28): set_steps_shape.
//
// The solve in 64 bits.  R_g = N 2^24 - NG rho_q[g] and its prefix sums P_g are
// below N NG 2^24 in magnitude, so they fit 64 bits for N NG <= 2^38 (the
// launch's runs stay below 2^36); sum_g P_g = sum_k (NG - k) R_k and M_g = NG P_g - sum P
// take 128.  The sum over the lanes of a warp is taken in three 26-bit pieces by
// redux.sync.  E_g = k_e (M_g + M_{g-1}) must be the same float32 as the
// float64 chain of field.cu gives, (float)(k_e (double)(M_g + M_{g-1})):
// GB300's float64 pipe takes 2 lanes per clock, so the product is formed from
// the two 64-bit mantissas in integers and rounded once; within 2^14 units of
// 2^-64 of a rounding boundary of float32, where the chain's own three
// roundings (each 2^-53) could matter, the chain itself is evaluated.
//
// Every wait has a limit (kStepsWaitLimit polls, some seconds), after which the block
// sets kErrWait and all blocks return.
#include "steps_common.cuh"

namespace pic {
namespace {

constexpr int kResident = 2;               // groups of particles a thread keeps

// Sum over a warp of 78-bit signed integers, in every lane.
__device__ __forceinline__ i128 warp_sum_i78(i128 v) {
    const unsigned m = (1u << 26) - 1u;
    const unsigned s0 = __reduce_add_sync(kFull, (unsigned)v & m);
    const unsigned s1 = __reduce_add_sync(kFull, (unsigned)(v >> 26) & m);
    const int s2 = __reduce_add_sync(kFull, (int)(v >> 52));
    return (i128)s0 + ((i128)s1 << 26) + ((i128)s2 << 52);
}

__device__ __forceinline__ long long warp_sum_i64(long long v) {
    const unsigned m = (1u << 26) - 1u;
    const unsigned s0 = __reduce_add_sync(kFull, (unsigned)v & m);
    const unsigned s1 = __reduce_add_sync(kFull, (unsigned)(v >> 26) & m);
    const int s2 = __reduce_add_sync(kFull, (int)(v >> 52));
    return (long long)s0 + ((long long)s1 << 26) + ((long long)s2 << 52);
}

// (float)(k (double)m), k > 0 (see above): kmant the mantissa of k with its top
// bit set, k = kmant 2^(kexp - 63).
__device__ __forceinline__ float scaled_f32(i128 m, double k, unsigned long long kmant, int kexp) {
    const bool neg = m < 0;
    const unsigned __int128 a = neg ? (unsigned __int128)(-m) : (unsigned __int128)m;
    const unsigned long long hi = (unsigned long long)(a >> 64), lo = (unsigned long long)a;
    if ((hi | lo) == 0ull) return 0.0f;
    const int n = hi ? __clzll((long long)hi) : 64 + __clzll((long long)lo);
    const unsigned long long A = n >= 64 ? lo << (n - 64) : n ? (hi << n) | (lo >> (64 - n)) : hi;
    unsigned long long p = __umul64hi(A, kmant);
    const int norm = __clzll((long long)p);              // 0 or 1
    p <<= norm;
    // a k = p 2^(65 - n - norm + kexp), p in [2^63, 2^64)
    const int e = 63 + 65 - n - norm + kexp + 127;        // biased float32 exponent
    const unsigned long long rem = p & ((1ull << 40) - 1ull), half = 1ull << 39;
    const unsigned long long dist = rem > half ? rem - half : half - rem;
    if (dist <= (1ull << 14) || e < 1 || e > 253) return (float)(k * i128_to_f64(m));
    const unsigned mant = (unsigned)(p >> 40) + (rem > half ? 1u : 0u);   // 2^24: exponent + 1
    const unsigned bits = ((unsigned)e << 23) + (mant - (1u << 23));
    return __uint_as_float(bits | (neg ? 0x80000000u : 0u));
}

// The W particles of a lane's group, as one word.
template <int W> struct Group { using T = float4; };
template <> struct Group<1> { using T = float; };

// Push and deposit a group's W particles.  The v_old v_new and v_new of a group of 4
// are summed before they join the thread's sums, whose chain of
// float32 adds, the longest part of the rows' error, is so a quarter as long
// (kinetic energy against float64 sums, rms: 2.3e7 Maxwellian particles 1.1e-9
// without and 2.8e-10 so, 5.6e-10 in the push kernel's chains, of two thirds the
// length, without).
template <bool NGP, int W>
__device__ __forceinline__ void step_group(typename Group<W>::T &x, typename Group<W>::T &v,
                                           const float *sE, const Tile &t, const PushConsts &c,
                                           unsigned *err, float &ke, float &mom) {
    using T = typename Group<W>::T;
    alignas(16) float xs[W], vs[W];
    *reinterpret_cast<T *>(xs) = x;
    *reinterpret_cast<T *>(vs) = v;
    float gke = 0.0f, gmom = 0.0f;
#pragma unroll
    for (int k = 0; k < W; k++) {
        if (NGP) push_particle_ngp(xs[k], vs[k], sE, c, W > 1 ? gke : ke, W > 1 ? gmom : mom);
        else push_particle(xs[k], vs[k], sE, c, W > 1 ? gke : ke, W > 1 ? gmom : mom);
    }
    if (W > 1) {
        ke += gke;
        mom += gmom;
    }
    if (NGP) deposit_ngp<W>(t, xs, W, c, err);
    else deposit_cells<W>(t, xs, W, c, err);
    x = *reinterpret_cast<const T *>(xs);
    v = *reinterpret_cast<const T *>(vs);
}

// The field of the whole grid, in thread t's K nodes K t ... K t + K - 1.
template <int K>
struct NodeSolve {
    long long R[K], P[K];         // R_g and its inclusive prefix sums
    unsigned long long q[K];      // the consumed sums
    long long SR;                 // sum of R (threads of warp 0)
    i128 SP;                      // sum of P
    i128 m[K];                    // M_g + M_{g-1}
};

template <int K>
__device__ __forceinline__ void solve_nodes(NodeSolve<K> &s, const StepsArgs &a,
                                            const unsigned long long *acc, int ng,
                                            long long *wr, unsigned long long *ws) {
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, nw = blockDim.x >> 5;
    const int g0 = t * K;
    long long r = 0;
    i128 sp = 0;
#pragma unroll
    for (int j = 0; j < K; j++) s.q[j] = g0 + j < ng ? __ldcg(acc + g0 + j) : 0ull;
#pragma unroll
    for (int j = 0; j < K; j++) {
        const bool in = g0 + j < ng;
        s.R[j] = in ? a.weight_total - (long long)ng * (long long)s.q[j] : 0ll;
        r += s.R[j];
        sp += (i128)s.R[j] * (i128)(ng - (g0 + j));
    }
    long long inc = r;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += u;
    }
    const i128 wsp = warp_sum_i78(sp);
    if (lane == 31) {
        wr[w] = inc;
        ws[w] = (unsigned long long)wsp;
        ws[32 + w] = (unsigned long long)(wsp >> 64);
    }
    __syncthreads();
    const long long wv = lane < nw ? wr[lane] : 0ll;
    const long long before = warp_sum_i64(w == 0 || lane < w ? wv : 0ll);
    s.SR = before;                // in warp 0: the total
    const i128 wq = lane < nw ? (i128)(((unsigned __int128)ws[32 + lane] << 64) | ws[lane]) : (i128)0;
    s.SP = warp_sum_i78(wq);
    long long run = (w == 0 ? 0ll : before) + inc - r;
#pragma unroll
    for (int j = 0; j < K; j++) {
        // M_g = NG P_g - SP, M_{g-1} the same with P_{g-1}, M_{-1} = M_{NG-1}
        const i128 prev = g0 + j == 0 ? (i128)s.SR : (i128)run;
        run += s.R[j];
        s.P[j] = run;
        s.m[j] = (i128)ng * ((i128)run + prev) - 2 * s.SP;
    }
}

// The field of a step in a worker's shared copy of E.
template <int K>
__device__ __forceinline__ void field_step(const StepsArgs &a, const unsigned long long *acc, float *sE) {
    __shared__ long long wr[32];
    __shared__ unsigned long long ws[64];
    const int ng = a.c.ng, tid = threadIdx.x;
    const unsigned long long kb = (unsigned long long)__double_as_longlong(a.k_e);
    const unsigned long long kmant = ((kb & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 11;
    const int kexp = (int)(kb >> 52) - 1023;
    NodeSolve<K> ns;
    solve_nodes<K>(ns, a, acc, ng, wr, ws);
#pragma unroll
    for (int j = 0; j < K; j++) {
        const int g = tid * K + j;
        if (g >= ng) break;
        const float e = scaled_f32(ns.m[j], a.k_e, kmant, kexp);
        sE[g + 1] = e;
        if (g == ng - 1) sE[0] = e;
        if (g == 0) sE[ng + 1] = e;
    }
    __syncthreads();
}

// After the last step: the results, once the sums have been read (a worker's last
// arrival).
template <int K>
__device__ __forceinline__ void last_step(const StepsArgs &a, const unsigned long long *acc, int b,
                                          int workers) {
    __shared__ long long wr[32];
    __shared__ unsigned long long ws[64];
    NodeSolve<K> ns;
    solve_nodes<K>(ns, a, acc, a.c.ng, wr, ws);
    if (threadIdx.x == 0) red_release(a.sync);
    step_results<K, true>(a, ns, b, workers);
}

// The diagnostics of a step.
template <int K>
__device__ __forceinline__ void diag_step(const StepsArgs &a, int s, int workers,
                                          const unsigned long long *acc, const float4 *kv,
                                          unsigned char *smem_raw, unsigned h0) {
    __shared__ long long wr[32];
    __shared__ unsigned long long ws[64];
    NodeSolve<K> ns;
    solve_nodes<K>(ns, a, acc, a.c.ng, wr, ws);
    step_rows<K, true>(a, s, ns, smem_raw, h0, [&](double &k, double &m) {
        const int lane = threadIdx.x & 31;
        float4 p[kStepsMaxGrid / 32];                       // all loads in flight
#pragma unroll
        for (int i = 0; i < kStepsMaxGrid / 32; i++)
            p[i] = 32 * i + lane < workers ? __ldcg(kv + 32 * i + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 1; i < kStepsMaxGrid / 32; i++) {
            add_pair(p[0].x, p[0].y, p[i].x, p[i].y);
            add_pair(p[0].z, p[0].w, p[i].z, p[i].w);
        }
        warp_sum_pairs(p[0], 32);
        k = (double)p[0].x + (double)p[0].y;
        m = (double)p[0].z + (double)p[0].w;
    });
}

// With 4 nodes a thread it is called out of line, so that its registers (a node's
// 128-bit sums, 4 times) are not taken from the push loop: 1.2e7 particles on 4096
// cells 44.6 us a step, 50.2 inlined.  With 1 or 2 they fit beside it (512 cells 34.4
// inlined, 36.0 called).  The diagnostics have a loop of their own for the same
// reason.
template <int K>
__device__ __noinline__ void field_step_call(const StepsArgs &a, const unsigned long long *acc, float *sE) {
    field_step<K>(a, acc, sE);
}

// Block b of a run's workers + nd: all its steps.
template <int VARIANT, int K, bool SMALL>
__device__ __forceinline__ void run_many_steps(const StepsArgs &a, unsigned char *smem_raw, const int b,
                                               const int workers) {
    __shared__ float4 kvs[32];                    // per warp: (ke, ke low, mom, mom low)
    __shared__ int dead;
    constexpr bool kNgp = VARIANT == kDepositNgp;
    constexpr int kW = SMALL ? 1 : 4;             // particles of a group
    using G = typename Group<kW>::T;
    const PushConsts c = a.c;
    const int ng = c.ng;
    const int words = (ng + 2) << a.log_copies, K_ = 1 << a.log_copies;
    const Tile tile0 = make_tile(smem_raw, words, false);
    float *sE = reinterpret_cast<float *>(tile0.n + words);
    Tile tile = tile0;                            // this lane's copy
    tile.w += threadIdx.x & (K_ - 1);
    tile.n += threadIdx.x & (K_ - 1);
    tile.c = tile.n;
    tile.k = a.log_copies;
    const int tid = threadIdx.x, bs = blockDim.x, lane = tid & 31, w = tid >> 5, nw = bs >> 5;
    const int nd = a.diag_blocks;
    const bool diag = b >= workers;
    if (tid == 0) dead = 0;
    auto clear_tile = [&] {
        for (int j = tid; j < words; j += bs) {
            if (!kNgp) tile0.w[j] = 0u;
            tile0.n[j] = 0u;
        }
    };
    clear_tile();
    for (int j = tid; j < ng + 2; j += bs) sE[j] = a.E32[j == 0 ? ng - 1 : (j == ng + 1 ? 0 : j - 1)];
    if (diag) {
        __syncthreads();
        const unsigned h0 = (unsigned)(a.step0 % a.hist_len);             // history slot of the first step
        for (int s = b - workers; s < a.steps; s += nd) {
            const int slot = s % kStepsSlots;
            unsigned long long *acc = a.acc + (size_t)slot * ng;
            const float4 *kv = reinterpret_cast<const float4 *>(a.partials) + (size_t)slot * kStepsMaxGrid;
            if (!wait_step(a, s, workers, false, &dead)) return;
            diag_step<K>(a, s, workers, acc, kv, smem_raw, h0);
            // give the slot back, once no worker reads it any more
            if (!wait_step(a, s + 1, workers, false, &dead)) return;
            for (int g = tid; g < ng; g += bs) acc[g] = 0ull;
            __syncthreads();
            if (tid == 0) red_release(a.sync + 1 + (b - workers));
        }
        return;
    }
    // this block's groups [q0, q1); the thread's groups q0 + tid + i bs, the first
    // kResident of them in registers.  The last N mod kW particles are block 0's.
    const int nq = (int)(a.n / kW), left = (int)(a.n % kW);                     // nq <= 2^30
    const int q0 = (int)((long long)nq * b / workers);
    const int q1 = (int)((long long)nq * (b + 1) / workers);
    G *xg = reinterpret_cast<G *>(a.x);
    G *vg = reinterpret_cast<G *>(a.v);
    G rx[kResident], rv[kResident];
#pragma unroll
    for (int i = 0; i < kResident; i++) {
        const int q = q0 + tid + i * bs;
        rx[i] = q < q1 ? __ldcg(xg + q) : G{};
        rv[i] = q < q1 ? __ldcg(vg + q) : G{};
    }
    __syncthreads();
    for (int s = 0; s < a.steps; s++) {
        const bool last = s == a.steps - 1;
        const int slot = s % kStepsSlots;
        unsigned long long *acc = a.acc + (size_t)slot * ng;
        float4 *kv = reinterpret_cast<float4 *>(a.partials) + (size_t)slot * kStepsMaxGrid;
        float ke = 0.0f, mom = 0.0f;
        const int qs = q0 + tid + kResident * bs;
        G cx = qs < q1 ? __ldcg(xg + qs) : G{}, cv = qs < q1 ? __ldcg(vg + qs) : G{};
#pragma unroll
        for (int i = 0; i < kResident; i++) {
            if (q0 + tid + i * bs < q1) step_group<kNgp, kW>(rx[i], rv[i], sE, tile, c, a.err, ke, mom);
        }
        for (int q = qs; q < q1; q += bs) {
            G xx = cx, vv = cv;
            const int qn = q + bs;
            cx = qn < q1 ? __ldcg(xg + qn) : G{};
            cv = qn < q1 ? __ldcg(vg + qn) : G{};
            step_group<kNgp, kW>(xx, vv, sE, tile, c, a.err, ke, mom);
            __stcg(xg + q, xx);
            __stcg(vg + q, vv);
        }
        if (kW > 1 && b == 0 && tid < left) {
            float *px = a.x + (long long)kW * nq + tid, *pv = a.v + (long long)kW * nq + tid;
            float x1 = __ldcg(px), v1 = __ldcg(pv);
            step_group<kNgp, 1>(x1, v1, sE, tile, c, a.err, ke, mom);
            __stcg(px, x1);
            __stcg(pv, v1);
        }
        float4 sums = make_float4(ke, 0.0f, mom, 0.0f);
        warp_sum_pairs(sums, 32);
        if (lane == 0) kvs[w] = sums;
        __syncthreads();
        if (w == nw - 1) {                        // the block's sums, still as pairs
            float4 p = lane < nw ? kvs[lane] : make_float4(0.f, 0.f, 0.f, 0.f);
            warp_sum_pairs(p, nw);
            if (lane == 0) kv[b] = p;
        }
        // node g: the left weights of cell g + 1 and the right ones of cell g
        // (held by the lane below: a warp's first lane only reads them), node
        // NG - 1 also cell 0's left ones, node 0 cell NG's right ones (NGP: the
        // counts of word g + 1; word NG + 1 is node 0, word 0 stays empty)
        auto cell = [&](int j) {
            u64 n = 0ull, W = 0ull;
#pragma unroll 4
            for (int i = 0; i < K_; i++) {
                const int at = (j << a.log_copies) + ((i + lane) & (K_ - 1));
                if (kNgp) {
                    n += tile0.n[at];
                } else {
                    const CellSum cs = cell_sum(tile0.w[at], tile0.n[at], 0u, false);
                    n += cs.n;
                    W += cs.W;
                }
            }
            return ulonglong2{n, W};
        };
        constexpr int kPer = kNgp ? 32 : 31;                // nodes a warp
        for (int g0 = kPer * w; g0 < ng; g0 += kPer * nw) {
            const int g = kNgp ? g0 + lane : g0 + lane - 1;
            const ulonglong2 own = g < ng ? cell(g + 1) : ulonglong2{0ull, 0ull};
            u64 val = (own.x << kFixBits) - own.y;
            if (!kNgp) val += __shfl_up_sync(kFull, own.y, 1);
            if (g == (kNgp ? 0 : ng - 1)) {
                const ulonglong2 e = cell(kNgp ? ng + 1 : 0);
                val += (e.x << kFixBits) - e.y;
            }
            if (!kNgp && g == 0) val += cell(ng).y;
            if ((kNgp || lane > 0) && g < ng && val) atomicAdd(&acc[g], val);
        }
        __syncthreads();
        if (tid == 0) red_release(a.sync);        // the whole block's adds: after the barrier
        if (!last) clear_tile();                  // while the others arrive
        if (!wait_step(a, s, workers, true, &dead)) return;
        if (last) break;
        if (K >= 4) field_step_call<K>(a, acc, sE);
        else field_step<K>(a, acc, sE);
    }
#pragma unroll
    for (int i = 0; i < kResident; i++) {
        const int q = q0 + tid + i * bs;
        if (q >= q1) break;
        __stcg(xg + q, rx[i]);
        __stcg(vg + q, rv[i]);
    }
    const int slot = (a.steps - 1) % kStepsSlots;
    last_step<K>(a, a.acc + (size_t)slot * ng, b, workers);
}

template <int VARIANT, int K, bool SMALL>
__global__ void __launch_bounds__(1024, 1) pic_steps_kernel(const __grid_constant__ StepsArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    run_many_steps<VARIANT, K, SMALL>(a, smem_raw, blockIdx.x, (int)gridDim.x - a.diag_blocks);
}

// Several runs side by side, each on its own blocks (a.first_block on), none
// waiting for another: the pool's few active runs.
__global__ void __launch_bounds__(1024, 1) pic_steps_pool_kernel(const StepsArgs *runs, int nrun) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(16) StepsArgs a;
    int i = 0;
    while (i + 1 < nrun && (int)blockIdx.x >= runs[i + 1].first_block) i++;
    static_assert(sizeof(StepsArgs) % 4 == 0, "copied by words");
    for (int k = threadIdx.x; k < (int)(sizeof(StepsArgs) / 4); k += blockDim.x)
        reinterpret_cast<unsigned *>(&a)[k] = reinterpret_cast<const unsigned *>(runs + i)[k];
    __syncthreads();
    const int b = (int)blockIdx.x - a.first_block, workers = a.blocks - a.diag_blocks;
    // a lane's 4 particles or fewer: one by one (pic_api.cu, steps_shape)
    if (a.c.ng <= 1024 && a.n <= 4ll * workers * kStepsPoolBlock)
        run_many_steps<kDepositCells, 1, true>(a, smem_raw, b, workers);
    else if (a.c.ng <= 1024) run_many_steps<kDepositCells, 1, false>(a, smem_raw, b, workers);
    else if (a.c.ng <= 2048) run_many_steps<kDepositCells, 2, false>(a, smem_raw, b, workers);
    else run_many_steps<kDepositCells, 4, false>(a, smem_raw, b, workers);
}

using StepsKernel = void (*)(StepsArgs);

template <int V>
StepsKernel pick_nodes(int per_thread, bool small) {
    switch (per_thread) {
        case 1: return small ? &pic_steps_kernel<V, 1, true> : &pic_steps_kernel<V, 1, false>;
        case 2: return &pic_steps_kernel<V, 2, false>;
        case 4: return &pic_steps_kernel<V, 4, false>;
        default: return nullptr;
    }
}

StepsKernel pick_steps(int variant, int ng, int block, bool small) {
    int k = 1;
    while (k * block < ng) k *= 2;
    return variant == kDepositNgp ? pick_nodes<kDepositNgp>(k, small) : pick_nodes<kDepositCells>(k, small);
}

// Copies of a block's tile, lanes alternating between them: lanes of one cell
// then meet on a word half as often, for twice the words to clear and read.
// Two pay in blocks of 1024 threads (1e6 Maxwellian particles on 1024 cells:
// 10.7 against 11.2 us a step, 4e6 on 2048: 22.8 against 24.5; four 10.8 and
// 23.2), not in small ones (4.3 us either way), and not where the deposit only
// counts (NGP).
int log_copies(int variant, int block) { return variant != kDepositNgp && block == 1024 ? 1 : 0; }

size_t steps_smem(int variant, int ng, int block) {
    return (size_t)(ng + 2) * (4 + (8 << log_copies(variant, block)));
}

}  // namespace

cudaError_t steps_prepare(int variant, int ng, int block, bool small, int *per_sm) {
    *per_sm = 0;
    StepsKernel k = pick_steps(variant, ng, block, small);
    if (!k) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)steps_smem(variant, kStepsMaxCells, block));
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k, block,
                                                         steps_smem(variant, ng, block));
}

cudaError_t launch_steps(StepsArgs a, int variant, int grid, int block, bool small, cudaStream_t s) {
    StepsKernel k = pick_steps(variant, a.c.ng, block, small);
    if (!k) return cudaErrorInvalidValue;
    a.log_copies = log_copies(variant, block);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    cooperative(cfg, attr, grid, block, steps_smem(variant, a.c.ng, block), s);
    return cudaLaunchKernelEx(&cfg, k, a);
}

cudaError_t steps_pool_prepare(int *per_sm) {
    const int smem = (int)steps_smem(kDepositCells, kStepsMaxCells, kStepsPoolBlock);
    cudaError_t e = cudaFuncSetAttribute(&pic_steps_pool_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, &pic_steps_pool_kernel,
                                                         kStepsPoolBlock, smem);
}

int steps_pool_copies() { return log_copies(kDepositCells, kStepsPoolBlock); }

cudaError_t launch_steps_pool(const StepsArgs *runs, int nrun, int grid, int ng_max, cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    cooperative(cfg, attr, grid, kStepsPoolBlock, steps_smem(kDepositCells, ng_max, kStepsPoolBlock), s);
    return cudaLaunchKernelEx(&cfg, &pic_steps_pool_kernel, runs, nrun);
}

}  // namespace pic
