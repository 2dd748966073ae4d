// push.cu -- the fused particle kernel of one PIC step: field gather (Sec.
// 2.3), velocity update (Sec. 2.1, Eq. 3), position update and periodic wrap
// (Sec. 2.1, Eq. 2; Appendix A wrap), and the charge deposit of the new
// positions (Sec. 2.3).
//
// Design (GB300): one persistent grid of (SMs x resident blocks), each block
// streaming float4 groups of 4 particles (the cell coordinates u = x NG/L and
// the velocities v are separate float32 arrays,
// 16 B loads and stores, streaming cache hints: the particle arrays are read
// and written once per step and do not fit in L2).  The block stages E in
// shared memory and accumulates a private density tile there; the tile is
// added to the global density with one 64-bit atomic per non-zero node when
// the block ends.  The deposit is exact integer arithmetic (2^-24 fractions
// of a particle), so the density is the same integer whatever the launch
// shape, the particle order or the deposit variant.
//
// Deposit variants (all give the same integers):
//   ATOMIC        per cell, a count and a sum of right weights: an add of 1 and one
//                 fetch-add per particle (particle_ops.cuh, cell tiles);
//   MATCH         lanes of a warp whose particles share a left node are
//                 grouped by __match_any_sync; the group's weights are summed
//                 by __reduce_add_sync and its first lane does two atomics;
//   QUAD          runs of equal left node among a thread's 4 particles are
//                 summed in registers, then two atomics per run;
//   PAIR          the same with two open runs, so that particles of two
//                 interleaved cells (the two beams before the first sort)
//                 still combine.
// The nearest-grid-point shape (PIC_SHAPE_NGP) uses the same loop with the
// NGP gather and counts the particles of each cell.
// The tiles hold exact 64-bit sums in two 32-bit words (particle_ops.cuh).
#include "particle_ops.cuh"
#include "push64.cuh"

namespace pic {
namespace {


// Add the block's tile to the global density (ghost nodes folded onto their
// periodic images).
template <int VARIANT>
__device__ __forceinline__ void flush_tile(const Tile &t, u64 *rho_q, int ng) {
    __syncthreads();
    for (int j = threadIdx.x; j <= ng + 1; j += blockDim.x) {
        const u64 v = tile_node<VARIANT>(t, j, ng);
        if (v) atomicAdd(&rho_q[j == 0 ? ng - 1 : (j == ng + 1 ? 0 : j - 1)], v);
    }
}

// Sum two per-thread values over the block in a fixed order; thread 0 gets it.
__device__ __forceinline__ void block_sum2(double &a, double &b, double *scratch) {
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(kFull, a, o);
        b += __shfl_down_sync(kFull, b, o);
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = (blockDim.x + 31) >> 5;
    if (lane == 0) { scratch[2 * w] = a; scratch[2 * w + 1] = b; }
    __syncthreads();
    if (w == 0) {
        a = lane < nw ? scratch[2 * lane] : 0.0;
        b = lane < nw ? scratch[2 * lane + 1] : 0.0;
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(kFull, a, o);
            b += __shfl_down_sync(kFull, b, o);
        }
    }
}

// One block-iteration covers U*blockDim consecutive float4 groups; thread t
// takes groups q0 + u*blockDim + t (coalesced for each u).  The next
// iteration's groups are loaded before the current ones are processed.
template <int VARIANT, bool PUSH, int U>
__global__ void __launch_bounds__(512) pic_push_fixed_kernel(PushArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ double red[64];
    const PushConsts c = a.c;
    const int ng = c.ng;
    float *sE = reinterpret_cast<float *>(smem_raw);                 // ng + 2
    const Tile tile = make_tile(smem_raw + 4 * (ng + 2), ng + 2, a.wide);
    const int tid = threadIdx.x, bs = blockDim.x, lane = tid & 31;
    cudaTriggerProgrammaticLaunchCompletion();
    for (int j = tid; j < ng + 2; j += bs) {
        tile.w[j] = 0u;
        tile.n[j] = 0u;
        tile.c[j] = 0u;
    }
    cudaGridDependencySynchronize();
    if (PUSH)
        for (int j = tid; j < ng + 2; j += bs) sE[j] = a.E32[j == 0 ? ng - 1 : (j == ng + 1 ? 0 : j - 1)];
    __syncthreads();

    float ke = 0.0f, mom = 0.0f;
    const long long n4 = a.n >> 2;
    float4 *x4 = reinterpret_cast<float4 *>(a.x);
    float4 *v4 = reinterpret_cast<float4 *>(a.v);
    const long long span = (long long)bs * U;
    const long long stride = (long long)gridDim.x * span;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 cx[U], cv[U];
    long long q0 = (long long)blockIdx.x * span;
#pragma unroll
    for (int u = 0; u < U; u++) {
        const long long q = q0 + u * bs + tid;
        cx[u] = q < n4 ? __ldcs(x4 + q) : zero4;
        cv[u] = (PUSH && q < n4) ? __ldcs(v4 + q) : zero4;
    }
    // The trip count is uniform over the block (q0 is), so every warp is
    // converged for the MATCH variant's warp votes.
    for (; q0 < n4; q0 += stride) {
        float4 nx[U], nv[U];
        const long long q1 = q0 + stride;
#pragma unroll
        for (int u = 0; u < U; u++) {
            const long long q = q1 + u * bs + tid;
            nx[u] = q < n4 ? __ldcs(x4 + q) : zero4;
            nv[u] = (PUSH && q < n4) ? __ldcs(v4 + q) : zero4;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const long long q = q0 + u * bs + tid;
            const bool valid = q < n4;
            float4 xx = cx[u], vv = cv[u];
            if (PUSH && valid) {
                if (VARIANT == kDepositNgp) {
                    push_particle_ngp(xx.x, vv.x, sE, c, ke, mom);
                    push_particle_ngp(xx.y, vv.y, sE, c, ke, mom);
                    push_particle_ngp(xx.z, vv.z, sE, c, ke, mom);
                    push_particle_ngp(xx.w, vv.w, sE, c, ke, mom);
                } else {
                    push_particle(xx.x, vv.x, sE, c, ke, mom);
                    push_particle(xx.y, vv.y, sE, c, ke, mom);
                    push_particle(xx.z, vv.z, sE, c, ke, mom);
                    push_particle(xx.w, vv.w, sE, c, ke, mom);
                }
            }
            deposit4<VARIANT>(tile, xx, valid, c, a.err, lane);
            if (PUSH && valid) {
                __stcs(x4 + q, xx);
                __stcs(v4 + q, vv);
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++) { cx[u] = nx[u]; cv[u] = nv[u]; }
    }
    // The last N mod 4 particles: warp 0 of block 0, converged.
    if (blockIdx.x == 0 && tid < 32) {
        const long long i = n4 * 4 + lane;
        const bool valid = i < a.n;
        float xs = valid ? a.x[i] : 0.0f, vs = valid && PUSH ? a.v[i] : 0.0f;
        if (PUSH && valid) {
            if (VARIANT == kDepositNgp) push_particle_ngp(xs, vs, sE, c, ke, mom);
            else push_particle(xs, vs, sE, c, ke, mom);
        }
        deposit_one<VARIANT>(tile, xs, valid, c, a.err, lane);
        if (PUSH && valid) { a.x[i] = xs; a.v[i] = vs; }
    }
    if (PUSH) {
        double dke = ke, dmom = mom;
        __syncthreads();
        block_sum2(dke, dmom, red);
        if (tid == 0) {
            a.partials[2 * blockIdx.x] = dke;
            a.partials[2 * blockIdx.x + 1] = dmom;
        }
    }
    flush_tile<VARIANT>(tile, a.rho_q, ng);
}

// ---- the fused push on 8-particle groups (QUAD8, PAIR8) ---------------------
//
// The same step, each thread taking 8 consecutive particles per group: one
// 32-byte vector load (and store) per array, lanes of a warp on consecutive
// groups (1 KB per warp and array, coalesced), and the deposit's runs of
// equal cell merged over all 8 particles, which halves the shared-memory
// atomics where neighbours share a cell (a sorted state, cold beams).
template <int VARIANT, bool PUSH, int U>
__global__ void __launch_bounds__(512) pic_push_oct_kernel(PushArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ double red[64];
    const PushConsts c = a.c;
    const int ng = c.ng;
    float *sE = reinterpret_cast<float *>(smem_raw);                 // ng + 2
    const Tile tile = make_tile(smem_raw + 4 * (ng + 2), ng + 2, a.wide);
    const int tid = threadIdx.x, bs = blockDim.x, lane = tid & 31;
    cudaTriggerProgrammaticLaunchCompletion();
    for (int j = tid; j < ng + 2; j += bs) {
        tile.w[j] = 0u;
        tile.n[j] = 0u;
        tile.c[j] = 0u;
    }
    cudaGridDependencySynchronize();
    if (PUSH)
        for (int j = tid; j < ng + 2; j += bs) sE[j] = a.E32[j == 0 ? ng - 1 : (j == ng + 1 ? 0 : j - 1)];
    __syncthreads();

    float ke = 0.0f, mom = 0.0f;
    const long long n8 = a.n >> 3;
    const long long span = (long long)bs * U;
    const long long stride = (long long)gridDim.x * span;
    F8 zero8;
#pragma unroll
    for (int k = 0; k < 8; k++) zero8.v[k] = 0.0f;
    // no loads ahead: a group's 16 values per thread are its registers'
    // worth, and three resident blocks hide the load latency instead
    for (long long q0 = (long long)blockIdx.x * span; q0 < n8; q0 += stride) {
        F8 cx[U], cv[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const long long q = q0 + u * bs + tid;
            cx[u] = q < n8 ? ld8(a.x + 8 * q) : zero8;
            cv[u] = (PUSH && q < n8) ? ld8(a.v + 8 * q) : zero8;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const long long q = q0 + u * bs + tid;
            const bool valid = q < n8;
            F8 xx = cx[u], vv = cv[u];
            if (PUSH && valid) {
#pragma unroll
                for (int k = 0; k < 8; k++) push_particle(xx.v[k], vv.v[k], sE, c, ke, mom);
            }
            deposit_group<VARIANT, 8>(tile, xx.v, valid, c, a.err, lane);
            if (PUSH && valid) {
                st8(a.x + 8 * q, xx);
                st8(a.v + 8 * q, vv);
            }
        }
    }
    // The last N mod 8 particles: warp 0 of block 0, converged.
    if (blockIdx.x == 0 && tid < 32) {
        const long long i = n8 * 8 + lane;
        const bool valid = i < a.n;
        float xs = valid ? a.x[i] : 0.0f, vs = valid && PUSH ? a.v[i] : 0.0f;
        if (PUSH && valid) push_particle(xs, vs, sE, c, ke, mom);
        deposit_one<VARIANT>(tile, xs, valid, c, a.err, lane);
        if (PUSH && valid) { a.x[i] = xs; a.v[i] = vs; }
    }
    if (PUSH) {
        double dke = ke, dmom = mom;
        __syncthreads();
        block_sum2(dke, dmom, red);
        if (tid == 0) {
            a.partials[2 * blockIdx.x] = dke;
            a.partials[2 * blockIdx.x + 1] = dmom;
        }
    }
    flush_tile<VARIANT>(tile, a.rho_q, ng);
}

// ---- float32 push with float32 atomic deposit (precision study) -------------
//
// Groups of 4 particles per thread and loads ahead, as the fixed-point push.
// A float32 add on shared memory is a compare-and-swap loop, and lanes that hit
// one node go through it one after the other: that is what bounds the kernel.
// So two open runs per thread are summed in registers first (PAIR), and the
// block keeps `copies` sums per node, side by side, lane l adding to copy
// l mod copies: lanes of one cell then meet on an address copies times less
// often, and with 32 copies a warp's lanes never meet and use a bank each.
// Measured (2^24 particles, 1024 cells, the mean over sort periods): 60 us a push
// with 32 copies (2^24 on 4096 cells, 8 copies: 73), 68 with 16, against 295 us with one copy and a shuffle sum
// where a whole warp holds one run, and 140 us (sorted) to 380 us (lattice
// order) with two adds per particle.
// As many copies as fit beside E, at most 32: in 216 KB for a block of 1024
// threads (its 50 registers leave room for one per SM), in 72 KB for smaller
// ones, so that two of 512 keep their place; open shapes take the large block
// where it holds more copies.  us a push, 2^24 particles sorted every 20 steps, in
// two blocks of 512 and one of 1024: 256 cells (32 copies either way) 58.9, 62.3;
// 1024 66.9, 59.6; 1600 78.5, 62.8; 2048 77.2, 65.1; 4096 83.5, 70.3; 8192 82.7,
// 72.1; 4e6 on 1600 28.1, 25.1; 1e6 on 4096 18.1, 18.1.  (Three of 512 threads and
// 40 registers: 10 us more on 1024 cells, the loops fail more often.)
constexpr size_t kAtomicShared = 216 * 1024, kAtomicSharedSmall = 72 * 1024;

int atomic_copies(int ng, int block) {
    const size_t most = block > 512 ? kAtomicShared - 4 * (size_t)(ng + 2) : kAtomicSharedSmall;
    int k = 32;
    while (k > 1 && (size_t)(ng + 2) * 4 * k > most) k /= 2;
    return k;
}

// A thread takes 4 particles at a time where one block of 256 had one, so plain
// float32 sums of v_old v_new and v_new have longer chains, and more of their rounding
// in the rows.  The sums are therefore pairs of float32, to which few particles are
// added one by one (EXACT), many in groups of 4.  Kinetic energy against exact sums,
// rms: 2e4 particles 1.3e-10 (4.9e-10 with plain chains, 2.2e-10 with one particle a
// thread), 1e6 2.8e-11 (1.0e-10, 8.2e-11), 2^22 1.9e-11 (1.8e-10, 1.2e-10), in groups
// 3e-11, 2^24 2.2e-11 (3.8e-10, 1.5e-10).  us a step, one by one and in groups: 4e6 on
// 1600 cells 28.2, 26.4; 2^24 on 1024 (in an older loop) 67.4, 63.4.
constexpr long long kAtomicExact = 1 << 22;

template <bool PUSH, bool EXACT>
__global__ void __launch_bounds__(1024) pic_push_f32atomic_kernel(PushArgsF32Atomic a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ float4 red[32];                            // per warp: (ke, ke low, mom, mom low)
    const PushConsts c = a.c;
    const int ng = c.ng;
    float *sE = reinterpret_cast<float *>(smem_raw);      // ng + 2, ghost-padded
    float *sRho = sE + ng + 2;                            // [ng + 2][copies], ghost-padded
    const int tid = threadIdx.x, bs = blockDim.x, K = a.copies;
    cudaTriggerProgrammaticLaunchCompletion();
    for (int j = tid; j < (ng + 2) * K; j += bs) sRho[j] = 0.0f;
    cudaGridDependencySynchronize();
    for (int j = tid; j < ng + 2; j += bs)
        if (PUSH) sE[j] = a.E32[j == 0 ? ng - 1 : (j == ng + 1 ? 0 : j - 1)];
    __syncthreads();
    float *mine = sRho + (tid & (K - 1));                 // this lane's copy
    auto add = [&](unsigned key, float l, float r) {
        atomicAdd(&mine[key * K], l);
        atomicAdd(&mine[(key + 1) * K], r);
    };
    float4 sums = make_float4(0.f, 0.f, 0.f, 0.f);        // (ke, ke low, mom, mom low)
    float gke = 0.0f, gmom = 0.0f;                        // of a group
    auto join = [&] {
        if (EXACT) {
            add_pair(sums.x, sums.y, gke, 0.0f);
            add_pair(sums.z, sums.w, gmom, 0.0f);
        } else {
            add_fast(sums.x, sums.y, gke);
            add_fast(sums.z, sums.w, gmom);
        }
        gke = gmom = 0.0f;
    };
    auto push = [&](float &x, float &v) {
        push_particle(x, v, sE, c, gke, gmom);
        if (EXACT) join();
    };
    const unsigned n4 = (unsigned)(a.n >> 2), stride = gridDim.x * (unsigned)bs;     // N < 2^32
    float4 *x4 = reinterpret_cast<float4 *>(a.x);
    float4 *v4 = reinterpret_cast<float4 *>(a.v);
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const unsigned q0 = blockIdx.x * (unsigned)bs + (unsigned)tid;
    float4 cx = q0 < n4 ? __ldcs(x4 + q0) : zero4;
    float4 cv = PUSH && q0 < n4 ? __ldcs(v4 + q0) : zero4;
    for (unsigned q = q0; q < n4; q += stride) {
        const unsigned qn = q + stride;
        const float4 nx = qn < n4 ? __ldcs(x4 + qn) : zero4;
        const float4 nv = PUSH && qn < n4 ? __ldcs(v4 + qn) : zero4;
        float xs[4] = {cx.x, cx.y, cx.z, cx.w}, vs[4] = {cv.x, cv.y, cv.z, cv.w};
        unsigned ka = 0xffffffffu, kb = 0xffffffffu;      // open runs' left nodes + 1
        float la = 0.0f, ra = 0.0f, lb = 0.0f, rb = 0.0f;
        bool bad = false;
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (PUSH) push(xs[k], vs[k]);
        if (PUSH && !EXACT) join();
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const Loc l = locate(xs[k]);
            const bool ok = l.j <= (unsigned)ng;
            bad |= !ok;
            if (!ok) continue;
            const float wl = 1.0f - l.f;
            if (l.j == ka) {
                la += wl;
                ra += l.f;
            } else if (l.j == kb) {
                lb += wl;
                rb += l.f;
            } else {
                if (kb != 0xffffffffu) add(kb, lb, rb);
                kb = ka; lb = la; rb = ra;
                ka = l.j; la = wl; ra = l.f;
            }
        }
        if (PUSH) {
            __stcs(x4 + q, make_float4(xs[0], xs[1], xs[2], xs[3]));
            __stcs(v4 + q, make_float4(vs[0], vs[1], vs[2], vs[3]));
        }
        if (ka != 0xffffffffu) add(ka, la, ra);
        if (kb != 0xffffffffu) add(kb, lb, rb);
        if (bad) atomicOr(a.err, kErrPosition);
        cx = nx;
        cv = nv;
    }
    // the last N mod 4 particles
    if (blockIdx.x == 0 && tid < (int)(a.n & 3)) {
        const long long i = 4ll * n4 + tid;
        float x = a.x[i], v = PUSH ? a.v[i] : 0.0f;
        if (PUSH) push(x, v);
        const Loc l = locate(x);
        if (l.j <= (unsigned)ng) add(l.j, 1.0f - l.f, l.f);
        else atomicOr(a.err, kErrPosition);
        if (PUSH) { a.x[i] = x; a.v[i] = v; }
    }
    if (PUSH) {
        join();                                           // (block 0's last particles)
        // the block's sums as pairs: the float64 pipe would take 2.5 us
        warp_sum_pairs(sums, 32);
        if ((tid & 31) == 0) red[tid >> 5] = sums;
        __syncthreads();
        float4 p = tid < 32 && tid < ((bs + 31) >> 5) ? red[tid & 31] : make_float4(0.f, 0.f, 0.f, 0.f);
        if (tid < 32) warp_sum_pairs(p, 32);
        const double dke = (double)p.x + (double)p.y, dmom = (double)p.z + (double)p.w;
        if (tid == 0) {
            a.partials[2 * blockIdx.x] = dke;
            a.partials[2 * blockIdx.x + 1] = dmom;
        }
    }
    __syncthreads();
    for (int j = tid; j < ng + 2; j += bs) {
        float t = 0.0f;
        for (int k = 0; k < K; k++) t += sRho[j * K + ((k + tid) & (K - 1))];
        if (t == 0.0f) continue;
        const int node = j == 0 ? ng - 1 : (j == ng + 1 ? 0 : j - 1);
        atomicAdd(&a.rho_acc[node], t);
    }
}

// ---- float64 push and deposit (precision study; push64.cuh) --------------------

struct Tile96 {
    unsigned *lo, *mid, *hi;
};

__device__ __forceinline__ void tile_add96(const Tile96 &t, unsigned j, u64 val) {
    const unsigned vl = (unsigned)val;
    const unsigned ol = atomicAdd(&t.lo[j], vl);
    const unsigned vm = (unsigned)(val >> 32) + (ol + vl < ol ? 1u : 0u);   // < 2^27
    const unsigned om = atomicAdd(&t.mid[j], vm);
    if (om + vm < om) atomicAdd(&t.hi[j], 1u);
}

struct Run64 {
    unsigned key, cnt;            // left node + 1 (0xffffffff: none open), particles
    u64 r;                        // sum of the right weights
};

__device__ __forceinline__ void close_run(const Tile96 &t, const Run64 &w) {
    if (w.key == 0xffffffffu) return;
    tile_add96(t, w.key, w.cnt * kOne53 - w.r);
    tile_add96(t, w.key + 1, w.r);
}

struct D4 {
    double v[4];
};

__device__ __forceinline__ D4 ld4d(const double *p) {
    D4 r;
    asm volatile("ld.global.cs.v4.f64 {%0, %1, %2, %3}, [%4];"
                 : "=d"(r.v[0]), "=d"(r.v[1]), "=d"(r.v[2]), "=d"(r.v[3]) : "l"(p));
    return r;
}

__device__ __forceinline__ void st4d(double *p, const D4 &r) {
    asm volatile("st.global.cs.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(r.v[0]), "d"(r.v[1]),
                 "d"(r.v[2]), "d"(r.v[3]) : "memory");
}

template <bool PUSH>
__global__ void __launch_bounds__(1024) pic_push_f64_kernel(PushArgs64 a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ double red[64];
    const int tid = threadIdx.x, bs = blockDim.x, ng = a.ng;
    double2 *pair = reinterpret_cast<double2 *>(smem_raw);           // ng + 1
    Tile96 t;                                                        // ng + 2 each
    t.lo = reinterpret_cast<unsigned *>(pair + ng + 1);
    t.mid = t.lo + ng + 2;
    t.hi = t.mid + ng + 2;
    cudaTriggerProgrammaticLaunchCompletion();
    for (int j = tid; j < ng + 2; j += bs) {
        t.lo[j] = 0u;
        t.mid[j] = 0u;
        t.hi[j] = 0u;
    }
    cudaGridDependencySynchronize();
    for (int j = tid; j < ng + 2; j += bs) {
        if (PUSH && j <= ng) {
            const double el = a.E64[j == 0 ? ng - 1 : j - 1], er = a.E64[j == ng ? 0 : j];
            const double de = er - el;
            pair[j] = make_double2(el - de, de);
        }
    }
    __syncthreads();
    const Push64 c = push64_consts(a, pair);
    double ke = 0.0, mom = 0.0;
    const long long n4 = a.n >> 2;
    const long long stride = (long long)gridDim.x * bs;
    for (long long q = (long long)blockIdx.x * bs + tid; q < n4; q += stride) {
        D4 x = ld4d(a.x + 4 * q), v;
        if (PUSH) v = ld4d(a.v + 4 * q);
        Run64 ra = {0xffffffffu, 0u, 0ull}, rb = {0xffffffffu, 0u, 0ull};
        bool bad = false;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (PUSH) push_particle64(x.v[k], v.v[k], a, c, ke, mom);
            const Loc64 l = locate64(x.v[k], a.inv_dx, ng, c);
            bad |= !l.ok;
            if (!l.ok) continue;
            const u64 w = (((u64)l.fh << 32) | l.fl) >> 11;
            if (l.j == ra.key) {
                ra.cnt++;
                ra.r += w;
            } else if (l.j == rb.key) {
                rb.cnt++;
                rb.r += w;
            } else if (rb.key == 0xffffffffu) {
                rb = ra;
                ra = Run64{l.j, 1u, w};
            } else {
                close_run(t, ra);
                ra = Run64{l.j, 1u, w};
            }
        }
        if (PUSH) {
            st4d(a.x + 4 * q, x);
            st4d(a.v + 4 * q, v);
        }
        close_run(t, ra);
        close_run(t, rb);
        if (bad) atomicOr(a.err, kErrPosition);
    }
    if (blockIdx.x == 0 && tid < (int)(a.n & 3)) {          // the last N mod 4 particles
        const long long i = n4 * 4 + tid;
        double x = a.x[i], v = 0.0;
        if (PUSH) {
            v = a.v[i];
            push_particle64(x, v, a, c, ke, mom);
            a.x[i] = x;
            a.v[i] = v;
        }
        const Loc64 l = locate64(x, a.inv_dx, ng, c);
        if (l.ok) close_run(t, Run64{l.j, 1u, (((u64)l.fh << 32) | l.fl) >> 11});
        else atomicOr(a.err, kErrPosition);
    }
    if (PUSH) {
        __syncthreads();
        block_sum2(ke, mom, red);
        if (tid == 0) {
            a.partials[2 * blockIdx.x] = ke;
            a.partials[2 * blockIdx.x + 1] = mom;
        }
    }
    __syncthreads();
    for (int j = tid; j < ng + 2; j += bs) {
        const unsigned lo = t.lo[j], mid = t.mid[j];
        const u64 low40 = ((u64)(mid & 0xFFu) << 32) | lo;
        const u64 rest = ((u64)t.hi[j] << 24) | (mid >> 8);
        const int node = j == 0 ? ng - 1 : (j == ng + 1 ? 0 : j - 1);
        if (low40) atomicAdd(&a.rho_w[2 * node], low40);
        if (rest) atomicAdd(&a.rho_w[2 * node + 1], rest);
    }
}

using AtomicKernel = void (*)(PushArgsF32Atomic);

AtomicKernel atomic_kernel(bool push, long long n) {
    if (!push) return &pic_push_f32atomic_kernel<false, false>;
    return n <= kAtomicExact ? &pic_push_f32atomic_kernel<true, true> : &pic_push_f32atomic_kernel<true, false>;
}

using FixedKernel = void (*)(PushArgs);

template <int V>
FixedKernel pick_unroll(bool push, int unroll) {
    if (!push) return &pic_push_fixed_kernel<V, false, 1>;
    switch (unroll) {
        case 1: return &pic_push_fixed_kernel<V, true, 1>;
        case 2: return &pic_push_fixed_kernel<V, true, 2>;
        case 4: return &pic_push_fixed_kernel<V, true, 4>;
        default: return nullptr;
    }
}

template <int V>
FixedKernel pick_oct(bool push, int unroll) {
    if (!push) return &pic_push_oct_kernel<V, false, 1>;
    switch (unroll) {
        case 1: return &pic_push_oct_kernel<V, true, 1>;
        case 2: return &pic_push_oct_kernel<V, true, 2>;
        default: return nullptr;
    }
}

FixedKernel pick_fixed(int variant, bool push, int unroll) {
    switch (variant) {
        case PIC_DEPOSIT_QUAD8: return pick_oct<PIC_DEPOSIT_QUAD8>(push, unroll);
        case PIC_DEPOSIT_PAIR8: return pick_oct<PIC_DEPOSIT_PAIR8>(push, unroll);
        case PIC_DEPOSIT_ATOMIC: return pick_unroll<kDepositCells>(push, unroll);
        case PIC_DEPOSIT_MATCH: return pick_unroll<PIC_DEPOSIT_MATCH>(push, unroll);
        case PIC_DEPOSIT_QUAD: return pick_unroll<PIC_DEPOSIT_QUAD>(push, unroll);
        case PIC_DEPOSIT_PAIR: return pick_unroll<PIC_DEPOSIT_PAIR>(push, unroll);
        case kDepositNgp: return pick_unroll<kDepositNgp>(push, unroll);
        default: return nullptr;
    }
}

}  // namespace

bool push_wide_tile(long long n, int sms) {
    // a grid smaller than the SMs takes one group of particles per thread
    return n / sms > kPackedCount - 512 * 32;
}

size_t push_smem_bytes(int mode, int ng, bool wide, int block) {
    if (mode == PIC_FP64) return (size_t)(ng + 1) * 16 + (size_t)(ng + 2) * 12;
    if (mode == PIC_FP32_ATOMIC) return (size_t)(ng + 2) * 4 * (1 + atomic_copies(ng, block));
    return (size_t)(ng + 2) * (wide ? 16 : 12);
}

cudaError_t push_prepare_attributes(int mode) {
    const int bytes = mode == PIC_FP32_ATOMIC ? (int)kAtomicShared
                                              : (int)push_smem_bytes(mode, PIC_NCELL_MAX, true, 0);
    cudaError_t e = cudaSuccess;
    if (mode == PIC_FP32_FIXED) {
        const int unrolls[3] = {1, 2, 4};
        const int fixed_variants[] = {PIC_DEPOSIT_ATOMIC, PIC_DEPOSIT_MATCH, PIC_DEPOSIT_QUAD,
                                      PIC_DEPOSIT_PAIR, PIC_DEPOSIT_QUAD8, PIC_DEPOSIT_PAIR8,
                                      kDepositNgp};
        for (int v : fixed_variants)
            for (int p = 0; p < 2; p++)
                for (int u : unrolls) {
                    FixedKernel k = pick_fixed(v, p != 0, u);
                    if (!k) continue;
                    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
                    if (e != cudaSuccess) return e;
                }
    } else if (mode == PIC_FP32_ATOMIC) {
        for (AtomicKernel k : {atomic_kernel(true, 1), atomic_kernel(true, kAtomicExact + 1), atomic_kernel(false, 1)}) {
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
            if (e != cudaSuccess) return e;
        }
    } else {
        e = cudaFuncSetAttribute(&pic_push_f64_kernel<true>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(&pic_push_f64_kernel<false>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    }
    return e;
}

int push_max_blocks_per_sm(int mode, int variant, int unroll, int block, int ng, bool wide) {
    int nb = 0;
    const size_t smem = push_smem_bytes(mode, ng, wide, block);
    cudaError_t e;
    if (mode == PIC_FP32_FIXED) {
        FixedKernel k = pick_fixed(variant, true, unroll);
        if (!k) return 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, block, smem);
    }
    else if (mode == PIC_FP32_ATOMIC)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, &pic_push_f32atomic_kernel<true, false>, block, smem);
    else
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, &pic_push_f64_kernel<true>, block, smem);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();     // do not leave the error for a later launch check
        return 0;
    }
    return nb;
}

cudaError_t launch_push_fixed(const PushArgs &a, int grid, int block, int variant,
                              int unroll, bool push, cudaStream_t s) {
    FixedKernel k = pick_fixed(variant, push, unroll);
    if (!k) return cudaErrorInvalidValue;
    return launch_after(k, dim3(grid), block, push_smem_bytes(PIC_FP32_FIXED, a.c.ng, a.wide, block), s, 0, a);
}

cudaError_t launch_push_f32_atomic(PushArgsF32Atomic a, int grid, int block, bool push,
                                   cudaStream_t s) {
    const size_t smem = push_smem_bytes(PIC_FP32_ATOMIC, a.c.ng, false, block);
    a.copies = atomic_copies(a.c.ng, block);
    return launch_after(atomic_kernel(push, a.n), dim3(grid), block, smem, s, 0, a);
}

cudaError_t launch_push_f64(const PushArgs64 &a, int grid, int block, bool push,
                            cudaStream_t s) {
    const size_t smem = push_smem_bytes(PIC_FP64, a.ng, false, block);
    return launch_after(push ? &pic_push_f64_kernel<true> : &pic_push_f64_kernel<false>, dim3(grid), block, smem,
                        s, 0, a);
}

}  // namespace pic
