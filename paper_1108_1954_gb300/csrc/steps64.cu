// steps64.cu -- many steps of one float64 run in one cooperative launch: steps.cu's
// scheme (push into a private tile, flush, one grid barrier, every block solves
// the grid itself, two blocks for the diagnostics) for PIC_FP64, whose steps of
// a small run were a push and a solve of 7 and 8.4 us (2e4 particles, 64 cells).
//
// What differs:
//   * one particle per lane: a float64 instruction takes the pipe for 16 clocks a
//     warp whatever it holds, so particles are spread over warps and SMs, and a
//     particle's chain of five dependent instructions is 64 clocks each;
//   * the tile keeps per cell the number of particles and the sum of their
//     weights W in 2^-53 as three 32-bit words, in kCopies copies that the lanes
//     alternate between (an add of 1 costs nothing where lanes collide, the
//     fetch-adds of W a clock per lane);
//   * the solve is in 128-bit integers (R_g = N 2^53 - NG q_g, the bounds in
//     field.cu) with one node per thread, and E stays float64;
//   * the sums of v_old v_new and v_new are taken over a warp as aligned integers
//     (warp_sum_fixed), 200 clocks against 700 for a tree of float64 adds.
// 2e4 particles, 64 cells: 4.1 us a step, 15.3 with the two kernels.  The float64
// solve of all nodes by every block (6 instructions a warp of nodes) bounds large
// grids and the push's five instructions a particle large runs; those keep the
// two kernels (pic_api.cu, set_steps_shape).
#include "push64.cuh"
#include "steps_common.cuh"

namespace pic {
namespace {

constexpr int kResident = 2;               // particles a thread keeps in registers
constexpr int kLogCopies = 2, kCopies = 1 << kLogCopies;

struct Solved64 {
    i128 R[1], P[1], q[1], m[1];  // as NodeSolve, one node per thread
    i128 SR, SP;
};

__device__ __forceinline__ void solve_nodes64(Solved64 &s, const StepsArgs &a,
                                              const unsigned long long *acc, int ng,
                                              unsigned long long *scan64) {
    const int g = threadIdx.x;
    const bool in = g < ng;
    ulonglong2 w = make_ulonglong2(0ull, 0ull);
    if (in) w = __ldcg(reinterpret_cast<const ulonglong2 *>(acc) + g);
    s.q[0] = (i128)w.x + ((i128)w.y << 40);
    s.R[0] = in ? ((i128)a.n << 53) - (i128)ng * s.q[0] : (i128)0;
    const int used = (ng + 31) >> 5;                  // warps with nodes
    const I128Pair sc = block_inclusive_scan2_i128(s.R[0], s.R[0] * (i128)g, scan64, used);
    i128 S1 = 0;
    s.SR = 0;
    for (int i = 0; i < used; i++) {
        s.SR += (i128)(((unsigned __int128)scan64[32 + i] << 64) | scan64[i]);
        S1 += (i128)(((unsigned __int128)scan64[96 + i] << 64) | scan64[64 + i]);
    }
    s.SP = (i128)ng * s.SR - S1;                      // sum_k (NG - k) R_k
    s.P[0] = sc.a;
    const i128 prev = g == 0 ? s.SR : sc.a - s.R[0];   // P_{g-1}; M_{-1} = M_{NG-1}
    s.m[0] = (i128)ng * (sc.a + prev) - 2 * s.SP;
}

struct Tile64 {
    unsigned *n, *lo, *mid, *hi;  // counts; sums of W mod 2^32, of its upper half, carries
};

struct CellSum64 {
    u64 n;
    unsigned __int128 W;
};

__global__ void __launch_bounds__(1024, 1) pic_steps64_kernel(const __grid_constant__ StepsArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ unsigned long long scan64[4 * 32];
    __shared__ double2 kvs[32];
    __shared__ int dead;
    const int ng = a.c.ng, words = (ng + 2) << kLogCopies;
    double2 *pair = reinterpret_cast<double2 *>(smem_raw);       // ng + 1
    double *sE = reinterpret_cast<double *>(pair + ng + 1);      // ng + 2, ghost-padded
    unsigned *tw = reinterpret_cast<unsigned *>(sE + ng + 2);
    const Tile64 tile = {tw, tw + words, tw + 2 * words, tw + 3 * words};
    const int tid = threadIdx.x, bs = blockDim.x, lane = tid & 31, w = tid >> 5, nw = bs >> 5;
    const int nd = a.diag_blocks, workers = (int)gridDim.x - nd, b = blockIdx.x;
    const bool diag = b >= workers;
    if (tid == 0) dead = 0;
    auto clear_tile = [&] {
        for (int j = tid; j < 4 * words; j += bs) tw[j] = 0u;
    };
    // (E_l - dE, dE) of every cell from the ghost-padded E
    auto make_pairs = [&] {
        for (int j = tid; j <= ng; j += bs) {
            const double el = sE[j], de = sE[j + 1] - el;
            pair[j] = make_double2(el - de, de);
        }
    };
    clear_tile();
    for (int j = tid; j < ng + 2; j += bs) sE[j] = a.E64[j == 0 ? ng - 1 : (j == ng + 1 ? 0 : j - 1)];
    const int n = (int)a.n;
    const int q0 = diag ? 0 : (int)((long long)n * b / workers);
    const int q1 = diag ? 0 : (int)((long long)n * (b + 1) / workers);
    const unsigned h0 = diag ? (unsigned)(a.step0 % a.hist_len) : 0u;
    double *x = a.d.x, *v = a.d.v;
    double rx[kResident], rv[kResident];
#pragma unroll
    for (int i = 0; i < kResident; i++) {
        const int q = q0 + tid + i * bs;
        rx[i] = q < q1 ? __ldcg(x + q) : 0.0;
        rv[i] = q < q1 ? __ldcg(v + q) : 0.0;
    }
    const Push64 c = push64_consts(a.d, pair);
    const unsigned copy = lane & (kCopies - 1);
    __syncthreads();
    make_pairs();
    __syncthreads();
    auto step1 = [&](double &px, double &pv, double &ke, double &mom) {
        push_particle64(px, pv, a.d, c, ke, mom);
        const Loc64 l = locate64(px, a.d.inv_dx, ng, c);
        if (l.ok) {
            const unsigned j = (l.j << kLogCopies) + copy;
            const u64 W = (((u64)l.fh << 32) | l.fl) >> 11;
            atomicAdd(&tile.n[j], 1u);
            const unsigned wl = (unsigned)W, ol = atomicAdd(&tile.lo[j], wl);
            const unsigned wm = (unsigned)(W >> 32) + (ol + wl < ol ? 1u : 0u);
            const unsigned om = atomicAdd(&tile.mid[j], wm);
            if (om + wm < om) atomicAdd(&tile.hi[j], 1u);
        } else {
            atomicOr(a.err, kErrPosition);
        }
    };
    for (int s = diag ? b - workers : 0; s < a.steps; s += diag ? nd : 1) {
        const bool last = s == a.steps - 1;
        const int slot = s % kStepsSlots;
        unsigned long long *acc = a.acc + (size_t)slot * 2 * ng;
        double2 *kv = reinterpret_cast<double2 *>(a.partials) + (size_t)slot * kStepsMaxGrid;
        if (!diag) {
            double ke = 0.0, mom = 0.0;
#pragma unroll
            for (int i = 0; i < kResident; i++)
                if (q0 + tid + i * bs < q1) step1(rx[i], rv[i], ke, mom);
            for (int q = q0 + tid + kResident * bs; q < q1; q += bs) {
                double px = __ldcg(x + q), pv = __ldcg(v + q);
                step1(px, pv, ke, mom);
                __stcg(x + q, px);
                __stcg(v + q, pv);
            }
            ke = warp_sum_fixed(ke);
            mom = warp_sum_fixed(mom);
            if (lane == 0) kvs[w] = make_double2(ke, mom);
            __syncthreads();
            if (w == nw - 1) {
                const double2 p = lane < nw ? kvs[lane] : make_double2(0.0, 0.0);
                const double k = warp_sum_fixed(p.x), m = warp_sum_fixed(p.y);
                if (lane == 0) kv[b] = make_double2(k, m);
            }
            // node g: the left weights of cell g + 1 and the right ones of cell g, as
            // in steps.cu
            auto cell = [&](int j) {
                CellSum64 r = {0ull, 0};
#pragma unroll
                for (int i = 0; i < kCopies; i++) {
                    const int at = (j << kLogCopies) + ((i + lane) & (kCopies - 1));
                    r.n += tile.n[at];
                    r.W += ((unsigned __int128)tile.hi[at] << 64) | ((u64)tile.mid[at] << 32) | tile.lo[at];
                }
                return r;
            };
            auto left = [](const CellSum64 &r) { return ((unsigned __int128)r.n << 53) - r.W; };
            for (int g = tid; g < ng; g += bs) {
                unsigned __int128 val = left(cell(g + 1)) + cell(g).W;
                if (g == ng - 1) val += left(cell(0));
                if (g == 0) val += cell(ng).W;
                // two sums, of the low 40 bits and of the rest (push64.cuh)
                const u64 low40 = (u64)val & ((1ull << 40) - 1ull), rest = (u64)(val >> 40);
                if (low40) atomicAdd(&acc[2 * g], low40);
                if (rest) atomicAdd(&acc[2 * g + 1], rest);
            }
            __syncthreads();
            if (tid == 0) red_release(a.sync);        // the whole block's adds: after the barrier
            if (!last) clear_tile();                  // while the others arrive
        }
        if (!wait_step(a, s, workers, !diag, &dead)) return;
        Solved64 ns;
        solve_nodes64(ns, a, acc, ng, scan64);
        if (!diag && last) {
            if (tid == 0) red_release(a.sync);        // the sums have been read
            step_results<1, false>(a, ns, b, workers);
            break;
        }
        if (!diag) {
            if (tid < ng) {
                const double e = a.k_e * i128_to_f64(ns.m[0]);
                sE[tid + 1] = e;
                if (tid == ng - 1) sE[0] = e;
                if (tid == 0) sE[ng + 1] = e;
            }
            __syncthreads();
            make_pairs();
            __syncthreads();
            continue;
        }
        step_rows<1, false>(a, s, ns, smem_raw, h0, [&](double &k, double &m) {
            double2 p[kStepsMaxGrid / 32];                      // all loads in flight
#pragma unroll
            for (int i = 0; i < kStepsMaxGrid / 32; i++)
                p[i] = 32 * i + lane < workers ? __ldcg(kv + 32 * i + lane) : make_double2(0.0, 0.0);
            k = 0.0;
            m = 0.0;
#pragma unroll
            for (int i = 0; i < kStepsMaxGrid / 32; i++) {
                k += p[i].x;
                m += p[i].y;
            }
            k = warp_sum_fixed(k);
            m = warp_sum_fixed(m);
        });
        // give the slot back, once no worker reads it any more
        if (!wait_step(a, s + 1, workers, false, &dead)) return;
        for (int g = tid; g < 2 * ng; g += bs) acc[g] = 0ull;
        __syncthreads();
        if (tid == 0) red_release(a.sync + 1 + (b - workers));
    }
    if (!diag) {
#pragma unroll
        for (int i = 0; i < kResident; i++) {
            const int q = q0 + tid + i * bs;
            if (q >= q1) break;
            __stcg(x + q, rx[i]);
            __stcg(v + q, rv[i]);
        }
    }
}

size_t steps64_smem(int ng) {
    return (size_t)(ng + 1) * 16 + (size_t)(ng + 2) * (8 + 16 * kCopies);
}

}  // namespace

cudaError_t steps64_prepare(int ng, int block, int *per_sm) {
    *per_sm = 0;
    if (ng > block) return cudaSuccess;               // one node per thread
    cudaError_t e = cudaFuncSetAttribute(&pic_steps64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)steps64_smem(1024));
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, &pic_steps64_kernel, block, steps64_smem(ng));
}

cudaError_t launch_steps64(const StepsArgs &a, int grid, int block, cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    cooperative(cfg, attr, grid, block, steps64_smem(a.c.ng), s);
    return cudaLaunchKernelEx(&cfg, &pic_steps64_kernel, a);
}

}  // namespace pic
