// steps_common.cuh -- what the many-step launches of the fixed-point runs
// (steps.cu) and the float64 runs (steps64.cu) share: the waits between blocks,
// the diagnostics rows, the cooperative launch.
#pragma once

#include "field_ops.cuh"
#include "particle_ops.cuh"

namespace pic {
namespace {

// The launch's counters, never reset: arrivals of the workers (one a step, and one
// when the last step's sums have been read), and the steps that each diagnostics
// block is done with (StepsArgs::sync, on 16 bytes).
__device__ __forceinline__ uint4 ld_acquire(const unsigned *p) {
    uint4 v;
    asm volatile("ld.acquire.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_release(unsigned *p) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

// Steps t <= last with t mod nd == d.
__device__ __forceinline__ unsigned steps_of(int last, int d, int nd) {
    return last < d ? 0u : (unsigned)((last - d) / nd + 1);
}

// Waits until all workers have arrived for step s, and, for a worker, until the
// slot of step s + 1 has been given back by the diagnostics of step s + 1 -
// kStepsSlots.  All threads of the block; false when the wait ran out.
__device__ __forceinline__ bool wait_step(const StepsArgs &a, int s, int workers, bool worker,
                                          int *dead) {
    if (threadIdx.x == 0) {
        const int nd = a.diag_blocks;
        const unsigned target = a.base[0] + (unsigned)workers * (unsigned)(s + 1);
        const unsigned d0 = a.base[1] + steps_of(s + 1 - kStepsSlots, 0, nd);
        const unsigned d1 = a.base[2] + (nd > 1 ? steps_of(s + 1 - kStepsSlots, 1, nd) : 0u);
        unsigned polls = 0;
        for (;;) {
            const uint4 v = ld_acquire(a.sync);
            if ((int)(v.x - target) >= 0 && (!worker || ((int)(v.y - d0) >= 0 && (int)(v.z - d1) >= 0)))
                break;
            if (++polls >= a.wait_limit) {
                atomicOr(a.err, kErrWait);
                *dead = 1;
                break;
            }
        }
    }
    __syncthreads();
    return *dead == 0;
}

// The diagnostics of step s from the solved nodes ns (thread t's nodes K t ... ).
// sums: the push's two sums, by the
// block's last warp.  smem_raw: 8 NG bytes.
template <int K, bool FIXED, class Solved, class Sums>
__device__ __forceinline__ void step_rows(const StepsArgs &a, int s, const Solved &ns,
                                          unsigned char *smem_raw, unsigned h0, const Sums &sums) {
    const int ng = a.c.ng, tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
    const bool last = s == a.steps - 1;
    __shared__ float shf[2 * PIC_NMODES][32];
    __shared__ double shd[8], fchunk[256], tot[2];
    double *fe = reinterpret_cast<double *>(smem_raw);      // [ng], in the tile
    if (w == nw - 1) {       // the push's sums: the warp without nodes, where there is one
        double k, m;
        sums(k, m);
        if (lane == 0) {
            tot[0] = k;
            tot[1] = m;
        }
    }
    NodeDiag d;
    node_diag_reset(d);
#pragma unroll
    for (int j = 0; j < K; j++) {
        const int g = tid * K + j;
        if (g >= ng) break;
        const double E = a.k_e * i128_to_f64(ns.m[j]);
        d.fe = 0.0;
        node_diag(d, g, ng, E, (float)E);
        fe[g] = d.fe;
    }
    float md[2 * PIC_NMODES];
#pragma unroll
    for (int m = 0; m < PIC_NMODES; m++) { md[2 * m] = d.re[m]; md[2 * m + 1] = d.im[m]; }
    static_assert(2 * PIC_NMODES == 16, "16 mode sums per warp");
    const int used = (ng + 32 * K - 1) / (32 * K);          // warps with nodes
    if (w < used) {
        const float msum = warp_sum16_halving(md, lane);
        if ((lane & 1) == 0) shf[lane >> 1][w] = msum;
    }
    __syncthreads();
    const int chunks = (ng + 31) >> 5;
    for (int i = w; i < chunks; i += nw) {                  // field energy of 32 nodes
        const int g = 32 * i + lane;
        const double sum = warp_sum_fast(g < ng ? fe[g] : 0.0);
        if (lane == 0) fchunk[i] = sum;
    }
    __syncthreads();
    const double fe_total = chunk_sum_f64(tid < chunks ? fchunk[tid] : 0.0, chunks, shd);
    if (w == 0) {
        const long long n = a.step0 + s + 1;
        pic_diag_row *prev = &a.hist[(h0 + s) % a.hist_len], *row = &a.hist[(h0 + s + 1) % a.hist_len];
        // one value per lane: kinetic energy and momentum of the row before,
        // field energy and charge of this one
        const double coef = lane == 0 ? 0.5 * a.mass : lane == 1 ? a.mass
                            : lane == 2 ? 0.5 * a.dx : a.dx * a.k_rho;
        const double fe0 = __shfl_sync(kFull, fe_total, 0);
        const double val = coef * (lane < 2 ? tot[lane] : lane == 2 ? fe0 : i128_to_f64((i128)ns.SR));
        if (lane < 4 && (lane >= 2 || prev != row))       // (a ring of one row: only the new one)
            *(lane == 0 ? &prev->kinetic : lane == 1 ? &prev->momentum
              : lane == 2 ? &row->field : &row->charge) = val;
        if (lane == 4) row->step = n;
        // sum of rho_q: SR = NG (N 2^24 - it), 0 unless particles were lost
        if (lane == 5) row->charge_q = !FIXED ? 0 : ns.SR ? a.weight_total - (long long)ns.SR / ng : a.weight_total;
        if (last && lane >= 6 && lane < 8)       // (otherwise the next step's, perhaps written already)
            *(lane == 6 ? &row->kinetic : &row->momentum) = __longlong_as_double(0x7ff8000000000000ll);
        if (last && lane == 8) *a.dstep = n;
    }
    if (w == nw - 1) {
        // mode sums: float32 over 256 nodes (kRun warps), float64 over those, every
        // other of them by the upper half of the warp.  (Over 1024 nodes in float32
        // the error on 4096 cells was 1.4 times as large.)
        constexpr int kRun = K < 8 ? 8 / K : 1;
        double sum = 0.0;
        for (int i0 = (lane >> 4) * kRun; i0 < used; i0 += 2 * kRun) {
            float part = 0.0f;
#pragma unroll
            for (int i = 0; i < kRun; i++)
                part += i0 + i < used ? shf[lane & 15][(i0 + i) & 31] : 0.0f;
            sum += (double)part;
        }
        sum += __shfl_down_sync(kFull, sum, 16);
        const double im = __shfl_down_sync(kFull, sum, 1);
        if (lane < 2 * PIC_NMODES && !(lane & 1))
            a.hist[(h0 + s + 1) % a.hist_len].mode[lane >> 1] =
                sqrt(sum * sum + im * im) * a.k_mode;
    }
}

// The run's results after the last step, by worker b of the workers: its share of
// the nodes.  (Every worker has solved the whole grid; the float64 conversions,
// some 12 instructions a node at 16 clocks a warp, are what takes time: written by
// the one diagnostics block a single step took 14.3 us, not 12.3, with 3e5
// particles on 500 cells and 26.6, not 21.9, with 1e6 on 2048.)
template <int K, bool FIXED, class Solved>
__device__ __forceinline__ void step_results(const StepsArgs &a, const Solved &ns, int b, int workers) {
    __shared__ unsigned long long scan64[2 * 32];
    const int ng = a.c.ng, tid = threadIdx.x;
    const int own0 = (int)((long long)ng * b / workers), own1 = (int)((long long)ng * (b + 1) / workers);
    // Phi: sum_{k<g} M_k = NG (g P_g - sum_{j<=g} j R_j) - g SP
    i128 jr = 0;
#pragma unroll
    for (int j = 0; j < K; j++) jr += (i128)ns.R[j] * (i128)(tid * K + j);
    i128 run = block_inclusive_scan_i128(jr, scan64) - jr;
#pragma unroll
    for (int j = 0; j < K; j++) {
        const int g = tid * K + j;
        if (g >= own1) break;
        run += (i128)ns.R[j] * (i128)g;
        if (g < own0) continue;
        const double E = a.k_e * i128_to_f64(ns.m[j]);
        a.E64[g] = E;
        a.E32[g] = (float)E;
        a.rho[g] = a.k_rho * i128_to_f64((i128)ns.R[j]);
        if (FIXED) a.rho_q_last[g] = (unsigned long long)ns.q[j];
        const i128 sumM = (i128)ng * ((i128)g * (i128)ns.P[j] - run) - (i128)g * ns.SP;
        a.phi[g] = a.k_phi * i128_to_f64(sumM);
    }
}

// A launch whose blocks are all resident at once.
void cooperative(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int grid, int block, size_t smem,
                 cudaStream_t s) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

}  // namespace
}  // namespace pic
