// field.cu -- the field solve that closes a PIC step (Sec. 2.2) and the
// step's diagnostics.
//
// Poisson (Eq. 6) in flux form.  With D_{g+1/2} = Phi_{g+1} - Phi_g, Eq. 6 is
// D_{g+1/2} - D_{g-1/2} = -rho_g dx^2, so D_{g+1/2} = C - dx^2 S_g with the
// prefix sum S_g = sum_{k<=g} rho_k.  A periodic Phi needs sum_g D = 0, which
// fixes C = dx^2 mean(S); Phi_0 = 0 (the gauge the paper's CG pins) and
// Phi_g = sum_{k<g} D_{k+1/2}.  The field of Eq. 7 needs only D:
//   E_g = -(Phi_{g+1} - Phi_{g-1})/(2 dx) = -(D_{g+1/2} + D_{g-1/2})/(2 dx)
//       = (dx/2) (S_g + S_{g-1} - 2 mean(S)),   S_{-1} = S_{NG-1}.
// For a neutral box this is the exact solution of the linear system the
// paper's CG iterates on (with 2 global reductions per iteration).
//
// Fixed-point mode: exact integer prefix sums.  The density is
//   rho_g = K (N 2^24 - NG rho_q[g]) = K R_g,   K = rho_ion / (N 2^24),
// with R_g an integer and sum_g R_g = 0 exactly when every particle deposited.
// All prefix sums are taken on R in 128-bit integers, exactly:
//   P_g = sum_{k<=g} R_k,  M_g = NG P_g - sum_k P_k  ( = NG (S_g - mean S)/K ),
//   E_g   = (dx/2)(K/NG) (M_g + M_{g-1}),          M_{-1} = M_{NG-1}
//   Phi_g = -dx^2 (K/NG) sum_{k<g} M_k,
// and float64 arithmetic appears only in the final conversion of each value,
// so E is within an ulp or two of the exactly rounded solution.  GB300 runs
// float64 at a small fraction of its float32 rate; this keeps the solve cheap.
// The nodes are split over the blocks of one thread-block cluster (one node
// per thread); the blocks exchange their slice sums through distributed
// shared memory, and block 0 reduces the diagnostics and writes the history
// rows.
//
// The float modes (precision study) solve their density sums as integers of
// finer units by the same kernel (take_density).  The paper's CG solver
// (PIC_SOLVER_CG) runs on a thread-block cluster too (below).
//
// Diagnostics: field energy (1/2) dx sum E^2 in float64; mode amplitudes
// from the float32 field with float32 twiddles, summed per block in float32
// and over blocks in float64; kinetic energy and momentum from the push's
// per-block float64 sums, reduced in a fixed order.
#include <math.h>

#include <cooperative_groups.h>

#include "field_ops.cuh"

namespace cg = cooperative_groups;

namespace pic {
namespace {

constexpr int kClusterSolveThreads = 512;   // most nodes per block (one per thread)
// Nodes per block of the exact solve: its per-node float64 conversions and
// diagnostics are the critical path, so spread them over up to 16 SMs.  us a
// solve with 256, 128 and 64: 1024 nodes 9.4, 8.6, 8.5; 2048 9.2, 8.4, 8.4; 4096
// 8.9 each.
constexpr int kSolveNodesPerBlock = 128;
constexpr int kMaxSolveCluster = 16;        // blocks per cluster (16: non-portable)

// ---- the density as integers --------------------------------------------------
//
// Every precision mode solves the same integers: node g's particle sum is q_g
// units of 2^-B of a particle, and rho_g = K R_g with R_g = N 2^B - NG q_g and
// K = rho_ion / (N 2^B).
//   fixed point     B = 24: the deposit's own integers
//   float32 atomic  B = 30: the float32 sum, exactly: locate's fractions, and so all
//                   weights and their sums, are multiples of 2^-24
//   float64         B = 53: the deposit's own integers, kept as two 64-bit sums
//                   of the low 40 bits and of the rest (push64.cuh)
// Bounds of the 128-bit arithmetic below, worst at B = 53, N < 2^32, NG = 2^13
// with every particle in one cell: |P_g| <= NG N 2^53 < 2^98, |sum P| < 2^111,
// |M_g| < 2^112 and the two terms of sum M below 2^125 each.
// N 2^B (in 64 bits where it fits: N < 2^39 at B = 24)
template <int MODE>
__device__ __forceinline__ i128 whole_density(const SolveArgs &a) {
    if (MODE == PIC_FP32_FIXED) return (i128)(a.npart_total << kFixBits);
    constexpr int kBits = density_bits(MODE);
    return (i128)a.npart_total << kBits;
}

template <int MODE>
__device__ __forceinline__ i128 take_density(const SolveArgs &a, int g) {
    // read and cleared by this thread only
    if (MODE == PIC_FP32_FIXED) {
        const unsigned long long q = __ldcg(&a.rho_q[g]);
        a.rho_q[g] = 0ull;
        a.rho_q_last[g] = q;
        return (i128)q;
    }
    if (MODE == PIC_FP32_ATOMIC) {
        const float acc = __ldcg(&a.rho_f32[g]);
        a.rho_f32[g] = 0.0f;
        return (i128)__float2ll_rn(acc * 0x1p30f);
    }
    const ulonglong2 w = __ldcg(reinterpret_cast<const ulonglong2 *>(a.rho_w) + g);
    reinterpret_cast<ulonglong2 *>(a.rho_w)[g] = make_ulonglong2(0ull, 0ull);
    return (i128)w.x + ((i128)w.y << 40);
}

// ---- the cluster solves' common parts -------------------------------------

// The part of a block's shared memory that block 0 reads for the diagnostics.
struct ClusterDiag {
    double fe[kClusterSolveThreads / 32];   // field energy sums of the warps
    double kv[2];                 // the block's share of the push sums
    double diag[kDiagFields];     // slice diagnostics
    unsigned long long cq;        // slice sum of rho_q
};

// The block's share of the push's per-block sums, summed by warp 0 alone
// (a few dozen values; float64 adds are scarce); valid in lane 0 of warp 0.
// Issued first in the solves, so the loads overlap the rest.
__device__ __forceinline__ void push_sums_share(const SolveArgs &a, int C, int r, double (&kv)[2]) {
    kv[0] = 0.0;
    kv[1] = 0.0;
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    for (int i = r * 32 + lane; i < a.npartials; i += C * 32) {
        kv[0] += a.partials[2 * i];
        kv[1] += a.partials[2 * i + 1];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double u0 = __shfl_down_sync(kFull, kv[0], o);
        const double u1 = __shfl_down_sync(kFull, kv[1], o);
        if (lane < o) { kv[0] += u0; kv[1] += u1; }
    }
}

// Diagnostics of a cluster solve: block sums of the nodes' contributions,
// then block 0 sums the blocks in rank order (after a cluster barrier) and
// writes the history rows (scalars by thread 0, mode m by thread m); a last
// cluster barrier keeps every block's shared memory alive until block 0 has
// read it.  charge: this block's share of the charge diagnostic.
__device__ void cluster_finish(const SolveArgs &a, cg::cluster_group &cl, ClusterDiag &cd,
                               const double (&kv)[2], const NodeDiag &d, double charge,
                               unsigned long long q, long long step) {
    __shared__ __align__(16) double shd[8];
    __shared__ __align__(16) float shf[2 * PIC_NMODES][32];       // [value][warp]
    __shared__ __align__(16) unsigned long long cqw[32];
    const int C = (int)cl.num_blocks(), r = (int)cl.block_rank();
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, nw = blockDim.x >> 5;
    // The warps' sums of the field energy (float64, published: block 0 adds them
    // in node order, below) and the block's sums of the mode sums (float32) and
    // the integer charge, with one barrier: warp sums by shuffles (the 16 mode
    // sums by recursive halving), then warp 0 across the warps, each mode sum by
    // one lane in warp order.
    const double fe = warp_sum_fast(d.fe);
    unsigned long long cqb = q;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cqb += __shfl_down_sync(kFull, cqb, o);
    float md[2 * PIC_NMODES];
#pragma unroll
    for (int m = 0; m < PIC_NMODES; m++) { md[2 * m] = d.re[m]; md[2 * m + 1] = d.im[m]; }
    static_assert(2 * PIC_NMODES == 16, "16 mode sums per warp");
    const float msum = warp_sum16_halving(md, lane);   // value lane/2 in lanes 2i, 2i+1
    if ((lane & 1) == 0) shf[lane >> 1][w] = msum;
    if (lane == 0) {
        cd.fe[w] = fe;
        cqw[w] = cqb;
    }
    __syncthreads();
    if (w == 0) {
        if (lane < 2 * PIC_NMODES) {
            float sm = 0.0f;
            for (int j = 0; j < nw; j++) sm += shf[lane][j];
            cd.diag[kDiagModes + lane] = (double)sm;
        }
        if (lane == 0) {
            unsigned long long sc = 0;
            for (int j = 0; j < nw; j++) sc += cqw[j];
            cd.cq = sc;
            cd.kv[0] = kv[0];
            cd.kv[1] = kv[1];
            cd.diag[kDiagFE] = 0.0;               // (block 0 adds the warps' sums, below)
            cd.diag[kDiagCharge] = charge;
        }
    }
    cl.sync();
    if (r == 0) {
        __shared__ double tot[kDiagFields + 2];
        __shared__ unsigned long long tot_cq;
        cluster_diag_sums<kMaxSolveCluster>(cl, cd, tot, &tot_cq);
        // the warps' field energies in node order (C nw <= 32 nw threads)
        const double fes = t < C * nw ? cl.map_shared_rank(&cd, t / nw)->fe[t % nw] : 0.0;
        const double fe_total = chunk_sum_f64(fes, C * nw, shd);
        const long long n = a.npartials > 0 ? step + 1 : step;
        pic_diag_row *row = &a.hist[n % a.hist_len];
        if (t == 0) {
            if (a.npartials > 0) {
                pic_diag_row *prev = &a.hist[step % a.hist_len];
                prev->kinetic = 0.5 * a.mass * tot[kDiagFields];
                prev->momentum = a.mass * tot[kDiagFields + 1];
                *a.dstep = n;
            }
            const double qnan = __longlong_as_double(0x7ff8000000000000ll);
            row->step = n;
            row->kinetic = qnan;
            row->momentum = qnan;
            row->field = 0.5 * a.dx * fe_total;
            row->charge = tot[kDiagCharge];
            row->charge_q = (long long)tot_cq;
        }
        // the amplitudes on warp 1 (when there is one), beside thread 0's row
        const int mt = blockDim.x >= 64 ? t - 32 : t;
        if (mt >= 0 && mt < PIC_NMODES) {
            const double re = tot[kDiagModes + 2 * mt], im = tot[kDiagModes + 2 * mt + 1];
            row->mode[mt] = sqrt(re * re + im * im) * a.k_mode;
        }
    }
    cl.sync();
}

// ---- fixed-point solve on one thread-block cluster --------------------------
//
// The same exact integer solve with the nodes split into C <= 16 slices of
// ceil(NG/C) nodes: one slice per block of a cluster, one node per thread.
// Each block reads (and clears) only its own slice of the accumulator, takes
// one block pass of two inclusive scans over its slice, of R_k and of k R_k
// (I and J below, over b0 <= k <= g), and publishes its slice sums sum_k R_k
// and sum_k k R_k (the scans' warp totals, summed) in shared memory.  After a
// cluster barrier every block forms, from all slices' sums (one remote read
// per lane of warp 0; integer sums, so the order does not matter),
//   A0 = sum_{k<b0} R_k,  B = sum_{k<b0} k R_k,
//   SR = sum_k R_k,       SP = NG SR - sum_k k R_k,
// and solves its slice: P_g = A0 + I, M_g = NG P_g - SP,
// M_{g-1} = NG (P_g - R_g) - SP (M_{-1} = NG SR - SP), and
// sum_{k<g} P_k = g P_g - (B + J); then the diagnostics (cluster_finish).
// Three cluster barriers, no global atomics.
struct SliceSums {
    i128 s0, s1;                  // slice sums of R and k R
};

template <int MODE>
__global__ void __launch_bounds__(kClusterSolveThreads) pic_solve_cluster_kernel(SolveArgs a) {
    cg::cluster_group cl = cg::this_cluster();
    __shared__ SliceSums ex;
    __shared__ ClusterDiag cd;
    __shared__ i128 pre[4];
    __shared__ __align__(16) unsigned long long scan64[4 * 32];
    const int C = (int)cl.num_blocks(), r = (int)cl.block_rank();
    const int ng = a.ng, t = threadIdx.x;
    cudaGridDependencySynchronize();
    const long long step = *a.dstep;
    const i128 ntot = whole_density<MODE>(a);
    const int per = (int)blockDim.x;              // whole warps of nodes
    const int b0 = r * per;
    const int b1 = min(ng, b0 + per);
    const int g = b0 + t;
    const bool mine = g < b1;
    i128 q = 0;
    if (mine) q = take_density<MODE>(a, g);
    double kv[2];
    push_sums_share(a, C, r, kv);
    const i128 R = mine ? ntot - (i128)ng * q : (i128)0;
    // one pass of the slice's inclusive scans of R_k and k R_k
    const I128Pair sc = block_inclusive_scan2_i128(R, R * (i128)g, scan64);
    if (t == 0) {
        i128 S0 = 0, S1 = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
            S0 += (i128)(((unsigned __int128)scan64[32 + w] << 64) | scan64[w]);
            S1 += (i128)(((unsigned __int128)scan64[96 + w] << 64) | scan64[64 + w]);
        }
        ex.s0 = S0;
        ex.s1 = S1;
    }
    cl.sync();                                                        // #1

    if (t < 32) {
        i128 v0 = 0, v1 = 0;
        if (t < C) {
            const SliceSums *pe = cl.map_shared_rank(&ex, t);
            v0 = pe->s0;
            v1 = pe->s1;
        }
        i128 a0 = t < r ? v0 : (i128)0, bb = t < r ? v1 : (i128)0;
        // lanes C.. hold zeros: kMaxSolveCluster lanes carry the sums
        for (int o = kMaxSolveCluster / 2; o > 0; o >>= 1) {
            a0 += shfl_down_i128(a0, o);
            bb += shfl_down_i128(bb, o);
            v0 += shfl_down_i128(v0, o);
            v1 += shfl_down_i128(v1, o);
        }
        if (t == 0) { pre[0] = a0; pre[1] = bb; pre[2] = v0; pre[3] = v1; }
    }
    __syncthreads();
    const i128 A0 = pre[0], B = pre[1], SR = pre[2], SS1 = pre[3];
    const i128 SP = (i128)ng * SR - SS1;          // sum_k (NG-k) R_k
    const i128 P = A0 + sc.a;                                          // P_g
    const i128 M = (i128)ng * P - SP;                                  // M_g
    // M_{g-1} = NG P_{g-1} - SP with P_{g-1} = P_g - R_g; M_{-1} = M_{NG-1}
    const i128 Mprev = g == 0 ? (i128)ng * SR - SP : (i128)ng * (P - R) - SP;
    NodeDiag d;
    node_diag_reset(d);
    if (mine) {
        // sum_{k<g} P_k = sum_{j<g} (g - j) R_j = g P_g - sum_{j<=g} j R_j
        const i128 sumP = (i128)g * P - (B + sc.b);
        const i128 sumM = (i128)ng * sumP - (i128)g * SP;                // sum_{k<g} M_k
        const double E = a.k_e * i128_to_f64(M + Mprev);
        const float E32 = (float)E;
        a.rho[g] = a.k_rho * i128_to_f64(R);
        a.E64[g] = E;
        a.E32[g] = E32;
        a.phi[g] = a.k_phi * i128_to_f64(sumM);
        node_diag(d, g, ng, E, E32);
    }
    const double charge = r == 0 ? a.dx * a.k_rho * i128_to_f64(SR) : 0.0;
    cluster_finish(a, cl, cd, kv, d, charge,
                   MODE == PIC_FP32_FIXED ? (unsigned long long)q : 0ull, step);   // #2, #3
}

// ---- CG: the paper's field solver, on one thread-block cluster ------------
//
// Sec. 2.2 / Sec. 3.3 / Appendix A: the matrix-free conjugate gradient on the
// Eq. 6 system with Phi_0 = 0 pinned (row 0 the identity) and the last row
// taking Phi_NG = 0, from x = 0 with r = v = -rho dx^2 (r_0 = v_0 = 0),
// c = r.r; while the initial |r| > 1e-16, exactly maxit iterations of
//   z = A v, t = c / (z.v), x += t v, r -= t z, d = r.r, v = (d/c) v + r, c = d
// (the paper forces 150 and keeps the unconverged field).  Where the next
// step would divide by zero (z.v == 0, t not finite, d == 0) it stops early.
// Then Phi = x and E by Eq. 7 with periodic neighbours.  For a neutral box
// the converged x is the periodic solution in the Phi_0 = 0 gauge.
//
// The nodes are split over the blocks of one cluster, one node per thread,
// C = ceil(NG/32) <= 16 blocks, float64 throughout.  An iteration is a chain of
// dependent operations, and what bounds it is their latency: on GB300 a float64
// add, multiply or FMA takes 64 clocks, a division 1465, a cluster barrier
// about 400 and a read of another block's shared memory about 250.  So
//   * the sums z.v and r.r are taken in integers (warp_sum_fixed): the products
//     aligned to the warp's largest exponent and added by redux.sync, 200
//     clocks against 530 for a shuffle tree of float64 adds; they are exact to
//     2^-57 of the largest product, where the tree rounded each add;
//   * every warp stores its sum into all blocks' shared memory itself (st.async,
//     completing on a memory barrier there), so a sum over the cluster takes one
//     crossing instead of a barrier and a read; every block adds the same
//     integers, so all hold the same scalars;
//   * the two neighbour values of v that A v needs from other blocks are not
//     exchanged after the update: each block sends its boundary v (before the
//     update) and r (after it) with its part of r.r, and the neighbour forms
//     beta v + r itself, the same operation on the same numbers as the owner;
//   * t = c / z.v and beta = d / c are corrected products with reciprocals
//     (recip64, divide64), of which 1/c is formed while the sums cross.
// A step of 150 iterations takes 311 us on 1024 nodes, 549 with cluster barriers,
// float64 trees and divisions; an iteration's instructions, one after the other
// in 4200 clocks, are what bounds it now.
// A block's barrier of one sum cannot complete again before the block has added
// its own part of the next sum, which it sends only after reading the first, so
// one buffer per sum is enough.  Every wait has a limit (SolveArgs::wait_limit
// tries of up to a microsecond), after which the thread sets kErrWait and its sum is
// no number, with which its warp, the block at the end of the iteration (the only
// way out of the loop, so that the barriers of all warps match) and, for want of
// its sums, the other blocks stop.  What a block sent last has arrived by then.

constexpr int kCgParts = kMaxSolveCluster * kClusterSolveThreads / 32;    // warps of a cluster

struct CgExchange {
    double part[2][kCgParts];     // every warp's sum of z.v and of r.r
    double2 nbr[2];               // (v, r) at the left and the right neighbour's boundary
    unsigned long long bar[2];    // memory barriers of z.v and of r.r
    double x0, x1;                // Phi at the slice's first and last node
    i128 sr;                      // slice sum of R
};

__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned peer_addr(const void *p, int rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}

// Into another block's shared memory (peer_addr), counted on its barrier; and
// the bytes a barrier's phase waits for.  For the lanes with `on`, predicated:
// a branch around them costs a divergent warp more than they do.
__device__ __forceinline__ void send8(bool on, unsigned dst, double a, unsigned bar) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t"
                 "@p st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];\n\t}"
                 ::"r"(dst), "l"(__double_as_longlong(a)), "r"(bar), "r"((unsigned)on) : "memory");
}

__device__ __forceinline__ void send16(bool on, unsigned dst, double a, double b, unsigned bar) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
                 "@p st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];\n\t}"
                 ::"r"(dst), "l"(__double_as_longlong(a)), "l"(__double_as_longlong(b)), "r"(bar),
                 "r"((unsigned)on) : "memory");
}

__device__ __forceinline__ void expect_bytes(bool on, const void *bar, unsigned bytes) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t"
                 "@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}"
                 ::"r"(smem_addr(bar)), "r"(bytes), "r"((unsigned)on) : "memory");
}

__device__ __forceinline__ bool wait_phase(const void *bar, unsigned parity, unsigned limit) {
#pragma unroll 1
    for (unsigned i = 0; i < limit; i++) {
        unsigned done;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, 1000;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(smem_addr(bar)), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}

// 1/x: the hardware's approximation y0 (at least 20 bits) and one step of the
// cubic Newton iteration y0 (1 + e + e^2), e = 1 - x y0: e^3 is below 2^-60,
// the result within two units of the last place.  Three dependent FMAs.
__device__ __forceinline__ double recip64(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// a / b with y = recip64(b): the product, off by a few units of the last place, is
// corrected by its residual a - q b, which the FMA gives exactly (Markstein 1990).
// What is rounded at the end is then within 2^-48 units of a / b, so the result is
// the rounded quotient unless a / b lies that close to a rounding boundary (that in
// all cases, with two more steps each, took 355 us a step for 311).
__device__ __forceinline__ double divide64(double a, double b, double y) {
    const double q = a * y;
    return fma(fma(-q, b, a), y, q);
}

template <int MODE>
__global__ void __launch_bounds__(kClusterSolveThreads) pic_solve_cg_kernel(SolveArgs a) {
    cg::cluster_group cl = cg::this_cluster();
    __shared__ double sv[kClusterSolveThreads + 2];   // v of the slice, ghost-padded
    __shared__ __align__(16) CgExchange ex;
    __shared__ ClusterDiag cd;
    __shared__ i128 sh[96];
    __shared__ double scal[2];                        // t and beta; NaN: stop
    const int C = (int)cl.num_blocks(), r = (int)cl.block_rank();
    const int ng = a.ng, t = threadIdx.x, lane = t & 31, w = t >> 5, nw = blockDim.x >> 5;
    cudaGridDependencySynchronize();
    const long long step = *a.dstep;
    const double dx = a.dx;
    const int per = (ng + C - 1) / C;
    const int b0 = r * per;
    const int cnt = min(ng, b0 + per) - b0;
    const int g = b0 + t;
    const bool mine = t < cnt;
    if (t < 2) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&ex.bar[t])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    double kv[2];
    push_sums_share(a, C, r, kv);
    double rh = 0.0;
    i128 q = 0, R = 0;
    if (mine) {
        q = take_density<MODE>(a, g);
        R = whole_density<MODE>(a) - (i128)ng * q;
        rh = a.k_rho * i128_to_f64(R);
        a.rho[g] = rh;
    }
    {
        i128 z1 = 0, z2 = 0, sr = R;
        block_sum3_i128(sr, z1, z2, sh);
        if (t == 0) ex.sr = sr;
    }
    for (int i = t; i < kClusterSolveThreads + 2; i += blockDim.x) sv[i] = 0.0;
    cl.sync();                                        // barriers ready in all blocks
    // lane l of a warp sends the warp's sums to block l
    const int to = lane < C ? lane : 0;
    const unsigned dst[2] = {peer_addr(&ex.part[0][r * nw + w], to), peer_addr(&ex.part[1][r * nw + w], to)};
    const unsigned bar[2] = {peer_addr(&ex.bar[0], to), peer_addr(&ex.bar[1], to)};
    // the slice's first and last node send their (v, r) to the neighbour (a slice
    // with neighbours on both sides has at least 17 nodes)
    const bool first = t == 0 && r > 0, final = t == cnt - 1 && r < C - 1;
    const int nb = first ? r - 1 : final ? r + 1 : 0;
    const unsigned ndst = peer_addr(&ex.nbr[first ? 1 : 0], nb), nbar = peer_addr(&ex.bar[1], nb);
    const unsigned zv_bytes = 8u * ((unsigned)(C * nw) + a.wait_missing);
    const unsigned rr_bytes = zv_bytes + 16u * (unsigned)((r > 0 ? 1 : 0) + (r < C - 1 ? 1 : 0));
    double xg = 0.0;
    double rg = (mine && g >= 1) ? (-rh * dx) * dx : 0.0;
    double vg = 0.0;
    bool dead = false;                                // a wait of this thread ran out
    // Every warp takes the sums itself where a block has few (no block barrier
    // between the sum and its use); where it has many, their float64 scalars
    // would fill the pipe, and warp 0 hands them on.
    const bool every = nw <= 4;
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    auto publish = [&](int which, double p) {
        const double f = warp_sum_fixed(p);
        send8(lane < C, dst[which], f, bar[which]);
    };
    auto total = [&](int which, unsigned parity) {
        dead |= !wait_phase(&ex.bar[which], parity, a.wait_limit);
        double v = lane < C * nw ? ex.part[which][lane] : 0.0;
        for (int i = lane + 32; i < C * nw; i += 32) v += ex.part[which][i];
        return warp_sum_fixed(dead ? nan : v);        // in all lanes
    };
    double c = 0.0, rc = 0.0, beta = 0.0;
    for (int it = -1; it < a.cg_maxit; it++) {
        bool stop = false;                            // uniform over the warp, if not `every` the block
        if (it >= 0) {                                // (it = -1: r.r of the start)
            const double vc = sv[t + 1];
            double z = fma(-2.0, vc, sv[t]) + sv[t + 2];      // (Phi_NG = 0: the last ghost stays 0)
            z = g == 0 ? vc : z;
            z = mine ? z : 0.0;
            publish(0, z * vg);
            expect_bytes(t == 0, &ex.bar[0], zv_bytes);
            double tk = 0.0;
            if (every || w == 0) {
                rc = recip64(c);                      // for beta, while the sums cross
                const double zv = total(0, (unsigned)it & 1u);
                tk = divide64(c, zv, recip64(zv));
                // stop where the step would divide by zero
                tk = zv == 0.0 ? nan : tk;
            }
            if (!every) {
                if (t == 0) scal[0] = tk;
                __syncthreads();
                tk = scal[0];
            }
            stop = !isfinite(tk);
            if (!stop) {
                xg = fma(tk, vg, xg);
                rg = fma(-tk, z, rg);
            }
        }
        if (!stop) {
            publish(1, rg * rg);
            send16(first || final, ndst, vg, rg, nbar);
            expect_bytes(t == 0, &ex.bar[1], rr_bytes);
            if (every || w == 0) {
                const double d = total(1, (unsigned)(it + 1) & 1u);
                beta = it < 0 ? 0.0 : divide64(d, c, rc);
                // stop where the next step would divide by zero, and at the start where
                // |r| <= 1e-16
                if (!(d > 0.0) || (it < 0 && !(sqrt(d) > 1e-16 && ng > 1))) beta = nan;
                c = d;
            }
            if (!every) {
                if (t == 0) scal[1] = beta;
                __syncthreads();
                beta = scal[1];
            }
            stop = !isfinite(beta);
        }
        if (!stop) {
            vg = fma(beta, vg, rg);
            if (mine) sv[t + 1] = vg;
            // the neighbours' boundary v, formed as they form it
            const double2 nv = ex.nbr[final ? 1 : 0];
            const double gv = fma(beta, nv.x, nv.y);
            if (first || final) sv[final ? cnt + 1 : 0] = gv;
        }
        if (nw == 1) __syncwarp();
        else if (every) stop = __syncthreads_or(stop);
        else __syncthreads();
        if (stop) break;
    }
    if (dead) atomicOr(a.err, kErrWait);
    // Phi = x; E by Eq. 7 with periodic neighbours (across the blocks)
    __syncthreads();
    if (mine) sv[t + 1] = xg;
    if (t == 0) ex.x0 = xg;
    if (t == cnt - 1) ex.x1 = xg;
    cl.sync();
    if (t == 0) sv[0] = cl.map_shared_rank(&ex, r > 0 ? r - 1 : C - 1)->x1;
    if (t == cnt - 1) sv[cnt + 1] = cl.map_shared_rank(&ex, r < C - 1 ? r + 1 : 0)->x0;
    __syncthreads();
    NodeDiag dg;
    node_diag_reset(dg);
    if (mine) {
        const double E = -(sv[t + 2] - sv[t]) / (2.0 * dx);
        const float E32 = (float)E;
        a.phi[g] = xg;
        a.E64[g] = E;
        a.E32[g] = E32;
        node_diag(dg, g, ng, E, E32);
    }
    i128 sr = 0;
    if (r == 0)
        for (int b = 0; b < C; b++) sr += cl.map_shared_rank(&ex, b)->sr;
    const double charge = r == 0 ? dx * a.k_rho * i128_to_f64(sr) : 0.0;
    cluster_finish(a, cl, cd, kv, dg, charge,
                   MODE == PIC_FP32_FIXED ? (unsigned long long)q : 0ull, step);
}

using SolveKernel = void (*)(SolveArgs);

SolveKernel pick_solve(int mode, int solver) {
    const bool c = solver == PIC_SOLVER_CG;
    switch (mode) {
        case PIC_FP32_FIXED:
            return c ? &pic_solve_cg_kernel<PIC_FP32_FIXED> : &pic_solve_cluster_kernel<PIC_FP32_FIXED>;
        case PIC_FP32_ATOMIC:
            return c ? &pic_solve_cg_kernel<PIC_FP32_ATOMIC> : &pic_solve_cluster_kernel<PIC_FP32_ATOMIC>;
        default:
            return c ? &pic_solve_cg_kernel<PIC_FP64> : &pic_solve_cluster_kernel<PIC_FP64>;
    }
}

}  // namespace


// Cluster shape of the solves: C = ceil(NG / per_block) blocks (at most 16),
// ceil(NG / C) nodes each, rounded up to whole warps.  The exact solve takes
// up to 128 nodes per block, the CG 32 (both are float64-bound on GB300).  The
// exact solve's blocks take as many nodes as they have threads, so that every
// warp holds 32 nodes from a multiple of 32 on.
void solve_cluster_shape(int ng, int per_block, int *C, int *threads) {
    int c = (ng + per_block - 1) / per_block;
    c = c < 1 ? 1 : (c > kMaxSolveCluster ? kMaxSolveCluster : c);
    const int per = (ng + c - 1) / c;
    *C = c;
    *threads = ((per + 31) / 32) * 32;
}

cudaError_t solve_prepare_attributes() {
    for (int mode : {PIC_FP32_FIXED, PIC_FP32_ATOMIC, PIC_FP64})
        for (int solver : {PIC_SOLVER_EXACT, PIC_SOLVER_CG}) {
            const cudaError_t e = cudaFuncSetAttribute(
                pick_solve(mode, solver), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

cudaError_t launch_solve(const SolveArgs &a, cudaStream_t s) {
    int C = 1, threads = 32;
    solve_cluster_shape(a.ng, a.solver == PIC_SOLVER_CG ? 32 : kSolveNodesPerBlock, &C, &threads);
    return launch_after(pick_solve(a.mode, a.solver), dim3((unsigned)C), threads, 0, s, C, a);
}

}  // namespace pic
