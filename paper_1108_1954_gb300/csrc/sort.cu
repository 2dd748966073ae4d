// sort.cu -- periodic counting sort of the particles by cell.
//
// Not a step of the paper's method: it reorders the particle arrays so that
// the particles a warp handles share few cells, which makes the fused push's
// field reads broadcasts and lets its deposit aggregate equal nodes before the
// shared-memory atomics.  It changes no physical quantity.
//
// Four passes (five beyond 1024 cells), all deterministic and stable (particles
// of one cell keep their relative order):
//   count    block b counts the cells of its contiguous chunk -> hist[b][g]
//   colscan  per (segment of chunks, cell): exclusive prefix over the chunks
//            of the segment, in place, and the segment total
//   base     per cell: exclusive prefix over the segments, in place, and the
//            cell total (many cells: a pass of its own, segscan); exclusive prefix
//            of those over the cells -> base[g]
//   scatter  block b walks its chunk in order, 512 particles at a time
//            (64 consecutive per warp; long chunks 1024, 128); the warps take their slots from the
//            per-cell cursors one after the other, so the order within a
//            cell is the original order.
// A small sort is launches, not work (1e6 particles, 1024 cells: passes of 3, 3, 2
// and 8 us), so each pass but the first is launched with programmatic
// serialisation: its blocks come up while the pass ahead still runs, and wait
// for that pass (and so for all before it: each waits before it ends) where
// they first read its results.  The scatter has loaded its first particles by
// then; those are complete before the count begins, which waits for everything
// ahead of it in the stream.  A sort, us, five plain launches before and here: 2e4
// particles on 64 cells 24.5, 13.5; 1e6 on 1024 27.2, 19.9; 4.2e6 on 2048 47.3,
// 37.4; 1.2e7 on 4096 115.5, 108.7; 2^26 on 4096 390, 388 (353 with the long
// chunks' scatter, below).
// The destination index is bounds-checked; a violation sets the device error
// word instead of writing.
#include "pic_internal.cuh"

namespace pic {
namespace {

constexpr unsigned kNoKey = 0xffffffffu;

template <typename T>
__device__ __forceinline__ unsigned cell_key(T x, T inv_dx, int ng) {
    T u = x * inv_dx;
    u = u > (T)0 ? u : (T)0;                  // also maps NaN to 0
    const T top = (T)(ng - 1);
    u = u < top ? u : top;
    return (unsigned)u;
}

// The same for float64: one float64 instruction, the product, and the clamps and
// the truncation on its bits.  The comparisons and the conversion take the
// float64 pipe too, at 16 clocks a warp each, and bounded both passes (2^24
// particles: count 148 us, 42 so; scatter 162, 122 so).
__device__ __forceinline__ unsigned cell_key(double x, double inv_dx, int ng) {
    const double u = x * inv_dx;
    const int hi = __double2hiint(u);
    const unsigned top = (unsigned)(ng - 1);
    if (hi < 0x3ff00000) return 0u;                       // u < 1, negative
    if (hi >= 0x7ff00000) return hi == 0x7ff00000 && __double2loint(u) == 0 ? top : 0u;  // inf, NaN
    const int e = (hi >> 20) - 1023;
    const unsigned j = e > 20 ? top : (((unsigned)hi & 0xfffffu) | 0x100000u) >> (20 - e);
    return j < top ? j : top;
}

template <typename T>
__global__ void __launch_bounds__(kSortThreads) sort_count_kernel(SortArgs<T> a) {
    extern __shared__ unsigned sh_count[];
    cudaTriggerProgrammaticLaunchCompletion();
    const int ng = a.ng;
    for (int g = threadIdx.x; g < ng; g += blockDim.x) sh_count[g] = 0u;
    __syncthreads();
    const long long start = (long long)blockIdx.x * a.chunk;
    const long long end = min(a.n, start + a.chunk);
    if (sizeof(T) == 4 && (a.chunk & 3) == 0) {
        // float4 groups (the chunk starts on a group): equal cells among a
        // group's 4 particles are counted with one atomic, K groups in flight
        constexpr int K = 4;
        const float4 *x4 = reinterpret_cast<const float4 *>(a.x);
        const long long q0 = start >> 2, q1 = end >> 2;
        for (long long qb = q0; qb < q1; qb += K * blockDim.x) {
            float4 xv[K];
#pragma unroll
            for (int k = 0; k < K; k++) {
                const long long q = qb + k * blockDim.x + threadIdx.x;
                xv[k] = q < q1 ? __ldcs(x4 + q) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int k = 0; k < K; k++) {
                const long long q = qb + k * blockDim.x + threadIdx.x;
                if (q >= q1) continue;
                const float xs[4] = {xv[k].x, xv[k].y, xv[k].z, xv[k].w};
                unsigned key = cell_key((T)xs[0], a.inv_dx, ng), run = 1u;
#pragma unroll
                for (int j = 1; j < 4; j++) {
                    const unsigned kj = cell_key((T)xs[j], a.inv_dx, ng);
                    if (kj == key) {
                        run++;
                    } else {
                        atomicAdd(&sh_count[key], run);
                        key = kj;
                        run = 1u;
                    }
                }
                atomicAdd(&sh_count[key], run);
            }
        }
        // the chunk's last n mod 4 particles
        const long long i = (q1 << 2) + threadIdx.x;
        if (i < end) atomicAdd(&sh_count[cell_key(a.x[i], a.inv_dx, ng)], 1u);
    } else {
        constexpr int K = 8;   // loads in flight per thread
        for (long long i0 = start; i0 < end; i0 += K * blockDim.x) {
            T xv[K];
#pragma unroll
            for (int k = 0; k < K; k++) {
                const long long i = i0 + k * blockDim.x + threadIdx.x;
                xv[k] = i < end ? __ldcs(a.x + i) : (T)0;
            }
#pragma unroll
            for (int k = 0; k < K; k++) {
                const long long i = i0 + k * blockDim.x + threadIdx.x;
                if (i < end) atomicAdd(&sh_count[cell_key(xv[k], a.inv_dx, ng)], 1u);
            }
        }
    }
    __syncthreads();
    unsigned *row = a.hist + (size_t)blockIdx.x * ng;
    for (int g = threadIdx.x; g < ng; g += blockDim.x) row[g] = sh_count[g];
}

// Exclusive prefix, in place, of the column p[0], p[stride], ... p[(len-1)
// stride]; returns the column total.  Loads are issued 16 at a time.
__device__ __forceinline__ unsigned column_scan(unsigned *p, size_t stride, int len) {
    constexpr int kB = 16;
    unsigned run = 0;
    for (int k0 = 0; k0 < len; k0 += kB) {
        unsigned c[kB];
#pragma unroll
        for (int k = 0; k < kB; k++) c[k] = k0 + k < len ? p[(size_t)(k0 + k) * stride] : 0u;
#pragma unroll
        for (int k = 0; k < kB; k++) {
            if (k0 + k < len) p[(size_t)(k0 + k) * stride] = run;
            run += c[k];
        }
    }
    return run;
}

template <typename T>
__global__ void __launch_bounds__(256) sort_colscan_kernel(SortArgs<T> a) {
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= a.ng) return;
    const int seg = blockIdx.y;
    const int b0 = seg * a.seg_len, b1 = min(a.nchunk, b0 + a.seg_len);
    a.segtot[(size_t)seg * a.ng + g] = column_scan(a.hist + (size_t)b0 * a.ng + g, a.ng, b1 - b0);
}

// Per cell: exclusive prefix of the segment totals over the segments, in place,
// and the cell total.  Many cells only: few are done by the base pass itself.
template <typename T>
__global__ void __launch_bounds__(256) sort_segscan_kernel(SortArgs<T> a) {
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < a.ng) a.base[g] = column_scan(a.segtot + g, a.ng, a.nseg);
}

// One block.  The cell totals (SEGSCAN: as the pass above), then their exclusive
// prefix over the cells, the first slot of each cell (each thread scans a
// contiguous run of cells).
constexpr int kBaseThreads = 1024;

template <typename T, bool SEGSCAN>
__global__ void __launch_bounds__(kBaseThreads) sort_base_kernel(SortArgs<T> a) {
    __shared__ unsigned wt[kBaseThreads / 32], total[PIC_NCELL_MAX];
    // the scatter's blocks only now: brought up while the count's are resident they
    // would be spread unevenly over the SMs (2^26 particles: 406 us a sort, 386 so)
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
    const int ng = a.ng, t = threadIdx.x;
    for (int g = t; g < ng; g += kBaseThreads) total[g] = SEGSCAN ? column_scan(a.segtot + g, a.ng, a.nseg) : a.base[g];
    __syncthreads();
    const int k = (ng + kBaseThreads - 1) / kBaseThreads;
    const int g0 = min(ng, t * k), g1 = min(ng, g0 + k);
    unsigned local = 0;
    for (int g = g0; g < g1; g++) local += total[g];
    const int lane = t & 31, w = t >> 5;
    unsigned inc = local;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) wt[w] = inc;
    __syncthreads();
    unsigned run = __reduce_add_sync(kFull, lane < w ? wt[lane] : 0u) + inc - local;
    for (int g = g0; g < g1; g++) {
        a.base[g] = run;
        run += total[g];
    }
}

// The scatter walks its chunk in rounds of kSub x 256 particles: warp w owns
// the round's particles [32 kSub w, 32 kSub (w + 1)) as kSub steps of 32
// (lane l takes particle 32 j + l of step j).  Lanes of one cell in a step are
// ranked by __match_any_sync; in its turn a warp's leaders take their slots
// from the per-cell cursors, step after step; the warps take their turns in
// order, so a cell's particles keep their order in the chunk.  The next round's
// particles are loaded a round ahead.  The turns are a serial chain, which is
// what bounds the pass (2^25 particles: warps wait at barriers 3/4 of the time);
// what differs is what the other warps do meanwhile.
//   short chunks  the warps step through the turns together, a block barrier each;
//                 kSub = 2 (30 registers; 3, 4 and 8 leave fewer blocks per SM)
//   LONG          a warp hands its turn to the next over a barrier of the two and
//                 goes on to its stores and its next particles' keys; kSub = 4
//                 (2, 3 and 6 on 2^26 particles: 395, 373 and 383 us a sort against
//                 353).  The shorter the chunk, the more of it is the way to the
//                 last warp's first turn.
// us a sort, short and LONG: 3e6 particles on 777 cells 30.4, 31.9; 4.2e6 on 2048
// 37.6, 41.5; 8.4e6 on 512 51.6, 51.6, on 4096 85.6, 81.4; 1.2e7 on 4096 109, 102;
// 2^24 on 8192 246, 197; 2^26 on 4096 385, 353; float64 8.4e6 on 1024 94, 82, 2^24
// 174, 140.  Slots taken by fetch-adds: 379 on 2^26.
constexpr long long kLongChunk = 8192;

// A warp's turn: handed from one warp to the next over a barrier of their two (of
// the next one's number + 1; both threads' worth of one warp wait, the other's
// only arrive).  No barrier is used again before the turn has gone all round.
static_assert(kSortThreads / 32 <= 15, "a named barrier per warp");
__device__ __forceinline__ void turn_wait(int warp) {
    asm volatile("bar.sync %0, 64;" ::"r"(warp + 1) : "memory");
}
__device__ __forceinline__ void turn_pass(int warp) {
    __threadfence_block();
    asm volatile("bar.arrive %0, 64;" ::"r"(warp + 1) : "memory");
}

template <typename T, bool LONG>
__global__ void __launch_bounds__(kSortThreads) sort_scatter_kernel(SortArgs<T> a) {
    constexpr int kSub = LONG ? 4 : 2;
    extern __shared__ unsigned cursor[];
    const int ng = a.ng;
    const long long start = (long long)blockIdx.x * a.chunk;
    const long long end = min(a.n, start + a.chunk);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const long long round = (long long)kSub * blockDim.x;
    // this lane's particle of step j in the round beginning at r0
    const long long own = (long long)warp * (kSub * 32) + lane;
    auto ldx = [&](long long i) { return i < end ? __ldcs(a.x + i) : (T)0; };
    auto ldv = [&](long long i) { return i < end ? __ldcs(a.v + i) : (T)0; };
    T nx[kSub], nv[kSub];
#pragma unroll
    for (int j = 0; j < kSub; j++) {
        nx[j] = ldx(start + own + 32 * j);
        nv[j] = ldv(start + own + 32 * j);
    }
    cudaGridDependencySynchronize();
    const int seg = blockIdx.x / a.seg_len;
    const unsigned *row = a.hist + (size_t)blockIdx.x * ng;
    const unsigned *srow = a.segtot + (size_t)seg * ng;
    for (int g = threadIdx.x; g < ng; g += blockDim.x) cursor[g] = a.base[g] + srow[g] + row[g];
    __syncthreads();
    for (long long r0 = start; r0 < end; r0 += round) {
        T x[kSub], v[kSub];
#pragma unroll
        for (int j = 0; j < kSub; j++) {
            x[j] = nx[j];
            v[j] = nv[j];
            nx[j] = ldx(r0 + round + own + 32 * j);      // the next round, a round ahead
            nv[j] = ldv(r0 + round + own + 32 * j);
        }
        unsigned key[kSub], peers[kSub], base[kSub];
        int leader[kSub];
#pragma unroll
        for (int j = 0; j < kSub; j++) {
            const bool valid = r0 + own + 32 * j < end;
            key[j] = valid ? cell_key(x[j], a.inv_dx, ng) : kNoKey;
            peers[j] = __match_any_sync(kFull, key[j]);
            leader[j] = __ffs(peers[j]) - 1;
            base[j] = 0u;
        }
        auto take = [&] {
#pragma unroll
            for (int j = 0; j < kSub; j++) {
                if (key[j] != kNoKey && lane == leader[j]) {
                    base[j] = cursor[key[j]];
                    cursor[key[j]] = base[j] + (unsigned)__popc(peers[j]);
                }
                __syncwarp();
            }
        };
        if (LONG) {
            if (warp > 0 || r0 > start) turn_wait(warp);
            take();
            if (warp < nwarp - 1) turn_pass(warp + 1);
            else if (r0 + round < end) turn_pass(0);
        } else {
            for (int w = 0; w < nwarp; w++) {
                if (w == warp) take();
                __syncthreads();
            }
        }
#pragma unroll
        for (int j = 0; j < kSub; j++) {
            const unsigned b = __shfl_sync(kFull, base[j], leader[j]);
            if (key[j] != kNoKey) {
                const unsigned long long dst = (unsigned long long)b + __popc(peers[j] & lt);
                if (dst < (unsigned long long)a.n) {
                    a.x_out[dst] = x[j];
                    a.v_out[dst] = v[j];
                } else {
                    atomicOr(a.err, kErrSortKey);
                }
            }
        }
    }
}

template <typename T>
cudaError_t launch_sort_t(const SortArgs<T> &a, cudaStream_t s) {
    const size_t smem = (size_t)a.ng * sizeof(unsigned);
    sort_count_kernel<T><<<a.nchunk, kSortThreads, smem, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_after(&sort_colscan_kernel<T>, dim3((a.ng + 255) / 256, a.nseg), 256, 0, s, 0, a);
    // With several cells a thread the one block's column scans take longer than a
    // launch.  A sort, us, without and with the separate pass: 2e4 particles on 64
    // cells 13.5, 14.9; 1e6 on 1024 19.9, 20.1; 4.2e6 on 2048 40.1, 37.4.
    const bool one = a.ng <= kBaseThreads;
    if (e == cudaSuccess && !one) e = launch_after(&sort_segscan_kernel<T>, dim3((a.ng + 255) / 256), 256, 0, s, 0, a);
    if (e == cudaSuccess)
        e = launch_after(one ? &sort_base_kernel<T, true> : &sort_base_kernel<T, false>, dim3(1), kBaseThreads,
                         0, s, 0, a);
    if (e == cudaSuccess)
        e = launch_after(a.chunk >= kLongChunk ? &sort_scatter_kernel<T, true> : &sort_scatter_kernel<T, false>,
                         dim3(a.nchunk), kSortThreads, smem, s, 0, a);
    return e;
}

}  // namespace

cudaError_t sort_prepare_attributes(int ng) {
    (void)ng;
    const int bytes = PIC_NCELL_MAX * (int)sizeof(unsigned);
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(&sort_count_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes))) return e;
    if ((e = cudaFuncSetAttribute(&sort_count_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes))) return e;
    for (auto *k : {&sort_scatter_kernel<float, false>, &sort_scatter_kernel<float, true>})
        if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes))) return e;
    for (auto *k : {&sort_scatter_kernel<double, false>, &sort_scatter_kernel<double, true>})
        if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes))) return e;
    return cudaSuccess;
}

cudaError_t launch_sort_f32(const SortArgs<float> &a, cudaStream_t s) { return launch_sort_t(a, s); }
cudaError_t launch_sort_f64(const SortArgs<double> &a, cudaStream_t s) { return launch_sort_t(a, s); }

}  // namespace pic
