// particle_ops.cuh -- the per-particle arithmetic of the PIC step, shared by
// the single-run fused push (push.cu) and the batched cluster kernel
// (batch.cu), so that a run gives bit-identical particles in either.
//   locate         cell of a position by the fixed-point recipe
//   fixed_weight   the right node's share trunc(f * 2^24)
//   Tile           a block's private density in shared memory, and the deposits
//   push_particle  gather (Sec. 2.3), kick (Eq. 3), drift (Eq. 2), wrap
#pragma once

#include "pic_internal.cuh"

namespace pic {

using u64 = unsigned long long;

// 8 consecutive float32 values moved by one 32-byte vector load or store
// (the QUAD8 and PAIR8 variants; the address 32-byte aligned).  .cs:
// streamed (the single run's arrays pass once per step); .cg: cached in L2
// only (the batched kernel's runs).
struct F8 {
    float v[8];
};

template <bool CG = false>
__device__ __forceinline__ F8 ld8(const float *p) {
    F8 r;
    if (CG)
        asm volatile("ld.global.cg.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3]), "=f"(r.v[4]),
                       "=f"(r.v[5]), "=f"(r.v[6]), "=f"(r.v[7])
                     : "l"(p));
    else
        asm volatile("ld.global.cs.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3]), "=f"(r.v[4]),
                       "=f"(r.v[5]), "=f"(r.v[6]), "=f"(r.v[7])
                     : "l"(p));
    return r;
}

template <bool CG = false>
__device__ __forceinline__ void st8(float *p, const F8 &r) {
    if (CG)
        asm volatile("st.global.cg.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p),
                     "f"(r.v[0]), "f"(r.v[1]), "f"(r.v[2]), "f"(r.v[3]), "f"(r.v[4]),
                     "f"(r.v[5]), "f"(r.v[6]), "f"(r.v[7])
                     : "memory");
    else
        asm volatile("st.global.cs.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p),
                     "f"(r.v[0]), "f"(r.v[1]), "f"(r.v[2]), "f"(r.v[3]), "f"(r.v[4]),
                     "f"(r.v[5]), "f"(r.v[6]), "f"(r.v[7])
                     : "memory");
}

// Cell location of a float32 cell coordinate u (the fixed-point recipe):
//   s = u - 1/2, fl = floor(s), f = s - fl   (float ops, round to nearest)
// floor(s) is formed as (s + 1.5*2^23 rounded down) - 1.5*2^23, which equals
// floorf(s) exactly for |s| < 2^22 (NG <= 8192; checked for every float in
// [-1, 8193]) and runs on the FMA pipe instead of the conversion unit; the
// rounded-down sum's bit pattern is 0x4B400000 + fl, which gives the node index
// without a float-to-int conversion.
// j = fl + 1 is the index of the left node in the ghost-padded tiles (node -1,
// the periodic image of NG-1, is j = 0); a valid position has j in [0, NG].
// A NaN, infinite or far-out-of-range position fails that one unsigned test.
struct Loc {
    unsigned j;
    float f;
};

constexpr float kMagic = 12582912.0f;          // 1.5 * 2^23
constexpr int kMagicBitsMinus1 = 0x4B400000 - 1;

__device__ __forceinline__ Loc locate(float u) {
    Loc l;
    const float s = __fsub_rn(u, 0.5f);
    const float t = __fadd_rd(s, kMagic);
    const float fl = __fsub_rn(t, kMagic);
    l.f = __fsub_rn(s, fl);
    l.j = (unsigned)(__float_as_int(t) - kMagicBitsMinus1);
    return l;
}

// The right node's share W = trunc(f * 2^24) of a particle's 2^24.
__device__ __forceinline__ unsigned fixed_weight(float f) {
    return __float2uint_rz(__fmul_rn(f, 16777216.0f));
}

// Kick (Eq. 3), drift (Eq. 2, in cell units: u advances by v dt NG/L) and
// the periodic wrap to [0, NG) of one particle, given the field ep at the
// particle; accumulates v_old v_new and v_new.
__device__ __forceinline__ void kick_drift_wrap(float &u, float &v, float ep, const PushConsts &c,
                                                float &ke, float &mom) {
    const float vn = fmaf(c.qmdt, ep, v);
    ke = fmaf(v, vn, ke);
    mom += vn;
    float un = fmaf(vn, c.kdrift, u);
    un = un < 0.0f ? un + c.ngf : un;
    un = un >= c.ngf ? un - c.ngf : un;
    un = un >= c.ngf ? 0.0f : un;      // u + NG rounded up to NG: the point 0
    u = un;
    v = vn;
}

// Gather (left and right node), kick, drift, wrap.
// sE[j] = E_{(j-1) mod NG} for j = 0..NG+1 (ghost-padded).
__device__ __forceinline__ void push_particle(float &u, float &v, const float *sE,
                                              const PushConsts &c, float &ke,
                                              float &mom) {
    const Loc l = locate(u);
    const bool ok = l.j <= (unsigned)c.ng;
    const unsigned j = ok ? l.j : 0u;
    const float e0 = sE[j], e1 = sE[j + 1];
    const float ep = ok ? fmaf(l.f, e1 - e0, e0) : 0.0f;
    kick_drift_wrap(u, v, ep, c, ke, mom);
}

// Nearest-grid-point weighting (PIC_SHAPE_NGP; Sec. 2: a grid point's density
// counts the particles of its cell, and a particle feels its cell's field):
// with nodes at the cell centres the cell of u is floor(u), formed by the
// same rounded-down magic sum as locate (exact on [-1, 8193]).  Returns the
// ghost-padded tile index j = cell + 1; a valid position has j - 1 in
// [0, NG] (one unsigned test).
__device__ __forceinline__ unsigned locate_ngp(float u) {
    const float t = __fadd_rd(u, kMagic);
    return (unsigned)(__float_as_int(t) - kMagicBitsMinus1);
}

__device__ __forceinline__ void push_particle_ngp(float &u, float &v, const float *sE,
                                                  const PushConsts &c, float &ke,
                                                  float &mom) {
    const unsigned j = locate_ngp(u);
    const bool ok = j - 1u <= (unsigned)c.ng;
    const float ep = ok ? sE[j] : 0.0f;
    kick_drift_wrap(u, v, ep, c, ke, mom);
}

// s + e = a + b exactly (Knuth's two-sum); pairs (h, l) added over a warp
__device__ __forceinline__ void add_pair(float &h, float &l, float h2, float l2) {
    const float s = __fadd_rn(h, h2);
    const float t = __fsub_rn(s, h);
    const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, t)), __fsub_rn(h2, t));
    l = __fadd_rn(__fadd_rn(l, l2), e);
    h = s;
}

// The same for one value and three adds less, exact where |h| >= |v| (Dekker's fast
// two-sum); otherwise off by a rounding of v at most.
__device__ __forceinline__ void add_fast(float &h, float &l, float v) {
    const float s = __fadd_rn(h, v);
    l = __fadd_rn(l, __fsub_rn(v, __fsub_rn(s, h)));
    h = s;
}

// (x, y) and (z, w) summed over the first n lanes of a warp (the others hold
// zeros), in lane 0.
__device__ __forceinline__ void warp_sum_pairs(float4 &p, int n) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (o >= n) continue;                         // uniform
        add_pair(p.x, p.y, __shfl_down_sync(kFull, p.x, o), __shfl_down_sync(kFull, p.y, o));
        add_pair(p.z, p.w, __shfl_down_sync(kFull, p.z, o), __shfl_down_sync(kFull, p.w, o));
    }
}

// Shared-memory density tiles.  GB300 has no single-instruction 64-bit integer
// add on shared memory (it is a compare-and-swap loop), so sums are kept in 32
// bits by fetch-adds, and the one add that wraps a word counts a carry.
//
// Node tiles (the combining variants MATCH, QUAD, PAIR, and the batched kernel): per ghost-padded node j
// = 0..NG+1 (node j - 1 mod NG) the low word w and the carries n of its sum; a
// run of particles adds its left and its right weights.
//
// Cell tiles (kDepositCells: ATOMIC in the single run): a particle in the cell between nodes j - 1 and j (j =
// 0..NG, locate) gives its left node 2^24 - W and its right node W, so per cell
// the number of particles n and the sum w of W are kept, and the nodes formed
// when the tile is read.  An add of the constant 1 that returns nothing is
// counted over the lanes of a warp by the hardware: lanes on one word cost no
// more than one lane, where other adds take a clock per lane.  Measured, clocks
// per warp of particles on one SM (4 of them the loop's random numbers):
//   distinct cells in the warp      1     2     4     8    16   many
//   two fetch-adds per particle  63.0  36.2  22.2  14.5  10.1   9.1
//   count and fetch-add          32.8  19.3  12.5   8.6   6.8   6.8
// Runs add more than 1 at a time and gain nothing from it (QUAD 0.188 ms a push
// of 2^26 particles with cell tiles, 0.184 with node tiles; PAIR8 takes 48
// registers instead of 40), so they keep node tiles.
// Carries of one cell number at most n / 256, so while a tile takes fewer than
// 2^20 particles both fit the count's word: count below, carries from bit 20
// (cinc = 2^20, c = n).  A tile of more has words of its own for the carries
// (cinc = 1).
//
// The nearest-grid-point shape only counts, in n[j] for the node j - 1.
template <int VARIANT>
struct CellTile {
    static constexpr bool value = VARIANT == kDepositCells;
};

struct Tile {
    unsigned *w, *n, *c;    // low words; carries (node tiles) or counts; carries (cell tiles)
    unsigned cinc;          // one carry
    unsigned k;             // cell j's word is j << k (2^k copies of the tile, steps.cu)
};

// A tile of `words` words per array at mem; 8 or (wide) 12 bytes per word.
__device__ __forceinline__ Tile make_tile(unsigned char *mem, int words, bool wide) {
    Tile t;
    t.w = reinterpret_cast<unsigned *>(mem);
    t.n = t.w + words;
    t.c = wide ? t.n + words : t.n;
    t.cinc = wide ? 1u : 1u << kCountBits;
    t.k = 0u;
    return t;
}

// A node tile: val to node j.
__device__ __forceinline__ void tile_add(const Tile &t, unsigned j, unsigned val) {
    const unsigned old = atomicAdd(&t.w[j], val);
    if (old + val < old) atomicAdd(&t.n[j], 1u);
}

// A cell tile: one particle of right weight W in cell j.
__device__ __forceinline__ void tile_add_one(const Tile &t, unsigned j, unsigned W) {
    atomicAdd(&t.n[j << t.k], 1u);
    const unsigned old = atomicAdd(&t.w[j << t.k], W);
    if (old + W < old) atomicAdd(&t.c[j << t.k], t.cinc);
}

// A cell's count and sum of W from its three words (the carry word is the count
// word unless wide).
struct CellSum {
    unsigned n;
    u64 W;
};
__device__ __forceinline__ CellSum cell_sum(unsigned w, unsigned n, unsigned c, bool wide) {
    CellSum s;
    s.n = wide ? n : n & ((1u << kCountBits) - 1u);
    s.W = ((u64)(wide ? c : n >> kCountBits) << 32) | w;
    return s;
}

// (one copy)
__device__ __forceinline__ CellSum tile_cell(const Tile &t, int j) {
    return cell_sum(t.w[j], t.n[j], t.c[j], t.cinc == 1u);
}

// The tile's share of ghost-padded node j = 0..NG+1.
template <int VARIANT>
__device__ __forceinline__ u64 tile_node(const Tile &t, int j, int ng) {
    if (VARIANT == kDepositNgp) return (u64)t.n[j] << kFixBits;
    if (!CellTile<VARIANT>::value) return ((u64)t.n[j] << 32) | (u64)t.w[j];
    u64 v = 0ull;
    if (j <= ng) {
        const CellSum s = tile_cell(t, j);
        v = ((u64)s.n << kFixBits) - s.W;
    }
    if (j >= 1) v += tile_cell(t, j - 1).W;
    return v;
}

// Deposit one particle (all 32 lanes of the warp call this together for the
// MATCH variants).
template <int VARIANT>
__device__ __forceinline__ void deposit_one(const Tile &t, float x, bool valid,
                                            const PushConsts &c, unsigned *err, int lane) {
    if (VARIANT == kDepositNgp) {
        const unsigned j = locate_ngp(x);
        const bool ok = valid && j - 1u <= (unsigned)c.ng;
        if (valid && !ok) atomicOr(err, kErrPosition);
        if (ok) atomicAdd(&t.n[j << t.k], 1u);
        return;
    }
    const Loc l = locate(x);
    const bool ok = valid && l.j <= (unsigned)c.ng;
    if (valid && !ok) atomicOr(err, kErrPosition);
    const unsigned W = ok ? fixed_weight(l.f) : 0u;
    if (CellTile<VARIANT>::value) {
        if (ok) tile_add_one(t, l.j, W);
    } else if (VARIANT != PIC_DEPOSIT_MATCH) {
        if (ok) {
            tile_add(t, l.j, kFixOne - W);
            tile_add(t, l.j + 1, W);
        }
    } else {
        const unsigned key = ok ? l.j : 0xffffffffu;
        const unsigned peers = __match_any_sync(kFull, key);
        const unsigned wsum = __reduce_add_sync(peers, W);
        if (ok && lane == __ffs(peers) - 1) {
            const unsigned cnt = (unsigned)__popc(peers);
            // cnt * 2^24 - wsum <= 2^29: fits the 32-bit add
            tile_add(t, l.j, (cnt << kFixBits) - wsum);
            tile_add(t, l.j + 1, wsum);
        }
    }
}

// Deposit the first m of W particles into a cell tile: the fetch-adds in flight
// together, their carries after them.
template <int W>
__device__ __forceinline__ void deposit_cells(const Tile &t, const float (&xs)[W], int m,
                                              const PushConsts &c, unsigned *err) {
    unsigned j[W], w[W], old[W];
    bool ok[W], bad = false;
#pragma unroll
    for (int k = 0; k < W; k++) {
        const Loc l = locate(xs[k]);
        ok[k] = k < m && l.j <= (unsigned)c.ng;
        bad |= k < m && !ok[k];
        j[k] = l.j << t.k;
        w[k] = fixed_weight(l.f);
    }
#pragma unroll
    for (int k = 0; k < W; k++) {
        old[k] = 0u;
        if (ok[k]) {
            atomicAdd(&t.n[j[k]], 1u);
            old[k] = atomicAdd(&t.w[j[k]], w[k]);
        }
    }
#pragma unroll
    for (int k = 0; k < W; k++)
        if (ok[k] && old[k] + w[k] < old[k]) atomicAdd(&t.c[j[k]], t.cinc);
    if (bad) atomicOr(err, kErrPosition);
}

// The first m of W particles of the nearest-grid-point shape.
template <int W>
__device__ __forceinline__ void deposit_ngp(const Tile &t, const float (&xs)[W], int m,
                                            const PushConsts &c, unsigned *err) {
    bool bad = false;
#pragma unroll
    for (int k = 0; k < W; k++) {
        const unsigned j = locate_ngp(xs[k]);
        const bool ok = k < m && j - 1u <= (unsigned)c.ng;
        bad |= k < m && !ok;
        if (ok) atomicAdd(&t.n[j << t.k], 1u);
    }
    if (bad) atomicOr(err, kErrPosition);
}

// Deposit a thread's W consecutive particles (W = 4: a float4 group; W = 8:
// the 32-byte groups of the QUAD8 / PAIR8 variants), valid per lane.
template <int VARIANT, int W>
__device__ __forceinline__ void deposit_group(const Tile &t, const float (&xs)[W], bool valid,
                                              const PushConsts &c, unsigned *err, int lane) {
    if (VARIANT == kDepositNgp) {
        deposit_ngp<W>(t, xs, valid ? W : 0, c, err);
    } else if (VARIANT == PIC_DEPOSIT_PAIR || VARIANT == PIC_DEPOSIT_PAIR8) {
        // two open runs (key, left, right); a third key closes run a
        unsigned ka = 0xffffffffu, la = 0, ra = 0, kb = 0xffffffffu, lb = 0, rb = 0;
        bool bad = false;
#pragma unroll
        for (int k = 0; k < W; k++) {
            const Loc l = locate(xs[k]);
            const bool ok = valid && l.j <= (unsigned)c.ng;
            bad |= valid && !ok;
            const unsigned Wk = fixed_weight(l.f);
            if (!ok) continue;
            if (l.j == ka) {
                la += kFixOne - Wk;
                ra += Wk;
            } else if (l.j == kb) {
                lb += kFixOne - Wk;
                rb += Wk;
            } else if (ka == 0xffffffffu) {
                ka = l.j; la = kFixOne - Wk; ra = Wk;
            } else if (kb == 0xffffffffu) {
                kb = l.j; lb = kFixOne - Wk; rb = Wk;
            } else {
                tile_add(t, ka, la);
                tile_add(t, ka + 1, ra);
                ka = l.j; la = kFixOne - Wk; ra = Wk;
            }
        }
        if (ka != 0xffffffffu) { tile_add(t, ka, la); tile_add(t, ka + 1, ra); }
        if (kb != 0xffffffffu) { tile_add(t, kb, lb); tile_add(t, kb + 1, rb); }
        if (bad) atomicOr(err, kErrPosition);
    } else if (VARIANT == PIC_DEPOSIT_QUAD || VARIANT == PIC_DEPOSIT_QUAD8) {
        // consecutive particles of the group with equal left node are summed
        // in registers first (at most W 2^24 <= 2^27 per word), then added once
        unsigned key = 0xffffffffu, left = 0, right = 0;
        bool bad = false;
#pragma unroll
        for (int k = 0; k < W; k++) {
            const Loc l = locate(xs[k]);
            const bool ok = valid && l.j <= (unsigned)c.ng;
            bad |= valid && !ok;
            const unsigned Wk = fixed_weight(l.f);
            if (ok && l.j == key) {
                left += kFixOne - Wk;
                right += Wk;
            } else if (ok) {
                if (key != 0xffffffffu) {
                    tile_add(t, key, left);
                    tile_add(t, key + 1, right);
                }
                key = l.j;
                left = kFixOne - Wk;
                right = Wk;
            }
        }
        if (key != 0xffffffffu) {
            tile_add(t, key, left);
            tile_add(t, key + 1, right);
        }
        if (bad) atomicOr(err, kErrPosition);
    } else if (CellTile<VARIANT>::value) {
        deposit_cells<W>(t, xs, valid ? W : 0, c, err);
    } else {
#pragma unroll
        for (int k = 0; k < W; k++) deposit_one<VARIANT>(t, xs[k], valid, c, err, lane);
    }
}

// Deposit the 4 particles of a float4 group (valid per lane).
template <int VARIANT>
__device__ __forceinline__ void deposit4(const Tile &t, const float4 &xx, bool valid,
                                         const PushConsts &c, unsigned *err, int lane) {
    const float xs[4] = {xx.x, xx.y, xx.z, xx.w};
    deposit_group<VARIANT, 4>(t, xs, valid, c, err, lane);
}

}  // namespace pic
