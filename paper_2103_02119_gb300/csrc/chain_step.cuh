// chain_step.cuh -- two fused steps of a large FP32 lattice (Sec. 4; Sec. 3 for
// the raw-moment scheme): K = 2 warps in a chain, each one step behind the
// other, march up a strip of 64 columns.
//
// Why: a step that reads and writes the whole state is bound by memory (72 B a
// cell), and its row-band kernel by the row barrier and by instructions that
// are not the collision.  Here a launch reads and writes the state once for K
// steps, a strip needs no barrier wider than its K warps, and a row costs a
// warp about 350 instructions for 64 cells against 620.
//
// A lane holds two neighbouring cells.  Warp 0 of the chain copies the rows of
// the state into a ring of shared memory (cp.async, each lane its own cells,
// kChainDepth rows ahead), the other warps read the rows that the warp before
// them left in theirs.  When row q arrives, a warp
//   1. gathers what row q - 1 pulls: the planes with e_y = +1, 0, -1 from the
//      rows q - 2, q - 1, q of its ring, shifted along x by shuffles, and
//      sums its density;
//   2. collides row q - 2 (gathered a row earlier, kept in registers; its
//      density gradient needs rows q - 3 .. q - 1) and hands it on: to the
//      next warp's ring, or, the last warp, to the state.
// Rows come two a turn, with one block barrier a turn; a warp starts three
// turns after the one before it, when its first rows are there.
// The strip's outer columns (two per step and side) and the band's outer rows
// (two per step and end) are computed by both neighbours: 56 of 64 columns are
// stored.  The bounced-back population of a blocked link is the cell's own
// opposite one, in row q - 1 of the ring; rows without blocked links (most)
// skip the selection.  The link bits of a turn's two rows come with loads a
// turn ahead, which nothing touches meanwhile: an instruction between the load
// and the row (a conversion, a select, the move of a register rotation) waits
// for memory, also where it is predicated off.
//
// What bounds it: the FP32 pipe (55 to 60 % busy) with four warps a scheduler
// to hide the latency of a row; 128 registers and 23 KB a chain let no more in.
// Measured, MLUPS, against the row-band kernel (100 steps): periodic
// 2048 x 8192 105k / 75.6k and 2048 x 1024 75.5k / 52.8k, cavity 2048 x 8192
// 103k / 80.3k, raw-moment scheme 106k / 81.0k, cavities with obstacles
// 2048 x 8192 101k / 78.1k and 1543 x 3001 86k / 58.8k.  Not kept (2048 x 8192):
// one step per launch (75k) or three (82k: halo columns); populations shifted
// by the copies, 4 bytes at a time (80k: shared-memory bandwidth); previous
// rows carried in registers (86.6k); two rows ahead instead of one (92.5k: the
// L1 cache gets what shared memory leaves); 20 warps per SM (58k: spills); two
// or four chains per block (79k, 70k); a barrier every row (89k); the strips at
// the lattice's sides read cell by cell (98.6k; with obstacles 84k: now only
// where an odd width wraps around); tall bands first, then short ones for the
// last quarter (91k).
//
// The arithmetic is that of step_block in the same order, so a lattice goes
// through the same states bit for bit on either path.
#pragma once
#include <type_traits>
#include "lbm_device.cuh"
#include "lbm_launch.h"

namespace lbm {

namespace {

constexpr int kChainDepth = 1;     // rows fetched ahead
constexpr int kStrip = 64;         // columns of a warp: two a lane
constexpr int kRowPairs = 9 * 32;  // float2 of a row's populations

// 8 or 4 bytes global -> shared, asynchronously
__device__ __forceinline__ void fetch8(unsigned dst, const char* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void fetch4(unsigned dst, const char* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
// v at column x - 1 / x + 1 (lane pairs)
__device__ __forceinline__ float2 from_west(float2 v) {
    return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x);
}
__device__ __forceinline__ float2 from_east(float2 v) {
    return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1));
}
// per cell (low byte of b: first cell): b's bit ? a : v
__device__ __forceinline__ float2 pick(unsigned b, unsigned bit, float2 a, float2 v) {
    return make_float2((b & bit) ? a.x : v.x, (b & (bit << 8)) ? a.y : v.y);
}

constexpr int kFetchSlots = kChainDepth + 3;  // rows q - 2 .. q + kChainDepth of the first warp
constexpr int kHandSlots = 6;                 // rows q - 2 .. q + 1, and the two being written
template <int K>
__host__ __device__ constexpr size_t chain_smem_bytes() {  // of one chain
    return (size_t)(kFetchSlots + kHandSlots * (K - 1)) * kRowPairs * sizeof(float2);
}

// K steps of rows y0 .. y1 - 1 and the strip's columns by the chain's warp
// `stage`; sm: chain_smem_bytes<K>(); constants(): the collision's.  nx >= 64,
// ny >= 16, 4 plane < 2^32.  PB: the type of a plane's byte offset, unsigned
// where 36 plane < 2^32 (the tight variant, fewer registers).
template <int SCH, bool MASK, int K, bool PAIRS, typename PB, typename PT, typename CC>
__device__ __forceinline__ void march_strip(const float* __restrict__ fin, float* __restrict__ fout,
                                            const PT& p, int strip, int y0, int y1, int stage,
                                            float2* sm, CC constants) {
    constexpr int kHaloC = 2 * K, kValid = kStrip - 2 * kHaloC;
    const int lane = threadIdx.x & 31;
    const int nx = p.nx, ny = p.ny;
    const int xs = strip * kValid - kHaloC;
    const int c0 = xs + 2 * lane;       // logical column of the lane's first cell
    auto col = [&](int c) {             // where a logical column is stored
        if (p.px) return c < 0 ? c + nx : c >= nx ? c - nx : c;
        // beyond a wall: any column, which no link reads
        return min(max(c, 0), p.pitch - 2);
    };
    auto row_of = [&](int r) {
        if (p.py) return r < 0 ? r + ny : r >= ny ? r - ny : r;
        return min(max(r, 0), ny - 1);
    };
    const int ca = col(c0), cb = PAIRS ? ca + 1 : col(c0 + 1);
    const bool stores = lane >= kHaloC / 2 && lane < 32 - kHaloC / 2 && c0 < nx;
    // walls along x, as link bits of the two cells
    unsigned xb = 0;
    bool xwall = false;
    if (!p.px) {
        if (c0 == 0) xb |= 0x91u;
        if (c0 == nx - 1) xb |= 0x64u;
        if (c0 + 1 == nx - 1) xb |= 0x6400u;
        xwall = xs <= 0 || xs + kStrip >= nx;
    }
    const bool xmoves = p.wall_odd[0][0] != 0.0f || p.wall_odd[0][1] != 0.0f ||
                        p.wall_odd[0][2] != 0.0f || p.wall_odd[1][0] != 0.0f ||
                        p.wall_odd[1][1] != 0.0f || p.wall_odd[1][2] != 0.0f;
    // Link bits of the two rows of a turn, the first in the low half: with a
    // mask the loads of the next turn's rows are in flight meanwhile (put
    // together at its start: anything done to them earlier waits for them).
    unsigned in[MASK ? (PAIRS ? 2 : 4) : 1];
    auto fetch_bits = [&](int r) {
        if constexpr (MASK) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const uint8_t* m = p.lmask + (unsigned)row_of(r + k) * (unsigned)p.pitch;
                if constexpr (PAIRS) {
                    asm volatile("ld.global.nc.u16 %0, [%1];" : "=r"(in[k]) : "l"(m + (unsigned)ca));
                } else {
                    asm volatile("ld.global.nc.u8 %0, [%1];" : "=r"(in[2 * k]) : "l"(m + (unsigned)ca));
                    asm volatile("ld.global.nc.u8 %0, [%1];" : "=r"(in[2 * k + 1]) : "l"(m + (unsigned)cb));
                }
            }
        }
    };
    auto bits_of = [&]() -> unsigned {
        if constexpr (MASK && PAIRS) return in[0] | in[1] << 16;
        else if constexpr (MASK) return in[0] | in[1] << 8 | in[2] << 16 | in[3] << 24;
        else return 0;
    };
    // without a mask: of one row, made where they are used
    auto wall_bits = [&](int r) -> unsigned {
        unsigned b = xb;
        if (!p.py) b |= (r == 0 ? 0x3232u : 0u) | (r == ny - 1 ? 0xC8C8u : 0u);
        return b;
    };
    auto any_of = [&](unsigned b, int r) -> bool {
        // a fluid cell with blocked links (0xFF: solid)
        if constexpr (MASK)
            return __any_sync(0xffffffffu, (b & 0xFFu) - 1u < 0xFEu || (b >> 8) - 1u < 0xFEu);
        return xwall || (!p.py && (r == 0 || r == ny - 1));
    };
    // byte offsets of 32 bits from the planes' (uniform) addresses
    const char* fbase = reinterpret_cast<const char*>(fin);
    const PB pb = (PB)(p.plane * 4);
    auto at = [&](auto* base, int i, unsigned o) {  // byte o of plane i
        if constexpr (sizeof(PB) == 4) return base + (o + (unsigned)i * pb);
        else return base + i * pb + o;
    };
    const unsigned dst0 = (unsigned)__cvta_generic_to_shared(sm) + 8u * lane;
    bool bad = false;  // checked build: a failed bounds check (the access is skipped)
    auto issue = [&](int r, int s) {
        const unsigned dst = dst0 + (unsigned)(s * kRowPairs * 8);
        const unsigned row = (unsigned)row_of(r) * (unsigned)p.rstride;
        if constexpr (kChecked) {
            if (!(idx_ok(row_of(r), ny) && idx_ok(s, kFetchSlots) && idx_ok(ca, p.rstride) &&
                  idx_ok(cb, p.rstride) && (!PAIRS || (ca & 1) == 0))) {
                bad = true;
                return;
            }
        }
        if constexpr (PAIRS) {
            const unsigned o = (row + (unsigned)ca) * 4u;
#pragma unroll
            for (int i = 0; i < 9; ++i) fetch8(dst + i * 256, at(fbase, i, o));
        } else {
            const unsigned oa = (row + (unsigned)ca) * 4u, ob = (row + (unsigned)cb) * 4u;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                fetch4(dst + i * 256, at(fbase, i, oa));
                fetch4(dst + i * 256 + 4, at(fbase, i, ob));
            }
        }
    };

    // rows of this stage: first .. last arrive (and one more where their number
    // is odd), two a turn; a stage starts three turns after the one before it
    const int first = y0 - 2 * (K - stage), last = y1 - 1 + 2 * (K - stage);
    const int stop = first + (last - first + 2) / 2 * 2;
    const float2 z = make_float2(0.0f, 0.0f);
    float2 G[9] = {z, z, z, z, z, z, z, z, z}, dS = z, dC = z;
    unsigned bt = 0, bp = 0;  // link bits of this turn's rows and of the previous turn's
    bool a1 = false, a2 = false;
    fetch_bits(first);
    const int nslots = stage == 0 ? kFetchSlots : kHandSlots;
    // slots of rows q, q - 1, q - 2 of my ring, and of the row I write next
    int s0 = 0, s1 = nslots - 1, s2 = nslots - 2;
    int so = 2;  // the four rows before the next stage's first go to slots 2 .. 5
    if (stage == 0)
#pragma unroll
        for (int d = 0; d < kChainDepth; ++d) {
            issue(first + d, d);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
    float2* mine = sm + (stage == 0 ? 0 : kFetchSlots + kHandSlots * (stage - 1)) * kRowPairs + lane;
    float2* hout = sm + (kFetchSlots + kHandSlots * stage) * kRowPairs + lane;
    if constexpr (K > 1)
        for (int w = 0; w < 3 * stage; ++w) __syncthreads();
    for (int q = first; q < stop;) {
        bp = bt;
        bt = bits_of();
        fetch_bits(q + 2);
#pragma unroll
        for (int k = 0; k < 2; ++k, ++q) {
            if (stage == 0) {
                // into the slot of row q - 3
                int sn = s0 + kChainDepth;
                sn = sn >= kFetchSlots ? sn - kFetchSlots : sn;
                issue(q + kChainDepth, sn);
                asm volatile("cp.async.commit_group;" ::: "memory");
                asm volatile("cp.async.wait_group %0;" ::"n"(kChainDepth) : "memory");
            }
            if constexpr (sizeof(PB) == 4) {  // two registers fewer
                s1 = s0 >= 1 ? s0 - 1 : s0 - 1 + nslots;
                s2 = s0 >= 2 ? s0 - 2 : s0 - 2 + nslots;
            }
            const float2 *r0 = mine + s0 * kRowPairs, *r1 = mine + s1 * kRowPairs,
                         *r2 = mine + s2 * kRowPairs;
            // link bits of rows q - 1 and q - 2, from bit h1 and h2 on
            const int h1 = MASK && !k ? 16 : 0, h2 = MASK && k ? 16 : 0;
            const unsigned b1 = !MASK ? wall_bits(q - 1) : k ? bt : bp;
            const unsigned b2 = !MASK ? wall_bits(q - 2) : bp;
            const bool a0 = any_of(k ? bt >> 16 : bt & 0xFFFFu, q);
            // the pulled populations of row q - 1
            float2 g[9];
            g[0] = r1[0];
            g[1] = from_west(r1[1 * 32]);
            g[3] = from_east(r1[3 * 32]);
            g[2] = r2[2 * 32];
            g[5] = from_west(r2[5 * 32]);
            g[6] = from_east(r2[6 * 32]);
            g[4] = r0[4 * 32];
            g[7] = from_east(r0[7 * 32]);
            g[8] = from_west(r0[8 * 32]);
            if (a1) {  // bounced back: the cell's own opposite populations
#pragma unroll
                for (int i = 1; i < 9; ++i) g[i] = pick(b1, 1u << (i - 1 + h1), r1[opp(i) * 32], g[i]);
            }
            s2 = s1;
            s1 = s0;
            s0 = s0 + 1 == nslots ? 0 : s0 + 1;
            const float2 dN = vadd(vadd(vadd(vadd(g[0], g[1]), vadd(g[2], g[3])),
                                        vadd(vadd(g[4], g[5]), vadd(g[6], g[7]))),
                                   g[8]);
            // row q - 2 collides
            const int r = q - 2;
            {
                float2 w = from_west(dC), e = from_east(dC), sd = dS, nn = dN;
                if (a2) {
                    w = pick(b2, 1u << h2, dC, w);
                    sd = pick(b2, 2u << h2, dC, sd);
                    e = pick(b2, 4u << h2, dC, e);
                    nn = pick(b2, 8u << h2, dC, nn);
                }
                const float2 dxr = vmul(make_float2(0.5f, 0.5f), vsub(e, w));
                const float2 dyr = vmul(make_float2(p.iah, p.iah), vsub(nn, sd));
                const float2 rho = SCH == 1 ? collide_raw<float>(constants(), G, dC, dxr, dyr)
                                            : collide<float, SCH != 3>(constants(), G, dC, dxr, dyr);
                if (p.moving && a2 && (xmoves || r == 0 || r == ny - 1)) {
                    float fa[9], fb[9];
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        fa[i] = G[i].x;
                        fb[i] = G[i].y;
                    }
                    moving_wall(p, c0, r, rho.x, fa);
                    moving_wall(p, c0 + 1, r, rho.y, fb);
#pragma unroll
                    for (int i = 0; i < 9; ++i) G[i] = make_float2(fa[i], fb[i]);
                }
                if (stage < K - 1) {
                    float2* o = hout + so * kRowPairs;
                    if (kChecked && !idx_ok(so, kHandSlots)) {
                        bad = true;
                        o = hout;
                    }
                    so = so + 1 == kHandSlots ? 0 : so + 1;
#pragma unroll
                    for (int i = 0; i < 9; ++i) o[i * 32] = G[i];
                } else if (stores && r >= y0 && r < y1) {
                    const unsigned lo = 0xFFu << h2, hi = 0xFF00u << h2;
                    if (MASK && ((b2 & lo) == lo || (b2 & hi) == hi)) {
                        // a solid cell keeps its zeros
#pragma unroll
                        for (int i = 0; i < 9; ++i) {
                            if ((b2 & lo) == lo) G[i].x = 0.0f;
                            if ((b2 & hi) == hi) G[i].y = 0.0f;
                        }
                    }
                    const unsigned o = ((unsigned)r * (unsigned)p.rstride + (unsigned)c0) * 4u;
                    if (kChecked && !(idx_ok(r, ny) && idx_ok(c0, p.rstride, 2))) bad = true;
                    else
#pragma unroll
                    for (int i = 0; i < 9; ++i)
                        *reinterpret_cast<float2*>(at(reinterpret_cast<char*>(fout), i, o)) = G[i];
                }
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) G[i] = g[i];
            dS = dC;
            dC = dN;
            a2 = a1;
            a1 = a0;
        }
        if constexpr (K > 1) __syncthreads();
    }
    if constexpr (K > 1)
        for (int w = stage; w < K - 1; ++w) __syncthreads();
    if (kChecked && bad) atomicOr(p.status, kStatusBounds);
}

// The strip's lanes read their two cells as an aligned pair, but where an odd
// width wraps around.
template <int SCH, bool MASK, int K, typename PB, typename PT, typename CC>
__device__ __forceinline__ void chain_march(const float* fin, float* fout, const PT& p, int strip,
                                            int y0, int y1, int stage, float2* sm, CC constants) {
    const int xs = strip * (kStrip - 4 * K) - 2 * K;
    if (!p.px || (p.nx & 1) == 0 || (xs >= 0 && xs + kStrip <= p.nx))
        march_strip<SCH, MASK, K, true, PB>(fin, fout, p, strip, y0, y1, stage, sm, constants);
    else
        march_strip<SCH, MASK, K, false, PB>(fin, fout, p, strip, y0, y1, stage, sm, constants);
}

template <int SCH, bool MASK, int K>
__global__ void __launch_bounds__(32 * K, 16 / K)
chain_kernel(const float* __restrict__ fin, float* __restrict__ fout,
             const __grid_constant__ KParams<float> p, int nbands) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int band = blockIdx.y;
    const int y0 = (int)((long long)band * p.ny / nbands);
    const int y1 = (int)((long long)(band + 1) * p.ny / nbands);
    // the strips along the walls take longer: first in every band
    const int x = blockIdx.x, n = gridDim.x;
    chain_march<SCH, MASK, K, long long>(fin, fout, p, x == 0 ? n - 1 : x - 1, y0, y1, threadIdx.x >> 5,
                              reinterpret_cast<float2*>(smem), [&] { return to_lanes(p.cc); });
}

}  // namespace

}  // namespace lbm
