// small_step.cuh -- many steps of a small lattice by one thread-block cluster
// (Sec. 4, the same fused step as step_block.cuh), its state in the shared
// memory of the cluster's CTAs.  Included by small_step.cu (one lattice) and
// batch_table.cuh (a cluster per lattice).
//
// What bounds it: latency.  CTA b of C owns rows [b ny / C, (b+1) ny / C) and
// keeps the post-stream populations of its cells, and those of the next step,
// in two shared-memory buffers.  A step is:
//   1. the densities of the CTA's rows and of one row either side (whose
//      populations are read from the neighbour CTA's shared memory: nine
//      independent reads) go into a shared density field;
//   2. a block barrier;
//   3. every cell collides and pushes its nine populations to the slots they
//      stream to (or its own opposite slot at a wall or solid) in the other
//      buffer, a neighbour CTA's where the row is not the CTA's own;
//   4. one cluster barrier (release / acquire); the buffers swap.
// So a step waits for one cluster barrier and one round of reads from a
// neighbour CTA.  With the state in global memory, two barriers and three
// dependent L2 reads a step, 32 x 32 FP64 took 8.1 us a step and 61 x 53 FP32
// 5.1 us.
// The global state is read once and written after the last two steps (both
// buffers of the lattice then hold what single steps would have left there).
// Every CTA runs the same number of steps and barriers, with no early exit
// (a checked build skips an access that fails its bounds test and records
// bit 1 of the status word at the end).
// The arithmetic is that of step_block in the same order (FP32: two cells of
// a row in one float2), so a lattice goes through the same states bit for
// bit on either path.
#pragma once
#include <cooperative_groups.h>

#include "lbm_device.cuh"
#include "lbm_launch.h"

namespace lbm {

namespace {

// Shared memory of one CTA: two population buffers of 9 planes x R rows, the
// densities of R + 2 rows, for FP32 the slots that each pair of cells pushes
// to (kSmallTable words a pair; see small_run) and a word that solid cells
// push to, and the link bits of R rows.
constexpr int kSmallTable = 20;
template <typename T>
__host__ __device__ constexpr int small_row(int nx) { return (nx + 1) & ~1; }
template <typename T>
__host__ __device__ constexpr size_t small_smem_bytes(int nx, int ny, int C) {
    const int R = (ny + C - 1) / C, P = small_row<T>(nx);
    const size_t cells = ((size_t)(18 * R + R + 2) * P) * sizeof(T);
    const size_t table = sizeof(T) == 4 ? 16 + (size_t)kSmallTable * 4 * R * (P / 2) : 0;
    return (cells + 15) / 16 * 16 + table + (size_t)R * P;
}
// cells of a row one thread handles, and threads a CTA takes at most
template <typename T> constexpr int kSmallVec = sizeof(T) == 4 ? 2 : 1;
template <typename T> constexpr int kSmallMaxThreads = sizeof(T) == 4 ? 512 : 256;
template <typename T>
__host__ __device__ inline int small_threads(int nx, int ny, int C) {
    const int R = (ny + C - 1) / C, G = (nx + kSmallVec<T> - 1) / kSmallVec<T>;
    const int n = ((R + 2) * G + 31) / 32 * 32;  // a thread per own and halo group
    return n < kSmallMaxThreads<T> ? n : kSmallMaxThreads<T>;
}

// the cells of one group (FP32: two, 8-byte aligned)
__device__ __forceinline__ void group_ld(const float* p, float* v) {
    const float2 q = *reinterpret_cast<const float2*>(p);
    v[0] = q.x;
    v[1] = q.y;
}
__device__ __forceinline__ void group_ld(const double* p, double* v) { v[0] = *p; }
__device__ __forceinline__ unsigned cluster_map(unsigned addr, unsigned rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_ld(unsigned addr, float* v) {  // two cells
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(addr));
}
__device__ __forceinline__ void cluster_ld(unsigned addr, double* v) {
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[0]) : "r"(addr));
}
__device__ __forceinline__ void cluster_st(unsigned addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_st(unsigned addr, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_barrier() {
    cluster_arrive();
    cluster_wait();
}

// pull() with loads that bypass L1 (the buffers are written later in the launch)
template <typename S, typename P>
__device__ __forceinline__ void pull_l2(const S* fin, const P& p, int x, int y, unsigned sb,
                                        S f[9], bool& bad) {
    const int xm = x == 0 ? p.nx - 1 : x - 1;
    const int xp = x == p.nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? p.ny - 1 : y - 1;
    const int yp = y == p.ny - 1 ? 0 : y + 1;
    const long long pl = p.plane;
    const long long rc = (long long)y * p.rstride, rm = (long long)ym * p.rstride,
                    rp = (long long)yp * p.rstride;
    const long long c = rc + x;
    const long long idx[9] = {c,
                              (sb & 1u) ? 3 * pl + c : 1 * pl + rc + xm,
                              (sb & 2u) ? 4 * pl + c : 2 * pl + rm + x,
                              (sb & 4u) ? 1 * pl + c : 3 * pl + rc + xp,
                              (sb & 8u) ? 2 * pl + c : 4 * pl + rp + x,
                              (sb & 16u) ? 7 * pl + c : 5 * pl + rm + xm,
                              (sb & 32u) ? 8 * pl + c : 6 * pl + rm + xp,
                              (sb & 64u) ? 5 * pl + c : 7 * pl + rp + xp,
                              (sb & 128u) ? 6 * pl + c : 8 * pl + rp + xm};
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        if (kChecked && !idx_ok(idx[i], 9 * pl)) {
            bad = true;
            f[i] = S(0);
            continue;
        }
        f[i] = __ldcg(fin + idx[i]);
    }
}

// the deviations of a cell summed in step_block's order
template <typename T>
__device__ __forceinline__ T density(const T g[9]) {
    return ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8];
}

// nsteps steps of one lattice from buffer `from` (f0 or f1), by the CTAs of
// one cluster (this one: rank of C).  bits: the lattice's link bits (0xFF
// solid), rows bpitch apart.  smem: small_smem_bytes.
template <typename T, typename PT>
__device__ __forceinline__ void small_run(const PT& p, T* f0, T* f1,
                                          const uint8_t* __restrict__ bits, int bpitch, int from,
                                          int nsteps, unsigned char* smem, int rank, int C) {
    constexpr int VC = kSmallVec<T>;
    const int nx = p.nx, ny = p.ny;
    const int R = (ny + C - 1) / C, P = small_row<T>(nx);
    const int y0 = (int)((long long)rank * ny / C), y1 = (int)((long long)(rank + 1) * ny / C);
    const int rows = y1 - y0;
    const int G = (nx + VC - 1) / VC;                // groups of VC cells in a row
    const unsigned inv = 0xFFFFFFFFu / (unsigned)G + 1u;  // it / G = umulhi(it, inv), it < 2^16
    const int plane = R * P, bufn = 9 * plane;
    T* buf = reinterpret_cast<T*>(smem);
    T* dens = buf + 2 * bufn;                        // row r of the band at (r + 1) P
    // FP32: word 0 of `table` takes what solid cells push; pair q's slots follow
    const size_t cells = ((size_t)(18 * R + R + 2) * P * sizeof(T) + 15) / 16 * 16;
    unsigned* table = reinterpret_cast<unsigned*>(smem + cells) + 4;
    uint8_t* sbits = sizeof(T) == 4 ? reinterpret_cast<uint8_t*>(table + kSmallTable * R * (P / 2))
                                    : smem + cells;
    const int tid = threadIdx.x, nt = blockDim.x;
    bool bad = false;

    // shared-memory addresses of the rows y0 - 1 and y1 (column 0 of plane 0 of
    // buffer 0) in the CTAs that own them; hv: the row exists
    unsigned haddr[2];
    bool hv[2];
    const unsigned base = (unsigned)__cvta_generic_to_shared(buf);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        int yy = k == 0 ? y0 - 1 : y1;
        hv[k] = (yy >= 0 && yy < ny) || p.py;
        yy = yy < 0 ? ny - 1 : yy >= ny ? 0 : yy;
        const int owner = (int)(((long long)(yy + 1) * C - 1) / ny);
        const int first = (int)((long long)owner * ny / C);
        haddr[k] = cluster_map(base + (unsigned)((yy - first) * P * (int)sizeof(T)), (unsigned)owner);
        if (kChecked && !(owner >= 0 && owner < C && yy - first >= 0 && yy - first < R)) bad = true;
    }

    // the state: pulled from global memory once, the cells of a group together
    // (their reads in flight at once); an inactive last column counts as solid.  A
    // single step pulls the rows either side too, for their densities, and then needs
    // no neighbour CTA.
    const int own = rows * G, items = own + 2 * G;
    const bool one = nsteps == 1;
    {
        const T* fin = from ? f1 : f0;
        for (int it = tid; it < (one ? items : own); it += nt) {
            const int r = (int)__umulhi((unsigned)it, inv), x = (it - r * G) * VC;
            int y = y0 + r;
            if (r >= rows) {  // the row below the band, or the one above it
                if (!(r == rows ? hv[0] : hv[1])) continue;
                y = r == rows ? y0 - 1 : y1;
                y = y < 0 ? ny - 1 : y >= ny ? 0 : y;
            }
            unsigned sb[VC];
            T g[VC][9];
#pragma unroll
            for (int j = 0; j < VC; ++j)
                sb[j] = x + j >= nx ? 0xFFu
                        : p.lmask   ? bits[(long long)y * bpitch + x + j]
                                    : link_bits<false>(p, x + j, y);
#pragma unroll
            for (int j = 0; j < VC; ++j)
                if (sb[j] != 0xFFu) pull_l2(fin, p, x + j, y, sb[j], g[j], bad);
#pragma unroll
            for (int j = 0; j < VC; ++j) {
                if (r >= rows) {
                    if (sb[j] != 0xFFu)
                        dens[(r == rows ? 0 : rows + 1) * P + x + j] = density(g[j]);
                    continue;
                }
                sbits[r * P + x + j] = (uint8_t)sb[j];
                if (sb[j] == 0xFFu) continue;
#pragma unroll
                for (int i = 0; i < 9; ++i) buf[i * plane + r * P + x + j] = g[j][i];
            }
        }
    }
    __syncthreads();
    // FP32: where each population of each pair of cells goes: byte offsets in
    // the cluster's shared memory, of buffer 0 (bit 0 set: of no buffer, the
    // word for solid cells), so that a step pushes without a test.  What they
    // cost instead, tests of nine links and two edges a cell, was half of a
    // step.
    if (VC == 2 && !one) {  // (a single step pushes nothing)
        const unsigned self = cluster_map(base, (unsigned)rank);
        const unsigned dump = self + (unsigned)((unsigned char*)(table - 4) - smem) + 1u;
        for (int it = tid; it < own; it += nt) {
            const int r = (int)__umulhi((unsigned)it, inv), x = (it - r * G) * VC;
#pragma unroll
            for (int j = 0; j < VC; ++j) {
                const int xj = x + j;
                const unsigned sb = sbits[r * P + xj];
                const int xw = xj == 0 ? nx - 1 : xj - 1, xe = xj >= nx - 1 ? 0 : xj + 1;
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const int tx = ex(i) == 0 ? xj : ex(i) > 0 ? xe : xw, tr = r + ey(i);
                    unsigned a;
                    if (sb == 0xFFu)
                        a = dump;
                    else if (i > 0 && ((sb >> (opp(i) - 1)) & 1u))  // back into the cell
                        a = self + (unsigned)((opp(i) * plane + r * P + xj) * (int)sizeof(T));
                    else if (tr >= 0 && tr < rows)
                        a = self + (unsigned)((i * plane + tr * P + tx) * (int)sizeof(T));
                    else
                        a = (tr < 0 ? haddr[0] : haddr[1]) +
                            (unsigned)((i * plane + tx) * (int)sizeof(T));
                    if (kChecked && !(tx >= 0 && tx < P && tr >= -1 && tr <= rows)) {
                        bad = true;
                        a = dump;
                    }
                    table[it * kSmallTable + j * 9 + i] = a;
                }
            }
        }
    }
    if (!one) cluster_barrier();

    for (int s = 0; s < nsteps; ++s) {
        const T* cur = buf + (s & 1) * bufn;
        const int nxt = ((s & 1) ^ 1) * bufn;
        // 1. densities
        for (int it = tid; it < (one ? own : items); it += nt) {
            const int r = (int)__umulhi((unsigned)it, inv), x = (it - r * G) * VC;
            T g[9][VC];
            T* dst = dens;
            if (r < rows) {
                const T* q = cur + r * P + x;
#pragma unroll
                for (int i = 0; i < 9; ++i) group_ld(q + i * plane, g[i]);
                dst += (r + 1) * P + x;
            } else {
                const bool below = r == rows;  // the row below the band, or the one above it
                if (!(below ? hv[0] : hv[1])) continue;
                const unsigned a = (below ? haddr[0] : haddr[1]) + (unsigned)(((s & 1) * bufn + x) * (int)sizeof(T));
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    cluster_ld(a + (unsigned)(i * plane * (int)sizeof(T)), g[i]);
                dst += (below ? 0 : rows + 1) * P + x;
            }
            // summed in step_block's order
#pragma unroll
            for (int j = 0; j < VC; ++j)
                dst[j] = ((g[0][j] + g[1][j]) + (g[2][j] + g[3][j])) +
                         ((g[4][j] + g[5][j]) + (g[6][j] + g[7][j])) + g[8][j];
        }
        __syncthreads();
        // 3. collide and push
        const bool last = s + 1 == nsteps, global = s + 2 >= nsteps;
        // (the last step reads nothing more from its neighbours and pushes nothing)
        if (last && !one) cluster_arrive();
        T* fout = ((from + s) & 1) ? f0 : f1;
        for (int it = tid; it < own; it += nt) {
            const int r = (int)__umulhi((unsigned)it, inv), x = (it - r * G) * VC, y = y0 + r;
            const T* q = cur + r * P + x;
            const T* dq = dens + (r + 1) * P;
            T g[9][VC], d[VC], dxr[VC], dyr[VC], rho[VC];
            unsigned sb[VC];
#pragma unroll
            for (int i = 0; i < 9; ++i) group_ld(q + i * plane, g[i]);
#pragma unroll
            for (int j = 0; j < VC; ++j) {
                const int xj = x + j;
                sb[j] = sbits[r * P + xj];
                d[j] = dq[xj];
                const T w = dq[xj == 0 ? nx - 1 : xj - 1], e = dq[xj >= nx - 1 ? 0 : xj + 1];
                const T dW = (sb[j] & 1u) ? d[j] : w;
                const T dS = (sb[j] & 2u) ? d[j] : dq[xj - P];
                const T dE = (sb[j] & 4u) ? d[j] : e;
                const T dN = (sb[j] & 8u) ? d[j] : dq[xj + P];
                dxr[j] = T(0.5) * (dE - dW);
                dyr[j] = p.iah * (dN - dS);
                rho[j] = p.rho0 + d[j];
            }
            if (p.collide) {
                if constexpr (VC == 2) {
                    float2 F[9];
#pragma unroll
                    for (int i = 0; i < 9; ++i) F[i] = make_float2(g[i][0], g[i][1]);
                    const float2 D = make_float2(d[0], d[1]), Gx = make_float2(dxr[0], dxr[1]),
                                 Gy = make_float2(dyr[0], dyr[1]);
                    const float2 Q =
                        p.raw ? collide_raw<float>(to_lanes(p.cc), F, D, Gx, Gy)
                              : (p.forced ? collide<float, true>(to_lanes(p.cc), F, D, Gx, Gy)
                                          : collide<float, false>(to_lanes(p.cc), F, D, Gx, Gy));
                    rho[0] = Q.x;
                    rho[1] = Q.y;
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        g[i][0] = F[i].x;
                        g[i][1] = F[i].y;
                    }
                } else {
                    T F[9];
#pragma unroll
                    for (int i = 0; i < 9; ++i) F[i] = g[i][0];
                    rho[0] = p.raw ? collide_raw<T>(to_lanes(p.cc), F, d[0], dxr[0], dyr[0])
                                   : (p.forced ? collide<T, true>(to_lanes(p.cc), F, d[0], dxr[0], dyr[0])
                                               : collide<T, false>(to_lanes(p.cc), F, d[0], dxr[0], dyr[0]));
#pragma unroll
                    for (int i = 0; i < 9; ++i) g[i][0] = F[i];
                }
            }
            if constexpr (VC == 2) {
                // a moving wall acts on the cells along it alone
                if (p.moving && (x == 0 || x + VC >= nx || y == 0 || y == ny - 1)) {
#pragma unroll
                    for (int j = 0; j < VC; ++j) {
                        const int xj = x + j;
                        if (sb[j] == 0xFFu || !(xj == 0 || xj == nx - 1 || y == 0 || y == ny - 1))
                            continue;
                        T f[9];
#pragma unroll
                        for (int i = 0; i < 9; ++i) f[i] = g[i][j];
                        moving_wall(p, xj, y, rho[j], f);
#pragma unroll
                        for (int i = 0; i < 9; ++i) g[i][j] = f[i];
                    }
                }
                if (global) {
#pragma unroll
                    for (int j = 0; j < VC; ++j) {
                        const int xj = x + j;
                        if (xj >= nx) continue;
                        const long long o = (long long)y * p.rstride + xj;
                        if (kChecked && !(y >= 0 && y < ny && xj < p.rstride)) {
                            bad = true;
                            continue;
                        }
#pragma unroll
                        for (int i = 0; i < 9; ++i)
                            fout[i * p.plane + o] = sb[j] == 0xFFu ? T(0) : g[i][j];
                    }
                }
                if (!last) {
                    unsigned a[kSmallTable];
                    const uint4* tq = reinterpret_cast<const uint4*>(table + it * kSmallTable);
#pragma unroll
                    for (int k = 0; k < kSmallTable / 4; ++k) {
                        const uint4 v = tq[k];
                        a[4 * k] = v.x;
                        a[4 * k + 1] = v.y;
                        a[4 * k + 2] = v.z;
                        a[4 * k + 3] = v.w;
                    }
                    const unsigned off = (unsigned)(nxt * (int)sizeof(T));
#pragma unroll
                    for (int j = 0; j < VC; ++j)
#pragma unroll
                        for (int i = 0; i < 9; ++i) {
                            const unsigned w = a[j * 9 + i];
                            cluster_st((w & 1u) ? w - 1u : w + off, g[i][j]);
                        }
                }
                continue;
            }
#pragma unroll
            for (int j = 0; j < VC; ++j) {
                const int xj = x + j;
                if (xj >= nx) continue;
                T f[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) f[i] = sb[j] == 0xFFu ? T(0) : g[i][j];
                if (p.moving && sb[j] != 0xFFu && (xj == 0 || xj == nx - 1 || y == 0 || y == ny - 1))
                    moving_wall(p, xj, y, rho[j], f);
                if (global) {
                    const long long o = (long long)y * p.rstride + xj;
                    if (kChecked && !(y >= 0 && y < ny && xj < p.rstride)) {
                        bad = true;
                    } else {
#pragma unroll
                        for (int i = 0; i < 9; ++i) fout[i * p.plane + o] = f[i];
                    }
                }
                if (last || sb[j] == 0xFFu) continue;
                const int xw = xj == 0 ? nx - 1 : xj - 1, xe = xj == nx - 1 ? 0 : xj + 1;
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const int k = opp(i);
                    if (i > 0 && ((sb[j] >> (k - 1)) & 1u)) {  // back into the cell
                        buf[nxt + k * plane + r * P + xj] = f[i];
                        continue;
                    }
                    const int tx = ex(i) == 0 ? xj : ex(i) > 0 ? xe : xw, tr = r + ey(i);
                    if (kChecked && !(tx >= 0 && tx < nx && tr >= -1 && tr <= rows)) {
                        bad = true;
                        continue;
                    }
                    if (ey(i) == 0 || (tr >= 0 && tr < rows))
                        buf[nxt + i * plane + tr * P + tx] = f[i];
                    else
                        cluster_st((tr < 0 ? haddr[0] : haddr[1]) +
                                       (unsigned)((nxt + i * plane + tx) * (int)sizeof(T)),
                                   f[i]);
                }
            }
        }
        if (!last) cluster_arrive();
        if (!one) cluster_wait();
    }
    if (kChecked && bad) atomicOr(p.status, kStatusBounds);
}

}  // namespace

}  // namespace lbm
