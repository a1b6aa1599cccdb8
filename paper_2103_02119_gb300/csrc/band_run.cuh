// band_run.cuh -- many steps of a middle-sized FP32 lattice in one launch: a
// CTA per band of rows on as many SMs as there are bands, its state in shared
// memory (small_step.cuh, without the limit of one cluster).
//
// Why: with a launch per step such a lattice waits for launches, and for the
// row-band kernel's chain of loads and barriers.  Here a step is
//   1. wait for the two neighbour CTAs' flags; densities of the CTA's rows and
//      of one row either side;
//   2. every cell collides and pushes its populations to the slots they stream
//      to, all in the CTA's own buffer, which has a halo row at each end;
//   3. what a neighbour needs goes to its mailbox in global memory: the edge row
//      next to it (nine planes, for the density of its halo row) and the halo row
//      that the edge row pushed into (three planes, for its own edge row); then the
//      CTA's flag is raised.
// A halo row's density is summed from the neighbour's nine planes and, for the
// three directions that leave the band, from what the CTA pushed there itself,
// or, where the halo cell's link is blocked, from the neighbour's bounced one.
// So a step is one exchange between neighbours, and no barrier of the grid.
// Mailboxes alternate by parity: a CTA writes the mailbox of step s after its
// neighbour's flag s - 1, which is raised after the neighbour has read the one
// of step s - 2.  The launch is cooperative (all CTAs resident); every wait
// is bounded, and one that runs out ends the CTA with bit 0 of the status word.
//
// What bounds it: latency, 3 to 8 us a step (256 x 256: 4.1 against 7.1 with a
// launch per step; 16 x 2000 3.0 / 18; 100 x 1000 3.7 / 18): the exchange
// through the L2 (a release, a neighbour's acquire, its reads of the mailbox),
// about half of it, and the dependent instructions of a collision by two warps a
// scheduler.  A fence before the release, which the block barrier makes
// unnecessary, took 0.4 us of a step.
//
// The arithmetic is that of step_block in the same order, so a lattice goes
// through the same states bit for bit; both buffers hold at the end what single
// steps would have left there.
#pragma once
#include "small_step.cuh"

namespace lbm {

namespace {

// bytes of the two population buffers and the densities, rounded up to 16
__host__ __device__ constexpr size_t band_cells(int R, int P) {
    return ((size_t)19 * (R + 2) * P * sizeof(float) + 15) / 16 * 16;
}
constexpr int kMailRows = 12;  // an edge row's nine planes, a halo row's three

template <int SCH>
__global__ void __launch_bounds__(kBandThreads)
band_run_kernel(float* f0, float* f1, const __grid_constant__ KParams<float> p, int from,
                int nsteps, float* mail, unsigned* flags) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int quit;
    const int rank = blockIdx.x, C = gridDim.x, nx = p.nx, ny = p.ny;
    const int R = (ny + C - 1) / C, P = small_row<float>(nx), G = P / 2;
    const int y0 = (int)((long long)rank * ny / C), y1 = (int)((long long)(rank + 1) * ny / C);
    const int rows = y1 - y0;
    const unsigned inv = 0xFFFFFFFFu / (unsigned)G + 1u;  // it / G = umulhi(it, inv), it < 2^16
    const int plane = (R + 2) * P, bufn = 9 * plane;      // row r of the band at (r + 1) P
    float* buf = reinterpret_cast<float*>(smem);
    float* dens = buf + 2 * bufn;
    // (16 bytes before the table: what solid cells push to)
    unsigned* table = reinterpret_cast<unsigned*>(smem + band_cells(R, P)) + 4;
    uint8_t* sbits = reinterpret_cast<uint8_t*>(table + kSmallTable * R * G);
    const int tid = threadIdx.x, nt = blockDim.x;
    bool bad = false;
    if (tid == 0) quit = 0;

    // neighbours below (0) and above (1), and the mailboxes: [CTA][side][parity]
    bool hv[2];
    int nb[2];
    hv[0] = y0 > 0 || p.py;
    hv[1] = y1 < ny || p.py;
    nb[0] = rank == 0 ? C - 1 : rank - 1;
    nb[1] = rank == C - 1 ? 0 : rank + 1;
    auto box = [&](int cta, int side, int parity) {
        return mail + (((long long)cta * 2 + side) * 2 + parity) * kMailRows * P;
    };

    // the state and the rows either side: pulled from global memory once
    const float* fin = from ? f1 : f0;
    for (int c = tid; c < (rows + 2) * nx; c += nt) {
        const int r = c / nx - 1, x = c - (r + 1) * nx;
        if ((r < 0 && !hv[0]) || (r == rows && !hv[1])) continue;
        int y = y0 + r;
        y = y < 0 ? ny - 1 : y >= ny ? 0 : y;
        const unsigned sb = p.lmask ? link_bits<true>(p, x, y) : link_bits<false>(p, x, y);
        sbits[(r + 1) * P + x] = (uint8_t)sb;
        if (sb == 0xFFu) continue;
        float g[9];
        pull_l2(fin, p, x, y, sb, g, bad);
#pragma unroll
        for (int i = 0; i < 9; ++i) buf[i * plane + (r + 1) * P + x] = g[i];
    }
    if (nx < P) {
        // the inactive last column counts as solid; its populations are zero, and
        // nothing streams there
        for (int r = tid; r < rows + 2; r += nt) sbits[r * P + nx] = 0xFFu;
        for (int r = tid; r < 18 * (rows + 2); r += nt) {
            const int i = r / (rows + 2);
            buf[i * plane + (r - i * (rows + 2)) * P + nx] = 0.0f;
        }
    }
    __syncthreads();
    // where each population of each pair of cells goes (small_step.cuh)
    const int own = rows * G, items = own + 2 * G;
    const unsigned base = (unsigned)__cvta_generic_to_shared(buf);
    const unsigned dump = (unsigned)__cvta_generic_to_shared(table - 4) + 1u;
    for (int it = tid; it < own; it += nt) {
        const int r = (int)__umulhi((unsigned)it, inv), x = (it - r * G) * 2;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int xj = x + j;
            const unsigned sb = sbits[(r + 1) * P + xj];
            const int xw = xj == 0 ? nx - 1 : xj - 1, xe = xj >= nx - 1 ? 0 : xj + 1;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const int tx = ex(i) == 0 ? xj : ex(i) > 0 ? xe : xw, tr = r + ey(i);
                const bool back = i > 0 && ((sb >> (opp(i) - 1)) & 1u);  // into the cell itself
                unsigned a = sb == 0xFFu ? dump
                             : back      ? base + 4u * (unsigned)(opp(i) * plane + (r + 1) * P + xj)
                                         : base + 4u * (unsigned)(i * plane + (tr + 1) * P + tx);
                if (kChecked && !(tx >= 0 && tx < P && tr >= -1 && tr <= rows && xj < P)) {
                    bad = true;
                    a = dump;
                }
                table[it * kSmallTable + j * 9 + i] = a;
            }
        }
    }
    __syncthreads();

    for (int s = 0; s < nsteps; ++s) {
        float* cur = buf + (s & 1) * bufn;
        const int nxt = ((s & 1) ^ 1) * bufn;
        if (s > 0) {
            // the neighbours have finished step s - 1
            if ((tid & 31) == 0 && tid < 64 && hv[tid >> 5]) {
                const unsigned* flag = flags + 32 * nb[tid >> 5];
                bool there = false;
                for (unsigned k = 0; k < p.spin_limit && !there; ++k) {
                    unsigned v;
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
                    there = v >= (unsigned)s;
                }
                if (!there) quit = 1;
            }
            __syncthreads();
            if (quit) break;
        }
        // 1. densities
        for (int it = tid; it < items; it += nt) {
            int r = (int)__umulhi((unsigned)it, inv);
            const int x = (it - r * G) * 2;
            if (r >= rows) r = r == rows ? -1 : rows;  // the row below the band, the one above
            const bool south = r <= 0, north = r >= rows - 1;
            if ((r < 0 && !hv[0]) || (r == rows && !hv[1])) continue;
            float* q = cur + (r + 1) * P + x;
            float2 g[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = *reinterpret_cast<const float2*>(q + i * plane);
            if (s > 0 && (south ? hv[0] : north && hv[1])) {
                const unsigned ba = sbits[(r + 1) * P + x], bb = sbits[(r + 1) * P + x + 1];
                const float* m = box(rank, south ? 0 : 1, (s - 1) & 1) + x;
                if (r < 0 || r == rows) {
                    // the neighbour's edge row, but for what this CTA pushed there
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        const float2 v = __ldcg(reinterpret_cast<const float2*>(m + i * P));
                        const bool mine = ey(i) == (r < 0 ? -1 : 1);
                        const unsigned bit = i > 0 ? 1u << (i - 1) : 0u;
                        if (!mine || (ba & bit)) g[i].x = v.x;
                        if (!mine || (bb & bit)) g[i].y = v.y;
                    }
                } else {
                    // what the neighbour pushed into this row
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const int iS = k == 0 ? 2 : 4 + k, iN = k == 0 ? 4 : 6 + k;  // 2 5 6, 4 7 8
                        const float2 v = __ldcg(reinterpret_cast<const float2*>(m + (9 + k) * P));
                        const unsigned bit = south ? 1u << (iS - 1) : 1u << (iN - 1);
                        float2 w = south ? g[iS] : g[iN];
                        if (!(ba & bit)) w.x = v.x;
                        if (!(bb & bit)) w.y = v.y;
                        if (south) g[iS] = w;
                        else g[iN] = w;
                        *reinterpret_cast<float2*>(q + (south ? iS : iN) * plane) = w;
                    }
                }
            }
            // summed in step_block's order
            *reinterpret_cast<float2*>(dens + (r + 1) * P + x) =
                vadd(vadd(vadd(vadd(g[0], g[1]), vadd(g[2], g[3])),
                          vadd(vadd(g[4], g[5]), vadd(g[6], g[7]))),
                     g[8]);
        }
        __syncthreads();
        // 2. collide and push
        const bool last = s + 1 == nsteps, global = s + 2 >= nsteps;
        float* fout = ((from + s) & 1) ? f0 : f1;
        for (int it = tid; it < own; it += nt) {
            const int r = (int)__umulhi((unsigned)it, inv), x = (it - r * G) * 2, y = y0 + r;
            const float* q = cur + (r + 1) * P + x;
            const float* dq = dens + (r + 1) * P + x;
            float2 F[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) F[i] = *reinterpret_cast<const float2*>(q + i * plane);
            const unsigned ba = sbits[(r + 1) * P + x], bb = sbits[(r + 1) * P + x + 1];
            const float2 D = *reinterpret_cast<const float2*>(dq);
            const float2 S = *reinterpret_cast<const float2*>(dq - P), N = *reinterpret_cast<const float2*>(dq + P);
            const float w = x == 0 ? dens[(r + 1) * P + nx - 1] : dq[-1];
            const float e = x + 2 >= nx ? dens[(r + 1) * P] : dq[2];
            // (an odd width's last cell has no second one: e is its eastern neighbour)
            const float ea = x + 1 >= nx ? e : D.y;
            const float2 dW = make_float2((ba & 1u) ? D.x : w, (bb & 1u) ? D.y : D.x);
            const float2 dS = make_float2((ba & 2u) ? D.x : S.x, (bb & 2u) ? D.y : S.y);
            const float2 dE = make_float2((ba & 4u) ? D.x : ea, (bb & 4u) ? D.y : e);
            const float2 dN = make_float2((ba & 8u) ? D.x : N.x, (bb & 8u) ? D.y : N.y);
            const float2 gx = vmul(make_float2(0.5f, 0.5f), vsub(dE, dW));
            const float2 gy = vmul(make_float2(p.iah, p.iah), vsub(dN, dS));
            const float2 rho = SCH == 1 ? collide_raw<float>(to_lanes(p.cc), F, D, gx, gy)
                                        : collide<float, SCH != 3>(to_lanes(p.cc), F, D, gx, gy);
            float g[2][9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                g[0][i] = F[i].x;
                g[1][i] = F[i].y;
            }
            // a moving wall acts on the cells along it alone
            if (p.moving && (x == 0 || x + 2 >= nx || y == 0 || y == ny - 1)) {
                if (ba != 0xFFu && (x == 0 || x == nx - 1 || y == 0 || y == ny - 1))
                    moving_wall(p, x, y, rho.x, g[0]);
                if (bb != 0xFFu && (x + 1 == nx - 1 || y == 0 || y == ny - 1))
                    moving_wall(p, x + 1, y, rho.y, g[1]);
            }
            if (global) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    // (the row padding beside an odd width: as the row-band kernel
                    // leaves it, untouched with a mask, else what the collision
                    // makes of an empty cell)
                    if (x + j >= nx && p.lmask) continue;
                    const long long o = (long long)y * p.rstride + x + j;
                    if (kChecked && !(y >= 0 && y < ny && x + j < p.rstride)) {
                        bad = true;
                        continue;
                    }
#pragma unroll
                    for (int i = 0; i < 9; ++i)
                        fout[i * p.plane + o] =
                            p.lmask && (j ? bb : ba) == 0xFFu ? 0.0f : g[j][i];
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
                const unsigned off = (unsigned)nxt * 4u;
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        const unsigned t = a[j * 9 + i];
                        asm volatile("st.shared.f32 [%0], %1;" ::"r"((t & 1u) ? t - 1u : t + off),
                                     "f"(g[j][i])
                                     : "memory");
                    }
            }
        }
        if (last) break;
        __syncthreads();
        // 3. to the neighbours: below, this band's row 0 and the halo row -1's
        // planes 4 7 8; above, row rows - 1 and the halo row rows' planes 2 5 6
        for (int it = tid; it < 2 * kMailRows * G; it += nt) {
            const int k = (int)__umulhi((unsigned)it, inv), x = (it - k * G) * 2;
            const int side = k >= kMailRows ? 1 : 0, m = k - side * kMailRows;
            if (!hv[side]) continue;
            const int i = m < 9 ? m : side ? (m == 9 ? 2 : m - 5) : (m == 9 ? 4 : m - 3);
            const int r = side ? (m < 9 ? rows - 1 : rows) : (m < 9 ? 0 : -1);
            const float2 v = *reinterpret_cast<const float2*>(buf + nxt + i * plane + (r + 1) * P + x);
            __stcg(reinterpret_cast<float2*>(box(nb[side], side ^ 1, s & 1) + m * P + x), v);
        }
        __syncthreads();
        if (tid == 0) {
            // (the barrier orders the other threads' stores before this release)
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(flags + 32 * rank), "r"((unsigned)s + 1u)
                         : "memory");
        }
    }
    if (tid == 0 && quit) atomicOr(p.status, kStatusTimeout);
    if (kChecked && bad) atomicOr(p.status, kStatusBounds);
}

}  // namespace

}  // namespace lbm
