// nn.cu -- the warm-start surrogate of include/lbm_nn.h: a 3x3-convolution
// encoder-decoder trained and evaluated on the GPU.
//
// The three GEMMs of a convolution run on the fifth-generation tensor cores
// (tcgen05.mma, kind::f16: BF16 operands from shared memory, FP32
// accumulator in tensor memory) as implicit GEMMs over NHWC activations with
// channels padded to a multiple of 8:
//   forward      M = pixels, N = cout, K = 9 cin:
//                A[p][(tap, ci)] = in(p + s(tap))[ci], B[co][(tap, ci)] = W
//   input grad   M = pixels, N = cin, K = 9 cout:
//                A[q][(tap, co)] = g(q - s(tap))[co], B[ci][(tap, co)] = W
//   weight grad  M = 9 cin, N = cout, K = pixels (split over blocks, the
//                partial sums added in a fixed order), transposed so that the
//                taps and input channels fill the 128 rows of the MMA:
//                A[(tap, ci)][p] = in(p + s(tap))[ci], B[co][p] = g(p)[co]
// with s(tap) = (dy - 1, dx - 1) and zeros outside the grid.
// Forward and input gradient go over tiles of pixels (conv_tile_kernel) where the
// channels come in steps of 16 and the tile fits shared memory: a CTA of 256 threads
// copies 128 positions and their neighbours once, a tap's operand A is a start
// address in that tile, and one thread issues the MMAs of a tap as its weights land.
// The weight gradient, and the convolutions that the tiles do not take, go by
// umma_gemm_kernel: a CTA of 128 threads computes a 128 x N tile (N = 16 .. 256);
// the threads copy K chunks of 64 (cp.async) into a ring of three or four
// shared-memory stages in the tensor core's core-matrix layout, and one thread issues
// the MMAs of a chunk and commits them to the stage's mbarrier.  In both each warp
// reads its rows of the accumulator back with tcgen05.ld.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <random>
#include <vector>

#include "lbm_nn.h"
#include "dev_alloc.h"
#include "nvtx_range.h"

namespace {

using bf16 = __nv_bfloat16;

constexpr int kThreads = 256;
constexpr unsigned kBiasBlocks = 304;  // most blocks of one launch of the bias-gradient sums

// Division by a divisor fixed at launch, for dividends in [0, 2^31):
// q = (n m) >> s with m = ceil(2^s / d), s = 31 + ceil(log2 d) (exact in that
// range: the error of m / 2^s is below 2^-31 / d).
struct FastDiv {
    unsigned d = 1;
    unsigned m = 1u << 31;  // (below 2^32 for every d)
    int s = 31;
    FastDiv() = default;
    explicit FastDiv(unsigned dv) : d(dv) {
        int l = 0;
        while ((1ull << l) < dv) ++l;
        s = 31 + l;
        m = (unsigned)(((1ull << s) + dv - 1) / dv);
    }
    __device__ __forceinline__ unsigned div(unsigned n) const {
        return (unsigned)((unsigned long long)n * m >> s);
    }
};

struct Geo {
    int n, h, w;          // batch and grid
    long long P;          // pixels n h w (below 2^31: checked at creation)
    FastDiv fhw, fw;      // by h w and by w
};

Geo make_geo(int n, int h, int w, long long P) {
    Geo g;
    g.n = n;
    g.h = h;
    g.w = w;
    g.P = P;
    g.fhw = FastDiv((unsigned)(h * w));
    g.fw = FastDiv((unsigned)w);
    return g;
}

// Eight channels of one pixel (16 bytes; channel counts are padded to
// multiples of 8) at a time, with 32-bit index arithmetic: the scalar forms
// spent most of their time on 64-bit divisions.
struct Oct {
    float v[8];
};
__device__ __forceinline__ Oct load8(const bf16* p) {
    const uint4 q = *reinterpret_cast<const uint4*>(p);
    const unsigned w[4] = {q.x, q.y, q.z, q.w};
    Oct o;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        o.v[2 * k] = __uint_as_float(w[k] << 16);
        o.v[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
    }
    return o;
}
__device__ __forceinline__ void put8(bf16* p, const Oct& o) {
    unsigned w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(o.v[2 * k], o.v[2 * k + 1]);
        w[k] = *reinterpret_cast<const unsigned*>(&h);
    }
    *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}
// ---- operand tiles of the tensor-core GEMM ----
//
// A tile holds rows r (UM = 128 of A, BN of B) and the K chunk [k0, k0 + UK)
// in the tensor core's no-swizzle core-matrix layout: core matrices of
// 8 x 16 bytes stored contiguously (128 bytes), the core matrices of one
// group of 8 rows adjacent along K (leading byte offset 128) and the row
// groups 8 core matrices apart (stride byte offset 1024).  K-major: a core
// matrix row is 8 consecutive k of one row; MN-major: 8 consecutive rows at
// one k.  Every operand arrives in 16-byte pieces of one of those two kinds,
// copied by cp.async (zero-filled outside the operand).
constexpr int UM = 128, UK = 64, kGemmThreads = 128;
constexpr int kConvSmemMax = 227 * 1024;
constexpr unsigned kLBO = 128, kSBO = (UK / 8) * 128;

// byte offset of the 16-byte piece holding rows r .. r+7 at k (MN-major) or
// row r at k .. k+7 (K-major), within a tile
__device__ __forceinline__ unsigned kmajor_off(int r, int kc) {
    return (unsigned)(r >> 3) * kSBO + (unsigned)(kc >> 3) * kLBO + (unsigned)(r & 7) * 16;
}
__device__ __forceinline__ unsigned mnmajor_off(int r8, int kc) {
    return (unsigned)(r8 >> 3) * kSBO + (unsigned)(kc >> 3) * kLBO + (unsigned)(kc & 7) * 16;
}
__device__ __forceinline__ unsigned smem_addr(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
// 16 bytes global -> shared, or 16 zero bytes when !valid (any: an address
// inside the operand, for those)
__device__ __forceinline__ void cp16(unsigned dst, const bf16* src, const bf16* any, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(valid ? src : any),
                 "r"(valid ? 16 : 0)
                 : "memory");
}

// The A tile of a convolution over pixels, K-major: row r is pixel m0 + r,
// column k channel k mod c of tap k / c (TS = 1: the pixel's neighbour at the
// tap, TS = -1: its opposite).  A thread copies one 16-byte piece of eight
// rows, always the same rows and the same column of a chunk, so what depends on
// the row (whether each tap leaves the grid: nine bits) is found once, and a
// chunk costs one division and an add and a bit test per piece.  (With the
// pixel's and the tap's divisions at every piece the copies were what bounded
// the kernel: forward and input-gradient convolutions of a batch of 16 at
// 64 x 64, 32 to 256 channels, 546 and 472 us.)
template <int TS>
struct ConvRows {
    static constexpr int kRows = UM * UK / 8 / kGemmThreads;
    const bf16* in;
    const bf16* base;    // piece of row r0 at channel 0 of the centre tap
    long long stride;    // elements between the thread's rows
    unsigned mask[kRows];
    int c, w, kc;
    unsigned dst;
    FastDiv fk;
    __device__ __forceinline__ ConvRows(const Geo& g, const FastDiv& fk_, const bf16* in_, int c_,
                                        long long m0, int tid)
        : in(in_), c(c_), w(g.w), fk(fk_) {
        const int r0 = tid >> 3;
        kc = (tid & 7) * 8;
        base = in + (m0 + r0) * c;
        stride = (long long)(kGemmThreads / 8) * c;
        dst = kmajor_off(r0, kc);
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            const long long p = m0 + r0 + i * (kGemmThreads / 8);
            mask[i] = 0;
            if (p < g.P) {
                const unsigned pp = (unsigned)p, nn = g.fhw.div(pp), rem = pp - nn * g.fhw.d,
                               y = g.fw.div(rem), x = rem - y * g.fw.d;
                // taps (rows of three) that stay inside
                const unsigned row = (x > 0 ? 1u : 0u) | 2u | ((int)x < g.w - 1 ? 4u : 0u);
                mask[i] = (y > 0 ? row : 0u) | row << 3 | ((int)y < g.h - 1 ? row << 6 : 0u);
            }
        }
    }
    __device__ __forceinline__ void load(unsigned t, long long k0, long long kend) const {
        const unsigned k = (unsigned)k0 + kc;
        unsigned tap = fk.div(k);
        const int ci = (int)(k - tap * c);
        if (TS < 0) tap = 8 - tap;
        const unsigned ty = tap / 3;
        const bf16* src = base + (long long)(((int)ty - 1) * w + (int)(tap - 3 * ty) - 1) * c + ci;
        const unsigned bit = k < (unsigned)kend ? 1u << tap : 0u;
#pragma unroll
        for (int i = 0; i < kRows; ++i, src += stride)
            cp16(t + dst + i * (kGemmThreads / 64) * kSBO, src, in, (mask[i] & bit) != 0);
    }
};
// The B tile, K-major: row r is row n0 + r of a [n][kall] matrix.
template <int BN>
struct WeightRows {
    const bf16* wt;
    const bf16* base;
    long long stride;
    int left, kc;        // rows from the thread's first on
    unsigned dst;
    __device__ __forceinline__ WeightRows(const bf16* wt_, int n, long long kall, int n0, int tid)
        : wt(wt_) {
        const int r0 = tid >> 3;
        kc = (tid & 7) * 8;
        base = wt + (n0 + r0) * kall + kc;
        stride = kGemmThreads / 8 * kall;
        left = n - n0 - r0;
        dst = kmajor_off(r0, kc);
    }
    __device__ __forceinline__ void load(unsigned t, long long k0, long long kend) const {
        const bf16* src = base + k0;
        const bool in = k0 + kc < kend;
#pragma unroll
        for (int i = 0; i < BN / (kGemmThreads / 8); ++i, src += stride)
            cp16(t + dst + i * (kGemmThreads / 64) * kSBO, src, wt,
                 in && i * (kGemmThreads / 8) < left);
    }
};

// Forward: out = act(conv(in) + b).  M = pixels, N = cout, K = 9 cin:
// A[p][(tap, ci)] = in(p + s(tap))[ci], B[co][(tap, ci)] = W; both K-major.
struct FwdOp {
    static constexpr bool kAmn = false, kBmn = false;
    Geo g;
    FastDiv fk;        // by cin (the K index's channel count)
    const bf16* in;    // [P][cin]
    const bf16* wf;    // [cout][9 cin]
    const float* bias; // [cout]
    bf16* out;         // [P][cout]
    int cin, cout, relu;
    __host__ __device__ long long M() const { return g.P; }
    __host__ __device__ int N() const { return cout; }
    __host__ __device__ long long K() const { return 9LL * cin; }
    __device__ ConvRows<1> rows_a(long long m0, int tid) const {
        return ConvRows<1>(g, fk, in, cin, m0, tid);
    }
    template <int BN>
    __device__ WeightRows<BN> rows_b(int n0, int tid) const {
        return WeightRows<BN>(wf, cout, K(), n0, tid);
    }
    static constexpr int kTap = 1;  // sign of a tap's shift
    __host__ __device__ int channels() const { return cin; }
    __device__ const bf16* pixels() const { return in; }
    __device__ const bf16* weights() const { return wf; }
    // eight output channels (a multiple of 8 of them) of pixel p
    __device__ void store8(long long p, int col, const float* v) const {
        if (col >= cout) return;
        Oct o;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            o.v[j] = v[j] + bias[col + j];
            if (relu) o.v[j] = fmaxf(o.v[j], 0.0f);
        }
        put8(out + p * cout + col, o);
    }
    __device__ void store16(long long row, int col0, const float* v, int) const {
        if (row >= g.P) return;
        store8(row, col0, v);
        store8(row, col0 + 8, v + 8);
    }
};

// Input gradient: gin = conv^T(gpre).  M = pixels, N = cin, K = 9 cout:
// A[q][(tap, co)] = g(q - s(tap))[co], B[ci][(tap, co)] = W; both K-major.
struct DgradOp {
    static constexpr bool kAmn = false, kBmn = false;
    Geo g;
    FastDiv fk;        // by cout
    const bf16* gpre;  // [P][cout]
    const bf16* wd;    // [cin][9 cout]
    bf16* gin;         // [P][cin]
    int cin, cout;
    __host__ __device__ long long M() const { return g.P; }
    __host__ __device__ int N() const { return cin; }
    __host__ __device__ long long K() const { return 9LL * cout; }
    __device__ ConvRows<-1> rows_a(long long m0, int tid) const {
        return ConvRows<-1>(g, fk, gpre, cout, m0, tid);
    }
    template <int BN>
    __device__ WeightRows<BN> rows_b(int n0, int tid) const {
        return WeightRows<BN>(wd, cin, K(), n0, tid);
    }
    static constexpr int kTap = -1;
    __host__ __device__ int channels() const { return cout; }
    __device__ const bf16* pixels() const { return gpre; }
    __device__ const bf16* weights() const { return wd; }
    __device__ void store8(long long p, int col, const float* v) const {
        if (col >= cin) return;
        Oct o;
#pragma unroll
        for (int j = 0; j < 8; ++j) o.v[j] = v[j];
        put8(gin + p * cin + col, o);
    }
    __device__ void store16(long long row, int col0, const float* v, int) const {
        if (row >= g.P) return;
        store8(row, col0, v);
        store8(row, col0 + 8, v + 8);
    }
};

// The A tile of the weight gradient, MN-major: eight channels (one 16-byte
// piece) of tap m / cin at pixel k.  A thread's channels and tap are the same in
// every chunk; its eight pixels of a chunk lie eight apart.
struct PixelColumns {
    static constexpr int kPixels = UM * UK / 8 / kGemmThreads;
    const bf16* x0;
    const bf16* base;   // the channels, at the tap's neighbour of pixel 0
    const Geo& g;
    int c, dy, dx, kk;
    bool in;
    unsigned dst;
    __device__ __forceinline__ PixelColumns(const Geo& g_, const FastDiv& fk, const bf16* x, int c_,
                                            long long m0, long long M, int tid)
        : x0(x), g(g_), c(c_) {
        // consecutive threads on consecutive channel groups of one pixel
        const int grp = tid & 15;
        kk = tid >> 4;
        const long long m = m0 + grp * 8;
        in = m < M;
        const unsigned tap = fk.div((unsigned)m), ty = tap / 3;
        dy = (int)ty - 1;
        dx = (int)(tap - 3 * ty) - 1;
        base = x + (long long)(dy * g.w + dx) * c + ((int)m - (int)tap * c);
        dst = mnmajor_off(grp * 8, kk);
    }
    __device__ __forceinline__ void load(unsigned t, long long k0, long long kend) const {
#pragma unroll
        for (int i = 0; i < kPixels; ++i) {
            const long long p = k0 + kk + i * (kGemmThreads / 16);
            const unsigned pp = (unsigned)p, nn = g.fhw.div(pp), rem = pp - nn * g.fhw.d,
                           yy = g.fw.div(rem);
            const unsigned y = yy + dy, x = rem - yy * g.fw.d + dx;
            const bool ok = in && p < kend && y < (unsigned)g.h && x < (unsigned)g.w;
            cp16(t + dst + i * (kGemmThreads / 128) * kLBO, base + p * c, x0, ok);
        }
    }
};
// Its B tile, MN-major: eight channels of the output gradient at pixel k.
template <int BN>
struct GradColumns {
    static constexpr int kGroups = BN / 8, kStep = kGemmThreads / kGroups;  // threads of a pixel
    const bf16* g0;
    const bf16* base;
    int c, kk;
    bool in;
    unsigned dst;
    __device__ __forceinline__ GradColumns(const bf16* gpre, int c_, int n0, int tid)
        : g0(gpre), c(c_) {
        const int grp = tid % kGroups, co = n0 + grp * 8;
        kk = tid / kGroups;
        in = co < c;
        base = gpre + co;
        dst = mnmajor_off(grp * 8, 0);
    }
    __device__ __forceinline__ void load(unsigned t, long long k0, long long kend) const {
        static_assert(UK % kStep == 0);
#pragma unroll
        for (int i = 0; i < UK / kStep; ++i) {
            const int k = kk + i * kStep;
            const long long p = k0 + k;
            cp16(t + dst + (unsigned)(k >> 3) * kLBO + (unsigned)(k & 7) * 16, base + p * c, g0,
                 in && p < kend);
        }
    }
};

// Weight gradient, transposed so that the taps and input channels (9 cin,
// usually the larger side) fill the 128 rows: M = 9 cin, N = cout,
// K = pixels (one split of them per blockIdx.z):
// A[(tap, ci)][p] = in(p + s(tap))[ci], B[co][p] = g(p)[co], both MN-major
// (8 consecutive channels of one pixel are one 16-byte piece);
// part[z][co][(tap, ci)] = D[(tap, ci)][co].
struct WgradOp {
    static constexpr bool kAmn = true, kBmn = true;
    Geo g;
    FastDiv fk;        // by cin
    const bf16* gpre;  // [P][cout]
    const bf16* in;    // [P][cin]
    float* part;       // [splits][cout][9 cin]
    int cin, cout;
    __host__ __device__ long long M() const { return 9LL * cin; }
    __host__ __device__ int N() const { return cout; }
    __host__ __device__ long long K() const { return g.P; }
    __device__ PixelColumns rows_a(long long m0, int tid) const {
        return PixelColumns(g, fk, in, cin, m0, M(), tid);
    }
    template <int BN>
    __device__ GradColumns<BN> rows_b(int n0, int tid) const {
        return GradColumns<BN>(gpre, cout, n0, tid);
    }
    __device__ void store16(long long row, int col0, const float* v, int z) const {
        if (row >= M()) return;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int co = col0 + j;
            if (co >= cout) break;
            part[((long long)z * cout + co) * M() + row] = v[j];
        }
    }
};

// ---- the tensor-core GEMM: tcgen05.mma, accumulator in tensor memory ----

// shared memory matrix descriptor: start address, leading / stride byte
// offsets (all >> 4), version 1 at bits 46-47, no swizzle
__device__ __forceinline__ uint64_t smem_desc(unsigned addr, unsigned lbo, unsigned sbo) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}
// bounded wait on an mbarrier phase; false when it ran out
__device__ __forceinline__ bool mbar_wait_parity(unsigned bar, unsigned parity) {
    for (int it = 0; it < (1 << 22); ++it) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int BN>
__host__ __device__ constexpr int tmem_cols() { return BN <= 32 ? 32 : BN <= 64 ? 64 : BN <= 128 ? 128 : 256; }
// pipeline depth: four stages up to 64 columns, three above (two CTAs per
// SM up to 128 columns)
template <int BN>
__host__ __device__ constexpr int gemm_stages() { return BN <= 64 ? 4 : 3; }
template <int BN>
constexpr size_t umma_smem() { return (size_t)gemm_stages<BN>() * (UM + BN) * UK * 2 + 128; }

// One CTA computes a UM x BN tile of D = A B^T over its K range, in chunks of
// UK: the threads keep NS - 1 chunks in flight as cp.async groups, one
// thread issues the four MMAs (K = 16 each) of a landed chunk and commits
// them to its stage's mbarrier, which frees the stage for the chunk NS - 1
// ahead.  The accumulator lives in BN columns of tensor memory; each warp
// reads its 32 rows back.  Every wait is bounded; one that runs out sets
// *err and the tile is not stored.
template <class Op, int BN>
__global__ void __launch_bounds__(kGemmThreads) umma_gemm_kernel(const Op op, long long kchunk,
                                                                 int* err) {
    static_assert(BN % 16 == 0 && BN >= 16 && BN <= 256, "UMMA N for M = 128");
    constexpr int NS = gemm_stages<BN>();
    constexpr int TC = tmem_cols<BN>();
    constexpr unsigned kStage = (UM + BN) * UK * 2;  // A then B of one stage
    extern __shared__ __align__(1024) unsigned char sm[];
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + NS * kStage);
    unsigned* tslot = reinterpret_cast<unsigned*>(bars + NS);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long m0 = (long long)blockIdx.x * UM;
    const int n0 = blockIdx.y * BN;
    const long long kbeg = (long long)blockIdx.z * kchunk;
    const long long kend = min(op.K(), kbeg + kchunk);
    const int nkb = kend > kbeg ? (int)((kend - kbeg + UK - 1) / UK) : 0;
    const unsigned s0 = smem_addr(sm), bar0 = smem_addr(bars);
    if (tid == 0) {
        for (int s = 0; s < NS; ++s)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0 + 8u * s) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(tslot)),
                     "n"(TC)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned taddr = *tslot;
    // instruction descriptor: FP32 accumulator, BF16 A and B, their majors
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) |
                               ((Op::kAmn ? 1u : 0u) << 15) | ((Op::kBmn ? 1u : 0u) << 16) |
                               ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(UM >> 4) << 24);
    const auto rows_a = op.rows_a(m0, tid);
    const auto rows_b = op.template rows_b<BN>(n0, tid);
    auto load = [&](int kb) {
        const unsigned st = s0 + (unsigned)(kb % NS) * kStage;
        const long long k0 = kbeg + (long long)kb * UK;
        rows_a.load(st, k0, kend);
        rows_b.load(st + UM * UK * 2, k0, kend);
    };
#pragma unroll
    for (int kb = 0; kb < NS - 1; ++kb) {
        if (kb < nkb) load(kb);
        cp_commit();
    }
    bool ok = true;
    for (int kb = 0; kb < nkb; ++kb) {
        const int st = kb % NS;
        cp_wait<NS - 2>();  // this thread's pieces of chunk kb have landed
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();    // everyone's have
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const unsigned a0 = s0 + (unsigned)st * kStage, b0 = a0 + UM * UK * 2;
#pragma unroll
            for (int kk = 0; kk < UK / 16; ++kk) {
                const uint64_t ad = smem_desc(a0 + kk * 2 * kLBO, kLBO, kSBO);
                const uint64_t bd = smem_desc(b0 + kk * 2 * kLBO, kLBO, kSBO);
                const unsigned acc = (kb > 0 || kk > 0) ? 1u : 0u;
                asm volatile(
                    "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(taddr),
                    "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                    : "memory");
            }
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    bar0 + 8u * st)
                : "memory");
        }
        // the chunk NS - 1 ahead goes into the stage of chunk kb - 1, once
        // the MMAs that read it are done
        const int nk = kb + NS - 1;
        if (nk < nkb) {
            if (kb >= 1) {
                const int ps = (kb - 1) % NS;
                ok &= mbar_wait_parity(bar0 + 8u * ps, (unsigned)(((kb - 1) / NS) & 1));
            }
            load(nk);
        }
        cp_commit();
    }
    // the last commit tracks every MMA of the tile
    if (nkb > 0)
        ok &= mbar_wait_parity(bar0 + 8u * ((nkb - 1) % NS), (unsigned)(((nkb - 1) / NS) & 1));
    cp_wait<0>();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const long long row = m0 + 32 * warp + lane;
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 16) {
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
            "%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
              "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
              "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(taddr + ((unsigned)(32 * warp) << 16) + (unsigned)c0));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = nkb > 0 ? __uint_as_float(r[j]) : 0.0f;
        if (ok) op.store16(row, n0 + c0, v, (int)blockIdx.z);
    }
    if (!ok && lane == 0) atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr),
                     "n"(TC)
                     : "memory");
}

template <class Op, int BN>
cudaError_t launch_umma_bn(const Op& op, long long kchunk, int splits, int* err,
                           cudaStream_t s) {
    constexpr size_t smem = umma_smem<BN>();
    static bool configured = false;
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(umma_gemm_kernel<Op, BN>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const long long gm = (op.M() + UM - 1) / UM;
    const int gn = (op.N() + BN - 1) / BN;
    if (gm > 0x7fffffffLL) return cudaErrorInvalidValue;
    umma_gemm_kernel<Op, BN><<<dim3((unsigned)gm, gn, splits), kGemmThreads, smem, s>>>(op, kchunk,
                                                                                        err);
    return cudaGetLastError();
}

// ---- convolutions over a tile of pixels ----
//
// A 3 x 3 convolution as a GEMM reads every pixel nine times, and the copies of
// the nine shifted tiles are what bounds it.  Here a CTA copies its pixels and
// their neighbours once: the pixels of the batch are laid out as positions, one
// padding column after each row and one padding row after each image (zeros),
// so that a tap's neighbours of 128 consecutive positions are 128 consecutive
// positions too.  In shared memory eight channels of a position are 16 bytes,
// positions adjacent and channel groups a plane apart: the tensor core's
// no-swizzle K-major layout with row groups 128 bytes and K core matrices a
// plane apart, in which a tap's tile begins 16 bytes per position further.  So
// the nine taps' operands are nine start addresses in one tile.
// The CTA copies everything it needs up front (the tile and the first tap's
// weights, then the weights of each further tap, as cp.async groups) and issues
// a tap's MMAs as its weights land, in the order of the GEMM's K: taps, then
// channels in steps of 16, so the sums are the GEMM's, bit for bit.
// Planes are an odd number of 16-byte pieces apart (copies then write to
// distinct banks).
// Measured, a batch of 16 at 64 x 64, 32 to 256 channels: the 15 forward
// convolutions 546 us as GEMMs with divisions at every piece, 370 without them
// and in narrower tiles where the tiles are few, 249 here; the 14 input gradients
// 472, 342, 218.  What bounds it now is latency: a CTA's copies, nine taps and
// read-out follow one another (9 to 29 us a convolution of 1.2 GFLOP).
// (the copies are what the threads do: 256 of them take 729 us for a gradient pass
// of 4 at 32 x 32 and 271 for a prediction at 64 x 64, 128 take 758 and 282; a pass of
// 16 at 64 x 64 1,320 either way)
constexpr int kConvThreads = 256;
struct ConvTile {
    FastDiv fpitch, frows, fgroups;  // by w + 1, h + 1 and the channel groups
    unsigned positions;              // n (h + 1) (w + 1)
    int halo, pieces;                // w + 2; pieces of a plane
};
template <class Op>
ConvTile conv_tile(const Op& op) {
    ConvTile t;
    t.fpitch = FastDiv((unsigned)op.g.w + 1);
    t.frows = FastDiv((unsigned)op.g.h + 1);
    t.fgroups = FastDiv((unsigned)op.channels() / 8);
    t.positions = (unsigned)op.g.n * (op.g.h + 1) * (op.g.w + 1);
    t.halo = op.g.w + 2;
    t.pieces = (UM + 2 * t.halo) | 1;
    return t;
}
inline size_t conv_tile_smem(int pieces, int channels, int bn) {
    return (size_t)(channels / 8) * (pieces + 9 * (bn + 1)) * 16 + 16;
}

template <class Op, int BN>
__global__ void __launch_bounds__(kConvThreads) conv_tile_kernel(const Op op, const ConvTile ct,
                                                                 int* err) {
    constexpr int TC = tmem_cols<BN>();
    extern __shared__ __align__(1024) unsigned char sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int c = op.channels(), groups = c / 8;
    const unsigned m0 = blockIdx.x * UM;
    const int n0 = blockIdx.y * BN;
    const unsigned a0 = smem_addr(sm), plane = (unsigned)ct.pieces * 16;
    const unsigned b0 = a0 + groups * plane, bplane = (BN + 1) * 16;
    const unsigned bar = b0 + 9 * groups * bplane, tslot = bar + 8;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tslot),
                     "n"(TC)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // position pos: its pixel, or -1 for padding
    auto pixel = [&](unsigned pos) -> long long {
        if (pos >= ct.positions) return -1;  // (positions below 0 too)
        const unsigned row = ct.fpitch.div(pos), x = pos - row * ct.fpitch.d;
        const unsigned nn = ct.frows.div(row), y = row - nn * ct.frows.d;
        if (x == (unsigned)op.g.w || y == (unsigned)op.g.h) return -1;
        return ((long long)nn * op.g.h + y) * op.g.w + x;
    };
    {
        const bf16* in = op.pixels();
        const int total = (UM + 2 * ct.halo) * groups;
        for (int v = tid; v < total; v += kConvThreads) {
            const int px = (int)ct.fgroups.div((unsigned)v), cg = v - px * groups;
            const long long p = pixel(m0 + (unsigned)px - (unsigned)ct.halo);
            cp16(a0 + cg * plane + px * 16, in + p * c + cg * 8, in, p >= 0);
        }
    }
    const bf16* wt = op.weights();
#pragma unroll
    for (int t = 0; t < 9; ++t) {
        for (int v = tid; v < BN * groups; v += kConvThreads) {
            const int r = (int)ct.fgroups.div((unsigned)v), cg = v - r * groups;
            cp16(b0 + (t * groups + cg) * bplane + r * 16,
                 wt + (long long)(n0 + r) * 9 * c + t * c + cg * 8, wt, n0 + r < op.N());
        }
        cp_commit();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    unsigned taddr;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(taddr) : "r"(tslot) : "memory");
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                               ((uint32_t)(UM >> 4) << 24);
    auto tap = [&](int t) {  // after its cp.async group
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid != 0) return;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int shift = Op::kTap * ((t / 3 - 1) * (op.g.w + 1) + t % 3 - 1);
        const unsigned at = a0 + (unsigned)(ct.halo + shift) * 16, bt = b0 + t * groups * bplane;
        for (int k = 0; k < groups; k += 2) {
            const uint64_t ad = smem_desc(at + k * plane, plane, 128);
            const uint64_t bd = smem_desc(bt + k * bplane, bplane, 128);
            const unsigned acc = t > 0 || k > 0 ? 1u : 0u;
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(taddr),
                "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                : "memory");
        }
        if (t == 8)
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                : "memory");
    };
    cp_wait<8>(); tap(0);
    cp_wait<7>(); tap(1);
    cp_wait<6>(); tap(2);
    cp_wait<5>(); tap(3);
    cp_wait<4>(); tap(4);
    cp_wait<3>(); tap(5);
    cp_wait<2>(); tap(6);
    cp_wait<1>(); tap(7);
    cp_wait<0>(); tap(8);
    const bool ok = mbar_wait_parity(bar, 0);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // a warp reads the 32 rows of its place in its group of four, the second
    // group of warps the upper half of the columns
    constexpr int kCols = BN >= 32 ? BN / 2 : BN;
    const int quarter = warp & 3, cbeg = (warp >> 2) * kCols;
    const long long p = pixel(m0 + 32 * quarter + lane);
#pragma unroll 1
    for (int c0 = cbeg; c0 < cbeg + kCols && c0 < BN; c0 += 16) {
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
            "%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
              "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
              "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(taddr + ((unsigned)(32 * quarter) << 16) + (unsigned)c0));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
        if (ok && p >= 0) {
            op.store8(p, n0 + c0, v);
            op.store8(p, n0 + c0 + 8, v + 8);
        }
    }
    if (!ok && lane == 0) atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "n"(TC)
                     : "memory");
}

template <class Op, int BN>
cudaError_t launch_conv_bn(const Op& op, const ConvTile& t, int* err, cudaStream_t s) {
    static bool configured = false;
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(conv_tile_kernel<Op, BN>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kConvSmemMax);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const dim3 grid((t.positions + UM - 1) / UM, (op.N() + BN - 1) / BN);
    conv_tile_kernel<Op, BN>
        <<<grid, kConvThreads, conv_tile_smem(t.pieces, op.channels(), BN), s>>>(op, t, err);
    return cudaGetLastError();
}

// The tile width: the smallest UMMA N (16, 32, 64, 128, 256) that covers N,
// 256 above; narrower ones, down to 32, while the tiles are fewer than `fill`.
template <class Op>
cudaError_t launch_gemm(const Op& op, long long kchunk, int splits, int fill, int* err,
                        cudaStream_t s) {
    const int n = op.N();
    const long long gm = (op.M() + UM - 1) / UM * splits;
    int bn = n <= 16 ? 16 : n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : 256;
    while (bn > 32 && gm * ((n + bn - 1) / bn) < fill) bn /= 2;
    switch (bn) {
    case 16: return launch_umma_bn<Op, 16>(op, kchunk, splits, err, s);
    case 32: return launch_umma_bn<Op, 32>(op, kchunk, splits, err, s);
    case 64: return launch_umma_bn<Op, 64>(op, kchunk, splits, err, s);
    case 128: return launch_umma_bn<Op, 128>(op, kchunk, splits, err, s);
    default: return launch_umma_bn<Op, 256>(op, kchunk, splits, err, s);
    }
}

// A forward or input-gradient convolution: over tiles of pixels where the
// channels come in steps of 16 and a tile with its weights fits a CTA's shared
// memory (always the faster one then); else as a GEMM.  In columns that cover N,
// or fewer, down to 32, while the tiles are fewer than the SMs: of a batch of 16
// at 8 x 8 with 256 channels, eight tiles of 256 columns took 93 us, 64 of 32
// columns 33 (both as GEMMs).
template <class Op>
cudaError_t launch_conv(const Op& op, int sms, int* err, cudaStream_t s) {
    const int n = op.N(), c = op.channels();
    const ConvTile t = conv_tile(op);
    const double positions = (double)op.g.n * (op.g.h + 1) * (op.g.w + 1);
    int bn = n <= 16 ? 16 : n <= 32 ? 32 : n <= 64 ? 64 : 128;
    const long long gm = ((long long)t.positions + UM - 1) / UM;
    while (bn > 32 && (gm * ((n + bn - 1) / bn) < sms ||
                       conv_tile_smem(t.pieces, c, bn) > (size_t)kConvSmemMax))
        bn /= 2;
    if (c % 16 || positions >= 2147483648.0 ||
        conv_tile_smem(t.pieces, c, bn) > (size_t)kConvSmemMax)
        return launch_gemm(op, op.K(), 1, sms, err, s);
    switch (bn) {
    case 16: return launch_conv_bn<Op, 16>(op, t, err, s);
    case 32: return launch_conv_bn<Op, 32>(op, t, err, s);
    case 64: return launch_conv_bn<Op, 64>(op, t, err, s);
    default: return launch_conv_bn<Op, 128>(op, t, err, s);
    }
}

// ---- elementwise and reduction kernels ----

// Octet i of an (n, h, w, 8 c8) tensor: its pixel and channel group.
struct At {
    unsigned p, y, x, g;
    unsigned long long off;  // element offset
    __device__ __forceinline__ At(unsigned i, const FastDiv& c8, const FastDiv& fw,
                                  const FastDiv& fh) {
        p = c8.div(i);
        g = i - p * c8.d;
        const unsigned r = fw.div(p);
        x = p - r * fw.d;
        y = r - fh.div(r) * fh.d;
        off = 8ull * i;
    }
};

// 2x2 average: (((x00 + x10) + x01) + x11) / 4, rounded once.  total: output octets
__global__ void __launch_bounds__(kThreads)
pool_kernel(const bf16* in, bf16* out, unsigned total, FastDiv c8, FastDiv fwo, FastDiv fho) {
    const unsigned c = 8 * c8.d, row = 2 * fwo.d * c;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += gridDim.x * blockDim.x) {
        const At t(i, c8, fwo, fho);
        // output row r of (n, ho) has its input rows at 2 r, 2 r + 1 of (n, h)
        const bf16* q = in + 2ull * fwo.div(t.p) * row + 2ull * t.x * c + 8 * t.g;
        const Oct a = load8(q), b = load8(q + row), d = load8(q + c), e = load8(q + row + c);
        Oct o;
#pragma unroll
        for (int k = 0; k < 8; ++k) o.v[k] = 0.25f * (((a.v[k] + b.v[k]) + d.v[k]) + e.v[k]);
        put8(out + t.off, o);
    }
}

// gin(2y+a, 2x+b) = 0.25 g(y, x) + gin(2y+a, 2x+b) (the skip gradient already
// there).  total: octets of gin (n, h, w)
__global__ void __launch_bounds__(kThreads)
pool_back_kernel(const bf16* g, bf16* gin, unsigned total, FastDiv c8, FastDiv fw, FastDiv fh) {
    const unsigned c = 8 * c8.d;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += gridDim.x * blockDim.x) {
        const At t(i, c8, fw, fh);
        // rows come in pairs (h is even), so row r of (n, h) lies under r / 2
        const unsigned long long q =
            ((unsigned long long)(fw.div(t.p) / 2) * (fw.d / 2) + t.x / 2) * c + 8 * t.g;
        const Oct a = load8(g + q), b = load8(gin + t.off);
        Oct o;
#pragma unroll
        for (int k = 0; k < 8; ++k) o.v[k] = 0.25f * a.v[k] + b.v[k];
        put8(gin + t.off, o);
    }
}

// out (n, 2h, 2w) from in (n, h, w).  total: output octets
__global__ void __launch_bounds__(kThreads)
up_kernel(const bf16* in, bf16* out, unsigned total, FastDiv c8, FastDiv fwo, FastDiv fho) {
    const unsigned c = 8 * c8.d;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += gridDim.x * blockDim.x) {
        const At t(i, c8, fwo, fho);
        const unsigned long long q =
            ((unsigned long long)(fwo.div(t.p) / 2) * (fwo.d / 2) + t.x / 2) * c + 8 * t.g;
        *reinterpret_cast<uint4*>(out + t.off) = __ldg(reinterpret_cast<const uint4*>(in + q));
    }
}

// gin(y, x) = ((g(2y,2x) + g(2y+1,2x)) + g(2y,2x+1)) + g(2y+1,2x+1), rounded
// once.  total: octets of gin (n, h, w)
__global__ void __launch_bounds__(kThreads)
up_back_kernel(const bf16* g, bf16* gin, unsigned total, FastDiv c8, FastDiv fw, FastDiv fh) {
    const unsigned c = 8 * c8.d, row = 2 * fw.d * c;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += gridDim.x * blockDim.x) {
        const At t(i, c8, fw, fh);
        const bf16* q = g + 2ull * fw.div(t.p) * row + 2ull * t.x * c + 8 * t.g;
        const Oct a = load8(q), b = load8(q + row), d = load8(q + c), e = load8(q + row + c);
        Oct o;
#pragma unroll
        for (int k = 0; k < 8; ++k) o.v[k] = ((a.v[k] + b.v[k]) + d.v[k]) + e.v[k];
        put8(gin + t.off, o);
    }
}

__global__ void __launch_bounds__(kThreads)
add_kernel(const bf16* a, const bf16* b, bf16* out, unsigned total) {
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += gridDim.x * blockDim.x) {
        const Oct x = load8(a + 8ull * i), y = load8(b + 8ull * i);
        Oct o;
#pragma unroll
        for (int k = 0; k < 8; ++k) o.v[k] = x.v[k] + y.v[k];
        put8(out + 8ull * i, o);
    }
}

// The gradient before the ReLU, gpre = g where out > 0, else 0 (RELU; gpre may
// not alias g), and its sums over the pixels of every block: part[block][8 c8].
// A thread keeps one channel group (its octets are a multiple of c8 apart), so
// the bias gradient costs no pass of its own; the block adds its threads'
// sums in a fixed order.  blockDim.x is a multiple of c8.
template <bool RELU>
__global__ void __launch_bounds__(512)
relu_bias_kernel(const bf16* out, const bf16* g, bf16* gpre, unsigned total, int c8, float* part) {
    __shared__ float sh[512][9];
    Oct s;
#pragma unroll
    for (int k = 0; k < 8; ++k) s.v[k] = 0.0f;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += gridDim.x * blockDim.x) {
        Oct x = load8(g + 8ull * i);
        if (RELU) {
            const Oct o = load8(out + 8ull * i);
#pragma unroll
            for (int k = 0; k < 8; ++k) x.v[k] = o.v[k] > 0.0f ? x.v[k] : 0.0f;
            put8(gpre + 8ull * i, x);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) s.v[k] += x.v[k];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) sh[threadIdx.x][k] = s.v[k];
    __syncthreads();
    for (int c = threadIdx.x; c < 8 * c8; c += blockDim.x) {
        float t = 0.0f;
        for (int r = c >> 3; r < (int)blockDim.x; r += c8) t += sh[r][c & 7];
        part[(long long)blockIdx.x * 8 * c8 + c] = t;
    }
}

// host float inputs (n, h, w, 4) -> bf16 (n, h, w, 8) with zero channels 4..7
__global__ void pack_input_kernel(const float* x, bf16* out, long long pixels, int cin, int cp) {
    const long long total = pixels * cp;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int ch = (int)(i % cp);
        const long long p = i / cp;
        out[i] = __float2bfloat16_rn(ch < cin ? x[p * cin + ch] : 0.0f);
    }
}

template <typename V>
__device__ __forceinline__ V block_sum(V v) {
    __shared__ V sh[kThreads / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    V s = V(0);
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x / 32); ++i) s += sh[i];
    return s;  // valid in thread 0
}

// ---- the fixed output stage: masked smoothing and the staggered projection ----
//
// smooth:    out(p) = fl(p) sum_{dy,dx} w(dy) w(dx) fl(q) in(q), q = p + (dy, dx)
//            inside the grid, w = (1/4, 1/2, 1/4); fl from input channel 0
// unstagger: channel 1 minus its projection on (-1)^x, channel 2 minus its
//            projection on (-1)^y, over the fluid cells of each instance
// Both are self-adjoint: the backward pass applies unstagger, then smooth.

// Fluid flags: the network input's channel 0 (the solid flag) below 1/2, or
// a byte per cell (nonzero: fluid).
struct FluidIn {
    const bf16* x;
    int cp;
    __device__ __forceinline__ bool operator()(long long p) const {
        return __bfloat162float(x[p * cp]) < 0.5f;
    }
};
struct FluidBytes {
    const uint8_t* m;
    __device__ __forceinline__ bool operator()(long long p) const { return m[p] != 0; }
};

// in: bf16 [P][icp] or float [P][3]; out: float [P][3] or bf16 [P][ocp] (the
// channels past 3 zeroed)
template <bool IN_BF16, bool OUT_BF16, typename FL>
__global__ void out_smooth_kernel(const void* in, int icp, FL fluid, void* out, int ocp, int n,
                                  int h, int w) {
    const long long P = (long long)n * h * w;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P;
         p += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(p % w);
        const long long r = p / w;
        const int y = (int)(r % h);
        const long long base = r / h * h;
        float acc[3] = {0.0f, 0.0f, 0.0f};
        if (fluid(p)) {
            for (int dy = -1; dy <= 1; ++dy) {
                const int yy = y + dy;
                if (yy < 0 || yy >= h) continue;
                for (int dx = -1; dx <= 1; ++dx) {
                    const int xx = x + dx;
                    if (xx < 0 || xx >= w) continue;
                    const long long q = (base + yy) * w + xx;
                    if (!fluid(q)) continue;
                    const float wt = (dy == 0 ? 0.5f : 0.25f) * (dx == 0 ? 0.5f : 0.25f);
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const float v = IN_BF16
                                            ? __bfloat162float(static_cast<const bf16*>(in)[q * icp + c])
                                            : static_cast<const float*>(in)[q * 3 + c];
                        acc[c] = fmaf(wt, v, acc[c]);
                    }
                }
            }
        }
        if (OUT_BF16) {
            bf16* o = static_cast<bf16*>(out) + p * ocp;
            for (int c = 0; c < ocp; ++c) o[c] = __float2bfloat16_rn(c < 3 ? acc[c] : 0.0f);
        } else {
            float* o = static_cast<float*>(out) + p * 3;
#pragma unroll
            for (int c = 0; c < 3; ++c) o[c] = acc[c];
        }
    }
}

// How the cells of an instance are shared out: 2^lg threads, as many as it has cells
// and a block at most, and parts of kThreads cells, up to 16, for a block each.
// Block (k, j) takes part j of the instances whose threads fit a block, from k
// kThreads / 2^lg on.  (One block per instance took 26 us for 16 instances of
// 64 x 64; 16 parts of every instance cost a batch of 300 of 8 x 8 50 us a pass.
// Instances go along x: a batch may hold more than the 65,535 of a grid's y.)
constexpr int kStaggerParts = 16;
struct Stagger {
    int n, lg, parts;
    Stagger(int n_, long long cells) : n(n_), lg(0) {
        while ((1 << lg) < kThreads && (1 << lg) < cells) ++lg;
        const long long p = (cells + kThreads - 1) / kThreads;
        parts = p < kStaggerParts ? (int)p : kStaggerParts;
    }
    dim3 grid() const {
        const int each = kThreads >> lg;
        return dim3((unsigned)(((long long)n + each - 1) / each), parts);
    }
};
// v summed over each group of 2^lg threads, valid in its first one: over warps
// by shuffles, then in order
template <typename V>
__device__ __forceinline__ V group_sum(V v, int lg) {
    __shared__ V sh[kThreads / 32];
    const int width = lg < 5 ? 1 << lg : 32;
    for (int o = width >> 1; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, width);
    if (lg <= 5) return v;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    V s = V(0);
    if ((threadIdx.x & ((1 << lg) - 1)) == 0)
        for (int i = 0; i < 1 << (lg - 5); ++i) s += sh[(threadIdx.x >> 5) + i];
    return s;
}

// Sums over part j of the fluid cells of instance k of (-1)^x v1, (-1)^y v2 and
// the cell count, in a fixed order, to sums[k][j][3].
template <typename FL>
__global__ void __launch_bounds__(kThreads)
stagger_sum_kernel(const float* v, FL fluid, double* sums, int h, int w, const Stagger g) {
    const int lane = threadIdx.x & ((1 << g.lg) - 1);
    const int k = blockIdx.x * (kThreads >> g.lg) + (threadIdx.x >> g.lg);
    const long long hw = (long long)h * w, p0 = k * hw;
    double s1 = 0.0, s2 = 0.0, nf = 0.0;
    for (long long i = ((long long)blockIdx.y << g.lg) + lane; k < g.n && i < hw;
         i += (long long)g.parts << g.lg) {
        const long long p = p0 + i;
        if (!fluid(p)) continue;
        const unsigned y = (unsigned)i / (unsigned)w, x = (unsigned)i - y * (unsigned)w;
        s1 += (x & 1) ? -(double)v[p * 3 + 1] : (double)v[p * 3 + 1];
        s2 += (y & 1) ? -(double)v[p * 3 + 2] : (double)v[p * 3 + 2];
        nf += 1.0;
    }
    s1 = group_sum(s1, g.lg);
    s2 = group_sum(s2, g.lg);
    nf = group_sum(nf, g.lg);
    if (lane == 0 && k < g.n) {
        double* o = sums + 3 * ((long long)k * g.parts + blockIdx.y);
        o[0] = s1;
        o[1] = s2;
        o[2] = nf;
    }
}

// Applies the projection to part j of instance k.
template <typename FL>
__global__ void __launch_bounds__(kThreads)
stagger_apply_kernel(const float* v, FL fluid, const double* sums, float* out, int h, int w,
                     const Stagger g) {
    __shared__ float c[kThreads][2];
    const int lane = threadIdx.x & ((1 << g.lg) - 1), sub = threadIdx.x >> g.lg;
    const int k = blockIdx.x * (kThreads >> g.lg) + sub;
    const long long hw = (long long)h * w, p0 = k * hw;
    if (lane == 0 && k < g.n) {
        const double* q = sums + 3 * (long long)k * g.parts;
        double s1 = 0.0, s2 = 0.0, nf = 0.0;
        for (int j = 0; j < g.parts; ++j) {
            s1 += q[3 * j];
            s2 += q[3 * j + 1];
            nf += q[3 * j + 2];
        }
        // (without fluid cells nothing below uses them)
        c[sub][0] = nf > 0.0 ? (float)(s1 / nf) : 0.0f;
        c[sub][1] = nf > 0.0 ? (float)(s2 / nf) : 0.0f;
    }
    __syncthreads();
    for (long long i = ((long long)blockIdx.y << g.lg) + lane; k < g.n && i < hw;
         i += (long long)g.parts << g.lg) {
        const long long p = p0 + i;
        const unsigned y = (unsigned)i / (unsigned)w, x = (unsigned)i - y * (unsigned)w;
        float o1 = v[p * 3 + 1], o2 = v[p * 3 + 2];
        if (fluid(p)) {
            o1 -= (x & 1) ? -c[sub][0] : c[sub][0];
            o2 -= (y & 1) ? -c[sub][1] : c[sub][1];
        }
        out[p * 3] = v[p * 3];
        out[p * 3 + 1] = o1;
        out[p * 3 + 2] = o2;
    }
}

// Bilinear prolongation by an integer factor f of cell-centred fields:
// coarse [n][hc][wc][3] -> fine [n][hc f][wc f][3].  The centre of fine cell
// (Y, X) lies at coarse coordinates ((Y + 1/2) / f - 1/2, (X + 1/2) / f - 1/2),
// clamped to the coarse cell centres (constant beyond the outermost ones);
// solid fine cells get 0.
__global__ void prolong_kernel(const float* in, const uint8_t* fluid, float* out, int n, int hc,
                               int wc, int f) {
    const int H = hc * f, W = wc * f;
    const long long P = (long long)n * H * W;
    const float inv = 1.0f / (float)f;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P;
         p += (long long)gridDim.x * blockDim.x) {
        const int X = (int)(p % W);
        const long long r = p / W;
        const int Y = (int)(r % H);
        const long long k = r / H;
        float* o = out + p * 3;
        if (!fluid[p]) {
            o[0] = o[1] = o[2] = 0.0f;
            continue;
        }
        const float yc = fminf(fmaxf(((float)Y + 0.5f) * inv - 0.5f, 0.0f), (float)(hc - 1));
        const float xc = fminf(fmaxf(((float)X + 0.5f) * inv - 0.5f, 0.0f), (float)(wc - 1));
        const int y0 = (int)yc, x0 = (int)xc;
        const int y1 = min(y0 + 1, hc - 1), x1 = min(x0 + 1, wc - 1);
        const float ty = yc - (float)y0, tx = xc - (float)x0;
        const float* a = in + k * hc * wc * 3;
        const float* r0 = a + (long long)y0 * wc * 3;
        const float* r1 = a + (long long)y1 * wc * 3;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float lo = fmaf(tx, r0[x1 * 3 + c] - r0[x0 * 3 + c], r0[x0 * 3 + c]);
            const float hi = fmaf(tx, r1[x1 * 3 + c] - r1[x0 * 3 + c], r1[x0 * 3 + c]);
            o[c] = fmaf(ty, hi - lo, lo);
        }
    }
}

// Masked squared error of the network's output y (FP32 [P][3], after the
// output stage): per-block partial sums (FP64) and the output gradient
// 2 (y - t) fluid / cnt (FP32 [P][3]).
__global__ void __launch_bounds__(kThreads) loss_kernel(const float* y, const float* t,
                                                        const uint8_t* fluid, float* gy,
                                                        double* part, long long pixels,
                                                        float inv_cnt) {
    double s = 0.0;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < pixels;
         p += (long long)gridDim.x * blockDim.x) {
        const float m = fluid[p] ? 1.0f : 0.0f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float d = (y[p * 3 + c] - t[p * 3 + c]) * m;
            s += (double)d * (double)d;
            gy[p * 3 + c] = 2.0f * d * inv_cnt;
        }
    }
    const double b = block_sum(s);
    if (threadIdx.x == 0) part[blockIdx.x] = b;
}

__global__ void __launch_bounds__(kThreads) sum_kernel(const double* part, int n, double* out) {
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += part[i];
    const double b = block_sum(s);
    if (threadIdx.x == 0) *out = b;
}

// dW = sum over the splits, and gb = sum over the bias partials, in a fixed
// order: a block takes 32 values, each by eight threads whose sums (terms z =
// k, k + 8, ...) are added in order.  (One thread a value was a chain of 100 to
// 300 dependent rounds: 25 us a convolution on average.)
__global__ void __launch_bounds__(kThreads)
split_sum_kernel(const float* part, float* gw, int splits, long long n, const float* bpart,
                 float* gb, int bparts, int cout) {
    __shared__ float sh[8][33];
    const int x = threadIdx.x & 31, k = threadIdx.x >> 5;
    // blocks of weights, then blocks of biases
    const long long wblocks = (n + 31) / 32, blocks = wblocks + (cout + 31) / 32;
    for (long long b = blockIdx.x; b < blocks; b += gridDim.x) {
        const bool w = b < wblocks;
        const long long i = (w ? b : b - wblocks) * 32 + x, size = w ? n : cout;
        const int terms = w ? splits : bparts;
        float s = 0.0f;
        if (i < size) {
            const float* q = (w ? part : bpart) + i;
#pragma unroll 8
            for (int z = k; z < terms; z += 8) s += q[z * size];
        }
        sh[k][x] = s;
        __syncthreads();
        if (k == 0 && i < size) {
#pragma unroll
            for (int j = 1; j < 8; ++j) s += sh[j][x];
            (w ? gw : gb)[i] = s;
        }
        __syncthreads();
    }
}

// Adam on FP32 masters; counts t from 1.
__global__ void adam_kernel(float* p, const float* g, float* m, float* v, long long n,
                            float lr, float b1, float b2, float c1, float c2, float eps) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// BF16 copies of the weights: wf[co][tap][ci] and wd[ci][tap][co] from the
// master wm[co][tap][ci]
__global__ void weight_copies_kernel(const float* wm, bf16* wf, bf16* wd, int cin, int cout) {
    const long long n = 9LL * cin * cout;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int ci = (int)(i % cin);
        const long long r = i / cin;
        const int tap = (int)(r % 9);
        const int co = (int)(r / 9);
        const bf16 v = __float2bfloat16_rn(wm[i]);
        wf[i] = v;
        wd[((long long)ci * 9 + tap) * cout + co] = v;
    }
}

// The host's parameter order (dy, dx, cin, cout, then the biases) from or to the
// convolutions' device arrays w [coutp][9][cinp], b [coutp].  A block moves a
// tile of 32 input by 32 output channels of one tap through shared memory, so
// that both sides are read and written in rows; all convolutions in one launch
// (one launch each took 75 us more of a gradient pass of 16 at 64 x 64, now 1,250).
constexpr int kMaxConvs = 23;  // of six levels
struct ParamTable {
    struct Entry {
        float *w, *b;
        long long at;               // in the host's order
        int cin, cout, cinp, first; // first: its first block
    } e[kMaxConvs];
    int n;
};
template <bool TO_HOST>
__global__ void __launch_bounds__(kThreads)
param_order_kernel(float* vec, const __grid_constant__ ParamTable table) {
    __shared__ float t[32][33];
    int k = 0;
    while (k + 1 < table.n && table.e[k + 1].first <= (int)blockIdx.x) ++k;
    const ParamTable::Entry& c = table.e[k];
    float* const host = vec + c.at;
    float *const w = c.w, *const b = c.b;
    const int cin = c.cin, cout = c.cout, cinp = c.cinp;
    const int tx = (cout + 31) / 32, ty = (cin + 31) / 32, local = (int)blockIdx.x - c.first;
    const int tap = local / (tx * ty), ci0 = local / tx % ty * 32, co0 = local % tx * 32;
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    for (int r = y; r < 32; r += kThreads / 32) {
        if (TO_HOST) {  // rows of the device array: ci across
            const int co = co0 + r, ci = ci0 + x;
            if (co < cout && ci < cin) t[r][x] = w[((long long)co * 9 + tap) * cinp + ci];
        } else {        // rows of the host array: co across
            const int ci = ci0 + r, co = co0 + x;
            if (co < cout && ci < cin) t[x][r] = host[((long long)tap * cin + ci) * cout + co];
        }
    }
    __syncthreads();
    for (int r = y; r < 32; r += kThreads / 32) {
        if (TO_HOST) {
            const int ci = ci0 + r, co = co0 + x;
            if (co < cout && ci < cin) host[((long long)tap * cin + ci) * cout + co] = t[x][r];
        } else {
            const int co = co0 + r, ci = ci0 + x;
            if (co < cout && ci < cin) w[((long long)co * 9 + tap) * cinp + ci] = t[r][x];
        }
    }
    if (tap == 0 && ci0 == 0)
        for (int i = threadIdx.x; i < 32 && co0 + i < cout; i += kThreads) {
            float* hb = host + 9ll * cin * cout + co0 + i;
            if (TO_HOST) *hb = b[co0 + i];
            else b[co0 + i] = *hb;
        }
}

int grid_of(long long n) {
    long long b = (n + kThreads - 1) / kThreads;
    return (int)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

}  // namespace

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------

struct lbm_nn {
    struct Tensor {
        int h, w, c, cp;   // grid, logical and padded channels
        bf16* v = nullptr; // activation
        bf16* g = nullptr; // its gradient
    };
    struct Conv {
        int in, out, relu;
        int cin, cout, cinp, coutp;
        float *wm, *bm, *gw, *gb, *mw, *vw, *mb, *vb;  // [coutp][9][cinp], [coutp]
        bf16 *wf, *wd;
    };
    enum Kind { CONV, POOL, UP, ADD };
    struct Op {
        Kind k;
        int a, b, out;  // tensor ids (CONV: conv index in a)
    };
    int L = 0, nb = 0, H = 0, W = 0;
    std::vector<int> ch;
    std::vector<Tensor> t;
    std::vector<Conv> conv;
    std::vector<Op> ops;
    int x_id = 0, y_id = 0;
    cudaStream_t stream = nullptr;
    float* pbuf = nullptr;     // all FP32 parameter-sized arrays
    size_t pfloats = 0;
    bf16* wbuf = nullptr;      // BF16 weight copies
    unsigned char* abuf = nullptr;  // activations and gradients
    bf16* scratch[2] = {nullptr, nullptr};  // relu-masked gradients, in turn
    float* part = nullptr;     // weight-gradient split partials
    float* bpart[2] = {nullptr, nullptr};  // bias-gradient partials [runs kBiasBlocks][coutp], in turn
    // Parameter gradients run beside the chain of input gradients (backward())
    cudaStream_t side = nullptr;
    cudaEvent_t ready = nullptr, done[2] = {nullptr, nullptr};
    float* flat = nullptr;     // a parameter vector in the host's order
    int sms = 1;
    long long nfluid = 0;      // fluid cells of the batch at hand
    double* dpart = nullptr;   // loss partials (+1 for the total)
    float* xin = nullptr;      // staging of host inputs (float)
    float* tgt = nullptr;
    uint8_t* fl = nullptr;
    float* yout = nullptr;     // the network's output after the output stage [P][3]
    float* gout = nullptr;     // the loss gradient of yout [P][3]
    float* tmp3 = nullptr;     // the output stage's intermediate [P][3]
    double* ssum = nullptr;    // per instance and part: the staggered sums and fluid count
    float* fine = nullptr;     // lbm_nn_prolong: two fine fields [max_batch][H f][W f][3]
    uint8_t* fine_fl = nullptr;  // and their fluid flags
    long long fine_cells = 0;  // cells per fine field the buffers hold
    int* gemm_err = nullptr;   // set by a GEMM whose bounded wait ran out
    long long adam_t = 0;
    int64_t launches = 0;
    char err[512] = {0};
};

namespace {

thread_local char g_nn_err[512] = "no error";

void nn_err(lbm_nn* nn, const char* fmt, ...) {
    char* dst = nn ? nn->err : g_nn_err;
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(dst, 512, fmt, ap);
    va_end(ap);
}

#define NCK(nn, call, what)                                                    \
    do {                                                                       \
        cudaError_t e_ = (call);                                               \
        if (e_ != cudaSuccess) {                                               \
            nn_err(nn, "%s: %s", what, cudaGetErrorString(e_));                \
            return e_ == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA; \
        }                                                                      \
    } while (0)

int pad8(int c) { return (c + 7) / 8 * 8; }

long long pixels(const lbm_nn* nn, int id, int n) {
    return (long long)n * nn->t[id].h * nn->t[id].w;
}

// f(first instance, octets) over the batch in runs of instances whose tensor
// `id` has fewer than 2^31 groups of eight channels (one run but for the very
// largest batches; an instance has at most 2^30).
template <class F>
cudaError_t by_octets(const lbm_nn* nn, int id, int n, const F& f) {
    const long long one = (long long)nn->t[id].h * nn->t[id].w * (nn->t[id].cp / 8);
    const int most = (int)(((1LL << 31) - 1) / one);
    for (int i = 0; i < n; i += most) {
        const int m = n - i < most ? n - i : most;
        f(i, (unsigned)(m * one));
        if (cudaError_t e = cudaGetLastError(); e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
// the address of instance i of an activation or gradient of tensor `id`
const bf16* instance(const lbm_nn* nn, int id, const bf16* v, int i) {
    return v + (long long)i * nn->t[id].h * nn->t[id].w * nn->t[id].cp;
}
bf16* instance(const lbm_nn* nn, int id, bf16* v, int i) {
    return v + (long long)i * nn->t[id].h * nn->t[id].w * nn->t[id].cp;
}

int add_tensor(lbm_nn* nn, int h, int w, int c) {
    lbm_nn::Tensor T;
    T.h = h;
    T.w = w;
    T.c = c;
    T.cp = pad8(c);
    nn->t.push_back(T);
    return (int)nn->t.size() - 1;
}

int add_conv(lbm_nn* nn, int in, int cout, int relu) {
    const lbm_nn::Tensor X = nn->t[in];  // a copy: add_tensor grows nn->t
    const int out = add_tensor(nn, X.h, X.w, cout);
    lbm_nn::Conv c{};
    c.in = in;
    c.out = out;
    c.relu = relu;
    c.cin = X.c;
    c.cout = cout;
    c.cinp = X.cp;
    c.coutp = pad8(cout);
    nn->conv.push_back(c);
    nn->ops.push_back({lbm_nn::CONV, (int)nn->conv.size() - 1, 0, out});
    return out;
}

// Builds the network graph (see include/lbm_nn.h).
void build_graph(lbm_nn* nn) {
    nn->x_id = add_tensor(nn, nn->H, nn->W, 4);
    int x = nn->x_id;
    std::vector<int> e(nn->L);
    int h = nn->H, w = nn->W;
    for (int l = 0; l < nn->L; ++l) {
        x = add_conv(nn, x, nn->ch[l], 1);
        x = add_conv(nn, x, nn->ch[l], 1);
        e[l] = x;
        if (l < nn->L - 1) {
            h /= 2;
            w /= 2;
            const int p = add_tensor(nn, h, w, nn->ch[l]);
            nn->ops.push_back({lbm_nn::POOL, x, 0, p});
            x = p;
        }
    }
    for (int l = nn->L - 2; l >= 0; --l) {
        h *= 2;
        w *= 2;
        const int u = add_tensor(nn, h, w, nn->ch[l + 1]);
        nn->ops.push_back({lbm_nn::UP, x, 0, u});
        const int c = add_conv(nn, u, nn->ch[l], 1);
        const int s = add_tensor(nn, h, w, nn->ch[l]);
        nn->ops.push_back({lbm_nn::ADD, c, e[l], s});
        x = add_conv(nn, s, nn->ch[l], 1);
    }
    nn->y_id = add_conv(nn, x, 3, 0);
}

size_t conv_wsize(const lbm_nn::Conv& c) { return 9ull * c.cinp * c.coutp; }

lbm_status sync_weights(lbm_nn* nn) {
    for (auto& c : nn->conv) {
        weight_copies_kernel<<<grid_of((long long)conv_wsize(c)), kThreads, 0, nn->stream>>>(
            c.wm, c.wf, c.wd, c.cinp, c.coutp);
        NCK(nn, cudaGetLastError(), "weight copies");
        ++nn->launches;
    }
    return LBM_OK;
}

lbm_status upload_inputs(lbm_nn* nn, const float* x, const float* tgt, const uint8_t* fluid,
                         int n) {
    const long long P = (long long)n * nn->H * nn->W;
    NCK(nn, cudaMemcpyAsync(nn->xin, x, P * 4 * sizeof(float), cudaMemcpyHostToDevice, nn->stream),
        "cudaMemcpyAsync(H2D)");
    if (tgt)
        NCK(nn, cudaMemcpyAsync(nn->tgt, tgt, P * 3 * sizeof(float), cudaMemcpyHostToDevice,
                                nn->stream),
            "cudaMemcpyAsync(H2D)");
    if (fluid)
        NCK(nn, cudaMemcpyAsync(nn->fl, fluid, P, cudaMemcpyHostToDevice, nn->stream),
            "cudaMemcpyAsync(H2D)");
    const lbm_nn::Tensor& X = nn->t[nn->x_id];
    pack_input_kernel<<<grid_of(P * X.cp), kThreads, 0, nn->stream>>>(nn->xin, X.v, P, 4, X.cp);
    NCK(nn, cudaGetLastError(), "input packing");
    ++nn->launches;
    if (fluid) {
        nn->nfluid = 0;
        for (long long i = 0; i < P; ++i) nn->nfluid += fluid[i] != 0;
    }
    return LBM_OK;
}

// Splits of a weight gradient's pixels over CTAs, and pixels per split: two
// CTAs per SM, with at least 256 pixels each.  (Splits of 4096 pixels left most
// SMs idle: 94 us a convolution of 16 x 64 x 64 pixels on average.)
void wgrad_splits(const lbm_nn* nn, const lbm_nn::Conv& c, long long P, int& splits,
                  long long& kchunk) {
    const long long tiles = ((9LL * c.cinp + UM - 1) / UM) * ((c.coutp + 255) / 256);
    long long s = (2LL * nn->sms + tiles - 1) / tiles;
    if (s > (P + 255) / 256) s = (P + 255) / 256;
    kchunk = ((P + s - 1) / s + UK - 1) / UK * UK;
    splits = (int)((P + kchunk - 1) / kchunk);
}

// out = the staggered projection of v (FP32 [P][3] each), per instance.
lbm_status unstagger(lbm_nn* nn, int n, const float* v, float* out) {
    const lbm_nn::Tensor& X = nn->t[nn->x_id];
    const FluidIn fl{X.v, X.cp};
    const Stagger g(n, (long long)X.h * X.w);
    stagger_sum_kernel<<<g.grid(), kThreads, 0, nn->stream>>>(v, fl, nn->ssum, X.h, X.w, g);
    NCK(nn, cudaGetLastError(), "staggered sums");
    stagger_apply_kernel<<<g.grid(), kThreads, 0, nn->stream>>>(v, fl, nn->ssum, out, X.h, X.w, g);
    NCK(nn, cudaGetLastError(), "staggered projection");
    nn->launches += 3;  // with the smoothing launched beside it
    return LBM_OK;
}

lbm_status forward(lbm_nn* nn, int n) {
    const cudaStream_t s = nn->stream;
    for (const auto& op : nn->ops) {
        cudaError_t e = cudaSuccess;
        if (op.k == lbm_nn::CONV) {
            const lbm_nn::Conv& c = nn->conv[op.a];
            const lbm_nn::Tensor& X = nn->t[c.in];
            FwdOp f;
            f.g = make_geo(n, X.h, X.w, pixels(nn, c.in, n));
            f.fk = FastDiv((unsigned)c.cinp);
            f.in = X.v;
            f.wf = c.wf;
            f.bias = c.bm;
            f.out = nn->t[c.out].v;
            f.cin = c.cinp;
            f.cout = c.coutp;
            f.relu = c.relu;
            e = launch_conv(f, nn->sms, nn->gemm_err, s);
        } else if (op.k == lbm_nn::POOL) {
            const lbm_nn::Tensor& X = nn->t[op.a];
            const lbm_nn::Tensor& O = nn->t[op.out];
            e = by_octets(nn, op.out, n, [&](int i, unsigned t) {
                pool_kernel<<<grid_of(t), kThreads, 0, s>>>(
                    instance(nn, op.a, X.v, i), instance(nn, op.out, O.v, i), t, FastDiv(X.cp / 8),
                    FastDiv(O.w), FastDiv(O.h));
            });
        } else if (op.k == lbm_nn::UP) {
            const lbm_nn::Tensor& X = nn->t[op.a];
            const lbm_nn::Tensor& O = nn->t[op.out];
            e = by_octets(nn, op.out, n, [&](int i, unsigned t) {
                up_kernel<<<grid_of(t), kThreads, 0, s>>>(
                    instance(nn, op.a, X.v, i), instance(nn, op.out, O.v, i), t, FastDiv(X.cp / 8),
                    FastDiv(O.w), FastDiv(O.h));
            });
        } else {
            e = by_octets(nn, op.out, n, [&](int i, unsigned t) {
                add_kernel<<<grid_of(t), kThreads, 0, s>>>(
                    instance(nn, op.a, nn->t[op.a].v, i), instance(nn, op.b, nn->t[op.b].v, i),
                    instance(nn, op.out, nn->t[op.out].v, i), t);
            });
        }
        NCK(nn, e, "forward kernels");
        ++nn->launches;
    }
    // the fixed output stage: yout = unstagger(smooth(y))
    const lbm_nn::Tensor& X = nn->t[nn->x_id];
    const lbm_nn::Tensor& Y = nn->t[nn->y_id];
    const long long P = pixels(nn, nn->y_id, n);
    out_smooth_kernel<true, false><<<grid_of(P), kThreads, 0, s>>>(
        Y.v, Y.cp, FluidIn{X.v, X.cp}, nn->tmp3, 3, n, Y.h, Y.w);
    NCK(nn, cudaGetLastError(), "output smoothing");
    return unstagger(nn, n, nn->tmp3, nn->yout);
}

// Loss of the batch (synchronous) and, through the backward pass, the
// gradients of every convolution's parameters (c.gw, c.gb).
lbm_status backward(lbm_nn* nn, int n, float* loss) {
    const cudaStream_t s = nn->stream;
    const long long P = (long long)n * nn->H * nn->W;
    const long long nf = nn->nfluid;
    const float inv_cnt = nf > 0 ? (float)(1.0 / (3.0 * (double)nf)) : 0.0f;
    std::vector<bf16*> G(nn->t.size());
    for (size_t i = 0; i < nn->t.size(); ++i) G[i] = nn->t[i].g;
    const lbm_nn::Tensor& X = nn->t[nn->x_id];
    const lbm_nn::Tensor& Y = nn->t[nn->y_id];
    const int lb = grid_of(P) < 1024 ? grid_of(P) : 1024;
    loss_kernel<<<lb, kThreads, 0, s>>>(nn->yout, nn->tgt, nn->fl, nn->gout, nn->dpart, P,
                                        inv_cnt);
    NCK(nn, cudaGetLastError(), "loss kernel");
    sum_kernel<<<1, kThreads, 0, s>>>(nn->dpart, lb, nn->dpart + 1024);
    NCK(nn, cudaGetLastError(), "loss sum");
    nn->launches += 2;
    // the output stage backward: unstagger, then smooth into the gradient of
    // the last convolution's output (BF16, padded channels zeroed)
    if (lbm_status st = unstagger(nn, n, nn->gout, nn->tmp3); st != LBM_OK) return st;
    out_smooth_kernel<false, true><<<grid_of(P), kThreads, 0, s>>>(nn->tmp3, 3, FluidIn{X.v, X.cp},
                                                                   G[nn->y_id], Y.cp, n, Y.h, Y.w);
    NCK(nn, cudaGetLastError(), "output smoothing (backward)");
    // The chain of the pass (ReLU and bias partials, input gradient) stays on the
    // stream; a convolution's weight and bias gradients, which nothing in the
    // pass waits for, run beside it on a stream of lower priority: neither fills
    // the GPU (a dozen to 300 CTAs, latency-bound).  They read the masked gradient
    // and the partials from two buffers in turn; the stream waits for them before
    // a buffer is written again, and for the last at the end.  A gradient pass of
    // 16 at 64 x 64, 32 to 256 channels: 1.56 -> 1.34 ms; of 4 at 32 x 32 931 ->
    // 759 us.
    int turn = 0;
    cudaError_t e = cudaSuccess;
    for (int i = (int)nn->ops.size() - 1; i >= 0 && e == cudaSuccess; --i) {
        const lbm_nn::Op& op = nn->ops[i];
        if (op.k == lbm_nn::CONV) {
            const lbm_nn::Conv& c = nn->conv[op.a];
            const lbm_nn::Tensor& X = nn->t[c.in];
            const lbm_nn::Tensor& O = nn->t[c.out];
            const long long Pc = pixels(nn, c.in, n);
            const int buf = turn & 1;
            bf16* const scratch = nn->scratch[buf];
            float* const bpart = nn->bpart[buf];
            const bf16* gpre = c.relu ? scratch : G[c.out];
            if (turn >= 2 && (e = cudaStreamWaitEvent(s, nn->done[buf], 0)) != cudaSuccess) break;
            ++turn;
            // the gradient before the ReLU and the bias partials
            const int c8 = O.cp / 8, bt = 512 / c8 * c8;
            int bb = 0;  // partials so far
            e = by_octets(nn, c.out, n, [&](int i, unsigned t) {
                const unsigned want = (t + bt - 1) / bt;
                const int blocks = (int)(want < kBiasBlocks ? want : kBiasBlocks);
                float* part = bpart + (long long)bb * 8 * c8;
                const bf16* o = instance(nn, c.out, O.v, i);
                const bf16* g = instance(nn, c.out, (const bf16*)G[c.out], i);
                if (c.relu)
                    relu_bias_kernel<true><<<blocks, bt, 0, s>>>(
                        o, g, instance(nn, c.out, scratch, i), t, c8, part);
                else
                    relu_bias_kernel<false><<<blocks, bt, 0, s>>>(o, g, nullptr, t, c8, part);
                bb += blocks;
            });
            if (e != cudaSuccess) break;
            if ((e = cudaEventRecord(nn->ready, s)) != cudaSuccess) break;
            WgradOp wg;
            wg.g = make_geo(n, X.h, X.w, Pc);
            wg.fk = FastDiv((unsigned)c.cinp);
            wg.gpre = gpre;
            wg.in = X.v;
            wg.part = nn->part;
            wg.cin = c.cinp;
            wg.cout = c.coutp;
            if (c.in != nn->x_id) {
                DgradOp dg;
                dg.g = wg.g;
                dg.fk = FastDiv((unsigned)c.coutp);
                dg.gpre = gpre;
                dg.wd = c.wd;
                dg.gin = G[c.in];
                dg.cin = c.cinp;
                dg.cout = c.coutp;
                if ((e = launch_conv(dg, nn->sms, nn->gemm_err, s)) != cudaSuccess) break;
                ++nn->launches;
            }
            // weight gradient, split over pixels
            int splits;
            long long kchunk;
            wgrad_splits(nn, c, Pc, splits, kchunk);
            if ((e = cudaStreamWaitEvent(nn->side, nn->ready, 0)) != cudaSuccess) break;
            if ((e = launch_gemm(wg, kchunk, splits, 0, nn->gemm_err, nn->side)) != cudaSuccess) break;
            const long long nw = (long long)conv_wsize(c);
            split_sum_kernel<<<grid_of((nw + c.coutp + 64) * 8), kThreads, 0, nn->side>>>(
                nn->part, c.gw, splits, nw, bpart, c.gb, bb, c.coutp);
            if ((e = cudaGetLastError()) != cudaSuccess) break;
            if ((e = cudaEventRecord(nn->done[buf], nn->side)) != cudaSuccess) break;
            nn->launches += 3;
        } else if (op.k == lbm_nn::POOL) {
            const lbm_nn::Tensor& X = nn->t[op.a];
            // the skip addition of the decoder has set the gradient of op.a
            e = by_octets(nn, op.a, n, [&](int i, unsigned t) {
                pool_back_kernel<<<grid_of(t), kThreads, 0, s>>>(
                    instance(nn, op.out, G[op.out], i), instance(nn, op.a, G[op.a], i), t,
                    FastDiv(X.cp / 8), FastDiv(X.w), FastDiv(X.h));
            });
            ++nn->launches;
        } else if (op.k == lbm_nn::UP) {
            const lbm_nn::Tensor& X = nn->t[op.a];
            e = by_octets(nn, op.a, n, [&](int i, unsigned t) {
                up_back_kernel<<<grid_of(t), kThreads, 0, s>>>(
                    instance(nn, op.out, G[op.out], i), instance(nn, op.a, G[op.a], i), t,
                    FastDiv(X.cp / 8), FastDiv(X.w), FastDiv(X.h));
            });
            ++nn->launches;
        } else {
            // an addition passes its gradient to both inputs
            G[op.a] = G[op.out];
            G[op.b] = G[op.out];
        }
    }
    // join (after a failure too: the side stream may hold work of this pass)
    const cudaError_t joined = cudaEventRecord(nn->ready, nn->side);
    if (e == cudaSuccess) e = joined;
    if (joined == cudaSuccess) {
        const cudaError_t w = cudaStreamWaitEvent(s, nn->ready, 0);
        if (e == cudaSuccess) e = w;
    }
    if (e != cudaSuccess) {
        nn_err(nn, "backward kernels: %s", cudaGetErrorString(e));
        return LBM_ERR_CUDA;
    }
    double l = 0.0;
    NCK(nn, cudaMemcpyAsync(&l, nn->dpart + 1024, sizeof(double), cudaMemcpyDeviceToHost, s),
        "cudaMemcpyAsync(D2H)");
    NCK(nn, cudaStreamSynchronize(s), "cudaStreamSynchronize");
    if (loss) *loss = (float)(l * (double)inv_cnt);
    return LBM_OK;
}

// After a synchronisation: a GEMM whose bounded wait ran out leaves its word
// set (its tile was not stored).
lbm_status check_gemm(lbm_nn* nn) {
    int e = 0;
    NCK(nn, cudaMemcpy(&e, nn->gemm_err, sizeof(int), cudaMemcpyDeviceToHost), "cudaMemcpy(D2H)");
    if (e) {
        NCK(nn, cudaMemset(nn->gemm_err, 0, sizeof(int)), "cudaMemset");
        nn_err(nn, "a tensor-core GEMM gave up waiting for its MMAs");
        return LBM_ERR_TIMEOUT;
    }
    return LBM_OK;
}

bool bad_batch(lbm_nn* nn, int n) {
    if (n < 1 || n > nn->nb) {
        nn_err(nn, "batch size %d outside [1, %d]", n, nn->nb);
        return true;
    }
    return false;
}

}  // namespace

extern "C" {

lbm_status lbm_nn_create(int levels, const int* channels, int max_batch, int height, int width,
                         uint64_t seed, void* cuda_stream, lbm_nn** out) {
    LBM_RANGE("lbm_nn_create");
    if (!out) {
        nn_err(nullptr, "out is NULL");
        return LBM_ERR_INVALID;
    }
    *out = nullptr;
    if (levels < 1 || levels > 6 || !channels || max_batch < 1 || height < 1 || width < 1 ||
        height > 4096 || width > 4096 || height % (1 << (levels - 1)) ||
        width % (1 << (levels - 1))) {
        nn_err(nullptr, "invalid network shape (levels 1..6, height and width multiples of "
                        "2^(levels-1), at most 4096)");
        return LBM_ERR_INVALID;
    }
    for (int l = 0; l < levels; ++l)
        if (channels[l] < 1 || channels[l] > 512) {
            nn_err(nullptr, "channels must lie in [1, 512]");
            return LBM_ERR_INVALID;
        }
    if ((double)max_batch * height * width > 1.0e8) {
        nn_err(nullptr, "batch of more than 1e8 cells");
        return LBM_ERR_INVALID;
    }
    lbm_nn* nn = new (std::nothrow) lbm_nn();
    if (!nn) {
        nn_err(nullptr, "host allocation failed");
        return LBM_ERR_OOM;
    }
    nn->L = levels;
    nn->ch.assign(channels, channels + levels);
    nn->nb = max_batch;
    nn->H = height;
    nn->W = width;
    nn->stream = (cudaStream_t)cuda_stream;
    build_graph(nn);
    auto fail = [&](lbm_status s) {
        std::snprintf(g_nn_err, sizeof(g_nn_err), "%s", nn->err);
        lbm_nn_destroy(nn);
        return s;
    };
#define NCKC(call, what)                                                        \
    do {                                                                        \
        cudaError_t e_ = (call);                                                \
        if (e_ != cudaSuccess) {                                                \
            nn_err(nn, "%s: %s", what, cudaGetErrorString(e_));                 \
            return fail(e_ == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA); \
        }                                                                       \
    } while (0)
    // parameters: 8 FP32 arrays per convolution (w, b, gw, gb, mw, vw, mb, vb)
    size_t pf = 0, wb = 0;
    for (auto& c : nn->conv) {
        pf += 4 * (conv_wsize(c) + c.coutp);
        wb += 2 * conv_wsize(c);
    }
    nn->pfloats = pf;
    NCKC(lbm::dev_alloc(&nn->pbuf, pf * sizeof(float)), "cudaMalloc(parameters)");
    NCKC(cudaMemsetAsync(nn->pbuf, 0, pf * sizeof(float), nn->stream), "cudaMemset");
    NCKC(lbm::dev_alloc(&nn->wbuf, wb * sizeof(bf16)), "cudaMalloc(weights)");
    {
        float* q = nn->pbuf;
        bf16* r = nn->wbuf;
        for (auto& c : nn->conv) {
            const size_t w = conv_wsize(c), b = c.coutp;
            c.wm = q; q += w;
            c.gw = q; q += w;
            c.mw = q; q += w;
            c.vw = q; q += w;
            c.bm = q; q += b;
            c.gb = q; q += b;
            c.mb = q; q += b;
            c.vb = q; q += b;
            c.wf = r; r += w;
            c.wd = r; r += w;
        }
    }
    // activations and their gradients, 256-byte aligned parts
    size_t ab = 0, maxt = 0;
    for (auto& T : nn->t) {
        const size_t e = (size_t)nn->nb * T.h * T.w * T.cp;
        ab += 2 * ((e * sizeof(bf16) + 255) / 256 * 256);
        maxt = e > maxt ? e : maxt;
    }
    NCKC(lbm::dev_alloc(&nn->abuf, ab), "cudaMalloc(activations)");
    NCKC(cudaMemsetAsync(nn->abuf, 0, ab, nn->stream), "cudaMemset");
    {
        unsigned char* q = nn->abuf;
        for (auto& T : nn->t) {
            const size_t e = ((size_t)nn->nb * T.h * T.w * T.cp * sizeof(bf16) + 255) / 256 * 256;
            T.v = reinterpret_cast<bf16*>(q);
            q += e;
            T.g = reinterpret_cast<bf16*>(q);
            q += e;
        }
    }
    for (auto& b : nn->scratch) NCKC(lbm::dev_alloc(&b, maxt * sizeof(bf16)), "cudaMalloc(scratch)");
    int least = 0, greatest = 0;
    NCKC(cudaDeviceGetStreamPriorityRange(&least, &greatest), "cudaDeviceGetStreamPriorityRange");
    NCKC(cudaStreamCreateWithPriority(&nn->side, cudaStreamNonBlocking, least), "cudaStreamCreate");
    for (cudaEvent_t* e : {&nn->ready, &nn->done[0], &nn->done[1]})
        NCKC(cudaEventCreateWithFlags(e, cudaEventDisableTiming), "cudaEventCreate");
    const long long Pmax = (long long)nn->nb * nn->H * nn->W;
    int dev = 0;
    NCKC(cudaGetDevice(&dev), "cudaGetDevice");
    NCKC(cudaDeviceGetAttribute(&nn->sms, cudaDevAttrMultiProcessorCount, dev),
         "cudaDeviceGetAttribute");
    // weight-gradient partials: the most of any convolution and batch size
    // (the splits grow with the pixels, up to two CTAs per SM)
    size_t pfl = 0, maxc = 0;
    for (auto& c : nn->conv) {
        const long long tiles = ((9LL * c.cinp + UM - 1) / UM) * ((c.coutp + 255) / 256);
        const long long most = (2LL * nn->sms + tiles - 1) / tiles;
        const long long px = (pixels(nn, c.in, nn->nb) + 255) / 256;
        const size_t need = (size_t)(most < px ? most : px) * conv_wsize(c);
        pfl = need > pfl ? need : pfl;
        maxc = (size_t)c.coutp > maxc ? (size_t)c.coutp : maxc;
    }
    NCKC(lbm::dev_alloc(&nn->part, pfl * sizeof(float)), "cudaMalloc(partials)");
    size_t runs = 1;  // of by_octets
    for (auto& T : nn->t) {
        const size_t r = (size_t)nn->nb * T.h * T.w * (T.cp / 8) / (1u << 30) + 1;
        runs = r > runs ? r : runs;
    }
    for (auto& b : nn->bpart)
        NCKC(lbm::dev_alloc(&b, runs * kBiasBlocks * maxc * sizeof(float)), "cudaMalloc(partials)");
    NCKC(lbm::dev_alloc(&nn->flat, lbm_nn_param_count(nn) * sizeof(float)),
         "cudaMalloc(parameter vector)");
    NCKC(lbm::dev_alloc(&nn->dpart, 1025 * sizeof(double)), "cudaMalloc(loss)");
    NCKC(lbm::dev_alloc(&nn->xin, Pmax * 4 * sizeof(float)), "cudaMalloc(inputs)");
    NCKC(lbm::dev_alloc(&nn->tgt, Pmax * 3 * sizeof(float)), "cudaMalloc(targets)");
    NCKC(lbm::dev_alloc(&nn->fl, Pmax), "cudaMalloc(fluid)");
    NCKC(lbm::dev_alloc(&nn->yout, Pmax * 3 * sizeof(float)), "cudaMalloc(outputs)");
    NCKC(lbm::dev_alloc(&nn->gout, Pmax * 3 * sizeof(float)), "cudaMalloc(output gradient)");
    NCKC(lbm::dev_alloc(&nn->tmp3, Pmax * 3 * sizeof(float)), "cudaMalloc(output stage)");
    // (of the finest grid that lbm_nn_prolong takes: a factor of 16)
    NCKC(lbm::dev_alloc(&nn->ssum, (size_t)nn->nb * Stagger(1, 256LL * nn->H * nn->W).parts * 3 *
                                       sizeof(double)),
         "cudaMalloc(output sums)");
    NCKC(lbm::dev_alloc(&nn->gemm_err, sizeof(int)), "cudaMalloc(error word)");
    NCKC(cudaMemsetAsync(nn->gemm_err, 0, sizeof(int), nn->stream), "cudaMemset");
#undef NCKC
    // He-normal initial weights (host generator), zero biases
    std::vector<float> params(lbm_nn_param_count(nn));
    std::mt19937_64 rng(seed);
    std::normal_distribution<double> N01(0.0, 1.0);
    size_t k = 0;
    for (auto& c : nn->conv) {
        const double sd = std::sqrt(2.0 / (9.0 * c.cin));
        for (size_t i = 0; i < 9ull * c.cin * c.cout; ++i) params[k++] = (float)(sd * N01(rng));
        for (int i = 0; i < c.cout; ++i) params[k++] = 0.0f;
    }
    lbm_status st = lbm_nn_set_params(nn, params.data());
    if (st != LBM_OK) return fail(st);
    *out = nn;
    return LBM_OK;
}

void lbm_nn_destroy(lbm_nn* nn) {
    if (!nn) return;
    cudaFree(nn->pbuf);
    cudaFree(nn->wbuf);
    cudaFree(nn->abuf);
    if (nn->side) {
        cudaStreamSynchronize(nn->side);
        cudaStreamDestroy(nn->side);
    }
    for (cudaEvent_t e : {nn->ready, nn->done[0], nn->done[1]})
        if (e) cudaEventDestroy(e);
    for (auto b : nn->scratch) cudaFree(b);
    cudaFree(nn->part);
    for (auto b : nn->bpart) cudaFree(b);
    cudaFree(nn->flat);
    cudaFree(nn->dpart);
    cudaFree(nn->xin);
    cudaFree(nn->tgt);
    cudaFree(nn->fl);
    cudaFree(nn->yout);
    cudaFree(nn->gout);
    cudaFree(nn->tmp3);
    cudaFree(nn->ssum);
    cudaFree(nn->gemm_err);
    cudaFree(nn->fine);
    cudaFree(nn->fine_fl);
    delete nn;
}

size_t lbm_nn_param_count(const lbm_nn* nn) {
    if (!nn) return 0;
    size_t n = 0;
    for (auto& c : nn->conv) n += 9ull * c.cin * c.cout + c.cout;
    return n;
}

// Host parameter vector (dy, dx, cin, cout per convolution, then biases) <->
// device masters [coutp][tap][cinp]: reordered on the GPU, one copy.  (The
// padding of the device arrays is zero from creation and stays so.)
static lbm_status transfer_params(lbm_nn* nn, float* host, bool to_device, bool grads) {
    const size_t bytes = lbm_nn_param_count(nn) * sizeof(float);
    if (to_device)
        NCK(nn, cudaMemcpyAsync(nn->flat, host, bytes, cudaMemcpyHostToDevice, nn->stream),
            "cudaMemcpyAsync(H2D)");
    ParamTable table;
    table.n = 0;
    long long at = 0;
    int blocks = 0;
    for (auto& c : nn->conv) {
        table.e[table.n++] = {grads ? c.gw : c.wm, grads ? c.gb : c.bm, at, c.cin, c.cout, c.cinp, blocks};
        at += 9ll * c.cin * c.cout + c.cout;
        blocks += (c.cout + 31) / 32 * ((c.cin + 31) / 32) * 9;
    }
    if (to_device) param_order_kernel<false><<<blocks, kThreads, 0, nn->stream>>>(nn->flat, table);
    else param_order_kernel<true><<<blocks, kThreads, 0, nn->stream>>>(nn->flat, table);
    NCK(nn, cudaGetLastError(), "parameter order");
    ++nn->launches;
    if (!to_device)
        NCK(nn, cudaMemcpyAsync(host, nn->flat, bytes, cudaMemcpyDeviceToHost, nn->stream),
            "cudaMemcpyAsync(D2H)");
    NCK(nn, cudaStreamSynchronize(nn->stream), "cudaStreamSynchronize");
    return LBM_OK;
}

lbm_status lbm_nn_get_params(lbm_nn* nn, float* params) {
    if (!nn || !params) return LBM_ERR_INVALID;
    return transfer_params(nn, params, false, false);
}

lbm_status lbm_nn_set_params(lbm_nn* nn, const float* params) {
    if (!nn || !params) return LBM_ERR_INVALID;
    lbm_status s = transfer_params(nn, const_cast<float*>(params), true, false);
    if (s != LBM_OK) return s;
    for (auto& c : nn->conv) {
        const size_t w = conv_wsize(c);
        NCK(nn, cudaMemsetAsync(c.mw, 0, w * sizeof(float), nn->stream), "cudaMemset");
        NCK(nn, cudaMemsetAsync(c.vw, 0, w * sizeof(float), nn->stream), "cudaMemset");
        NCK(nn, cudaMemsetAsync(c.mb, 0, c.coutp * sizeof(float), nn->stream), "cudaMemset");
        NCK(nn, cudaMemsetAsync(c.vb, 0, c.coutp * sizeof(float), nn->stream), "cudaMemset");
    }
    nn->adam_t = 0;
    s = sync_weights(nn);
    if (s != LBM_OK) return s;
    NCK(nn, cudaStreamSynchronize(nn->stream), "cudaStreamSynchronize");
    return LBM_OK;
}

lbm_status lbm_nn_forward(lbm_nn* nn, const float* x, int n, float* y) {
    LBM_RANGE("lbm_nn_forward");
    if (!nn || !x || !y) return LBM_ERR_INVALID;
    if (bad_batch(nn, n)) return LBM_ERR_INVALID;
    lbm_status s = upload_inputs(nn, x, nullptr, nullptr, n);
    if (s == LBM_OK) s = forward(nn, n);
    if (s != LBM_OK) return s;
    const long long P = (long long)n * nn->H * nn->W;
    NCK(nn, cudaMemcpyAsync(y, nn->yout, P * 3 * sizeof(float), cudaMemcpyDeviceToHost,
                            nn->stream),
        "cudaMemcpyAsync(D2H)");
    NCK(nn, cudaStreamSynchronize(nn->stream), "cudaStreamSynchronize");
    return check_gemm(nn);
}

lbm_status lbm_nn_prolong(lbm_nn* nn, const float* y, int n, int factor, const uint8_t* fluid,
                          float* out) {
    LBM_RANGE("lbm_nn_prolong");
    if (!nn || !y || !fluid || !out) return LBM_ERR_INVALID;
    if (bad_batch(nn, n)) return LBM_ERR_INVALID;
    if (factor < 1 || factor > 16) {
        nn_err(nn, "factor %d outside [1, 16]", factor);
        return LBM_ERR_INVALID;
    }
    const int H = nn->H * factor, W = nn->W * factor;
    const long long cells = (long long)H * W;
    const cudaStream_t s = nn->stream;
    if (cells > nn->fine_cells) {
        // grown on demand, kept until the network is destroyed
        NCK(nn, cudaStreamSynchronize(s), "cudaStreamSynchronize");
        cudaFree(nn->fine);
        cudaFree(nn->fine_fl);
        nn->fine = nullptr;
        nn->fine_fl = nullptr;
        nn->fine_cells = 0;
        NCK(nn, lbm::dev_alloc(&nn->fine, 2 * (size_t)nn->nb * cells * 3 * sizeof(float)),
            "cudaMalloc(fine fields)");
        NCK(nn, lbm::dev_alloc(&nn->fine_fl, (size_t)nn->nb * cells), "cudaMalloc(fine fluid)");
        nn->fine_cells = cells;
    }
    const long long Pc = (long long)n * nn->H * nn->W, P = (long long)n * cells;
    float* f0 = nn->fine;
    float* f1 = nn->fine + (size_t)nn->nb * cells * 3;
    // the coarse fields go through the output stage's buffer, free between calls
    NCK(nn, cudaMemcpyAsync(nn->tmp3, y, Pc * 3 * sizeof(float), cudaMemcpyHostToDevice, s),
        "cudaMemcpyAsync(H2D)");
    NCK(nn, cudaMemcpyAsync(nn->fine_fl, fluid, P, cudaMemcpyHostToDevice, s),
        "cudaMemcpyAsync(H2D)");
    const FluidBytes fl{nn->fine_fl};
    prolong_kernel<<<grid_of(P), kThreads, 0, s>>>(nn->tmp3, nn->fine_fl, f0, n, nn->H, nn->W,
                                                   factor);
    NCK(nn, cudaGetLastError(), "prolongation");
    out_smooth_kernel<false, false><<<grid_of(P), kThreads, 0, s>>>(f0, 3, fl, f1, 3, n, H, W);
    NCK(nn, cudaGetLastError(), "output smoothing (fine)");
    const Stagger g(n, cells);
    stagger_sum_kernel<<<g.grid(), kThreads, 0, s>>>(f1, fl, nn->ssum, H, W, g);
    NCK(nn, cudaGetLastError(), "staggered sums (fine)");
    stagger_apply_kernel<<<g.grid(), kThreads, 0, s>>>(f1, fl, nn->ssum, f0, H, W, g);
    NCK(nn, cudaGetLastError(), "staggered projection (fine)");
    nn->launches += 4;
    NCK(nn, cudaMemcpyAsync(out, f0, P * 3 * sizeof(float), cudaMemcpyDeviceToHost, s),
        "cudaMemcpyAsync(D2H)");
    NCK(nn, cudaStreamSynchronize(s), "cudaStreamSynchronize");
    return LBM_OK;
}

lbm_status lbm_nn_gradients(lbm_nn* nn, const float* x, const float* target,
                            const uint8_t* fluid, int n, float* loss, float* grads) {
    LBM_RANGE("lbm_nn_gradients");
    if (!nn || !x || !target || !fluid) return LBM_ERR_INVALID;
    if (bad_batch(nn, n)) return LBM_ERR_INVALID;
    lbm_status s = upload_inputs(nn, x, target, fluid, n);
    if (s == LBM_OK) s = forward(nn, n);
    if (s == LBM_OK) s = backward(nn, n, loss);
    if (s == LBM_OK) s = check_gemm(nn);
    if (s == LBM_OK && grads) s = transfer_params(nn, grads, false, true);
    return s;
}

lbm_status lbm_nn_train_step(lbm_nn* nn, const float* x, const float* target,
                             const uint8_t* fluid, int n, float lr, float* loss) {
    LBM_RANGE("lbm_nn_train_step");
    if (!nn || !x || !target || !fluid) return LBM_ERR_INVALID;
    if (bad_batch(nn, n)) return LBM_ERR_INVALID;
    if (!(lr > 0.0f) || !std::isfinite(lr)) {
        nn_err(nn, "learning rate must be finite and > 0");
        return LBM_ERR_INVALID;
    }
    lbm_status s = upload_inputs(nn, x, target, fluid, n);
    if (s == LBM_OK) s = forward(nn, n);
    if (s == LBM_OK) s = backward(nn, n, loss);
    if (s != LBM_OK) return s;
    ++nn->adam_t;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - (float)std::pow(0.9, (double)nn->adam_t);
    const float c2 = 1.0f - (float)std::pow(0.999, (double)nn->adam_t);
    for (auto& c : nn->conv) {
        const long long w = (long long)conv_wsize(c);
        adam_kernel<<<grid_of(w), kThreads, 0, nn->stream>>>(c.wm, c.gw, c.mw, c.vw, w, lr, b1, b2,
                                                             c1, c2, 1e-8f);
        NCK(nn, cudaGetLastError(), "adam");
        adam_kernel<<<grid_of(c.coutp), kThreads, 0, nn->stream>>>(c.bm, c.gb, c.mb, c.vb, c.coutp,
                                                                   lr, b1, b2, c1, c2, 1e-8f);
        NCK(nn, cudaGetLastError(), "adam");
        nn->launches += 2;
    }
    s = sync_weights(nn);
    if (s != LBM_OK) return s;
    NCK(nn, cudaStreamSynchronize(nn->stream), "cudaStreamSynchronize");
    return check_gemm(nn);
}

int64_t lbm_nn_launch_count(const lbm_nn* nn) { return nn ? nn->launches : -1; }

const char* lbm_nn_last_error(const lbm_nn* nn) { return nn ? nn->err : g_nn_err; }

}  // extern "C"
