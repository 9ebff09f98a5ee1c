// One-axis transforms of real fields on the tensor cores, exact to more than
// the double-float FFT stages they replace: spectral derivatives, and the
// real Fourier transform (cosines and sines) along an axis and back.
//
// Each is a real n x n matrix applied to a batch of lines, so a contraction.
// With h = n/2 it splits into two h x h blocks, e and o, that act on the
// functions of even and of odd frequency: on a field these are the sums and
// differences s = x_lo + x_hi, d = x_lo - x_hi of its halves (and back
// out_lo = e + o, out_hi = e - o); the coefficients of a transformed line
// are stored even frequencies first, then odd ones.
//   derivative: e = De s, o = Do d, De, Do = (D(j - l) +- D(j - l - h)) / 2
//   forward:    the orthonormal cosines and sines of even (odd) frequency
//   inverse:    their transposes
//
// The products are taken in integers.  Each line is scaled by the power of
// two of its largest magnitude to 53-bit integers, the matrices are rounded
// to 54-bit integers once, and both are cut into seven signed digits of
// radix 256.  A digit is exact in f16, a product of two is at most 2^14,
// and the sums over h <= 72 and up to seven digit pairs (two of them with a
// leading digit, at most 64) stay below 2^24, so the f32 accumulators of
// tcgen05.mma (kind::f16) hold exact integers.  Digit products of equal
// weight share one accumulator: 7 accumulators, 28 products; the first
// products dropped, six for each term, are each at most about 2^-51 of the
// line's largest value times the largest matrix entry.  Fields are double-float pairs in memory (8 bytes).
#include <math.h>

#include <algorithm>

#include "digits.cuh"
#include "kernels.h"
#include "pdl.cuh"
#include "tcgen.cuh"

namespace ofdft {

namespace {

constexpr int kLines = 64;    // lines of a tile: the rows of one M = 64 accumulator
constexpr int kTlThreads = 640;   // converting and reading-out threads at most; one more warp issues the products
constexpr int kMaxChunks = 3;     // column chunks of a matrix
constexpr int kMaxUnits = 2 * kMaxChunks;

// Shared-memory distance between 8-wide K chunks of the lines' digits: one
// 16-byte row more than the 64 lines, so that threads that walk the chunks
// of one line (z axis) store to different banks.
constexpr uint32_t kALbo = (kLines + 1) * 16;

// Sizes of the operands for an axis of n points.  The outputs come in column
// chunks of up to 4 groups of 8 (their 7 accumulators then fit one product's
// N <= 256); chunk c of e and of o are units 2c and 2c + 1 of the matrix,
// which pass through nslot shared-memory slots.
struct TlShape {
    int h, np, nc;            // half length; padded to 8 (N); 8-wide K chunks (an even number)
    int chunks, g;            // column chunks; groups of 8 in each (the last may have fewer)
    int nslot;
    uint32_t a_dig;           // bytes of one digit of a tile half
    uint32_t unit;            // bytes of a slot (a full chunk's unit)
    uint32_t cols;            // tensor-memory columns
    uint32_t smem;
};

__host__ __device__ __forceinline__ int tl_width(const TlShape &s, int c) { return 8 * min(s.g, s.np / 8 - c * s.g); }
__host__ __device__ __forceinline__ uint32_t tl_unit_bytes(const TlShape &s, int c)
{
    return (uint32_t)(s.nc * kDig * tl_width(s, c) * 16);
}

constexpr size_t kTlSmemMax = 227 * 1024 - 2048;   // static shared memory of the kernel beside it

TlShape tl_shape(int n)
{
    TlShape s;
    s.h = n / 2;
    s.np = (s.h + 7) / 8 * 8;
    s.nc = (s.h + 15) / 16 * 2;
    const int groups = s.np / 8;
    s.chunks = std::max((groups + 3) / 4, groups > 1 ? 2 : 1);
    s.g = (groups + s.chunks - 1) / s.chunks;
    s.a_dig = (uint32_t)s.nc * kALbo;
    s.unit = (uint32_t)(s.nc * kDig * s.g * 128);
    s.cols = 32;
    while (s.cols < (uint32_t)(kDig * s.np)) s.cols *= 2;
    const uint32_t a = 2 * kDig * s.a_dig;
    s.nslot = a < kTlSmemMax ? (int)std::min<size_t>(2 * s.chunks, (kTlSmemMax - a) / s.unit) : 0;
    s.smem = a + s.nslot * s.unit;
    return s;
}

// One transform of a launch.
struct TlJob {
    TlShape sh;
    int nlines, tiles, zlen;       // lines; tiles of 64; lines of one outer index (x, y: consecutive in memory)
    int zaxis;                     // lines contiguous in memory
    int direct_in, direct_out;     // coefficients instead of a field's halves
    long long ostride, rstride;    // between outer indices; between a line's points
    int mexp;
    const unsigned char *mat;
    const float2 *in;
    float2 *out;
};
constexpr int kMaxJobs = 4;
struct TlJobs {
    TlJob job[kMaxJobs];
    int count;
};

// x + sgn y of two such pairs, normalised, times sc (a power of two).
__device__ __forceinline__ float2 butterfly(ff::f2 x, ff::f2 y, float sgn, float sc)
{
    const float s = ff::ffma(sgn, y.hi, x.hi);
    const float bb = ff::fsub(s, x.hi);
    const float e = ff::fadd(ff::fsub(x.hi, ff::fsub(s, bb)), ff::ffma(sgn, y.hi, -bb));
    const float l = ff::fadd(ff::ffma(sgn, y.lo, x.lo), e);
    const ff::f2 r = ff::fast_two_sum(s, l);
    return make_float2(r.hi * sc, r.lo * sc);
}

__device__ __forceinline__ void bar_arrive(int id, int count) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory"); }
__device__ __forceinline__ void bar_sync(int id, int count) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory"); }

// The issuing warp: for every unit of the matrix, digit i of the lines meets
// digits 0 .. 6 - i of the unit, which lie side by side along N as their
// accumulators i .. 6 do.  e accumulates in lanes 0-15 of each quarter of
// the tensor memory, o in lanes 16-31.  KS: 16-wide K steps; unrolled, so
// that the descriptors are built in uniform registers (with run-time loops
// the products of n = 96 took 9,400 cycles to issue, from a single thread
// 19,100; so they run at the tensor cores' rate, 0.46 cycles a column).  A
// wait that runs out raises *bad before the products that it stood for are
// committed: whoever sees them done sees *bad.
template <int KS>
__device__ __forceinline__ void issue(const TlShape &sh, const unsigned char *mat, uint32_t full, uint32_t done, uint32_t sa,
                                      uint32_t sb, uint32_t tmem, int nthreads, volatile int *bad)
{
    const int units = 2 * sh.chunks;
    const uint32_t a_dig = sh.a_dig;
    auto wait = [&](uint32_t bar) {
        if (!tc::mbar_wait(bar, 0)) {
            *bad = 1;
            __threadfence_block();
        }
        __syncwarp();
    };
#pragma unroll 1
    for (int u = 0; u < units; ++u) {
        const int c = u >> 1, width = tl_width(sh, c);
        wait(full + 8 * u);
        if (u < 2) bar_sync(1 + u, nthreads);     // the digits of s (u = 0), of d (u = 1)
        tc::fence_after_sync();
        const uint32_t blb = (uint32_t)(kDig * width) * 16;
        const uint64_t a0 = tc::operand(sa + (u & 1) * kDig * a_dig, kALbo, 128);
        const uint64_t b0 = tc::operand(sb + (u % sh.nslot) * sh.unit, blb, 128);
        const uint32_t acc = tmem + ((uint32_t)(u & 1) << 20) + c * sh.g * 8 * kDig;
#pragma unroll
        for (int i = 0; i < kDig; ++i) {
            const uint32_t idesc = tc::idesc_f16(kLines, (kDig - i) * width);
#pragma unroll
            for (int k = 0; k < KS; ++k)
                tc::mma_f16(acc + i * width, a0 + ((i * a_dig + k * 2 * kALbo) >> 4), b0 + ((k * 2 * blb) >> 4), idesc,
                            (i | k) != 0);
        }
        tc::mma_commit(done + 8 * u);
        const int next = u - 1 + sh.nslot;        // the unit that takes over slot (u - 1)
        if (u >= 1 && next < units) {
            wait(done + 8 * (u - 1));
            if ((threadIdx.x & 31) == 0) {
                const uint32_t bytes = tl_unit_bytes(sh, next >> 1);
                tc::mbar_expect(full + 8 * next, bytes);
                tc::bulk_load(sb + (next % sh.nslot) * sh.unit, mat + (size_t)next * sh.unit, bytes, full + 8 * next);
            }
            __syncwarp();
        }
    }
}

// Eight consecutive outputs of a line (left: how many lie in the half).
__device__ __forceinline__ void store_lines(const float2 (&y)[8], float2 *p, long long rstride, int left, bool wide, bool ok)
{
    if (!ok) return;
    if (left >= 8) {
        if (wide) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                reinterpret_cast<float4 *>(p)[i] = make_float4(y[2 * i].x, y[2 * i].y, y[2 * i + 1].x, y[2 * i + 1].y);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) p[i * rstride] = y[i];
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < left) p[i * rstride] = y[i];
    }
}

// The transforms of a launch's jobs, one block per tile of 64 lines.  out
// may be in: a block reads its lines whole before it writes them.
//
// M = 64 because at 96^3 tiles of 128 lines would leave half the SMs idle
// (144 tiles of 64 for 152 SMs).  Measured (GB300, in a graph): one axis at
// 96^3 7.8 us (z 10), three derivatives in one launch 24 us, one axis at
// 48^3 5.5 us; the double-float FFT passes took about 19 us a derivative and
// 12-32 us a Fourier pass at 96^3.  Of the 12,000 cycles of a tile the
// products are 6,000 (0.5-0.7 cycles a column, M = 64 runs at half rate),
// the conversion 2,800, the load 1,600, the read-out 1,700 behind the last
// product; instruction fetch is the largest stall, since each warp runs the
// code once.
__global__ void __launch_bounds__(kTlThreads + 32, 1) k_tline(const __grid_constant__ TlJobs jobs)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ __align__(8) uint64_t s_bar[2 * kMaxUnits];   // units of the matrix in place; their products done
    __shared__ uint32_t s_tmem;
    __shared__ uint32_t s_max[kLines];
    __shared__ int s_bad;                          // a bounded wait ran out: the tile's output is NaN
    int ji = 0, tile = blockIdx.x;
    while (ji + 1 < jobs.count && tile >= jobs.job[ji].tiles) tile -= jobs.job[ji++].tiles;
    const TlJob &jb = jobs.job[ji];
    const TlShape &sh = jb.sh;
    const int h = sh.h, nc = sh.nc, zaxis = jb.zaxis;
    const uint32_t a_dig = sh.a_dig;
    unsigned char *A = smraw, *B = smraw + 2 * kDig * (size_t)a_dig;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nconv = blockDim.x - 32;             // the last warp issues the products
    const uint32_t full = tc::smem_addr(s_bar), done = full + 8 * kMaxUnits;
    const uint32_t sa = tc::smem_addr(A), sb = tc::smem_addr(B);
    const long long rstride = jb.rstride;
    const int nlines = jb.nlines, zlen = jb.zlen;
    if (tid >= nconv) {
        const int units = 2 * sh.chunks;
        if (lane == 0) {
            s_bad = 0;
            for (int i = 0; i < 2 * kMaxUnits; ++i) tc::mbar_init(full + 8 * i, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            for (int u = 0; u < min(units, sh.nslot); ++u) {
                const uint32_t bytes = tl_unit_bytes(sh, u >> 1);
                tc::mbar_expect(full + 8 * u, bytes);
                tc::bulk_load(sb + u * sh.unit, jb.mat + (size_t)u * sh.unit, bytes, full + 8 * u);
            }
        }
        __syncwarp();
        tc::tmem_alloc(tc::smem_addr(&s_tmem), sh.cols);
        __syncwarp();
        tc::fence_before_sync();
        bar_arrive(4, blockDim.x);                 // barriers and tensor memory are there
        const uint32_t tmem = __shfl_sync(0xffffffffu, *(volatile uint32_t *)&s_tmem, 0);
        switch (nc / 2) {
        case 1: issue<1>(sh, jb.mat, full, done, sa, sb, tmem, blockDim.x, &s_bad); break;
        case 2: issue<2>(sh, jb.mat, full, done, sa, sb, tmem, blockDim.x, &s_bad); break;
        case 3: issue<3>(sh, jb.mat, full, done, sa, sb, tmem, blockDim.x, &s_bad); break;
        case 4: issue<4>(sh, jb.mat, full, done, sa, sb, tmem, blockDim.x, &s_bad); break;
        default: issue<5>(sh, jb.mat, full, done, sa, sb, tmem, blockDim.x, &s_bad); break;
        }
        __syncthreads();                           // every accumulator has been read
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, sh.cols);
        return;
    }

    // thread = (line, K chunk): consecutive threads walk the lines of an x or
    // y tile, the chunks of a z line, so that loads coalesce
    const int row = zaxis ? tid / nc : tid & (kLines - 1);
    const int chunk = zaxis ? tid - row * nc : tid >> 6;
    const bool mine = tid < kLines * nc;           // (a shorter job may share the launch)
    // read-out: a warp takes its quarter's 16 lines of e (lanes 0-15) and of o
    const int half = lane >> 4, quarter = warp & 3, set = warp >> 2, nset = nconv >> 7;
    const int r = quarter * 16 + (lane & 15);
    const int ln = tile * kLines + r;
    const bool w_ok = ln < nlines;
    const int ou = ln / zlen;
    const long long ln_off = (w_ok ? ou * jb.ostride + (zaxis ? 0 : ln - ou * zlen) : 0) + (half ? h * rstride : 0);
    const bool wide = zaxis && (h & 1) == 0;
    if (tid < kLines) s_max[tid] = 27u << 23;      // 2^-100: the least exponent of the scale
    pdl_wait();                                    // (the issuing warp reads nothing that another kernel writes)
    float2 v[16];
    if (mine) {
        const int line = tile * kLines + row;
        const bool ok = line < nlines;
        const int outer = ok ? line / zlen : 0, left = min(8, h - chunk * 8);
        const float2 *src = jb.in + (ok ? outer * jb.ostride + (zaxis ? 0 : line - outer * zlen) : 0) + chunk * 8 * rstride;
        const float2 *srh = src + h * rstride;
        if (ok && left == 8) {
            if (wide) {                        // 16-byte aligned halves
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 x = reinterpret_cast<const float4 *>(src)[i], y = reinterpret_cast<const float4 *>(srh)[i];
                    v[2 * i] = make_float2(x.x, x.y);
                    v[2 * i + 1] = make_float2(x.z, x.w);
                    v[8 + 2 * i] = make_float2(y.x, y.y);
                    v[8 + 2 * i + 1] = make_float2(y.z, y.w);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    v[i] = src[i * rstride];
                    v[8 + i] = srh[i * rstride];
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const bool in_line = ok && i < left;
                v[i] = in_line ? src[i * rstride] : make_float2(0.0f, 0.0f);
                v[8 + i] = in_line ? srh[i * rstride] : make_float2(0.0f, 0.0f);
            }
        }
    }
    bar_sync(4, blockDim.x);                       // s_max is set too; the loads are under way
    tc::fence_after_sync();
    const uint32_t tmem = s_tmem;
    pdl_trigger();                                 // the block has its tensor memory: see pdl.cuh
    if (mine) {
        uint32_t m = 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) m = max(m, __float_as_uint(v[i].x) & 0x7fffffffu);
        if (m > (27u << 23)) atomicMax(&s_max[row], m);
    }
    bar_sync(3, nconv);
    // digits of the first operand (s), then of the second (d): the
    // products of e start in between
    unsigned char *dsta = A + chunk * kALbo + row * 16;
    uint64_t q[8];
    if (mine) {
        const float u = ff::int_bits_float((254u - (s_max[row] >> 23)) << 23 | (s_max[row] >> 23 == 254u ? 0x400000u : 0u));
        if (jb.direct_in) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                q[i] = to_fixed(v[i], u) + (kDigBias - fixed_off<52>());
                const uint64_t y = to_fixed(v[8 + i], u) + (kDigBias - fixed_off<52>());
                v[i] = make_float2(__uint_as_float((uint32_t)y), __uint_as_float((uint32_t)(y >> 32)));
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint64_t x = to_fixed(v[i], u), y = to_fixed(v[8 + i], u);
                q[i] = x + y + (kDigBias - 2 * fixed_off<52>());
                const uint64_t d = x - y + kDigBias;
                v[i] = make_float2(__uint_as_float((uint32_t)d), __uint_as_float((uint32_t)(d >> 32)));
            }
        }
        store_digits(q, dsta, a_dig);
    }
    tc::fence_async();
    bar_arrive(1, blockDim.x);
    if (mine) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            q[i] = (uint64_t)__float_as_uint(v[i].x) | (uint64_t)__float_as_uint(v[i].y) << 32;
        store_digits(q, dsta + kDig * a_dig, a_dig);
    }
    tc::fence_async();
    bar_arrive(2, blockDim.x);

    const uint32_t m = s_max[r];
    // weight 1 stands for 2^96 times the integers' units 2^(E - 52) and 2^-mexp
    float sc = ff::pow2i((int)(m >> 23) - 127 + 44 - jb.mexp);
    if (m >= 0x7f800000u) sc = __uint_as_float(0x7fc00000u);   // inf, NaN
    const float sgn = half ? -1.0f : 1.0f;
    float2 *dst = jb.out + ln_off;
#pragma unroll 1
    for (int ch = 0; ch < sh.chunks; ++ch) {
        const int width = tl_width(sh, ch), j0 = ch * sh.g * 8;
        if (!tc::mbar_wait(done + 8 * (2 * ch + 1), 0) || *(volatile int *)&s_bad) sc = __uint_as_float(0x7fc00000u);
        tc::fence_after_sync();
        const uint32_t tacc = tmem + ((uint32_t)(quarter * 32) << 16) + j0 * kDig;
#pragma unroll 1
        for (int c0 = set * 8; c0 < width; c0 += nset * 8) {
            float a[kDig][8];
#pragma unroll
            for (int d = 0; d < kDig; ++d) tc::tmem_ld8(tacc + d * width + c0, a[d]);
            tc::tmem_wait_ld();
#pragma unroll
            for (int d = 0; d < kDig; ++d) tc::pin8(a[d]);
            float2 y[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float t[kDig];
#pragma unroll
                for (int d = 0; d < kDig; ++d) t[d] = a[d][i];
                const ff::f2 own = combine(t);
                if (jb.direct_out) {
                    y[i] = scaled(own, sc);
                } else {
                    ff::f2 other;
                    other.hi = __shfl_xor_sync(0xffffffffu, own.hi, 16);
                    other.lo = __shfl_xor_sync(0xffffffffu, own.lo, 16);
                    y[i] = butterfly(other, own, sgn, sc);
                }
            }
            const int j = j0 + c0;
            store_lines(y, dst + j * rstride, rstride, h - j, wide, w_ok);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
}

}  // namespace

bool tline_supported(int n)
{
    const TlShape s = tl_shape(n);
    return s.nslot >= 2 && kDig * s.np <= 512 && kLines * s.nc <= kTlThreads;
}

// The derivative matrix's largest entry is scale / (2 sin(2 pi / n)), both
// blocks' sums of cot and tan; its exponent has to keep a line's scale (2^-100
// to 2^127, times 2^(44 - mexp)) within binary32.  Grid spacings from 2^14
// bohr leave that range.
bool tline_derivative_supported(int n, double scale)
{
    if (!tline_supported(n)) return false;
    int e = 0;
    frexp(fabs(scale) / (2.0 * sin(6.283185307179586477 / n)), &e);
    return 54 - e >= -60 && 54 - e <= 68;
}

// A double-float set's transforms: the derivatives of a GGA take the tensor
// cores along every axis that they support; the Hartree chain does when all
// three axes (and for a GGA their derivatives) are supported.  ftTF has the
// chain alone and five kernels more in this form, which on the smallest grids
// cost more than they save, FFT passes -> here: an evaluation at 8^3 51 -> 56
// us, 16^3 62 -> 55, 32^3 64 -> 58, 48^3 73 -> 70, 54^3 86 -> 79, a solve's
// evaluation at 32^3 119 -> 102 us.  (GGA: 96^3 291 -> 255 us, 48^3 95 -> 92,
// 32^3 72 -> 73 before the launches of a chain overlapped.)
constexpr long long kRealTfPoints = 2048;
TlPlan tline_plan(const GridInfo &g, bool gga)
{
    const int n3[3] = {g.nx, g.ny, g.nz};
    const bool on = g.dd && !g.dws;
    TlPlan p{{false, false, false}, on && (gga || g.N >= kRealTfPoints)};
    for (int a = 0; a < 3; ++a) {
        p.der[a] = on && gga && tline_derivative_supported(n3[a], g.ds[a] * n3[a]);
        p.real_basis = p.real_basis && (gga ? p.der[a] : tline_supported(n3[a]));
    }
    return p;
}

size_t tline_matrix_bytes(int n)
{
    const TlShape s = tl_shape(n);
    return 2 * (size_t)s.chunks * s.unit;
}

namespace {

// The matrix blocks e and o (h x h each; at(half, output, input) indexes a
// table of the distinct entries) times 2^mexp as seven f16 digits each, laid
// out as the kernel's shared-memory image ([column chunk][e, o][K chunk]
// [digit][output][8]); returns mexp.
// On fixed arrays: the allocation-free entry point's first call fills its
// matrices too.
constexpr int kTlMaxEdge = 2 * (512 / kDig / 8 * 8);   // tline_supported: the accumulators of np <= 72
struct DigitF16 {
    uint16_t f[256];                               // f16 of -128 .. 127
    constexpr DigitF16() : f{}
    {
        for (int b = 0; b < 256; ++b) {
            int a = b < 128 ? 128 - b : b - 128, ex = 0;
            while ((a >> ex) > 1) ++ex;
            f[b] = a == 0 ? 0 : (uint16_t)((b < 128 ? 0x8000 : 0) | ((ex + 15) << 10) | ((a << (10 - ex)) & 0x3ff));
        }
    }
};
template <typename F> int pack_matrix(int n, const long double *entry, int entries, F at, uint16_t *img)
{
    const TlShape s = tl_shape(n);
    const int h = s.h;
    static constexpr DigitF16 digit;
    long double big = 0.0L;
    for (int i = 0; i < entries; ++i) big = std::max(big, fabsl(entry[i]));
    int e = 0;
    frexpl(big, &e);                               // big in [2^(e-1), 2^e)
    const int mexp = 54 - e;                       // integers up to 2^54
    uint64_t fixed[3 * kTlMaxEdge];
    for (int i = 0; i < entries; ++i) fixed[i] = (uint64_t)llroundl(ldexpl(entry[i], mexp)) + kDigBias;
    std::fill(img, img + tline_matrix_bytes(n) / 2, (uint16_t)0);
    for (int half = 0; half < 2; ++half)
        for (int j = 0; j < h; ++j) {
            const int ch = j / (8 * s.g), width = tl_width(s, ch), jj = j - ch * 8 * s.g;
            uint16_t *base = img + (size_t)(2 * ch + half) * s.unit / 2;
            for (int l = 0; l < h; ++l) {
                const uint64_t b = fixed[at(half, j, l)];
                uint16_t *p = base + ((size_t)(l / 8) * kDig * width + jj) * 8 + l % 8;
                for (int d = 0; d < kDig; ++d) p[(size_t)d * width * 8] = digit.f[(b >> (8 * (6 - d))) & 0xff];
            }
        }
    return mexp;
}

const long double kTwoPiL = 6.283185307179586476925286766559005768L;

}  // namespace

// D(m) = (scale/2) (-1)^m cot(pi m/n), period n.
int tline_derivative_matrix(int n, double scale, uint16_t *img)
{
    const int h = n / 2;
    long double D[kTlMaxEdge] = {}, t[2 * kTlMaxEdge];
    for (int m = 1; m < n; ++m) {
        const long double x = 0.5L * kTwoPiL * m / n;
        D[m] = (long double)scale * 0.5L * ((m & 1) ? -1.0L : 1.0L) * (2 * m == n ? 0.0L : cosl(x) / sinl(x));
    }
    for (int m = 0; m < n; ++m) {                  // De, Do by m = j - l (mod n)
        const long double a = D[m], b = D[(m + n - h) % n];
        t[m] = 0.5L * (a + b);
        t[n + m] = 0.5L * (a - b);
    }
    return pack_matrix(n, t, 2 * n, [&](int half, int j, int l) { return (size_t)half * n + (j - l + n) % n; }, img);
}

int tline_fourier_matrix(int n, bool inverse, uint16_t *img)
{
    const int h = n / 2;
    const long double edge = 1.0L / sqrtl((long double)n), mid = sqrtl(2.0L / (long double)n);
    long double t[3 * kTlMaxEdge];                 // cosines, sines, cosines of the end frequencies
    for (int m = 0; m < n; ++m) {
        t[m] = mid * cosl(kTwoPiL * m / n);
        t[n + m] = mid * sinl(kTwoPiL * m / n);
        t[2 * n + m] = edge * cosl(kTwoPiL * m / n);
    }
    int k[kTlMaxEdge], type[kTlMaxEdge];
    for (int a = 0; a < n; ++a) {
        bool sine;
        k[a] = real_freq(n, a, sine);
        type[a] = sine ? 1 : (k[a] == 0 || 2 * k[a] == n ? 2 : 0);
    }
    return pack_matrix(n, t, 3 * n, [&](int half, int out, int in) {
        const int a = (inverse ? in : out) + half * h, j = inverse ? out : in;
        return (size_t)type[a] * n + (size_t)(k[a] * j) % n;
    }, img);
}

cudaError_t tline_smem_limits()
{
    return cudaFuncSetAttribute(k_tline, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTlSmemMax);
}

namespace {

TlJob make_job(const GridInfo &g, int axis, const TlMat &m, const float2 *in, float2 *out, int direct_in, int direct_out)
{
    const long long plane = (long long)g.ny * g.nz;
    const int n = axis == 0 ? g.nx : (axis == 1 ? g.ny : g.nz);
    TlJob j{};
    j.sh = tl_shape(n);
    j.nlines = (int)(g.N / n);
    j.tiles = (j.nlines + kLines - 1) / kLines;
    j.zaxis = axis == 2;
    j.zlen = axis == 0 ? (int)plane : (axis == 1 ? g.nz : 1);
    j.ostride = axis == 2 ? g.nz : plane;                // (x: one outer index)
    j.rstride = axis == 0 ? plane : (axis == 1 ? g.nz : 1);
    j.direct_in = direct_in;
    j.direct_out = direct_out;
    j.mexp = m.mexp;
    j.mat = (const unsigned char *)m.img;
    j.in = in;
    j.out = out;
    return j;
}

}  // namespace

void launch_tline(const GridInfo &g, int count, const TlPass *pass, cudaStream_t st)
{
    TlJobs jobs{};
    int blocks = 0, items = 0;
    uint32_t smem = 0;
    for (int i = 0; i < count; ++i) {
        const TlPass &p = pass[i];
        TlJob &j = jobs.job[jobs.count++];
        j = make_job(g, p.axis, *p.mat, p.in, p.out, p.kind == TlPass::kInverse, p.kind == TlPass::kForward);
        blocks += j.tiles;
        items = std::max(items, kLines * j.sh.nc);
        smem = std::max(smem, j.sh.smem);
    }
    if (blocks == 0) return;
    pdl_launch(k_tline, blocks, items + 32, smem, st, jobs);
}

}  // namespace ofdft
