// Local-pseudopotential forces (Eq. (M12)) on the tensor cores, orthorhombic
// double-float contexts.
//
// In the real Fourier basis v_ext of an ion at R has the coefficients Z N w(k)
// f_a(X) f_b(Y) f_c(Z) (f: the cosine or sine of each axis's frequency), so
//   F_I = Z_I grad sum_abc g[a][b][c] f_a(X) f_b(Y) f_c(Z),
//   g = -Omega w(k) n_abc,
// with n_abc the cosine and sine coefficients of n.  The sum over c of every
// row (a, b) for every ion, and the same with f_c' for the z force, is a
// contraction (rows x nz x ions, 2 N nat products): the double-float kernel
// took 34.3 ms for 1024 ions at 256^3, bound by instruction issue.  Here the
// phases f_c, f_c' of 64 ions over 64 values of c stay in shared memory as
// exact f16 digits (A), rows of g are cut into digits 32 at a time (B), and a
// tile's accumulators T, T' hold ions in lanes and rows in columns, so that
// each thread sums its ion's f_b T and f_b' T over the rows without
// shuffles.  Digits and accumulators as in kernels_tline.cu.
//
// Blocks: (64 ions x 64 c) x row splits; warps 0-7 read out (two halves of a
// tile's columns), 8-11 convert, 12 issues; two tiles in flight.  Measured
// (GB300): 1024 ions at 256^3 2.9 ms, with the coefficients 0.48 and the
// phases and corners 0.17 (the double-float kernel 34.3); 512 ions at 192^3
// 0.55 ms with the tensor pipe 61 % and the issue slots 59 % active.
#include <algorithm>

#include "digits.cuh"
#include "kernels.h"
#include "pdl.cuh"
#include "tcgen.cuh"

namespace ofdft {

namespace {

constexpr int kIons = 64, kKc = 64, kRows = 32;
constexpr uint32_t kALbo = (kIons + 1) * 16, kADig = kKc / 8 * kALbo, kAHalf = kDig * kADig;
constexpr uint32_t kImage = 2 * kAHalf;                        // f, f' of one (ion group, c block)
constexpr int kAcc = kDig + 1;                                 // accumulators: one weight more for T'
constexpr uint32_t kBLbo = kAcc * kRows * 16 + 16, kBBuf = kKc / 8 * kBLbo;
constexpr uint32_t kForceSmem = kImage + 2 * kBBuf;
constexpr int kReadWarps = 8, kConvThreads = 128, kForceThreads = kReadWarps * 32 + kConvThreads + 32;

struct ForceLayout {
    int groups, kblocks, splits, natp;
    size_t image, tx, ty, bytes;   // offsets; total
};

ForceLayout force_layout(const GridInfo &g, int nat)
{
    ForceLayout f;
    f.groups = (nat + kIons - 1) / kIons;
    f.kblocks = (g.nz + kKc - 1) / kKc;
    f.natp = f.groups * kIons;
    const int tiles = g.nx * ((g.ny + kRows - 1) / kRows), ab = f.groups * f.kblocks;
    // Up to three waves of the 152 SMs (one block an SM); at least two tiles a
    // block, and eight once that fills the SMs.
    const int most = std::max(1, 3 * 152 / ab), fill = std::max(1, 152 / ab);
    f.splits = std::max(std::min(fill, std::max(1, tiles / 2)), std::min(most, std::max(1, tiles / 8)));
    f.image = 0;
    f.tx = f.image + (size_t)ab * kImage;
    f.ty = f.tx + (size_t)g.nx * f.natp * sizeof(float4);
    f.bytes = f.ty + (size_t)g.ny * f.natp * sizeof(float4);
    return f;
}

// Cosine (c = 0 and odd c) or sine of frequency (c + 1) / 2 at an ion, from
// its phase table p[k] = exp(-i k theta), and the derivative per theta.
__device__ __forceinline__ void ion_phase(int c, const double2 *__restrict__ p, double &f, double &df)
{
    const bool sine = c > 0 && !(c & 1);
    const int k = (c + 1) / 2;
    const double2 e = p[k];
    f = sine ? -e.y : e.x;
    df = k * (sine ? e.x : e.y);
}

// f_c' enters divided by the block's highest frequency and times 7/4 (below
// 2^55: the leading digit still fits).  The fixed-point errors of T' are
// relative to that frequency while its sum comes from lower ones, so T' keeps
// the products of one weight more than T, and rows of g an eighth digit (in
// units of 2^-60 of the row's largest value, which is often the coefficient of
// frequency 0, whose f' is zero).  Error of the forces along x, y, z in 1e-15
// Ha/bohr rms, 64 ions at 64^3: 1.9, 1.6, 1.7; with seven digits 1.9, 1.6,
// 2.5; the double-float kernel 2.1, 1.8, 2.0.
__host__ __device__ __forceinline__ double block_top(int nz, int kb) { return 0.5 * min((kb + 1) * kKc, nz) / 1.75; }

// The coefficients on two or three Nyquist frequencies, whose phases do not
// factor by axis: dv/dR is the mean over G and its partner G' (the Nyquist
// components of opposite sign), summed in binary64 over the half spectrum's
// lines; a warp per ion.  The last of the chunks of part.
__device__ void corners(const GridInfo &g, int I, const double *__restrict__ Z, const double2 *__restrict__ px,
                        const double2 *__restrict__ py, const double2 *__restrict__ pz, const double2 *__restrict__ nG,
                        int nchunk, double *__restrict__ part)
{
    const int lane = threadIdx.x & 31;
    double F[3] = {0.0, 0.0, 0.0};
    const int hx = g.nx / 2, hy = g.ny / 2, hz = g.nz / 2;
    for (int i = lane; i < g.K + g.ny + g.nx; i += 32) {
        // (hx, hy, kz); (hx, y, hz) and (x, hy, hz) without the first's last point
        int x = hx, y = hy, z = hz;
        if (i < g.K) z = i;
        else if (i < g.K + g.ny) y = i - g.K;
        else x = i - g.K - g.ny;
        if (i >= g.K && x == hx && y == hy) continue;
        const bool qx = x == hx, qy = y == hy, qz = z == hz;
        const double2 a = px[(size_t)I * g.nx + x], b = py[(size_t)I * g.ny + y], c = pz[(size_t)I * g.K + z];
        const double kx = (x <= hx ? x : x - g.nx) * g.bx, ky = (y <= hy ? y : y - g.ny) * g.by, kz = z * g.bz;
        const double s = -0.5 * g.omega * (z == 0 || qz ? 1.0 : 2.0) * lpp_w(g, kx * kx + ky * ky + kz * kz);
        const double2 n = nG[((size_t)x * g.ny + y) * g.K + z];
        double e[2];                                   // Im(conj(n) P), Im(conj(n) P')
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const double ay = p && qx ? -a.y : a.y, by = p && qy ? -b.y : b.y, cy = p && qz ? -c.y : c.y;
            const double re = a.x * b.x - ay * by, im = a.x * by + ay * b.x;
            e[p] = s * (n.x * (re * cy + im * c.x) - n.y * (re * c.x - im * cy));
        }
        F[0] += kx * (qx ? e[0] - e[1] : e[0] + e[1]);
        F[1] += ky * (qy ? e[0] - e[1] : e[0] + e[1]);
        F[2] += kz * (qz ? e[0] - e[1] : e[0] + e[1]);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        for (int o = 16; o > 0; o >>= 1) F[a] += __shfl_down_sync(0xffffffffu, F[a], o);
        if (lane == 0) part[((size_t)I * nchunk + nchunk - 1) * 3 + a] = Z[I] * F[a];
    }
}

// The A images (f_c and f_c' / block_top, times 2^54), eight c
// a thread, and the pairs (f, f') of the x and y coefficients; the first
// blocks sum the corners.
__global__ void k_force_phases(GridInfo g, int nat, int natp, int kblocks, const double *Z,
                               const double2 *px, const double2 *py,
                               const double2 *pz, const double2 *nG, unsigned char *image,
                               float4 *tx, float4 *ty, int nchunk, double *part)
{
    pdl_enter();
    const int ncorner = (nat + 3) / 4;
    if (blockIdx.x < ncorner) {
        const int I = blockIdx.x * 4 + (threadIdx.x >> 5);
        if (I < nat) corners(g, I, Z, px, py, pz, nG, nchunk, part);
        return;
    }
    const int zc = kblocks * (kKc / 8), total = natp * (zc + g.nx + g.ny);
    for (int i = (blockIdx.x - ncorner) * blockDim.x + threadIdx.x; i < total; i += (gridDim.x - ncorner) * blockDim.x) {
        const int I = i % natp, j = i / natp;
        if (j < zc) {
            uint64_t q[8], d[8];
            const double sz = 18014398509481984.0 / block_top(g.nz, j / (kKc / 8));
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int c = j * 8 + t;
                double f = 0.0, df = 0.0;
                if (I < nat && c < g.nz) ion_phase(c, pz + (size_t)I * g.K, f, df);
                q[t] = (uint64_t)(long long)rint(f * 18014398509481984.0) + kDigBias;
                d[t] = (uint64_t)(long long)rint(df * sz) + kDigBias;
            }
            unsigned char *dst = image + ((size_t)(I / kIons) * kblocks + j / (kKc / 8)) * kImage + (j % (kKc / 8)) * kALbo +
                                 (I % kIons) * 16;
            store_digits(q, dst, kADig);
            store_digits(d, dst + kAHalf, kADig);
        } else {
            const bool y = j >= zc + g.nx;
            const int a = y ? j - zc - g.nx : j - zc;
            double f = 0.0, df = 0.0;
            if (I < nat) ion_phase(a, y ? py + (size_t)I * g.ny : px + (size_t)I * g.nx, f, df);
            const ff::f2 u = ff::from_double(f), v = ff::from_double(df);
            (y ? ty : tx)[(size_t)a * natp + I] = make_float4(u.hi, u.lo, v.hi, v.lo);
        }
    }
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__global__ void __launch_bounds__(kForceThreads, 1)
    k_force(GridInfo g, int nat, int natp, int kblocks, const double *Z, const float2 *coef,
            const unsigned char *image, const float4 *tx, const float4 *ty,
            double *part)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    // A in place; B tile converted, its products done, its accumulators read (per buffer); scales written (four tiles deep)
    __shared__ __align__(8) uint64_t s_bar[1 + 2 + 2 + 2 + 4];
    __shared__ uint32_t s_tmem;
    __shared__ float s_scale[4][kRows];
    __shared__ int s_bad;
    const uint32_t b_a = tc::smem_addr(s_bar), b_full = b_a + 8, b_done = b_full + 16, b_read = b_done + 16, b_scale = b_read + 16;
    unsigned char *A = smraw, *B = smraw + kImage;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int group = blockIdx.x / kblocks, kb = blockIdx.x - group * kblocks;
    const int nbt = (g.ny + kRows - 1) / kRows, tiles = g.nx * nbt;
    pdl_wait();
    if (tid == 0) {
        s_bad = 0;
        tc::mbar_init(b_a, 1);
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(b_full + 8 * i, kConvThreads);
            tc::mbar_init(b_done + 8 * i, 1);
            tc::mbar_init(b_read + 8 * i, kReadWarps);
        }
        for (int i = 0; i < 4; ++i) tc::mbar_init(b_scale + 8 * i, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tc::mbar_expect(b_a, kImage);
        tc::bulk_load(tc::smem_addr(A), image + ((size_t)group * kblocks + kb) * kImage, kImage, b_a);
    }
    __syncwarp();
    if (warp == 0) tc::tmem_alloc(tc::smem_addr(&s_tmem), 512);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    pdl_trigger();                                     // the block has its tensor memory: see pdl.cuh
    const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);

    if (warp < kReadWarps) {
        // lanes 0-15: T of the quarter's 16 ions, lanes 16-31: T' of the same
        const int half = lane >> 4, quarter = warp & 3, set = warp >> 2;
        const int I = group * kIons + quarter * 16 + (lane & 15);
        const ff::f2 z0(0.0f, 0.0f);
        ff::f2 F1 = z0, F2 = z0;
        bool good = true;
        int it = 0;
        for (int t = blockIdx.y; t < tiles && good; t += gridDim.y, ++it) {
            const int a = t / nbt, b0 = (t - a * nbt) * kRows, buf = it & 1;
            const float4 fa = tx[(size_t)a * natp + I];
            good = tc::mbar_wait(b_scale + 8 * (it & 3), (it >> 2) & 1) && tc::mbar_wait(b_done + 8 * buf, (it >> 1) & 1);
            tc::fence_after_sync();
            ff::f2 S1 = z0, S2 = z0;
#pragma unroll 1
            for (int c0 = set * 16; c0 < set * 16 + 16; c0 += 8) {
                float v[kAcc][8];
                const uint32_t at = tmem + ((uint32_t)(quarter * 32) << 16) + buf * (kAcc * kRows) + c0;
#pragma unroll
                for (int d = 0; d < kAcc; ++d) tc::tmem_ld8(at + d * kRows, v[d]);
                tc::tmem_wait_ld();
#pragma unroll
                for (int d = 0; d < kAcc; ++d) tc::pin8(v[d]);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int b = b0 + c0 + i;
                    float x[kAcc];
#pragma unroll
                    for (int d = 0; d < kDig; ++d) x[d] = v[d][i];
                    x[kDig] = half ? v[kDig][i] : 0.0f;    // T has none
                    const float2 y = scaled(combine(x), s_scale[it & 3][c0 + i]);
                    const ff::f2 T(y.x, y.y);
                    const float4 f = b < g.ny ? ty[(size_t)b * natp + I] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    S1 += ff::mul(ff::f2(f.x, f.y), T);
                    S2 += ff::mul(ff::f2(f.z, f.w), T);
                }
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(b_read + 8 * buf);
            // x force: f_a' sum f_b T; y: f_a sum f_b' T; z: f_a sum f_b T'
            F1 += ff::mul(half ? ff::f2(fa.x, fa.y) : ff::f2(fa.z, fa.w), S1);
            F2 += ff::mul(ff::f2(fa.x, fa.y), S2);
        }
        if (!good) s_bad = 1;
        __syncthreads();
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        if (I < nat) {
            const size_t nchunk = (size_t)kblocks * gridDim.y * 2 + 1;
            double *p = part + ((size_t)I * nchunk + ((size_t)kb * gridDim.y + blockIdx.y) * 2 + set) * 3;
            const double z = s_bad ? nan : Z[I];
            if (half) {
                p[2] = z * g.bz * block_top(g.nz, kb) * ff::to_double(F1);
            } else {
                p[0] = z * g.bx * ff::to_double(F1);
                p[1] = z * g.by * ff::to_double(F2);
            }
        }
    } else if (warp < kReadWarps + kConvThreads / 32) {
        // thread = (row, 16 of the 64 coefficients)
        const int ct = tid - kReadWarps * 32, row = ct >> 2, part4 = ct & 3;
        bool good = true;
        int it = 0;
        for (int t = blockIdx.y; t < tiles && good; t += gridDim.y, ++it) {
            const int a = t / nbt, b = (t - a * nbt) * kRows + row, buf = it & 1;
            const int c0 = kb * kKc + part4 * 16;
            const float2 *src = coef + ((size_t)a * g.ny + b) * g.nz + c0;
            float2 v[16];
            if (b < g.ny && c0 + 16 <= g.nz) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 x = reinterpret_cast<const float4 *>(src)[i];   // nz and c0 are even: 16-byte aligned
                    v[2 * i] = make_float2(x.x, x.y);
                    v[2 * i + 1] = make_float2(x.z, x.w);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = b < g.ny && c0 + i < g.nz ? src[i] : make_float2(0.0f, 0.0f);
            }
            uint32_t m = 27u << 23;                        // 2^-100: the least exponent of the scale
#pragma unroll
            for (int i = 0; i < 16; ++i) m = max(m, __float_as_uint(v[i].x) & 0x7fffffffu);
            m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
            m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
            const uint32_t e = m >> 23;
            const float u = ff::int_bits_float(e == 254u ? 0x400000u : (254u - e) << 23);
            if (it >= 2) good = tc::mbar_wait(b_done + 8 * buf, ((it >> 1) - 1) & 1);
            // weight 1 stands for 2^96 times the units 2^-54 and 2^(E - 52)
            if (part4 == 0)
                s_scale[it & 3][row] = m >= 0x7f800000u ? __uint_as_float(0x7fc00000u) : ff::pow2i((int)e - 127 - 10);
            unsigned char *dst = B + buf * kBBuf + part4 * 2 * kBLbo + row * 16;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint64_t q[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) q[i] = to_fixed<60>(v[8 * h + i], u) + (kDigBias8 - fixed_off<60>());
                store_digits<8>(q, dst + h * kBLbo, kRows * 16);
            }
            tc::fence_async();
            mbar_arrive(b_full + 8 * buf);
        }
        if (!good) s_bad = 1;
        __syncthreads();
    } else {
        const uint32_t sa = tc::smem_addr(A), sb = tc::smem_addr(B);
        bool good = tc::mbar_wait(b_a, 0);
        int it = 0;
        for (int t = blockIdx.y; t < tiles && good; t += gridDim.y, ++it) {
            const int buf = it & 1;
            good = tc::mbar_wait(b_full + 8 * buf, (it >> 1) & 1);
            if (it >= 2) good = tc::mbar_wait(b_read + 8 * buf, ((it >> 1) - 1) & 1) && good;
            if (lane == 0) mbar_arrive(b_scale + 8 * (it & 3));
            __syncwarp();
            tc::fence_after_sync();
            const uint64_t b0 = tc::operand(sb + buf * kBBuf, kBLbo, 128);
#pragma unroll 1
            for (int p = 0; p < 2; ++p) {                  // f, f'
                const uint64_t a0 = tc::operand(sa + p * kAHalf, kALbo, 128);
                const uint32_t acc = tmem + ((uint32_t)p << 20) + buf * (kAcc * kRows);
#pragma unroll
                for (int i = 0; i < kDig; ++i)
#pragma unroll
                    for (int k = 0; k < kKc / 16; ++k)
                        tc::mma_f16(acc + i * kRows, a0 + ((i * kADig + k * 2 * kALbo) >> 4), b0 + ((k * 2 * kBLbo) >> 4),
                                    tc::idesc_f16(64, (kDig - i + p) * kRows), (i | k) != 0);
            }
            tc::mma_commit(b_done + 8 * buf);
        }
        // nothing in flight when the tensor memory is given back
        if (it > 0) good = tc::mbar_wait(b_done + 8 * ((it - 1) & 1), ((it - 1) >> 1) & 1) && good;
        if (!good) s_bad = 1;
        __syncthreads();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

}  // namespace

// Its three launches and their set-up cost more than the double-float kernel's
// sums on small grids.  Forces with their evaluation, double-float -> here:
// 20^3, 8 ions 130 -> 140 us; 40^3, 8 154 -> 158, 54 163 -> 160, 128 178 ->
// 160; 64^3, 4 226 -> 206; 96^3, 8 370 -> 303, 128 535 -> 318; 180^3, 8 1554
// -> 1137.
bool force_tc_takes(const GridInfo &g, int nat) { return g.dd && !g.tri && (long long)g.nx * g.ny * g.nz * ((nat + 31) / 32 * 32) >= 4000000; }

size_t force_tc_bytes(const GridInfo &g, int nat) { return force_layout(g, nat).bytes; }

int force_tc_chunks(const GridInfo &g, int nat)
{
    const ForceLayout f = force_layout(g, nat);
    return f.kblocks * f.splits * 2 + 1;
}

int launch_force_tc(const GridInfo &g, int nat, const double *Z, const double2 *px, const double2 *py, const double2 *pz,
                    const double2 *nG, const float2 *coef, void *scratch, double *part, cudaStream_t st)
{
    const ForceLayout f = force_layout(g, nat);
    unsigned char *s = (unsigned char *)scratch;
    float4 *tx = (float4 *)(s + f.tx), *ty = (float4 *)(s + f.ty);
    const int total = f.natp * (f.kblocks * (kKc / 8) + g.nx + g.ny), nchunk = force_tc_chunks(g, nat);
    pdl_launch(k_force_phases, (nat + 3) / 4 + std::min((total + 127) / 128, 4864), 128, 0, st, g, nat, f.natp, f.kblocks, Z, px, py,
               pz, nG, s + f.image, tx, ty, nchunk, part);
    pdl_launch(k_force, dim3(f.groups * f.kblocks, f.splits), kForceThreads, kForceSmem, st, g, nat, f.natp, f.kblocks, Z, coef,
               s + f.image, tx, ty, part);
    return nchunk;
}

cudaError_t force_tc_smem_limits()
{
    return cudaFuncSetAttribute(k_force, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kForceSmem);
}

}  // namespace ofdft
