// Allocation-free energy and potential: ofdft_energy_potential_static.
//
// Same arithmetic and kernels as ofdft_setup + ofdft_energy_potential, but all
// device scratch (fields, local potential, phases, reduction partials,
// transform matrices, temperature table) lives in one file-scope __device__
// array, so a call allocates nothing.  Callers that cannot allocate device memory (tight
// loops where cudaMalloc could synchronise the GPU, or programs whose device
// memory belongs to another allocator) pass their own phi and v buffers.
//
// Host code reaches the array only through the address cudaGetSymbolAddress
// returns for the current device (the symbol itself is a host-side stand-in).
// The first call on a device does that lookup and uploads the tables
// and matrices, under a mutex, so first calls from several host threads do not race
// on the host.  Every call reuses the same array; calls that overlap on the
// GPU race.
#include <math.h>
#include <string.h>

#include <mutex>

#include "kernels.h"
#include "pointwise.cuh"

using namespace ofdft;

namespace {

// Limits of the static path.
constexpr int kSMaxEdge = kStaticEdge;
constexpr long long kSMaxN = 32768;
constexpr int kSMaxAtoms = kStaticAtoms;
constexpr long long kSMaxPart = 3LL * kSMaxEdge * 5 + 15LL * (kSMaxN / 16) + 64;

constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Byte offsets inside the scratch array.
constexpr size_t kFieldBytes = align256((size_t)kSMaxN * sizeof(float2));   // a field of pairs: n's coefficients, three derivatives
constexpr size_t kOffVre = 4 * kFieldBytes;                                 // v_ext's coefficients
constexpr size_t kOffVpart = kOffVre + kFieldBytes;                         // n, then v_part
constexpr size_t kOffT = kOffVpart + kFieldBytes;
constexpr size_t kOffEg = kOffT + align256((size_t)kSMaxAtoms * (3 * kSMaxEdge + 3) * sizeof(float2));
constexpr size_t kOffG2 = kOffEg + align256(3 * kSMaxEdge * sizeof(double2));
constexpr size_t kOffIons = kOffG2 + align256(3 * kSMaxEdge * sizeof(float2));
constexpr size_t kOffZ = kOffIons + align256(3 * kSMaxAtoms * sizeof(double));
constexpr size_t kOffFrac = kOffZ + align256(kSMaxAtoms * sizeof(double));
constexpr size_t kOffPart = kOffFrac + align256(3 * kSMaxAtoms * sizeof(float));
constexpr size_t kOffScal = kOffPart + align256((size_t)kSMaxPart * sizeof(double));
constexpr int kEdges[] = {8, 10, 12, 16, 18, 20, 24, 30, 32, 36, 40, 48, 50, 54, 60, 64};   // the path takes
constexpr size_t kOffEwTab = kOffScal + align256(64 * sizeof(double));
constexpr size_t kOffEwPart = kOffEwTab + align256((size_t)kEwTabRows * kSMaxAtoms * sizeof(double2));
// tensor-core matrices of every edge: derivative per lattice period, forward
// and inverse real Fourier transform
constexpr size_t kMatBytes = 768 * 1024;
constexpr size_t kOffMat = kOffEwPart + align256(kEwBlocks * sizeof(double));
constexpr size_t kOffTab = kOffMat + kMatBytes;
constexpr size_t kScratchBytes = kOffTab + align256((size_t)kDdTabSize * sizeof(double));   // + splits

static __device__ __align__(256) unsigned char g_ofdft_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
struct DevState {
    bool ready;
    unsigned char *base;
};
DevState g_dev[kMaxDevices];
double g_tab_host[kDdTabSize];    // host temperature table + double-float tables, filled once
struct EdgeMats {                 // transform matrices, filled once
    size_t at[3];                 // offsets in the matrices' block
    int mexp[3];
} g_mat[sizeof(kEdges) / sizeof(kEdges[0])];
unsigned char g_mat_host[kMatBytes];
bool g_tab_ready = false;
std::mutex g_setup_mu;            // guards g_dev, g_tab_host, g_mat, g_mat_host and g_tab_ready (locking allocates nothing)

// The matrices of every edge, filled once with the other tables.
bool matrices_fill()
{
    size_t at = 0;
    for (size_t i = 0; i < sizeof(kEdges) / sizeof(kEdges[0]); ++i) {
        const int n = kEdges[i];
        for (int k = 0; k < 3; ++k) {
            const size_t b = align256(tline_matrix_bytes(n));
            if (!tline_supported(n) || at + b > kMatBytes) return false;
            uint16_t *img = (uint16_t *)(g_mat_host + at);
            g_mat[i].at[k] = at;
            g_mat[i].mexp[k] = k == 0 ? tline_derivative_matrix(n, 1.0, img) : tline_fourier_matrix(n, k == 2, img);
            at += b;
        }
    }
    return true;
}

TlAxis axis_matrices(int n, unsigned char *dev)
{
    TlAxis a;
    TlMat *m[3] = {&a.der, &a.fwd, &a.inv};
    for (size_t i = 0; i < sizeof(kEdges) / sizeof(kEdges[0]); ++i)
        if (kEdges[i] == n)
            for (int k = 0; k < 3; ++k) {
                m[k]->img = dev + g_mat[i].at[k];
                m[k]->mexp = g_mat[i].mexp[k];
            }
    return a;
}

// Status only: the documented limits say what OFDFT_EINVAL means here.
ofdft_status serr(ofdft_status s, const char *, cudaError_t = cudaSuccess) { return s; }

#define SCK(call, what)                                            \
    do {                                                           \
        cudaError_t e_ = (call);                                   \
        if (e_ != cudaSuccess) return serr(OFDFT_EDEVICE, what, e_); \
    } while (0)

bool edge_ok(int n)
{
    if (n < 8 || n > kSMaxEdge || (n & 1)) return false;
    for (int p : {2, 3, 5})
        while (n % p == 0) n /= p;
    return n == 1;
}

// One-time set-up on the current device: scratch address, tables, smem limits.
// The uploads run on the caller's stream and are waited for: a copy from
// pageable memory may return before its data have arrived, and a later call
// may come on any stream.
ofdft_status device_setup(int dev, cudaStream_t st, unsigned char **base)
{
    if (dev < 0 || dev >= kMaxDevices) return serr(OFDFT_EINVAL, "device ordinal out of range");
    std::lock_guard<std::mutex> lk(g_setup_mu);
    DevState &d = g_dev[dev];
    if (!d.ready) {
        void *p = nullptr;
        SCK(cudaGetSymbolAddress(&p, g_ofdft_scratch), "cudaGetSymbolAddress of the static scratch failed");
        d.base = (unsigned char *)p;
        if (!g_tab_ready) {
            static double ttab[kTfSize];
            tfunc_table_fill(ttab);
            dd_tables_fill(ttab, g_tab_host);
            if (!matrices_fill()) return serr(OFDFT_EDEVICE, "no transform matrices");
            g_tab_ready = true;
        }
        SCK(cudaMemcpyAsync(d.base + kOffTab, g_tab_host, sizeof(g_tab_host), cudaMemcpyHostToDevice, st),
            "temperature table upload failed");
        SCK(cudaMemcpyAsync(d.base + kOffMat, g_mat_host, sizeof(g_mat_host), cudaMemcpyHostToDevice, st),
            "matrix upload failed");
        SCK(cudaStreamSynchronize(st), "table upload failed");
        SCK(tline_smem_limits(), "shared-memory limit set-up failed");
        d.ready = true;
    }
    *base = d.base;
    return OFDFT_OK;
}

// Self and background terms of the Ewald energy.
double ewald_consts(const double L[3], int nat, const double *Z)
{
    const double pi = 3.14159265358979323846;
    const double om = L[0] * L[1] * L[2];
    const double a = 1.2 * sqrt(pi) * pow((double)nat / (om * om), 1.0 / 6.0);
    double z2 = 0.0, zs = 0.0;
    for (int I = 0; I < nat; ++I) {
        z2 += Z[I] * Z[I];
        zs += Z[I];
    }
    return -a / sqrt(pi) * z2 - pi * zs * zs / (2.0 * om * a * a);
}

// Textbook Ewald sums on the host, no heap: real-space erfc sum and
// reciprocal sum over the box of G with |G| < gcut (cells too uneven for
// launch_static_ions's tables).
double ewald_host(const double L[3], int nat, const double *R, const double *Z)
{
    const double pi = 3.14159265358979323846;
    double om = L[0] * L[1] * L[2];
    double a = 1.2 * sqrt(pi) * pow((double)nat / (om * om), 1.0 / 6.0);
    double rcut = 6.3 / a, gcut = 2.0 * a * 6.3;
    int ni[3], km[3];
    for (int k = 0; k < 3; ++k) {
        ni[k] = (int)ceil(rcut / L[k] + 0.5);
        km[k] = (int)ceil(gcut * L[k] / (2.0 * pi));
    }
    double E = 0.0;
    for (int I = 0; I < nat; ++I)
        for (int J = 0; J < nat; ++J) {
            double d0[3];
            for (int k = 0; k < 3; ++k) {
                d0[k] = R[3 * I + k] - R[3 * J + k];
                d0[k] -= L[k] * rint(d0[k] / L[k]);
            }
            for (int i = -ni[0]; i <= ni[0]; ++i)
                for (int j = -ni[1]; j <= ni[1]; ++j)
                    for (int k = -ni[2]; k <= ni[2]; ++k) {
                        double dx = d0[0] - i * L[0], dy = d0[1] - j * L[1], dz = d0[2] - k * L[2];
                        double r2 = dx * dx + dy * dy + dz * dz;
                        if (r2 < 1e-24 || r2 >= rcut * rcut) continue;
                        double r = sqrt(r2);
                        E += 0.5 * Z[I] * Z[J] * erfc(a * r) / r;
                    }
        }
    for (int i = -km[0]; i <= km[0]; ++i)
        for (int j = -km[1]; j <= km[1]; ++j)
            for (int k = -km[2]; k <= km[2]; ++k) {
                double gx = 2 * pi * i / L[0], gy = 2 * pi * j / L[1], gz = 2 * pi * k / L[2];
                double g2 = gx * gx + gy * gy + gz * gz;
                if (g2 == 0.0 || g2 >= gcut * gcut) continue;
                double sr = 0.0, si = 0.0;
                for (int I = 0; I < nat; ++I) {
                    double ph = gx * R[3 * I] + gy * R[3 * I + 1] + gz * R[3 * I + 2];
                    sr += Z[I] * cos(ph);
                    si += Z[I] * sin(ph);
                }
                E += 2.0 * pi / om * exp(-g2 / (4.0 * a * a)) / g2 * (sr * sr + si * si);
            }
    return E;
}

}  // namespace

extern "C" ofdft_status ofdft_energy_potential_static(const double cell[9], const int grid[3], int nat,
                                                      const double *ions, const double *Z, double T_kelvin,
                                                      int functional, int xc, double rc,
                                                      const double *phi_dev, double *v_dev,
                                                      ofdft_energy *E, void *stream)
{
    if (!cell || !grid || !ions || !Z || !phi_dev || !v_dev)
        return serr(OFDFT_EINVAL, "NULL argument");
    if ((((uintptr_t)phi_dev) | ((uintptr_t)v_dev)) & 15)
        return serr(OFDFT_EINVAL, "phi_dev and v_dev must be 16-byte aligned");
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            if (i != j && cell[3 * i + j] != 0.0) return serr(OFDFT_EINVAL, "cell is not orthorhombic");
    if (!(cell[0] > 0 && cell[4] > 0 && cell[8] > 0)) return serr(OFDFT_EINVAL, "non-positive cell edge");
    for (int a = 0; a < 3; ++a)
        if (!edge_ok(grid[a]))
            return serr(OFDFT_EINVAL, "static path: grid edges must be even, {2,3,5}-smooth, 8..64");
    long long N = (long long)grid[0] * grid[1] * grid[2];
    if (N > kSMaxN) return serr(OFDFT_EINVAL, "static path: nx*ny*nz exceeds 32768 grid points");
    if (nat <= 0 || nat > kSMaxAtoms) return serr(OFDFT_EINVAL, "static path: nat must be in 1..64");
    if (!(T_kelvin > 0.0) || !isfinite(T_kelvin) || !(rc > 0.0) || !isfinite(rc))
        return serr(OFDFT_EINVAL, "temperature and rc must be finite and > 0");
    for (int i = 0; i < nat; ++i) {   // the per-ion checks of ofdft_setup
        if (!(Z[i] > 0.0) || !isfinite(Z[i])) return serr(OFDFT_EINVAL, "ion charges must be finite and > 0");
        for (int k = 0; k < 3; ++k)
            if (!isfinite(ions[3 * i + k])) return serr(OFDFT_EINVAL, "ion positions must be finite");
    }
    FuncParams fp = functional_params(functional);
    if (fp.kind < 0) return serr(OFDFT_EINVAL, "unknown functional");
    cudaStream_t st = (cudaStream_t)stream;
    {
        // the call copies to host memory and synchronises: not capturable
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone)
            return serr(OFDFT_EINVAL, "the stream is being captured");
    }
    int dev = 0;
    SCK(cudaGetDevice(&dev), "cudaGetDevice failed");
    unsigned char *base = nullptr;
    ofdft_status s = device_setup(dev, st, &base);
    if (s != OFDFT_OK) return s;

    GridInfo g{};
    g.nx = grid[0];
    g.ny = grid[1];
    g.nz = grid[2];
    g.K = g.nz / 2 + 1;
    g.N = N;
    g.NH = (long long)g.nx * g.ny * g.K;
    g.Lx = cell[0];
    g.Ly = cell[4];
    g.Lz = cell[8];
    g.omega = g.Lx * g.Ly * g.Lz;
    g.dV = g.omega / (double)N;
    g.rc = rc;
    grid_reciprocal(g);
    g.dd = 1;   // double-float transforms and pointwise arithmetic, as ofdft_setup's default
    const double T = T_kelvin * 3.166811563e-6;

    // ions -> tables -> Ewald sums and v_ext
    const double L[3] = {g.Lx, g.Ly, g.Lz};
    StaticIons arg;
    memcpy(arg.R, ions, 3 * nat * sizeof(double));
    memcpy(arg.Z, Z, nat * sizeof(double));
    for (int i = 0; i < 3 * nat; ++i) {
        const double f = ions[i] / L[i % 3];
        arg.frac[i] = (float)(f - floor(f));
    }
    StaticIonTables it;
    it.R = (double *)(base + kOffIons);
    it.Z = (double *)(base + kOffZ);
    it.frac = (float *)(base + kOffFrac);
    it.t = (float2 *)(base + kOffT);
    it.eg = (double2 *)(base + kOffEg);
    it.g2 = (float2 *)(base + kOffG2);
    it.ewtab = (double2 *)(base + kOffEwTab);
    it.ewpart = (double *)(base + kOffEwPart);
    float2 *vre = (float2 *)(base + kOffVre);
    const int newald = launch_static_ions(g, nat, arg, it, vre, st);

    const double *tab = (const double *)(base + kOffTab);
    double *scal = (double *)(base + kOffScal);   // 18 sums of the evaluation, then the Ewald sum
    double *vpart = (double *)(base + kOffVpart);
    double *pA = (double *)(base + kOffPart);
    const bool fttf = fp.kind == 0;
    // The context path's sequence in the real Fourier basis.  The matrices are
    // those of unit spacing, shared by all cells of an edge: the derivatives
    // are per lattice period, and the pointwise stage takes them (and gives the
    // fields of div W) through the reciprocal basis, as in a general cell.
    unsigned char *mat = base + kOffMat;
    const TlAxis tl[3] = {axis_matrices(g.nx, mat), axis_matrices(g.ny, mat), axis_matrices(g.nz, mat)};
    float2 *coef = (float2 *)base, *nf = (float2 *)vpart;
    double *d[3];
    TlPass grad[4], div[3];
    for (int a = 0; a < 3; ++a) {
        d[a] = (double *)(base + (a + 1) * kFieldBytes);
        grad[a] = {TlPass::kDerivative, a, &tl[a].der, nf, (float2 *)d[a]};
        div[a] = {TlPass::kDerivative, a, &tl[a].der, (float2 *)d[a], (float2 *)d[a]};
    }
    const TlPass zf = {TlPass::kForward, 2, &tl[2].fwd, nf, coef};
    grad[3] = zf;
    launch_density(g.N, phi_dev, nullptr, 1.0, 0.0, nullptr, nullptr, nf, st);
    launch_tline(g, fttf ? 1 : 4, fttf ? &zf : grad, st);
    for (int a = 1; a >= 0; --a) {
        const TlPass fwd = {TlPass::kForward, a, &tl[a].fwd, coef, coef};
        launch_tline(g, 1, &fwd, st);
    }
    TlHartree hl{};
    for (int a = 0; a < 3; ++a) hl.g2[a] = it.g2 + a * kSMaxEdge;
    hl.ve = vre;
    hl.hr = make_float2(g.hr2[0], g.hr2[1]);
    hl.half_dv = 0.5 * g.dV;
    hl.dv = g.dV;
    hl.ploc = g.dV / g.omega / 3.0;
    hl.part = pA;
    const int nbx = launch_hartree(g, coef, hl, st);
    for (int a = 0; a < 3; ++a) {
        const TlPass inv = {TlPass::kInverse, a, &tl[a].inv, coef, coef};
        launch_tline(g, 1, &inv, st);
    }
    // partial sums of the Hartree, the pointwise and the final stage
    double *pB = pA + 3 * nbx, *pC = pB + 6 * ((long long)g.nx * g.ny / 2);
    int nbg = 0, nbz;
    if (fttf) {
        nbz = launch_ptf(g, coef, phi_dev, nullptr, nullptr, 1.0, 0.0, nullptr, T, fp, tab, xc, v_dev, pC, st);
    } else {
        GridInfo gp = g;
        gp.tri = 1;
        for (int i = 0; i < 9; ++i) gp.Bm[i] = 0.0;
        gp.Bm[0] = g.bx;
        gp.Bm[4] = g.by;
        gp.Bm[8] = g.bz;
        nbg = launch_pw<double>(gp, d[0], d[1], d[2], phi_dev, T, fp, tab, xc, vpart, pB, false, st);
        launch_tline(g, 3, div, st);
        TlFinal fin{};
        fin.vhl = coef;
        fin.vpart = nf;
        for (int a = 0; a < 3; ++a) fin.d[a] = (const float2 *)d[a];
        fin.phit = phi_dev;
        fin.c = 1.0;
        fin.vout = v_dev;
        fin.part = pC;
        nbz = launch_final(g, fin, st);
    }
    launch_reduce_eval(pA, nbx, pB, nbg, pC, nbz, !fttf, scal, st, it.ewpart, newald);
    double h[19];
    SCK(cudaMemcpyAsync(h, scal, sizeof(h), cudaMemcpyDeviceToHost, st), "scalar read-back failed");
    SCK(cudaStreamSynchronize(st), "stream synchronisation failed");
    SCK(cudaGetLastError(), "kernel launch failed");

    const double *f = fttf ? h + 9 : h + 3;
    const double dV = g.dV, om = g.omega;
    double Ne = 0.0, zs = 0.0;
    for (int i = 0; i < nat; ++i) {
        Ne += Z[i];
        zs += 3.14159265358979323846 * Z[i] * rc * rc;
    }
    const double E_ion = (newald ? h[18] : ewald_host(L, nat, ions, Z)) + ewald_consts(L, nat, Z);
    ofdft_energy e;
    memset(&e, 0, sizeof(e));
    e.F_s = dV * f[0];
    e.minus_TS = -dV * f[1];
    e.E_H = h[0];
    e.E_loc = h[1];
    e.F_xc = dV * f[2];
    e.E_ion = E_ion;
    e.F_tot = e.F_s + e.E_H + e.E_loc + e.F_xc + e.E_ion;
    e.E_int = e.F_tot + dV * f[1];
    e.mu = h[15] / h[16];
    e.E_alphaZ = Ne * zs / om;
    e.P_s = (dV * f[3] + (4.0 / 3.0) * dV * (fttf ? 0.0 : f[4])) / om;
    e.P_xc = dV * f[5] / om;
    e.P_H = h[0] / (3.0 * om);
    e.P_loc = h[2];
    e.P_ion = E_ion / (3.0 * om);
    e.P = e.P_s + e.P_xc + e.P_H + e.P_loc + e.P_ion;
    if (!isfinite(e.F_tot + e.mu)) return serr(OFDFT_ENUMERIC, "non-finite energy or potential");
    if (E) *E = e;
    return OFDFT_OK;
}
