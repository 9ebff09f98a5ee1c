// Host-side launchers of the libofdft kernels (templated on the field type).
#pragma once

#include "ofdft_internal.h"

namespace ofdft {

// Frequency of real-Fourier coefficient a of an axis of n points, and whether
// it is the sine's: coefficients 0 .. n/2 - 1 are the even frequencies 0, 2
// (cosine, sine), 4, ..., the others the odd ones; the Nyquist frequency has
// a cosine only.
__host__ __device__ __forceinline__ int real_freq(int n, int a, bool &sine)
{
    const int h = n / 2;
    const bool odd = a >= h;
    const int i = odd ? a - h : a;
    sine = odd ? (i & 1) != 0 : (i > 0 && (i & 1) == 0);
    return odd ? 2 * (i / 2) + 1 : 2 * ((i + 1) / 2);
}

// Index of the cosine of frequency k (the sine's is the next).
__host__ __device__ __forceinline__ int real_cosine(int n, int k) { return (k & 1 ? n / 2 : 0) + (k > 0 ? k - 1 : 0); }

#ifdef __CUDACC__
// Local pseudopotential form factor per unit charge, 0 at G = 0.
// Gaussian ion: w(G) = -4 pi exp(-G^2 rc^2/4) / (Omega G^2).
// Heine-Abarenkov, Eq. (E4A), q = |G|, divided by the common charge Z:
// w(q) = -4 pi/(Omega q^2 Z) [(Z - A rc) cos(q rc) + (A/q) sin(q rc)] exp(-(q/qc)^6).
__device__ __forceinline__ double lpp_w(const GridInfo &g, double g2)
{
    if (!(g2 > 0.0)) return 0.0;
    if (g.lpp == 0) return -12.566370614359172954 * exp(-0.25 * g2 * g.rc * g.rc) / (g.omega * g2);
    const double q = sqrt(g2), u = q / g.ha_qc, u2 = u * u;
    double s, c;
    sincos(q * g.rc, &s, &c);
    const double B = (g.ha_Z - g.ha_A * g.rc) * c + g.ha_A * s / q;
    return -12.566370614359172954 * B * exp(-u2 * u2 * u2) / (g.omega * g2 * g.ha_Z);
}
#endif

// ---- grid fields (kernels_fields.cu)
// z pass, forward: n = phi^2 (mode 1), the trial rotation phi cos + dhat sin
// written to phit (mode 2) or a plain field (mode 0), R2C along z into the
// half spectrum out; with dz also d_z n into the real field dz, with nout
// also n.
template <typename T>
void launch_zfwd(const GridInfo &g, const FftAxis &az, int mode, const T *in, const T *phi,
                 const T *dhat, T c, T s, const void *cs, T *phit, cplx<T> *out, cudaStream_t st,
                 T *dz = nullptr, T *nout = nullptr);
// Derivative of a real field along grid axis 0 (x) or 1 (y) by 1-D
// transforms along that axis: out = d f, f = phi^2 for mode 0 and f = in for
// mode 1 (scale GridInfo::ds).  Derivative fields (this out, zfwd's dz,
// zfinal_gga's dx, dy, dz) are double-float pairs in a
// double-float grid (two binary32 words in a double's place).
template <typename T>
void launch_dline(const GridInfo &g, const FftAxis &fa, int axis, int mode, const T *in, T *out,
                  cudaStream_t st);
// ---- one-axis transforms on the tensor cores (kernels_tline.cu).  Fields
// and coefficients are double-float pairs (float2).
// A matrix's digits in device memory and their binary exponent.
struct TlMat {
    const void *img = nullptr;
    int mexp = 0;
};
// Matrices of one axis (null: the axis is too long, or not asked for) and
// (k b)^2 of its real-Fourier coefficients.
struct TlAxis {
    TlMat der, fwd, inv;
    const float2 *g2 = nullptr;
};
bool tline_supported(int n);
bool tline_derivative_supported(int n, double scale);
struct TlPlan {
    bool der[3];        // derivatives along the axis
    bool real_basis;    // the Hartree chain in the real Fourier basis
};
TlPlan tline_plan(const GridInfo &g, bool gga);
size_t tline_matrix_bytes(int n);
// Fill img (tline_matrix_bytes(n)) and return the exponent: the derivative
// times scale; the orthonormal real Fourier transform, or its inverse.
int tline_derivative_matrix(int n, double scale, uint16_t *img);
int tline_fourier_matrix(int n, bool inverse, uint16_t *img);
cudaError_t tline_smem_limits();
// Up to four transforms, each along one axis, in one launch; out may be in.
struct TlPass {
    enum Kind { kDerivative, kForward, kInverse } kind;
    int axis;
    const TlMat *mat;
    const float2 *in;
    float2 *out;
};
void launch_tline(const GridInfo &g, int count, const TlPass *pass, cudaStream_t st);
// coef: coefficients of n -> of v_HL = 4 pi n / G^2 + v_ext; partials E_H,
// E_loc, P_loc in three rows of the returned number of columns.
struct TlHartree {
    const float2 *g2[3];       // (k b)^2 per coefficient and axis (orthorhombic cells)
    const float2 *ve, *vp;     // v_ext's coefficients; pressure weights or null (Gaussian ion, orthorhombic cell)
    float2 hr;                 // rc^2 / 2
    double half_dv, dv, ploc;  // factors of the three sums
    double *part;
};
int launch_hartree(const GridInfo &g, float2 *coef, const TlHartree &hl, cudaStream_t st);
// v = v_HL + v_part - (d[0] + d[1] + d[2]), partials as launch_zfinal_gga.
struct TlFinal {
    const float2 *vhl, *vpart, *d[3];
    const double *phit, *phi, *dhat, *cs;
    double c, s, *vout, *part;
};
int launch_final(const GridInfo &g, const TlFinal &fin, cudaStream_t st);
// n = phi^2 (with dhat: of the trial phi c + dhat s, written to phit), as pairs.
void launch_density(long long n, const double *phi, const double *dhat, double c, double s, const double *cs,
                    double *phit, float2 *dens, cudaStream_t st);
// ftTF: v = v_HL + df/dn + v_xc; partials as launch_zfinal's.
int launch_ptf(const GridInfo &g, const float2 *vhl, const double *phit, const double *phi, const double *dhat, double c,
               double s, const double *cs, double temp, const FuncParams &fp, const double *tab, int xc, double *vout,
               double *part, cudaStream_t st);
// Real-Fourier coefficients (pairs) of the real field whose half spectrum is
// v (its Nyquist planes Hermitian).
void launch_real_coefficients(const GridInfo &g, const double2 *v, float2 *coef, cudaStream_t st);
// Pointwise functional + XC: reads phi and the derivatives of n in d0..d2,
// writes v_part and, over d0..d2, the fields U_j whose derivatives sum to
// div W.  Partials: 6 rows (12 with stress: sum W_a d_b n in rows 6..11, FP64
// sets only) of the returned number of columns.
template <typename T>
int launch_pw(const GridInfo &g, T *d0, T *d1, T *d2, const T *phit, T temp, const FuncParams &fp, const T *tab,
              int xc, T *vpart, double *part, bool stress, cudaStream_t st);
// z pass, final (ftTF): C2R of v_HL, pointwise functional, potential and sums.
template <typename T>
int launch_zfinal(const GridInfo &g, const FftAxis &az, bool fttf, const cplx<T> *dspec,
                  const T *vpart, const T *phit, const T *phi, const T *dhat, T c, T s,
                  const void *cs, T temp, const FuncParams &fp, const T *tab, int xc, T *vout,
                  double *part, cudaStream_t st);
// z pass, final (GGA): v = v_HL + v_part - dx - dy - d_z U_z; with uz null, dz
// is that last term.
template <typename T>
int launch_zfinal_gga(const GridInfo &g, const FftAxis &az, const cplx<T> *dspec, const T *uz, const T *vpart,
                      const T *dx, const T *dy, const T *dz, const T *phit, const T *phi, const T *dhat, T c,
                      T s, const void *cs, T *vout, double *part, cudaStream_t st);
template <typename T>
void launch_ypass(const GridInfo &g, const FftAxis &ay, bool inv, cplx<T> *data, int nfields,
                  long long fstride, cudaStream_t st);
template <typename T>
int launch_xhl(const GridInfo &g, const FftAxis &ax, cplx<T> *spec, const cplx<T> *vext,
               cplx<T> *nG_out, int inverse, double *part, cudaStream_t st);
size_t field_smem_max(const GridInfo &g, size_t csize);
// blocks (and partial sums per quantity) of the x passes
int xpass_blocks(const GridInfo &g);
// Largest block the transform kernels were built for.
int fft_max_threads();
template <typename T> cudaError_t set_field_smem_limits(size_t bytes);

// ---- vectors, reductions, ions (kernels_misc.cu)
// Sum part[q * nblk + b] over b for q < nq into out[q] (one block per q, fixed order).
void launch_reduce(const double *part, int nblk, int nq, double *out, cudaStream_t st);
// The three reductions of an evaluation in one launch: rows 0..2 of pA (na
// columns) into out[0..2], rows 0..5 of pB (nb columns, GGA only) into
// out[3..8], rows 0..8 of pC (nc columns) into out[9..17]; with ne also the
// ne sums of pE into out[18].
void launch_reduce_eval(const double *pA, int na, const double *pB, int nb, const double *pC, int nc, bool gga,
                        double *out, cudaStream_t st, const double *pE = nullptr, int ne = 0);
template <typename T> void launch_fill(long long n, T *x, T val, cudaStream_t st);
template <typename T> void launch_scale(long long n, T *x, double s, const double *sp, cudaStream_t st);
// if *accepted: phi <- phit, v <- vt, gprev <- g; then g = 2 phi (v - *mup);
// part: sum g^2, sum g.gprev (returns blocks)
template <typename T>
int launch_cg_update(long long n, const int *accepted, T *phi, const T *phit, T *v, const T *vt,
                     const double *mup, T *g, T *gprev, double *part, cudaStream_t st);
template <typename T, typename U> void launch_convert(long long n, const T *x, U *y, cudaStream_t st);
// sum x^2 -> part (returns blocks)
template <typename T> int launch_sumsq(long long n, const T *x, double *part, cudaStream_t st);
// y = 2 x - xp; part: sum y^2
template <typename T>
int launch_extrap(long long n, const T *x, const T *xp, T *y, double *part, cudaStream_t st);
// part <- block sums of a.b (returns blocks); out = alpha x + beta y
template <typename T> int launch_dot(long long n, const T *a, const T *b, double *part, cudaStream_t st);
template <typename T>
void launch_axpby(long long n, double alpha, const T *x, double beta, const T *y, T *out, cudaStream_t st);
// g = 2 phi (v - mu); part: sum g^2, sum g.gprev
template <typename T>
int launch_cg_grad(long long n, const T *phi, const T *v, double mu, const double *mup, T *g,
                   const T *gprev, double *part, cudaStream_t st);
// d = -g + beta d; part: sum phi d, sum d^2, sum d g, sum phi^2, sum phi g
template <typename T>
int launch_cg_dir(long long n, const T *g, T *d, double beta, const double *betap, const T *phi,
                  double *part, cudaStream_t st);
// restart: d = -g; else d -= c1 phi; dhat = c2 d; part: sum 2 phi v dhat
template <typename T>
int launch_cg_dhat(long long n, const T *g, T *d, const T *phi, const T *v, double c1, double c2,
                   int restart, const double *c12r, T *dhat, double *part, cudaStream_t st);

// Local-pseudopotential forces on the tensor cores (kernels_force.cu): coef
// from launch_force_coefficients (pairs, N), scratch of force_tc_bytes, part
// as launch_lpp_forces; returns the chunk count (= force_tc_chunks).  Taken
// when force_tc_takes.
bool force_tc_takes(const GridInfo &g, int nat);
size_t force_tc_bytes(const GridInfo &g, int nat);
int force_tc_chunks(const GridInfo &g, int nat);
cudaError_t force_tc_smem_limits();
void launch_force_coefficients(const GridInfo &g, const double2 *nG, float2 *coef, cudaStream_t st);
int launch_force_tc(const GridInfo &g, int nat, const double *Z, const double2 *px, const double2 *py, const double2 *pz,
                    const double2 *nG, const float2 *coef, void *scratch, double *part, cudaStream_t st);

// Double-float copies of the phase tables (16 bytes per complex entry, the
// size of a double2): xT[ix][I], yT[iy][I], zT[kz][I] (atoms fastest) and
// zd[I][kz].
struct PhaseTablesDD {
    double2 *xT, *yT, *zT, *zd;
};
// Per-ion axis phase tables exp(-i G_a R_a) for a = x, y, z (complex double,
// [nat][nx], [nat][ny], [nat][K]); with dd also their double-float copies.
void launch_phases(const GridInfo &g, int nat, const double *R, double2 *px, double2 *py,
                   double2 *pz, const PhaseTablesDD *dd, cudaStream_t st);
// v_ext(G) on the half spectrum, Hermitian-symmetrised on Nyquist planes:
// sums over atoms in double-float when dd is given and the grid computes in
// double-float, else binary64.  (A single-precision copy is made with
// launch_convert.)
void launch_vext(const GridInfo &g, int nat, const double *Z, const double2 *px,
                 const double2 *py, const double2 *pz, const PhaseTablesDD *dd, double2 *vext, cudaStream_t st);
// Local-pseudopotential forces from n(G): part[(I * nchunk + c) * 3 + a];
// returns nchunk (= lpp_force_chunks(g, nat, dd != nullptr)).  cn is
// scratch of NH double2.  Double-float sums as launch_vext.
template <typename T>
int launch_lpp_forces(const GridInfo &g, int nat, const double *Z, const double2 *px,
                      const double2 *py, const double2 *pz, const PhaseTablesDD *dd, const cplx<T> *nG,
                      double2 *cn, double *part, cudaStream_t st);
int lpp_force_chunks(const GridInfo &g, int nat, bool dd);
// Chunks of the double-float force kernel for nx * ny = rows (footprints).
int lpp_force_chunks_dd(long long rows, int nat);
// Sum force partials over chunks into F[nat][3] (+= if accumulate).
void launch_force_reduce(int nat, int nchunk, const double *part, double *F, int accumulate,
                         cudaStream_t st);

// The cell of the Ewald real-space sums: rows a_j of a (bohr), ai = a^-1;
// tri = 0 for an orthorhombic cell (a diagonal).
struct EwCell {
    double a[9], ai[9];
    int tri;
};

// Ewald: real-space part per ion -> eparts[nat], F[nat][3];
// reciprocal part over the G list -> S[nG], energy partials, forces added.

void launch_ewald_real(int nat, const double *R, const double *Z, const EwCell &cl, double alpha,
                       double rcut, int3 nimg, double *eion, double *F, cudaStream_t st);
int launch_ewald_recip(int nat, const double *R, const double *Z, int nG, const double *Gv,
                       const double *wG, double2 *S, double *epart, double *F, cudaStream_t st);

// The ions of the allocation-free entry point, by value in a kernel's
// arguments (a copy from pageable memory would wait for the stream), and the
// tables made of them: t nat (nx + ny + nz + 3), eg and g2 3 kStaticEdge,
// ewtab kEwTabRows nat, ewpart kEwBlocks entries.
constexpr int kStaticEdge = 64, kStaticAtoms = 64, kEwTabRows = 256, kEwBlocks = 304;
struct StaticIons {
    double R[3 * kStaticAtoms], Z[kStaticAtoms];
    float frac[3 * kStaticAtoms];   // fractional coordinates in [0, 1], for screening the pairs
};
struct StaticIonTables {
    double *R, *Z;
    float *frac;
    float2 *t;
    double2 *eg;
    float2 *g2;                     // (k b)^2 of each axis's coefficients, kStaticEdge apart
    double2 *ewtab;
    double *ewpart;
};
// v_ext's coefficients into vre (N) and the Ewald energy, without its self
// and background terms, as the returned number of sums in ewpart: 0 for cells
// so uneven that an axis needs more images or reciprocal planes than fit.
int launch_static_ions(const GridInfo &g, int nat, const StaticIons &ions, const StaticIonTables &t, float2 *vre, cudaStream_t st);

// MD: half step A (thermostat half, kick, drift) and B (kick, thermostat half).
void launch_md_a(int nat, const double *m, double *R, double *V, const double *F, double dt,
                 double kT, double Q, int ndof, int thermo, double *nh, cudaStream_t st);
void launch_md_b(int nat, const double *m, double *V, const double *F, double dt, double kT,
                 double Q, int ndof, int thermo, double *nh, cudaStream_t st);
void launch_andersen(int nat, const double *m, double *V, double kT, double prob, const double *u,
                     const double *xi, double *nh, cudaStream_t st);
// Stress tensor parts: Hartree and LPP sums over the half spectrum (12
// partial rows, nx ny columns; returns the column count), and the Ewald
// real-space (6 rows, nat columns) and reciprocal (7 rows; returns the
// column count) sums.
int launch_gstress(const GridInfo &g, int nat, const double *Z, const double2 *px, const double2 *py,
                   const double2 *pz, const PhaseTablesDD *dd, const double2 *nG, double *part, cudaStream_t st);
int launch_ewald_stress(int nat, const double *R, const double *Z, const EwCell &cl, double alpha, double rcut,
                        int3 nimg, int nG, const double *Gv, const double *wG, const double2 *S,
                        double *preal, double *precip, cudaStream_t st);

// ---- device CG controller (cg_control.cu); single-thread kernels.
// use_cond = 0 outside a graph (the handles are then ignored).
void launch_ctl_norm(CgState *s, cudaStream_t st);
void launch_ctl_init(CgState *s, cudaStream_t st);
void launch_ctl_grad(CgState *s, int first, cudaGraphConditionalHandle outer, int use_cond,
                     cudaStream_t st);
void launch_ctl_dir(CgState *s, cudaStream_t st);
void launch_ctl_dhat(CgState *s, cudaGraphConditionalHandle ls, int use_cond, cudaStream_t st);
void launch_ctl_ls(CgState *s, cudaGraphConditionalHandle ls, int use_cond, cudaStream_t st);

}  // namespace ofdft
