// Internal definitions shared by the libgbfd translation units: the padded
// field layout in HBM, the stencil coefficient tables, the Williamson RK3
// coefficients and the per-point right-hand side of Eqs. 1-3.
#pragma once

#include <cmath>
#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>
#include <stdint.h>

namespace gbfd {

// ---------------------------------------------------------------------------
// Padded field layout.
//
// Each field is stored as [z][Y][X] with ghost columns/rows in x and y only:
// interior point (x, y, z) lives at X = x + GX, Y = y + GY.  The ghosts hold
// periodic copies (X in [0, GX) is x = nx-GX.., X in [nx+GX, nx+2GX) is
// x = 0..GX-1; same in y with GY) so that a tile plus its 3-cell halo is one
// rectangular, in-bounds box for TMA.  z needs no ghosts: a plane is fetched
// by its wrapped index.  The row pitch P is a multiple of 128 bytes and the
// origin is offset so that every interior row starts 128-byte aligned
// (whole-sector warp accesses).  GX = 4 (not 3) keeps the TMA box origin
// X = x0 16-byte aligned.
//
// With walls in z (the ghost-zone boundary variant) each field also holds
// gz = 3 ghost planes below and above its nz interior planes: interior plane
// z sits at plane index z + gz of the field, the origin points at interior
// plane 0, so element offsets of interior points are unchanged, and ghost
// planes are z = -3..-1 and nz..nz+2.  A ghost-fill kernel writes them (the
// parity mirror of the interior about the wall points) after every substep.
// ---------------------------------------------------------------------------
constexpr int GX = 4;
constexpr int GY = 3;
constexpr int R = 3;  // stencil radius (sixth order, n = 2R)

struct Layout {
    int nx, ny, nz;
    int w;              // bytes per value
    long long P;        // row pitch, elements
    long long rows;     // rows per plane, ny + 2 GY
    long long plane;    // P * rows
    long long fpitch;   // elements between consecutive fields
    long long origin;   // byte offset of element (f=0,z=0,Y=0,X=0) in the region
    long long bytes;    // region bytes for `nf` fields
    int gz;             // ghost planes below and above in z: 0 (periodic z) or
                        // GZW (walls in z)
};

constexpr int GZW = 3;  // ghost planes per side with walls in z

inline Layout make_layout(int nx, int ny, int nz, int w, int nf, int gz = 0)
{
    Layout L;
    L.nx = nx;
    L.ny = ny;
    L.nz = nz;
    L.w = w;
    L.gz = gz;
    const long long q = 128 / w;  // elements per 128 bytes
    L.P = ((nx + 2 * GX + q - 1) / q) * q;
    L.rows = ny + 2 * GY;
    L.plane = L.P * L.rows;
    L.fpitch = L.plane * (nz + 2 * gz);  // P*w is a multiple of 128, so is this
    L.origin = 128 - GX * w + (long long)gz * L.plane * w;
    L.bytes = 128 + (long long)nf * L.fpitch * w;
    return L;
}

// Index of the plane holding local z (which may lie in [-3, nz + 3) for a
// stencil arm): the wrapped index for periodic z, the plane itself (ghost
// planes included) with walls.  TMA maps of a walled layout start at ghost
// plane -gz, so their z coordinate is zplane + gz.
__host__ __device__ __forceinline__ int zplane(const Layout &L, int z)
{
    if (L.gz)
        return z;
    return z < 0 ? z + L.nz : (z >= L.nz ? z - L.nz : z);
}

// Element index of interior point (x, y, z) of field f relative to origin.
__host__ __device__ inline long long lidx(const Layout &L, int f, int z, int y, int x)
{
    return (long long)f * L.fpitch + (long long)z * L.plane + (long long)(y + GY) * L.P + (x + GX);
}

// ---------------------------------------------------------------------------
// Stencil coefficients (Eqs. 6-8) with the grid spacing folded in.
//   D1 f = sum_k d1[a][k-1] (f_{+k} - f_{-k})                      (Eq. 6)
//   D2 f = d2c[a] f_0 + sum_k d2[a][k-1] (f_{+k} + f_{-k})         (Eq. 7)
//   Dab f = sum_k mx[p][k-1] (f_{+k,+k} - f_{-k,+k} + f_{-k,-k} - f_{+k,-k})
//                                                                  (Eq. 8)
// pair p: 0 = (x,y), 1 = (x,z), 2 = (y,z).
// ---------------------------------------------------------------------------
template <class T>
struct Coef {
    T d1[3][3];
    T d2c[3];
    T d2[3][3];
    T mx[3][3];
    T cs2;     // c_s^2
    T nu;      // nu
    T nu3;     // nu / 3
    T nu2;     // 2 nu
    T nu23;    // (2/3) nu
    // accessors shared with CubicCoef (axis a, pair p, arm k = 1..3)
    __host__ __device__ __forceinline__ T D1(int a, int k) const { return d1[a][k - 1]; }
    __host__ __device__ __forceinline__ T D2c(int a) const { return d2c[a]; }
    __host__ __device__ __forceinline__ T D2(int a, int k) const { return d2[a][k - 1]; }
    __host__ __device__ __forceinline__ T MX(int p, int k) const { return mx[p][k - 1]; }
};

// Coefficients of a box with the same spacing h on every axis: one set of
// stencil weights serves all axes (10 values plus 4 physics scalars), small
// enough to live in registers when it changes from box to box.
template <class T>
struct CubicCoef {
    T d1[3], d2c, d2[3], mx[3];
    T cs2, nu, nu3, nu23;
    __host__ __device__ __forceinline__ T D1(int, int k) const { return d1[k - 1]; }
    __host__ __device__ __forceinline__ T D2c(int) const { return d2c; }
    __host__ __device__ __forceinline__ T D2(int, int k) const { return d2[k - 1]; }
    __host__ __device__ __forceinline__ T MX(int, int k) const { return mx[k - 1]; }
};

template <class T>
inline Coef<T> make_coef(double hx, double hy, double hz, double cs, double nu)
{
    Coef<T> c;
    const double h[3] = {hx, hy, hz};
    const double d1w[3] = {45.0, -9.0, 1.0};
    const double d2w[3] = {270.0, -27.0, 2.0};
    const double mxw[3] = {270.0, -27.0, 2.0};
    for (int a = 0; a < 3; ++a) {
        for (int k = 0; k < 3; ++k) {
            c.d1[a][k] = (T)(d1w[k] / (60.0 * h[a]));
            c.d2[a][k] = (T)(d2w[k] / (180.0 * h[a] * h[a]));
        }
        c.d2c[a] = (T)(-490.0 / (180.0 * h[a] * h[a]));
    }
    const double hp[3][2] = {{hx, hy}, {hx, hz}, {hy, hz}};
    for (int p = 0; p < 3; ++p)
        for (int k = 0; k < 3; ++k)
            c.mx[p][k] = (T)(mxw[k] / (720.0 * hp[p][0] * hp[p][1]));
    c.cs2 = (T)(cs * cs);
    c.nu = (T)nu;
    c.nu3 = (T)(nu / 3.0);
    c.nu2 = (T)(2.0 * nu);
    c.nu23 = (T)(2.0 * nu / 3.0);
    return c;
}

// True when the weights are the same on every axis (equal grid spacing);
// cubic_of then carries exactly the same values in the isotropic form.
template <class T>
inline bool coef_is_cubic(const Coef<T> &c)
{
    bool iso = c.d2c[1] == c.d2c[0] && c.d2c[2] == c.d2c[0];
    for (int k = 0; k < 3; ++k)
        iso = iso && c.d1[1][k] == c.d1[0][k] && c.d1[2][k] == c.d1[0][k] &&
              c.d2[1][k] == c.d2[0][k] && c.d2[2][k] == c.d2[0][k] &&
              c.mx[1][k] == c.mx[0][k] && c.mx[2][k] == c.mx[0][k];
    return iso;
}

template <class T>
inline CubicCoef<T> cubic_of(const Coef<T> &c)
{
    CubicCoef<T> q;
    for (int k = 0; k < 3; ++k) {
        q.d1[k] = c.d1[0][k];
        q.d2[k] = c.d2[0][k];
        q.mx[k] = c.mx[0][k];
    }
    q.d2c = c.d2c[0];
    q.cs2 = c.cs2;
    q.nu = c.nu;
    q.nu3 = c.nu3;
    q.nu23 = c.nu23;
    return q;
}

template <class T>
inline CubicCoef<T> make_cubic_coef(double h, double cs, double nu)
{
    Coef<T> c = make_coef<T>(h, h, h, cs, nu);
    CubicCoef<T> q;
    for (int k = 0; k < 3; ++k) {
        q.d1[k] = c.d1[0][k];
        q.d2[k] = c.d2[0][k];
        q.mx[k] = c.mx[0][k];
    }
    q.d2c = c.d2c[0];
    q.cs2 = c.cs2;
    q.nu = c.nu;
    q.nu3 = c.nu3;
    q.nu23 = c.nu23;
    return q;
}

// Weights of the FP64 lagged kernel with everything that multiplies a linear term
// folded in: the time step s (1 where the update multiplies by dt itself), the
// viscosity and the signs.  With gm = -s grad u (weights N1) and nng = -nu
// grad lnrho, Eqs. 1-3 of component i become
//   s rhs_i = sum_j gm_ij (u_j + nng_j) + sum_j gm_ji nng_j          (Eq. 3)
//           + (nu23 dvm + ncs2) d_i lnrho                    dvm = sum gm_jj
//           + sum_a [V2 or, for a = i, X2] + sum Eq. 8 terms with M3,
//   s rhs_lnrho = ns (u . grad lnrho) + dvm,   s rhs_s = sum_j u_j (gm_s)_j:
// no separate Laplacian, divergence, advection and update multiplications
// (245 instead of 285 FP64 operations per point and substep).  Built in FP64
// and rounded once.  VC is minus the sum of the second-derivative weights, so that
// they cancel on a constant as they do in Eq. 7; the arms X2 take what rounding
// VC left over, the first arm as much of it as its last bit shows, the next ones
// the rest (no arm moves by more than about one unit of the first one's last
// place).  Left over, it adds the same multiple of u in every substep.
template <class T>
struct FoldCoef {
    T l1[3][3];  // d1
    T n1[3][3];  // -s d1
    T v2[3][3];  // s nu d2
    T x2[3][3];  // s (4/3) nu d2 (Eq. 7's part of grad div included)
    T vc[3];     // centre weight of component i
    T m3[3][3];  // s (nu/3) mx
    T nnu, nu23, ncs2, ns;  // -nu, (2/3) nu, -s c_s^2, -s
    __host__ __device__ __forceinline__ T L1(int a, int k) const { return l1[a][k - 1]; }
    __host__ __device__ __forceinline__ T N1(int a, int k) const { return n1[a][k - 1]; }
    __host__ __device__ __forceinline__ T V2(int a, int k) const { return v2[a][k - 1]; }
    __host__ __device__ __forceinline__ T X2(int a, int k) const { return x2[a][k - 1]; }
    __host__ __device__ __forceinline__ T VC(int i) const { return vc[i]; }
    __host__ __device__ __forceinline__ T M3(int p, int k) const { return m3[p][k - 1]; }
};

// The same for equal spacing on every axis (the same values, 20 instead of 52).
template <class T>
struct FoldCubic {
    T l1[3], n1[3], v2[3], x2[3], vc, m3[3];
    T nnu, nu23, ncs2, ns;
    __host__ __device__ __forceinline__ T L1(int, int k) const { return l1[k - 1]; }
    __host__ __device__ __forceinline__ T N1(int, int k) const { return n1[k - 1]; }
    __host__ __device__ __forceinline__ T V2(int, int k) const { return v2[k - 1]; }
    __host__ __device__ __forceinline__ T X2(int, int k) const { return x2[k - 1]; }
    __host__ __device__ __forceinline__ T VC(int) const { return vc; }
    __host__ __device__ __forceinline__ T M3(int, int k) const { return m3[k - 1]; }
};

// The batch's FP32 form of the folding, for equal spacing: every axis has a centre
// weight of its own (cx beside X2, cv beside V2), so that each axis' sum cancels
// by itself before the three are added.  In one sum with the common centre weight
// VC the partial sums round against VC u until the last arm: at the viscous limit
// of the time step (VC = 2.3) two FP32 steps were 2.1e-7 off (rms of the velocity at
// 20^3 to 48^3), with three sums 1.16e-7, the two-plane routine's unfolded
// second derivatives 1.19e-7.
struct FoldAxes {
    float l1[3], n1[3], v2[3], x2[3], cv, cx, m3[3];
    float nnu, nu23, ncs2, ns;
    __host__ __device__ __forceinline__ float L1(int, int k) const { return l1[k - 1]; }
    __host__ __device__ __forceinline__ float N1(int, int k) const { return n1[k - 1]; }
    __host__ __device__ __forceinline__ float V2(int, int k) const { return v2[k - 1]; }
    __host__ __device__ __forceinline__ float X2(int, int k) const { return x2[k - 1]; }
    __host__ __device__ __forceinline__ float M3(int, int k) const { return m3[k - 1]; }
};

template <class C>
struct is_fold : std::is_same<C, FoldAxes> {};

// Centre weight of the arms w, which take what its rounding left over (as above).
inline float centre_of(float (&w)[3])
{
    const double sum = 2.0 * ((double)w[0] + ((double)w[1] + (double)w[2]));
    const float c = (float)(-sum);
    double left = (double)c + sum;  // exact: 24-bit terms of few binades apart
    for (int k = 0; k < 3; ++k) {
        const float arm = (float)((double)w[k] - 0.5 * left);
        left += 2.0 * ((double)arm - (double)w[k]);
        w[k] = arm;
    }
    return c;
}

inline FoldAxes make_fold_axes(const Coef<double> &c, double s)
{
    FoldAxes f;
    for (int k = 0; k < 3; ++k) {
        f.l1[k] = (float)c.d1[0][k];
        f.n1[k] = (float)(-s * c.d1[0][k]);
        f.v2[k] = (float)(s * c.nu * c.d2[0][k]);
        f.x2[k] = (float)(s * c.nu * (4.0 / 3.0) * c.d2[0][k]);
        f.m3[k] = (float)(s * (c.nu / 3.0) * c.mx[0][k]);
    }
    f.cv = centre_of(f.v2);
    f.cx = centre_of(f.x2);
    f.nnu = (float)(-c.nu);
    f.nu23 = (float)(2.0 * c.nu / 3.0);
    f.ncs2 = (float)(-s * c.cs2);
    f.ns = (float)(-s);
    return f;
}

template <class T>
inline FoldCoef<T> make_fold(const Coef<double> &c, double s)
{
    FoldCoef<T> f;
    for (int a = 0; a < 3; ++a)
        for (int k = 0; k < 3; ++k) {
            f.l1[a][k] = (T)c.d1[a][k];
            f.n1[a][k] = (T)(-s * c.d1[a][k]);
            f.v2[a][k] = (T)(s * c.nu * c.d2[a][k]);
            f.x2[a][k] = (T)(s * c.nu * (4.0 / 3.0) * c.d2[a][k]);
            f.m3[a][k] = (T)(s * (c.nu / 3.0) * c.mx[a][k]);
        }
    for (int i = 0; i < 3; ++i) {
        double sum[3];  // per arm, in an order that equal spacings make the same for every i
        for (int k = 0; k < 3; ++k)
            sum[k] = (double)f.x2[i][k] +
                     ((double)f.v2[(i + 1) % 3][k] + (double)f.v2[(i + 2) % 3][k]);
        f.vc[i] = (T)(-2.0 * (sum[0] + (sum[1] + sum[2])));
        // what is left over, by a sum that carries its rounding errors along
        double hi = (double)f.vc[i], lo = 0.0;
        for (int j = 0; j < 3; ++j)
            for (int k = 0; k < 3; ++k) {
                const double v = 2.0 * (double)(j == 0 ? f.x2[i][k] : f.v2[(i + j) % 3][k]);
                const double t = hi + v, w = t - hi;
                lo += (hi - (t - w)) + (v - w);
                hi = t;
            }
        double left = hi + lo;
        for (int k = 0; k < 3; ++k) {
            const T arm = (T)((double)f.x2[i][k] - 0.5 * left);
            left += 2.0 * ((double)arm - (double)f.x2[i][k]);
            f.x2[i][k] = arm;
        }
    }
    f.nnu = (T)(-c.nu);
    f.nu23 = (T)(2.0 * c.nu / 3.0);
    f.ncs2 = (T)(-s * c.cs2);
    f.ns = (T)(-s);
    return f;
}

template <class T>
inline bool fold_is_cubic(const FoldCoef<T> &f)
{
    bool iso = f.vc[1] == f.vc[0] && f.vc[2] == f.vc[0];
    for (int a = 1; a < 3; ++a)
        for (int k = 0; k < 3; ++k)
            iso = iso && f.l1[a][k] == f.l1[0][k] && f.n1[a][k] == f.n1[0][k] &&
                  f.v2[a][k] == f.v2[0][k] && f.x2[a][k] == f.x2[0][k] && f.m3[a][k] == f.m3[0][k];
    return iso;
}

template <class T>
inline FoldCubic<T> cubic_of(const FoldCoef<T> &f)
{
    FoldCubic<T> q;
    for (int k = 0; k < 3; ++k) {
        q.l1[k] = f.l1[0][k];
        q.n1[k] = f.n1[0][k];
        q.v2[k] = f.v2[0][k];
        q.x2[k] = f.x2[0][k];
        q.m3[k] = f.m3[0][k];
    }
    q.vc = f.vc[0];
    q.nnu = f.nnu;
    q.nu23 = f.nu23;
    q.ncs2 = f.ncs2;
    q.ns = f.ns;
    return q;
}

// Williamson (1980) 2N-storage RK3: the paper's Eq. 10 leaves alpha, beta to
// the chosen scheme and fixes alpha_1 = 0.
constexpr double RK3_ALPHA[3] = {0.0, -5.0 / 9.0, -153.0 / 128.0};
constexpr double RK3_BETA[3] = {1.0 / 3.0, 15.0 / 16.0, 8.0 / 15.0};

// ---------------------------------------------------------------------------
// Right-hand side of Eqs. 1-3 (f = 0) at one point from its derivatives.
// gu[i][j] = d_j u_i.  lap[i] = sum_j D2_j u_i.  gd[i] = d_i(div u), the
// grad-div term (left 0 by the 19-point first pass, which adds it in pass 2).
// ---------------------------------------------------------------------------
template <class T>
struct PointDerivs {
    T u[3];
    T gl[3];
    T gu[3][3];
    T gs[3];
    T lap[3];
    T gd[3];
};

template <class T, int NF>
__device__ __forceinline__ void rhs_point(const PointDerivs<T> &d, const Coef<T> &c, T *out)
{
    const T div = d.gu[0][0] + d.gu[1][1] + d.gu[2][2];
    // Eq. 1
    out[0] = -(d.u[0] * d.gl[0] + d.u[1] * d.gl[1] + d.u[2] * d.gl[2]) - div;
    // Eq. 3 and Eq. 2:  2 (S . grad lnrho)_i
    //   = sum_j (d_j u_i + d_i u_j) d_j lnrho - (2/3) div d_i lnrho
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        T adv = d.u[0] * d.gu[i][0] + d.u[1] * d.gu[i][1] + d.u[2] * d.gu[i][2];
        T s2 = (d.gu[i][0] + d.gu[0][i]) * d.gl[0] + (d.gu[i][1] + d.gu[1][i]) * d.gl[1] +
               (d.gu[i][2] + d.gu[2][i]) * d.gl[2];
        T visc = c.nu * (d.lap[i] + s2) + c.nu3 * d.gd[i] - c.nu23 * div * d.gl[i];
        out[1 + i] = -adv - c.cs2 * d.gl[i] + visc;
    }
    if (NF == 5)
        out[4] = -(d.u[0] * d.gs[0] + d.u[1] * d.gs[1] + d.u[2] * d.gs[2]);
}

// Eq. 10 update of one value: w <- alpha w + dt r (the first substep ignores
// the old w, alpha_1 = 0), u_out <- u + beta w; arithmetic in TA.
template <class TA, class TW, class TS>
__device__ __forceinline__ void rk3_update(bool first, TA alpha, TA beta, TA dt, TA r, TS u,
                                           TW &w, TS &out)
{
    TA wn = first ? dt * r : alpha * (TA)w + dt * r;
    w = (TW)wn;
    out = (TS)((TA)u + beta * wn);
}

// A value carried as an unevaluated sum of two FP32 numbers, hi + lo with
// |lo| <= ulp(hi) / 2 ("float-float", Dekker 1971): the precision form's
// Eq. 10 update in compensated FP32 arithmetic.  Built from an FP64 value
// (the RK3 coefficients and dt) or from an FP32 one (lo = 0).
struct ffloat {
    float hi, lo;
    __host__ __device__ ffloat() : hi(0.f), lo(0.f) {}
    __host__ __device__ ffloat(double v) : hi((float)v), lo((float)(v - (double)(float)v)) {}
};

// Error-free transformations (round-to-nearest FP32; explicit _rn operations
// so that nothing is contracted into a fused multiply-add):
// a * b = p + e exactly (fused multiply-add form of Dekker's product) ...
__device__ __forceinline__ void two_prod(float a, float b, float &p, float &e)
{
    p = __fmul_rn(a, b);
    e = __fmaf_rn(a, b, -p);
}
// ... a + b = s + e exactly (Knuth's TwoSum, no ordering of a and b needed) ...
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// ... and a + b = s + e exactly when |a| >= |b| (Dekker's FastTwoSum).
__device__ __forceinline__ void fast_two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}

// Eq. 10 for one FP32 value in float-float arithmetic: w_new = alpha w + dt r
// kept as hi + lo (the products and their sum error-free, the low-order
// terms summed in FP32), w stored as its FP32 rounding hi, and
// u_out = u + beta (hi + lo) rounded once to FP32 from an error-free sum.
// About 48 significant bits, so the result matches the FP64 update of the
// same inputs except where the two roundings of a near-tie differ.
__device__ __forceinline__ void rk3_update_ff(bool first, ffloat alpha, ffloat beta, ffloat dt,
                                              float r, float u, float &w, float &out)
{
    float p2, e2, hi, lo;
    two_prod(dt.hi, r, p2, e2);
    e2 = __fmaf_rn(dt.lo, r, e2);
    if (first) {
        fast_two_sum(p2, e2, hi, lo);
    } else {
        float p1, e1, s, t;
        two_prod(alpha.hi, w, p1, e1);
        e1 = __fmaf_rn(alpha.lo, w, e1);
        two_sum(p1, p2, s, t);
        // s can be small after cancellation: renormalise with the full TwoSum
        two_sum(s, __fadd_rn(t, __fadd_rn(e1, e2)), hi, lo);
    }
    w = hi;
    float q, f, s2, t2;
    two_prod(beta.hi, hi, q, f);
    f = __fmaf_rn(beta.hi, lo, f);
    f = __fmaf_rn(beta.lo, hi, f);
    two_sum(u, q, s2, t2);
    out = __fadd_rn(s2, __fadd_rn(t2, f));
}

template <>
__device__ __forceinline__ void rk3_update<ffloat, float, float>(bool first, ffloat alpha,
                                                                 ffloat beta, ffloat dt, ffloat r,
                                                                 float u, float &w, float &out)
{
    rk3_update_ff(first, alpha, beta, dt, r.hi, u, w, out);
}

// The FP64 update of Eq. 10 (FP32 storage) reached through float-float
// arithmetic: carries the coefficient in both forms.  Below 2^-100 the low half
// runs into the subnormals and the pair no longer holds the value to 48 bits: an
// infinite high half then makes every result fail rk3_pair_ff's check, so that
// all take the FP64 update.
struct fexact {
    ffloat f;
    double d;
    __host__ __device__ fexact() : d(0.0) {}
    __host__ __device__ fexact(double v) : f(v), d(v)
    {
        if (v != 0.0 && fabs(v) < 0x1p-100) {
            f.hi = INFINITY;
            f.lo = 0.f;
        }
    }
};

// Exact IEEE-754 conversions between binary32 and binary64 done with integer
// instructions, so that GB300's narrow FP64 pipe is left to the arithmetic.
// binary32 (sign, 8-bit exponent e, 23-bit fraction m) -> binary64: exponent
// e + 896 (= e - 127 + 1023), fraction m << 29.  binary64 -> binary32: exponent
// E - 896, the top 23 fraction bits, rounded to nearest, ties to even, on the
// 29 dropped bits (a carry out of the fraction bumps the exponent, and past
// the largest finite value gives infinity, as round-to-nearest requires).
// Zero, subnormal, infinite and NaN operands, and results below the normal
// binary32 range, take the hardware conversion.
__device__ __forceinline__ double f32_to_f64_int(float x)
{
    const uint32_t b = __float_as_uint(x);
    const uint32_t e = (b >> 23) & 0xffu;
    if (e == 0u || e == 0xffu)
        return (double)x;
    const uint32_t hi = (b & 0x80000000u) | ((e + 896u) << 20) | ((b & 0x7fffffu) >> 3);
    return __hiloint2double((int)hi, (int)(b << 29));
}

__device__ __forceinline__ float f64_to_f32_int(double v)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const int e = (int)((hi >> 20) & 0x7ffu) - 896;
    if (e <= 0 || e >= 255)
        return __double2float_rn(v);
    const uint32_t m = ((hi & 0xfffffu) << 3) | (lo >> 29);
    const uint32_t rest = lo & 0x1fffffffu;
    const uint32_t up = (rest > 0x10000000u) || (rest == 0x10000000u && (m & 1u));
    return __uint_as_float(((hi & 0x80000000u) | ((uint32_t)e << 23) | m) + up);
}

// Eq. 10 in FP64 for FP32 state: the same arithmetic with explicit fused
// multiply-adds whichever conversions are used (ICVT: the integer routines
// above, else the hardware conversions), so the two give identical bits.
template <bool ICVT, class TW>
__device__ __forceinline__ void rk3_update_f64(bool first, double alpha, double beta, double dt,
                                               float r, float u, TW &w, float &out)
{
    auto up = [](float v) { return ICVT ? f32_to_f64_int(v) : (double)v; };
    auto down = [](double v) { return ICVT ? f64_to_f32_int(v) : __double2float_rn(v); };
    const double rd = up(r);
    double wd;
    if constexpr (sizeof(TW) == 8)
        wd = w;
    else
        wd = up(w);
    const double wn = first ? dt * rd : fma(alpha, wd, dt * rd);
    if constexpr (sizeof(TW) == 8)
        w = wn;
    else
        w = down(wn);
    out = down(fma(beta, wn, up(u)));
}

// rk3_update_ff for two points at once in packed FP32x2 instructions (the same
// operations and bits; constants are broadcast pairs, n* negated ones, so that
// error terms come out negated by one fused multiply-add).
//
// CHECK: `safe` tells, per point, whether both results are also those of the
// FP64 update (rk3_update_f64).  The float-float value and the FP64 one differ
// by less than E = 2^-43 M + 2^-146, M the sum of the magnitudes of the terms
// added (float-float: 2^-46 M by Dekker's and Knuth's bounds, FP64: 2^-52 M; the
// constant covers products whose error terms leave the binary32 range), so
// when the lowest and the highest value within E round to the same binary32
// number, so does the FP64 one.  M = 0 is exact.  Infinities and NaN fail the
// comparison.  About 4 in 10^6 values do; they take the FP64 update.
struct FfConst {
    float2 dh, ndh, ndl, ah, nah, nal, bh, nbh, nbl;
    __device__ __forceinline__ FfConst(const ffloat &dt, const ffloat &a, const ffloat &b)
        : dh(make_float2(dt.hi, dt.hi)), ndh(make_float2(-dt.hi, -dt.hi)),
          ndl(make_float2(-dt.lo, -dt.lo)), ah(make_float2(a.hi, a.hi)),
          nah(make_float2(-a.hi, -a.hi)), nal(make_float2(-a.lo, -a.lo)),
          bh(make_float2(b.hi, b.hi)), nbh(make_float2(-b.hi, -b.hi)),
          nbl(make_float2(-b.lo, -b.lo))
    {
    }
};
template <bool CHECK>
__device__ __forceinline__ void rk3_pair_ff(const bool first, const FfConst &c, const float2 r,
                                            const float2 u, float2 &w, float2 &out, bool &safe0,
                                            bool &safe1)
{
    const float2 N1 = make_float2(-1.f, -1.f);
    auto sub = [&](float2 a, float2 b) { return __ffma2_rn(b, N1, a); };
    auto two_sum2 = [&](float2 a, float2 b, float2 &s, float2 &e) {
        s = __fadd2_rn(a, b);
        const float2 bb = sub(s, a);
        e = __fadd2_rn(sub(a, sub(s, bb)), sub(b, bb));
    };
    // negated errors of the products: -(a b - p) = (-a) b + p
    const float2 p2 = __fmul2_rn(c.dh, r);
    const float2 n2 = __ffma2_rn(c.ndl, r, __ffma2_rn(c.ndh, r, p2));
    float2 hi, lo, m;
    if (CHECK)
        m = make_float2(fabsf(p2.x), fabsf(p2.y));
    if (first) {
        hi = sub(p2, n2);
        lo = __fmul2_rn(__fadd2_rn(n2, sub(hi, p2)), N1);
    } else {
        const float2 p1 = __fmul2_rn(c.ah, w);
        const float2 n1 = __ffma2_rn(c.nal, w, __ffma2_rn(c.nah, w, p1));
        float2 s, t;
        two_sum2(p1, p2, s, t);
        two_sum2(s, sub(t, __fadd2_rn(n1, n2)), hi, lo);
        if (CHECK)
            m = make_float2(m.x + fabsf(p1.x), m.y + fabsf(p1.y));
    }
    const float2 q = __fmul2_rn(c.bh, hi);
    float2 nf = __ffma2_rn(c.nbh, hi, q);
    nf = __ffma2_rn(c.nbh, lo, nf);
    nf = __ffma2_rn(c.nbl, hi, nf);
    float2 s2, t2;
    two_sum2(u, q, s2, t2);
    const float2 g = sub(t2, nf);
    out = __fadd2_rn(s2, g);
    w = hi;
    if (CHECK) {
        const float2 C = make_float2(0x1p-43f, 0x1p-43f), K = make_float2(0x1p-146f, 0x1p-146f);
        const float2 e = __ffma2_rn(C, m, K);
        const float2 wa = __fadd2_rn(hi, __fadd2_rn(lo, e)), wb = __fadd2_rn(hi, sub(lo, e));
        const float2 mo = make_float2(fabsf(q.x) + fabsf(u.x), fabsf(q.y) + fabsf(u.y));
        const float2 eo = __ffma2_rn(C, mo, __ffma2_rn(c.bh, e, K));
        const float2 oa = __fadd2_rn(s2, __fadd2_rn(g, eo)), ob = __fadd2_rn(s2, sub(g, eo));
        safe0 = (wa.x == wb.x || m.x == 0.f) && (oa.x == ob.x || mo.x == 0.f);
        safe1 = (wa.y == wb.y || m.y == 0.f) && (oa.y == ob.y || mo.y == 0.f);
    }
}

// Store v at interior (x, y, z) of field f and at its periodic ghost copies.
template <class T>
__device__ __forceinline__ void store_ghosted(T *base, const Layout &L, int f, int z, int y, int x,
                                              T v)
{
    const long long i0 = lidx(L, f, z, y, x);
    base[i0] = v;
    long long dx = 0, dy = 0;
    if (x < GX)
        dx = L.nx;
    else if (x >= L.nx - GX)
        dx = -L.nx;
    if (y < GY)
        dy = (long long)L.ny * L.P;
    else if (y >= L.ny - GY)
        dy = -(long long)L.ny * L.P;
    if (dx)
        base[i0 + dx] = v;
    if (dy) {
        base[i0 + dy] = v;
        if (dx)
            base[i0 + dy + dx] = v;
    }
}

// Host-side launch helpers implemented in the kernel translation units.
struct StateBufs {
    void *in;    // padded state, storage type
    void *out;   // padded state, storage type
    void *w;     // padded 2N register (u-tilde)
    void *div;   // padded divergence field (19-point form)
    Layout Ls;   // layout of in/out/div (div uses one field)
    Layout Lw;   // layout of w
    int zc;      // planes per CTA of the default tiled kernel on this grid
};

}  // namespace gbfd
