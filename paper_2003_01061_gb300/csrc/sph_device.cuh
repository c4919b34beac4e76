// sph_device.cuh -- device-side data layout and inline helpers of the relaxation kernels.
//
// Layout in HBM (a batch of instances packed into n slots; per-instance slot ranges):
//   stored state (in the order of the previous step's sort):
//     C[a][n] int32   finest-level cell of the position;  O[a][n] T  offset inside that cell
//                     (position = origin + C*c0 + O, reconstructed in FP64 where needed)
//     V[a][n] T       velocities;  H[n] T smoothing length;  G[n] uint32 meta;  ID[n] int32
//   sorted state (written by the gather of the rebuild, read by the pair passes):
//     Cs, Os, IDs as above, VH[n] T4 = (v, h), Ks[n] cell key, Ms[n] meta word,
//     P[n] T4 = offsets inside the particle's own level cell + h (FP32 build, 2D:
//     (ox, oy, h, meta word)), A[n] T4 = (a_p.x, a_p.y, a_p.z, V~) from the pressure pass.
//   meta bits: 0-5 group (feature index), 6-7 intrinsic dimension; in the sorted arrays the meta
//   word also holds the low bits of the particle's level-cell corner (MetaWord).
// T is float (FP32 pair sums) or double (FP64 build); D is 2 or 3.
#pragma once
#include <cuda_runtime.h>
#include <math_constants.h>
#include <climits>
#include <stdint.h>

namespace sph {

constexpr int MAXF = 64;
constexpr int MAXH = 8;
constexpr int MAXL = 8;
// words per occupancy cell: per level, the largest half support of its particles in the cell
// (the search records' w, float bits; 0: none there)
constexpr int OCCW = MAXL;
#ifndef SPH_BLOCK
#define SPH_BLOCK 128
#endif
constexpr int BLOCK = SPH_BLOCK;   // threads per block of the per-slot and pair-pass kernels

enum { K_VOLUME = 0, K_POINT = 1, K_SEGMENT = 2, K_CIRCLE = 3, K_RECT = 4, K_SPHERE = 5 };
enum { PH1 = 1, PH_RAMP = 2, PH2 = 3, PH_DONE = 4 };
enum { ST_NONFINITE = 1u, ST_OUTSIDE_GRID = 2u, ST_H_RANGE = 4u, ST_SCAN = 8u };

struct Feat {
    int kind, dim;
    double g[12];
    double nb[3];
    double orient;
    float fnb[3];        // float copies used by the FP32 pair sums
    float ftg[3];        // SEGMENT: unit tangent; RECT: unit normal
    float fc[3];         // CIRCLE / SPHERE centre
    float forient;
};

struct Domain {
    int D, base;
    double lo[3], hi[3], bc[3], br;
    int nh;
    double hc[MAXH][3];
    double hr[MAXH];
    float flo[3], fhi[3], fbc[3], fbr;   // float copies for the FP32 level-set pre-check
    float fhc[MAXH][3], fhr[MAXH];
    int nf;
    Feat f[MAXF];
};

struct Sizing {
    int kind;
    double a, b, lo, hi;
    double q[3];
    int nref;
    double rc[MAXH][3];
    double rr[MAXH];
    float fa, fb, flo, fhi, fq[3];       // float copies for the FP32 evaluation of h_t
    float frc[MAXH][3], frr[MAXH];
};

struct Grid {
    int D, L;
    float c0;
    float origin[3];
    double c[MAXL];      // c0 * 2^l
    double inv_c[MAXL];  // 1 / c_l rounded once in FP64
    float cf[MAXL];      // c0 * 2^l as float (exact)
    float thr[MAXL];
    int dims[MAXL][3];
    int base[MAXL + 1];  // first key of each level; base[MAXL]: the instance's dummy key
    int ncell;           // cells of the instance (its keys are base[0] .. base[0]+ncell-1)
    int sm;              // log2 of the cells per support m: level l holds kappa h <= m c_l
    int osh;             // occupancy cells of 2^osh finest cells per axis
    int od[3];           // occupancy grid dimensions
    int occ_base;        // first entry of the instance's occupancy cells in the occupancy array
};

struct Params {
    double kappa, p0, visc, cfl_a, cfl_v, eps1, dt_cap, dt_collapse, threshold;
    int reset_period, sample_every, window, ramp_len, boundary_rho;
    int boundary_corr;   // 0: the boundary sum of Eq. 19 is left out (earlier method, Sec. 4.1)
    int group_conv;      // 1: every group runs its own phases (Algorithm 1's per-feature check)
    int feature_order;   // 1: Algorithm 1's feature loop in sequence: the step runs one pass per
                         // intrinsic dimension (curves, surfaces, volume), each reading the lower
                         // classes' new positions; 0: one pass for all (Jacobi)
    int G;
    int gdim[MAXF];      // intrinsic dimension of every group (feature)
    float kappa_f, p0_f, visc_f, cfl_a_f, cfl_v_f;   // float copies for the FP32 kernels
};

// controller state + per-step accumulators (one per instance, in device memory; 16-byte
// aligned so that it is copied in vectors)
struct alignas(16) Ctrl {
    int phase, wcount, nwin, sample_now;
    long long n, ramp_start;
    unsigned long long escapes;
    unsigned int status;
    int pad;
    double wsum[MAXF], A_last[MAXF], A_prev[MAXF], Vbar[MAXF], dt_prev[MAXF], dt[MAXF];
    int reset[MAXF];
    double E_t, E_avg, E_sys, eps, f;
    float dt_f[MAXF], eps_f, f_f;      // float copies of dt, eps, f for the FP32 update
    unsigned long long dta_bits[MAXF], dtv_bits[MAXF];   // per-group minima of Eq. 24 terms
    // per group, used only with group_convergence = 1 (kept last: the instance controller
    // copies the part before it): phase, damping and attenuation of the last step, window
    // counters, switch step, last error
    int gphase[MAXF];
    double geps[MAXF], gf[MAXF];
    float geps_f[MAXF], gf_f[MAXF];
    int gwcount[MAXF], gnwin[MAXF];
    long long gramp_start[MAXF];
    double gE[MAXF];
    // feature order: the step's largest errors of the groups evaluated in the earlier class passes
    double seq_et, seq_ea;
    int seq_ev, seq_pad[3];
};

template <typename T> struct alignas(4 * sizeof(T)) Vec4 { T x, y, z, w; };

// ---- rounding-explicit arithmetic (the neighbour predicate must be evaluated op by op) ----
__device__ __forceinline__ float rn_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float rn_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float rn_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rn_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double rn_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double rn_mul(double a, double b) { return __dmul_rn(a, b); }

__device__ __forceinline__ float rn_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rn_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

__device__ __forceinline__ unsigned long long min_bits(float v) { return (unsigned long long)__float_as_uint(v); }
__device__ __forceinline__ unsigned long long min_bits(double v) { return (unsigned long long)__double_as_longlong(v); }
template <typename T> __device__ __forceinline__ T from_bits(unsigned long long b);
template <> __device__ __forceinline__ float from_bits<float>(unsigned long long b) { return __uint_as_float((unsigned)b); }
template <> __device__ __forceinline__ double from_bits<double>(unsigned long long b) { return __longlong_as_double((long long)b); }
template <typename T> __host__ __device__ __forceinline__ unsigned long long inf_bits();
template <> __host__ __device__ __forceinline__ unsigned long long inf_bits<float>() { return 0x7f800000ull; }
template <> __host__ __device__ __forceinline__ unsigned long long inf_bits<double>() { return 0x7ff0000000000000ull; }

template <typename T> __device__ __forceinline__ T t_sqrt(T v);
template <> __device__ __forceinline__ float t_sqrt<float>(float v) { return sqrtf(v); }
template <> __device__ __forceinline__ double t_sqrt<double>(double v) { return sqrt(v); }
template <typename T> __device__ __forceinline__ T t_floor(T v);
template <> __device__ __forceinline__ float t_floor<float>(float v) { return floorf(v); }
template <> __device__ __forceinline__ double t_floor<double>(double v) { return floor(v); }

// a constant in the working precision: the float copy in the FP32 build (a double-to-float
// conversion runs on the FP64 pipe, which is narrow on this GPU), the double in the FP64 build
template <typename T> __device__ __forceinline__ T wp(double d, float f);
template <> __device__ __forceinline__ float wp<float>(double, float f) { return f; }
template <> __device__ __forceinline__ double wp<double>(double d, float) { return d; }

// h^d and h^(2d) for an intrinsic dimension d in {1, 2, 3}
template <typename T> __device__ __forceinline__ void hpow(T h, int d, T& hd, T& h2d) {
    const T h2 = h * h;
    hd = d == 1 ? h : (d == 2 ? h2 : h2 * h);
    h2d = hd * hd;
}

// Wendland C2 normalisation alpha_d / (its R-dependence): alpha_1 = 3/(2R), alpha_2 = 7/(pi R^2),
// alpha_3 = 21/(2 pi R^3); given invR = 1/R.
template <typename T> __device__ __forceinline__ T wendland_alpha(int d, T invR) {
    if (d == 1) return T(1.5) * invR;
    if (d == 2) return T(7.0 / CUDART_PI) * invR * invR;
    return T(21.0 / (2.0 * CUDART_PI)) * invR * invR * invR;
}

// ---- particle record access (sorted arrays) ----
// The meta word of a sorted particle holds the group and intrinsic dimension (8 bits) and the
// low bits of the corner of the particle's own level cell, counted in finest cells: 12 bits per
// axis in 2D (one 32-bit word), 16 in 3D (two).  Two cells of one search lie fewer than 2,048
// finest cells apart (the largest support is 512, a cell 128), so the difference of two corners
// is exact from these bits, and a pair needs no other array for it.
template <int D> struct MetaWord;
template <> struct MetaWord<2> {
    typedef unsigned type;
    __device__ __forceinline__ static type make(unsigned meta, const int P[3]) {
        return (meta & 255u) | (((unsigned)P[0] & 0xfffu) << 8) | ((unsigned)P[1] << 20);
    }
    __device__ __forceinline__ static unsigned meta(type w) { return w & 255u; }
    // P - (the corner in w), per axis
    __device__ __forceinline__ static void rel(type w, const int P[3], int m[3]) {
        m[0] = (int)(((unsigned)P[0] - (w >> 8)) << 20) >> 20;
        m[1] = (int)(((unsigned)P[1] - (w >> 20)) << 20) >> 20;
        m[2] = 0;
    }
};
template <> struct MetaWord<3> {
    typedef uint2 type;
    __device__ __forceinline__ static type make(unsigned meta, const int P[3]) {
        return make_uint2(((unsigned)P[0] & 0xffffu) | ((unsigned)P[1] << 16),
                          ((unsigned)P[2] & 0xffffu) | ((meta & 255u) << 16));
    }
    __device__ __forceinline__ static unsigned meta(type w) { return w.y >> 16; }
    __device__ __forceinline__ static void rel(type w, const int P[3], int m[3]) {
        m[0] = (int)(short)((unsigned)P[0] - w.x);
        m[1] = (int)(short)((unsigned)P[1] - (w.x >> 16));
        m[2] = (int)(short)((unsigned)P[2] - w.y);
    }
};
template <int D> using Meta = typename MetaWord<D>::type;

template <typename T, int D> struct Rec {
    // (float, 2D): P = (ox, oy, h, meta word); every other case: P = (ox, oy, oz, h) + M
    static constexpr bool packed = (sizeof(T) == 4 && D == 2);
    __device__ __forceinline__ static void load(const Vec4<T>* __restrict__ P, const Meta<D>* __restrict__ M, int j,
                                                T off[3], T& h, Meta<D>& w) {
        Vec4<T> p = P[j];
        off[0] = p.x;
        off[1] = p.y;
        if constexpr (packed) {
            off[2] = T(0);
            h = p.z;
            w = __float_as_uint((float)p.w);
        } else {
            off[2] = p.z;
            h = p.w;
            w = M[j];
        }
    }
    __device__ __forceinline__ static void store(Vec4<T>* P, Meta<D>* M, int j, const T off[3], T h, Meta<D> w) {
        Vec4<T> p;
        p.x = off[0];
        p.y = off[1];
        if constexpr (packed) {
            p.z = h;
            p.w = (T)__uint_as_float(w);
        } else {
            p.z = off[2];
            p.w = h;
        }
        P[j] = p;
        M[j] = w;
    }
};

__device__ __forceinline__ int meta_group(unsigned m) { return (int)(m & 63u); }
__device__ __forceinline__ int meta_dim(unsigned m) { return (int)((m >> 6) & 3u); }

// level of a smoothing length: first l with h <= thr[l] (the top level takes the rest)
template <typename T> __device__ __forceinline__ int level_of(const Grid& g, T h) {
    int l = 0;
    while (l < g.L - 1 && h > (T)g.thr[l]) ++l;
    return l;
}

// Positions are stored as the finest-level cell (integers) and the offset from that cell's
// origin in the working precision.  From an FP64 position:
//   c = floor((x - origin) * inv_c0) (clamped into the finest grid), o = (x - origin) - c * c0
template <typename T, int D>
__device__ __forceinline__ bool fine_of(const Grid& g, const double x[3], int c[3], T o[3]) {
    bool clamped = false;
    for (int a = 0; a < 3; ++a) {
        if (a >= D) { c[a] = 0; o[a] = T(0); continue; }
        double rel = __dsub_rn(x[a], (double)g.origin[a]);
        double t = floor(__dmul_rn(rel, g.inv_c[0]));
        int ca = (int)fmax(fmin(t, 2.0e9), -2.0e9);
        if (ca < 0) { ca = 0; clamped = true; }
        if (ca > g.dims[0][a] - 1) { ca = g.dims[0][a] - 1; clamped = true; }
        c[a] = ca;
        o[a] = (T)__dsub_rn(rel, __dmul_rn((double)ca, g.c[0]));
    }
    return clamped;
}

// the FP64 position of a stored (finest cell, offset) pair
template <typename T, int D> __device__ __forceinline__ void pos64(const Grid& g, const int c[3], const T o[3], double x[3]) {
    for (int a = 0; a < 3; ++a)
        x[a] = a < D ? __dadd_rn(__dadd_rn((double)g.origin[a], __dmul_rn((double)c[a], g.c[0])), (double)o[a]) : 0.0;
}

// the same position in the working precision (for the sizing function, the level-set
// pre-check and tangent directions; absolute error ~ the precision of |x|)
template <typename T, int D> __device__ __forceinline__ void pos_t(const Grid& g, const int c[3], const T o[3], T x[3]) {
    for (int a = 0; a < 3; ++a) x[a] = a < D ? (T)g.origin[a] + (T)c[a] * (T)g.c0 + o[a] : T(0);
}

// level-l representation derived from the stored one, each operation rounded in T:
//   cell = c >> l, off = o + (c - (cell << l)) * c0
template <typename T, int D>
__device__ __forceinline__ void level_repr(const Grid& g, int l, const int c[3], const T o[3], int cell[3], T off[3]) {
    for (int a = 0; a < 3; ++a) {
        if (a >= D) { cell[a] = 0; off[a] = T(0); continue; }
        cell[a] = c[a] >> l;
        off[a] = rn_add(o[a], rn_mul((T)(c[a] - (cell[a] << l)), (T)g.c0));
    }
}

__device__ __forceinline__ int key_of(const Grid& g, int l, const int cell[3]) {
    return g.base[l] + (cell[2] * g.dims[l][1] + cell[1]) * g.dims[l][0] + cell[0];
}

// ---- analytic geometry (FP64) ----
__device__ __forceinline__ double dnorm3(const double v[3]) { return sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]); }

__device__ inline double sizing_h(const Sizing& s, const double x[3]) {
    if (s.kind == 0) return s.a;
    double h;
    if (s.kind == 1) {
        double dmin = 1e300;
        for (int k = 0; k < s.nref; ++k) {
            double d[3] = {x[0] - s.rc[k][0], x[1] - s.rc[k][1], x[2] - s.rc[k][2]};
            double dk = fabs(dnorm3(d) - s.rr[k]);
            dmin = fmin(dmin, dk);
        }
        h = s.a + s.b * dmin;
    } else {
        double d[3] = {x[0] - s.q[0], x[1] - s.q[1], x[2] - s.q[2]};
        h = s.a + s.b * dnorm3(d);
    }
    return fmin(fmax(h, s.lo), s.hi);
}

// level set of the domain and its gradient (positive inside)
__device__ inline double domain_phi(const Domain& dom, const double x[3], double grad[3]) {
    double phi = 1e300;
    grad[0] = grad[1] = grad[2] = 0.0;
    if (dom.base == 0) {
        for (int a = 0; a < dom.D; ++a) {
            double dlo = x[a] - dom.lo[a], dhi = dom.hi[a] - x[a];
            if (dlo < phi) { phi = dlo; grad[0] = grad[1] = grad[2] = 0.0; grad[a] = 1.0; }
            if (dhi < phi) { phi = dhi; grad[0] = grad[1] = grad[2] = 0.0; grad[a] = -1.0; }
        }
    } else {
        double d[3] = {x[0] - dom.bc[0], x[1] - dom.bc[1], dom.D == 3 ? x[2] - dom.bc[2] : 0.0};
        double r = dnorm3(d);
        phi = dom.br - r;
        for (int a = 0; a < 3; ++a) grad[a] = r > 0 ? -d[a] / r : (a == 0 ? -1.0 : 0.0);
    }
    for (int k = 0; k < dom.nh; ++k) {
        double d[3] = {x[0] - dom.hc[k][0], x[1] - dom.hc[k][1], dom.D == 3 ? x[2] - dom.hc[k][2] : 0.0};
        double r = dnorm3(d);
        double pk = r - dom.hr[k];
        if (pk < phi) {
            phi = pk;
            for (int a = 0; a < 3; ++a) grad[a] = r > 0 ? d[a] / r : (a == 0 ? 1.0 : 0.0);
        }
    }
    return phi;
}

// closest point on a curve / surface / point feature (FP64)
__device__ inline void project_feature(const Feat& f, int D, double x[3]) {
    if (f.kind == K_POINT) {
        for (int a = 0; a < 3; ++a) x[a] = a < D ? f.g[a] : 0.0;
    } else if (f.kind == K_SEGMENT) {
        double ab[3], ax[3];
        for (int a = 0; a < 3; ++a) { ab[a] = f.g[3 + a] - f.g[a]; ax[a] = x[a] - f.g[a]; }
        double t = (ax[0] * ab[0] + ax[1] * ab[1] + ax[2] * ab[2]) / (ab[0] * ab[0] + ab[1] * ab[1] + ab[2] * ab[2]);
        t = fmin(fmax(t, 0.0), 1.0);
        for (int a = 0; a < 3; ++a) x[a] = f.g[a] + t * ab[a];
    } else if (f.kind == K_CIRCLE || f.kind == K_SPHERE) {
        double c[3] = {f.g[0], f.g[1], f.kind == K_SPHERE ? f.g[2] : 0.0};
        double R = f.kind == K_SPHERE ? f.g[3] : f.g[2];
        double d[3] = {0, 0, 0};
        for (int a = 0; a < D; ++a) d[a] = x[a] - c[a];
        double r = dnorm3(d);
        for (int a = 0; a < 3; ++a) {
            double u = r > 0 ? d[a] / r : (a == 0 ? 1.0 : 0.0);
            x[a] = a < D ? c[a] + R * u : 0.0;
        }
    } else if (f.kind == K_RECT) {
        double ox[3];
        for (int a = 0; a < 3; ++a) ox[a] = x[a] - f.g[a];
        double s = ox[0] * f.g[3] + ox[1] * f.g[4] + ox[2] * f.g[5];
        double t = ox[0] * f.g[6] + ox[1] * f.g[7] + ox[2] * f.g[8];
        s = fmin(fmax(s, 0.0), f.g[9]);
        t = fmin(fmax(t, 0.0), f.g[10]);
        for (int a = 0; a < 3; ++a) x[a] = f.g[a] + s * f.g[3 + a] + t * f.g[6 + a];
    }
}

// the tangent-space descriptor of a particle of feature f at position x: unit tangent for
// curves (SEGMENT, CIRCLE), unit normal for surfaces (RECT, SPHERE)
template <typename T> __device__ inline void feature_tangent(const Feat& f, const T x[3], T tg[3]) {
    tg[0] = tg[1] = tg[2] = T(0);
    if (f.kind == K_SEGMENT || f.kind == K_RECT) {
        for (int a = 0; a < 3; ++a) tg[a] = (T)f.ftg[a];
        if (sizeof(T) == 8) {   // FP64 build: exact descriptor
            if (f.kind == K_RECT) { for (int a = 0; a < 3; ++a) tg[a] = (T)f.nb[a]; }
            else {
                double ab[3] = {f.g[3] - f.g[0], f.g[4] - f.g[1], f.g[5] - f.g[2]};
                double L = dnorm3(ab);
                for (int a = 0; a < 3; ++a) tg[a] = (T)(ab[a] / L);
            }
        }
    } else if (f.kind == K_CIRCLE) {
        T d0 = x[0] - (T)f.g[0], d1 = x[1] - (T)f.g[1];
        T r = t_sqrt(d0 * d0 + d1 * d1);
        T u0 = r > T(0) ? d0 / r : T(1), u1 = r > T(0) ? d1 / r : T(0);
        tg[0] = -u1;
        tg[1] = u0;
    } else if (f.kind == K_SPHERE) {
        T d[3] = {x[0] - (T)f.g[0], x[1] - (T)f.g[1], x[2] - (T)f.g[2]};
        T r = t_sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
        for (int a = 0; a < 3; ++a) tg[a] = r > T(0) ? d[a] / r : (a == 0 ? T(1) : T(0));
    }
}

// v <- Pi v : identity (volume), t t^T (curves), I - n n^T (surfaces), 0 (points)
template <typename T> __device__ __forceinline__ void tangent_map(int dim, int D, const T tg[3], T v[3]) {
    if (dim == D) return;
    if (dim == 0) { v[0] = v[1] = v[2] = T(0); return; }
    T s = v[0] * tg[0] + v[1] * tg[1] + v[2] * tg[2];
    if (dim == 1) { for (int a = 0; a < 3; ++a) v[a] = s * tg[a]; }
    else { for (int a = 0; a < 3; ++a) v[a] = v[a] - s * tg[a]; }
}

// outward normal n_b of a boundary particle of feature f at (absolute) position x
template <typename T> __device__ __forceinline__ void boundary_normal(const Feat& f, const T x[3], T nb[3]) {
    if (f.kind == K_CIRCLE || f.kind == K_SPHERE) {
        T d[3] = {x[0] - (T)f.fc[0], x[1] - (T)f.fc[1], f.kind == K_SPHERE ? x[2] - (T)f.fc[2] : T(0)};
        if (sizeof(T) == 8) {
            d[0] = x[0] - (T)f.g[0];
            d[1] = x[1] - (T)f.g[1];
            if (f.kind == K_SPHERE) d[2] = x[2] - (T)f.g[2];
        }
        T r = t_sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
        T s = (T)f.forient / (r > T(0) ? r : T(1));
        for (int a = 0; a < 3; ++a) nb[a] = s * d[a];
    } else {
        for (int a = 0; a < 3; ++a) nb[a] = sizeof(T) == 8 ? (T)f.nb[a] : (T)f.fnb[a];
    }
}

// the two predicates of the pair sums, evaluated op by op:
//   pair: r2 < ((h_i + h_j) * kappa/2)^2   (j != i);   self: r2 < (kappa h_i)^2
template <typename T> __device__ __forceinline__ T pair_rc2(T hi, T hj, T half_kappa) {
    T rc = rn_mul(rn_add(hi, hj), half_kappa);
    return rn_mul(rc, rc);
}
template <typename T> __device__ __forceinline__ T self_rc2(T hi, T kappa) {
    T rc = rn_mul(hi, kappa);
    return rn_mul(rc, rc);
}

// ---- reciprocal / reciprocal square root for the pair arithmetic (not the predicate) ----
__device__ __forceinline__ float fast_rcp(float v) {   // normal v: within 1 ulp
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
// correctly rounded: the FP64 build is the one that reference results come from (one Newton step from
// the hardware's estimate, a few results in ten thousand an ulp off and NaN for 0 and infinity: 916 us
// per step against 960 on the 40k cube)
__device__ __forceinline__ double fast_rcp(double v) { return 1.0 / v; }
__device__ __forceinline__ float fast_rsqrt(float v) { return rsqrtf(v); }
__device__ __forceinline__ double fast_rsqrt(double v) { return 1.0 / sqrt(v); }
// sqrt(v) for v >= 0 (float: v times its reciprocal root, within 2 ulp for normal v)
__device__ __forceinline__ float root_of(float v) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaxf(v, 1.2e-38f)));
    return v * r;
}
__device__ __forceinline__ double root_of(double v) { return sqrt(v); }

__device__ __forceinline__ float pos_part(float v) { return fmaxf(v, 0.0f); }
__device__ __forceinline__ double pos_part(double v) { return fmax(v, 0.0); }

// The kernel factor of a pair, S2 W'(r)/r for the Wendland C2 kernel with support 1/invR in d
// dimensions and S2 = rho_i^-2 + rho_j^-2: -20 alpha_d S2 (1-q)^3 / R^2, zero outside the support.
// S2 ~ h^(2d) meets part of R^-(d+2) first: alone, that power leaves the single-precision range for
// 2D spacings below 2e-10, where S2 is still a number.
template <typename T> __device__ __forceinline__ T kernel_factor(int d, T S2, T r, T invR) {
    const T t = pos_part(T(1) - r * invR), i2 = invR * invR;
    const T a = d == 1 ? T(-30) * invR : d == 2 ? T(-140.0 / CUDART_PI) * i2 : T(-210.0 / CUDART_PI) * (i2 * invR);
    return (S2 * i2) * a * (t * t * t);
}

// 2 a b / (a + b) for a, b >= 0 (0 where the sum is 0)
template <typename T> __device__ __forceinline__ T harmonic(T a, T b) {
    const T s = rn_add(a, b);
    return s > T(0) ? rn_mul(rn_mul(T(2), a), b) / s : T(0);
}

// sum over the LPP lanes of one particle (xor butterfly: every lane gets the same bits).  The
// lanes of a particle are consecutive and aligned, and the mask names only them: a caller may
// branch per particle (all lanes of a particle take the same branch).
template <int LPP, typename T> __device__ __forceinline__ T sub_sum(T v) {
    static_assert(LPP >= 1 && LPP <= 32 && (LPP & (LPP - 1)) == 0, "lanes per particle: a power of two");
    const unsigned mask =
        LPP == 32 ? 0xffffffffu : ((1u << (LPP & 31)) - 1u) << ((threadIdx.x & 31u) & ~(unsigned)(LPP - 1));
#pragma unroll
    for (int o = 1; o < LPP; o <<= 1) v += __shfl_xor_sync(mask, v, o);
    return v;
}

}  // namespace sph
