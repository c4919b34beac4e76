// sample.cu -- the initial particle set on the device (Sec. 3.6; Algorithm 1: "calculate the
// target information (Eqs. 10, 11)" and "allocate particles ... initial particle sampling").
//
// Target counts: N_k = integral over feature k of rho_t = h_t^-d (Eqs. 10, 11), by the midpoint
// rule on a fixed grid of the feature's parameter space (volume: the bounding box, cells whose
// centre has phi > 0); per-block FP64 partial sums added on the host in block order.
//
// Sampling: particles of feature k are drawn with probability proportional to rho_t by
// rejection.  Candidate c of feature k takes the four 32-bit outputs of Philox4x32-10 (Salmon,
// Moraes, Dror, Shaw, SC 2011) for counter (c, c >> 32, k, 0) under the key (seed, seed >> 32),
// as uniforms u = (x + 1/2) 2^-32; it is accepted with probability (h_min/h_t(x))^d (h_min the
// sizing's lower bound), volume candidates only where phi(x) > h_t(x)/4, face candidates only
// h_t/4 inside the face's edges, and feature k keeps its first N_k accepted candidates in
// candidate order.  Every FP64 operation that decides acceptance is rounded one by one, so a
// candidate is accepted or rejected exactly as by any other correctly rounded evaluation of
// the same expressions.
#include "sph_internal.cuh"

#include <algorithm>
#include <vector>

namespace sph {

namespace {

constexpr int SB = 256;   // threads per block of the sampling kernels

__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double ddiv(double a, double b) { return __ddiv_rn(a, b); }

// |x - c| over the first n components, summed in component order
__device__ double dist_n(const double x[3], const double* c, int n) {
    double s = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double d = a < n ? dsub(x[a], c[a]) : 0.0;
        s = dadd(s, dmul(d, d));
    }
    return __dsqrt_rn(s);
}

// h_t(x) (Eq. 2, the analytic sizing) in FP64
__device__ double samp_h(const Sizing& z, const double x[3]) {
    if (z.kind == 0) return z.a;
    double h;
    if (z.kind == 1) {
        double dmin = 1.7976931348623157e308;
        for (int k = 0; k < z.nref; ++k) {
            const double dk = fabs(dsub(dist_n(x, z.rc[k], 3), z.rr[k]));
            if (dk < dmin) dmin = dk;
        }
        h = dadd(z.a, dmul(z.b, dmin));
    } else {
        h = dadd(z.a, dmul(z.b, dist_n(x, z.q, 3)));
    }
    if (h < z.lo) h = z.lo;
    if (h > z.hi) h = z.hi;
    return h;
}

// the level set phi(x) (Eq. 1): box or ball minus the holes, in FP64
__device__ double samp_phi(const Domain& dm, const double x[3]) {
    double phi = 1.7976931348623157e308;
    if (dm.base == 0) {
        for (int a = 0; a < dm.D; ++a) {
            const double dlo = dsub(x[a], dm.lo[a]), dhi = dsub(dm.hi[a], x[a]);
            if (dlo < phi) phi = dlo;
            if (dhi < phi) phi = dhi;
        }
    } else {
        phi = dsub(dm.br, dist_n(x, dm.bc, dm.D));
    }
    for (int k = 0; k < dm.nh; ++k) {
        const double pk = dsub(dist_n(x, dm.hc[k], dm.D), dm.hr[k]);
        if (pk < phi) phi = pk;
    }
    return phi;
}

// Philox4x32-10: ten rounds of the Philox S-box, the key advanced by the Weyl constants between
// rounds (Salmon et al., SC 2011)
__device__ __forceinline__ void philox(unsigned c[4], unsigned k0, unsigned k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const unsigned lo0 = 0xD2511F53u * c[0], hi0 = __umulhi(0xD2511F53u, c[0]);
        const unsigned lo1 = 0xCD9E8D57u * c[2], hi1 = __umulhi(0xCD9E8D57u, c[2]);
        const unsigned n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = lo1;
        c[2] = n2;
        c[3] = lo0;
    }
}

__device__ __forceinline__ void uniforms(unsigned long long seed, int k, long long c, double u[4]) {
    unsigned w[4] = {(unsigned)c, (unsigned)((unsigned long long)c >> 32), (unsigned)k, 0u};
    philox(w, (unsigned)seed, (unsigned)(seed >> 32));
#pragma unroll
    for (int a = 0; a < 4; ++a) u[a] = ((double)w[a] + 0.5) * (1.0 / 4294967296.0);
}

// acceptance of candidate u of feature f, and its position
__device__ bool accept(const Domain& dm, const Sizing& z, const Feat& f, const double u[4], double x[3]) {
    x[0] = x[1] = x[2] = 0.0;
    const int D = dm.D;
    switch (f.kind) {
        case SPH_FEAT_VOLUME: {
            for (int a = 0; a < D; ++a) x[a] = dadd(dm.lo[a], dmul(u[a], dsub(dm.hi[a], dm.lo[a])));
            const double h = samp_h(z, x);
            if (!(samp_phi(dm, x) > dmul(0.25, h))) return false;
            const double r = ddiv(z.lo, h);
            double rd = dmul(r, r);
            if (D == 3) rd = dmul(rd, r);
            return u[3] < rd;
        }
        case SPH_FEAT_SEGMENT:
            for (int a = 0; a < 3; ++a) x[a] = dadd(f.g[a], dmul(u[0], dsub(f.g[3 + a], f.g[a])));
            return u[1] < ddiv(z.lo, samp_h(z, x));
        case SPH_FEAT_CIRCLE: {
            const double p0 = dsub(dmul(2.0, u[0]), 1.0), p1 = dsub(dmul(2.0, u[1]), 1.0);
            const double q = dadd(dmul(p0, p0), dmul(p1, p1));
            if (!(q > 0.0 && q <= 1.0)) return false;
            const double r = __dsqrt_rn(q);
            x[0] = dadd(f.g[0], dmul(f.g[2], ddiv(p0, r)));
            x[1] = dadd(f.g[1], dmul(f.g[2], ddiv(p1, r)));
            return u[2] < ddiv(z.lo, samp_h(z, x));
        }
        case SPH_FEAT_SPHERE: {
            const double p0 = dsub(dmul(2.0, u[0]), 1.0), p1 = dsub(dmul(2.0, u[1]), 1.0),
                         p2 = dsub(dmul(2.0, u[2]), 1.0);
            const double q = dadd(dadd(dmul(p0, p0), dmul(p1, p1)), dmul(p2, p2));
            if (!(q > 0.0 && q <= 1.0)) return false;
            const double r = __dsqrt_rn(q);
            x[0] = dadd(f.g[0], dmul(f.g[3], ddiv(p0, r)));
            x[1] = dadd(f.g[1], dmul(f.g[3], ddiv(p1, r)));
            x[2] = dadd(f.g[2], dmul(f.g[3], ddiv(p2, r)));
            const double acc = ddiv(z.lo, samp_h(z, x));
            return u[3] < dmul(acc, acc);
        }
        case SPH_FEAT_RECT: {
            const double sv = dmul(u[0], f.g[9]), tv = dmul(u[1], f.g[10]);
            for (int a = 0; a < 3; ++a) x[a] = dadd(dadd(f.g[a], dmul(sv, f.g[3 + a])), dmul(tv, f.g[6 + a]));
            const double h = samp_h(z, x);
            const double m = dmul(0.25, h);
            if (!(sv > m && sv < dsub(f.g[9], m) && tv > m && tv < dsub(f.g[10], m))) return false;
            const double acc = ddiv(z.lo, h);
            return u[2] < dmul(acc, acc);
        }
        default:
            for (int a = 0; a < D; ++a) x[a] = f.g[a];
            return true;
    }
}

// One pass over candidates of several features: blocks block0[q] .. block0[q + 1] take the next
// candidates, from c0[q] on, of feature k[q], which wants its first want[q] accepted ones at
// out0[q] (particles).
struct SamplePass {
    int n;
    int k[MAXF];
    int block0[MAXF + 1];
    long long c0[MAXF], want[MAXF], out0[MAXF];
};
__device__ __forceinline__ int pass_entry(const SamplePass& ps) {
    int q = 0;
    while (q + 1 < ps.n && (int)blockIdx.x >= ps.block0[q + 1]) ++q;
    return q;
}

// pass 1: accepted candidates per block
__global__ void __launch_bounds__(SB) k_sample_count(const Domain* dmp, const Sizing* zp, unsigned long long seed,
                                                     const __grid_constant__ SamplePass ps, int* block_count) {
    const Domain& dm = *dmp;
    const int q = pass_entry(ps), k = ps.k[q];
    double u[4], x[3];
    uniforms(seed, k, ps.c0[q] + (long long)(blockIdx.x - ps.block0[q]) * SB + threadIdx.x, u);
    const int n = __syncthreads_count(accept(dm, *zp, dm.f[k], u, x) ? 1 : 0);
    if (threadIdx.x == 0) block_count[blockIdx.x] = n;
}

// pass 2: accepted candidates written in candidate order, the first `want` of them (block_off: the
// accepted candidates of the block's feature before it)
__global__ void __launch_bounds__(SB) k_sample_emit(const Domain* dmp, const Sizing* zp, unsigned long long seed,
                                                    const __grid_constant__ SamplePass ps, const long long* block_off,
                                                    double* out) {
    __shared__ int wsum[SB / 32];
    const Domain& dm = *dmp;
    const int q = pass_entry(ps), k = ps.k[q];
    double u[4], x[3] = {0.0, 0.0, 0.0};
    uniforms(seed, k, ps.c0[q] + (long long)(blockIdx.x - ps.block0[q]) * SB + threadIdx.x, u);
    const bool ok = accept(dm, *zp, dm.f[k], u, x);
    const unsigned bal = __ballot_sync(0xffffffffu, ok);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) wsum[wid] = __popc(bal);
    __syncthreads();
    int before = 0;
    for (int w = 0; w < wid; ++w) before += wsum[w];
    const long long rank = block_off[blockIdx.x] + before + __popc(bal & ((1u << lane) - 1u));
    if (ok && rank < ps.want[q])
        for (int a = 0; a < 3; ++a) out[3 * (ps.out0[q] + rank) + a] = x[a];
}

// phi(x) > 0 as samp_phi has it.  Single precision decides wherever the level set is clearly off
// zero (by far more than its rounding, 2^-20 of the domain's size); the FP64 expressions only
// close to the boundary.
__device__ __forceinline__ bool inside(const Domain& dm, const double x[3], const float xf[3], float size) {
    float phi = 3e38f;
    if (dm.base == 0) {
        for (int a = 0; a < dm.D; ++a) phi = fminf(phi, fminf(xf[a] - dm.flo[a], dm.fhi[a] - xf[a]));
    } else {
        float s = 0.0f;
        for (int a = 0; a < dm.D; ++a) s = fmaf(xf[a] - dm.fbc[a], xf[a] - dm.fbc[a], s);
        phi = dm.fbr - sqrtf(s);
    }
    for (int k = 0; k < dm.nh; ++k) {
        float s = 0.0f;
        for (int a = 0; a < dm.D; ++a) s = fmaf(xf[a] - dm.fhc[k][a], xf[a] - dm.fhc[k][a], s);
        phi = fminf(phi, sqrtf(s) - dm.fhr[k]);
    }
    if (fabsf(phi) > size * 0x1p-16f) return phi > 0.0f;
    return samp_phi(dm, x) > 0.0;
}

// h_t(x) of a point of the volume, bit for bit as samp_h has it (sx2: (x_0 - c_0)^2 of the one
// reference, formed before the loop).  With several reference circles or spheres, only the nearest
// one's distance is formed in FP64 where single precision shows which it is (by far more than its
// rounding, 2^-20 of the domain's size).
__device__ __forceinline__ double quad_h(const Sizing& z, const double x[3], const float xf[3], float size, double sx2) {
    if (z.kind != 1 || z.nref < 1) return samp_h(z, x);
    double d;
    if (z.nref == 1) {
        const double d1 = dsub(x[1], z.rc[0][1]), d2 = dsub(x[2], z.rc[0][2]);
        d = fabs(dsub(__dsqrt_rn(dadd(dadd(sx2, dmul(d1, d1)), dmul(d2, d2))), z.rr[0]));
    } else {
        float best = 3e38f, next = 3e38f;
        int kb = 0;
        for (int k = 0; k < z.nref; ++k) {
            float s = 0.0f;
            for (int a = 0; a < 3; ++a) s = fmaf(xf[a] - z.frc[k][a], xf[a] - z.frc[k][a], s);
            const float dk = fabsf(sqrtf(s) - z.frr[k]);
            if (dk < best) {
                next = best;
                best = dk;
                kb = k;
            } else {
                next = fminf(next, dk);
            }
        }
        if (!(next - best > size * 0x1p-16f)) return samp_h(z, x);
        d = fabs(dsub(dist_n(x, z.rc[kb], 3), z.rr[kb]));
    }
    double h = dadd(z.a, dmul(z.b, d));
    if (h < z.lo) h = z.lo;
    if (h > z.hi) h = z.hi;
    return h;
}

// i + 1/2 for 0 <= i < 2^31, exactly, in one FP64 subtraction (a conversion from an integer runs on the
// same narrow pipe, and the addition comes on top)
__device__ __forceinline__ double mid(int i) { return dsub(__hiloint2double(0x43300000, i), 4503599627370495.5); }

// Midpoint-rule integral of rho_t over feature k (Eqs. 10, 11), per-block partial sums.  The
// quadrature sizes are powers of two (nq = 2^ln), so the divisions by nq are exact and a point's
// indices are bits of its number; what does not depend on the point is computed before the loop.
// Where a feature's measure over h^d is an odd multiple of 1/2 (constant spacing) the rounding of
// the terms and the order of their sum decide the rounded count: the terms use correctly rounded
// roots and quotients, and every feature is summed over the same QUAD_BLOCKS blocks of SB threads
// whatever its size.  (Roots and reciprocals by one Newton step, within an ulp, and fewer blocks for
// the small features gave other counts in 14 of 821 such features.)
// Bound by the FP64 pipe, two multiply-adds per SM and clock: a volume point costs one root and one
// quotient, and two coordinates, since a thread's points share their first one (its stride is a
// multiple of nq); the single-precision coordinates that decide the filters come from the indices.
// All features of a cube take 1.82 ms, of a disk 0.35 (coordinates and conversions per point: 2.19
// and 0.43; one launch per feature, with quotients per point for the cell size and a second root for
// the level set: 4.41 and 1.49).
constexpr int QUAD_BLOCKS = 4 * 152;
template <int KIND>
__device__ __forceinline__ double integral_share(const Domain& dm, const Sizing& z, const Feat& f, long long npts, int ln,
                                                 int block) {
    const int D = dm.D, nq = 1 << ln, last = nq - 1;
    const double inq = 1.0 / nq;
    float size = 0.0f;   // of the domain, with its distance from the origin
    for (int a = 0; a < D; ++a) size = fmaxf(size, fmaxf(fabsf(dm.flo[a]), fabsf(dm.fhi[a])));
    for (int q = 0; q < z.nref; ++q)
        for (int a = 0; a < 3; ++a) size = fmaxf(size, fabsf(z.frc[q][a]) + z.frr[q]);
    for (int q = 0; q < dm.nh; ++q)
        for (int a = 0; a < D; ++a) size = fmaxf(size, fabsf(dm.fhc[q][a]) + dm.fhr[q]);
    if (dm.base != 0)
        for (int a = 0; a < D; ++a) size = fmaxf(size, fabsf(dm.fbc[a]) + dm.fbr);
    double dx[3] = {0.0, 0.0, 0.0}, cell = 1.0;
    if (KIND == SPH_FEAT_VOLUME)
        for (int a = 0; a < D; ++a) {
            dx[a] = (dm.hi[a] - dm.lo[a]) * inq;
            cell *= dx[a];
        }
    if (KIND == SPH_FEAT_SEGMENT) {
        double L2 = 0.0;
        for (int a = 0; a < 3; ++a) {
            dx[a] = f.g[3 + a] - f.g[a];
            L2 += dx[a] * dx[a];
        }
        cell = sqrt(L2) * inq;
    }
    if (KIND == SPH_FEAT_CIRCLE) cell = 2.0 * CUDART_PI * f.g[2] * inq;
    if (KIND == SPH_FEAT_RECT) cell = (f.g[9] * inq) * (f.g[10] * inq);
    double x0 = 0.0, sx2 = 0.0;
    float xf0 = 0.0f, dxf[3] = {0.0f, 0.0f, 0.0f};
    if (KIND == SPH_FEAT_VOLUME) {
        static_assert(QUAD_BLOCKS * SB % SPH_QUAD_VOLUME == 0 && QUAD_BLOCKS * SB % SPH_QUAD_AREA == 0,
                      "the points of a thread share their first coordinate");
        x0 = fma(mid((block * SB + (int)threadIdx.x) & last), dx[0], dm.lo[0]);
        xf0 = (float)x0;
        const double d0 = dsub(x0, z.rc[0][0]);
        sx2 = dmul(d0, d0);
        for (int a = 0; a < D; ++a) dxf[a] = (float)dx[a];
    }
    double acc = 0.0;
    for (long long i = (long long)block * SB + threadIdx.x; i < npts; i += (long long)QUAD_BLOCKS * SB) {
        double x[3] = {0.0, 0.0, 0.0};
        if (KIND == SPH_FEAT_VOLUME) {
            x[0] = x0;
            float xf[3] = {xf0, 0.0f, 0.0f};
            for (int a = 1; a < D; ++a) {
                const int ia = (int)(i >> (a * ln)) & last;
                x[a] = fma(mid(ia), dx[a], dm.lo[a]);
                xf[a] = fmaf((float)ia + 0.5f, dxf[a], dm.flo[a]);
            }
            if (inside(dm, x, xf, size)) {
                const double h = quad_h(z, x, xf, size, sx2);
                acc += cell / (D == 3 ? h * h * h : h * h);
            }
        } else if (KIND == SPH_FEAT_SEGMENT) {
            const double t = (i + 0.5) * inq;
            for (int a = 0; a < 3; ++a) x[a] = f.g[a] + t * dx[a];
            acc += cell / samp_h(z, x);
        } else if (KIND == SPH_FEAT_CIRCLE) {
            const double th = 2.0 * CUDART_PI * (i + 0.5) * inq;
            x[0] = f.g[0] + f.g[2] * cos(th);
            x[1] = f.g[1] + f.g[2] * sin(th);
            acc += cell / samp_h(z, x);
        } else if (KIND == SPH_FEAT_RECT) {
            const double si = (((int)i & last) + 0.5) * inq * f.g[9], tj = ((int)(i >> ln) + 0.5) * inq * f.g[10];
            for (int a = 0; a < 3; ++a) x[a] = f.g[a] + si * f.g[3 + a] + tj * f.g[6 + a];
            const double h = samp_h(z, x);
            acc += cell / (h * h);
        } else if (KIND == SPH_FEAT_SPHERE) {
            const int ii = (int)(i >> (ln + 1)), jj = (int)i & (2 * nq - 1);
            const double th = CUDART_PI * (ii + 0.5) * inq, ph = CUDART_PI * (jj + 0.5) * inq;
            const double R = f.g[3];
            double st, ct, sp, cp;
            sincos(th, &st, &ct);
            sincos(ph, &sp, &cp);
            x[0] = f.g[0] + R * st * cp;
            x[1] = f.g[1] + R * st * sp;
            x[2] = f.g[2] + R * ct;
            const double h = samp_h(z, x);
            acc += R * R * st * (CUDART_PI * inq) * (CUDART_PI * inq) / (h * h);
        }
    }
    return acc;
}

// all features in one launch: blocks block0[q] .. block0[q + 1] share the points of feature k[q]
struct IntegralPass {
    int n;
    int k[MAXF], ln[MAXF], block0[MAXF + 1];
    long long npts[MAXF];
};
__global__ void __launch_bounds__(SB) k_feature_integrals(const Domain* dmp, const Sizing* zp,
                                                          const __grid_constant__ IntegralPass ip, double* partial) {
    __shared__ double ws[SB / 32];
    int q = 0;
    while (q + 1 < ip.n && (int)blockIdx.x >= ip.block0[q + 1]) ++q;
    const Domain& dm = *dmp;
    const Feat& f = dm.f[ip.k[q]];
    const int block = blockIdx.x - ip.block0[q], ln = ip.ln[q];
    double acc = 0.0;
    switch (f.kind) {
        case SPH_FEAT_VOLUME: acc = integral_share<SPH_FEAT_VOLUME>(dm, *zp, f, ip.npts[q], ln, block); break;
        case SPH_FEAT_SEGMENT: acc = integral_share<SPH_FEAT_SEGMENT>(dm, *zp, f, ip.npts[q], ln, block); break;
        case SPH_FEAT_CIRCLE: acc = integral_share<SPH_FEAT_CIRCLE>(dm, *zp, f, ip.npts[q], ln, block); break;
        case SPH_FEAT_RECT: acc = integral_share<SPH_FEAT_RECT>(dm, *zp, f, ip.npts[q], ln, block); break;
        case SPH_FEAT_SPHERE: acc = integral_share<SPH_FEAT_SPHERE>(dm, *zp, f, ip.npts[q], ln, block); break;
        default: break;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < SB / 32; ++w) s += ws[w];
        partial[blockIdx.x] = s;
    }
}

constexpr bool power_of_two(int n) { return n > 0 && (n & (n - 1)) == 0; }
static_assert(power_of_two(SPH_QUAD_AREA) && power_of_two(SPH_QUAD_VOLUME) && power_of_two(SPH_QUAD_CURVE) &&
                  power_of_two(SPH_QUAD_FACE) && power_of_two(SPH_QUAD_SPHERE),
              "integral_share takes a point's indices from the bits of its number");

}  // namespace

int quad_points(int kind, int D, long long* npts) {
    int nq = 0;
    switch (kind) {
        case SPH_FEAT_VOLUME:
            nq = D == 2 ? SPH_QUAD_AREA : SPH_QUAD_VOLUME;
            *npts = D == 2 ? (long long)nq * nq : (long long)nq * nq * nq;
            break;
        case SPH_FEAT_SEGMENT:
        case SPH_FEAT_CIRCLE:
            nq = SPH_QUAD_CURVE;
            *npts = nq;
            break;
        case SPH_FEAT_RECT:
            nq = SPH_QUAD_FACE;
            *npts = (long long)nq * nq;
            break;
        case SPH_FEAT_SPHERE:
            nq = SPH_QUAD_SPHERE;
            *npts = 2LL * nq * nq;
            break;
        default:
            *npts = 0;
    }
    return nq;
}

cudaError_t feature_integrals(const Domain& dm, const Domain* d_dom, const Sizing* d_siz, cudaStream_t st,
                              double* integral) {
    // One launch, one copy back and one wait for all features: the curves and faces, each too small
    // to fill the GPU, run beside the volume.  Blocks without a point are left out (their sums are 0).
    IntegralPass ip;
    ip.n = 0;
    ip.block0[0] = 0;
    for (int k = 0; k < dm.nf; ++k) {
        if (dm.f[k].kind == SPH_FEAT_POINT) continue;
        long long npts = 0;
        const int nq = quad_points(dm.f[k].kind, dm.D, &npts);
        if (npts == 0) continue;
        int ln = 0;
        while ((1 << ln) < nq) ++ln;
        ip.k[ip.n] = k;
        ip.ln[ip.n] = ln;
        ip.npts[ip.n] = npts;
        ip.block0[ip.n + 1] = ip.block0[ip.n] + (int)std::min<long long>(QUAD_BLOCKS, (npts + SB - 1) / SB);
        ip.n += 1;
    }
    for (int k = 0; k < dm.nf; ++k) integral[k] = dm.f[k].kind == SPH_FEAT_POINT ? 1.0 : 0.0;
    if (ip.n == 0) return cudaSuccess;
    const int nb = ip.block0[ip.n];
    double* d_part = nullptr;
    cudaError_t e = cudaMallocAsync(&d_part, sizeof(double) * nb, st);
    if (e != cudaSuccess) return e;
    std::vector<double> part(nb, 0.0);
    k_feature_integrals<<<nb, SB, 0, st>>>(d_dom, d_siz, ip, d_part);
    e = cudaMemcpyAsync(part.data(), d_part, sizeof(double) * nb, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    for (int q = 0; q < ip.n; ++q) {
        double sum = 0.0;
        for (int b = ip.block0[q]; b < ip.block0[q + 1]; ++b) sum += part[b];
        integral[ip.k[q]] = sum;
    }
    cudaError_t f = cudaFreeAsync(d_part, st);
    if (e == cudaSuccess) e = f;
    if (e == cudaSuccess) e = cudaGetLastError();
    return e;
}

// Expected fraction of accepted candidates of feature k when it holds n particles (n is close to
// the integral of rho_t, so the acceptance (h_min/h)^d averages to n h_min^d / measure), times
// the fraction its geometry keeps (the disc in its square, the ball in its cube)
double acceptance_estimate(const Domain& dm, const Sizing& z, int k, long long n) {
    const Feat& f = dm.f[k];
    const int d = f.dim;
    double meas = 1.0, geo = 1.0;
    switch (f.kind) {
        case SPH_FEAT_VOLUME:
            for (int a = 0; a < dm.D; ++a) meas *= dm.hi[a] - dm.lo[a];
            break;
        case SPH_FEAT_SEGMENT: {
            double L2 = 0.0;
            for (int a = 0; a < 3; ++a) L2 += (f.g[3 + a] - f.g[a]) * (f.g[3 + a] - f.g[a]);
            meas = std::sqrt(L2);
            break;
        }
        case SPH_FEAT_CIRCLE:
            meas = 2.0 * CUDART_PI * f.g[2];
            geo = CUDART_PI / 4.0;
            break;
        case SPH_FEAT_RECT:
            meas = f.g[9] * f.g[10];
            break;
        case SPH_FEAT_SPHERE:
            meas = 4.0 * CUDART_PI * f.g[3] * f.g[3];
            geo = CUDART_PI / 6.0;
            break;
        default:
            return 1.0;
    }
    const double p = geo * (double)n * std::pow(z.lo, d) / meas;
    return std::min(1.0, std::max(p, 1e-9));
}

cudaError_t sample_features(const Domain& dm, const Sizing& z, const Domain* d_dom, const Sizing* d_siz,
                            unsigned long long seed, const int64_t* counts, cudaStream_t st, double* d_out) {
    // Candidates per pass: enough for the remaining count at the expected acceptance, so that one
    // pass usually suffices; a short one is followed by another sized by the acceptance seen so
    // far.  All features share the passes (two kernels and one host round trip each, where one pass
    // per feature took 28 round trips for a cube: 1.2 ms).  The result does not depend on the pass
    // sizes: it is always the first accepted candidates in candidate order.
    constexpr long long MAXB = 1LL << 26;   // candidates per pass
    struct Feature {
        long long got = 0, c0 = 0, seen = 0, taken = 0;
        double p = 1.0;
    };
    std::vector<Feature> fs(dm.nf);
    std::vector<long long> base(dm.nf + 1, 0);
    for (int k = 0; k < dm.nf; ++k) {
        base[k + 1] = base[k] + counts[k];
        if (counts[k] > 0) fs[k].p = acceptance_estimate(dm, z, k, counts[k]);
    }
    int* d_cnt = nullptr;
    long long* d_off = nullptr;
    size_t cap = 0;   // blocks d_cnt and d_off hold
    std::vector<int> cnt;
    std::vector<long long> off;
    cudaError_t e = cudaSuccess;
    while (e == cudaSuccess) {
        SamplePass ps;
        ps.n = 0;
        ps.block0[0] = 0;
        long long room = MAXB;
        for (int k = 0; k < dm.nf; ++k) {
            Feature& f = fs[k];
            if (f.got >= counts[k] || room == 0) continue;
            const double need = (double)(counts[k] - f.got) / f.p;
            long long nc = (long long)(1.05 * need + 6.0 * std::sqrt(need)) + 4096;
            if (dm.f[k].kind == SPH_FEAT_POINT) nc = counts[k];   // every candidate is the point itself
            nc = std::min(room, (nc + SB - 1) / SB * SB);
            ps.k[ps.n] = k;
            ps.c0[ps.n] = f.c0;
            ps.want[ps.n] = counts[k];
            ps.out0[ps.n] = base[k];
            ps.block0[ps.n + 1] = ps.block0[ps.n] + (int)(nc / SB);
            room -= nc;
            ps.n += 1;
        }
        if (ps.n == 0) break;
        const int nblk = ps.block0[ps.n];
        if ((size_t)nblk > cap) {
            if (d_cnt) cudaFreeAsync(d_cnt, st);
            if (d_off) cudaFreeAsync(d_off, st);
            d_cnt = nullptr;
            d_off = nullptr;
            cap = (size_t)nblk;
            e = cudaMallocAsync(&d_cnt, sizeof(int) * cap, st);
            if (e == cudaSuccess) e = cudaMallocAsync(&d_off, sizeof(long long) * cap, st);
            if (e != cudaSuccess) break;
            cnt.resize(cap);
            off.resize(cap);
        }
        k_sample_count<<<nblk, SB, 0, st>>>(d_dom, d_siz, seed, ps, d_cnt);
        e = cudaMemcpyAsync(cnt.data(), d_cnt, sizeof(int) * nblk, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) break;
        for (int q = 0; q < ps.n; ++q) {
            Feature& f = fs[ps.k[q]];
            long long run = f.got;
            for (int b = ps.block0[q]; b < ps.block0[q + 1]; ++b) {
                off[b] = run;
                run += cnt[b];
            }
            const long long nc = (long long)(ps.block0[q + 1] - ps.block0[q]) * SB;
            f.seen += nc;
            f.taken += run - f.got;
            f.got = std::min<long long>(run, counts[ps.k[q]]);
            f.c0 += nc;
            f.p = std::max(1e-9, (double)std::max<long long>(f.taken, 1) / (double)f.seen);
            if (f.got < counts[ps.k[q]] && f.c0 >= (1LL << 36)) e = cudaErrorInvalidValue;   // acceptance too small
        }
        if (e != cudaSuccess) break;
        e = cudaMemcpyAsync(d_off, off.data(), sizeof(long long) * nblk, cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) break;
        k_sample_emit<<<nblk, SB, 0, st>>>(d_dom, d_siz, seed, ps, d_off, d_out);
        e = cudaStreamSynchronize(st);   // off is reused by the next pass
    }
    if (d_cnt) cudaFreeAsync(d_cnt, st);
    if (d_off) cudaFreeAsync(d_off, st);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e;
}

}  // namespace sph
