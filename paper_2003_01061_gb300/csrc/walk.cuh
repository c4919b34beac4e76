// walk.cuh -- what the search and the pair passes share: packed arithmetic, the pair geometry, and
// the search of one warp (by itself in search.cu; in the pair passes for the particles whose
// neighbour list overflowed).
#pragma once
#include "sph_internal.cuh"

namespace sph {

// two single-precision operations in one instruction
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ f32x2 neg2(f32x2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return add2(a, neg2(b)); }

// the warp's smallest value of the Eq. 24 minima's bits (working precision)
template <typename T> __device__ __forceinline__ unsigned long long warp_min_bits(unsigned long long v) {
    if constexpr (sizeof(T) == 4) {
        return __reduce_min_sync(0xffffffffu, (unsigned)v);
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, o);
            v = u < v ? u : v;
        }
        return v;
    }
}

// (T)m for |m| < 2^22 (float: off the conversion pipe, which is narrow)
template <typename T> __device__ __forceinline__ T small_int(int m) {
    if (sizeof(T) == 4) return (T)(__int_as_float(0x4b400000 + m) - 12582912.0f);
    return (T)m;
}

// the lane of the warp, in a register for good (recomputing it from the thread index is slow)
__device__ __forceinline__ int lane_id() {
    int l;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(l));
    return l;
}

// dx = x_i - x_j = (off_i - off_j) + m c0 and r2 = |dx|^2, op by op, m the exact difference of the
// two cell corners
template <typename T, int D>
__device__ __forceinline__ T pair_dx(const T offi[3], const T offj[3], const int m[3], T c0, T dx[3]) {
    dx[0] = rn_add(rn_sub(offi[0], offj[0]), rn_mul(small_int<T>(m[0]), c0));
    dx[1] = rn_add(rn_sub(offi[1], offj[1]), rn_mul(small_int<T>(m[1]), c0));
    dx[2] = D == 3 ? rn_add(rn_sub(offi[2], offj[2]), rn_mul(small_int<T>(m[2]), c0)) : T(0);
    T r2 = rn_add(rn_mul(dx[0], dx[0]), rn_mul(dx[1], dx[1]));
    if (D == 3) r2 = rn_add(r2, rn_mul(dx[2], dx[2]));
    return r2;
}

// two or four consecutive list entries of a lane (aligned to their size)
__device__ __forceinline__ void list_load(const int* p, int (&j)[4]) {
    const int4 v = *reinterpret_cast<const int4*>(p);
    j[0] = v.x, j[1] = v.y, j[2] = v.z, j[3] = v.w;
}
__device__ __forceinline__ void list_load(const int* p, int (&j)[2]) {
    const int2 v = *reinterpret_cast<const int2*>(p);
    j[0] = v.x, j[1] = v.y;
}
template <int U> __device__ __forceinline__ void list_load(const double* p, double (&f)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) f[u] = p[u];
}
__device__ __forceinline__ void list_load(const float* p, float (&f)[4]) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    f[0] = v.x, f[1] = v.y, f[2] = v.z, f[3] = v.w;
}
__device__ __forceinline__ void list_store(float* p, const float (&f)[2]) {
    *reinterpret_cast<float2*>(p) = make_float2(f[0], f[1]);
}
template <int U> __device__ __forceinline__ void list_store(double* p, const double (&f)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) p[u] = f[u];
}
__device__ __forceinline__ void list_store(float* p, const float (&f)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(f[0], f[1], f[2], f[3]);
}

// ---- the search of one warp ----
// Longest segment, in cells of its row, of a warp that searches for cl particles: a longer one has a
// wider bounding box, a shorter one splits more warps.  Measured, whole step in us: 3D, cl = 2 with 1 /
// 2 / 3 / 6, 26k ball in three passes 280 / 280 / 315 / 351; cl = 8 with 3 / 4 / 5 / 6, batch of 340k 724 /
// 728 / 732 / 744; cl = 16 with 4 / 6 / 10, 1.2M cube 1941 / 1925 / 1953; 2D, cl = 8 with 6 / 8 / 10 / 14,
// 120k disk 136.2 / 133.9 / 133.4 / 135.4; cl = 16 with 6 / 12 / 16 / 24, 1M disk 668 / 658 / 655 / 656.
constexpr int seg_span(int D, int cl) {
    return D == 2 ? (cl <= 4 ? 6 : cl == 8 ? 10 : 16) : (cl <= 4 ? 2 : cl == 8 ? 3 : 6);
}

template <int CL> struct alignas(16) SearchWarp {
    float4 me[CL];                   // pairs of particles: (-x, -x', -y, -y'), (-z, -z', a, a')
    float4 near_f[64];               // candidates near the segment's box, a ring
    int near_j[64];
    int delta[32];                   // per non-empty row: its first index minus its offset in the batch
    unsigned long long xid[CL];      // the particles' list blocks so far
};

__device__ __forceinline__ float warp_min_nn(float v) {   // v >= 0: ordered as its bits
    return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ float warp_max_nn(float v) {
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

// Shared memory by its 32-bit address, kept in a register (the compiler would form the address
// anew from the block's window at every access), and stores under a predicate, without a branch.
__device__ __forceinline__ unsigned shared_address(const void* p) {
    unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
    asm volatile("mov.u32 %0, %1;" : "=r"(r) : "r"(a));
    return r;
}
__device__ __forceinline__ float4 lds_f4(unsigned at) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ ulonglong2 lds_u2(unsigned at) {
    ulonglong2 v;
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ int lds_i(unsigned at) {
    int v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ void sts_f(unsigned at, float v) {
    asm volatile("st.shared.f32 [%0], %1;" :: "r"(at), "f"(v) : "memory");
}
__device__ __forceinline__ void sts_if(bool on, unsigned at, int v) {
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n @p st.shared.u32 [%1], %2;\n}"
                 :: "r"((unsigned)on), "r"(at), "r"(v) : "memory");
}
// if (a < b): v to shared address at, j to jat
__device__ __forceinline__ void sts_if_less(float a, float b, unsigned at, float4 v, unsigned jat, int j) {
    asm volatile("{\n .reg .pred p;\n setp.lt.f32 p, %0, %1;\n @p st.shared.v4.f32 [%2], {%3, %4, %5, %6};\n"
                 " @p st.shared.u32 [%7], %8;\n}"
                 :: "f"(a), "f"(b), "r"(at), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(jat), "r"(j) : "memory");
}
// if (a < b): j to p
__device__ __forceinline__ void stg_if_less(float a, float b, char* p, int j) {
    asm volatile("{\n .reg .pred p;\n setp.lt.f32 p, %0, %1;\n @p st.global.u32 [%2], %3;\n}"
                 :: "f"(a), "f"(b), "l"(p), "r"(j) : "memory");
}

// One warp searches for the CL particles of CL consecutive sorted slots k0 .. at once; lane t serves
// particle t / LPP (active: it takes part; k its slot, f its search record, li and ci its level
// and cell).  All lanes call this together.
//
// The particles of a warp that lie in one stencil row of cells (a segment; nearly always all of
// them, since sorted neighbours share a row) have almost the same neighbourhood, so the warp
// walks the cells around their bounding box once.  A few lanes per level find the level's search
// radius and cell box; the lanes then cut one stencil row each, of whatever level, to the cells
// that reach the box widened by the level's radius.  The rows' concatenated candidates are taken
// 32 at a time, one per lane: those within a pair's radius of the box (about a third) are packed
// together, and again 32 at a time tested against every particle of the segment (broadcast from
// shared memory, two particles per packed operation).  The hits of a particle are appended, in
// candidate order, to its row of the neighbour lists.
//
// What bounds it: the instruction stream, about 5.5k warp instructions per 8 particles on a 300k cube
// (issue slots 68 % busy), a third of it in the ~27 groups of candidates, a third in the ~10 groups
// tested, the rest in segments and rows; on small states the slowest warp's chain of loads.
// Loading the next candidates ahead of the tests gained nothing at 32 warps per SM (605 us per step
// with, 597 without, on that cube).  The walk it replaces, 8 lanes searching for
// their own particle and working off its pairs as they came, took 2.9k per particle for search and
// pair sums together (pressure pass of the 1.2M cube 3.6 ms; search and pressure pass now 1.38 ms).
// Measured on the way: testing every candidate against all particles without the box test 211 M
// instead of 172 M instructions on that cube; pair sums inside the search kernel, from pools in
// shared memory, 80 registers with spills in both and 1.8 ms.
//
// The test is a filter on the search records F (positions and half supports in finest cells, in
// single precision also in the FP64 build), with the radius widened by more than the rounding
// (below).  The exact predicate, evaluated op by op on the stored representation, is applied by
// whoever reads the list.
//
// At level l all particles have kappa h_j <= m c_l, and those in the occupancy cells around the
// box have h_j <= H_l (recorded by the gather; a level with none there is skipped), so
// R_l = max((kappa h_max + min(m c_l, kappa H_l))/2, kappa h_max), h_max the segment's largest h,
// bounds every pair of the level.
//
// FLUSH = false: a list takes the first list_most hits, blocks beyond its row taken as they are
// needed; returns the number of hits of the lane's particle, and adds the candidate pairs tested to
// `tested`.  FLUSH = true (lists that overflowed): whenever a row is nearly full, and at the end,
// work(n) is called by all lanes, with n hits of the lane's particle in its row, and the rows start
// again.  WIDE = false: for grids of at most SEARCH_WRAP cells along x (the general form there: a step
// of the 300k cube 599 us against 590).
template <typename T, int D, int CL, bool FLUSH, bool WIDE = true, typename F>
__device__ __forceinline__ int warp_search(const Grid& g, const State<T>& s, SearchWarp<CL>& ww, int lane, int k0,
                                           bool active, float4 fi, int li, const int ci[3],
                                           unsigned long long& tested, F&& work) {
    typedef ListShape<D> L;
    constexpr int LPP = 32 / CL, ROW = L::ROW;
    constexpr unsigned FULL = 0xffffffffu;
    const int p = lane / LPP, sub = lane % LPP;
    const unsigned lt = (1u << lane) - 1u;
    const unsigned sh_me = shared_address(&ww);
    constexpr unsigned NEAR_F = sizeof(float4) * CL, NEAR_J = NEAR_F + 64 * sizeof(float4), DELTA = NEAR_J + 256;
    char* const list = reinterpret_cast<char*>(s.vj + (size_t)k0 * ROW);
    // Search records are off by less than 2^-24 of the grid's extent X per coordinate and
    // particle (X at most SEARCH_WRAP cells), their difference and the exact predicate's own rounding
    // by as much again: less than 2^-20.6 X in the distance.  A pair's radius is widened by 2^-20 X
    // here, and by a relative 2^-12 where the record is written.
    const float pad = (float)max(min(g.dims[0][0], SEARCH_WRAP), max(g.dims[0][1], g.dims[0][2])) * 0x1p-20f;
    unsigned end[CL];   // byte offset in `list` of the next hit of every particle
#pragma unroll
    for (int q = 0; q < CL; ++q) end[q] = q * ROW * 4;
    auto hits = [&]() {
        int n = 0;
#pragma unroll
        for (int q = 0; q < CL; ++q) n = q == p ? (int)(end[q] / 4 - q * ROW) : n;
        return n;
    };
    // The hits h (this lane's: j) of particle q that do not all fit its row, `old` of them before:
    // into the row, and into blocks of the chunk, taken as the list grows.
    auto append_long = [&](int q, int old, unsigned h, int j) {
        auto blocks = [](int n) { return n <= ROW ? 0 : min((n - ROW + L::XB - 1) / L::XB, XMAX); };
        const int need = blocks(old + __popc(h));
        for (int b = blocks(old); b < need; ++b) {
            if (lane == 0) {
                const int id = atomicAdd(s.xcnt + k0 / CHUNK, 1);
                const unsigned long long v = (unsigned long long)min(id, 255) << (8 * b);
                ww.xid[q] = b == 0 ? v : ww.xid[q] | v;
            }
        }
        __syncwarp();
        const int at = old + __popc(h & lt);
        if (((h >> lane) & 1u) && at < list_most<D>()) {
            const unsigned long long x = ww.xid[q];
            if (at < ROW || ((int)(x >> (8 * ((at - ROW) / L::XB))) & 255) < L::NXB)
                s.vj[list_entry<T, D>(s, k0 + q, at, x)] = j;
        }
        __syncwarp();
    };
    int head = 0, held = 0;   // the ring of candidates near the box
    unsigned pend = __ballot_sync(FULL, active && sub == 0);
    while (pend) {
        // ---- next segment: its box ----
        const int ll = __ffs(pend) - 1;
        const int sl = __shfl_sync(FULL, li, ll);
        int sc[3] = {0, 0, 0};
        for (int a = 0; a < D; ++a) sc[a] = __shfl_sync(FULL, ci[a], ll);
        const bool in = active && ((pend >> (lane - sub)) & 1u) && li == sl && ci[1] == sc[1] &&
                        (D == 2 || ci[2] == sc[2]) && (unsigned)(ci[0] - sc[0]) <= (unsigned)seg_span(D, CL);
        const unsigned seg = __ballot_sync(FULL, in && sub == 0);
        pend &= ~seg;
        // x counts from x0, in grids beyond SEARCH_WRAP a quarter of it before the segment, where the
        // records' x start again in between
        const bool wide = WIDE && g.dims[0][0] > SEARCH_WRAP;
        const int x0 = wide ? (sc[0] << sl) - SEARCH_WRAP / 4 : 0;
        auto from_x0 = [&](float v) {
            if (wide) {
                v -= (float)(x0 & (SEARCH_WRAP - 1));
                v = v < 0.0f ? v + (float)SEARCH_WRAP : v;
            }
            return v;
        };
        const float x[3] = {from_x0(fi.x), fi.y, fi.z};
        float b0[3] = {0, 0, 0}, b1[3] = {0, 0, 0};
        for (int a = 0; a < D; ++a) {
            b0[a] = warp_min_nn(in ? fmaxf(x[a], 0.0f) : 3e38f);
            b1[a] = warp_max_nn(in ? fmaxf(x[a], 0.0f) : 0.0f);
        }
        const float amax = warp_max_nn(in ? fi.w : 0.0f) + pad;
        __syncwarp();
        if (sub == 0) {   // a particle outside the segment lies out of every radius
            const unsigned m = sh_me + (p >> 1) * 32 + (p & 1) * 4;
            sts_f(m, in ? -x[0] : -1e18f);
            sts_f(m + 8, in ? -x[1] : 0.0f);
            sts_f(m + 16, in ? -x[2] : 0.0f);
            sts_f(m + 24, fi.w + pad);
        }
        __syncwarp();
        // ---- search radius and cell box of every level, four lanes per level ----
        float R = 0.0f;
        int lo[3] = {0, 0, 0}, hx = 0, ny = 1, rows = 0;
        {
            const int l = lane >> 2;
            if (l < g.L) {
                // every particle of level l has kappa h_j / 2 <= acap
                const float acap = 0.5f * (float)(1 << (l + g.sm));
                int hb[3] = {0, 0, 0};
                auto box = [&]() -> bool {
                    bool some = true;
                    for (int a = 0; a < D; ++a) {
                        const int s0 = a == 0 ? x0 : 0;
                        lo[a] = max((__float2int_rd(b0[a] - R) + s0) >> l, 0);
                        hb[a] = min((__float2int_rd(b1[a] + R) + s0) >> l, g.dims[l][a] - 1);
                        some = some && lo[a] <= hb[a];
                    }
                    return some;
                };
                R = (amax + fmaxf(amax, acap)) * (1.0f + 0x1p-10f);
                if (box()) {
                    // half the largest support of the level's particles in the occupancy cells
                    // over the box (0: none there); a box of many occupancy cells is searched
                    // without it (it would cost more loads than it can save), and so is a grid of
                    // one level, where all supports reach the cap (constant spacing, 127k particles:
                    // 108.4 us per step against 112.4)
                    const unsigned four = 0xfu << (lane & ~3);
                    const int sh = g.osh;
                    int o0[3] = {0, 0, 0}, no[3] = {1, 1, 1};
                    for (int a = 0; a < D; ++a) {   // a particle past the last cell is counted in it
                        o0[a] = min((lo[a] << l) >> sh, g.od[a] - 1);
                        no[a] = min((hb[a] << l) >> sh, g.od[a] - 1) - o0[a] + 1;
                    }
                    unsigned hm = 0x7f800000u;
                    if (s.occ && g.L > 1 && no[0] * no[1] * no[2] <= 256) {
                        hm = 0u;   // positive floats order as their bits
                        const int nyz = no[1] * no[2];
                        // rows of occupancy cells in turn over the four lanes
                        int yy = lane & 3, zz = 0;
                        while (yy >= no[1]) yy -= no[1], ++zz;
                        for (int t = lane & 3; t < nyz; t += 4) {
                            const unsigned* q =
                                s.occ + (size_t)(g.occ_base + ((o0[2] + zz) * g.od[1] + o0[1] + yy) * g.od[0] + o0[0]) * OCCW + l;
                            for (int xx = 0; xx < no[0]; ++xx) hm = max(hm, __ldg(q + xx * OCCW));
                            yy += 4;
                            while (yy >= no[1]) yy -= no[1], ++zz;
                        }
                        hm = max(hm, __shfl_xor_sync(four, hm, 1));
                        hm = max(hm, __shfl_xor_sync(four, hm, 2));
                    }
                    const float ah = __uint_as_float(hm);
                    if (ah > 0.0f) {
                        bool some = true;
                        if (ah < acap) {
                            R = (amax + fmaxf(amax, ah)) * (1.0f + 0x1p-10f);
                            some = box();
                        }
                        ny = hb[1] - lo[1] + 1;
                        hx = hb[0];
                        if (some) rows = ny * (hb[2] - lo[2] + 1);
                    }
                }
            }
        }
        int rend = rows;   // rows of the levels before and with this one
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL, rend, o);
            if (lane >= o) rend += v;
        }
        const int nrows = __shfl_sync(FULL, rend, 31);
        for (int r0 = 0; r0 < nrows; r0 += 32) {
            // ---- one row per lane, cut to the cells within R of the box ----
            int r = r0 + lane, len = 0, first = 0;
            const bool row_in = r < nrows;
            int l = 0, before = 0;
            for (int q = 0; q < g.L; ++q) {
                const int e = __shfl_sync(FULL, rend, 4 * q);
                if (r >= e) {
                    l = q + 1;
                    before = e;
                }
            }
            l = min(l, g.L - 1);
            const float Rl = __shfl_sync(FULL, R, 4 * l);
            const int nyl = __shfl_sync(FULL, ny, 4 * l), hxl = __shfl_sync(FULL, hx, 4 * l);
            int lol[3] = {0, 0, 0};
            for (int a = 0; a < D; ++a) lol[a] = __shfl_sync(FULL, lo[a], 4 * l);
            if (row_in) {
                r -= before;
                const int rz = D == 2 ? 0 : (int)(((float)r + 0.5f) * __fdividef(1.0f, (float)nyl));
                const int cy = lol[1] + (r - rz * nyl), cz = lol[2] + rz;
                const float w1 = (float)(1 << l);
                const float oy = (float)(cy << l);
                const float dy = fmaxf(fmaxf(oy - b1[1], b0[1] - (oy + w1)), 0.0f);
                float d2 = dy * dy;
                if (D == 3) {
                    const float oz = (float)(cz << l);
                    const float dz = fmaxf(fmaxf(oz - b1[2], b0[2] - (oz + w1)), 0.0f);
                    d2 = fmaf(dz, dz, d2);
                }
                const float rem = fmaf(Rl, Rl, -d2);
                if (rem > 0.0f) {
                    const float w = rem * rsqrtf(rem);
                    const int a0 = max((__float2int_rd(b0[0] - w) + x0) >> l, lol[0]);
                    const int a1 = min((__float2int_rd(b1[0] + w) + x0) >> l, hxl);
                    if (a0 <= a1) {
                        const int row = g.base[l] + (cz * g.dims[l][1] + cy) * g.dims[l][0];
                        first = max(__ldg(s.cell_start + row + a0), 0);
                        len = max(min(__ldg(s.cell_start + row + a1 + 1), s.n) - first, 0);
                    }
                }
            }
            int incl = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += v;
            }
            const int total = __shfl_sync(FULL, incl, 31), excl = incl - len;
            const unsigned some = __ballot_sync(FULL, len > 0);
            __syncwarp();   // the lanes are done with the previous batch's rows
            sts_if(len > 0, sh_me + DELTA + 4 * __popc(some & lt), first - excl);
            __syncwarp();
            tested += (unsigned long long)total * (unsigned)__popc(seg);
            const bool last = r0 + 32 >= nrows;
            int c = 0, started = 0;
            do {
                if (c < total) {
                    // ---- 32 candidates, one per lane: those near the box into the ring ----
                    const unsigned first_at = (unsigned)(excl - c);   // rows that start here
                    const unsigned heads = __reduce_or_sync(FULL, len > 0 && first_at < 32u ? 1u << first_at : 0u);
                    const int ord = started + __popc(heads & (lt | (1u << lane))) - 1;
                    started += __popc(heads);
                    // past the end: the last candidate again
                    const int j = min(c + lane, total - 1) + lds_i(sh_me + DELTA + 4 * ord);
                    float4 f = s.F[j];
                    f.x = from_x0(f.x);
                    const bool there = c + lane < total;
                    c += 32;
                    const float dx = fmaxf(fmaxf(b0[0] - f.x, f.x - b1[0]), 0.0f);
                    const float dy = fmaxf(fmaxf(b0[1] - f.y, f.y - b1[1]), 0.0f);
                    float d2 = fmaf(dy, dy, dx * dx);
                    if (D == 3) {
                        const float dz = fmaxf(fmaxf(b0[2] - f.z, f.z - b1[2]), 0.0f);
                        d2 = fmaf(dz, dz, d2);
                    }
                    float a = fmaxf(f.w, amax) + amax;
                    a = there ? a * a : 0.0f;
                    const unsigned nb = __ballot_sync(FULL, d2 < a);
                    const unsigned at = (unsigned)(head + held + __popc(nb & lt)) & 63u;
                    sts_if_less(d2, a, sh_me + NEAR_F + at * 16, f, sh_me + NEAR_J + at * 4, j);
                    held += __popc(nb);
                }
                while (held >= 32 || (held > 0 && last && c >= total)) {
                    // ---- 32 candidates, one per lane, against every particle of the segment ----
                    __syncwarp();
                    const unsigned at = (unsigned)(head + lane) & 63u;
                    float4 f = lds_f4(sh_me + NEAR_F + at * 16);
                    const int j = lds_i(sh_me + NEAR_J + at * 4);
                    if (lane >= held) f = make_float4(-1e18f, 0.0f, 0.0f, 0.0f);   // out of every radius
                    __syncwarp();
                    head += 32;
                    held = max(held - 32, 0);
                    if (held == 0) head = 0;
                    const f32x2 X = pack2(f.x, f.x), Y = pack2(f.y, f.y), Z = pack2(f.z, f.z);
#pragma unroll
                    for (int q = 0; q < CL; q += 2) {
                        const ulonglong2 A = lds_u2(sh_me + q * 16), B = lds_u2(sh_me + q * 16 + 16);
                        const f32x2 dx = add2(X, A.x), dy = add2(Y, A.y);
                        f32x2 r2 = fma2(dy, dy, mul2(dx, dx));
                        if (D == 3) {
                            const f32x2 dz = add2(Z, B.x);
                            r2 = fma2(dz, dz, r2);
                        }
                        float a0, a1, d0, d1, s0, s1;
                        unpack2(B.y, a0, a1);
                        f32x2 sum = add2(pack2(fmaxf(f.w, a0), fmaxf(f.w, a1)), B.y);
                        sum = mul2(sum, sum);
                        unpack2(sum, s0, s1);
                        unpack2(r2, d0, d1);
                        const unsigned h0 = __ballot_sync(FULL, d0 < s0), h1 = __ballot_sync(FULL, d1 < s1);
                        const unsigned n0 = end[q] + 4 * __popc(h0), n1 = end[q + 1] + 4 * __popc(h1);
                        if (!FLUSH && (n0 > (q + 1) * ROW * 4 || n1 > (q + 2) * ROW * 4)) {
                            append_long(q, end[q] / 4 - q * ROW, h0, j);
                            append_long(q + 1, end[q + 1] / 4 - (q + 1) * ROW, h1, j);
                        } else {
                            stg_if_less(d0, s0, list + (end[q] + 4 * __popc(h0 & lt)), j);
                            stg_if_less(d1, s1, list + (end[q + 1] + 4 * __popc(h1 & lt)), j);
                        }
                        end[q] = n0;
                        end[q + 1] = n1;
                    }
                    if (FLUSH) {
                        unsigned most = 0;
#pragma unroll
                        for (int q = 0; q < CL; ++q) most = max(most, end[q] - q * ROW * 4);
                        if (most > (ROW - 32) * 4) {
                            __syncwarp();
                            work(hits());
                            __syncwarp();
#pragma unroll
                            for (int q = 0; q < CL; ++q) end[q] = q * ROW * 4;
                        }
                    }
                }
            } while (c < total);
        }
    }
    if (FLUSH) {
        __syncwarp();
        work(hits());
        __syncwarp();
    }
    return hits();
}

}  // namespace sph
