// interact.cu -- the fused pressure pass of one relaxation step (Algorithm 1: renormalisation
// gamma_i, pressure force with the feature-boundary correction, map onto the feature, step-size
// candidates) over the neighbour lists of the search (search.cu).  LPP consecutive lanes handle
// one particle (sorted order) and split its list, a few consecutive entries per lane and turn;
// their partial sums are combined with a fixed shuffle butterfly.
//
// For particle i of group g (intrinsic dimension d, kernel W_d, rho = h^-d, P = p0 h^(2d)):
//   sigma_i = sum_{j in g, r < kappa h_i} W_d(r_ij, h_i)             (Eq. 20 denominator, j = i included)
//   gamma_i = sum_{j in g, r < kappa h_i} W_d(r_ij, h_i) h_j^d         (Eq. 18)
//   F_i     = sum_{j in g, j != i, r < kappa h_ij} (P_i + P_j) W_d'(r_ij, h_ij) e_ij          (Eq. 19, 1st sum)
//           + sum_{b: d_b < d, r < kappa h_ib} rho_b (P_i + P_b) W_d(r_ib, h_ib) n_b|i A_b  (Eq. 19, 2nd sum;
//             left out with boundary_correction = 0, the earlier method compared in Sec. 4.1)
//   a_p,i   = Pi_i(-F_i / gamma_i),  V~_i = 1 / sigma_i
// and the Eq. 24 candidates 0.25 sqrt(r_c/|a_p|), r_c/(40 |v|), reduced to per-group minima.  On
// sampling steps the last warp of every chunk of slots sums V~ over it (Eq. 22) in a fixed order.
// Every list entry gets the pair's kernel factor of Eq. 7 for the viscous pass.
//
// A block serves BLOCK/LPP consecutive slots, which lie in one chunk and so in one instance:
// the instance's grid and parameters are copied into shared memory once per block (a batch of
// one passes them as kernel parameters instead).
#include <type_traits>

#include "walk.cuh"

namespace sph {

// fn(j, h_i, r2, h_j, meta_i, meta_j) for the candidates of particle k (on: it has some), shared out
// among its LPP lanes; all lanes of the warp call this together
template <typename T, int D, int LPP, typename F>
__device__ __forceinline__ void for_pairs(const Grid& g, const State<T>& s, SearchWarp<32 / LPP>& ww, int lane, int k0,
                                          bool on, F&& fn) {
    const Meta<D>* const Ms = meta_words<D>(s);
    const int k = k0 + lane / LPP;
    T offi[3] = {T(0), T(0), T(0)}, hi = T(1);
    unsigned mi = 0;
    int li = 0, ci[3] = {0, 0, 0}, Pi[3], n = 0;
    if (on) {
        Meta<D> wi;
        Rec<T, D>::load(s.P, Ms, k, offi, hi, wi);
        own_cell<T, D>(g, s, k, hi, li, ci);
        mi = MetaWord<D>::meta(wi);
        n = s.vcnt[k];
    }
    for (int a = 0; a < 3; ++a) Pi[a] = ci[a] << li;
    unsigned long long xid = 0;
    const bool dense = list_overflowed<T, D>(s, k, n);
    if (!dense && n > ListShape<D>::ROW) xid = s.xid[k];
    auto row = [&](int m_) {
        for (int t = lane % LPP; t < m_; t += LPP) {
            const int j = s.vj[list_entry<T, D>(s, k, t, xid)];
            T offj[3], hj, dx[3];
            Meta<D> w;
            int m[3];
            Rec<T, D>::load(s.P, Ms, j, offj, hj, w);
            MetaWord<D>::rel(w, Pi, m);
            const T r2 = pair_dx<T, D>(offi, offj, m, (T)g.c0, dx);
            fn(j, hi, r2, hj, mi, MetaWord<D>::meta(w));
        }
    };
    if (!dense) row(n);
    if (__any_sync(0xffffffffu, dense)) {
        unsigned long long none = 0;
        warp_search<T, D, 32 / LPP, true>(g, s, ww, lane, k0, dense,
                                          dense ? s.F[k] : make_float4(0.0f, 0.0f, 0.0f, 0.0f), li, ci, none, row);
    }
}

// One particle's sums of the pressure pass without their common factors (F without p0, sig and gam
// without the normalisation alpha_i of W(r, h_i)).
template <typename T, int D> struct Pressure {
    const State<T>& s;
    const Grid& g;
    const Params& p;
    const Domain& dom;
    T hi, hk, invRi, hi2d, offi[3], tg[3];
    int gi, di, Pi[3];
    T F[3], sig, gam;

    __device__ __forceinline__ void init(T h, unsigned meta, const T off[3], int li, const int ci[3]) {
        const T kappa = wp<T>(p.kappa, p.kappa_f);
        hi = h;
        hk = T(0.5) * kappa;
        invRi = fast_rcp(kappa * hi);
        gi = meta_group(meta);
        di = meta_dim(meta);
        T hid;
        hpow(hi, di > 0 ? di : 1, hid, hi2d);
        for (int a = 0; a < 3; ++a) {
            offi[a] = off[a];
            tg[a] = F[a] = T(0);
            Pi[a] = ci[a] << li;
        }
        sig = gam = T(0);
        if (di > 0 && di < D) {
            T xi[3] = {T(0), T(0), T(0)};
            for (int a = 0; a < D; ++a) xi[a] = (T)g.origin[a] + (T)Pi[a] * (T)g.c0 + offi[a];
            feature_tangent<T>(dom.f[gi], xi, tg);
        }
    }
    // Eq. 19's second sum: boundary particle j (of lower dimension than d)
    __device__ __forceinline__ void wall(int d, T r, T R, T S2, T hj, unsigned mj, const T offj[3], const int m[3]) {
        const T invR = fast_rcp(R);
        const T q = r * invR;
        const T t = T(1) - q;
        const T w = wendland_alpha<T>(d, invR) * (t * t) * (t * t) * (T(1) + T(4) * q);
        T xb[3] = {T(0), T(0), T(0)};
        for (int a = 0; a < D; ++a) xb[a] = (T)g.origin[a] + (T)(Pi[a] - m[a]) * (T)g.c0 + offj[a];
        T nb[3];
        boundary_normal<T>(dom.f[meta_group(mj)], xb, nb);
        tangent_map<T>(d, D, tg, nb);
        const T nn2 = nb[0] * nb[0] + nb[1] * nb[1] + nb[2] * nb[2];
        if (nn2 > T(1e-12)) {
            T hjd, hj2d;
            hpow(hj, d, hjd, hj2d);
            const T Ab = p.boundary_rho != 0 ? fast_rcp(hj) : hjd * fast_rcp(hj);
            const T c2 = Ab * S2 * w * fast_rsqrt(nn2);
            F[0] += c2 * nb[0];
            F[1] += c2 * nb[1];
            if (D == 3) F[2] += c2 * nb[2];
        }
    }
    // any candidate; returns the pair's kernel factor of Eq. 7, (rho_i^-2 + rho_j^-2) W'(r, h_ij) / r
    // (0: not a pair of the viscous sum)
    __device__ __forceinline__ T pair(const T dx[3], T r2, T hj, unsigned mj, const T offj[3], const int m[3]) {
        const T R = rn_mul(rn_add(hi, hj), hk);   // the pair's support, as pair_rc2 has it
        const bool near = r2 < rn_mul(R, R);
        T hjd, hj2d;
        hpow(hj, di, hjd, hj2d);
        const T S2 = hi2d + hj2d;   // rho_i^-2 + rho_j^-2; times p0: P_i + P_j
        const T r = root_of(r2);
        if (meta_group(mj) == gi) {
            // outside its support each kernel is zero, so the two sums need no predicate
            const T q = pos_part(T(1) - r * invRi);
            const T w4 = (q * q) * (q * q) * (T(5) - T(4) * q);   // (1 - r/R)^4 (1 + 4 r/R)
            sig += w4;
            gam += w4 * hjd;
            const T kv = kernel_factor<T>(di, S2, r, fast_rcp(R));
            for (int a = 0; a < D; ++a) F[a] += kv * dx[a];
            return near && r2 > T(0) ? kv : T(0);
        }
        if (near && p.boundary_corr != 0 && meta_dim(mj) < di) wall(di, r, R, S2, hj, mj, offj, m);
        return T(0);
    }
    // N candidates: their records are all loaded before the first is used
    template <int N> __device__ __forceinline__ void candidates(const Meta<D>* Ms, const int (&j)[N], int n, T (&kv)[N]) {
        T off[N][3], hj[N];
        Meta<D> w[N];
#pragma unroll
        for (int u = 0; u < N; ++u)
            if (u < n) Rec<T, D>::load(s.P, Ms, j[u], off[u], hj[u], w[u]);
#pragma unroll
        for (int u = 0; u < N; ++u) {
            kv[u] = T(0);
            if (u >= n) continue;
            T dx[3];
            int m[3];
            MetaWord<D>::rel(w[u], Pi, m);
            const T r2 = pair_dx<T, D>(offi, off[u], m, (T)g.c0, dx);
            kv[u] = pair(dx, r2, hj[u], MetaWord<D>::meta(w[u]), off[u], m);
        }
    }
};

// The pair sums of the warp's particles whose list overflowed (over), from a second search; all lanes
// call it together, and it adds to sums (F, sig, gam).  Not inlined: rarely needed, and its
// registers would weigh on k_interact.
template <typename T, int D>
__device__ __noinline__ void pressure_again(const State<T>& s, const Grid& g, const Params& p, const Domain& dom,
                                            SearchWarp<32 / Lpp<D>::v>& ww, int lane, int k0, bool over, T* sums) {
    constexpr int LPP = Lpp<D>::v, CL = 32 / LPP;
    const int k = k0 + lane / LPP, sub = lane % LPP;
    const Meta<D>* const Ms = meta_words<D>(s);
    Pressure<T, D> c{s, g, p, dom};
    int li = 0, ci[3] = {0, 0, 0};
    unsigned mi = 0;
    T offi[3] = {T(0), T(0), T(0)}, hi = T(1);
    if (over) {
        Meta<D> wi;
        Rec<T, D>::load(s.P, Ms, k, offi, hi, wi);
        own_cell<T, D>(g, s, k, hi, li, ci);
        mi = MetaWord<D>::meta(wi);
    }
    c.init(hi, mi, offi, li, ci);
    unsigned long long none = 0;
    warp_search<T, D, CL, true>(g, s, ww, lane, k0, over, over ? s.F[k] : make_float4(0.0f, 0.0f, 0.0f, 0.0f), li, ci,
                                none, [&](int n) {
                                    for (int t = sub; t < n; t += LPP) {
                                        const int j[1] = {s.vj[(size_t)k * ListShape<D>::ROW + t]};
                                        T kv[1];
                                        c.candidates(Ms, j, 1, kv);
                                    }
                                });
    for (int a = 0; a < 3; ++a) sums[a] += c.F[a];
    sums[3] += c.sig;
    sums[4] += c.gam;
}

template <typename T, int D> constexpr int interact_minb() {
    return sizeof(T) == 4 ? (D == 2 ? SPH_INTERACT_MINB : SPH_INTERACT_MINB_3D) : SPH_INTERACT_MINB_F64;
}

template <typename T, int D, bool ONE>
__global__ void __launch_bounds__(BLOCK, (interact_minb<T, D>()))
    k_interact(const __grid_constant__ State<T> s, const __grid_constant__ One one, T* dbg_sigma, T* dbg_gamma, int cls) {
    dep_launch();
    dep_wait();
    constexpr int LPP = Lpp<D>::v, CL = 32 / LPP, U = pressure_listu<D>();
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ SearchWarp<CL> ww[BLOCK / 32];
    __shared__ Grid gsh;
    __shared__ Params psh;
    const int lane = lane_id(), sub = lane % LPP;
    const int k0 = (blockIdx.x * (BLOCK / 32) + (threadIdx.x >> 5)) * CL;   // the warp's first slot
    const int k = k0 + lane / LPP;
    const int inst = ONE ? 0 : __ldg(s.chunk_inst + k0 / CHUNK);
    Ctrl* const ctrl = s.ctrls + inst;
    const Domain& dom = s.doms[inst];
    if (!ONE) {
        block_copy(&gsh, s.grids + inst);
        block_copy(&psh, s.params + inst);
        __syncthreads();
    }
    const Grid& g = ONE ? one.g : gsh;
    const Params& p = ONE ? one.p : psh;

    const bool lead = sub == 0;
    const bool inrange = k < s.n && live(s, inst, k);
    const int n = inrange ? s.vcnt[k] : 0;
    T offi[3] = {T(0), T(0), T(0)}, hi = T(1);
    unsigned mi = 0;
    int li = 0, ci[3] = {0, 0, 0};
    const Meta<D>* const Ms = meta_words<D>(s);
    if (inrange) {
        Meta<D> wi;
        Rec<T, D>::load(s.P, Ms, k, offi, hi, wi);
        mi = MetaWord<D>::meta(wi);
        own_cell<T, D>(g, s, k, hi, li, ci);
    }
    const int gi = inrange ? meta_group(mi) : -1;
    const int di = inrange ? meta_dim(mi) : 0;
    // a converged (DONE) instance is frozen: no pair work
    bool active = inrange && di > 0 && ctrl->phase != PH_DONE && in_pass(p, cls, di, D);
    if (p.group_conv && active) active = ctrl->gphase[gi] != PH_DONE;   // the group itself converged
    const T kappa = wp<T>(p.kappa, p.kappa_f), p0 = wp<T>(p.p0, p.p0_f);
    Pressure<T, D> c{s, g, p, dom};
    c.init(hi, mi, offi, li, ci);
    const bool over = active && list_overflowed<T, D>(s, k, n);
    if constexpr (sizeof(T) == 4) {
        // single precision: packed arithmetic, two pairs per operation (for each pair the operations
        // of Pressure::pair); compiled for warps whose particles are all of full dimension (most)
        // and for mixed ones, whose powers and constants depend on the lane
        auto sums_of = [&](auto full) {
            constexpr bool FD = decltype(full)::value;
            const int d = FD ? D : di;
            // x1, x2 or x3 by the particle's dimension
            auto pick = [&](f32x2 x1, f32x2 x2, f32x2 x3) -> f32x2 {
                if (FD) return D == 2 ? x2 : x3;
                const f32x2 low = d == 1 ? x1 : x2;
                return D == 3 && d == 3 ? x3 : low;
            };
            const float A = d == 1 ? -20.0f * 1.5f
                                   : d == 2 ? (float)(-20.0 * 7.0 / CUDART_PI) : (float)(-20.0 * 21.0 / (2.0 * CUDART_PI));
            const f32x2 A2 = pack2(A, A);
            const f32x2 c02 = pack2(g.c0, g.c0), hi2 = pack2(hi, hi), hk2 = pack2(T(0.5) * kappa, T(0.5) * kappa), one2 = pack2(1.0f, 1.0f);
            const f32x2 nRi = pack2(-c.invRi, -c.invRi), hid2 = pack2(c.hi2d, c.hi2d);
            const unsigned long long xid = n > ListShape<D>::ROW ? s.xid[k] : 0ull;
            f32x2 F0 = 0, F1 = 0, F2 = 0, S0 = 0, G0 = 0;
            for (int t = sub * U; t < n; t += LPP * U) {
                int jj[U];
                const size_t e = list_entry<T, D>(s, k, t, xid);
                list_load(s.vj + e, jj);
                T off[U][3], hj[U];
                Meta<D> w[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (t + u >= n) jj[u] = k;   // past the end: the particle itself, without weight
                    Rec<T, D>::load(s.P, Ms, jj[u], off[u], hj[u], w[u]);
                }
                T fac[U];
#pragma unroll
                for (int u = 0; u < U; u += 2) {
                    int ma[3], mb[3];
                    MetaWord<D>::rel(w[u], c.Pi, ma);
                    MetaWord<D>::rel(w[u + 1], c.Pi, mb);
                    // dx, r2, R op by op, as pair_dx and pair_rc2 have them
                    auto axis = [&](int a) {
                        return add2(sub2(pack2(offi[a], offi[a]), pack2(off[u][a], off[u + 1][a])),
                                    mul2(pack2(small_int<T>(ma[a]), small_int<T>(mb[a])), c02));
                    };
                    const f32x2 dx = axis(0), dy = axis(1);
                    f32x2 r2 = add2(mul2(dx, dx), mul2(dy, dy));
                    f32x2 dz = 0;
                    if (D == 3) {
                        dz = axis(2);
                        r2 = add2(r2, mul2(dz, dz));
                    }
                    const f32x2 h = pack2(hj[u], hj[u + 1]);
                    const f32x2 R = mul2(add2(hi2, h), hk2), Rq = mul2(R, R);
                    float r2a, r2b, Ra, Rb, qa, qb, xa, xb;
                    unpack2(r2, r2a, r2b);
                    unpack2(R, Ra, Rb);
                    unpack2(Rq, qa, qb);
                    const unsigned ea = MetaWord<D>::meta(w[u]), eb = MetaWord<D>::meta(w[u + 1]);
                    const bool ia = t + u < n, ib = t + u + 1 < n;
                    const bool sa = ia && meta_group(ea) == gi, sb = ib && meta_group(eb) == gi;
                    const f32x2 r = pack2(root_of(r2a), root_of(r2b));
                    const f32x2 invR = pack2(fast_rcp(Ra), fast_rcp(Rb));
                    const f32x2 h2 = mul2(h, h), hd = pick(h, h2, mul2(h2, h));
                    const f32x2 S2 = add2(hid2, mul2(hd, hd));   // rho_i^-2 + rho_j^-2
                    // outside its support each kernel is zero, so the two sums need no predicate
                    f32x2 q = fma2(r, nRi, one2);
                    unpack2(q, xa, xb);
                    q = pack2(sa ? fmaxf(xa, 0.0f) : 0.0f, sb ? fmaxf(xb, 0.0f) : 0.0f);
                    const f32x2 q2 = mul2(q, q);
                    const f32x2 w4 = mul2(mul2(q2, q2), fma2(q, pack2(-4.0f, -4.0f), pack2(5.0f, 5.0f)));
                    S0 = add2(S0, w4);
                    G0 = fma2(w4, hd, G0);
                    q = fma2(r, neg2(invR), one2);
                    unpack2(q, xa, xb);
                    q = pack2(sa ? fmaxf(xa, 0.0f) : 0.0f, sb ? fmaxf(xb, 0.0f) : 0.0f);
                    const f32x2 i2 = mul2(invR, invR);   // products in the order of kernel_factor
                    const f32x2 kv = mul2(mul2(mul2(S2, i2), mul2(pick(invR, i2, mul2(i2, invR)), A2)), mul2(mul2(q, q), q));
                    F0 = fma2(kv, dx, F0);
                    F1 = fma2(kv, dy, F1);
                    if (D == 3) F2 = fma2(kv, dz, F2);
                    unpack2(kv, xa, xb);
                    const bool na = r2a < qa, nb = r2b < qb;
                    fac[u] = na && r2a > 0.0f ? xa : 0.0f;
                    fac[u + 1] = nb && r2b > 0.0f ? xb : 0.0f;
                    const bool wa = ia && na && meta_dim(ea) < d, wb = ib && nb && meta_dim(eb) < d;
                    if ((wa || wb) && p.boundary_corr != 0) {
                        float sx, sy;
                        unpack2(S2, sx, sy);
                        if (wa) c.wall(d, root_of(r2a), Ra, sx, hj[u], ea, off[u], ma);
                        if (wb) c.wall(d, root_of(r2b), Rb, sy, hj[u + 1], eb, off[u + 1], mb);
                    }
                }
                list_store(s.vr + e, fac);   // the pairs' kernel factors of Eq. 7
            }
            auto fold = [&](f32x2 v) {
                float a, b;
                unpack2(v, a, b);
                return a + b;
            };
            c.F[0] += fold(F0);
            c.F[1] += fold(F1);
            if (D == 3) c.F[2] += fold(F2);
            c.sig += fold(S0);
            c.gam += fold(G0);
        };
        const bool full = __all_sync(FULL, !active || di == D);
        if (active && !over) {
            if (full) sums_of(std::true_type());
            else sums_of(std::false_type());
        }
    } else if (active && !over) {   // pair by pair
        const unsigned long long xid = n > ListShape<D>::ROW ? s.xid[k] : 0ull;
        constexpr int N = 2;
        for (int t = sub * N; t < n; t += LPP * N) {
            const size_t e = list_entry<T, D>(s, k, t, xid);
            int jj[N];
            T kv[N];
            list_load(s.vj + e, jj);
            c.candidates(Ms, jj, n - t, kv);
            list_store(s.vr + e, kv);
        }
    }
    T sums[5] = {c.F[0], c.F[1], c.F[2], c.sig, c.gam};
    if (__any_sync(FULL, over)) pressure_again<T, D>(s, g, p, dom, ww[threadIdx.x >> 5], lane, k0, over, sums);
    const T alpha_i = wendland_alpha<T>(di > 0 ? di : 1, c.invRi);
    T F[3] = {T(0), T(0), T(0)};
    for (int a = 0; a < D; ++a) F[a] = p0 * sub_sum<LPP>(sums[a]);
    const T sig = alpha_i * sub_sum<LPP>(sums[3]), gam = alpha_i * sub_sum<LPP>(sums[4]);

    T ap[3] = {T(0), T(0), T(0)};
    T vtil = T(0);
    unsigned long long dta = inf_bits<T>(), dtv = inf_bits<T>();
    if (active && lead) {
        const T ig = T(1) / gam;
        for (int a = 0; a < 3; ++a) ap[a] = -F[a] * ig;
        tangent_map<T>(di, D, c.tg, ap);
        vtil = T(1) / sig;
        const T rc = kappa * hi;
        const T an = t_sqrt(ap[0] * ap[0] + ap[1] * ap[1] + ap[2] * ap[2]);
        const Vec4<T> vh = s.VH[k];
        const T v0 = vh.x, v1 = vh.y, v2 = vh.z;
        const T vn = t_sqrt(v0 * v0 + v1 * v1 + v2 * v2);
        if (an > T(0)) dta = min_bits(wp<T>(p.cfl_a, p.cfl_a_f) * t_sqrt(rc / an));
        if (vn > T(0)) dtv = min_bits(wp<T>(p.cfl_v, p.cfl_v_f) * rc / vn);
        if (!(an == an) || !isfinite(an)) atomicOr(&ctrl->status, ST_NONFINITE);
    }
    if (inrange && lead) {
        Vec4<T> a4;
        a4.x = ap[0];
        a4.y = ap[1];
        a4.z = ap[2];
        a4.w = vtil;
        s.A[k] = a4;
        if (dbg_sigma) dbg_sigma[k] = sig;
        if (dbg_gamma) dbg_gamma[k] = gam;
    }
    // per-group minima of the Eq. 24 terms: one pass per group present in the warp (mostly one).
    // A minimum that is no lower than the one already there needs no atomic (it only falls).
    unsigned pending = __ballot_sync(FULL, active && lead);
    while (pending) {
        const int gg = __shfl_sync(FULL, gi, __ffs(pending) - 1);
        const bool mine = active && lead && gi == gg;
        const unsigned long long a = warp_min_bits<T>(mine ? dta : inf_bits<T>());
        const unsigned long long v = warp_min_bits<T>(mine ? dtv : inf_bits<T>());
        if (lane == 0) {
            if (a < __ldcg(&ctrl->dta_bits[gg])) atomicMin(&ctrl->dta_bits[gg], a);
            if (v < __ldcg(&ctrl->dtv_bits[gg])) atomicMin(&ctrl->dtv_bits[gg], v);
        }
        pending &= ~__ballot_sync(FULL, mine);
    }
    if (ctrl->sample_now != 0) {
        // the last warp of this chunk of slots to finish sums V~ over the chunk, group by group in
        // a fixed order, into the chunk's row, which the controller reads (a chunk lies in one
        // instance; particles that took no part have V~ = 0)
        constexpr int WPC = CHUNK / CL;
        const int c = k0 / CHUNK;
        __threadfence();
        __syncwarp();
        int old = 0;
        if (lane == 0) old = atomicAdd(s.pticket + c, 1);
        if (__shfl_sync(FULL, old, 0) == WPC - 1) {
            __threadfence();
            double* const row = s.partials2 + (size_t)c * MAXF;
            for (int t = lane; t < p.G; t += 32) row[t] = 0.0;
            __syncwarp();
            double v[CHUNK / 32];
            int gr[CHUNK / 32];
#pragma unroll
            for (int i = 0; i < CHUNK / 32; ++i) {
                const int q = c * CHUNK + i * 32 + lane;
                const bool on = q < s.n && live(s, inst, q);
                v[i] = on ? (double)__ldcg(&s.A[q].w) : 0.0;
                gr[i] = on ? meta_group(slot_meta<T, D>(s, q)) : -1;
            }
            for (int i = 0; i < CHUNK / 32; ++i) {
                unsigned left = __ballot_sync(FULL, gr[i] >= 0);
                while (left) {   // every group is summed where it first appears
                    const int gg = __shfl_sync(FULL, gr[i], __ffs(left) - 1);
                    double acc = 0.0;
#pragma unroll
                    for (int q = 0; q < CHUNK / 32; ++q) {
                        if (gr[q] == gg) {
                            acc += v[q];
                            gr[q] = -1;
                        }
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(FULL, acc, o);
                    if (lane == 0) row[gg] = acc;
                    left = __ballot_sync(FULL, gr[i] >= 0);
                }
            }
            if (lane == 0) s.pticket[c] = 0;
        }
    }
}

// neighbour sets for inspection, from the lists of a search over all particles: mode 0 pair
// predicate (j != i), mode 1 self predicate (j = i included), over all groups.  lists == nullptr:
// counts only; otherwise counts (of the first call) are counted down to place the entries.
template <typename T, int D>
__global__ void __launch_bounds__(BLOCK) k_neighbors(State<T> s, int mode, int* counts, const long long* offsets,
                                                     int* lists) {
    constexpr int LPP = Lpp<D>::v;
    __shared__ SearchWarp<32 / LPP> ww[BLOCK / 32];
    const int lane = lane_id(), wid = threadIdx.x >> 5;
    const int k0 = (blockIdx.x * (BLOCK / 32) + wid) * (32 / LPP), k = k0 + lane / LPP;
    const int inst = k0 < s.n ? inst_of(s, k0) : 0;   // a warp's slots lie in one instance
    const Grid& g = s.grids[inst];
    const Params& p = s.params[inst];
    const bool active = k < s.n && live(s, inst, k);
    const T kappa = wp<T>(p.kappa, p.kappa_f), hk = T(0.5) * kappa;
    int cnt = 0;
    const long long base = lists && active ? offsets[k] : 0;
    for_pairs<T, D, LPP>(g, s, ww[wid], lane, k0, active, [&](int j, T hi, T r2, T hj, unsigned, unsigned) {
        if (!(mode == 0 ? (j != k && r2 < pair_rc2(hi, hj, hk)) : (r2 < self_rc2(hi, kappa)))) return;
        if (lists) lists[base + atomicSub(counts + k, 1) - 1] = j;
        ++cnt;
    });
    cnt = sub_sum<LPP>(cnt);
    if (k < s.n && !lists && lane % LPP == 0) counts[k] = cnt;
}

// pairs inside the interaction support of the pressure pass, summed over all particles
template <typename T, int D>
__global__ void __launch_bounds__(BLOCK) k_pair_counts(State<T> s, unsigned long long* out) {
    constexpr int LPP = Lpp<D>::v;
    __shared__ SearchWarp<32 / LPP> ww[BLOCK / 32];
    const int lane = lane_id(), wid = threadIdx.x >> 5;
    const int k0 = (blockIdx.x * (BLOCK / 32) + wid) * (32 / LPP), k = k0 + lane / LPP;
    const int inst = k0 < s.n ? inst_of(s, k0) : 0;   // a warp's slots lie in one instance
    const Grid& g = s.grids[inst];
    const Params& p = s.params[inst];
    const bool active = k < s.n && live(s, inst, k);
    const T kappa = wp<T>(p.kappa, p.kappa_f), hk = T(0.5) * kappa;
    unsigned long long accd = 0;
    for_pairs<T, D, LPP>(g, s, ww[wid], lane, k0, active, [&](int j, T hi, T r2, T hj, unsigned mi, unsigned mj) {
        if (meta_dim(mi) > 0 && (meta_group(mj) == meta_group(mi) || meta_dim(mj) < meta_dim(mi)) && j != k &&
            r2 < pair_rc2(hi, hj, hk))
            ++accd;
    });
    for (int o = 16; o > 0; o >>= 1) accd += __shfl_down_sync(0xffffffffu, accd, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, accd);
}

template <typename T, int D>
void launch_interact(const State<T>& s, const One* one, T* dbg_sigma, T* dbg_gamma, cudaStream_t st, bool pdl,
                     int cls) {
    if (one) launch_k(k_interact<T, D, true>, div_up((long long)s.n * Lpp<D>::v, BLOCK), BLOCK, st, pdl, s, *one, dbg_sigma, dbg_gamma, cls);
    else launch_k(k_interact<T, D, false>, div_up((long long)s.n * Lpp<D>::v, BLOCK), BLOCK, st, pdl, s, One(), dbg_sigma, dbg_gamma, cls);
}
template <typename T, int D>
void launch_neighbors(const State<T>& s, int mode, int* counts, const long long* offsets, int* lists, cudaStream_t st) {
    k_neighbors<T, D><<<div_up((long long)s.n * Lpp<D>::v, BLOCK), BLOCK, 0, st>>>(s, mode, counts, offsets, lists);
}
template <typename T, int D> void launch_pair_counts(const State<T>& s, unsigned long long* out, cudaStream_t st) {
    k_pair_counts<T, D><<<div_up((long long)s.n * Lpp<D>::v, BLOCK), BLOCK, 0, st>>>(s, out);
}

#define SPH_INST(T, D)                                                                                        \
    template void launch_interact<T, D>(const State<T>&, const One*, T*, T*, cudaStream_t, bool, int);        \
    template void launch_neighbors<T, D>(const State<T>&, int, int*, const long long*, int*, cudaStream_t);   \
    template void launch_pair_counts<T, D>(const State<T>&, unsigned long long*, cudaStream_t);
SPH_INST(float, 2)
SPH_INST(float, 3)
SPH_INST(double, 2)
SPH_INST(double, 3)

}  // namespace sph
