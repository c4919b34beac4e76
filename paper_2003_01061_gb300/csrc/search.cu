// search.cu -- neighbour search of a step: per particle the list of the candidates within a pair's
// radius, which the pressure pass and the viscous pass then work through (warp_search in walk.cuh).
#include "walk.cuh"

namespace sph {

// One warp per block, two where a warp takes two particles (search_warps): a block holds its slots
// until its slowest warp is done, and neighbourhoods differ by the levels around.
// cls: the dimension class of the pass (in_pass), or -1 for every particle, whatever its dimension
// or its instance's phase (inspection).  tested: if not null, the candidate pairs tested are
// counted in it.
template <typename T, int D, bool ONE, int CL, bool WIDE>
__global__ void __launch_bounds__(32 * search_warps(CL), 32 / search_warps(CL))
k_search(State<T> s, One one, int cls, unsigned long long* tested) {
    dep_launch();
    dep_wait();
    constexpr int LPP = 32 / CL, WARPS = search_warps(CL);
    static_assert(CHUNK % (CL * WARPS) == 0, "a block's slots lie in one chunk");
    __shared__ SearchWarp<CL> sh[WARPS];
    SearchWarp<CL>& ww = sh[WARPS == 1 ? 0 : threadIdx.x >> 5];
    __shared__ Grid gsh;
    __shared__ Params psh;
    const int lane = lane_id(), p = lane / LPP, sub = lane % LPP;
    const int k0 = (blockIdx.x * WARPS + (WARPS == 1 ? 0 : threadIdx.x >> 5)) * CL, k = k0 + p;
    const int inst = ONE ? 0 : __ldg(s.chunk_inst + k0 / CHUNK);
    if (!ONE) {
        block_copy(&gsh, s.grids + inst);
        block_copy(&psh, s.params + inst);
        __syncthreads();
    }
    const Grid& g = ONE ? one.g : gsh;
    const Params& prm = ONE ? one.p : psh;
    const Ctrl* const ctrl = s.ctrls + inst;
    bool active = k < s.n && live(s, inst, k);
    float4 fi = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    int li = 0, ci[3] = {0, 0, 0};
    if (active) {
        fi = s.F[k];
        own_cell<T, D>(g, s, k, s.VH[k].w, li, ci);
        if (cls >= 0) {
            const unsigned meta = slot_meta<T, D>(s, k);
            const int di = meta_dim(meta);
            // a converged (DONE) instance is frozen: no pair work
            active = di > 0 && ctrl->phase != PH_DONE && in_pass(prm, cls, di, D);
            if (prm.group_conv && active) active = ctrl->gphase[meta_group(meta)] != PH_DONE;
        }
    }
    unsigned long long count = 0;
    const int n = warp_search<T, D, CL, false, WIDE>(g, s, ww, lane, k0, active, fi, li, ci, count, [](int) {});
    __syncwarp();
    if (sub == 0 && k < s.n) {
        s.vcnt[k] = n;
        if (n > ListShape<D>::ROW) s.xid[k] = ww.xid[p];
    }
    if (tested && lane == 0) atomicAdd(tested, count);
}

template <typename T, int D, int CL, bool WIDE>
void launch_search_wide(const State<T>& s, const One* one, cudaStream_t st, bool pdl, int cls, unsigned long long* tested) {
    const int nb = div_up(s.n, CL * search_warps(CL)), nt = 32 * search_warps(CL);
    if (one) launch_k(k_search<T, D, true, CL, WIDE>, nb, nt, st, pdl, s, *one, cls, tested);
    else launch_k(k_search<T, D, false, CL, WIDE>, nb, nt, st, pdl, s, One(), cls, tested);
}
template <typename T, int D, int CL>
void launch_search_cl(const State<T>& s, const One* one, cudaStream_t st, bool pdl, int cls, unsigned long long* tested) {
    if (s.wide) launch_search_wide<T, D, CL, true>(s, one, st, pdl, cls, tested);
    else launch_search_wide<T, D, CL, false>(s, one, st, pdl, cls, tested);
}
template <typename T, int D>
void launch_search(const State<T>& s, const One* one, cudaStream_t st, bool pdl, int cls, unsigned long long* tested) {
    const int cl = search_width(D, s.n, s.levels);
    if constexpr (D == 3)
        if (cl == 2) return launch_search_cl<T, D, 2>(s, one, st, pdl, cls, tested);
    if (cl == 4) launch_search_cl<T, D, 4>(s, one, st, pdl, cls, tested);
    else if (cl == 8) launch_search_cl<T, D, 8>(s, one, st, pdl, cls, tested);
    else launch_search_cl<T, D, 16>(s, one, st, pdl, cls, tested);
}

#define SPH_INST(T, D) \
    template void launch_search<T, D>(const State<T>&, const One*, cudaStream_t, bool, int, unsigned long long*);
SPH_INST(float, 2)
SPH_INST(float, 3)
SPH_INST(double, 2)
SPH_INST(double, 3)

}  // namespace sph
