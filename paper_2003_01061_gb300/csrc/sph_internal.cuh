// sph_internal.cuh -- device pointers of a batch of instances and the kernel launchers shared by
// the translation units of libsphmesh.so.  Not part of the public ABI.
//
// A batch packs NI independent instances (same dimension and precision) into one particle
// array.  Instance i owns the slots [inst_off[i], inst_off[i+1]) -- its particle count rounded up
// to a multiple of CHUNK, none while it is empty -- of which the first inst_n[i] hold its
// particles in the current order; the rest are padding (hashed to the instance's dummy cell,
// which sorts last and is never searched).  Its cells are the global keys grids[i].base[0] ..
// grids[i].base[MAXL]-1, followed by its dummy key grids[i].base[MAXL].  Every kernel serves all
// instances in one launch over the n slots in use.
#pragma once
#include "../../include/sphmesh.h"
#include "sph_device.cuh"

namespace sph {

constexpr int CHUNK = SPH_SLOT_CHUNK;   // slot alignment of instances (a multiple of every pair-pass block)

// Search records hold x modulo this many finest cells (y and z have fewer): beyond it single precision
// would be too coarse, and the search radius, widened by its rounding, would take in whole cells of
// strangers (2D ribbons of 2^18, 2^20 and 2^21 cells: 1,043, 4,064 and 8,074 us per step, with x as it is
// 1,219, 10,424 and 32,887).  A search spans less than a quarter of it.
constexpr int SEARCH_WRAP = 1 << 14;

template <typename T> struct State {
    int n;             // total slots of the batch
    int NI;            // instances
    int levels;        // most grid levels of a loaded instance
    bool wide;         // one of them has a grid longer than SEARCH_WRAP cells along x
    const int* inst_off;    // [NI+1]
    const int* inst_n;      // [NI]
    const int* chunk_inst;  // [n / CHUNK] instance of every chunk of slots
    const Grid* grids;      // [NI]
    const Params* params;   // [NI]
    const Domain* doms;     // [NI]
    const Sizing* sizs;     // [NI]
    Ctrl* ctrls;            // [NI]
    // stored state (order of the previous sort): position = finest cell C + offset O
    int* C[3];
    T* O[3];
    T* V[3];
    T* H;
    unsigned* G;
    int* ID;           // index of the particle in its instance's input order (-1: padding)
    int* K;            // cell key of every stored particle (written by the hash)
    // sorted state
    int* Cs[3];
    T* Os[3];
    Vec4<T>* VH;       // (v.x, v.y, v.z, h): one 16-byte (FP64: 32-byte) load per neighbour
    unsigned* Ms;
    int* IDs;
    int* Ks;
    Vec4<T>* P;
    float4* F;         // search records: position (x modulo SEARCH_WRAP) and kappa h / 2 in finest
                       // cells (padding: stale)
    Vec4<T>* A;
    // rebuild scratch: per-cell counts (down to zero after the scatter) and cell starts
    int* count;
    int* cell_start;
    // one-pass scan: per-tile status words (flag << 62 | value) and the tile ticket, cleared by
    // whichever kernel produces the histogram
    unsigned long long* tstate;
    int* ticket;
    int ntile;
    int* perm;         // slot -> stored index as left by the scatter (unordered inside a cell)
    int* sperm;        // slot -> stored index, stable (ordered inside a cell; written by the gather)
    int ncell;         // total keys (all instances' cells and dummy cells)
    // per occupancy cell, OCCW words: per level the largest half support (F's w) of its
    // particles in the cell (float bits, 0 for none; built by the gather)
    unsigned* occ;
    int nocc;
    // neighbour lists (ListShape): the rows by slot, then, from entry xbase, the blocks by chunk;
    // per entry the candidate (search) and the pair's kernel factor of Eq. 7,
    // (rho_i^-2 + rho_j^-2) W'(r, h_ij) / r (pressure pass; 0: no pair of the viscous sum); per slot
    // the number of candidates and, for a list longer than its row, its blocks (a byte each); per
    // chunk the number of blocks asked for
    int* vj;
    T* vr;
    int* vcnt;
    unsigned long long* xid;
    int* xcnt;
    size_t xbase;
    // sums of V~ per chunk of CHUNK slots and group (sample steps), [chunk][MAXF]: written by the
    // chunk's last pressure-pass warp (counted in pticket), read by the controller
    double* partials2;
    int* pticket;
};

// The grid and parameters of a batch of one, passed to the kernels by value so that they are
// read as constant-bank operands; with more instances the kernels read the per-instance tables.
struct One {
    Grid g;
    Params p;
};

// output set of the update kernel (the stored state, or scratch for inspection calls)
template <typename T> struct Out {
    int* C[3];
    T* O[3];
    T* V[3];
    T* H;
    unsigned* G;
    int* ID;
    T* av[3];          // optional: viscous acceleration (inspection only)
    int* K;            // optional (stored state): the next rebuild's cell keys ...
    int* count;        // ... and per-cell histogram, so that the next step needs no hash pass
};

// lanes per particle in the pair passes over the neighbour lists (measured, whole step in us with
// 4 / 8 / 16: 20k disk 76 / 78 / 84, 120k disk 144 / 159 / 206, 83k cube 320 / 328 / 363, 300k cube
// 706 / 778 / 935; a result must not depend on the batch, so the number is the same at every size)
#ifndef SPH_LPP_2D
#define SPH_LPP_2D 4
#endif
#ifndef SPH_LPP_3D
#define SPH_LPP_3D 4
#endif
template <int D> struct Lpp {
    static constexpr int v = D == 2 ? SPH_LPP_2D : SPH_LPP_3D;
};
// Neighbour lists: the candidates within the larger of a particle's own and the pair's radius,
// itself included, about 24 in 2D and 80 in 3D.  A particle has a row of ROW entries; a longer list
// goes on in up to XMAX blocks of XB entries, taken from the NXB blocks of its chunk of slots
// (coarse particles beside much finer ones: a few per mille of a graded 3D mesh).  A list that
// needs more, or any list with blocks in a chunk that ran out of them, counts as overflowed (which
// lists got blocks there depends on timing, whether the chunk ran out does not): the pair passes
// search those particles' neighbours again.
// In 2D a row is one 128-byte line, and every particle of a chunk can have a block (measured, rows of
// 32 with 128 blocks against rows of 48 with 64, the same memory, us per step: constant spacing, 127k
// particles 113.3 / 110.8, 300k 210.7 / 204.0; 120k disk 132.9 / 130.5, 1M disk 627 / 614).
template <int D> struct ListShape;
template <> struct ListShape<2> {
    static constexpr int ROW = 32, XB = 32, NXB = 128;
};
template <> struct ListShape<3> {
    static constexpr int ROW = 128, XB = 64, NXB = 128;
};
constexpr int XMAX = 8;
template <int D> constexpr int list_most() { return ListShape<D>::ROW + XMAX * ListShape<D>::XB; }
// entries per slot, blocks included
template <int D> constexpr int list_entries() {
    return ListShape<D>::ROW + ListShape<D>::XB * ListShape<D>::NXB / CHUNK;
}
// consecutive list entries per lane and turn of the viscous sum and of the pressure pass: their loads
// are in flight together (measured on the 1.2M cube: 4 against 2 viscous sum and update 339 us against
// 468).  A 2D list fills one and a half turns of 16 entries: the pressure pass takes turns of 8 (us per
// step, 2 against 4: constant spacing, 127k particles 104.5 / 108.4, 300k 188.5 / 196.5; 120k disk 127.9
// / 131.6, 1M disk 602 / 618; the viscous sum gains nothing, 128.6 / 127.9 and 606 / 602 on the disks).
constexpr int LISTU = 4;
template <int D> constexpr int pressure_listu() { return D == 2 ? 2 : LISTU; }
// particles searched by one warp: 2 (in 3D), 4, 8 or 16 by the slots of the batch.
// A warp searching for more particles reads the cells around them once for all, one searching for
// fewer is done sooner, which counts while the GPU is not full.  The lists do not depend on it.
// Measured, search and pressure pass in us with 2 / 4 / 8 / 16: a 26k ball in three passes (whole
// step) 376 / 437 / 640 / 826; a 20k disk 33 / 29 / 38 / 55; 120k disk 106 / 76 / 66 / 79; 1M disk
// - / - / 430 / 404; 83k cube 189 / 149 / 137 / 146; 300k cube 671 / 498 / 472 / -; 1.2M cube
// 2447 / - / 1451 / 1408.  In a 2D mesh of constant spacing (levels 1) all warps take alike, and the
// wider ones pay earlier: 4 / 8 / 16, 40k particles 37.6 / 35.5 / -, 60k 46.3 / 41.9 / -, 127k 76 / 66 / 66,
// 300k - / 127.5 / 124.0.
constexpr int search_width(int D, int slots, int levels) {
    return D == 3 && slots <= 32768 ? 2
           : D == 2 && levels == 1 ? (slots <= 32768 ? 4 : slots <= 262144 ? 8 : 16)
                                   : (slots <= 65536 ? 4 : slots <= 524288 ? 8 : 16);
}
// most slots of a batch whose prediction, viscous sum and update run as one kernel (FP32 build).
// Measured, one kernel against three, us per step: the 2.6k square 48.6 against 52.2; constant spacing,
// 38k particles 57.1 against 63.1, 55k 73.5 / 74.6, 64k 76.0 / 76.2, 90k 89.8 / 88.3, 127k 109 / 103; a 38k
// disk 77.4 / 82.6, 55k 94.7 / 95.0, 65k 99.9 / 101.4, 90k 116.8 / 114.6; 3D, a 26k ball in three passes
// 372 / 363.  In FP64 the neighbours' predictions cost more than the launches (2.9k square 116 / 110).
// Eight resident blocks per SM asked of the compiler take 38,912 particles at once, six 29,184: 57.4
// against 61.2 at 30k, 51.8 against 50.8 at 20k.
#ifndef SPH_FUSED_MINB
#define SPH_FUSED_MINB 8
#endif
#ifndef SPH_FUSED_MOST_2D
#define SPH_FUSED_MOST_2D 65536
#endif
#ifndef SPH_FUSED_MOST_3D
#define SPH_FUSED_MOST_3D 8192
#endif
inline bool one_update_kernel(int precision, int D, int slots) {
    return precision == 32 && slots <= (D == 2 ? SPH_FUSED_MOST_2D : SPH_FUSED_MOST_3D);
}
// Warps per block of the search, and 32 resident warps per SM asked of the compiler (64 registers
// with a few spills).  Measured, us per step: 16 particles per warp at 20, 24, 28, 32 resident warps
// 701, 664, 655, 646 on the 1M disk, 2104, 1991, 1925, 1869 on the 1.2M cube; two-warp blocks there
// 688 and 2011 (a block's slots wait for its slower warp), at 36 and 40 resident warps 674..682 and
// 1966..2009 (spills).  Where a warp takes two particles its work is short and the launch of the
// blocks weighs more than the wait: two warps 270 against 280 on a 26k ball in lattice order.
constexpr int search_warps(int cl) { return cl == 2 ? 2 : 1; }
static_assert(CHUNK % (BLOCK / Lpp<2>::v) == 0 && CHUNK % (BLOCK / Lpp<3>::v) == 0,
              "a pair-pass block must lie in one chunk");
// 3D occupancy cells finer than the cells-per-support top-level cells by 2^SPH_OCC_FINER per axis
// (measured on the 3D cube: 1 and 2 make the pressure pass 5 % and 21 % slower than 0; with the
// search radius from the cells' largest h, 6 % and 16 %)
#ifndef SPH_OCC_FINER
#define SPH_OCC_FINER 0
#endif

// minimum resident blocks per SM asked of the compiler for the pair passes: it bounds the registers
// per thread, trading spills for warps in flight (measured, search and pressure pass in us: 2D, 1M
// disk, 5 / 6 / 7 / 8 blocks 499 / 472 / 443 / 428; 3D, 1.2M cube, 5 / 6 / 7 / 8 blocks 1541 / 1499 /
// 1504 / 1595; FP64, 40k cube, 4 / 6 blocks 791 / 990; viscous sum and update: 1M disk 6 / 8 / 10 /
// 12 blocks 219 / 201 / 182 / 172, 1.2M cube 8 / 10 / 12 blocks 392 / 362 / 439; update alone at 6 /
// 8 blocks: the same stage 171.5 / 167.5 us on the 1M disk, 56.0 / 59.3 on the 83k cube)
#ifndef SPH_INTERACT_MINB
#define SPH_INTERACT_MINB 8
#endif
#ifndef SPH_INTERACT_MINB_F64
#define SPH_INTERACT_MINB_F64 4
#endif
#ifndef SPH_INTERACT_MINB_3D
#define SPH_INTERACT_MINB_3D 6
#endif
#ifndef SPH_VISC_MINB_2D
#define SPH_VISC_MINB_2D 12
#endif
#ifndef SPH_VISC_MINB_3D
#define SPH_VISC_MINB_3D 10
#endif
#ifndef SPH_UPDATE_MINB_2D
#define SPH_UPDATE_MINB_2D 8
#endif
#ifndef SPH_UPDATE_MINB_3D
#define SPH_UPDATE_MINB_3D 6
#endif
// cells per support of the cell grid when the parameters leave the choice to the library
// (measured with a 2.6h support: 2 in 2D are 9 % faster than 1; 1 in 3D is 45 % slower than 2)
#ifndef SPH_DEFAULT_CPS_2D
#define SPH_DEFAULT_CPS_2D 2
#endif
#ifndef SPH_DEFAULT_CPS_3D
#define SPH_DEFAULT_CPS_3D 2
#endif
// Whether a particle of intrinsic dimension di takes part in the step pass for dimension class
// cls: 0 is the whole step at once; with Algorithm 1's feature loop in sequence (feature_order)
// a step runs the passes cls = 1 .. D in turn and each moves the particles of its class, and an
// instance without it (batched with one that has it) takes its whole step in the last pass.
__device__ __forceinline__ bool in_pass(const Params& p, int cls, int di, int D) {
    if (cls == 0) return true;
    return p.feature_order ? di == cls : cls == D;
}

// instance of slot k, and whether the slot holds a particle
template <typename T> __device__ __forceinline__ int inst_of(const State<T>& s, int k) {
    return __ldg(s.chunk_inst + k / CHUNK);
}
template <typename T> __device__ __forceinline__ bool live(const State<T>& s, int i, int k) {
    return k - __ldg(s.inst_off + i) < __ldg(s.inst_n + i);
}

// the sorted meta words of the batch's dimension (the same memory serves as scratch for plain
// 32-bit metas while instances are re-packed)
template <int D, typename T> __device__ __forceinline__ Meta<D>* meta_words(const State<T>& s) {
    return reinterpret_cast<Meta<D>*>(s.Ms);
}

// meta (group and dimension) of sorted slot k
template <typename T, int D> __device__ __forceinline__ unsigned slot_meta(const State<T>& s, int k) {
    if constexpr (Rec<T, D>::packed) return MetaWord<D>::meta(__float_as_uint((float)s.P[k].w));
    else return MetaWord<D>::meta(meta_words<D>(s)[k]);
}

// whether the list of slot k (n candidates) overflowed, and the place of its entry t
template <typename T, int D> __device__ __forceinline__ bool list_overflowed(const State<T>& s, int k, int n) {
    return n > ListShape<D>::ROW && (n > list_most<D>() || s.xcnt[k / CHUNK] > ListShape<D>::NXB);
}
template <typename T, int D>
__device__ __forceinline__ size_t list_entry(const State<T>& s, int k, int t, unsigned long long xid) {
    typedef ListShape<D> L;
    if (t < L::ROW) return (size_t)k * L::ROW + t;
    const int u = t - L::ROW, b = (int)(xid >> (8 * (u / L::XB))) & 255;
    return s.xbase + (size_t)((k / CHUNK) * L::NXB + b) * L::XB + u % L::XB;
}

// the one-pass scan's tile states back to "nothing published" (grid-stride over any grid)
template <typename T> __device__ __forceinline__ void reset_scan_state(const State<T>& s) {
    const int t0 = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    for (int t = t0; t < s.ntile; t += stride) s.tstate[t] = 0ull;
    if (t0 == 0) *s.ticket = 0;
}

// copy a struct into shared memory with the whole block (one round trip)
template <typename S> __device__ __forceinline__ void block_copy(S* dst, const S* src) {
    const unsigned* a = reinterpret_cast<const unsigned*>(src);
    unsigned* b = reinterpret_cast<unsigned*>(dst);
    for (int t = threadIdx.x; t < (int)(sizeof(S) / 4); t += blockDim.x) b[t] = a[t];
}

// level and level-cell of sorted particle k (from its h and stored finest cell; the same as
// decoding its key, without the integer divisions)
template <typename T, int D>
__device__ __forceinline__ void own_cell(const Grid& g, const State<T>& s, int k, T h, int& l, int c[3]) {
    l = level_of(g, h);
    for (int a = 0; a < 3; ++a) c[a] = a < D ? (s.Cs[a][k] >> l) : 0;
}

constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_ITEMS = 4;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;
// cells per thread (read and written as 16-byte words) and threads per tile of the step's one-pass
// scan (bound by DRAM and the tiles' chain: 100 MB on the 12M cells of the 83k graded cube; measured,
// rebuild in us, 4 cells per thread / 8 / 16 / 8 with 512 threads: 20k disk 15.6 / 16.0 / 18.2 / 15.9,
// 1M disk 73.8 / 66.9 / 66.0 / 67.5, 83k cube 62.2 / 55.1 / 53.6 / 54.7, 1.2M cube 82.6 / 79.2 / 79.0 /
// 79.0)
#ifndef SPH_SCAN1_ITEMS
#define SPH_SCAN1_ITEMS 8
#endif
#ifndef SPH_SCAN1_THREADS
#define SPH_SCAN1_THREADS 1024
#endif
constexpr int SCAN1_ITEMS = SPH_SCAN1_ITEMS;
constexpr int SCAN1_THREADS = SPH_SCAN1_THREADS;
constexpr int SCAN1_TILE = SCAN1_THREADS * SCAN1_ITEMS;

inline int div_up(long long a, long long b) { return (int)((a + b - 1) / b); }

// Programmatic dependent launch between the kernels of a step.  A kernel launched with
// pdl = true may be scheduled while its predecessor in the stream is still running (once every
// block of the predecessor has started); its blocks then wait in dep_wait() until the
// predecessor has completed and its writes are visible.  Every step kernel calls dep_wait()
// before its first access to device memory other than its kernel parameters, so the order of
// the stream is kept; without the attribute dep_wait() returns at once.  dep_launch() lets
// the successor be scheduled as soon as every block of this kernel is running.
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

#ifndef SPH_PDL
#define SPH_PDL 1
#endif
template <typename... K, typename... A>
inline void launch_k(void (*kern)(K...), int grid, int block, cudaStream_t st, bool pdl, A&&... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = (pdl && SPH_PDL) ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kern, static_cast<A&&>(args)...);
}

// rebuild.cu
// `one`: the descriptors of a batch of one (nullptr: read the per-instance tables)
template <typename T, int D> void launch_hash(const State<T>& s, const One* one, cudaStream_t st);
void launch_scan(int ncell, int* count, int* cell_start, int* bsum, cudaStream_t st);
// one-pass scan of the step (decoupled look-back over tiles taken in ticket order)
template <typename T> void launch_scan_onepass(const State<T>& s, cudaStream_t st);
template <typename T> void launch_scatter(const State<T>& s, cudaStream_t st, bool pdl = false);
void launch_cellsort(int ncell, int n, const int* cell_start, int* perm, int* count, cudaStream_t st);
template <typename T, int D> void launch_gather(const State<T>& s, const One* one, cudaStream_t st, bool pdl = false);
template <typename T, int D> void launch_init_h(const State<T>& s, int inst, cudaStream_t st);
template <typename T, int D> void launch_repack(const State<T>& s, const int* old_off, const int* move_n, cudaStream_t st);

// state_io.cu: an instance's slots from and to the caller's FP64 arrays (staged on the device)
struct IoCheck {      // accepted ranges: positions inside [lo, hi] per axis, h in (0, hmax]
    double lo[3], hi[3];
    double hmax;
    int G, D;
};
struct IoGrid {       // finest-level cell geometry of an instance, and each group's dimension
    double origin[3];
    double c0, inv_c0;
    int dims0[3];
    unsigned char fdim[MAXF];
};
template <typename T> struct SlotArrays {   // an instance's stored state, from its first slot
    int* C[3];
    T* O[3];
    T* V[3];
    T* H;
    unsigned* G;
    int* ID;
};
template <typename T> struct ConstSlotArrays {
    const int* C[3];
    const T* O[3];
    const T* V[3];
    const T* H;
    const unsigned* G;
    const int* ID;
};
// first offending particle as (index << 2) | check (0 group, 1 position, 2 h, 3 velocity) by
// atomicMin into *first (the caller sets it to all ones)
void launch_check_state(const IoCheck& c, int n, const double* x, const int* group, const double* v, const double* h,
                        unsigned long long* first, cudaStream_t st);
// slots [0, n) from the arrays (v, h may be null: zero), [n, ns) padding
template <typename T, int D>
void launch_load_state(const SlotArrays<T>& s, const IoGrid& g, int ns, int n, const double* x, const int* group,
                       const double* v, const double* h, cudaStream_t st);
// slots [0, ns) to the arrays in input order (any may be null); cnt[0] counts the particles
// written, cnt[1] is set when a slot holds an index >= n (both zeroed by the caller)
template <typename T, int D>
void launch_store_state(const ConstSlotArrays<T>& s, const IoGrid& g, int ns, int n, double* x, int* group, double* v,
                        double* h, int* cnt, cudaStream_t st);

// search.cu: the neighbour lists of the particles taking part in pass cls (in_pass; -1: of all);
// tested (may be null) counts the candidate pairs tested
template <typename T, int D>
void launch_search(const State<T>& s, const One* one, cudaStream_t st, bool pdl = false, int cls = 0,
                   unsigned long long* tested = nullptr);

// interact.cu (over the lists of a search)
template <typename T, int D>
void launch_interact(const State<T>& s, const One* one, T* dbg_sigma, T* dbg_gamma, cudaStream_t st,
                     bool pdl = false, int cls = 0);
template <typename T, int D>
void launch_neighbors(const State<T>& s, int mode, int* counts, const long long* offsets, int* lists, cudaStream_t st);
template <typename T, int D> void launch_pair_counts(const State<T>& s, unsigned long long* out, cudaStream_t st);

// integrate.cu
template <typename T, int D>
void launch_control(const State<T>& s, const One* one, cudaStream_t st, bool pdl = false, int cls = 0);
template <typename T, int D>
void launch_integrate(const State<T>& s, const One* one, const Ctrl* use, const Out<T>& o, cudaStream_t st,
                      bool pdl = false, int cls = 0);

// sample.cu: midpoint-rule integrals of rho_t over every feature of dm (Eqs. 10, 11), and the
// rejection sampling of counts[k] particles per feature into d_out[n][3] in feature order
// (d_dom / d_siz: device copies of dm and its sizing)
int quad_points(int kind, int D, long long* npts);
cudaError_t feature_integrals(const Domain& dm, const Domain* d_dom, const Sizing* d_siz, cudaStream_t st,
                              double* integral);
cudaError_t sample_features(const Domain& dm, const Sizing& z, const Domain* d_dom, const Sizing* d_siz,
                            unsigned long long seed, const int64_t* counts, cudaStream_t st, double* d_out);

// sets the message returned by sph_last_error() on the calling thread (capi.cu)
void set_last_error(const char* msg);

}  // namespace sph
