// mrlt_tree.cu -- tree kernels of the MRLT library: projections and tree
// refreshing (Eqs. 3, 15-22; Algs. 3, 4, 6, 8, 9), the multiresolution
// adaptation (details Eq. 5, thresholding Alg. 2, graded closure Alg. 1),
// compaction of the per-level leaf / internal-node / tile lists,
// conservative flux registers, reductions and read-back packing.
#include "mrlt_tree.cuh"

namespace mrlt {

static inline int blocks_dense(long long n)
{
    long long b = (n + NTHREADS - 1) / NTHREADS;
    return (int)(b < 1 ? 1 : (b > 65535 ? 65535 : b));
}
// blocks of the passes that take 16 cells per thread
static inline int blocks_step(const Grid& g, int l)
{
    return blocks_dense(l < kStepLevel ? g.N[l] : g.N[l] / kStep);
}
static inline int blocks_list(const Grid& g, int l)
{
    long long b = (g.N[l] + NTHREADS - 1) / NTHREADS;
    return (int)(b < 1 ? 1 : (b > 1216 ? 1216 : b));
}

#define GRID_STRIDE(i, n) MRLT_GRID_STRIDE(i, n)

// ------------------------------------------------------------ kernels
// Each kernel waits for its predecessor (programmatic dependent launch) and
// runs one device body of mrlt_tree_dev.cuh over its own grid; kernels that leave
// the tree alone look it up before they wait (tree_enter).  Most launches
// are short chains of dependent trips, so that takes two or three of five trips
// off them (figures at tree_enter).
// (T: the storage type of the fields, double or float)
template <int M, class T>
__global__ void k_leaf_copy(const __grid_constant__ Grid g, int lo, int hi, int from, int to)
{
    MRLT_ENTER(g);
    dev_leaf_copy<M, T>(g, lo, hi, from, to);
}

// Up-sweep of levels hi..lo (one level: hi = lo).
template <int D, int M, class T>
__global__ void k_project_up(const __grid_constant__ Grid g, int hi, int lo, int mode, int top, TreeSync sync)
{
    const bool waited = tree_enter<D>(g, sync);
    const int steps = up_steps(g, hi, lo);
    UpRefs<D> r = up_lookup<D>(g, hi, lo, blockIdx.x);
    if (!waited) pdl_enter();
    if (halted(g)) return;
    for (int c = blockIdx.x; c < steps; c += gridDim.x) { // uniform across the CTA
        if (c != (int)blockIdx.x) r = up_lookup<D>(g, hi, lo, c);
        up_project<D, M, T>(g, r, hi - lo, mode, top);
    }
}

// The beginning of an iteration: q^n := end value of the leaves of levels
// lo..L and, beside it, the up-sweep of levels uhi..ulo (which reads leaf
// children's end values; ulo with mode top): one launch where the copy and the
// sweep were two.
template <int D, int M, class T>
__global__ void k_begin(const __grid_constant__ Grid g, int lo, bool next, int uhi, int ulo, int top, TreeSync sync)
{
    const bool waited = tree_enter<D>(g, sync);
    const int steps = uhi >= ulo ? up_steps(g, uhi, ulo) : 0;
    UpRefs<D> r;
    if (uhi >= ulo) r = up_lookup<D>(g, uhi, ulo, blockIdx.x);
    kernel_list<0>(
        g, lo, g.L, waited, [&](int l, long long id) { return slot_of(g, l, id); },
        [&](int sl) {
            T q[M];
            load_row<M, T>(nd<T>(g, F_QE, sl), q);
            store_row<M, T>(nd<T>(g, F_Q0, sl), q);
        });
    if (halted(g)) return;
    if (next && blockIdx.x == 0 && threadIdx.x == 0) ++g.room[4]; // the next iteration of the macro step
    for (int c = blockIdx.x; c < steps; c += gridDim.x) { // uniform across the CTA
        if (c != (int)blockIdx.x) r = up_lookup<D>(g, uhi, ulo, c);
        up_project<D, M, T>(g, r, uhi - ulo, PM_BEG, top);
    }
}

template <int D, int M, class T>
__global__ void k_detail(const __grid_constant__ Grid g, int lo, int hi, TreeSync sync)
{
    kernel_list<1>(
        g, lo, hi, tree_enter<D>(g, sync), [&](int l, long long id) { return lookup_detail<D>(g, l, id); },
        [&](const DetailRefs<D>& e) { detail_node<D, M, T>(g, e); });
}

// Desired and admissible refinements in one pass: desire reads only the detail
// bits, which the stores of the refinement bit keep.
// count: the tree's size is checked (room_count); last: this launch finalises
// the flags (a remesh at level la = L-1 has no closure) and decides.
template <int D>
__global__ void k_mark(const __grid_constant__ Grid g, int lo, int hi, int la, bool count, bool last)
{
    MRLT_ENTER(g);
    const int c = dev_mark<D>(g, lo, hi, la);
    if (last) room_decide(g, c, la);
    else if (count) room_count(g, c);
}

// last: the last closure (level l-1 = la)
template <int D>
__global__ void k_close(const __grid_constant__ Grid g, int l, bool count, bool last)
{
    MRLT_ENTER(g);
    const int c = dev_close<D>(g, l);
    if (last) room_decide(g, c, l - 1);
    else if (count) room_count(g, c);
}

template <int D, int M, class T>
__global__ void k_apply(const __grid_constant__ Grid g, int l, int la)
{
    MRLT_ENTER(g);
    dev_apply<D, M, T, NTHREADS>(g, l, la);
}

// the releases of a remesh and its installation on level la in one launch:
// level la creates no node (its nodes stay; only leaf and internal swap), so
// it takes no slot, and the released nodes (levels above la) are not its
template <int D, int M, class T>
__global__ void k_release_apply(const __grid_constant__ Grid g, int la)
{
    MRLT_ENTER(g);
    dev_release(g, la);
    dev_apply<D, M, T, NTHREADS>(g, la, la);
}

// A small 1D tree (at most kOneBlock cells on the finest level: one step per
// thread) is flagged and installed by one block each, its levels separated by
// barriers instead of launches.  Measured on a GB300, a launch per level against
// this: 1D Burgers L = 9 15.84 / 14.95 ms, L = 10 17.8 / 17.1, L = 12 10.99 /
// 10.20; with as many cells in 2D (Euler L = 6) 6.08 / 6.06 and in 3D (Burgers
// L = 4) 0.80 / 0.84 ms, whose nodes hold more work than one block has threads.
// Whether the new tree fits is not asked: at most 8191 nodes of at most 244 bytes
// always have a slot for every cell (kDenseBytes).
constexpr int kOneBlockThreads = 256;
constexpr long long kOneBlock = kOneBlockThreads * kStep;

template <int D>
__global__ void __launch_bounds__(kOneBlockThreads) k_flag_small(const __grid_constant__ Grid g, int la)
{
    MRLT_ENTER(g);
    dev_mark<D>(g, la, g.L - 1, la);
    for (int l = g.L - 1; l > la; --l) {
        __syncthreads();
        dev_close<D>(g, l);
    }
}

template <int D, int M, class T>
__global__ void __launch_bounds__(kOneBlockThreads) k_install_small(const __grid_constant__ Grid g, int la)
{
    MRLT_ENTER(g);
    dev_release(g, la);
    __syncthreads();
    for (int l = la; l <= g.L; ++l) dev_apply<D, M, T, kOneBlockThreads>(g, l, la); // ends with a barrier
}

// compaction of levels lo..hi: one block per chunk
__global__ void k_cmp_count(const __grid_constant__ Grid g, LevelChunks lc, int* bc)
{
    MRLT_ENTER(g);
    chunk_count<NTHREADS>(g, lc, blockIdx.x, bc);
}

// the tile lists (the longest single blocks) first, then one block per chunk
__global__ void k_cmp_scatter(const __grid_constant__ Grid g, LevelChunks lc, const int* bc)
{
    MRLT_ENTER(g);
    const int levels = lc.hi - lc.lo + 1;
    if ((int)blockIdx.x < levels) level_tile_list<NTHREADS>(g, lc.hi - blockIdx.x);
    else chunk_scatter<NTHREADS>(g, lc, blockIdx.x - levels, bc);
}

template <int D, int M, class T>
__global__ void k_reflux(const __grid_constant__ Grid g, int lo, int hi, TreeSync sync)
{
    kernel_list<0>(
        g, lo, hi, tree_enter<D>(g, sync), [&](int l, long long id) { return lookup_reflux<D>(g, l, id); },
        [&](const RefluxRefs<D>& e) { reflux_leaf<D, M, T>(g, e); });
}

// ------------------------------------------------------------ reductions
template <int M, class T>
__global__ void k_scale(const __grid_constant__ Grid g)
{
    MRLT_ENTER(g);
    dev_scale<M, T>(g, g.lb, g.L);
}

template <int M, class T>
__global__ void k_finite(const __grid_constant__ Grid g)
{
    MRLT_ENTER(g);
    dev_finite<M, T>(g, g.lb, g.L);
}

// fixed-shape partial sums (deterministic): part[block * m + v]
template <class T>
__global__ void k_mass(Grid g, int l, double* part)
{
    pdl_enter();
    __shared__ double sh[NTHREADS];
    const int cnt = g.counts[l];
    const int* list = g.leaves + g.off[l];
    const long long N = g.N[l];
    for (int v = 0; v < g.m; ++v) {
        double acc = 0.0;
        for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < cnt;
             t += (long long)gridDim.x * blockDim.x) {
            const long long id = list[t];
            if (id >= 0 && id < N) acc += double(nd<T>(g, F_QE, slot_of(g, l, id))[v]);
        }
        sh[threadIdx.x] = acc;
        __syncthreads();
        for (int o = NTHREADS / 2; o > 0; o >>= 1) {
            if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) part[blockIdx.x * g.m + v] = sh[0];
        __syncthreads();
    }
}

template <int M, class T>
__global__ void k_pack(const __grid_constant__ Grid g, int* keys, double* vals)
{
    pdl_enter();
    for_list<0>(g, g.lb, g.L, [&](int l, long long id, long long t) {
        if (keys) {
            int c[3];
            cell_xyz(g, l, id, c);
            reinterpret_cast<int4*>(keys)[t] = make_int4(l, c[0], c[1], c[2]);
        }
        if (vals) {
            T q[M];
            load_row<M, T>(nd<T>(g, F_QE, slot_of(g, l, id)), q);
            double r[M];
#pragma unroll
            for (int v = 0; v < M; ++v) r[v] = double(q[v]);
            store_row<M, double>(vals + t * M, r);
        }
    });
}

// inverse MR transform onto the finest level, in scratch pyramids T / us:
// bottom-up projection of the leaves' q^{n+1} into internal nodes, then
// top-down prediction of every absent cell from the level above
template <int D, class F>
__global__ void k_uni_up(Grid g, int l, double* T, uint8_t* us)
{
    pdl_enter();
    const long long N = g.N[l];
    const long long Nc = l < g.L ? g.N[l + 1] : 0;
    double* Tl = T + g.off[l] * g.m;
    const double* Tc = l < g.L ? T + g.off[l + 1] * g.m : nullptr;
    GRID_STRIDE(id, N)
    {
        const int s = status(g, l, id);
        us[g.off[l] + id] = s != 0;
        if (s == 1) {
            for (int v = 0; v < g.m; ++v) Tl[v * N + id] = double(nd<F>(g, F_QE, slot_of(g, l, id))[v]);
        } else if (s == 2) {
            int c[3];
            cell_xyz(g, l, id, c);
            for (int v = 0; v < g.m; ++v) {
                double acc = 0.0;
                for (int k = 0; k < (1 << D); ++k)
                    acc += Tc[v * Nc + cell_id(g, l + 1, 2 * c[0] + (k & 1), D > 1 ? 2 * c[1] + ((k >> 1) & 1) : 0,
                                                D > 2 ? 2 * c[2] + ((k >> 2) & 1) : 0)];
                Tl[v * N + id] = acc * (1.0 / (1 << D));
            }
        }
    }
}

template <int D>
__global__ void k_uni_down(Grid g, int l, double* T, uint8_t* us)
{
    pdl_enter();
    const long long N = g.N[l], Np = g.N[l - 1];
    double* Tl = T + g.off[l] * g.m;
    const double* Tp = T + g.off[l - 1] * g.m;
    GRID_STRIDE(id, N)
    {
        if (us[g.off[l] + id]) continue;
        int c[3];
        cell_xyz(g, l, id, c);
        const int P[3] = {c[0] >> 1, c[1] >> 1, c[2] >> 1};
        for (int v = 0; v < g.m; ++v) {
            double acc = 0.0;
            MRLT_FOR3(D, dx, dy, dz)
            {
                int neg = 0;
                const int x = wrap_or_mirror(g, l - 1, 0, P[0] + dx, neg);
                const int y = D > 1 ? wrap_or_mirror(g, l - 1, 1, P[1] + dy, neg) : 0;
                const int z = D > 2 ? wrap_or_mirror(g, l - 1, 2, P[2] + dz, neg) : 0;
                const double w0 = pw(c[0] & 1, dx) * (D > 1 ? pw(c[1] & 1, dy) : 1.0) * (D > 2 ? pw(c[2] & 1, dz) : 1.0);
                const double w = neg ? -w0 : w0;
                acc += w * Tp[v * Np + cell_id(g, l - 1, x, y, z)];
            }
            Tl[v * N + id] = acc;
        }
        us[g.off[l] + id] = 1;
    }
}

// ------------------------------------------------------------ launchers
// fn<D, M>(...) for the solver's dimension and number of variables
#define MRLT_DM_DISPATCH(fn, ...)                                   \
    do {                                                            \
        if (g.d == 1 && g.m == 1) fn<1, 1>(__VA_ARGS__);            \
        else if (g.d == 1) fn<1, 3>(__VA_ARGS__);                   \
        else if (g.d == 2 && g.m == 1) fn<2, 1>(__VA_ARGS__);       \
        else if (g.d == 2) fn<2, 4>(__VA_ARGS__);                   \
        else if (g.m == 1) fn<3, 1>(__VA_ARGS__);                   \
        else fn<3, 5>(__VA_ARGS__);                                 \
    } while (0)

// launch k<..., T> with the fields' storage type: float in the mixed mode
#define MRLT_T_LAUNCH(L, blocks, args, ...)                                                                    \
    do {                                                                                                       \
        if ((L).g.prec) pdl_launch(__VA_ARGS__, float>, blocks, NTHREADS, 0, (L).st, MRLT_UNPACK args);        \
        else pdl_launch(__VA_ARGS__, double>, blocks, NTHREADS, 0, (L).st, MRLT_UNPACK args);                  \
    } while (0)
#define MRLT_UNPACK(...) __VA_ARGS__

// Up-sweep hi -> lo in groups of at most 6 / d + 1 levels per launch: a group
// [glo, ghi] has 2^{d (ghi - glo)} <= 64 descendants per top node, so two top
// nodes fit the NTHREADS = 128 threads of a CTA.  Level lo takes mode `top`.
static int up_blocks(const Grid& g, int ghi, int glo)
{
    if (ghi <= glo) return blocks_list(g, glo);
    const int tops = NTHREADS >> (g.d * (ghi - glo));
    const long long b = (g.N[glo] + tops - 1) / tops;
    return (int)(b > 1216 ? 1216 : b);
}

template <int D, int M>
static void project_up_dm(Launcher& L, int hi, int lo, int mode, int top)
{
    static_assert((1 << (D * kUpDepth<D>)) * 2 <= NTHREADS, "two top nodes per CTA");
    for (int ghi = hi; ghi >= lo;) {
        const int glo = ghi - kUpDepth<D> > lo ? ghi - kUpDepth<D> : lo;
        MRLT_T_LAUNCH(L, up_blocks(L.g, ghi, glo), (L.g, ghi, glo, mode, glo == lo ? top : mode, L.enter()),
                      k_project_up<D, M);
        ++L.n;
        ghi = glo - 1;
    }
}

void Launcher::project(int l, int mode) { MRLT_DM_DISPATCH(project_up_dm, *this, l, l, mode, mode); }

void Launcher::project_up(int hi, int lo, int mode, int top)
{
    if (hi >= lo) MRLT_DM_DISPATCH(project_up_dm, *this, hi, lo, mode, top < 0 ? mode : top);
}

template <int D, int M>
static void begin_dm(Launcher& L, int lmin, bool next, int lo, int top)
{
    const Grid& g = L.g;
    const int ghi = g.L - 1, glo = ghi - kUpDepth<D> > lo ? ghi - kUpDepth<D> : lo;
    const int b0 = blocks_list(g, g.L), b1 = ghi >= lo ? up_blocks(g, ghi, glo) : 1;
    MRLT_T_LAUNCH(L, b0 > b1 ? b0 : b1, (g, lmin, next, ghi, glo, glo == lo ? top : (int)PM_BEG, L.enter()),
                  k_begin<D, M);
    ++L.n;
    if (glo > lo) project_up_dm<D, M>(L, glo - 1, lo, PM_BEG, top);
}

void Launcher::begin(int lmin, bool next, int lo, int top) { MRLT_DM_DISPATCH(begin_dm, *this, lmin, next, lo, top); }

template <int D, int M>
static void leaf_copy_dm(Launcher& L, int lo, int hi, int from, int to)
{
    MRLT_T_LAUNCH(L, blocks_list(L.g, hi), (L.g, lo, hi, from, to), k_leaf_copy<M);
    ++L.n;
}

void Launcher::leaf_copy(int lo, int hi, int from, int to) { MRLT_DM_DISPATCH(leaf_copy_dm, *this, lo, hi, from, to); }

template <int D, int M>
static void adapt_dm(Launcher& L, int la, bool check)
{
    const Grid& g = L.g;
    const int hi = g.L - 1; // levels whose nodes may own children
    MRLT_T_LAUNCH(L, blocks_list(g, hi), (g, la, hi, L.enter()), k_detail<D, M);
    ++L.n;
    if constexpr (D == 1) {
        if (g.N[g.L] <= kOneBlock) {
            pdl_launch(k_flag_small<D>, 1, kOneBlockThreads, 0, L.st, g, la);
            ++L.n;
            return;
        }
    }
    pdl_launch(k_mark<D>, blocks_step(g, hi), NTHREADS, 0, L.st, g, la, hi, la, check, check && la == hi);
    ++L.n;
    for (int l = g.L - 1; l > la; --l, ++L.n)
        pdl_launch(k_close<D>, blocks_step(g, l - 1), NTHREADS, 0, L.st, g, l, check, check && l == la + 1);
}


template <int D, int M>
static void apply_dm(Launcher& L, int la)
{
    const Grid& g = L.g;
    if constexpr (D == 1) {
        if (g.N[g.L] <= kOneBlock) {
            if (g.prec) pdl_launch(k_install_small<D, M, float>, 1, kOneBlockThreads, 0, L.st, g, la);
            else pdl_launch(k_install_small<D, M, double>, 1, kOneBlockThreads, 0, L.st, g, la);
            ++L.n;
            return;
        }
    }
    const int b0 = blocks_list(g, g.L), b1 = blocks_step(g, la);
    if (g.prec) pdl_launch(k_release_apply<D, M, float>, b0 > b1 ? b0 : b1, NTHREADS, 0, L.st, g, la);
    else pdl_launch(k_release_apply<D, M, double>, b0 > b1 ? b0 : b1, NTHREADS, 0, L.st, g, la);
    ++L.n;
    for (int l = la + 1; l <= g.L; ++l, ++L.n) {
        if (g.prec) pdl_launch(k_apply<D, M, float>, blocks_step(g, l), NTHREADS, 0, L.st, g, l, la);
        else pdl_launch(k_apply<D, M, double>, blocks_step(g, l), NTHREADS, 0, L.st, g, l, la);
    }
}

void Launcher::mark_refinements(int la, bool check) { MRLT_DM_DISPATCH(adapt_dm, *this, la, check); }
void Launcher::apply_tree(int la) { MRLT_DM_DISPATCH(apply_dm, *this, la); }

void Launcher::compact(int lo, int hi)
{
    LevelChunks lc;
    const int total = number_chunks(g, lc, lo, hi);
    pdl_launch(k_cmp_count, total, NTHREADS, 0, st, g, lc, bc);
    pdl_launch(k_cmp_scatter, total + hi - lo + 1, NTHREADS, 0, st, g, lc, (const int*)bc);
    n += 2;
    stale = true;
}

template <int D, int M>
static void reflux_dm(Launcher& L, int lo, int hi)
{
    MRLT_T_LAUNCH(L, blocks_list(L.g, hi), (L.g, lo, hi, L.enter()), k_reflux<D, M);
    ++L.n;
}

void Launcher::reflux(int lo, int hi) { MRLT_DM_DISPATCH(reflux_dm, *this, lo, hi); }

__global__ void k_scale_init(Grid g)
{
    MRLT_ENTER(g);
    if (threadIdx.x < MMAX) g.scale_bits[threadIdx.x] = (unsigned long long)__double_as_longlong(1e-14);
}

__global__ void k_set_dt(Grid g, double dt)
{
    pdl_enter();
    if (threadIdx.x == 0) {
        *g.dtp = dt;
        g.room[4] = 0; // iteration 0
    }
}

// leaf values from (level, i, j, k) keys: q^n and the end value of each leaf
// (restoring a state saved at a macro-step boundary); a key that is not a
// leaf of the installed tree sets ERR_INDEX
template <class T>
__global__ void k_set_leaves(Grid g, const int* keys, const double* vals, long long n)
{
    pdl_enter();
    GRID_STRIDE(t, n)
    {
        const int* K = keys + 4 * t;
        const int l = K[0];
        if (l < g.lb || l > g.L || K[1] < 0 || K[1] >= g.n[l] || (g.d > 1 && (K[2] < 0 || K[2] >= g.n[l])) ||
            (g.d > 2 && (K[3] < 0 || K[3] >= g.n[l]))) {
            atomicOr(g.err, ERR_INDEX);
            continue;
        }
        const long long id = cell_id(g, l, K[1], g.d > 1 ? K[2] : 0, g.d > 2 ? K[3] : 0);
        if (status(g, l, id) != 1) {
            atomicOr(g.err, ERR_INDEX);
            continue;
        }
        const int sl = slot_of(g, l, id);
        T* q0 = nd<T>(g, F_Q0, sl);
        T* qe = nd<T>(g, F_QE, sl);
        for (int v = 0; v < g.m; ++v) q0[v] = qe[v] = T(vals[t * g.m + v]);
    }
}

void Launcher::set_leaves(const int* keys, const double* vals, long long count)
{
    if (g.prec) pdl_launch(k_set_leaves<float>, blocks_dense(count), NTHREADS, 0, st, g, keys, vals, count);
    else pdl_launch(k_set_leaves<double>, blocks_dense(count), NTHREADS, 0, st, g, keys, vals, count);
    ++n;
}

// finest-level data (double, host layout [v][cell], in device memory or read
// from the host's) stored in q^n of the finest nodes, in the fields' type
template <int M, class T>
__global__ void k_store_finest(const __grid_constant__ Grid g, const double* src)
{
    pdl_enter();
    const long long N = g.N[g.L];
    GRID_STRIDE(id, N)
    {
        T q[M];
#pragma unroll
        for (int v = 0; v < M; ++v) q[v] = T(src[v * N + id]);
        store_row<M, T>(nd<T>(g, F_Q0, slot_of(g, g.L, id)), q);
    }
}

template <int D, int M>
static void store_finest_dm(Launcher& L, const double* src)
{
    MRLT_T_LAUNCH(L, blocks_dense(L.g.N[L.g.L]), (L.g, src), k_store_finest<M);
    ++L.n;
}
void Launcher::store_finest(const double* src) { MRLT_DM_DISPATCH(store_finest_dm, *this, src); }

// every cell of levels lb..L a node, in level and cell order from slot 1 on:
// the full tree of a new solver; the free stack holds the rest
__global__ void k_slots_full(Grid g, long long ntot)
{
    pdl_enter();
    long long first = 1;
    for (int l = g.lb; l <= g.L; ++l) {
        GRID_STRIDE(i, g.N[l]) g.slot[g.off[l] + i] = (int)(first + i);
        first += g.N[l];
    }
    const long long nfree = g.cap - 1 - ntot;
    GRID_STRIDE(k, nfree) g.fstack[k] = (int)(g.cap - 1 - k);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        g.ftop[0] = (int)nfree;
        g.ftop[1] = 0;
    }
}

void Launcher::slots_full(long long ntot)
{
    pdl_launch(k_slots_full, blocks_dense(ntot), NTHREADS, 0, st, g, ntot);
    ++n;
}

// Refinement flags of levels la..L-1, added into *out: after the closure of an
// adaptation at level la every flagged cell owns 2^d nodes of the new tree.
__global__ void k_count_ref(const __grid_constant__ Grid g, int la, int* out)
{
    MRLT_ENTER(g);
    const int c = __reduce_add_sync(0xffffffffu, refined_here(g, la));
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

void Launcher::count_refined(int la, int* out)
{
    cudaMemsetAsync(out, 0, sizeof(int), st);
    pdl_launch(k_count_ref, blocks_dense((g.off[g.L] - g.off[la]) / kStep), NTHREADS, 0, st, g, la, out);
    ++n;
}


// Compacting copy into node arrays of a new capacity: the nodes of level l
// (leaves, then internal nodes, in list order) take the consecutive slots
// from base[l] + 1; their fields and registers are copied from the old
// arrays (`from`), the slot map rewritten.  The free stack of the new arrays
// holds every slot above the nodes.
template <class T>
__global__ void k_renumber(Grid g, Grid from, LevelChunks base, long long used)
{
    pdl_enter();
    for (int l = g.lb; l <= g.L; ++l) {
        const long long N = g.N[l];
        const int nl = g.counts[l], ni = g.counts[LMAX + 1 + l];
        GRID_STRIDE(t, nl + ni)
        {
            const long long id = t < nl ? g.leaves[g.off[l] + t] : g.inner[g.off[l] + t - nl];
            if (id < 0 || id >= N) {
                atomicOr(g.err, ERR_INDEX);
                continue;
            }
            const int os = slot_of(from, l, id), ns = (int)(1 + base.base[l] + t);
            for (int f = 0; f < NFIELD; ++f) {
                const T* a = nd<T>(from, f, os);
                T* b = nd<T>(g, f, ns);
                for (int v = 0; v < g.m; ++v) b[v] = a[v];
            }
            if (g.rg) {
                const double* a = regs(from.rg, from, os);
                double* b = regs(g.rg, g, ns);
                for (int r = 0; r < g.nf * g.m; ++r) b[r] = a[r];
            }
            g.slot[g.off[l] + id] = ns;
        }
    }
    const long long nfree = g.cap - 1 - used;
    GRID_STRIDE(k, nfree) g.fstack[k] = (int)(g.cap - 1 - k);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        g.ftop[0] = (int)nfree;
        g.ftop[1] = 0;
    }
}

void Launcher::renumber(const Grid& from, const int* counts_host, long long used)
{
    LevelChunks base;
    base.lo = g.lb;
    base.hi = g.L;
    int acc = 0;
    for (int l = g.lb; l <= g.L; ++l) {
        base.base[l] = acc;
        acc += counts_host[l] + counts_host[LMAX + 1 + l];
    }
    base.base[g.L + 1] = acc;
    long long cnt = used > g.cap - 1 - used ? used : g.cap - 1 - used;
    if (g.prec) pdl_launch(k_renumber<float>, blocks_dense(cnt), NTHREADS, 0, st, g, from, base, used);
    else pdl_launch(k_renumber<double>, blocks_dense(cnt), NTHREADS, 0, st, g, from, base, used);
    stale = true;
    ++n;
}

void Launcher::scale_init()
{
    pdl_launch(k_scale_init, 1, 32, 0, st, g);
    ++n;
}

// the words of g.built that a captured piece used, after all its kernels
__global__ void k_piece_end(const __grid_constant__ Grid g, int stages)
{
    pdl_enter(); // each kernel of the piece waited for the one before it
    if (threadIdx.x == 0) g.built[0] = 0;
    for (int i = threadIdx.x; i < stages; i += blockDim.x) g.built[kFirstTick + i] = 0;
}

void Launcher::piece_begin()
{
    capturing = true;
    stale = false;
    published[0] = 0;
    stages = 0;
}

void Launcher::piece_end()
{
    if (published[0] || stages) {
        pdl_launch(k_piece_end, 1, NTHREADS, 0, st, g, stages);
        ++n;
    }
    capturing = false;
    stale = true;
}

void Launcher::set_dt(double dt)
{
    pdl_launch(k_set_dt, 1, 32, 0, st, g, dt);
    stale = true;
    ++n;
}

template <int D, int M>
static void scale_dm(Launcher& L)
{
    MRLT_T_LAUNCH(L, blocks_list(L.g, L.g.L), (L.g), k_scale<M);
    ++L.n;
}
void Launcher::scale() { MRLT_DM_DISPATCH(scale_dm, *this); }

template <int D, int M>
static void finite_dm(Launcher& L)
{
    MRLT_T_LAUNCH(L, blocks_list(L.g, L.g.L), (L.g), k_finite<M);
    ++L.n;
}
void Launcher::finite() { MRLT_DM_DISPATCH(finite_dm, *this); }
void Launcher::mass(int l, double* part)
{
    ++n;
    if (g.prec) k_mass<float><<<MASS_BLOCKS, NTHREADS, 0, st>>>(g, l, part);
    else k_mass<double><<<MASS_BLOCKS, NTHREADS, 0, st>>>(g, l, part);
}
template <int D, int M>
static void pack_dm(Launcher& L, int* keys, double* vals)
{
    MRLT_T_LAUNCH(L, blocks_list(L.g, L.g.L), (L.g, keys, vals), k_pack<M);
    ++L.n;
}
void Launcher::pack(int* keys, double* vals) { MRLT_DM_DISPATCH(pack_dm, *this, keys, vals); }
void Launcher::uniform(double* T, uint8_t* us)
{
    for (int l = g.L; l >= g.lb; --l, ++n) {
        const int nb = blocks_dense(g.N[l]);
        if (g.prec) {
            if (g.d == 1) k_uni_up<1, float><<<nb, NTHREADS, 0, st>>>(g, l, T, us);
            else if (g.d == 2) k_uni_up<2, float><<<nb, NTHREADS, 0, st>>>(g, l, T, us);
            else k_uni_up<3, float><<<nb, NTHREADS, 0, st>>>(g, l, T, us);
        } else {
            if (g.d == 1) k_uni_up<1, double><<<nb, NTHREADS, 0, st>>>(g, l, T, us);
            else if (g.d == 2) k_uni_up<2, double><<<nb, NTHREADS, 0, st>>>(g, l, T, us);
            else k_uni_up<3, double><<<nb, NTHREADS, 0, st>>>(g, l, T, us);
        }
    }
    for (int l = g.lb + 1; l <= g.L; ++l, ++n) {
        if (g.d == 1) k_uni_down<1><<<blocks_dense(g.N[l]), NTHREADS, 0, st>>>(g, l, T, us);
        else if (g.d == 2) k_uni_down<2><<<blocks_dense(g.N[l]), NTHREADS, 0, st>>>(g, l, T, us);
        else k_uni_down<3><<<blocks_dense(g.N[l]), NTHREADS, 0, st>>>(g, l, T, us);
    }
}

} // namespace mrlt
