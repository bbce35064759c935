// mrlt_tree_dev.cuh -- device bodies of the tree work of the MRLT library:
// projections and tree refreshing (Eqs. 3, 14-22; Algs. 3, 4, 6, 8, 9), the
// multiresolution adaptation (details Eq. 5, thresholding Alg. 2, graded
// closure Alg. 1), list compaction, conservative flux registers and the
// per-macro-step reductions.  Each body distributes its work over the
// launch's grid (grid-stride loops over blockIdx / gridDim), so the same body
// serves a kernel of its own (mrlt_tree.cu) and a phase of the persistent
// macro-step kernel (mrlt_macro.cuh).
#pragma once
#include "mrlt_impl.cuh"

namespace mrlt {

enum ProjMode { PM_Q0 = 0, PM_BEG, PM_Q1, PM_Q2, PM_REF2, PM_PRJ2, PM_REF3, PM_PRJ3, PM_MID };

#define MRLT_GRID_STRIDE(i, n) \
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += (long long)gridDim.x * blockDim.x)

// ------------------------------------------------------------ lists and rows
// f(l, id, t) for every entry of the leaf lists (KIND 0) or internal-node
// lists (KIND 1) of levels lo..hi, level by level as one range t = 0, 1, ...
// over the launch's threads: one pass whatever the number of levels, where a
// loop over the levels costs a chain of dependent loads for each.  Every thread
// of the CTA takes part.
template <int KIND, class F>
__device__ __forceinline__ void for_list(const Grid& g, int lo, int hi, F f)
{
    const int* list = KIND ? g.inner : g.leaves;
    if (lo == hi) { // the first entry and the count in one trip (the list has room for every cell)
        const long long N = g.N[lo], t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        const int* mine = list + g.off[lo];
        int e = t0 < N ? mine[t0] : -1;
        const int total = g.counts[KIND * (LMAX + 1) + lo];
        for (long long t = t0; t < total; t += (long long)gridDim.x * blockDim.x) {
            if (t != t0) e = mine[t];
            if (e < 0 || e >= N) atomicOr(g.err, ERR_INDEX);
            else f(lo, (long long)e, t);
        }
        return;
    }
    __shared__ int base[LMAX + 2]; // level lo + k starts at base[k]
    __syncthreads();               // base may hold an earlier call's
    if (threadIdx.x < 32) {
        const int k = threadIdx.x, n = hi - lo + 1;
        int inc = k < n ? g.counts[KIND * (LMAX + 1) + lo + k] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, inc, o);
            if (k >= o) inc += x;
        }
        if (k < n) base[k + 1] = inc;
        if (k == 0) base[0] = 0;
    }
    __syncthreads();
    const int total = base[hi - lo + 1];
    MRLT_GRID_STRIDE(t, total)
    {
        int k = hi - lo; // most entries are on the finest levels
        while (t < base[k]) --k;
        const long long id = list[g.off[lo + k] + t - base[k]];
        if (id < 0 || id >= g.N[lo + k]) {
            atomicOr(g.err, ERR_INDEX);
            continue;
        }
        f(lo + k, id, t);
    }
}

// for_list for a kernel's whole body, with the tree's share of an entry's work,
// lookup(l, id), apart from the use(entry) of its result: the first entries are
// looked up before the wait for the predecessor's values where the tree is
// visible by then (waited: what tree_enter returned).
template <int KIND, class Lookup, class Use>
__device__ __forceinline__ void kernel_list(const Grid& g, int lo, int hi, bool waited, Lookup lookup, Use use)
{
    bool stop = waited && halted(g);
    const auto enter = [&]() {
        if (waited) return;
        pdl_enter();
        waited = true;
        stop = halted(g);
    };
    for_list<KIND>(g, lo, hi, [&](int l, long long id, long long) {
        auto e = lookup(l, id);
        enter();
        if (!stop) use(e);
    });
    enter(); // a thread without entries: the kernels after this one rely on its wait
}

// a node's row of M values: 16-byte accesses where rows are whole vectors
template <int M, class T>
__device__ __forceinline__ void load_row(const T* p, T (&r)[M])
{
    if constexpr (M * sizeof(T) % 16 == 0) {
        constexpr int E = 16 / sizeof(T);
#pragma unroll
        for (int k = 0; k < M / E; ++k) {
            const int4 x = reinterpret_cast<const int4*>(p)[k];
            memcpy(&r[k * E], &x, 16);
        }
    } else {
#pragma unroll
        for (int v = 0; v < M; ++v) r[v] = p[v];
    }
}
template <int M, class T>
__device__ __forceinline__ void store_row(T* p, const T (&r)[M])
{
    if constexpr (M * sizeof(T) % 16 == 0) {
        constexpr int E = 16 / sizeof(T);
#pragma unroll
        for (int k = 0; k < M / E; ++k) {
            int4 x;
            memcpy(&x, &r[k * E], 16);
            reinterpret_cast<int4*>(p)[k] = x;
        }
    } else {
#pragma unroll
        for (int v = 0; v < M; ++v) p[v] = r[v];
    }
}

// T: storage type of the fields (double, or float in the mixed mode); the
// arithmetic of a body is in T except where it says otherwise
template <int M, class T>
__device__ __forceinline__ void dev_leaf_copy(const Grid& g, int lo, int hi, int from, int to)
{
    for_list<0>(g, lo, hi, [&](int l, long long id, long long) {
        const int sl = slot_of(g, l, id);
        T r[M];
        load_row<M, T>(nd<T>(g, from, sl), r);
        store_row<M, T>(nd<T>(g, to, sl), r);
    });
}

// ------------------------------------------------------------ projections
// Every internal node of level l combines its 2^d children (Eq. 3 mean):
//  PM_Q0 / PM_Q1 / PM_Q2: plain projection of that field (Alg. 3; GTS stages)
//  PM_BEG: q^n as an iteration begins, reading the end value of leaf children
//           (the q^n that the leaf copy gives them in the same launch)
//  PM_REF2: Alg. 8 -- XH = mean q* (Eq. 17), q* = 2 XH - q^n (Eq. 18)
//  PM_PRJ2: Alg. 4 -- q* = mean(leaf: Eq. 14 value, internal: Eq. 15 value)
//  PM_REF3: Alg. 9 -- N1 = mean q**, N3 by Eq. 20, q** by Eq. 21
//  PM_PRJ3: Alg. 6 -- q** = mean(children at t^n + dt_{l+1}), end value
//           2 q** - q^n (Eq. 16 with the theta values implied by q**)
//  PM_MID:  Alg. 3 / Sec. 4.3 refresh of the mid-step level lmin-1, from its
//           children's q^n, read likewise
// one internal node (l, id): the projection of the given mode.  Bound by its
// dependent trips (list, child slots, rows), so the rows of all children are
// loaded before any is used; a loop over the variables that stored each before
// loading the next took 8.8 us per launch over the opening of the 2D Euler
// L = 10 solve on a GB300 (14 k nodes on level 9), this takes 6.0 us.  The
// roundings are written out: which multiply-adds are fused must not depend on
// what else the compiler finds to share.
// What a projection looks up in the tree: the node's slot, its children's
// slots, and which of them are leaves.
template <int D>
struct NodeRefs {
    int sl, csl[1 << D];
    unsigned leaf;
};

template <int D>
__device__ __forceinline__ NodeRefs<D> lookup_node(const Grid& g, int l, long long id)
{
    NodeRefs<D> r;
    int c[3];
    cell_xyz(g, l, id, c);
    r.leaf = 0;
#pragma unroll
    for (int k = 0; k < (1 << D); ++k) {
        const long long ch = cell_id(g, l + 1, 2 * c[0] + (k & 1), D > 1 ? 2 * c[1] + ((k >> 1) & 1) : 0,
                                     D > 2 ? 2 * c[2] + ((k >> 2) & 1) : 0);
        r.leaf |= (status(g, l + 1, ch) == 1 ? 1u : 0u) << k;
        r.csl[k] = slot_of(g, l + 1, ch);
    }
    r.sl = slot_of(g, l, id);
    return r;
}

template <int D, int M, class T>
__device__ __forceinline__ void project_node(const Grid& g, const NodeRefs<D>& n, int mode)
{
    constexpr int NCH = 1 << D;
    const int sl = n.sl;
    const int child = mode == PM_Q1 || mode == PM_REF2   ? F_Q1
                      : mode == PM_Q2 || mode == PM_REF3 ? F_Q2
                      : mode == PM_PRJ3                  ? F_QE
                                                         : F_Q0;
    const int leaf = mode == PM_BEG || mode == PM_MID ? F_QE : child; // a leaf child's q^n is its end value
    T w[NCH][M], acc[M], a0[M], a1[M];
    if (mode == PM_PRJ2) {
        T x[NCH][M];
#pragma unroll
        for (int k = 0; k < NCH; ++k) {
            load_row<M, T>(nd<T>(g, F_Q0, n.csl[k]), w[k]);
            load_row<M, T>(nd<T>(g, !(n.leaf >> k & 1) ? F_Q1 : (g.rk == 2 ? F_QE : F_Q2), n.csl[k]), x[k]);
        }
#pragma unroll
        for (int k = 0; k < NCH; ++k)
#pragma unroll
            for (int v = 0; v < M; ++v) {
                if ((n.leaf >> k & 1) && g.rk != 2) w[k][v] = fma(T(4), x[k][v], -mul_rn(T(3), w[k][v]));
                else w[k][v] = T(2) * x[k][v] - w[k][v];
            }
    } else {
#pragma unroll
        for (int k = 0; k < NCH; ++k) load_row<M, T>(nd<T>(g, n.leaf >> k & 1 ? leaf : child, n.csl[k]), w[k]);
        if (mode >= PM_REF2) {
            load_row<M, T>(nd<T>(g, F_Q0, sl), a0);
            if (mode == PM_REF3 || mode == PM_MID) load_row<M, T>(nd<T>(g, F_Q1, sl), a1);
        }
    }
#pragma unroll
    for (int v = 0; v < M; ++v) {
        acc[v] = T(0);
#pragma unroll
        for (int k = 0; k < NCH; ++k) acc[v] += w[k][v];
        acc[v] = acc[v] * T(1.0 / NCH); // the mean
    }
    switch (mode) {
    case PM_Q0: case PM_BEG: store_row<M, T>(nd<T>(g, F_Q0, sl), acc); break;
    case PM_Q1: case PM_PRJ2: store_row<M, T>(nd<T>(g, F_Q1, sl), acc); break;
    case PM_Q2: store_row<M, T>(nd<T>(g, F_Q2, sl), acc); break;
    case PM_REF2:
        store_row<M, T>(nd<T>(g, F_XH, sl), acc);
#pragma unroll
        for (int v = 0; v < M; ++v) acc[v] = T(2) * acc[v] - a0[v];
        store_row<M, T>(nd<T>(g, F_Q1, sl), acc);
        break;
    case PM_REF3: {
        T r[M];
        store_row<M, T>(nd<T>(g, F_N1, sl), acc);
#pragma unroll
        for (int v = 0; v < M; ++v) r[v] = fma(T(9), acc[v], fma(T(-6.5), a0[v], -mul_rn(T(1.5), a1[v])));
        store_row<M, T>(nd<T>(g, F_N3, sl), r);
#pragma unroll
        for (int v = 0; v < M; ++v) r[v] = fma(T(8), acc[v], fma(T(-5.5), a0[v], -mul_rn(T(1.5), a1[v])));
        store_row<M, T>(nd<T>(g, F_Q2, sl), r);
        break;
    }
    case PM_PRJ3:
        store_row<M, T>(nd<T>(g, F_Q2, sl), acc);
#pragma unroll
        for (int v = 0; v < M; ++v) acc[v] = T(2) * acc[v] - a0[v];
        store_row<M, T>(nd<T>(g, F_QE, sl), acc);
        break;
    default: { // PM_MID
        T r[M];
        if (g.rk == 2) {
            store_row<M, T>(nd<T>(g, F_NH, sl), acc);
#pragma unroll
            for (int v = 0; v < M; ++v) r[v] = T(-2) * a0[v] - a1[v] + T(4) * acc[v];
            store_row<M, T>(nd<T>(g, F_QE, sl), r);
        } else {
            T n1[M];
            store_row<M, T>(nd<T>(g, F_Q2, sl), acc);
#pragma unroll
            for (int v = 0; v < M; ++v) {
                r[v] = T(2) * acc[v] - a0[v];
                n1[v] = fma(T(1.5), a1[v], fma(T(5.5), a0[v], acc[v])) * T(0.125);
            }
            store_row<M, T>(nd<T>(g, F_QE, sl), r);
            store_row<M, T>(nd<T>(g, F_N1, sl), n1);
#pragma unroll
            for (int v = 0; v < M; ++v)
                r[v] = fma(T(9), n1[v], fma(T(-6.5), a0[v], -mul_rn(T(1.5), a1[v])));
            store_row<M, T>(nd<T>(g, F_N3, sl), r);
        }
    }
    }
}

// An up-sweep of one mode over levels hi..lo in one launch.  Each step of a CTA
// takes `tops` internal nodes of level lo and projects their internal
// descendants bottom-up, level by level, with a CTA barrier between levels: a
// node's projection reads only its own children, which lie in the same subtree.
// Thread t of a step owns descendant t % sub of top node t / sub on each level
// (sub = 2^{d (u - lo)} on level u), so 2^{d (hi - lo)} <= blockDim.x, and at
// most 6 / d levels above lo (kUpDepth).  The nodes of all levels are looked up
// together (one trip for the list, one for statuses, one for slots), so a level
// costs the trip of its rows.
template <int D> constexpr int kUpDepth = 6 / D;

template <int D>
struct UpRefs {
    NodeRefs<D> n[kUpDepth<D> + 1];
    unsigned have; // bit s: this thread projects a node of level lo + s
};

template <int D>
__device__ __forceinline__ UpRefs<D> up_lookup(const Grid& g, int hi, int lo, int step)
{
    UpRefs<D> r;
    r.have = 0;
    const int depth = hi - lo, tops = blockDim.x >> (D * depth), t = threadIdx.x;
    const int* list = g.inner + g.off[lo];
    const long long N = g.N[lo];
    const int cnt = g.counts[LMAX + 1 + lo];
#pragma unroll
    for (int s = 0; s <= kUpDepth<D>; ++s) {
        if (s > depth) continue;
        const int sub = 1 << (D * s);
        const long long ti = (long long)step * tops + t / sub;
        if (t >= tops * sub || ti >= N) continue;
        const long long top = list[ti]; // with the count: the list has room for every cell
        if (ti >= cnt) continue;
        if (top < 0 || top >= N) {
            atomicOr(g.err, ERR_INDEX);
            continue;
        }
        int tc[3];
        cell_xyz(g, lo, top, tc);
        const int q = t % sub, msk = (1 << s) - 1, u = lo + s;
        const long long id = cell_id(g, u, (tc[0] << s) + (q & msk), D > 1 ? (tc[1] << s) + ((q >> s) & msk) : 0,
                                     D > 2 ? (tc[2] << s) + (q >> (2 * s)) : 0);
        if (s && status(g, u, id) != 2) continue;
        r.have |= 1u << s;
        r.n[s] = lookup_node<D>(g, u, id);
    }
    return r;
}

// the projections of one step: level lo with mode topmode, the others with mode
template <int D, int M, class T>
__device__ __forceinline__ void up_project(const Grid& g, const UpRefs<D>& r, int depth, int mode, int topmode)
{
#pragma unroll
    for (int s = kUpDepth<D>; s >= 0; --s) {
        if (s > depth) continue;
        if (r.have >> s & 1) project_node<D, M, T>(g, r.n[s], s ? mode : topmode);
        if (s) __syncthreads();
    }
}

__device__ __forceinline__ int up_steps(const Grid& g, int hi, int lo)
{
    const int tops = blockDim.x >> (g.d * (hi - lo));
    return (g.counts[LMAX + 1 + lo] + tops - 1) / tops;
}

// one level (the persistent macro-step kernel's phases)
template <int D, int M, class T>
__device__ __forceinline__ void dev_project(const Grid& g, int l, int mode)
{
    for_list<1>(g, l, l, [&](int, long long id, long long) { project_node<D, M, T>(g, lookup_node<D>(g, l, id), mode); });
}

// ------------------------------------------------------------ adaptation
__device__ __forceinline__ double eps_level(const Grid& g, int l)
{
    return g.eps_mode == 1 ? ldexp(g.eps, g.d * (l - g.L)) : g.eps;
}

// Predictions (Eq. 4) of the 2^D children of a node from the 3^D block b of
// values around it (x fastest), direction by direction: a row (l, m, r) gives
// the two children m -+ (r - l) / 8.  3 operations per row and direction
// instead of a weighted sum over the block for each child: 15 against 36
// per variable in 2D, 57 against 216 in 3D, and FP64 operations (2 per clock
// and SM) are what the details cost.  Child k has offset bits (x, y, z).
template <int D>
__device__ __forceinline__ void predict_block(const double* b, double* out)
{
    auto split = [](double l, double m, double r, double& lo, double& hi) {
        const double d = r - l;
        lo = fma(-0.125, d, m);
        hi = fma(0.125, d, m);
    };
    constexpr int NY = D > 1 ? 3 : 1, NZ = D > 2 ? 3 : 1;
    double x[NY * NZ][2], y[NZ][4];
#pragma unroll
    for (int r = 0; r < NY * NZ; ++r) split(b[3 * r], b[3 * r + 1], b[3 * r + 2], x[r][0], x[r][1]);
    if constexpr (D == 1) {
        out[0] = x[0][0];
        out[1] = x[0][1];
    } else {
#pragma unroll
        for (int z = 0; z < NZ; ++z)
#pragma unroll
            for (int a = 0; a < 2; ++a)
                split(x[3 * z][a], x[3 * z + 1][a], x[3 * z + 2][a], y[z][a], y[z][2 + a]);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            if constexpr (D == 2) out[a] = y[0][a];
            else split(y[0][a], y[1][a], y[2][a], out[a], out[4 + a]);
        }
    }
}

// detail norm (Eq. 5) of every internal node of levels lo..hi (< L): max over
// children and variables of |q_child - prediction| / s_v; flags significance
// (> eps_{l+1}) and the scale-safety bound (> 8 eps_{l+1}).  The predictions
// and the test are FP64 whatever the storage type T.  The maximum over the
// children is taken on the bit patterns and before the division, which keeps
// the order (one division per variable, and it rounds monotonically).
// Measured on a GB300, per launch: 30 us with weighted sums against 13.8 us in
// the opening of the 2D Euler L = 10 solve (all depths of remesh), 80 against
// 11 us at full remeshes of 2D L = 9, 234 against 68 us in the 3D blast at L = 7.
template <int D>
struct DetailRefs {
    static constexpr int NB = D == 1 ? 3 : (D == 2 ? 9 : 27);
    int l, sl[NB], csl[1 << D];
    unsigned minus; // block cells that enter negated (an odd count of odd mirrors)
    long long id;
};

template <int D>
__device__ __forceinline__ DetailRefs<D> lookup_detail(const Grid& g, int l, long long id)
{
    DetailRefs<D> r;
    r.l = l;
    r.id = id;
    r.minus = 0;
    int c[3];
    cell_xyz(g, l, id, c);
    int q[3][3], neg[3][3]; // in-box coordinate and mirror parity of the neighbours per direction
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            neg[k][j] = 0;
            q[k][j] = k < D ? wrap_or_mirror(g, l, k, c[k] + j - 1, neg[k][j]) : 0;
        }
    bool missing = false;
#pragma unroll
    for (int b = 0; b < DetailRefs<D>::NB; ++b) {
        const int i = b % 3, j = D > 1 ? b / 3 % 3 : 0, k = D > 2 ? b / 9 : 0;
        const long long bid = cell_id(g, l, q[0][i], q[1][j], q[2][k]);
        missing = missing || status(g, l, bid) == 0;
        r.sl[b] = slot_of(g, l, bid);
        r.minus |= (unsigned)(neg[0][i] ^ (D > 1 ? neg[1][j] : 0) ^ (D > 2 ? neg[2][k] : 0)) << b;
    }
    if (missing && g.eps > 0.0) atomicOr(g.err, ERR_SOURCE);
#pragma unroll
    for (int k = 0; k < (1 << D); ++k)
        r.csl[k] = slot_of(g, l + 1, cell_id(g, l + 1, 2 * c[0] + (k & 1), D > 1 ? 2 * c[1] + ((k >> 1) & 1) : 0,
                                             D > 2 ? 2 * c[2] + ((k >> 2) & 1) : 0));
    return r;
}

template <int D, int M, class T>
__device__ __forceinline__ void detail_node(const Grid& g, const DetailRefs<D>& e)
{
    constexpr int NB = DetailRefs<D>::NB, NCH = 1 << D;
    uint8_t fl = 0;
    if (g.eps <= 0.0) {
        fl = FL_SIG;
    } else {
        const double el = eps_level(g, e.l + 1);
        double nrm = 0.0;
#pragma unroll(D > 2 ? 1 : M)
        for (int v = 0; v < M; ++v) {
            const double sc = __longlong_as_double((long long)g.scale_bits[v]);
            double b[NB], p[NCH];
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                b[k] = double(nd<T>(g, F_Q0, e.sl[k])[v]);
                if (e.minus >> k & 1) b[k] = -b[k];
            }
            predict_block<D>(b, p);
            unsigned long long mx = 0;
#pragma unroll
            for (int k = 0; k < NCH; ++k) {
                const double d = double(nd<T>(g, F_Q0, e.csl[k])[v]) - p[k];
                const unsigned long long a = abs_bits(d);
                if (a > mx && a <= 0x7ff0000000000000ull << 1) mx = a; // a NaN is no detail
            }
            nrm = fmax(nrm, __longlong_as_double((long long)(mx >> 1)) / sc);
        }
        if (fabs(nrm - el) <= 1e-10 * el || fabs(nrm - 8.0 * el) <= 8e-10 * el) atomicAdd(g.near, 1ull);
        if (nrm > el) fl |= FL_SIG;
        if (nrm > 8.0 * el) fl |= FL_BIG;
    }
    g.flag[g.off[e.l] + e.id] |= fl;
}

template <int D, int M, class T>
__device__ __forceinline__ void dev_detail(const Grid& g, int lo, int hi)
{
    for_list<1>(g, lo, hi, [&](int l, long long id, long long) { detail_node<D, M, T>(g, lookup_detail<D>(g, l, id)); });
}

template <int D>
__device__ __forceinline__ bool nb3(const Grid& g, int l, const int c[3], int dx, int dy, int dz, long long* id)
{
    int q[3] = {0, 0, 0};
    if (!in_box(g, l, 0, c[0] + dx, &q[0])) return false;
    if (D > 1 && !in_box(g, l, 1, c[1] + dy, &q[1])) return false;
    if (D > 2 && !in_box(g, l, 2, c[2] + dz, &q[2])) return false;
    *id = cell_id(g, l, q[0], q[1], q[2]);
    return true;
}

#define MRLT_FOR3(D, dx, dy, dz)                                  \
    for (int dz = (D > 2 ? -1 : 0); dz <= (D > 2 ? 1 : 0); ++dz) \
        for (int dy = (D > 1 ? -1 : 0); dy <= (D > 1 ? 1 : 0); ++dy) \
            for (int dx = -1; dx <= 1; ++dx)

// ------------------------------------------------------------ 16 cells at a time
// The passes over the dense byte maps (status, flags) take a step of 16
// consecutive cells per thread with 16-byte loads, and keep a bit per cell.
// Almost every step holds nothing and ends there; with one byte per thread the
// passes were bound by the number of their loads.  On a GB300, marking and
// applying took 98 + 80 us at 3D L = 8 (330 k leaves) and 9.9 + 5.5 us at 2D
// L = 10 (5 k leaves), and take 16 + 28 and 4.5 + 2.4 us.  A step lies in one
// row of cells where a row has 16 (levels >= 4, hence the line); the few cells
// below go one by one.
constexpr int kStep = 16;          // cells per step
constexpr int kStepLevel = 4;      // rows hold whole steps from this level on

// bit j: byte j of the 16 has bit `bit` set (a status byte is 1 for a leaf and
// 2 for an internal node, so bit 0 and bit 1 select the two)
__device__ __forceinline__ unsigned byte_mask(const uint4& s, int bit)
{
    auto four = [&](unsigned w) { return (((w >> bit) & 0x01010101u) * 0x10204080u) >> 28; };
    return four(s.x) | four(s.y) << 4 | four(s.z) << 8 | four(s.w) << 12;
}

// bytes j = 1 where bit j of the low four bits of m is set
__device__ __forceinline__ unsigned mask_bytes(unsigned m)
{
    return (m & 0xfu) * 0x00204081u & 0x01010101u;
}

// bit j of 8 to bits 2j, 2j + 1 of 16 (the children's row of a row of parents)
__device__ __forceinline__ unsigned double_bits(unsigned m)
{
    m = (m | m << 4) & 0x0f0fu;
    m = (m | m << 2) & 0x3333u;
    m = (m | m << 1) & 0x5555u;
    return m | m << 1;
}

// bits 2j, 2j + 1 of 32 combined (or) to bit j of 16
__device__ __forceinline__ unsigned halve_bits(unsigned m)
{
    m = (m | m >> 1) & 0x55555555u;
    m = (m | m >> 1) & 0x33333333u;
    m = (m | m >> 2) & 0x0f0f0f0fu;
    m = (m | m >> 4) & 0x00ff00ffu;
    return (m | m >> 8) & 0xffffu;
}

// byte-bit `bit` of the 16 cells from x0 (bits 1..16) and of the cell to
// either side of them (bits 0 and 17) in row (y, z) of a map of level l;
// past a wall: 0
__device__ __forceinline__ unsigned row_bits(const Grid& g, const uint8_t* map, int l, int x0, int y, int z, int bit)
{
    const int n = g.n[l];
    const uint8_t* r = map + cell_id(g, l, 0, y, z);
    unsigned m = byte_mask(*reinterpret_cast<const uint4*>(r + x0), bit) << 1;
    const bool wrap = g.bc[0] == 0;
    if (x0 > 0 || wrap) m |= (unsigned)(r[x0 > 0 ? x0 - 1 : n - 1] >> bit & 1);
    if (x0 + kStep < n || wrap) m |= (unsigned)(r[x0 + kStep < n ? x0 + kStep : 0] >> bit & 1) << 17;
    return m;
}

// byte-bit `bit` of the parents (level l - 1) of cells i..i+15, for each cell
__device__ __forceinline__ unsigned parent_bits(const Grid& g, const uint8_t* map, int l, const int c[3], int bit)
{
    const uint2 p = *reinterpret_cast<const uint2*>(map + cell_id(g, l - 1, c[0] >> 1, c[1] >> 1, c[2] >> 1));
    return double_bits(byte_mask(make_uint4(p.x, p.y, 0, 0), bit));
}

// Desired refinement (space safety: a significant node in the 3^d
// neighbourhood; scale safety: a parent, of level >= la, flagged by it; eps =
// 0 refines all) of one cell, and of the 16 cells from c (bit per cell)
template <int D>
__device__ __forceinline__ bool desired(const Grid& g, int l, const int c[3], int la)
{
    if (g.eps <= 0.0) return true;
    const uint8_t* fl = g.flag + g.off[l];
    bool want = false;
    MRLT_FOR3(D, dx, dy, dz)
    {
        long long j;
        if (nb3<D>(g, l, c, dx, dy, dz, &j) && (fl[j] & FL_SIG)) want = true;
    }
    if (!want && l - 1 >= la) {
        const long long p = cell_id(g, l - 1, c[0] >> 1, c[1] >> 1, c[2] >> 1);
        want = g.flag[g.off[l - 1] + p] & FL_BIG;
    }
    return want;
}

template <int D>
__device__ __forceinline__ unsigned desired16(const Grid& g, int l, const int c[3], int la)
{
    if (g.eps <= 0.0) return 0xffffu;
    unsigned m = 0;
#pragma unroll
    for (int dz = (D > 2 ? -1 : 0); dz <= (D > 2 ? 1 : 0); ++dz)
#pragma unroll
        for (int dy = (D > 1 ? -1 : 0); dy <= (D > 1 ? 1 : 0); ++dy) {
            int y = 0, z = 0;
            if (D > 1 && !in_box(g, l, 1, c[1] + dy, &y)) continue;
            if (D > 2 && !in_box(g, l, 2, c[2] + dz, &z)) continue;
            m |= row_bits(g, g.flag + g.off[l], l, c[0], y, z, 0); // FL_SIG
        }
    unsigned want = (m | m >> 1 | m >> 2) & 0xffffu;
    if (l - 1 >= la) want |= parent_bits(g, g.flag + g.off[l - 1], l, c, 1); // FL_BIG
    return want;
}
static_assert(FL_SIG == 1 && FL_BIG == 2 && FL_REF == 16, "flag bits read by position");

// Admissible refinements: a node (l, i) may be refined if every node of the
// frozen level la-1 its grading chain requires is refined already.  Unrolling
// the rule "refining (m, j) needs (m-1, floor(j/2) + delta), |delta| <= 1"
// from level l down to la-1 gives, per direction, the interval [a, b] obtained
// by a -> floor(a/2) - 1, b -> floor(b/2) + 1 (l - la + 1 times), wrapped when
// periodic and clipped at walls.  At a full adaptation (la = min level)
// everything is admissible.
__device__ __forceinline__ void chain_interval(int l, int la, int& a, int& b)
{
    for (int m = l; m >= la; --m) {
        a = (a >> 1) - 1; // arithmetic shift: floor for negatives
        b = (b >> 1) + 1;
    }
}

template <int D>
__device__ __forceinline__ bool allowed(const Grid& g, int l, const int c[3], int la)
{
    if (la <= g.lb) return true;
    const int pl = la - 1, n = g.n[pl];
    int lo3[3] = {0, 0, 0}, cnt3[3] = {1, 1, 1};
    for (int k = 0; k < D; ++k) {
        int a = c[k], b = c[k];
        chain_interval(l, la, a, b);
        if (g.bc[k] == 0) {
            lo3[k] = a;
            cnt3[k] = min(b - a + 1, n);
        } else {
            lo3[k] = max(a, 0);
            cnt3[k] = min(b, n - 1) - lo3[k] + 1;
        }
    }
    bool ok = true;
    for (int tz = 0; tz < cnt3[2] && ok; ++tz)
        for (int ty = 0; ty < cnt3[1] && ok; ++ty)
            for (int tx = 0; tx < cnt3[0] && ok; ++tx) {
                int q[3] = {lo3[0] + tx, lo3[1] + ty, lo3[2] + tz};
                for (int k = 0; k < D; ++k)
                    if (g.bc[k] == 0) q[k] &= n - 1; // periodic wrap (n = 2^l)
                ok = status(g, pl, cell_id(g, pl, q[0], q[1], q[2])) == 2;
            }
    return ok;
}

// The same for those of the 16 cells from c that `want` selects: they share
// the intervals across the rows, so the statuses of the (at most 10) columns
// that any of them needs are combined over the rows first.
template <int D>
__device__ __forceinline__ unsigned allowed16(const Grid& g, int l, const int c[3], int la, unsigned want)
{
    if (la <= g.lb) return want;
    const int pl = la - 1;
    int a0 = c[0], b0 = c[0] + kStep - 1, a1 = c[1], b1 = c[1], a2 = c[2], b2 = c[2];
    chain_interval(l, la, a0, b0);
    if (D > 1) chain_interval(l, la, a1, b1);
    if (D > 2) chain_interval(l, la, a2, b2);
    unsigned cols = ~0u; // bit k: every row of column a0 + k is refined
    for (int z = a2; z <= b2; ++z) {
        int qz = 0;
        if (D > 2 && !in_box(g, pl, 2, z, &qz)) continue; // clipped at walls
#pragma unroll
        for (int j = 0; j < (D > 1 ? 5 : 1); ++j) { // at most 5 rows; their loads in one trip
            int qy = 0;
            if (D > 1 && (a1 + j > b1 || !in_box(g, pl, 1, a1 + j, &qy))) continue;
            const uint8_t* row = g.st + g.off[pl] + cell_id(g, pl, 0, qy, qz);
            uint8_t s[10];
#pragma unroll
            for (int k = 0; k < 10; ++k) {
                int qx = 0;
                s[k] = a0 + k <= b0 && in_box(g, pl, 0, a0 + k, &qx) ? row[qx] : 2;
            }
#pragma unroll
            for (int k = 0; k < 10; ++k)
                if (s[k] != 2) cols &= ~(1u << k);
        }
    }
    if (cols == ~0u) return want;
    unsigned ok = 0;
    for (unsigned m = want; m; m &= m - 1) {
        const int j = __ffs(m) - 1;
        int a = c[0] + j, b = a;
        chain_interval(l, la, a, b);
        const unsigned need = ((2u << (b - a)) - 1u) << (a - a0);
        if ((cols & need) == need) ok |= 1u << j;
    }
    return ok;
}

// FL_REF set on the cells of mask m of the 16 at f
__device__ __forceinline__ void refine16(uint8_t* f, unsigned m)
{
    uint4* p = reinterpret_cast<uint4*>(f);
    uint4 v = *p;
    v.x |= mask_bytes(m) * FL_REF;
    v.y |= mask_bytes(m >> 4) * FL_REF;
    v.z |= mask_bytes(m >> 8) * FL_REF;
    v.w |= mask_bytes(m >> 12) * FL_REF;
    *p = v;
}

// Refinements of levels lo..hi: desired and admissible.  A step's stores keep
// the detail bits that other threads read.  Returns how many cells this thread
// flagged.
template <int D>
__device__ __forceinline__ int dev_mark(const Grid& g, int lo, int hi, int la)
{
    int count = 0;
    for (int l = lo; l <= hi; ++l) {
        uint8_t* fl = g.flag + g.off[l];
        int c[3];
        if (l < kStepLevel) {
            MRLT_GRID_STRIDE(id, g.N[l])
            {
                cell_xyz(g, l, id, c);
                if (desired<D>(g, l, c, la) && allowed<D>(g, l, c, la)) {
                    fl[id] |= FL_REF;
                    ++count;
                }
            }
        } else {
            MRLT_GRID_STRIDE(s, g.N[l] / kStep)
            {
                cell_xyz(g, l, s * kStep, c);
                unsigned m = desired16<D>(g, l, c, la);
                if (m) m = allowed16<D>(g, l, c, la, m);
                if (m) refine16(fl + s * kStep, m);
                count += __popc(m);
            }
        }
    }
    return count;
}

// grading closure, one level: refining (l, i) refines (l-1, floor(i/2) + delta)
// for |delta|_inf <= 1 -- gathered at the coarse node.  Returns how many cells
// this thread flagged.
template <int D>
__device__ __forceinline__ int dev_close(const Grid& g, int l)
{
    int count = 0;
    const int pl = l - 1;
    uint8_t* fp = g.flag + g.off[pl];
    const uint8_t* fc = g.flag + g.off[l];
    if (pl < kStepLevel) {
        MRLT_GRID_STRIDE(pid, g.N[pl])
        {
            if (fp[pid] & FL_REF) continue;
            int c[3];
            cell_xyz(g, pl, pid, c);
            bool hit = false;
            MRLT_FOR3(D, dx, dy, dz)
            {
                long long j;
                if (!nb3<D>(g, pl, c, -dx, -dy, -dz, &j)) continue;
                int q[3];
                cell_xyz(g, pl, j, q);
                for (int k = 0; k < (1 << D); ++k) {
                    const long long cid = cell_id(g, l, 2 * q[0] + (k & 1), D > 1 ? 2 * q[1] + ((k >> 1) & 1) : 0,
                                                  D > 2 ? 2 * q[2] + ((k >> 2) & 1) : 0);
                    if (fc[cid] & FL_REF) hit = true;
                }
            }
            if (hit) {
                fp[pid] |= FL_REF;
                ++count;
            }
        }
        return count;
    }
    MRLT_GRID_STRIDE(s, g.N[pl] / kStep)
    {
        int c[3];
        cell_xyz(g, pl, s * kStep, c);
        const unsigned own = byte_mask(*reinterpret_cast<const uint4*>(fp + s * kStep), 4);
        const bool wrap = g.bc[0] == 0;
        const int n = g.n[l], x0 = 2 * c[0]; // first child
        unsigned m = 0; // parents x0/2 - 1 (bit 0) .. x0/2 + 16 (bit 17) with a refined child in the rows
#pragma unroll
        for (int dz = (D > 2 ? -1 : 0); dz <= (D > 2 ? 1 : 0); ++dz)
#pragma unroll
            for (int dy = (D > 1 ? -1 : 0); dy <= (D > 1 ? 1 : 0); ++dy) {
                int py = 0, pz = 0;
                if (D > 1 && !in_box(g, pl, 1, c[1] + dy, &py)) continue;
                if (D > 2 && !in_box(g, pl, 2, c[2] + dz, &pz)) continue;
#pragma unroll
                for (int k = 0; k < (1 << (D - 1)); ++k) {
                    const uint8_t* r = fc + cell_id(g, l, 0, D > 1 ? 2 * py + (k & 1) : 0, D > 2 ? 2 * pz + (k >> 1) : 0);
                    const uint4* v = reinterpret_cast<const uint4*>(r + x0);
                    m |= halve_bits(byte_mask(v[0], 4) | byte_mask(v[1], 4) << 16) << 1;
                    constexpr unsigned kBoth = FL_REF | FL_REF << 8;
                    if ((x0 > 0 || wrap) && (*reinterpret_cast<const uint16_t*>(r + (x0 > 0 ? x0 : n) - 2) & kBoth)) m |= 1u;
                    const int xr = x0 + 2 * kStep;
                    if ((xr < n || wrap) && (*reinterpret_cast<const uint16_t*>(r + (xr < n ? xr : 0)) & kBoth)) m |= 1u << 17;
                }
            }
        const unsigned hit = (m | m >> 1 | m >> 2) & 0xffffu & ~own;
        if (hit) refine16(fp + s * kStep, hit);
        count += __popc(hit);
    }
    return count;
}

// Does the tree flagged by a remesh at level la fit the node arrays?  The
// threads of its mark and closure passes count the cells c that they flag, and
// the blocks add their counts into room[0] (counting the flags again in the last
// pass, which has few blocks when la is a coarse level, took up to 20 us).
// The new tree has 2^d nodes above level la per refined cell, and the slots
// it may take are the free ones plus those of the nodes above level la now
// (the remesh releases them first).  The last block of the last pass to finish
// (ticket room[3]) decides: short of slots, the solver halts at this iteration
// (room[4], counted on by its first kernel), room[1] = it + 1, room[2] = the
// nodes of the new tree (see halted()).  Called by every thread of the block.
__device__ __forceinline__ void room_count(const Grid& g, int c)
{
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&g.room[0], c);
}

__device__ __forceinline__ void room_decide(const Grid& g, int c, int la)
{
    __shared__ int blk;
    if (threadIdx.x == 0) blk = 0;
    __syncthreads();
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&blk, c);
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (blk) atomicAdd(&g.room[0], blk);
    __threadfence();
    if (atomicAdd(&g.room[3], 1) != (int)gridDim.x - 1) return;
    __threadfence();
    const long long fresh = (long long)atomicExch(&g.room[0], 0) << g.d;
    g.room[3] = 0;
    long long above = 0, below = 0;
    for (int l = g.lb; l <= g.L; ++l) {
        const long long n = (long long)g.counts[l] + g.counts[LMAX + 1 + l];
        if (l > la) above += n;
        else below += n;
    }
    if (fresh > g.ftop[0] + above) {
        g.room[2] = (int)(below + fresh);
        g.room[1] = g.room[4] + 1;
    }
}

// refined cells among this thread's share of levels la..L-1
__device__ __forceinline__ int refined_here(const Grid& g, int la)
{
    int c = 0;
    long long from = g.off[la];
    if (la < kStepLevel) {
        MRLT_GRID_STRIDE(i, g.N[la]) c += (g.flag[from + i] & FL_REF) ? 1 : 0;
        from = g.off[la + 1];
    }
    MRLT_GRID_STRIDE(s, (g.off[g.L] - from) / kStep)
        c += __popc(byte_mask(*reinterpret_cast<const uint4*>(g.flag + from + s * kStep), 4));
    return c;
}

// Slots of the nodes a remesh removes (levels la+1..L: a node whose parent
// is not refined any more), pushed on the free stack before the apply passes
// pop slots for new nodes.  Walks the node lists of the tree being replaced.
static __device__ __forceinline__ void dev_release(const Grid& g, int la)
{
    for (int l = la + 1; l <= g.L; ++l) {
        const long long N = g.N[l];
        for (int which = 0; which < 2; ++which) {
            const int cnt = g.counts[which * (LMAX + 1) + l];
            const int* list = (which ? g.inner : g.leaves) + g.off[l];
            MRLT_GRID_STRIDE(t, cnt)
            {
                const long long id = list[t];
                if (id < 0 || id >= N) {
                    atomicOr(g.err, ERR_INDEX);
                    continue;
                }
                int c[3];
                cell_xyz(g, l, id, c);
                const long long p = cell_id(g, l - 1, c[0] >> 1, c[1] >> 1, c[2] >> 1);
                if (g.flag[g.off[l - 1] + p] & FL_REF) continue; // stays
                const int sl = slot_of(g, l, id);
                if (sl > 0) g.fstack[atomicAdd(&g.ftop[0], 1)] = sl;
                g.slot[g.off[l] + id] = -1;
            }
        }
    }
}

// install the new tree on level l (top-down): status from the refinement
// flags; new nodes take a free slot (the sink, with ERR_CAPACITY, when none
// is left) and are predicted from level l-1 (Sec. 2, in FP64, stored as T);
// new leaves and merged nodes get q^{n+1} = q^n; registers of changed nodes
// cleared.  A CTA of NT threads finds the changed cells of its steps first and
// then shares the nodes among them evenly between its threads.
template <int D, int M, class T, int NT>
__device__ __forceinline__ void dev_apply(const Grid& g, int l, int la)
{
    __shared__ uint16_t item[NT * kStep]; // offset | existed before << 12 | leaf << 13
    __shared__ int nitem;
    static_assert(NT * kStep <= 4096, "offsets of 12 bits");
    const long long N = g.N[l];
    const int top = g.ftop[0]; // free slots after this remesh's releases
    const bool wide = l >= kStepLevel;
    const int per = wide ? kStep : 1;
    uint8_t* st = g.st + g.off[l];
    for (long long base = (long long)blockIdx.x * NT * per; base < N; base += (long long)gridDim.x * NT * per) {
        if (threadIdx.x == 0) nitem = 0;
        __syncthreads();
        const long long i = base + threadIdx.x * per;
        if (i < N) {
            int c[3];
            cell_xyz(g, l, i, c);
            unsigned ol, oi, ex, ref = 0; // leaves and internal nodes before, nodes of the new tree, refined cells
            if (wide) {
                const uint4 s = *reinterpret_cast<const uint4*>(st + i);
                ol = byte_mask(s, 0);
                oi = byte_mask(s, 1);
                ex = l == la ? ol | oi : parent_bits(g, g.flag + g.off[l - 1], l, c, 4);
                if (l < g.L) ref = byte_mask(*reinterpret_cast<const uint4*>(g.flag + g.off[l] + i), 4);
            } else {
                ol = st[i] & 1;
                oi = st[i] >> 1;
                ex = l == la ? ol | oi
                             : (unsigned)(g.flag[g.off[l - 1] + cell_id(g, l - 1, c[0] >> 1, c[1] >> 1, c[2] >> 1)] >> 4 & 1);
                if (l < g.L) ref = g.flag[g.off[l] + i] >> 4 & 1;
            }
            if (ref & ~ex) atomicOr(g.err, ERR_SOURCE);
            const unsigned nl = ex & ~ref, ni = ex & ref;
            const unsigned changed = (ol ^ nl) | (oi ^ ni);
            if (changed) {
                if (wide)
                    *reinterpret_cast<uint4*>(st + i) =
                        make_uint4(mask_bytes(nl) | mask_bytes(ni) << 1, mask_bytes(nl >> 4) | mask_bytes(ni >> 4) << 1,
                                   mask_bytes(nl >> 8) | mask_bytes(ni >> 8) << 1,
                                   mask_bytes(nl >> 12) | mask_bytes(ni >> 12) << 1);
                else
                    st[i] = (uint8_t)(nl | ni << 1);
                unsigned m = changed & ex; // removed nodes: their slots were released before the apply passes
                int at = m ? atomicAdd(&nitem, __popc(m)) : 0;
                for (; m; m &= m - 1) {
                    const int j = __ffs(m) - 1;
                    item[at++] = (uint16_t)(threadIdx.x * per + j | ((ol | oi) >> j & 1) << 12 | (nl >> j & 1) << 13);
                }
            }
        }
        __syncthreads();
        for (int t = threadIdx.x; t < nitem; t += NT) {
            const int it = item[t];
            const long long id = base + (it & 4095);
            const bool old = it >> 12 & 1;
            int sl = 0, k = 0;
            double p[M];
            if (old) {
                sl = slot_of(g, l, id);
            } else { // the pop is on its way while the prediction's sources are read
                k = atomicAdd(&g.ftop[1], 1);
                int c[3];
                cell_xyz(g, l, id, c);
                const Ctx x{l, 0, g.lb};
                predict<D, M, T, double>(g, x, l, c, p);
                if (k < top) sl = g.fstack[top - 1 - k];
                else atomicOr(g.err, ERR_CAPACITY);
                g.slot[g.off[l] + id] = sl;
            }
            T* q0 = nd<T>(g, F_Q0, sl);
            if (!old) {
#pragma unroll
                for (int v = 0; v < M; ++v) q0[v] = T(p[v]);
            }
            if (it >> 13) {
                T* qe = nd<T>(g, F_QE, sl);
#pragma unroll
                for (int v = 0; v < M; ++v) qe[v] = q0[v];
            }
            if (g.rg) {
                double* rg = regs(g.rg, g, sl);
                for (int r = 0; r < g.nf * M; ++r) rg[r] = 0.0;
            }
        }
        __syncthreads(); // the list is written again
    }
}

// adaptation flags of levels >= la cleared (grid-stride)
static __device__ __forceinline__ void dev_clear_flags(const Grid& g, long long from, long long to)
{
    MRLT_GRID_STRIDE(i, to - from) g.flag[from + i] = 0;
}

// ------------------------------------------------------------ compaction
// Leaf, node and active-tile lists of levels lo..hi in two passes over the
// status bytes, 16 cells per thread and step (one 16-byte load).  Bound by
// those bytes and the launches: a level is cut into at most kMaxChunks chunks,
// so a block of the second pass sums the counts of the chunks before its own
// itself and no scan pass is needed; the first pass flags the tiles, so their
// lists are built by extra blocks of the second.  On a GB300, with 46 k finest
// leaves at 2D L = 10 and 330 k at 3D L = 8, one byte per thread and a scan
// and a tile-list launch beside took 11 + 19 + 12 + 3 and 150 + 430 + 150 +
// 131 us; this takes 2.7 + 4.0 and 8 + 19 us.
constexpr int kChunk = 128 * kStep; // cells of a chunk at least
constexpr int kMaxChunkLog = 10;   // at most 2^10 chunks per level
static_assert(kTile1X % kStep == 0 && kTile2X % kStep == 0 && kTile3X * 2 == kStep,
              "a step lies in one tile row in 1D and 2D and in two tiles in 3D");

// cells of a chunk of level l: 2^11, doubled until 2^10 chunks cover the level
__host__ __device__ __forceinline__ long long chunk_cells(const Grid& g, int l)
{
    const int sh = g.d * l - kMaxChunkLog - 11;
    return (long long)kChunk << (sh > 0 ? sh : 0);
}

// Chunks numbered over levels lo..hi: level l owns [base[l], base[l+1]).
struct LevelChunks {
    int lo, hi;
    int base[LMAX + 2];
};

__host__ __device__ __forceinline__ int number_chunks(const Grid& g, LevelChunks& b, int lo, int hi)
{
    int total = 0;
    b.lo = lo;
    b.hi = hi;
    for (int l = lo; l <= hi; ++l) {
        b.base[l] = total;
        total += (int)((g.N[l] + chunk_cells(g, l) - 1) / chunk_cells(g, l));
    }
    b.base[hi + 1] = total;
    return total;
}

__device__ __forceinline__ int chunk_level(const LevelChunks& b, int c)
{
    int l = b.lo;
    while (l < b.hi && c >= b.base[l + 1]) ++l;
    return l;
}

// Exclusive sum of v over the block's threads in thread order; total: the
// sum.  Every thread of the block takes part.
template <int NT>
__device__ __forceinline__ unsigned block_scan(unsigned v, unsigned* total)
{
    __shared__ unsigned ws[NT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += x;
    }
    if (lane == 31) ws[warp] = inc;
    __syncthreads();
    unsigned before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        before += w < warp ? ws[w] : 0u;
        all += ws[w];
    }
    __syncthreads(); // ws may be written again
    *total = all;
    return before + inc - v;
}

// the leaf's tile of the tiled stage kernel is active
__device__ __forceinline__ void mark_tile(const Grid& g, int l, long long i)
{
    const int tx = g.d == 1 ? kTile1X : (g.d == 2 ? kTile2X : kTile3X);
    const int ty = g.d == 2 ? kTile2Y : kTile3Y;
    const long long mask = (1LL << l) - 1;
    const long long x = i & mask, y = g.d >= 2 ? (i >> l) & mask : 0, z = g.d == 3 ? i >> (2 * l) : 0;
    g.tflag[g.toff[l] + x / tx + (long long)g.ntx[l] * (y / ty + (long long)g.nty[l] * (z / kTile3Z))] = 1;
}

// the tiles of the leaves among cells i..i+15 (i a multiple of 16, leaf mask m)
__device__ __forceinline__ void mark_tiles(const Grid& g, int l, long long i, unsigned m)
{
    if (l < 4) { // several rows
        for (; m; m &= m - 1) mark_tile(g, l, i + __ffs(m) - 1);
    } else if (g.d == 3) {
        if (m & 0xffu) mark_tile(g, l, i);
        if (m >> 8) mark_tile(g, l, i + 8);
    } else if (m) {
        mark_tile(g, l, i);
    }
}

// Per chunk (a CTA of NT threads): number of leaves and of internal nodes,
// into bc[2 chunk], bc[2 chunk + 1]; their tiles flagged, the spent
// refinement flags cleared.
template <int NT>
__device__ __forceinline__ void chunk_count(const Grid& g, const LevelChunks& lc, int chunk, int* bc)
{
    const int l = chunk_level(lc, chunk);
    const long long cells = chunk_cells(g, l), c0 = (chunk - lc.base[l]) * cells;
    const long long c1 = min(c0 + cells, g.N[l]);
    unsigned nl = 0, ni = 0;
    for (long long i = c0 + threadIdx.x * kStep; i < c1; i += NT * kStep) {
        const uint4 s = *reinterpret_cast<const uint4*>(g.st + g.off[l] + i);
        *reinterpret_cast<uint4*>(g.flag + g.off[l] + i) = make_uint4(0, 0, 0, 0); // the remesh is installed
        if (!(s.x | s.y | s.z | s.w)) continue;
        const unsigned m = byte_mask(s, 0);
        nl += __popc(m);
        ni += __popc(byte_mask(s, 1));
        mark_tiles(g, l, i, m);
    }
    unsigned a, b;
    block_scan<NT>(nl, &a);
    block_scan<NT>(ni, &b);
    if (threadIdx.x == 0) {
        bc[2 * chunk] = (int)a;
        bc[2 * chunk + 1] = (int)b;
        if (chunk == 0) { // the slots popped by the remesh leave the free stack
            const int k = g.ftop[1], top = g.ftop[0];
            g.ftop[0] = top - (k < top ? k : top);
            g.ftop[1] = 0;
        }
    }
}

// Per chunk: leaves and internal nodes written to the level lists behind those
// of the chunks before it (ascending cell id); the last chunk of a level
// writes the level's counts.
template <int NT>
__device__ __forceinline__ void chunk_scatter(const Grid& g, const LevelChunks& lc, int chunk, const int* bc)
{
    const int l = chunk_level(lc, chunk);
    const int ownl = bc[2 * chunk], owni = bc[2 * chunk + 1];
    const bool last = chunk + 1 == lc.base[l + 1];
    if (!(ownl | owni) && !last) return; // uniform across the CTA
    unsigned a = 0, b = 0;
    for (int k = lc.base[l] + threadIdx.x; k < chunk; k += NT) {
        a += bc[2 * k];
        b += bc[2 * k + 1];
    }
    unsigned pl, pi;
    block_scan<NT>(a, &pl);
    block_scan<NT>(b, &pi);
    if (last && threadIdx.x == 0) {
        g.counts[l] = (int)pl + ownl;
        g.counts[LMAX + 1 + l] = (int)pi + owni;
    }
    const long long cells = chunk_cells(g, l), c0 = (chunk - lc.base[l]) * cells;
    const long long c1 = min(c0 + cells, g.N[l]);
    int* leaves = g.leaves + g.off[l];
    int* inner = g.inner + g.off[l];
    for (long long i0 = c0; i0 < c1; i0 += NT * kStep) { // uniform across the CTA
        const long long i = i0 + threadIdx.x * kStep;
        uint4 s = make_uint4(0, 0, 0, 0);
        if (i < c1) s = *reinterpret_cast<const uint4*>(g.st + g.off[l] + i);
        unsigned ml = byte_mask(s, 0), mi = byte_mask(s, 1);
        unsigned all; // at most 16 x 256 of each: two 16-bit sums in one
        const unsigned ex = block_scan<NT>(__popc(ml) | __popc(mi) << 16, &all);
        unsigned at = pl + (ex & 0xffffu);
        for (; ml; ml &= ml - 1) leaves[at++] = (int)(i + __ffs(ml) - 1);
        at = pi + (ex >> 16);
        for (; mi; mi &= mi - 1) inner[at++] = (int)(i + __ffs(mi) - 1);
        pl += all & 0xffffu;
        pi += all >> 16;
    }
}

// ordered list of the flagged tiles of level l by one CTA of NT threads, the
// flags cleared again; each thread takes up to 8 x 16 consecutive flags
template <int NT>
__device__ __forceinline__ void level_tile_list(const Grid& g, int l)
{
    const int nt = g.ntx[l] * g.nty[l] * g.ntz[l];
    uint4* fl = reinterpret_cast<uint4*>(g.tflag + g.toff[l]);
    int* list = g.tlist + g.toff[l];
    const int words = (nt + kStep - 1) / kStep; // 16 flags each; the padding holds none
    const int per = min(8, (words + NT - 1) / NT);
    unsigned pos = 0;
    for (int w0 = 0; w0 < words; w0 += NT * per) { // uniform across the CTA
        const int w = w0 + threadIdx.x * per;
        unsigned m[8], c = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            m[k] = k < per && w + k < words ? byte_mask(fl[w + k], 0) : 0u;
            c += __popc(m[k]);
        }
        unsigned all, at = pos + block_scan<NT>(c, &all);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (m[k]) fl[w + k] = make_uint4(0, 0, 0, 0);
            for (unsigned x = m[k]; x; x &= x - 1) list[at++] = (w + k) * kStep + __ffs(x) - 1;
        }
        pos += all;
    }
    if (threadIdx.x == 0) g.counts[2 * (LMAX + 1) + l] = (int)pos;
}

// ------------------------------------------------------------ registers
// conservative correction of the coarse leaves of levels lo..hi whose step
// ended: q += +-(coarse time-integrated flux - mean of the fine ones) / dx; the
// registers read are cleared for the next step.  Bound by the dependent trips
// of a leaf (neighbours' statuses, children's slots, registers), so each trip
// loads all it can: the statuses of all faces at once, the rows of a face's
// children at once.  One face, variable and child after the other took 40 us
// per launch over the opening of the 2D Euler L = 10 solve on a GB300 (73 k
// leaves), and 142 us in the 3D blast at L = 7; this takes 13 and 36 us.
template <int D>
struct RefluxRefs {
    unsigned finer; // faces to an internal node
    int l, c[3], sl;
};

template <int D>
__device__ __forceinline__ RefluxRefs<D> lookup_reflux(const Grid& g, int l, long long id)
{
    RefluxRefs<D> r;
    r.l = l;
    cell_xyz(g, l, id, r.c);
    uint8_t st[2 * D];
#pragma unroll
    for (int fi = 0; fi < 2 * D; ++fi) {
        int nb[3] = {r.c[0], r.c[1], r.c[2]};
        st[fi] = in_box(g, l, fi >> 1, r.c[fi >> 1] + (fi & 1 ? 1 : -1), &nb[fi >> 1])
                     ? status(g, l, cell_id(g, l, nb[0], nb[1], nb[2]))
                     : 0;
    }
    r.sl = slot_of(g, l, id);
    r.finer = 0;
#pragma unroll
    for (int fi = 0; fi < 2 * D; ++fi) r.finer |= (st[fi] == 2 ? 1u : 0u) << fi;
    return r;
}

template <int D, int M, class T>
__device__ __forceinline__ void reflux_leaf(const Grid& g, const RefluxRefs<D>& e)
{
    constexpr int NT = 1 << (D - 1);
    if (!e.finer) return;
    const int l = e.l;
    const int* c = e.c;
    double* rc = regs(g.rg, g, e.sl);
    T q[M];
    load_row<M, T>(nd<T>(g, F_QE, e.sl), q);
    for (unsigned finer = e.finer; finer; finer &= finer - 1) {
        const int fi = __ffs(finer) - 1, k = fi >> 1, side = (fi & 1) ? 1 : -1;
        const int opp = 2 * k + (side > 0 ? 0 : 1);
        int nk; // the neighbour's coordinate along k
        in_box(g, l, k, (k == 0 ? c[0] : (k == 1 ? c[1] : c[2])) + side, &nk);
        double* rf[NT];
#pragma unroll
        for (int tt = 0; tt < NT; ++tt) {
            int p[3] = {0, 0, 0}, bit = 0;
#pragma unroll
            for (int j = 0; j < D; ++j) {
                if (j == k) p[j] = 2 * nk + (side > 0 ? 0 : 1);
                else p[j] = 2 * c[j] + ((tt >> bit++) & 1);
            }
            const long long ch = cell_id(g, l + 1, p[0], p[1], p[2]);
            if (status(g, l + 1, ch) != 1) atomicOr(g.err, ERR_REFLUX);
            rf[tt] = regs(g.rg, g, slot_of(g, l + 1, ch)) + opp * M;
        }
        double r[NT][M], own[M];
        const double none[M] = {};
        load_row<M, double>(rc + fi * M, own);
#pragma unroll
        for (int tt = 0; tt < NT; ++tt) load_row<M, double>(rf[tt], r[tt]);
        const double idx = g.rdx[l][k];
#pragma unroll
        for (int v = 0; v < M; ++v) {
            double sum = 0.0;
#pragma unroll
            for (int tt = 0; tt < NT; ++tt) sum += r[tt][v];
            // the correction from the FP64 registers, rounded to T once
            q[v] = T(double(q[v]) + side * (own[v] - sum * (1.0 / NT)) * idx);
        }
        store_row<M, double>(rc + fi * M, none);
#pragma unroll
        for (int tt = 0; tt < NT; ++tt) store_row<M, double>(rf[tt], none);
    }
    store_row<M, T>(nd<T>(g, F_QE, e.sl), q);
}

template <int D, int M, class T>
__device__ __forceinline__ void dev_reflux(const Grid& g, int lo, int hi)
{
    for_list<0>(g, lo, hi, [&](int l, long long id, long long) { reflux_leaf<D, M, T>(g, lookup_reflux<D>(g, l, id)); });
}

// ------------------------------------------------------------ reductions
// *at = max(*at, x), for the bit patterns of non-negative doubles; most calls
// find a larger value already there and skip the atomic
__device__ __forceinline__ void max_bits(unsigned long long* at, double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    if (b > *(volatile unsigned long long*)at) atomicMax(at, b);
}

// running max |q^n_v| over the leaves of levels lo..hi (detail normalisation)
template <int M, class T>
__device__ __forceinline__ void dev_scale(const Grid& g, int lo, int hi)
{
    double mx[M] = {};
    for_list<0>(g, lo, hi, [&](int l, long long id, long long) {
        T q0[M];
        load_row<M, T>(nd<T>(g, F_Q0, slot_of(g, l, id)), q0);
#pragma unroll
        for (int v = 0; v < M; ++v) mx[v] = fmax(mx[v], fabs(double(q0[v])));
    });
#pragma unroll
    for (int v = 0; v < M; ++v) {
        double a = mx[v];
        for (int o = 16; o > 0; o >>= 1) a = fmax(a, __shfl_xor_sync(0xffffffffu, a, o));
        if ((threadIdx.x & 31) == 0 && a > 0.0) max_bits(&g.scale_bits[v], a);
    }
}

// non-finite end values of the leaves of levels lo..hi set ERR_NONFINITE
template <int M, class T>
__device__ __forceinline__ void dev_finite(const Grid& g, int lo, int hi)
{
    for_list<0>(g, lo, hi, [&](int l, long long id, long long) {
        T qe[M];
        load_row<M, T>(nd<T>(g, F_QE, slot_of(g, l, id)), qe);
        bool ok = true;
#pragma unroll
        for (int v = 0; v < M; ++v) ok = ok && isfinite(double(qe[v]));
        if (!ok) atomicOr(g.err, ERR_NONFINITE);
    });
}

// largest sum of characteristic speeds over the leaves of levels lo..hi (CFL
// step), as the bit pattern of a positive double in *g.wmax
template <int EQ, int D, class T>
__device__ __forceinline__ void dev_wave(const Grid& g, int lo, int hi)
{
    constexpr int M = EQ == 2 ? D + 2 : 1;
    double w = 0.0;
    for_list<0>(g, lo, hi, [&](int l, long long id, long long) {
        T qe[M];
        load_row<M, T>(nd<T>(g, F_QE, slot_of(g, l, id)), qe);
        double q[M];
#pragma unroll
        for (int v = 0; v < M; ++v) q[v] = double(qe[v]);
        const double s = wave_speed<EQ, D, M>(g, q);
        w = fmax(w, s != s ? 1e300 : s);
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w = fmax(w, __shfl_xor_sync(0xffffffffu, w, o));
    if ((threadIdx.x & 31) == 0 && w > 0.0) max_bits(g.wmax, w);
}

} // namespace mrlt
