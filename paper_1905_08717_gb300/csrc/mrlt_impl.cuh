// mrlt_impl.cuh -- device data layout and shared device routines of the
// MRLT/NERK library (private to the library; the public C-ABI is mrlt.h).
//
// Data layout in HBM (one solver instance):
//   every level l in [min_level, L] indexes its N_l = 2^{d l} cells as
//   id = i + n_l (j + n_l k), n_l = 2^l; the per-cell maps of all levels live
//   in one "pyramid" allocation at offset off[l] (cells):
//   - status (uint8): 0 absent, 1 leaf, 2 internal node; refinement flags (uint8)
//   - slot (int32): the node's slot in the node arrays, -1 when absent
//   The values live only where nodes exist: node arrays of `cap` slots, each
//   node's m variables contiguous ([slot][v]); slot 0 is a sink that never
//   belongs to a node (see the capacity rule in mrlt_api.cu):
//   - fields, float64, or float32 in the mixed-precision mode (the state is
//     stored, and the stage arithmetic done, in FP32; registers and the detail
//     test stay FP64):
//       Q0 q^n, Q1 q*, Q2 q**, QE q^{n+1} (leaves: compact RK stages of Sec. 3;
//       internal nodes: the projections / refreshed values of Algs. 3-9),
//       XH half-step value (Eq. 17), NH, N1, N3 the NERK theta = 1/2, 1/4, 3/4
//       values of internal nodes.  Leaves never store NERK values: they are
//       recomputed from Q0, Q1, Q2, QE where needed (same polynomial).
//   - registers (float64, [slot][face][v]): the time-integrated flux through
//       each face of a leaf whose neighbour across it is on another level (a
//       coarse leaf at a face to finer nodes, or a fine leaf at a face to a
//       coarser leaf).  One array serves both roles: the kind of a face cannot
//       change while its register holds a value (the restricted remesh keeps
//       both sides until the coarse step ends, when the reflux clears them).
//   - per-level compact lists (int32) of leaves and internal nodes, ascending
//     cell id, rebuilt after every remesh by a two-pass stream compaction.
//   Free slots form a stack (fstack, ftop[0] entries); a remesh releases the
//   slots of removed nodes, then pops slots for new nodes (ftop[1] counts the
//   pops until the next compaction commits them).
#pragma once
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

namespace mrlt {

constexpr int LMAX = 16;
constexpr int MMAX = 5;
constexpr int NTHREADS = 128;
// tiles of the tiled stage kernel (d = 1: 48 cells; d = 2: 16 x 8; d = 3: 8 x 4 x 4)
constexpr int kTile1X = 48;
constexpr int kTile2X = 16, kTile2Y = 8;
constexpr int kTile3X = 8, kTile3Y = 4, kTile3Z = 4;
// threads per tile CTA: two per cell (measured: 3D blast L=8 -10 to -13%, 2D
// Euler L=10 -1.5% against one per cell; four per cell was slower)
constexpr int kTileThreads1 = 64, kTileThreads2 = 256, kTileThreads3 = 256;

enum Field { F_Q0 = 0, F_Q1, F_Q2, F_QE, F_XH, F_NH, F_N1, F_N3, NFIELD };
enum FlagBits { FL_SIG = 1, FL_BIG = 2, FL_REF = 16 };
enum ErrBits { ERR_INDEX = 1, ERR_SOURCE = 2, ERR_NONFINITE = 4, ERR_REFLUX = 8, ERR_TIMEOUT = 16, ERR_CAPACITY = 32 };

struct Grid {
    uint8_t* st;
    uint8_t* flag;
    int* slot;                      // per cell: node slot, -1 when absent
    int* fstack;                    // free slots
    int* ftop;                      // [0] free slots on the stack, [1] pops not yet committed
    long long cap;                  // node slots (slot 0 is the sink)
    void* f[NFIELD];                // node fields: double, or float when prec = 1
    double* rg;                     // flux registers of the nodes, [slot][face][v]
    int* leaves;
    int* inner;
    int* counts;                    // [0..LMAX] leaves, [LMAX+1..] internal nodes, [2(LMAX+1)..] active tiles
    uint8_t* tflag;                 // per-level tile flags (tile holds a leaf)
    int* tlist;                     // per-level lists of active tiles, ascending
    double* scale;                  // [MMAX] detail normalisation s_v
    unsigned long long* scale_bits; // [MMAX] running max |q_v| (bit pattern)
    int* err;
    unsigned long long* near;
    unsigned long long* wmax;
    unsigned long long* updates;
    unsigned long long* work;       // [(LMAX+1) * 4]: leaf-stages per level and stage
    unsigned* built;                // [0] publications of the running captured piece, [1] of direct launches (see
                                    // TreeSync); tile tickets: [2] of direct stage launches, [3..] of the piece's
    double* dtp;                    // fine step dt of the current macro step (device scalar)
    int* room;                      // [0] refinement flags being counted, [1] halt: iteration + 1, [2] nodes needed,
                                    // [3] blocks that counted, [4] iteration of the macro step
    long long off[LMAX + 1];
    long long N[LMAX + 1];
    int n[LMAX + 1];
    double dx[LMAX + 1][3];
    double rdx[LMAX + 1][3];        // 1 / dx
    long long toff[LMAX + 1];       // tile offset of each level in tflag / tlist
    int ntx[LMAX + 1], nty[LMAX + 1], ntz[LMAX + 1]; // tiles per direction
    int d, m, nf, L, lb, eq, rk, gts;
    int bc[3];
    double phys[8];
    double eps;
    int eps_mode;
    int prec;                       // 0 FP64, 1 mixed: state, fluxes and stage updates in FP32
    int flux;                       // Euler: 0 HLL, 1 AUSM+
    double igm;                     // Euler: 1 / (gamma - 1)
    double cstar;                   // Euler: 2 (gamma - 1) / (gamma + 1)
    int gcap;                       // CTAs per stage launch at most (0: resident capacity)
};

// Programmatic dependent launch (sm_90 and later).  Every thread of every kernel
// waits until the kernel before it in the stream has completed and its writes are
// visible (griddepcontrol.wait), then allows the next kernel's launch to begin
// (griddepcontrol.launch_dependents).  The launch and the CTA setup of the next
// kernel thus overlap the tail of this one.  Most kernels wait first; those that
// leave the tree alone may look it up before (tree_enter).  Both are no-ops in a
// kernel launched without a programmatic dependency.
__device__ __forceinline__ void pdl_enter()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A remesh inside a macro step whose new tree would need more node slots than
// the arrays hold halts the solver's device work (room[1] != 0): every later
// kernel of the fine iterations returns at its start, until the host has
// grown the arrays, cleared the halt and resumed at the halted iteration.
// Read after pdl_enter, or after tree_enter: the remesh that sets it comes before
// the publication that follows the remesh.
__device__ __forceinline__ bool halted(const Grid& g) { return g.room[1] != 0; }

// Lookups before the wait: the tree (counts, lists, statuses, slots), the halt
// and the fine step.  A kernel's own wait makes its predecessor's writes visible;
// those of the launches before that one have to be known to be visible in another
// way, which TreeSync holds for each launch of a kernel that leaves the tree alone:
//  - kVisible: captured in a piece of a macro step, with no remesh before it in
//    the piece.  A graph launch is ordered with the stream, so a piece starts
//    after everything before it.
//  - kPublish: the first kernel after a remesh, or after anything else of the
//    kind.  It waits first, and then adds one to g.built[word] with release order.
//  - kAcquire: it reads g.built[word] with acquire order, and a count of at least
//    `need` shows that the last publication before it, and with it all that is
//    looked up, is visible; otherwise it waits first.  No older value can be
//    taken for that count: word 0, of captured launches, counts within a piece and
//    is cleared at the end of each (k_piece_end); word 1, of direct launches, only
//    grows, and the host knows the count.
//  - kWait: it waits first.  For instances of a large batch, which fill the GPU
//    for one another: nothing is gained there by starting early, and the acquire
//    (which drops the L1 cache) slows the neighbours.
// tree_enter is called by every thread of the CTA and returns whether this one has
// waited.  Measured on a GB300 against waiting first everywhere: 1D Burgers L = 10
// 17.9 / 20.9 ms, 2D Burgers L = 10 83.5 / 95.3, global step L = 9 72.0 / 77.1, 3D
// blast L = 7 35.6 / 39.1, 2D Euler L = 10 opening, FP64 179 / 204 and mixed 73.7 /
// 85.3 ms.  In 2D and 3D one thread reads the count for its CTA (with a read by
// every warp 2D Burgers took 1% and 2D Euler 1.5% longer); the small CTAs of 1D
// read it with every thread (one thread and a barrier: 2% longer).
enum TreeMode { kVisible = 0, kAcquire, kPublish, kWait };
struct TreeSync {
    int mode, word;
    unsigned need;
};
template <int D>
__device__ __forceinline__ bool tree_enter(const Grid& g, const TreeSync& t)
{
    if (t.mode == kVisible) return false;
    if (t.mode == kAcquire) {
        unsigned n = t.need - 1;
        if (D == 1 || threadIdx.x == 0)
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(n) : "l"(g.built + t.word) : "memory");
        const bool there = (int)(n - t.need) >= 0;
        if (D == 1 ? there : __syncthreads_or(there) != 0) return false;
    } else if (t.mode == kPublish) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (blockIdx.x == 0) { // before this CTA lets the next kernel start
            if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(g.built + t.word) : "memory");
            __syncthreads();
        }
    }
    pdl_enter();
    return true;
}

#define MRLT_ENTER(g)         \
    do {                      \
        pdl_enter();          \
        if (halted(g)) return; \
    } while (0)

// Launch with programmatic stream serialisation: the kernel may be launched
// before its predecessor in the stream has finished; it waits in pdl_enter().
template <class... KArgs, class... Args>
inline cudaError_t pdl_launch(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

// exposure context: level u being updated, stage s (0 = plain q^n), lmin
struct Ctx {
    int u, s, lmin;
};

// Ghost rule, the same on every level: periodic wrap; homogeneous Neumann as
// an even mirror; zero Dirichlet (scalar equations) as an odd mirror, the
// ghost taking the negated value: the parity neg flips at every reflection
// on a Dirichlet wall (an odd count negates the value).
__device__ __forceinline__ int wrap_or_mirror(const Grid& g, int l, int k, int p, int& neg)
{
    const int n = g.n[l];
    if (g.bc[k] == 0) return p & (n - 1); // periodic wrap (n = 2^l)
    const int odd = g.bc[k] == 2;
#pragma unroll 1
    for (int it = 0; it < 8 && (p < 0 || p >= n); ++it) {
        p = p < 0 ? -1 - p : 2 * n - 1 - p;
        neg ^= odd;
    }
    return p < 0 ? 0 : (p >= n ? n - 1 : p);
}

// neighbourhood rule of the tree: wrap when periodic, drop cells past a wall
__device__ __forceinline__ bool in_box(const Grid& g, int l, int k, int p, int* q)
{
    const int n = g.n[l];
    if (g.bc[k] == 0) {
        *q = p & (n - 1); // periodic wrap (n = 2^l)
        return true;
    }
    if (p < 0 || p >= n) return false;
    *q = p;
    return true;
}

__device__ __forceinline__ long long cell_id(const Grid& g, int l, int x, int y, int z)
{
    const long long n = g.n[l];
    return (long long)x + n * ((long long)y + n * (long long)z);
}

// coordinates of cell id on level l (n = 2^l cells per direction)
__device__ __forceinline__ void cell_xyz(const Grid& g, int l, long long id, int c[3])
{
    const long long mask = (1LL << l) - 1;
    c[0] = (int)(id & mask);
    c[1] = g.d > 1 ? (int)((id >> l) & mask) : 0;
    c[2] = g.d > 2 ? (int)(id >> (2 * l)) : 0;
}

// the m values of field f of the node in slot sl, stored as T (double, or
// float in the mixed mode); a negative slot (an absent cell) reads the sink
template <class T>
__device__ __forceinline__ T* nd(const Grid& g, int f, int sl)
{
    return static_cast<T*>(g.f[f]) + (long long)(sl < 0 ? 0 : sl) * g.m;
}

__device__ __forceinline__ int slot_of(const Grid& g, int l, long long id)
{
    return g.slot[g.off[l] + id];
}

// registers of the node in slot sl: [face][v]
__device__ __forceinline__ double* regs(double* r, const Grid& g, int sl)
{
    return r + (long long)(sl < 0 ? 0 : sl) * g.nf * g.m;
}

__device__ __forceinline__ uint8_t status(const Grid& g, int l, long long id)
{
    return g.st[g.off[l] + id];
}

// Value of the stored node of level l in slot sl (status st) as seen by the stencil of a
// level-u leaf at stage x.s of the current iteration: the exposure table of
// Secs. 4.1-4.3 / Algs. 3-9.  Leaves recompute their NERK values from the
// stage values: with k1 = q* - q^n and k2 the second stage increment
// (RK2: k2 = 2 q^{n+1} - q^n - q*, RK3: k2 = 4 q** - 3 q^n - q*),
// q(theta) = q^n + (theta - theta^2/2) k1 + theta^2/2 k2 (Sec. 3 NERK2).
// T is the storage type of the fields, O the arithmetic type of the result.
template <int M, class T, class O>
__device__ __forceinline__ void expose(const Grid& g, const Ctx& x, int l, int sl, int st, O* out)
{
    const T* q0 = nd<T>(g, F_Q0, sl);
    const T* q1 = nd<T>(g, F_Q1, sl);
    const T* q2 = nd<T>(g, F_Q2, sl);
    const T* qe = nd<T>(g, F_QE, sl);
    const int s = x.s;
    const int rel = l - x.u;
    if (s == 0 || (s == 1 && g.gts) || (s == 1 && (rel >= 0 || l >= x.lmin))) {
#pragma unroll
        for (int v = 0; v < M; ++v) out[v] = O(q0[v]);
        return;
    }
    if (g.gts) {
        const T* a = s == 2 ? q1 : q2;
#pragma unroll
        for (int v = 0; v < M; ++v) out[v] = O(a[v]);
        return;
    }
    if (s == 1) { // coarser level lmin-1, mid-step: theta = 1/2 value
        if (g.rk == 3) {
#pragma unroll
            for (int v = 0; v < M; ++v) out[v] = O(q2[v]);
        } else if (st == 1) {
#pragma unroll
            for (int v = 0; v < M; ++v)
                out[v] = O(0.5) * O(q0[v]) + O(0.25) * O(q1[v]) + O(0.25) * O(qe[v]);
        } else {
            const T* nh = nd<T>(g, F_NH, sl);
#pragma unroll
            for (int v = 0; v < M; ++v) out[v] = O(nh[v]);
        }
        return;
    }
    if (s == 2) {
        if (rel == 0) {
#pragma unroll
            for (int v = 0; v < M; ++v) out[v] = O(q1[v]);
        } else if (rel == 1) {
            if (st == 1) { // Eq. 14: q* + k2
                if (g.rk == 2) {
#pragma unroll
                    for (int v = 0; v < M; ++v) out[v] = O(2) * O(qe[v]) - O(q0[v]);
                } else {
#pragma unroll
                    for (int v = 0; v < M; ++v) out[v] = O(4) * O(q2[v]) - O(3) * O(q0[v]);
                }
            } else { // Eq. 15
#pragma unroll
                for (int v = 0; v < M; ++v) out[v] = O(2) * O(q1[v]) - O(q0[v]);
            }
        } else if (l >= x.lmin) { // half step of the coarser level
            if (st == 1) {
#pragma unroll
                for (int v = 0; v < M; ++v) out[v] = O(q0[v]) + O(0.5) * (O(q1[v]) - O(q0[v]));
            } else {
                const T* xh = nd<T>(g, F_XH, sl);
#pragma unroll
                for (int v = 0; v < M; ++v) out[v] = O(xh[v]);
            }
        } else { // end of the mid-step coarser level
#pragma unroll
            for (int v = 0; v < M; ++v) out[v] = O(qe[v]);
        }
        return;
    }
    // stage 3
    if (rel == 0) {
#pragma unroll
        for (int v = 0; v < M; ++v) out[v] = O(q2[v]);
    } else if (rel == 1) {
#pragma unroll
        for (int v = 0; v < M; ++v) out[v] = O(qe[v]);
    } else {
        const bool act = l >= x.lmin;
        if (st == 1) {
            const O b1 = act ? O(7.0 / 32.0) : O(15.0 / 32.0);
            const O b2 = act ? O(1.0 / 32.0) : O(9.0 / 32.0);
#pragma unroll
            for (int v = 0; v < M; ++v) {
                const O a0 = O(q0[v]), a1 = O(q1[v]);
                const O k1 = a1 - a0;
                const O k2 = O(4) * O(q2[v]) - O(3) * a0 - a1;
                out[v] = a0 + b1 * k1 + b2 * k2;
            }
        } else {
            const T* nn = nd<T>(g, act ? F_N1 : F_N3, sl);
#pragma unroll
            for (int v = 0; v < M; ++v) out[v] = O(nn[v]);
        }
    }
}

// Eq. 4 along one direction in FP64: the child of offset a (0 left, 1 right) of
// m between its neighbours l and r.  Predictions in FP64 apply it direction by
// direction (2 operations each) instead of weighting every cell of the block.
__device__ __forceinline__ double child(double l, double m, double r, int a)
{
    return fma(a ? 0.125 : -0.125, r - l, m);
}

// 1D prediction weights of Eq. 4 for child offset a (0 left, 1 right):
// child = parent + s (right - left) / 8, s = -1 for a = 0, +1 for a = 1.
__device__ __forceinline__ double pw(int a, int delta)
{
    if (delta == 0) return 1.0;
    const double s = a ? 0.125 : -0.125;
    return delta > 0 ? s : -s;
}

// Tensor-product prediction (Eq. 4 applied along each direction) of the cell
// at in-box coordinates q of level l from the 3^d stored nodes of level l-1
// around its parent, using their exposures.
template <int D, int M, class T, class O>
__device__ __forceinline__ void predict(const Grid& g, const Ctx& x, int l, const int q[3], O* out)
{
    const int pl = l - 1;
#pragma unroll
    for (int v = 0; v < M; ++v) out[v] = O(0);
    if (pl < g.lb) {
        atomicOr(g.err, ERR_SOURCE);
        return;
    }
    const int P0 = q[0] >> 1, P1 = q[1] >> 1, P2 = q[2] >> 1;
    const int a0 = q[0] & 1, a1 = q[1] & 1, a2 = q[2] & 1;
    // in 3D the outer loops stay rolled: 27 inlined exposures per prediction
    // site cost far more compile time than the loop overhead they save
#pragma unroll(D > 2 ? 1 : 3)
    for (int dz = (D > 2 ? -1 : 0); dz <= (D > 2 ? 1 : 0); ++dz) {
        int nz = 0;
        const int z = D > 2 ? wrap_or_mirror(g, pl, 2, P2 + dz, nz) : 0;
        const O wz = D > 2 ? O(pw(a2, dz)) : O(1);
#pragma unroll(D > 2 ? 1 : 3)
        for (int dy = (D > 1 ? -1 : 0); dy <= (D > 1 ? 1 : 0); ++dy) {
            int nyz = nz;
            const int y = D > 1 ? wrap_or_mirror(g, pl, 1, P1 + dy, nyz) : 0;
            const O wyz = wz * (D > 1 ? O(pw(a1, dy)) : O(1));
#pragma unroll
            for (int dxx = -1; dxx <= 1; ++dxx) {
                int neg = nyz;
                const int xx = wrap_or_mirror(g, pl, 0, P0 + dxx, neg);
                const long long id = cell_id(g, pl, xx, y, z);
                const int st = status(g, pl, id);
                const int sl = slot_of(g, pl, id);
                if (st == 0) {
                    atomicOr(g.err, ERR_SOURCE);
                    continue;
                }
                O val[M];
                expose<M, T, O>(g, x, pl, sl, st, val);
                const O w0 = wyz * O(pw(a0, dxx));
                const O w = neg ? -w0 : w0; // an odd-mirror ghost enters negated
#pragma unroll
                for (int v = 0; v < M; ++v) out[v] += w * val[v];
            }
        }
    }
}

// value of the cell at (possibly out-of-box) coordinates p on level l
template <int D, int M, class T, class O>
__device__ __forceinline__ void value_at(const Grid& g, const Ctx& x, int l, const int p[3], O* out)
{
    int q[3] = {0, 0, 0};
    int neg = 0;
#pragma unroll
    for (int k = 0; k < D; ++k) q[k] = wrap_or_mirror(g, l, k, p[k], neg);
    const long long id = cell_id(g, l, q[0], q[1], q[2]);
    const int st = status(g, l, id);
    if (st) expose<M, T, O>(g, x, l, slot_of(g, l, id), st, out);
    else predict<D, M, T, O>(g, x, l, q, out);
    if (neg) {
#pragma unroll
        for (int v = 0; v < M; ++v) out[v] = -out[v];
    }
}

// ---------------------------------------------------------------- physics
// FP64 operations issue at 2 lanes per clock and SM on this GPU (one warp
// instruction every 16 cycles), integer operations at 64: comparisons, signs and
// selections of doubles are done on their bit patterns below.
__device__ __forceinline__ long long ordered_bits(double a) // ordered as the values are (-0 below +0)
{
    const long long x = __double_as_longlong(a);
    return x ^ (x >> 63 & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ bool less(double a, double b) { return ordered_bits(a) < ordered_bits(b); }
__device__ __forceinline__ bool negative(double a) { return __double2hiint(a) < 0; } // sign bit
__device__ __forceinline__ bool positive(double a) { return __double_as_longlong(a) > 0; } // and not +0
// bits of |a|, one place up: ordered as the magnitudes are.  (Masking the sign bit
// instead is recognised as fabs, which is an FP64 instruction.)
__device__ __forceinline__ unsigned long long abs_bits(double a)
{
    return (unsigned long long)__double_as_longlong(a) << 1;
}
__device__ __forceinline__ bool below_abs(double a, double b) { return abs_bits(a) < abs_bits(b); } // |a| < |b|

// A product and a sum rounded by themselves, never contracted into a
// multiply-add.  Where an expression could be contracted in two ways, the one
// meant is written out: the FP32 results must not depend on what the compiler
// finds around it.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }

template <class R>
__device__ __forceinline__ R minmod(R a, R b)
{
    if (a * b <= R(0)) return R(0);
    return fabs(a) < fabs(b) ? a : b;
}
// The same on the bit patterns.  A NaN leaves b, as in the comparisons above: a NaN
// in b passes on to the slope.  (Differences hold quiet NaNs only, whose high word
// lies above infinity's.)
__device__ __forceinline__ double minmod(double a, double b)
{
    const unsigned ha = (unsigned)__double2hiint(a) << 1, hb = (unsigned)__double2hiint(b) << 1;
    const bool take_a = below_abs(a, b);
    const double m = take_a ? a : b;
    const double r = (__double2hiint(a) ^ __double2hiint(b)) < 0 ? 0.0 : m;
    return (take_a ? hb : ha) > 0xffe00000u ? b : r;
}

// 1 / x and 1 / sqrt(x) for the fluxes, correctly rounded and CUDA's rsqrt: over
// all of FP64, subnormal densities and pressures included.  A third-order step
// from the hardware's approximation, which takes 4% fewer FP64 operations in a
// full-grid stage launch, loses both: it is good to one unit in the last place
// only and gives a NaN for subnormals and infinities.
template <class R>
__device__ __forceinline__ R recip(R x) { return R(1) / x; }
__device__ __forceinline__ double recip_sqrt(double x) { return rsqrt(x); }

// a[k] for a run-time direction k < D: selects, where an indexed register
// array would have to live in local memory
template <int D, class R>
__device__ __forceinline__ R along(const R* a, int k)
{
    R x = a[0];
    if (D > 1 && k == 1) x = a[1];
    if (D > 2 && k == 2) x = a[2];
    return x;
}

// Variables that MUSCL reconstructs: primitives (rho, u_1..u_d, p) for Euler,
// the conserved variable itself otherwise.  R is the arithmetic type of the
// flux evaluation: double, or float in the mixed-precision mode; W holds the
// conservative values (type WT).
template <int EQ, int D, int M, class R, class WT>
__device__ __forceinline__ void recon_vars(const Grid& g, const WT* W, R* P)
{
    if constexpr (EQ == 2) {
        const R gam = R(g.phys[0]);
        const R rho = R(W[0]);
        const R ir = recip(rho);
        R ke = R(0);
        P[0] = rho;
#pragma unroll
        for (int c = 0; c < D; ++c) {
            P[1 + c] = R(W[1 + c]) * ir;
            ke += R(W[1 + c]) * P[1 + c];
        }
        P[D + 1] = (gam - R(1)) * (R(W[D + 1]) - R(0.5) * ke);
    } else {
#pragma unroll
        for (int v = 0; v < M; ++v) P[v] = R(W[v]);
    }
}

// AUSM+ (Liou 1996), the paper's Euler flux (Sec. 5), across a face normal
// to direction k, from the reconstructed primitives (rho, u_1..u_d, p) of both
// sides.  With total enthalpy H = (E + p)/rho
// and critical speed a*^2 = 2 (g-1)/(g+1) H, the interface speed is
// a = min(a*_L^2 / max(a*_L, u_L), a*_R^2 / max(a*_R, -u_R)); the Mach
// numbers M = u/a are split as M+-(M) = +-(M +- 1)^2/4 +- (M^2 - 1)^2/8 and
// pressure as P+-(M) = (M +- 1)^2 (2 -+ M)/4 +- 3/16 M (M^2 - 1)^2 when
// |M| < 1 (upwind values otherwise); the flux is
// a (max(m, 0) Psi_L + min(m, 0) Psi_R) + p_half e_k, Psi = rho (1, u, H),
// m = M+(M_L) + M-(M_R), p_half = P+(M_L) p_L + P-(M_R) p_R.
template <class R>
__device__ __forceinline__ R ausm_split_mach(R M, R sgn)
{
    if (fabs(M) >= R(1)) return R(0.5) * (M + sgn * fabs(M));
    const R t = M * M - R(1);
    return sgn * R(0.25) * (M + sgn) * (M + sgn) + sgn * R(0.125) * t * t;
}

template <class R>
__device__ __forceinline__ R ausm_split_pres(R M, R sgn)
{
    if (fabs(M) >= R(1)) return M * sgn > R(0) ? R(1) : R(0);
    const R t = M * M - R(1);
    return R(0.25) * (M + sgn) * (M + sgn) * (R(2) - sgn * M) + sgn * R(0.1875) * M * t * t;
}

template <int D, class R>
__device__ __forceinline__ void ausm_plus(R gam, int k, const R* PL, const R* PR, const R* UL, const R* UR, R* F)
{
    const R pL = PL[D + 1], pR = PR[D + 1];
    const R HL = (UL[D + 1] + pL) / PL[0], HR = (UR[D + 1] + pR) / PR[0];
    const R uL = along<D>(PL + 1, k), uR = along<D>(PR + 1, k);
    const R cst = R(2) * (gam - R(1)) / (gam + R(1));
    const R asL = sqrt(cst * HL), asR = sqrt(cst * HR);
    const R atL = asL * asL / fmax(asL, uL);
    const R atR = asR * asR / fmax(asR, -uR);
    const R a = fmin(atL, atR);
    const R ML = uL / a, MR = uR / a;
    const R mh = ausm_split_mach(ML, R(1)) + ausm_split_mach(MR, R(-1));
    const R ph = ausm_split_pres(ML, R(1)) * pL + ausm_split_pres(MR, R(-1)) * pR;
    const R mp = fmax(mh, R(0)), mm = fmin(mh, R(0));
    F[0] = a * (mp * PL[0] + mm * PR[0]);
#pragma unroll
    for (int c = 0; c < D; ++c) {
        F[1 + c] = mul_rn(a, mp * UL[1 + c] + mm * UR[1 + c]);
        if (c == k) F[1 + c] = add_rn(F[1 + c], ph);
    }
    F[D + 1] = a * (mp * (PL[0] * HL) + mm * (PR[0] * HR));
}

// The same in FP64 with fewer operations: four divisions instead of six (a*^2
// / a* = a* unless the normal flow is above critical), the polynomials of a side
// shared by its two splits, and the flux from the two mass fluxes.
__device__ __forceinline__ void ausm_split(double M, double sgn, double& mach, double& pres)
{
    if (!below_abs(M, 1.0)) {
        const bool with = !negative(M * sgn);
        mach = with ? M : 0.0;
        pres = with ? 1.0 : 0.0;
        return;
    }
    const double t = fma(M, M, -1.0), t2 = t * t, q = M + sgn, q2 = 0.25 * q * q;
    mach = sgn * fma(0.125, t2, q2);
    pres = fma(q2, fma(-sgn, M, 2.0), (sgn * 0.1875) * M * t2);
}

template <int D, int M>
__device__ __forceinline__ void ausm_plus64(const Grid& g, int k, const double* PL, const double* PR, double* F)
{
    const double pL = PL[D + 1], pR = PR[D + 1];
    double keL = 0.0, keR = 0.0;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        keL = fma(PL[1 + c], PL[1 + c], keL);
        keR = fma(PR[1 + c], PR[1 + c], keR);
    }
    const double hp = g.igm + 1.0; // enthalpy of pressure: p g / (g - 1)
    const double HL = fma(hp, pL / PL[0], 0.5 * keL), HR = fma(hp, pR / PR[0], 0.5 * keR);
    const double uL = along<D>(PL + 1, k), uR = along<D>(PR + 1, k);
    const double cst = g.cstar; // 2 (g - 1) / (g + 1)
    const double aL2 = cst * HL, aR2 = cst * HR;
    // a side without a critical speed leaves the interface speed to the other
    const bool okL = positive(aL2), okR = positive(aR2);
    double aL = sqrt(aL2), aR = sqrt(aR2);
    if (okL && less(aL, uL)) aL = aL2 / uL;
    if (okR && less(aR, -uR)) aR = aR2 / -uR;
    const double a = !okL ? aR : (!okR || less(aL, aR) ? aL : aR);
    double m1, p1, m2, p2;
    ausm_split(uL / a, 1.0, m1, p1);
    ausm_split(uR / a, -1.0, m2, p2);
    const double mh = a * (m1 + m2), ph = fma(p1, pL, p2 * pR);
    const bool back = negative(mh);
    const double fL = back ? 0.0 : mh * PL[0], fR = back ? mh * PR[0] : 0.0; // mass fluxes
    F[0] = fL + fR;
#pragma unroll
    for (int c = 0; c < D; ++c) F[1 + c] = fma(fL, PL[1 + c], fma(fR, PR[1 + c], c == k ? ph : 0.0));
    F[D + 1] = fma(fL, HL, fR * HR);
}

// HLL in FP64 from the reconstructed primitives, by its weights: with
// w_L = s_R / (s_R - s_L) and w_R = -s_L / (s_R - s_L) (1 and 0 when both waves
// run one way) the flux is w_L F(U_L) + w_R F(U_R) + d (U_R - U_L), d = s_L w_L =
// -s_R w_R: each side gives U (w u_n -+ d), - on the left, plus w times the
// pressure terms.  The two mass fluxes rho (w u_n -+ d) carry momentum and kinetic
// energy, so neither the conservative states nor the physical fluxes are formed;
// with one d for both sides its rounding cancels between like states (with
// w (u_n - s) for each side, one operation more, the root mean square error of
// the mass flux is 0.238 x 2^-53 of rho (|u| + c) against 0.195; rho, u and p of
// order one, neighbours within 10%).  Measured on a GB300 when this, the
// comparisons above and child() replaced the general forms, mean stage-2 launch:
// 2D Euler L = 10 from 43.9 to 35.8 us on level 10 and 33.3 to 24.9 us on level
// 9, 3D blast L = 7 from 308 to 243 us on level 7.
template <int D, int M>
__device__ __forceinline__ void hll64(const Grid& g, int k, const double* PL, const double* PR, double* F)
{
    const double gam = g.phys[0], igm = g.igm, pL = PL[D + 1], pR = PR[D + 1];
    const double uL = along<D>(PL + 1, k), uR = along<D>(PR + 1, k);
    // sound speeds sqrt(gamma p / rho) = gamma p rsqrt(gamma p rho)
    const double gpL = gam * pL, gpR = gam * pR, xL = gpL * PL[0], xR = gpR * PR[0];
    const double cL = gpL * recip_sqrt(xL), cR = gpR * recip_sqrt(xR);
    double lL = uL - cL, lR = uR - cR, rL = uL + cL, rR = uR + cR;
    // a side without a sound speed (no positive pressure, as a prediction at a
    // strong shock may give) leaves the wave speeds to the other
    const bool okL = positive(xL), okR = positive(xR);
    if (!okL) lL = lR, rL = rR;
    if (!okR) lR = lL, rR = rL;
    const double sL = less(lL, lR) ? lL : lR, sR = less(rL, rR) ? rR : rL;
    const bool allL = (okL || okR) && !negative(sL), allR = (okL || okR) && !allL && !positive(sR);
    const double ids = recip(sR - sL);
    double wL = sR * ids, wR = -sL * ids;
    const double d = sL * wL;
    double aL = fma(wL, uL, -d), aR = fma(wR, uR, d);
    if (allL || allR) {
        wL = allL ? 1.0 : 0.0;
        wR = allL ? 0.0 : 1.0;
        aL = allL ? uL : 0.0;
        aR = allL ? 0.0 : uR;
    }
    const double mL = aL * PL[0], mR = aR * PR[0]; // mass fluxes
    F[0] = mL + mR;
    const double pw2 = fma(wL, pL, wR * pR);
    double keL = 0.0, keR = 0.0;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        F[1 + c] = fma(mL, PL[1 + c], fma(mR, PR[1 + c], c == k ? pw2 : 0.0));
        keL = fma(PL[1 + c], PL[1 + c], keL);
        keR = fma(PR[1 + c], PR[1 + c], keR);
    }
    // energy: m ke / 2 + p (a / (g - 1) + w u_n), each side
    const double eL = pL * fma(aL, igm, wL * uL), eR = pR * fma(aR, igm, wR * uR);
    F[D + 1] = fma(0.5 * mL, keL, fma(0.5 * mR, keR, eL + eR));
}

// Numerical flux along direction k across the face between stencil cells 1
// and 2 of a 4-cell stencil, from their reconstruction variables P(i, v).
template <int EQ, int D, int M, class R, class Acc>
__device__ __forceinline__ void flux_recon(const Grid& g, int k, double dxf, const Acc& P, R* F)
{
    const R h = R(0.5);
    if constexpr (EQ == 0) { // linear advection, centred flux
        F[0] = R(g.phys[k]) * (P(1, 0) + P(2, 0)) * h;
    } else if constexpr (EQ == 3) { // two-point diffusive flux
        F[0] = -R(g.phys[0]) * (P(2, 0) - P(1, 0)) / R(dxf);
    } else if constexpr (EQ == 1) { // Burgers: MUSCL-minmod + Godunov
        const R u0 = P(0, 0), u1 = P(1, 0), u2 = P(2, 0), u3 = P(3, 0);
        const R uL = u1 + h * minmod(u1 - u0, u2 - u1);
        const R uR = u2 - h * minmod(u2 - u1, u3 - u2);
        const R fL = h * uL * uL, fR = h * uR * uR;
        if (uL <= uR) F[0] = uL > R(0) ? fL : (uR < R(0) ? fR : R(0));
        else F[0] = fmax(fL, fR);
    } else { // Euler: MUSCL-minmod on (rho, u_1..u_d, p) + HLL
        const R gam = R(g.phys[0]);
        R PL[M], PR[M];
#pragma unroll
        for (int v = 0; v < M; ++v) {
            const R a0 = P(0, v), a1 = P(1, v), a2 = P(2, v), a3 = P(3, v);
            PL[v] = a1 + h * minmod(a1 - a0, a2 - a1);
            PR[v] = a2 - h * minmod(a2 - a1, a3 - a2);
        }
        if constexpr (sizeof(R) == 8) {
            if (g.flux == 1) ausm_plus64<D, M>(g, k, PL, PR, F);
            else hll64<D, M>(g, k, PL, PR, F);
        } else {
            R UL[M], UR[M], FL[M], FR[M];
            R keL = R(0), keR = R(0);
            UL[0] = PL[0];
            UR[0] = PR[0];
#pragma unroll
            for (int c = 0; c < D; ++c) {
                UL[1 + c] = PL[0] * PL[1 + c];
                UR[1 + c] = PR[0] * PR[1 + c];
                keL += PL[1 + c] * PL[1 + c];
                keR += PR[1 + c] * PR[1 + c];
            }
            const R igm = R(g.igm);
            UL[D + 1] = fma(PL[D + 1], igm, mul_rn(h * PL[0], keL));
            UR[D + 1] = fma(PR[D + 1], igm, mul_rn(h * PR[0], keR));
            const R unL = along<D>(PL + 1, k), unR = along<D>(PR + 1, k);
            if (g.flux == 1) { // AUSM+
                ausm_plus<D, R>(gam, k, PL, PR, UL, UR, F);
                return;
            }
#pragma unroll
            for (int v = 0; v <= D; ++v) {
                FL[v] = mul_rn(UL[v], unL);
                FR[v] = mul_rn(UR[v], unR);
                if (v == 1 + k) {
                    FL[v] = add_rn(FL[v], PL[D + 1]);
                    FR[v] = add_rn(FR[v], PR[D + 1]);
                }
            }
            // energy flux (E + p) u_n: which product is rounded first differs by
            // dimension, as FP32 solves have always had it
            const R eL = UL[D + 1], eR = UR[D + 1], pL = PL[D + 1], pR = PR[D + 1];
            FL[D + 1] = D == 2 ? fma(eL, unL, mul_rn(pL, unL)) : fma(pL, unL, mul_rn(eL, unL));
            FR[D + 1] = D == 2 ? fma(eR, unR, mul_rn(pR, unR)) : fma(pR, unR, mul_rn(eR, unR));
            // sound speeds sqrt(gamma p / rho) = gamma p rsqrt(gamma p rho)
            const R gpL = gam * PL[D + 1], gpR = gam * PR[D + 1];
            const R cL = gpL * rsqrt(gpL * PL[0]);
            const R cR = gpR * rsqrt(gpR * PR[0]);
            const R sL = fmin(unL - cL, unR - cR);
            const R sR = fmax(unL + cL, unR + cR);
            if (sL >= R(0)) {
#pragma unroll
                for (int v = 0; v < M; ++v) F[v] = FL[v];
            } else if (sR <= R(0)) {
#pragma unroll
                for (int v = 0; v < M; ++v) F[v] = FR[v];
            } else {
                const R ids = R(1) / (sR - sL);
#pragma unroll
                for (int v = 0; v < M; ++v)
                    F[v] = fma(sL * sR, UR[v] - UL[v], fma(sR, FL[v], -mul_rn(sL, FR[v]))) * ids;
            }
        }
    }
}

template <int EQ, int D, int M>
__device__ __forceinline__ double wave_speed(const Grid& g, const double* q)
{
    double s = 0.0;
    if constexpr (EQ == 0) {
#pragma unroll
        for (int k = 0; k < D; ++k) s += fabs(g.phys[k]);
    } else if constexpr (EQ == 1) {
        s = D * fabs(q[0]);
    } else if constexpr (EQ == 2) {
        const double gam = g.phys[0], rho = q[0];
        double ke = 0.0;
#pragma unroll
        for (int k = 0; k < D; ++k) ke += q[1 + k] * q[1 + k] / rho;
        const double p = (gam - 1.0) * (q[D + 1] - 0.5 * ke);
        const double c = sqrt(gam * p / rho);
#pragma unroll
        for (int k = 0; k < D; ++k) s += fabs(q[1 + k] / rho) + c;
    }
    return s;
}

// ---------------------------------------------------------------- host side
struct Launch; // fwd

// kernel launchers (defined in the .cu files), all on stream `st`
// one compact RK stage s on every leaf of the levels lo..hi (independent
// levels only), fine step dt = *g.dtp (level u steps dt, or 2^{L-u} dt in LT
// mode), RK weight b of the stage; returns the number of kernel launches issued
// (-1 when the kernel could not be set up).  lo > hi only sets the kernel up.
// sync: see TreeSync; tick: the index of its tile tickets in g.built.
int launch_stage(const Grid& g, cudaStream_t st, int lo, int hi, int s, int lmin, double b, int reg, TreeSync sync,
                 int tick);
// iterations of the longest captured piece and its lead (see run_macro).  Measured
// on a GB300, whole passes with 8 / 16 / 32: 1D Burgers L = 10 from creation 19.2 /
// 19.1 / 19.8 ms, mixed 2D Euler opening 78.1 / 78.9 / 80.5, 2D Burgers 83.9 / 83.8 /
// 85.0, a batch of 24 66.6 / 67.7 / 72.5, a server's 12 requests 55.4 / 56.4 / 58.7.
constexpr int kBlockIters = 16;
// words of g.built: three, and one for each stage launch of a captured piece (at
// most kBlockIters iterations of one launch and two for each level)
constexpr int kDirectTick = 2, kFirstTick = 3;
constexpr int kBuiltWords = kFirstTick + kBlockIters * (1 + 2 * (LMAX + 1));
void launch_wave(const Grid& g, cudaStream_t st);
// one persistent macro-step kernel launch (mrlt_macro.cuh); a == nullptr sets
// the kernel up only.  Returns 1 when launched, 0 after set-up, -1 on failure.
struct MacroArgs;
int launch_macro(const Grid& g, cudaStream_t st, const MacroArgs* a);
// the bounded grid barrier with `missing` CTAs that never arrive (self-test)
int launch_grid_wait_test(cudaStream_t st, int ctas, int missing, unsigned long long limit_ns, unsigned* bar,
                          int* err);
} // namespace mrlt
