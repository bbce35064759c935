// mrlt_stage.cuh -- the stage kernels of the MR/MRLT time evolution: face
// fluxes from the exposures of Secs. 4.1-4.3, the compact RK update of Sec. 3
// and the flux-register epilogue.
// k_stage_tile (d = 1, 2, 3) works on one tile of one level per CTA: the
// halo is staged in shared memory and every face flux is computed once.  It is
// instantiated for R = double and, for the mixed-precision mode, R = float:
// the stored state, the exposures, the reconstruction, the numerical fluxes,
// the right-hand side and the RK update are all in R; the flux registers
// accumulate in double.
#pragma once
#include "mrlt_impl.cuh"
#include "mrlt_tree_dev.cuh"

namespace mrlt {

// Compact RK update of one variable of a leaf from its right-hand side f (Sec. 3):
//   s = 1: q*  = q^n + dt_l f
//   s = 2: RK2 q^{n+1} = q^n/2 + q*/2 + dt_l f/2 ; RK3 q** = 3q^n/4 + q*/4 + dt_l f/4
//   s = 3: q^{n+1} = q^n/3 + 2q**/3 + 2 dt_l f/3
// qs is the leaf's own value at stage s (q^n, q*, q** for s = 1, 2, 3: its
// exposure, already staged in shared memory) and q0 its q^n (s >= 2).
// The roundings are written out (see mul_rn); with one variable the product of
// the larger weight is rounded first.
template <int M, class R>
__device__ __forceinline__ void rk_update(const Grid& g, int sl, int v, int s, R dtl, R f, R q0, R qs)
{
    const R kk = mul_rn(dtl, f);
    if (s == 1) {
        nd<R>(g, F_Q1, sl)[v] = qs + kk;
        return;
    }
    R a, b, c; // weights of q0, qs, kk
    int to = F_QE;
    if (s == 2 && g.rk == 2) {
        a = b = c = R(0.5);
    } else if (s == 2) {
        a = R(0.75);
        b = c = R(0.25);
        to = F_Q2;
    } else {
        a = R(1.0 / 3.0);
        b = c = R(2.0 / 3.0);
    }
    const R q = M == 1 ? fma(b, qs, mul_rn(a, q0)) : fma(a, q0, mul_rn(b, qs));
    nd<R>(g, to, sl)[v] = fma(c, kk, q);
}

// Tile shapes of the tiled stage kernel: a CTA of THREADS threads owns
// TX x TY x TZ cells of one level (the same shapes index the per-level
// active-tile lists); THREADS may exceed the cell count, so that the list,
// exposure and face phases spread over more threads.  Bits holds a row of
// the tile and its ring, one bit per cell.
template <int D> struct Tile;
template <> struct Tile<1> {
    static constexpr int TX = kTile1X, TY = 1, TZ = 1, THREADS = kTileThreads1;
    using Bits = unsigned long long;
};
template <> struct Tile<2> {
    static constexpr int TX = kTile2X, TY = kTile2Y, TZ = 1, THREADS = kTileThreads2;
    using Bits = unsigned;
};
template <> struct Tile<3> {
    static constexpr int TX = kTile3X, TY = kTile3Y, TZ = kTile3Z, THREADS = kTileThreads3;
    using Bits = unsigned;
};
__device__ __forceinline__ int popc(unsigned m) { return __popc(m); }
__device__ __forceinline__ int popc(unsigned long long m) { return __popcll(m); }
__device__ __forceinline__ int first_bit(unsigned m) { return __ffs(m) - 1; }
__device__ __forceinline__ int first_bit(unsigned long long m) { return __ffsll(m) - 1; }

// Block (tile + 2-cell ring) and face counts of one tile; the large shared
// arrays (conservative values, reconstruction variables, face fluxes) live in
// dynamic shared memory, SMEM bytes.
template <int EQ, int D, class R>
struct TileShape {
    static constexpr int M = EQ == 2 ? D + 2 : 1;
    static constexpr int TX = Tile<D>::TX, TY = Tile<D>::TY, TZ = Tile<D>::TZ, H = 2;
    static constexpr int NC = TX * TY * TZ, NT = Tile<D>::THREADS; // cells, threads
    static constexpr int BX = TX + 2 * H, BY = D > 1 ? TY + 2 * H : 1, BZ = D > 2 ? TZ + 2 * H : 1;
    static constexpr int NB = BX * BY * BZ, NR = BY * BZ; // cells and rows of the block
    static_assert(NT % 32 == 0 && NT >= NC && NT >= NR + 32, "one thread per cell and per row, a warp for the faces");
    static_assert(TX % 2 == 0 && (D < 2 || TY % 2 == 0) && (D < 3 || TZ % 2 == 0), "tiles hold whole siblings");
    static_assert(BX <= 8 * (int)sizeof(typename Tile<D>::Bits) && TX + 1 <= BX, "a row fits a mask");
    // entries of a variable of the block: padded so that the variables of a
    // leaf, taken by adjacent lanes, fall in different banks (M = 4)
    static constexpr int NBP = (NB + 15) / 16 * 16 + (sizeof(R) == 8 ? 4 : 8);
    static constexpr int NFX = (TX + 1) * TY * TZ;
    static constexpr int NFY = D > 1 ? TX * (TY + 1) * TZ : 0;
    static constexpr int NFZ = D > 2 ? TX * TY * (TZ + 1) : 0;
    static constexpr int NF = NFX + NFY + NFZ;
    // rows of faces: normal to x, y, z
    static constexpr int RFX = TY * TZ, RFY = D > 1 ? (TY + 1) * TZ : 0, RFZ = D > 2 ? TY * (TZ + 1) : 0;
    static constexpr int NFR = RFX + RFY + RFZ;
    static_assert(NB <= 1024 && NF <= 1024, "packed face entries");
    // parent-level block: the cells of level u-1 whose exposures predict the
    // virtual cells of the block (Eq. 4 reads a 3^d neighbourhood of the parent)
    static constexpr int PBX = TX / 2 + 4, PBY = D > 1 ? TY / 2 + 4 : 1, PBZ = D > 2 ? TZ / 2 + 4 : 1;
    static constexpr int PB = PBX * PBY * PBZ;
    // sub-face tasks whose two finer-side cells are fetched with the exposures
    static constexpr int NPF = D > 2 ? 64 : (D > 1 ? 128 : 32);
    static_assert(NPF <= NT - 32, "fetched by the warps after the first");
    // dynamic shared memory (all R): conservative values of the block and of
    // the parent block, reconstruction variables, face fluxes and the
    // prefetched finer-side variables
    static constexpr size_t SMEM = sizeof(R) * M * (2 * NBP + PB + NF + 2 * NPF);
    // CTAs per SM that the registers are shared out for.  Measured on a GB300,
    // solves of the benchmark cases: 2D FP32 4 / 5 / 6 per SM 99.3 / 97.1 / 97.4
    // ms, 3D FP32 2 / 3 / 4 24.6 / 22.7 / 22.8 ms; 2D FP64 2 / 3 / 4 / 5 240 /
    // 221.5 / 221.7 / 222.8 ms, 3D FP64 1 / 2 48.2 / 43.3 ms (bound by FP64 issue);
    // 1D FP64 4 / 8 / 16: Sod L = 10 18.63 / 18.46 / 19.20 ms, its full grid at L = 14
    // 4.48 / 4.97 / 5.31 ms, Burgers L = 14 2.84 / 2.84 / 3.01 ms.
    static constexpr int PERSM = D == 1 ? 8 : (D == 2 ? (sizeof(R) == 4 ? 5 : 3) : (sizeof(R) == 4 ? 3 : 2));
};

// Value, as the level-u stencil sees it at stage x.s (the rel = +1 rows of
// expose()), of the stored node of level u + 1 in slot sl (status st != 0):
// every field the choice may need, loaded at once.
template <int M, class T>
__device__ __forceinline__ void finer_exposure(const Grid& g, const Ctx& x, int st, int sl, T* out)
{
    const T* q0 = nd<T>(g, F_Q0, sl);
    if (x.s <= 1) {
#pragma unroll
        for (int v = 0; v < M; ++v) out[v] = q0[v];
        return;
    }
    if (g.gts || x.s == 3) { // global step: q* / q**; LT stage 3: q^{n+1} of the first sub-step
        const T* a = nd<T>(g, g.gts ? (x.s == 2 ? F_Q1 : F_Q2) : F_QE, sl);
#pragma unroll
        for (int v = 0; v < M; ++v) out[v] = a[v];
        return;
    }
    // LT stage 2: leaf Eq. 14 (q* + k2), internal node Eq. 15 (2 q* - q^n)
    const T* q1 = nd<T>(g, F_Q1, sl);
    const T* qx = nd<T>(g, g.rk == 2 ? F_QE : F_Q2, sl);
    T a0[M], a1[M], ax[M];
#pragma unroll
    for (int v = 0; v < M; ++v) {
        a0[v] = q0[v];
        a1[v] = q1[v];
        ax[v] = qx[v];
    }
    if (st == 1) {
        if (g.rk == 2) {
#pragma unroll
            for (int v = 0; v < M; ++v) out[v] = T(2) * ax[v] - a0[v];
        } else {
#pragma unroll
            for (int v = 0; v < M; ++v) out[v] = T(4) * ax[v] - T(3) * a0[v];
        }
    } else {
#pragma unroll
        for (int v = 0; v < M; ++v) out[v] = T(2) * a1[v] - a0[v];
    }
}

// value_at() out of line, for the rare cells whose sources are not staged
// (inlined, its registers would be those of the whole kernel)
template <int D, int M, class R>
__device__ __noinline__ void far_value(const Grid& g, Ctx x, int l, int p0, int p1, int p2, R* out)
{
    const int p[3] = {p0, p1, p2};
    value_at<D, M, R, R>(g, x, l, p, out);
}

// Tiled stage (d = 1, 2, 3).  The CTA works on one tile of one level at a
// time, in phases separated by CTA barriers, with as few dependent trips to
// memory as the data allow:
//  1. status and slot of the tile, its 2-cell ring and the parent-level block
//     (one trip), the statuses as bit sets by warp ballots;
//  2. the work of the tile as row masks, a thread per row of cells or faces:
//     the cells some tile leaf reads -- its radius-2 cross stencil and the
//     3^d block of a leaf facing an internal node -- split into stored nodes
//     and virtual cells (absent nodes and ghosts past a wall); the
//     parent-block cells the virtual cells' predictions (Eq. 4) read; the
//     faces touching a tile leaf, split into faces against an internal node
//     (2^{d-1} sub-faces on level u+1, Sec. 2) and plain faces;
//  3. one trip for everything the stage reads from memory: exposures
//     (Secs. 4.1-4.3) of the stored cells and of the parent-block cells and
//     the finer-side cells of the sub-faces (their slots were fetched during
//     phase 2); the lists written from the masks meanwhile;
//  4. virtual cells predicted in shared memory from the parent block (a ghost
//     whose mirror image is stored takes that image's value), and the
//     reconstruction variables of every needed cell;
//  5. every face touching a tile leaf computed once, one thread per face or
//     sub-face (the 2^{d-1} threads of a face are adjacent lanes, combined by
//     shuffles), the leaf's own virtual children predicted from its shared
//     3^d block;
//  6. the compact RK update and the flux-register epilogue, one thread per
//     variable of a leaf.
// The chain of these phases is what an adaptive launch costs beside its FP64
// work (a few hundred tiles, one to three per CTA).  With masks a row of
// cells is one word, so phase 2 is some 50 instructions of one thread per
// row, where each cell's and face's neighbourhood was tested by itself and
// appended to the lists with a block barrier per step.  Measured on a GB300,
// mean over the stage-2 launches of the opening of a solve: 2D Euler L = 10
// mixed from 13.9 to 12.1 us, FP64 from 38.9 to 37 us (bound by its FP64
// operations), 3D blast L = 8 mixed from 160 to 117 us, L = 7 FP64 from 234
// to 216 us.
// Work lists keep every warp on one kind of work.  In FP32 each value is
// computed by the same operations in the same order as the direct definitions
// (expose, predict, value_at); in FP64, whose operations bound the kernel, the
// predictions go direction by direction (child()).
// The tiles of levels lo..hi are distributed over the CTAs of the launch; smem
// is the dynamic shared memory of TileShape::SMEM bytes.  Called by
// k_stage_tile and by the persistent macro-step kernel.
//
// EARLY (k_stage_tile): phases 1 and 2 read nothing but the tree, so they run
// before the wait for the predecessor's results where the tree is visible by
// then (tree_enter).  The first tile's status trips, masks and lookups thus
// overlap the predecessor.  CTAs that start early land on SMs unevenly, so a
// launch with more tiles than CTAs hands out those after every CTA's first by a
// counter, in the order the CTAs ask (tiles fixed to CTAs made an early start 10%
// slower).  Every launch of a captured piece has a counter of its own, 0 since
// before the piece, and asks before the wait; direct launches share one, ask
// after the wait, and the CTA that takes the last ticket clears it for the next.
template <int EQ, int D, class R, bool EARLY>
__device__ __forceinline__ void stage_tiles(const Grid& g, int lo, int hi, int s, int lmin, double bstage, int reg,
                                            const TreeSync& sync, int tick, unsigned char* smem)
{
    bool waited = !EARLY || tree_enter<D>(g, sync);
    const bool halt = halted(g); // with the loads below in one trip
    // the fine step, set by a launch of its own before the macro step's pieces;
    // direct launches publish it like a tree (on a tree of one level a stage may
    // follow directly on the launch that sets the step)
    const double dt = *g.dtp;
    using S = TileShape<EQ, D, R>;
    using Bits = typename Tile<D>::Bits;
    constexpr int M = S::M, TX = S::TX, TY = S::TY, TZ = S::TZ, NT = S::NT, H = S::H, NC = S::NC;
    constexpr int BX = S::BX, BY = S::BY, BZ = S::BZ, NB = S::NB, NBP = S::NBP, NR = S::NR;
    constexpr int NFX = S::NFX, NFY = S::NFY, NF = S::NF, RFX = S::RFX, RFY = S::RFY, NFR = S::NFR;
    constexpr int PBX = S::PBX, PBY = S::PBY, PBZ = S::PBZ, PB = S::PB, NPF = S::NPF;
    constexpr int NTS = 1 << (D - 1); // sub-faces per face
    constexpr int OUT = 3;            // status code of a cell past a wall
    constexpr int SY = BX, SZ = BX * BY;      // block strides in y and z
    constexpr int PSY = PBX, PSZ = PBX * PBY; // parent-block strides
    constexpr int NW = (NB + 31) / 32;        // words of a bit set over the block
    constexpr int PER = (NC * M + NT - 1) / NT; // (leaf, variable) pairs of a thread at most
    R (*sW)[NBP] = reinterpret_cast<R (*)[NBP]>(smem);
    R (*sP)[NBP] = reinterpret_cast<R (*)[NBP]>(smem + sizeof(R) * M * NBP);
    R (*sPW)[PB] = reinterpret_cast<R (*)[PB]>(smem + sizeof(R) * M * 2 * NBP);
    // x faces [0, NFX), y faces [NFX, NFX + NFY), z faces [NFX + NFY, NF)
    R (*sF)[NF] = reinterpret_cast<R (*)[NF]>(smem + sizeof(R) * M * (2 * NBP + PB));
    R (*sFine)[M][NPF] = reinterpret_cast<R (*)[M][NPF]>(smem + sizeof(R) * M * (2 * NBP + PB + NF));
    __shared__ unsigned sWord[2][NW + 1];   // leaves, internal nodes of the block as bits
    __shared__ Bits sTile[NR], sFacing[NR]; // per row: tile leaves, those facing an internal node
    __shared__ Bits sStored[NR], sVirt[NR]; // per row: needed cells
    __shared__ Bits sPlain[NFR];            // per row of faces: plain faces
    __shared__ short sTileAt[NR], sStoredAt[NR], sVirtAt[NR], sPlainAt[NFR]; // their places in the lists
    __shared__ unsigned sPar[PBY * PBZ];    // per row of the parent block: cells read by predictions
    __shared__ int sCount[5];               // stored, virtual, tile leaves, sub-faced, plain faces
    __shared__ uint8_t sSt[NB], sPSt[PB], sPNeg[PB];
    __shared__ int sSlot[NB], sPSlot[PB];
    __shared__ short sList[NB], sLeaf[NC];  // stored then virtual cells; tile leaves
    __shared__ int sFace[NF];               // sub-faced then plain: face | lo cell << 10 | direction << 20 | leaf is lo << 22

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // The CTA walks the active tiles (tiles holding a leaf) of levels lo..hi,
    // in level order; one launch may cover several independent levels.
    int ntask = 0;
    for (int l = lo; l <= hi; ++l) ntask += g.counts[2 * (LMAX + 1) + l];
    // the first tile of a one-level launch comes with the counts (its list has
    // an entry for every tile of the level)
    const bool one = lo == hi && (int)blockIdx.x < g.ntx[lo] * g.nty[lo] * g.ntz[lo];
    const int tile0 = one ? g.tlist[g.toff[lo] + blockIdx.x] : 0;
    if (halt) ntask = 0;
    const bool handed = EARLY && ntask > (int)gridDim.x; // tiles beyond the first by tickets
    __shared__ int sNext;
    for (int task = blockIdx.x; task < ntask;) {
    int u = lo, at = task;
    for (int c; at >= (c = g.counts[2 * (LMAX + 1) + u]); ++u) at -= c;
    const int tile = one && task == (int)blockIdx.x ? tile0 : g.tlist[g.toff[u] + at];
    const int n = g.n[u];
    const int ntx = g.ntx[u], nty = g.nty[u];
    const int ox = (tile % ntx) * TX;
    const int oy = D > 1 ? ((tile / ntx) % nty) * TY : 0;
    const int oz = D > 2 ? (tile / (ntx * nty)) * TZ : 0;
    const Ctx x{u, s, lmin};
    const bool finer = u < g.L;   // internal nodes of level u have children
    const bool pstage = u > g.lb; // a parent level exists
    // parent-block origin (level u-1 coordinates, before wrapping)
    const int pox = (ox >> 1) - 2, poy = D > 1 ? (oy >> 1) - 2 : 0, poz = D > 2 ? (oz >> 1) - 2 : 0;

    // 1. status and slot of the tile, its ring and the parent-level block
#pragma unroll
    for (int b0 = 0; b0 < NW * 32; b0 += NT) {
        const int b = b0 + tid;
        int st = 0, sl = -1;
        if (b < NB) {
            const int bx = b % BX, by = (b / BX) % BY, bz = b / SZ;
            int qx, qy = 0, qz = 0;
            const bool inb = in_box(g, u, 0, ox + bx - H, &qx) && (D < 2 || in_box(g, u, 1, oy + by - H, &qy)) &&
                             (D < 3 || in_box(g, u, 2, oz + bz - H, &qz));
            st = OUT;
            if (inb) {
                const long long id = cell_id(g, u, qx, qy, qz);
                st = status(g, u, id);
                sl = slot_of(g, u, id);
            }
            sSt[b] = (uint8_t)st;
            sSlot[b] = sl;
        }
        if (b0 + 32 * warp < NW * 32) {
            const unsigned wl = __ballot_sync(0xffffffffu, st == 1), wi = __ballot_sync(0xffffffffu, st == 2);
            if (lane == 0) {
                sWord[0][b >> 5] = wl;
                sWord[1][b >> 5] = wi;
            }
        }
    }
    if (pstage)
        for (int pb = tid; pb < PB; pb += NT) {
            const int i = pb % PBX, j = (pb / PBX) % PBY, kk = pb / PSZ;
            int neg = 0;
            const int px = wrap_or_mirror(g, u - 1, 0, pox + i, neg);
            const int py = D > 1 ? wrap_or_mirror(g, u - 1, 1, poy + j, neg) : 0;
            const int pz = D > 2 ? wrap_or_mirror(g, u - 1, 2, poz + kk, neg) : 0;
            const long long pid = cell_id(g, u - 1, px, py, pz);
            sPSt[pb] = status(g, u - 1, pid);
            sPSlot[pb] = slot_of(g, u - 1, pid);
            sPNeg[pb] = (uint8_t)neg;
        }
    if (tid < PBY * PBZ) sPar[tid] = 0;
    if (tid == 0) sWord[0][NW] = sWord[1][NW] = 0;
    __syncthreads();
    if (handed && tid == 0 && tick != kDirectTick) sNext = (int)(gridDim.x + atomicAdd(&g.built[tick], 1u));

    // 2. row masks.  row(k, by, bz): the leaves (k = 0) or internal nodes (1)
    // of a row of the block, empty past it; tile_row: the tile's leaves in it
    auto row = [&](int k, int by, int bz) -> Bits {
        if (by < 0 || by >= BY || bz < 0 || bz >= BZ) return 0;
        const int o = (bz * BY + by) * BX;
        if constexpr (D == 1) return sWord[k][0] | (Bits)sWord[k][1] << 32;
        else return __funnelshift_r(sWord[k][o >> 5], sWord[k][(o >> 5) + 1], o & 31) & ((1u << BX) - 1u);
    };
    const int tw = n - ox < TX ? n - ox : TX; // a level may be smaller than a tile
    const Bits xmask = (((Bits)1 << tw) - 1) << H;
    auto tile_row = [&](int by, int bz) -> Bits {
        if (D > 1 && (by < H || by >= H + TY || oy + by - H >= n)) return 0;
        if (D > 2 && (bz < H || bz >= H + TZ || oz + bz - H >= n)) return 0;
        return row(0, by, bz) & xmask;
    };
    if (tid < NR) { // tile leaves, and those with an internal node across a face
        const int by = tid % BY, bz = tid / BY;
        const Bits t = tile_row(by, bz);
        Bits in = 0;
        if (finer && t) {
            const Bits m = row(1, by, bz);
            in = m << 1 | m >> 1;
            if (D > 1) in |= row(1, by - 1, bz) | row(1, by + 1, bz);
            if (D > 2) in |= row(1, by, bz - 1) | row(1, by, bz + 1);
        }
        sTile[tid] = t;
        sFacing[tid] = t & in;
    } else if (warp == NT / 32 - 1) { // faces, by the last warp
        constexpr int RPL = (NFR + 31) / 32; // rows per lane
        Bits sub[RPL], islo[RPL];
        int cnt = 0; // sub-faced | plain << 16
#pragma unroll
        for (int k = 0; k < RPL; ++k) {
            const int q = lane * RPL + k;
            sub[k] = islo[k] = 0;
            if (q >= NFR) continue;
            Bits tl, th, il, ih; // tile leaves and internal nodes on the low and high side
            if (q < RFX) {
                const int by = D > 1 ? H + q % TY : 0, bz = D > 2 ? H + q / TY : 0;
                const Bits t = tile_row(by, bz), m = row(1, by, bz);
                constexpr Bits full = ((Bits)1 << (TX + 1)) - 1;
                tl = t >> (H - 1) & full;
                th = t >> H & full;
                il = m >> (H - 1);
                ih = m >> H;
            } else {
                const bool isy = D < 3 || q < RFX + RFY;
                const int r = isy ? q - RFX : q - RFX - RFY;
                const int hy = isy ? H + r % (TY + 1) : H + r % TY, ly = isy ? hy - 1 : hy;
                const int hz = D < 3 ? 0 : H + r / (isy ? TY + 1 : TY), lz = isy ? hz : hz - 1;
                tl = tile_row(ly, lz) >> H;
                th = tile_row(hy, hz) >> H;
                il = row(1, ly, lz) >> H;
                ih = row(1, hy, hz) >> H;
            }
            if (finer) {
                islo[k] = tl & ih;
                sub[k] = islo[k] | (th & il);
            }
            const Bits plain = (tl | th) & ~sub[k];
            sPlain[q] = plain;
            cnt += popc(sub[k]) | popc(plain) << 16;
        }
        int inc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        const int nsb = __shfl_sync(0xffffffffu, inc, 31) & 0xffff;
        int ps = (inc - cnt) & 0xffff, pp = (inc - cnt) >> 16;
#pragma unroll
        for (int k = 0; k < RPL; ++k) {
            const int q = lane * RPL + k;
            if (q >= NFR) continue;
            sPlainAt[q] = (short)(nsb + pp);
            pp += popc(sPlain[q]);
            const bool isx = q < RFX, isy = D > 1 && !isx && (D < 3 || q < RFX + RFY);
            for (Bits m = sub[k]; m; m &= m - 1) {
                const int i = first_bit(m);
                int f, lc; // face and its low cell
                if (isx) {
                    f = i + (TX + 1) * q;
                    lc = (D > 2 ? H + q / TY : 0) * SZ + (D > 1 ? H + q % TY : 0) * SY + H + i - 1;
                } else if (isy) {
                    const int r = q - RFX;
                    f = NFX + i + TX * r;
                    lc = (D > 2 ? H + r / (TY + 1) : 0) * SZ + (H + r % (TY + 1) - 1) * SY + H + i;
                } else {
                    const int r = q - RFX - RFY;
                    f = NFX + NFY + i + TX * r;
                    lc = (H + r / TY - 1) * SZ + (H + r % TY) * SY + H + i;
                }
                sFace[ps++] = f | lc << 10 | (isx ? 0 : (isy ? 1 : 2)) << 20 | (int)(islo[k] >> i & 1) << 22;
            }
        }
        if (lane == 31) {
            sCount[3] = nsb;
            sCount[4] = inc >> 16;
        }
    }
    __syncthreads();
    const int nsb = sCount[3], nfl = sCount[4];
    const int nsub = nsb * NTS; // sub-face tasks come first; NTS divides 32

    // the finer-side cells (r = 0, 1) of sub-face task k: in-box coordinates, or
    // the leaf's side of the face and its cell
    struct Sub {
        int k, bl, side, t;
        int c[3];
    };
    auto sub_task = [&](int task) -> Sub {
        const int e = sFace[task / NTS];
        Sub z;
        z.t = task % NTS;
        z.k = e >> 20 & 3;
        const int lc = e >> 10 & 1023;
        z.side = e >> 22 ? 1 : -1;
        z.bl = e >> 22 ? lc : lc + (z.k == 0 ? 1 : (z.k == 1 ? SY : SZ)); // the leaf
        z.c[0] = ox + z.bl % BX - H;
        z.c[1] = D > 1 ? oy + (z.bl / BX) % BY - H : 0;
        z.c[2] = D > 2 ? oz + z.bl / SZ - H : 0;
        return z;
    };
    // stencil cell i = 0..3 across the face on level u+1
    auto sub_cell = [&](const Sub& z, int i, int p[3]) {
        const int j1 = z.k == 0 ? 1 : 0, j2 = z.k == 2 ? 1 : 2;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            p[j] = 0;
            if (j >= D) continue;
            if (j == z.k) p[j] = 2 * z.c[j] + (z.side > 0 ? i : i - 2);
            else if (j == j1) p[j] = 2 * z.c[j] + (z.t & 1);
            else if (j == j2) p[j] = 2 * z.c[j] + (z.t >> 1);
        }
    };
    int fst[2] = {0, 0}, fsl[2] = {-1, -1}, fneg[2] = {0, 0}; // status, slot and mirror parity of this thread's finer cells
    const int ftask = tid - 32;                               // its sub-face task
    const bool fetch = ftask >= 0 && ftask < NPF && ftask < nsub;
    if (warp == 0) { // needed cells, by the first warp
        constexpr int RPL = (NR + 31) / 32;
        int cnt = 0, nlf = 0; // stored | virtual << 16; tile leaves
        constexpr Bits full = BX == 8 * sizeof(Bits) ? ~(Bits)0 : ((Bits)1 << BX) - 1;
#pragma unroll
        for (int k = 0; k < RPL; ++k) {
            const int r = lane * RPL + k;
            if (r >= NR) continue;
            const int by = r % BY, bz = r / BY;
            const Bits t = sTile[r];
            Bits need = t | t << 1 | t >> 1 | t << 2 | t >> 2;
#pragma unroll
            for (int d = -2; d <= 2; ++d) {
                if (d == 0) continue;
                if (D > 1 && by + d >= 0 && by + d < BY) need |= sTile[r + d];
                if (D > 2 && bz + d >= 0 && bz + d < BZ) need |= sTile[r + d * BY];
            }
            if (finer) {
#pragma unroll
                for (int dz = (D > 2 ? -1 : 0); dz <= (D > 2 ? 1 : 0); ++dz)
#pragma unroll
                    for (int dy = (D > 1 ? -1 : 0); dy <= (D > 1 ? 1 : 0); ++dy) {
                        if (by + dy < 0 || by + dy >= BY || bz + dz < 0 || bz + dz >= BZ) continue;
                        const Bits m = sFacing[r + dy + dz * BY];
                        need |= m | m << 1 | m >> 1;
                    }
            }
            need &= full;
            const Bits there = row(0, by, bz) | row(1, by, bz);
            sStored[r] = need & there;
            sVirt[r] = need & ~there;
            cnt += popc(need & there) | popc(need & ~there) << 16;
            nlf += popc(t);
            // parents of the virtual cells: cell column bx reads the columns
            // bx/2 .. bx/2 + 2 of the parent block, likewise for the rows
            Bits h = need & ~there;
            if (pstage && h) {
                unsigned ph = 0;
#pragma unroll
                for (int j = 0; j < BX / 2; ++j) ph |= (unsigned)((h >> (2 * j) & 3) != 0) << j;
                ph |= ph << 1 | ph << 2;
#pragma unroll
                for (int dz = 0; dz < (D > 2 ? 3 : 1); ++dz)
#pragma unroll
                    for (int dy = 0; dy < (D > 1 ? 3 : 1); ++dy)
                        atomicOr(&sPar[(D > 1 ? (by >> 1) + dy : 0) + (D > 2 ? (bz >> 1) + dz : 0) * PBY], ph);
            }
        }
        int inc = cnt, incl = nlf;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o), z = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) {
                inc += y;
                incl += z;
            }
        }
        const int nst = __shfl_sync(0xffffffffu, inc, 31) & 0xffff;
        int as = (inc - cnt) & 0xffff, av = nst + ((inc - cnt) >> 16), al = incl - nlf;
#pragma unroll
        for (int k = 0; k < RPL; ++k) {
            const int r = lane * RPL + k;
            if (r >= NR) continue;
            sStoredAt[r] = (short)as;
            sVirtAt[r] = (short)av;
            sTileAt[r] = (short)al;
            as += popc(sStored[r]);
            av += popc(sVirt[r]);
            al += popc(sTile[r]);
        }
        if (lane == 31) {
            sCount[0] = nst;
            sCount[1] = inc >> 16;
            sCount[2] = incl;
            if (s == 1) atomicAdd(g.updates, (unsigned long long)incl);
            atomicAdd(&g.work[u * 4 + s], (unsigned long long)incl);
        }
    } else { // meanwhile: the plain faces' list, status and slot of the finer-side cells
        if (fetch) {
            const Sub z = sub_task(ftask);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                int p[3], q[3] = {0, 0, 0};
                sub_cell(z, z.side > 0 ? 2 + r : r, p); // the cells on the internal node's side
#pragma unroll
                for (int j = 0; j < D; ++j) q[j] = wrap_or_mirror(g, u + 1, j, p[j], fneg[r]);
                const long long id = cell_id(g, u + 1, q[0], q[1], q[2]);
                fst[r] = status(g, u + 1, id);
                fsl[r] = slot_of(g, u + 1, id);
            }
        }
        for (int f = tid - 32; f < NF; f += NT - 32) {
            int q, i, k, lc;
            if (f < NFX) {
                q = f / (TX + 1);
                i = f % (TX + 1);
                k = 0;
                lc = (D > 2 ? H + q / TY : 0) * SZ + (D > 1 ? H + q % TY : 0) * SY + H + i - 1;
            } else if (D < 3 || f < NFX + NFY) {
                const int r = (f - NFX) / TX;
                q = RFX + r;
                i = (f - NFX) % TX;
                k = 1;
                lc = (D > 2 ? H + r / (TY + 1) : 0) * SZ + (H + r % (TY + 1) - 1) * SY + H + i;
            } else {
                const int r = (f - NFX - NFY) / TX;
                q = RFX + RFY + r;
                i = (f - NFX - NFY) % TX;
                k = 2;
                lc = (H + r / TY - 1) * SZ + (H + r % TY) * SY + H + i;
            }
            const Bits m = sPlain[q];
            if (m >> i & 1) sFace[sPlainAt[q] + popc(m & (((Bits)1 << i) - 1))] = f | lc << 10 | k << 20;
        }
    }
    __syncthreads();
    if (!waited) { // from here on values are read
        pdl_enter();
        waited = true;
    }
    if (handed && tid == 0 && tick == kDirectTick) {
        const int ticket = (int)atomicAdd(&g.built[tick], 1u);
        if (ticket == ntask - 1) g.built[tick] = 0;
        sNext = (int)gridDim.x + ticket;
    }
    const double dtl = g.gts ? dt : ldexp(dt, g.L - u); // Eq. 13 step of level u
    const double bw = dtl * bstage; // register weight dt_l b_s
    const int nst = sCount[0], nvc = sCount[1], nlf = sCount[2];

    // 3. one trip: exposures of stored and parent cells and of the finer-side
    //    cells; the lists of cells.  On its own level a node exposes the
    //    stage's own field (q^n, q*, q**).
    const int own = s == 1 ? F_Q0 : (s == 2 ? F_Q1 : F_Q2);
    for (int b = tid; b < NB; b += NT) {
        const int r = b / BX, i = b % BX;
        const Bits below = ((Bits)1 << i) - 1;
        const Bits ms = sStored[r], mv = sVirt[r], mt = sTile[r];
        if (ms >> i & 1) {
            R W[M];
            load_row<M, R>(nd<R>(g, own, sSlot[b]), W);
            sList[sStoredAt[r] + popc(ms & below)] = (short)b;
#pragma unroll
            for (int v = 0; v < M; ++v) sW[v][b] = W[v];
        }
        if (mv >> i & 1) sList[sVirtAt[r] + popc(mv & below)] = (short)b;
        if (mt >> i & 1) sLeaf[sTileAt[r] + popc(mt & below)] = (short)b;
    }
    if (pstage)
        for (int pb = tid; pb < PB; pb += NT) {
            const int st = sPSt[pb];
            if (!(sPar[pb / PBX] >> (pb % PBX) & 1) || st == 0) continue; // an absent source is flagged when it is read
            R W[M];
            expose<M, R, R>(g, x, u - 1, sPSlot[pb], st, W);
            // an odd-mirror ghost enters negated: (-w) v = w (-v) exactly
            const bool neg = sPNeg[pb] != 0;
#pragma unroll
            for (int v = 0; v < M; ++v) sPW[v][pb] = neg ? -W[v] : W[v];
        }
    if (fetch) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            R W[M];
            if (fst[r] == 0) { // absent: predicted (flags the missing source)
                const Sub z = sub_task(ftask);
                int p[3];
                sub_cell(z, z.side > 0 ? 2 + r : r, p);
                R far[M];
                far_value<D, M, R>(g, x, u + 1, p[0], p[1], p[2], far);
#pragma unroll
                for (int v = 0; v < M; ++v) W[v] = far[v];
            } else {
                finer_exposure<M, R>(g, x, fst[r], fsl[r], W);
                if (fneg[r]) {
#pragma unroll
                    for (int v = 0; v < M; ++v) W[v] = -W[v];
                }
            }
            R P[M];
            recon_vars<EQ, D, M, R>(g, W, P);
#pragma unroll
            for (int v = 0; v < M; ++v) sFine[r][v][ftask] = P[v];
        }
    }
    __syncthreads();

    // q^n of the leaves this thread updates in phase 6 (one variable each),
    // on its way while the next phases compute
    R q0r[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int t = tid + k * NT;
        q0r[k] = R(0);
        if (s >= 2 && t < nlf * M) q0r[k] = nd<R>(g, F_Q0, sSlot[sLeaf[t / M]])[t % M];
    }

    // 4. virtual cells: predicted from the parent block (the terms of
    //    predict() in its order), or a stored mirror image, else value_at();
    //    reconstruction variables of all needed cells
    for (int t = tid; t < nst + nvc; t += NT) {
        const int e = t < nvc ? nst + t : t - nvc; // virtual cells, the longer tasks, first
        const int b = sList[e];
        R W[M];
        if (t < nvc) {
            int pc[3] = {b % BX, (b / BX) % BY, b / SZ}; // the block cell whose parents predict
            int neg = 0;
            bool predicted = pstage, copied = false;
            int bq = b;
            if (sSt[b] == OUT) { // a ghost: its mirror image, if that is in the block
                const int o3[3] = {ox, oy, oz}, B3[3] = {BX, BY, BZ}, bs3[3] = {1, SY, SZ};
                bq = 0;
                bool inb = true;
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    const int q = wrap_or_mirror(g, u, k, o3[k] + pc[k] - H, neg);
                    if (g.bc[k] != 0) pc[k] = q - o3[k] + H; // a periodic direction keeps the block cell
                    inb = inb && pc[k] >= 0 && pc[k] < B3[k];
                    bq += pc[k] * bs3[k];
                }
                predicted = copied = false;
                if (inb) {
                    predicted = pstage && (sVirt[bq / BX] >> (bq % BX) & 1) && sSt[bq] == 0;
                    copied = sStored[bq / BX] >> (bq % BX) & 1;
                }
            }
            if (predicted) {
                const int pb0 = (D > 2 ? (pc[2] >> 1) * PSZ : 0) + (D > 1 ? (pc[1] >> 1) * PSY : 0) + (pc[0] >> 1);
                const int a0 = pc[0] & 1, a1 = pc[1] & 1, a2 = pc[2] & 1;
                if constexpr (sizeof(R) == 8) {
                    bool missing = false;
#pragma unroll
                    for (int v = 0; v < M; ++v) {
                        R z3[3];
#pragma unroll
                        for (int dz = 0; dz < (D > 2 ? 3 : 1); ++dz) {
                            R y3[3];
#pragma unroll
                            for (int dy = 0; dy < (D > 1 ? 3 : 1); ++dy) {
                                const int pb = pb0 + dz * PSZ + dy * PSY;
                                if (v == 0) missing = missing || !sPSt[pb] || !sPSt[pb + 1] || !sPSt[pb + 2];
                                y3[dy] = child(sPW[v][pb], sPW[v][pb + 1], sPW[v][pb + 2], a0);
                            }
                            z3[dz] = D > 1 ? child(y3[0], y3[1], y3[2], a1) : y3[0];
                        }
                        W[v] = D > 2 ? child(z3[0], z3[1], z3[2], a2) : z3[0];
                    }
                    if (missing) atomicOr(g.err, ERR_SOURCE);
                } else {
#pragma unroll
                    for (int v = 0; v < M; ++v) W[v] = R(0);
#pragma unroll(D > 2 ? 1 : 3)
                    for (int dz = (D > 2 ? -1 : 0); dz <= (D > 2 ? 1 : 0); ++dz) {
                        const R wz = D > 2 ? R(pw(a2, dz)) : R(1);
#pragma unroll(D > 2 ? 1 : 3)
                        for (int dy = (D > 1 ? -1 : 0); dy <= (D > 1 ? 1 : 0); ++dy) {
                            const R wyz = wz * (D > 1 ? R(pw(a1, dy)) : R(1));
#pragma unroll
                            for (int dxx = -1; dxx <= 1; ++dxx) {
                                const int pb = pb0 + (D > 2 ? (dz + 1) * PSZ : 0) + (D > 1 ? (dy + 1) * PSY : 0) + dxx + 1;
                                if (sPSt[pb] == 0) {
                                    atomicOr(g.err, ERR_SOURCE);
                                    continue;
                                }
                                const R w0 = wyz * R(pw(a0, dxx));
#pragma unroll
                                for (int v = 0; v < M; ++v) W[v] += w0 * sPW[v][pb];
                            }
                        }
                    }
                }
                if (neg) {
#pragma unroll
                    for (int v = 0; v < M; ++v) W[v] = -W[v];
                }
            } else if (copied) { // a ghost whose mirror image is a staged stored cell
#pragma unroll
                for (int v = 0; v < M; ++v) W[v] = neg ? -sW[v][bq] : sW[v][bq];
            } else {
                const int p[3] = {ox + b % BX - H, D > 1 ? oy + (b / BX) % BY - H : 0, D > 2 ? oz + b / SZ - H : 0};
                R far[M];
                far_value<D, M, R>(g, x, u, p[0], p[1], p[2], far);
#pragma unroll
                for (int v = 0; v < M; ++v) W[v] = far[v];
            }
#pragma unroll
            for (int v = 0; v < M; ++v) sW[v][b] = W[v];
        } else {
#pragma unroll
            for (int v = 0; v < M; ++v) W[v] = sW[v][b];
        }
        R P[M];
        recon_vars<EQ, D, M, R>(g, W, P);
#pragma unroll
        for (int v = 0; v < M; ++v) sP[v][b] = P[v];
    }
    __syncthreads();

    // 5. the faces touching a tile leaf, one pass: faces of a leaf against an
    //    internal node (2^{d-1} sub-face tasks each, in adjacent lanes), then
    //    plain faces on level u, one thread per face
    for (int base = 0; base < nsub + nfl; base += NT) {
        const int task = base + tid;
        const bool isSub = task < nsub, act = task < nsub + nfl;
        const int e = act && !isSub ? sFace[nsb + task - nsub] : (act ? sFace[task / NTS] : 0);
        const int f = e & 1023;
        const int t = isSub ? task % NTS : 0;
        R F[M];
#pragma unroll
        for (int v = 0; v < M; ++v) F[v] = R(0);
        if (act) {
            const int k = e >> 20 & 3;
            if (!isSub) {
                const int lc = e >> 10 & 1023;
                const int stride = k == 0 ? 1 : (k == 1 ? SY : SZ);
                flux_recon<EQ, D, M, R>(g, k, g.dx[u][k], [&](int c, int v) { return sP[v][lc + (c - 1) * stride]; },
                                        F);
            } else {
                // stencil on level u+1: the leaf's own children (virtual, predicted;
                // low and high) and the two cells of the finer side
                const Sub z = sub_task(task);
                R Pc[2][M], Pf[2][M];
                if constexpr (sizeof(R) == 8) {
                    const int sk = k == 0 ? 1 : (k == 1 ? SY : SZ); // strides along the face's normal
                    const int s1 = k == 0 ? SY : 1, s2 = k == 2 ? SY : SZ; // and its tangential directions
                    R W[2][M];
#pragma unroll
                    for (int v = 0; v < M; ++v) {
                        R c3[3];
#pragma unroll
                        for (int i = 0; i < 3; ++i) {
                            const R* w = &sW[v][z.bl + (i - 1) * sk];
                            if constexpr (D == 1) {
                                c3[i] = w[0];
                            } else if constexpr (D == 2) {
                                c3[i] = child(w[-s1], w[0], w[s1], z.t);
                            } else {
                                R y3[3];
#pragma unroll
                                for (int j = 0; j < 3; ++j) {
                                    const R* y = w + (j - 1) * s2;
                                    y3[j] = child(y[-s1], y[0], y[s1], z.t & 1);
                                }
                                c3[i] = child(y3[0], y3[1], y3[2], z.t >> 1);
                            }
                        }
                        const R d = c3[2] - c3[0];
                        W[0][v] = fma(-0.125, d, c3[1]);
                        W[1][v] = fma(0.125, d, c3[1]);
                    }
                    recon_vars<EQ, D, M, R>(g, W[0], Pc[0]);
                    recon_vars<EQ, D, M, R>(g, W[1], Pc[1]);
                } else {
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        int p[3];
                        sub_cell(z, z.side > 0 ? r : 2 + r, p);
                        R W[M];
                        const int ax = p[0] & 1, ay = p[1] & 1, az = p[2] & 1;
#pragma unroll
                        for (int v = 0; v < M; ++v) W[v] = R(0);
#pragma unroll
                        for (int dz = (D > 2 ? -1 : 0); dz <= (D > 2 ? 1 : 0); ++dz)
#pragma unroll
                            for (int dy = (D > 1 ? -1 : 0); dy <= (D > 1 ? 1 : 0); ++dy)
#pragma unroll
                                for (int dx = -1; dx <= 1; ++dx) {
                                    const R w = R((D > 2 ? pw(az, dz) : 1.0) * (D > 1 ? pw(ay, dy) : 1.0)) *
                                                R(pw(ax, dx));
                                    const int bs = z.bl + dz * SZ + dy * SY + dx;
#pragma unroll
                                    for (int v = 0; v < M; ++v) W[v] += w * sW[v][bs];
                                }
                        recon_vars<EQ, D, M, R>(g, W, Pc[r]);
                    }
                }
                if (task < NPF) { // finer side fetched in phase 3
#pragma unroll
                    for (int r = 0; r < 2; ++r)
#pragma unroll
                        for (int v = 0; v < M; ++v) Pf[r][v] = sFine[r][v][task];
                } else {
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        int p[3];
                        sub_cell(z, z.side > 0 ? 2 + r : r, p);
                        R far[M];
                        far_value<D, M, R>(g, x, u + 1, p[0], p[1], p[2], far);
                        recon_vars<EQ, D, M, R>(g, far, Pf[r]);
                    }
                }
                const bool up = z.side > 0;
                flux_recon<EQ, D, M, R>(
                    g, k, g.dx[u + 1][k],
                    [&](int c, int v) { return c < 2 ? (up ? Pc[c][v] : Pf[c][v]) : (up ? Pf[c - 2][v] : Pc[c - 2][v]); },
                    F);
            }
        }
        // mean of the sub-face fluxes of a face: in the warps that hold any (their
        // every lane takes part in the shuffles; plain faces keep their own flux)
        if (NTS > 1 && base + 32 * warp < nsub) {
#pragma unroll
            for (int v = 0; v < M; ++v) {
                R sum = F[v] + __shfl_xor_sync(0xffffffffu, F[v], 1);
                if (NTS == 4) sum += __shfl_xor_sync(0xffffffffu, sum, 2);
                if (isSub) F[v] = sum * R(1.0 / NTS);
            }
        }
        if (act && t == 0) {
#pragma unroll
            for (int v = 0; v < M; ++v) sF[v][f] = F[v];
        }
    }
    __syncthreads();

    // 6. compact RK update of the tile's leaves, and the flux registers
    //    (conservation across levels): dt_l b_s F at coarse-fine faces
#pragma unroll
    for (int kk = 0; kk < PER; ++kk) {
        const int t = tid + kk * NT;
        if (t >= nlf * M) break;
        const int b = sLeaf[t / M], v = t % M;
        const int i = b % BX - H, j = D > 1 ? (b / BX) % BY - H : 0, kz = D > 2 ? b / SZ - H : 0;
        const int sl = sSlot[b];
        const R self = sW[v][b];
        const R q0p = s >= 2 ? q0r[kk] : self; // the stage value is the staged exposure
        R f = R(0);
#pragma unroll
        for (int k = 0; k < D; ++k) {
            const int stride = k == 0 ? 1 : (k == 1 ? SY : SZ);
            int fm, fp;
            if (k == 0) {
                fm = i + (TX + 1) * (j + TY * kz);
                fp = fm + 1;
            } else if (k == 1) {
                fm = NFX + i + TX * (j + (TY + 1) * kz);
                fp = fm + TX;
            } else {
                fm = NFX + NFY + i + TX * (j + TY * kz);
                fp = fm + TX * TY;
            }
            const R Fm = sF[v][fm], Fp = sF[v][fp];
            const R idx = R(g.rdx[u][k]);
            if (EQ == 3 && k == 0) { // the reaction k u (1 - u) (u - a)
                f = fma(R(g.phys[1]) * self * (R(1) - self), self - R(g.phys[2]), mul_rn(Fm - Fp, idx));
            } else {
                f = fma(Fm - Fp, idx, f);
            }
            if (reg) {
                // a face to another level: a coarser leaf (absent here), or an
                // internal node (finer leaves; on the finest level there is none)
                double* rg = regs(g.rg, g, sl) + 2 * k * M + v;
                const int sm = sSt[b - stride], sp = sSt[b + stride];
                if (sm == 0 || (sm == 2 && finer)) rg[0] += bw * double(Fm);
                if (sp == 0 || (sp == 2 && finer)) rg[M] += bw * double(Fp);
            }
        }
        rk_update<M, R>(g, sl, v, s, R(dtl), f, q0p, self);
    }
    __syncthreads(); // shared arrays are reused by the next tile
    task = handed ? sNext : task + (int)gridDim.x;
    }
    if (!waited) pdl_enter(); // no tile: the kernels after this one rely on its wait
}

template <int EQ, int D, class R>
__global__ void __launch_bounds__(Tile<D>::THREADS, TileShape<EQ, D, R>::PERSM)
k_stage_tile(const __grid_constant__ Grid g, int lo, int hi, int s, int lmin, double bstage, int reg, TreeSync sync,
             int tick)
{
    extern __shared__ __align__(16) unsigned char smem[];
    stage_tiles<EQ, D, R, true>(g, lo, hi, s, lmin, bstage, reg, sync, tick, smem);
}

static inline int grid_for(const Grid& g, int l)
{
    long long b = (g.N[l] + NTHREADS - 1) / NTHREADS;
    return (int)(b < 1216 ? (b < 1 ? 1 : b) : 1216);
}

// One launch of the tiled stage kernel over the active tiles of levels lo..hi;
// the persistent grid is the device's resident capacity for this instantiation
// (occupancy API, once per device), capped by the tile count and by g.gcap
// when that is set.  Every cell's update and flux registers are written by one
// thread, so the result does not depend on the grid size or on which CTA
// takes a tile.
template <int EQ, int D, class R>
static int stage_dispatch(const Grid& g, cudaStream_t st, int lo, int hi, int s, int lmin, double b, int reg, TreeSync sync,
                          int tick)
{
    using S = TileShape<EQ, D, R>;
    constexpr int kMaxDev = 64;
    static int resident[kMaxDev] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return -1;
    if (!resident[dev]) {
        if (cudaFuncSetAttribute(k_stage_tile<EQ, D, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)S::SMEM) != cudaSuccess)
            return -1;
        int per_sm = 0, sms = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_stage_tile<EQ, D, R>, S::NT, S::SMEM) !=
                cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || per_sm < 1)
            return -1;
        resident[dev] = per_sm * sms;
    }
    if (lo > hi) return 0; // set-up only
    long long total = 0;
    for (int l = lo; l <= hi; ++l) total += (long long)g.ntx[l] * g.nty[l] * g.ntz[l];
    long long grid = total < resident[dev] ? total : resident[dev];
    if (g.gcap > 0 && grid > g.gcap) grid = g.gcap;
    if (grid < 1) grid = 1;
    if (pdl_launch(k_stage_tile<EQ, D, R>, dim3((unsigned)grid), dim3(S::NT), S::SMEM, st, g, lo, hi, s, lmin, b, reg,
                   sync, tick) !=
        cudaSuccess)
        return -1;
    return 1;
}

// stage launcher of one equation (all dimensions, both precisions); each is
// defined in its own translation unit so that they compile in parallel
template <int EQ>
int launch_stage_eq(const Grid& g, cudaStream_t st, int lo, int hi, int s, int lmin, double b, int reg, TreeSync sync,
                    int tick);
template <> int launch_stage_eq<0>(const Grid&, cudaStream_t, int, int, int, int, double, int, TreeSync, int);
template <> int launch_stage_eq<1>(const Grid&, cudaStream_t, int, int, int, int, double, int, TreeSync, int);
template <> int launch_stage_eq<2>(const Grid&, cudaStream_t, int, int, int, int, double, int, TreeSync, int);
template <> int launch_stage_eq<3>(const Grid&, cudaStream_t, int, int, int, int, double, int, TreeSync, int);

} // namespace mrlt
