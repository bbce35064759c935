// mrlt_tree.cuh -- host-side launcher of the tree kernels (private).
#pragma once
#include "mrlt_tree_dev.cuh"

namespace mrlt {

constexpr int MASS_BLOCKS = 64;

struct Launcher {
    Grid g;
    cudaStream_t st = nullptr;
    int* bc = nullptr; // compaction scratch, 2 ints per block over all levels
    long long n = 0;   // kernel launches issued
    // what the next kernel can rely on (see TreeSync)
    bool capturing = false;
    unsigned published[2] = {0, 0}; // publications, of the piece being captured and of direct launches
    bool stale = true;              // something to look up has changed since the last publication
    int stages = 0;                 // stage launches of the piece
    bool wait_first = false;        // one of many solvers that share the GPU

    // how the next kernel that looks the tree up enters
    TreeSync enter()
    {
        if (wait_first) return {kWait, 0, 0};
        const int word = capturing ? 0 : 1;
        if (!stale) return {capturing && !published[0] ? kVisible : kAcquire, word, published[word]};
        stale = false;
        return {kPublish, word, ++published[word]};
    }
    // the index of a stage launch's tile tickets in g.built
    int tick() { return capturing ? kFirstTick + stages++ : kDirectTick; }
    // a captured piece begins; ends, with the words of g.built that it used cleared
    void piece_begin();
    void piece_end();

    void project(int l, int mode);
    // levels hi..lo in fewer launches; level lo with mode top (mode if top < 0)
    void project_up(int hi, int lo, int mode, int top = -1);
    // an iteration begins: leaf copy of levels lmin..L, up-sweep of levels L-1..lo
    // (level lo with mode top); next: it is not the macro step's first
    void begin(int lmin, bool next, int lo, int top);
    void leaf_copy(int lo, int hi, int from, int to); // leaves of levels lo..hi
    void mark_refinements(int la, bool check = false); // check that the tree fits (halt)
    void apply_tree(int la);
    void compact(int lo, int hi);                      // leaf / node / tile lists of levels lo..hi
    void reflux(int lo, int hi);                       // coarse levels lo..hi
    void scale();                                      // running max |q_v| over all leaves
    void scale_init();                                 // running max |q_v| := 1e-14
    void set_dt(double dt);                            // *g.dtp := dt, iteration 0
    void set_leaves(const int* keys, const double* vals, long long count); // leaf q^n and end values
    void store_finest(const double* src); // finest-level q^n from double data [v][cell]
    void slots_full(long long ntot);      // every cell of every level a node (a new solver's tree)
    // compacting copy of the nodes from `from` into the arrays of g (a new capacity)
    void renumber(const Grid& from, const int* counts_host, long long used);
    void count_refined(int la, int* out);   // *out = refinement flags of levels la..L-1
    void finite();                                     // all leaves
    void mass(int l, double* part);
    void pack(int* keys, double* vals);                // all leaves, in level and list order
    void uniform(double* T, uint8_t* us);
};

} // namespace mrlt
