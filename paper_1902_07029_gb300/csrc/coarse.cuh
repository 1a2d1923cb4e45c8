// The coarse levels of a V-cycle on the equation for s (schur.cuh) resident in
// the shared memory of one thread-block cluster, one launch per cycle.
//
// On levels of up to some ten thousand nodes every phase of the cycle (a
// colour, the ghosts, the defect, a transfer) is shorter as work than the
// launch and memory latency it pays as a kernel of its own (2.2 us in the
// 65^2 disk's cycle, 14 such phases per level).  Here the nodes of the levels
// l0 .. L-1 are dealt to the CTAs of a cluster in bands of the box order; each
// CTA keeps its rows, tables and values in shared memory, reads a neighbour's
// value from its owner's shared memory, and a cluster barrier separates the
// phases.  Levels too small for that (`narrow` nodes in build_coarse) run on CTA 0
// alone with CTA barriers.  The rows (gt, dd, 1/dd, rho, C) and the tables are fixed
// during a linear solve and are copied in while the previous kernel runs.
#pragma once

#include "schur.cuh"

namespace sulf {

constexpr int kCoarseThreads = 512;
constexpr int kCoarseMaxCta = 16;

// rows of one table, longest first, dealt to `nw` warps: job (u32) says a
// warp's rows and the lanes of each; idx (u16): the ghost of a row
struct CTab {
    int ptr, ref, val, idx, job;  // byte offsets
    int nw;
};

// one level as one CTA sees it: counts, byte offsets into its shared memory
// (values: the same in every CTA; the others its own)
struct CLev {
    int cr, cbn, cb, cg;  // own red nodes, black ones away from the ghosts, all black ones, ghosts
    int nr, nx;           // rows (cr + cb), nodes (nr + cg)
    int wide;             // dealt to all CTAs (else to CTA 0)
    int x, y, d2, b, snap;
    int coef;             // gt/dd[2D][nr], dd[nr], 1/dd[nr], rho[nx], C[nx]
    int nbr;              // u16 [2D][nr]
    CTab g;               // composed ghost rows: owner << kAddrBits | byte offset of the value
    CTab r;               // ghost rows of the defect
    int pro;              // u16 [2^D][cb + cg]: coarse corners
    int cptr, cref, cval;  // rows of the restriction onto the own inside nodes
    CTab c;               // and onto the own ghosts
    int ainv;             // coarsest level: own rows of the inverse (-1: in global memory)
    int m;                // coarsest level: order of the matrix
};

template <typename T>
struct CDesc {
    const char* head;       // per CTA: its levels (CLev), then the program
    int head_len, nop;
    const char* tab;        // tables, per CTA from tab_off[cta]
    const T* coef;          // rows, per CTA from coef_off[cta]
    const T* ainv;
    T* b;                   // right-hand side of the first level, per CTA from b_off[cta]
    const int* slot;        // slots of the first level's nodes, same order
    T* X;                   // the first level's x by slot
    double* acc;            // finest level of mixed precision: X is added to it (else null)
    const int* skip;        // the first level is the finest: X is its start, set: its first sweep is done (else null)
    const int* cnt_m;       // coarsest level: own nodes of each CTA
    int nlev;
    int ncta;
    int tab_off[kCoarseMaxCta], tab_len[kCoarseMaxCta];    // bytes
    int coef_off[kCoarseMaxCta], coef_len[kCoarseMaxCta];  // elements
    int ainv_off[kCoarseMaxCta], ainv_len[kCoarseMaxCta];  // elements copied into shared memory
    int b_off[kCoarseMaxCta];
    int tab_at, coef_at, ainv_at;  // where they go in shared memory (bytes)
};

// the fused levels of one handle and precision
template <typename T>
struct CoarseSet {
    int l0 = -1;
    int want = -2, nu1 = 0, nu2 = 0, max_cta = 0;  // what it was built for
    bool rows = false;      // built, and for the current boundary rows
    int own_want = -2, own = 0;  // lock step: the first level fused with no regard to the class, and what it was found for
    size_t smem = 0;
    int ncta = 0;
    bool wide = false;      // the first level is dealt to all CTAs (else CTA 0 runs it)
    CDesc<T>* dev = nullptr;
    CPerm* perm[SULF_MAXLEV] = {};  // device, per level
    T* coef = nullptr;
    T* b = nullptr;
    int* bpos = nullptr;    // list position -> position in b (level l0)
    int* cpos = nullptr;    // coarsest level: list position -> row of the inverse
    char* tab = nullptr;
    size_t tab_cap = 0, coef_cap = 0, b_cap = 0;
    int* slot = nullptr;
    char* head = nullptr;
    int* cnt_m = nullptr;
    std::vector<std::pair<void*, size_t>> kept;  // the uploaded arrays and their sizes
};

// (re)builds the set for levels l0 .. L-1 (the smallest l0 >= want that fits);
// l0 = -1 where none does
template <int D, typename T>
int build_coarse(CoarseSet<T>& S, const LevelGeo* G, const SGeo* SG, const SVec<T>* V, int L, int want, int nu1,
                 int nu2, int max_cta, double* acc, const int* skip, DevMem& mem, cudaStream_t s, std::string& err);
template <int D, typename T>
int launch_coarse(const CoarseSet<T>& S, cudaStream_t s);
// the fused levels of K domains (device array of their descriptors), a cluster
// each; masked ones skipped
template <int D, typename T>
int launch_coarse_batched(const CDesc<T>* const* descs, int K, const int* active, int ncta, size_t smem,
                          cudaStream_t s);

}  // namespace sulf
