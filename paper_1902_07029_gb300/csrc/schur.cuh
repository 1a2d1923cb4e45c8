// The collective red-black multigrid cycle on the equation for s alone
// (arXiv:1902.07029, Sec. 3.4 and 3.5), the production path of both
// precisions.
//
// The c rows of the Jacobian couple only a node's own two unknowns, J^cs_pp
// x^s + J^cc_pp x^c = b^c, and the collective (2x2 block) Gauss-Seidel update
// leaves the c row of the node it updates satisfied, as the ghost relaxation
// does.  So wherever a node's neighbours have been relaxed, x^c_q = t_q -
// rho_q x^s_q with rho = J^cs/J^cc and t = b^c/J^cc, and the collective update
// of x^s is the point Gauss-Seidel update of the Schur complement
//
//   dd_p x_p - sum_q gt_pq x_q = b~_p,
//   gt_pq = g_pq + e_pq rho_q,   dd_p = J^ss_pp - J^sc_pp rho_p,
//   b~_p  = b^s_p - J^sc_pp t_p - sum_q e_pq t_q
//
// (g, e: the edge terms of J^ss, J^sc): the same iterates with half the
// unknowns, 7 instead of 16 FP64 instructions and about half the bytes per
// 3-D update.  Only right after a prolongation (and at the zero start of a
// linear solve) do nodes hold an x^c off their c row by a known delta_q; the
// first sweep after it subtracts sum_q e_pq delta_q = C_p sum delta_q - sum
// C_q delta_q, C = kappa alpha s (the DELTA form below).  The defect of the c
// rows is zero, so every coarse right-hand side has t = 0 and the coarse
// levels are scalar throughout; the defect of the s rows is zero at the black
// nodes without a ghost neighbour (relaxed last, from the red values they
// still see), so the defect, the restriction and the finest defect norm visit
// the red nodes, the black nodes next to a ghost, and the ghosts only; and as
// no update reads the node's own old value, the prolongation visits the black
// nodes and the ghosts only.
//
// Layout: values by node live in checkerboard arrays, the nodes of one colour
// (parity of i+j+k) packed along x: slot = colour * Hn + (i >> 1) + H (j + n k),
// H = (n + 1) / 2, so that a colour's update reads whole sectors of the other
// colour and writes whole sectors of its own.  What belongs to one row of the
// system (gt, dd, 1/dd, b~) is stored in the order of the row list: red inside
// nodes, black inside nodes, ghosts; in each colour the nodes with a regular
// restriction first and those next to a ghost last, so that the cases of a
// kernel fall into different warps.
#pragma once

#include "mg_stages.cuh"

namespace sulf {

// A list entry: (half index << 3) | all coarse corners active << 2 | next to a
// ghost << 1 | parity of i.  nn < 2^29 (checked by the builder).
constexpr int kEntHalf = 3;

// where a node of a level fused into the cluster kernel (coarse.cuh) lies in
// that kernel's rows: gt[q] at off + q stride, then dd and 1/dd; rho at roff, C
// at roff + nx; in the order of the level's list
struct CPerm {
    int off, stride, roff, nx;
};

// one level as the kernels read it
template <int D, typename T>
struct SLev {
    typedef typename V2<T>::t T2;
    int n, H, P, Hn;   // nodes per axis, row and plane pitch, half size
    int n0, n1, ng;    // red and black inside nodes, ghosts
    int nga;           // black nodes next to a ghost (the last ones)
    int nreg0, nreg1;  // red and black nodes with a regular restriction (the first ones)
    const int* hl;     // entries of the inside nodes
    const int* gslot;  // slots of the ghosts
    const int* gidx;   // box nodes of the ghosts
    const int8_t* type;
    // values by slot
    T* X;
    T2* D2;            // (delta, C delta) of the nodes off their c row
    T* R;              // defect
    T* rho;
    T* cs;             // C = kappa alpha s
    // values by list position; gt[q * gs + t], q = +x, -x, +y, -y, +z, -z
    T* gt;
    long long gs;
    T* dd;
    T* di;             // 1 / dd
    T* b;
    T* snap;           // ghosts' s before a sweep's ghost relaxation
    // composed ghost relaxation: code >= 0 slot of an inside member, else
    // u = ~code: snap[u >> 1] (u even) or b[n0 + n1 + (u >> 1)] (u odd)
    const int* gptr;
    const int* gcode;
    const T* gval;
    // the ghosts by the length of that row: ng1 of up to 4 entries, ng8 of up
    // to 32, the longer ones
    const int* gord;
    int ng1, ng8;
    // ghost rows: slot and weight of the members
    const int* rptr;
    const int* rslot;
    const T* rval;
    // restriction onto this level (from the next finer one): slot of an inside
    // node's fine twin; bits of the 3^D fine members that are inside nodes (a
    // regular node's are all, its black ones away from the ghosts); and the
    // ghosts' rows over the finer level's ghost defects (extension along the
    // normal, then outside weighting)
    const int* twin;
    const int* mask;
    const int* cptr;
    const int* cslot;
    const T* cval;
    // a fused level (else null): its rows, and on the first of them where the
    // right-hand side goes (then x is not started)
    const CPerm* perm;
    T* cf;
    const int* bpos;
    T* bf;
    const T* Ainv;  // coarsest level
    int* skip;      // finest level: set where the first sweep of the cycle has been done
    double* acc;    // finest FP32 level: the FP64 update its error is added to
};

// phases of the cycle over a level (restriction and prolongation: a level and
// the next coarser one)
enum class SPhase { correct, red, black, ghosts, residual, outer, restrict_to, prolong_from, solve };

// geometry of a level in these terms (precision independent)
struct SGeo {
    int H = 0, P = 0, Hn = 0, n0 = 0, n1 = 0, nga = 0, nreg0 = 0, nreg1 = 0, ng1 = 0, ng8 = 0;
    int* hl = nullptr;
    int* gslot = nullptr;
    int* gcode = nullptr;
    int* gord = nullptr;
    long long gcap = 0;
    int *rptr = nullptr, *rslot = nullptr;
    double* rval = nullptr;
    float* rval32 = nullptr;
    int *twin = nullptr, *mask = nullptr;
    int *cptr = nullptr, *cslot = nullptr;
    double* cval = nullptr;
    float* cval32 = nullptr;
    int* spos = nullptr;  // coarsest level: list position (ghosts after the inside nodes) of a slot
    int bc = -1, passes = 0;
    double tau = 0;
};

// vectors of a level
template <typename T>
struct SVec {
    typedef typename V2<T>::t T2;
    T2* Wc = nullptr;  // coefficient source in box order (FP32: coarse levels only)
    T *X = nullptr, *R = nullptr, *rho = nullptr, *cs = nullptr;
    T2* D2 = nullptr;
    T *gt = nullptr, *dd = nullptr, *di = nullptr, *b = nullptr, *snap = nullptr;
    T *A = nullptr, *Ainv = nullptr;  // coarsest level: work matrix (where it does not fit on chip) and inverse
    T *tt = nullptr, *uu = nullptr;   // finest level, FP64: t and u = kappa phi by slot
};

template <int D, typename T>
SLev<D, T> make_slev(const LevelGeo& G, const SGeo& S, const SVec<T>& V) {
    const bool f = std::is_same<T, float>::value;
    SLev<D, T> s;
    s.n = G.n;
    s.H = S.H;
    s.P = S.P;
    s.Hn = S.Hn;
    s.n0 = S.n0;
    s.n1 = S.n1;
    s.ng = G.ng;
    s.nga = S.nga;
    s.nreg0 = S.nreg0;
    s.nreg1 = S.nreg1;
    s.gord = S.gord;
    s.ng1 = S.ng1;
    s.ng8 = S.ng8;
    s.hl = S.hl;
    s.gslot = S.gslot;
    s.gidx = G.gidx;
    s.type = G.type;
    s.X = V.X;
    s.D2 = V.D2;
    s.R = V.R;
    s.rho = V.rho;
    s.cs = V.cs;
    s.gt = V.gt;
    s.gs = (long long)S.n0 + S.n1;
    s.dd = V.dd;
    s.di = V.di;
    s.b = V.b;
    s.snap = V.snap;
    s.gptr = G.gop_ptr;
    s.gcode = S.gcode;
    s.gval = f ? (const T*)G.gop_val32 : (const T*)G.gop_val;
    s.rptr = S.rptr;
    s.rslot = S.rslot;
    s.rval = f ? (const T*)S.rval32 : (const T*)S.rval;
    s.twin = S.twin;
    s.mask = S.mask;
    s.cptr = S.cptr;
    s.cslot = S.cslot;
    s.cval = f ? (const T*)S.cval32 : (const T*)S.cval;
    s.perm = nullptr;
    s.cf = nullptr;
    s.bpos = nullptr;
    s.bf = nullptr;
    s.Ainv = V.Ainv;
    s.skip = nullptr;
    s.acc = nullptr;
    return s;
}

// builds a level's SGeo (coarser: the next coarser level or null; finer: the
// next finer one or null); false in `ok` where the level does not fit the
// form (the caller then keeps the two-unknown kernels)
int build_sgeo(SGeo& S, const LevelGeo& L, const LevelGeo* finer, const SGeo* sfiner, const LevelGeo* coarser,
               DevMem& mem, cudaStream_t s, std::string& err, long long& launches, bool& ok);
// what depends on the boundary rows and the composed ghost relaxation
int build_sgeo_rows(SGeo& S, const LevelGeo& L, DevMem& mem, cudaStream_t s, std::string& err, long long& launches);

// ---- kernels; each launcher returns the kernels launched ----

// rho, C (and on the finest level t, the ghosts' right-hand sides and zero
// starts) of every active node from Wc; F: the finest right-hand side in box
// order.  Mixed precision: U the FP32 finest level beside the FP64 one.
template <int D, typename T>
int launch_s_rho(const SLev<D, T>& L, const typename V2<T>::t* Wc, const Coef<T>& c, cudaStream_t s);
template <int D>
int launch_s_rho_fine(const SLev<D, double>& L, const double2* Wc, const Coef<double>& c, const double2* F, double* tt,
                      double* uu, const SLev<D, float>* U, cudaStream_t s);
// the rows gt, dd, 1/dd of the inside nodes (and on the finest level b~ and
// the start of the first sweep)
template <int D, typename T>
int launch_s_coefs(const SLev<D, T>& L, const typename V2<T>::t* Wc, const Coef<T>& c, cudaStream_t s);
template <int D>
int launch_s_coefs_fine(const SLev<D, double>& L, const double2* Wc, const Coef<double>& c, const double2* F,
                        const double* tt, const double* uu, const SLev<D, float>* U, cudaStream_t s);
// threads of a phase
template <int D, typename T>
long long s_threads(SPhase ph, const SLev<D, T>& L, const SLev<D, T>* C);
// one colour; snap: also the ghosts' s into snap; skip: return at once where
// *L.skip is set; acc: the new values are added to L.acc
template <int D, typename T>
int launch_s_relax(const SLev<D, T>& L, int colour, bool delta, bool snap, bool skip, bool acc, cudaStream_t s);
template <int D, typename T>
int launch_s_ghosts(const SLev<D, T>& L, bool skip, bool acc, cudaStream_t s);
// the red half-sweep that opens an FP64 cycle, from the defects that the norm
// of the cycle before left in R
template <int D, typename T>
int launch_s_correct(const SLev<D, T>& L, cudaStream_t s);
// defect of the red nodes, of the black ones next to a ghost and of the
// ghosts into R (norm null), or its max-norm, with the red nodes' defects in R
// and *L.skip set to 0
template <int D, typename T>
int launch_s_residual(const SLev<D, T>& L, unsigned long long* norm, cudaStream_t s);
// mixed precision: the FP64 defect of every row with its max-norm, stored as
// the FP32 right-hand side, and the FP32 error's start (and *U.skip set to 0)
template <int D>
int launch_s_outer(const SLev<D, double>& L, const SLev<D, float>& U, unsigned long long* norm, cudaStream_t s);
template <int D, typename T>
int launch_s_restrict(const SLev<D, T>& F, const SLev<D, T>& C, cudaStream_t s);
template <int D, typename T>
int launch_s_prolong(const SLev<D, T>& F, const SLev<D, T>& C, cudaStream_t s);
// coarsest level: the dense Schur complement inverted (rows and columns in
// list order, or at cpos of it), and applied
template <int D, typename T>
int launch_s_factor(const SLev<D, T>& L, const int* spos, const int* cpos, T* A, T* Ainv, int* singular,
                    cudaStream_t s);
template <int D, typename T>
int launch_s_solve(const SLev<D, T>& L, cudaStream_t s);
// a phase of K domains in one launch (CTAs of kNodeThreads; masked domains are
// skipped; a residual with norms is the finest one's norms)
template <int D, typename T>
int launch_s_batched(SPhase ph, bool delta, const SLev<D, T>* lv, const SLev<D, T>* lc, const int* pre, int nblocks,
                     int K, const int* active, bool skip, bool acc, unsigned long long* norms, cudaStream_t s);
template <int D>
int launch_s_batched_outer(const SLev<D, double>* l64, const SLev<D, float>* l32, const int* pre, int nblocks, int K,
                           const int* active, unsigned long long* norms, cudaStream_t s);
// W -= (x, t - rho x) on the active nodes with the norms of launch_newton_update
// (nothing where *on is zero)
template <int D>
int launch_s_update(const SLev<D, double>& L, const double* tt, double2* W, unsigned long long* norms, const int* on,
                    cudaStream_t s);
// (x, t - rho x) in box order (debug outputs)
template <int D>
int launch_s_export(const SLev<D, double>& L, const double* tt, double2* x, cudaStream_t s);
// coarse (s, c) by injection, from FP64 or FP32 into either
template <int D, typename TF, typename T>
int launch_inject_to(const LevelGeo& F, const typename V2<TF>::t* fW, const LevelGeo& C, typename V2<T>::t* cW,
                     cudaStream_t s);

}  // namespace sulf
