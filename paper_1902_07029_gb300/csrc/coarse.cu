// The cluster-resident coarse levels (coarse.cuh): kernel and tables.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "coarse.cuh"

namespace sulf {

using stages::fmadd;
using stages::kGopLanes;

namespace {

constexpr int kRefBits = 12;  // a reference: owner << kRefBits | index in its values
constexpr unsigned kRefMask = (1u << kRefBits) - 1;
constexpr unsigned kNoRef = 0xffffu;
constexpr size_t kCoarseSmem = 224 * 1024;
// words of the cycle's program: phase | level << 8 | flags; kOpAll: by every
// CTA (else CTA 0), kOpFar: values of other CTAs are read, kOpWide: a cluster
// barrier follows (else one of CTA 0)
enum { kOpNone = 0, kOpRed, kOpBlack, kOpGhosts, kOpDefect, kOpRestrict, kOpSolve, kOpProlong, kOpVisit };
constexpr unsigned kOpDelta = 1u << 16, kOpLast = 1u << 17, kOpAll = 1u << 18, kOpFar = 1u << 19, kOpWide = 1u << 20;
constexpr unsigned kOpSkipRed = 1u << 21, kOpDown = 1u << 22;  // of a visit: first red half-sweep done; defect after
constexpr unsigned kOpTop = 1u << 23;                           // the cycle's first visit of the finest level
// a table entry that names a value of any array: owner << kAddrBits | byte
// offset in the owner's shared memory
constexpr int kAddrBits = 20;
constexpr unsigned kAddrMask = (1u << kAddrBits) - 1;
// entries a lane of a table's row has, up to 32 lanes a row: with four the
// longest row is one round of loads, while an SM's two FP64 lanes make the
// partial sums dear (33^3 box, rows of 1 to 90 entries, four lanes a row and a
// warp above 64: 6000 cycles a phase)
template <typename T>
constexpr int kRowEntries = sizeof(T) == 4 ? 4 : 8;
// a table's warp: its first row | log2 lanes per row << 16 | rows << 20
__host__ __device__ constexpr unsigned row_job(int row, int lg, int cnt) {
    return (unsigned)row | (unsigned)lg << 16 | (unsigned)cnt << 20;
}

__device__ __forceinline__ unsigned cta_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned map_rank(unsigned a, unsigned r) {
    unsigned o;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(a), "r"(r));
    return o;
}
__device__ __forceinline__ void ld_remote(unsigned a, float& v) {
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
}
__device__ __forceinline__ void ld_remote(unsigned a, double& v) {
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
}
__device__ __forceinline__ void ld_remote(unsigned a, float2& v) {
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
}
__device__ __forceinline__ void ld_remote(unsigned a, double2& v) {
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a));
}

// own shared memory (W false) or the cluster's, by address
template <bool W>
__device__ __forceinline__ void ld_at(unsigned a, float& v) {
    if (W)
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
    else
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
}
template <bool W>
__device__ __forceinline__ void ld_at(unsigned a, double& v) {
    if (W)
        asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
    else
        asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a));
}
template <bool W>
__device__ __forceinline__ void ld_at(unsigned a, float2& v) {
    if (W)
        asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    else
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
}
template <bool W>
__device__ __forceinline__ void ld_at(unsigned a, double2& v) {
    if (W)
        asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a));
    else
        asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a));
}
template <bool W>
__device__ __forceinline__ void phase_barrier() {
    if (W)
        cluster_barrier();
    else
        __syncthreads();
}

// copy into shared memory in 16-byte pieces (both ends aligned) by the CTA
__device__ __forceinline__ void stage(char* dst, const void* src, size_t bytes) {
    const size_t n16 = (bytes + 15) / 16;
    for (size_t c = threadIdx.x; c < n16; c += blockDim.x) {
        const unsigned d = (unsigned)__cvta_generic_to_shared(dst + 16 * c);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"((const char*)src + 16 * c) : "memory");
    }
}

template <int D, typename T>
struct Coarse {
    typedef typename V2<T>::t T2;
    char* sm;
    unsigned sa;  // shared address of sm
    int tid, nthr;

    template <typename V>
    __device__ __forceinline__ V* at(int off) const {
        return reinterpret_cast<V*>(sm + off);
    }
    // the values N references name in the array at byte offset off (the same
    // offset in every CTA); w: an owner may be another CTA (uniform)
    template <int N, typename V>
    __device__ __forceinline__ void get(bool w, int off, const unsigned* ref, V* v) const {
        if (w) {
#pragma unroll
            for (int q = 0; q < N; q++)
                ld_remote(map_rank(sa + off + (ref[q] & kRefMask) * (unsigned)sizeof(V), ref[q] >> kRefBits), v[q]);
        } else {
#pragma unroll
            for (int q = 0; q < N; q++) v[q] = at<const V>(off)[ref[q]];
        }
    }

    // address of a table entry's value (an array at byte offset off, or by kAddrBits)
    template <class R>
    __device__ __forceinline__ unsigned where(bool w, int off, R u) const {
        if (sizeof(R) == 4) {
            const unsigned a = sa + (u & kAddrMask);
            return w ? map_rank(a, u >> kAddrBits) : a;
        }
        const unsigned a = sa + off + (u & kRefMask) * (unsigned)sizeof(T);
        return w ? map_rank(a, u >> kRefBits) : a;
    }

    // entries beg, beg + step, ... < end of a CSR table times the values they name
    template <class R>
    __device__ __forceinline__ T entries(bool w, int beg, int end, int step, const R* ref, const T* val,
                                         int off) const {
        T v = 0;
        for (int j0 = beg; j0 < end; j0 += 4 * step) {
            unsigned u[4];
            T c[4], x[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int j = j0 + q * step < end ? j0 + q * step : j0;
                u[q] = where<R>(w, off, ref[j]);
                c[q] = val[j];
            }
            if (w) {
#pragma unroll
                for (int q = 0; q < 4; q++) ld_at<true>(u[q], x[q]);
            } else {
#pragma unroll
                for (int q = 0; q < 4; q++) ld_at<false>(u[q], x[q]);
            }
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (j0 + q * step < end) v = fmadd(c[q], x[q], v);
        }
        return v;
    }

    // the rows of a table, by `stride` threads, after the `skip` first threads'
    // own work first(t) (a multiple of 32); done(ghost, sum)
    template <class R, class First, class Done>
    __device__ __forceinline__ void rows(bool w, int stride, int skip, const CTab& tab, int off, const First& first,
                                         const Done& done) const {
        const int tot = skip + 32 * tab.nw;
        const int* ptr = at<const int>(tab.ptr);
        for (int t = tid; t < tot; t += stride) {
            if (t < skip) {
                first(t);
                continue;
            }
            const unsigned job = at<const unsigned>(tab.job)[(t - skip) >> 5];
            const int lg = job >> 16 & 15, lane = t & 31, i = lane >> lg, ln = lane & ((1 << lg) - 1);
            const bool on = i < (int)(job >> 20);
            const int r = (int)(job & 0xffff) + i;
            T v = 0;
            if (on)
                v = entries<R>(w, ptr[r] + ln, ptr[r + 1], 1 << lg, at<const R>(tab.ref), at<const T>(tab.val), off);
            for (int o = 1 << lg >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (on && ln == 0) done(at<const uint16_t>(tab.idx)[r], v);
        }
    }

    // a row's neighbour sum: gt/dd . x over the axis neighbours added to r
    __device__ __forceinline__ T couple(bool w, const T* coef, int nr, int i, int x, const unsigned* u, T r) const {
        T xv[2 * D];
        get<2 * D, T>(w, x, u, xv);
#pragma unroll
        for (int q = 0; q < 2 * D; q++) r = fmadd(coef[q * nr + i], xv[q], r);
        return r;
    }

    __device__ __forceinline__ void colour(const CLev& L, bool w, int c, bool delta, bool last) const {
        const T* coef = at<const T>(L.coef);
        const uint16_t* nbr = at<const uint16_t>(L.nbr);
        const int nr = L.nr, i1 = c ? nr : L.cr, near = L.cr + L.cbn, xo = L.x, cg = L.cg;
        const T* b = at<const T>(L.b);
        T* x = at<T>(xo);
        T* y = at<T>(L.y);
        const int d2 = L.d2, nx = L.nx;
        for (int i = (c ? L.cr : 0) + tid; i < i1; i += nthr) {
            unsigned u[2 * D];
#pragma unroll
            for (int q = 0; q < 2 * D; q++) u[q] = nbr[q * nr + i];
            T r = b[i];
            if (delta && (c == 0 || i >= near)) {
                T2 d[2 * D];
                get<2 * D, T2>(w, d2, u, d);
                T sd = d[0].x, sc = d[0].y;
#pragma unroll
                for (int q = 1; q < 2 * D; q++) {
                    sd += d[q].x;
                    sc += d[q].y;
                }
                r = fmadd(-coef[(2 * D + 2) * nr + nx + i], sd, r + sc);
            }
            r = couple(w, coef, nr, i, xo, u, r * coef[(2 * D + 1) * nr + i]);
            x[i] = r;
            if (last) y[i] = coef[(2 * D + 2) * nr + i] * r;
        }
        if (c)
            for (int g = nthr - 1 - tid; g < cg; g += nthr) at<T>(L.snap)[g] = x[nr + g];
    }

    __device__ __forceinline__ void ghosts(const CLev& L, bool w, bool last) const {
        const T* rho = at<const T>(L.coef) + (2 * D + 3) * L.nr;  // of the ghosts
        T* x = at<T>(L.x) + L.nr;
        T* y = at<T>(L.y) + L.nr;
        rows<unsigned>(
            w, nthr, 0, L.g, 0, [](int) {},
            [&](int g, T v) {
                x[g] = v;
                if (last) y[g] = rho[g] * v;
            });
    }

    // defect of the red nodes, of the black ones next to a ghost and of the ghosts
    __device__ __forceinline__ void defect(const CLev& L, bool w) const {
        const T* coef = at<const T>(L.coef);
        const uint16_t* nbr = at<const uint16_t>(L.nbr);
        const int nr = L.nr, cr = L.cr, cbn = L.cbn, own = nr - cbn, xo = L.x;
        const T* x = at<const T>(xo);
        const T* b = at<const T>(L.b);
        T* R = at<T>(L.y);
        rows<uint16_t>(
            w, nthr, (own + 31) / 32 * 32, L.r, xo,
            [&](int t) {
                if (t >= own) return;
                const int i = t < cr ? t : cbn + t;
                unsigned u[2 * D];
#pragma unroll
                for (int q = 0; q < 2 * D; q++) u[q] = nbr[q * nr + i];
                R[i] = coef[2 * D * nr + i] * couple(w, coef, nr, i, xo, u, fmadd(b[i], coef[(2 * D + 1) * nr + i], -x[i]));
            },
            [&](int g, T v) { R[nr + g] = b[nr + g] - v; });
    }

    // the defect of level F onto the right-hand side of the next coarser level
    // C, whose x starts with its red half-sweep from zero
    __device__ __forceinline__ void restrict_to(const CLev& F, const CLev& C, bool w) const {
        const int* ptr = at<const int>(C.cptr);
        const uint16_t* ref = at<const uint16_t>(C.cref);
        const T* val = at<const T>(C.cval);
        const int nr = C.nr, cr = C.cr, yo = F.y;
        const T* di = at<const T>(C.coef) + (2 * D + 1) * nr;
        T* b = at<T>(C.b);
        T* x = at<T>(C.x);
        // a row's entries are a chain of loads and multiply-adds: up to four
        // lanes share it where the threads suffice
        const int lg = 4 * nr <= nthr ? 2 : (2 * nr <= nthr ? 1 : 0);
        rows<uint16_t>(
            w, nthr, ((nr << lg) + 31) / 32 * 32, C.c, yo,
            [&](int t) {
                const int i = t >> lg, ln = t & ((1 << lg) - 1);
                T v = 0;
                if (i < nr) v = entries<uint16_t>(w, ptr[i] + ln, ptr[i + 1], 1 << lg, ref, val, yo);
                for (int o = 1 << lg >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (i >= nr || ln) return;
                b[i] = v;
                x[i] = i < cr ? v * di[i] : (T)0;
            },
            [&](int g, T v) {
                b[nr + g] = v;
                x[nr + g] = 0;
            });
    }

    __device__ __forceinline__ void prolong(const CLev& F, const CLev& C, bool w) const {
        const uint16_t* pro = at<const uint16_t>(F.pro);
        const int n = F.cb + F.cg, cr = F.cr, nx = F.nx, xc = C.x, yc = C.y;
        const T* rho = at<const T>(F.coef) + (2 * D + 2) * F.nr;
        T* x = at<T>(F.x);
        T2* d2 = at<T2>(F.d2);
        for (int t = tid; t < n; t += nthr) {
            const int i = cr + t;  // black nodes, then ghosts
            unsigned u[1 << D];
            T v[1 << D];
            int cnt = 0;
            bool has[1 << D];
#pragma unroll
            for (int cc = 0; cc < (1 << D); cc++) {
                u[cc] = pro[cc * n + t];
                has[cc] = u[cc] != kNoRef;
                cnt += has[cc];
                if (!has[cc]) u[cc] = 0;  // read and dropped
            }
            T ps = 0, py = 0;
            get<1 << D, T>(w, xc, u, v);
#pragma unroll
            for (int cc = 0; cc < (1 << D); cc++)
                if (has[cc]) ps += v[cc];
            get<1 << D, T>(w, yc, u, v);
#pragma unroll
            for (int cc = 0; cc < (1 << D); cc++)
                if (has[cc]) py += v[cc];
            T2 d;
            d.x = 0;
            d.y = 0;
            if (cnt) {
                const T r = stages::inv_count<T>(cnt);
                x[i] = fmadd(ps, r, x[i]);
                d.x = fmadd(rho[i], ps, -py) * r;
                d.y = rho[nx + i] * d.x;
            }
            d2[i] = d;
        }
    }

    // address of a reference in the array at byte offset off
    template <bool W, typename V>
    __device__ __forceinline__ unsigned addr(int off, unsigned ref) const {
        if (!W) return sa + off + ref * (unsigned)sizeof(V);
        return map_rank(sa + off + (ref & kRefMask) * (unsigned)sizeof(V), ref >> kRefBits);
    }

    // The sweeps of one visit of a level whose rows fit the threads, and after
    // the down sweeps the defect: a thread has a red row, a black row and a
    // lane of a ghost's row, kept in registers (coefficients and
    // addresses) over the visit, so a phase is a handful of loads and
    // multiply-adds between two barriers.  What a warp executes between two
    // barriers is its latency and what all warps execute the CTA's, so nothing
    // else is left there and the warps without a row do nothing.  Measured
    // (clock stamps, levels of 100 to 5000 nodes, a visit of two sweeps and the
    // defect, its loads of the rows included, per phase): 570 to 680 cycles on
    // CTA 0 and 1200 to 1300 on the cluster in FP32, 1200 to 1400 and 2000 to
    // 2150 in FP64.
    template <bool W>
    __device__ __forceinline__ void visit(const CLev& L, int nsw, bool skip_red, bool delta, bool last,
                                          bool dft) const {
        const int nr = L.nr, cr = L.cr;
        const int nact = max((max(cr, L.cb) + 31) & ~31, 32 * L.g.nw);
        auto barrier = [&] {
            if (W)
                cluster_barrier();
            else
                asm volatile("bar.sync 1, %0;" ::"r"(nact) : "memory");
        };
        const int nph = 3 * nsw - (skip_red ? 1 : 0);
        const int nbar = nph - (dft ? 0 : 1);  // (before the defect: one more)
        if (tid >= nact) {
            if (W)
                for (int q = 0; q < nbar; q++) cluster_barrier();
            return;
        }
        const T* coef = at<const T>(L.coef);
        const int xo = L.x;
        const T* bs = at<const T>(L.b);
        T* xs = at<T>(xo);
        T* y = at<T>(L.y);
        const bool gwarp = tid >> 5 < L.g.nw;
        const unsigned job = gwarp ? at<const unsigned>(L.g.job)[tid >> 5] : 0;
        const int lg = job >> 16 & 15, ln = tid & ((1 << lg) - 1), gr = (int)(job & 0xffff) + ((tid & 31) >> lg);
        const bool rowg = (tid & 31) >> lg < (int)(job >> 20);
        int gi = 0;
        constexpr bool kRegs = sizeof(T) == 4;  // FP64 coefficients stay in shared memory (registers)
        unsigned u[2][2 * D], a[4];
        T g[2][2 * D], bb[2], c[4];  // bb: b/dd, at first with what the neighbours are off their c rows by
        bool on[2], own[2];
        {
            const uint16_t* nbr = at<const uint16_t>(L.nbr);
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const int i = k ? cr + tid : tid;
                on[k] = tid < (k ? L.cb : cr);
                own[k] = on[k] && (k == 0 || tid >= L.cbn);  // has a defect, sees values off their c rows
                if (!on[k]) continue;
                T r = bs[i];
#pragma unroll
                for (int q = 0; q < 2 * D; q++) {
                    u[k][q] = nbr[q * nr + i];
                    if (kRegs) g[k][q] = coef[q * nr + i];
                }
                if (delta && own[k]) {
                    // what the neighbours are off their c rows by
                    T2 d[2 * D];
#pragma unroll
                    for (int q = 0; q < 2 * D; q++) ld_at<W>(addr<W, T2>(L.d2, u[k][q]), d[q]);
                    T sd = 0, sc = 0;
#pragma unroll
                    for (int q = 0; q < 2 * D; q++) {
                        sd += d[q].x;
                        sc += d[q].y;
                    }
                    r = fmadd(-coef[(2 * D + 2) * nr + L.nx + i], sd, r + sc);
                }
                bb[k] = r * coef[(2 * D + 1) * nr + i];
#pragma unroll
                for (int q = 0; q < 2 * D; q++) u[k][q] = addr<W, T>(xo, u[k][q]);
            }
        }
        const unsigned* ref = at<const unsigned>(L.g.ref);
        const T* val = at<const T>(L.g.val);
        int beg = 0, end = 0;
        // address of entry k of the ghost's row (past the end: its last one's, times 0)
        auto entry = [&](int k) { return where<unsigned>(W, 0, ref[min(k, end - 1)]); };
        if (rowg) {
            const int* ptr = at<const int>(L.g.ptr);
            gi = at<const uint16_t>(L.g.idx)[gr];
            beg = ptr[gr] + ln;
            end = ptr[gr + 1];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int k = beg + (q << lg);
                a[q] = entry(k);
                c[q] = k < end ? val[k] : (T)0;
            }
        }
        const int plast = last ? nph - 3 : nph;  // from here on y = rho s is kept
        auto row = [&](int k, int p) {
            const int i = k ? cr + tid : tid;
            T v[2 * D], r = bb[k];
#pragma unroll
            for (int e = 0; e < 2 * D; e++) ld_at<W>(u[k][e], v[e]);
#pragma unroll
            for (int e = 0; e < 2 * D; e++) r = fmadd(kRegs ? g[k][e] : coef[e * nr + i], v[e], r);
            xs[i] = r;
            if (p >= plast) y[i] = coef[(2 * D + 2) * nr + i] * r;
            if (p < 3 && delta) bb[k] = bs[i] * coef[(2 * D + 1) * nr + i];
        };
        // phases: red, black, ghosts, red, ...; one copy of each phase's code
        int kind = skip_red ? 1 : 0;
#pragma unroll 1
        for (int p = 0; p < nph; p++) {
            if (kind == 0) {
                if (on[0]) row(0, p);
            } else if (kind == 1) {
                if (rowg && ln == 0) at<T>(L.snap)[gi] = xs[nr + gi];
                if (on[1]) row(1, p);
            } else if (gwarp) {
                T v = 0;
                if (rowg) {
                    T w[4];
#pragma unroll
                    for (int q = 0; q < 4; q++) ld_at<W>(a[q], w[q]);
#pragma unroll
                    for (int q = 0; q < 4; q++) v = fmadd(c[q], w[q], v);
#pragma unroll 1
                    for (int j = beg + (4 << lg); j < end; j += 4 << lg) {
#pragma unroll
                        for (int q = 0; q < 4; q++) ld_at<W>(entry(j + (q << lg)), w[q]);
#pragma unroll
                        for (int q = 0; q < 4; q++) {
                            const int k = j + (q << lg);
                            v = fmadd(k < end ? val[k] : (T)0, w[q], v);
                        }
                    }
                }
                for (int o = 1 << lg >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (rowg && ln == 0) {
                    xs[nr + gi] = v;
                    if (p >= plast) y[nr + gi] = coef[(2 * D + 3) * nr + gi] * v;
                }
            }
            kind = kind == 2 ? 0 : kind + 1;
            if (p < nbar) barrier();
        }
        if (dft) {
#pragma unroll
            for (int k = 0; k < 2; k++) {
                if (!own[k]) continue;
                const int i = k ? cr + tid : tid;
                T v[2 * D];
#pragma unroll
                for (int q = 0; q < 2 * D; q++) ld_at<W>(u[k][q], v[q]);
                T r = bb[k] - xs[i];
#pragma unroll
                for (int q = 0; q < 2 * D; q++) r = fmadd(kRegs ? g[k][q] : coef[q * nr + i], v[q], r);
                y[i] = r * coef[2 * D * nr + i];
            }
            rows<uint16_t>(
                W, nact, 0, L.r, xo, [](int) {}, [&](int g, T v) { y[nr + g] = bs[nr + g] - v; });
        }
        // (the caller's barrier follows)
    }

    // coarsest level: x = A^{-1} b, kGopLanes lanes per row
    __device__ __forceinline__ void solve(const CLev& L, bool w, const CDesc<T>& d, const T* ag) const {
        const T* A = L.ainv >= 0 ? at<const T>(L.ainv) : ag;
        const int* cnt = d.cnt_m;
        const T* rho = at<const T>(L.coef) + (2 * D + 2) * L.nr;
        const int ln = tid % kGopLanes, nx = L.nx, m = L.m, bo = L.b;
        for (int base = 0; base < nx; base += nthr / kGopLanes) {
            const int i = base + tid / kGopLanes;
            T v = 0;
            if (i < nx) {
                const T* a = A + (size_t)i * m;
                for (unsigned o = 0; o < (w ? (unsigned)d.ncta : 1u); o++) {
                    const int n = cnt[o];
                    for (int j0 = ln; j0 < n; j0 += 4 * kGopLanes) {
                        unsigned u[4];
                        T x[4];
#pragma unroll
                        for (int q = 0; q < 4; q++)
                            u[q] = o << kRefBits | (unsigned)(j0 + q * kGopLanes < n ? j0 + q * kGopLanes : j0);
                        get<4, T>(w, bo, u, x);
#pragma unroll
                        for (int q = 0; q < 4; q++)
                            if (j0 + q * kGopLanes < n) v = fmadd(a[j0 + q * kGopLanes], x[q], v);
                    }
                    a += n;
                }
            }
            v = stages::gop_reduce<T>(v);
            if (i < nx && ln == 0) {
                at<T>(L.x)[i] = v;
                at<T>(L.y)[i] = rho[i] * v;
            }
        }
    }
};

// The phases of a cycle run as a program of (phase, level, flags, barrier)
// words: each phase's code exists once and stays in the instruction cache
// (inlined per call site and per kind of level the kernel had 144 KB of code
// and its phases took two to three times as long).
template <int D, typename T>
__global__ void __launch_bounds__(kCoarseThreads, 1) k_s_coarse(const CDesc<T>* __restrict__ one,
                                                                   const CDesc<T>* const* __restrict__ many,
                                                                   const int* __restrict__ active) {
    extern __shared__ __align__(16) char coarse_smem[];
    // many domains (lock-step batching): a cluster each, masked ones skipped
    const int inst = many ? (int)(blockIdx.x / cluster_size()) : 0;
    if (many && masked(active, inst)) return;
    const CDesc<T>& d = many ? *many[inst] : *one;
    Coarse<D, T> k;
    k.sm = coarse_smem;
    k.sa = (unsigned)__cvta_generic_to_shared(coarse_smem);
    k.tid = threadIdx.x;
    k.nthr = blockDim.x;
    const int me = (int)cta_rank(), n = d.nlev, nop = d.nop;
    // fixed during the linear solve: copied while the previous kernel runs
    stage(k.sm, d.head + (size_t)me * d.head_len, d.head_len);
    stage(k.sm + d.tab_at, d.tab + d.tab_off[me], d.tab_len[me]);
    stage(k.sm + d.coef_at, d.coef + d.coef_off[me], sizeof(T) * (size_t)d.coef_len[me]);
    if (d.ainv_len[me]) stage(k.sm + d.ainv_at, d.ainv + d.ainv_off[me], sizeof(T) * (size_t)d.ainv_len[me]);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const T* bg = d.b + d.b_off[me];
    const int* slot = d.slot + d.b_off[me];
    const T* ag = d.ainv + d.ainv_off[me];
    T* X = d.X;
    double* acc = d.acc;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const CLev* lev = reinterpret_cast<const CLev*>(k.sm);
    const unsigned* prog = reinterpret_cast<const unsigned*>(k.sm + n * sizeof(CLev));
    // the red nodes stay on their c rows
    for (int l = 0; l + 1 < n; l++)
        for (int i = threadIdx.x; i < 2 * lev[l].cr; i += blockDim.x) k.template at<T>(lev[l].d2)[i] = 0;
    const int nx = lev[0].nx;
    pdl_enter();
    const bool done = d.skip && *(const volatile int*)d.skip;  // the finest level's first sweep
    {
        // the first level's right-hand side, and its red half-sweep from zero
        const CLev& L = lev[0];
        const T* di = k.template at<const T>(L.coef) + (2 * D + 1) * L.nr;
        const int cr = L.cr;
        for (int i = threadIdx.x; i < nx; i += blockDim.x) {
            const T v = __ldcg(bg + i);
            k.template at<T>(L.b)[i] = v;
            k.template at<T>(L.x)[i] = d.skip ? __ldcg(X + slot[i]) : (i < cr ? v * di[i] : (T)0);
        }
    }
    for (int pc = 0; pc < nop; pc++) {
        const unsigned o = prog[pc];
        const CLev& L = lev[(o >> 8) & 0xff];
        if ((o & kOpAll) || me == 0) {
            const bool w = o & kOpFar, delta = o & kOpDelta, last = o & kOpLast;
            switch (o & 0xff) {
                case kOpRed:
                case kOpBlack: k.colour(L, w, (o & 0xff) == kOpBlack, delta, last); break;
                case kOpGhosts: k.ghosts(L, w, last); break;
                case kOpDefect: k.defect(L, w); break;
                case kOpRestrict: k.restrict_to(*(&L - 1), L, w); break;
                case kOpSolve: k.solve(L, w, d, ag); break;
                case kOpProlong: k.prolong(L, *(&L + 1), w); break;
                case kOpVisit: {
                    const bool first = done && (o & kOpTop);
                    const int nsw = (int)(o >> 24) - (first ? 1 : 0);
                    const bool skip_red = (o & kOpSkipRed) && !first;
                    if (w)
                        k.template visit<true>(L, nsw, skip_red, delta, last, o & kOpDown);
                    else
                        k.template visit<false>(L, nsw, skip_red, delta, last, o & kOpDown);
                    break;
                }
                default: break;
            }
        }
        if (o & kOpWide)
            cluster_barrier();
        else if (me == 0)
            __syncthreads();
    }
    {
        const T* x = k.template at<const T>(lev[0].x);
        for (int i = threadIdx.x; i < nx; i += blockDim.x) {
            if (acc)
                acc[slot[i]] += (double)x[i];
            else
                X[slot[i]] = x[i];
        }
    }
    cluster_barrier();  // no CTA leaves while another may still read its shared memory
}

// ---------------------------------------------------------------------------
// tables (host)

// the kernel's limits raised once per device (a per-launch value would race
// with other threads' launches)
template <int D, typename T>
void raise_limits() {
    static std::mutex mu;
    static bool raised[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    if (dev >= 0 && dev < 64 && raised[dev]) return;
    cudaFuncSetAttribute(k_s_coarse<D, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCoarseSmem);
    cudaFuncSetAttribute(k_s_coarse<D, T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (dev >= 0 && dev < 64) raised[dev] = true;
}

// whether the device can hold a cluster of C such CTAs
template <int D, typename T>
bool cluster_fits(int C, size_t smem) {
    raise_limits<D, T>();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(kCoarseThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_s_coarse<D, T>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n > 0;
}

inline size_t up16(size_t n) { return (n + 15) & ~size_t(15); }

// the warps of a table's rows, given their lengths, longest first
template <typename T>
std::vector<unsigned> row_jobs(const std::vector<int>& len) {
    std::vector<unsigned> jobs;
    for (int i = 0, n = (int)len.size(); i < n;) {
        int lg = 0;
        while (lg < 5 && kRowEntries<T> << lg < len[i]) lg++;
        const int cnt = std::min(32 >> lg, n - i);
        jobs.push_back(row_job(i, lg, cnt));
        i += cnt;
    }
    return jobs;
}

template <typename T>
struct Download {
    std::vector<T> v;
    void get(const T* dev, size_t n, cudaStream_t s, bool& ok) {
        v.resize(n + 1);
        if (n && cudaMemcpyAsync(v.data(), dev, sizeof(T) * n, cudaMemcpyDeviceToHost, s) != cudaSuccess) ok = false;
    }
};

// a level's device data on the host
struct HostLevel {
    Download<int> hl, gslot, gptr, gcode, rptr, rslot, cptr, cslot;
    Download<double> gval, rval, cval;
    Download<int8_t> type;
    std::vector<uint16_t> ref;                  // slot -> reference
    std::vector<std::vector<int>> own;          // per CTA: list positions, red, black away, black near, ghosts
    std::vector<int> cr, cbn, cb, cg;
    int wide = 1;
};

}  // namespace

template <int D, typename T>
int build_coarse(CoarseSet<T>& S, const LevelGeo* G, const SGeo* SG, const SVec<T>* V, int L, int want, int nu1,
                 int nu2, int max_cta, double* acc, const int* skip, DevMem& mem, cudaStream_t s, std::string& err) {
    S.l0 = -1;
    S.want = want;
    S.nu1 = nu1;
    S.nu2 = nu2;
    S.max_cta = max_cta;
    S.rows = false;  // (the caller's note of success)
    if (want < 0 || want > L - 1) return SULF_OK;
    const bool f32 = std::is_same<T, float>::value;
    // Levels of up to this many nodes run on CTA 0, whose phases take half as
    // long as the cluster's (see visit), while an SM's two FP64 lanes or the
    // ghosts of 3-D levels make them long sooner.  Two CN steps with 300 /
    // 600 / 1200: 257^2 star, mixed 7.49 / 7.47 / 7.77 and 5.81 / 5.81 / 5.70 ms;
    // 1025^2 star, FP64 8.77 / 8.62 / 8.63, mixed 5.92 / 5.79 / 5.80; 321^2 star
    // (Neumann), FP64 8.33 / 7.87 / 7.89; 65^3 box, mixed 17.2 / 18.4 / 18.4;
    // 129^3 box, FP64 28.0 / 28.7 / 28.7.
    const int narrow = D == 3 ? 300 : (f32 ? 1200 : 600);
    // The finest level joins where its rows fit the threads (a visit, else its
    // phases are no shorter there than as kernels of their own).
    auto top_fits = [&](int C) { return std::max(SG[0].n0, SG[0].n1) <= kCoarseThreads * C; };
    // the first level that fits, with the smallest cluster
    int l0 = want, ncta = 0;
    for (; l0 < L; l0++) {
        size_t nodes = 0;
        for (int l = l0; l < L; l++) nodes += (size_t)G[l].nin[0] + G[l].nin[1] + G[l].ng;
        if (nodes > 40000 || (l0 == 0 && !top_fits(std::min(max_cta, kCoarseMaxCta)))) continue;
        break;
    }
    if (l0 >= L) return SULF_OK;
    std::vector<HostLevel> H(L);
    bool ok = true;
    for (int l = l0; l < L; l++) {
        HostLevel& h = H[l];
        const SGeo& g = SG[l];
        const size_t nin = (size_t)g.n0 + g.n1, ng = G[l].ng;
        h.hl.get(g.hl, nin, s, ok);
        h.gslot.get(g.gslot, ng, s, ok);
        h.type.get(G[l].type, (size_t)G[l].nn, s, ok);
        if (ng) {
            h.gptr.get(G[l].gop_ptr, ng + 1, s, ok);
            h.gcode.get(g.gcode, (size_t)G[l].gop_nnz, s, ok);
            h.gval.get(G[l].gop_val, (size_t)G[l].gop_nnz, s, ok);
            h.rptr.get(g.rptr, ng + 1, s, ok);
            if (l > 0) h.cptr.get(g.cptr, ng + 1, s, ok);
        }
    }
    if (!ok || cudaStreamSynchronize(s) != cudaSuccess) {
        err = "coarse-level tables failed";
        return SULF_EDEVICE;
    }
    for (int l = l0; l < L; l++) {
        HostLevel& h = H[l];
        if (!G[l].ng) continue;
        h.rslot.get(SG[l].rslot, (size_t)h.rptr.v[G[l].ng], s, ok);
        h.rval.get(SG[l].rval, (size_t)h.rptr.v[G[l].ng], s, ok);
        if (l > l0) {
            h.cslot.get(SG[l].cslot, (size_t)h.cptr.v[G[l].ng], s, ok);
            h.cval.get(SG[l].cval, (size_t)h.cptr.v[G[l].ng], s, ok);
        }
    }
    if (!ok || cudaStreamSynchronize(s) != cudaSuccess) {
        err = "coarse-level tables failed";
        return SULF_EDEVICE;
    }
    std::vector<char> tab;
    std::vector<CLev> lev;
    std::vector<unsigned> prog;
    CDesc<T> d;
    std::vector<int> slots;
    size_t smem = 0, coef_tot = 0;
    bool fit = false;
    for (; l0 < L && !fit; l0++) {
        for (int C : {8, 16}) {
            if (C > max_cta) break;
            if (l0 == 0 && !top_fits(C)) continue;
            const int n = L - l0;
            ncta = C;
            // deal the nodes: bands of the box order (slots are box order up to
            // the colour: half indices compare as box rows do)
            bool refs_ok = true;
            for (int l = l0; l < L && refs_ok; l++) {
                HostLevel& h = H[l];
                const SGeo& g = SG[l];
                const int nin = g.n0 + g.n1, ng = G[l].ng, tot = nin + ng;
                h.wide = tot > narrow || (l == L - 1 && !f32 && tot > 40);
                const int w = h.wide ? C : 1;
                auto half = [&](int t) {
                    if (t < nin) return h.hl.v[t] >> kEntHalf;
                    const int sl = h.gslot.v[t - nin];
                    return sl >= g.Hn ? sl - g.Hn : sl;
                };
                // counting sort by half index
                std::vector<int> cnt(g.Hn + 1, 0), ord(tot);
                for (int t = 0; t < tot; t++) cnt[half(t) + 1]++;
                for (int q = 0; q < g.Hn; q++) cnt[q + 1] += cnt[q];
                for (int t = 0; t < tot; t++) ord[cnt[half(t)]++] = t;
                h.own.assign(C, {});
                h.cr.assign(C, 0);
                h.cbn.assign(C, 0);
                h.cb.assign(C, 0);
                h.cg.assign(C, 0);
                h.ref.assign(2 * (size_t)g.Hn, (uint16_t)kNoRef);
                for (int r = 0; r < w; r++) {
                    const int a = (int)((long long)tot * r / w), b = (int)((long long)tot * (r + 1) / w);
                    std::vector<int> part[4];
                    for (int q = a; q < b; q++) {
                        const int t = ord[q];
                        part[t >= nin ? 3 : (t < g.n0 ? 0 : (t < nin - g.nga ? 1 : 2))].push_back(t);
                    }
                    h.cr[r] = (int)part[0].size();
                    h.cbn[r] = (int)part[1].size();
                    h.cb[r] = (int)(part[1].size() + part[2].size());
                    h.cg[r] = (int)part[3].size();
                    std::vector<int>& o = h.own[r];
                    for (auto& p : part) o.insert(o.end(), p.begin(), p.end());
                    if (o.size() > kRefMask) refs_ok = false;
                    for (size_t i = 0; i < o.size(); i++) {
                        const int t = o[i];
                        const int sl = t >= nin ? h.gslot.v[t - nin] : (t >= g.n0 ? g.Hn : 0) + (h.hl.v[t] >> kEntHalf);
                        h.ref[sl] = (uint16_t)(r << kRefBits | (int)i);
                    }
                }
            }
            if (!refs_ok) continue;
            // uniform offsets of the values
            std::vector<CLev> base(n);
            // levels whose rows fit the threads are swept a visit at a time
            auto visit_fits = [&](int l) {
                const HostLevel& h = H[l0 + l];
                const int nin = SG[l0 + l].n0 + SG[l0 + l].n1;
                for (int r = 0; r < C; r++) {
                    std::vector<int> len;
                    for (int q = 0; q < h.cg[r]; q++) {
                        const int gi = h.own[r][h.cr[r] + h.cb[r] + q] - nin;
                        len.push_back(h.gptr.v[gi + 1] - h.gptr.v[gi]);
                        if (!len.back()) return false;
                    }
                    std::sort(len.begin(), len.end(), std::greater<int>());
                    if (std::max(h.cr[r], h.cb[r]) > kCoarseThreads ||
                        32 * row_jobs<T>(len).size() > (size_t)kCoarseThreads)
                        return false;
                }
                return nu1 < 256 && nu2 < 256;
            };
            std::vector<char> fits_(n);
            for (int l = 0; l < n; l++) fits_[l] = visit_fits(l);
            auto fits = [&](int l) { return fits_[l] != 0; };
            if (l0 == 0 && !fits(0)) continue;
            // the program
            prog.clear();
            {
                auto wide = [&](int l) { return H[l0 + l].wide != 0; };
                // a phase that reads level a and writes level b
                auto op = [&](unsigned code, int lv, int a, int b, unsigned fl, bool sync) {
                    const bool far = wide(a) || wide(b);
                    prog.push_back(code | (unsigned)lv << 8 | fl | (wide(b) ? kOpAll : 0u) | (far ? kOpFar : 0u) |
                                   (sync ? kOpWide : 0u));
                };
                auto sweep = [&](int l, bool red, unsigned fl, bool after) {
                    if (red) op(kOpRed, l, l, l, fl, wide(l));
                    op(kOpBlack, l, l, l, fl, wide(l));
                    op(kOpGhosts, l, l, l, fl, wide(l) || after);
                };
                op(kOpNone, 0, 0, 0, 0, wide(0));
                for (int l = 0; l + 1 < n; l++) {
                    const bool both = wide(l) || wide(l + 1);
                    if (fits(l)) {
                        const unsigned top = l0 + l > 0 ? kOpSkipRed : (f32 ? kOpSkipRed | kOpTop : kOpTop);
                        op(kOpVisit, l, l, l, (unsigned)nu1 << 24 | top | kOpDown, both);
                    } else {
                        for (int q = 0; q < nu1; q++) sweep(l, q > 0, 0, false);
                        op(kOpDefect, l, l, l, 0, both);
                    }
                    op(kOpRestrict, l + 1, l, l + 1, 0, both);
                }
                op(kOpSolve, n - 1, n - 1, n - 1, 0, wide(n - 1) || (n > 1 && wide(n - 2)));
                for (int l = n - 2; l >= 0; l--) {
                    op(kOpProlong, l, l + 1, l, 0, wide(l) || wide(l + 1));
                    if (fits(l))
                        op(kOpVisit, l, l, l, (unsigned)nu2 << 24 | kOpDelta | (l > 0 ? kOpLast : 0u),
                           wide(l) || (l > 0 && wide(l - 1)));
                    else
                    for (int q = 0; q < nu2; q++)
                        sweep(l, true, (q == 0 ? kOpDelta : 0u) | (q == nu2 - 1 && l > 0 ? kOpLast : 0u),
                              q == nu2 - 1 && l > 0 && wide(l - 1));
                }
            }
            d.nop = (int)prog.size();
            d.head_len = (int)up16(n * sizeof(CLev) + 4 * prog.size());
            size_t off = d.head_len;
            for (int l = l0; l < L; l++) {
                const HostLevel& h = H[l];
                CLev& c = base[l - l0];
                memset(&c, 0, sizeof c);
                size_t nx = 0, ng = 0;
                for (int r = 0; r < C; r++) {
                    nx = std::max(nx, h.own[r].size());
                    ng = std::max(ng, (size_t)h.cg[r]);
                }
                c.wide = h.wide;
                auto take = [&](int& o, size_t bytes) {
                    o = (int)off;
                    off += up16(bytes);
                };
                take(c.x, sizeof(T) * nx);
                take(c.y, sizeof(T) * nx);
                take(c.b, sizeof(T) * nx);
                take(c.d2, 2 * sizeof(T) * nx);
                take(c.snap, sizeof(T) * ng);
            }
            d.coef_at = (int)off;
            // coefficients: own offsets, the tables after the largest of them
            lev.assign((size_t)C * n, CLev{});
            size_t coef_max = 0, lists_max = 0;
            coef_tot = 0;
            for (int r = 0; r < C; r++) {
                size_t e = 0, lists = 0;
                d.coef_off[r] = (int)coef_tot;
                for (int l = l0; l < L; l++) {
                    CLev& c = lev[(size_t)r * n + l - l0];
                    const HostLevel& h = H[l];
                    c = base[l - l0];
                    c.cr = h.cr[r];
                    c.cbn = h.cbn[r];
                    c.cb = h.cb[r];
                    c.cg = h.cg[r];
                    c.nr = c.cr + c.cb;
                    c.nx = c.nr + c.cg;
                    c.coef = d.coef_at + (int)(sizeof(T) * e);
                    lists += 4 * D * (size_t)c.nr + (l + 1 < L ? 2 * (size_t)(c.cb + c.cg) << D : 0);
                    e += up16(sizeof(T) * ((size_t)(2 * D + 2) * c.nr + 2 * (size_t)c.nx)) / sizeof(T);
                }
                d.coef_len[r] = (int)e;
                coef_tot += e;
                coef_max = std::max(coef_max, e);
                lists_max = std::max(lists_max, lists);
            }
            d.tab_at = d.coef_at + (int)up16(sizeof(T) * coef_max);
            if (d.tab_at + lists_max > kCoarseSmem) continue;  // (before the tables are built)
            tab.clear();
            tab.reserve((size_t)C * (kCoarseSmem - d.tab_at));
            size_t tab_max = 0;
            for (int r = 0; r < C; r++) {
                const size_t t0 = tab.size();
                d.tab_off[r] = (int)t0;
                auto put = [&](const void* p, size_t bytes) {
                    const size_t o = tab.size();
                    tab.resize(o + up16(bytes));
                    if (bytes) memcpy(tab.data() + o, p, bytes);
                    return d.tab_at + (int)(o - t0);
                };
                // rows given in ghost order, stored longest first
                auto put_tab = [&](CTab& tb, const std::vector<int>& rp, const auto& ref, const std::vector<T>& val) {
                    const int cnt = (int)rp.size() - 1;
                    std::vector<uint16_t> idx(cnt);
                    for (int i = 0; i < cnt; i++) idx[i] = (uint16_t)i;
                    auto len = [&](int i) { return rp[i + 1] - rp[i]; };
                    std::stable_sort(idx.begin(), idx.end(), [&](int a, int b) { return len(a) > len(b); });
                    std::vector<int> p(1, 0), ln;
                    auto rf = ref;
                    std::vector<T> vl;
                    rf.clear();
                    for (int i : idx) {
                        rf.insert(rf.end(), ref.begin() + rp[i], ref.begin() + rp[i + 1]);
                        vl.insert(vl.end(), val.begin() + rp[i], val.begin() + rp[i + 1]);
                        p.push_back((int)rf.size());
                        ln.push_back(len(i));
                    }
                    tb.ptr = put(p.data(), 4 * p.size());
                    tb.ref = put(rf.data(), sizeof(rf[0]) * rf.size());
                    tb.val = put(vl.data(), sizeof(T) * vl.size());
                    tb.idx = put(idx.data(), 2 * idx.size());
                    const std::vector<unsigned> jobs = row_jobs<T>(ln);
                    tb.nw = (int)jobs.size();
                    tb.job = put(jobs.data(), 4 * jobs.size());
                };
                for (int l = l0; l < L; l++) {
                    CLev& c = lev[(size_t)r * n + l - l0];
                    const HostLevel& h = H[l];
                    const SGeo& g = SG[l];
                    const int nin = g.n0 + g.n1, nn = G[l].n;
                    std::vector<uint16_t> u;
                    std::vector<int> ptr;
                    std::vector<T> val;
                    // neighbours
                    u.assign((size_t)2 * D * c.nr + 1, 0);
                    for (int i = 0; i < c.nr; i++) {
                        const int t = h.own[r][i], e = h.hl.v[t], a = e & 1;
                        const int so = (t >= g.n0 ? 0 : g.Hn) + (e >> kEntHalf);
                        const int o[6] = {a, a - 1, g.H, -g.H, g.P, -g.P};
                        for (int q = 0; q < 2 * D; q++) u[(size_t)q * c.nr + i] = h.ref[so + o[q]];
                    }
                    c.nbr = put(u.data(), 2 * (size_t)2 * D * c.nr);
                    // composed ghost rows and rows of the defect
                    std::vector<unsigned> gr;
                    std::vector<uint16_t> rr;
                    std::vector<T> rv;
                    std::vector<int> rp;
                    ptr.assign(1, 0);
                    rp.assign(1, 0);
                    for (int q = 0; q < c.cg; q++) {
                        const int gi = h.own[r][c.nr + q] - nin;
                        for (int j = h.gptr.v[gi]; j < h.gptr.v[gi + 1]; j++) {
                            const int code = h.gcode.v[j];
                            unsigned ref;
                            int base = c.x;
                            if (code >= 0) {
                                ref = h.ref[code];
                            } else {
                                const unsigned w = ~(unsigned)code;
                                ref = h.ref[h.gslot.v[w >> 1]];
                                base = c.b;
                                if (!(w & 1u)) {  // snap holds the ghosts only
                                    const int o = (int)(ref >> kRefBits);
                                    ref -= (unsigned)(h.cr[o] + h.cb[o]);
                                    base = c.snap;
                                }
                            }
                            gr.push_back((ref >> kRefBits) << kAddrBits |
                                         (unsigned)(base + (int)(ref & kRefMask) * (int)sizeof(T)));
                            val.push_back((T)h.gval.v[j]);
                        }
                        ptr.push_back((int)gr.size());
                        for (int j = h.rptr.v[gi]; j < h.rptr.v[gi + 1]; j++) {
                            rr.push_back(h.ref[h.rslot.v[j]]);
                            rv.push_back((T)h.rval.v[j]);
                        }
                        rp.push_back((int)rr.size());
                    }
                    put_tab(c.g, ptr, gr, val);
                    put_tab(c.r, rp, rr, rv);
                    // coarse corners of the black nodes and the ghosts
                    auto coords = [&](int t, int* ii) {
                        int sl = t >= nin ? h.gslot.v[t - nin] : (t >= g.n0 ? g.Hn : 0) + (h.hl.v[t] >> kEntHalf);
                        const int col = sl >= g.Hn;
                        if (col) sl -= g.Hn;
                        const int row = sl / g.H;
                        ii[1] = D == 3 ? row % nn : row;
                        ii[2] = D == 3 ? row / nn : 0;
                        ii[0] = 2 * (sl % g.H) + ((col + ii[1] + ii[2]) & 1);
                    };
                    auto slot_of = [](const SGeo& q, int n_, int i, int j, int k) {
                        return ((i + j + k) & 1) * q.Hn + (i >> 1) + q.H * (j + n_ * k);
                    };
                    if (l + 1 < L) {
                        const HostLevel& hc = H[l + 1];
                        const SGeo& gc = SG[l + 1];
                        const int np = c.cb + c.cg;
                        u.assign(((size_t)np << D) + 1, (uint16_t)kNoRef);
                        for (int q = 0; q < np; q++) {
                            int ii[3];
                            coords(h.own[r][c.cr + q], ii);
                            for (int cc = 0; cc < (1 << D); cc++) {
                                int v[3] = {0, 0, 0};
                                bool dup = false;
                                for (int a = 0; a < D; a++) {
                                    const int upper = (cc >> a) & 1;
                                    dup = dup || (upper && !(ii[a] & 1));
                                    v[a] = (ii[a] >> 1) + (upper && (ii[a] & 1) ? 1 : 0);
                                }
                                if (!dup) u[(size_t)cc * np + q] = hc.ref[slot_of(gc, G[l + 1].n, v[0], v[1], v[2])];
                            }
                        }
                        c.pro = put(u.data(), 2 * ((size_t)np << D));
                    }
                    // rows of the restriction onto this level
                    if (l > l0) {
                        const HostLevel& hf = H[l - 1];
                        const SGeo& gf = SG[l - 1];
                        const int fn = G[l - 1].n, st[3] = {1, fn, fn * fn};
                        const int8_t* ft = hf.type.v.data();
                        ptr.assign(1, 0);
                        rr.clear();
                        rv.clear();
                        for (int i = 0; i < c.nr; i++) {
                            int ci[3];
                            coords(h.own[r][i], ci);
                            const int f[3] = {2 * ci[0], 2 * ci[1], 2 * ci[2]};
                            int p = 0, w[3][3] = {{0, 1, 0}, {0, 1, 0}, {0, 1, 0}};
                            for (int a = 0; a < D; a++) p += f[a] * st[a];
                            for (int a = 0; a < D; a++) {
                                const bool vl = ft[p - st[a]] == T_IN, vr = ft[p + st[a]] == T_IN;
                                w[a][0] = vl ? (vr ? 1 : 2) : 0;
                                w[a][1] = vl || vr ? 2 : 4;
                                w[a][2] = vr ? (vl ? 1 : 2) : 0;
                            }
                            int wc = 0;
                            auto add = [&](int a0, int a1, int a2, int iw) {
                                // black nodes away from the ghosts have no defect
                                const uint16_t ref = hf.ref[slot_of(gf, fn, a0, a1, a2)];
                                const int o = ref >> kRefBits, x = ref & (int)kRefMask;
                                if (x >= hf.cr[o] && x < hf.cr[o] + hf.cbn[o]) return;
                                rr.push_back(ref);
                                rv.push_back((T)iw / (T)(D == 2 ? 16 : 64));
                            };
                            for (int kk = 0; kk < (D == 2 ? 9 : 27); kk++) {
                                const int k0 = kk % 3 - 1, k1 = (kk / 3) % 3 - 1, k2 = D == 3 ? kk / 9 - 1 : 0;
                                const int iw = w[0][k0 + 1] * w[1][k1 + 1] * (D == 3 ? w[2][k2 + 1] : 1);
                                if (!iw) continue;
                                const int q = p + k0 + k1 * st[1] + k2 * st[2];
                                if ((!k0 && !k1 && !k2) || ft[q] != T_IN)
                                    wc += iw;
                                else
                                    add(f[0] + k0, f[1] + k1, f[2] + k2, iw);
                            }
                            add(f[0], f[1], f[2], wc);
                            ptr.push_back((int)rr.size());
                        }
                        c.cptr = put(ptr.data(), 4 * ptr.size());
                        c.cref = put(rr.data(), 2 * rr.size());
                        c.cval = put(rv.data(), sizeof(T) * rv.size());
                        ptr.assign(1, 0);
                        rr.clear();
                        rv.clear();
                        for (int q = 0; q < c.cg; q++) {
                            const int gi = h.own[r][c.nr + q] - nin;
                            for (int j = h.cptr.v[gi]; j < h.cptr.v[gi + 1]; j++) {
                                rr.push_back(hf.ref[h.cslot.v[j]]);
                                rv.push_back((T)h.cval.v[j]);
                            }
                            ptr.push_back((int)rr.size());
                        }
                        put_tab(c.c, ptr, rr, rv);
                    }
                }
                d.tab_len[r] = (int)(tab.size() - t0);
                tab_max = std::max(tab_max, tab.size() - t0);
            }
            // the coarsest inverse: own rows in shared memory where they fit
            d.ainv_at = d.tab_at + (int)up16(tab_max);
            const HostLevel& hc = H[L - 1];
            const int m = SG[L - 1].n0 + SG[L - 1].n1 + G[L - 1].ng;
            size_t rows_max = 0;
            int row0 = 0;
            for (int r = 0; r < C; r++) {
                CLev& c = lev[(size_t)r * n + n - 1];
                c.m = m;
                d.ainv_off[r] = row0 * m;
                d.ainv_len[r] = c.nx * m;
                row0 += c.nx;
                rows_max = std::max(rows_max, (size_t)c.nx * m);
            }
            (void)hc;
            // a copied piece starts on 16 bytes: rows of odd length may not
            bool stage_inv = d.ainv_at + up16(sizeof(T) * rows_max) <= kCoarseSmem;
            for (int r = 0; r < C; r++)
                if ((sizeof(T) * (size_t)d.ainv_off[r]) % 16) stage_inv = false;
            for (int r = 0; r < C; r++) {
                lev[(size_t)r * n + n - 1].ainv = stage_inv ? d.ainv_at : -1;
                if (!stage_inv) d.ainv_len[r] = 0;
            }
            smem = d.ainv_at + (stage_inv ? up16(sizeof(T) * rows_max) : 0);
            if (smem <= kCoarseSmem && cluster_fits<D, T>(C, smem)) {
                fit = true;
                break;
            }
        }
        if (fit) break;
    }
    if (!fit) return SULF_OK;
    const int n = L - l0, C = ncta;
    // device copies
    auto oom = [&] {
        err = "out of device memory";
        return SULF_ENOMEM;
    };
    auto grow = [&](auto*& p, size_t& cap, size_t bytes) {
        if (bytes <= cap && p) return true;
        p = (std::remove_reference_t<decltype(p)>)mem.get(bytes + 64);
        cap = bytes;
        return p != nullptr;
    };
    if (!grow(S.tab, S.tab_cap, tab.size()) || !grow(S.coef, S.coef_cap, sizeof(T) * coef_tot)) return oom();
    const int nb = SG[l0].n0 + SG[l0].n1 + G[l0].ng, nc = SG[L - 1].n0 + SG[L - 1].n1 + G[L - 1].ng;
    if (!grow(S.b, S.b_cap, sizeof(T) * nb)) return oom();
    std::vector<int> bpos(nb), cpos(nc), cntm(C);
    slots.resize(nb);
    {
        int at = 0;
        for (int r = 0; r < C; r++) {
            d.b_off[r] = at;
            for (int t : H[l0].own[r]) {
                const SGeo& g = SG[l0];
                const int nin = g.n0 + g.n1;
                bpos[t] = at;
                slots[at++] =
                    t >= nin ? H[l0].gslot.v[t - nin] : (t >= g.n0 ? g.Hn : 0) + (H[l0].hl.v[t] >> kEntHalf);
            }
        }
        at = 0;
        for (int r = 0; r < C; r++) {
            cntm[r] = (int)H[L - 1].own[r].size();
            for (int t : H[L - 1].own[r]) cpos[t] = at++;
        }
    }
    for (int r = C; r < kCoarseMaxCta; r++)
        d.tab_off[r] = d.tab_len[r] = d.coef_off[r] = d.coef_len[r] = d.ainv_off[r] = d.ainv_len[r] = d.b_off[r] = 0;
    std::vector<std::vector<CPerm>> perm(L);
    for (int l = l0; l < L; l++) {
        const SGeo& g = SG[l];
        perm[l].resize((size_t)g.n0 + g.n1 + G[l].ng);
        for (int r = 0; r < C; r++) {
            const CLev& c = lev[(size_t)r * n + l - l0];
            const int base = d.coef_off[r] + (int)((c.coef - d.coef_at) / (int)sizeof(T));
            for (int i = 0; i < c.nx; i++)
                perm[l][H[l].own[r][i]] = CPerm{base + i, c.nr, base + (2 * D + 2) * c.nr + i, c.nx};
        }
    }
    // (rebuilt for another threshold or cluster size: the old set's arrays,
    // which nothing in flight reads, where they are large enough)
    size_t used = 0;
    auto upload = [&](auto*& dst, const auto& v) {
        const size_t nb = sizeof(v[0]) * v.size();
        if (used == S.kept.size()) S.kept.push_back({nullptr, 0});
        auto& k = S.kept[used++];
        if (!k.first || k.second < nb) k = {mem.get(nb + 64), nb};
        dst = (std::remove_reference_t<decltype(dst)>)k.first;
        return dst && cudaMemcpyAsync(dst, v.data(), nb, cudaMemcpyHostToDevice, s) == cudaSuccess;
    };
    for (int l = 0; l < SULF_MAXLEV; l++) S.perm[l] = nullptr;
    for (int l = L - 1; l >= l0; l--)
        if (!upload(S.perm[l], perm[l])) return oom();
    std::vector<char> head((size_t)C * d.head_len, 0);
    for (int r = 0; r < C; r++) {
        memcpy(head.data() + (size_t)r * d.head_len, &lev[(size_t)r * n], n * sizeof(CLev));
        memcpy(head.data() + (size_t)r * d.head_len + n * sizeof(CLev), prog.data(), 4 * prog.size());
    }
    if (!upload(S.bpos, bpos) || !upload(S.cpos, cpos) || !upload(S.slot, slots) || !upload(S.head, head) ||
        !upload(S.cnt_m, cntm))
        return oom();
    d.head = S.head;
    d.tab = S.tab;
    d.coef = S.coef;
    d.ainv = V[L - 1].Ainv;
    d.b = S.b;
    d.slot = S.slot;
    d.X = V[l0].X;
    d.acc = l0 == 0 ? acc : nullptr;
    d.skip = l0 == 0 ? skip : nullptr;
    d.cnt_m = S.cnt_m;
    d.nlev = n;
    d.ncta = C;
    std::vector<CDesc<T>> dd(1, d);
    if (!upload(S.dev, dd)) return oom();
    if (cudaMemcpyAsync(S.tab, tab.data(), tab.size(), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemsetAsync(S.coef, 0, sizeof(T) * coef_tot, s) != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) {
        err = "coarse-level tables failed";
        return SULF_EDEVICE;
    }
    S.smem = smem;
    S.ncta = C;
    S.wide = H[l0].wide != 0;
    S.l0 = l0;
    return SULF_OK;
}

namespace {
template <int D, typename T>
int launch_clusters(int K, int ncta, size_t smem, const CDesc<T>* one, const CDesc<T>* const* many, const int* active,
                    cudaStream_t s) {
    raise_limits<D, T>();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(K * ncta);
    cfg.blockDim = dim3(kCoarseThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ncta;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = launch_pdl() ? 1 : 0;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_s_coarse<D, T>, one, many, active);
    if (e != cudaSuccess) note_launch_error(e, K * ncta, kCoarseThreads, smem);
    return 1;
}
}  // namespace

template <int D, typename T>
int launch_coarse(const CoarseSet<T>& S, cudaStream_t s) {
    return launch_clusters<D, T>(1, S.ncta, S.smem, S.dev, nullptr, nullptr, s);
}

template <int D, typename T>
int launch_coarse_batched(const CDesc<T>* const* descs, int K, const int* active, int ncta, size_t smem,
                          cudaStream_t s) {
    return launch_clusters<D, T>(K, ncta, smem, nullptr, descs, active, s);
}

#define SULF_INST_COARSE(D, T)                                                                                      \
    template int build_coarse<D, T>(CoarseSet<T>&, const LevelGeo*, const SGeo*, const SVec<T>*, int, int, int, int, \
                                    int, double*, const int*, DevMem&, cudaStream_t, std::string&);                                            \
    template int launch_coarse<D, T>(const CoarseSet<T>&, cudaStream_t);                                          \
    template int launch_coarse_batched<D, T>(const CDesc<T>* const*, int, const int*, int, size_t, cudaStream_t);
SULF_INST_COARSE(2, double)
SULF_INST_COARSE(2, float)
SULF_INST_COARSE(3, double)
SULF_INST_COARSE(3, float)

}  // namespace sulf
