// Kernels and per-level data of the multigrid cycle on the equation for s
// (schur.cuh).
#include <mutex>

#include <cooperative_groups.h>

#include "schur.cuh"

namespace sulf {

using stages::abs_bits;
using stages::block_max;
using stages::find_instance;
using stages::fmadd;
using stages::kGopLanes;

namespace {

constexpr int kT = kNodeThreads;

// node coordinates of a half index
template <int D>
__device__ __forceinline__ void half_coords(int h, int a, int H, int n, int* ii) {
    const unsigned row = (unsigned)h / (unsigned)H;
    ii[0] = 2 * (int)((unsigned)h - row * (unsigned)H) + a;
    if (D == 3) {
        const unsigned k = row / (unsigned)n;
        ii[1] = (int)(row - k * (unsigned)n);
        ii[2] = (int)k;
    } else {
        ii[1] = (int)row;
        ii[2] = 0;
    }
}

template <int D>
__device__ __forceinline__ int slot_of(int i, int j, int k, int H, int P, int Hn) {
    return ((i + j + (D == 3 ? k : 0)) & 1) * Hn + (i >> 1) + H * j + (D == 3 ? P * k : 0);
}

// the node at list position t (inside nodes, then ghosts): its slot and box node
template <int D, typename T>
__device__ __forceinline__ int list_slot(const SLev<D, T>& L, int t, int& p) {
    if (t < L.n0 + L.n1) {
        const int e = L.hl[t], h = e >> kEntHalf;
        int ii[3];
        half_coords<D>(h, e & 1, L.H, L.n, ii);
        p = ii[0] + L.n * (ii[1] + (D == 3 ? L.n * ii[2] : 0));
        return (t >= L.n0 ? L.Hn : 0) + h;
    }
    const int g = t - L.n0 - L.n1;
    p = L.gidx[g];
    return L.gslot[g];
}

// half-index offsets of the axis neighbours (all of the other colour) of a
// node whose x index has parity a
template <int D, typename T>
__device__ __forceinline__ void nbr_offsets(const SLev<D, T>& L, int a, int* o) {
    o[0] = a;
    o[1] = a - 1;
    o[2] = L.H;
    o[3] = -L.H;
    if (D == 3) {
        o[4 % (2 * D)] = L.P;
        o[5 % (2 * D)] = -L.P;
    }
}

// ---------------------------------------------------------------------------
// set-up of a linear solve

template <typename T>
__device__ __forceinline__ void c_row(const Coef<T>& c, T s, T cp, T& ph, T& pcs, T& pcc) {
    ph = c.alpha * cp + c.beta;
    pcs = c.a2ms * ph * cp;
    pcc = c.idt + c.a2ms * (c.alpha * s * cp + ph * s);
}

// FINE: the finest level of a linear solve (T = double), U the FP32 finest
// level of mixed precision (MIXED)
template <int D, typename T, bool FINE, bool MIXED>
__global__ void __launch_bounds__(kT) k_s_rho(SLev<D, T> L, SLev<D, float> U, const typename V2<T>::t* __restrict__ Wc,
                                               Coef<T> c, const double2* __restrict__ F, double* __restrict__ tt,
                                               double* __restrict__ uu) {
    pdl_enter();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int nin = L.n0 + L.n1;
    if (t >= nin + L.ng) return;
    int p;
    const int sl = list_slot<D, T>(L, t, p);
    const typename V2<T>::t w = Wc[p];
    T ph, pcs, pcc;
    c_row<T>(c, w.x, w.y, ph, pcs, pcc);
    const T inv = (T)1 / pcc;
    const T rho = pcs * inv, C = c.kap * c.alpha * w.x;
    L.rho[sl] = rho;
    L.cs[sl] = C;
    if (!MIXED && L.perm) {
        const CPerm q = L.perm[t];
        L.cf[q.roff] = rho;
        L.cf[q.roff + q.nx] = C;
    }
    if (FINE) {
        const double2 f = F[p];
        const double t0 = f.y * (double)inv;
        tt[sl] = t0;
        uu[sl] = (double)(c.kap * ph);
        if (MIXED) {
            U.rho[sl] = (float)rho;
            U.cs[sl] = (float)C;
            if (U.perm) {
                const CPerm q = U.perm[t];
                U.cf[q.roff] = (float)rho;
                U.cf[q.roff + q.nx] = (float)C;
            }
            L.X[sl] = 0;
            if (t >= nin) {
                L.b[t] = (T)f.x;
                U.b[t] = (float)f.x;
                if (U.bpos) U.bf[U.bpos[t]] = (float)f.x;
                U.X[sl] = 0.f;
                U.D2[sl] = make_float2((float)-t0, (float)(-(double)C * t0));
            }
        } else if (t >= nin) {
            // x = 0 is off the ghosts' c rows by -t in the first sweep
            typename V2<T>::t d;
            d.x = (T)-t0;
            d.y = (T)(-(double)C * t0);
            L.D2[sl] = d;
            L.X[sl] = 0;
            L.b[t] = (T)f.x;
            if (L.bpos) L.bf[L.bpos[t]] = (T)f.x;
        }
    }
}

template <int D, typename T>
__global__ void __launch_bounds__(kT) k_s_coefs(SLev<D, T> L, const typename V2<T>::t* __restrict__ Wc, Coef<T> c) {
    pdl_enter();
    typedef typename V2<T>::t T2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= L.n0 + L.n1) return;
    const int colour = t >= L.n0;
    const int e = L.hl[t], h = e >> kEntHalf;
    int ii[3], o[2 * D];
    half_coords<D>(h, e & 1, L.H, L.n, ii);
    nbr_offsets<D, T>(L, e & 1, o);
    const int p = ii[0] + L.n * (ii[1] + (D == 3 ? L.n * ii[2] : 0));
    const int st[3] = {1, L.n, L.n * L.n};
    const int sl = colour * L.Hn + h, so = (1 - colour) * L.Hn + h;
    const T2 w = Wc[p];
    const T s = w.x, cp = w.y;
    T ph, pcs, pcc;
    c_row<T>(c, s, cp, ph, pcs, pcc);
    T sg = 0, se = 0;
    T2 wq[2 * D];
    T rq[2 * D];
#pragma unroll
    for (int q = 0; q < 2 * D; q++) {
        wq[q] = Wc[(q & 1) ? p - st[q >> 1] : p + st[q >> 1]];
        rq[q] = L.rho[so + o[q]];
    }
    T g[2 * D];
#pragma unroll
    for (int q = 0; q < 2 * D; q++) {
        const T gq = c.kap * ((c.alpha * wq[q].y + c.beta) + ph);
        const T eq = c.kap * c.alpha * (s - wq[q].x);
        sg += gq;
        se += eq;
        g[q] = fmadd(eq, rq[q], gq);
        L.gt[q * L.gs + t] = g[q];
    }
    const T Pss = ph * c.idt + c.a2mc * ph * cp + sg;
    const T Psc = c.alpha * s * c.idt + c.a2mc * (c.alpha * s * cp + ph * s) + se;
    const T dd = Pss - Psc * L.rho[sl];
    const T di = (T)1 / dd;
    L.dd[t] = dd;
    L.di[t] = di;
    if (L.perm) {
        const CPerm q = L.perm[t];
#pragma unroll
        for (int a = 0; a < 2 * D; a++) L.cf[q.off + a * q.stride] = g[a] * di;
        L.cf[q.off + 2 * D * q.stride] = dd;
        L.cf[q.off + (2 * D + 1) * q.stride] = di;
    }
}

// The finest level's rows in FP64, with the right-hand side b~ and the start
// of the first sweep, and in mixed precision the FP32 copies.  The FP64 pipe
// bounds it, so what a node gives its neighbours (u = kappa phi, C, rho, t)
// comes from k_s_rho: six FP64 instructions per neighbour (g = u_q + u_p, e =
// C_p - C_q, gt = g + e rho_q, the sums of u_q, C_q and e t_q).
template <int D, bool MIXED>
__global__ void __launch_bounds__(kT) k_s_coefs_fine(const __grid_constant__ SLev<D, double> L,
                                                      const __grid_constant__ SLev<D, float> U,
                                                      const double2* __restrict__ Wc, Coef<double> c,
                                                      const double2* __restrict__ F, const double* __restrict__ tt,
                                                      const double* __restrict__ uu) {
    pdl_enter();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= L.n0 + L.n1) return;
    const int colour = t >= L.n0;
    const int e = L.hl[t], h = e >> kEntHalf;
    int ii[3], o[2 * D];
    half_coords<D>(h, e & 1, L.H, L.n, ii);
    nbr_offsets<D, double>(L, e & 1, o);
    const int p = ii[0] + L.n * (ii[1] + (D == 3 ? L.n * ii[2] : 0));
    const int sl = colour * L.Hn + h, so = (1 - colour) * L.Hn + h;
    const double2 w = Wc[p], f = F[p];
    const double up = uu[sl], Cp = L.cs[sl], rho = L.rho[sl], tp = tt[sl];
    double uq[2 * D], cq[2 * D], rq[2 * D], tq[2 * D];
#pragma unroll
    for (int q = 0; q < 2 * D; q++) {
        uq[q] = uu[so + o[q]];
        cq[q] = L.cs[so + o[q]];
        rq[q] = L.rho[so + o[q]];
        tq[q] = tt[so + o[q]];
    }
    double su = 0, sc = 0, et = 0, g[2 * D];
#pragma unroll
    for (int q = 0; q < 2 * D; q++) {
        const double eq = Cp - cq[q];
        su += uq[q];
        sc += eq;
        g[q] = fma(eq, rq[q], uq[q] + up);
        et = fma(eq, tq[q], et);
        L.gt[q * L.gs + t] = g[q];
    }
    const double ph = fma(c.alpha, w.y, c.beta), as = c.alpha * w.x;
    const double Pss = fma(ph, fma(c.a2mc, w.y, c.idt), fma(2.0 * D, up, su));
    const double Psc = fma(as, c.idt, fma(c.a2mc, fma(as, w.y, ph * w.x), sc));
    const double dd = fma(-Psc, rho, Pss), di = 1.0 / dd;
    const double bs = fma(-Psc, tp, f.x), b = bs - et;
    L.dd[t] = dd;
    L.di[t] = di;
    L.b[t] = b;
    if (MIXED) {
#pragma unroll
        for (int q = 0; q < 2 * D; q++) U.gt[q * U.gs + t] = (float)g[q];
        const float df = (float)di;
        U.dd[t] = (float)dd;
        U.di[t] = df;
        U.b[t] = (float)b;
        if (U.perm) {
            const CPerm q = U.perm[t];
#pragma unroll
            for (int a = 0; a < 2 * D; a++) U.cf[q.off + a * q.stride] = (float)g[a] * df;
            U.cf[q.off + 2 * D * q.stride] = (float)dd;
            U.cf[q.off + (2 * D + 1) * q.stride] = df;
            U.bf[U.bpos[t]] = (float)b;
        }
        // the first red half-sweep from zero, the neighbours' x^c = 0 off their c rows
        if (!colour) U.X[sl] = (float)bs * df;
    } else {
        if (L.perm) {
            const CPerm q = L.perm[t];
#pragma unroll
            for (int a = 0; a < 2 * D; a++) L.cf[q.off + a * q.stride] = g[a] * di;
            L.cf[q.off + 2 * D * q.stride] = dd;
            L.cf[q.off + (2 * D + 1) * q.stride] = di;
            L.bf[L.bpos[t]] = b;
        }
        if (!colour) L.X[sl] = bs * di;
    }
}

// ---------------------------------------------------------------------------
// relaxation

// Each phase of the cycle is a function of a level and a thread's place in its
// work; one kernel takes the level of one domain, another the levels of many
// (lock-step batching): CTA b serves the domain i with pre[i] <= b < pre[i+1].
template <int D, typename T, bool DELTA>
__device__ __forceinline__ void s_relax(const SLev<D, T>& L, int t, int colour, bool snap, bool use_skip,
                                        bool use_acc) {
    typedef typename V2<T>::t T2;
    const int cnt = colour ? L.n1 : L.n0, pos = (colour ? L.n0 : 0) + t;
    // the row is fixed during the linear solve: fetched while the previous
    // kernel is still running
    int e = 0, o[2 * D];
    T g[2 * D], di = 0, cp = 0;
    if (t < cnt) {
        e = L.hl[pos];
#pragma unroll
        for (int q = 0; q < 2 * D; q++) g[q] = L.gt[q * L.gs + pos];
        di = L.di[pos];
        if (DELTA && (colour == 0 || (e & 2))) cp = L.cs[colour * L.Hn + (e >> kEntHalf)];
    }
    nbr_offsets<D, T>(L, e & 1, o);
    const int sg = snap && t < L.ng ? L.gslot[t] : 0;
    pdl_enter();
    if (use_skip && *L.skip) return;
    if (snap && t < L.ng) L.snap[t] = L.X[sg];
    if (t >= cnt) return;
    const int h = e >> kEntHalf, so = (1 - colour) * L.Hn + h, sl = colour * L.Hn + h;
    T r = L.b[pos];
    T x[2 * D];
#pragma unroll
    for (int q = 0; q < 2 * D; q++) x[q] = L.X[so + o[q]];
    if (DELTA) {
        // red inside nodes are on their c rows (their entries of D2 stay
        // zero): only a black node next to a ghost has terms
        if (colour == 0 || (e & 2)) {
            T2 d[2 * D];
#pragma unroll
            for (int q = 0; q < 2 * D; q++) d[q] = L.D2[so + o[q]];
            T sd = d[0].x, sc = d[0].y;
#pragma unroll
            for (int q = 1; q < 2 * D; q++) {
                sd += d[q].x;
                sc += d[q].y;
            }
            r = fmadd(-cp, sd, r + sc);
        }
    }
#pragma unroll
    for (int q = 0; q < 2 * D; q++) r = fmadd(g[q], x[q], r);
    r *= di;
    L.X[sl] = r;
    if (use_acc) L.acc[sl] += (double)r;
}

// The red half-sweep that opens an FP64 cycle, from the defects that the norm
// of the cycle before left in R: x + r / dd is what the row gives, and takes 36
// instead of 84 bytes a node (3-D) and one FP64 instruction instead of seven
// (257^3 box, two CN steps: 77.4 -> 76.2 and 80.6 -> 79.6 ms).
template <int D, typename T>
__device__ __forceinline__ void s_correct(const SLev<D, T>& L, int t) {
    int h = 0;
    T di = 0;
    if (t < L.n0) {
        h = L.hl[t] >> kEntHalf;
        di = L.di[t];
    }
    pdl_enter();
    if (*L.skip || t >= L.n0) return;
    L.X[h] = fmadd(L.R[h], di, L.X[h]);
}

template <int D, typename T>
__device__ __forceinline__ T ghost_input(const SLev<D, T>& L, int code) {
    if (code >= 0) return L.X[code];
    const unsigned u = ~(unsigned)code;
    return (u & 1u) ? L.b[L.n0 + L.n1 + (u >> 1)] : L.snap[u >> 1];
}

// The threads of a kernel over the ghosts' rows: one for each of the ng1 short
// rows, `mid` lanes for each of the ng8 next, `most` for each longer one, every
// part rounded up to whole warps.  On the flat parts of a boundary a composed
// row has 4 entries, on an edge of a box 50 to 500: eight lanes for all left
// most lanes idle and the long rows as a tail (257^3 box FP64: 37.6 us).
struct GhostPart {
    int g, lane, lanes;
    bool on;
};
__host__ __device__ __forceinline__ int up32(int n) { return (n + 31) & ~31; }
template <int D, typename T>
__host__ __device__ __forceinline__ int ghost_threads(const SLev<D, T>& L, int mid, int most) {
    return up32(L.ng1) + up32(L.ng8 * mid) + up32((L.ng - L.ng1 - L.ng8) * most);
}
template <int D, typename T>
__device__ __forceinline__ GhostPart ghost_part(const SLev<D, T>& L, int t, int mid, int most) {
    GhostPart p;
    const int t8 = up32(L.ng1), tx = t8 + up32(L.ng8 * mid);
    if (t < t8) {
        p.lanes = 1;
        p.lane = 0;
        p.g = t;
        p.on = t < L.ng1;
    } else if (t < tx) {
        p.lanes = mid;
        p.lane = (t - t8) % mid;
        p.g = L.ng1 + (t - t8) / mid;
        p.on = p.g < L.ng1 + L.ng8;
    } else {
        p.lanes = most;
        p.lane = (t - tx) % most;
        p.g = L.ng1 + L.ng8 + (t - tx) / most;
        p.on = p.g < L.ng;
    }
    p.g = p.on ? L.gord[p.g] : 0;
    return p;
}
// sum over the lanes of a part (every lane of the warp calls it)
template <typename T>
__device__ __forceinline__ T part_sum(T v, int lanes) {
    for (int o = lanes >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// all passes of a sweep's ghost relaxation, one composed row per ghost
constexpr int kGopPre = 4;
template <int D, typename T>
__device__ __forceinline__ void s_ghosts(const SLev<D, T>& L, int t, bool use_skip, bool use_acc) {
    const GhostPart p = ghost_part<D, T>(L, t, kGopLanes, 32);
    int beg = 0, end = 0, sl = 0;
    int cd[kGopPre];
    T w[kGopPre];
    if (p.on) {
        beg = L.gptr[p.g] + p.lane;
        end = L.gptr[p.g + 1];
#pragma unroll
        for (int i = 0; i < kGopPre; i++) {
            const int j = beg + i * p.lanes;
            cd[i] = j < end ? L.gcode[j] : 0;
            w[i] = j < end ? L.gval[j] : (T)0;
        }
        sl = L.gslot[p.g];
    }
    pdl_enter();
    if (use_skip && *L.skip) return;
    T v = 0;
    if (p.on) {
        for (int j = beg;;) {
            T u[kGopPre];
#pragma unroll
            for (int i = 0; i < kGopPre; i++) u[i] = j + i * p.lanes < end ? ghost_input<D, T>(L, cd[i]) : (T)0;
#pragma unroll
            for (int i = 0; i < kGopPre; i++)
                if (j + i * p.lanes < end) v = fmadd(w[i], u[i], v);
            j += kGopPre * p.lanes;
            if (j >= end) break;
#pragma unroll
            for (int i = 0; i < kGopPre; i++) {
                const int q = j + i * p.lanes < end ? j + i * p.lanes : j;
                cd[i] = L.gcode[q];
                w[i] = L.gval[q];
            }
        }
    }
    v = part_sum<T>(v, p.lanes);
    if (!p.on || p.lane != 0) return;
    L.X[sl] = v;
    if (use_acc) L.acc[sl] += (double)v;
}

// ---------------------------------------------------------------------------
// defect

template <int D, typename T>
__device__ __forceinline__ T inside_defect(const SLev<D, T>& L, int pos, int colour, int h, int a, const T* g, T dd) {
    int o[2 * D];
    nbr_offsets<D, T>(L, a, o);
    const int so = (1 - colour) * L.Hn + h;
    T x[2 * D];
#pragma unroll
    for (int q = 0; q < 2 * D; q++) x[q] = L.X[so + o[q]];
    T r = fmadd(-dd, L.X[colour * L.Hn + h], L.b[pos]);
#pragma unroll
    for (int q = 0; q < 2 * D; q++) r = fmadd(g[q], x[q], r);
    return r;
}

// b - row . x of a ghost by its lanes; every lane of the warp calls it, lane 0
// holds the result
template <int D, typename T>
__device__ __forceinline__ T ghost_defect(const SLev<D, T>& L, const GhostPart& p) {
    T v = 0;
    if (p.on) {
        const int end = L.rptr[p.g + 1];
        for (int j = L.rptr[p.g] + p.lane; j < end; j += p.lanes) v = fmadd(L.rval[j], L.X[L.rslot[j]], v);
    }
    v = part_sum<T>(v, p.lanes);
    return p.on && p.lane == 0 ? L.b[L.n0 + L.n1 + p.g] - v : (T)0;
}

template <int D, typename T, bool NORM>
__device__ __forceinline__ void s_residual(const SLev<D, T>& L, int t, unsigned long long* norm) {
    const int nin = L.n0 + L.nga, nrow = up32(nin);  // rows of inside nodes, in whole warps
    int e = 0, pos = 0, colour = 0;
    T g[2 * D], dd = 0;
    if (t < nin) {
        colour = t >= L.n0;
        pos = colour ? L.n1 - L.nga + t : t;
        e = L.hl[pos];
#pragma unroll
        for (int q = 0; q < 2 * D; q++) g[q] = L.gt[q * L.gs + pos];
        dd = L.dd[pos];
    }
    pdl_enter();
    if (NORM && t == 0) *L.skip = 0;  // the next cycle runs its first sweep
    T r = 0;
    if (t < nrow) {
        if (t < nin) {
            r = inside_defect<D, T>(L, pos, colour, e >> kEntHalf, e & 1, g, dd);
            // (with the norm: the red ones for the next cycle, s_correct)
            if (!NORM || !colour) L.R[colour * L.Hn + (e >> kEntHalf)] = r;
        }
    } else {
        const GhostPart p = ghost_part<D, T>(L, t - nrow, kGopLanes, kGopLanes);
        r = ghost_defect<D, T>(L, p);
        if (!NORM && p.on && p.lane == 0) L.R[L.gslot[p.g]] = r;
    }
    if (NORM) block_max(abs_bits(r), norm);
}

// mixed precision: the FP64 defect of every row into the FP32 right-hand
// side; the FP32 error starts with its red half-sweep from zero
template <int D>
__device__ __forceinline__ void s_outer(const SLev<D, double>& L, const SLev<D, float>& U, int t,
                                        unsigned long long* norm) {
    const int nin = L.n0 + L.n1, nrow = up32(nin);
    int e = 0;
    double g[2 * D], dd = 0;
    float df = 0;
    const int colour = t >= L.n0;
    if (t < nin) {
        e = L.hl[t];
#pragma unroll
        for (int q = 0; q < 2 * D; q++) g[q] = L.gt[q * L.gs + t];
        dd = L.dd[t];
        if (!colour) df = U.di[t];
    }
    pdl_enter();
    if (t == 0) *U.skip = 0;
    double r = 0;
    if (t < nrow) {
        if (t < nin) {
            const int h = e >> kEntHalf;
            r = inside_defect<D, double>(L, t, colour, h, e & 1, g, dd);
            U.b[t] = (float)r;
            if (U.bpos) U.bf[U.bpos[t]] = (float)r;
            if (!colour) U.X[h] = (float)r * df;
        }
    } else {
        const GhostPart p = ghost_part<D, double>(L, t - nrow, kGopLanes, kGopLanes);
        r = ghost_defect<D, double>(L, p);
        if (p.on && p.lane == 0) {
            U.b[nin + p.g] = (float)r;
            if (U.bpos) U.bf[U.bpos[nin + p.g]] = (float)r;
            U.X[L.gslot[p.g]] = 0.f;
        }
    }
    block_max(abs_bits(r), norm);
}

// ---------------------------------------------------------------------------
// transfers

// boundary-aware full weighting of the finer level's defect (Eqs. Fstencil,
// Fstencilgen) at a coarse inside node whose fine neighbourhood holds nodes
// that are not inside, or black nodes with a defect of their own; m: the
// members that are inside nodes.  Weights are powers of two over 4^D, built
// from their exponents (mg_stages.cuh).
template <int D, typename T>
__device__ __forceinline__ T restrict_near(const SLev<D, T>& F, int tw, unsigned m) {
    constexpr int K = D == 2 ? 9 : 27, mid = K / 2, pw[3] = {1, 3, 9};
    int e[3][3];  // per axis: log2 of the weight times 4, or -16 (weight 0)
#pragma unroll
    for (int a = 0; a < D; a++) {
        const bool vl = (m >> (mid - pw[a])) & 1u, vr = (m >> (mid + pw[a])) & 1u;
        e[a][0] = vl ? (vr ? 0 : 1) : -16;
        e[a][1] = vl || vr ? 1 : 2;
        e[a][2] = vr ? (vl ? 0 : 1) : -16;
    }
    // the twin (2I, 2J, 2K) is red at an even x index: the members along x lie
    // at half indices -1, 0 (odd x) or 0 (even x) of its row
    T v[K];
#pragma unroll
    for (int kk = 0; kk < K; kk++) {
        const int k0 = kk % 3 - 1, k1 = (kk / 3) % 3 - 1, k2 = D == 3 ? kk / 9 - 1 : 0;
        const int odd = (k0 + k1 + k2) & 1;
        v[kk] = (m >> kk) & 1u ? F.R[tw + odd * F.Hn + (k0 < 0 ? -1 : 0) + k1 * F.H + (D == 3 ? k2 * F.P : 0)] : (T)0;
    }
    T acc = 0;
    int wc = 0;
#pragma unroll
    for (int kk = 0; kk < K; kk++) {
        const int s = e[0][kk % 3] + e[1][(kk / 3) % 3] + (D == 3 ? e[2][kk / 9] : 0);
        if (s < 0) continue;
        if (kk == mid || !((m >> kk) & 1u))
            wc += 1 << s;
        else
            acc = fmadd(stages::pow2_weight<D, T>(s), v[kk], acc);
    }
    return fmadd((T)wc * stages::pow2_weight<D, T>(0), v[mid], acc);
}

// the finer level's defect onto the coarse level's right-hand side; the coarse
// error starts with its red half-sweep from zero
template <int D, typename T>
__device__ __forceinline__ void s_restrict(const SLev<D, T>& F, const SLev<D, T>& C, int t) {
    const int nin = C.n0 + C.n1, nreg = C.nreg0 + C.nreg1, freg = up32(nreg), nrow = freg + up32(nin - nreg);
    // regular nodes, then (from a whole warp on) the others
    int pos = -1, tw = 0, e = 0;
    unsigned m = 0;
    T di = 0;
    if (t < nreg) {
        pos = t < C.nreg0 ? t : C.n0 + t - C.nreg0;
    } else if (t >= freg && t < nrow) {
        const int u = t - freg, near0 = C.n0 - C.nreg0;
        if (u < nin - nreg) pos = u < near0 ? C.nreg0 + u : C.n0 + C.nreg1 + u - near0;
    }
    if (pos >= 0) {
        tw = C.twin[pos];
        e = C.hl[pos];
        if (t >= freg) m = (unsigned)C.mask[pos];
        if (pos < C.n0) di = C.di[pos];
    }
    pdl_enter();
    if (t < nrow) {
        if (pos < 0) return;
        T r;
        if (t < freg) {
            // black members (weights of the faces and corners) have no defect
            const T* R = F.R + tw;
            const int H = F.H, P = F.P;
            const T c0 = R[0];
            T s = (R[H] + R[H - 1]) + (R[-H] + R[-H - 1]);
            if (D == 3) {
                s += (R[P] + R[P - 1]) + (R[-P] + R[-P - 1]);
                s += (R[P + H] + R[P - H]) + (R[H - P] + R[-H - P]);
                r = (T)0.125 * c0 + (T)0.03125 * s;
            } else {
                r = (T)0.25 * c0 + (T)0.0625 * s;
            }
        } else {
            r = restrict_near<D, T>(F, tw, m);
        }
        if (C.bpos) {
            C.bf[C.bpos[pos]] = r;
        } else {
            C.b[pos] = r;
            C.X[(pos >= C.n0 ? C.Hn : 0) + (e >> kEntHalf)] = pos < C.n0 ? r * di : (T)0;
        }
    } else {
        const int gi = (t - nrow) / kGopLanes, ln = (t - nrow) % kGopLanes;
        T v = 0;
        if (gi < C.ng) {
            const int end = C.cptr[gi + 1];
            for (int j = C.cptr[gi] + ln; j < end; j += kGopLanes) v = fmadd(C.cval[j], F.R[C.cslot[j]], v);
        }
        v = stages::gop_reduce<T>(v);
        if (gi < C.ng && ln == 0) {
            if (C.bpos) {
                C.bf[C.bpos[nin + gi]] = v;
            } else {
                C.b[nin + gi] = v;
                C.X[C.gslot[gi]] = 0;
            }
        }
    }
}

// (bi/tri)linear interpolation of the coarse error, renormalised over the
// active corners (Sec. 3.5.3), at the black nodes and the ghosts; the
// corners' x^c is -rho x^s
template <int D, typename T>
__device__ __forceinline__ void s_prolong(const SLev<D, T>& F, const SLev<D, T>& C, int t) {
    typedef typename V2<T>::t T2;
    const bool on = t < F.n1 + F.ng;
    int cn[1 << D];
    T cr[1 << D];
    unsigned use = 0;
    int sl = 0, pair = -1;  // a black node on a coarse line: the two corners along this axis
    T rho = 0, Cs = 0;
    if (on) {
        int ii[3];
        bool all = false;
        if (t < F.n1) {
            const int e = F.hl[F.n0 + t];
            sl = F.Hn + (e >> kEntHalf);
            half_coords<D>(e >> kEntHalf, e & 1, F.H, F.n, ii);
            all = e & 4;
            if (all && (D == 2 || !(ii[0] & ii[1] & ii[2] & 1))) pair = ii[0] & 1 ? 0 : (ii[1] & 1 ? 1 : 2);
        } else {
            sl = F.gslot[t - F.n1];
            stages::box_coords<D>(F.gidx[t - F.n1], F.n, ii);
        }
        rho = F.rho[sl];
        Cs = F.cs[sl];
        if (pair >= 0) {
            int q[3] = {ii[0] >> 1, ii[1] >> 1, D == 3 ? ii[2] >> 1 : 0};
            cn[0] = slot_of<D>(q[0], q[1], q[2], C.H, C.P, C.Hn);
            cn[1] = slot_of<D>(q[0] + (pair == 0), q[1] + (pair == 1), q[2] + (pair == 2), C.H, C.P, C.Hn);
            cr[0] = C.rho[cn[0]];
            cr[1] = C.rho[cn[1]];
        } else {
#pragma unroll
            for (int cc = 0; cc < (1 << D); cc++) {
                int q[3] = {0, 0, 0};
                bool dup = false;
#pragma unroll
                for (int a = 0; a < D; a++) {
                    const int up = (cc >> a) & 1;
                    if (up && !(ii[a] & 1)) dup = true;
                    q[a] = (ii[a] >> 1) + (up && (ii[a] & 1) ? 1 : 0);
                }
                cn[cc] = slot_of<D>(q[0], q[1], q[2], C.H, C.P, C.Hn);
                if (dup) continue;
                if (!all) {
                    const int8_t ty = C.type[q[0] + C.n * (q[1] + (D == 3 ? C.n * q[2] : 0))];
                    if (ty != T_IN && ty != T_GHOST) continue;
                }
                use |= 1u << cc;
                cr[cc] = C.rho[cn[cc]];
            }
        }
    }
    pdl_enter();
    if (!on) return;
    T2 d;
    d.x = 0;
    d.y = 0;
    T x = F.X[sl], ps = 0, pc = 0, r = 0;
    if (pair >= 0) {
        const T v0 = C.X[cn[0]], v1 = C.X[cn[1]];
        ps = v0 + v1;
        pc = fmadd(-cr[1], v1, -cr[0] * v0);
        r = (T)0.5;
    } else if (use) {
        T v[1 << D];
#pragma unroll
        for (int cc = 0; cc < (1 << D); cc++) v[cc] = (use >> cc) & 1u ? C.X[cn[cc]] : (T)0;
#pragma unroll
        for (int cc = 0; cc < (1 << D); cc++)
            if ((use >> cc) & 1u) {
                ps += v[cc];
                pc = fmadd(-cr[cc], v[cc], pc);
            }
        r = stages::inv_count<T>(__popc(use));
    }
    if (pair >= 0 || use) {
        F.X[sl] = fmadd(ps, r, x);
        // off the c row by delta = x^c + rho x^s of the correction
        d.x = fmadd(rho, ps, pc) * r;
        d.y = Cs * d.x;
    }
    F.D2[sl] = d;
}

// coarse (s, c) by injection; a coarse ghost whose fine twin is inactive takes
// the mean over the active fine 3^d neighbourhood
template <int D, typename TF, typename T>
__global__ void __launch_bounds__(kT) k_inject_to(stages::Lists ls, int cn, const int8_t* __restrict__ ftype, int fn,
                                                   const typename V2<TF>::t* __restrict__ fW,
                                                   typename V2<T>::t* __restrict__ cW) {
    pdl_enter();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ls.n0 + ls.n1 + ls.ng) return;
    int kind, gi, ii[3];
    const long long I = stages::list_node(ls, t, kind, gi);
    stages::box_coords<D>(I, cn, ii);
    const int f = 2 * ii[0] + fn * (2 * ii[1] + (D == 3 ? fn * 2 * ii[2] : 0));
    typename V2<T>::t out;
    const int8_t tf = ftype[f];
    if (tf == T_IN || tf == T_GHOST) {
        const typename V2<TF>::t v = fW[f];
        out.x = (T)v.x;
        out.y = (T)v.y;
        cW[I] = out;
        return;
    }
    constexpr int K = D == 2 ? 9 : 27;
    int8_t ty[K];
    typename V2<TF>::t v[K];
    int q[K];
#pragma unroll
    for (int kk = 0; kk < K; kk++) {
        const int k[3] = {kk % 3 - 1, (kk / 3) % 3 - 1, D == 3 ? kk / 9 - 1 : 0};
        bool ok = true;
#pragma unroll
        for (int a = 0; a < D; a++) ok = ok && 2 * ii[a] + k[a] >= 0 && 2 * ii[a] + k[a] < fn;
        q[kk] = f + k[0] + fn * (k[1] + (D == 3 ? fn * k[2] : 0));
        ty[kk] = ok ? ftype[q[kk]] : (int8_t)T_OUT;
    }
    TF ss = 0, sc = 0;
    int cnt = 0;
#pragma unroll
    for (int kk = 0; kk < K; kk++)
        if (ty[kk] == T_IN || ty[kk] == T_GHOST) v[kk] = fW[q[kk]];
#pragma unroll
    for (int kk = 0; kk < K; kk++)
        if (ty[kk] == T_IN || ty[kk] == T_GHOST) {
            ss += v[kk].x;
            sc += v[kk].y;
            cnt++;
        }
    out.x = (T)(cnt ? ss / (TF)cnt : (TF)0);
    out.y = (T)(cnt ? sc / (TF)cnt : (TF)0);
    cW[I] = out;
}

// ---------------------------------------------------------------------------
// coarsest level

// The dense Schur complement in list order (inside nodes, then ghosts)
// assembled and inverted by Gauss-Jordan elimination with partial pivoting on
// a thread-block cluster: CTA r of C owns the columns j with j % C == r, in
// its shared memory where they fit (SMEM) or in A.  Step k: the owner of
// column k finds the pivot row (first of largest magnitude, i >= k) and writes
// the interchanged column, its pivot's reciprocal and the pivot row index into
// every CTA's shared memory (double-buffered by the parity of k); one cluster
// barrier; then each CTA interchanges, scales and eliminates in its own
// columns.  The row interchanges are undone as column interchanges at the end.
// Eliminating c first halves the order of the matrix: half the pivot steps.
constexpr int kFacCluster = 8;
constexpr int kFacThreads = 512;

template <typename T>
inline size_t factor_smem(int m, bool columns) {
    const size_t mc = ((size_t)m + kFacCluster - 1) / kFacCluster;
    return sizeof(T) * ((columns ? (size_t)m * mc : 0) + 2 * ((size_t)m + 1)) + sizeof(int) * 3 * (size_t)m;
}

template <int D, typename T, bool SMEM>
__global__ void __launch_bounds__(kFacThreads) k_s_factor(SLev<D, T> L, const int* __restrict__ spos,
                                                          const int* __restrict__ cpos, T* Ag, T* Ainv,
                                                          int* singular) {
    namespace cg = cooperative_groups;
    pdl_enter();
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), me = (int)cl.block_rank();
    const int nin = L.n0 + L.n1, m = nin + L.ng;
    const int mc = (m + C - 1) / C;  // local column jl is global column jl * C + me
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* A = SMEM ? reinterpret_cast<T*>(smem_raw) : Ag + (size_t)me * m * mc;  // m x mc, row-major
    T* fac = reinterpret_cast<T*>(smem_raw) + (SMEM ? (size_t)m * mc : 0);    // two buffers of m + 1
    int* piv = reinterpret_cast<int*>(fac + 2 * (m + 1));
    int* idx = piv + m;
    int* pos = idx + m;
    for (int i = threadIdx.x; i < m * mc; i += blockDim.x) A[i] = 0;
    __syncthreads();
    auto add = [&](int i, int j, T v) {
        if (j % C == me) A[(size_t)i * mc + j / C] += v;
    };
    for (int r = threadIdx.x; r < m; r += blockDim.x) {
        if (r < nin) {
            const int colour = r >= L.n0, e = L.hl[r];
            int o[2 * D];
            nbr_offsets<D, T>(L, e & 1, o);
            const int so = (1 - colour) * L.Hn + (e >> kEntHalf);
            for (int q = 0; q < 2 * D; q++) add(r, spos[so + o[q]], -L.gt[q * L.gs + r]);
            add(r, r, L.dd[r]);
        } else {
            for (int j = L.rptr[r - nin]; j < L.rptr[r - nin + 1]; j++) add(r, spos[L.rslot[j]], L.rval[j]);
        }
    }
    // (all of the cluster: another CTA's shared memory may be written only once
    // that CTA is known to run)
    cl.sync();
    __shared__ int s_piv;
    // a thread's elements (row, local column) of the elimination, packed: a
    // half-empty FP64 instruction costs as much as a full one
    constexpr int kEl = 4;
    const int nel = m * mc, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int er[kEl], ec[kEl];
#pragma unroll
    for (int q = 0; q < kEl; q++) {
        const int t = threadIdx.x + q * kFacThreads;
        er[q] = t / mc;
        ec[q] = t % mc;
    }
    for (int k = 0; k < m; k++) {
        T* fb = fac + (size_t)(k & 1) * (m + 1);
        if (k % C == me) {
            const int kl = k / C;
            __syncthreads();  // this CTA's updates of column k in the previous step
            if (warp == 0) {
                // magnitudes compared as integers (an FP64 compare takes the
                // FP64 pipe); a NaN is no pivot
                unsigned long long bv = 0;
                int bi = k;
                for (int i = k + lane; i < m; i += 32) {
                    unsigned long long v = abs_bits(A[(size_t)i * mc + kl]);
                    if (v > 0x7ff0000000000000ULL) v = 0;
                    if (v > bv) {
                        bv = v;
                        bi = i;
                    }
                }
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long ov = __shfl_down_sync(0xffffffffu, bv, o);
                    const int oi = __shfl_down_sync(0xffffffffu, bi, o);
                    if (ov > bv || (ov == bv && oi < bi)) {
                        bv = ov;
                        bi = oi;
                    }
                }
                if (lane == 0) {
                    s_piv = bi;
                    if (bv == 0) *singular = 1;
                }
            }
            __syncthreads();
            const int pr = s_piv;
            if (warp < C) {
                T* dst = cl.map_shared_rank(fb, warp);
                for (int i = lane; i < m; i += 32) {
                    const int src = i == k ? pr : (i == pr ? k : i);
                    dst[i] = A[(size_t)src * mc + kl];
                }
            } else if (warp == C && lane < C) {
                cl.map_shared_rank(fb, lane)[m] = (T)1 / A[(size_t)pr * mc + kl];
                cl.map_shared_rank(piv, lane)[k] = pr;
            }
        }
        cl.sync();
        // rows k and pr change places, row k is scaled by the reciprocal pivot,
        // column k eliminated from the others: all reads, then all writes
        const int pr = piv[k];
        const T inv = fb[m];
        auto value = [&](int i, int jl) -> T {
            const T top = A[(size_t)pr * mc + jl] * inv;
            const bool own = jl * C + me == k;
            if (i == k) return own ? inv : top;
            if (own) return -fb[i] * inv;
            const T v = i == pr ? A[(size_t)k * mc + jl] : A[(size_t)i * mc + jl];
            return fmadd(-fb[i], top, v);
        };
        if (nel <= kEl * kFacThreads) {
            T v[kEl];
#pragma unroll
            for (int q = 0; q < kEl; q++)
                if ((int)threadIdx.x + q * kFacThreads < nel) v[q] = value(er[q], ec[q]);
            __syncthreads();
#pragma unroll
            for (int q = 0; q < kEl; q++)
                if ((int)threadIdx.x + q * kFacThreads < nel) A[(size_t)er[q] * mc + ec[q]] = v[q];
        } else {
            // larger matrices: a column at a time per thread group
            for (int jl = warp; jl < mc; jl += kFacThreads / 32) {
                const T rowk = A[(size_t)k * mc + jl], top = A[(size_t)pr * mc + jl] * inv;
                const bool own = jl * C + me == k;
                __syncwarp();
                for (int i = lane; i < m; i += 32) {
                    const T v = i == pr ? rowk : A[(size_t)i * mc + jl];
                    A[(size_t)i * mc + jl] =
                        i == k ? (own ? inv : top) : (own ? -fb[i] * inv : fmadd(-fb[i], top, v));
                }
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int j = 0; j < m; j++) idx[j] = j;
        for (int k = m - 1; k >= 0; k--) {
            const int p = piv[k], t = idx[k];
            idx[k] = idx[p];
            idx[p] = t;
        }
        for (int j = 0; j < m; j++) pos[idx[j]] = j;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < m * mc; t += blockDim.x) {
        const int i = t / mc, jl = t % mc;
        const int j = jl * C + me;
        if (j < m)
            Ainv[(size_t)(cpos ? cpos[i] : i) * m + (cpos ? cpos[pos[j]] : pos[j])] = A[(size_t)i * mc + jl];
    }
    cl.sync();  // no CTA leaves while another may still write its shared memory
}

// x = A^{-1} b: one warp per row
template <int D, typename T>
__device__ __forceinline__ void s_solve(const SLev<D, T>& L, int t) {
    const int nin = L.n0 + L.n1, m = nin + L.ng;
    const int r = t >> 5, lane = t & 31;
    pdl_enter();
    if (r >= m) return;
    const T* row = L.Ainv + (size_t)r * m;
    T v = 0;
    for (int j = lane; j < m; j += 32) v = fmadd(row[j], L.b[j], v);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) {
        int p;
        L.X[list_slot<D, T>(L, r, p)] = v;
    }
}

// ---------------------------------------------------------------------------
// the phases as kernels, of one domain and of many

enum { kPhRelax = 0, kPhCorrect, kPhDelta, kPhGhosts, kPhResidual, kPhNorm, kPhRestrict, kPhProlong, kPhSolve };

// flags: 1 black colour, 2 snap, 4 skip on the flag, 8 accumulate
template <int D, typename T, int PH>
__device__ __forceinline__ void s_phase(const SLev<D, T>& L, const SLev<D, T>& C, int t, int flags,
                                        unsigned long long* norm) {
    if (PH == kPhRelax) s_relax<D, T, false>(L, t, flags & 1, flags & 2, flags & 4, flags & 8);
    if (PH == kPhCorrect) s_correct<D, T>(L, t);
    if (PH == kPhDelta) s_relax<D, T, true>(L, t, flags & 1, flags & 2, flags & 4, flags & 8);
    if (PH == kPhGhosts) s_ghosts<D, T>(L, t, flags & 4, flags & 8);
    if (PH == kPhResidual) s_residual<D, T, false>(L, t, norm);
    if (PH == kPhNorm) s_residual<D, T, true>(L, t, norm);
    if (PH == kPhRestrict) s_restrict<D, T>(L, C, t);
    if (PH == kPhProlong) s_prolong<D, T>(L, C, t);
    if (PH == kPhSolve) s_solve<D, T>(L, t);
}

template <int D, typename T, int PH>
__global__ void __launch_bounds__(kT) k_s_phase(const __grid_constant__ SLev<D, T> L,
                                                 const __grid_constant__ SLev<D, T> C, int flags,
                                                 unsigned long long* norm) {
    s_phase<D, T, PH>(L, C, blockIdx.x * blockDim.x + threadIdx.x, flags, norm);
}

// (single-level phases: one level parameter less to copy per launch)
template <int D, typename T, int PH>
__global__ void __launch_bounds__(kT) k_s_phase1(const __grid_constant__ SLev<D, T> L, int flags,
                                                  unsigned long long* norm) {
    s_phase<D, T, PH>(L, L, blockIdx.x * blockDim.x + threadIdx.x, flags, norm);
}

template <int D>
__global__ void __launch_bounds__(kT) k_s_outer(const __grid_constant__ SLev<D, double> L,
                                                 const __grid_constant__ SLev<D, float> U, unsigned long long* norm) {
    s_outer<D>(L, U, blockIdx.x * blockDim.x + threadIdx.x, norm);
}

template <int D, typename T, int PH>
__global__ void __launch_bounds__(kT) kb_s_phase(const SLev<D, T>* __restrict__ lv, const SLev<D, T>* __restrict__ lc,
                                                  const int* __restrict__ pre, int K, const int* __restrict__ active,
                                                  int flags, unsigned long long* norms) {
    const int i = find_instance(pre, K, blockIdx.x);
    if (masked(active, i)) return;
    s_phase<D, T, PH>(lv[i], lc[i], (blockIdx.x - pre[i]) * kT + threadIdx.x, flags, norms + i);
}

template <int D>
__global__ void __launch_bounds__(kT) kb_s_outer(const SLev<D, double>* __restrict__ l64,
                                                  const SLev<D, float>* __restrict__ l32, const int* __restrict__ pre,
                                                  int K, const int* __restrict__ active, unsigned long long* norms) {
    const int i = find_instance(pre, K, blockIdx.x);
    if (masked(active, i)) return;
    s_outer<D>(l64[i], l32[i], (blockIdx.x - pre[i]) * kT + threadIdx.x, norms + i);
}

// ---------------------------------------------------------------------------
// end of a linear solve

template <int D>
__global__ void __launch_bounds__(kT) k_s_update(SLev<D, double> L, const double* __restrict__ tt,
                                                  double2* __restrict__ W, unsigned long long* norms,
                                                  const int* __restrict__ on) {
    pdl_enter();
    if (on && !*on) return;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long nx = 0, nw = 0;
    if (t < L.n0 + L.n1 + L.ng) {
        int p;
        const int sl = list_slot<D, double>(L, t, p);
        double2 w = W[p];
        const double xs = L.X[sl], xc = fmadd(-L.rho[sl], xs, tt[sl]);
        unsigned long long a0 = abs_bits(w.x), a1 = abs_bits(w.y);
        nw = a0 > a1 ? a0 : a1;
        a0 = abs_bits(xs);
        a1 = abs_bits(xc);
        nx = a0 > a1 ? a0 : a1;
        w.x -= xs;
        w.y -= xc;
        W[p] = w;
    }
    block_max(nx, norms);
    __syncthreads();
    block_max(nw, norms + 1);
}

template <int D>
__global__ void __launch_bounds__(kT) k_s_export(SLev<D, double> L, const double* __restrict__ tt, double2* x) {
    pdl_enter();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= L.n0 + L.n1 + L.ng) return;
    int p;
    const int sl = list_slot<D, double>(L, t, p);
    x[p] = make_double2(L.X[sl], fmadd(-L.rho[sl], L.X[sl], tt[sl]));
}

// ---------------------------------------------------------------------------
// per-level data

constexpr int kChunk = 1024;

__device__ __forceinline__ bool near_ghost(const int8_t* type, int p, int n, int dim) {
    bool g = type[p - 1] == T_GHOST || type[p + 1] == T_GHOST || type[p - n] == T_GHOST || type[p + n] == T_GHOST;
    if (dim == 3) g = g || type[p - n * n] == T_GHOST || type[p + n * n] == T_GHOST;
    return g;
}

// bits of the 3^d fine members of a coarse node (its fine twin at box node p)
// that are inside nodes; regular: all of them are, the black ones (odd index
// sum) away from the ghosts
__device__ __forceinline__ int member_mask(const int8_t* ftype, int p, int fn, int dim, bool& regular) {
    int m = 0;
    regular = true;
    for (int kk = 0; kk < (dim == 2 ? 9 : 27); kk++) {
        const int k[3] = {kk % 3 - 1, (kk / 3) % 3 - 1, dim == 3 ? kk / 9 - 1 : 0};
        const int q = p + k[0] + fn * (k[1] + fn * k[2]);
        const bool in = ftype[q] == T_IN;
        if (in) m |= 1 << kk;
        if (!in || (((k[0] + k[1] + k[2]) & 1) && near_ghost(ftype, q, fn, dim))) regular = false;
    }
    return m;
}

// class of an inside node: 2 next to a ghost, else 0 where its restriction
// from the finer level (if any) is regular, 1 where it is not
__device__ __forceinline__ int node_class(const int8_t* type, int p, int n, int dim, const int8_t* ftype, int fn) {
    if (near_ghost(type, p, n, dim)) return 2;
    if (!ftype) return 0;
    bool regular;
    member_mask(ftype, 2 * (p % n) + fn * (2 * ((p / n) % n) + (dim == 3 ? fn * 2 * (p / (n * n)) : 0)), fn, dim,
                regular);
    return regular ? 0 : 1;
}

// nodes of a colour's list of class 0 and 1, per chunk
__global__ void k_class_count(const int* __restrict__ list, int cnt, const int8_t* __restrict__ type, int n, int dim,
                              const int8_t* __restrict__ ftype, int fn, int* __restrict__ out) {
    const int t = blockIdx.x * kChunk + threadIdx.x;
    const int k = t < cnt ? node_class(type, list[t], n, dim, ftype, fn) : 3;
    const int c0 = __syncthreads_count(k == 0), c1 = __syncthreads_count(k == 1);
    if (threadIdx.x == 0) {
        out[2 * blockIdx.x] = c0;
        out[2 * blockIdx.x + 1] = c1;
    }
}

// entries of a colour's nodes by class, each class in list order; off: the
// chunk's offsets within classes 0 and 1, first: where classes 1 and 2 begin
__global__ void k_entries(const int* __restrict__ list, int cnt, const int8_t* __restrict__ type, int n, int dim,
                          const int8_t* __restrict__ ftype, int fn, const int8_t* __restrict__ ctype, int cn,
                          const int* __restrict__ off, int first1, int first2, int H, int* __restrict__ hl) {
    __shared__ int wsum[2][32];
    const int t = blockIdx.x * kChunk + threadIdx.x;
    const bool on = t < cnt;
    const int p = on ? list[t] : 0;
    const int k = on ? node_class(type, p, n, dim, ftype, fn) : 3;
    const unsigned m0 = __ballot_sync(0xffffffffu, k == 0), m1 = __ballot_sync(0xffffffffu, k == 1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        wsum[0][warp] = __popc(m0);
        wsum[1][warp] = __popc(m1);
    }
    __syncthreads();
    if (!on) return;
    const unsigned below = (1u << lane) - 1u;
    int r0 = off[2 * blockIdx.x] + __popc(m0 & below), r1 = off[2 * blockIdx.x + 1] + __popc(m1 & below);
    for (int w = 0; w < warp; w++) {
        r0 += wsum[0][w];
        r1 += wsum[1][w];
    }
    const int ii[3] = {p % n, (p / n) % n, dim == 3 ? p / (n * n) : 0};
    bool all = ctype != nullptr;
    for (int cc = 0; cc < (1 << dim) && all; cc++) {
        int q = 0, st = 1;
        for (int d = 0; d < dim; d++) {
            q += ((ii[d] + ((cc >> d) & 1)) >> 1) * st;
            st *= cn;
        }
        all = ctype[q] == T_IN || ctype[q] == T_GHOST;
    }
    const int h = (ii[0] >> 1) + H * (ii[1] + n * ii[2]);
    hl[k == 0 ? r0 : (k == 1 ? first1 + r1 : first2 + t - r0 - r1)] =
        (h << kEntHalf) | (all ? 4 : 0) | (k == 2 ? 2 : 0) | (ii[0] & 1);
}

__device__ __forceinline__ int box_slot(int p, int n, int dim, int H, int Hn) {
    const int i = p % n, j = (p / n) % n, k = dim == 3 ? p / (n * n) : 0;
    return ((i + j + k) & 1) * Hn + (i >> 1) + H * (j + n * k);
}

__global__ void k_ghost_slots(const int* __restrict__ gidx, int ng, int n, int dim, int H, int Hn,
                              int* __restrict__ gslot) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < ng) gslot[g] = box_slot(gidx[g], n, dim, H, Hn);
}

__global__ void k_gop_codes(const int* __restrict__ code, int nnz, const int* __restrict__ gpos, int n, int dim,
                            int H, int Hn, int* __restrict__ out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nnz) return;
    const int c = code[j];
    if (c >= 0) {
        out[j] = box_slot(c, n, dim, H, Hn);
        return;
    }
    const unsigned u = ~(unsigned)c;
    out[j] = (u & 1u) ? ~(int)(2u * (unsigned)gpos[u >> 1] + 1u) : c;
}

// members of the ghosts' rows: count, then fill
__global__ void k_rows(int ng, int K, const double* __restrict__ wk, const float* __restrict__ wk32,
                       const int* __restrict__ node, const int* __restrict__ ptr, int n, int dim, int H, int Hn,
                       int* __restrict__ cnt, int* __restrict__ slot, double* __restrict__ val,
                       float* __restrict__ val32) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ng) return;
    int j = ptr ? ptr[g] : 0;
    for (int kk = 0; kk < K; kk++) {
        const long long o = (long long)kk * ng + g;
        if (wk[o] == 0.0 && wk32[o] == 0.f) continue;
        if (ptr) {
            slot[j] = box_slot(node[o], n, dim, H, Hn);
            val[j] = wk[o];
            val32[j] = wk32[o];
        }
        j++;
    }
    if (!ptr) cnt[g] = j;
}

// slot of a coarse inside node's fine twin (a red node) and its members
__global__ void k_twins(const int* __restrict__ hl, int nin, int cn, int cH, const int8_t* __restrict__ ftype, int fn,
                        int fH, int dim, int* __restrict__ twin, int* __restrict__ mask) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nin) return;
    const int e = hl[t], h = e >> kEntHalf, row = h / cH;
    const int f[3] = {2 * (2 * (h - row * cH) + (e & 1)), 2 * (row % cn), dim == 3 ? 2 * (row / cn) : 0};
    bool regular;
    mask[t] = member_mask(ftype, f[0] + fn * (f[1] + fn * f[2]), fn, dim, regular);
    twin[t] = (f[0] >> 1) + fH * (f[1] + fn * f[2]);
}

// A coarse ghost's right-hand side: the outside weighting (Sec. 3.5.2) of the
// fine ghosts' defects and of their extension into the band, as one row over
// the fine ghosts (entries of one ghost merged).  Workspace in shared memory.
constexpr int kOutCap = 192;
struct OutWork {
    double w[kOutCap];
    int g[kOutCap];
};
constexpr int kOutThreads = 16;

__global__ void k_outside_rows(const int* __restrict__ cgidx, int cng, int cn, const int8_t* __restrict__ ftype,
                               int fn, int dim, const int* __restrict__ bpos, const int* __restrict__ eptr,
                               const int* __restrict__ eidx, const double* __restrict__ eval, int fH, int fHn,
                               const int* __restrict__ ptr, int* __restrict__ cnt, int* __restrict__ slot,
                               double* __restrict__ val, float* __restrict__ val32) {
    extern __shared__ OutWork out_ws[];
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= cng) return;
    OutWork& W = out_ws[threadIdx.x];
    int m = 0;
    bool over = false;
    auto add = [&](int g, double w) {
        int j = 0;
        while (j < m && W.g[j] != g) j++;
        if (j == m) {
            if (m == kOutCap) {
                over = true;
                return;
            }
            W.g[m] = g;
            W.w[m] = 0.0;
            m++;
        }
        W.w[j] += w;
    };
    auto node = [&](int q, double w) {
        if (ftype[q] == T_GHOST)
            add(q, w);
        else if (ftype[q] == T_BAND)
            for (int j = eptr[bpos[q]]; j < eptr[bpos[q] + 1]; j++) add(eidx[j], w * eval[j]);
    };
    const int I = cgidx[gi];
    const int ci[3] = {I % cn, (I / cn) % cn, dim == 3 ? I / (cn * cn) : 0};
    const int st[3] = {1, fn, fn * fn};
    int p = 0;
    for (int a = 0; a < dim; a++) p += 2 * ci[a] * st[a];
    auto outside = [&](int q) { return ftype[q] == T_GHOST || ftype[q] == T_BAND; };
    int w[3][3] = {{0, 1, 0}, {0, 1, 0}, {0, 1, 0}};
    for (int a = 0; a < dim; a++) {
        const bool vl = ci[a] > 0 && outside(p - st[a]), vr = 2 * ci[a] < fn - 1 && outside(p + st[a]);
        w[a][0] = vl ? (vr ? 1 : 2) : (vr ? 0 : 0);
        w[a][1] = vl || vr ? 2 : 4;
        w[a][2] = vr ? (vl ? 1 : 2) : 0;
    }
    const double scale = dim == 2 ? 1.0 / 16 : 1.0 / 64;
    int wc = 0;
    for (int kk = 0; kk < (dim == 2 ? 9 : 27); kk++) {
        const int k[3] = {kk % 3, (kk / 3) % 3, dim == 3 ? kk / 9 : 1};
        const int iw = w[0][k[0]] * w[1][k[1]] * w[2][k[2]];
        if (iw == 0) continue;
        int q = p;
        for (int a = 0; a < dim; a++) q += (k[a] - 1) * st[a];
        if (q == p || !outside(q))
            wc += iw;
        else
            node(q, iw * scale);
    }
    node(p, wc * scale);
    if (!ptr) {
        cnt[gi] = over ? -1 : m;
        return;
    }
    for (int j = 0; j < m; j++) {
        slot[ptr[gi] + j] = box_slot(W.g[j], fn, dim, fH, fHn);
        val[ptr[gi] + j] = W.w[j];
        val32[ptr[gi] + j] = (float)W.w[j];
    }
}

__global__ void k_positions(const int* __restrict__ hl, int n0, int nin, const int* __restrict__ gslot, int ng, int Hn,
                            int* __restrict__ spos) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nin)
        spos[(t >= n0 ? Hn : 0) + (hl[t] >> kEntHalf)] = t;
    else if (t < nin + ng)
        spos[gslot[t - nin]] = t;
}

inline unsigned nblk(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// host scan of n counts at dcnt into offsets (in place, dcnt has n + 1
// entries); the total, or -1 on a negative count or error
long long host_scan(int* dcnt, int n, cudaStream_t s, bool& bad) {
    std::vector<int> c(n + 1, 0);
    bad = false;
    if (cudaMemcpyAsync(c.data(), dcnt, sizeof(int) * n, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return -1;
    long long tot = 0;
    for (int i = 0; i < n; i++) {
        if (c[i] < 0) bad = true;
        const int v = c[i];
        c[i] = (int)tot;
        tot += v;
    }
    c[n] = (int)tot;
    if (bad) return 0;
    if (cudaMemcpyAsync(dcnt, c.data(), sizeof(int) * (n + 1), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return -1;
    return tot;
}

}  // namespace

int build_sgeo(SGeo& S, const LevelGeo& L, const LevelGeo* finer, const SGeo* sfiner, const LevelGeo* coarser,
               DevMem& mem, cudaStream_t s, std::string& err, long long& launches, bool& ok) {
    ok = false;
    auto oom = [&] {
        err = "out of device memory";
        return SULF_ENOMEM;
    };
    auto fail = [&] {
        err = "level lists failed";
        return SULF_EDEVICE;
    };
    if (L.nn >= (1LL << 28)) return SULF_OK;  // entries hold 29-bit half indices
    S.H = (L.n + 1) / 2;
    S.P = S.H * L.n;
    S.Hn = L.dim == 3 ? S.P * L.n : S.P;
    S.n0 = L.nin[0];
    S.n1 = L.nin[1];
    const int nin = S.n0 + S.n1;
    S.hl = (int*)mem.get(sizeof(int) * (nin + 1));
    S.gslot = (int*)mem.get(sizeof(int) * (L.ng + 1));
    const int nch = (int)nblk(S.n0 > S.n1 ? S.n0 : S.n1, kChunk);
    int* dc = (int*)mem.get(sizeof(int) * 4 * (nch + 1));
    if (!S.hl || !S.gslot || !dc) return oom();
    std::vector<int> c(4 * (nch + 1), 0);
    const int8_t* ft = finer ? finer->type : nullptr;
    const int fn = finer ? finer->n : 0;
    for (int k = 0; k < 2; k++)
        if (L.nin[k] > 0) {
            k_class_count<<<nblk(L.nin[k], kChunk), kChunk, 0, s>>>(L.inl[k], L.nin[k], L.type, L.n, L.dim, ft, fn,
                                                                    dc + 2 * k * (nch + 1));
            launches++;
        }
    if (cudaMemcpyAsync(c.data(), dc, sizeof(int) * c.size(), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return fail();
    int tot[2][2] = {{0, 0}, {0, 0}};
    for (int k = 0; k < 2; k++)
        for (int b = 0; b < (int)nblk(L.nin[k], kChunk); b++)
            for (int q = 0; q < 2; q++) {
                int& v = c[2 * k * (nch + 1) + 2 * b + q];
                const int w = v;
                v = tot[k][q];
                tot[k][q] += w;
            }
    S.nreg0 = tot[0][0];
    S.nreg1 = tot[1][0];
    S.nga = S.n1 - tot[1][0] - tot[1][1];
    if (cudaMemcpyAsync(dc, c.data(), sizeof(int) * c.size(), cudaMemcpyHostToDevice, s) != cudaSuccess) return fail();
    for (int k = 0; k < 2; k++)
        if (L.nin[k] > 0) {
            k_entries<<<nblk(L.nin[k], kChunk), kChunk, 0, s>>>(
                L.inl[k], L.nin[k], L.type, L.n, L.dim, ft, fn, coarser ? coarser->type : nullptr,
                coarser ? coarser->n : 0, dc + 2 * k * (nch + 1), tot[k][0], tot[k][0] + tot[k][1], S.H,
                S.hl + (k ? S.n0 : 0));
            launches++;
        }
    if (L.ng > 0) {
        k_ghost_slots<<<nblk(L.ng), 256, 0, s>>>(L.gidx, L.ng, L.n, L.dim, S.H, S.Hn, S.gslot);
        launches++;
    }
    if (finer) {
        S.twin = (int*)mem.get(sizeof(int) * (nin + 1));
        S.cptr = (int*)mem.get(sizeof(int) * (L.ng + 1));
        S.mask = (int*)mem.get(sizeof(int) * (nin + 1));
        if (!S.twin || !S.cptr || !S.mask) return oom();
        k_twins<<<nblk(nin), 256, 0, s>>>(S.hl, nin, L.n, S.H, finer->type, finer->n, sfiner->H, L.dim, S.twin,
                                          S.mask);
        launches++;
        long long tot = 0;
        const size_t shm = sizeof(OutWork) * kOutThreads;
        if (L.ng > 0) {
            k_outside_rows<<<nblk(L.ng, kOutThreads), kOutThreads, shm, s>>>(
                L.gidx, L.ng, L.n, finer->type, finer->n, L.dim, finer->bpos, finer->eptr, finer->eidx, finer->eval,
                sfiner->H, sfiner->Hn, nullptr, S.cptr, nullptr, nullptr, nullptr);
            launches++;
            bool bad;
            tot = host_scan(S.cptr, L.ng, s, bad);
            if (tot < 0) return fail();
            if (bad) return SULF_OK;
        }
        S.cslot = (int*)mem.get(sizeof(int) * (tot + 1));
        S.cval = (double*)mem.get(sizeof(double) * (tot + 1));
        S.cval32 = (float*)mem.get(sizeof(float) * (tot + 1));
        if (!S.cslot || !S.cval || !S.cval32) return oom();
        if (L.ng > 0) {
            k_outside_rows<<<nblk(L.ng, kOutThreads), kOutThreads, shm, s>>>(
                L.gidx, L.ng, L.n, finer->type, finer->n, L.dim, finer->bpos, finer->eptr, finer->eidx, finer->eval,
                sfiner->H, sfiner->Hn, S.cptr, nullptr, S.cslot, S.cval, S.cval32);
            launches++;
        }
    }
    if (!coarser) {
        S.spos = (int*)mem.get(sizeof(int) * 2 * (size_t)S.Hn);
        if (!S.spos) return oom();
        if (cudaMemsetAsync(S.spos, 0, sizeof(int) * 2 * (size_t)S.Hn, s) != cudaSuccess) return fail();
        k_positions<<<nblk(nin + L.ng), 256, 0, s>>>(S.hl, S.n0, nin, S.gslot, L.ng, S.Hn, S.spos);
        launches++;
    }
    if (cudaStreamSynchronize(s) != cudaSuccess) return fail();
    ok = true;
    return SULF_OK;
}

int build_sgeo_rows(SGeo& S, const LevelGeo& L, DevMem& mem, cudaStream_t s, std::string& err, long long& launches) {
    auto oom = [&] {
        err = "out of device memory";
        return SULF_ENOMEM;
    };
    // what the rows are built for: known once they are there
    S.bc = -1;
    auto built = [&] {
        S.bc = L.gop_bc;
        S.passes = L.gop_passes;
        S.tau = L.gop_tau;
        return SULF_OK;
    };
    if (L.ng == 0) return built();
    if (L.gop_nnz > S.gcap) {
        S.gcode = (int*)mem.get(sizeof(int) * (L.gop_nnz + 1));
        if (!S.gcode) return oom();
        S.gcap = L.gop_nnz;
    }
    {
        // the ghosts by the length of their composed row
        if (!S.gord) S.gord = (int*)mem.get(sizeof(int) * (L.ng + 1));
        if (!S.gord) return oom();
        std::vector<int> p(L.ng + 1), ord(L.ng);
        if (cudaMemcpyAsync(p.data(), L.gop_ptr, sizeof(int) * (L.ng + 1), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) {
            err = "ghost rows failed";
            return SULF_EDEVICE;
        }
        int n[4] = {0, 0, 0, 0};
        auto part = [&](int g) {
            const int len = p[g + 1] - p[g];
            return len <= kGopPre ? 0 : (len <= kGopPre * kGopLanes ? 1 : 2);
        };
        for (int g = 0; g < L.ng; g++) n[part(g) + 1]++;
        S.ng1 = n[1];
        S.ng8 = n[2];
        n[2] += n[1];
        for (int g = 0; g < L.ng; g++) ord[n[part(g)]++] = g;
        if (cudaMemcpyAsync(S.gord, ord.data(), sizeof(int) * L.ng, cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) {
            err = "ghost rows failed";
            return SULF_EDEVICE;
        }
    }
    k_gop_codes<<<nblk(L.gop_nnz), 256, 0, s>>>(L.gop_code, (int)L.gop_nnz, L.gpos, L.n, L.dim, S.H, S.Hn, S.gcode);
    const int K = L.dim == 2 ? 9 : 27;
    if (!S.rptr) {
        S.rptr = (int*)mem.get(sizeof(int) * (L.ng + 1));
        // at most K members a row: sized once, the boundary condition may change
        S.rslot = (int*)mem.get(sizeof(int) * (size_t)K * (L.ng + 1));
        S.rval = (double*)mem.get(sizeof(double) * (size_t)K * (L.ng + 1));
        S.rval32 = (float*)mem.get(sizeof(float) * (size_t)K * (L.ng + 1));
        if (!S.rptr || !S.rslot || !S.rval || !S.rval32) return oom();
    }
    k_rows<<<nblk(L.ng), 256, 0, s>>>(L.ng, K, L.gwk, L.gwk32, L.gnode, nullptr, L.n, L.dim, S.H, S.Hn, S.rptr,
                                      nullptr, nullptr, nullptr);
    bool bad;
    if (host_scan(S.rptr, L.ng, s, bad) < 0 || bad) {
        err = "ghost rows failed";
        return SULF_EDEVICE;
    }
    k_rows<<<nblk(L.ng), 256, 0, s>>>(L.ng, K, L.gwk, L.gwk32, L.gnode, S.rptr, L.n, L.dim, S.H, S.Hn, nullptr,
                                      S.rslot, S.rval, S.rval32);
    launches += 3;
    if (cudaStreamSynchronize(s) != cudaSuccess) {
        err = "ghost rows failed";
        return SULF_EDEVICE;
    }
    return built();
}

// ---------------------------------------------------------------------------
// launchers

template <int D, typename T>
int launch_s_rho(const SLev<D, T>& L, const typename V2<T>::t* Wc, const Coef<T>& c, cudaStream_t s) {
    const int tot = L.n0 + L.n1 + L.ng;
    launch_k(k_s_rho<D, T, false, false>, grid_for(tot), block_for(tot), 0, s, L, SLev<D, float>{}, Wc, c,
             (const double2*)nullptr, (double*)nullptr, (double*)nullptr);
    return 1;
}

template <int D>
int launch_s_rho_fine(const SLev<D, double>& L, const double2* Wc, const Coef<double>& c, const double2* F, double* tt,
                      double* uu, const SLev<D, float>* U, cudaStream_t s) {
    const int tot = L.n0 + L.n1 + L.ng;
    if (U)
        launch_k(k_s_rho<D, double, true, true>, grid_for(tot), block_for(tot), 0, s, L, *U, Wc, c, F, tt, uu);
    else
        launch_k(k_s_rho<D, double, true, false>, grid_for(tot), block_for(tot), 0, s, L, SLev<D, float>{}, Wc, c, F,
                 tt, uu);
    return 1;
}

template <int D, typename T>
int launch_s_coefs(const SLev<D, T>& L, const typename V2<T>::t* Wc, const Coef<T>& c, cudaStream_t s) {
    const int tot = L.n0 + L.n1;
    launch_k(k_s_coefs<D, T>, grid_for(tot), block_for(tot), 0, s, L, Wc, c);
    return 1;
}

template <int D>
int launch_s_coefs_fine(const SLev<D, double>& L, const double2* Wc, const Coef<double>& c, const double2* F,
                        const double* tt, const double* uu, const SLev<D, float>* U, cudaStream_t s) {
    const int tot = L.n0 + L.n1;
    if (U)
        launch_k(k_s_coefs_fine<D, true>, grid_for(tot), block_for(tot), 0, s, L, *U, Wc, c, F, tt, uu);
    else
        launch_k(k_s_coefs_fine<D, false>, grid_for(tot), block_for(tot), 0, s, L, SLev<D, float>{}, Wc, c, F, tt, uu);
    return 1;
}

namespace {
template <int D, typename T, int PH>
int launch_one(const SLev<D, T>& L, long long threads, int flags, unsigned long long* norm, cudaStream_t s) {
    if (threads <= 0) return 0;
    launch_k(k_s_phase1<D, T, PH>, grid_for(threads), block_for(threads), 0, s, L, flags, norm);
    return 1;
}
inline int relax_flags(int colour, bool snap, bool skip, bool acc) {
    return (colour ? 1 : 0) | (snap ? 2 : 0) | (skip ? 4 : 0) | (acc ? 8 : 0);
}
}  // namespace

template <int D, typename T>
long long s_threads(SPhase ph, const SLev<D, T>& L, const SLev<D, T>* C) {
    switch (ph) {
        case SPhase::correct:
        case SPhase::red: return L.n0;
        case SPhase::black: return L.n1 > L.ng ? L.n1 : L.ng;
        case SPhase::ghosts: return ghost_threads<D, T>(L, kGopLanes, 32);
        case SPhase::residual: return up32(L.n0 + L.nga) + (long long)ghost_threads<D, T>(L, kGopLanes, kGopLanes);
        case SPhase::outer: return up32(L.n0 + L.n1) + (long long)ghost_threads<D, T>(L, kGopLanes, kGopLanes);
        case SPhase::restrict_to:
            return up32(C->nreg0 + C->nreg1) + up32(C->n0 + C->n1 - C->nreg0 - C->nreg1) + (long long)C->ng * kGopLanes;
        case SPhase::prolong_from: return (long long)L.n1 + L.ng;
        case SPhase::solve: return 32LL * (L.n0 + L.n1 + L.ng);
    }
    return 0;
}

template <int D, typename T>
int launch_s_relax(const SLev<D, T>& L, int colour, bool delta, bool snap, bool skip, bool acc, cudaStream_t s) {
    const long long n = colour && snap ? s_threads<D, T>(SPhase::black, L, nullptr) : (colour ? L.n1 : L.n0);
    const int fl = relax_flags(colour, snap, skip, acc);
    return delta ? launch_one<D, T, kPhDelta>(L, n, fl, nullptr, s) : launch_one<D, T, kPhRelax>(L, n, fl, nullptr, s);
}

template <int D, typename T>
int launch_s_ghosts(const SLev<D, T>& L, bool skip, bool acc, cudaStream_t s) {
    return launch_one<D, T, kPhGhosts>(L, s_threads<D, T>(SPhase::ghosts, L, nullptr), relax_flags(0, false, skip, acc),
                                       nullptr, s);
}

template <int D, typename T>
int launch_s_correct(const SLev<D, T>& L, cudaStream_t s) {
    return launch_one<D, T, kPhCorrect>(L, L.n0, 0, nullptr, s);
}

template <int D, typename T>
int launch_s_residual(const SLev<D, T>& L, unsigned long long* norm, cudaStream_t s) {
    const long long n = s_threads<D, T>(SPhase::residual, L, nullptr);
    return norm ? launch_one<D, T, kPhNorm>(L, n, 0, norm, s) : launch_one<D, T, kPhResidual>(L, n, 0, norm, s);
}

template <int D>
int launch_s_outer(const SLev<D, double>& L, const SLev<D, float>& U, unsigned long long* norm, cudaStream_t s) {
    const long long n = s_threads<D, double>(SPhase::outer, L, nullptr);
    launch_k(k_s_outer<D>, grid_for(n), block_for(n), 0, s, L, U, norm);
    return 1;
}

template <int D, typename T>
int launch_s_restrict(const SLev<D, T>& F, const SLev<D, T>& C, cudaStream_t s) {
    const long long n = s_threads<D, T>(SPhase::restrict_to, F, &C);
    launch_k(k_s_phase<D, T, kPhRestrict>, grid_for(n), block_for(n), 0, s, F, C, 0, (unsigned long long*)nullptr);
    return 1;
}

template <int D, typename T>
int launch_s_prolong(const SLev<D, T>& F, const SLev<D, T>& C, cudaStream_t s) {
    const long long n = s_threads<D, T>(SPhase::prolong_from, F, &C);
    if (n == 0) return 0;
    launch_k(k_s_phase<D, T, kPhProlong>, grid_for(n), block_for(n), 0, s, F, C, 0, (unsigned long long*)nullptr);
    return 1;
}

template <int D, typename T>
int launch_s_solve(const SLev<D, T>& L, cudaStream_t s) {
    return launch_one<D, T, kPhSolve>(L, s_threads<D, T>(SPhase::solve, L, nullptr), 0, nullptr, s);
}

template <int D, typename T>
int launch_s_batched(SPhase ph, bool delta, const SLev<D, T>* lv, const SLev<D, T>* lc, const int* pre, int nblocks,
                     int K, const int* active, bool skip, bool acc, unsigned long long* norms, cudaStream_t s) {
    if (nblocks <= 0) return 0;
    const unsigned nb = (unsigned)nblocks;
    if (!lc) lc = lv;
    const int fl = relax_flags(ph == SPhase::black, ph == SPhase::black, skip, acc);
    switch (ph) {
        case SPhase::correct:
            launch_k(kb_s_phase<D, T, kPhCorrect>, nb, kT, 0, s, lv, lc, pre, K, active, fl, norms);
            break;
        case SPhase::red:
        case SPhase::black:
            if (delta)
                launch_k(kb_s_phase<D, T, kPhDelta>, nb, kT, 0, s, lv, lc, pre, K, active, fl, norms);
            else
                launch_k(kb_s_phase<D, T, kPhRelax>, nb, kT, 0, s, lv, lc, pre, K, active, fl, norms);
            break;
        case SPhase::ghosts:
            launch_k(kb_s_phase<D, T, kPhGhosts>, nb, kT, 0, s, lv, lc, pre, K, active, fl, norms);
            break;
        case SPhase::residual:
            if (norms)
                launch_k(kb_s_phase<D, T, kPhNorm>, nb, kT, 0, s, lv, lc, pre, K, active, fl, norms);
            else
                launch_k(kb_s_phase<D, T, kPhResidual>, nb, kT, 0, s, lv, lc, pre, K, active, fl, norms);
            break;
        case SPhase::restrict_to:
            launch_k(kb_s_phase<D, T, kPhRestrict>, nb, kT, 0, s, lv, lc, pre, K, active, fl, norms);
            break;
        case SPhase::prolong_from:
            launch_k(kb_s_phase<D, T, kPhProlong>, nb, kT, 0, s, lv, lc, pre, K, active, fl, norms);
            break;
        case SPhase::solve:
            launch_k(kb_s_phase<D, T, kPhSolve>, nb, kT, 0, s, lv, lc, pre, K, active, fl, norms);
            break;
        default:
            return 0;
    }
    return 1;
}

template <int D>
int launch_s_batched_outer(const SLev<D, double>* l64, const SLev<D, float>* l32, const int* pre, int nblocks, int K,
                           const int* active, unsigned long long* norms, cudaStream_t s) {
    if (nblocks <= 0) return 0;
    launch_k(kb_s_outer<D>, (unsigned)nblocks, kT, 0, s, l64, l32, pre, K, active, norms);
    return 1;
}

template <int D, typename T>
int launch_s_factor(const SLev<D, T>& L, const int* spos, const int* cpos, T* A, T* Ainv, int* singular,
                    cudaStream_t s) {
    const int m = L.n0 + L.n1 + L.ng;
    constexpr size_t kMaxSmem = 220 * 1024;
    const bool smem = factor_smem<T>(m, true) <= kMaxSmem;
    auto kern = smem ? k_s_factor<D, T, true> : k_s_factor<D, T, false>;
    // set once to the largest size ever used (a per-launch value would race
    // with other threads' launches of different sizes)
    static std::mutex mu;
    static bool raised[2][64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    {
        std::lock_guard<std::mutex> lock(mu);
        if (dev < 0 || dev >= 64 || !raised[smem][dev]) {
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
            if (dev >= 0 && dev < 64) raised[smem][dev] = true;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kFacCluster);
    cfg.blockDim = dim3(kFacThreads);
    cfg.dynamicSmemBytes = factor_smem<T>(m, smem);
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kFacCluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = launch_pdl() ? 1 : 0;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kern, L, spos, cpos, A, Ainv, singular);
    if (e != cudaSuccess) note_launch_error(e, kFacCluster, kFacThreads, cfg.dynamicSmemBytes);
    return 1;
}

template <int D>
int launch_s_update(const SLev<D, double>& L, const double* tt, double2* W, unsigned long long* norms, const int* on,
                    cudaStream_t s) {
    const int tot = L.n0 + L.n1 + L.ng;
    launch_k(k_s_update<D>, grid_for(tot), block_for(tot), 0, s, L, tt, W, norms, on);
    return 1;
}

template <int D>
int launch_s_export(const SLev<D, double>& L, const double* tt, double2* x, cudaStream_t s) {
    const int tot = L.n0 + L.n1 + L.ng;
    launch_k(k_s_export<D>, grid_for(tot), block_for(tot), 0, s, L, tt, x);
    return 1;
}

template <int D, typename TF, typename T>
int launch_inject_to(const LevelGeo& F, const typename V2<TF>::t* fW, const LevelGeo& C, typename V2<T>::t* cW,
                     cudaStream_t s) {
    stages::Lists ls = stages::make_lists(C);
    const int tot = ls.n0 + ls.n1 + ls.ng;
    launch_k(k_inject_to<D, TF, T>, grid_for(tot), block_for(tot), 0, s, ls, C.n, F.type, F.n, fW, cW);
    return 1;
}

#define SULF_INST_S(D, T)                                                                                          \
    template int launch_s_rho<D, T>(const SLev<D, T>&, const typename V2<T>::t*, const Coef<T>&, cudaStream_t);     \
    template int launch_s_coefs<D, T>(const SLev<D, T>&, const typename V2<T>::t*, const Coef<T>&, cudaStream_t);   \
    template long long s_threads<D, T>(SPhase, const SLev<D, T>&, const SLev<D, T>*);                              \
    template int launch_s_relax<D, T>(const SLev<D, T>&, int, bool, bool, bool, bool, cudaStream_t);               \
    template int launch_s_ghosts<D, T>(const SLev<D, T>&, bool, bool, cudaStream_t);                               \
    template int launch_s_correct<D, T>(const SLev<D, T>&, cudaStream_t);                                          \
    template int launch_s_residual<D, T>(const SLev<D, T>&, unsigned long long*, cudaStream_t);                    \
    template int launch_s_restrict<D, T>(const SLev<D, T>&, const SLev<D, T>&, cudaStream_t);                      \
    template int launch_s_prolong<D, T>(const SLev<D, T>&, const SLev<D, T>&, cudaStream_t);                       \
    template int launch_s_factor<D, T>(const SLev<D, T>&, const int*, const int*, T*, T*, int*, cudaStream_t);     \
    template int launch_s_solve<D, T>(const SLev<D, T>&, cudaStream_t);                                            \
    template int launch_s_batched<D, T>(SPhase, bool, const SLev<D, T>*, const SLev<D, T>*, const int*, int, int,  \
                                        const int*, bool, bool, unsigned long long*, cudaStream_t);
SULF_INST_S(2, double)
SULF_INST_S(2, float)
SULF_INST_S(3, double)
SULF_INST_S(3, float)
#define SULF_INST_SD(D)                                                                                            \
    template int launch_s_rho_fine<D>(const SLev<D, double>&, const double2*, const Coef<double>&, const double2*, \
                                      double*, double*, const SLev<D, float>*, cudaStream_t);                      \
    template int launch_s_coefs_fine<D>(const SLev<D, double>&, const double2*, const Coef<double>&,               \
                                        const double2*, const double*, const double*, const SLev<D, float>*,       \
                                        cudaStream_t);                                                             \
    template int launch_s_outer<D>(const SLev<D, double>&, const SLev<D, float>&, unsigned long long*,             \
                                   cudaStream_t);                                                                  \
    template int launch_s_batched_outer<D>(const SLev<D, double>*, const SLev<D, float>*, const int*, int, int,    \
                                           const int*, unsigned long long*, cudaStream_t);                         \
    template int launch_s_update<D>(const SLev<D, double>&, const double*, double2*, unsigned long long*,          \
                                    const int*, cudaStream_t);                                                     \
    template int launch_s_export<D>(const SLev<D, double>&, const double*, double2*, cudaStream_t);                \
    template int launch_inject_to<D, double, double>(const LevelGeo&, const double2*, const LevelGeo&, double2*,   \
                                                     cudaStream_t);                                                \
    template int launch_inject_to<D, double, float>(const LevelGeo&, const double2*, const LevelGeo&, float2*,     \
                                                    cudaStream_t);                                                 \
    template int launch_inject_to<D, float, float>(const LevelGeo&, const float2*, const LevelGeo&, float2*,       \
                                                   cudaStream_t);
SULF_INST_SD(2)
SULF_INST_SD(3)

}  // namespace sulf
