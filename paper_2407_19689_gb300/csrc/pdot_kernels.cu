// pdot_kernels.cu -- sm_103a kernels of restarted PDHG for optimal transport
// (arXiv 2407.19689, Algorithm 2 with the Sec. 5 controller).
//
// One iteration, as two launches over a multi-instance work queue:
//   plan pass (plan tiles): forms the projected primal step of Algorithm 2,
//           X+ = max(0, X - tau (C - p 1^T - 1 q^T)), and in registers the row
//           and column sums of X+ - X and ||X+ - X||^2.  FP32 plans and their
//           averages are written by every third pass (k_pass_lag,
//           pdot_pass.cuh), FP64 ones by each (k_pass).
//   k_dual  (vector tiles, O(m+n)): fixed-order reduction of the partial sums,
//           the dual updates p+ = p + sigma (f - (2 r+ - r)),
//           q+ = q + sigma (g - (2 c+ - c)) (r = X 1, c = X^T 1 of the current
//           plan, so 2X+ - X is never re-read), the average of (p, q), and the
//           step-size reductions.  The last vector tile of each instance
//           (atomic ticket) runs the scalar controller: PDLP step-size test,
//           accept/reject by swapping slot roles.
// or, where all tiles are resident at once, the passes and dual updates of a
// check period in one cooperative launch (k_persist, pdot_persist.cuh).
// Every K passes:
//   k_kkt      (plan tiles): reads C, X, Xbar, anchor once; <C,X>, <C,Xbar>,
//              ||[p1^T+1q^T-C]^+||^2 for the current and the average duals,
//              distances to the restart anchor, and exact row/column sums of
//              the stored average.
//   k_checkvec (vector tiles): primal residuals, dual objectives, dual
//              distances; the last tile per instance runs the restart /
//              termination / primal-weight logic of Sec. 5.
// The path is a streaming stencil plus reductions: no tensor cores.  Plan
// tiles are one warp wide (128 columns, 16-byte loads per lane) and
// `tile_rows` tall, handed out by an atomic queue so uneven batches balance.
#include <cuda_runtime.h>
#include <math_constants.h>

#include <type_traits>

#include "pdot_internal.h"

namespace pdot {

constexpr int KU = 2;   // rows per load batch in the register KKT pass
// Rows a plan pass (KKT pass) accumulates in FP32 per lane before adding into
// its FP64 partial sums: FP64 is a narrow pipe on this part, and the FP32
// partial over 32 (64) rows of one column carries a relative error of order
// 1e-7, far below what the FP64 sums it feeds are compared against.
constexpr int FLUSH_ROWS = 32;
constexpr int KKT_FLUSH_ROWS = 64;

// ---------------------------------------------------------------------------
// loads and stores of 4 consecutive elements
// ---------------------------------------------------------------------------
__device__ __forceinline__ void ld4(const float* p, float (&v)[4]) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void ld4(const double* p, double (&v)[4]) {
    const double2 a = reinterpret_cast<const double2*>(p)[0];
    const double2 b = reinterpret_cast<const double2*>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void st4(float* p, const float (&v)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(double* p, const double (&v)[4]) {
    reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}

__device__ __forceinline__ float bf16_bits_to_f32(unsigned int h) { return __uint_as_float(h << 16); }

// Cost entries (read-only for the whole solve: non-coherent path).
template <typename A>
__device__ __forceinline__ void ldc4(const float* p, A (&v)[4]) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = (A)t.x; v[1] = (A)t.y; v[2] = (A)t.z; v[3] = (A)t.w;
}
template <typename A>
__device__ __forceinline__ void ldc4(const unsigned short* p, A (&v)[4]) {
    const uint2 t = __ldg(reinterpret_cast<const uint2*>(p));
    v[0] = (A)bf16_bits_to_f32(t.x & 0xffffu);
    v[1] = (A)bf16_bits_to_f32(t.x >> 16);
    v[2] = (A)bf16_bits_to_f32(t.y & 0xffffu);
    v[3] = (A)bf16_bits_to_f32(t.y >> 16);
}
template <typename A>
__device__ __forceinline__ void ldc4(const double* p, A (&v)[4]) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p));
    const double2 b = __ldg(reinterpret_cast<const double2*>(p) + 1);
    v[0] = (A)a.x; v[1] = (A)a.y; v[2] = (A)b.x; v[3] = (A)b.y;
}
// Ragged right edge: only the first `cnt` (< 4) entries exist.
template <typename A>
__device__ __forceinline__ void ldc4_tail(const float* p, long long cnt, A (&v)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = e < cnt ? (A)__ldg(p + e) : A(0);
}
template <typename A>
__device__ __forceinline__ void ldc4_tail(const unsigned short* p, long long cnt, A (&v)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = e < cnt ? (A)bf16_bits_to_f32(__ldg(p + e)) : A(0);
}
template <typename A>
__device__ __forceinline__ void ldc4_tail(const double* p, long long cnt, A (&v)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = e < cnt ? (A)__ldg(p + e) : A(0);
}

// Tag type of the generated cost (TT_GEN): C_ij comes from coordinates of at
// most DM dimensions (the pass kernel has a 4-dimension variant that keeps
// fewer coordinates in registers).
template <int DM>
struct GenC {};
template <typename TC>
struct GenDims { static constexpr int value = 0; };
template <int DM>
struct GenDims<GenC<DM>> { static constexpr int value = DM; };
using GenC8 = GenC<GEN_DMAX>;
using GenC4 = GenC<4>;

// One lane's four cost entries C[i][j0..j0+3]: read from the stored matrix,
// or generated from the coordinates (the four columns' coordinates are kept in
// registers; the row's are read per call).
template <typename TC, typename A>
struct CostRow {
    const TC* C;
    long long ldc, cnt;
    bool full;
    __device__ __forceinline__ CostRow(const Inst& I, long long j0)
        : C(reinterpret_cast<const TC*>(I.C) + j0), ldc(I.ldc), cnt(I.n - j0), full(j0 + 4 <= I.n) {}
    __device__ __forceinline__ void get(long long i, A (&c)[4]) const {
        if (full) ldc4<A>(C + i * ldc, c);
        else ldc4_tail<A>(C + i * ldc, cnt, c);
    }
};
template <int DM, typename A>
struct CostRow<GenC<DM>, A> {
    GenSpec g;
    float y[4][DM];
    __device__ __forceinline__ CostRow(const Inst& I, long long j0) : g(I.gen) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
#pragma unroll
            for (int k = 0; k < DM; ++k)
                y[e][k] = (k < g.d && j0 + e < I.n) ? __ldg(g.ys + (j0 + e) * g.d + k) : 0.f;
        }
    }
    __device__ __forceinline__ void get(long long i, A (&c)[4]) const {
        float x[DM];
#pragma unroll
        for (int k = 0; k < DM; ++k) x[k] = k < g.d ? __ldg(g.xs + i * g.d + k) : 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) c[e] = (A)gen_cost<DM>(g.kind, g.d, x, y[e], g.div, g.inv);
    }
};

// ---------------------------------------------------------------------------
// Reduced cost C_ij - p_i - q_j of the plan pass (reading C9)
// ---------------------------------------------------------------------------
// FP32 plans take the FP64 duals as FP32 pairs, y = hi + lo with hi = RN(y)
// and lo = RN(y - hi).  With `comp` the reduced cost is then formed so that
// its error is of its own size, not of the size of p and q: the rounding
// error e of s = c - p_hi is recovered exactly (Knuth's TwoSum: c - p_hi =
// s + e), s - q_hi is exact where the reduced cost is small (Sterbenz: s is
// then within a factor 2 of q_hi), and the small terms e, p_lo, q_lo are
// added last.  Without `comp`: (c - p_hi) - q_hi, two FP32 roundings of the
// size of p and q (the plan's fixed point is then only as accurate as that).
// FP64 plans use the FP64 duals directly.
__device__ __forceinline__ void split_dual(double y, float& hi, float& lo) {
    hi = (float)y;
    lo = (float)(y - (double)hi);
}
__device__ __forceinline__ void split_dual(double y, double& hi, double& lo) {
    hi = y;
    lo = 0.0;
}
__device__ __forceinline__ float reduced_cost(float c, float ph, float pl, float qh, float ql, bool comp) {
    if (!comp) return (c - ph) - qh;
    const float s = c - ph;
    const float bv = s - c;
    const float e = (c - (s - bv)) + (-ph - bv);   // c - ph = s + e exactly
    return (s - qh) + (e - (pl + ql));
}
__device__ __forceinline__ double reduced_cost(double c, double ph, double, double qh, double, bool) {
    return (c - ph) - qh;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
    // Butterfly: every lane ends with the same, order-fixed sum.
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <typename TX>
__device__ __forceinline__ TX* slot_x(const Inst& I, int s) {
    return reinterpret_cast<TX*>(I.X) + (long long)s * I.xslot;
}
__device__ __forceinline__ double* slot_v(const Inst& I, int s) { return I.V + (long long)s * I.vslot; }

// Warp-level work queue.
__device__ __forceinline__ int warp_next(unsigned* ctr) {
    int t = 0;
    if ((threadIdx.x & 31) == 0) t = (int)atomicAdd(ctr, 1u);
    return __shfl_sync(0xffffffffu, t, 0);
}

// Tile queue of the plan kernels: a warp's first tile is its global warp
// index (no atomic on the path to the first load); later tiles come from the
// counter, after all first tiles.  Which warp runs a tile does not change its
// arithmetic, so results do not depend on the assignment.
__device__ __forceinline__ int tile_next(unsigned* ctr, bool& first) {
    const int W = (int)(gridDim.x * (blockDim.x >> 5));
    if (first) {
        first = false;
        return (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    }
    return W + warp_next(ctr);
}

// Arrival on an instance's ticket: the atomic releases this thread's earlier
// writes and, for the last arrival, acquires the others' (one acquire-release
// atomic instead of two sequentially consistent fences).
__device__ __forceinline__ unsigned ticket_arrive(unsigned* ctr) {
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(ctr) : "memory");
    return old;
}

// Programmatic dependent launch: wait for the previous grid in the stream
// (completion and memory visibility; a no-op without the launch attribute).
// Every solve-loop kernel calls this before touching any data or work counter.
__device__ __forceinline__ void pdl_enter() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Let the next grid start launching: called when a CTA has finished its work
// (a CTA that exits without calling it counts as having called it).
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Before the wait of a dependent launch: pull the warp's first tile reference
// and its instance descriptor into L1.  Both are written by the host before
// the launch, never by the preceding kernel, so this may run while that
// kernel finishes.
__device__ __forceinline__ void prefetch_first_tile(const Inst* insts, const TileRef* tmap, int T) {
    const int t = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    if (t >= T || (threadIdx.x & 31) != 0) return;
    const TileRef tr = tmap[t];
    const char* ip = reinterpret_cast<const char*>(insts + tr.inst);
    asm volatile("prefetch.global.L1 [%0];" ::"l"(ip));
    asm volatile("prefetch.global.L1 [%0];" ::"l"(ip + 128));
}

__device__ __forceinline__ void reset_other_counters(unsigned* wctr, int mine) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        for (int c = 0; c < WC_N; ++c)
            if (c != mine) wctr[c] = 0u;
    }
}

// ---------------------------------------------------------------------------
// Plan pass: Algorithm 2 primal step + running average + partial sums
// ---------------------------------------------------------------------------
// Row order of a plan tile: every other pass walks its tiles bottom-up, so the
// rows a pass reads first are the ones the previous pass touched last, which
// are still in L2 (C read, X+ and Xbar+ just written) when the plan does not
// fit in it.  Which order a pass takes changes only the order of its FP32
// column partial sums; it is a function of the instance's pass count (and of
// `dir_xor`, a launch parameter used by the pass timer), so runs stay
// reproducible and an instance gives the same result alone or in a batch.
__device__ __forceinline__ bool pass_reversed(const Ctrl& S, int dir_xor) {
    return ((S.passes ^ (long long)dir_xor) & 1) != 0;
}

// Uniform running average of Algorithm 2, kept as its deviation from the
// current plan, D = Xbar - X: Xbar+ = Xbar + w (X+ - Xbar) becomes
// D+ = (1 - w)(D - d) with d = X+ - X, and D+ = 0 for the first iterate of an
// epoch (Xbar+ = X+).  Stored this way, the rounding of each update is
// relative to |D| (the spread of the iterates around their mean, which
// shrinks as the solve converges), not to |Xbar|: an FP32 average updated in
// place loses the late iterates' weight w = 1/(k+1) below its last bit.
__device__ __forceinline__ float avg_dev_next(float dbar, float d, float w, bool first) {
    const float s = dbar - d;
    return first ? 0.f : fmaf(-w, s, s);
}
__device__ __forceinline__ double avg_dev_next(double dbar, double d, double w, bool first) {
    const double s = dbar - d;
    return first ? 0.0 : fma(-w, s, s);
}

// CP: compensated reduced cost (a kernel template parameter, so the plain
// path is compiled without the compensated one and costs nothing extra).
template <typename TC, typename TX, int U, bool CP>
__device__ __forceinline__ void pass_tile(const Inst& I, const Ctrl& S, int lt, int lane, bool rev) {
    typedef TX A;
    const long long m = I.m, n = I.n, ldx = I.ldx;
    const int strip = lt % I.nstrips, chunk = lt / I.nstrips;
    const long long j0 = (long long)strip * STRIP + lane * 4;
    const long long i0 = (long long)chunk * I.tile_rows;
    const long long i1 = min(i0 + (long long)I.tile_rows, m);
    const bool on = j0 < n;
    const CostRow<TC, A> cr(I, j0);
    const TX* X = slot_x<TX>(I, S.cur);
    const TX* Xb = slot_x<TX>(I, S.bar);
    TX* Xn = slot_x<TX>(I, S.nxt);
    TX* Xbn = slot_x<TX>(I, S.barn);
    const double* p = slot_v(I, S.cur);
    const double* q = p + m;
    const bool first = S.k == 0;
    const A tau = (A)S.tau;
    const A w = (A)S.wavg;

    A qv[4], ql[4];
    bool valid[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        valid[e] = j0 + e < n;
        split_dual(valid[e] ? q[j0 + e] : 0.0, qv[e], ql[e]);
    }
    double cs[4] = {0.0, 0.0, 0.0, 0.0};
    double dx2 = 0.0;
    double* rowpart = I.rowpart + (long long)strip * m;
    const long long nb = (i1 - i0 + U - 1) / U;   // batches of U rows, walked in either order

    for (long long bi = 0; bi < nb; ++bi) {
        const long long ib = i0 + (rev ? nb - 1 - bi : bi) * U;
        // Row pointers of the batch (lanes past n never dereference).
        const long long xo = ib * ldx + j0;
        const TX* Xr = X + xo;
        const TX* Xbr = Xb + xo;
        TX* Xnr = Xn + xo;
        TX* Xbnr = Xbn + xo;
        A c[U][4], x[U][4], xb[U][4], pv[U], pl[U];
        // Issue every load of the U-row batch before any arithmetic.
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool rv = ib + u < i1;
            split_dual(rv ? p[ib + u] : 0.0, pv[u], pl[u]);
            if (rv && on) {
                cr.get(ib + u, c[u]);
                ld4(Xr + u * ldx, x[u]);
                if (!first) ld4(Xbr + u * ldx, xb[u]);
                else {
#pragma unroll
                    for (int e = 0; e < 4; ++e) xb[u][e] = A(0);
                }
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) { c[u][e] = A(0); x[u][e] = A(0); xb[u][e] = A(0); }
            }
        }
        A csa[4] = {A(0), A(0), A(0), A(0)};
        A dxa = A(0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool rv = ib + u < i1;
            A xn[4], xbn[4];
            A rs = A(0);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const A R = reduced_cost(c[u][e], pv[u], pl[u], qv[e], ql[e], CP);   // C - p - q
                A v = x[u][e] - tau * R;
                v = v > A(0) ? v : A(0);                         // projection onto X >= 0
                v = (valid[e] && rv) ? v : A(0);                 // padding columns / rows past the tile stay 0
                const A d = v - x[u][e];
                dxa += d * d;
                rs += d;                                          // row / column sums of X+ - X
                csa[e] += d;
                xn[e] = v;
                xbn[e] = avg_dev_next(xb[u][e], d, w, first);
            }
            if (rv && on) {
                st4(Xnr + u * ldx, xn);
                st4(Xbnr + u * ldx, xbn);
            }
            rs = warp_sum(rs);
            if (rv && lane == 0) rowpart[ib + u] = (double)rs;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) cs[e] += (double)csa[e];
        dx2 += (double)dxa;
    }
    if (on) {
        double* cp = I.colpart + (long long)chunk * ldx + j0;
        reinterpret_cast<double2*>(cp)[0] = make_double2(cs[0], cs[1]);
        reinterpret_cast<double2*>(cp)[1] = make_double2(cs[2], cs[3]);
    }
    dx2 = warp_sum(dx2);
    if (lane == 0) I.tpart[(long long)lt * TP + 0] = dx2;
}

template <typename TC, typename TX, int U, bool CP>
__global__ void __launch_bounds__(TWARPS * 32, sizeof(TX) == 4 ? 2 : 1)
k_pass(const Inst* __restrict__ insts, const TileRef* __restrict__ tmap, const int* __restrict__ Tp, unsigned* wctr, int wc,
       int dir_xor) {
    pdl_enter();
    const int T = *Tp;
    reset_other_counters(wctr, wc);
    const int lane = threadIdx.x & 31;
    bool first = true;
    for (;;) {
        const int t = tile_next(&wctr[wc], first);
        if (t >= T) break;
        const TileRef tr = tmap[t];
        const Inst& I = insts[tr.inst];
        const Ctrl& S = *I.ctrl;
        if (S.status != ST_RUNNING) continue;
        pass_tile<TC, TX, U, CP>(I, S, tr.local, lane, pass_reversed(S, dir_xor));
    }
}

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Row duals staged per window of PWIN rows (the KKT pass).
constexpr int PWIN = 128;

struct RowRef {       // what a stage holds
    int tile;         // global tile index (into tmap), -1 = none
    int row;          // matrix row
};

}  // namespace pdot

#include "pdot_pass.cuh"

namespace pdot {

// ---------------------------------------------------------------------------
// Slot bookkeeping
// ---------------------------------------------------------------------------
// nxt and barn <- the two lowest slots not in use as cur, bar or anc.
__device__ __forceinline__ void assign_free(Ctrl* S, int cur, int bar, int anc) {
    const int used = (1 << cur) | (1 << bar) | (1 << anc);
    int picks[2] = {0, 0};
    int np = 0;
    for (int s = 0; s < NSLOT && np < 2; ++s)
        if (!(used & (1 << s))) picks[np++] = s;
    S->nxt = picks[0];
    S->barn = picks[1];
}


// ---------------------------------------------------------------------------
// Dual step + PDLP step-size controller
// ---------------------------------------------------------------------------
// The schedule factors of attempted iteration t1 = total + 2 (reading C6).
struct SchedFactors {
    double f3, f6;   // t1^-0.3, t1^-0.6
};
__device__ __forceinline__ SchedFactors sched_factors(const Ctrl* S, long long total) {
    SchedFactors r;
    if (total < S->sched_len) {
        r.f3 = __ldg(S->sched + 2 * total);
        r.f6 = __ldg(S->sched + 2 * total + 1);
    } else {
        const double t1 = (double)(total + 2);
        r.f3 = pow(t1, -0.3);
        r.f6 = pow(t1, -0.6);
    }
    return r;
}

// The controller fields the step decision reads.  Only the decision itself
// writes them during a dual update, so a copy taken when the update starts
// is current when the instance's last tile decides; taking it early keeps
// those reads off the serial path (after the ticket's acquire they would go
// to L2 again).
struct StepPre {
    double eta, omega;
    long long passes, k, total, rejected;
    int cur, nxt, bar, barn, anc, adaptive_step;
    int lag, npend, h0, xcur, xbar, xanc, xdst;
    float tau, wavg;
};
__device__ __forceinline__ StepPre step_pre(const Ctrl* S) {
    StepPre P;
    P.eta = S->eta;
    P.omega = S->omega;
    P.passes = S->passes;
    P.k = S->k;
    P.total = S->total;
    P.rejected = S->rejected;
    P.cur = S->cur;
    P.nxt = S->nxt;
    P.bar = S->bar;
    P.barn = S->barn;
    P.anc = S->anc;
    P.adaptive_step = S->adaptive_step;
    P.lag = S->lag;
    P.npend = S->npend;
    P.h0 = S->h0;
    P.xcur = S->xcur;
    P.xbar = S->xbar;
    P.xanc = S->xanc;
    P.xdst = S->xdst;
    P.tau = (float)S->tau;
    P.wavg = (float)S->wavg;
    return P;
}

// isfinite in integer arithmetic (an FP64 comparison takes the FP64 pipe 64
// cycles on the controller's serial path).
__device__ __forceinline__ bool finite_bits(double v) {
    return (((unsigned)__double2hiint(v) >> 20) & 2047u) != 2047u;
}

// w_next: 1 / (k + 2), the averaging weight after an accepted step (computed
// by the caller early, off this serial path).  P: step_pre(S), taken at any
// point after the previous decision.
__device__ void finalize_step(Ctrl* S, const StepPre& P, double dX2, double dy2, double inter, SchedFactors fac,
                              double w_next) {
    S->passes = P.passes + 1;
    S->fix = 0;   // the plan a restart picked has been formed before this pass, also where the pass ends the solve
    S->last_dX2 = dX2;
    S->last_dy2 = dy2;
    S->last_inter = inter;
    bool accept = true;
    double eta = P.eta;
    if (P.adaptive_step) {
        // Sec. 5 step-size rule in the PDLP form (reading C6); the exponent base
        // is the 1-based index of the attempted iteration plus one.
        // The accept/reject decision is discrete: it is taken in FP64 with
        // the same expression as the FP64 reference of the rule, so that
        // both sides decide alike away from exact ties.
        const double om = P.omega;
        const double etabar = inter != 0.0 ? (om * dX2 + dy2 / om) / (2.0 * fabs(inter)) : CUDART_INF;
        const double a = (1.0 - fac.f3) * etabar;
        const double b = (1.0 + fac.f6) * eta;
        const double eta_next = a < b ? a : b;
        accept = eta <= etabar;
        S->last_etabar = etabar;
        eta = eta_next;
    }
    if (!finite_bits(dX2) || !finite_bits(dy2) || !finite_bits(eta) || !(eta > 0.0)) {
        S->status = ST_NUMERIC;
        S->res_slot = P.cur;
        S->res_avg = 0;
        // The current plan: with deferred writes, where this pass or the
        // final pass has applied the pending steps.
        S->res_xslot = !P.lag ? P.cur : P.npend ? P.xdst : P.xcur;
        if (P.lag && P.npend == P.lag) {
            S->xcur = P.xdst;
            S->npend = 0;
        }
        return;
    }
    if (P.lag) {
        // Deferred plan writes: this pass has applied the pending steps if
        // there were `lag` of them; an accepted step becomes pending.
        int np = P.npend;
        const int c = (P.h0 + np) % YRING;   // ring index of this pass's duals
        if (np == P.lag) {
            np = 0;
            S->h0 = c;
            S->xcur = P.xdst;
            S->xdst = plan_dst(P.xdst, P.xbar, P.xanc);
        }
        if (accept) {
            if (np == 0) S->pfirst = P.k == 0;
            S->ptau[c] = P.tau;
            S->pw[c] = P.wavg;
            ++np;
        }
        S->npend = np;
    }
    if (accept) {
        S->cur = P.nxt;
        S->bar = P.barn;
        if (!P.lag) {
            S->xcur = P.nxt;
            S->xbar = P.barn;
        }
        assign_free(S, P.nxt, P.barn, P.anc);
        S->k = P.k + 1;
        S->wavg = w_next;
        S->total = P.total + 1;
    } else {
        S->rejected = P.rejected + 1;
    }
    if (P.adaptive_step) {   // (a constant step keeps tau and sigma)
        S->eta = eta;
        S->tau = eta / P.omega;
        S->sigma = eta * P.omega;
    }
}

__device__ __forceinline__ void finalize_step(Ctrl* S, double dX2, double dy2, double inter, SchedFactors fac,
                                              double w_next) {
    finalize_step(S, step_pre(S), dX2, dy2, inter, fac, w_next);
}

// Group sum of FP64 (or FP32) partials k = grp, grp + VG, ... < count in order,
// at part + k * stride, U of them requested together.  A partial that is zero
// in all 32 lanes is not added (it changes nothing, and an FP64 addition takes
// 64 cycles of its scheduler): the plan of a solve is sparse, so most tiles
// leave most columns as they were.
__device__ __forceinline__ bool nonzero(double v) {
    return ((unsigned)__double2hiint(v) << 1 | (unsigned)__double2loint(v)) != 0u;
}
__device__ __forceinline__ bool nonzero(float v) { return v != 0.f; }
__device__ __forceinline__ double as_double(double v) { return v; }
__device__ __forceinline__ double as_double(float v) { return lagp::widen(v); }
// (The loads are volatile: the compiler otherwise moves each one behind the
// test that uses it.)
__device__ __forceinline__ double ld_part(const double* p, bool in) {
    double v;
    asm volatile("{ .reg .pred t; setp.ne.u32 t, %2, 0; mov.b64 %0, 0; @t ld.global.cg.f64 %0, [%1]; }"
                 : "=d"(v) : "l"(p), "r"((unsigned)in));
    return v;
}
__device__ __forceinline__ float ld_part(const float* p, bool in) {
    float v;
    asm volatile("{ .reg .pred t; setp.ne.u32 t, %2, 0; mov.b32 %0, 0; @t ld.global.cg.f32 %0, [%1]; }"
                 : "=f"(v) : "l"(p), "r"((unsigned)in));
    return v;
}
// off: added to the group of some lanes (whose groups' indexes are not smaller).
template <int U, typename T>
__device__ __forceinline__ double group_sum(const T* part, int stride, int count, int grp, bool active, int off = 0) {
    double s = 0.0;
#pragma unroll 1
    for (int k = grp; k < count; k += U * VG) {
        T v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            v[u] = ld_part(part + (long long)(k + off + u * VG) * stride, active && k + off + u * VG < count);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k + u * VG >= count) break;
            if (__any_sync(0xffffffffu, nonzero(v[u]))) s += as_double(v[u]);
        }
    }
    return s;
}

// One vector tile (VE = 32 entries of [p; q]) per CTA.  All warps add the
// FP64 partial sums of the tile's row or column sums (group g: partials g,
// g + VG, ...).  FP64 takes 64 cycles per warp instruction on each of an SM's
// four schedulers, so what follows is spread over four warps: warps 0, 1 and 3
// combine the groups in order and form the duals and ||dy||^2, dy^T A dx, and
// the new sums and averages; warp 2 has the tile's slice of ||dX||^2 and warp 4
// what the controller needs besides the sums.  The instance's last tile (a
// ticket) adds the tiles' scalars, one per warp, and runs the step controller.
// (One warp for all of it: 19.0 us a launch with 16 uneven instances, here 16.6.)
struct DualShared {
    double grp[VG * 32];
    double sum[3];
    double w_next;
    SchedFactors fac;
    StepPre pre;
    int last;
};
__device__ void dual_tile(const Inst& I, Ctrl* S, int lvt, DualShared& sh) {
    const long long m = I.m, n = I.n;
    const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const long long e = (long long)lvt * VE + lane;
    const bool row = e < m, col = !row && e < m + n;
    const long long idx = row ? e : e - m;
    const long long so = m + n + e;                             // r_i or c_j
    const bool upd = grp == 0 || grp == 1 || grp == 3;
    if (S->status != ST_RUNNING) return;
    double sigma = 0.0, b = 0.0, r = 0.0, y = 0.0, ybar = 0.0, wavg = 1.0;
    long long k = 0;
    double* Vn = nullptr;
    double* Vbn = nullptr;
    float2* yfn = nullptr;
    if (upd) {
        sigma = S->sigma;
        k = S->k;
        wavg = S->wavg;
        const double* Vc = slot_v(I, S->cur);
        const double* Vb = slot_v(I, S->bar);
        Vn = slot_v(I, S->nxt);
        Vbn = slot_v(I, S->barn);
        if (S->lag) yfn = I.yf + (long long)((S->h0 + S->npend + 1) % YRING) * I.yslot;
        if (row || col) {
            b = row ? I.f[idx] : I.g[idx];
            r = Vc[so];
            y = Vc[e];
            if (k != 0 && grp == 3) ybar = Vb[e];
        }
    }
    // (a tile can hold the last rows and the first columns: two runs then)
    const bool any_row = (long long)lvt * VE < m, any_col = (long long)lvt * VE + VE > m;
    double s = 0.0;
    if (any_row) s = group_sum<4>(I.rowpart + idx, (int)m, I.nstrips, grp, row);
    if (any_col) {
        const double c = group_sum<8>(I.colpart + idx, (int)I.ldx, I.nchunks, grp, col);
        if (col) s = c;
    }
    sh.grp[grp * 32 + lane] = s;
    double* vp = I.vpart + (long long)lvt * VP;
    if (grp == 2) {
        // This tile's slice of the plan tiles' ||X+ - X||^2 partials.
        const int t0 = (int)((long long)I.ntiles * lvt / I.nvt), t1 = (int)((long long)I.ntiles * (lvt + 1) / I.nvt);
        double a2 = 0.0;
        for (int tt = t0 + lane; tt < t1; tt += 32) a2 += I.tpart[(long long)tt * TP];
        a2 = warp_sum(a2);
        if (lane == 0) vp[2] = a2;
    }
    __syncthreads();
    if (upd) {
        double t = sh.grp[lane];
#pragma unroll
        for (int g2 = 1; g2 < VG; ++g2) t += sh.grp[g2 * 32 + lane];
        // t: this row's or column's sum of X+ - X (the pass sums the change
        // itself, so the step-size term dy^T A dX below is not a difference
        // of two nearly equal sums); (2X+ - X) 1 = r + 2t, X+ 1 = r + t.
        const double yn = y + sigma * (b - (r + 2.0 * t));
        const bool in = row || col;
        if (grp == 3) {
            if (in) {
                Vn[so] = r + t;
                Vbn[e] = k == 0 ? yn : ybar + wavg * (yn - ybar);
            }
        } else {
            const double dy = yn - y;
            double a = 0.0;
            if (in) a = grp == 0 ? dy * dy : dy * t;
            if (grp == 0 && in) {
                Vn[e] = yn;
                if (yfn) {   // the next pass reads the duals as FP32 pairs: split once here, not in every plan tile
                    float2 v;
                    split_dual(yn, v.x, v.y);
                    yfn[e] = v;
                }
            }
            a = warp_sum(a);
            if (lane == 0) vp[grp] = a;
        }
    } else if (threadIdx.x == 4 * 32) {
        // Used by the instance's last tile.  Only the step decision itself
        // writes these fields during a dual update.
        sh.w_next = 1.0 / (double)(S->k + 2);
        if (S->adaptive_step) sh.fac = sched_factors(S, S->total);
        sh.pre = step_pre(S);
    }
    __syncthreads();
    if (threadIdx.x == 0) sh.last = ticket_arrive(I.ticket) == (unsigned)(I.nvt - 1) ? 1 : 0;
    __syncthreads();
    if (!sh.last) return;
    if (grp < 3) {
        double t = 0.0;
        for (int v = lane; v < I.nvt; v += 32) {
            const double a = __ldcg(I.vpart + (long long)v * VP + grp);
            t = v == lane ? a : t + a;
        }
        t = warp_sum(t);
        if (lane == 0) sh.sum[grp] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        *I.ticket = 0u;
        finalize_step(S, sh.pre, sh.sum[2], sh.sum[0], sh.sum[1], sh.fac, sh.w_next);
    }
}

__global__ void __launch_bounds__(VT) k_dual(const Inst* __restrict__ insts, const TileRef* __restrict__ vmap,
                                             const int* __restrict__ NVp, unsigned* wctr, int direct) {
    // One CTA per vector tile (no work queue): the grid covers the tile count.
    // direct: one instance whose vector tiles are exactly the grid (no map or
    // count to read before the work).
    __shared__ DualShared sh;
    pdl_enter();
    // The next pass may start launching now: it waits for this grid to
    // complete before it reads anything this grid writes, and its CTAs use
    // the time to set up (a no-op without programmatic dependent launch).
    pdl_release();
    // No work counter of its own, but it still resets the others for the
    // kernels that follow (block 0, before any early exit).
    reset_other_counters(wctr, wc_index(WC_DUAL, 0));
    TileRef tr;
    if (direct) {
        tr.inst = 0;
        tr.local = (int)blockIdx.x;
    } else {
        const int NV = *NVp;
        if ((int)blockIdx.x >= NV) return;
        tr = vmap[blockIdx.x];
    }
    const Inst& I = insts[tr.inst];
    // (a finished instance's tile does nothing)
    dual_tile(I, I.ctrl, tr.local, sh);
}

// ---------------------------------------------------------------------------
// KKT pass (every K passes, and once at the start)
// ---------------------------------------------------------------------------
template <typename TC, typename TX>
__device__ __forceinline__ void kkt_tile(const Inst& I, const Ctrl& S, int lt, int lane, int mode) {
    typedef TX A;
    const long long m = I.m, n = I.n, ldx = I.ldx;
    const int strip = lt % I.nstrips, chunk = lt / I.nstrips;
    const long long j0 = (long long)strip * STRIP + lane * 4;
    const long long i0 = (long long)chunk * I.tile_rows;
    const long long i1 = min(i0 + (long long)I.tile_rows, m);
    const bool on = j0 < n;
    const CostRow<TC, A> cr(I, j0);
    const bool init = mode == MODE_INIT;
    const bool avg = !init && S.k > 0;      // the running average exists
    const bool sums = init || avg;          // exact row/col sums of X (init) or Xbar (check)
    const TX* X = slot_x<TX>(I, plan_slot(S));
    const TX* Xb = slot_x<TX>(I, S.xbar);
    const TX* Xa = slot_x<TX>(I, S.xanc);
    const double* p = slot_v(I, S.cur);
    const double* q = p + m;
    const double* pb = slot_v(I, S.bar);
    const double* qb = pb + m;

    // The check's dual residual [p + q - C]^+ takes the plain reduced cost:
    // its FP32 rounding (of the size of p and q) is far below ||C||_F, the
    // scale this term is measured against.
    A qv[4], qbv[4];
    bool valid[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        valid[e] = j0 + e < n;
        qv[e] = valid[e] ? (A)q[j0 + e] : A(0);
        qbv[e] = (valid[e] && avg) ? (A)qb[j0 + e] : A(0);
    }
    double acc[TP] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};   // cxc, rd2c, cxb, rd2b, dXac, dXab
    double cs[4] = {0.0, 0.0, 0.0, 0.0};
    double cs2[4] = {0.0, 0.0, 0.0, 0.0};   // check: exact column sums of the current plan
    double* rowpart = I.rowpart + (long long)strip * m;
    double* rowpart2 = I.rowpart2 + (long long)strip * m;

    // FP32 plans accumulate in FP32 over KKT_FLUSH_ROWS rows before adding
    // into the FP64 partials (an FP64 add per batch of two rows would make
    // this pass bound by the narrow FP64 pipe) -- the same grouping as
    // k_kkt_staged, so both give the same bits.
    constexpr int KFLUSH = sizeof(A) == 4 ? KKT_FLUSH_ROWS / KU : 1;
    A t[TP] = {A(0), A(0), A(0), A(0), A(0), A(0)};
    A csa[4] = {A(0), A(0), A(0), A(0)}, csa2[4] = {A(0), A(0), A(0), A(0)};
    int nbatch = 0;
    for (long long ib = i0; ib < i1; ib += KU) {
        A c[KU][4], x[KU][4], xb[KU][4], xa[KU][4], pv[KU], pbv[KU];
#pragma unroll
        for (int u = 0; u < KU; ++u) {
            const long long i = ib + u;
            const bool rv = i < i1;
            pv[u] = rv ? (A)p[i] : A(0);
            pbv[u] = (rv && avg) ? (A)pb[i] : A(0);
#pragma unroll
            for (int e = 0; e < 4; ++e) { c[u][e] = A(0); x[u][e] = A(0); xb[u][e] = A(0); xa[u][e] = A(0); }
            if (rv && on) {
                cr.get(i, c[u]);
                ld4(X + i * ldx + j0, x[u]);
                if (avg) {
                    ld4(Xb + i * ldx + j0, xb[u]);
                    ld4(Xa + i * ldx + j0, xa[u]);
#pragma unroll
                    for (int e = 0; e < 4; ++e) xb[u][e] = x[u][e] + xb[u][e];   // the average: X + D
                } else if (!init) {
                    ld4(Xa + i * ldx + j0, xa[u]);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < KU; ++u) {
            const long long i = ib + u;
            const bool rv = i < i1;
            A rs = A(0), rs2 = A(0);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (!valid[e] || !rv) continue;
                const A Rc = (c[u][e] - pv[u]) - qv[e];
                t[0] += c[u][e] * x[u][e];
                t[1] += Rc < A(0) ? Rc * Rc : A(0);             // [p + q - C]^+ squared
                const A da = x[u][e] - xa[u][e];
                t[4] += da * da;
                if (init) t[2] += c[u][e] * c[u][e];             // ||C||_F^2 (once per solve)
                if (avg) {
                    const A Rb = (c[u][e] - pbv[u]) - qbv[e];
                    t[2] += c[u][e] * xb[u][e];
                    t[3] += Rb < A(0) ? Rb * Rb : A(0);
                    const A db = xb[u][e] - xa[u][e];
                    t[5] += db * db;
                }
                const A sv = init ? x[u][e] : xb[u][e];
                rs += sv;
                csa[e] += sv;
                rs2 += x[u][e];
                csa2[e] += x[u][e];
            }
            if (sums) {
                rs = warp_sum(rs);
                if (rv && lane == 0) rowpart[i] = (double)rs;
            }
            if (!init) {
                rs2 = warp_sum(rs2);
                if (rv && lane == 0) rowpart2[i] = (double)rs2;
            }
        }
        if (++nbatch == KFLUSH || ib + KU >= i1) {
#pragma unroll
            for (int k = 0; k < TP; ++k) {
                acc[k] += (double)t[k];
                t[k] = A(0);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                cs[e] += (double)csa[e];
                cs2[e] += (double)csa2[e];
                csa[e] = A(0);
                csa2[e] = A(0);
            }
            nbatch = 0;
        }
    }
    if (sums && on) {
        double* cp = I.colpart + (long long)chunk * ldx + j0;
        reinterpret_cast<double2*>(cp)[0] = make_double2(cs[0], cs[1]);
        reinterpret_cast<double2*>(cp)[1] = make_double2(cs[2], cs[3]);
    }
    if (!init && on) {
        double* cp = I.colpart2 + (long long)chunk * ldx + j0;
        reinterpret_cast<double2*>(cp)[0] = make_double2(cs2[0], cs2[1]);
        reinterpret_cast<double2*>(cp)[1] = make_double2(cs2[2], cs2[3]);
    }
#pragma unroll
    for (int k = 0; k < TP; ++k) acc[k] = warp_sum(acc[k]);
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < TP; ++k) I.tpart[(long long)lt * TP + k] = acc[k];
    }
}

template <typename TC, typename TX>
__global__ void __launch_bounds__(TWARPS * 32, sizeof(TX) == 4 ? 2 : 1)
k_kkt(const Inst* __restrict__ insts, const TileRef* __restrict__ tmap, const int* __restrict__ Tp, unsigned* wctr, int wc, int mode) {
    pdl_enter();
    const int T = *Tp;
    reset_other_counters(wctr, wc);
    const int lane = threadIdx.x & 31;
    bool first = true;
    for (;;) {
        const int t = tile_next(&wctr[wc], first);
        if (t >= T) break;
        const TileRef tr = tmap[t];
        const Inst& I = insts[tr.inst];
        const Ctrl& S = *I.ctrl;
        if (S.status != ST_RUNNING) continue;
        kkt_tile<TC, TX>(I, S, tr.local, lane, mode);
    }
}

// ---------------------------------------------------------------------------
// KKT pass, staged (FP32 plans with a stored FP32 or BF16 cost): the
// arithmetic of kkt_tile, with each warp streaming its tile's rows of C, X, D
// and the restart anchor through KS shared-memory stages.  Every lane copies
// the 16 bytes it reads itself (cp.async; by bulk copies the rows took 40
// cycles each of an SM's copy engine: this kernel at 4096 x 4096 74 us, here 61).
// The FP32 accumulators are added into FP64 every 64 rows.
// ---------------------------------------------------------------------------
constexpr int KS = 4;                     // stages per warp (two CTAs per SM: 64 rows of 4 arrays in flight)
constexpr int KSTAGE = 4 * STRIP * 4;     // C (<= 512 B), X, Xbar, anchor (512 B each)
constexpr int KACC = TP + 8;              // FP64 accumulators per lane kept in shared memory (6 scalars, 2 x 4 columns)
__host__ __device__ constexpr int kkt_warp_smem() {
    return KS * KSTAGE + KS * 16 + PWIN * 8 + KACC * 32 * 8;
}
constexpr int kkt_smem() { return TWARPS * kkt_warp_smem(); }

template <typename TC>
__global__ void __launch_bounds__(TWARPS * 32, 2)
k_kkt_staged(const Inst* __restrict__ insts, const TileRef* __restrict__ tmap, const int* __restrict__ Tp,
           unsigned* wctr, int wc, int mode) {
    const int T = *Tp;   // host-written: read before the wait
    extern __shared__ __align__(128) unsigned char dsm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char* wbase = dsm + warp * kkt_warp_smem();
    RowRef* refs = reinterpret_cast<RowRef*>(wbase + KS * KSTAGE);
    float2* pbuf = reinterpret_cast<float2*>(wbase + KS * KSTAGE + KS * 16);   // (p_i, pbar_i) of a row window
    // The lane's FP64 accumulators (kept out of registers): [k * 32 + lane],
    // k < TP the tile scalars, then 4 column sums (average / initial plan), 4
    // column sums (current plan).
    double* sacc = reinterpret_cast<double*>(wbase + KS * KSTAGE + KS * 16 + PWIN * 8);
    const unsigned wbase_s = smem_u32(wbase);
    prefetch_first_tile(insts, tmap, T);
    pdl_enter();
    reset_other_counters(wctr, wc);
    const bool init = mode == MODE_INIT;

    // ---- producer ----
    int p_tile = T;
    int p_row = 0, p_end = 0, p_last = -1;
    const TC* p_c = nullptr;        // this lane's columns of C and X in the row to copy; D and the anchor as offsets from X
    const float* p_x = nullptr;
    long long p_cstride = 0, p_xstride = 0, p_db = 0, p_da = 0;
    unsigned p_cb = 0, p_xb = 0;    // bytes of C and X this lane has in a row
    bool p_avg = false;
    bool q_first = true;
    auto next_tile = [&]() {
        for (;;) {
            p_tile = tile_next(&wctr[wc], q_first);
            if (p_tile >= T) return;
            const TileRef tr = tmap[p_tile];
            const Inst& I = insts[tr.inst];
            const Ctrl& Sc = *I.ctrl;
            if (Sc.status != ST_RUNNING) continue;
            const unsigned strip = (unsigned)tr.local % (unsigned)I.nstrips, chunk = (unsigned)tr.local / (unsigned)I.nstrips;
            const long long c0 = (long long)strip * STRIP;
            const int mine = (int)min(4LL, I.n - c0 - lane * 4);   // columns of this lane (<= 0: none)
            const long long j = c0 + (mine > 0 ? lane * 4 : 0);
            p_row = (int)chunk * I.tile_rows;
            p_end = min(p_row + I.tile_rows, (int)I.m);
            p_xstride = I.ldx;
            p_cstride = I.ldc;
            p_c = reinterpret_cast<const TC*>(I.C) + p_row * p_cstride + j;
            const float* Xb = reinterpret_cast<const float*>(I.X);
            const int sx = plan_slot(Sc);
            p_x = Xb + (long long)sx * I.xslot + p_row * p_xstride + j;
            p_db = (long long)(Sc.xbar - sx) * I.xslot;
            p_da = (long long)(Sc.xanc - sx) * I.xslot;
            p_xb = mine > 0 ? 16u : 0u;
            p_cb = mine > 0 ? (unsigned)mine * (unsigned)sizeof(TC) : 0u;
            p_last = mine < 4 ? (int)I.m - 1 : -1;   // the row whose padding may be past the allocation
            p_avg = !init && Sc.k > 0;
            return;
        }
    };
    long long issued = 0, consumed = 0;
    auto issue = [&]() {
        const int st = (int)(issued % KS);
        const unsigned dst = wbase_s + st * KSTAGE + (unsigned)lane * 16u;
        const bool off = p_xb == 0u;
        lagp::cp16z(dst + STRIP * 4, p_x, off);
        if (p_avg) lagp::cp16z(dst + 2 * STRIP * 4, p_x + p_db, off);
        if (!init) lagp::cp16z(dst + 3 * STRIP * 4, p_x + p_da, off);
        if constexpr (sizeof(TC) == 4) lagp::cp16(dst, p_c, p_row == p_last ? p_cb : p_xb);
        else lagp::cp8(dst - lane * 8u, p_c, p_row == p_last ? p_cb : p_xb / 2u);
        lagp::cp_commit();
        if (lane == 0) {
            refs[st].tile = p_tile;
            refs[st].row = p_row;
        }
        ++issued;
        p_x += p_xstride;
        p_c += p_cstride;
        if (++p_row >= p_end) next_tile();
    };
    next_tile();
    while (issued < KS && p_tile < T) issue();

    // ---- consumer ----
    int c_tile = -1, c_local = 0;
    const Inst* CI = nullptr;
    long long c_i0 = 0, c_i1 = 0, c_n = 0, c_chunk = 0, c_win = -1, j0 = 0;
    bool on = false, c_avg = false, valid[4] = {false, false, false, false};
    float qv[4] = {0.f, 0.f, 0.f, 0.f}, qbv[4] = {0.f, 0.f, 0.f, 0.f};
    const double* c_p = nullptr;
    const double* c_pb = nullptr;
    double* c_rowpart = nullptr;
    double* c_rowpart2 = nullptr;
    float t[TP], csa[4], csa2[4];
    int rows_in_batch = 0;
    bool flushed = false;
    auto flush_acc = [&]() {
#pragma unroll
        for (int k = 0; k < TP; ++k) {
            const double v = lagp::widen(t[k]);
            sacc[k * 32 + lane] = flushed ? sacc[k * 32 + lane] + v : v;
            t[k] = 0.f;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const double v = lagp::widen(csa[e]), v2 = lagp::widen(csa2[e]);
            sacc[(TP + e) * 32 + lane] = flushed ? sacc[(TP + e) * 32 + lane] + v : v;
            sacc[(TP + 4 + e) * 32 + lane] = flushed ? sacc[(TP + 4 + e) * 32 + lane] + v2 : v2;
            csa[e] = 0.f;
            csa2[e] = 0.f;
        }
        flushed = true;
        rows_in_batch = 0;
    };
    auto flush_tile = [&]() {
        if (c_tile < 0) return;
        flush_acc();
        const double* cs = sacc + TP * 32;
        if (on && (init || c_avg)) {
            double* cp = CI->colpart + c_chunk * CI->ldx + j0;
            reinterpret_cast<double2*>(cp)[0] = make_double2(cs[0 * 32 + lane], cs[1 * 32 + lane]);
            reinterpret_cast<double2*>(cp)[1] = make_double2(cs[2 * 32 + lane], cs[3 * 32 + lane]);
        }
        if (on && !init) {
            double* cp = CI->colpart2 + c_chunk * CI->ldx + j0;
            reinterpret_cast<double2*>(cp)[0] = make_double2(cs[4 * 32 + lane], cs[5 * 32 + lane]);
            reinterpret_cast<double2*>(cp)[1] = make_double2(cs[6 * 32 + lane], cs[7 * 32 + lane]);
        }
#pragma unroll
        for (int k = 0; k < TP; ++k) {
            if (init ? k > 2 : (!c_avg && (k == 2 || k == 3 || k == 5))) continue;   // not read by the check
            const double a = warp_sum(sacc[k * 32 + lane]);
            if (lane == 0) CI->tpart[(long long)c_local * TP + k] = a;
        }
    };
    auto open_consumer = [&](int tt) {
        flush_tile();
        c_tile = tt;
        const TileRef tr = tmap[tt];
        CI = &insts[tr.inst];
        const Ctrl& Sc = *CI->ctrl;
        c_local = tr.local;
        const int strip = tr.local % CI->nstrips;
        c_chunk = tr.local / CI->nstrips;
        const long long c0 = (long long)strip * STRIP;
        c_n = CI->n;
        c_i0 = c_chunk * CI->tile_rows;
        c_i1 = min(c_i0 + (long long)CI->tile_rows, CI->m);
        j0 = c0 + lane * 4;
        on = j0 < c_n;
        c_avg = !init && Sc.k > 0;
        c_p = slot_v(*CI, Sc.cur);
        c_pb = slot_v(*CI, Sc.bar);
        const double* q = c_p + CI->m;
        const double* qb = c_pb + CI->m;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            valid[e] = j0 + e < c_n;
            qv[e] = valid[e] ? (float)q[j0 + e] : 0.f;
            qbv[e] = (valid[e] && c_avg) ? (float)qb[j0 + e] : 0.f;
        }
        c_rowpart = CI->rowpart + (long long)strip * CI->m;
        c_rowpart2 = CI->rowpart2 + (long long)strip * CI->m;
        c_win = -1;
        flushed = false;
#pragma unroll
        for (int k = 0; k < TP; ++k) t[k] = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) { csa[e] = 0.f; csa2[e] = 0.f; }
        rows_in_batch = 0;
    };

    while (consumed < issued) {
        const int st = (int)(consumed % KS);
        // The oldest row's copies (wait_group counts the newer ones).
        const long long newer = issued - consumed - 1;
        if (newer >= 3) lagp::cp_wait<3>();
        else if (newer == 2) lagp::cp_wait<2>();
        else if (newer == 1) lagp::cp_wait<1>();
        else lagp::cp_wait<0>();
        __syncwarp();
        const RowRef ref = refs[st];
        if (ref.tile != c_tile) open_consumer(ref.tile);
        const long long i = ref.row;
        const long long di = i - c_i0;
        const unsigned char* stage = wbase + st * KSTAGE;
        float c[4], x[4], xb[4], xa[4];
        if (on) {
            if (sizeof(TC) == 4) {
                const float4 v = *reinterpret_cast<const float4*>(stage + lane * 16);
                c[0] = v.x; c[1] = v.y; c[2] = v.z; c[3] = v.w;
            } else {
                const uint2 v = *reinterpret_cast<const uint2*>(stage + lane * 8);
                c[0] = bf16_bits_to_f32(v.x & 0xffffu);
                c[1] = bf16_bits_to_f32(v.x >> 16);
                c[2] = bf16_bits_to_f32(v.y & 0xffffu);
                c[3] = bf16_bits_to_f32(v.y >> 16);
            }
            const float4 vx = *reinterpret_cast<const float4*>(stage + STRIP * 4 + lane * 16);
            x[0] = vx.x; x[1] = vx.y; x[2] = vx.z; x[3] = vx.w;
            if (c_avg) {
                const float4 vb = *reinterpret_cast<const float4*>(stage + 2 * STRIP * 4 + lane * 16);
                xb[0] = x[0] + vb.x; xb[1] = x[1] + vb.y; xb[2] = x[2] + vb.z; xb[3] = x[3] + vb.w;   // X + D
            } else {
                xb[0] = xb[1] = xb[2] = xb[3] = 0.f;
            }
            if (!init) {
                const float4 va = *reinterpret_cast<const float4*>(stage + 3 * STRIP * 4 + lane * 16);
                xa[0] = va.x; xa[1] = va.y; xa[2] = va.z; xa[3] = va.w;
            } else {
                xa[0] = xa[1] = xa[2] = xa[3] = 0.f;
            }
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) { c[e] = 0.f; x[e] = 0.f; xb[e] = 0.f; xa[e] = 0.f; }
        }
        // Row duals (current and average) staged per window of PWIN rows.
        const long long win = di / PWIN;
        if (win != c_win) {
            const long long r0 = c_i0 + win * PWIN;
            const long long r1 = min(r0 + (long long)PWIN, c_i1);
            __syncwarp();
            for (long long r = r0 + lane; r < r1; r += 32)
                pbuf[r - r0] = make_float2((float)c_p[r], c_avg ? (float)c_pb[r] : 0.f);
            __syncwarp();
            c_win = win;
        }
        const float2 pp = pbuf[di - win * PWIN];
        // The stage has been read: release it to the producer.
        __syncwarp();
        ++consumed;
        if (p_tile < T) issue();

        float rs = 0.f, rs2 = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (!valid[e]) continue;
            const float Rc = (c[e] - pp.x) - qv[e];
            t[0] += c[e] * x[e];
            t[1] += Rc < 0.f ? Rc * Rc : 0.f;                  // [p + q - C]^+ squared
            const float da = x[e] - xa[e];
            t[4] += da * da;
            if (init) t[2] += c[e] * c[e];                      // ||C||_F^2 (once per solve)
            if (c_avg) {
                const float Rb = (c[e] - pp.y) - qbv[e];
                t[2] += c[e] * xb[e];
                t[3] += Rb < 0.f ? Rb * Rb : 0.f;
                const float db = xb[e] - xa[e];
                t[5] += db * db;
            }
            const float sv = init ? x[e] : xb[e];
            rs += sv;
            csa[e] += sv;
            rs2 += x[e];
            csa2[e] += x[e];
        }
        if (init || c_avg) {
            rs = warp_sum(rs);
            if (lane == 0) c_rowpart[i] = lagp::widen(rs);
        }
        if (!init) {
            rs2 = warp_sum(rs2);
            if (lane == 0) c_rowpart2[i] = lagp::widen(rs2);
        }
        if (++rows_in_batch == KKT_FLUSH_ROWS) flush_acc();
    }
    pdl_release();
    flush_tile();
}

// ---------------------------------------------------------------------------
// Check: KKT of current and average, restart / termination / primal weight
// ---------------------------------------------------------------------------
struct KP {
    double rp2, rd2, cx, dual, gap, kkt, rel_p, rel_d, rel_gap, rel;
};

__device__ void kkt_parts(const Ctrl* S, double rp2, double rd2, double cx, double dual, KP& o) {
    // KKT error of Sec. 3.1 and the relative measures of reading C5.
    o.rp2 = rp2;
    o.rd2 = rd2;
    o.cx = cx;
    o.dual = dual;
    o.gap = cx - dual;
    const double gr = o.gap / S->R;
    o.kkt = sqrt(rp2 + rd2 + gr * gr);
    double dp = S->norm_b, dd = S->norm_C, dg = fabs(cx) + fabs(dual);
    if (S->rel_mode == 1) { dp += 1.0; dd += 1.0; dg += 1.0; }
    if (!(dp > 0.0)) dp = 1.0;
    if (!(dd > 0.0)) dd = 1.0;
    if (!(dg > 0.0)) dg = 1.0;
    o.rel_p = sqrt(rp2) / dp;
    o.rel_d = sqrt(rd2) / dd;
    o.rel_gap = fabs(o.gap) / dg;
    o.rel = fmax(o.rel_p, fmax(o.rel_d, o.rel_gap));
}

__device__ void report(Ctrl* S, const KP& k) {
    S->r_rp2 = k.rp2; S->r_rd2 = k.rd2; S->r_cx = k.cx; S->r_dual = k.dual; S->r_gap = k.gap;
    S->r_kkt = k.kkt; S->r_rel_p = k.rel_p; S->r_rel_d = k.rel_d; S->r_rel_gap = k.rel_gap; S->r_rel = k.rel;
}

// A: 0 rp2 cur, 1 rp2 avg, 2 dual cur, 3 dual avg, 4 ||dy_anchor||^2 cur, 5 avg,
//    6 <C,X>, 7 rd2 cur, 8 <C,Xbar>, 9 rd2 avg, 10 ||X - Xa||^2, 11 ||Xbar - Xa||^2.
// In MODE_INIT: 1 sum f, 3 sum g, 4 ||[f;g]||^2, 5 invalid marginal entries,
//    8 ||C||_F^2.
// Report the current iterate.
__device__ __forceinline__ void set_result(Ctrl* S) {
    S->res_slot = S->cur;
    S->res_xslot = S->xcur;
    S->res_avg = 0;
}

// pre: the measures of the current point and of the average, where the caller
// has formed them (kkt_parts of the same sums).
__device__ void finalize_check(Ctrl* S, const double* A, int mode, const KP* pre = nullptr) {
    if (S->lag && S->npend) {
        // The final pass before this check has applied the pending steps.
        S->h0 = (S->h0 + S->npend) % YRING;
        S->npend = 0;
        S->xcur = S->xdst;
        S->xdst = plan_dst(S->xcur, S->xbar, S->xanc);
    }
    if (mode == MODE_INIT) {
        // Data norms for the relative measures, and the marginal checks of the ABI.
        S->norm_b = sqrt(A[4]);
        S->norm_C = sqrt(A[8]);
        const double sf = A[1], sg = A[3];
        if (A[5] > 0.0 || !(fabs(sf - sg) <= 1e-9 * fmax(sf, 1.0))) {
            S->status = ST_ARG;
            set_result(S);
            return;
        }
    }
    KP c;
    if (pre) c = pre[0];
    else kkt_parts(S, A[0], A[7], A[6], A[2], c);
    S->checks += 1;
    if (mode == MODE_CHECK && S->stop_req) {
        // Stopped by the host (time limit): the current iterate, with the
        // measures this check has just computed for it.
        report(S, c);
        S->status = ST_TIMEOUT;
        set_result(S);
        return;
    }
    if (mode == MODE_INIT) {
        report(S, c);
        S->kkt0 = c.kkt;
        S->kkt_prev = c.kkt;
        if (!isfinite(c.kkt)) { S->status = ST_NUMERIC; set_result(S); }
        else if (c.rel <= S->tol) { S->status = ST_OK; set_result(S); }
        return;
    }
    if (S->k == 0) {
        // No accepted step since the last restart: only the pass budget is checked.
        if (S->passes >= S->max_passes) {
            report(S, c);
            S->status = ST_MAX_ITER;
            set_result(S);
        }
        return;
    }
    KP b;
    if (pre) b = pre[1];
    else kkt_parts(S, A[1], A[9], A[8], A[3], b);
    if (!isfinite(c.kkt) || !isfinite(b.kkt)) {
        report(S, c);
        S->status = ST_NUMERIC;
        set_result(S);
        return;
    }
    // Restart candidate (Sec. 5): current iff its KKT is strictly smaller.
    const bool use_avg = S->adaptive_restart ? !(c.kkt < b.kkt) : true;
    const KP& kk = use_avg ? b : c;
    const int cand = use_avg ? S->bar : S->cur;       // vector set
    const int candx = use_avg ? S->xbar : S->xcur;    // plan slot
    report(S, kk);
    if (kk.rel <= S->tol || S->passes >= S->max_passes) {
        S->status = kk.rel <= S->tol ? ST_OK : ST_MAX_ITER;
        S->res_slot = cand;
        S->res_xslot = candx;
        S->res_avg = use_avg ? 1 : 0;
        if (use_avg) {
            // The reported plan X + D is formed into a free slot, so
            // the current plan, D and the anchor stay as they are (a solve
            // stopped by its pass budget can be resumed from them).
            S->fix = 1;
            S->fix_x = S->xcur;
            S->fix_d = S->xbar;
            S->fix_dst = S->lag ? free_slot(S->xcur, S->xbar, S->xanc) : S->nxt;
            S->res_xslot = S->fix_dst;
        }
        return;
    }
    bool restart;
    if (S->adaptive_restart) {
        restart = (kk.kkt <= S->beta_suff * S->kkt0) ||
                  (kk.kkt <= S->beta_nec * S->kkt0 && kk.kkt > S->kkt_prev) ||
                  ((double)S->k >= S->beta_art * (double)S->total);
    } else {
        restart = b.kkt <= S->beta * S->kkt0;   // Eq. (6)
    }
    if (!restart) {
        S->kkt_prev = kk.kkt;
        return;
    }
    if (S->pw_update) {
        // PrimalWeightUpdate of Sec. 5 against the previous restart point.
        const double dX = sqrt(use_avg ? A[11] : A[10]);
        const double dy = sqrt(use_avg ? A[5] : A[4]);
        if (dX > S->eps_zero && dy > S->eps_zero)
            S->omega = exp(S->theta * log(dy / dX) + (1.0 - S->theta) * log(S->omega));
    }
    if (use_avg) {
        // Restart to the average: its slot becomes X + D in place before the
        // next pass (the vector set of that slot already holds the averaged
        // duals and the exact sums of X + D).
        S->fix = 1;
        S->fix_x = S->xcur;
        S->fix_d = candx;
        S->fix_dst = candx;
    }
    S->cur = cand;
    S->anc = cand;
    // The average restarts empty: its slot content is not read while k == 0.
    {
        int used = 1 << cand;
        int picks[3] = {0, 0, 0};
        int np = 0;
        for (int s = 0; s < NSLOT && np < 3; ++s)
            if (!(used & (1 << s))) picks[np++] = s;
        S->bar = picks[0];
        S->nxt = picks[1];
        S->barn = picks[2];
    }
    S->xcur = S->xanc = candx;
    S->xbar = S->lag ? free_slot(candx, candx, candx) : S->bar;
    S->xdst = plan_dst(S->xcur, S->xbar, S->xanc);
    S->k = 0;
    S->wavg = 1.0;
    S->kkt0 = kk.kkt;
    S->kkt_prev = kk.kkt;
    S->restarts += 1;
    S->tau = S->eta / S->omega;
    S->sigma = S->eta * S->omega;
}

// One vector tile of the check: the exact row / column sums (both partial
// sets: A the plan's at the initial check, the average's at a check; B the
// current plan's, which the passes carry forward by sums of changes between
// checks), the residual, dual-objective and distance terms, the plan tiles'
// partials, twelve scalars and the instance's ticket; the last tile runs the
// restart / termination logic.  Group g (warp g) adds partials g, g + VG, ...
// of each set, warp 0 combines the groups in order.  FP64 takes 64 cycles per
// warp instruction on each of an SM's four schedulers, so the sums over the
// plan tiles, the twelve reductions, the last tile's and the two points'
// measures are spread over the warps (all on one warp: 24 us at 4096 x 4096; here 18).
struct CheckShared {
    double grp[2 * VG * 32];
    double a[VP][32];
    double tot[VP];
    KP kp[2];
    int last;
};
__device__ void checkvec_tile(const Inst& I, Ctrl* S, int lvt, int mode, CheckShared& sh) {
    const long long m = I.m, n = I.n;
    const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const long long e = (long long)lvt * VE + lane;
    const bool init = mode == MODE_INIT;
    const bool avg = !init && S->k > 0;
    const bool row = e < m, col = !row && e < m + n;
    const long long idx = row ? e : e - m;          // i or j
    {
        const double* pa = row ? I.rowpart : I.colpart;
        const double* pb = row ? I.rowpart2 : I.colpart2;
        const long long stride = row ? m : I.ldx;
        const int count = row ? I.nstrips : I.nchunks;
        double a = 0.0, b = 0.0;
        if (row || col) {
#pragma unroll 4
            for (int k = grp; k < count; k += VG) {
                if (init || avg) a += pa[(long long)k * stride + idx];
                if (!init) b += pb[(long long)k * stride + idx];
            }
        }
        sh.grp[grp * 32 + lane] = a;
        sh.grp[(VG + grp) * 32 + lane] = b;
    }
    if (grp >= 1 && grp <= TP) {   // the plan tiles' scalars: one per warp
        const int k = grp - 1;
        const int t0 = (int)((long long)I.ntiles * lvt / I.nvt), t1 = (int)((long long)I.ntiles * (lvt + 1) / I.nvt);
        double a = 0.0;
        for (int t = t0 + lane; t < t1; t += 32) a += I.tpart[(long long)t * TP + k];
        sh.a[6 + k][lane] = a;
    }
    __syncthreads();
    if (grp == 0) {
        double s = 0.0, s2 = 0.0;
#pragma unroll
        for (int g2 = 0; g2 < VG; ++g2) {
            if (init || avg) s += sh.grp[g2 * 32 + lane];
            if (!init) s2 += sh.grp[(VG + g2) * 32 + lane];
        }
        double* Vc = slot_v(I, S->cur);
        double* Vb = slot_v(I, S->bar);
        const double* Va = slot_v(I, S->anc);
        double a[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        if (row || col) {
            const long long yo = row ? idx : m + idx;                   // offset of p_i / q_j in a vector set
            const long long so = row ? m + n + idx : 2 * m + n + idx;   // offset of r_i / c_j
            const double b = row ? I.f[idx] : I.g[idx];
            const double y = Vc[yo];
            if (init) {
                Vc[so] = s;
                a[0] = (s - b) * (s - b);
                a[2] = b * y;
                // marginal statistics: sum f, sum g, ||[f;g]||^2, invalid entries
                if (row) a[1] = b; else a[3] = b;
                a[4] = b * b;
                a[5] = (b >= 0.0 && isfinite(b)) ? 0.0 : 1.0;
                if (S->lag) {   // the first pass's duals as FP32 pairs
                    float2 v;
                    split_dual(y, v.x, v.y);
                    I.yf[(long long)S->h0 * I.yslot + e] = v;
                }
            } else {
                Vc[so] = s2;
                a[0] = (s2 - b) * (s2 - b);
                a[2] = b * y;
                const double ya = Va[yo];
                a[4] = (y - ya) * (y - ya);
                if (avg) {
                    Vb[so] = s;
                    const double yb = Vb[yo];
                    a[1] = (s - b) * (s - b);
                    a[3] = b * yb;
                    a[5] = (yb - ya) * (yb - ya);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) sh.a[k][lane] = a[k];
    }
    __syncthreads();
    for (int k = grp; k < VP; k += VG) {
        const double t = warp_sum(sh.a[k][lane]);
        if (lane == 0) I.vpart[(long long)lvt * VP + k] = t;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) sh.last = ticket_arrive(I.ticket) == (unsigned)(I.nvt - 1) ? 1 : 0;
    __syncthreads();
    if (sh.last) {
        for (int k = grp; k < VP; k += VG) {
            double t = 0.0;
            for (int v = lane; v < I.nvt; v += 32) t += __ldcg(I.vpart + (long long)v * VP + k);
            t = warp_sum(t);
            if (lane == 0) sh.tot[k] = t;
        }
        __syncthreads();
        if (!init) {
            if (threadIdx.x == 0) kkt_parts(S, sh.tot[0], sh.tot[7], sh.tot[6], sh.tot[2], sh.kp[0]);
            if (threadIdx.x == 32) kkt_parts(S, sh.tot[1], sh.tot[9], sh.tot[8], sh.tot[3], sh.kp[1]);
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            *I.ticket = 0u;
            finalize_check(S, sh.tot, mode, init ? nullptr : sh.kp);
        }
    }
}

__global__ void __launch_bounds__(VT) k_checkvec(const Inst* __restrict__ insts, const TileRef* __restrict__ vmap,
                                                 const int* __restrict__ NVp, unsigned* wctr, int mode) {
    // One CTA per vector tile (no work queue): the grid covers the tile count.
    __shared__ CheckShared sh;
    pdl_enter();
    // No work counter of its own, but it still resets the others for the
    // kernels that follow (block 0, before any early exit).
    reset_other_counters(wctr, wc_index(WC_CHECK, 0));
    const int NV = *NVp;
    if ((int)blockIdx.x >= NV) return;
    const TileRef tr = vmap[blockIdx.x];
    const Inst& I = insts[tr.inst];
    Ctrl* S = I.ctrl;
    if (S->status != ST_RUNNING) return;
    checkvec_tile(I, S, tr.local, mode, sh);
}

// ---------------------------------------------------------------------------
// After every check: where the check picked the running average (a restart to
// it, or the reported point), write X[fix_dst] = X[fix_x] + X[fix_d] -- the
// current plan plus the stored deviation, with the rounding the checks used
// for the same value -- and, for deferred plan writes, split the current
// duals for the next pass (a restart may have changed them).  One warp per
// plan tile; the tiles of the first strip and chunk cover the duals.
// ---------------------------------------------------------------------------
template <typename TX>
__global__ void __launch_bounds__(TWARPS * 32)
k_avgfix(const Inst* __restrict__ insts, const TileRef* __restrict__ tmap, const int* __restrict__ Tp) {
    pdl_enter();
    const int T = *Tp;
    const int lane = threadIdx.x & 31;
    const int nw = (int)gridDim.x * TWARPS;
    for (int t = (int)blockIdx.x * TWARPS + (int)(threadIdx.x >> 5); t < T; t += nw) {
        const TileRef tr = tmap[t];
        const Inst& I = insts[tr.inst];
        Ctrl& S = *I.ctrl;
        const int strip = tr.local % I.nstrips, chunk = tr.local / I.nstrips;
        const long long j0 = (long long)strip * STRIP + lane * 4;
        const long long i0 = (long long)chunk * I.tile_rows;
        const long long i1 = min(i0 + (long long)I.tile_rows, I.m);
        if (S.lag) {
            if (S.status == ST_NUMERIC && S.npend > 0) {
                // A step with a non-finite value ended the solve: the final
                // pass has applied the steps before it.
                if (tr.local == 0 && lane == 0) {
                    S.xcur = S.xdst;
                    S.npend = 0;
                }
                continue;
            }
            if (S.status == ST_RUNNING) {
                float2* yf = I.yf + (long long)S.h0 * I.yslot;
                const double* y = slot_v(I, S.cur);
                if (strip == 0)
                    for (long long i = i0 + lane; i < i1; i += 32) split_dual(y[i], yf[i].x, yf[i].y);
                if (chunk == 0)
                    for (int e = 0; e < 4; ++e)
                        if (j0 + e < I.n) split_dual(y[I.m + j0 + e], yf[I.m + j0 + e].x, yf[I.m + j0 + e].y);
            }
        }
        if (!S.fix || j0 >= I.n) continue;
        const TX* Xa = slot_x<TX>(I, S.fix_x);
        const TX* Xd = slot_x<TX>(I, S.fix_d);
        TX* Xo = slot_x<TX>(I, S.fix_dst);
        for (long long i = i0; i < i1; ++i) {
            TX a[4], d[4];
            ld4(Xa + i * I.ldx + j0, a);
            ld4(Xd + i * I.ldx + j0, d);
#pragma unroll
            for (int e = 0; e < 4; ++e) a[e] = a[e] + d[e];
            st4(Xo + i * I.ldx + j0, a);
        }
    }
}

// out = a + d over `count` elements (a multiple of 4): a plan formed from
// the current plan and the average's deviation, for the host's copies.
template <typename TX>
__global__ void k_combine(const TX* __restrict__ a, const TX* __restrict__ d, TX* out, long long count) {
    const long long stride = (long long)gridDim.x * blockDim.x * 4;
    for (long long e = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * 4; e < count; e += stride) {
        TX x[4], y[4];
        ld4(a + e, x);
        ld4(d + e, y);
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = x[k] + y[k];
        st4(out + e, x);
    }
}

// Snapshot of every live instance's controller (one D2H copy per chunk).
__global__ void k_snapshot(const Inst* __restrict__ insts, const int* __restrict__ count, Ctrl* out) {
    pdl_enter();
    const int n = *count;
    const int words = (int)(sizeof(Ctrl) / sizeof(int));
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n * words; t += gridDim.x * blockDim.x) {
        const int i = t / words, w = t % words;
        reinterpret_cast<int*>(out + i)[w] = reinterpret_cast<const int*>(insts[i].ctrl)[w];
    }
}

}  // namespace pdot

#include "pdot_resident.cuh"
#include "pdot_persist.cuh"


namespace pdot {

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static int err(cudaError_t e) { return e == cudaSuccess ? 0 : (int)e; }

// Launch with the programmatic-stream-serialization attribute when enabled.
template <typename... KArgs, typename... Args>
static int launch_k(bool pdl, void (*kern)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                    Args... args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute attr[1];
    if (pdl) {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        c.attrs = attr;
        c.numAttrs = 1;
    }
    return err(cudaLaunchKernelEx(&c, kern, args...));
}

// The pass kernel of FP32 plans with deferred writes; FINAL: apply and write
// the pending steps only.  Generated costs take the variant with room for
// their coordinates.
template <bool CP, bool FINAL>
static int launch_lag(int ttype, const Inst* d_insts, const TileRef* d_tmap, const int* T, unsigned* wctr, int wc,
                      int dir_xor, const LaunchCfg& cfg, cudaStream_t st) {
    const bool pdl = cfg.pdl != 0;
    const unsigned nb = (unsigned)cfg.lag_blocks, th = TWARPS * 32;
    const int ro = cfg.pass_form == 1 ? 1 : 0;
    constexpr int sm = lagp::smem_bytes();
    if (ttype == TT_BF16)
        return launch_k(pdl, k_pass_lag<unsigned short, CP, FINAL>, nb, th, sm, st, d_insts, d_tmap, T, wctr, wc, dir_xor, ro);
    if (ttype == TT_F32)
        return launch_k(pdl, k_pass_lag<float, CP, FINAL>, nb, th, sm, st, d_insts, d_tmap, T, wctr, wc, dir_xor, ro);
    if (cfg.gen_dims <= 2)
        return launch_k(pdl, k_pass_lag<GenC<2>, CP, FINAL>, nb, th, sm, st, d_insts, d_tmap, T, wctr, wc, dir_xor, ro);
    if (cfg.gen_dims <= 4)
        return launch_k(pdl, k_pass_lag<GenC4, CP, FINAL>, nb, th, sm, st, d_insts, d_tmap, T, wctr, wc, dir_xor, ro);
    return launch_k(pdl, k_pass_lag<GenC8, CP, FINAL>, nb, th, sm, st, d_insts, d_tmap, T, wctr, wc, dir_xor, ro);
}

template <bool CP>
static int launch_pass_t(int ttype, const Inst* d_insts, const TileRef* d_tmap, const int* T, unsigned* wctr,
                         const LaunchCfg& cfg, void* stream, int wc_override, int dir_xor) {
    const cudaStream_t st = (cudaStream_t)stream;
    const int wc = wc_override >= 0 ? wc_override : wc_index(WC_PASS, ttype);
    const bool pdl = cfg.pdl != 0;
    const unsigned tb = (unsigned)cfg.tile_blocks, th = TWARPS * 32;
    if (ttype == TT_F64)
        return launch_k(pdl, k_pass<double, double, 2, CP>, (unsigned)cfg.tile_blocks_f64, th, 0, st, d_insts, d_tmap, T,
                        wctr, wc, dir_xor);
    if (cfg.pass_form)
        return launch_lag<CP, false>(ttype, d_insts, d_tmap, T, wctr, wc, dir_xor, cfg, st);
    if (ttype == TT_GEN)
        return launch_k(pdl, k_pass<GenC8, float, 2, CP>, tb, th, 0, st, d_insts, d_tmap, T, wctr, wc, dir_xor);
    if (ttype == TT_BF16) {
        if (cfg.pass_u == 4)
            return launch_k(pdl, k_pass<unsigned short, float, 4, CP>, tb, th, 0, st, d_insts, d_tmap, T, wctr, wc, dir_xor);
        return launch_k(pdl, k_pass<unsigned short, float, 2, CP>, tb, th, 0, st, d_insts, d_tmap, T, wctr, wc, dir_xor);
    }
    if (cfg.pass_u == 4) return launch_k(pdl, k_pass<float, float, 4, CP>, tb, th, 0, st, d_insts, d_tmap, T, wctr, wc, dir_xor);
    return launch_k(pdl, k_pass<float, float, 2, CP>, tb, th, 0, st, d_insts, d_tmap, T, wctr, wc, dir_xor);
}
int launch_pass(int ttype, const Inst* d_insts, const TileRef* d_tmap, const int* T, unsigned* wctr,
                const LaunchCfg& cfg, void* stream, int wc_override, int dir_xor) {
    if (cfg.comp) return launch_pass_t<true>(ttype, d_insts, d_tmap, T, wctr, cfg, stream, wc_override, dir_xor);
    return launch_pass_t<false>(ttype, d_insts, d_tmap, T, wctr, cfg, stream, wc_override, dir_xor);
}
int launch_plan_final(int ttype, const Inst* d_insts, const TileRef* d_tmap, const int* T, unsigned* wctr,
                      const LaunchCfg& cfg, void* stream) {
    const int wc = wc_index(WC_AUX, ttype);
    const cudaStream_t st = (cudaStream_t)stream;
    if (cfg.comp) return launch_lag<true, true>(ttype, d_insts, d_tmap, T, wctr, wc, 0, cfg, st);
    return launch_lag<false, true>(ttype, d_insts, d_tmap, T, wctr, wc, 0, cfg, st);
}

int launch_dual(const Inst* d_insts, const TileRef* d_vmap, const int* NV, int nv_hint, unsigned* wctr,
                const LaunchCfg& cfg, void* stream, bool direct) {
    // nv_hint: an upper bound of the vector-tile count (one CTA each); with
    // direct, exactly the count of the single instance's vector tiles.
    int blocks = nv_hint;
    if (blocks < 1) blocks = 1;
    return launch_k(cfg.pdl != 0, k_dual, (unsigned)blocks, VT, 0, (cudaStream_t)stream, d_insts, d_vmap, NV, wctr,
                    direct ? 1 : 0);
}
int launch_kkt(int ttype, const Inst* d_insts, const TileRef* d_tmap, const int* T, unsigned* wctr, int mode,
               const LaunchCfg& cfg, void* stream) {
    const cudaStream_t st = (cudaStream_t)stream;
    const int wc = wc_index(WC_KKT, ttype);
    const bool pdl = cfg.pdl != 0;
    const unsigned th = TWARPS * 32;
    if (ttype == TT_F64)
        return launch_k(pdl, k_kkt<double, double>, (unsigned)cfg.tile_blocks_f64, th, 0, st, d_insts, d_tmap, T, wctr,
                        wc, mode);
    if (ttype == TT_GEN)
        return launch_k(pdl, k_kkt<GenC8, float>, (unsigned)cfg.tile_blocks, th, 0, st, d_insts, d_tmap, T, wctr, wc,
                        mode);
    if (cfg.kkt_blocks > 0) {   // stored FP32 / BF16 costs
        if (ttype == TT_BF16)
            return launch_k(pdl, k_kkt_staged<unsigned short>, (unsigned)cfg.kkt_blocks, th, kkt_smem(), st, d_insts,
                            d_tmap, T, wctr, wc, mode);
        return launch_k(pdl, k_kkt_staged<float>, (unsigned)cfg.kkt_blocks, th, kkt_smem(), st, d_insts, d_tmap, T, wctr,
                        wc, mode);
    }
    if (ttype == TT_BF16)
        return launch_k(pdl, k_kkt<unsigned short, float>, (unsigned)cfg.tile_blocks, th, 0, st, d_insts, d_tmap, T,
                        wctr, wc, mode);
    return launch_k(pdl, k_kkt<float, float>, (unsigned)cfg.tile_blocks, th, 0, st, d_insts, d_tmap, T, wctr, wc,
                    mode);
}
int launch_checkvec(const Inst* d_insts, const TileRef* d_vmap, const int* NV, int nv_hint, unsigned* wctr, int mode,
                    const LaunchCfg& cfg, void* stream) {
    int blocks = nv_hint;
    if (blocks < 1) blocks = 1;
    return launch_k(cfg.pdl != 0, k_checkvec, (unsigned)blocks, VT, 0, (cudaStream_t)stream, d_insts, d_vmap, NV,
                    wctr, mode);
}
int launch_avgfix(int ttype, const Inst* d_insts, const TileRef* d_tmap, const int* T, const LaunchCfg& cfg,
                  void* stream) {
    const cudaStream_t st = (cudaStream_t)stream;
    if (ttype == TT_F64)
        return launch_k(cfg.pdl != 0, k_avgfix<double>, (unsigned)cfg.tile_blocks_f64, TWARPS * 32, 0, st, d_insts,
                        d_tmap, T);
    return launch_k(cfg.pdl != 0, k_avgfix<float>, (unsigned)cfg.tile_blocks, TWARPS * 32, 0, st, d_insts, d_tmap, T);
}
int launch_combine(int xtype, const void* a, const void* d, void* out, long long count, void* stream) {
    if (count <= 0) return 0;
    long long blocks = (count / 4 + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (xtype == 2)
        k_combine<double><<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(
            static_cast<const double*>(a), static_cast<const double*>(d), static_cast<double*>(out), count);
    else
        k_combine<float><<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(
            static_cast<const float*>(a), static_cast<const float*>(d), static_cast<float*>(out), count);
    return err(cudaGetLastError());
}
int launch_watchdog_selftest(int polls, int* d_status, unsigned* d_count, void* stream) {
    k_watchdog_selftest<<<4, 64, 0, (cudaStream_t)stream>>>(d_count, polls, d_status);
    return err(cudaGetLastError());
}

int launch_snapshot(const Inst* d_insts, const int* count, int max_count, Ctrl* out, void* stream) {
    const int words = (int)(sizeof(Ctrl) / sizeof(int));
    int blocks = (max_count * words + 255) / 256;
    if (blocks < 1) blocks = 1;
    if (blocks > 1024) blocks = 1024;
    k_snapshot<<<blocks, 256, 0, (cudaStream_t)stream>>>(d_insts, count, out);
    return err(cudaGetLastError());
}

static int occ(const void* fn, int threads) {
    int a = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, fn, threads, 0);
    return a > 0 ? a : 1;
}
int occupancy_tile_blocks_per_sm(int ttype) {
    if (ttype == TT_F64) {
        const int a = occ((const void*)k_pass<double, double, 2, true>, TWARPS * 32);
        const int b = occ((const void*)k_kkt<double, double>, TWARPS * 32);
        return a < b ? a : b;
    }
    const void* fns[] = {(const void*)k_pass<float, float, 2, true>,          (const void*)k_pass<float, float, 2, false>,
                         (const void*)k_pass<unsigned short, float, 4, true>,  (const void*)k_pass<unsigned short, float, 4, false>,
                         (const void*)k_pass<GenC8, float, 2, true>,           (const void*)k_pass<GenC8, float, 2, false>,
                         (const void*)k_kkt<float, float>,                     (const void*)k_kkt<unsigned short, float>,
                         (const void*)k_kkt<GenC8, float>};
    int r = 1 << 20;
    for (const void* f : fns) {
        const int a = occ(f, TWARPS * 32);
        if (a < r) r = a;
    }
    return r;
}

// Opt every instantiation of a kernel with dynamic shared memory into `bytes`;
// returns minus the fewest CTAs per SM any of them holds, or a positive
// cudaError_t code.
static int setup_dyn(const void* const* fns, int nf, int bytes) {
    int r = 1 << 20;
    for (int i = 0; i < nf; ++i) {
        const cudaError_t e = cudaFuncSetAttribute(fns[i], cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return (int)e;
        int a = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, fns[i], TWARPS * 32, bytes);
        if (a < r) r = a;
    }
    return -(r > 0 ? r : 1);
}

// Resident kernel: its shared-memory size, and how many of its clusters the
// device holds at once (-count; 0: cannot run, a positive value: an error).
int setup_resident() {
    const void* fns[] = {(const void*)k_resident<float, false>, (const void*)k_resident<float, true>,
                         (const void*)k_resident<unsigned short, false>, (const void*)k_resident<unsigned short, true>};
    int r = 1 << 20;
    for (const void* fn : fns) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, res::RSMEM);
        if (e != cudaSuccess) return (int)e;
        cudaLaunchConfig_t c = {};
        c.gridDim = dim3(res::RCS);
        c.blockDim = dim3(res::RT);
        c.dynamicSmemBytes = res::RSMEM;
        int nc = 0;
        e = cudaOccupancyMaxActiveClusters(&nc, fn, &c);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        if (nc < r) r = nc;
    }
    return -r;
}
bool resident_fits(long long m, long long n) { return res::fits(m, n); }
int launch_resident(int ttype, const Inst* d_insts, const int* list, const int* count, int max_count, int passes,
                    int K, int replay, const LaunchCfg& cfg, void* stream) {
    if (max_count < 1) return 0;
    const cudaStream_t st = (cudaStream_t)stream;
    const dim3 grid((unsigned)(res::RCS * max_count)), block(res::RT);
    if (ttype == TT_BF16) {
        if (cfg.comp)
            k_resident<unsigned short, true><<<grid, block, res::RSMEM, st>>>(d_insts, list, count, passes, K, replay);
        else
            k_resident<unsigned short, false><<<grid, block, res::RSMEM, st>>>(d_insts, list, count, passes, K, replay);
    } else if (ttype == TT_F32) {
        if (cfg.comp)
            k_resident<float, true><<<grid, block, res::RSMEM, st>>>(d_insts, list, count, passes, K, replay);
        else
            k_resident<float, false><<<grid, block, res::RSMEM, st>>>(d_insts, list, count, passes, K, replay);
    } else {
        return (int)cudaErrorInvalidValue;   // FP32 plans with stored FP32 / BF16 costs only
    }
    return err(cudaGetLastError());
}

int setup_kkt_staged() {
    const void* fns[] = {(const void*)k_kkt_staged<float>, (const void*)k_kkt_staged<unsigned short>};
    return setup_dyn(fns, 2, kkt_smem());
}

template <typename TC>
static int setup_lag() {
    const void* fns[] = {(const void*)k_pass_lag<TC, true, false>, (const void*)k_pass_lag<TC, false, false>,
                         (const void*)k_pass_lag<TC, true, true>, (const void*)k_pass_lag<TC, false, true>};
    return setup_dyn(fns, 4, lagp::smem_bytes());
}
int setup_lag_pass() {
    const int r[] = {setup_lag<float>(), setup_lag<unsigned short>(), setup_lag<GenC<2>>(), setup_lag<GenC4>(),
                     setup_lag<GenC8>()};
    int worst = r[0];
    for (int v : r) worst = v > worst ? v : worst;   // an error, or the fewest blocks per SM (negative)
    return worst;
}

template <typename TC>
static int setup_pers() {
    const void* plain[] = {(const void*)k_persist<TC, false>};
    const void* comp[] = {(const void*)k_persist<TC, true>};
    const int a = setup_dyn(plain, 1, pers::Lay<false>::CTA), b = setup_dyn(comp, 1, pers::Lay<true>::CTA);
    return a > b ? a : b;
}
int setup_persist() {
    const int r[] = {setup_pers<float>(), setup_pers<unsigned short>(), setup_pers<GenC<2>>(), setup_pers<GenC4>()};
    int worst = r[0];
    for (int v : r) worst = v > worst ? v : worst;
    return worst;
}
int persist_rows(bool comp) { return (comp ? pers::Lay<true>::NS : pers::Lay<false>::NS) * pers::R; }
template <typename TC>
static int launch_pers(const Inst* d_insts, const CtaRef* refs, int ctas, GridSync* gs, int epoch, int npass, const LaunchCfg& cfg,
                       cudaStream_t st) {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)ctas);
    c.blockDim = dim3(TWARPS * 32);
    c.dynamicSmemBytes = cfg.comp ? pers::Lay<true>::CTA : pers::Lay<false>::CTA;
    c.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    c.attrs = attr;
    c.numAttrs = 1;
    const int ro = cfg.pass_form == 1 ? 1 : 0;
    return err(cfg.comp ? cudaLaunchKernelEx(&c, k_persist<TC, true>, d_insts, refs, gs, epoch, npass, ro, cfg.barrier_polls)
                        : cudaLaunchKernelEx(&c, k_persist<TC, false>, d_insts, refs, gs, epoch, npass, ro, cfg.barrier_polls));
}
int launch_persist(int ttype, const Inst* d_insts, const CtaRef* refs, int ctas, bool on_chip, GridSync* gs, int epoch,
                   int npass, const LaunchCfg& cfg, void* stream) {
    const cudaStream_t st = (cudaStream_t)stream;
    if (ttype == TT_BF16) return launch_pers<unsigned short>(d_insts, refs, ctas, gs, epoch, npass, cfg, st);
    // A generated cost whose tiles stay on the chip is computed once and then
    // served as a stored one.
    if (ttype == TT_F32 || on_chip) return launch_pers<float>(d_insts, refs, ctas, gs, epoch, npass, cfg, st);
    if (cfg.gen_dims <= 2) return launch_pers<GenC<2>>(d_insts, refs, ctas, gs, epoch, npass, cfg, st);
    return launch_pers<GenC4>(d_insts, refs, ctas, gs, epoch, npass, cfg, st);
}

int occupancy_vec_blocks_per_sm() {
    const int a = occ((const void*)k_dual, VT);
    const int b = occ((const void*)k_checkvec, VT);
    return a < b ? a : b;
}

}  // namespace pdot
